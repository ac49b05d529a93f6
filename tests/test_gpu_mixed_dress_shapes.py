"""The mixed dressing's launch forms at the sizes where they change: vvvv tiles of 32 and 64 (one and two
tiles a side), groups of four virtuals with a remainder, vvvo products within the other blocks' launch and
in their own, T1 passes with 64 and 256 threads a block and with a remainder of eight rows.

Tolerance: an element of the T1-dressed integrals carries FP32 sums of at most n terms |t1| |W| <= 0.04,
n 0.04 2^-24 < 2e-7 at n = 70, the T2 terms FP32 products below that; f and E0 add 3 o of them with
random signs: 1e-6 for all."""
import numpy as np
import pytest

from oracle import hbar
from paper_2606_04186_gb300 import synth

from gpu_util import library, vvvv_four_distinct

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,no", [(6, 2), (9, 3), (34, 2), (35, 2), (36, 3), (50, 16), (56, 5), (70, 4)])
def test_mixed_dressing_at_launch_sizes(n, no):
    qf = library()
    eps, h, g = synth.make_system(n, no, 0.05, 7)
    t1, t2 = synth.random_amplitudes(no, n - no, 3, 0.01, 0.01)
    k = min(no, n - no, 2)
    f = qf.Flow(h, g, no, synth.all_spaces(n, no, k, k)[:20], precision="mixed")
    f.set_amplitudes(t1, t2)
    e0, F, W = f.dressed()
    f.close()
    e0r, Fr, Wr = hbar.hbar2(h, g, t1, t2, no)
    assert abs(e0 - e0r) < 1e-6
    assert np.abs(F - Fr).max() < 1e-6
    v = slice(no, n)  # vvvv elements with four distinct virtuals are not dressed: left out
    diff = W - Wr
    diff[v, v, v, v][vvvv_four_distinct(n - no)] = 0.0
    assert np.abs(diff).max() < 1e-6
