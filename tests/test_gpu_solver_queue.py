"""The mixed solver's work queue: a block of items per thread block, taken one by one by its warps.  Every
class, list length (shorter than one block, no multiple of one, many blocks), warp count and block
length gives the sweep of the per-class schedule bit for bit (a space's arithmetic does not depend on
the warp that takes it or on the elements a warp keeps from its previous space)."""
import numpy as np
import pytest

from paper_2606_04186_gb300 import synth

from gpu_util import library

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_class,warps,chunk", [(1, 15, 1), (7, 15, 3), (44, 1, 1), (60, 12, 16), (1000, 2, 5),
                                                   (1000, 15, 4)])
def test_queue_gives_the_per_class_sweep(per_class, warps, chunk):
    qf = library()
    n, no = 15, 4
    eps, h, g = synth.make_system(n, no, 0.05, 3)
    sp = synth.mixed_spaces(n, no, per_class, 9) if per_class <= 60 else synth.all_spaces(n, no, 3, 3)[:per_class]
    t1, t2 = synth.random_amplitudes(no, n - no, 2, 0.01, 0.02)
    runs = []
    for kw in (dict(schedule="per_class", warps=warps), dict(schedule="persistent", warps=warps, chunk=chunk)):
        f = qf.Flow(h, g, no, sp, precision="mixed", graph=False, **kw)
        f.set_amplitudes(t1, t2)
        f.sweep(raise_on_fail=False)
        runs.append((f.energy(per_space=True)[1], *f.amplitudes()))
        f.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b, equal_nan=True)
