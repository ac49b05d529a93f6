"""Spaces that the FP64 solver's fixed-point kernel hands to the general kernel, among spaces it keeps:
long lists of 6e6o spaces (two warps a block, several items per block), some of whose blocks lack pair
symmetry or hold a non-finite integral, in an order that makes every block meet both kinds.

Tolerance: as in test_gpu_fixed_solver.py (both kernels round like FP64 on O(1) quantities); spaces both
runs give to the general kernel are equal bit for bit.
"""
import numpy as np
import pytest

from paper_2606_04186_gb300 import synth

from gpu_util import dev
from test_gpu_fixed_solver import _solve, _system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["bent", "non_finite", "both"])
def test_deferred_spaces_among_others(kind):
    import torch
    n, no, k = 24, 5, 3
    qf, h, g, t1, t2, e0, F, W = _system(n, no, 4.0, 41, 0.02)
    sp = synth.all_spaces(n, no)
    sp = sp[np.random.default_rng(2).permutation(len(sp))]
    perm, o1, o2, _ = qf.plan(h, g, no, sp)
    sp, own = sp[perm], (dev(o1), dev(o2))
    w = W.clone()
    if kind != "non_finite":  # spaces with occupied 1 and virtual 9
        w[1, 9, 2:, 3:] += 1e-3 * torch.rand_like(w[1, 9, 2:, 3:])
    if kind != "bent":        # spaces with virtuals 12 and 15
        w[12, 15, 12, 15] = w[15, 12, 15, 12] = float("inf")
    has = lambda *orb: np.all([(sp[:, 2:] == o).any(axis=1) for o in orb], axis=0)  # noqa: E731
    off = np.zeros(len(sp), dtype=bool)
    if kind != "non_finite":
        off |= has(1, 9)
    if kind != "bent":
        off |= has(12, 15)
    assert 0.01 < off.mean() < 0.5
    a = _solve(qf, n, no, e0, F, w, k, dev(sp), t1, t2, own, False)
    b = _solve(qf, n, no, e0, F, w, k, dev(sp), t1, t2, own, True)
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    assert (a[1][~off] == 0).all()
    assert np.array_equal(a[0][off], b[0][off], equal_nan=True)
    assert np.abs(a[0][~off] - b[0][~off]).max() < 1e-12
    for x, y in zip(a[3:], b[3:]):
        ok = np.isfinite(y)
        assert np.array_equal(np.isnan(x), np.isnan(y)) and np.abs(x[ok] - y[ok]).max() < 1e-12
    # the kept spaces' energies do not depend on the others
    c = _solve(qf, n, no, e0, F, W, k, dev(sp), t1, t2, own, False)
    assert np.array_equal(a[0][~off], c[0][~off])
