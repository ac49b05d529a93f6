"""FP64 dressings under a diagonal similarity transform of the orbitals: creators times d_p, annihilators by
1 / d_p, amplitudes t_i^a d_a / d_i.  The dressed integrals transform like the bare ones, so with powers of two
every element of the result, scaled back, is the untransformed one: rows of the products' operands then
differ in their scale exponents by up to 2^40, and integrals and amplitudes oppose each other along the
sums, down to elements that an absolute bound on the largest integral would not see.

Tolerance: the transform is exact, so it is the one of the untransformed dressing, 1e-12 of the largest integral
(test_gpu_fixed_dress.py); halved exponents cost up to two bits a digit of a summed pair.
"""
import numpy as np
import pytest

from oracle import hbar
from paper_2606_04186_gb300 import synth

from gpu_util import library
from test_gpu_fixed_dress import _dress

pytestmark = pytest.mark.gpu


def _transform(h, g, t1, t2, no, x):
    """Exponents x: everything times 2^(creators - annihilators)."""
    up, dn = np.exp2(x), np.exp2(-x)
    o, v = slice(0, no), slice(no, None)
    h = h * up[:, None] * dn[None, :]
    g = g * np.einsum("p,q,r,s->pqrs", up, dn, up, dn)
    t1 = t1 * dn[o, None] * up[None, v]
    t2 = t2 * np.einsum("i,j,a,b->ijab", dn[o], dn[o], up[v], up[v])
    return h, g, t1, t2


# sizes on the integer pipe and on the tensor cores (the last three), one above the T1 passes' 16 occupied orbitals
@pytest.mark.parametrize("n,no", [(4, 1), (19, 5), (24, 3), (22, 17), (26, 13), (44, 6), (47, 5)])
@pytest.mark.parametrize("which", ["virtual", "occupied", "all", "one"])
def test_scaled_orbitals(n, no, which):
    qf = library()
    _, h, g = synth.make_system(n, no, 4.0, 70 + n)
    t1, t2 = synth.random_amplitudes(no, n - no, n, 0.05, 0.1)
    rng = np.random.default_rng(n)
    x = -np.round(20.0 * rng.permutation(n) / (n - 1))
    if which == "virtual":
        x[:no] = 0.0
    elif which == "occupied":
        x[no:] = 0.0
    elif which == "one":
        x[:] = 0.0
        x[n - 1] = -18.0
    ref = hbar.hbar2(h, g, t1, t2, no)
    e0, F, W = _dress(qf, *_transform(h, g, t1, t2, no, x), no)
    up, dn = np.exp2(x), np.exp2(-x)
    F = F * dn[:, None] * up[None, :]
    W = W * np.einsum("p,q,r,s->pqrs", dn, up, dn, up)
    scale = max(1.0, np.abs(ref[2]).max())
    for y, r in zip((e0, F, W), ref):
        assert np.abs(np.asarray(y) - r).max() < 1e-12 * scale
