"""The FP64 solver's FP32-seeded helpers and what keeps their arguments in range: a space whose integrals are
2^30 and more goes to the general kernel, so both forms of the call give the same bits there, and large scales
below that limit agree to rounding.  So do spaces whose couplings' rounding comes near the tolerance and spaces with
pair asymmetry above rounding (64 units of 2^-54 of the largest coupling).

Tolerances: recip and rsqrt_nr as derived beside them in csrc/fixed.cuh (2^-44 and 2^-52; the references
are themselves within 2^-52); scaled solves as in test_gpu_fixed_solver.py, times the scale.
"""
import os
import subprocess

import numpy as np
import pytest

from paper_2606_04186_gb300 import build, synth

from gpu_util import dev
from test_gpu_fixed_solver import _solve, _system

pytestmark = pytest.mark.gpu


def test_seeded_reciprocal_and_root(tmp_path):
    exe = str(tmp_path / "seed_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", "seed_check.cu")
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, src, "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert float(out[0]) < 2.0 ** -44 + 2.0 ** -52 and float(out[1]) < 2.0 ** -52 + 2.0 ** -52


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("bits", [20, 36, 140, 700])
def test_solver_at_large_scales(k, bits):
    """Integrals times 2^bits with the tolerance scaled along."""
    n, no = 13, 4
    qf, h, g, t1, t2, e0, F, W = _system(n, no, 5.0, 5, 0.02)
    sp = synth.sampled_spaces(n, no, 36, 4, no=k, nv=k)
    perm, o1, o2, _ = qf.plan(h, g, no, sp)
    sp, own = dev(sp[perm]), (dev(o1), dev(o2))
    s = 2.0 ** bits
    kw = {"tol": 1e-9 * s}
    a = _solve(qf, n, no, e0 * s, F * s, W * s, k, sp, t1, t2, own, False, **kw)
    b = _solve(qf, n, no, e0 * s, F * s, W * s, k, sp, t1, t2, own, True, **kw)
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    if bits > 32:  # the largest integrals (about 0.2) are above 2^30: the general kernel both times
        for x, y in zip((a[0], a[3], a[4]), (b[0], b[3], b[4])):
            assert np.array_equal(x, y, equal_nan=True)
    else:
        assert (a[1] == 0).all()
        for x, y, u in ((a[0], b[0], s), (a[3], b[3], 1.0), (a[4], b[4], 1.0)):
            assert np.abs(x - y).max() < 1e-12 * u


def _system13(seed, k):
    n, no = 13, 4
    qf, h, g, t1, t2, e0, F, W = _system(n, no, 5.0, seed, 0.02)
    sp = synth.sampled_spaces(n, no, 36, 4, no=k, nv=k)
    perm, o1, o2, _ = qf.plan(h, g, no, sp)
    return qf, n, no, t1, t2, e0, F, W, sp[perm], (dev(o1), dev(o2))


@pytest.mark.parametrize("k", [1, 2, 3])
def test_pair_asymmetry_above_rounding(k):
    """One element of each pair, (pp|rr) among them, times 1 + 2^-45: spaces where that is more than 64 units of
    the largest coupling (which an element paired with itself or the F block may hold) are the general kernel's."""
    import torch
    qf, n, no, t1, t2, e0, F, W, sp, own = _system13(5, k)
    pq = torch.arange(n * n, device="cuda").reshape(n, n)
    upper = pq[:, :, None, None] < pq[None, None, :, :]
    w = W * (1.0 + 2.0 ** -45 * upper.to(torch.float64))
    a = _solve(qf, n, no, e0, F, w, k, dev(sp), t1, t2, own, False)
    b = _solve(qf, n, no, e0, F, w, k, dev(sp), t1, t2, own, True)
    f, w = F.cpu().numpy(), w.cpu().numpy()
    units = []
    for s in sp:
        o, m = s[2:2 + 2 * k], 2 * k
        block = w[np.ix_(o, o, o, o)].reshape(m * m, m * m)
        dd = np.zeros(m * m, dtype=bool)
        dd[:: m + 1] = True
        c = np.where(dd[:, None] & dd[None, :], 0.0, block)
        one = f[np.ix_(o, o)] * (1 - np.eye(m))
        sx = np.frexp(max(np.abs(c).max(), np.abs(one).max()))[1]
        units.append(np.abs(c - c.T).max() / 2.0 ** (sx - 54))
    over = np.array(units) > 65.0
    assert over.any() and (a[1] == 0).all() and np.array_equal(a[1], b[1])
    assert np.array_equal(a[0][over], b[0][over]) and np.array_equal(a[2][over], b[2][over])
    for x, y in zip((a[0], a[3], a[4]), (b[0], b[3], b[4])):
        assert np.abs(x - y).max() < 1e-12


@pytest.mark.parametrize("k", [2, 3])
def test_couplings_that_span_many_decades(k):
    """A diagonal similarity transform of the operator (creators times d, annihilators by 1 / d, d = 2^-14 on
    two virtuals): couplings out of the scaled orbitals reach 2^28, where 2^-54 of them is above the tolerance."""
    import torch
    qf, n, no, t1, t2, e0, F, W, sp, own = _system13(6, k)
    d = torch.ones(n, dtype=torch.float64, device="cuda")
    d[no] = d[no + 3] = 2.0 ** -14
    f = F * d[:, None] / d[None, :]
    w = W * torch.einsum("p,q,r,s->pqrs", d, 1 / d, d, 1 / d)
    assert float(w.abs().max()) < 2.0 ** 29 and float(f.abs().max()) < 2.0 ** 29
    a = _solve(qf, n, no, e0, f, w, k, dev(sp), t1, t2, own, False)
    b = _solve(qf, n, no, e0, f, w, k, dev(sp), t1, t2, own, True)
    for x, y in zip(a, b):
        assert np.abs(x - y).max() < 1e-12
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    assert (b[1] == 0).mean() > 0.3
