"""The FP64 solver's two kernels against each other: spaces started from Phi run on fixed-point
products (solve_fixed.cu), an all-zero start vector (which also means Phi) takes the general kernel.
Both run the same Davidson iteration, so statuses and iteration counts are equal and energies and
increments differ by rounding only.

Tolerances: sigma is exact to 2^-54 of the space's largest coupling per term (the general kernel's
rounding is of the same size), amplified by the few iterations and the division by gaps of 0.3 Eh
and more: 1e-12 leaves two orders of magnitude.
"""
import numpy as np
import pytest

from paper_2606_04186_gb300 import synth

from gpu_util import dev, library

pytestmark = pytest.mark.gpu


def _solve(qf, n, no, e0, F, W, k, sp, t1, t2, own, general, **kw):
    import torch
    ns = len(sp)
    ndet = {1: 4, 2: 36, 3: 400}[k]
    energy = torch.full((ns,), 7.0, dtype=torch.float64, device="cuda")
    status = torch.full((ns,), -1, dtype=torch.int32, device="cuda")
    iters = torch.full((ns,), -1, dtype=torch.int32, device="cuda")
    t1n, t2n = t1.clone(), t2.clone()
    guess = torch.zeros((ns, ndet), dtype=torch.float64, device="cuda") if general else None
    qf.solve_device(n, no, e0, F, W, k, sp, energy, status, iters, owner1=own[0], owner2=own[1], t1_old=t1,
                    t2_old=t2, t1_new=t1n, t2_new=t2n, guess=guess, **kw)
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in (energy, status, iters, t1n, t2n)]


def _system(n, no, xi, seed, amp):
    import torch
    qf = library()
    _, h, g = synth.make_system(n, no, xi, seed)
    t1, t2 = (dev(a) for a in synth.random_amplitudes(no, n - no, seed, amp, amp))
    e0 = torch.zeros(1, dtype=torch.float64, device="cuda")
    F = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    W = torch.zeros((n,) * 4, dtype=torch.float64, device="cuda")
    work = torch.zeros(qf.dress_workspace(n, no), dtype=torch.uint8, device="cuda")
    qf.dress_device(dev(h), dev(g), t1, t2, no, e0, F, W, work)
    return qf, h, g, t1, t2, e0, F, W


@pytest.mark.parametrize("n,no,xi,amp,count", [(10, 3, 3.0, 0.0, 35), (13, 4, 8.0, 0.03, 211), (24, 5, 4.0, 0.02, 1531)])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_fixed_point_solver_equals_general_kernel(n, no, xi, amp, count, k):
    qf, h, g, t1, t2, e0, F, W = _system(n, no, xi, 17 + n, amp)
    import math
    most = math.comb(no, k) * math.comb(n - no, k)
    sp = synth.sampled_spaces(n, no, min(count, most), 3, no=k, nv=k)
    perm, o1, o2, _ = qf.plan(h, g, no, sp)
    sp = sp[perm]
    if len(sp) > 4:
        sp[2] = sp[2][[0, 1, 3, 2, 4, 5, 6, 7]] if k > 1 else sp[2]  # any orbital order is accepted
        sp[3, 0] = k + 1  # malformed: skipped with status 4
    own = (dev(o1), dev(o2))
    a = _solve(qf, n, no, e0, F, W, k, dev(sp), t1, t2, own, False)
    b = _solve(qf, n, no, e0, F, W, k, dev(sp), t1, t2, own, True)
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    assert (a[1] == 0).sum() >= len(sp) - 1
    for x, y in zip((a[0], a[3], a[4]), (b[0], b[3], b[4])):
        assert np.abs(x - y).max() < 1e-12


@pytest.mark.parametrize("k", [1, 2, 3])
def test_spaces_the_fixed_point_kernel_passes_on(k):
    """Integrals without pair symmetry, non-finite integrals and an iteration limit of one."""
    import torch
    qf, h, g, t1, t2, e0, F, W = _system(13, 4, 5.0, 5, 0.02)
    n, no = 13, 4
    sp = synth.sampled_spaces(n, no, 25, 4, no=k, nv=k)
    perm, o1, o2, _ = qf.plan(h, g, no, sp)
    sp, own = dev(sp[perm]), (dev(o1), dev(o2))
    rng = np.random.default_rng(0)
    bent = W + dev(1e-3 * rng.standard_normal((n,) * 4))
    broken = W.clone()
    broken[1, 5, 2, 6] = float("nan")
    broken[0, 7, 0, 7] = float("inf")
    tiny = W * 0.0
    for w, kw in ((bent, {}), (broken, {}), (tiny, {}), (W, {"max_iter": 1}), (W, {"tol": 1e-6})):
        a = _solve(qf, n, no, e0, F, w, k, sp, t1, t2, own, False, **kw)
        b = _solve(qf, n, no, e0, F, w, k, sp, t1, t2, own, True, **kw)
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
        for x, y in zip((a[0], a[3], a[4]), (b[0], b[3], b[4])):
            ok = np.isfinite(y)
            assert np.array_equal(np.isnan(x), np.isnan(y))
            assert np.abs(x[ok] - y[ok]).max(initial=0.0) < 1e-12
