"""The FP64 dressing's fixed-point products (fix_gemm.cuh) against the oracle at sizes on both sides
of the 32- and 64-wide tiles and of the stage depths, with one occupied or one virtual orbital, and
for integrals whose rows span many orders of magnitude.

Tolerance: an element of a product is off by at most 2^-54 sqrt(K) of the product of its operand rows'
norms (K <= 2 n^2 terms); with norms below 10 and about ten products per element this stays below
1e-13 of the largest integral.  The oracle's own FP64 sums are of the same size.
"""
import numpy as np
import pytest

from oracle import hbar
from paper_2606_04186_gb300 import synth

from gpu_util import dev, library

pytestmark = pytest.mark.gpu


def _dress(qf, h, g, t1, t2, no):
    import torch
    n = h.shape[0]
    e0 = torch.zeros(1, dtype=torch.float64, device="cuda")
    F = torch.full((n, n), np.nan, dtype=torch.float64, device="cuda")
    W = torch.full((n,) * 4, np.nan, dtype=torch.float64, device="cuda")
    work = torch.full((qf.dress_workspace(n, no),), 0xff, dtype=torch.uint8, device="cuda")  # NaN everywhere
    qf.dress_device(dev(h), dev(g), dev(t1), dev(t2), no, e0, F, W, work)
    torch.cuda.synchronize()
    return e0.item(), F.cpu().numpy(), W.cpu().numpy()


@pytest.mark.parametrize("n,no", [(2, 1), (5, 1), (5, 4), (9, 8), (11, 3), (13, 6), (17, 2), (20, 9), (20, 16), (22, 17), (29, 5), (33, 8)])
def test_dressing_at_tile_edges(n, no):
    qf = library()
    _, h, g = synth.make_system(n, no, 4.0, 100 + n)
    t1, t2 = synth.random_amplitudes(no, n - no, n, 0.05, 0.1)
    got, ref = _dress(qf, h, g, t1, t2, no), hbar.hbar2(h, g, t1, t2, no)
    scale = max(1.0, np.abs(ref[2]).max())
    for x, y in zip(got, ref):
        assert np.abs(np.asarray(x) - y).max() < 1e-13 * scale * 10


def test_dressing_with_rows_of_many_magnitudes():
    """Orbitals scaled by 10^0 .. 10^-6: every element to 1e-13 of what its own row scales allow."""
    qf = library()
    n, no = 19, 5
    _, h, g = synth.make_system(n, no, 4.0, 7)
    s = 10.0 ** -(6.0 * np.arange(n)[np.random.default_rng(1).permutation(n)] / (n - 1))
    h = h * s[:, None] * s[None, :]
    g = g * np.einsum("p,q,r,s->pqrs", s, s, s, s)
    t1, t2 = synth.random_amplitudes(no, n - no, 3, 0.05, 0.1)
    got, ref = _dress(qf, h, g, t1, t2, no), hbar.hbar2(h, g, t1, t2, no)
    for x, y in zip(got, ref):
        assert np.abs(np.asarray(x) - y).max() < 1e-13 * max(1.0, np.abs(ref[2]).max()) * 10


def test_non_finite_integral_reaches_the_dressed_blocks():
    qf = library()
    n, no = 12, 4
    _, h, g = synth.make_system(n, no, 4.0, 8)
    t1, t2 = synth.random_amplitudes(no, n - no, 3, 0.0, 0.1)
    g = g.copy()
    g[5, 6, 7, 8] = g[7, 8, 5, 6] = np.inf   # a vvvv element: reaches the doubles block through the ladder
    e0, F, W = _dress(qf, h, g, t1, t2, no)
    assert np.isfinite(e0) and np.isfinite(F[:no, :no]).all()
    assert not np.isfinite(W[5, :no, 7, :no]).any()
    ok = np.ones(n - no, dtype=bool)
    ok[[5 - no, 7 - no]] = False
    assert np.isfinite(W[no:, :no, no:, :no][np.ix_(ok, range(no), ok, range(no))]).all()


@pytest.mark.parametrize("n,no", [(26, 13), (43, 6), (47, 5), (50, 11)])
def test_tensor_core_products_equal_integer_pipe_products(n, no):
    """Problems above the work limit run on packed slices (oz_gemm.cuh); the static-scratch entry point
    computes the same products without packing (43 x 6 fits it), and torch's FP64 gives the ladder of the
    others.  Both forms are exact to 2^-54 sqrt(K) of the operand rows' norms, see above."""
    import torch
    qf = library()
    _, h, g = synth.make_system(n, no, 5.0, 300 + n)
    t1, t2 = synth.random_amplitudes(no, n - no, n, 0.05, 0.1)
    e0, F, W = _dress(qf, h, g, t1, t2, no)
    scale = max(1.0, np.abs(W).max())
    if (n, no) == (43, 6):
        f64 = lambda *s: torch.full(s, np.nan, dtype=torch.float64, device="cuda")  # noqa: E731
        e0s, Fs, Ws = f64(1), f64(n, n), f64(n, n, n, n)
        qf.dress_device_static(dev(h), dev(g), dev(t1), dev(t2), no, e0s, Fs, Ws)
        torch.cuda.synchronize()
        assert np.abs(F - Fs.cpu().numpy()).max() < 1e-12 * scale and np.abs(W - Ws.cpu().numpy()).max() < 1e-12 * scale
        return
    ref = hbar.hbar2(h, g, t1, t2, no)
    for x, y in zip((e0, F, W), ref):
        assert np.abs(np.asarray(x) - y).max() < 1e-12 * scale


def test_tensor_core_products_pass_non_finite_integrals_on():
    qf = library()
    n, no = 44, 6
    _, h, g = synth.make_system(n, no, 4.0, 8)
    t1, t2 = synth.random_amplitudes(no, n - no, 3, 0.0, 0.1)
    g = g.copy()
    g[15, 16, 17, 18] = g[17, 18, 15, 16] = np.nan
    e0, F, W = _dress(qf, h, g, t1, t2, no)
    assert np.isfinite(e0) and np.isfinite(F[:no, :no]).all()
    assert not np.isfinite(W[15, :no, 17, :no]).any()
    ok = np.ones(n - no, dtype=bool)
    ok[[15 - no, 17 - no]] = False
    assert np.isfinite(W[no:, :no, no:, :no][np.ix_(ok, range(no), ok, range(no))]).all()
