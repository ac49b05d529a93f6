"""Workspaces aligned to their element type only: packed operands are read by TMA, which needs 16 bytes, so
these calls place them, or choose the products that pack nothing, by the address they get.

Tolerances: the two forms of the FP64 products are exact to 2^-54 sqrt(K) of the operand rows' norms (1e-12
of the largest integral, as in test_gpu_fixed_dress.py); the network's as in test_gpu_mlp.py.
"""
import numpy as np
import pytest

from oracle import mlp
from paper_2606_04186_gb300 import synth

from gpu_util import dev, library

pytestmark = pytest.mark.gpu


def test_fp64_dressing_with_an_8_byte_aligned_workspace():
    import torch
    qf = library()
    n, no = 44, 6  # above the work limit of the tensor-core products
    _, h, g = synth.make_system(n, no, 5.0, 17)
    t1, t2 = synth.random_amplitudes(no, n - no, 18, 0.05, 0.1)
    nb, out = qf.dress_workspace(n, no), []
    buf = torch.full((nb + 16,), 0xff, dtype=torch.uint8, device="cuda")
    for off in (0, 8):
        e0 = torch.zeros(1, dtype=torch.float64, device="cuda")
        F = torch.full((n, n), np.nan, dtype=torch.float64, device="cuda")
        W = torch.full((n,) * 4, np.nan, dtype=torch.float64, device="cuda")
        qf.dress_device(dev(h), dev(g), dev(t1), dev(t2), no, e0, F, W, buf[off:off + nb])
        torch.cuda.synchronize()
        out.append((e0, F, W))
    scale = max(1.0, out[0][2].abs().max().item())
    for a, b in zip(*out):
        assert (a - b).abs().max().item() < 1e-12 * scale


@pytest.mark.parametrize("off", [4, 8])
def test_network_with_an_unaligned_workspace(off):
    import torch
    qf = library()
    (I, H, O), rows = (708, 45, 54), 1300  # above the row count of the FP32 tiles
    rng = np.random.default_rng(off)
    p = synth.mlp_init_params(I, H, O, 5).astype(np.float32)
    x = rng.standard_normal((rows, I)).astype(np.float32)
    t = rng.standard_normal((rows, O)).astype(np.float32)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    nb = qf.mlp_workspace(I, H, O, rows)
    work = torch.full((nb + 16,), 0xff, dtype=torch.uint8, device="cuda")[off:off + nb]
    y = torch.zeros((rows, O), dtype=torch.float32, device="cuda")
    qf.mlp_forward_device(I, H, O, cu(p), cu(x), y, work)
    grad = torch.zeros(p.size, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    qf.mlp_grad_device(I, H, O, cu(p), cu(x), cu(t), grad, loss, work)
    torch.cuda.synchronize()
    p64, x64, t64 = (a.astype(np.float64) for a in (p, x, t))
    y_ref, _ = mlp.forward(p64, x64, I, H, O)
    l_ref, g_ref = mlp.loss_and_grad(p64, x64, t64, I, H, O)
    for got, ref in ((y, y_ref), (grad, g_ref), (loss, np.array([l_ref]))):
        assert np.abs(got.cpu().numpy() - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())
