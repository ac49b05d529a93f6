"""The network's two product forms at the row counts where they change over and at ragged sizes: FP32
tiles up to 1,024 rows, tensor-core row streaming above (layer widths that are no multiple of four are
held in padded rows; an odd input width takes the functor engine).

Tolerances: tests/test_gpu_mlp.py's 2e-5 of the largest value (three-term TF32 products and FP32 sums of
up to 3,000 rows; the FP32 tiles are more accurate).
"""
import numpy as np
import pytest

from oracle import mlp
from paper_2606_04186_gb300 import synth

from gpu_util import library

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,rows", [((708, 256, 54), 1024), ((708, 256, 54), 1025), ((708, 319, 54), 1300),
                                        ((708, 45, 54), 2111), ((35, 130, 7), 1500), ((64, 64, 300), 1153),
                                        ((708, 33, 54), 31), ((5, 3, 1), 65)])
def test_products_at_row_counts(sizes, rows):
    import torch
    qf = library()
    I, H, O = sizes
    rng = np.random.default_rng(rows)
    p = (synth.mlp_init_params(I, H, O, 5) + 0.05 * rng.standard_normal(mlp.param_count(I, H, O))).astype(np.float32)
    x = rng.standard_normal((rows, I)).astype(np.float32)
    t = rng.standard_normal((rows, O)).astype(np.float32)
    keep = rng.random(rows) < 0.9
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    work = torch.full((qf.mlp_workspace(I, H, O, rows),), 0xff, dtype=torch.uint8, device="cuda")  # NaN everywhere
    y = torch.zeros((rows, O), dtype=torch.float32, device="cuda")
    qf.mlp_forward_device(I, H, O, cu(p), cu(x), y, work)
    grad = torch.zeros(p.size, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    qf.mlp_grad_device(I, H, O, cu(p), cu(x), cu(t), grad, loss, work, mask=cu(keep.astype(np.uint8)))
    torch.cuda.synchronize()
    p64, x64, t64 = (a.astype(np.float64) for a in (p, x, t))
    y_ref, _ = mlp.forward(p64, x64, I, H, O)
    l_ref, g_ref = mlp.loss_and_grad(p64, x64[keep], t64[keep], I, H, O)
    f = keep.sum() / rows
    for got, ref in ((y, y_ref), (grad, f * g_ref), (loss, np.array([f * l_ref]))):
        assert np.abs(got.cpu().numpy() - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())
