"""A layer whose split weights exceed the workspace's 128 MiB stays on the functor engine: 1,100 rows (above
the FP32 tiles) through 2,100 x 9,000, forward and gradient.  Tolerance: test_gpu_mlp.py's 2e-5."""
import numpy as np
import pytest

from oracle import mlp
from paper_2606_04186_gb300 import synth

from gpu_util import library

pytestmark = pytest.mark.gpu


def test_layer_beyond_the_split_weights():
    import torch
    qf = library()
    I, H, O, rows = 16, 2100, 9000, 1100
    rng = np.random.default_rng(1)
    p = synth.mlp_init_params(I, H, O, 5).astype(np.float32)
    x = rng.standard_normal((rows, I)).astype(np.float32)
    t = rng.standard_normal((rows, O)).astype(np.float32)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    work = torch.full((qf.mlp_workspace(I, H, O, rows),), 0xff, dtype=torch.uint8, device="cuda")  # NaN everywhere
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
