"""The network's row-streaming products against the functor engine, bit for bit: both split the same elements
the same way and sum in the same order.  Inputs and workspace 4 bytes off 16 cannot be read by TMA, so
that call takes the functor engine for every product; aligned ones stream rows.  Gradients take these forms at
every row count, inference above the 1,024 rows of the FP32 tiles."""
import numpy as np
import pytest

from paper_2606_04186_gb300 import synth

from gpu_util import library

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(708, 256, 54), (708, 45, 54), (64, 130, 300)])
@pytest.mark.parametrize("rows", [1, 31, 128, 1000, 1025, 4097])
def test_streamed_rows_equal_the_functor_engine(sizes, rows):
    import torch
    qf = library()
    I, H, O = sizes
    gen = torch.Generator(device="cuda").manual_seed(rows)
    p = torch.as_tensor(synth.mlp_init_params(I, H, O, 5).astype(np.float32), device="cuda")
    x = torch.randn((rows, I), generator=gen, device="cuda")
    t = torch.randn((rows, O), generator=gen, device="cuda")
    nb, out = qf.mlp_workspace(I, H, O, rows), []
    work = torch.full((nb + 16,), 0xff, dtype=torch.uint8, device="cuda")  # NaN everywhere
    xbuf = torch.empty(rows * I + 4, device="cuda")
    for off in (0, 1):
        xs = xbuf[off:off + rows * I].view(rows, I)
        xs.copy_(x)
        assert xs.data_ptr() % 16 == 4 * off and work.data_ptr() % 16 == 0
        w = work[4 * off:4 * off + nb]
        y = torch.zeros((rows, O), device="cuda")
        grad, loss = torch.zeros_like(p), torch.zeros(1, device="cuda")
        qf.mlp_forward_device(I, H, O, p, xs, y, w)
        qf.mlp_grad_device(I, H, O, p, xs, t, grad, loss, w)
        torch.cuda.synchronize()
        out.append((y, grad, loss))
    for a, b in zip(*out):
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)
