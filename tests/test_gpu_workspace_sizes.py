"""FP64 dressings with smaller workspaces: the arrays alone (what the call took before the products packed
operands), the arrays and the scale exponents, and all; 256 bytes less than the arrays are refused.

Tolerances: without packed operands the products differ by their tiles only, which round a sum up to four times
at 2^-56 of the operand rows' norms (below 10, about ten products an element): 1e-13 of the largest integral.
Against the packed form 1e-12, as in test_gpu_fixed_dress.py.
"""
import numpy as np
import pytest

from paper_2606_04186_gb300 import synth

from gpu_util import dev, library

pytestmark = pytest.mark.gpu


def arrays_bytes(n, o):
    """The twelve arrays of a dressing, each rounded up to 256 bytes (include/qflow.h)."""
    v = n - o
    counts = [n * n, o * o, v * v, o ** 4, v * o, *([o * o * v * v] * 6), 256]
    return sum(-(-8 * c // 256) * 256 for c in counts)


@pytest.mark.parametrize("n,no", [(2, 1), (3, 2), (9, 8), (13, 4), (24, 5), (33, 30), (44, 6), (57, 7)])
def test_dressing_with_the_arrays_alone(n, no):
    import torch
    qf = library()
    _, h, g = synth.make_system(n, no, 4.0, 100 + n)
    t1, t2 = synth.random_amplitudes(no, n - no, n, 0.05, 0.1)
    args = [dev(a) for a in (h, g, t1, t2)]
    full, least = qf.dress_workspace(n, no), arrays_bytes(n, no)
    assert least < full
    o, v = no, n - no
    scales = 4 * (5 * o * o + 6 * v * v + 20 * o * v + 2 * o * o * v + v)
    out = []
    for size in (least, min(full, least + scales + 512), full):
        buf = torch.full((size + 512,), 0xff, dtype=torch.uint8, device="cuda")  # NaN everywhere
        e0 = torch.zeros(1, dtype=torch.float64, device="cuda")
        F = torch.full((n, n), np.nan, dtype=torch.float64, device="cuda")
        W = torch.full((n,) * 4, np.nan, dtype=torch.float64, device="cuda")
        qf.dress_device(*args, no, e0, F, W, buf[:size])
        torch.cuda.synchronize()
        assert bool((buf[size:] == 0xff).all())
        out.append((e0, F, W))
    for a, b, c in zip(*out):
        scale = max(1.0, out[2][2].abs().max().item())
        assert (a - b).abs().max().item() < 1e-13 * scale and (a - c).abs().max().item() < 1e-12 * scale
    with pytest.raises(RuntimeError):
        qf.dress_device(*args, no, e0, F, W, buf[: least - 256])
