"""The network's workspace over the accepted sizes: the activations and what the backward pass keeps of them
(3 hidden and 2 output rows per batch row), at most 128 MiB of split weights, and alignment.  Widest layer
times longest sum, a product no layer has, would be 32 GiB for one row of 8 x 4,096 x 65,536."""
import pytest

from paper_2606_04186_gb300 import qflow

MIB = 1 << 20


@pytest.mark.parametrize("sizes", [(708, 256, 54), (708, 1024, 54), (1, 1, 1), (8, 4096, 65536), (65536, 4096, 8),
                                   (65536, 4096, 65536), (65536, 1, 65536), (300, 2048, 2048)])
@pytest.mark.parametrize("rows", [0, 1, 128, 100_000])
def test_workspace_is_activations_and_bounded_weights(sizes, rows):
    I, H, O = sizes
    got = qflow.mlp_workspace(I, H, O, rows)
    batch = 4 * rows * (3 * (H + 3) + 2 * O)
    assert 4 * rows * (3 * H + 2 * O) <= got <= batch + 128 * MIB + 16 * 256 + 512
    # no more than twice the network's own (padded) layers
    pad = lambda x, m: -(-x // m) * m  # noqa: E731
    layers = max(pad(n, 256) * pad(k, 32) for n, k in ((H, I), (H, H), (O, H), (H, O)))
    assert got - batch <= 2 * 4 * layers + 16 * 256 + 512
