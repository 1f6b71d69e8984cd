"""512 hidden units, the most the fused layers take: the GEMM chain splits that
sum of the second layer into two chunks that it adds, and so do they; outputs
and gradients are its bits (channels in multiples of 16)."""
import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("base,channels,hidden,batch", [
    (8, (16,), 512, 1), (8, (16,), 512, 200), (4, (32, 16), 512, 33),
    (8, (16,), 512, 6000),            # so many tiles that the sum is not split
    (8, (16,), 504, 40),              # below the chain's limit for a split
    (3, (16,), 512, 40),
])
def test_the_second_layer_sums_in_the_chains_chunks(base, channels, hidden, batch):
    import torch
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=base, channels=channels, hidden=hidden, seed=7)
    z = np.random.default_rng(batch).standard_normal((batch, 16)).astype(np.float32)
    got = []
    for fused in (True, False):
        net.fused = fused
        y = net.forward(z)
        dy = torch.randn(y.shape, device="cuda",
                         generator=torch.Generator("cuda").manual_seed(batch))
        got.append((y, {k: v.clone() for k, v in net.backward(dy).items()}))
    (y, g), (yr, gr) = got
    assert torch.equal(y, yr)
    for k in ("W1", "b1", "W2", "b2"):
        assert torch.equal(g[k], gr[k]), k
