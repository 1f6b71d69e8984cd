"""Sums over the batch in the gradients of the fully connected layers.

They are taken in the order of the GEMM chain (steps of 16 samples on the
tensor cores, its chunks of samples, eight interleaved lanes for the biases), so
from equal inputs they are its bits at every batch size: one step and several,
the first batch that splits the sum, several chunks of the biases (2,048
samples), ragged ends.  The networks' layers have channels in multiples of 16,
where everything handed down to these layers is the same bits.  Their
error against FP64 is then the chain's.
"""
import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("hidden,batch", [
    (64, 1), (64, 16), (64, 33), (64, 511), (64, 512), (64, 1040), (64, 4100),
    (72, 16), (72, 700),               # hidden units that do not fill the last tile
    (50, 40), (50, 600), (50, 2049),   # leading dimensions of the chain's mma.sync form
])
def test_fully_connected_gradients_are_the_chain(hidden, batch):
    import torch
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=4, channels=(32, 16), hidden=hidden, seed=3)
    z = np.random.default_rng(batch).standard_normal((batch, 16)).astype(np.float32)
    got = []
    for fused in (True, False):
        net.fused = fused
        y = net.forward(z)
        dy = torch.randn(y.shape, device="cuda",
                         generator=torch.Generator("cuda").manual_seed(batch))
        got.append({k: v.clone() for k, v in net.backward(dy).items()})
    for k in ("W1", "b1", "W2", "b2"):
        assert torch.equal(got[0][k], got[1][k]), k


def _lanes(d):
    """FP32 sums of the rows of d by eight interleaved lanes in chunks of 2,048."""
    total = np.zeros(d.shape[1], np.float32)
    for m in range(0, len(d), 2048):
        part = np.zeros(d.shape[1], np.float32)
        for r in range(8):
            lane = np.zeros(d.shape[1], np.float32)
            for row in d[m:m + 2048][r::8]:
                lane = lane + row
            part = part + lane
        total = total + part
    return total


@pytest.mark.parametrize("batch", [16, 256, 4096])
def test_bias_sums_against_fp64(batch):
    """A network that hands dy down to the second layer unchanged (the centre tap
    is the identity, its input 0): b2's gradient is the sum of dy over the batch."""
    import torch
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=1, channels=(16,), hidden=16, out_ch=16, seed=5)
    net.params["Wc0"].zero_()[4 * 16:5 * 16].copy_(torch.eye(16))
    net.params["W1"].zero_()
    net.params["W2"].zero_()
    for k in ("Wc0", "W1", "W2"):
        net._to_bf16(net.params[k], net.bf[k])
    rng = np.random.default_rng(batch)
    err = np.zeros(2)                                   # squares: these sums, one chain
    for _ in range(16):
        dy = torch.from_numpy(rng.standard_normal((batch, 1, 1, 16))).bfloat16().float()
        net.forward(np.zeros((batch, 16), np.float32))
        got = net.backward(dy.cuda())["b2"].cpu().numpy()
        d = dy.view(batch, 16).numpy()
        assert np.array_equal(got, _lanes(d))
        exact = d.astype(np.float64).sum(axis=0)
        chain = np.add.accumulate(d, axis=0)[-1]        # one FP32 chain over the batch
        err += [((got - exact) ** 2).sum(), ((chain - exact) ** 2).sum()]
    assert err[0] <= err[1]
