"""Large batches: the fully connected layers of the fused network.

The features of up to 32 samples, of up to 480, and of more than four times 480
reach the kernel in three ways, and a block then takes several tiles of 16
samples; every sample is the bits of the GEMM chain at the ends of these ranges
(channels in multiples of 16), within a captured graph too, where no copy from
pageable memory is possible.  A small network at 16,384 samples has to stay
below the chain's time, as at small batches (one launch for every 32 samples
would take 37 times as long there; half of the chain's time is the margin).
"""
import time

import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


def _net(**kw):
    from paper_2509_01099_gb300.cnn import WarmStartNet
    return WarmStartNet(seed=2, **kw)


def _z(batch):
    return np.random.default_rng(batch).standard_normal((batch, 16)).astype(np.float32)


@pytest.mark.parametrize("hidden", [64, 50])
@pytest.mark.parametrize("batch", [31, 32, 33, 479, 480, 481, 961, 1920, 1921, 5000])
def test_every_sample_is_the_chain(hidden, batch):
    import torch
    net = _net(base=2, channels=(16,), hidden=hidden)
    z = _z(batch)
    y = net.forward(z)
    zk = net.cache["flat"][:16 * batch].view(batch, 16).cpu()
    assert torch.equal(zk, torch.from_numpy(z).bfloat16().float())
    assert torch.equal(y, net._forward_chain(z, False))


def test_a_captured_forward_of_a_large_batch():
    import torch
    net = _net(base=2, channels=(16,), hidden=64)
    z = _z(2500)
    net.forward(z)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y = net.forward(z, keep=False)
    y.zero_()
    g.replay()
    assert torch.equal(y, net._forward_chain(z, False))


@pytest.mark.parametrize("batch", [512, 16384])
def test_a_small_network_at_large_batches_is_no_slower_than_the_chain(batch):
    import torch
    net = _net(base=2, channels=(16,), hidden=256)
    z = _z(batch)

    def best(fn):
        t = []
        for _ in range(12):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            fn()
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t)

    assert best(lambda: net.forward(z)) <= 1.5 * best(lambda: net._forward_chain(z, True))


@pytest.mark.parametrize("base,channels,batch,fused", [
    (1, (16,), 8192, True), (1, (16,), 8193, False), (2, (64,), 16384, False),
    (1, (16, 16), 20000, False), (2, (16, 16), 20000, True), (3, (16,), 20000, True),
    (1, (2,), 65535 * 64 + 1, True),        # beyond the chain's grids
])
def test_tiny_images_in_large_batches_take_the_chain(base, channels, batch, fused):
    net = _net(base=base, channels=channels, hidden=16)
    net.forward(_z(batch))
    assert ("flat" in net.cache) == fused


def test_tiny_images_in_a_captured_large_batch():
    """A graph keeps the fused layers: the chain's copy of the features cannot be captured."""
    import torch
    net = _net(base=1, channels=(16,), hidden=16)
    z = _z(9000)
    net._forward_fused(z, False)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y = net.forward(z, keep=False)
    y.zero_()
    g.replay()
    assert torch.equal(y, net._forward_chain(z, False))
