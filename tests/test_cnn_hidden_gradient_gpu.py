"""The hidden layer's gradient (k_fc_dh): a block's 16 warps share its tiles by
the number of chunks of the sum and the size of the batch.  Every way of
sharing gives the bits of the GEMM chain (W1 and b1 sum what it hands down), at
tiles that do not fill a block and ragged batches, and large batches take no
longer than the chain (half its time measured; one warp of sixteen working
takes 1.4 times as long; the margin is a tenth)."""
import time

import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


def _both(base, channels, hidden, batch):
    import torch
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=base, channels=channels, hidden=hidden, seed=7)
    z = np.random.default_rng(batch).standard_normal((batch, 16)).astype(np.float32)
    dy = torch.randn((batch, net.size, net.size, 3), device="cuda",
                     generator=torch.Generator("cuda").manual_seed(batch))
    grads, times = [], []
    for fused in (True, False):
        net.fused = fused
        net.forward(z)
        grads.append({k: v.clone() for k, v in net.backward(dy).items()})
        t = []
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            net.backward(dy)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        times.append(min(t))
    return grads, times


@pytest.mark.parametrize("base,hidden,batch", [
    (2, 256, 4096), (4, 256, 16384 + 7),      # one chunk: a warp a tile
    (6, 256, 2000), (8, 256, 700),            # two and four chunks: as many warps a tile
    (8, 256, 100),                            # too few samples to share a block
    (2, 136, 8000), (2, 40, 8100),            # hidden units that do not fill a block's tiles
    (2, 264, 2500), (4, 72, 5000),
])
def test_every_sharing_is_the_chain(base, hidden, batch):
    import torch
    (got, ref), _ = _both(base, (16,), hidden, batch)
    for k in ("W1", "b1", "W2", "b2"):
        assert torch.equal(got[k], ref[k]), k


@pytest.mark.parametrize("base,hidden,batch", [(8, 256, 16384), (16, 512, 4096)])
def test_large_batches_are_no_slower_than_the_chain(base, hidden, batch):
    _, (fused, chain) = _both(base, (16,), hidden, batch)
    assert fused <= 1.1 * chain
