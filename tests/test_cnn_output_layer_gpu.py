"""A last convolution of 64 input channels and 3 output channels: its sum of 576
products is split where the GEMM chain splits it.  (A width that is not a
multiple of 8 takes the chain's mma.sync product, whose tiles and chunks differ
from those of the tensor-memory one.)  Outputs are the chain's bits below, at
and above the sizes where either product stops splitting (19,456 and 38,912
pixels), and at widths in multiples of 8."""
import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("out_ch", [3, 5, 8])
@pytest.mark.parametrize("batch", [1, 75, 76, 77, 100, 151, 152, 153, 300])
def test_the_last_layer_sums_in_the_chains_chunks(batch, out_ch):
    import torch
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=16, channels=(64,), hidden=32, out_ch=out_ch, seed=9)
    z = np.random.default_rng(batch).standard_normal((batch, 16)).astype(np.float32)
    assert torch.equal(net._forward_fused(z, False), net._forward_chain(z, False))
