"""The fused layers at the ends of their batch range: the library refuses the
batches whose padded pixels pass a 32-bit index (images of one or two rows are
padded to 16 pixels), and takes more samples than 65535 blocks of 16.
"""
import ctypes

import numpy as np
import pytest

from paper_2509_01099_gb300 import build as B
from paper_2509_01099_gb300.islbm import load_library
from tests.helpers import gpu_available


@pytest.mark.parametrize("base,batch,taken", [
    (1, 1 << 26, True), (1, 1 << 27, False), (1, 1 << 30, False),
    (2, 1 << 26, True), (2, 1 << 27, False), (2, 1 << 28, False),
    (4, 1 << 24, True), (4, (1 << 26) + 1, False),
])
def test_batches_beyond_a_32_bit_index_are_refused(base, batch, taken):
    B.build()
    lib = load_library()
    chan = (ctypes.c_int * 2)(64, 64)
    n = ctypes.c_ulonglong()
    st = lib.islbm_cnn_backward_scratch(1, chan, base, 8, batch, ctypes.byref(n))
    assert (st == 0) == taken


@pytest.mark.gpu
@pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")
def test_a_million_samples_of_a_tiny_network():
    import torch
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=1, channels=(2,), hidden=8, seed=1)
    batch = 16 * 65535 + 1
    z = np.random.default_rng(0).standard_normal((batch, 16)).astype(np.float32)
    dy = torch.randn((batch, 1, 1, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    out = []
    for fused in (True, False):
        y = (net._forward_fused if fused else net._forward_chain)(z, True)
        out.append((y, {k: v.clone() for k, v in net.backward(dy).items()}))
    (y, g), (yr, gr) = out
    assert float((y - yr).norm() / yr.norm()) <= 1e-5
    # FP32 sums of 10^6 terms of random sign: 0.4 sqrt(10^6) 2^-24 = 2.4e-5 RMS in one chain
    for k in g:
        assert float((g[k] - gr[k]).norm() / gr[k].norm()) <= 1e-3, k
