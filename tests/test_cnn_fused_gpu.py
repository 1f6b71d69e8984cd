"""The network's fused layers against the chain of im2col GEMMs.

The fused kernels sum their products in the chain's order, so activations,
gradients handed down and weight gradients are the same bits wherever the input
channels are a multiple of 16 (else a 16-wide step of the sum crosses a tap in
the chain and not here: a few FP32 roundings, checked at 1e-5 of the norm, 40
times the largest of them, sqrt(576) 2^-24 of a sum of 576 terms, unless a BF16
rounding of a layer's input flips).  The sums over the batch of the fully
connected layers are short FP32 sums in another order (16 terms: 4 x 2^-24).
"""
import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


def _both(net, batch, seed):
    import torch
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((batch, 16)).astype(np.float32)
    out = []
    for fused in (True, False):
        assert net.fused
        net.fused = fused
        y = net.forward(z)
        dy = torch.randn(y.shape, device="cuda",
                         generator=torch.Generator("cuda").manual_seed(seed))
        g = {k: v.clone() for k, v in net.backward(dy).items()}
        out.append((y, g))
        net.fused = True
    return out


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm().clamp_min(1e-300))


@pytest.mark.parametrize("base,channels,hidden,batch", [
    (8, (64, 64, 48, 32, 16, 16), 256, 1),     # the warm-start network, its smallest call
    (8, (64, 64, 48, 32, 16, 16), 256, 5),
    (4, (32, 16, 16), 64, 33),                 # several launches of the first layers
    (8, (16, 64), 72, 2),
    (16, (48,), 32, 3),                        # a single layer, no upsampling
])
def test_fused_layers_are_the_chain(base, channels, hidden, batch):
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=base, channels=channels, hidden=hidden, seed=3)
    (y, g), (yr, gr) = _both(net, batch, seed=batch)
    assert _rel(y, yr) <= 4 * 2 ** -24
    for k in g:
        assert _rel(g[k], gr[k]) <= 4 * 2 ** -24 * (1 if k[:2] in ("Wc", "bc") else 4), k


@pytest.mark.parametrize("base,channels,hidden,out_ch,batch", [
    (3, (10, 7, 40, 5), 50, 2, 5),             # ragged channels, images of 6, 12 and 24 pixels
    (5, (24, 3), 30, 64, 2),
])
def test_ragged_layers_agree_with_the_chain(base, channels, hidden, out_ch, batch):
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=base, channels=channels, hidden=hidden, out_ch=out_ch, seed=4)
    (y, g), (yr, gr) = _both(net, batch, seed=7)
    assert _rel(y, yr) <= 1e-5
    for k in g:
        assert _rel(g[k], gr[k]) <= 1e-5, k


def test_wide_networks_take_the_chain():
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(base=4, channels=(80, 16), hidden=64)
    assert not net.fused
    assert net.forward(np.zeros((2, 16), np.float32)).shape == (2, 8, 8, 3)


def test_adam_of_all_tensors_is_adam_of_each():
    """Same operations on every value: the same bits, across block borders."""
    import ctypes
    import torch
    from paper_2509_01099_gb300.cnn import _p
    from paper_2509_01099_gb300.cnn import WarmStartNet
    a, b = (WarmStartNet(base=8, channels=(16, 24), hidden=40, seed=5) for _ in range(2))
    for k in a.names:
        gen = torch.Generator("cuda").manual_seed(len(k) + a.params[k].numel())
        a.grads[k].copy_(torch.randn(a.grads[k].shape, device="cuda", generator=gen))
        b.grads[k].copy_(a.grads[k])
    for t in (1, 2):
        a.adam(lr=1e-2)
        for k in b.names:
            f = ctypes.c_float
            assert b.lib.islbm_cnn_adam(_p(b.params[k]), _p(b.bf.get(k)), _p(b.grads[k]), _p(b.m[k]),
                                        _p(b.v[k]), b.params[k].numel(), f(1e-2), f(0.9), f(0.999),
                                        f(1e-8), t, b._stream()) == 0
    for k in a.names:
        for x, y in ((a.params, b.params), (a.m, b.m), (a.v, b.v), (a.bf, b.bf)):
            if k in x:
                assert torch.equal(x[k], y[k]), k
