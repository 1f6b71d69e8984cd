"""The forward layers start before the layer below has finished, so they read
its output with ordinary loads behind grid_wait: the read-only path (__ldg) is
for data that no kernel writes meanwhile, and its loads are not ordered by the
wait.  The source is read for that (a wrong load shows in the results only by
chance); on a GPU, predictions enqueued one after the other without a pause,
with other features and batch sizes, are the bits of the GEMM chain.
"""
import os
import re

import numpy as np
import pytest

from tests.helpers import gpu_available

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_2509_01099_gb300", "csrc", "islbm_cnn_net.cu")


def _function(text, name):
    """The body of the function `name` (its definition's braces)."""
    at = re.search(r"\b%s\([^;{}]*\)\s*\{" % name, text)
    assert at, name
    depth, k = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        k += 1
    return text[at.end():k]


def test_early_layers_read_their_input_with_ordinary_loads():
    text = re.sub(r"//[^\n]*", "", open(SOURCE).read())
    after = _function(text, "k_conv_fwd").split("grid_wait()", 1)[1]
    assert "__ldg" not in after and "p.x" in after
    calls = re.findall(r"stage_window(\S*?)\(", after)
    assert calls == ["<true>"]
    assert "__ldg" not in _function(text, "stage_window")
    live = _function(text, "load_image").split("else")[0]
    assert "LIVE" in live and "__ldg" not in live


@pytest.mark.gpu
@pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")
def test_predictions_without_a_pause():
    from paper_2509_01099_gb300.cnn import WarmStartNet
    net = WarmStartNet(seed=6)
    rng = np.random.default_rng(8)
    z = [rng.standard_normal((1 + k % 3, 16)).astype(np.float32) for k in range(24)]
    net.forward(z[0], keep=False)
    got = [net.forward(v, keep=False) for v in z]
    for v, y in zip(z, got):
        ref = net._forward_chain(v, False)
        assert float((y - ref).norm() / ref.norm()) <= 4 * 2 ** -24
