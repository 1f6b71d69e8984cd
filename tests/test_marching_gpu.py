"""The marching 2-D step (two steps a launch) against the tile kernel's single steps.

The two kernels perform the same operations in the same order on every node,
so the states have to be equal bit for bit, in every storage form (stochastic
rounding included): meshes at and around the strip width (62 columns) and the
chunk rules (odd and even row counts, short and long chunks), and step counts
that mix launches of two steps, a single one and graphs of 64.
"""
import numpy as np
import pytest

from oracle import islbm_oracle as O
from synthetic import random_populations, random_signed
from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


def _pkg():
    from paper_2509_01099_gb300 import build as B
    B.build()
    import paper_2509_01099_gb300 as pkg
    return pkg


def _mesh(nx, ny):
    x, y = O.mesh_tanh(nx, 1.5), O.mesh_erf(ny, 1.0)
    return x, y * ((x[1] - x[0]) / (y[1] - y[0]))       # one lattice unit


# FP32 and FP16NEQ take the kernel from 600,000 nodes, the 16-bit deviations from 1,500,000
FP32 = [(16, 37501), (62, 9700), (63, 9601), (64, 9377), (125, 4801), (775, 777), (1030, 601),
        (4099, 151), (20001, 31)]
HALF = [(63, 23811), (1225, 1226), (9967, 151)]


@pytest.mark.parametrize("precision,nx,ny", [(p, *s) for p in ("fp32", "fp16neq") for s in FP32] +
                         [(p, *s) for p in ("fp16dev", "bf16dev") for s in HALF])
def test_two_steps_a_launch_are_single_steps(nx, ny, precision):
    pkg = _pkg()
    x, y = _mesh(nx, ny)
    f = random_populations(9, (ny, nx), seed=nx, spread=0.2)
    g = random_signed(5, (ny, nx), seed=ny, amplitude=0.12)
    states = []
    for kernel in ("auto", "tma_r2s2"):
        # the height sets the length scale: a Rayleigh number with a moderate viscosity
        s = pkg.Solver(x, y, Ra=1e6 * max(1.0, (ny / 200) ** 2), precision=precision, kernel=kernel)
        s.set_populations(f, g)
        got = []
        for steps in (2, 1, 67):
            s.step(steps)
            got.append(s.populations())
        s.close()
        states.append(got)
    for a, b in zip(*states):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("sizes", [(600, 511, 27), (128,) * 37, (1030, 64, 333)])
def test_batch_pairs_are_single_steps_of_each_cavity(sizes):
    """600,000 nodes and more: the batch advances two steps a launch."""
    pkg = _pkg()
    cavs = [dict(n=n, mesh=("tanh", "erf", "uniform")[k % 3], a=1.5, Ra=1e6 * (1 + k))
            for k, n in enumerate(sizes)]
    b = pkg.Batch(cavs, "fp32")
    alone = []
    for k, (c, m) in enumerate(zip(cavs, b.members)):
        n = c["n"]
        f = random_populations(9, (n, n), seed=k, spread=0.2)
        g = random_signed(5, (n, n), seed=k + 100, amplitude=0.12)
        xi = getattr(O, "mesh_" + c["mesh"])(n, *([] if c["mesh"] == "uniform" else [1.5]))
        s = pkg.Solver(xi, xi, Ra=c["Ra"], precision="fp32", kernel="tma_r2s2")
        for h in (m, s):
            h.set_populations(f, g)
        alone.append(s)
    for steps in (2, 1, 67):
        b.step(steps)
        b.synchronize()
        for m, s in zip(b.members, alone):
            s.step(steps)
            for x, y in zip(m.populations(), s.populations()):
                assert np.array_equal(x, y)
    for s in alone:
        s.close()
    b.close()
