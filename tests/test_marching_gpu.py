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


# FP32 takes the kernel from 600,000 nodes, the 16-bit forms from 1,500,000
FP32 = [(16, 37501), (62, 9700), (63, 9601), (64, 9377), (125, 4801), (775, 777), (1030, 601),
        (4099, 151), (20001, 31)]
HALF = [(63, 23811), (1225, 1226), (9967, 151)]


@pytest.mark.parametrize("precision,nx,ny", [("fp32", *s) for s in FP32] +
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
