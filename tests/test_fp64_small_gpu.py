"""FP64 steps at the sizes where the four-warp kernel of small meshes takes over.

Up to two rows of 32 nodes an SM go to it: partial warps, one and several of
them a row, and the first size that the one-warp kernel keeps, on stretched
and uniform meshes and with the upwind stencil, every population against the
oracle.  Both sides round at 2^-53; ten steps of fewer than 300 operations on
values of order one stay within 1e-13 (the bound of the FP64 parity tests).
"""
import numpy as np
import pytest

from oracle import islbm_oracle as O
from synthetic import random_populations, random_signed
from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("mesh", ["tanh", "uniform"])
@pytest.mark.parametrize("n", [4, 31, 32, 33, 64, 96, 101])
def test_small_fp64_steps(n, mesh):
    from paper_2509_01099_gb300 import build as B
    B.build()
    import paper_2509_01099_gb300 as pkg
    xi = O.mesh_tanh(n, 1.5) if mesh == "tanh" else O.mesh_uniform(n)
    cav = O.Cavity(xi, xi, params=O.Params(Ra=1e5))
    f = random_populations(9, cav.shape, seed=n, spread=0.2)
    g = random_signed(5, cav.shape, seed=n + 1, amplitude=0.12)
    cav.init_populations(f, g)
    cav.step(10)
    fr, gr = cav.post_collision()
    s = pkg.Solver(xi, xi, Ra=1e5, precision="fp64")
    s.set_populations(f, g)
    s.step(10)
    fp, gp = s.populations()
    s.close()
    assert np.abs(fp - fr).max() / np.abs(fr).max() <= 1e-13
    assert np.abs(gp - gr).max() / np.abs(gr).max() <= 1e-13
