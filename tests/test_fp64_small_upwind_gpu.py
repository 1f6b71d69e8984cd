"""FP64 steps of small meshes with the upwind stencil: the four-warp kernel takes
them too (it pulls through the tables of either stencil).  Partial warps, several
warps a row and the first size that the one-warp kernel keeps, every population
against the oracle within the bound of the FP64 parity tests."""
import numpy as np
import pytest

from oracle import islbm_oracle as O
from synthetic import random_populations, random_signed
from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]


@pytest.mark.parametrize("mesh", ["tanh", "uniform"])
@pytest.mark.parametrize("n", [4, 31, 33, 64, 101])
def test_small_fp64_upwind_steps(n, mesh):
    import paper_2509_01099_gb300 as pkg
    xi = O.mesh_tanh(n, 1.5) if mesh == "tanh" else O.mesh_uniform(n)
    cav = O.Cavity(xi, xi, params=O.Params(Ra=1e5, stencil="upwind"))
    f = random_populations(9, cav.shape, seed=n, spread=0.2)
    g = random_signed(5, cav.shape, seed=n + 1, amplitude=0.12)
    cav.init_populations(f, g)
    cav.step(10)
    fr, gr = cav.post_collision()
    s = pkg.Solver(xi, xi, Ra=1e5, precision="fp64", stencil="upwind")
    s.set_populations(f, g)
    s.step(10)
    fp, gp = s.populations()
    s.close()
    assert np.abs(fp - fr).max() / np.abs(fr).max() <= 1e-13
    assert np.abs(gp - gr).max() / np.abs(gr).max() <= 1e-13
