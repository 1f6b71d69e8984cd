"""Rounding of the output velocities: no larger than that of FP64 arithmetic.

The stored FP32 populations are read back bit for bit and the velocities formed
from them in extended precision.  A plain FP64 evaluation (sums, force, division
by rho) is the yardstick: the RMS error of the library's velocities, whose sums
are formed on the integer units and whose division goes by a reciprocal, may not
exceed its error.  The quotient is exact to 2^-74 before it is rounded, so about
one in 2^20 rounds the other way: by at most 2^-20 of its half ulp, which is also
the margin of the comparison and of the largest error.
"""
import os

import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not gpu_available(), reason="needs a CUDA device")]

E2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
E3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
      (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


def _velocity(f, g, e, gbeta, t_ref, dtype):
    """u, v[, w] of post-collision deviations f, g, evaluated in dtype."""
    f, g = f.astype(dtype), g.astype(dtype)
    gbeta, t_ref = dtype(gbeta), dtype(t_ref)
    rho = 1 + f.sum(axis=0)
    force = rho * gbeta * (g.sum(axis=0) - t_ref)
    out = []
    for axis in range(len(e[0])):
        j = sum(dtype(c[axis]) * f[i] for i, c in enumerate(e) if c[axis])
        out.append((j - force / 2 if axis == 1 else j) / rho)
    return out


def _state(s, q, path):
    """The stored state [q][nodes shape], from a checkpoint (planes of padded rows)."""
    s.save(path)
    n = s.shape
    pitch = (n[-1] + 31) // 32 * 32
    count = q * pitch * int(np.prod(n[:-1]))
    raw = np.fromfile(path, dtype=np.uint8)[-4 * count:].view(np.float32)
    return raw.reshape((q,) + n[:-1] + (pitch,))[..., :n[-1]]


@pytest.mark.parametrize("dim,n,speed,shift", [(2, 96, 0.05, 0.0), (2, 96, 1e-4, 0.0),
                                               (2, 96, 0.05, 0.03), (2, 96, 0.05, -0.4),
                                               (3, 24, 0.05, 0.0)])
def test_velocities_round_no_worse_than_fp64(dim, n, speed, shift, tmp_path):
    import paper_2509_01099_gb300 as pkg
    xi = pkg.islbm_mesh_tanh(n, 1.5)
    s = pkg.Solver(*([xi] * dim), Ra=1e6, precision="fp32")
    rng = np.random.default_rng(n + dim)
    rho = 1 + shift + 0.005 * rng.uniform(-1, 1, s.shape)
    vel = [speed * rng.uniform(-1, 1, s.shape) for _ in range(dim)]
    s.set_fields(rng.uniform(-0.5, 0.5, s.shape), *vel, rho=rho)
    e = E2 if dim == 2 else E3
    d = _state(s, len(e) + 2 * dim + 1, os.path.join(tmp_path, "state"))
    f, g = d[:len(e)], d[len(e):]
    args = (f, g, e, s.info.gbeta, -0.5)
    exact = _velocity(*args, np.longdouble)
    plain = _velocity(*args, np.float64)
    got = s.fields()
    s.close()
    for k, name in enumerate("uvw"[:dim]):
        new = (got[name] - exact[k]).astype(np.float64)
        old = (plain[k] - exact[k]).astype(np.float64)
        assert np.abs(new).max() <= 2.0 ** -40 * np.abs(exact[k]).max()   # the same numbers
        assert (new ** 2).mean() <= (old ** 2).mean() * (1 + 2.0 ** -20), name
        if name != "v":
            ulp = np.spacing(np.abs(exact[k]).astype(np.float64))
            assert (np.abs(new) <= 0.5 * ulp * (1 + 2.0 ** -19)).all()
