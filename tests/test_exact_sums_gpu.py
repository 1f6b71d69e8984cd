"""Field output, reductions and time averages formed from FP32 states on the
integer units (csrc/islbm_exactsum.cuh, csrc/islbm_reduce.cuh).

The stored populations are read back bit for bit (islbm_get_rows) and the fields
formed from them in extended precision.  Sums: each of up to 14 values is
aligned to 58 bits and the sum rounded once, so rho, T and j are within
14 * 2^-58 max|f| + 2^-53 |sum| of the true sums; the velocity adds the
reciprocal and the products, each below 2^-52 relative: 8 * 2^-53 of
(|j| + |F|) / rho + 14 * 2^-58 max|f| / rho bounds them together.
"""
import numpy as np
import pytest

from tests.helpers import gpu_available

pytestmark = pytest.mark.gpu

if gpu_available():
    from paper_2509_01099_gb300 import build as _B
    _B.build()
import paper_2509_01099_gb300 as pkg  # noqa: E402

EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])


def _state(s, ny, nx, spread, seed):
    """A random FP32 state whose populations span 2^-spread .. 1, with zeros."""
    import torch
    rng = np.random.default_rng(seed)
    pitch = (nx + 31) // 32 * 32
    f = (0.1 * rng.uniform(-1, 1, (14, ny, pitch))
         * 2.0 ** -rng.uniform(0, spread, (14, ny, pitch))).astype(np.float32)
    f[rng.random(f.shape) < 0.05] = 0.0
    s.set_rows(0, ny, torch.from_numpy(f).cuda())
    return f[:, :, :nx].astype(np.longdouble)


@pytest.mark.parametrize("n,spread", [(33, 0), (70, 24), (128, 60), (5, 3)])
def test_fields_of_fp32_state(n, spread):
    import torch
    xi = pkg.islbm_mesh_tanh(n, 1.5)
    s = pkg.Solver(xi, xi, Ra=1e6, precision="fp32")
    f = _state(s, n, n, spread, seed=n)
    o = s.info
    top = np.abs(f[:9]).max(axis=0)
    rho = 1 + f[:9].sum(axis=0)
    T = f[9:].sum(axis=0)
    jx, jy = np.tensordot(EX, f[:9], 1), np.tensordot(EY, f[:9], 1)
    F = rho * o.gbeta * (T + 0.5)
    ref = {"rho": rho, "T": T, "u": jx / rho, "v": (jy - F / 2) / rho}
    eps, cut = np.longdouble(2.0) ** -53, 14 * np.longdouble(2.0) ** -58
    tol = {"rho": cut * top + 2 * eps * np.abs(rho) + eps,
           "T": cut * np.abs(f[9:]).max(axis=0) + eps * np.abs(T),
           "u": (cut * top + 8 * eps * np.abs(jx)) / rho,
           "v": (cut * top + 8 * eps * (np.abs(jy) + np.abs(F))) / rho}
    got = {k: torch.empty((n, n), dtype=torch.float64, device="cuda") for k in ref}
    s.fields_device(**got)
    for k in ref:
        err = np.abs(got[k].cpu().numpy().astype(np.longdouble) - ref[k])
        assert (err <= tol[k]).all(), (k, float((err - tol[k]).max()))
    # the time average of one state is that state, of three equal ones within 2 ulp
    s.average_reset()
    s.average_add()
    avg, count = s.average()
    assert count == 1 and np.array_equal(avg["T"], got["T"].cpu().numpy())
    s.average_add()
    s.average_add()
    avg, count = s.average()
    u = got["u"].cpu().numpy()
    assert count == 3 and (np.abs(avg["u"] - u) <= 4 * 2.0 ** -53 * np.abs(u)).all()
    s.close()


def test_fields_of_a_diverged_state():
    """Infinities and NaN reach the outputs, and the reductions report them."""
    import torch
    n = 40
    xi = pkg.islbm_mesh_tanh(n, 1.5)
    s = pkg.Solver(xi, xi, Ra=1e6, precision="fp32")
    f = np.zeros((14, n, 64), dtype=np.float32)
    f[3, 5, 7] = np.inf
    f[9, 6, 8] = np.nan
    f[0, 9, 9] = -1.0                       # rho = 0
    s.set_rows(0, n, torch.from_numpy(f).cuda())
    got = {k: torch.empty((n, n), dtype=torch.float64, device="cuda") for k in ("rho", "T", "u", "v")}
    s.fields_device(**got)
    got = {k: v.cpu().numpy() for k, v in got.items()}
    assert np.isinf(got["rho"][5, 7]) and not np.isfinite(got["u"][5, 7])
    assert np.isnan(got["T"][6, 8]) and np.isnan(got["v"][6, 8])
    assert got["rho"][9, 9] == 0.0 and not np.isfinite(got["u"][9, 9])
    assert np.isfinite(got["u"]).sum() == n * n - 2
    with pytest.raises(pkg.IslbmError):
        s.reduce()
    assert s.reduce(check=False)["nonfinite"] == 3
    s.close()


@pytest.mark.parametrize("nx,ny,nz", [(4, 4, 0), (31, 31, 0), (65, 65, 0), (64, 64, 0), (1000, 1000, 0),
                                      (9, 9, 9), (34, 34, 34)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_reductions_against_fields(nx, ny, nz, precision):
    """The sums over strips and blocks against FP64 sums of the output fields.
    FP32 node values carry a rounding of 2^-23 each; the sums add 2^-53."""
    shape = (ny, nx) if nz == 0 else (nz, ny, nx)
    xi = pkg.islbm_mesh_tanh(nx, 1.5)
    Ra = 1e5 if nx < 100 else 1e8           # the diffusivity has to fit the mesh
    s = pkg.Solver(*([xi] * (3 if nz else 2)), Ra=Ra, precision=precision)
    rng = np.random.default_rng(nx)
    T = rng.uniform(-0.5, 0.5, shape)
    vel = [0.02 * rng.uniform(-1, 1, shape) for _ in range(3 if nz else 2)]
    s.set_fields(T, *vel)
    fl = s.fields()
    r = s.reduce()
    o = s.info
    X = (xi - xi[0]) / (xi[1] - xi[0])
    W1 = 0.5 * (X[2:] - X[:-2])
    W = W1[:, None] * W1[None, :] if nz == 0 else W1[:, None, None] * W1[:, None] * W1
    u2 = sum(fl[k] ** 2 for k in ("u", "v", "w")[:len(vel)])
    vol = W.sum()
    tol = 1e-5 if precision == "fp32" else 1e-11
    sra = np.sqrt(Ra / 0.71)
    assert abs(r["mass"] / (W * fl["rho"]).sum() - 1) <= tol
    assert abs(r["Re"] / (sra * np.sqrt((W * u2).sum() / vol) / o.u_f) - 1) <= tol
    assert abs(r["Re_mean"] / (sra * (W * np.sqrt(u2)).sum() / vol / o.u_f) - 1) <= tol
    assert abs(r["max_speed"] / (np.sqrt(u2.max()) / o.u_f) - 1) <= tol
    scale = np.sqrt(Ra * 0.71) * (W * np.abs(fl["u"] * (fl["T"] + 0.5))).sum() / (o.u_f * vol)
    nu = np.sqrt(Ra * 0.71) * (W * fl["u"] * (fl["T"] + 0.5)).sum() / (o.u_f * vol) + 1
    assert abs(r["Nu"] - nu) <= tol * scale
    if nz == 0:                              # the centre-line and wall columns
        conv = fl["u"] * (fl["T"] + 0.5)
        m = nx // 2
        line = 0.5 * (conv[:, m - 1] + conv[:, m]) if nx % 2 == 0 else conv[:, m]
        lo, hi = (m - 1, m) if nx % 2 == 0 else (m - 1, m + 1)
        dT = (W1 * (fl["T"][:, hi] - fl["T"][:, lo])).sum() / (X[hi + 1] - X[lo + 1])
        want = (np.sqrt(Ra * 0.71) * (W1 * line).sum() / o.u_f - o.L * dT) / o.L
        big = (np.sqrt(Ra * 0.71) * (W1 * np.abs(line)).sum() / o.u_f
               + o.L * (W1 * (np.abs(fl["T"][:, hi]) + np.abs(fl["T"][:, lo]))).sum()
               / (X[hi + 1] - X[lo + 1])) / o.L
        assert abs(r["Nu_middle"] - want) <= tol * big
    # steady change: none yet, an unchanged state, a changed one
    assert s.steady_change() == (float("inf"), float("inf"))
    assert s.steady_change() == (0.0, 0.0)
    s.step(3)
    du, dT = s.steady_change()
    now = s.fields()
    names = ("u", "v", "w")[:len(vel)]
    d = np.sqrt(sum((now[k] - fl[k]) ** 2 for k in names)).sum()
    u0 = np.sqrt(sum(fl[k] ** 2 for k in names)).sum()
    # each term within 4 ulp, fields against the snapshot bit for bit
    assert abs(du / (d / u0) - 1) <= 1e-11
    assert abs(dT / (np.abs(now["T"] - fl["T"]).sum() / np.abs(fl["T"] + 0.5).sum()) - 1) <= 1e-11
    s.close()
