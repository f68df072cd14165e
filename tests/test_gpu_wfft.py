"""The register transforms of pp_wfft.cuh, every length as x and as y
(periodic and between walls), with row counts that leave warps and blocks
partly filled, against the oracle.  FP64: 1e-11 relative L2, as every FP64
solve; mixed plans: the FP32 rounding bound of one solve."""
import numpy as np
import pytest

import oracle.pressure_oracle as orc
from paper_2005_11806_gb300 import workloads as wl
from tests.fp32_bounds import mixed_solve_bound

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = (32, 36, 40, 48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128, 144, 150, 160, 180, 192, 240, 256)


def _rel(a, b):
    return float(np.linalg.norm((np.asarray(a) - b).ravel()) / np.linalg.norm(b.ravel()))


def _solve_error(dims, precision, ywalls):
    from paper_2005_11806_gb300 import pressure as pp
    nx, ny, nz = dims
    zf = wl.tanh_zfaces(nz, 1.2, 1.3)
    g = orc.Grid(nx, ny, nz, 1.0, 0.75, zf, ywalls=ywalls)
    f = np.random.default_rng(31 * nx + 7 * ny + nz).standard_normal(g.shape)
    plan = pp.Plan(nx, ny, nz, 1.0, 0.75, 1.2, zfaces=zf, precision=precision, ywalls=ywalls)
    p = torch.empty(g.shape, dtype=torch.float64, device="cuda")
    pp.pressure_solve(plan.handle, torch.from_numpy(f).cuda(), p)
    return _rel(p.cpu().numpy(), orc.solve_constant(g, f))


@pytest.mark.parametrize("precision", ["fp64", "mixed_z64"])
@pytest.mark.parametrize("n", LENGTHS)
def test_constant_solve(n, precision):
    for nx, ny, nz, ywalls in ((n, 6, 5, False), (n, 1, 3, False), (8, n, 3, False), (18, n, 2, False),
                               (18, n, 2, True), (n, n, 2, True)):
        bound = 1e-11 if precision == "fp64" else mixed_solve_bound(nx, ny, ywalls=ywalls)
        assert _solve_error((nx, ny, nz), precision, ywalls) < bound, (nx, ny, nz, ywalls)


@pytest.mark.parametrize("ny", [5, 6])
@pytest.mark.parametrize("n", LENGTHS)
def test_projection(n, ny):
    """The residual of the warp kernels: FP64 iterates equal the oracle's, and
    a mixed plan converges to the same fields (exact and updated residuals,
    even and odd ny)."""
    from paper_2005_11806_gb300 import pressure as pp
    nz = 4
    zf = wl.tanh_zfaces(nz, 0.1, 1.2)
    g = orc.Grid(n, ny, nz, 1.0, ny / n, zf)
    rng = np.random.default_rng(n + ny)
    rho = np.where(rng.random(g.shape) < 0.3, 1.0, 8.0)
    us, vs, ws = wl.random_faces(n, ny, nz, 0.1, 5)
    S = -0.01 * (rho < 2.0)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731

    def run(precision, **kw):
        plan = pp.Plan(n, ny, nz, 1.0, ny / n, 0.1, zfaces=zf, precision=precision)
        p = torch.empty(g.shape, dtype=torch.float64, device="cuda")
        u, v = torch.empty_like(p), torch.empty_like(p)
        w = torch.empty((nz + 1, ny, n), dtype=torch.float64, device="cuda")
        pp.pressure_correct(plan.handle, dev(us), dev(vs), dev(ws), dev(rho), dev(S), 1e-3, p, u, v, w, **kw)
        return [t.cpu().numpy() for t in (p, u, v, w)]

    ref = orc.method3(g, us, vs, ws, rho, S, 1e-3, rtol=0.0, maxit=6)[:4]
    for a, b in zip(run("fp64", rtol=0.0, maxit=6, allow_not_converged=True), ref):
        assert _rel(a, b) < 1e-11
    full = orc.method3(g, us, vs, ws, rho, S, 1e-3, rtol=1e-13, maxit=5000)[1:4]
    for a, b in zip(run("mixed_z64", rtol=1e-11, maxit=5000)[1:], full):
        assert _rel(a, b) < 1e-9
