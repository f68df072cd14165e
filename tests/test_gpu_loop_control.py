"""The loop control inside the residual kernels and the graph of passes: the
reported residual with one block, around a full group of blocks and over
several groups, on register and shared-memory lengths; the stopping pass
around the first graph; a plan called twice with other fields and arguments."""
import numpy as np
import pytest

import oracle.pressure_oracle as orc
from paper_2005_11806_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _fields(dims, seed):
    nx, ny, nz = dims
    lz = 0.03 * nz
    zf = wl.uniform_zfaces(nz, lz)
    g = orc.Grid(nx, ny, nz, 1.0, ny / nx, zf)
    rng = np.random.default_rng(seed)
    rho = np.where(rng.random(g.shape) < 0.3, 1.0, 6.0)
    us, vs, ws = wl.random_faces(nx, ny, nz, 0.1, seed)
    return g, zf, lz, us, vs, ws, rho


def _run(plan, g, us, vs, ws, rho, **kw):
    from paper_2005_11806_gb300 import pressure as pp
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    p = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    u, v = torch.empty_like(p), torch.empty_like(p)
    w = torch.empty((g.nz + 1, g.ny, g.nx), dtype=torch.float64, device="cuda")
    info = pp.pressure_correct(plan.handle, dev(us), dev(vs), dev(ws), dev(rho), None, 1e-3, p, u, v, w,
                               allow_not_converged=True, **kw)
    return info, p.cpu().numpy()


# 32 x 8 rows: eight rows a block while the grid is small, so nz blocks
@pytest.mark.parametrize("dims", [(32, 8, 1), (32, 8, 127), (32, 8, 128), (32, 8, 129), (32, 8, 257), (32, 5, 40),
                                  (18, 6, 5), (18, 8, 150), (320, 4, 70)])
def test_reported_residual(dims):
    from paper_2005_11806_gb300 import pressure as pp
    g, zf, lz, us, vs, ws, rho = _fields(dims, 3)
    plan = pp.Plan(*dims, 1.0, dims[1] / dims[0], lz, zfaces=zf)
    info, p = _run(plan, g, us, vs, ws, rho, rtol=0.0, maxit=3)
    ref = orc.method3(g, us, vs, ws, rho, np.zeros(g.shape), 1e-3, rtol=0.0, maxit=3)
    assert info["iters"] == 3
    assert info["res_final"] == pytest.approx(ref[4]["res_hist"][-1], rel=1e-9)
    assert info["res0"] == pytest.approx(ref[4]["res0"], rel=1e-12)
    assert np.linalg.norm(p - ref[0]) <= 1e-11 * np.linalg.norm(ref[0])


@pytest.mark.parametrize("maxit", [0, 1, 7, 8, 9, 11, 12, 13, 16, 21])
def test_pass_counts_around_graphs(maxit):
    from paper_2005_11806_gb300 import pressure as pp
    dims = (32, 6, 9)
    g, zf, lz, us, vs, ws, rho = _fields(dims, 4)
    plan = pp.Plan(*dims, 1.0, dims[1] / dims[0], lz, zfaces=zf)
    for seed in (4, 5):  # the second call updates the first one's graph
        _, _, _, us, vs, ws, rho = _fields(dims, seed)
        info, p = _run(plan, g, us, vs, ws, rho, rtol=0.0, maxit=maxit)
        ref = orc.method3(g, us, vs, ws, rho, np.zeros(g.shape), 1e-3, rtol=0.0, maxit=maxit)
        assert info["iters"] == maxit and info["status"] == pp.PP_ERR_NOT_CONVERGED
        if maxit:
            assert np.linalg.norm(p - ref[0]) <= 1e-11 * np.linalg.norm(ref[0])
    plain = pp.Plan(*dims, 1.0, dims[1] / dims[0], lz, zfaces=zf)
    pp.pressure_profile_enable(plain.handle)  # kernel timing: single launches, the same iterates
    _, q = _run(plain, g, us, vs, ws, rho, rtol=0.0, maxit=maxit)
    assert np.array_equal(p, q)
