"""Forms of the register transforms that walls in y bring: the cosine
transform of a batch (two tiles a block for the lengths with 8 threads a
line, one for those with 16; the last block half filled), and the residual of
a stretched y with an odd number of rows."""
import numpy as np
import pytest

import oracle.pressure_oracle as orc
from paper_2005_11806_gb300 import workloads as wl
from tests import test_gpu_batch as tb
from tests import test_gpu_ystretch as ts

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# nx = 32 and 36: 3 tiles of 8 columns a plane, an odd number of tiles with odd nz
@pytest.mark.parametrize("dims", [[(32, 32, 13), (32, 48, 11)], [(16, 100, 9), (36, 144, 5)],
                                  [(32, 32, 13), (16, 100, 9), (24, 20, 18), (18, 64, 7)]])
def test_batch_cosine_matches_single_grid_plans(dims):
    """A fixed pass count; the tolerance is that of the other batch tests (the same arithmetic on both sides)."""
    from paper_2005_11806_gb300 import pressure as pp
    cases = []
    for i, (nx, ny, nz) in enumerate(dims):
        w = wl.channel_bubble_case(nx, ny, nz, seed=1400 + i, rho_ratio=1000.0, stretched=i % 2 == 0)
        cases.append((w, orc.mixture_density(w.phi, w.rho_g, w.rho_l)))
    infos, res = tb._run_batch(pp, cases, 0.0, 25)
    for k, (w, rho) in enumerate(cases):
        assert infos[k]["iters"] == 25
        plan = pp.Plan(w.nx, w.ny, w.nz, w.lx, w.ly, float(w.zf[-1]), zfaces=w.zf, precision="mixed",
                       ywalls=w.ywalls)
        p = torch.empty(w.shape, dtype=torch.float64, device="cuda")
        u, v = torch.empty_like(p), torch.empty_like(p)
        ww = torch.empty((w.nz + 1, w.ny, w.nx), dtype=torch.float64, device="cuda")
        pp.pressure_correct(plan.handle, ts.dev(w.us), ts.dev(w.vs), ts.dev(w.ws), ts.dev(rho), ts.dev(w.S), w.dt, p,
                            u, v, ww, rtol=0.0, maxit=25, allow_not_converged=True)
        for got, ref in zip(res[k], (p, u, v, ww)):
            assert tb._rel(got, ref.cpu().numpy()) < 1e-12, k
        assert np.all(res[k][2][:, 0, :] == 0.0)
        plan.close()


@pytest.mark.parametrize("precision", ["mixed", "mixed_z64", "mixed_tc"])
def test_stretched_odd_rows_vs_oracle(precision):
    """Tolerances of the stretched-y tests of mixed plans."""
    from paper_2005_11806_gb300 import pressure as pp
    w, rho = ts._case(32, 21, 18, ratio=10.0)
    g = ts._grid(w)
    _, u0, v0, w0, _ = orc.method3(g, w.us, w.vs, w.ws, rho, w.S, w.dt, rtol=1e-12, maxit=8000)
    info, p, u, v, ww = ts._run(pp, w, rho, precision, rtol=1e-10, maxit=8000)
    assert info["status"] == 0 and info["res_final"] <= 1e-10
    Sc = w.S - orc.volume_mean(g, w.S)
    d0 = orc.divergence(g, w.us, w.vs, w.ws) - Sc
    assert np.linalg.norm(orc.divergence(g, u, v, ww) - Sc) <= 1e-10 * np.linalg.norm(d0) * 1.0001
    assert max(ts._rel(a, b) for a, b in ((u, u0), (v, v0), (ww, w0))) < 1e-9
    assert np.all(v[:, 0, :] == 0.0)
