"""The marching predictor at the edges of its tiles (30 cells of a row a warp)
and chunks of layers, periodic and walled y, with a force and a history,
against the oracle (1e-12 relative L2, as the other predictor tests)."""
import numpy as np
import pytest

import oracle.pressure_oracle as orc
from paper_2005_11806_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ywalls", [False, True])
@pytest.mark.parametrize("dims", [(8, 4, 2), (30, 4, 3), (32, 2, 4), (36, 6, 5), (60, 4, 8), (90, 4, 9), (96, 2, 65),
                                  (240, 40, 70)])
def test_tiles_and_chunks(dims, ywalls):
    from paper_2005_11806_gb300 import pressure as pp
    nx, ny, nz = dims
    zf = wl.tanh_zfaces(nz, 1.0, 1.4)
    g = orc.Grid(nx, ny, nz, 1.0, ny / nx, zf, ywalls=ywalls)
    rng = np.random.default_rng(nx + nz)
    u, v, w = wl.random_faces(nx, ny, nz, 1.0, 11, ywalls=ywalls)
    rho, mu = 1.0 + 9.0 * rng.random(g.shape), 0.1 + rng.random(g.shape)
    force = wl.random_faces(nx, ny, nz, 1.0, 21, ywalls=ywalls)
    prev = wl.random_faces(nx, ny, nz, 1.0, 31, ywalls=ywalls)
    grav = (0.3, -0.2, -9.81)
    ref, ref_ru = orc.predictor(g, u, v, w, rho, mu, grav, 1e-3, 1.3e-3, prev, force)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    plan = pp.Plan(nx, ny, nz, 1.0, ny / nx, 1.0, zfaces=zf, ywalls=ywalls)
    star, ru = ([torch.full(a.shape, float("nan"), dtype=torch.float64, device="cuda") for a in (u, v, w)]
                for _ in range(2))
    pp.pressure_predictor(plan.handle, dev(u), dev(v), dev(w), dev(rho), dev(mu), grav, 1e-3, star, dt_old=1.3e-3,
                          ru_prev=[dev(a) for a in prev], ru_out=ru, force=[dev(a) for a in force])
    for a, b in zip(star + ru, list(ref) + list(ref_ru)):
        assert np.linalg.norm(a.cpu().numpy() - b) <= 1e-12 * np.linalg.norm(b)
