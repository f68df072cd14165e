"""The streamed z sweeps (pp_zsweep.cuh) at the edges of their ring: line
lengths around the row group and the group count, odd and single rows in y,
and both forms (one and two columns a thread) of the mixed_z64 solve, against
the oracle's constant solve.  FP64: 1e-11 relative L2, as every FP64 solve;
mixed plans: the FP32 rounding bound of one solve."""
import numpy as np
import pytest

import oracle.pressure_oracle as orc
from paper_2005_11806_gb300 import workloads as wl
from tests.fp32_bounds import mixed_solve_bound

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve_error(dims, precision, ywalls=False):
    from paper_2005_11806_gb300 import pressure as pp
    nx, ny, nz = dims
    lx, ly, lz = 1.0, 0.75, 1.2
    zf = wl.tanh_zfaces(nz, lz, 1.3)
    g = orc.Grid(nx, ny, nz, lx, ly, zf, ywalls=ywalls)
    f = np.random.default_rng(31 * nx + 7 * ny + nz).standard_normal(g.shape)
    ref = orc.solve_constant(g, f)
    plan = pp.Plan(nx, ny, nz, lx, ly, lz, zfaces=zf, precision=precision, ywalls=ywalls)
    p = torch.empty(g.shape, dtype=torch.float64, device="cuda")
    pp.pressure_solve(plan.handle, torch.from_numpy(f).cuda(), p)
    return float(np.linalg.norm(p.cpu().numpy() - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("precision", ["fp64", "mixed_z64", "mixed"])
@pytest.mark.parametrize("nz", [2, 3, 4, 5, 8, 11, 12, 13, 15, 16, 17, 21, 64])
def test_line_lengths(nz, precision):
    for nx, ny, ywalls in ((8, 6, False), (10, 3, False), (16, 1, False), (12, 4, True)):
        err = _solve_error((nx, ny, nz), precision, ywalls)
        assert err < (1e-11 if precision == "fp64" else mixed_solve_bound(nx, ny)), (nx, ny, nz, ywalls)


@pytest.mark.parametrize("dims", [(256, 480, 17), (320, 405, 6), (256, 432, 5)])
def test_column_pairs(dims):
    """Enough columns for two a thread (even and odd ny), and just too few."""
    assert _solve_error(dims, "mixed_z64") < mixed_solve_bound(dims[0], dims[1])
