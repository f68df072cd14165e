"""Device memory of a plan: an FP64 plan holds no more than its fields, its
spectrum and two full tables of the z solve, also where walls in y leave the
tables no shared columns."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ywalls", [False, True])
def test_fp64_plan_bytes(ywalls):
    from paper_2005_11806_gb300 import pressure as pp
    nx, ny, nz = 256, 256, 256
    cells, columns = nx * ny * nz, (nx // 2 + 1) * ny * nz
    make = lambda: pp.Plan(nx, ny, nz, 1.0, 1.0, 1.0, precision="fp64", ywalls=ywalls)  # noqa: E731
    make().close()  # the kernels' code is loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plan = make()
    used = before - torch.cuda.mem_get_info()[0]
    plan.close()
    # spectrum 16 B and tables 2 x 8 B a column; right-hand side, three face
    # coefficients, diagonal (8 B each) and 4 B a cell; up to 2 MB of rounding
    # for each of at most twelve allocations
    assert used <= 32 * columns + (5 * 8 + 4) * cells + 12 * (2 << 20)
