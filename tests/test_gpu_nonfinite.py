"""Inf and NaN in the input reach the caller, whatever form the z sweeps give
them: a projection ends with the numeric error, a plain solve leaves no value
finite.  The plan serves the next call as before."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# a register and a shared-memory length; 40 layers: the decay away from a bad row is long over
PLANS = [((32, 32, 40), "mixed_z64"), ((18, 20, 40), "mixed_z64"), ((32, 32, 40), "fp64"), ((32, 32, 40), "mixed"),
         ((32, 512, 4), "mixed_z64")]


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf"), 1e200])
@pytest.mark.parametrize("dims,precision", PLANS)
def test_bad_value_reaches_the_caller(dims, precision, bad):
    from paper_2005_11806_gb300 import pressure as pp
    if precision == "fp64" and bad == 1e200:
        bad = float("nan")
    nx, ny, nz = dims
    plan = pp.Plan(nx, ny, nz, 1.0, ny / nx, 0.03 * nz, precision=precision)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    field = lambda *s: torch.rand(*s, dtype=torch.float64, device="cuda", generator=g) - 0.5  # noqa: E731
    f = field(nz, ny, nx)
    good = torch.empty_like(f)
    pp.pressure_solve(plan.handle, f, good)
    p = torch.empty_like(f)
    for k in (0, nz // 2, nz - 1):
        h = f.clone()
        h[k, ny // 3, nx // 5] = bad
        pp.pressure_solve(plan.handle, h, p)
        assert not torch.isfinite(p).any()
    rho = torch.where(field(nz, ny, nx) < 0.0, 1.0, 6.0).double()
    us, vs, ws = field(nz, ny, nx), field(nz, ny, nx), field(nz + 1, ny, nx)
    us[nz // 2, ny // 3, nx // 5] = bad
    u, v, w = torch.empty_like(us), torch.empty_like(vs), torch.empty_like(ws)
    with pytest.raises(pp.PressureError) as e:
        pp.pressure_correct(plan.handle, us, vs, ws, rho, None, 1e-3, p, u, v, w, rtol=1e-10, maxit=50)
    assert e.value.code == pp.PP_ERR_NUMERIC
    pp.pressure_solve(plan.handle, f, p)
    assert torch.equal(p, good)
    plan.close()
