"""Host threads: one projects while another waits for the device; and the graph
of passes, built from kernel nodes, against single launches for every kernel
that a pass can hold."""
import threading
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(dims, stream=0, seed=1, yfaces=None, **kw):
    """A plan and a call that runs a projection of maxit passes on it."""
    from paper_2005_11806_gb300 import pressure as pp
    nx, ny, nz = dims
    if yfaces is not None:
        kw["yfaces"] = yfaces
    plan = pp.Plan(nx, ny, nz, 1.0, ny / nx, 0.03 * nz, stream=stream, **kw)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    field = lambda *s: torch.rand(*s, dtype=torch.float64, device="cuda", generator=g)  # noqa: E731
    rho = torch.where(field(nz, ny, nx) < 0.3, 1.0, 6.0).double()
    us, vs, ws = field(nz, ny, nx), field(nz, ny, nx), field(nz + 1, ny, nx)
    p = torch.zeros_like(rho)
    out = [torch.empty_like(us), torch.empty_like(vs), torch.empty_like(ws)]
    torch.cuda.synchronize()

    def call(maxit):
        info = pp.pressure_correct(plan.handle, us, vs, ws, rho, None, 1e-3, p, *out, rtol=0.0, maxit=maxit,
                                   allow_not_converged=True)
        assert info["iters"] == maxit
    return plan, call, p


def _together(calls, seconds):
    """Runs each call over and over in a thread of its own; returns the errors and the counts."""
    stop, errors, counts = threading.Event(), [], [0] * len(calls)

    def loop(i):
        try:
            while not stop.is_set():
                calls[i]()
                counts[i] += 1
        except Exception as e:  # noqa: BLE001 - reported by the test
            errors.append((i, repr(e)))
    threads = [threading.Thread(target=loop, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    end = time.monotonic() + seconds
    while time.monotonic() < end and not errors:
        time.sleep(0.02)
    stop.set()
    for t in threads:
        t.join(60)
        assert not t.is_alive()
    return errors, counts


def test_device_wait_in_another_thread():
    stream = torch.cuda.Stream()
    plan, call, p = _case((32, 32, 32), stream.cuda_stream)
    call(20)
    torch.cuda.synchronize()
    first = p.clone()
    torch.cuda.synchronize()
    errors, counts = _together([lambda: call(20), torch.cuda.synchronize], 4.0)
    assert not errors and min(counts) > 100
    torch.cuda.synchronize()
    assert torch.equal(first, p)
    plan.close()


_yf = np.cumsum([0.0] + [1.0 + 0.1 * j for j in range(21)])
_GRAPHS = [
    ((32, 20, 9), dict(precision="fp64")),            # x in registers, y by shared-memory passes
    ((18, 32, 9), dict(precision="fp64")),            # the other way round
    ((18, 32, 9), dict(precision="mixed_z64")),
    ((32, 48, 9), dict(precision="mixed_z64", ywalls=True)),
    ((32, 20, 9), dict(precision="fp64", ywalls=True)),
    ((32, 20, 9), dict(precision="mixed_z64", ywalls=True)),
    ((32, 32, 40), dict(precision="mixed")),
    ((32, 32, 40), dict(precision="mixed_tc")),
    ((512, 6, 5), dict(precision="mixed_z64")),
    ((32, 512, 4), dict(precision="mixed_z64")),
    ((512, 6, 5), dict(precision="fp64")),
    ((32, 21, 8), dict(precision="fp64", ywalls=True, yfaces=_yf * (21 / 32 / _yf[-1]))),
    ((32, 21, 8), dict(precision="mixed_z64", ywalls=True, yfaces=_yf * (21 / 32 / _yf[-1]))),
    ((32, 20, 16), dict(precision="fp64", cosine=True)),
]


@pytest.mark.parametrize("dims,kw", _GRAPHS)
def test_graph_equals_single_launches(dims, kw):
    from paper_2005_11806_gb300 import pressure as pp
    kw = dict(kw)
    cosine = kw.pop("cosine", False)
    found = []
    for profile in (False, True):  # kernel timing keeps single launches
        plan, call, p = _case(dims, seed=7, **kw)
        if cosine:
            pp.pressure_plan_set_zsolve(plan.handle, "cosine")
        if profile:
            pp.pressure_profile_enable(plan.handle)
        call(14)
        call(17)  # updates the graph of the first call
        torch.cuda.synchronize()
        found.append(p.clone())
        plan.close()
    assert torch.equal(found[0], found[1])
    assert torch.isfinite(found[0]).all() and found[0].abs().max() > 0


def test_two_plans_with_other_shared_memory():
    """Two threads whose plans take the same y kernel with 76.8 and 96 KB of shared memory."""
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    cases = [_case((16, ny, 8), s.cuda_stream, precision="fp64") for ny, s in zip((200, 250), streams)]
    errors, counts = _together([lambda c=c: c[1](3) for c in cases], 4.0)
    assert not errors and min(counts) > 100
    for plan, _, _ in cases:
        plan.close()
