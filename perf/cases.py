"""The calls whose speed is followed from change to change.

Each case is one call (or one time step's calls) of a low-Mach two-phase flow
solver that uses this library, through the public entry points of
``paper_2005_11806_gb300``: sizes, boundary conditions, precisions and density
ratios are those of the repository's configurations, tests and benchmark.
Inputs are drawn on the GPU from the seed; ``exact`` computes what a case
returns in 64 bits with plain torch (conjugate gradients on the symmetric
form of the variable-coefficient equation, dense or Fourier eigenbases).
"""
import math

import numpy as np
import torch

from paper_2005_11806_gb300 import autograd
from paper_2005_11806_gb300 import pressure as pp

DT = 1e-3
GAMMA, P0, DP0DT = 1.4, 1.0, 1e-2
GRAVITY = (0.1, -0.2, -0.981)
RTOL, MAXIT = 1e-12, 50000     # the tolerance the tests and autograd.project converge to


def listed():
    def project(name, nx, ny, nz, precision, y="periodic", zbeta=1.5, ratio=100.0, bubbles=3):
        return dict(name=name, kind="project", nx=nx, ny=ny, nz=nz, precision=precision, y=y, zbeta=zbeta,
                    ratio=ratio, bubbles=bubbles)

    return [
        # the smallest call: one constant-coefficient solve (e.g. a preconditioner or a single-phase step)
        dict(name="solve_fp64_32", kind="solve", nx=32, ny=32, nz=32, precision="fp64", y="periodic", zbeta=0.0),
        # a small projection in full precision: parameter studies, regression runs
        project("project_fp64_32", 32, 32, 32, "fp64", zbeta=0.0, ratio=1000.0, bubbles=1),
        # a rising bubble at moderate resolution, full precision, liquid/gas ratio of water and air
        project("project_fp64_128", 128, 128, 128, "fp64", zbeta=0.0, ratio=833.0, bubbles=1),
        # the single-sphere configuration with the benchmark's precision
        project("project_z64_256", 256, 256, 256, "mixed_z64", zbeta=0.0, ratio=833.0, bubbles=1),
        # the benchmark's bubble swarm at full size, at the largest ratio the method was published for
        project("project_z64_512", 512, 512, 512, "mixed_z64", ratio=10.0, bubbles=200),
        # a box whose lengths have factors 3 and 5, hybrid z solve
        project("project_mixed_ragged", 192, 160, 144, "mixed", ratio=100.0, bubbles=8),
        # a duct: walls in y, uniform spacing
        project("duct_z64_walls", 256, 192, 128, "mixed_z64", y="walls", ratio=100.0, bubbles=5),
        # a duct resolved at its walls: stretched y (dense eigenbasis on the tensor cores)
        project("duct_z64_stretched", 256, 200, 128, "mixed_z64", y="stretched", ratio=100.0, bubbles=5),
        # training or data assimilation: projection and its gradient (u*, rho) through autograd
        dict(name="gradient_fp64", kind="gradient", nx=128, ny=128, nz=64, precision="fp64", y="periodic", zbeta=2.0,
             ratio=100.0, bubbles=4),
        # data generation: many independent grids of uneven sizes in one call
        dict(name="batch_mixed", kind="batch", grids=12, smallest=64, largest=192, ratio=100.0),
        # the explicit part of a time step: predictor with its history, pressure rate and divergence source
        dict(name="explicit_256", kind="explicit", nx=256, ny=256, nz=256, zbeta=1.5, ratio=833.0, bubbles=4),
        # one whole time step of a stretched, ragged box
        dict(name="step_z64", kind="step", nx=240, ny=192, nz=180, precision="mixed_z64", zbeta=1.5, ratio=10.0,
             bubbles=8),
    ]


_LENGTHS = [n for n in range(8, 513, 2) if not [1 for q in (7, 11, 13, 17, 19) if n % q == 0]
            and max([q for q in range(2, n + 1) if n % q == 0 and all(q % r for r in range(2, int(q ** 0.5) + 1))]) <= 5]


def _box(rng, lo, hi, most=512):
    """nx, ny (even, factors 2, 3, 5) and nz (any) of a box of lo .. hi cells, drawn over the logarithm."""
    while True:
        cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        edge = cells ** (1 / 3)
        nx = min(_LENGTHS, key=lambda n: abs(math.log(n / (edge * math.exp(rng.uniform(-0.6, 0.6))))))
        ny = min(_LENGTHS, key=lambda n: abs(math.log(n / (edge * math.exp(rng.uniform(-0.6, 0.6))))))
        nz = int(round(cells / (nx * ny)))
        if 8 <= nz <= most and nx <= most and ny <= most:
            return nx, ny, nz


def draw(rng):
    kind = rng.choice(["solve", "project", "project", "project", "duct", "gradient", "batch", "explicit", "step"])
    zbeta = rng.choice([0.0, round(rng.uniform(1.0, 2.0), 2)])
    ratio = round(math.exp(rng.uniform(math.log(3.0), math.log(100.0))), 1)
    bubbles = rng.randint(1, 6)
    if kind == "batch":
        lo = rng.choice([32, 48, 64])
        return dict(kind="batch", grids=rng.randint(2, 20), smallest=lo, largest=rng.choice([96, 128, 160]), ratio=ratio)
    if kind == "solve":
        nx, ny, nz = _box(rng, 16 ** 3, 256 ** 3)
        return dict(kind="solve", nx=nx, ny=ny, nz=nz, precision="fp64", y=rng.choice(["periodic", "walls"]), zbeta=zbeta)
    if kind == "explicit":
        nx, ny, nz = _box(rng, 16 ** 3, 256 ** 3)
        return dict(kind="explicit", nx=nx, ny=ny, nz=nz, zbeta=zbeta, ratio=ratio, bubbles=bubbles)
    if kind == "gradient":
        nx, ny, nz = _box(rng, 16 ** 3, 80 ** 3)
        return dict(kind="gradient", nx=nx, ny=ny, nz=nz, precision="fp64", y="periodic", zbeta=zbeta, ratio=ratio,
                    bubbles=bubbles)
    if kind == "step":
        nx, ny, nz = _box(rng, 32 ** 3, 200 ** 3)
        return dict(kind="step", nx=nx, ny=ny, nz=nz, precision=rng.choice(["mixed_z64", "mixed"]), zbeta=zbeta,
                    ratio=ratio, bubbles=bubbles)
    if kind == "duct":
        nx, ny, nz = _box(rng, 24 ** 3, 200 ** 3)
        return dict(kind="project", nx=nx, ny=ny, nz=nz, precision=rng.choice(["mixed_z64", "mixed"]),
                    y=rng.choice(["walls", "stretched"]), zbeta=zbeta, ratio=min(ratio, 50.0), bubbles=bubbles)
    precision = rng.choice(["mixed_z64", "mixed_z64", "mixed", "fp64"])
    nx, ny, nz = _box(rng, 16 ** 3, 96 ** 3 if precision == "fp64" else 288 ** 3)
    return dict(kind="project", nx=nx, ny=ny, nz=nz, precision=precision, y="periodic", zbeta=zbeta, ratio=ratio,
                bubbles=bubbles)


# ---- inputs ------------------------------------------------------------------------------------

def _tanh_faces(n, length, beta):
    if beta <= 0:
        return np.linspace(0.0, length, n + 1)
    xi = np.arange(n + 1) / n
    f = 0.5 * length * (1.0 + np.tanh(beta * (2.0 * xi - 1.0)) / math.tanh(beta))
    f[0], f[-1] = 0.0, length
    return f


def _geometry(case):
    """Lengths (cubic cells before stretching, lx = 1) and face coordinates."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    y = case.get("y", "periodic")
    g = dict(nx=nx, ny=ny, nz=nz, lx=1.0, ly=ny / nx, lz=nz / nx, ywalls=y != "periodic")
    g["zf"] = _tanh_faces(nz, g["lz"], case.get("zbeta", 0.0))
    g["yf"] = _tanh_faces(ny, g["ly"], 1.5) if y == "stretched" else None
    return g


def _gas_fraction(g, bubbles, seed):
    """Volume fraction of non-overlapping gas spheres, each cell sampled at 4 x 4 x 4 points."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nx, ny, nz, h = g["nx"], g["ny"], g["nz"], g["lx"] / g["nx"]
    least = min(g["lx"], g["ly"], g["lz"])
    lo, hi = (0.008, 0.019) if bubbles > 50 else (0.08, 0.16)
    yf = np.linspace(0.0, g["ly"], ny + 1) if g["yf"] is None else g["yf"]
    placed = []
    for _ in range(400 * bubbles):
        if len(placed) == bubbles:
            break
        r = rng.uniform(lo, hi) * least
        c = np.array([rng.uniform(0, g["lx"]), rng.uniform(r + h, g["ly"] - r - h), rng.uniform(r + h, g["lz"] - r - h)])
        c[0] = min(max(c[0], r + h), g["lx"] - r - h)
        if all(np.linalg.norm(c - q) > r + s + 2 * h for q, s in placed):
            placed.append((c, r))
    phi = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    off = (np.arange(4) + 0.5) / 4
    for c, r in placed:
        box, pts = [], []
        for faces, q in ((g["zf"], c[2]), (yf, c[1]), (np.linspace(0.0, g["lx"], nx + 1), c[0])):
            a = max(int(np.searchsorted(faces, q - r)) - 1, 0)
            b = min(int(np.searchsorted(faces, q + r)) + 1, len(faces) - 1)
            box.append(slice(a, b))
            s = faces[a:b, None] + off[None, :] * (faces[a + 1:b + 1] - faces[a:b])[:, None] - q
            pts.append(torch.from_numpy((s * s).reshape(-1)).cuda())
        inside = (pts[0][:, None, None] + pts[1][None, :, None] + pts[2][None, None, :] <= r * r).double()
        n = [len(p) // 4 for p in pts]
        phi[box[0], box[1], box[2]] += inside.view(n[0], 4, n[1], 4, n[2], 4).mean(dim=(1, 3, 5))
    return phi.clamp_(max=1.0)


def _faces(g, gen, sigma):
    """Random face velocities, no flow through the walls."""
    s = (g["nz"], g["ny"], g["nx"])
    u, v = (sigma * torch.randn(s, dtype=torch.float64, device="cuda", generator=gen) for _ in range(2))
    w = sigma * torch.randn((s[0] + 1,) + s[1:], dtype=torch.float64, device="cuda", generator=gen)
    w[0] = 0.0
    w[-1] = 0.0
    if g["ywalls"]:
        v[:, 0] = 0.0
    return u, v, w


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _two_phase(case, g, seed):
    """(gas fraction, density, random face velocities, divergence source) of a projection."""
    phi = _gas_fraction(g, case["bubbles"], seed)
    if case["kind"] == "gradient":
        phi = 1.0 - phi     # liquid drops in gas
    rho = phi + case["ratio"] * (1.0 - phi)
    u, v, w = _faces(g, _generator(seed), 0.1)
    return phi, rho, u, v, w, phi * (-DP0DT / (GAMMA * P0))


def _flow(case, g, seed):
    """Fields of one explicit step: a smooth flow with small-scale noise, gas properties from the fraction."""
    phi, rho, u, v, w, _ = _two_phase(case, g, seed)
    x, y, z = (torch.arange(n, dtype=torch.float64, device="cuda") / n for n in (g["nx"], g["ny"], g["nz"]))
    sx, sy, sz = torch.sin(2 * math.pi * x), torch.sin(2 * math.pi * y), torch.sin(math.pi * z)
    u = 0.1 * u + sy[None, :, None] * sz[:, None, None]
    v = 0.1 * v + sx[None, None, :] * sz[:, None, None]
    w = 0.1 * w
    mu = 1.8e-2 * phi + 1.0 * (1.0 - phi)
    kc = 0.05 * phi + 1.0 * (1.0 - phi)
    T = 1.0 + 0.1 * sx[None, None, :] * sy[None, :, None] + 0.2 * torch.cos(math.pi * z)[:, None, None] + 0.0 * phi
    ru = _faces(g, _generator(seed + 1), 0.1)
    return dict(phi=phi, rho=rho, mu=mu, kc=kc, T=T.contiguous(), vel=(u.contiguous(), v.contiguous(), w.contiguous()),
                ru=ru)


def _batch_grids(case):
    rng = np.random.Generator(np.random.PCG64(case["grids"]))
    sizes = [n for n in (32, 48, 64, 96, 128, 160, 192) if case["smallest"] <= n <= case["largest"]]
    out = []
    for _ in range(case["grids"]):
        n = int(sizes[rng.integers(0, len(sizes))])
        nz = int(math.ceil(n * rng.uniform(1.0, 2.0) / 8.0) * 8)
        out.append(dict(nx=n, ny=n, nz=nz, lx=1.0, ly=1.0, lz=nz / n, ywalls=False, zf=np.linspace(0, nz / n, nz + 1),
                        yf=None))
    return out


def _batch_fields(case, seed):
    per = []
    for k, g in enumerate(_batch_grids(case)):
        drop = _gas_fraction(g, 1, 1000 * seed + k)
        gen = _generator(1000 * seed + k)
        per.append((g, case["ratio"] * drop + (1.0 - drop), _faces(g, gen, 1.0)))
    return per


def _empty(g):
    p, u, v = (torch.empty((g["nz"], g["ny"], g["nx"]), dtype=torch.float64, device="cuda") for _ in range(3))
    return p, u, v, torch.empty((g["nz"] + 1, g["ny"], g["nx"]), dtype=torch.float64, device="cuda")


def _plan(case, g):
    return pp.Plan(g["nx"], g["ny"], g["nz"], g["lx"], g["ly"], g["lz"], zfaces=g["zf"],
                   precision=case.get("precision", "fp64"), ywalls=g["ywalls"], yfaces=g["yf"])


def prepare(case, seed):
    kind, st = case["kind"], dict(kind=case["kind"])
    if kind == "batch":
        per = _batch_fields(case, seed)
        st["batch"] = pp.Batch([dict(nx=g["nx"], ny=g["ny"], nz=g["nz"], lx=g["lx"], ly=g["ly"], lz=g["lz"], zfaces=g["zf"])
                                for g, _, _ in per])
        st["rho"] = torch.cat([r.reshape(-1) for _, r, _ in per])
        st["us"], st["vs"], st["ws"] = (torch.cat([f[q].reshape(-1) for _, _, f in per]) for q in range(3))
        st["S"] = torch.zeros_like(st["rho"])
        st["p"], st["u"], st["v"], st["w"] = (torch.empty_like(st[k]) for k in ("rho", "us", "vs", "ws"))
        return st
    g = _geometry(case)
    st["plan"] = _plan(case, g)
    st["out"] = _empty(g)
    if kind == "solve":
        st["f"] = torch.randn((g["nz"], g["ny"], g["nx"]), dtype=torch.float64, device="cuda", generator=_generator(seed))
    elif kind == "project":
        _, st["rho"], st["us"], st["vs"], st["ws"], st["S"] = _two_phase(case, g, seed)
    elif kind == "gradient":
        _, st["rho"], st["us"], st["vs"], st["ws"], _ = _two_phase(case, g, seed)
        for k in ("rho", "us", "vs", "ws"):
            st[k].requires_grad_(True)
        st["cot"] = _faces(g, _generator(seed + 7), 1.0)
    else:
        st.update(_flow(case, g, seed))
        st["star"], st["ru_out"], st["S"] = _empty(g)[1:], _empty(g)[1:], torch.empty_like(st["phi"])
        st["ratio"] = case["ratio"]
        st["dens"] = torch.empty_like(st["phi"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        st["batch"].correct(st["us"], st["vs"], st["ws"], st["rho"], st["S"], DT, st["p"], st["u"], st["v"], st["w"],
                            rtol=RTOL, maxit=MAXIT)
        return [st["p"], st["u"], st["v"], st["w"]]
    plan = st["plan"].handle
    p, u, v, w = st["out"]
    if kind == "solve":
        pp.pressure_solve(plan, st["f"], p)
        return [p]
    if kind == "project":
        pp.pressure_correct(plan, st["us"], st["vs"], st["ws"], st["rho"], st["S"], DT, p, u, v, w, rtol=RTOL,
                            maxit=MAXIT)
        return [p, u, v, w]
    if kind == "gradient":
        ins = [st["us"], st["vs"], st["ws"], st["rho"]]
        un, vn, wn, pn = autograd.project(*ins, st["plan"], dt=DT, rtol=RTOL, maxit=MAXIT)
        grads = torch.autograd.grad([un, vn, wn], ins, grad_outputs=list(st["cot"]))
        return [pn, un, vn, wn, *grads]
    vel, rho = st["vel"], st["rho"]
    if kind == "step":
        pp.pressure_mixture_density(plan, st["phi"], 1.0, st["ratio"], st["dens"])
        rho = st["dens"]
    rp = pp.pressure_p0_rate(plan, st["phi"], st["kc"], st["T"], *vel, P0, GAMMA)
    rate = pp.pressure_dp0dt_extrapolate(rp, 0.5 * rp, DT, 0.8 * DT)
    pp.pressure_divergence_source(plan, st["phi"], st["kc"], st["T"], P0, GAMMA, rate, st["S"])
    pp.pressure_predictor(plan, *vel, rho, st["mu"], GRAVITY, DT, st["star"], dt_old=0.8 * DT, ru_prev=st["ru"],
                          ru_out=st["ru_out"])
    if kind == "explicit":
        return [rp, st["S"], *st["star"], *st["ru_out"]]
    pp.pressure_correct(plan, *st["star"], rho, st["S"], DT, p, u, v, w, rtol=RTOL, maxit=MAXIT)
    return [rp, st["S"], p, u, v, w]


# ---- work --------------------------------------------------------------------------------------

def _passes(case):
    """About how many constant-coefficient solves the iteration needs at this density ratio."""
    return 45.0 * max(1.0, case["ratio"] / 10.0) ** 0.5


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = sum(g["nx"] * g["ny"] * g["nz"] for g in _batch_grids(case))
        line = 5.0 * 4 * math.log2(case["largest"])
        return dict(bytes=72.0 * n, flops=_passes(case) * n * (line + 40.0))
    n = case["nx"] * case["ny"] * case["nz"]
    solve = 5.0 * (math.log2(case["nx"]) + math.log2(case["ny"])) * 2 + 10.0   # transforms there and back, z solve
    if kind == "solve":
        return dict(bytes=16.0 * n, flops=n * solve)
    if kind == "project":   # u*, rho, S in; p, u out; a residual of 25 flops a pass
        return dict(bytes=72.0 * n, flops=n * _passes(case) * (solve + 25.0))
    if kind == "gradient":  # and the cotangents in, the gradients out
        return dict(bytes=136.0 * n, flops=2.4 * n * _passes(case) * (solve + 25.0))
    if kind == "explicit":  # u, rho, mu, phi, k, T, RU in; S, u*, RU out
        return dict(bytes=8.0 * 18 * n, flops=n * 330.0)
    return dict(bytes=8.0 * 18 * n, flops=n * (330.0 + _passes(case) * (solve + 25.0)))


# ---- exact values ------------------------------------------------------------------------------

class _Reference:
    """The discrete operators on one grid in plain 64-bit torch."""

    def __init__(self, g):
        self.g, self.dx, self.yw = g, g["lx"] / g["nx"], g["ywalls"]
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        zf, ny = g["zf"], g["ny"]
        zc = 0.5 * (zf[1:] + zf[:-1])
        yf = np.linspace(0.0, g["ly"], ny + 1) if g["yf"] is None else g["yf"]
        yc = 0.5 * (yf[1:] + yf[:-1])
        dyc = np.full(ny, g["ly"] / ny)
        if g["yf"] is not None:
            dyc[1:] = np.diff(yc)
        self.hz, self.hy = np.diff(zf), np.diff(yf) if g["yf"] is not None else np.full(ny, g["ly"] / ny)
        self.dzf, self.dyf = t(self.hz)[:, None, None], t(self.hy)[None, :, None]
        self.dzc, self.dyc = t(np.diff(zc))[:, None, None], t(dyc)[None, :, None]
        self.W = self.dzf * self.dyf                       # cell volume over dx
        k = np.arange(g["nx"] // 2 + 1)
        lam = t(-4.0 / self.dx ** 2 * np.sin(math.pi * k / g["nx"]) ** 2)[None, None, :]
        lz, self.Qz = self._basis(self.hz, np.diff(zc))
        if self.yw:
            ly, self.Qy = self._basis(self.hy, dyc[1:])
        else:
            ly, self.Qy = t(-4.0 / dyc[0] ** 2 * np.sin(math.pi * np.arange(ny) / ny) ** 2), None
        self.lam = lam + ly[None, :, None] + lz[:, None, None]
        self.zero = self.lam.abs().argmin()

    @staticmethod
    def _basis(h, dc):
        """Eigenvalues and (V, V^T W) of the Neumann second difference with widths h and centre distances dc."""
        n = len(h)
        T = np.zeros((n, n))
        for j in range(n - 1):
            T[j, j] -= 1 / dc[j]
            T[j + 1, j + 1] -= 1 / dc[j]
            T[j, j + 1] = T[j + 1, j] = 1 / dc[j]
        s = 1 / np.sqrt(h)
        w, Q = np.linalg.eigh(s[:, None] * T * s[None, :])
        V = s[:, None] * Q
        put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        return put(w), (put(V), put((V * h[:, None]).T))

    @staticmethod
    def _along(M, a, axis):
        r = torch.view_as_real(a)
        if axis == 0:
            return torch.view_as_complex((M @ r.reshape(r.shape[0], -1)).view(r.shape))
        return torch.view_as_complex(torch.matmul(M, r.reshape(r.shape[0], r.shape[1], -1)).view(r.shape))

    def constant_solve(self, f, pinned=True):
        """L^{-1} f: zero mean (pinned), or with the zero eigenvalue replaced by the next one."""
        F = torch.fft.rfft(f, dim=2)
        F = self._along(self.Qy[1], F, 1) if self.yw else torch.fft.fft(F, dim=1)
        F = self._along(self.Qz[1], F, 0)
        F = F / self.lam
        z = self.zero
        if pinned:
            F.view(-1)[z] = 0.0
        else:
            F.view(-1)[z] *= 0.0
        F = self._along(self.Qz[0], F, 0)
        F = self._along(self.Qy[0], F, 1) if self.yw else torch.fft.ifft(F, dim=1)
        return torch.fft.irfft(F, n=self.g["nx"], dim=2)

    def mean(self, a):
        return (self.W * a).sum() / (self.W.sum() * self.g["nx"])

    def div(self, u, v, w):
        if self.yw:
            v = v.clone()
            v[:, 0] = 0.0
        return ((torch.roll(u, -1, 2) - u) / self.dx + (torch.roll(v, -1, 1) - v) / self.dyf
                + (w[1:] - w[:-1]) / self.dzf)

    def grad(self, p):
        gx = (p - torch.roll(p, 1, 2)) / self.dx
        gy = (p - torch.roll(p, 1, 1)) / self.dyc
        if self.yw:
            gy[:, 0] = 0.0
        gz = torch.zeros((p.shape[0] + 1,) + tuple(p.shape[1:]), dtype=p.dtype, device=p.device)
        gz[1:-1] = (p[1:] - p[:-1]) / self.dzc
        return gx, gy, gz

    def beta(self, rho):
        bz = torch.zeros((rho.shape[0] + 1,) + tuple(rho.shape[1:]), dtype=rho.dtype, device=rho.device)
        bz[1:-1] = 2.0 / (rho[1:] + rho[:-1])
        return 2.0 / (rho + torch.roll(rho, 1, 2)), 2.0 / (rho + torch.roll(rho, 1, 1)), bz

    def variable_solve(self, rho, rhs):
        """D(beta G p) = rhs, zero mean: conjugate gradients on -W D beta G, preconditioned by
        sqrt(rho) L^{-1} sqrt(rho)."""
        beta, root = self.beta(rho), rho.sqrt()
        op = lambda p: -self.W * self.div(*(b * q for b, q in zip(beta, self.grad(p))))  # noqa: E731

        def pre(r):
            q = root * r / self.W
            m = self.mean(q)
            return root * (-self.constant_solve(q - m) + m * self.g["lz"] ** 2)

        def residual(x):
            r = -self.W * (rhs - self.mean(rhs)) - op(x)
            return r - self.W * (r.sum() / (self.W.sum() * self.g["nx"]))

        x = torch.zeros_like(rhs)
        r = residual(x)
        norm = last = float(r.norm())
        for _ in range(6):              # conjugate gradients, started again from the true residual
            d = rz = None
            for _ in range(400):
                z = pre(r)
                new = (r * z).sum()
                d = z if d is None else z + (new / rz) * d
                rz = new
                q = op(d)
                a = rz / (d * q).sum()
                x += a * d
                r -= a * q
                if float(r.norm()) <= max(1e-9 * last, 1e-15 * norm):
                    break
            r = residual(x)
            now = float(r.norm())
            if now <= 1e-14 * norm or now > 0.3 * last:
                break
            last = now
        return x - self.mean(x)

    def project(self, u, v, w, rho, S, dt=DT):
        d = self.div(u, v, w)
        if S is not None:
            d = d - (S - self.mean(S))
        p = self.variable_solve(rho, d / dt)
        b, g = self.beta(rho), self.grad(p)
        out = [q - dt * bb * gg for q, bb, gg in zip((u, v, w), b, g)]
        if self.yw:
            out[1][:, 0] = 0.0
        return [p, *out]

    def conduction(self, kc, T):
        gx, gy, gz = self.grad(T)
        kz = torch.zeros_like(gz)
        kz[1:-1] = 0.5 * (kc[1:] + kc[:-1])
        return self.div(0.5 * (kc + torch.roll(kc, 1, 2)) * gx, 0.5 * (kc + torch.roll(kc, 1, 1)) * gy, kz * gz)

    def p0_rate(self, phi, kc, T, vel):
        dv = self.dx * self.W
        vg = (phi * dv).sum()
        return GAMMA / vg * ((GAMMA - 1) / GAMMA * (phi * self.conduction(kc, T) * dv).sum()
                             - P0 * (phi * self.div(*vel) * dv).sum())

    def source(self, phi, kc, T, rate):
        return ((GAMMA - 1) / GAMMA * self.conduction(kc, T) - rate / GAMMA) * phi / P0

    def momentum(self, u, v, w, rho, mu):
        """-C(u) + div tau / rho_f + g on the faces (periodic y, no-slip z walls)."""
        r, dx, dy = torch.roll, self.dx, self.g["ly"] / self.g["ny"]
        D = self.div(u, v, w)
        inner = lambda a: 0.5 * (a[1:] + a[:-1])  # noqa: E731

        def planes(mid, lo=None, hi=None):
            out = torch.zeros_like(w)
            out[1:-1] = mid
            if lo is not None:
                out[0], out[-1] = lo, hi
            return out

        fxx, fyy, fzz = (0.5 * (u + r(u, -1, 2))) ** 2, (0.5 * (v + r(v, -1, 1))) ** 2, inner(w) ** 2
        fxy = 0.25 * (u + r(u, 1, 1)) * (v + r(v, 1, 2))
        fxz = planes(inner(u) * 0.5 * (w + r(w, 1, 2))[1:-1])
        fyz = planes(inner(v) * 0.5 * (w + r(w, 1, 1))[1:-1])
        txx, tyy, tzz = (mu * (2.0 * d - 2.0 / 3.0 * D) for d in (
            (r(u, -1, 2) - u) / dx, (r(v, -1, 1) - v) / dy, (w[1:] - w[:-1]) / self.dzf))
        m4 = 0.25 * (mu + r(mu, 1, 2) + r(mu, 1, 1) + r(mu, (1, 1), (1, 2)))
        txy = m4 * ((u - r(u, 1, 1)) / dy + (v - r(v, 1, 2)) / dx)

        def shear(a, axis, h):
            m2, half = 0.5 * (mu + r(mu, 1, axis)), 0.5 * self.dzf
            return planes(inner(m2) * ((a[1:] - a[:-1]) / self.dzc + ((w - r(w, 1, axis)) / h)[1:-1]),
                          m2[0] * a[0] / half[0], -m2[-1] * a[-1] / half[-1])

        txz, tyz = shear(u, 2, dx), shear(v, 1, dy)
        bx, by, bz = self.beta(rho)
        ru = (-((fxx - r(fxx, 1, 2)) / dx + (r(fxy, -1, 1) - fxy) / dy + (fxz[1:] - fxz[:-1]) / self.dzf
                - u * 0.5 * (D + r(D, 1, 2)))
              + bx * ((txx - r(txx, 1, 2)) / dx + (r(txy, -1, 1) - txy) / dy + (txz[1:] - txz[:-1]) / self.dzf)
              + GRAVITY[0])
        rv = (-((r(fxy, -1, 2) - fxy) / dx + (fyy - r(fyy, 1, 1)) / dy + (fyz[1:] - fyz[:-1]) / self.dzf
                - v * 0.5 * (D + r(D, 1, 1)))
              + by * ((r(txy, -1, 2) - txy) / dx + (tyy - r(tyy, 1, 1)) / dy + (tyz[1:] - tyz[:-1]) / self.dzf)
              + GRAVITY[1])
        mid = lambda a: a[1:-1]  # noqa: E731
        rw = planes(-((r(mid(fxz), -1, 2) - mid(fxz)) / dx + (r(mid(fyz), -1, 1) - mid(fyz)) / dy
                      + (fzz[1:] - fzz[:-1]) / self.dzc - mid(w) * inner(D))
                    + mid(bz) * ((r(mid(txz), -1, 2) - mid(txz)) / dx + (r(mid(tyz), -1, 1) - mid(tyz)) / dy
                                 + (tzz[1:] - tzz[:-1]) / self.dzc) + GRAVITY[2])
        return ru, rv, rw

    def gradient(self, rho, p, cot, dt=DT):
        """dL/d(u*, v*, w*, rho) of the projection for the cotangents of u, v, w."""
        # u = u* - dt beta G p, W D(beta G p) = W (D u*)/dt; with G = -(W_f)^{-1} D^T W on the faces
        beta = self.beta(rho)
        wf = [self.W.expand_as(rho), (self.dzf * self.dyc).expand_as(rho), None]
        wz = torch.zeros_like(cot[2])
        wz[1:-1] = self.dzc * self.dyf
        wf[2] = wz
        iw = [1.0 / wf[0], 1.0 / wf[1], torch.where(wz > 0, 1.0 / wz, torch.zeros_like(wz))]
        lam = self.variable_solve(rho, self.div(*(b * i * c for b, i, c in zip(beta, iw, cot))))
        gl, gp = self.grad(lam), self.grad(p)
        star = [c - w_ * q for c, w_, q in zip(cot, wf, gl)]
        star[2][0] = star[2][-1] = 0.0
        face = [0.5 * b * b * dt * q * s for b, q, s in zip(beta, gp, star)]   # d beta/d rho = -beta^2 / 2 a cell
        grho = (face[0] + torch.roll(face[0], -1, 2) + face[1] + torch.roll(face[1], -1, 1)
                + face[2][1:] + face[2][:-1])
        return [*star, grho]


def exact(case, seed):
    kind = case["kind"]
    if case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0) > 300 ** 3:
        return None     # over a minute
    if kind == "batch":
        per = [_Reference(g).project(*f, rho, None) for g, rho, f in _batch_fields(case, seed)]
        return [torch.cat([o[q].reshape(-1) for o in per]) for q in range(4)]
    g = _geometry(case)
    ref = _Reference(g)
    if kind == "solve":
        f = torch.randn((g["nz"], g["ny"], g["nx"]), dtype=torch.float64, device="cuda", generator=_generator(seed))
        p = ref.constant_solve(f - ref.mean(f))
        return [p - ref.mean(p)]
    if kind == "project":
        _, rho, u, v, w, S = _two_phase(case, g, seed)
        return ref.project(u, v, w, rho, S)
    if kind == "gradient":
        _, rho, u, v, w, _ = _two_phase(case, g, seed)
        out = ref.project(u, v, w, rho, None)
        return [*out, *ref.gradient(rho, out[0], _faces(g, _generator(seed + 7), 1.0))]
    f = _flow(case, g, seed)
    rp = ref.p0_rate(f["phi"], f["kc"], f["T"], f["vel"])
    r = DT / (0.8 * DT)
    S = ref.source(f["phi"], f["kc"], f["T"], (1 + r) * rp - r * 0.5 * rp)
    ru = ref.momentum(*f["vel"], f["rho"], f["mu"])
    star = [q + DT * ((1 + 0.5 * r) * a - 0.5 * r * b) for q, a, b in zip(f["vel"], ru, f["ru"])]
    star[2][0] = star[2][-1] = 0.0
    if kind == "explicit":
        return [float(rp), S, *star, *ru]
    return [float(rp), S, *ref.project(*star, f["rho"], S)]
