"""Performance cases: what a user of the solver has it do, through its public entry points.

Families (a case's "family"), each with the sizes, schemes, boundaries and precisions it is used with:
  reconstruct  face values of a field set (npweno_reconstruct), the building block of a user's own solver
  step1d       one TVD-RK3 step of a user's own time loop (npweno_rk3_step)
  solve1d      one instance to its end time (npweno_solve): convergence studies, single runs
  batch1d      many uneven instances of one flux (npweno_batch_solve): parameter studies
  queue1d      1D Euler batches (npweno_queue_solve), component- or characteristic-wise
  queue2d      batches of 2D Euler squares (npweno_queue_solve)
  step2d       one step of a 2D grid (npweno_rk3_step_2d), the paper's 2D examples and larger grids
  serve        a mix of requests of both precisions through the request server

Inputs are made on the GPU from the seed: cell averages of Fourier modes with jumps (Burgers,
advection), Riemann and Shu-Osher-type data (1D Euler), vortices and four-quadrant data (2D Euler).
A case's sizes do not depend on the seed.  A pass of a solve copies the kept initial state into the
arena it advances, as a program that runs one set-up repeatedly does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1602_00182_gb300.npweno as npw

GAMMA = 1.4
CFL = 0.5
MIXED_GUARD = 8.0 * 2.0 ** -24  # the float state's automatic round-off guard of the shape parameter
EPS_M, EPS_WENO = 1e-12, 1e-6

ADV, BURG, EUL1, EUL2 = (npw.NPW_FLUX_ADVECTION, npw.NPW_FLUX_BURGERS, npw.NPW_FLUX_EULER1D, npw.NPW_FLUX_EULER2D)
PER, TRA = npw.NPW_BC_PERIODIC, npw.NPW_BC_TRANSMISSIVE
SCHEMES = {"eno": npw.NPW_ENO, "weno-js": npw.NPW_WENO_JS, "rbf-eno": npw.NPW_RBF_ENO, "rbf-weno": npw.NPW_RBF_WENO}
FLUXES = {"advection": ADV, "burgers": BURG, "euler1d": EUL1, "euler2d": EUL2}
FIELDS = {"advection": 1, "burgers": 1, "euler1d": 3, "euler2d": 4}


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one step of the paper's advection example (Sec. 5.2 Ex. 1) in a user's time loop
        dict(name="step1d advection fp64 200", family="step1d", flux="advection", n=200, scheme="rbf-weno", k=3,
             fp64=True),
        # the paper's convergence study: N = 200, FP64 (the default precision), 100 steps
        dict(name="solve1d advection fp64 200", family="solve1d", flux="advection", n=200, scheme="rbf-weno", k=3,
             fp64=True, steps=100),
        # one ordinary instance of the Burgers family in the float state, odd size
        dict(name="solve1d burgers mixed 5613", family="solve1d", flux="burgers", n=5613, scheme="rbf-weno", k=3,
             fp64=False, steps=150),
        # face values of a large 1D Euler field, flags included (the default)
        dict(name="reconstruct euler mixed", family="reconstruct", m=3, n=300007, scheme="rbf-weno", k=3, fp64=False),
        # a single FP64 gas-dynamics step, ordinary size, ragged
        dict(name="step1d euler fp64 20011", family="step1d", flux="euler1d", n=20011, scheme="rbf-weno", k=3,
             fp64=True),
        # the batched Burgers study: N log-uniform in [64, 8192]
        dict(name="batch1d burgers mixed", family="batch1d", flux="burgers", count=1024, nmin=64, nmax=8192,
             scheme="rbf-weno", k=3, fp64=False, steps=300),
        # the 1D Euler batch, N log-uniform in [256, 65536], component-wise
        dict(name="queue1d euler mixed", family="queue1d", count=96, nmin=256, nmax=65536, scheme="rbf-weno",
             characteristic=False, fp64=False, steps=60),
        # the same family characteristic-wise
        dict(name="queue1d euler characteristic", family="queue1d", count=64, nmin=256, nmax=16384,
             scheme="rbf-weno", characteristic=True, fp64=False, steps=60),
        # 2D Euler squares, vortices and four-quadrant data
        dict(name="queue2d euler mixed 256", family="queue2d", count=16, n=256, scheme="rbf-weno", fp64=False,
             steps=20),
        # the largest grid: one step of 2048 x 2048 cells
        dict(name="step2d euler mixed 2048", family="step2d", flux="euler2d", nx=2048, ny=2048, scheme="rbf-weno", k=3,
             cross=False, fp64=False),
        # the paper's 2D advection (Sec. 7 Ex. 1): k = 2 RBF-ENO on the five-cell cross, FP64, ragged
        dict(name="step2d advection k2 cross fp64", family="step2d", flux="advection", nx=321, ny=300,
             scheme="rbf-eno", k=2, cross=True, fp64=True),
        # a burst of requests of both tolerance classes, 1D and 2D
        dict(name="serve mixed requests", family="serve", count=24, nmin=64, nmax=4096, squares=2, nsq=128, steps=40),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the families above over their ranges."""
    fam = rng.choice(["reconstruct", "step1d", "solve1d", "batch1d", "queue1d", "queue2d", "step2d", "serve"])
    scheme = rng.choice(["rbf-weno", "rbf-weno", "rbf-eno", "weno-js", "eno"])
    fp64 = rng.random() < 0.4
    if fam == "reconstruct":
        return dict(family=fam, m=rng.choice([1, 3, 4]), n=_log(rng, 100, 1000000), scheme=scheme, k=rng.choice([3, 3, 2]),
                    fp64=fp64)
    if fam == "step1d":
        return dict(family=fam, flux=rng.choice(["advection", "burgers", "euler1d"]), n=_log(rng, 20, 300000),
                    scheme=scheme, k=rng.choice([3, 3, 2]), fp64=fp64)
    if fam == "solve1d":
        return dict(family=fam, flux=rng.choice(["advection", "burgers"]), n=_log(rng, 25, 20000), scheme=scheme, k=3,
                    fp64=fp64, steps=_log(rng, 20, 120))
    if fam == "batch1d":
        return dict(family=fam, flux="burgers", count=_log(rng, 16, 1024), nmin=64, nmax=_log(rng, 1024, 8192),
                    scheme=scheme, k=3, fp64=False, steps=_log(rng, 40, 300))
    if fam == "queue1d":
        char = rng.random() < 0.4
        return dict(family=fam, count=_log(rng, 4, 96), nmin=256, nmax=_log(rng, 2048, 16384 if char else 65536),
                    scheme="rbf-weno", characteristic=char, fp64=False, steps=_log(rng, 20, 60))
    if fam == "queue2d":
        n = _log(rng, 100, 512)
        return dict(family=fam, count=max(1, min(64, (1 << 20) // (n * n))), n=n, scheme="rbf-weno", fp64=False,
                    steps=_log(rng, 4, 20))
    if fam == "step2d":
        k2 = rng.random() < 0.4
        nx = _log(rng, 40, 400 if fp64 else 2048)
        return dict(family=fam, flux="advection" if k2 else "euler2d", nx=nx, ny=max(16, int(nx * rng.uniform(0.5, 1.0))),
                    scheme="rbf-eno" if k2 else "rbf-weno", k=2 if k2 else 3, cross=k2, fp64=fp64)
    return dict(family=fam, count=_log(rng, 8, 24), nmin=64, nmax=_log(rng, 512, 4096), squares=rng.choice([0, 1, 2]),
                nsq=_log(rng, 48, 128), steps=_log(rng, 10, 40))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _sizes(case):
    """Log-uniform sizes over [nmin, nmax], largest first."""
    c, lo, hi = case["count"], math.log(case["nmin"]), math.log(case["nmax"])
    return [int(round(math.exp(lo + (hi - lo) * (i + 0.5) / c))) for i in reversed(range(c))]


def _params(case):
    k = case.get("k", 3)
    p = npw.Params(scheme=SCHEMES[case["scheme"]], k=k, precision=npw.NPW_FP64 if case["fp64"] else npw.NPW_FP32_MIXED)
    p.rbf = npw.NPW_RBF_MQ if case["fp64"] else npw.NPW_RBF_GA
    p.characteristic = int(bool(case.get("characteristic")))
    p.cross_2d = int(bool(case.get("cross")))
    if case["family"] in ("queue1d", "queue2d") or (k == 2 and not p.cross_2d):
        p.eta_max = 1.0  # runs through shocks and k = 2, whose printed shape parameter is singular, bound it
    if p.cross_2d:
        p.eta_max = 100.0
    return p


def _waves(ns, g, dev):
    """Packed cell averages on [0, 2 pi]: 1 + four Fourier modes + up to two jumps per line."""
    nt = torch.tensor(ns, device=dev)
    inst = torch.repeat_interleave(torch.arange(len(ns), device=dev), nt)
    start = torch.cumsum(nt, 0) - nt
    j = torch.arange(int(nt.sum()), device=dev, dtype=torch.float64) - start[inst]
    w = (2.0 * math.pi / nt.double())[inst]
    a, b = j * w, (j + 1.0) * w
    pick = lambda x: torch.tensor(x, device=dev)[inst]  # noqa: E731
    u = torch.ones_like(a)
    for mode in range(1, 5):
        amp, ph = pick(g.uniform(0.0, 0.5, len(ns))), pick(g.uniform(0.0, 2.0 * math.pi, len(ns)))
        u += amp * (torch.cos(mode * a + ph) - torch.cos(mode * b + ph)) / (mode * w)
    nj = pick(g.integers(0, 3, len(ns)))
    for q in range(2):
        x, h = pick(g.uniform(0.0, 2.0 * math.pi, len(ns))), pick(g.uniform(-0.5, 0.5, len(ns)))
        u += torch.where(nj > q, h * torch.clamp((b - x) / w, 0.0, 1.0), 0.0)
    return u


def _cons(rho, u, p, v=None):
    f = [rho, rho * u] + ([] if v is None else [rho * v])
    return f + [p / (GAMMA - 1.0) + 0.5 * rho * (u * u + (0.0 if v is None else v * v))]


def _euler_line(i, n, g, dev):
    """[3][n] cell averages and dx: Riemann data on [0, 1] (even i), Shu-Osher-type on [-5, 5] (odd i)."""
    if i % 2 == 0:
        rho, vel, pr, x0 = g.uniform(0.1, 1.0, 2), g.uniform(-1.0, 1.0, 2), g.uniform(0.1, 1.0, 2), g.uniform(0.3, 0.7)
        dx = 1.0 / n
        a = torch.arange(n, device=dev, dtype=torch.float64) * dx
        fl = torch.clamp((x0 - a) / dx, 0.0, 1.0)
        L, R = _cons(rho[0], vel[0], pr[0]), _cons(rho[1], vel[1], pr[1])
        return torch.stack([L[q] * fl + R[q] * (1.0 - fl) for q in range(3)]), dx
    kk, M, x0 = int(g.integers(2, 9)), 3.0, -4.0 + g.uniform(-0.2, 0.2)
    p2 = 1.0 + 2.0 * GAMMA / (GAMMA + 1.0) * (M * M - 1.0)
    r2 = (GAMMA + 1.0) * M * M / ((GAMMA - 1.0) * M * M + 2.0)
    L = _cons(r2, M * math.sqrt(GAMMA) * (1.0 - 1.0 / r2), p2)
    dx = 10.0 / n
    a = -5.0 + torch.arange(n, device=dev, dtype=torch.float64) * dx
    b = a + dx
    fl = torch.clamp((x0 - a) / dx, 0.0, 1.0)
    ar = torch.clamp(a, min=x0)
    right = torch.where(b > x0, (b - ar) + 0.2 * (torch.cos(kk * ar) - torch.cos(kk * b)) / kk, 0.0) / dx
    return torch.stack([L[0] * fl + right, L[1] * fl, L[2] * fl + (1.0 - fl) / (GAMMA - 1.0)]), dx


def _square(i, nx, ny, g, dev):
    """[4][ny][nx] and the cell size: an isentropic vortex (even i) or four-quadrant data (odd i)."""
    n = max(nx, ny)
    if i % 2 == 0:
        d, s = 10.0 / n, g.uniform(3.0, 5.0)
        x = (torch.arange(nx, device=dev, dtype=torch.float64) + 0.5) * d - g.uniform(3.0, 4.0) * nx / n
        y = ((torch.arange(ny, device=dev, dtype=torch.float64) + 0.5) * d - g.uniform(3.0, 4.0) * ny / n)[:, None]
        x, y = x[None].expand(ny, nx), y.expand(ny, nx)
        r2 = x * x + y * y
        e = s / (2.0 * math.pi) * torch.exp(0.5 * (1.0 - r2))
        T = 1.0 - (GAMMA - 1.0) / (2.0 * GAMMA) * e * e
        rho = T ** (1.0 / (GAMMA - 1.0))
        return torch.stack(_cons(rho, 1.0 - e * y, rho * T, 1.0 + e * x)), d
    d = 1.0 / n
    U = torch.empty((4, ny, nx), dtype=torch.float64, device=dev)
    for ys in (slice(0, ny // 2), slice(ny // 2, ny)):
        for xs in (slice(0, nx // 2), slice(nx // 2, nx)):
            c = _cons(*g.uniform(0.1, 1.0, 1), g.uniform(-1.0, 1.0), g.uniform(0.1, 1.0), g.uniform(-1.0, 1.0))
            for q in range(4):
                U[q, ys, xs] = c[q]
    return U, d


def _problem(case, seed):
    """Initial states and the run's numbers, all in FP64: dict(u = packed initial state, ...)."""
    g, dev, fam = np.random.default_rng(seed), torch.device("cuda"), case["family"]
    if fam == "reconstruct":
        if case["m"] == 3:
            return dict(u=_euler_line(1, case["n"], g, dev)[0])
        return dict(u=torch.stack([_waves([case["n"]], g, dev) for _ in range(case["m"])]))
    if fam in ("step1d", "solve1d"):
        n = case["n"]
        if case["flux"] == "euler1d":
            u, dx = _euler_line(1, n, g, dev)
        else:
            u, dx = _waves([n], g, dev)[None], 2.0 * math.pi / n
        speed = {"advection": 1.0, "burgers": 2.5, "euler1d": 4.8}[case["flux"]]
        return dict(u=u, dx=dx, dt=0.4 * dx / speed, t_end=(case.get("steps", 0) - 0.5) * CFL * dx / speed)
    if fam == "batch1d":
        ns = _sizes(case)
        t = case["steps"] * CFL * 2.0 * math.pi / ns[0] / 2.5
        return dict(u=_waves(ns, g, dev), ns=ns, dx=[2.0 * math.pi / n for n in ns], t_end=[t] * len(ns))
    if fam == "queue1d":
        ns = _sizes(case)
        lines = [_euler_line(i, n, g, dev) for i, n in enumerate(ns)]
        # the share of each instance's run that the largest takes `steps` steps for
        dx = [d for _, d in lines]
        t = [case["steps"] * CFL * (1.0 if i % 2 == 0 else 10.0) / ns[0] / (2.5 if i % 2 == 0 else 4.8)
             for i in range(len(ns))]
        return dict(u=torch.cat([u.reshape(-1) for u, _ in lines]), ns=ns, dx=dx, t_end=t)
    if fam == "queue2d":
        sq = [_square(i, case["n"], case["n"], g, dev) for i in range(case["count"])]
        return dict(u=torch.stack([u for u, _ in sq]), dx=[d for _, d in sq],
                    t_end=[case["steps"] * CFL * d / (2.0 * 2.4) for _, d in sq])
    if fam == "step2d":
        nx, ny = case["nx"], case["ny"]
        if case["flux"] == "euler2d":
            u, d = _square(0, nx, ny, g, dev)
        else:
            d, ph = 1.0 / max(nx, ny), g.uniform(0.0, 1.0, 2)
            x = (torch.arange(nx, device=dev, dtype=torch.float64) + 0.5) * d + ph[0]
            y = (torch.arange(ny, device=dev, dtype=torch.float64) + 0.5) * d + ph[1]
            avg = (math.sin(math.pi * d) / (math.pi * d)) ** 2  # exact cell averages of the sine
            u = (avg * torch.sin(2.0 * math.pi * (x[None, :] + y[:, None])))[None]
        return dict(u=u, dx=d, dt=0.2 * d / (2.4 if case["flux"] == "euler2d" else 1.0))
    reqs = []  # serve: Burgers and Euler lines, a quarter of them in FP64, and 2D Euler squares
    for i, n in enumerate(_sizes(case)):
        if i % 3 == 2 and n >= 128:
            u, d = _euler_line(i, n, g, dev)
            reqs.append(dict(u=u, flux=EUL1, bc=TRA, dx=d, t_end=case["steps"] * CFL * d / 4.8, fp64=i % 4 == 3))
        else:
            d = 2.0 * math.pi / n
            reqs.append(dict(u=_waves([n], g, dev)[None], flux=BURG, bc=PER, dx=d, t_end=case["steps"] * CFL * d / 2.5,
                             fp64=i % 4 == 3))
    for i in range(case["squares"]):
        u, d = _square(i, case["nsq"], case["nsq"], g, dev)
        reqs.append(dict(u=u, flux=EUL2, bc=PER, dx=d, t_end=case["steps"] * CFL * d / (2.0 * 2.4), fp64=False))
    return dict(reqs=reqs)


def prepare(case, seed):
    fam, q = case["family"], _problem(case, seed)
    if fam == "serve":
        p = npw.Params(rbf=npw.NPW_RBF_GA, precision=npw.NPW_FP32_MIXED, eta_max=1.0)
        for r in q["reqs"]:
            r["u"] = r["u"].cpu().numpy().astype(np.float64 if r["fp64"] else np.float32)
        cells = sum(r["u"].size for r in q["reqs"])
        return dict(family=fam, reqs=q["reqs"], server=npw.Server(heap_cells=cells + 4096, max_slots=64, params=p))
    p = _params(case)
    u0 = q["u"].to(torch.float64 if case["fp64"] else torch.float32).contiguous()
    s = dict(q, family=fam, params=p, u0=u0, u=torch.empty_like(u0), flux=FLUXES.get(case.get("flux", ""), EUL1))
    s["bc"] = TRA if s["flux"] == EUL1 or case.get("m") == 3 else PER
    if fam in ("step1d", "solve1d"):
        nbytes = npw.npw_workspace_size(case["n"], u0.shape[0], p)
    elif fam == "batch1d":
        s["table"], _ = npw.make_instances(q["ns"], q["dx"], q["t_end"], [CFL] * len(q["ns"]), [PER] * len(q["ns"]))
        nbytes = npw.npw_batch_workspace_size(s["table"], 1, p)
    elif fam in ("queue1d", "queue2d"):
        if fam == "queue1d":
            specs = [dict(kind=EUL1, nx=n, dx=d, t_end=t, cfl=CFL, bc=TRA) for n, d, t in zip(q["ns"], q["dx"], q["t_end"])]
        else:
            specs = [dict(kind=EUL2, nx=case["n"], ny=case["n"], dx=d, dy=d, t_end=t, cfl=CFL, bc=PER)
                     for d, t in zip(q["dx"], q["t_end"])]
        s["table"], _, _ = npw.make_queue_instances(specs)
        nbytes = npw.npw_queue_workspace_size(s["table"], p)
    elif fam == "step2d":
        nbytes = npw.npw_workspace_size_2d(case["nx"], case["ny"], u0.shape[0], p)
    else:
        return s
    s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    fam = s["family"]
    if fam == "reconstruct":
        return npw.npweno_reconstruct(s["u0"], s["bc"], s["params"])
    if fam == "serve":
        srv = s["server"]
        for i, r in enumerate(s["reqs"]):
            srv.submit(r["u"], r["flux"], r["bc"], r["dx"], r["t_end"], CFL, tag=i,
                       dy=r["dx"] if r["flux"] == EUL2 else 0.0, tolerance=1e-8 if r["fp64"] else 1e-4)
        active = queued = 1
        got = []
        while active or queued:
            active, queued = srv.step(32)
            got += srv.poll()
        return [r["u"] for r in sorted(got, key=lambda r: r["tag"])]
    u, p = s["u"], s["params"]
    u.copy_(s["u0"])
    if fam == "step1d":
        npw.npweno_rk3_step(u, s["dx"], s["dt"], s["flux"], s["bc"], p, workspace=s["ws"])
    elif fam == "solve1d":
        npw.npweno_solve(u, s["dx"], s["t_end"], CFL, s["flux"], s["bc"], p, workspace=s["ws"])
    elif fam == "batch1d":
        npw.npweno_batch_solve(u, s["table"], 1, s["flux"], p, workspace=s["ws"])
    elif fam == "step2d":
        npw.npweno_rk3_step_2d(u, s["dx"], s["dx"], s["dt"], s["flux"], s["bc"], p, workspace=s["ws"])
    else:
        npw.npweno_queue_solve(u, s["table"], p, workspace=s["ws"])
    return u


# ---------------------------------------------------------------------------------------
# the work of a pass: state in and out once, and the flops of the method's formulas
# ---------------------------------------------------------------------------------------
def _face_flops(case):
    """Flops per face, field and stage: k = 3: shape parameter 12, switch 12, candidates 30, indicators 15,
    weights 25; k = 2 about half; flux, difference and stage update 16."""
    rbf, weno = case["scheme"].startswith("rbf"), "weno" in case["scheme"]
    full = (24 if rbf else 0) + 30 + (40 if weno else 12)
    return (full if case.get("k", 3) == 3 else full // 2) + 16


def work(case):
    fam = case["family"]
    if fam == "serve":
        r = _serve_sizes(case)
        c3 = dict(scheme="rbf-weno")
        return dict(bytes=sum(2 * b * c for c, b, _, _ in r),
                    flops=sum(c * st * 3 * d * _face_flops(c3) for c, _, st, d in r))
    b = 8 if case["fp64"] else 4
    if fam == "reconstruct":
        return dict(bytes=case["m"] * case["n"] * (3 * b + 1), flops=case["m"] * case["n"] * _face_flops(case))
    if fam in ("step1d", "solve1d"):
        cells, steps, dims, fsteps = case["n"] * FIELDS[case["flux"]], case.get("steps", 1), 1, None
    elif fam == "step2d":
        cells, steps, dims, fsteps = case["nx"] * case["ny"] * FIELDS[case["flux"]], 1, 2, None
    elif fam == "queue2d":
        cells, steps, dims, fsteps = case["count"] * case["n"] ** 2 * 4, case["steps"], 2, None
    else:
        ns, m = _sizes(case), 1 if fam == "batch1d" else 3
        cells, steps, dims = m * sum(ns), 1, 1
        fsteps = m * sum(n * max(1.0, case["steps"] * n / ns[0]) for n in ns)
    return dict(bytes=2 * b * cells, flops=(fsteps or cells * steps) * 3 * dims * _face_flops(case))


def _serve_sizes(case):
    """(values, bytes each, steps, directions) of every request."""
    r = []
    for i, n in enumerate(_sizes(case)):
        r.append((n * (3 if i % 3 == 2 and n >= 128 else 1), 8 if i % 4 == 3 else 4, case["steps"], 1))
    return r + [(4 * case["nsq"] ** 2, 4, case["steps"], 2)] * case["squares"]


# ---------------------------------------------------------------------------------------
# the method in FP64, plain torch: the same inputs, rounded to the state's type
# ---------------------------------------------------------------------------------------
class _Method:
    def __init__(self, scheme, k, fp64, characteristic=False, cross=False, eta_max=0.0, gaussian=None):
        self.scheme, self.k, self.char, self.cross, self.eta_max = scheme, k, characteristic, cross, eta_max
        self.gauss = (not fp64) if gaussian is None else gaussian
        self.guard = 0.0 if fp64 else MIXED_GUARD
        self.rbf, self.weno = scheme.startswith("rbf"), "weno" in scheme

    def _limit(self, num, den, mag):
        eta = num / (den + EPS_M)
        if self.guard > 0.0:
            eta = torch.where(den.abs() <= self.guard * mag, 0.0, eta)
        return torch.where(eta.abs() > self.eta_max, 0.0, eta) if self.eta_max > 0.0 else eta

    def _eta3(self, w0, w1, w2, w3):
        eta = self._limit(w0 - 3.0 * w1 + 3.0 * w2 - w3, w0 - 15.0 * w1 + 15.0 * w2 - w3,
                          w0.abs() + 15.0 * w1.abs() + 15.0 * w2.abs() + w3.abs())
        A = 6.0 * ((w3 - w0) + 3.0 * (w1 - w2))
        B = 6.0 * ((w0 - w1) + (w3 - w2))
        C = (w0 - w3) + 15.0 * (w2 - w1)
        lo, hi = torch.minimum(4.0 * A - 2.0 * B + C, 4.0 * A + 2.0 * B + C), torch.maximum(4.0 * A - 2.0 * B + C, 4.0 * A + 2.0 * B + C)
        inside = (A != 0.0) & (B.abs() < 4.0 * A.abs())
        v = C - B * B / torch.where(A == 0.0, 1.0, 4.0 * A)
        lo, hi = torch.where(inside, torch.minimum(lo, v), lo), torch.where(inside, torch.maximum(hi, v), hi)
        return torch.where((lo < 0.0) & (hi > 0.0), 0.0, eta)

    def _cell3(self, c, eta, side):
        poly = [(11 / 6, -7 / 6, 1 / 3), (1 / 3, 5 / 6, -1 / 6), (-1 / 6, 5 / 6, 1 / 3), (1 / 3, -7 / 6, 11 / 6)]
        pert = ([(-3.0, 3.0, 0.0), (2 / 3, -1 / 3, -1 / 3), (-1 / 3, -1 / 3, 2 / 3), (0.0, 3.0, -3.0)] if self.gauss else
                [(-9 / 2, 6.0, -3 / 2), (5 / 6, -2 / 3, -1 / 6), (-1 / 6, -2 / 3, 5 / 6), (-3 / 2, 6.0, -9 / 2)])
        cand = []
        for r in range(3):
            row = r + 1 - side
            cand.append(sum((poly[row][j] + pert[row][j] * eta) * c[2 - r + j] for j in range(3)))
        if not self.weno:
            left = (c[2] - c[1]).abs() < (c[3] - c[2]).abs()
            dd = [(c[i] - 2.0 * c[i + 1] + c[i + 2]).abs() for i in range(3)]
            return torch.where(left, torch.where(dd[0] < dd[1], cand[2], cand[1]), torch.where(dd[1] < dd[2], cand[1], cand[0]))
        ab = [(c[2] - 2.0 * c[3] + c[4], 3.0 * c[2] - 4.0 * c[3] + c[4]), (c[1] - 2.0 * c[2] + c[3], c[1] - c[3]),
              (c[0] - 2.0 * c[1] + c[2], c[0] - 4.0 * c[1] + 3.0 * c[2])]
        d = (0.3, 0.6, 0.1) if side == 0 else (0.1, 0.6, 0.3)
        al = [d[r] / (EPS_WENO + 13.0 / 12.0 * a * a + 0.25 * b * b) ** 2 for r, (a, b) in enumerate(ab)]
        return sum(al[r] * cand[r] for r in range(3)) / (al[0] + al[1] + al[2])

    def _cell2(self, c, side, trans):
        a, b, d = (c[0], c[1], c[2]) if side == 0 else (c[2], c[1], c[0])
        ec = ex = torch.zeros_like(b)
        if self.rbf:
            f = 1.0 if self.gauss else 2.0
            den, mag = -a + 5.0 * b + 2.0 * d, a.abs() + 5.0 * b.abs() + 2.0 * d.abs()
            ec = self._limit(f * (-a + 2.0 * b - d - 0.25 * trans), den, mag)
            ex = self._limit(f * (-a + 2.0 * b - d + 0.125 * trans), den, mag)
            dn = -c[0] + 2.0 * c[1] - c[2]
            ratio = (-2.0 * c[0] + 3.0 * c[1] - c[2]) / torch.where(dn == 0.0, 1.0, dn)
            off = (dn != 0.0) & (ratio > 0.0) & (ratio < 3.0)
            ec, ex = torch.where(off, 0.0, ec), torch.where(off, 0.0, ex)
        poly = [(1.5, -0.5), (0.5, 0.5), (-0.5, 1.5)]
        pert = [(-2.0, 0.0), (0.5, 0.5), (0.0, -2.0)] if self.gauss else [(-1.5, 0.5), (0.25, 0.25), (0.5, -1.5)]
        cand = []
        for r in range(2):
            row, eta = r + 1 - side, ec if r - side == 0 else ex
            cand.append(sum((poly[row][j] + pert[row][j] * eta) * c[1 - r + j] for j in range(2)))
        if not self.weno:
            return torch.where((c[1] - c[0]).abs() < (c[2] - c[1]).abs(), cand[1], cand[0])
        dw = (2 / 3, 1 / 3) if side == 0 else (1 / 3, 2 / 3)
        a0, a1 = dw[0] / (EPS_WENO + (c[2] - c[1]) ** 2) ** 2, dw[1] / (EPS_WENO + (c[1] - c[0]) ** 2) ** 2
        return (a0 * cand[0] + a1 * cand[1]) / (a0 + a1)

    def face(self, w, tl=0.0, tr=0.0):
        """v^-, v^+ of one field set from the six cells around a face (tl, tr: transverse differences)."""
        if self.k == 2:
            return self._cell2(w[1:4], 0, tl), self._cell2(w[2:5], 1, tr)
        eta = self._eta3(*w[1:5]) if self.rbf else torch.zeros_like(w[0])
        return self._cell3(w[:5], eta, 0), self._cell3(w[1:], eta, 1)

    def face_char(self, w):
        """The same in Roe characteristic fields: w[j] is [3][...]."""
        L, R = w[2], w[3]
        vel, rt = [x[1] / x[0] for x in (L, R)], [torch.sqrt(x[0]) for x in (L, R)]
        pr = [(GAMMA - 1.0) * (x[2] - 0.5 * x[0] * v * v) for x, v in zip((L, R), vel)]
        H = [(x[2] + p) / x[0] for x, p in zip((L, R), pr)]
        u = (rt[0] * vel[0] + rt[1] * vel[1]) / (rt[0] + rt[1])
        h = (rt[0] * H[0] + rt[1] * H[1]) / (rt[0] + rt[1])
        c2 = (GAMMA - 1.0) * (h - 0.5 * u * u)
        c = torch.sqrt(c2)
        b1 = (GAMMA - 1.0) / c2
        b2 = 0.5 * b1 * u * u
        one = torch.ones_like(u)
        rows = [(0.5 * (b2 + u / c), -0.5 * (b1 * u + 1.0 / c), 0.5 * b1), (1.0 - b2, b1 * u, -b1),
                (0.5 * (b2 - u / c), -0.5 * (b1 * u - 1.0 / c), 0.5 * b1)]
        cols = [(one, one, one), (u - c, u, u + c), (h - u * c, 0.5 * u * u, h + u * c)]
        wc = [torch.stack([sum(rw[q] * x[q] for q in range(3)) for rw in rows]) for x in w]
        return tuple(torch.stack([sum(cl[q] * v[q] for q in range(3)) for cl in cols]) for v in self.face(wc))


def _flux(U, flux, d):
    if flux == ADV:
        return U
    if flux == BURG:
        return 0.5 * U * U
    rho, E = U[0], U[-1]
    vel = [U[q] / rho for q in range(1, U.shape[0] - 1)]
    p = (GAMMA - 1.0) * (E - 0.5 * rho * sum(v * v for v in vel))
    return torch.stack([rho * vel[d]] + [U[1 + q] * vel[d] + (p if q == d else 0.0) for q in range(len(vel))] + [(E + p) * vel[d]])


def _speed(U, flux, d):
    if flux == ADV:
        return torch.ones_like(U[0])
    if flux == BURG:
        return U[0].abs()
    rho = U[0]
    vel = [U[q] / rho for q in range(1, U.shape[0] - 1)]
    p = (GAMMA - 1.0) * (U[-1] - 0.5 * rho * sum(v * v for v in vel))
    return vel[d].abs() + torch.sqrt(GAMMA * p / rho)


def _neighbours(ns, bc, dev):
    """(line, k -> index of the cell k places right of each packed cell, by the boundary rule)."""
    nt = torch.tensor(ns, device=dev)
    line = torch.repeat_interleave(torch.arange(len(ns), device=dev), nt)
    start, n = (torch.cumsum(nt, 0) - nt)[line], nt[line]
    j = torch.arange(int(nt.sum()), device=dev) - start
    at = {k: start + (torch.remainder(j + k, n) if bc == PER else torch.minimum(torch.clamp(j + k, min=0), n - 1))
          for k in range(-3, 4)}
    return line, at


def _difference(U, M, flux, d, alpha, at, h, trans):
    """-(h_right - h_left) / dx of every cell: at(U, k) the cells k places along direction d."""
    T = trans(U) if M.k == 2 and M.cross else None
    fl = []
    for o in (0, -1):  # the right and the left face of each cell
        w = [at(U, k + o) for k in range(-2, 4)]
        if M.char:
            vm, vp = M.face_char(w)
        else:
            vm, vp = M.face(w, *((at(T, o), at(T, o + 1)) if T is not None else (0.0, 0.0)))
        fl.append(0.5 * (_flux(vm, flux, d) + _flux(vp, flux, d) - alpha * (vp - vm)))
    return -(fl[0] - fl[1]) / h


def _rk3(U, dt, L):
    u1 = U + dt * L(U)
    u2 = 0.75 * U + 0.25 * (u1 + dt * L(u1))
    return U / 3.0 + 2.0 / 3.0 * (u2 + dt * L(u2))


def _run_exact(U, groups, dims, M, flux, dx, at, trans, t_end=None, dt=None, top=None):
    """One step of dt, or steps to each group's t_end.  top(speed): the largest of each group, spread to
    the cells by groups(); dx, t_end and dt: per cell tensors or numbers."""
    t = 0.0
    for _ in range(1 if dt is not None else 5000):
        al = [groups(top(_speed(U, flux, d))) for d in range(dims)]
        if dt is None:
            step = CFL / sum(a / dx for a in al)
            left = t_end - t
            step = torch.where(step * (1.0 + 1e-10) >= left, left, step)
            if float(left.max()) <= 0.0:
                return U
        else:
            step = dt
        U = _rk3(U, step, lambda V: sum(_difference(V, M, flux, d, al[d], at[d], dx, trans[d]) for d in range(dims)))
        t = t + step
    return U


def _exact_lines(u, ns, flux, bc, M, dx, t_end=None, dt=None):
    """u: [m][cells], lines packed."""
    line, idx = _neighbours(ns, bc, u.device)
    spread = lambda x: torch.tensor(x, dtype=torch.float64, device=u.device)[line]  # noqa: E731
    top = lambda s: torch.zeros(len(ns), dtype=s.dtype, device=s.device).scatter_reduce(0, line, s, "amax")  # noqa: E731
    return _run_exact(u, lambda a: a[line], 1, M, flux, spread(dx), [lambda V, k: V[..., idx[k]]], [None],
                      None if t_end is None else spread(t_end), dt, top)


def _exact_squares(u, flux, M, dx, t_end=None, dt=None):
    """u: [m][squares][ny][nx], periodic."""
    dev = u.device
    spread = lambda x: torch.tensor(x, dtype=torch.float64, device=dev)[:, None, None]  # noqa: E731
    at = [lambda V, k: torch.roll(V, -k, -1), lambda V, k: torch.roll(V, -k, -2)]
    second = lambda a: (lambda V: a(V, -1) - 2.0 * V + a(V, 1))  # noqa: E731
    return _run_exact(u, lambda a: a[:, None, None], 2, M, flux, spread(dx), at, [second(at[1]), second(at[0])],
                      None if t_end is None else spread(t_end), dt, lambda s: s.amax((-2, -1)))


def exact(case, seed):
    fam, q = case["family"], _problem(case, seed)
    rounded = lambda u, fp64: u if fp64 else u.float().double()  # noqa: E731
    if fam == "serve":
        out = []
        for r in q["reqs"]:
            u, M = rounded(r["u"], r["fp64"]), _Method("rbf-weno", 3, r["fp64"], eta_max=1.0, gaussian=True)
            if r["flux"] == EUL2:
                v = _exact_squares(u[:, None], EUL2, M, [r["dx"]], t_end=[r["t_end"]])[:, 0]
            else:
                v = _exact_lines(u, [u.shape[1]], r["flux"], r["bc"], M, [r["dx"]], t_end=[r["t_end"]])
            out.append(v.cpu().numpy())
        return out
    u, p = rounded(q["u"], case["fp64"]), _params(case)
    M = _Method(case["scheme"], case.get("k", 3), case["fp64"], bool(p.characteristic), bool(p.cross_2d), p.eta_max)
    flux = FLUXES.get(case.get("flux", ""), EUL1)
    if fam == "reconstruct":
        n, bc = case["n"], TRA if case["m"] == 3 else PER
        f = torch.arange(n + 1, device=u.device)
        pick = (lambda j: torch.remainder(j, n)) if bc == PER else (lambda j: torch.clamp(j, 0, n - 1))
        return (*M.face([u[:, pick(f + k)] for k in range(-3, 3)]), None)
    if fam in ("step1d", "solve1d"):
        to = dict(dt=q["dt"]) if fam == "step1d" else dict(t_end=[q["t_end"]])
        return _exact_lines(u, [case["n"]], flux, TRA if flux == EUL1 else PER, M, [q["dx"]], **to)
    if fam == "batch1d":
        return _exact_lines(u[None], q["ns"], BURG, PER, M, q["dx"], t_end=q["t_end"])[0]
    if fam == "queue1d":
        lines = [x.reshape(3, n) for n, x in zip(q["ns"], torch.split(u, [3 * n for n in q["ns"]]))]
        v = _exact_lines(torch.cat(lines, 1), q["ns"], EUL1, TRA, M, q["dx"], t_end=q["t_end"])
        return torch.cat([x.reshape(-1) for x in torch.split(v, q["ns"], 1)])
    if fam == "queue2d":
        return _exact_squares(u.transpose(0, 1).contiguous(), EUL2, M, q["dx"], t_end=q["t_end"]).transpose(0, 1)
    return _exact_squares(u[:, None], flux, M, [q["dx"]], dt=q["dt"])[:, 0]
