"""Workloads of the Chebyshev-Jacobi library as its users run them, for timing.

Every case goes through the public binding (``paper_1705_00103_gb300``): whole solves in each
precision, the sweeps alone, a batch and a burst of served requests.  Inputs are synthetic and
seeded: right-hand sides are sums of sine modes with Gaussian coefficients whose amplitude decays
as |k|^-2 up to |k| <= 64 (the repository's smooth random right-hand side), or the paper's test
problem with its Dirichlet data.

``exact`` gives the 64-bit value of each computed grid, from numpy and torch alone: a solve
converges to the discrete solution, which the discrete sine transform gives in closed form, and
sweeps are written out on whole arrays.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

import paper_1705_00103_gb300 as cj

_PREC = {"f64": cj.CJ_FP64, "mixed": cj.CJ_FP32_INNER, "mixed_dd": cj.CJ_FP32_INNER_DD,
         "f64_dd": cj.CJ_FP64_INNER_DD}
# arithmetic operations of one node update u + w (L u - b), by stencil
_OPS = {5: 9, 9: 14, 17: 24}


def listed():
    return [
        # the smallest everyday solve: a coarse Poisson problem to full accuracy, latency-bound
        dict(name="solve_f64_5pt_64", kind="solve", prec="f64", st=5, Nx=64, Ny=64, tol=1e-10, bc="zero"),
        # a small high-order grid (the paper's 17-point N = 128 regime), ragged and not square
        dict(name="solve_f64_17pt_129x200", kind="solve", prec="f64", st=17, Nx=129, Ny=200, tol=1e-8, bc="zero"),
        # the paper's timing run: its test problem with Dirichlet data, N = 1024, tol = N^-2
        dict(name="solve_f64_9pt_paper_1024", kind="solve", prec="f64", st=9, Nx=1024, Ny=1024, tol=2.0 ** -20,
             bc="data"),
        # an all-FP64 solve below one array's rounding floor, medium grid with odd sides
        dict(name="solve_f64dd_9pt_1001x701", kind="solve", prec="f64_dd", st=9, Nx=1001, Ny=701, tol=1e-10,
             bc="zero"),
        # a quick loose-tolerance solve of a small grid in mixed precision (the served 1e-6 requests)
        dict(name="solve_mixed_5pt_333x250", kind="solve", prec="mixed", st=5, Nx=333, Ny=250, tol=1e-6, bc="zero"),
        # a medium grid to 1e-10 in mixed precision
        dict(name="solve_mixed_dd_9pt_1023", kind="solve", prec="mixed_dd", st=9, Nx=1023, Ny=1023, tol=1e-10,
             bc="zero"),
        # the large mixed-precision solve to 1e-10
        dict(name="solve_mixed_dd_9pt_4096", kind="solve", prec="mixed_dd", st=9, Nx=4096, Ny=4096, tol=1e-10,
             bc="zero"),
        # part of an FP32 inner cycle of the high-order stencil at its full size
        dict(name="sweeps_f32_17pt_8192", kind="sweeps", prec="mixed", st=17, Nx=8192, Ny=8192, tol=1e-10,
             inner=8192, first=0, count=64),
        # plain FP64 sweeps of the large grid (a smoother called from another solver)
        dict(name="sweeps_f64_9pt_4096", kind="sweeps", prec="f64", st=9, Nx=4096, Ny=4096, tol=1e-10, first=0,
             count=16),
        # the same in float-float, ragged in both directions
        dict(name="sweeps_ff_9pt_4095x4001", kind="sweeps", prec="ff", st=9, Nx=4095, Ny=4001, tol=1e-10, first=5,
             count=32),
        # independent problems of uneven sizes solved together
        dict(name="batch_32", kind="batch", n=32, lo=64, hi=1024, tol=1e-8, pick=3),
        # a burst of served requests of all stencils and both tolerances, host arrays in and out
        dict(name="serve_24", kind="serve", n=24, lo=32, hi=1024, pick=4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choice(["solve", "solve", "solve", "sweeps", "sweeps", "sweeps", "batch", "serve"])
        if kind == "solve":
            prec = rng.choice(["f64", "mixed", "mixed_dd", "f64_dd"])
            big = 4096 if prec.startswith("mixed") else 1100
            st = rng.choice([5, 9, 17])
            bc = rng.choice(["zero", "zero", "data"]) if st != 17 else "zero"
            tol = {"f64": 10.0 ** rng.uniform(-8, -5), "mixed": 10.0 ** rng.uniform(-7, -5)}.get(prec, 1e-10)
            c = dict(kind=kind, prec=prec, st=st, Nx=_log_int(rng, 40, big), Ny=_log_int(rng, 40, big), tol=tol, bc=bc)
            # about the time of the pass: no longer than the largest listed solve
            rate = 2e11 if prec.startswith("mixed") else 3e10
            if st == 17:
                rate *= 0.5
            M = _sweeps_needed(st, c["Nx"], c["Ny"], tol)
            if 2 * M * (c["Nx"] * c["Ny"] / rate + 4e-6) <= 0.5:
                return c
        elif kind == "sweeps":
            prec = rng.choice(["f64", "mixed", "ff"])
            c = dict(kind=kind, prec=prec, st=rng.choice([5, 9, 17]), Nx=_log_int(rng, 200, 8192),
                     Ny=_log_int(rng, 200, 8192), tol=1e-10, first=rng.randint(0, 9), count=rng.randint(8, 64))
            if prec == "mixed":
                c["inner"] = rng.choice([1024, 4096, 8192])
            if c["Nx"] * c["Ny"] * c["count"] <= 64 * 8192 * 8192 // (8 if prec == "f64" else 1):
                return c
        elif kind == "batch":
            return dict(kind=kind, n=rng.randint(8, 32), lo=64, hi=rng.choice([300, 600, 1024]),
                        tol=10.0 ** rng.uniform(-8, -6), pick=rng.randint(0, 10 ** 6))
        else:
            return dict(kind=kind, n=rng.randint(6, 24), lo=32, hi=rng.choice([300, 600, 1024]),
                        pick=rng.randint(0, 10 ** 6))


# ------------------------------------------------------------------------------------- inputs

def _rhs(Nx, Ny, seed, device="cuda"):
    """Smooth random right-hand side (Ny, Nx): sine modes, Gaussian amplitudes / |k|^2, |k| <= 64."""
    rs = np.random.RandomState(seed % (2 ** 32))
    k = np.arange(1, min(64, Nx) + 1)[None, :]
    l = np.arange(1, min(64, Ny) + 1)[:, None]
    k2 = (k * k + l * l).astype(np.float64)
    A = np.where(k2 <= 64.0 ** 2, rs.standard_normal(k2.shape) / k2, 0.0)
    A = torch.from_numpy(A).to(device)
    kk = torch.from_numpy(k.astype(np.float64)).to(device)
    ll = torch.from_numpy(l.astype(np.float64)).to(device)
    i = torch.arange(1, Nx + 1, dtype=torch.float64, device=device)
    j = torch.arange(1, Ny + 1, dtype=torch.float64, device=device)
    Sx = torch.sin(math.pi / (Nx + 1) * kk.T * i[None, :])
    Sy = torch.sin(math.pi / (Ny + 1) * j[:, None] * ll.T)
    return (Sy @ A @ Sx).contiguous()


def _paper_problem(Nx, Ny, seed, device="cuda"):
    """(f, u) of the paper's test problem scaled by a seeded factor: u = -a e^{xy} on (Ny+4, Nx+4)
    nodes i, j = -1 .. N+2, f = -a (x^2 + y^2) e^{xy} at the interior nodes."""
    a = 0.5 + np.random.RandomState(seed % (2 ** 32)).uniform()
    h = 1.0 / (Nx + 1)
    x = torch.arange(-1, Nx + 3, dtype=torch.float64, device=device)[None, :] * h
    y = torch.arange(-1, Ny + 3, dtype=torch.float64, device=device)[:, None] * h
    e = a * torch.exp(x * y)
    f = -((x * x + y * y) * e)[2:-2, 2:-2].contiguous()
    return f, -e


def _problems(case, seed):
    """(Nx, Ny, st, tol, seed of the right-hand side) of a batch's or burst's problems."""
    rs = np.random.RandomState(case["pick"])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    out = []
    for q in range(case["n"]):
        nx, ny = (int(round(math.exp(v))) for v in rs.uniform(lo, hi, 2))
        if case["kind"] == "batch":
            st, tol = int(rs.choice([5, 9])), case["tol"]
        else:
            st, tol = int(rs.choice([5, 9, 17])), float(rs.choice([1e-6, 1e-10]))
        out.append((nx, ny, st, tol, 1000 * seed + q))
    return out


def _sweep_inputs(case, seed):
    """(right-hand side, start iterate) of the sweeps: FP32 inner cycles start at 0 on a smooth
    defect; FP64 and float-float sweeps smooth a rough iterate."""
    Nx, Ny = case["Nx"], case["Ny"]
    r = _rhs(Nx, Ny, seed)
    if case["prec"] == "mixed":
        return (r * 1e-6).float(), torch.zeros((Ny, Nx), dtype=torch.float32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = _rhs(Nx, Ny, seed + 17) * 0.05
    u += 1e-4 * torch.randn((Ny, Nx), generator=g, dtype=torch.float64, device="cuda")
    return r, u


# ------------------------------------------------------------------------------------ run side

class _Served:
    """A server that is closed with the state that holds it."""

    def __init__(self, budget, slots):
        self.s = cj.Server(budget, slots)

    def __del__(self):
        self.s.close()


def prepare(case, seed):
    if case["kind"] == "solve":
        Nx, Ny = case["Nx"], case["Ny"]
        data = case["bc"] == "data"
        plan = cj.Plan(Nx, Ny, case["st"], case["tol"], precision=_PREC[case["prec"]],
                       bc=cj.CJ_BC_DIRICHLET if data else cj.CJ_BC_DIRICHLET0)
        if data:
            f, g = _paper_problem(Nx, Ny, seed)
            cj.cj_set_boundary(plan.handle, g.contiguous())
        else:
            f = _rhs(Nx, Ny, seed)
        return dict(case=case, plan=plan, f=f, u=torch.zeros_like(f))
    if case["kind"] == "sweeps":
        kw = dict(precision=cj.CJ_FP32_INNER, inner_cycle=case["inner"]) if case["prec"] == "mixed" else {}
        plan = cj.Plan(case["Nx"], case["Ny"], case["st"], case["tol"], **kw)
        f, u0 = _sweep_inputs(case, seed)
        return dict(case=case, plan=plan, f=f, u0=u0, u=torch.empty_like(u0))
    probs = _problems(case, seed)
    if case["kind"] == "batch":
        ps = []
        for nx, ny, st, tol, s in probs:
            f = _rhs(nx, ny, s)
            ps.append(dict(Nx=nx, Ny=ny, st=st, tol=tol, f=f, u=torch.zeros_like(f)))
        return dict(case=case, problems=ps)
    reqs = [(_rhs(nx, ny, s, "cpu").numpy(), st, tol) for nx, ny, st, tol, s in probs]
    return dict(case=case, server=_Served(8 << 30, 64), requests=reqs)


def _told(res):
    """The numbers of a result that depend on the inputs alone."""
    return [res["sweeps"], res["cycles"], res["rc"], res["rel_res_l2"]]


def _together(us, results):
    """The grids of several problems, then their results' numbers in two arrays."""
    told = [_told(r) for r in results]
    return us + [np.array([t[:3] for t in told], dtype=np.int64), np.array([t[3] for t in told])]


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        u = state["u"].zero_()
        res = cj.cj_solve(state["plan"].handle, state["f"], u)
        return [u, _told(res)]
    if case["kind"] == "sweeps":
        u = state["u"].copy_(state["u0"])
        sweeps = {"f64": cj.cj_sweeps, "ff": cj.cj_sweeps_ff, "mixed": cj.cj_sweeps_f32}[case["prec"]]
        sweeps(state["plan"].handle, state["f"], u, case["first"], case["count"])
        return u
    if case["kind"] == "batch":
        for p in state["problems"]:
            p["u"].zero_()
        res = cj.cj_solve_batch(state["problems"])
        return _together([p["u"] for p in state["problems"]], res)
    server = state["server"].s
    tickets = [server.submit(f, st, tol) for f, st, tol in state["requests"]]
    us, told = [None] * len(tickets), [None] * len(tickets)
    waiting = list(range(len(tickets)))
    while waiting:
        for q in list(waiting):
            got = server.poll(tickets[q], state["requests"][q][0].shape)
            if got is not None:
                us[q], told[q] = got
                waiting.remove(q)
        if waiting:
            time.sleep(2e-4)
    return _together(us, told)


# ------------------------------------------------------------------------------- what it takes

def _kappa(st, Nx, Ny):
    """Ends of the spectrum of the Jacobi-normalised operator on the Nx x Ny grid."""
    def s2(x):
        return math.sin(x) ** 2
    hx, hy = math.pi / (2.0 * (Nx + 1)), math.pi / (2.0 * (Ny + 1))
    if st == 5:
        return s2(hx) + s2(hy), 2.0
    if st == 9:
        return 0.8 * (s2(hx) + s2(hy)) + 0.2 * (s2(hx + hy) + s2(hx - hy)), 1.6
    fx, fy = 2 * hx, 2 * hy
    return (-4.0 / 75.0 * (s2(fx) + s2(fy)) + 64.0 / 75.0 * (s2(hx) + s2(hy))
            - 1.0 / 75.0 * (s2(fx + fy) + s2(fx - fy)) + 16.0 / 75.0 * (s2(hx + hy) + s2(hx - hy))), 128.0 / 75.0


def _sweeps_needed(st, Nx, Ny, tol):
    """Smallest degree whose Chebyshev bound reaches tol."""
    a, b = _kappa(st, Nx, Ny)
    return math.ceil(math.acosh(1.0 / tol) / math.acosh((b + a) / (b - a)))


def _weights(st, Nx, Ny, M):
    """The M sweep weights, mirror-paired: every j of one level is followed by 2m + 1 - j."""
    a, b = _kappa(st, Nx, Ny)
    o = [1]
    while len(o) < M:
        m = len(o)
        o = [v for j in o for v in (j, 2 * m + 1 - j)]
    c = {5: 4.0, 9: 20.0 / 6.0, 17: 300.0 / 72.0}[st]
    th = (2.0 * np.array(o, dtype=np.float64) - 1.0) * math.pi / (2 * M)
    return 1.0 / (c * (0.5 * (b + a) + 0.5 * (b - a) * np.cos(th)))


def work(case):
    """Every grid read once and written once; a solve's operations are those of the sweeps whose
    Chebyshev bound reaches its tolerance."""
    if case["kind"] == "sweeps":
        n = case["Nx"] * case["Ny"]
        return {"bytes": n * (12 if case["prec"] == "mixed" else 24), "flops": n * case["count"] * _OPS[case["st"]]}
    if case["kind"] == "solve":
        probs = [(case["Nx"], case["Ny"], case["st"], case["tol"])]
    else:
        probs = [p[:4] for p in _problems(case, 0)]
    return {"bytes": sum(24 * nx * ny for nx, ny, _, _ in probs),
            "flops": sum(nx * ny * _OPS[st] * _sweeps_needed(st, nx, ny, tol) for nx, ny, st, tol in probs)}


# --------------------------------------------------------------------------------- exact values

def _padded(u, st, ring=None):
    """u with two rings around it: the given values, or homogeneous Dirichlet data (0, and the odd
    reflection in the outer ring, which only the 17-point stencil reads)."""
    Ny, Nx = u.shape
    if ring is not None:
        P = ring.clone()
    else:
        P = torch.zeros((Ny + 4, Nx + 4), dtype=torch.float64, device=u.device)
    P[2:-2, 2:-2] = u
    if ring is None and st == 17:
        P[2:-2, 0] = -u[:, 0]
        P[2:-2, -1] = -u[:, -1]
        P[0] = -P[2]
        P[-1] = -P[-3]
    return P


def _apply(P, st):
    """h^2 Delta_h on the interior of a padded array."""
    Ny, Nx = P.shape[0] - 4, P.shape[1] - 4

    def at(dx, dy):
        return P[2 + dy:2 + dy + Ny, 2 + dx:2 + dx + Nx]

    def axis(s):
        return at(s, 0) + at(-s, 0) + at(0, s) + at(0, -s)

    def diag(s):
        return at(s, s) + at(-s, s) + at(s, -s) + at(-s, -s)
    if st == 5:
        return axis(1) - 4.0 * at(0, 0)
    if st == 9:
        return (4.0 * axis(1) + diag(1) - 20.0 * at(0, 0)) / 6.0
    return (64.0 * axis(1) + 16.0 * diag(1) - 4.0 * axis(2) - diag(2) - 300.0 * at(0, 0)) / 72.0


def _dst(x):
    """Discrete sine transform along the last axis: sum_i x_i sin(pi k i / (N + 1))."""
    z = torch.zeros(x.shape[:-1] + (1,), dtype=x.dtype, device=x.device)
    return -0.5 * torch.fft.rfft(torch.cat([z, x, z, -x.flip(-1)], dim=-1)).imag[..., 1:-1]


def _solution(st, b):
    """The u with h^2 Delta_h u = b, u = 0 on the boundary."""
    Ny, Nx = b.shape
    cx = torch.cos(math.pi / (Nx + 1) * torch.arange(1, Nx + 1, dtype=torch.float64, device=b.device))[None, :]
    cy = torch.cos(math.pi / (Ny + 1) * torch.arange(1, Ny + 1, dtype=torch.float64, device=b.device))[:, None]
    if st == 5:
        lam = 2.0 * (cx - 1.0) + 2.0 * (cy - 1.0)
    elif st == 9:
        lam = (8.0 * (cx + cy) + 4.0 * cx * cy - 20.0) / 6.0
    else:
        dx, dy = 2.0 * cx * cx - 1.0, 2.0 * cy * cy - 1.0
        lam = (128.0 * (cx + cy) + 64.0 * cx * cy - 8.0 * (dx + dy) - 4.0 * dx * dy - 300.0) / 72.0
    t = _dst(_dst(b).T.contiguous()).T / lam
    t = _dst(_dst(t.contiguous()).T.contiguous()).T
    return (t * (4.0 / ((Nx + 1) * (Ny + 1)))).contiguous()


def exact(case, seed):
    if case["kind"] == "solve":
        Nx, Ny, st = case["Nx"], case["Ny"], case["st"]
        if case["bc"] == "data":
            f, g = _paper_problem(Nx, Ny, seed)
            b = f / (Nx + 1) ** 2 - _apply(_padded(torch.zeros_like(f), st, g), st)
        else:
            b = _rhs(Nx, Ny, seed) / (Nx + 1) ** 2
        return [_solution(st, b), [None] * 4]
    if case["kind"] == "sweeps":
        f, u = _sweep_inputs(case, seed)
        st, Nx, Ny = case["st"], case["Nx"], case["Ny"]
        if case["prec"] == "mixed":
            w = _weights(st, Nx, Ny, case["inner"]).astype(np.float32).astype(np.float64)
            b, u = f.double(), u.double()
        else:
            M = 1
            while M < _sweeps_needed(st, Nx, Ny, case["tol"]):
                M *= 2
            w, b = _weights(st, Nx, Ny, M), f / (Nx + 1) ** 2
        for n in range(case["first"], case["first"] + case["count"]):
            u = u + float(w[n % len(w)]) * (_apply(_padded(u, st), st) - b)
        return u
    out = []
    for nx, ny, st, tol, s in _problems(case, seed):
        dev = "cuda" if case["kind"] == "batch" else "cpu"
        u = _solution(st, _rhs(nx, ny, s, dev).cuda() / (nx + 1) ** 2)
        out.append(u if case["kind"] == "batch" else u.cpu().numpy())
    return out + [None, None]
