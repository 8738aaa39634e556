"""The calls this library's performance is measured on.

Each case is one pass through public entry points, at sizes of the workloads
this repository benchmarks and tests (the double integrator, the 2-D point
mass, the 4096-problem batch, the differentiable n = 8 problem, the n = 64
problem and the falling body on a state grid), from the smallest solve, where
launches and latency count, to the longest horizon.  Inputs are synthetic and
made from the seed alone.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what a program holds before the call
    run(state)          one pass; its outputs
    work(case)          bytes and FP64 operations the pass cannot do without
    exact(case, seed)   the outputs in plain 64-bit torch
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2212_11744_gb300 as lqt

CONST, PER_INTERVAL, PER_STAGE = 0, 1, 2
DEV = "cuda"
F64 = torch.float64


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------


def listed():
    return [
        # one control-loop solve: two states, a short horizon; latency and launches
        {"name": "solve_n2_T1024", "kind": "solve", "model": "integrator", "n": 2, "T": 1024, "K": 10},
        # the paper's experiment: the point mass, ten RK4 steps per block, an ordinary (ragged) block count
        {"name": "solve_n4_T10007", "kind": "solve", "model": "point_mass", "n": 4, "T": 10007, "K": 10},
        # the longest horizon: the benchmark's own workload
        {"name": "solve_n4_T1048576", "kind": "solve", "model": "point_mass", "n": 4, "T": 1 << 20, "K": 4},
        # every coefficient a function of time, an output matrix, a drift, an uneven grid
        {"name": "solve_general_n3_T3001", "kind": "solve", "model": "general", "n": 3, "T": 3001, "K": 4},
        # learning through the solver: forward, backward, all gradients
        {"name": "train_n8_T16384", "kind": "train", "model": "members", "n": 8, "T": 1 << 14, "K": 4},
        # one problem of middle size
        {"name": "solve_n16_T8192", "kind": "solve", "model": "members", "n": 16, "T": 8192, "K": 4},
        # a large state
        {"name": "solve_n64_T4096", "kind": "solve", "model": "large", "n": 64, "T": 4096, "K": 2},
        # the mixed-precision option on the same model, a shorter horizon
        {"name": "mixed_n64_T1000", "kind": "mixed", "model": "large", "n": 64, "T": 1000, "K": 2},
        # many independent problems of several state dimensions in one pass
        {"name": "batch_256", "kind": "batch", "model": "members", "count": 256, "T": 8192},
        # the solution at every RK4 step: a solve, then the dense output
        {"name": "densify_n4_T131072", "kind": "densify", "model": "point_mass", "n": 4, "T": 1 << 17, "K": 4},
        # host buffers in and out, the copies included
        {"name": "host_n4_T131072", "kind": "host", "model": "point_mass", "n": 4, "T": 1 << 17, "K": 4},
        # the nonlinear example on a state grid
        {"name": "grid_G201_T10000", "kind": "grid", "G": 201, "T": 10000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "train", "mixed", "batch", "densify", "host", "grid"])
    if kind == "batch":
        return {"kind": kind, "model": "members", "count": _log_int(rng, 16, 256), "T": _log_int(rng, 512, 8192)}
    if kind == "grid":
        return {"kind": kind, "G": _log_int(rng, 20, 201), "T": _log_int(rng, 100, 10000)}
    if kind == "train":
        return {"kind": kind, "model": "members", "n": rng.choice([2, 4, 8]), "T": _log_int(rng, 128, 1 << 14), "K": 4}
    if kind == "mixed":
        return {"kind": kind, "model": "large", "n": 64, "T": _log_int(rng, 64, 1000), "K": 2}
    if kind in ("densify", "host"):
        return {"kind": kind, "model": "point_mass", "n": 4, "T": _log_int(rng, 256, 1 << 17), "K": 4}
    model = rng.choice(["integrator", "point_mass", "general", "members", "members", "large"])
    if model == "integrator":
        return {"kind": kind, "model": model, "n": 2, "T": _log_int(rng, 64, 65536), "K": rng.choice([4, 10])}
    if model == "point_mass":
        return {"kind": kind, "model": model, "n": 4, "T": _log_int(rng, 256, 1 << 19), "K": rng.choice([4, 10])}
    if model == "general":
        return {"kind": kind, "model": model, "n": rng.choice([1, 2, 3, 4, 8]), "T": _log_int(rng, 100, 30000),
                "K": rng.choice([2, 4])}
    if model == "members":
        n = rng.choice([2, 4, 8, 16])
        return {"kind": kind, "model": model, "n": n, "T": _log_int(rng, 256, 8192 if n == 16 else 65536), "K": 4}
    return {"kind": kind, "model": "large", "n": 64, "T": _log_int(rng, 64, 4096), "K": 2}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------


class _Coef:
    def __init__(self, values, mode):
        self.values, self.mode = values, mode


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=F64)


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _problem(n, m, nr, T, K, t, co, Xf, rf, x0, Hf=None):
    """A problem object with torch (GPU) arrays; co: name -> (samples, mode)."""
    p = SimpleNamespace(n=n, m=m, nr=nr, T=T, K=K, t=t, Xf=Xf, rf=rf, Hf=Hf, x0=x0)
    for name in ("F", "L", "c", "H", "X", "U", "r"):
        v = co.get(name)
        setattr(p, name, None if v is None else _Coef(v[0].contiguous(), v[1]))
    return p


def _stage_times(t, K):
    f = torch.arange(2 * K, device=DEV, dtype=F64) / (2 * K)
    return torch.cat([(t[:-1, None] + (t[1:] - t[:-1])[:, None] * f).reshape(-1), t[-1:]])


def _sinusoids(g, tt, count):
    amp, freq, ph = _uniform(g, 0.5, 2.0, count), _uniform(g, 0.1, 1.0, count), _uniform(g, 0.0, 2 * math.pi, count)
    out = torch.zeros_like(tt)
    for a, f, q in zip(amp.tolist(), freq.tolist(), ph.tolist()):
        out += a * torch.sin(2 * math.pi * f * tt + q)
    return out


def _box(g, T, n, width):
    return _randn(g, T + width - 1, n).unfold(0, width, 1).mean(-1)


def _integrator(T, K, g):
    t = torch.linspace(0.0, 10.0, T + 1, device=DEV, dtype=F64)
    pos = _sinusoids(g, _stage_times(t, K), 3)
    r = torch.stack([pos, torch.zeros_like(pos)], 1)
    d = lambda *v: torch.tensor(v, device=DEV, dtype=F64)
    co = {"F": (d(0, 1, 0, 0).view(1, 2, 2), CONST), "L": (d(0, 1).view(1, 2, 1), CONST),
          "X": (torch.diag(d(1.0, 0.1))[None], CONST), "U": (d(0.01).view(1, 1, 1), CONST), "r": (r, PER_STAGE)}
    return _problem(2, 1, 2, T, K, t, co, 10.0 * torch.eye(2, device=DEV, dtype=F64), r[-1].clone(), _randn(g, 2))


def _point_mass(T, K, g):
    tf = 100.0 if K == 4 else 50.0
    t = torch.linspace(0.0, tf, T + 1, device=DEV, dtype=F64)
    ts = _stage_times(t, K)
    z = torch.zeros_like(ts)
    r = torch.stack([_sinusoids(g, ts, 5), _sinusoids(g, ts, 5), z, z], 1)
    phase = float(_uniform(g, 0.0, 2 * math.pi, 1))
    Xd = torch.diag(torch.tensor([1.0, 1.0, 0.01, 0.01], device=DEV, dtype=F64))
    X = (1.0 + 0.5 * torch.sin(ts + phase))[:, None, None] * Xd
    F = torch.zeros(1, 4, 4, device=DEV, dtype=F64)
    L = torch.zeros(1, 4, 2, device=DEV, dtype=F64)
    F[0, 0, 2] = F[0, 1, 3] = 1.0
    L[0, 2, 0] = L[0, 3, 1] = 1.0
    I = torch.eye(4, device=DEV, dtype=F64)
    co = {"F": (F, CONST), "L": (L, CONST), "X": (X, PER_STAGE), "U": (0.1 * I[None, :2, :2], CONST),
          "r": (r, PER_STAGE)}
    return _problem(4, 2, 4, T, K, t, co, I, r[-1].clone(), _randn(g, 4))


def _rotations(g, n, lo, hi):
    P, _ = torch.linalg.qr(_randn(g, n, n))
    D = torch.zeros(n, n, device=DEV, dtype=F64)
    a, w = _uniform(g, lo, hi, n), _uniform(g, 0.0, 1.0, n)
    for i in range(0, n - 1, 2):
        D[i, i] = D[i + 1, i + 1] = a[i]
        D[i, i + 1], D[i + 1, i] = w[i], -w[i]
    if n % 2:
        D[-1, -1] = a[-1]
    return P @ D @ P.T


def _member(n, T, K, g, step=0.05, stable=False):
    """A time-invariant problem with dense random F, L, X, U and a smoothed
    random reference, one sample per sub-interval."""
    m = max(1, n // 2)
    F = _rotations(g, n, -1.0, -0.1 if stable else 0.2)
    L = _randn(g, n, m) / math.sqrt(n)
    if stable:
        X, U = torch.diag(_uniform(g, 0.5, 2.0, n)), torch.diag(_uniform(g, 0.05, 0.5, m))
    else:
        G, H = _randn(g, n, n), _randn(g, m, m)
        X = G @ G.T + 0.1 * torch.eye(n, device=DEV, dtype=F64)
        U = H @ H.T + 0.1 * torch.eye(m, device=DEV, dtype=F64)
    r = _box(g, T, n, 32)
    t = torch.linspace(0.0, step * T, T + 1, device=DEV, dtype=F64)
    co = {"F": (F[None], CONST), "L": (L[None], CONST), "X": (X[None], CONST), "U": (U[None], CONST),
          "r": (r, PER_INTERVAL)}
    return _problem(n, m, n, T, K, t, co, X.clone(), None if stable else r[-1].clone(), _randn(g, n))


def _large(n, T, K, g):
    m = n // 4
    I = torch.eye(n, device=DEV, dtype=F64)
    r = _box(g, T, n, 64)
    t = torch.linspace(0.0, 0.02 * T, T + 1, device=DEV, dtype=F64)
    co = {"F": (-0.5 * I[None] + _randn(g, 1, n, n) / math.sqrt(n), CONST),
          "L": (_randn(g, 1, n, m) / math.sqrt(n), CONST), "X": (I[None], CONST), "U": (0.1 * I[None, :m, :m], CONST),
          "r": (r, PER_INTERVAL)}
    return _problem(n, m, n, T, K, t, co, I, r[-1].clone(), _randn(g, n))


def _general(n, T, K, g):
    """Every coefficient a smooth function of time on the half-step grid, an
    output matrix H, a drift c, full X and U, uneven sub-intervals."""
    m, nr = max(1, n // 2), max(1, n - 1)
    d = _uniform(g, 0.5, 1.5, T)
    t = torch.cat([torch.zeros(1, device=DEV, dtype=F64), d.cumsum(0)])
    t = t * (2.0 / t[-1])
    ts = _stage_times(t, K)
    w = _uniform(g, 0.5, 2.0, 6).tolist()
    s = lambda i: torch.sin(w[i] * ts)
    GX, GU, GF = _randn(g, nr, nr), _randn(g, m, m), _randn(g, nr, nr)
    I = lambda k: torch.eye(k, device=DEV, dtype=F64)
    mix = lambda a, b, f: a[None] + b[None] * f.view((-1,) + (1,) * a.dim())
    X0, U0 = GX @ GX.T / nr + 0.2 * I(nr), GU @ GU.T / m + 0.3 * I(m)
    co = {"F": (mix(0.6 * _randn(g, n, n), 0.3 * _randn(g, n, n), s(0)), PER_STAGE),
          "L": (mix(_randn(g, n, m), 0.3 * _randn(g, n, m), s(1)), PER_STAGE),
          "c": (mix(_randn(g, n), 0.5 * _randn(g, n), s(2)), PER_STAGE),
          "H": (mix(_randn(g, nr, n), 0.2 * _randn(g, nr, n), s(3)), PER_STAGE),
          "X": (mix(X0, 0.5 * X0, s(4)), PER_STAGE), "U": (mix(U0, 0.3 * U0, s(5)), PER_STAGE),
          "r": (_randn(g, nr) * torch.sin(ts[:, None] * _uniform(g, 0.5, 3.0, nr) + 1.0), PER_STAGE)}
    return _problem(n, m, nr, T, K, t, co, GF @ GF.T / nr + 0.5 * I(nr), _randn(g, nr), _randn(g, n),
                    Hf=_randn(g, nr, n))


def _make(case, g):
    T, K, n = case["T"], case["K"], case["n"]
    if case["model"] == "integrator":
        return _integrator(T, K, g)
    if case["model"] == "point_mass":
        return _point_mass(T, K, g)
    if case["model"] == "general":
        return _general(n, T, K, g)
    if case["model"] == "large":
        return _large(n, T, K, g)
    return _member(n, T, K, g, 0.01, True) if case["kind"] == "train" else _member(n, T, K, g)


def _batch_shapes(case):
    """(n, T) of each problem: dimensions 2, 4, 8, 16 in turn, lengths spread
    over T/32 .. T (the golden ratio's multiples, so no order in them)."""
    lo = max(2, case["T"] // 32)
    return [((2, 4, 8, 16)[b % 4], lo + int((b * 0.6180339887498949) % 1.0 * (case["T"] - lo)))
            for b in range(case["count"])]


def _batch_problems(case, seed):
    g = _gen(seed)
    return [_member(n, T, 4, g) for n, T in _batch_shapes(case)]


def _grid_problem(case, seed):
    """The falling body on [-6, 6]; gravity and weights vary with the seed."""
    rng = np.random.default_rng(seed)
    G = case["G"]
    return SimpleNamespace(G=G, x_min=-6.0, dx=12.0 / (G - 1), d0=float(rng.uniform(0.8, 1.2)), d1=0.0,
                           d2=-float(rng.uniform(0.08, 0.12)), q=float(rng.uniform(0.8, 1.2)), rho=1.0, qf=4.0,
                           tau=0.1, substeps=10, T=case["T"], interp=True)


def _to_numpy(p):
    """The same problem with numpy arrays, as the binding's constructors take them."""
    num = lambda a: None if a is None else a.cpu().numpy()
    q = SimpleNamespace(n=p.n, m=p.m, nr=p.nr, T=p.T, K=p.K, t=num(p.t), Xf=num(p.Xf), rf=num(p.rf), Hf=num(p.Hf),
                        x0=num(p.x0))
    for name in ("F", "L", "c", "H", "X", "U", "r"):
        co = getattr(p, name)
        setattr(q, name, None if co is None else _Coef(num(co.values), co.mode))
    return q


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(kind=kind)
    if kind == "grid":
        s.g = _grid_problem(case, seed)
        s.wb = torch.empty(lqt.lqt_grid_workspace_size(s.g, 0), dtype=torch.uint8, device=DEV)
        s.wv = torch.empty(lqt.lqt_grid_workspace_size(s.g, 1), dtype=torch.uint8, device=DEV)
        s.Vb = torch.empty(s.g.G, s.g.G, dtype=F64, device=DEV)
        s.V = torch.empty(s.g.T + 1, s.g.G, dtype=F64, device=DEV)
        return s
    if kind == "batch":
        from paper_2212_11744_gb300.batch import BatchSet
        s.batch = BatchSet([_to_numpy(p) for p in _batch_problems(case, seed)])
        s.out = s.batch.new_outputs()
        return s
    p = _make(case, _gen(seed))
    if kind == "train":
        s.template = p
        s.target = _randn(_gen(seed + 1), p.n)
        s.params = [a.requires_grad_() for a in (p.F.values, p.L.values, p.X.values, p.U.values, p.r.values, p.Xf, p.x0)]
        return s
    q = _to_numpy(p)
    if kind == "host":
        s.hp = lqt.HostProblem(q)
        s.out = lqt.host_solution(s.hp)
        s.ws = torch.empty(lqt.lqt_workspace_size(s.hp, lqt.LQT_WS_SOLVE) + lqt.lqt_host_staging_size(s.hp) + 4096,
                           dtype=torch.uint8, device=DEV)
        return s
    s.dp = lqt.DeviceProblem(q)
    s.ws = torch.empty(lqt.lqt_workspace_size(s.dp, lqt.LQT_WS_SOLVE), dtype=torch.uint8, device=DEV)
    s.out = lqt.new_solution(s.dp)
    if kind == "densify":
        s.dense = lqt.new_dense(s.dp)
        s.wd = torch.empty(lqt.lqt_workspace_size(s.dp, lqt.LQT_WS_DENSIFY), dtype=torch.uint8, device=DEV)
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------


def run(s):
    if s.kind == "solve":
        return lqt.lqt_solve(s.dp, out=s.out, ws=s.ws)
    if s.kind == "mixed":
        return lqt.lqt_solve_mixed(s.dp, out=s.out, ws=s.ws)
    if s.kind == "densify":
        sol = lqt.lqt_solve(s.dp, out=s.out, ws=s.ws)
        return {"sol": sol, "dense": lqt.lqt_densify(s.dp, sol, out=s.dense, ws=s.wd)}
    if s.kind == "host":
        return lqt.lqt_solve_host(s.hp, s.ws, out=s.out)
    if s.kind == "batch":
        return {"n%d" % n: o for n, o in s.batch.solve(s.out).items()}
    if s.kind == "grid":
        lqt.lqt_grid_block(s.g, out=s.Vb, ws=s.wb)
        return {"block": s.Vb, "values": lqt.lqt_grid_values(s.g, s.Vb, out=s.V, ws=s.wv)}
    from paper_2212_11744_gb300.autograd import LQTSolve
    F, L, X, U, r, Xf, x0 = s.params
    S, v, zeta, x, cost = LQTSolve.apply(s.template, F, L, X, U, r, Xf, None, x0)
    loss = cost + ((x[-1] - s.target) ** 2).sum()
    grads = torch.autograd.grad(loss, s.params)
    return {"S": S.detach(), "v": v.detach(), "zeta": zeta.detach(), "x": x.detach(), "cost": cost.detach(),
            "grads": dict(zip(("F", "L", "X", "U", "r", "Xf", "x0"), grads))}


# --------------------------------------------------------------------------
# the work
# --------------------------------------------------------------------------


def _flops_build(n, m, K):
    return K * (40.0 * n ** 3 + 60.0 * n ** 2)


def _flops_solve(n, m, K):
    return _flops_build(n, m, K) + 31.0 * n ** 3 + 2.0 * m * n


def _bytes_problem(case):
    """Inputs read and outputs written by one solve, in doubles."""
    n, T, K = case["n"], case["T"], case["K"]
    model = case["model"]
    m = {"integrator": 1, "large": n // 4}.get(model, max(1, n // 2))
    stages = 2 * K * T + 1
    ins = {"integrator": stages * n, "point_mass": stages * (n * n + n), "members": T * n, "large": T * n,
           "general": stages * (n * n + n * m + n + max(1, n - 1) * n + max(1, n - 1) ** 2 + m * m + max(1, n - 1))}[model]
    return m, T + ins, (T + 1) * (n * n + 2 * n + 1 + m)


def work(case):
    kind = case["kind"]
    if kind == "grid":
        G, T = case["G"], case["T"]
        L = T.bit_length()
        pops = sum(bin(e).count("1") for e in range(1, T + 1))
        flops = (9 + L - 1) * (float(G) ** 3 + 16.0 * G * G) + pops * (float(G) * G + 16.0 * G)
        return {"bytes": 8.0 * (G * G + (T + 1) * G), "flops": flops}
    if kind == "batch":
        flops = nbytes = 0.0
        for n, T in _batch_shapes(case):
            flops += T * _flops_solve(n, n // 2, 4)
            nbytes += 8.0 * T * (1 + n + n * n + 2 * n + 1 + n // 2)
        return {"bytes": nbytes, "flops": flops}
    n, T, K = case["n"], case["T"], case["K"]
    m, ins, outs = _bytes_problem(case)
    flops = T * _flops_solve(n, m, K)
    if kind == "train":
        flops += T * (3.0 * _flops_build(n, m, K) + 62.0 * n ** 3)
        outs += T * n
    elif kind == "densify":
        flops += T * K * (4.0 * (2 * n ** 3 + 4 * n * n * m + 2 * n * n + 4 * n * m) + 4.0 * (2 * n * n + 4 * n * m))
        outs += (T * K + 1) * (n * n + 2 * n + 1 + m)
    return {"bytes": 8.0 * (ins + outs), "flops": flops}


# --------------------------------------------------------------------------
# the same results in plain 64-bit torch
# --------------------------------------------------------------------------


def _sym(a):
    return 0.5 * (a + a.mT)


def _mv(a, x):
    return (a @ x.unsqueeze(-1)).squeeze(-1)


def _sample(co, T, K, p):
    """The samples of every sub-interval at half-step p: [T, ...]."""
    if co.mode == CONST:
        return co.values[0].expand((T,) + tuple(co.values.shape[1:]))
    if co.mode == PER_INTERVAL:
        return co.values
    return co.values[torch.arange(T, device=DEV) * (2 * K) + p]


def _at(prob, p):
    """(F, B, c, Q, q, rho, G) of every sub-interval at half-step p, with
    B = L U^-1 L', Q = H'XH, q = H'Xr, rho = r'Xr, G = U^-1 L'."""
    T, K, n = prob.T, prob.K, prob.n
    F, L, X, U = (_sample(getattr(prob, k), T, K, p) for k in ("F", "L", "X", "U"))
    G = torch.linalg.solve(U, L.mT)
    r = _sample(prob.r, T, K, p)
    Xr = _mv(X, r)
    Q, q = X, Xr
    if prob.H is not None:
        H = _sample(prob.H, T, K, p)
        Q, q = H.mT @ X @ H, _mv(H.mT, Xr)
    c = _sample(prob.c, T, K, p) if prob.c is not None else torch.zeros(T, n, device=DEV, dtype=F64)
    return F, _sym(L @ G), c, _sym(Q), q, (r * Xr).sum(-1), G


def _element_rhs(y, k):
    A, b, C, eta, J, z = y
    F, B, c, Q, q, rho, _ = k
    BJ = B @ J
    Be = _mv(B, eta) + c
    return (A @ BJ - A @ F, -_mv(A, Be), _sym(-(A @ B) @ A.mT),
            -q - _mv(F.mT, eta) + _mv(J, Be), _sym(J @ BJ - F.mT @ J - J @ F - Q),
            -0.5 * rho + 0.5 * (eta * _mv(B, eta)).sum(-1) + (eta * c).sum(-1))


def _value_rhs(y, k):
    S, v, z = y
    F, B, c, Q, q, rho, _ = k
    Bv = _mv(B, v) + c
    return (_sym(S @ B @ S - F.mT @ S - S @ F - Q), -q - _mv(F.mT, v) + _mv(S, Bv),
            -0.5 * rho + 0.5 * (v * _mv(B, v)).sum(-1) + (v * c).sum(-1))


def _axpy(y, s, k):
    return tuple(a + s.view((-1,) + (1,) * (a.dim() - 1)) * d for a, d in zip(y, k))


def _rk4_back(rhs, y, h, c2, c1, c0):
    """One step from s + h to s; also the slope at its start."""
    k1 = rhs(y, c2)
    k2 = rhs(_axpy(y, -0.5 * h, k1), c1)
    k3 = rhs(_axpy(y, -0.5 * h, k2), c1)
    k4 = rhs(_axpy(y, -h, k3), c0)
    return _axpy(y, -h / 6.0, [a + 2.0 * b + 2.0 * c + d for a, b, c, d in zip(k1, k2, k3, k4)]), k1


def _elements(prob):
    """The T conditional value functions and the terminal element: [T+1, ...]."""
    n, T, K = prob.n, prob.T, prob.K
    h = (prob.t[1:] - prob.t[:-1]) / K
    z = lambda *s: torch.zeros(T, *s, device=DEV, dtype=F64)
    y = (torch.eye(n, device=DEV, dtype=F64).expand(T, n, n), z(n), z(n, n), z(n), z(n, n), z())
    constant = all(co is None or co.mode != PER_STAGE for co in (prob.F, prob.L, prob.c, prob.H, prob.X, prob.U, prob.r))
    k2 = k1 = k0 = _at(prob, 2 * K)
    for i in range(K - 1, -1, -1):
        if not constant:
            k1, k0 = _at(prob, 2 * i + 1), _at(prob, 2 * i)
        y, _ = _rk4_back(_element_rhs, y, h, k2, k1, k0)
        k2 = k0
    Hf = prob.Hf if prob.Hf is not None else torch.eye(n, device=DEV, dtype=F64)
    rf = prob.rf if prob.rf is not None else torch.zeros(prob.nr, device=DEV, dtype=F64)
    o = lambda *s: torch.zeros(*s, device=DEV, dtype=F64)
    end = (o(n, n), o(n), o(n, n), Hf.T @ (prob.Xf @ rf), _sym(Hf.T @ prob.Xf @ Hf), 0.5 * rf @ (prob.Xf @ rf))
    return tuple(torch.cat([a, e[None]]) for a, e in zip(y, end))


def _combine(e1, e2):
    A1, b1, C1, n1, J1, z1 = e1
    A2, b2, C2, n2, J2, z2 = e2
    n = A1.shape[-1]
    W = C1 @ J2 + torch.eye(n, device=DEV, dtype=F64)
    R = torch.linalg.solve(W, torch.cat([A1, C1, (b1 + _mv(C1, n2)).unsqueeze(-1)], -1))
    M, MC, z0 = R[..., :n], R[..., n:2 * n], R[..., 2 * n]
    Jz = _mv(J2, z0)
    lam = Jz - n2
    return (A2 @ M, _mv(A2, z0) + b2, _sym(A2 @ MC @ A2.mT + C2), _mv(M.mT, n2 - _mv(J2, b1)) + n1,
            _sym(M.mT @ (J2 @ A1) + J1),
            z1 + z2 + 0.5 * (lam * _mv(C1, lam)).sum(-1) + 0.5 * (z0 * Jz).sum(-1) - (z0 * n2).sum(-1))


def _scan(op, e):
    """Inclusive prefixes along the leading axis."""
    N = e[0].shape[0]
    if N == 1:
        return e
    half = _scan(op, op(tuple(a[0:N - 1:2] for a in e), tuple(a[1::2] for a in e)))
    out = [e_[:1] for e_ in e]
    if N > 2:
        more = op(tuple(a[:(N - 1) // 2] for a in half), tuple(a[2::2] for a in e))
        out = [torch.cat([a, b]) for a, b in zip(out, more)]
    full = []
    for even, odd in zip(out, half):
        k = odd.shape[0]
        both = torch.stack([even[:k], odd], 1).reshape((2 * k,) + tuple(odd.shape[1:]))
        full.append(both if even.shape[0] == k else torch.cat([both, even[k:]]))
    return tuple(full)


def _compose(f, g):
    """x -> g(f(x)) of affine maps."""
    return g[0] @ f[0], _mv(g[0], f[1]) + g[1]


def _solve64(el, x0):
    """Values, states and cost from elements [N, *batch, ...] and x0 [*batch, n]."""
    back = tuple(a.flip(0) for a in el)
    suf = _scan(lambda a, b: _combine(b, a), back)
    S, v, zeta = (suf[i].flip(0) for i in (4, 3, 5))
    A, b, C = (a[:-1] for a in el[:3])
    n = A.shape[-1]
    W = C @ S[1:] + torch.eye(n, device=DEV, dtype=F64)
    R = torch.linalg.solve(W, torch.cat([A, (b + _mv(C, v[1:])).unsqueeze(-1)], -1))
    P, a = _scan(_compose, (R[..., :n], R[..., n]))
    x = torch.cat([x0[None], _mv(P, x0) + a])
    cost = zeta[0] + 0.5 * (x0 * _mv(S[0], x0)).sum(-1) - (v[0] * x0).sum(-1)
    return S, v, zeta, x, cost


def _gains(prob):
    """U^-1 L' at the T+1 boundaries."""
    G0, GT = _at(prob, 0)[6], _at(prob, 2 * prob.K)[6][-1:]
    return torch.cat([G0, GT])


def _solution64(prob):
    S, v, zeta, x, cost = _solve64(_elements(prob), prob.x0)
    u = _mv(_gains(prob), v - _mv(S, x))
    return {"S": S, "v": v, "zeta": zeta, "x": x, "u": u, "cost": cost.reshape(1)}


def _dense64(prob, sol):
    """The solution at every RK4 step: values backward from each boundary, the
    closed loop forward with cubic Hermite midpoints."""
    T, K = prob.T, prob.K
    h = (prob.t[1:] - prob.t[:-1]) / K
    co = [_at(prob, p) for p in range(2 * K + 1)]
    Y, D = [None] * (K + 1), [None] * (K + 1)
    Y[K] = tuple(sol[k][1:] for k in ("S", "v", "zeta"))
    for i in range(K - 1, -1, -1):
        Y[i], D[i + 1] = _rk4_back(_value_rhs, Y[i + 1], h, co[2 * i + 2], co[2 * i + 1], co[2 * i])
    D[0] = _value_rhs(Y[0], co[0])
    loop = lambda y, x, k: _mv(k[0], x) + _mv(k[1], y[1] - _mv(y[0], x)) + k[2]
    hv = h[:, None]
    x = sol["x"][:-1]
    parts = {k: [] for k in ("S", "v", "zeta", "x", "u")}
    for i in range(K):
        y = tuple(sol[k][:-1] for k in ("S", "v", "zeta")) if i == 0 else Y[i]
        for k, a in zip(("S", "v", "zeta", "x", "u"), y + (x, _mv(co[2 * i][6], y[1] - _mv(y[0], x)))):
            parts[k].append(a)
        mid = tuple(0.5 * (a + b) + _axpy((torch.zeros_like(da),), h / 8.0, (da - db,))[0]
                    for a, b, da, db in zip(Y[i], Y[i + 1], D[i], D[i + 1]))
        k1 = loop(Y[i], x, co[2 * i])
        k2 = loop(mid, x + 0.5 * hv * k1, co[2 * i + 1])
        k3 = loop(mid, x + 0.5 * hv * k2, co[2 * i + 1])
        k4 = loop(Y[i + 1], x + hv * k3, co[2 * i + 2])
        x = x + hv / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    return {k: torch.cat([torch.stack(a, 1).reshape((T * K,) + tuple(a[0].shape[1:])), sol[k][-1:]])
            for k, a in parts.items()}


def _train64(prob, target):
    prm = [prob.F.values, prob.L.values, prob.X.values, prob.U.values, prob.r.values, prob.Xf, prob.x0]
    for a in prm:
        a.requires_grad_()
    S, v, zeta, x, cost = _solve64(_elements(prob), prob.x0)
    grads = torch.autograd.grad(cost + ((x[-1] - target) ** 2).sum(), prm)
    return {"S": S.detach(), "v": v.detach(), "zeta": zeta.detach(), "x": x.detach(), "cost": cost.detach(),
            "grads": dict(zip(("F", "L", "X", "U", "r", "Xf", "x0"), grads))}


def _batch64(problems):
    """Per dimension, the problems' results laid end to end.  Problems of one
    dimension are padded behind their terminal element with identities."""
    out = {}
    for n in sorted({p.n for p in problems}):
        ps = [p for p in problems if p.n == n]
        N = max(p.T for p in ps) + 1
        pad = []
        for p in ps:
            el = _elements(p)
            k = N - el[0].shape[0]
            eye = torch.eye(n, device=DEV, dtype=F64).expand(k, n, n)
            pad.append([torch.cat([a, eye if i == 0 else a.new_zeros((k,) + tuple(a.shape[1:]))])
                        for i, a in enumerate(el)])
        el = tuple(torch.stack([q[i] for q in pad], 1) for i in range(6))
        del pad
        S, v, zeta, x, cost = _solve64(el, torch.stack([p.x0 for p in ps]))
        G = torch.stack([p_[6][0] for p_ in (_at(p, 0) for p in ps)])
        u = _mv(G.expand((N,) + tuple(G.shape)), v - _mv(S, x))
        out["n%d" % n] = {k: torch.cat([a[:p.T + 1, b] for b, p in enumerate(ps)])
                          for k, a in (("S", S), ("v", v), ("zeta", zeta), ("x", x), ("u", u))}
        out["n%d" % n]["cost"] = cost
    return out


def _grid_refine(best, k, gm, g0, gp, fm, f0, fp, G, dx):
    a = (gp + gm - 2.0 * g0) / (2.0 * dx * dx) + (fp + fm - 2.0 * f0) / (2.0 * dx * dx)
    b = (gp - gm) / (2.0 * dx) + (fp - fm) / (2.0 * dx)
    ok = (k > 0) & (k < G - 1) & (a > 0)
    return torch.where(ok, best - b * b / (4.0 * torch.where(ok, a, torch.ones_like(a))), best)


def _grid_combine(A, B, dx):
    G = A.shape[0]
    best, k = (A[:, :, None] + B[None]).min(1)
    i = torch.arange(G, device=DEV)[:, None]
    j = torch.arange(G, device=DEV)[None]
    lo, hi = (k - 1).clamp_min(0), (k + 1).clamp_max(G - 1)
    return _grid_refine(best, k, A[i, lo], A[i, k], A[i, hi], B[lo, j], B[k, j], B[hi, j], G, dx)


def _grid64(g):
    G, dt = g.G, g.tau / g.substeps
    x = g.x_min + g.dx * torch.arange(G, device=DEV, dtype=F64)
    drift = g.d0 + g.d1 * x + g.d2 * x * x
    u = (x[None] - x[:, None]) / dt - drift[:, None]
    C = dt * 0.5 * (g.q * x[:, None] ** 2 + g.rho * u * u)
    V = C
    for _ in range(1, g.substeps):
        V = _grid_combine(V, C, g.dx)
    w = (0.5 * g.qf * x * x).repeat(g.T + 1, 1)
    e = g.T - torch.arange(g.T + 1, device=DEV)
    P, l, j = V, 0, torch.arange(G, device=DEV)[None]
    while (1 << l) <= g.T:
        if l:
            P = _grid_combine(P, P, g.dx)
        for rows in torch.nonzero((e >> l) & 1).squeeze(1).split(1024):
            f = w[rows]
            best, k = (P[None] + f[:, None, :]).min(2)
            lo, hi = (k - 1).clamp_min(0), (k + 1).clamp_max(G - 1)
            w[rows] = _grid_refine(best, k, P[j, lo], P[j, k], P[j, hi], f.gather(1, lo), f.gather(1, k),
                                   f.gather(1, hi), G, g.dx)
        l += 1
    return {"block": V, "values": w}


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        return _grid64(_grid_problem(case, seed))
    if kind == "batch":
        with torch.no_grad():
            return _batch64(_batch_problems(case, seed))
    p = _make(case, _gen(seed))
    if kind == "train":
        return _train64(p, _randn(_gen(seed + 1), p.n))
    with torch.no_grad():
        sol = _solution64(p)
        return {"sol": sol, "dense": _dense64(p, sol)} if kind == "densify" else sol
