"""Measured cases of the HOSC cavity solver: what a program that uses the library has it do.

Every case goes through the public entry points (the binding's functions, ``Cavity`` and
``serve.Pool``), from state tensors on the GPU to result tensors on the GPU:

* ``march``: load a state (velocity, temperature, pressure), take ``steps`` pseudo-time steps, read
  the state back. All-FP64 and mixed precision, FP32 sweeps and FP64 defect sweeps, Newtonian and
  power-law fluids, cubes and boxes, the options of the parameters (time-level history, Jacobi row
  scaling, BiCGSTAB(2)).
* ``solve``: march to the steady state from a start state and evaluate the diagnostics.
* ``batch``: one round of a pool of uneven cavities.
* ``systems``: the allocation-free solve of four caller-owned linear systems.

All-FP64 runs and FP64 defect sweeps hand back the state in 64 bits. A mixed run in FP32 sweeps hands
back 32-bit snapshots, as a program that keeps or draws them does: its increments are solved in
32 bits, and so is what ``exact`` (64 bits throughout) is compared with.

Start states are seeded, smooth and shaped like developed cavity flow: no-slip solenoidal rolls at
the speeds of converged cavities, a temperature between the hot and the cold wall with adiabatic
side walls, a pressure with zero normal gradient.
"""

import math
import random

import torch

from paper_2411_06563_gb300 import hosc as H
from paper_2411_06563_gb300 import serve as S

STATE = (("u", H.HOSC_U), ("v", H.HOSC_V), ("w", H.HOSC_W), ("th", H.HOSC_THETA), ("p", H.HOSC_P))
PREV = (("L", H.HOSC_PREV_L), ("u", H.HOSC_PREV_U), ("v", H.HOSC_PREV_V), ("w", H.HOSC_PREV_W),
        ("Eu", H.HOSC_PREV_EU), ("Ev", H.HOSC_PREV_EV), ("Ew", H.HOSC_PREV_EW))


def _march(name, N, Ra, n, steps, precision="mixed", phase=0, history=0, Ly=1.0, Lz=1.0,
           precond=0, solver=0):
    c = dict(kind="march", N=N, Ra=Ra, n=n, steps=steps, precision=precision, phase=phase,
             history=history, Ly=Ly, Lz=Lz, precond=precond, solver=solver)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the Newtonian 21^3 cavity, one step per call: a program that looks at the state after
        # every step; the smallest call, launches and latency count
        _march("newtonian21_fp64", 21, 1e3, 1.0, 1, "fp64"),
        # the same cavity solved to its steady state in FP64, with the Nusselt, entropy and Bejan
        # numbers: a whole solve as it is served
        dict(kind="solve", name="steady21_fp64", N=21, Ra=1e3, n=1.0),
        # the shear-thickening 41^3 cavity in FP64: the reference run of a parameter study
        _march("thickening41_fp64", 41, 1e4, 1.25, 4, "fp64"),
        # a box with three spacings and BiCGSTAB(2), restarted between writes of the state; an
        # even grid
        _march("box34_fp64_bicgstab2", 34, 5e3, 0.8, 2, "fp64", Ly=0.7, Lz=1.4, solver=1),
        # the paper's finest grid with the three-level time terms, FP64, restarted from a
        # checkpoint with its history: the time-accurate march
        _march("history91_fp64", 91, 1e4, 0.75, 1, "fp64", history=1),
        # the caller's own linear systems on the largest grid of the allocation-free solve
        dict(kind="systems", name="noalloc41", N=41, Ra=1e4, n=0.8),
        # the shear-thinning 41^3 cavity in mixed precision: a member of a study, many steps per
        # call
        _march("thinning41_mixed", 41, 1e4, 0.75, 8),
        # an even, mid-sized grid with Jacobi row scaling
        _march("jacobi64_mixed", 64, 2e4, 1.25, 4, precond=1),
        # the single large cavity of the benchmark, FP32 sweeps (the start of its solve)
        _march("cavity101_mixed", 101, 1e5, 0.75, 4),
        # the same cavity in FP64 defect sweeps: most steps of its steady solve
        _march("cavity101_defect", 101, 1e5, 0.75, 2, phase=1),
        # a cavity whose vectors are far larger than the L2 cache
        _march("cavity257_mixed", 257, 1e5, 0.75, 1),
        # a round of a pool of uneven cavities (the sizes of the batch workload)
        dict(kind="batch", name="batch16_mixed", members=16, largest=61, rounds=1),
    ]


def draw(rng):
    """One more case of the same ranges: sizes over the logarithm of their range, odd and even,
    Ra over three decades, the indices and options in use."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    Ra = 10.0 ** rng.uniform(2.0, 5.0)
    n = rng.choice((0.75, 0.9, 1.0, 1.1, 1.25))
    kind = rng.choice(("fp64", "fp64", "mixed", "mixed", "defect", "box", "batch", "systems"))
    if kind == "fp64":
        return _march(None, size(9, 101), Ra, n, rng.randint(1, 4), "fp64",
                      history=rng.randint(0, 1), solver=rng.choice((0, 0, 1)))
    if kind == "mixed":
        return _march(None, size(11, 200), Ra, n, rng.randint(1, 8), precond=rng.choice((0, 0, 1)))
    if kind == "defect":
        return _march(None, size(21, 110), Ra, n, rng.randint(1, 4), phase=1)
    if kind == "box":
        return _march(None, size(13, 70), Ra, n, rng.randint(1, 4), rng.choice(("fp64", "mixed")),
                      Ly=rng.uniform(0.6, 1.6), Lz=rng.uniform(0.6, 1.6))
    if kind == "batch":
        return dict(kind="batch", members=rng.randint(2, 16), largest=rng.choice((31, 41, 61)),
                    rounds=rng.randint(1, 2))
    return dict(kind="systems", N=size(9, 41), Ra=Ra, n=n)


# ------------------------------------------------------------------ start states

def _outer(fx, fy, fz):
    return fz[:, None, None] * fy[None, :, None] * fx[None, None, :]


def _state(N, Ra, n, seed, Ly=1.0, Lz=1.0):
    """u, v, w, th, p on N^3 nodes of the box 1 x Ly x Lz, tensors indexed [z, y, x]."""
    rng = random.Random(seed)
    x = torch.linspace(0.0, 1.0, N, dtype=torch.float64, device="cuda")
    pi = math.pi

    def bump(k):   # zero with its slope at both ends, and its derivative
        f = torch.sin(pi * x) * torch.sin(k * pi * x)
        d = pi * torch.cos(pi * x) * torch.sin(k * pi * x) + \
            k * pi * torch.sin(pi * x) * torch.cos(k * pi * x)
        f[0] = f[-1] = d[0] = d[-1] = 0.0
        return f, d

    env = torch.sin(pi * x)
    env[0] = env[-1] = 0.0
    u = torch.zeros(N, N, N, dtype=torch.float64, device="cuda")
    v, w = torch.zeros_like(u), torch.zeros_like(u)
    for kx, ky, a in ((1, 1, 1.0), (2, 1, 0.3), (1, 2, 0.3), (2, 3, 0.15)):   # rolls in x-y
        a *= rng.uniform(0.6, 1.0) * rng.choice((-1.0, 1.0) if kx + ky > 2 else (1.0,))
        (fx, dx), (fy, dy) = bump(kx), bump(ky)
        u += a * _outer(fx, dy / Ly, env)
        v -= a * _outer(dx, fy, env)
    for ky, kz, a in ((1, 2, 0.2), (2, 1, 0.2)):                              # and in y-z
        a *= rng.uniform(-1.0, 1.0)
        (fy, dy), (fz, dz) = bump(ky), bump(kz)
        v += a * _outer(env, fy, dz / Lz)
        w -= a * _outer(env, dy / Ly, fz)
    # peak speed of converged cavities: 0.12 * 2^(4 (1 - n)) sqrt(Ra)
    scale = 0.12 * 2.0 ** (4.0 * (1.0 - n)) * math.sqrt(max(Ra, 1.0))
    scale /= max(float(u.abs().max()), float(v.abs().max()))
    u, v, w = u * scale, v * scale, w * scale
    one = torch.ones_like(x)
    th = _outer(1.0 - x, one, one)
    p = torch.zeros_like(u)
    for ky, kz in ((1, 0), (0, 1), (1, 1), (2, 1)):
        cy, cz = torch.cos(ky * pi * x), torch.cos(kz * pi * x)
        th += rng.uniform(-0.12, 0.12) * _outer(torch.sin(rng.randint(1, 2) * pi * x), cy, cz)
        p += 0.05 * max(Ra, 1.0) * rng.uniform(-1.0, 1.0) * \
            _outer(torch.cos(rng.randint(0, 2) * pi * x), cy, cz)
    th[:, :, 0], th[:, :, -1] = 1.0, 0.0
    return dict(u=u, v=v, w=w, th=th, p=p)


def _params(case):
    """The library's steady-solve rule, with the options of the case."""
    p = H.hosc_steady_params(case["N"], case["Ra"], 1.0, case["n"])
    p.tol_lin = 1e-10
    p.max_lin_iter = 4000
    p.auto_defect = 0
    p.precision = H.HOSC_FP64 if case.get("precision", "fp64") == "fp64" else H.HOSC_MIXED
    p.use_history = case.get("history", 0)
    p.precond, p.solver = case.get("precond", 0), case.get("solver", 0)
    Ly, Lz = case.get("Ly", 1.0), case.get("Lz", 1.0)
    if (Ly, Lz) != (1.0, 1.0):
        p.Ly, p.Lz = Ly, Lz
        h = min(1.0, Ly, Lz) / (case["N"] - 1)
        p.dt = min(p.dt, 0.9 * h * h / p.lambda_)
    return p


def _members(case):
    """The pool's cavities: sizes of the batch workload up to the largest, Ra and n spread over
    their ranges."""
    sizes = [N for N in (21, 31, 41, 61) if N <= case["largest"]]
    return [dict(N=sizes[q % len(sizes)], Ra=10.0 ** (2.0 + 3.0 * ((7 * q + 3) % 16) / 15.0),
                 n=0.75 + 0.5 * ((5 * q + 1) % 11) / 10.0, precision="mixed")
            for q in range(case["members"])]


def _ok(status, where):
    if status:
        raise H.HoscError(status, where)


# ------------------------------------------------------------------ the cases

def _inputs(case, seed):
    """What a case starts from: the state, the level before it (history), and the scheme."""
    q = _scheme(_params(case))
    make = lambda: _state(case["N"], case["Ra"], case["n"], seed, case.get("Ly", 1.0),   # noqa: E731
                          case.get("Lz", 1.0))
    first, prev = make(), None
    if case.get("history"):
        old = make()
        for k in ("u", "v", "w"):
            old[k] *= 0.995
        prev = _level(old, q)
    return first, prev, q


def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    stream = torch.cuda.Stream()
    p = _params(case)
    p.cuda_stream = stream.cuda_stream
    first, prev, q = _inputs(case, seed)
    st = dict(kind=case["kind"], stream=stream)
    if case["kind"] == "systems":
        Am, Ae, rhs = _assemble(first, _level(first, q), None, q)
        full = lambda a: torch.nn.functional.pad(a, (1,) * 6)   # noqa: E731
        st.update(N=case["N"], tol=p.tol_lin, limit=p.max_lin_iter,
                  weights=[full(a) for a in Am + Ae], rhs=[full(a) for a in rhs],
                  out=[torch.zeros_like(first["u"]) for _ in range(4)])
        return st
    st.update(first=first, prev=prev, out={k: torch.empty_like(a) for k, a in first.items()},
              snapshot=None)
    if case.get("precision") == "mixed" and not case["phase"]:
        st["snapshot"] = {k: torch.empty_like(a, dtype=torch.float32) for k, a in first.items()}
    torch.cuda.synchronize()
    st["cavity"] = H.Cavity(p, workspace="torch")
    st["steps"] = case.get("steps", 0)
    if case.get("phase"):
        _ok(H.hosc_set_phase(st["cavity"].h, case["phase"]), "hosc_set_phase")
    return st


def _prepare_batch(case, seed):
    members = _members(case)
    params = []
    for m in members:
        p = _params(m)
        p.tol_steady = p.div_steady = 0.0   # a fixed number of steps for every member
        params.append(p)
    pool = S.Pool(sum(H.hosc_workspace_bytes(p) for p in params) + 1, steps_per_round=8,
                  autotune=False)
    slots, ctxs = [], []
    for q, (m, p) in enumerate(zip(members, params)):
        slots.append(pool.admit(p, 10 ** 9))
        st, _, _, _, ctx = H.hosc_pool_result(pool.h, slots[-1])
        _ok(st, "hosc_pool_result")
        ctxs.append(ctx)
        first = _state(m["N"], m["Ra"], m["n"], 1000 * seed + q)
        torch.cuda.synchronize()
        for name, which in STATE:
            _ok(H.hosc_set_field(ctx, which, first[name].cpu().numpy()), "hosc_set_field")
    sizes = [m["N"] ** 3 for m in members]
    out = {name: torch.empty(sum(sizes), dtype=torch.float64, device="cuda") for name, _ in STATE}
    ptrs, at = [], 0
    for s in sizes:
        ptrs.append({name: out[name].data_ptr() + 8 * at for name, _ in STATE})
        at += s
    snapshot = {name: torch.empty_like(a, dtype=torch.float32) for name, a in out.items()}
    return dict(kind="batch", pool=pool, ctxs=ctxs, ptrs=ptrs, out=out, snapshot=snapshot,
                rounds=case["rounds"])


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["pool"].run(state["rounds"])
        for ctx, ptr in zip(state["ctxs"], state["ptrs"]):
            for name, which in STATE:
                _ok(H.hosc_get_field_device(ctx, which, ptr[name]), "hosc_get_field_device")
        torch.cuda.synchronize()   # the members' fields arrive on streams of their own
        for name, a in state["snapshot"].items():
            a.copy_(state["out"][name])
        return state["snapshot"]
    if kind == "systems":
        st, _ = H.hosc_bicgstab_noalloc(
            state["N"], [a.data_ptr() for a in state["weights"]],
            [a.data_ptr() for a in state["rhs"]], [a.data_ptr() for a in state["out"]],
            state["tol"], state["limit"], state["stream"].cuda_stream)
        _ok(st, "hosc_bicgstab_noalloc")
        return state["out"]
    cav = state["cavity"]
    for name, which in STATE:
        _ok(H.hosc_set_field_device(cav.h, which, state["first"][name].data_ptr()), "set")
    if state["prev"] is not None:
        for name, which in PREV:
            _ok(H.hosc_set_field_device(cav.h, which, state["prev"][name].data_ptr()), "set")
    if kind == "solve":
        cav.solve_steady(20000, allow=())
    else:
        cav.step(state["steps"], allow=())
    for name, which in STATE:
        _ok(H.hosc_get_field_device(cav.h, which, state["out"][name].data_ptr()), "get")
    if kind == "solve":
        return dict(state=state["out"], diagnostics=cav.diagnostics())
    if state["snapshot"] is None:
        return state["out"]
    with torch.cuda.stream(state["stream"]):
        for name, a in state["snapshot"].items():
            a.copy_(state["out"][name])
    return state["snapshot"]


# Iterations of the level-(n+1) solves that the work of a step is counted with: about what the
# four systems of a developed cavity take to the tolerance of each precision.
ITERS = {"fp64": 12, "mixed": 7}


def work(case):
    """Bytes: the state read once and written once (the systems: weights and right-hand sides in,
    solutions out). Flops per node and step: viscosity, sources, right-hand sides and weights of
    the four systems about 700; a BiCGSTAB iteration applies two seven-point operators and updates
    three vectors with four dot products, 2 (7 + 7 + 10) a system."""
    if case["kind"] == "batch":
        out = dict(bytes=0.0, flops=0.0)
        for m in _members(case):
            one = work(_march(None, m["N"], m["Ra"], m["n"], 8 * case["rounds"]))
            out = {k: out[k] + one[k] for k in out}
        return out
    n3, ni3 = case["N"] ** 3, (case["N"] - 2) ** 3
    solve = ITERS[case.get("precision", "fp64")] * 4 * 48.0
    if case["kind"] == "systems":
        return dict(bytes=8.0 * (14 + 4 + 4) * ni3, flops=solve * ni3)
    # a steady solve of the listed size takes about 1100 steps
    steps = case["steps"] if case["kind"] == "march" else 1100
    return dict(bytes=80.0 * n3, flops=steps * (700.0 + solve) * ni3)


# ------------------------------------------------------------------ the scheme in plain torch

class _scheme:
    """Parameters of the scheme (Punia & Ray, arXiv:2411.06563, Eqs. 5-8) as plain numbers."""

    def __init__(self, p):
        self.N, self.Ra, self.Pr, self.n, self.dt, self.lam = p.N, p.Ra, p.Pr, p.n, p.dt, p.lambda_
        self.ref, self.eps, self.tol_div = p.theta_ref, p.I2_eps, p.tol_div
        self.a_limit, self.a_boost, self.history = p.a_limit, p.a_boost, p.use_history
        d = 1.0 / (p.N - 1)
        self.h = (d, d * (p.Ly or 1.0), d * (p.Lz or 1.0))   # x, y, z


def _diff(f, axis, h):
    """First derivative at every node: central inside, second-order one-sided on the walls."""
    f = f.movedim(2 - axis, -1)
    d = torch.empty_like(f)
    d[..., 1:-1] = (f[..., 2:] - f[..., :-2]) / (2 * h)
    d[..., 0] = (-3 * f[..., 0] + 4 * f[..., 1] - f[..., 2]) / (2 * h)
    d[..., -1] = (3 * f[..., -1] - 4 * f[..., -2] + f[..., -3]) / (2 * h)
    return d.movedim(-1, 2 - axis)


def _level(s, q):
    """Viscosity, L = 1/(Pr eta) and the momentum sources E* of one time level."""
    g = [[_diff(s[c], a, q.h[a]) for a in range(3)] for c in ("u", "v", "w")]
    strain = [[0.5 * (g[a][b] + g[b][a]) for b in range(3)] for a in range(3)]
    if q.n == 1.0:
        eta = torch.ones_like(s["u"])
    else:
        I2 = 2.0 * sum(strain[a][b] ** 2 for a in range(3) for b in range(3))
        N = q.N
        i = torch.arange(N, device=I2.device)
        inner = i.clamp(1, N - 2)
        wall = (i != inner).to(torch.int64)
        edge = wall[:, None, None] + wall[None, :, None] + wall[None, None, :] >= 2
        I2 = torch.where(edge, I2[inner][:, inner][:, :, inner], I2)   # edges from one node inside
        eta = (I2 + q.eps) ** (0.5 * (q.n - 1.0))
    de = [_diff(eta, a, q.h[a]) for a in range(3)]
    E = [-_diff(s["p"], a, q.h[a]) / (q.Pr * eta) +
         2.0 / eta * sum(strain[b][a] * de[b] for b in range(3)) for a in range(3)]
    E[1] = E[1] + q.Ra * (s["th"] - q.ref) / eta
    return dict(L=1.0 / (q.Pr * eta), u=s["u"], v=s["v"], w=s["w"], Eu=E[0], Ev=E[1], Ew=E[2])


def _in(f, o=(0, 0, 0)):
    """Interior nodes of f shifted by o = (x, y, z)."""
    N = f.shape[0]
    return f[1 + o[2]:N - 1 + o[2], 1 + o[1]:N - 1 + o[1], 1 + o[0]:N - 1 + o[0]]


def _unit(a, s=1):
    o = [0, 0, 0]
    o[a] = s
    return tuple(o)


def _d1(f, a, h):
    return (_in(f, _unit(a)) - _in(f, _unit(a, -1))) / (2 * h[a])


def _d2(f, a, h):
    return (_in(f, _unit(a)) - 2 * _in(f) + _in(f, _unit(a, -1))) / h[a] ** 2


def _mixed(f, a, b, h, ka, kb):
    """d_a^ka d_b^kb f (ka, kb = 1 or 2) at interior nodes."""
    ca = {1: ((1, 0.5 / h[a]), (-1, -0.5 / h[a])),
          2: ((1, h[a] ** -2), (0, -2 * h[a] ** -2), (-1, h[a] ** -2))}[ka]
    cb = {1: ((1, 0.5 / h[b]), (-1, -0.5 / h[b])),
          2: ((1, h[b] ** -2), (0, -2 * h[b] ** -2), (-1, h[b] ** -2))}[kb]
    out = 0.0
    for sa, wa in ca:
        for sb, wb in cb:
            o = [0, 0, 0]
            o[a], o[b] = sa, sb
            out = out + wa * wb * _in(f, tuple(o))
    return out


def _systems(V, Vp, h):
    """The coefficients of Eq. (5) for the convective coefficients V = (G*, H*, I*)."""
    def bracket(f, fp):
        return _in(f) + sum(h[a] ** 2 / 12 * (_d2(f, a, h) - _in(V[a]) * _d1(f, a, h))
                            for a in range(3)) + 0.5 * (_in(f) - _in(fp))
    c = dict(V=[_in(f) for f in V], bracket=bracket)
    c["diag"] = [1 + h[a] ** 2 / 12 * (c["V"][a] ** 2 - 2 * _d1(V[a], a, h)) for a in range(3)]
    c["M"] = [bracket(V[a], Vp[a]) for a in range(3)]
    c["cross"] = []
    for a in range(3):
        b = (a + 1) % 3
        s = h[a] ** 2 + h[b] ** 2
        c["cross"].append(-c["V"][a] * c["V"][b] + 2 * h[b] ** 2 / s * _d1(V[a], b, h) +
                          2 * h[a] ** 2 / s * _d1(V[b], a, h))
    return c


def _apply_B(c, f, h):
    out = sum(c["M"][a] * _d1(f, a, h) - c["diag"][a] * _d2(f, a, h) for a in range(3))
    for a in range(3):
        b = (a + 1) % 3
        out = out - (h[a] ** 2 + h[b] ** 2) / 12 * (
            _mixed(f, a, b, h, 2, 2) - c["V"][b] * _mixed(f, a, b, h, 2, 1) -
            c["V"][a] * _mixed(f, a, b, h, 1, 2) - c["cross"][a] * _mixed(f, a, b, h, 1, 1))
    return out


def _weights(V, L, extra, L_d, q):
    """Seven level-(n+1) weights: centre, x+, x-, y+, y-, z+, z-."""
    h, dt = q.h, q.dt
    M = [-dt / (2 * L) + h[a] ** 2 / 12 for a in range(3)]
    centre = L * (1 - 2 * sum(M[a] / h[a] ** 2 for a in range(3))) + extra
    if q.a_boost > 0:
        g2 = sum(v ** 2 for v in V)
        s3 = sum(1 / x ** 2 for x in h) / 3
        centre = centre + q.a_boost * torch.clamp(
            torch.maximum(dt * (g2 / 6 - s3), dt * g2 / 6 - 2 * L / 3), min=0.0)
    out = [centre]
    for a in range(3):
        odd = (M[a] * V[a] - h[a] ** 2 / (6 * L) * L_d[a]) / (2 * h[a])
        out += [L * (M[a] / h[a] ** 2 - odd), L * (M[a] / h[a] ** 2 + odd)]
    return out


def _assemble(s, lev, prev, q):
    """Momentum and energy operators (seven weights each) and the four right-hand sides
    dt (R - B chi^n) at interior nodes."""
    h = q.h
    prev = lev if prev is None else prev
    L, Lp = lev["L"], prev["L"]
    vel, old = [s[c] for c in ("u", "v", "w")], [prev[c] for c in ("u", "v", "w")]
    cm = _systems([f * L for f in vel], [f * Lp for f in old], h)
    ce = _systems(vel, old, h)
    rhs = []
    for c in ("u", "v", "w"):
        E = "E" + c
        rhs.append(q.dt * (cm["bracket"](lev[E], prev[E]) - _apply_B(cm, s[c], h)))
    rhs.append(-q.dt * _apply_B(ce, s["th"], h))
    Lc = _in(L)
    L_d = [_d1(L, a, h) for a in range(3)]
    m18 = 0.5 * (Lc - _in(Lp)) + sum(h[a] ** 2 / 12 * (_d2(L, a, h) - cm["V"][a] * L_d[a])
                                     for a in range(3))
    if q.a_limit > 0:
        m18 = torch.maximum(m18, -q.a_limit * Lc)
    one = torch.ones_like(Lc)
    Am = _weights(cm["V"], Lc, m18, L_d, q)
    Ae = _weights(ce["V"], one, 0.0, [0.0 * one] * 3, q)
    return Am, Ae, rhs


def _apply_A(W, f):
    f = torch.nn.functional.pad(f, (1,) * 6)
    out = W[0] * _in(f)
    for a in range(3):
        out = out + W[1 + 2 * a] * _in(f, _unit(a)) + W[2 + 2 * a] * _in(f, _unit(a, -1))
    return out


def _krylov(W, b, tol=3e-15, limit=500):
    """Textbook BiCGSTAB with row scaling, to the rounding of 64 bits."""
    x = torch.zeros_like(b)
    b = b / W[0]
    W = [a / W[0] for a in W]
    r = b.clone()
    r0, p, v = r.clone(), torch.zeros_like(b), torch.zeros_like(b)
    dot = lambda a, c: float((a * c).sum())   # noqa: E731
    rho, alpha, om, stop = 1.0, 1.0, 1.0, tol * math.sqrt(dot(b, b))
    for _ in range(limit):
        if math.sqrt(dot(r, r)) <= stop:
            break
        rho1 = dot(r0, r)
        p = r + rho1 / rho * alpha / om * (p - om * v)
        v = _apply_A(W, p)
        rho, alpha = rho1, rho1 / dot(r0, v)
        s = r - alpha * v
        t = _apply_A(W, s)
        om = dot(t, s) / max(dot(t, t), 1e-300)
        x += alpha * p + om * s
        r = s - om * t
        if om == 0.0:
            break
    return x


def _walls(f, axes):
    """Zero normal derivative on the walls of the axes (x, y, z = 0, 1, 2): (4 f_1 - f_2)/3."""
    for a in axes:
        g = f.movedim(2 - a, -1)
        g[..., 0] = (4 * g[..., 1] - g[..., 2]) / 3
        g[..., -1] = (4 * g[..., -2] - g[..., -3]) / 3
    return f


def _step(s, prev, q):
    lev = _level(s, q)
    Am, Ae, rhs = _assemble(s, lev, prev, q)
    new = {k: a.clone() for k, a in s.items()}
    for k, (c, b) in enumerate(zip(("u", "v", "w", "th"), rhs)):
        _in(new[c]).add_(_krylov(Ae if c == "th" else Am, b))
    inside = new["th"][:, :, 1:-1]                 # the hot and cold walls keep their values
    new["th"][:, :, 1:-1] = _walls(inside.clone(), (1, 2))
    div = sum(_d1(new[c], a, q.h) for a, c in enumerate(("u", "v", "w")))
    if float(div.abs().max()) > q.tol_div:
        _in(new["p"]).sub_(q.lam * div)
        _walls(new["p"], (0, 1, 2))
    return new, (lev if q.history else None)


def exact(case, seed):
    """The outputs in 64 bits, from the scheme written out in plain torch. None for the steady
    solve (a thousand steps)."""
    kind = case["kind"]
    if kind == "solve":
        return None
    if kind == "batch":
        got = []
        for k, m in enumerate(_members(case)):
            q = _scheme(_params(m))
            s, prev = _state(m["N"], m["Ra"], m["n"], 1000 * seed + k), None
            for _ in range(8 * case["rounds"]):
                s, prev = _step(s, prev, q)
            got.append(s)
        return {name: torch.cat([s[name].reshape(-1) for s in got]) for name, _ in STATE}
    s, prev, q = _inputs(case, seed)
    if kind == "systems":
        Am, Ae, rhs = _assemble(s, _level(s, q), None, q)
        return [torch.nn.functional.pad(_krylov(Ae if k == 3 else Am, b), (1,) * 6)
                for k, b in enumerate(rhs)]
    for _ in range(case["steps"]):
        s, prev = _step(s, prev, q)
    return s
