"""The work that is measured: calls of the library's public entry points over
the sizes, element types and options that its configurations, tests and
benchmark use.

A case is a dict of plain values. Its "call" says which entry point a pass goes
through:
  step      one RK step in place on a device array (solver.rk3_step): the unit
            of every time loop, and what a control loop calls by itself
  solve     a whole solve from a device or pinned host V0 to its time slices
            (solver.solve)
  batch     many solves of uneven sizes at once (solver.solve_batch)
  gradient  the one-sided derivatives along every dimension (solver.upwind):
            what a feedback law reads off a solved value function
  term      the Hamiltonian term with its dissipation (solver.term)
  surface   an initial surface from primitives (solver.implicit_surface)
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2507_11542_gb300 import _lib as L
from paper_2507_11542_gb300 import solver, workloads as W

PI = math.pi

# Domains of the workloads: bounds, periodic dimensions, dynamics and its
# parameters, target radius and the dimensions that the target spans.
DOMAINS = {
    "di": ((-1.0, -1.0), (1.0, 1.0), (), L.HJ_DYN_DOUBLE_INTEGRATOR, (1.0,), (0.2, 0.8), 2),
    "air3d": ((-6.0, -10.0, 0.0), (20.0, 10.0, 2 * PI), (2,), L.HJ_DYN_AIR3D, (5.0, 5.0, 1.0, 1.0), (3.0, 5.5), 2),
    "rockets": ((-64.0, -64.0, -PI / 2), (64.0, 64.0, PI / 2), (), L.HJ_DYN_ROCKETS, (1.0, 32.0, 1.0, 1.0), (1.5, 20.0), 2),
    "dubins": ((-5.0, -5.0, 0.0, 0.0), (5.0, 5.0, 2 * PI, 2.0), (2,), L.HJ_DYN_DUBINS4D, (1.0, 0.5), (0.5, 1.5), 2),
    "sphere": ((-1.0, -1.0, -1.0), (1.0, 1.0, 1.0), (), L.HJ_DYN_NORM, (1.0,), (0.2, 0.4), 3),
}
# Floating-point operations of both one-sided derivatives along one dimension,
# per node (the method as stated; an FMA counts two), and of the rest of a stage.
DERIVATIVE_FLOPS = {1: 2, 2: 14, 3: 36, 5: 141}
NODE_FLOPS = 50
CFL = 0.8


def _case(call, dyn, n, dtype, scheme=5, brt=1, **more):
    c = {"call": call, "dyn": dyn, "dtype": dtype, "scheme": scheme, "brt": brt, "extrap": 0, "alpha": 0, "order": 3}
    for d, k in enumerate(n):
        c["n%d" % d] = k
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: a safety filter that advances a coarse planar value function every cycle
        _case("step", "di", (51, 51), "float32", name="step_di_51_f32"),
        # the double-integrator tube, whole: 11 slices over its horizon, in the paper's precision
        _case("solve", "di", (101, 101), "float64", tau=1.0, slices=11, host=False, name="solve_di_101_f64"),
        # the pursuit-evasion game in the paper's precision, one step of its time loop
        _case("step", "air3d", (101, 101, 101), "float64", name="step_air3d_101_f64"),
        # the same game in FP32 as a user with host arrays solves it up to a slice
        _case("solve", "air3d", (101, 101, 101), "float32", tau=0.14, slices=2, host=True, name="solve_air3d_101_f32_host"),
        # a finer grid with a different node count along every dimension
        _case("step", "air3d", (161, 113, 79), "float32", name="step_air3d_ragged_f32"),
        # the paper's rockets game with its ENO2 scheme, in its precision
        _case("step", "rockets", (100, 100, 100), "float64", scheme=2, name="step_rockets_100_f64_eno2"),
        # the car with speed state on the largest 4-D grid
        _case("step", "dubins", (81, 81, 81, 81), "float32", name="step_dubins_81_f32"),
        # the same car in FP64, the reference that its FP32 results are held against
        _case("step", "dubins", (61, 61, 61, 61), "float64", name="step_dubins_61_f64"),
        # the expanding front on the largest grid, arrays far larger than L2, no tube rule
        _case("step", "sphere", (512, 512, 512), "float32", brt=0, name="step_sphere_512_f32"),
        # many independent solves of uneven sizes, as parameter studies and requests come
        {"call": "batch", "dtype": "float32", "scheme": 5, "brt": 1, "extrap": 0, "alpha": 0, "order": 3, "count": 24, "mix": 42,
         "tau_di": 0.2, "tau_air": 0.15, "name": "batch_mix_f32"},
        # gradients of a solved game for a feedback law, every dimension
        _case("gradient", "air3d", (101, 101, 101), "float64", name="gradient_air3d_101_f64"),
        # the initial surface of the largest grid: two spheres and a box joined, a ball cut out
        _case("surface", "sphere", (512, 512, 512), "float32", name="surface_512_f32"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step"] * 6 + ["solve", "solve", "batch", "gradient", "term", "surface"])
    dtype = rng.choice(["float32", "float64"])
    scheme = rng.choice([5, 5, 5, 2, 1, 3])
    brt = rng.choice([1, 1, 0, 2])
    extrap = rng.choice([0, 0, 1])
    if call == "batch":
        return {"call": "batch", "dtype": dtype, "scheme": 5, "brt": brt, "extrap": 0, "alpha": 0, "order": 3,
                "count": rng.randint(4, 24 if dtype == "float32" else 8), "mix": rng.randint(0, 10 ** 6),
                "tau_di": round(rng.uniform(0.02, 0.2), 3), "tau_air": round(rng.uniform(0.01, 0.05), 3)}
    dyn = rng.choice(["di", "air3d", "air3d", "rockets", "dubins", "sphere"])
    if dyn == "di":
        n = [_spread(rng, 51, 301) for _ in range(2)]
    elif dyn == "dubins":
        n = [rng.randint(31, 61) for _ in range(4)]
    elif dyn == "sphere" and dtype == "float32":
        n = [_spread(rng, 64, 400) for _ in range(3)]
    else:
        n = [_spread(rng, 41, 161) for _ in range(3)]
    alpha = rng.choice([0, 0, 1]) if dyn == "rockets" else 0
    order = rng.choice([3, 3, 3, 2])
    c = _case(call, dyn, n, dtype, scheme=scheme, brt=brt, extrap=extrap, alpha=alpha, order=order)
    if call == "solve":
        # a few tens of steps in one to eleven slices
        steps = rng.randint(6, 40) if dyn == "di" else rng.randint(4, 12)
        c.update(tau=round(steps * CFL / _bound(c), 5), slices=rng.choice([1, 2, 11 if dyn == "di" else 3]), host=rng.random() < 0.3)
    return c


# ---------------------------------------------------------------------------
# Grids, targets and what they cost
# ---------------------------------------------------------------------------

def _n(case):
    return tuple(int(case["n%d" % d]) for d in range(len(DOMAINS[case["dyn"]][0])))


def _spec(dyn, n):
    lo, hi, periodic = DOMAINS[dyn][:3]
    return W.GridSpec(tuple(n), lo, hi, periodic)


def _spacing(spec):
    return [(spec.hi[d] - spec.lo[d]) / (spec.n[d] if d in spec.periodic else spec.n[d] - 1) for d in range(spec.ndim)]


def _members(case):
    """(dynamics, nodes, horizon) of a batch: half of them planar, half games."""
    r = random.Random(int(case["mix"]))
    got = []
    for k in range(int(case["count"])):
        if k % 2 == 0:
            got.append(("di", (r.randint(51, 201),) * 2, case["tau_di"]))
        else:
            got.append(("air3d", (r.randint(41, 121),) * 3, case["tau_air"]))
    return got


def _method(case, dyn):
    return solver.method(scheme=case["scheme"], dynamics=DOMAINS[dyn][3], params=DOMAINS[dyn][4], brt=case["brt"],
                         extrap=case["extrap"], cfl=CFL, order=case["order"], alpha_mode=case["alpha"])


def _target(spec, dyn, seed, device, bumps):
    """Signed distance to a seeded ball (a cylinder where the target spans fewer
    dimensions than the grid); bumps: a smooth relief on top of it, as a value
    function has after a while."""
    rng = np.random.default_rng(seed)
    dims = DOMAINS[dyn][6]
    radius = rng.uniform(*DOMAINS[dyn][5])
    V = torch.zeros([1] * spec.ndim, dtype=torch.float64, device=device)
    X = [_axis(spec, d, device) for d in range(spec.ndim)]
    for d in range(dims):
        span = spec.hi[d] - spec.lo[d]
        center = rng.uniform(-0.05, 0.05) * span
        V = V + (X[d] - center) ** 2
    V = torch.sqrt(V) - radius
    for _ in range(3 if bumps else 0):
        arg = rng.uniform(0.0, 2 * PI)
        for d in range(spec.ndim):
            span = spec.hi[d] - spec.lo[d]
            k = rng.integers(1, 3) if d in spec.periodic else rng.uniform(0.4, 2.0)
            arg = arg + 2 * PI * float(k) * (X[d] - spec.lo[d]) / span
        V = V + rng.uniform(0.02, 0.06) * (spec.hi[0] - spec.lo[0]) * torch.sin(arg)
    return V.expand(tuple(reversed(spec.n))).contiguous().view(-1)


def _axis(spec, d, device):
    """Node positions along dimension d, shaped to broadcast (dimension 0 is the last axis)."""
    x = spec.lo[d] + torch.arange(spec.n[d], dtype=torch.float64, device=device) * _spacing(spec)[d]
    shape = [1] * spec.ndim
    shape[spec.ndim - 1 - d] = spec.n[d]
    return x.view(shape)


def _alphas(spec, dyn, device):
    """alpha_d(x), the largest speed along each dimension at a node."""
    X = [_axis(spec, d, device) for d in range(spec.ndim)]
    q = DOMAINS[dyn][4]
    one = torch.ones([1] * spec.ndim, dtype=torch.float64, device=device)
    if dyn == "di":
        return [X[1].abs(), q[0] * one]
    if dyn == "air3d":
        f0, f1 = -q[0] + q[1] * torch.cos(X[2]), q[1] * torch.sin(X[2])
        return [f0.abs() + q[2] * X[1].abs(), f1.abs() + q[2] * X[0].abs(), (q[2] + q[3]) * one]
    if dyn == "rockets":
        f0, f1 = q[0] * torch.cos(X[2]), q[0] * torch.sin(X[2]) + q[0] - q[1]
        return [f0.abs() + q[2] * X[0].abs(), f1.abs() + q[3] * X[0].abs(), (q[2] + q[3]) * one]
    if dyn == "dubins":
        return [(X[3] * torch.cos(X[2])).abs(), (X[3] * torch.sin(X[2])).abs(), q[0] * one, q[1] * one]
    return [q[0] * one] * spec.ndim


def _bound(case, dyn=None, n=None):
    """max over the grid of sum_d alpha_d / dx_d."""
    dyn, n = dyn or case["dyn"], n or _n(case)
    spec = _spec(dyn, n)
    dx = _spacing(spec)
    a = _alphas(spec, dyn, "cpu")
    if case["alpha"] == L.HJ_ALPHA_GLOBAL:
        return sum(float(a[d].max()) / dx[d] for d in range(spec.ndim))
    return float(sum(a[d] / dx[d] for d in range(spec.ndim)).max())


def _steps(bound, tau, slices):
    """Step sizes up to each slice: full steps, the last of a slice clipped to land on it."""
    t, out = 0.0, []
    for ts in _slice_times(tau, slices):
        dts = []
        while ts > t and ts - t >= 100 * np.finfo(np.float64).eps * ts:
            dts.append(min(ts - t, CFL * (1.0 / bound)))
            t += dts[-1]
        out.append((dts, t))
    return out


def _slice_times(tau, slices):
    return [tau] if slices == 1 else [float(t) for t in W.slice_times(tau, slices)]


def work(case):
    size = 4 if case["dtype"] == "float32" else 8
    if case["call"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for dyn, n, tau in _members(case):
            N = math.prod(n)
            steps = sum(len(d) for d, _ in _steps(_bound(case, dyn, n), tau, 1))
            total["bytes"] += 2 * N * size
            total["flops"] += steps * case["order"] * N * (len(n) * DERIVATIVE_FLOPS[case["scheme"]] + NODE_FLOPS)
        return total
    n = _n(case)
    N, D = math.prod(n), len(n)
    stage = D * DERIVATIVE_FLOPS[case["scheme"]] + NODE_FLOPS
    if case["call"] == "surface":
        return {"bytes": N * size, "flops": N * 4 * (2 * D + 3)}
    if case["call"] == "gradient":
        return {"bytes": (1 + 2 * D) * N * size, "flops": N * D * DERIVATIVE_FLOPS[case["scheme"]]}
    if case["call"] == "term":
        return {"bytes": 2 * N * size, "flops": N * stage}
    if case["call"] == "step":
        return {"bytes": 2 * N * size, "flops": case["order"] * N * stage}
    steps = sum(len(d) for d, _ in _steps(_bound(case), case["tau"], case["slices"]))
    return {"bytes": (1 + case["slices"]) * N * size, "flops": steps * case["order"] * N * stage}


# ---------------------------------------------------------------------------
# A pass
# ---------------------------------------------------------------------------

_context = None


def _ctx():
    """The context that a program keeps for as long as it runs."""
    global _context
    if _context is None:
        _context = solver.Context(0)
    return _context


def _shapes(seed):
    """Two balls and a box joined, a ball cut out of them."""
    rng = np.random.default_rng(seed)
    three = (0, 1, 2)

    def at(reach):
        return tuple(rng.uniform(-reach, reach, 3))

    return [
        {"kind": L.HJ_SHAPE_SPHERE, "op": L.HJ_SHAPE_UNION, "dims": three, "center": at(0.5), "radius": rng.uniform(0.2, 0.4)},
        {"kind": L.HJ_SHAPE_SPHERE, "op": L.HJ_SHAPE_UNION, "dims": three, "center": at(0.5), "radius": rng.uniform(0.2, 0.4)},
        {"kind": L.HJ_SHAPE_RECTANGLE, "op": L.HJ_SHAPE_UNION, "dims": three, "center": at(0.5), "axes": tuple(rng.uniform(0.1, 0.4, 3))},
        {"kind": L.HJ_SHAPE_SPHERE, "op": L.HJ_SHAPE_SUBTRACT, "dims": three, "center": at(0.3), "radius": rng.uniform(0.1, 0.2)},
    ]


def _surface_spec(case):
    # the primitives of _shapes live in three dimensions, whatever the grid's bounds
    return W.GridSpec(_n(case)[:3] + (32,) * (3 - len(_n(case)[:3])), (-1.0,) * 3, (1.0,) * 3, ())


def prepare(case, seed):
    dtype = getattr(torch, case["dtype"])
    ctx = _ctx()
    if case["call"] == "surface":
        return {"call": "surface", "ctx": ctx, "spec": _surface_spec(case), "shapes": _shapes(seed), "dtype": case["dtype"]}
    if case["call"] == "batch":
        s = {"call": "batch", "ctx": ctx, "specs": [], "methods": [], "V0": [], "times": []}
        for k, (dyn, n, tau) in enumerate(_members(case)):
            spec = _spec(dyn, n)
            s["specs"].append(spec)
            s["methods"].append(_method(case, dyn))
            s["V0"].append(_target(spec, dyn, 1000 * seed + k, "cuda", False).to(dtype))
            s["times"].append([tau])
        return s
    spec, m = _spec(case["dyn"], _n(case)), _method(case, case["dyn"])
    s = {"call": case["call"], "ctx": ctx, "spec": spec, "method": m}
    if case["call"] == "solve":
        V0 = _target(spec, case["dyn"], seed, "cuda", False).to(dtype)
        s["times"] = _slice_times(case["tau"], case["slices"])
        s["out"] = torch.empty((len(s["times"]), V0.numel()), dtype=dtype, device="cpu" if case["host"] else "cuda",
                               pin_memory=case["host"])
        s["V0"] = V0.cpu().pin_memory() if case["host"] else V0
        return s
    s["V"] = _target(spec, case["dyn"], seed, "cuda", True).to(dtype)
    s["dt"] = CFL / solver.step_bound(ctx, spec, m)
    return s


def run(state):
    call = state["call"]
    if call == "step":
        return solver.rk3_step(state["ctx"], state["spec"], state["method"], state["V"], state["dt"])
    if call == "solve":
        out, times, _ = solver.solve(state["ctx"], state["spec"], state["method"], state["V0"], state["times"], state["out"])
        return out, times
    if call == "batch":
        outs, times, _ = solver.solve_batch(state["ctx"], state["specs"], state["methods"], state["V0"], state["times"])
        return outs
    if call == "gradient":
        return [solver.upwind(state["ctx"], state["spec"], state["method"], state["V"], d) for d in range(state["spec"].ndim)]
    if call == "term":
        return solver.term(state["ctx"], state["spec"], state["method"], state["V"])
    return solver.implicit_surface(state["ctx"], state["spec"], state["shapes"], state["dtype"])


# ---------------------------------------------------------------------------
# The same in plain 64-bit torch
# ---------------------------------------------------------------------------

def _padded(V, axis, periodic, extrap):
    """V with three ghost values on each side along an axis."""
    n = V.shape[axis]

    def part(a, b):
        return V.narrow(axis, a, b - a)

    if periodic:
        return torch.cat([part(n - 3, n), V, part(0, 3)], axis)

    def ghosts(edge, inner):
        slope = edge - inner if extrap == L.HJ_EXTRAP_LINEAR else (edge - inner).abs() * torch.sign(edge)
        return [edge + m * slope for m in (1, 2, 3)]

    low = ghosts(part(0, 1), part(1, 2))
    high = ghosts(part(n - 1, n), part(n - 2, n - 1))
    return torch.cat([low[2], low[1], low[0], V] + high, axis)


def _weno5(a, b, c, d, e):
    s1 = 13 / 12 * (a - 2 * b + c) ** 2 + (a - 4 * b + 3 * c) ** 2 / 4
    s2 = 13 / 12 * (b - 2 * c + d) ** 2 + (b - d) ** 2 / 4
    s3 = 13 / 12 * (c - 2 * d + e) ** 2 + (3 * c - 4 * d + e) ** 2 / 4
    big = a.abs()
    for v in (b, c, d, e):
        big = torch.maximum(big, v.abs())
    eps = 1e-6 * big ** 2 + 1e-99
    w1, w2, w3 = 0.1 / (s1 + eps) ** 2, 0.6 / (s2 + eps) ** 2, 0.3 / (s3 + eps) ** 2
    q1, q2, q3 = 2 * a - 7 * b + 11 * c, -b + 5 * c + 2 * d, 2 * c + 5 * d - e
    return (w1 * q1 + w2 * q2 + w3 * q3) / (6 * (w1 + w2 + w3))


def _sides(V, axis, dx, scheme, periodic, extrap):
    """p- and p+ along an axis."""
    P = _padded(V, axis, periodic, extrap)
    n = V.shape[axis]

    def part(x, start, size=n):
        return x.narrow(axis, start, size)

    D1 = (part(P, 1, n + 5) - part(P, 0, n + 5)) / dx  # D1[k]: between padded nodes k and k + 1
    if scheme == 1:
        return part(D1, 2), part(D1, 3)
    if scheme == 5:
        e = [part(D1, k) for k in range(6)]
        return _weno5(*e[:5]), _weno5(*e[:0:-1])
    D2 = (part(D1, 1, n + 4) - part(D1, 0, n + 4)) / (2 * dx)  # at padded nodes 1 .. n + 4
    D3 = (part(D2, 1, n + 3) - part(D2, 0, n + 3)) / (3 * dx)
    sides = []
    for first, sign in ((0, 1.0), (1, -1.0)):
        # candidates: second differences at the stencil's first node k and at k + 1
        l2, r2 = part(D2, first + 1), part(D2, first + 2)
        left = l2.abs() <= r2.abs()
        p = part(D1, 2 + first) + sign * torch.where(left, l2, r2) * dx
        if scheme == 3:
            t = [part(D3, first + k) for k in range(3)]
            a, b = torch.where(left, t[0], t[1]), torch.where(left, t[1], t[2])
            best = torch.where(a.abs() <= b.abs(), a, b)
            coef = torch.where(left, 2.0, -1.0) if first == 0 else torch.where(left, -1.0, 2.0)
            p = p + best * coef * dx * dx
        sides.append(p)
    return sides[0], sides[1]


def _exact_term(case, dyn, spec, V):
    dx = _spacing(spec)
    X = [_axis(spec, d, V.device) for d in range(spec.ndim)]
    alpha = _alphas(spec, dyn, V.device)
    if case["alpha"] == L.HJ_ALPHA_GLOBAL:
        alpha = [a.max() for a in alpha]
    p, diss = [], 0.0
    for d in range(spec.ndim):
        lo, hi = _sides(V, spec.ndim - 1 - d, dx[d], case["scheme"], d in spec.periodic, case["extrap"])
        p.append((lo + hi) / 2)
        diss = diss + alpha[d] * (hi - lo) / 2
    q = DOMAINS[dyn][4]
    if dyn == "di":
        H = p[0] * X[1] - q[0] * p[1].abs()
    elif dyn == "air3d":
        H = (p[0] * (-q[0] + q[1] * torch.cos(X[2])) + p[1] * (q[1] * torch.sin(X[2]))
             + q[2] * (p[0] * X[1] - p[1] * X[0] - p[2]).abs() - q[3] * p[2].abs())
    elif dyn == "rockets":
        H = (p[0] * q[0] * torch.cos(X[2]) + p[1] * (q[0] * torch.sin(X[2]) + q[0] - q[1])
             + q[2] * (p[0] * X[0] - p[2]).abs() - q[3] * (p[1] * X[0] + p[2]).abs())
    elif dyn == "dubins":
        H = X[3] * (p[0] * torch.cos(X[2]) + p[1] * torch.sin(X[2])) - q[0] * p[2].abs() - q[1] * p[3].abs()
    else:
        H = -q[0] * torch.sqrt(sum(x * x for x in p))
    y = H + diss
    return y.clamp(max=0.0) if case["brt"] == L.HJ_BRT_MIN0 else y


def _exact_step(case, dyn, spec, V, dt):
    def euler(u):
        return u + dt * _exact_term(case, dyn, spec, u)

    if case["order"] == 2:
        new = 0.5 * V + 0.5 * euler(euler(V))
    else:
        u = 0.75 * V + 0.25 * euler(euler(V))
        new = V / 3 + 2 / 3 * euler(u)
    return torch.minimum(new, V) if case["brt"] == L.HJ_BRT_MINV else new


def _exact_solve(case, dyn, spec, V0, tau, slices):
    V, outs, times = V0, [], []
    for dts, t in _steps(_bound(case, dyn, spec.n), tau, slices):
        for dt in dts:
            V = _exact_step(case, dyn, spec, V, dt)
        outs.append(V.reshape(-1))
        times.append(t)
    return torch.stack(outs), np.array(times)


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    dtype = getattr(torch, case["dtype"])
    if case["call"] == "surface":
        spec = _surface_spec(case)
        X, V = [_axis(spec, d, device) for d in range(3)], None
        for s in _shapes(seed):
            r = [X[d] - s["center"][d] for d in range(3)]
            if s["kind"] == L.HJ_SHAPE_SPHERE:
                f = torch.sqrt(r[0] ** 2 + r[1] ** 2 + r[2] ** 2) - s["radius"]
            else:
                f = torch.maximum(torch.maximum(r[0].abs() - s["axes"][0], r[1].abs() - s["axes"][1]), r[2].abs() - s["axes"][2])
            V = f if V is None else torch.minimum(V, f) if s["op"] == L.HJ_SHAPE_UNION else torch.maximum(V, -f)
        return V.reshape(-1)
    if case["call"] == "batch":
        outs = []
        for k, (dyn, n, tau) in enumerate(_members(case)):
            spec = _spec(dyn, n)
            V0 = _target(spec, dyn, 1000 * seed + k, device, False).to(dtype).double()
            outs.append(_exact_solve(case, dyn, spec, V0.view(tuple(reversed(n))), tau, 1)[0])
        return outs
    dyn, spec = case["dyn"], _spec(case["dyn"], _n(case))
    V = _target(spec, dyn, seed, device, case["call"] != "solve").to(dtype).double().view(tuple(reversed(spec.n)))
    if case["call"] == "solve":
        return _exact_solve(case, dyn, spec, V, case["tau"], case["slices"])
    if case["call"] == "step":
        return _exact_step(case, dyn, spec, V, CFL / _bound(case)).reshape(-1)
    if case["call"] == "term":
        return _exact_term(case, dyn, spec, V).reshape(-1)
    dx = _spacing(spec)
    return [tuple(p.reshape(-1) for p in _sides(V, spec.ndim - 1 - d, dx[d], case["scheme"], d in spec.periodic, case["extrap"]))
            for d in range(spec.ndim)]
