"""The calls a user of libsfac makes, as measurable cases.

A case is one pass through a public entry point: a call of `Plan.step` on a
device field (most cases), of `Plan.step_host` on a pinned host field, of
`Plan.step` followed by `Plan.diagnostics` (a monitored run), or one launch of
a prepared `Batch`. Grids, orders and time steps come from the repository's
workloads (`sfac_inputs`), the paper's examples and the GPU tests.
"""
import math

import numpy as np
import torch

import paper_2209_08437_gb300 as S
import sfac_inputs as I


def _grid(name, kind, prec, n, alpha, eps, tau, steps, field, lo=-1.0, hi=1.0, **more):
    case = {"name": name, "kind": kind, "prec": prec, "dim": len(n), "eps": eps, "tau": tau, "steps": steps,
            "field": field, "lo": lo, "hi": hi, **more}
    for l, (nl, al) in enumerate(zip(n, alpha)):
        case[f"n{l + 1}"], case[f"alpha{l + 1}"] = nl, al
    return case


def listed():
    return [
        # The 2D n = 64 workload: one call runs the whole 100-step solve; the
        # smallest grid, where launches, barriers and latency count.
        _grid("2d64_fp64_call100", "step", "fp64", (64, 64), (1.5, 1.5), 0.1, 0.01, 100, "uniform"),
        # Example 5 of the paper: h = 1/128 on (0,1)^2, the energy and max|u|
        # read after every step (a monitored run on n = 2^k - 1 lines).
        _grid("2d127_fp64_monitored", "monitored", "fp64", (127, 127), (1.5, 1.7), 0.01, 0.01, 1, "small", 0.0, 1.0),
        # Example 1 (Table 2): two Gaussian bumps on (0,2)^2, n = 255, a few
        # steps of a solve per call.
        _grid("2d255_fp64_step10", "step", "fp64", (255, 255), (1.2, 1.8), 0.1, 0.005, 10, "bumps", 0.0, 2.0),
        # Example 2 (Table 4): two narrow bumps in 3D, h = 1/64 on (0,1)^3.
        _grid("3d63_fp64_step5", "step", "fp64", (63, 63, 63), (1.2, 1.3, 1.4), 0.1, 0.05, 5, "bumps", 0.0, 1.0),
        # The 2D n = 1024 workload in both precisions: a step per call (FP64),
        # ten steps between two looks at the field (FP32).
        _grid("2d1024_fp64_step", "step", "fp64", (1024, 1024), (1.3, 1.7), 0.05, 1e-3, 1, "wave"),
        _grid("2d1024_fp32_step10", "step", "fp32", (1024, 1024), (1.3, 1.7), 0.05, 1e-3, 10, "wave"),
        # The 3D n = 256 workload, the headline, one step per call.
        _grid("3d256_fp64_step", "step", "fp64", (256, 256, 256), (1.2, 1.5, 1.8), 0.08, 2e-3, 1, "uniform"),
        _grid("3d256_fp32_step", "step", "fp32", (256, 256, 256), (1.2, 1.5, 1.8), 0.08, 2e-3, 1, "uniform"),
        # The same step end to end from pinned host memory.
        _grid("3d256_fp32_host", "host", "fp32", (256, 256, 256), (1.2, 1.5, 1.8), 0.08, 2e-3, 1, "uniform"),
        # Uneven 3D extents, none a power of two, two of them odd.
        _grid("3d_ragged_fp32_step2", "step", "fp32", (255, 100, 127), (1.3, 1.7, 1.5), 0.07, 2e-3, 2, "uniform"),
        # Long lines: a fine 2D grid, fields of 64 MB.
        _grid("2d4096_fp32_step", "step", "fp32", (4096, 4096), (1.3, 1.7), 0.05, 1e-3, 1, "wave"),
        # The batched workload: the first 64 of the 512 uneven 2D instances, a
        # tenth of each one's steps per launch.
        {"name": "batch64_fp32", "kind": "batch", "prec": "fp32", "count": 64, "first_seed": 100, "div": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["host", "monitored", "batch"])
    if kind == "batch":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        return {"kind": kind, "prec": prec, "count": _log_int(rng, 8, 40) if prec == "fp32" else rng.randint(2, 3),
                "first_seed": rng.randrange(100, 600), "div": rng.choice([15, 25, 40])}
    prec = rng.choice(["fp64", "fp32"])
    most = 0.5 * max(_cost(c) for c in listed() if c["kind"] != "batch")
    while True:
        dim = rng.choice([2, 2, 3, 3])
        hi = 2048 if dim == 2 else 256
        n = []
        for _ in range(dim):
            v = _log_int(rng, 24, hi)
            # half of the extents are powers of two, a quarter the paper's 2^k - 1
            r = rng.random()
            if r < 0.75:
                v = 2 ** max(5, round(math.log2(v))) - (0 if r < 0.5 else 1)
            n.append(v)
        alpha = [round(rng.uniform(1.1, 1.9), 3) for _ in n]
        steps = _log_int(rng, 1, 50) if kind == "step" else 1
        side = rng.choice([(-1.0, 1.0), (0.0, 1.0), (0.0, 2.0)])
        case = _grid("", kind, prec, n, alpha, round(rng.uniform(0.02, 0.1), 4),
                     rng.choice([1e-3, 2e-3, 0.01, 0.05]), steps, rng.choice(["uniform", "wave", "bumps"]), *side)
        del case["name"]
        if _cost(case) <= most:
            return case


def _points(case):
    return math.prod(_n(case))


def _n(case):
    return tuple(case[f"n{l + 1}"] for l in range(case["dim"]))


def _alpha(case):
    return tuple(case[f"alpha{l + 1}"] for l in range(case["dim"]))


def _cost(case):
    """A bound on a case's size: point updates along one axis, times the
    logarithm of the line, doubled where it is not a power of two, 30 times as
    many for FP64, and no less than 20000 points' worth a step."""
    per = sum(math.log2(v) * (1 if v & (v - 1) == 0 else 2.2) for v in _n(case))
    return max(_points(case), 20000) * case["steps"] * per * (30 if case["prec"] == "fp64" else 1)


def _problem(case):
    return I.Problem(n=_n(case), alpha=_alpha(case), eps=case["eps"], tau=case["tau"], a=case["lo"], b=case["hi"],
                     steps=case["steps"])


def _instances(case):
    out = []
    for seed, p in I.batched_instances(case["count"], case["first_seed"]):
        out.append((p, max(1, p.steps // case["div"])))
    return out


def _u0(prob, field, prec, gen):
    """The initial field, on the GPU: axis 1 is the last index."""
    dev = "cuda"
    rand = lambda lo, hi: lo + (hi - lo) * torch.rand(prob.shape, generator=gen, device=dev, dtype=torch.float64)
    if field == "uniform":
        u = rand(-0.95, 0.95)
    elif field == "small":
        u = rand(-0.4, 0.4)
    else:
        d = prob.dim
        xs = []
        for ax in range(d):
            shp = [1] * d
            shp[d - 1 - ax] = prob.n[ax]
            xs.append(torch.tensor(prob.nodes(ax), device=dev).reshape(shp))
        if field == "wave":
            u = 0.9 * torch.ones(prob.shape, device=dev, dtype=torch.float64)
            for x in xs:
                u = u * torch.sin(math.pi * x)
            u = u + rand(-0.05, 0.05)
        else:  # two Gaussian bumps, their centres moved a little by the seed
            u = torch.zeros(prob.shape, device=dev, dtype=torch.float64)
            side, width = prob.b - prob.a, 500.0 if d == 3 else 400.0
            for c in (3 / 8, 5 / 8):
                mid = c + 0.05 * (torch.rand(d, generator=gen, device=dev, dtype=torch.float64) - 0.5)
                r2 = sum(((x - prob.a) / side - mid[k]) ** 2 for k, x in enumerate(xs))
                u = u + 0.5 * torch.exp(-width * r2)
    return u.to(torch.float64 if prec == "fp64" else torch.float32).contiguous()


def _fields(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "batch":
        return [_u0(p, "uniform", case["prec"], gen) for p, _ in _instances(case)]
    return [_u0(_problem(case), case["field"], case["prec"], gen)]


def prepare(case, seed):
    prec = S.SFAC_FP64 if case["prec"] == "fp64" else S.SFAC_FP32
    fields = _fields(case, seed)
    if case["kind"] == "batch":
        inst = _instances(case)
        batch = S.Batch([p for p, _ in inst], prec)
        batch.prepare(fields, [k for _, k in inst])
        return {"kind": "batch", "batch": batch, "fields": fields}
    state = {"kind": case["kind"], "plan": S.Plan.for_problem(_problem(case), prec), "u": fields[0],
             "steps": case["steps"]}
    if case["kind"] == "host":
        state["u"] = fields[0].cpu().pin_memory()
    return state


def run(state):
    if state["kind"] == "batch":
        state["batch"].launch()
        return list(state["fields"])
    plan, u = state["plan"], state["u"]
    if state["kind"] == "host":
        plan.step_host(u.numpy(), state["steps"])
        return u
    plan.step(u, state["steps"])
    if state["kind"] == "monitored":
        umax, energy = plan.diagnostics(u)
        return [u, umax, energy]
    return u


def work(case):
    """Bytes: the field read once and written once. Flops: per point, axis and
    step six complex FFTs per two real lines, 5 N log2 N each, and ten for the
    multipliers, the twist and the nonlinear flow."""
    w = 8 if case["prec"] == "fp64" else 4
    if case["kind"] == "batch":
        items = [(p.n, k) for p, k in _instances(case)]
    else:
        items = [(_n(case), case["steps"])]
    nbytes = flops = 0
    for n, k in items:
        pts = math.prod(n)
        nbytes += 2 * w * pts
        flops += pts * k * sum(15 * math.log2(v) + 10 for v in n)
    return {"bytes": nbytes, "flops": int(flops)}


# ---- the same in 64 bits, in plain torch and numpy ----------------------------

def _factor_increment(n, alpha, eps, tau, a, b):
    """D = e^{tau/2 C} e^{tau S} e^{tau/2 C} - I of one axis, dense, and B's
    first column. The exponentials of the circulant and skew-circulant parts
    come from expm1 of their spectra, so D has the precision of its own size."""
    h = (b - a) / (n + 1)
    k = np.arange(n + 2, dtype=np.float64)
    g = np.cumprod(np.concatenate([[1.0], 1.0 - (alpha + 1.0) / k[1:]]))
    w = 0.5 * alpha * g
    w[1:] += 0.5 * (2.0 - alpha) * g[:-1]
    r = -eps * eps / (2.0 * h ** alpha * math.cos(alpha * math.pi / 2.0))
    bcol = np.zeros(n)
    bcol[0] = 2.0 * r * w[1]
    if n > 1:
        bcol[1] = r * (w[0] + w[2])
    bcol[2:] = r * w[3:n + 1]
    wrap = np.concatenate([[0.0], bcol[:0:-1]])
    c, s = 0.5 * (bcol + wrap), 0.5 * (bcol - wrap)
    c[0] = s[0] = 0.5 * bcol[0]
    j = np.arange(n)
    twist = np.exp(1j * math.pi * j / n)
    lam, mu = np.fft.fft(c).real, np.fft.fft(s * twist).real
    gc = np.fft.ifft(np.expm1(0.5 * tau * lam)).real
    hs = (np.fft.ifft(np.expm1(tau * mu)) * twist.conj()).real
    d = np.abs(j[:, None] - j[None, :])
    dev = "cuda"
    G, H = (torch.tensor(v[d], device=dev) for v in (gc, hs))
    W = H + G + H @ G
    return G + W + G @ W, torch.tensor(bcol[d], device=dev)


def _along(M, u, ax):
    dim = u.dim() - 1 - ax
    return torch.movedim(torch.tensordot(u, M, dims=([dim], [0])), -1, dim)


def _flow(v, s):
    q = -math.expm1(-2.0 * s) * (1.0 - v * v)
    r = torch.sqrt(1.0 - q)
    return v + v * q / (r * (1.0 + r))


def _solve(prob, u, steps, D):
    for _ in range(steps):
        u = _flow(u, 0.5 * prob.tau)
        for ax in range(prob.dim):
            u = u + _along(D[ax], u, ax)
        u = _flow(u, 0.5 * prob.tau)
    return u


def exact(case, seed):
    fields = [u.double() for u in _fields(case, seed)]
    items = _instances(case) if case["kind"] == "batch" else [(_problem(case), case["steps"])]
    out, seconds = [], 0.0
    for (p, steps), _ in zip(items, fields):
        seconds += p.points * steps * 2.0 * sum(p.n) / 1e12
    if seconds > 10.0:
        return None
    for (p, steps), u in zip(items, fields):
        DB = [_factor_increment(p.n[ax], p.alpha[ax], p.eps, p.tau, p.a, p.b) for ax in range(p.dim)]
        v = _solve(p, u, steps, [d for d, _ in DB])
        out.append(v)
        if case["kind"] == "monitored":
            Au = sum(_along(B, v, ax) for ax, (_, B) in enumerate(DB))
            vol = math.prod(p.h(ax) for ax in range(p.dim))
            energy = vol * float((0.25 * (v * v - 1.0) ** 2 - 0.5 * v * Au).sum())
            return [v, float(v.abs().max()), energy]
    return out if case["kind"] == "batch" else out[0].cpu() if case["kind"] == "host" else out[0]
