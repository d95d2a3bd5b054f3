"""What a user of the group explicit solver has it do, as measurable passes.

Every case goes through the ctypes binding as a program would call it: a
context, a batch plan or a surrogate model is made once and kept; a pass
loads new data, advances it and reads the result.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1310_3422_gb300 import binding as B

PREC = {"f64": B.GE_F64, "f32": B.GE_F32, "f32c": B.GE_F32_COMP}
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f32c": torch.float32}

# The surrogate's shape: 1024 points, 64 channels, 16 modes, 4 layers, 128 hidden.
SNO = (1024, 64, 16, 4, 128)


def listed():
    return [
        # one small problem to its final time: the first configuration (n = 1024, r = 1, 1000 steps from sin(pi x)),
        # where latency and launches are everything
        {"name": "solve_f64_small", "kind": "solve", "prec": "f64", "n": 1024, "r": 1.0, "steps": 1000,
         "bl": 0.0, "br": 0.0, "init": "sine"},
        # an odd mid-size problem with two wall values, the size of the tests' accuracy runs
        {"name": "solve_f64_mid", "kind": "solve", "prec": "f64", "n": 100003, "r": 0.7, "steps": 2000,
         "bl": 0.3, "br": -0.6, "init": "fourier"},
        # the headline problem: 2^24 points, r = 2, from a sum of sine modes
        {"name": "solve_f64_large", "kind": "solve", "prec": "f64", "n": 1 << 24, "r": 2.0, "steps": 2000,
         "bl": 0.0, "br": 0.0, "init": "modes"},
        # a program that looks at its field every few steps: few steps per call on a large grid
        {"name": "solve_f64_few_steps", "kind": "solve", "prec": "f64", "n": 1 << 22, "r": 0.5, "steps": 24,
         "bl": -0.2, "br": 0.9, "init": "fourier"},
        # the headline problem in single precision
        {"name": "solve_f32_large", "kind": "solve", "prec": "f32", "n": 1 << 24, "r": 2.0, "steps": 2000,
         "bl": 0.0, "br": 0.0, "init": "modes"},
        # a long single-precision run with compensated sums, from rough data (the accuracy option)
        {"name": "solve_f32c_long", "kind": "solve", "prec": "f32c", "n": 300001, "r": 1.7, "steps": 5000,
         "bl": 0.5, "br": -0.7, "init": "random"},
        # one-shot solve from host memory and back, context and all
        {"name": "host_solve_f64", "kind": "host", "prec": "f64", "n": 1 << 20, "r": 1.0, "steps": 1000,
         "bl": 0.0, "br": 0.0, "init": "modes"},
        # the batched configuration: 4096 uneven problems of 256 .. 65536 points, each with its own r and walls
        {"name": "batch_f32", "kind": "batch", "prec": "f32", "problems": 4096, "n_min": 256, "n_max": 65536,
         "steps": 2000},
        # a smaller batch at reference accuracy
        {"name": "batch_f64", "kind": "batch", "prec": "f64", "problems": 512, "n_min": 256, "n_max": 65536,
         "steps": 500},
        # the paper's own sub-domains of 16 points
        {"name": "width16_f64", "kind": "width", "prec": "f64", "n": 1 << 20, "r": 2.0, "steps": 200, "k": 16,
         "bl": 0.0, "br": 0.0, "init": "modes"},
        # one jump of the learned surrogate for a batch of problems (inference)
        {"name": "surrogate_forward", "kind": "sno_forward", "problems": 4096},
        # loss and gradient of one training batch of the surrogate (forward and backward)
        {"name": "surrogate_grad", "kind": "sno_grad", "problems": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["host", "batch", "batch", "width", "sno_forward", "sno_grad"])
    walls = {"bl": round(rng.uniform(-1, 1), 3), "br": round(rng.uniform(-1, 1), 3)}
    r = round(math.exp(rng.uniform(math.log(0.25), math.log(4.0))), 4)
    if kind in ("solve", "host"):
        n = _log_int(rng, 1000, 1 << (24 if kind == "solve" else 21))
        steps = min(_log_int(rng, 16, 5000), max(16, 33_000_000_000 // n))
        prec = rng.choice(["f64", "f64", "f32", "f32c"])
        return {"kind": kind, "prec": prec, "n": n, "r": r, "steps": steps,
                "init": rng.choice(["modes", "fourier", "random", "tents"]), **walls}
    if kind == "batch":
        prec = rng.choice(["f32", "f64", "f32c"])
        problems = _log_int(rng, 16, 4096 if prec == "f32" else 1024)
        return {"kind": kind, "prec": prec, "problems": problems, "n_min": 256,
                "n_max": _log_int(rng, 1024, 65536), "steps": _log_int(rng, 32, 2000 if prec == "f32" else 500)}
    if kind == "width":
        return {"kind": kind, "prec": rng.choice(["f64", "f32"]), "n": _log_int(rng, 1000, 1 << 21), "r": r,
                "steps": _log_int(rng, 8, 200), "k": rng.randint(2, 40), "init": "fourier", **walls}
    if kind == "sno_forward":
        return {"kind": kind, "problems": _log_int(rng, 1, 4096)}
    return {"kind": kind, "problems": _log_int(rng, 4, 128)}


# ---------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 13)
    return g


def _initial(init, n, bl, br, seed):
    """float64 state on the interior points x_i = (i + 1) / (n + 1)."""
    rng = np.random.default_rng(seed + 101)
    x = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") / float(n + 1)
    if init == "sine":
        return torch.sin(math.pi * x) * (1.0 + 0.1 * rng.uniform(-1, 1))
    if init == "modes":  # eight modes of 1 .. 64, amplitudes in (-1, 1)
        u = torch.zeros_like(x)
        for k, a in zip(rng.choice(np.arange(1, 65), size=8, replace=False), rng.uniform(-1, 1, 8)):
            u += float(a) * torch.sin(float(k) * math.pi * x)
        return u
    if init == "random":  # rough data, the worst case for round-off
        return torch.randn(n, dtype=torch.float64, device="cuda", generator=_gen(seed))
    u = bl + (br - bl) * x  # fourier, tents: the wall profile and a decaying series
    for k, a in enumerate(rng.standard_normal(16), 1):
        u += float(a) / (k * k) * torch.sin(k * math.pi * x)
    if init == "tents":
        for _ in range(2):
            c, w, h = rng.uniform(0.1, 0.9), rng.uniform(0.02, 0.2), rng.normal(0.0, 0.5)
            u += float(h) * torch.clamp(1.0 - (x - float(c)).abs() / float(w), min=0.0)
    return u


def _sizes(case):
    """Even problem sizes, log-uniform in the case's range: the case's own, whatever the data."""
    rng = np.random.default_rng(case["problems"])
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    n = np.exp(rng.uniform(lo, hi, case["problems"])).round().astype(np.int64) // 2 * 2
    return np.maximum(n, case["n_min"])


def _batch_inputs(case, seed):
    """Uneven problems packed on 32-element boundaries, and the packed state."""
    p = case["problems"]
    n = _sizes(case)
    rng = np.random.default_rng(seed + 202)
    r, bl, br = rng.uniform(0.25, 4.0, p), rng.uniform(-1, 1, p), rng.uniform(-1, 1, p)
    padded = (n + 31) // 32 * 32
    off = np.concatenate([[0], np.cumsum(padded)[:-1]]).astype(np.int64)
    total = int(padded.sum())

    def per_point(v):
        return torch.repeat_interleave(torch.from_numpy(np.ascontiguousarray(v)).cuda(),
                                       torch.from_numpy(padded).cuda(), output_size=total)

    nn = per_point(n)
    j = torch.arange(total, device="cuda") - per_point(off)
    x = (j + 1).double() / (nn + 1).double()
    u = per_point(bl) + per_point(br - bl) * x
    amps = rng.standard_normal((16, p))
    for k in range(1, 17):
        u += per_point(amps[k - 1] / (k * k)) * torch.sin(k * math.pi * x)
    u = torch.where(j < nn, u, torch.zeros_like(u))
    return n, r, bl, br, off, total, u, j, nn, per_point


def _sno_inputs(case, seed):
    """Surrogate problems: r in [0.5, 4], walls in (-1, 1), Fourier series and two tents."""
    n, p, g = SNO[0], case["problems"], _gen(seed + 303)

    def uni(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)

    x = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") / float(n + 1)
    r, bl, br = uni(0.5, 4.0, p), uni(-1, 1, p), uni(-1, 1, p)
    u0 = bl[:, None] + (br - bl)[:, None] * x
    for k in range(1, 17):
        a = torch.randn(p, 1, dtype=torch.float64, device="cuda", generator=g)
        u0 = u0 + a / (k * k) * torch.sin(k * math.pi * x)
    for _ in range(2):
        c, w = uni(0.1, 0.9, p, 1), uni(0.02, 0.2, p, 1)
        h = 0.5 * torch.randn(p, 1, dtype=torch.float64, device="cuda", generator=g)
        u0 = u0 + h * torch.clamp(1.0 - (x - c).abs() / w, min=0.0)
    return [t.float().contiguous() for t in (u0, r, bl, br)]


def _sno_target(u0, r, bl, br):
    """The state 256 group explicit steps later (the surrogate's training target)."""
    p, n = u0.shape
    off = np.arange(p, dtype=np.int64) * n
    u = u0.reshape(-1).clone()
    cpu = [t.double().cpu().numpy() for t in (r, bl, br)]
    B.ge_solve_batch(np.full(p, n, np.int64), *cpu, off, p * n, u, 256, B.GE_F32)
    torch.cuda.synchronize()
    return u.view(p, n)


# ---------------------------------------------------------------- a pass


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "width", "host"):
        dt = DTYPE[case["prec"]]
        u0 = _initial(case["init"], case["n"], case["bl"], case["br"], seed).to(dt)
        if kind == "host":
            host = u0.cpu().numpy()
            return {"case": case, "u0": host, "out": np.empty_like(host)}
        torch.cuda.synchronize()
        ctx = B.ge_create(case["n"], case["r"], case["bl"], case["br"], PREC[case["prec"]], u0)
        if kind == "width":
            B.ge_set_subdomain_width(ctx, case["k"])
        return {"case": case, "ctx": ctx, "u0": u0, "out": torch.empty_like(u0)}
    if kind == "batch":
        n, r, bl, br, off, total, u, *_ = _batch_inputs(case, seed)
        u0 = u.to(DTYPE[case["prec"]])
        torch.cuda.synchronize()
        plan = B.ge_batch_create(n, r, bl, br, off, total, PREC[case["prec"]])
        return {"case": case, "plan": plan, "u0": u0, "u": torch.empty_like(u0)}
    u0, r, bl, br = _sno_inputs(case, seed)
    p = case["problems"]
    state = {"case": case, "args": (u0, r, bl, br), "pred": torch.empty_like(u0)}
    if kind == "sno_grad":
        state["target"] = _sno_target(u0, r, bl, br)
        state["loss"] = torch.empty(p, device="cuda")
    torch.cuda.synchronize()
    state["model"] = B.ge_sno_create(*SNO, p, 1 + seed % 1000)
    if kind == "sno_grad":
        state["grads"] = torch.empty(B.ge_sno_num_params(state["model"]), device="cuda")
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("solve", "width"):
        B.ge_write_state(state["ctx"], state["u0"], 0)
        B.ge_step_n(state["ctx"], case["steps"])
        B.ge_read_state(state["ctx"], state["out"])
        return state["out"]
    if kind == "host":
        B.ge_solve(case["n"], case["r"], case["bl"], case["br"], PREC[case["prec"]], B.GE_KERNEL_AUTO, 0,
                   case["steps"], state["u0"], state["out"])
        return state["out"]
    if kind == "batch":
        state["u"].copy_(state["u0"])
        B.ge_batch_run(state["plan"], state["u"], case["steps"])
        return state["u"]
    if kind == "sno_forward":
        B.ge_sno_forward(state["model"], case["problems"], *state["args"], state["pred"])
        return state["pred"]
    B.ge_sno_loss_grad(state["model"], case["problems"], *state["args"], state["target"], state["loss"],
                       state["grads"])
    return [state["loss"], state["grads"]]


def work(case):
    kind = case["kind"]
    if kind.startswith("sno"):
        n, c, m, layers, h = SNO
        macs = n * (4 * c + layers * (c * c + 2 * c * 2 * m) + c * h + h) + layers * m * 4 * c * c
        params = 5 * c + layers * (2 * m * c * c + c * c + c) + c * h + 2 * h + 1
        p = case["problems"]
        if kind == "sno_forward":
            return {"bytes": 8.0 * p * n + 4.0 * params, "flops": 2.0 * macs * p}
        return {"bytes": 8.0 * p * n + 8.0 * params, "flops": 6.0 * macs * p}
    size = 8.0 if case["prec"] == "f64" else 4.0
    points = float(_sizes(case).sum()) if kind == "batch" else case["n"]
    # the state read once and written once; one multiply-add per point and step (the group form of the scheme),
    # three for sub-domains wider than one point
    return {"bytes": 2.0 * size * points, "flops": (6.0 if kind == "width" else 2.0) * points * case["steps"]}


# ---------------------------------------------------------------- 64-bit values


def _swap(x, parity):
    """x with every group's two points exchanged; a point without a partner keeps its place."""
    y = x.clone()
    if parity == 0:
        m = x.numel() // 2 * 2
        y[:m] = x[:m].view(-1, 2).flip(1).reshape(-1)
    else:
        m = (x.numel() - 1) // 2 * 2
        y[1:1 + m] = x[1:1 + m].view(-1, 2).flip(1).reshape(-1)
    return y


def _group_steps(u, j, n, r, bl, br, steps):
    """`steps` group explicit steps of problems packed at even offsets: j the
    point's index in its problem, n, r, bl, br its problem's numbers (tensors
    of every point, or numbers).  With w = (I - r G') u + f the right-hand side
    of a step's groups, a step is w <- (I - r G)(I + r G)^-1 w + f."""
    inside = j < n
    paired = []
    for p in (0, 1):
        partner = (j + p) % 2 * -2 + 1 + j
        paired.append((partner >= 0) & (partner < n) & inside)
    one = torch.ones_like(u)
    f = one * (j == 0) * (r * bl) + one * (j == n - 1) * (r * br)
    g = paired[1]
    w = torch.where(g, (1 - r) * u + r * _swap(u, 1), (1 - r) * u) + f
    coef = []
    for p in (0, 1):
        # as w + a w + b (partner - w) + f: what a group's points exchange cancels exactly
        a = torch.where(paired[p], 0.0 * one, one * -2 * r / (1 + r)) * inside
        b = torch.where(paired[p], one * 2 * r / (1 + 2 * r), 0.0 * one)
        coef.append((a, b))
    for s in range(steps - 1):
        a, b = coef[s & 1]
        w = (w + f).addcmul_(a, w).addcmul_(b, _swap(w, s & 1).sub_(w))
    p = (steps - 1) & 1
    return torch.where(paired[p], ((1 + r) * w + r * _swap(w, p)) / (1 + 2 * r), w / (1 + r)) * inside


def _width_steps(u, k, r, bl, br, steps):
    """`steps` steps with sub-domains of k points.  Paper node i = 1 .. n lies
    in sub-domain i // k; at parity p it takes Saul'yev A when i // k + p is
    even, else B; each B run and the A run to its right meet in a coupled pair."""
    n = u.numel()
    x = torch.zeros(n + 2, dtype=torch.float64, device=u.device)
    x[0], x[-1], x[1:-1] = bl, br, u
    node = np.arange(1, n + 1)
    plans = []
    for p in (0, 1):
        is_a = (node // k + p) % 2 == 0
        # order of each node: distance from its run's first computed node
        rank = np.zeros(n, np.int64)
        pair = np.zeros(n, bool)  # left members of the coupled pairs
        pair[:-1] = ~is_a[:-1] & is_a[1:]
        member = pair.copy()
        member[1:] |= pair[:-1]
        start = np.flatnonzero(np.concatenate([[True], is_a[1:] != is_a[:-1]]))
        first = np.zeros(n, np.int64)
        first[start] = start
        first = np.maximum.accumulate(first)
        end = np.concatenate([start[1:], [n]]) - 1
        last = end[np.searchsorted(start, node - 1, side="right") - 1]
        rank = np.where(is_a, node - 1 - first, last - (node - 1))
        todo = []
        for t in range(int(rank.max()) + 1):
            sel = (rank == t) & ~member
            todo.append([torch.from_numpy(np.ascontiguousarray(node[sel & m])).to(u.device)
                         for m in (is_a, ~is_a)])
        plans.append((torch.from_numpy(np.ascontiguousarray(node[pair])).to(u.device), todo))
    for s in range(steps):
        left, todo = plans[s & 1]
        y = x.clone()
        bi = (1 - r) * x[left] + r * x[left - 1]
        ai = (1 - r) * x[left + 1] + r * x[left + 2]
        y[left] = ((1 + r) * bi + r * ai) / (1 + 2 * r)
        y[left + 1] = ((1 + r) * ai + r * bi) / (1 + 2 * r)
        for ia, ib in todo:
            if ia.numel():
                y[ia] = ((1 - r) * x[ia] + r * x[ia + 1] + r * y[ia - 1]) / (1 + r)
            if ib.numel():
                y[ib] = ((1 - r) * x[ib] + r * x[ib - 1] + r * y[ib + 1]) / (1 + r)
        x = y
    return x[1:-1]


def _network(p, u0, r, bl, br):
    """The surrogate in float64 from its flat parameter vector."""
    n, c, m, layers, h = SNO
    at = 0

    def take(*shape):
        nonlocal at
        size = int(np.prod(shape))
        at += size
        return p[at - size:at].view(*shape)

    x = (torch.arange(1, n + 1, dtype=torch.float64, device=u0.device) / (n + 1)).expand_as(u0)
    v = torch.stack([u0, x, r[:, None].expand_as(u0), bl[:, None] + (br - bl)[:, None] * x], -1)
    v = v @ take(4, c) + take(c)
    # the truncated transform as products with its cosines and sines
    ang = 2 * math.pi / n * torch.outer(torch.arange(m, dtype=torch.float64, device=u0.device),
                                        torch.arange(n, dtype=torch.float64, device=u0.device))
    cos, sin = torch.cos(ang), torch.sin(ang)
    scale = torch.full((m, 1), 2.0 / n, dtype=torch.float64, device=u0.device)
    scale[0] = 1.0 / n
    for layer in range(layers):
        rr, ri = take(m, c, c), take(m, c, c)
        w, b = take(c, c), take(c)
        re, im = torch.einsum("mn,pnc->pmc", cos, v), -torch.einsum("mn,pnc->pmc", sin, v)
        yr = torch.einsum("moi,pmi->pmo", rr, re) - torch.einsum("moi,pmi->pmo", ri, im)
        yi = torch.einsum("moi,pmi->pmo", rr, im) + torch.einsum("moi,pmi->pmo", ri, re)
        v = torch.einsum("mn,pmc->pnc", cos * scale, yr) - torch.einsum("mn,pmc->pnc", sin * scale, yi) + v @ w + b
        if layer < layers - 1:
            v = torch.nn.functional.gelu(v, approximate="tanh")
    hid = torch.nn.functional.gelu(v @ take(c, h) + take(h), approximate="tanh")
    return u0 + hid @ take(h) + take(1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "host"):
        u = _initial(case["init"], case["n"], case["bl"], case["br"], seed).to(DTYPE[case["prec"]]).double()
        j = torch.arange(case["n"], device="cuda")
        out = _group_steps(u, j, case["n"], case["r"], case["bl"], case["br"], case["steps"])
        return out.cpu().numpy() if kind == "host" else out
    if kind == "width":
        u = _initial(case["init"], case["n"], case["bl"], case["br"], seed).to(DTYPE[case["prec"]]).double()
        return _width_steps(u, case["k"], case["r"], case["bl"], case["br"], case["steps"])
    if kind == "batch":
        n, r, bl, br, off, total, u, j, nn, per_point = _batch_inputs(case, seed)
        u = u.to(DTYPE[case["prec"]]).double()
        return _group_steps(u, j, nn, per_point(r), per_point(bl), per_point(br), case["steps"])
    state = prepare(case, seed)
    params = torch.empty(B.ge_sno_num_params(state["model"]), device="cuda")
    B.ge_sno_get_params(state["model"], params)
    torch.cuda.synchronize()
    p = params.bfloat16().double()  # the network's weights are BF16 values
    u0, r, bl, br = (t.double() for t in state["args"])
    if kind == "sno_forward":
        with torch.no_grad():
            return torch.cat([_network(p, *(t[i:i + 256] for t in (u0, r, bl, br))) for i in range(0, len(u0), 256)])
    p.requires_grad_(True)
    target = state["target"].double()
    loss = torch.linalg.vector_norm(_network(p, u0, r, bl, br) - target, dim=1) / torch.linalg.vector_norm(target, dim=1)
    loss.mean().backward()
    return [loss.detach(), p.grad]
