"""What this library is timed on: calls of its public entry points as user
programs make them, over the range of sizes and options in use.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  what a program has in hand before the call
    run(state)           one pass; returns every output
    work(case)           the bytes and operations one pass cannot do without
    exact(case, seed)    the outputs in 64-bit arithmetic, where they have such a value

All inputs are made on the GPU from the seed: jittered lattices that carry a
mixture of Gaussian vortices, Lamb-Oseen vortices on uniform lattices, and
input rows of the weight-proposal network.
"""
import math

import numpy as np
import torch

import paper_1508_06379_gb300 as vrm
from paper_1508_06379_gb300 import learn

NU = 1e-3


def listed():
    return [
        # the smallest run a user makes: the paper's Lamb-Oseen lattice of spacing 0.02 (about 870
        # particles), where the latency of one step is what counts
        {"name": "step_vortex_870", "kind": "step", "field": "vortex", "h": 0.02, "order": 1, "precision": "fp64",
         "learned": False},
        # an ordinary cloud of a run that is still growing, odd-sized, with the fp32 application
        {"name": "step_cloud_20k_mixed", "kind": "step", "field": "mixture", "side": 143, "order": 1,
         "precision": "mixed", "learned": False},
        # the benchmark's cloud: a million jittered particles, every option at its default
        {"name": "step_cloud_1m", "kind": "step", "field": "mixture", "side": 1001, "order": 1, "precision": "fp64",
         "learned": False},
        # the third-order operator (nine moment rows), whose LPs need the full neighbourhoods
        {"name": "step_order2_250k", "kind": "step", "field": "mixture", "side": 501, "order": 2,
         "precision": "fp64", "learned": False},
        # a step whose weights a trained network proposes
        {"name": "step_learned_500k", "kind": "step", "field": "mixture", "side": 707, "order": 1,
         "precision": "fp64", "learned": True},
        # one step of the viscous run with advection, on the sheared particles a few steps in
        {"name": "rk3_vortex_500k", "kind": "rk3", "h": 7 * 2.0 ** -13, "velocity": "lamb_oseen",
         "precision": "fp64"},
        # many independent clouds of uneven size advanced together
        {"name": "batch_32_clouds", "kind": "batch", "clouds": 32, "n_lo": 10000, "n_hi": 300000},
        # thinning of a crowded cloud
        {"name": "remove_close_1m", "kind": "remove", "side": 1001},
        # the operator in its own calls, as a program with its own time integrator makes them:
        # neighbourhoods, weights and one application
        {"name": "operator_300k", "kind": "operator", "side": 547, "order": 1},
        # the particles' velocity on a 200 x 200 evaluation grid by direct summation
        {"name": "velocity_250k_on_40k", "kind": "velocity", "side": 501, "targets": 40000},
        # proposals of the network for a large cloud's rows
        {"name": "net_forward_500k", "kind": "forward", "rows": 499999},
        # a training step of the network: forward, backward, AdamW
        {"name": "net_train_4096", "kind": "train", "batch": 4096, "rows": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "order2", "learned", "rk3", "batch", "remove", "operator", "velocity",
                       "forward", "train"])
    if kind == "step" and rng.random() < 0.3:
        return {"kind": "step", "field": "vortex", "h": math.exp(rng.uniform(math.log(0.002), math.log(0.03))),
                "order": 1, "precision": rng.choice(["fp64", "mixed"]), "learned": False}
    if kind == "step":
        return {"kind": "step", "field": "mixture", "side": _log_int(rng, 30, 1001), "order": 1,
                "precision": rng.choice(["fp64", "mixed"]), "learned": False}
    if kind == "order2":
        return {"kind": "step", "field": "mixture", "side": _log_int(rng, 30, 501), "order": 2, "precision": "fp64",
                "learned": False}
    if kind == "learned":
        return {"kind": "step", "field": "mixture", "side": _log_int(rng, 40, 707), "order": 1,
                "precision": rng.choice(["fp64", "mixed"]), "learned": True}
    if kind == "rk3":
        own = rng.random() < 0.3
        return {"kind": "rk3", "h": math.exp(rng.uniform(math.log(3e-3 if own else 7 * 2.0 ** -13), math.log(1e-2))),
                "velocity": "self" if own else "lamb_oseen", "precision": rng.choice(["fp64", "mixed"])}
    if kind == "batch":
        lo = _log_int(rng, 1000, 20000)
        return {"kind": "batch", "clouds": rng.randint(2, 32), "n_lo": lo, "n_hi": _log_int(rng, 2 * lo, 200000)}
    if kind == "remove":
        return {"kind": "remove", "side": _log_int(rng, 40, 1001)}
    if kind == "operator":
        return {"kind": "operator", "side": _log_int(rng, 40, 547), "order": rng.choice([1, 1, 2])}
    if kind == "velocity":
        return {"kind": "velocity", "side": _log_int(rng, 30, 400), "targets": _log_int(rng, 300, 60000)}
    if kind == "forward":
        return {"kind": "forward", "rows": _log_int(rng, 1000, 499999)}
    batch = 128 * _log_int(rng, 4, 128)
    return {"kind": "train", "batch": batch, "rows": batch - rng.choice([0, 0, rng.randint(1, 127)])}


# ---- inputs ---------------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * (hi - lo) + lo


def _mixture_cloud(g, side, h, jitter=0.3, modes=8):
    """A side x side lattice of spacing h about the origin, jittered by up to
    0.3 h per coordinate, with the circulations of a mixture of Gaussians."""
    half = 0.5 * (side - 1) * h
    c = torch.arange(side, dtype=torch.float64, device="cuda") * h - half
    x = c.repeat(side) + _uniform(g, side * side, -jitter * h, jitter * h)
    y = c.repeat_interleave(side) + _uniform(g, side * side, -jitter * h, jitter * h)
    centre = _uniform(g, 2 * modes, -0.8 * half, 0.8 * half).view(2, modes)
    strength = torch.randn(modes, generator=g, dtype=torch.float64, device="cuda")
    sigma = _uniform(g, modes, 0.05 * half, 0.15 * half)
    w = torch.zeros_like(x)
    for k in range(modes):
        r2 = (x - centre[0, k]) ** 2 + (y - centre[1, k]) ** 2
        w += strength[k] / (2 * math.pi * sigma[k] ** 2) * torch.exp(-r2 / (2 * sigma[k] ** 2))
    return x, y, w * (h * h)


def _vortex_lattice(g, h, nu, lo, hi):
    """Lamb-Oseen vortex on the lattice k h + lo, where that of unit strength
    and age has |omega| > 1e-10; strength and age vary with the seed."""
    gamma, t = _uniform(g, 2, 0.9, 1.1).tolist()
    side = int(round((hi - lo) / h)) + 1
    c = torch.arange(side, dtype=torch.float64, device="cuda") * h + lo
    x, y = c.repeat(side), c.repeat_interleave(side)
    r2 = x * x + y * y
    keep = torch.exp(-r2 / (4 * nu)) / (4 * math.pi * nu) > 1e-10
    x, y, r2 = x[keep], y[keep], r2[keep]
    return x, y, gamma / (4 * math.pi * nu * t) * torch.exp(-r2 / (4 * nu * t)) * (h * h), gamma, t


def _padded(v, cap):
    out = torch.zeros(cap, dtype=torch.float64, device="cuda")
    out[:v.numel()] = v
    return out


def _net_rows(g, rows):
    """Input rows as the neighbourhoods of a jittered cloud give them: 8 to 32
    filled slots, offsets in the annulus from 0.5 to 2 spacings."""
    pad = (rows + 127) // 128 * 128
    filled = torch.randint(8, 33, (pad, 1), generator=g, device="cuda")
    mask = (torch.arange(32, device="cuda") < filled).float()
    mask[rows:] = 0
    r = torch.sqrt(torch.rand(pad, 32, generator=g, device="cuda") * 3.75 + 0.25)
    a = torch.rand(pad, 32, generator=g, device="cuda") * (2 * math.pi)
    return torch.cat([r * torch.cos(a) * mask, r * torch.sin(a) * mask, mask, torch.zeros_like(mask)],
                     1).to(torch.bfloat16)


SHAPES = ((256, 96), (256, 256), (256, 256), (32, 256))


def _net_params(g):
    parts = []
    for out, inp in SHAPES:
        parts.append(torch.randn(out * inp, generator=g, device="cuda") / math.sqrt(inp))
        parts.append(torch.randn(out, generator=g, device="cuda") * 0.05)
    return torch.cat(parts)


def _layers(theta):
    at, out = 0, []
    for o, i in SHAPES:
        out.append((theta[at:at + o * i].view(o, i), theta[at + o * i:at + o * i + o]))
        at += o * i + o
    return out


def _network(theta, X):
    a = X[:, :96]
    for k, (w, b) in enumerate(_layers(theta)):
        a = a @ w.T + b
        if k < 3:
            a = torch.nn.functional.gelu(a, approximate="tanh")
    return a


_TRAINED = []


def _trained():
    """A program's trained network, the same for every cloud: a few hundred
    Adam steps on LP solutions, in torch."""
    if not _TRAINED:
        X, T, n = learn.make_dataset(150_000, side=401)
        X, T = X[:n].float(), T[:n]
        g = _gen(1508007)
        theta = _net_params(g).requires_grad_(True)
        opt = torch.optim.Adam([theta], lr=2e-3)
        steps = 400
        for k in range(steps):
            for q in opt.param_groups:
                q["lr"] = 2e-3 * 0.5 * (1 + math.cos(math.pi * k / steps)) + 1e-5
            idx = torch.randint(0, n, (8192,), generator=g, device="cuda")
            x, t = X[idx], T[idx]
            mask = x[:, 64:96]
            loss = (mask * (_network(theta, x) - t) ** 2).sum() / mask.sum()
            opt.zero_grad(set_to_none=True)
            loss.backward()
            opt.step()
        _TRAINED.append(theta.detach())
    return _TRAINED[0]


def _step_dt(h, nu):
    return (0.5 * h) ** 2 / (4 * nu) / 8


def _step_cloud(case, g):
    if case["field"] == "vortex":
        x, y, w, _, _ = _vortex_lattice(g, case["h"], NU, -1.0, 1.0)
        return x, y, w, case["h"], 0.25 * case["h"] ** 2 / NU
    h = 2.0 / (case["side"] - 1)
    return (*_mixture_cloud(g, case["side"], h), h, _step_dt(h, NU))


def _annulus(order):
    return 2.5 if order == 2 else 2.0


# ---- the cases' states ------------------------------------------------------------------


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, _gen(seed))


def run(state):
    return state["run"](state)


def _prepare_step(case, g):
    x, y, w, h, dt = _step_cloud(case, g)
    n = x.numel()
    cap = 2 * n + 1024
    ctx = vrm.VRM(h=h, nu=NU, R=_annulus(case["order"]), order=case["order"], precision=case["precision"])
    net = None
    if case["learned"]:
        net = vrm.MLP(batch_rows=128)
        net.set_params(_trained())
        ctx.set_mlp(net)
    return {"run": _run_step, "ctx": ctx, "net": net, "x": _padded(x, cap), "y": _padded(y, cap), "n": n, "gamma": w,
            "out": torch.zeros(cap, dtype=torch.float64, device="cuda"), "dt": dt}


COUNTS = ("n_diffused", "open_segments", "small_ok", "full_ok", "no_stencil", "learned_ok", "rounds", "max_dt_ratio")


def _run_step(s):
    n, st = s["ctx"].step(s["x"], s["y"], s["n"], s["gamma"], s["out"], s["dt"])
    return {"x": s["x"], "y": s["y"], "gamma": s["out"], "n": n, "stats": [st[k] for k in COUNTS]}


def _prepare_rk3(case, g):
    nu, h = 5e-4, case["h"]
    x, y, w, gamma, t = _vortex_lattice(g, h, nu, -0.25, 0.25)
    n = x.numel()
    cap = 3 * n + 4096
    umax = 0.64 * gamma / (2 * math.pi * 2.24 * math.sqrt(nu * t))
    dt = min((0.5 * h) ** 2 / (4 * nu), 0.25 * h / umax)
    vel = dict(gamma=gamma, nu=nu) if case["velocity"] == "lamb_oseen" else dict(eps=3 * h)
    ctx = vrm.VRM(h=h, nu=nu, precision=case["precision"])
    x, y, bufs = _padded(x, cap), _padded(y, cap), [_padded(w, cap), torch.zeros(cap, dtype=torch.float64,
                                                                                 device="cuda")]
    for k in range(2):  # the run's first steps, which shear the lattice and fill it up
        n, _ = ctx.rk3_step(x, y, n, bufs[k], bufs[1 - k], t, dt, vel)
        t += dt
    return {"run": _run_rk3, "ctx": ctx, "x0": x[:n].clone(), "y0": y[:n].clone(), "x": x, "y": y, "n": n,
            "gamma": bufs[0][:n].clone(), "out": bufs[1], "t": t, "dt": dt, "vel": vel}


def _run_rk3(s):
    # the step moves the particles in place: every pass starts from the same ones
    s["x"][:s["n"]].copy_(s["x0"])
    s["y"][:s["n"]].copy_(s["y0"])
    n, st = s["ctx"].rk3_step(s["x"], s["y"], s["n"], s["gamma"], s["out"], s["t"], s["dt"], s["vel"])
    return {"x": s["x"], "y": s["y"], "gamma": s["out"], "n": n, "stats": [st[k] for k in COUNTS]}


def _batch_sizes(case):
    """Log-uniform sizes and uniform spacings, the case's own."""
    rng, k = np.random.default_rng([case["clouds"], case["n_lo"], case["n_hi"]]), case["clouds"]
    n = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), k))
    return [max(2, int(round(math.sqrt(v)))) for v in n], rng.uniform(1e-3, 4e-3, k).tolist()


def _prepare_batch(case, g):
    sides, hs = _batch_sizes(case)
    caps = [(2 * s * s + 1024 + 63) // 64 * 64 for s in sides]
    x, y, out = (torch.zeros(sum(caps), dtype=torch.float64, device="cuda") for _ in range(3))
    clouds, at = [], 0
    for side, h, cap in zip(sides, hs, caps):
        n = side * side
        cx, cy, w = _mixture_cloud(g, side, h)
        x[at:at + n], y[at:at + n] = cx, cy
        clouds.append({"x": x[at:at + cap], "y": y[at:at + cap], "gamma_in": w, "gamma_out": out[at:at + cap], "n": n,
                       "h": h, "dt": _step_dt(h, NU)})
        at += cap
    return {"run": _run_batch, "batch": vrm.VRMBatch(case["clouds"], NU), "clouds": clouds, "x": x, "y": y, "out": out}


def _run_batch(s):
    per_cloud, st = s["batch"].step(s["clouds"])
    return {"x": s["x"], "y": s["y"], "gamma": s["out"], "n": np.array([n for n, _ in per_cloud]),
            "stats": [st[k] for k in COUNTS]}


def _prepare_remove(case, g):
    h = 2.0 / (case["side"] - 1)
    x, y, w = _mixture_cloud(g, case["side"], h)
    n = x.numel()
    m = max(1, n // 10)  # a tenth of the particles has a close neighbour
    k = torch.randperm(n, generator=g, device="cuda")[:m]
    x = torch.cat([x, x[k] + _uniform(g, m, -0.3 * h, 0.3 * h)])
    y = torch.cat([y, y[k] + _uniform(g, m, -0.3 * h, 0.3 * h)])
    w = torch.cat([w, w[k] * _uniform(g, m, -1.0, 1.0)])
    kept = torch.zeros(3, n + m, dtype=torch.float64, device="cuda")
    return {"run": _run_remove, "ctx": vrm.VRM(h=h, nu=NU), "x": x, "y": y, "gamma": w, "n": n + m, "kept": kept}


def _run_remove(s):
    *kept, n, st = s["ctx"].remove_close(s["x"], s["y"], s["gamma"], s["n"])
    for buf, v in zip(s["kept"], kept):  # the program's own arrays, whose length stays
        buf[:n].copy_(v)
    return {"kept": s["kept"], "n": n, "candidates": st["remove_candidates"]}


def _prepare_operator(case, g):
    h = 2.0 / (case["side"] - 1)
    order = case["order"]
    x0, y0, w = _mixture_cloud(g, case["side"], h)
    n0 = x0.numel()
    cap = 2 * n0 + 1024
    x, y = _padded(x0, cap), _padded(y0, cap)
    ctx = vrm.VRM(h=h, nu=NU, R=_annulus(order), order=order)
    n, diffused, _ = ctx.insert_reduce(x, y, n0, w)
    width = ctx.W

    def buf(count, dtype, fill):
        return torch.full((count,), fill, dtype=dtype, device="cuda")

    nb = {"count": buf(cap, torch.int32, 0), "idx": buf(32 * cap, torch.int32, -1), "mask": buf(cap, torch.uint8, 0),
          "small": buf(8 * cap, torch.int32, -1)}
    wt = {"cols": buf(width * cap, torch.int32, -1), "f": buf(width * cap, torch.float64, 0.0),
          "fii": buf(cap, torch.float64, 0.0), "status": buf(cap, torch.uint8, 0)}
    return {"run": _run_operator, "ctx": ctx, "x": x, "y": y, "n": n, "n0": n0, "gamma": w, "diffused": diffused,
            "nb": nb, "wt": wt, "dgamma": buf(cap, torch.float64, 0.0)}


def _run_operator(s):
    ctx, n = s["ctx"], s["n"]
    nb = ctx.build_neighbourhoods(s["x"], s["y"], n, out=s["nb"])
    w = ctx.solve_weights(s["x"], s["y"], n, s["diffused"], nb, out=s["wt"])
    dg = ctx.apply(n, s["n0"], s["gamma"], s["diffused"], nb, w, s["dgamma"])
    return {"dgamma": dg, "count": nb["count"], "idx": nb["idx"], "mask": nb["mask"], "small": nb["small"],
            "cols": w["cols"], "f": w["f"], "fii": w["fii"], "status": w["status"]}


def _prepare_velocity(case, g):
    h = 2.0 / (case["side"] - 1)
    x, y, w = _mixture_cloud(g, case["side"], h)
    m = case["targets"]
    side = int(math.ceil(math.sqrt(m)))
    shift = _uniform(g, 1, 0.0, 3.0 / side)
    c = (torch.arange(side, dtype=torch.float64, device="cuda") + 0.5) * (3.0 / side) - 1.5
    u, v = (torch.zeros(m, dtype=torch.float64, device="cuda") for _ in range(2))
    return {"run": _run_velocity, "ctx": vrm.VRM(h=h, nu=NU), "x": x, "y": y, "gamma": w, "n": x.numel(),
            "xt": (c + shift).repeat(side)[:m].contiguous(), "yt": c.repeat_interleave(side)[:m].contiguous(), "m": m,
            "eps": 3 * h, "u": u, "v": v}


def _run_velocity(s):
    u, v = s["ctx"].biot_savart(s["x"], s["y"], s["gamma"], s["n"], s["xt"], s["yt"], s["m"], s["eps"], s["u"], s["v"])
    return {"u": u, "v": v}


def _prepare_forward(case, g):
    net = vrm.MLP(batch_rows=128)
    theta = _net_params(g)
    net.set_params(theta)
    return {"run": _run_forward, "net": net, "theta": theta, "X": _net_rows(g, case["rows"]), "rows": case["rows"]}


def _run_forward(s):
    return {"Y": s["net"].forward(s["X"], s["rows"])}


TRAIN_SET = 100_000


def _prepare_train(case, g):
    net = vrm.MLP(batch_rows=case["batch"])
    theta = _net_params(g)
    net.set_params(theta)
    X = _net_rows(g, TRAIN_SET)
    xi, eta, mask = X[:, :32].float(), X[:, 32:64].float(), X[:, 64:96].float()
    T = (mask * (torch.relu(xi) / 2 + eta * eta / 8))[:TRAIN_SET].contiguous()
    rows = case["rows"]
    perm = torch.randperm(TRAIN_SET, generator=g, device="cuda").to(torch.int32)
    batches = [perm[k:k + rows].contiguous() for k in range(0, max(1, TRAIN_SET - rows + 1), rows)]
    return {"run": _run_train, "net": net, "theta": theta, "X": X, "T": T, "batches": batches, "t": 0,
            "loss": torch.zeros(2, dtype=torch.float32, device="cuda")}


def _run_train(s):
    s["t"] += 1
    idx = s["batches"][(s["t"] - 1) % len(s["batches"])]
    s["net"].train_step(s["X"], s["T"], idx, s["t"], loss_out=s["loss"], lr=1e-3)
    return {"theta": s["net"].get_params(), "loss": s["loss"]}


# ---- what a pass cannot do without ---------------------------------------------------------


def _step_work(n, order=1, stages=1):
    """Per particle given: position and circulation in, circulation out, and
    a third of it again for the inserted ones; the LP of the 0.7 that diffuse
    (the column offsets and the solve of the final basis), 36 pair tests, and
    the stencil's sums."""
    after = 1.3 * n
    lp = 203 if order == 1 else 900
    return {"bytes": 24 * n + 8 * after + 16 * (after - n),
            "flops": stages * (0.7 * n * (lp + 36 * 6) + 2 * 5.5 * 0.7 * n)}


def work(case):
    kind = case["kind"]
    if kind == "step":
        n = math.pi * 0.106 / case["h"] ** 2 if case["field"] == "vortex" else case["side"] ** 2
        w = _step_work(n, case["order"])
        if case["learned"]:
            w["flops"] += 0.7 * n * 2 * vrm.MLP_PARAMS
        return w
    if kind == "rk3":
        n = 2 * math.pi * 0.056 / case["h"] ** 2
        w = _step_work(n, stages=3)
        w["bytes"] += 16 * n
        if case["velocity"] == "self":
            w["flops"] += 3 * 20 * n * n
        return w
    if kind == "batch":
        lo, hi = case["n_lo"], case["n_hi"]
        return _step_work(case["clouds"] * (hi - lo) / math.log(hi / lo))
    if kind == "remove":
        n = 1.1 * case["side"] ** 2
        return {"bytes": 24 * n + 24 * n, "flops": n * 40 * 6}
    if kind == "operator":
        n = 1.3 * case["side"] ** 2
        width = 8 if case["order"] == 1 else 12
        out = 4 + 4 * 13 + 1 + 32 + width * 12 + 8 + 1 + 8
        return {"bytes": n * (24 + out), "flops": n * (36 * 6 + (203 if case["order"] == 1 else 900))}
    if kind == "velocity":
        n, m = case["side"] ** 2, case["targets"]
        return {"bytes": 24 * n + 32 * m, "flops": 20.0 * n * m}
    if kind == "forward":
        return {"bytes": case["rows"] * (192 + 128) + 4 * vrm.MLP_PARAMS, "flops": 2.0 * vrm.MLP_PARAMS * case["rows"]}
    return {"bytes": case["rows"] * (192 + 128) + 4 * 7 * vrm.MLP_PARAMS, "flops": 6.0 * vrm.MLP_PARAMS * case["rows"]}


# ---- 64-bit values -------------------------------------------------------------------------


def exact(case, seed):
    if case["kind"] not in ("velocity", "forward", "train"):
        return None  # which vertex of an LP's solutions is taken is the method's own choice
    s = prepare(case, seed)
    if case["kind"] == "velocity":
        return _exact_velocity(s)
    theta = s["theta"].double()
    if case["kind"] == "forward":
        return {"Y": _network(theta, s["X"][:s["rows"]].double())}
    idx = s["batches"][0].long()
    x, t = s["X"][idx].double(), s["T"][idx].double()
    mask = x[:, 64:96]
    theta.requires_grad_(True)
    loss = ((mask * (_network(theta, x) - t)) ** 2).sum() / mask.sum()
    (grad,) = torch.autograd.grad(loss, theta)
    # the first AdamW step: the corrected moments are the gradient and its square
    new = theta.detach() - 1e-3 * grad / (grad.abs() + 1e-8)
    return {"theta": new, "loss": torch.stack([loss.detach(), mask.sum()])}


def _exact_velocity(s):
    u, v = torch.zeros_like(s["u"]), torch.zeros_like(s["v"])
    c = 1 / (2 * math.pi)
    per = max(1, (1 << 26) // s["n"])
    for k in range(0, s["m"], per):
        dx = s["xt"][k:k + per, None] - s["x"][None]
        dy = s["yt"][k:k + per, None] - s["y"][None]
        r2 = dx * dx + dy * dy
        kern = -torch.expm1(-r2 / s["eps"] ** 2) / torch.where(r2 > 0, r2, torch.ones_like(r2)) * s["gamma"] * c
        u[k:k + per] = -(dy * kern).sum(1)
        v[k:k + per] = (dx * kern).sum(1)
    return {"u": u, "v": v}
