"""What a user of this framework has it do, as cases that can be timed and checked.

A case names a kind of call, the instances it is made on and the arithmetic.  Sizes are those of the
benchmark's workloads: one instance of 50 circles (plain binary64), one of 1000, the batch of 4096
instances of 300 to 1000 circles, one of 100000 circles, the container adjustment's 304 instances,
and the learned form's sets of 512 (training) and 1024 (evaluation) instances.  The densities
n / R^2 lie in [0.80, 0.84].

Layouts are drawn here, from a seed: "packed" ones (a hexagonal lattice of the instance's density,
shifted, rotated and jittered: every circle with about six neighbors, as near the end of a descent)
and "random" ones (uniform in the disk, as a descent starts).  Their coordinates are binary32 values
held in binary64, so that every arithmetic form sees the same layout.
"""
import math

import numpy as np
import torch

from paper_2303_02650_gb300 import pecc

PREC = {"fp64": pecc.FP64, "fp32": pecc.FP32, "mixed": pecc.FP32_POLISH64}
L_CUT = 2.5       # neighbor cutoff of every context (the default)
DEGREE = 6.0      # list entries of a circle in a packed layout
# the settings of the benchmark's descents
BATCH = {"k_batches": 2, "step_max": 0.3, "polish_gate": 1e-5, "stall_window": 5, "polish_stall_window": 50,
         "lbfgs_m": 5}
H, FEATURES, KNN, KNN_CUT = 128, 25, 12, 4.5


def listed():
    return [
        # one evaluation of the smallest instance in plain binary64: latency and launches
        dict(name="evaluate_50_fp64", kind="evaluate", num=1, n_lo=50, n_hi=50, prec="fp64", layout="packed"),
        # energy and gradient of the batch over lists in hand: the hot kernel by itself
        dict(name="energy_grad_4096", kind="energy_grad", num=4096, n_lo=300, n_hi=1000, prec="fp32", layout="packed"),
        # a caller's own optimiser step on the batch: new positions, lists, energy and gradient
        dict(name="evaluate_4096", kind="evaluate", num=4096, n_lo=300, n_hi=1000, prec="fp32", layout="packed"),
        # the same on one large instance
        dict(name="evaluate_100k", kind="evaluate", num=1, n_lo=100000, n_hi=100000, prec="fp32", layout="packed"),
        # the judge of finished layouts: largest overlap of every instance in binary64
        dict(name="feasible_4096", kind="feasible", num=4096, n_lo=300, n_hi=1000, layout="packed"),
        # one instance from host memory to host memory: the latency a single search sees
        dict(name="solve_1000", kind="solve", num=1, n_lo=1000, n_hi=1000),
        # the plain method: one small instance in binary64, up to 2000 sweeps
        dict(name="descend_50_fp64", kind="descend", num=1, n_lo=50, n_hi=50, prec="fp64"),
        # the batch: every instance drawn, descended, polished and checked in one call sequence
        dict(name="descend_4096", kind="descend", num=4096, n_lo=300, n_hi=1000, prec="mixed"),
        # one large instance, descended by the whole GPU
        dict(name="descend_100k", kind="descend", num=1, n_lo=100000, n_hi=100000, prec="fp32"),
        # container adjustment of finished layouts: the first rounds of its schedule
        dict(name="adjust_304", kind="adjust", num=304, n_lo=300, n_hi=1000, layout="packed", rounds=6,
             max_iter=50),
        # gradient of the learned form's loss over the circles of one training round
        dict(name="mlp_grad_333k", kind="mlp_grad", rows=333001),
        # the learned form's proposals for the circles of its evaluation set
        dict(name="propose_1024", kind="propose", num=1024, n_lo=300, n_hi=1000, layout="packed"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _instances(rng, num_hi, n_lo, n_hi, circles):
    """A number of instances and a range of sizes, at most `circles` circles in all."""
    lo = _log_int(rng, n_lo, n_hi)
    hi = min(n_hi, _log_int(rng, lo, max(lo, min(n_hi, 3 * lo))))
    return dict(num=_log_int(rng, 1, max(1, min(num_hi, circles // hi))), n_lo=lo, n_hi=hi)


def draw(rng):
    kind = rng.choice(["energy_grad", "evaluate", "evaluate_large", "feasible", "descend", "descend_large", "solve",
                       "adjust", "mlp_grad", "propose"])
    layout = rng.choice(["packed", "packed", "random"])
    prec = rng.choice(["fp32", "fp32", "fp64", "mixed"])
    if kind in ("energy_grad", "evaluate"):
        return dict(kind=kind, prec=prec, layout=layout, **_instances(rng, 4096, 50, 1000, 2600000))
    if kind == "evaluate_large":
        n = _log_int(rng, 1001, 100000)
        return dict(kind="evaluate", prec=prec, layout=layout, num=1, n_lo=n, n_hi=n)
    if kind == "feasible":
        return dict(kind=kind, layout=layout, **_instances(rng, 4096, 50, 1000, 2600000))
    if kind == "descend":
        prec = rng.choice(["mixed", "mixed", "fp32", "fp64"])
        if prec == "fp64":  # small instances: every one runs its 2000 sweeps
            return dict(kind=kind, prec=prec, **_instances(rng, 32, 20, 50, 1600))
        return dict(kind=kind, prec=prec, **_instances(rng, 2048, 50, 600, 1200000))
    if kind == "descend_large":
        n = _log_int(rng, 16384, 90000)
        return dict(kind="descend", prec="fp32", num=1, n_lo=n, n_hi=n)
    if kind == "solve":
        n = _log_int(rng, 50, 1000)
        return dict(kind=kind, num=1, n_lo=n, n_hi=n)
    if kind == "adjust":
        return dict(kind=kind, layout="packed", rounds=rng.randint(2, 6), max_iter=50,
                    **_instances(rng, 304, 50, 1000, 190000))
    if kind == "mlp_grad":
        return dict(kind=kind, rows=_log_int(rng, 1000, 333000))
    return dict(kind=kind, layout=layout, **_instances(rng, 1024, 50, 1000, 600000))


# ---------------------------------------------------------------------------------------- inputs
def _sizes(case):
    """Sizes and radii of a case's instances (the same for every seed)."""
    g = np.random.Generator(np.random.Philox([case["num"], case["n_lo"] * 1000003 + case["n_hi"]]))
    n = g.integers(case["n_lo"], case["n_hi"] + 1, size=case["num"]).astype(np.int32)
    return n, np.sqrt(n / g.uniform(0.80, 0.84, size=case["num"]))


def _layout(case, n, R, seed, jitter):
    """Centres of every instance, instances concatenated: float64 [sum n, 2] of binary32 values."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    f64 = dict(dtype=torch.float64, device=dev)
    nt = torch.as_tensor(n, dtype=torch.int64, device=dev)
    Rt = torch.as_tensor(R, **f64)
    total, num, nmax = int(n.sum()), len(n), int(n.max())
    if case["layout"] == "random":
        rad = torch.sqrt(torch.rand(total, generator=g, **f64)) * torch.repeat_interleave(Rt - 1.0, nt)
        phi = 2.0 * math.pi * torch.rand(total, generator=g, **f64)
        xy = torch.stack([rad * torch.cos(phi), rad * torch.sin(phi)], 1)
        return xy.float().double().contiguous()
    # the n lattice points nearest to a random centre, scaled to the disk of radius R - 1
    reach = int(math.sqrt(nmax * math.sqrt(0.75) / math.pi)) + 3
    a = torch.arange(-2 * reach, 2 * reach + 1, **f64)
    px = (a[None, :] + 0.5 * a[:, None]).reshape(-1)
    py = (math.sqrt(0.75) * a[:, None]).expand(-1, a.numel()).reshape(-1)
    near = px * px + py * py <= (reach + 1.0) ** 2
    px, py = px[near], py[near]
    out = []
    step = max(1, 20000000 // px.numel())
    for q0 in range(0, num, step):
        q1 = min(num, q0 + step)
        c = torch.rand((q1 - q0, 2), generator=g, **f64) - 0.5
        phi = 2.0 * math.pi * torch.rand(q1 - q0, generator=g, **f64)[:, None]
        dx, dy = px[None, :] - c[:, :1], py[None, :] - c[:, 1:]
        r, order = torch.sort(dx * dx + dy * dy, dim=1, stable=True)
        m = nt[q0:q1]
        last = torch.sqrt(torch.gather(r, 1, (m - 1)[:, None]))
        scale = ((Rt[q0:q1, None] - 1.0) / last.clamp_min(1e-9))
        x, y = torch.gather(dx, 1, order) * scale, torch.gather(dy, 1, order) * scale
        x, y = x * torch.cos(phi) - y * torch.sin(phi), x * torch.sin(phi) + y * torch.cos(phi)
        # the circles of an instance in no particular order
        key = torch.rand(x.shape, generator=g, **f64)
        inside = torch.arange(px.numel(), device=dev)[None, :] < m[:, None]
        shuffle = torch.argsort(torch.where(inside, key, 2.0 + key), dim=1)
        x, y = torch.gather(x, 1, shuffle), torch.gather(y, 1, shuffle)
        out.append(torch.stack([x[inside], y[inside]], 1))
    xy = torch.cat(out)
    xy += jitter * (2.0 * torch.rand(xy.shape, generator=g, **f64) - 1.0)
    return xy.float().double().contiguous()


def _jitter(case):
    # checked layouts are finished ones, some of them feasible; the others still overlap a little
    return {"feasible": 0.01, "adjust": 0.05}.get(case["kind"], 0.1)


def _network(seed):
    """He-uniform weights and small biases: W1[128][25] b1 W2[128][128] b2 W3[128][128] b3 W4[2][128] b4."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    parts = []
    for o, i in ((H, FEATURES), (H, H), (H, H), (2, H)):
        parts.append((2.0 * torch.rand(o * i, generator=g, device="cuda") - 1.0) * math.sqrt(6.0 / i))
        parts.append(0.05 * torch.randn(o, generator=g, device="cuda"))
    return torch.cat(parts)


def _samples(rows, seed):
    """Feature rows (offsets of the nearest neighbors, the wall distance) and displacement targets."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    rad = torch.sort(1.5 + 3.0 * torch.rand((rows, KNN), generator=g, device="cuda"), dim=1).values
    phi = 2.0 * math.pi * torch.rand((rows, KNN), generator=g, device="cuda")
    off = torch.stack([rad * torch.cos(phi), rad * torch.sin(phi)], 2)
    off[rad > 4.3] = 0.0  # fewer than twelve neighbors within the cutoff
    wall = (30.0 * torch.rand((rows, 1), generator=g, device="cuda")).clamp_max(KNN_CUT)
    feat = torch.cat([off.reshape(rows, 2 * KNN), wall], 1).contiguous()
    return feat, (0.3 * torch.randn((rows, 2), generator=g, device="cuda")).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp_grad":
        mlp = pecc.MLP()
        mlp.set_params(_network(seed))
        feat, target = _samples(case["rows"], seed + 1)
        return dict(kind=kind, mlp=mlp, feat=feat, target=target)
    n, R = _sizes(case)
    s = dict(kind=kind, seed=seed)
    if kind in ("descend", "solve"):
        prec = PREC[case.get("prec", "mixed")]
        cfg = dict(BATCH)
        if case.get("prec") == "fp64" and case["num"] == 1:
            cfg = {}  # the plain method with the library's settings
        elif case["num"] > 256:
            cfg.update(block_threads=128, blocks_per_sm=4)  # the shape the autotuner picks for the batch
        s["ctx"] = pecc.Context(n, precision=prec, **cfg)
        s["R"] = np.ascontiguousarray(R)
        s["ctx"].set_radius(R)
        return s
    if kind == "adjust":
        s["ctx"] = pecc.Context(n, precision=pecc.FP32_POLISH64, max_iter=case["max_iter"])
        s["rounds"] = case["rounds"]
    elif kind == "feasible":
        s["ctx"] = pecc.Context(n, precision=pecc.FP64)
    elif kind == "propose":
        s["ctx"] = pecc.Context(n, precision=pecc.FP32)
        s["mlp"] = pecc.MLP()
        s["mlp"].set_params(_network(seed + 1))
    else:
        s["ctx"] = pecc.Context(n, precision=PREC[case["prec"]])
        s["eval"] = PREC[case["prec"]]
    s["R"] = torch.as_tensor(R, dtype=torch.float64, device="cuda")
    s["xy"] = _layout(case, n, R, seed, _jitter(case))
    s["ctx"].set_radius(s["R"])
    if kind == "energy_grad":
        s["ctx"].set_positions(s["xy"])
        s["ctx"].rebuild_neighbors(force=True, eval=s["eval"])
    return s


def run(state):
    kind = state["kind"]
    if kind == "mlp_grad":
        return state["mlp"].grad(state["feat"], state["target"])
    ctx = state["ctx"]
    if kind == "solve":
        return ctx.solve_host(state["R"], state["seed"])
    if kind == "descend":
        ctx.init_random(state["seed"])
        iters, status = ctx.descend()
        feasible, overlap = ctx.check_feasible()
        return ctx.get_positions(), ctx.get_energy(), iters, status, feasible, overlap
    if kind == "energy_grad":
        return ctx.energy_grad(eval=state["eval"])
    ctx.set_positions(state["xy"])
    if kind == "evaluate":
        ctx.rebuild_neighbors(force=True, eval=state["eval"])
        return ctx.energy_grad(eval=state["eval"])
    if kind == "feasible":
        return ctx.check_feasible()
    if kind == "adjust":
        R, iters, status = ctx.adjust_container(state["R"], rounds=state["rounds"])
        return R, iters, status, ctx.get_positions()
    feat = ctx.features()  # propose
    return feat, state["mlp"].forward(feat)


# ------------------------------------------------------------------------------------------ work
def work(case):
    kind = case["kind"]
    net = FEATURES * H + 2 * H * H + 2 * H  # multiply-adds of one row of the network
    if kind == "mlp_grad":
        params = net + 3 * H + 2
        return {"bytes": case["rows"] * 4 * (FEATURES + 2) + 8 * params, "flops": 6 * net * case["rows"]}
    num = case["num"]
    N = num * (case["n_lo"] + case["n_hi"]) / 2.0
    pair = 16.0 * DEGREE * N  # one visit of every list entry
    wide = case.get("prec") == "fp64"
    if kind == "energy_grad":
        return {"bytes": N * ((36 if wide else 20) + 4 * DEGREE) + 12 * num, "flops": pair}
    if kind == "evaluate":
        return {"bytes": N * (32 if wide else 24) + 16 * num, "flops": 3 * pair}
    if kind == "feasible":
        return {"bytes": 16 * N + 17 * num, "flops": 2 * pair}
    if kind == "adjust":
        # an iteration: an evaluation and a two-loop recursion over ten stored pairs
        its = case["rounds"] * case["max_iter"]
        return {"bytes": 32 * N + 24 * num, "flops": its * (pair + 10 * 16 * N)}
    if kind == "propose":
        return {"bytes": N * (16 + 4 * FEATURES + 8), "flops": 2 * net * N}
    # a descent: the sweeps it takes on average (small binary64 instances never end early), each an
    # evaluation, a trial and a quasi-Newton direction
    sweeps = 2000 if N < 300 else (600 if N / num < 16384 else 1100)
    m = 10 if (wide and num == 1) else BATCH["lbfgs_m"]
    return {"bytes": 16 * N + 33 * num, "flops": sweeps * (2 * pair + 24.0 * m * N)}


# ------------------------------------------------------------------- the same in 64 bits, in torch
def _cells(xy, inst, R, side):
    """Circles sorted by (instance, cell): cell of each circle, its first and last entry, the order."""
    nc = torch.ceil(2.0 * R.max() / side).long() + 3
    ij = torch.floor((xy + R[inst][:, None]) / side).long().clamp(-1, nc - 2) + 1
    key = (inst * nc + ij[:, 1]) * nc + ij[:, 0]
    order = torch.argsort(key, stable=True)
    count = torch.bincount(key, minlength=int(nc * nc * R.numel()) + 2 * int(nc) + 2)
    start = torch.cumsum(count, 0) - count
    return key, nc, start, count, order


def _pairs(xy, inst, R, reach, side):
    """Candidate neighbors: yields for every circle one other index (or -1) at a time."""
    key, nc, start, count, order = _cells(xy, inst, R, side)
    own = torch.arange(xy.shape[0], device=xy.device)
    for oy in range(-reach, reach + 1):
        for ox in range(-reach, reach + 1):
            cell = (key + oy * nc + ox).clamp(0, count.numel() - 1)
            c, s = count[cell], start[cell]
            for k in range(int(c.max())):
                j = order[(s + k).clamp_max(order.numel() - 1)]
                yield torch.where((k < c) & (j != own) & (inst[j] == inst), j, -1)


def _in_hand(case, seed):
    n, R = _sizes(case)
    xy = _layout(case, n, R, seed, _jitter(case))
    nt = torch.as_tensor(n, dtype=torch.int64, device="cuda")
    inst = torch.repeat_interleave(torch.arange(len(n), device="cuda"), nt)
    return xy, inst, torch.as_tensor(R, dtype=torch.float64, device="cuda")


def _exact_energy(case, seed):
    xy, inst, R = _in_hand(case, seed)
    own = torch.arange(xy.shape[0], device="cuda")
    g = torch.zeros_like(xy)
    e = torch.zeros_like(xy[:, 0])
    for j in _pairs(xy, inst, R, 1, 2.0):
        d = xy - xy[j.clamp_min(0)]
        l = torch.sqrt((d * d).sum(1))
        depth = torch.where(j >= 0, (2.0 - l).clamp_min(0.0), 0.0)
        g -= 2.0 * (depth / l.clamp_min(1e-300))[:, None] * d
        e += torch.where(j < own, depth * depth, 0.0)
    r = torch.sqrt((xy * xy).sum(1))
    wall = (r + 1.0 - R[inst]).clamp_min(0.0)
    g += 2.0 * (wall / r.clamp_min(1e-300))[:, None] * xy
    e += wall * wall
    return torch.zeros_like(R).index_add_(0, inst, e), g


def _exact_overlap(case, seed):
    xy, inst, R = _in_hand(case, seed)
    m = (torch.sqrt((xy * xy).sum(1)) + 1.0 - R[inst]).clamp_min(0.0)
    for j in _pairs(xy, inst, R, 1, 2.0):
        d = xy - xy[j.clamp_min(0)]
        m = torch.maximum(m, torch.where(j >= 0, 2.0 - torch.sqrt((d * d).sum(1)), 0.0))
    top = torch.zeros_like(R).scatter_reduce_(0, inst, m, "amax")
    return (top <= 1e-9).to(torch.uint8), top


def _weights(seed):
    p = _network(seed).double()
    out, o = [], 0
    for a, b in ((H, FEATURES), (H, H), (H, H), (2, H)):
        out.append((p[o:o + a * b].reshape(a, b), p[o + a * b:o + a * b + a]))
        o += a * b + a
    return out


def _forward(w, x):
    acts = [x]
    for i, (W, b) in enumerate(w):
        x = x @ W.T + b
        if i < 3:
            x = x.clamp_min(0.0)
        acts.append(x)
    return acts


def _exact_grad(case, seed):
    w = _weights(seed)
    feat, target = _samples(case["rows"], seed + 1)
    acts = _forward(w, feat.double())
    diff = acts[4] - target.double()
    loss = (diff * diff).sum() / case["rows"]
    dz = 2.0 * diff / case["rows"]
    grads = []
    for i in (3, 2, 1, 0):
        grads = [(dz.T @ acts[i]).reshape(-1), dz.sum(0)] + grads
        if i:
            dz = (dz @ w[i][0]) * (acts[i] > 0.0)
    return torch.cat(grads), loss.reshape(1)


def _exact_proposals(case, seed):
    xy, inst, R = _in_hand(case, seed)
    # the twelve nearest by (binary32 squared distance, index), as one integer key each
    none = torch.iinfo(torch.int64).max
    near = torch.full((xy.shape[0], KNN), none, dtype=torch.int64, device="cuda")
    x32 = xy.float()
    for j in _pairs(xy, inst, R, 2, L_CUT):
        d = x32[j.clamp_min(0)] - x32
        s = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]
        key = (s.view(torch.int32).long() << 32) | j
        key = torch.where((j >= 0) & (s < KNN_CUT * KNN_CUT), key, none)
        near = torch.sort(torch.cat([near, key[:, None]], 1), dim=1).values[:, :KNN].contiguous()
    who = near & 0xFFFFFFFF
    has = near != none
    r = torch.sqrt((xy * xy).sum(1))
    er = xy / r.clamp_min(1e-300)[:, None]
    d = torch.where(has[:, :, None], xy[torch.where(has, who, 0)] - xy[:, None, :], 0.0)
    u = d[:, :, 0] * er[:, :1] + d[:, :, 1] * er[:, 1:]
    v = d[:, :, 1] * er[:, :1] - d[:, :, 0] * er[:, 1:]
    wall = (R[inst] - r - 1.0).clamp_max(KNN_CUT)
    feat = torch.cat([torch.stack([u, v], 2).reshape(-1, 2 * KNN), wall[:, None]], 1)
    return feat, _forward(_weights(seed + 1), feat)[4]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("energy_grad", "evaluate"):
        return _exact_energy(case, seed)
    if kind == "feasible":
        return _exact_overlap(case, seed)
    if kind == "mlp_grad":
        return _exact_grad(case, seed)
    if kind == "propose":
        return _exact_proposals(case, seed)
    return None  # a descent or an adjustment: no value but the one its own rounding leads to
