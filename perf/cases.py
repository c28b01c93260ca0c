"""The calls whose speed matters, each through the package's public entry points.

A case names what a user's program does with the lattice sum u(m) = sum_n phi(m - n) f(n):
solve a point set once (plan + evaluation, or the one-shot call on host buffers), evaluate
a plan it keeps (one charge vector or several), solve a forest of small problems, apply a
boundary operator inside a Krylov iteration.  Points follow the recipes of
paper_1105_3505_gb300/workloads.py, drawn here on the GPU.

  prepare(case, seed)  inputs, and the plan where a program keeps one
  run(state)           one pass
  work(case)           bytes and operations that the pass cannot do without
  exact(case, seed)    the same sum in binary64 without the package: by FFT on the grid of
                       a box, by plain summation over a table of phi otherwise
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1105_3505_gb300 import lfmm

PRECISION = {"mixed": lfmm.LFMM_MIXED, "float-float": lfmm.LFMM_DF, "binary64": lfmm.LFMM_FP64}


def _case(call, points, n_src, n_tgt, side, precision="mixed", p=8, leaf=64, k=1, **more):
    """n_tgt = 0: the targets are the sources.  p, leaf: the options of the plan."""
    return {"call": call, "points": points, "n_src": n_src, "n_tgt": n_tgt, "side": side, "precision": precision,
            "p": p, "leaf": leaf, "k": k, **more}


def listed():
    def named(name, case):
        return {"name": name, **case}

    return [
        # the smallest configuration, one step of a program that solves small boxes one by
        # one: launches and round trips count
        named("solve_4k", _case("solve", "uniform", 4096, 0, 256)),
        # a served request at tolerance 1e-6 in the middle of the stream's sizes
        named("request_30k", _case("one_shot", "four_clusters", 31623, 7905, 712)),
        # a served request at tolerance 1e-10, with the options that the server gives it
        named("request_178k_1e10", _case("one_shot", "four_clusters", 177828, 44457, 1687, "float-float", 16, 192)),
        # the headline: a million sources and as many other targets, inputs on the device
        named("solve_1m", _case("solve", "uniform", 1 << 20, 1 << 20, 4096)),
        # the same from and to pinned host memory, odd sizes in a box that is no power of two
        named("solve_host", _case("host", "uniform", 786433, 524287, 3500)),
        # a plan that is kept while the loads change: odd sizes, fewer targets than sources
        named("eval_1m", _case("eval", "uniform", 1000003, 250001, 4000)),
        # eight loads on one plan
        named("multi_8", _case("multi", "uniform", 1 << 20, 1 << 20, 4096, k=8)),
        # clusters and segments in a box 65,536 wide: pruned tree, 14 levels
        named("clustered_4m", _case("solve", "clustered", 4194304, 0, 65536)),
        # 4,096 small problems in one forest
        named("forest_4096", _case("solve", "forest", 512, 0, 0, problems=4096, n_max=8192)),
        # one Krylov iteration of a Dirichlet problem on a disk: recorded graph, host vectors
        named("dirichlet_disk", _case("iteration", "circle", 1500, 0, 0, "float-float", 16)),
        # the accurate path on a plan that is kept
        named("eval_df_400k", _case("eval", "uniform", 400009, 400009, 2530, "float-float", 16, 128)),
        # the plain binary64 path that the others are compared with
        named("eval_fp64_100k", _case("eval", "uniform", 100003, 100003, 1265, "binary64", 16, 128)),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def side_for(n):
        return int(math.ceil(rng.uniform(2.5, 6.0) * math.sqrt(n)))

    kind = rng.choice(["solve", "one_shot", "one_shot_1e10", "host", "eval", "multi", "clustered", "forest", "iteration",
                       "eval_df", "eval_fp64"])
    if kind == "solve":
        n = size(1000, 1 << 20)
        return _case("solve", "uniform", n, rng.choice([0, size(max(1, n // 8), n)]), side_for(n))
    if kind in ("one_shot", "one_shot_1e10"):  # the served stream
        n = size(1000, 1000000 if kind == "one_shot" else 400000)
        points, side = rng.choice(["uniform", "four_clusters"]), int(math.ceil(4 * math.sqrt(n)))
        if kind == "one_shot":
            return _case("one_shot", points, n, n // 4, side)
        return _case("one_shot", points, n, n // 4, side, "float-float", 16, 192)
    if kind == "host":
        n = size(4096, 1 << 20)
        return _case("host", "uniform", n, size(n // 4, n), side_for(n))
    if kind == "eval":
        n = size(4096, 1 << 20)
        return _case("eval", "uniform", n, size(n // 4, n), side_for(n), p=rng.choice([6, 7, 8, 12, 16]),
                     leaf=rng.choice([32, 64, 64, 128]))
    if kind == "multi":
        n, k = size(4096, 1 << 19), rng.randint(2, 16)
        return _case("multi", "uniform", n, n, side_for(n), k=k)
    if kind == "clustered":
        return _case("solve", "clustered", size(100000, 4000000), 0, rng.choice([16384, 32768, 65536]))
    if kind == "forest":
        return _case("solve", "forest", size(100, 512), 0, 0, problems=size(48, 3000), n_max=size(1000, 8192),
                     p=rng.choice([7, 8]))
    if kind == "iteration":
        return _case("iteration", "circle", size(100, 3000), 0, 0, "float-float", 16)
    n = size(4096, 500000 if kind == "eval_df" else 150000)
    return _case("eval", "uniform", n, size(n // 4, n), side_for(n),
                 "float-float" if kind == "eval_df" else "binary64", rng.choice([12, 14, 16]), rng.choice([64, 128, 192]))


# ---- inputs ------------------------------------------------------------------------------


def _distinct(keys, n, gen):
    """n of the distinct values among `keys`, in random order."""
    keys = torch.unique(keys)
    return keys[torch.randperm(keys.shape[0], generator=gen, device=keys.device)[:n]]


def _xy(keys, width):
    return torch.stack([keys % width, keys // width], 1).to(torch.int32)


def _zero_sum(f):
    f = f - f.mean(-1, keepdim=True)
    f[..., -1] -= f.sum(-1)
    return f


def _forest_sizes(case):
    """Points of each problem, log-uniform between n_src and n_max."""
    u = np.random.default_rng(case["problems"]).uniform(math.log(case["n_src"]), math.log(case["n_max"]), case["problems"])
    return np.rint(np.exp(u)).astype(np.int64)


def _points(case, gen, dev):
    """(src, tgt, offsets): int32 points on the device; offsets of a forest's problems."""
    kind, n, m, side = case["points"], case["n_src"], case["n_tgt"], case["side"]

    def integers(hi, count):
        return torch.randint(0, hi, (count,), generator=gen, device=dev, dtype=torch.int64)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device=dev, dtype=torch.float64)

    def uniform(*shape):
        return torch.rand(*shape, generator=gen, device=dev, dtype=torch.float64)

    def in_box(count):
        return _xy(_distinct(integers(side * side, count + count // 3 + 64), count, gen), side)

    if kind == "uniform":
        src = in_box(n)
        return src, in_box(m) if m else src.clone(), None
    if kind == "four_clusters":  # standard deviation side / 16, targets anywhere in the box
        k = n + n // 2 + 64
        c = uniform(4, 2)[torch.arange(k, device=dev) % 4] * side
        q = (c + normal(k, 2) * (side / 16)).round().to(torch.int64) + side
        src = _xy(_distinct(q[:, 1] * (4 * side) + q[:, 0], n, gen), 4 * side) - side
        return src, torch.stack([integers(side, m), integers(side, m)], 1).to(torch.int32), None
    if kind == "clustered":  # 64 Gaussian clusters, and one point in a hundred on 16 segments
        k, on_lines = n + n // 3, n // 80
        c = uniform(64, 2)[torch.arange(k, device=dev) % 64] * side
        q = c + normal(k, 2) * 200.0
        seg = torch.arange(on_lines, device=dev) % 16
        angle, mid = uniform(16)[seg] * math.pi, (uniform(16, 2) * side)[seg]
        along = (uniform(on_lines) - 0.5) * 4000
        line = mid + along[:, None] * torch.stack([angle.cos(), angle.sin()], 1)
        q = torch.cat([q, line]).round().to(torch.int64) + 8192
        width = side + 16384
        src = _xy(_distinct(q[:, 1] * width + q[:, 0], n, gen), width) - 8192
        return src, src.clone(), None
    if kind == "forest":  # each in its own box of side 4 sqrt(N)
        sizes = torch.from_numpy(_forest_sizes(case)).to(dev)
        sides = (4 * sizes.double().sqrt()).ceil().to(torch.int64)
        drawn = sizes + sizes // 5 + 32
        pid = torch.repeat_interleave(torch.arange(sizes.shape[0], device=dev), drawn)
        cell = torch.minimum((uniform(pid.shape[0]) * (sides * sides)[pid]).to(torch.int64), (sides * sides)[pid] - 1)
        keys = torch.unique(pid * (1 << 20) + cell)
        keys = keys[torch.randperm(keys.shape[0], generator=gen, device=dev)]
        pid, order = torch.sort(keys >> 20, stable=True)
        start = torch.searchsorted(pid, torch.arange(sizes.shape[0], device=dev))
        keep = torch.arange(pid.shape[0], device=dev) - start[pid] < sizes[pid]
        pid, cell = pid[keep], (keys[order] & ((1 << 20) - 1))[keep]
        src = torch.stack([cell % sides[pid], cell // sides[pid]], 1).to(torch.int32)
        offsets = np.concatenate([[0], np.cumsum(_forest_sizes(case))]).astype(np.int64)
        return src, src.clone(), offsets
    raise ValueError(kind)


def _dipoles(radius, gen, dev):
    """The sources (boundary nodes of a disk, then the nodes next to them outside), the
    boundary nodes, and the charges of a random double-layer density."""
    r = torch.arange(-radius - 2, radius + 3, device=dev)
    inside = (r[:, None] ** 2 + r[None, :] ** 2) <= radius * radius
    steps = [(1, 0), (-1, 0), (0, 1), (0, -1)]
    out_of = [torch.roll(~inside, (-a, -b), (0, 1)) & inside for a, b in steps]
    edge = out_of[0] | out_of[1] | out_of[2] | out_of[3]
    q = torch.zeros(inside.shape, dtype=torch.float64, device=dev)
    q[edge] = torch.randn(int(edge.sum()), generator=gen, device=dev, dtype=torch.float64)
    charge = torch.zeros_like(q)
    outside = torch.zeros_like(inside)
    for (a, b), o in zip(steps, out_of):
        moved = torch.where(o, q, torch.zeros_like(q))
        charge += torch.roll(moved, (a, b), (0, 1)) - moved
        outside |= torch.roll(o, (a, b), (0, 1))
    gamma, outer = edge.nonzero(), outside.nonzero()
    at = torch.cat([gamma, outer])
    xy = (at - (radius + 2)).to(torch.int32)
    return xy, xy[: gamma.shape[0]].clone(), charge[at[:, 0], at[:, 1]]


def _inputs(case, seed):
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    if case["points"] == "circle":
        src, tgt, f = _dipoles(case["n_src"], gen, dev)
        return src, tgt, f, None
    src, tgt, offsets = _points(case, gen, dev)
    shape = (case["k"], src.shape[0]) if case["call"] == "multi" else (src.shape[0],)
    if case["points"] == "clustered":
        f = torch.rand(shape, generator=gen, device=dev, dtype=torch.float64) * 2 - 1
    else:
        f = torch.randn(shape, generator=gen, device=dev, dtype=torch.float64)
    if offsets is None:
        return src.contiguous(), tgt.contiguous(), _zero_sum(f), None
    sizes = torch.from_numpy(np.diff(offsets)).to(dev)
    pid = torch.repeat_interleave(torch.arange(sizes.shape[0], device=dev), sizes)
    for _ in range(2):  # the charges of each problem add up to nothing
        f -= (torch.zeros(sizes.shape[0], dtype=f.dtype, device=dev).index_add_(0, pid, f) / sizes)[pid]
    return src, tgt, f, offsets


def prepare(case, seed):
    src, tgt, f, offsets = _inputs(case, seed)
    opts = lfmm.make_opts(PRECISION[case["precision"]], case["p"], case["leaf"], graph=case["call"] == "iteration")
    state = {"call": case["call"], "src": src, "tgt": tgt, "f": f, "offsets": offsets, "opts": opts}
    if case["call"] in ("eval", "multi", "iteration"):
        if case["call"] == "iteration":  # a Krylov solver's vectors are numpy arrays
            src, tgt, state["f"] = (a.cpu().numpy() for a in (src, tgt, f))
        state["plan"] = lfmm.Plan(src, tgt, opts=opts)
    elif case["call"] == "host":
        for name in ("src", "tgt", "f"):
            state[name] = state[name].cpu().pin_memory()
        state["u"] = torch.empty(tgt.shape[0], dtype=torch.float64).pin_memory()
    return state


def run(state):
    call, src, tgt, f = (state[k] for k in ("call", "src", "tgt", "f"))
    if call == "solve":
        if state["offsets"] is not None:
            plan = lfmm.Forest(src, state["offsets"], tgt, state["offsets"], opts=state["opts"])
        else:
            plan = lfmm.Plan(src, tgt, opts=state["opts"])
        with plan:
            return plan.eval(f)
    if call == "one_shot":
        u = torch.empty(tgt.shape[0], dtype=torch.float64, device=f.device)
        lfmm.lfmm_solve(src, tgt, f, u, state["opts"])
        return u
    if call == "host":
        lfmm.lfmm_solve(src, tgt, f, state["u"], state["opts"])
        return state["u"]
    if call == "multi":
        return state["plan"].eval_multi(f)
    return state["plan"].eval(f)


# ---- what a pass cannot do without ---------------------------------------------------------


def work(case):
    """Each coordinate and charge read once, each result written once; multiply-adds (two
    operations) of the near field and of the expansions for leaves that are half full."""
    if case["points"] == "forest":
        n = m = int(_forest_sizes(case).sum())
    elif case["points"] == "circle":
        m = int(5.66 * case["n_src"])
        n = 2 * m
    else:
        n = case["n_src"]
        m = case["n_tgt"] or n
    k, P, full = case["k"], 4 * (case["p"] - 1), case["leaf"] / 2
    leaves = max(1.0, n / full)
    adds = m * min(float(n), 9 * full) + (n + m) * P + (leaves * 4 / 3) * (27 + 2) * P * P
    return {"bytes": 8 * (n + m) + 8 * k * (n + m), "flops": 2 * k * adds}


# ---- the sum in binary64 -------------------------------------------------------------------


def _phi_table(size, dev):
    """phi(i, j) for 0 <= i, j < size: an integral over one period where max(i, j) < 192,
    its expansion for large arguments beyond (error near 1e-14 there)."""
    x, y = (a.to(torch.float64) for a in torch.meshgrid(torch.arange(size, device=dev), torch.arange(size, device=dev),
                                                       indexing="ij"))
    r2 = (x * x + y * y).clamp_(min=1.0)
    x2, y2 = x * x / r2, y * y / r2
    c4 = x2 * x2 - 6 * x2 * y2 + y2 * y2  # cos 4t
    c8 = 2 * c4 * c4 - 1
    table = -(0.5 * r2.log() + np.euler_gamma + 1.5 * math.log(2)) / (2 * math.pi)
    table += c4 / (24 * math.pi * r2) + (18 * c4 + 25 * c8) / (480 * math.pi * r2 * r2)
    near = min(size, 192)
    node, weight = np.polynomial.legendre.leggauss(24)
    cuts = np.linspace(0.0, math.pi, 129)
    t = (cuts[:-1, None] + (cuts[1] - cuts[0]) * (node + 1) / 2).reshape(-1)
    w = np.tile(weight * (cuts[1] - cuts[0]) / 2, 128) / math.pi
    t, w = torch.from_numpy(t).to(dev), torch.from_numpy(w).to(dev)
    h = 2 * (t / 2).sin() ** 2  # 1 - cos t
    a = 2 * (h / 2).sqrt().asinh()  # cosh a = 1 + h
    w = w / (2 * a.sinh())
    at = torch.arange(near, device=dev, dtype=torch.float64)
    for i in range(near):  # exp(-a i) cos(j t) - 1 for j <= i, without cancellation near t = 0
        down = torch.expm1(-a * i)
        turn = -2 * (at[: i + 1, None] * (t / 2)).sin() ** 2
        row = ((down + turn + down * turn) * w).sum(1)
        table[i, : i + 1] = row
        table[: i + 1, i] = row
    return table


def _by_fft(src, tgt, f):
    lo = torch.minimum(src.amin(0), tgt.amin(0)).to(torch.int64)
    hi = torch.maximum(src.amax(0), tgt.amax(0)).to(torch.int64)
    size = int((hi - lo).max()) + 1
    n = 2 * size
    table = _phi_table(size + 1, src.device)
    mean = float(table.mean())  # phi without its mean: less to cancel
    i = torch.arange(n, device=src.device)
    i = torch.minimum(i, n - i)
    kernel = torch.fft.rfft2((table - mean)[i][:, i])
    s, t = src.to(torch.int64) - lo, tgt.to(torch.int64) - lo
    rows = []
    for row in f.reshape(-1, f.shape[-1]):
        grid = torch.zeros(n * n, dtype=torch.float64, device=src.device)
        grid.index_add_(0, s[:, 0] * n + s[:, 1], row)
        u = torch.fft.irfft2(torch.fft.rfft2(grid.reshape(n, n)) * kernel, s=(n, n))
        rows.append(u[t[:, 0], t[:, 1]] + mean * row.sum())
    return torch.stack(rows).reshape(f.shape[:-1] + (tgt.shape[0],))


def _by_sum(src, tgt, f, table):
    n = table.shape[0]
    flat, u = table.reshape(-1), torch.empty(tgt.shape[0], dtype=torch.float64, device=src.device)
    step = max(1, (1 << 28) // max(1, src.shape[0]))
    for i in range(0, tgt.shape[0], step):
        d = (tgt[i:i + step, None, 0] - src[None, :, 0]).abs_() * n
        d += (tgt[i:i + step, None, 1] - src[None, :, 1]).abs_()
        u[i:i + step] = flat[d] @ f
    return u


def exact(case, seed):
    src, tgt, f, offsets = _inputs(case, seed)
    if case["points"] == "clustered":
        return None  # neither a grid of the box nor the sum over all pairs is affordable
    if offsets is not None:
        table = _phi_table(int(src.max()) + 1, src.device)
        cuts = offsets.tolist()
        return torch.cat([_by_sum(src[a:b], tgt[a:b], f[a:b], table) for a, b in zip(cuts, cuts[1:])])
    if f.dim() == 1 and (case["precision"] != "mixed" or src.shape[0] <= 65536):
        both = torch.cat([src, tgt])
        u = _by_sum(src, tgt, f, _phi_table(int((both.amax(0) - both.amin(0)).max()) + 1, src.device))
        return u.cpu().numpy() if case["call"] == "iteration" else u
    return _by_fft(src, tgt, f)
