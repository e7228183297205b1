"""Timed workloads of the box FMM: what a program that uses this package has it do.

Trees of the three kinds the package builds (uniform, refined to a tolerance, refined to a leaf
count), operators of every size it supports (k = 4..16, p up to 60), both arithmetics (FP64 and
split BF16) and every way of calling a solve (one call, many right-hand sides, a replayed graph, a
batch), besides the tree build and the two kinds of evaluation away from the leaf nodes. A program
keeps its tree, operators and buffers and solves for one f after another, so those are the state;
f (and points) come from the seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1610_00823_gb300 as v
from paper_1610_00823_gb300 import api

GAUSS_SUM, KINKED = 1, 2
CFG2 = dict(tree="tail", n_src=20, s_min=1e-3, s_max=1e-1, spread=0.45, tol=1e-10, max_depth=16, src_seed=20161005)


def listed():
    return [
        # the smallest solve of the repository: 64 leaves, a launch-bound call in plain FP64
        dict(name="solve_fp64_uniform_d3", kind="solve", form="fp64", call="direct", nrhs=1, tree="uniform", depth=3,
             n_src=3, s_min=0.1, s_max=0.1, spread=0.3, src_seed=20161004, k=8, p=20),
        # the same tree in the split form, replayed as a graph (a time stepper on a small grid)
        dict(name="graph_mixed_uniform_d3", kind="solve", form="mixed", call="graph", nrhs=1, tree="uniform", depth=3,
             n_src=3, s_min=0.1, s_max=0.1, spread=0.3, src_seed=20161004, k=8, p=20),
        # 64 right-hand sides that share this tree (many densities on one grid)
        dict(name="rhs64_mixed_uniform_d3", kind="solve", form="mixed", call="direct", nrhs=64, tree="uniform",
             depth=3, n_src=3, s_min=0.1, s_max=0.1, spread=0.3, src_seed=20161004, k=8, p=20),
        # the benchmark's default workload: 20 Gaussians refined to 1e-10, tuned and replayed
        dict(name="graph_mixed_gauss20", kind="solve", form="mixed", call="graph", nrhs=1, k=16, p=40, **CFG2),
        # the same in plain FP64: the accuracy reference a user checks the split form against
        dict(name="solve_fp64_gauss20", kind="solve", form="fp64", call="direct", nrhs=1, k=16, p=40, **CFG2),
        # an odd operator size on a leaf-count tree (k not a multiple of 4, k*k not of 32)
        dict(name="solve_mixed_leaves_k11", kind="solve", form="mixed", call="direct", nrhs=1, tree="leaves",
             n_leaves=2500, n_src=3, s_min=0.1, s_max=0.1, spread=0.3, src_seed=20161013, k=11, p=27),
        # the FP64 form with its plane-wave M2L on a uniform grid of 4,096 leaves (a dense smooth density)
        dict(name="solve_fp64_pw_uniform_d6", kind="solve", form="fp64_pw", call="direct", nrhs=1, tree="uniform",
             depth=6, n_src=3, s_min=0.1, s_max=0.1, spread=0.3, src_seed=20161004, k=16, p=40),
        # the largest: a source with a kink on a curve, 200,104 leaves and 51 million targets
        dict(name="solve_mixed_kinked", kind="solve", form="mixed", call="direct", nrhs=1, tree="kinked", tol=1e-10,
             max_depth=14, src_seed=20161006, k=16, p=40),
        # a dozen uneven problems in one batch (leaf counts 100 to 5e4, k = 8 and 16)
        dict(name="batch_mixed_12", kind="batch", form="mixed", members=12, lo=100, hi=50000, src_seed=20161003),
        # the potential at points that are not nodes, from the expansions a solve left
        dict(name="points_gauss20", kind="points", n_points=1000, form="fp64", k=16, p=40, **CFG2),
        # interpolated u, u_x, u_y at a million points (a plot, a particle push)
        dict(name="interp_gauss20", kind="interp", n_points=1 << 20, fields=3, k=16, p=40, **CFG2),
        # the tree, its lists and the leaf values of a new density
        dict(name="tree_gauss20", kind="tree", k=16, **CFG2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    k = rng.randint(4, 16)
    p = min(60, max(8, int(round(2.5 * k + rng.uniform(-4, 4)))))
    seed = rng.randint(1, 10 ** 6)
    kind = rng.choices(["solve", "points", "interp", "tree", "batch"], [10, 1, 2, 2, 1])[0]
    if kind == "batch":
        form = rng.choice(["fp64", "mixed"])
        return dict(kind="batch", form=form, members=rng.randint(3, 12), lo=rng.randint(50, 200),
                    hi=_log(rng, 500, 20000 if form == "mixed" else 3000), src_seed=seed)
    t = rng.choice(["uniform", "leaves", "tail"]) if kind != "tree" else rng.choice(["leaves", "tail"])
    c = dict(kind=kind, tree=t, n_src=rng.randint(2, 20), src_seed=seed, k=k)
    if t == "uniform":
        c.update(depth=rng.randint(1, 6), s_min=0.1, s_max=0.1, spread=0.3)
    elif t == "leaves":
        c.update(n_leaves=_log(rng, 30, 20000), s_min=0.05, s_max=0.1, spread=0.3)
    else:
        s = math.exp(rng.uniform(math.log(2e-3), math.log(3e-2)))
        # a k-point interpolant reaches about 10^(1 - 0.7 k) on boxes of a few widths
        c.update(s_min=s, s_max=0.1, spread=0.45, tol=max(1e-10, 10.0 ** (1.0 - 0.7 * k)), max_depth=12)
    if kind == "tree":
        return c
    c["p"] = p
    if kind == "interp":
        c.update(n_points=_log(rng, 1000, 1 << 21), fields=rng.randint(1, 8))
        return c
    c["form"] = rng.choice(["fp64", "fp64_pw", "mixed", "mixed"])
    if kind == "points":
        c["n_points"] = _log(rng, 10, 1000)
        return c
    small = t == "uniform" and c["depth"] <= 3
    c.update(call=rng.choice(["direct", "graph"]), nrhs=rng.randint(1, 64) if small else rng.choice([1, 1, 2]))
    return c


# ---------------------------------------------------------------- what a program keeps
@functools.lru_cache(maxsize=None)
def _ops(k, p, form):
    ops = v.ops_create(k, p, v.MIXED if form == "mixed" else v.FP64)
    if form == "fp64_pw":
        ops.set_m2l(v.M2L_PLANEWAVE)
    return ops


def _source(case, amp_seed=None):
    """The case's source; another amp_seed keeps its places and widths and draws other amplitudes."""
    rng = np.random.default_rng(case["src_seed"])
    amp = rng if amp_seed is None else np.random.default_rng([case["src_seed"], amp_seed])
    if case.get("tree") == "kinked":
        a, c = rng.uniform(0.0, 0.03, 7), rng.uniform(0.0, 2.0 * math.pi, 7)
        rows = [np.column_stack([rng.uniform(-0.6, 0.6, (5, 2)), np.full(5, 0.2), amp.normal(0.0, 1.0, 5)])
                for _ in range(2)]
        return KINKED, 5, np.concatenate([a, c, rows[0].ravel(), rows[1].ravel()])
    n = case["n_src"]
    xy = rng.uniform(-case["spread"], case["spread"], (n, 2))
    s = np.exp(rng.uniform(math.log(case["s_min"]), math.log(case["s_max"]) + 1e-12, n))
    a = amp.uniform(0.3, 1.0, n) * np.where(amp.uniform(size=n) < 0.5, -1.0, 1.0)
    return GAUSS_SUM, n, np.column_stack([xy, s, a]).ravel()


def _new_source(case, seed):
    """The case's source at another strength: a new density whose tree has the same size."""
    kind, n, prm = _source(case)
    rows = prm.reshape(-1, 4).copy()
    rows[:, 3] *= np.random.default_rng(int(seed)).uniform(0.5, 2.0)
    return kind, n, rows.ravel()


def _build(case, source):
    w = 2.0 if case["tree"] == "kinked" else 1.0
    if case["tree"] == "uniform":
        return v.tree_build_uniform(0.0, 0.0, w, case["k"], case["depth"])
    if case["tree"] == "leaves":
        return v.tree_build_leaves(0.0, 0.0, w, case["k"], source, case["n_leaves"])
    return v.tree_build(0.0, 0.0, w, case["k"], source, case["tol"], case["max_depth"])


@functools.lru_cache(maxsize=3)
def _plan_of(items):
    case = dict(items)
    return _build(case, _source(case))


def _plan(case):
    """The case's tree: built once, as a program that solves for one f after another does."""
    return _plan_of(tuple(sorted((a, b) for a, b in case.items() if a not in ("name", "call", "form", "kind", "p"))))


def _f(case, tree, seed, nrhs=1):
    return torch.stack([v.source_sample(tree, _source(case, 1000 * seed + r)) for r in range(nrhs)]).reshape(-1)


@functools.lru_cache(maxsize=2)
def _members(src_seed, members, lo, hi):
    rng = np.random.default_rng(src_seed)
    specs = []
    for i in range(members):
        k = 8 if rng.uniform() < 0.5 else 16
        c = dict(tree="leaves", n_src=3, s_min=0.1, s_max=0.1, spread=0.3, src_seed=src_seed + i, k=k)
        # leaf counts spread over the logarithm of the range, from its lower to its upper end
        c["n_leaves"] = int(round(lo * (hi / lo) ** (i / max(1, members - 1))))
        specs.append(c)
    trees = v.tree_build_many([dict(cx=0.0, cy=0.0, width=1.0, k=c["k"], source=_source(c), max_depth=16,
                                    n_leaves=c["n_leaves"]) for c in specs])
    return list(zip(specs, trees))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "tree":
        return dict(case=case, source=_new_source(case, seed))
    if kind == "batch":
        items = []
        for c, tree in _members(case["src_seed"], case["members"], case["lo"], case["hi"]):
            ops = _ops(c["k"], 20 if c["k"] == 8 else 40, case["form"])
            f = _f(c, tree, seed)
            items.append((tree, ops, f, tuple(torch.empty_like(f) for _ in range(3)), v.workspace(tree, ops)))
        return dict(case=case, items=items, batch=api.Batch(8))
    tree = _plan(case)
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    half = 1.0 if case["tree"] == "kinked" else 0.5
    if kind == "interp":
        n = tree.n_leaves * case["k"] ** 2
        fields = [_f(case, tree, seed + 17 * q) for q in range(case["fields"])]
        xy = (torch.rand(2, case["n_points"], generator=g, dtype=torch.float64, device="cuda") - 0.5) * 2 * half
        assert fields[0].numel() == n
        return dict(case=case, tree=tree, fields=fields, x=xy[0].contiguous(), y=xy[1].contiguous())
    ops = _ops(case["k"], case["p"], case["form"])
    nrhs = case.get("nrhs", 1)
    f = _f(case, tree, seed, nrhs)
    out = tuple(torch.empty_like(f) for _ in range(3))
    ws = v.workspace(tree, ops, nrhs)
    s = dict(case=case, tree=tree, ops=ops, f=f, out=out, ws=ws)
    if kind == "points":
        v.volume_potential(tree, ops, f, out, ws)
        xy = (torch.rand(2, case["n_points"], generator=g, dtype=torch.float64, device="cuda") - 0.5) * 2 * half
        s.update(x=xy[0].contiguous(), y=xy[1].contiguous())
    elif case["call"] == "graph":
        side = torch.cuda.Stream()
        torch.cuda.synchronize()
        api.tune(tree, ops, f, out, ws, side)
        s["graph"] = api.SolveGraph(tree, ops, f, out, ws, side)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "tree":
        t = _build(case, s["source"])
        return [*t.export_boxes(), *t.leaf_nodes(), v.source_sample(t, s["source"])]
    if kind == "batch":
        s["batch"].potential(s["items"])
        return [o for it in s["items"] for o in it[3]]
    if kind == "interp":
        return v.leaf_interpolate(s["tree"], s["fields"], s["x"], s["y"])
    if kind == "points":
        return list(v.evaluate_points(s["tree"], s["ops"], s["f"], s["ws"], s["x"], s["y"]))
    if "graph" in s:
        s["graph"].launch()
        return list(s["out"])
    return list(v.volume_potential(s["tree"], s["ops"], s["f"], s["out"], s["ws"]))


def work(case):
    """f read once and the results written once. Products: per pair of adjacent leaves a k^2 x 3 k^2
    table apply, of which the reflections of the square leave a quarter to do."""
    kind = case["kind"]
    if kind == "batch":
        ms = _members(case["src_seed"], case["members"], case["lo"], case["hi"])
        return {"bytes": float(sum(32 * t.n_leaves * c["k"] ** 2 for c, t in ms)),
                "flops": float(sum(1.5 * c["k"] ** 4 * t.list_len[0] for c, t in ms))}
    tree = _build(case, _new_source(case, 0)) if kind == "tree" else _plan(case)
    kk = case["k"] ** 2
    n = tree.n_leaves * kk
    if kind == "tree":  # the coefficients of every box, its numbers, its nodes and values
        return {"bytes": 12.0 * tree.n_boxes + 24.0 * n, "flops": 4.0 * tree.n_boxes * case["k"] ** 3}
    if kind == "interp":  # a tensor sum of k^2 terms per point and field
        return {"bytes": 8.0 * (case["n_points"] * (2 + case["fields"]) + case["fields"] * n),
                "flops": 2.0 * case["n_points"] * case["fields"] * kk}
    if kind == "points":  # a weight per value of every adjacent leaf, for three results
        near = tree.list_len[0] / tree.n_leaves
        return {"bytes": 40.0 * case["n_points"] + 8.0 * n, "flops": 6.0 * kk * near * case["n_points"]}
    return {"bytes": 32.0 * n * case["nrhs"], "flops": 1.5 * kk * kk * tree.list_len[0] * case["nrhs"]}


# ---------------------------------------------------------------- the same numbers in plain 64-bit torch
D = torch.float64


def _gl(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.tensor(0.5 * (x + 1), dtype=D, device="cuda"), torch.tensor(0.5 * w, dtype=D, device="cuda")


def _nodes(k):
    return -torch.cos(math.pi * (2 * torch.arange(k, dtype=D, device="cuda") + 1) / (2 * k)) / 2


def _cheb(x, k):
    """T_0..T_{k-1} at 2x, last axis."""
    t = [torch.ones_like(x), 2 * x]
    while len(t) < k:
        t.append(4 * x * t[-1] - t[-2])
    return torch.stack(t[:k], -1)


def _coeffs(f, k):
    """Chebyshev coefficients [..., m (x), n (y)] of values [..., j (y), i (x)]."""
    C = _cheb(_nodes(k), k).T * (2.0 / k)
    C[0] /= 2
    return torch.einsum("mi,nj,...ji->...mn", C, C, f)


def _moments(t, k):
    """int over the unit box of (log|t-y|, (t-y)/|t-y|^2) T_m T_n dy, t [n, 2] anywhere: [n, 3, k, k].

    Triangles with apex at the box's point nearest t, two per edge, graded in both directions."""
    q, w = _gl(96)
    s, ws = q ** 6, 6 * q ** 5 * w
    out = []
    for tc in t.split(48):
        acc = torch.zeros(tc.shape[0], 3, k, k, dtype=D, device="cuda")
        c = tc.clamp(-0.5, 0.5)
        for axis in (0, 1):
            for side in (-0.5, 0.5):
                foot = c.clone()
                foot[:, axis] = side
                for end in (-0.5, 0.5):
                    e1 = foot - c  # across, then along the edge
                    along = end - c[:, 1 - axis]
                    area = (e1[:, axis] * along).abs()
                    across = s[:, None] * torch.ones_like(s)[None, :]
                    d = [None, None]
                    d[axis] = e1[:, axis, None, None] * across
                    d[1 - axis] = along[:, None, None] * (s[:, None] * s[None, :])
                    wt = area[:, None, None] * (s * ws)[:, None] * ws[None, :]
                    gap = tc - c
                    rx, ry = gap[:, 0, None, None] - d[0], gap[:, 1, None, None] - d[1]
                    r2 = rx * rx + ry * ry
                    ok = (wt > 0) & (r2 > 0)
                    r2 = torch.where(ok, r2, torch.ones_like(r2))
                    n = tc.shape[0]
                    tx = _cheb((c[:, 0, None, None] + d[0]).reshape(n, -1), k)
                    ty = _cheb((c[:, 1, None, None] + d[1]).reshape(n, -1), k)
                    for j, kern in enumerate((0.5 * torch.log(r2), rx / r2, ry / r2)):
                        g = torch.where(ok, kern * wt, torch.zeros_like(wt)).reshape(n, -1, 1)
                        acc[:, j] += torch.bmm((tx * g).transpose(1, 2), ty)
        out.append(acc)
    return torch.cat(out)


def _far(tz, cz, h, a, skip):
    """Phi and Phi' at tz [n] from multipoles a [ns, P] about cz, pairs in skip [n, ns] left out."""
    phi = torch.zeros_like(tz)
    dphi = torch.zeros_like(tz)
    step = max(1, (1 << 22) // max(1, len(cz)))
    P = a.shape[1]
    for i in range(0, len(tz), step):
        z = (tz[i:i + step, None] - cz[None]) / h[None]
        no = skip[i:i + step]
        z = torch.where(no, torch.full_like(z, 1e3), z)
        zi = 1 / z
        s = torch.zeros_like(z)
        g = torch.zeros_like(z)
        for n in range(P - 1, 0, -1):
            s = (s + a[None, :, n] * (-1.0 / n)) * zi
            g = (g + a[None, :, n]) * zi
        s = s + a[None, :, 0] * (torch.log(z.abs()) + torch.log(h)[None])
        g = (g + a[None, :, 0]) * zi / h[None]
        phi[i:i + step] = torch.where(no, torch.zeros_like(s), s).sum(1)
        dphi[i:i + step] = torch.where(no, torch.zeros_like(g), g).sum(1)
    return phi, dphi


def _mid(t, src, cx, cy, h, C, k):
    """Phi and Phi' at t [n, 2] of the source leaves src [n] (not adjacent) by a product rule."""
    q, w = _gl(28)
    y = q - 0.5
    B = _cheb(y, k)
    W2 = w[:, None] * w[None, :]
    phi, dphi = [], []
    for i in range(0, len(t), 20000):
        sl = src[i:i + 20000]
        g = torch.einsum("am,bn,pmn->pab", B, B, C[sl]) * W2 * (h[sl] ** 2)[:, None, None]
        hs = h[sl][:, None, None]
        rx = (t[i:i + 20000, 0] - cx[sl])[:, None, None] - hs * y[None, :, None]
        ry = (t[i:i + 20000, 1] - cy[sl])[:, None, None] - hs * y[None, None, :]
        r2 = rx * rx + ry * ry
        phi.append((0.5 * torch.log(r2) * g).sum((1, 2)))
        dphi.append(torch.complex((rx / r2 * g).sum((1, 2)), -(ry / r2 * g).sum((1, 2))))
    return torch.cat(phi), torch.cat(dphi)


def _leaf_boxes(tree, width):
    lv, ix, iy = tree.export_boxes()
    have = set(zip(lv.tolist(), ix.tolist(), iy.tolist()))
    leaf = np.array([(l + 1, 2 * x, 2 * y) not in have for l, x, y in zip(lv.tolist(), ix.tolist(), iy.tolist())])
    lv, ix, iy = lv[leaf], ix[leaf], iy[leaf]
    h = width / 2.0 ** lv
    return lv, ix, iy, h


def _potential_of(tree, width, k, f, points=None):
    """V f~ and its gradient, f [R, leaves, k, k], at every leaf node or at points [n, 2]."""
    lv, ix, iy, hn = _leaf_boxes(tree, width)
    h = torch.tensor(hn, device="cuda")
    cx = torch.tensor(-width / 2 + hn * (ix + 0.5), device="cuda")
    cy = torch.tensor(-width / 2 + hn * (iy + 0.5), device="cuda")
    cz = torch.complex(cx, cy)
    C = _coeffs(f, k)
    q, w = _gl(60)
    y = q - 0.5
    B = _cheb(y, k)
    z = torch.complex(y[:, None].expand(60, 60), y[None].expand(60, 60))
    g = torch.einsum("am,bn,rsmn->rsab", B, B, C) * (w[:, None] * w[None, :]) * (h ** 2)[None, :, None, None]
    a, zp = [], torch.ones_like(z)
    for n in range(61):
        a.append((g * zp).sum((2, 3)))
        zp = zp * z
    a = torch.stack(a, -1)  # [R, leaves, 61]
    one = _cheb(y, k).T @ w
    mass = torch.einsum("m,n,rsmn->rs", one, one, C)
    R = f.shape[0]
    if points is None:
        xn = _nodes(k)
        tx = (cx[:, None, None] + h[:, None, None] * xn[None, None, :]).expand(-1, k, k).reshape(-1)
        ty = (cy[:, None, None] + h[:, None, None] * xn[None, :, None]).expand(-1, k, k).reshape(-1)
        t = torch.stack([tx, ty], 1)
    else:
        t = points
    tz = torch.complex(t[:, 0], t[:, 1])
    gap = torch.maximum((t[:, 0, None] - cx[None]).abs(), (t[:, 1, None] - cy[None]).abs()) / h[None] - 0.5
    close = gap < (0.49 if points is not None else 2.0)
    if points is None:  # adjacent leaves, by their integer corners at the finest level
        m = int(lv.max())
        s = torch.tensor(1 << (m - lv), device="cuda")
        X, Y = torch.tensor(ix, device="cuda") * s, torch.tensor(iy, device="cuda") * s
        adj = (X[:, None] <= X[None] + s[None]) & (X[None] <= X[:, None] + s[:, None])
        adj &= (Y[:, None] <= Y[None] + s[None]) & (Y[None] <= Y[:, None] + s[:, None])
        close = adj.repeat_interleave(k * k, 0)
    mid = ~close & ((tz[:, None] - cz[None]).abs() < 1.45 * h[None])
    skip = close | mid
    ti, si = torch.nonzero(mid, as_tuple=True)
    phi = torch.zeros(R, len(t), dtype=D, device="cuda")
    dphi = torch.zeros(R, len(t), dtype=torch.complex128, device="cuda")
    for r in range(R):
        p0, d0 = _far(tz, cz, h, a[r], skip)
        phi[r], dphi[r] = p0.real, d0
        if len(ti):
            p1, d1 = _mid(t[ti], si, cx, cy, h, C[r], k)
            phi[r].index_add_(0, ti, p1)
            dphi[r].index_add_(0, ti, d1)
    if points is None:  # one table per kind of neighbour
        pt, ps = torch.nonzero(adj, as_tuple=True)
        key = torch.stack([((cx[pt] - cx[ps]) / h[ps] * 8).round(), ((cy[pt] - cy[ps]) / h[ps] * 8).round(),
                           (h[pt] / h[ps] * 2).round()], 1)
        kinds, which = torch.unique(key, dim=0, return_inverse=True)
        for c in range(len(kinds)):
            ox, oy, rel = float(kinds[c, 0]) / 8, float(kinds[c, 1]) / 8, float(kinds[c, 2]) / 2
            loc = torch.stack([(ox + rel * xn)[None, :].expand(k, k).reshape(-1),
                               (oy + rel * xn)[:, None].expand(k, k).reshape(-1)], 1)
            M = _moments(loc, k)
            tt, ss = pt[which == c], ps[which == c]
            v3 = torch.einsum("tqmn,rpmn->qrpt", M, C[:, ss])
            at = (tt[:, None] * k * k + torch.arange(k * k, device="cuda")[None]).reshape(-1)
            pot = (v3[0] + (torch.log(h[ss]) * mass[:, ss])[..., None]) * (h[ss] ** 2)[None, :, None]
            phi.index_add_(1, at, pot.reshape(R, -1))
            dphi.index_add_(1, at, (torch.complex(v3[1], -v3[2]) * h[ss][None, :, None]).reshape(R, -1))
    else:
        pt, ps = torch.nonzero(close, as_tuple=True)
        for i in range(0, len(pt), 4096):
            tt, ss = pt[i:i + 4096], ps[i:i + 4096]
            M = _moments(torch.stack([(t[tt, 0] - cx[ss]) / h[ss], (t[tt, 1] - cy[ss]) / h[ss]], 1), k)
            v3 = torch.einsum("pqmn,rpmn->qrp", M, C[:, ss])
            phi.index_add_(1, tt, (v3[0] + torch.log(h[ss]) * mass[:, ss]) * h[ss] ** 2)
            dphi.index_add_(1, tt, torch.complex(v3[1], -v3[2]) * h[ss])
    c = -1 / (2 * math.pi)
    return [(c * phi).reshape(-1), (c * dphi.real).reshape(-1), (-c * dphi.imag).reshape(-1)]


def _interp_of(tree, width, k, fields, x, y):
    lv, ix, iy, hn = _leaf_boxes(tree, width)
    m = int(lv.max())
    X = ((x + width / 2) / width * 2 ** m).floor().clamp(0, 2 ** m - 1).to(torch.int64)
    Y = ((y + width / 2) / width * 2 ** m).floor().clamp(0, 2 ** m - 1).to(torch.int64)
    leaf = torch.full_like(X, -1)
    for l in range(m + 1):
        ids = np.nonzero(lv == l)[0]
        if len(ids) == 0:
            continue
        code = torch.tensor(ix[ids].astype(np.int64) << l | iy[ids], device="cuda")
        code, order = code.sort()
        want = (X >> (m - l)) << l | (Y >> (m - l))
        at = torch.searchsorted(code, want).clamp(max=len(ids) - 1)
        leaf = torch.where(code[at] == want, torch.tensor(ids, device="cuda")[order[at]], leaf)
    h = torch.tensor(hn, device="cuda")[leaf]
    px = (x + width / 2 - h * torch.tensor(ix, device="cuda")[leaf]) / h - 0.5
    py = (y + width / 2 - h * torch.tensor(iy, device="cuda")[leaf]) / h - 0.5
    Tx, Ty = _cheb(px, k), _cheb(py, k)
    out = []
    for f in fields:
        C = _coeffs(f.reshape(-1, k, k), k)
        out.append(torch.cat([torch.einsum("pm,pn,pmn->p", Tx[i:i + 65536], Ty[i:i + 65536], C[leaf[i:i + 65536]])
                              for i in range(0, len(x), 65536)]))
    return out


def exact(case, seed):
    """The leaf interpolants' potential by direct sums: tables and points by graded quadrature,
    other leaves by order-60 multipoles. None where that would take long."""
    kind = case["kind"]
    if kind == "batch":
        return None
    width = 2.0 if case["tree"] == "kinked" else 1.0
    k = case["k"]
    if kind == "tree":
        src = _new_source(case, seed)
        t = _build(case, src)
        lv, ix, iy, h = _leaf_boxes(t, width)
        xn = _nodes(k).cpu().numpy()
        x = (-width / 2 + h * (ix + 0.5))[:, None, None] + h[:, None, None] * xn[None, None, :] + np.zeros((1, k, 1))
        y = (-width / 2 + h * (iy + 0.5))[:, None, None] + h[:, None, None] * xn[None, :, None] + np.zeros((1, 1, k))
        f = sum(a * np.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2 * s * s)) for cx, cy, s, a in src[2].reshape(-1, 4))
        return [None, None, None, x.reshape(-1), y.reshape(-1), f.reshape(-1)]
    tree = _plan(case)
    n = tree.n_leaves
    if kind == "interp":
        s = prepare(case, seed)
        return _interp_of(tree, width, k, s["fields"], s["x"], s["y"])
    if kind == "points":
        if n > 3000 or case["n_points"] > 2000:
            return None
        s = prepare(case, seed)
        return _potential_of(tree, width, k, s["f"].reshape(1, n, k, k), torch.stack([s["x"], s["y"]], 1))
    nrhs = case["nrhs"]
    if n > 4000 or float(n) * n * k * k * nrhs > 1.2e9:
        return None
    f = _f(case, tree, seed, nrhs)
    return _potential_of(tree, width, k, f.reshape(nrhs, n, k, k))
