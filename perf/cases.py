"""Performance cases of the sparse stress layout library.

Each case is one call chain a program makes through the public entry points of
``paper_1608_08909_gb300``, at the sizes of the repository's own workloads
(``inputs.workload``, the weighted, k-means and batching sections of
``bench.py``).  ``kind`` names the chain, the rest are sizes:

* ``layout``   -- the whole of Algorithm 1 on a small mesh (``layout``)
* ``prepare``  -- Algorithm 1 lines 1-4 from a host edge list (``prepare``)
* ``sweep``    -- Jacobi sweeps of Eq. 4 from a given layout (``ssm_iterate``)
* ``stress``   -- sampled (or exhaustive) full stress (``ssm_stress``)
* ``kmeans``   -- k-means sp pivots from max/min pivots (``ssm_kmeans_pivots``)
* ``wprepare`` -- weighted graph, pivots, distances and counts
* ``wlayout``  -- weighted PivotMDS, then weighted sweeps from a given layout
* ``wstress``  -- sampled stress over weighted distances
* ``batch``    -- many small graphs: batched preparation and sweeps

Layouts that sweeps start from are a seeded projection of the squared pivot
distances (what PivotMDS does with its eigenvectors) with a jitter of a third
of an edge length, formed here with torch: a start inside the value range the
sweep meets, with no coincident nodes, the same for every version of the code.
The number of sweeps in a case is below the 100 of a full layout because the
Jacobi iteration amplifies rounding differences with every step; outputs are
compared number by number.
"""
import math

import numpy as np
import torch

import paper_1608_08909_gb300 as ssm
from paper_1608_08909_gb300 import inputs

DEV = "cuda"


def listed():
    return [
        # the smallest call: one small mesh laid out from start to end (the 32 x 32 grid workload)
        {"name": "layout_grid32", "kind": "layout", "rows": 32, "cols": 32, "k": 50, "iters": 200},
        # preparation of a heavy-tailed network (the default benchmark workload)
        {"name": "prepare_ba1m", "kind": "prepare", "family": "ba", "n": 1 << 20, "k": 200},
        # preparation of a large-diameter mesh or road-like graph
        {"name": "prepare_rgg256k", "kind": "prepare", "family": "rgg", "n": 262144, "k": 200},
        # the sweep of the default benchmark workload
        {"name": "sweep_ba1m", "kind": "sweep", "family": "ba", "n": 1 << 20, "k": 200, "precision": 32, "iters": 10},
        # the sweep of the large-diameter workload
        {"name": "sweep_rgg256k", "kind": "sweep", "family": "rgg", "n": 262144, "k": 200, "precision": 32, "iters": 10},
        # the double-precision option, at the size of the precision study
        {"name": "sweep_ba64k_f64", "kind": "sweep", "family": "ba", "n": 65536, "k": 200, "precision": 64, "iters": 3},
        # evaluation of a layout on 1024 x 1024 sampled pairs
        {"name": "stress_rgg256k", "kind": "stress", "family": "rgg", "n": 262144, "k": 50, "sources": 1024, "targets": 1024},
        # the paper's recommended sampler on the benchmark workload (at most 50 passes)
        {"name": "kmeans_ba1m", "kind": "kmeans", "family": "ba", "n": 1 << 20, "k": 200, "passes": 50},
        # a weighted road-like graph: pivots, distances and counts
        {"name": "wprepare_rgg256k", "kind": "wprepare", "n": 262144, "k": 200},
        # its initial layout, and sweeps
        {"name": "wlayout_rgg256k", "kind": "wlayout", "n": 262144, "k": 200, "iters": 10},
        # its evaluation
        {"name": "wstress_rgg256k", "kind": "wstress", "n": 262144, "k": 50, "sources": 1024, "targets": 1024},
        # many small graphs at once (the batching workload's mix, an eighth of its count)
        {"name": "batch_512", "kind": "batch", "count": 512, "n_min": 64, "n_max": 8192, "iters": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layout", "prepare", "prepare", "sweep", "sweep", "stress", "kmeans", "wprepare", "wlayout", "wstress", "batch"])
    family = rng.choice(["ba", "rgg"])
    n = _log(rng, 4096, (1 << 20) if family == "ba" else 262144)
    k = _log(rng, 50, 200)
    if kind == "layout":
        return {"kind": kind, "rows": rng.randint(20, 64), "cols": rng.randint(20, 64), "k": rng.randint(20, 100), "iters": rng.randint(20, 200)}
    if kind == "prepare":
        return {"kind": kind, "family": family, "n": n, "k": k}
    if kind == "sweep":
        if rng.random() < 0.25:
            return {"kind": kind, "family": family, "n": _log(rng, 4096, 65536), "k": k, "precision": 64, "iters": rng.randint(1, 3)}
        return {"kind": kind, "family": family, "n": n, "k": k, "precision": 32, "iters": rng.randint(2, 10)}
    if kind == "stress":
        if rng.random() < 0.25:  # a small graph over all its pairs
            return {"kind": kind, "family": family, "n": _log(rng, 1024, 8192), "k": 50, "sources": 0, "targets": 0}
        return {"kind": kind, "family": family, "n": n, "k": 50, "sources": 1024, "targets": 1024}
    if kind == "kmeans":
        return {"kind": kind, "family": family, "n": n, "k": k, "passes": rng.choice([10, 20, 50])}
    n = _log(rng, 4096, 262144)
    if kind == "wprepare":
        return {"kind": kind, "n": n, "k": k}
    if kind == "wlayout":
        return {"kind": kind, "n": n, "k": k, "iters": rng.randint(2, 10)}
    if kind == "wstress":
        return {"kind": kind, "n": n, "k": 50, "sources": 1024, "targets": 1024}
    return {"kind": kind, "count": _log(rng, 32, 512), "n_min": 64, "n_max": rng.choice([1024, 4096, 8192]), "iters": rng.randint(5, 20)}


# ---------------------------------------------------------------- inputs
def _relabel(n, src, dst, seed, *more):
    """The same graph under a seeded relabelling, its edges in a seeded order."""
    rng = np.random.default_rng(seed)
    perm, order = rng.permutation(n).astype(np.int32), rng.permutation(len(src))
    return (n, perm[src[order]], perm[dst[order]], *(t[order] for t in more))


def _edges(family, n, seed):
    """A network of n nodes and as many edges for every seed: the heavy-tailed
    one generated anew, the geometric one (whose largest component varies in
    size) one point set whose labels, in no order there either, are drawn."""
    return inputs.ba(n, 4, seed) if family == "ba" else _relabel(*inputs.rgg(n, 8.0, 1), seed)


def _grid(case, seed):
    """A grid under a seeded relabelling: edge list, and every node's cell."""
    n, src, dst = inputs.grid(case["rows"], case["cols"])
    perm = np.random.default_rng(seed).permutation(n).astype(np.int32)
    cell = np.empty(n, np.int64)
    cell[perm] = np.arange(n)
    return n, perm[src], perm[dst], cell // case["cols"], cell % case["cols"]


def _batch_inputs(case, seed):
    rng = np.random.default_rng(1)
    graphs = []
    for j in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        graph = inputs.mixed_graph(inputs.FAMILIES[int(rng.integers(0, 3))], n, int(rng.integers(1, 1 << 40)))
        n, src, dst = _relabel(*graph, seed + 7919 * j)
        graphs.append((n, src, dst, max(2, min(100, n // 4))))
    return graphs


def _start(dist, src, dst, seed, dtype):
    """A layout: a seeded projection of the squared pivot distances, mean edge
    length 1, with a jitter of 0.3 of it."""
    k, n = dist.shape
    gen = torch.Generator().manual_seed(seed)
    v = torch.randn(k, 2, generator=gen, dtype=torch.float64)
    v -= v.mean(0)
    v = v.tolist()
    x = torch.zeros(n, 2, dtype=torch.float64, device=DEV)
    for a in range(k):
        d2 = dist[a].double().square()
        x[:, 0] += d2 * v[a][0]
        x[:, 1] += d2 * v[a][1]
    x -= x.mean(0)
    length = (x[src] - x[dst]).norm(dim=1).mean()
    jitter = torch.randn(n, 2, generator=torch.Generator(DEV).manual_seed(seed + 1), device=DEV, dtype=torch.float64)
    return (x / length + 0.3 * jitter).to(dtype).contiguous()


def _hops(dip):
    return dip.view(torch.int16)  # hop distances below 32768


def _table(cnt, most):
    """A count table, whose length depends on the pivots, in one of the length
    that no graph of this size exceeds."""
    out = torch.zeros(most, dtype=torch.int32, device=DEV)
    out[: cnt.numel()] = cnt.view(torch.int32)
    return out


def prepare(case, seed):
    kind, k = case["kind"], case.get("k")
    s = {"case": case, "seed": seed}
    if kind == "layout":
        s["n"], s["src"], s["dst"], _, _ = _grid(case, seed)
        return s
    if kind == "batch":
        s["graphs"] = _batch_inputs(case, seed)
        nodes = sum(g[0] for g in s["graphs"])
        s["jitter"] = 0.3 * torch.randn(nodes, 2, generator=torch.Generator(DEV).manual_seed(seed), device=DEV)
        return s
    if kind in ("wprepare", "wlayout", "wstress"):
        n, src, dst, length = inputs.rgg_lengths(case["n"], 8.0, 1)
        s["n"], src, dst, length = _relabel(n, src, dst, seed, length)
        s["src"], s["dst"], s["len"] = (torch.from_numpy(t).to(DEV) for t in (src, dst, length))
        if kind == "wprepare":
            return s
        g = s["g"] = ssm.ssm_build_wgraph(s["n"], s["src"], s["dst"], s["len"])
        s["piv"] = torch.from_numpy(np.random.default_rng(seed).permutation(g.n)[:k].astype(np.int32)).to(DEV)
        s["dist"] = ssm.ssm_pivot_sssp(g, s["piv"])
        if kind == "wlayout":
            s["region"], s["s"] = ssm.ssm_weighted_counts(g, s["piv"], s["dist"])
        s["x0"] = _start(s["dist"], s["src"], s["dst"], seed, torch.float32)
        return s
    s["n"], src, dst = _edges(case["family"], case["n"], seed)
    if kind == "prepare":
        s["src"], s["dst"] = src, dst
        return s
    s["src"], s["dst"] = torch.from_numpy(src).to(DEV), torch.from_numpy(dst).to(DEV)
    g = s["g"] = ssm.ssm_build_graph(s["n"], s["src"], s["dst"])
    piv = ssm.ssm_select_pivots(g, k)
    dip = ssm.ssm_pivot_bfs(g, piv)
    if kind == "kmeans":
        s["piv"], s["dip"] = piv, dip
        return s
    dtype = torch.float64 if case.get("precision") == 64 else torch.float32
    s["x0"] = _start(_hops(dip), s["src"], s["dst"], seed, dtype)
    if kind == "sweep":
        cnt_len, dmax = ssm.ssm_aggregate_size(dip, with_dmax=True)
        s["p"] = ssm.Pivots(k, piv, dip, *ssm.ssm_aggregate(dip, cnt_len), dmax)
        # the sweep's buffers, kept by a program that calls it repeatedly
        s["work"] = ssm.IterateWorkspace(g.n, g.m, k, cnt_len, case["precision"], DEV)
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "layout":
        return {"pos": ssm.layout(s["n"], s["src"], s["dst"], case["k"], case["iters"])}
    if kind == "prepare":
        g, p, pos, eig = ssm.prepare(s["n"], s["src"], s["dst"], case["k"])
        # eig also carries the solver's step count and residual: diagnostics, not results
        return {"rowptr": g.rowptr, "colidx": g.colidx, "pivots": p.pivots, "dip": _hops(p.dip), "region": p.region,
                "cnt_off": p.cnt_off, "cnt": _table(p.cnt, g.n + p.k), "pos": pos, "eig": eig[:2]}
    if kind == "sweep":
        pos = s["x0"].clone()
        ssm.ssm_iterate(s["g"], s["p"], pos, case["iters"], work=s["work"])
        return {"pos": pos}
    if kind == "stress":
        out, sums = ssm.ssm_stress(s["g"], s["x0"], case["sources"], case["targets"], s["seed"])
        return {"out": out, "sums": sums}
    if kind == "kmeans":
        piv, assign, passes = ssm.ssm_kmeans_pivots(s["dip"], s["piv"], case["passes"])
        return {"pivots": piv, "assign": assign, "passes": passes}
    if kind == "wprepare":
        g = ssm.ssm_build_wgraph(s["n"], s["src"], s["dst"], s["len"])
        piv = ssm.ssm_select_pivots_weighted(g, case["k"])
        dist = ssm.ssm_pivot_sssp(g, piv)
        region, cnt = ssm.ssm_weighted_counts(g, piv, dist)
        return {"rowptr": g.rowptr, "colidx": g.colidx, "elen": g.elen, "pivots": piv, "dist": dist, "region": region,
                "s": cnt.view(torch.int32)}
    if kind == "wlayout":
        init, eig = ssm.ssm_pivotmds_weighted(s["g"], s["dist"])
        pos = s["x0"].clone()
        ssm.ssm_iterate_weighted(s["g"], s["piv"], s["dist"], s["s"], pos, case["iters"])
        return {"init": init, "eig": eig[:2], "pos": pos}
    if kind == "wstress":
        out, sums = ssm.ssm_stress_weighted(s["g"], s["x0"], case["sources"], case["targets"], s["seed"])
        return {"out": out, "sums": sums}
    bp = ssm.ssm_batch_prepare(s["graphs"], DEV)
    init = bp.pos.clone()
    bp.pos.add_(s["jitter"])  # separates coincident nodes before the sweeps
    ssm.ssm_batch_iterate_packed(bp, case["iters"])
    return {"rowptr": bp.rowptr, "pivots": bp.pivots, "dip": _hops(bp.dip), "region": bp.region, "cnt": _table(bp.cnt, bp.pos.shape[0] + bp.pivots.numel()),
            "init": init, "eig": bp.eig, "pos": bp.pos}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind, k = case["kind"], case.get("k", 0)
    if kind == "layout":
        n = case["rows"] * case["cols"]
        return {"bytes": 16 * n + 8 * n, "flops": case["iters"] * 14.0 * n * (k + 4) + n * k * k}
    if kind == "batch":
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        nodes = case["count"] * (case["n_max"] - case["n_min"]) / (hi - lo)
        return {"bytes": nodes * (24 + 24 + 2 * 80 + 32), "flops": case["iters"] * 14.0 * nodes * 84 + nodes * 6400}
    n = case["n"]
    m = 4 * n  # both families: mean degree 8
    if kind == "prepare":  # edges in; CSR, distances, regions, layout out
        return {"bytes": 8 * m + 4 * n + 8 * m + 2 * k * n + 4 * n + 8 * n, "flops": n * k * (k + 1.0) + 4.0 * n * k}
    if kind == "sweep":  # an iteration reads every distance and edge once: the table does not stay on the SMs
        size = 2 * case["precision"] // 8
        return {"bytes": case["iters"] * (2 * k * n + 4 * n + 8 * m + 2 * size * n), "flops": case["iters"] * 14.0 * n * (k + 8)}
    if kind == "stress":
        pairs = case["sources"] * case["targets"] or n * (n - 1) // 2
        return {"bytes": 4 * n + 8 * m + 8 * n, "flops": 12.0 * pairs + 1.0 * (case["sources"] or n) * 2 * m}
    if kind == "kmeans":
        # a pass compares every node with every centre, and only a pass that changes nothing ends them early
        return {"bytes": 2 * k * n * case["passes"] + 4 * n, "flops": case["passes"] * 2.0 * n * k * k}
    if kind == "wprepare":
        return {"bytes": 12 * m + 4 * n + 16 * m + 4 * k * n + 4 * n + 4 * k * n, "flops": 2.0 * k * 2 * m}
    if kind == "wlayout":
        return {"bytes": (1 + case["iters"]) * 4 * k * n + case["iters"] * (4 * k * n + 16 * m + 20 * n) + 8 * n,
                "flops": n * k * (k + 1.0) + case["iters"] * 14.0 * n * (k + 8)}
    return {"bytes": 4 * n + 16 * m + 8 * n, "flops": 12.0 * case["sources"] * case["targets"] + 2.0 * case["sources"] * 2 * m}


# ---------------------------------------------------------------- the same in 64 bits
def _mds(delta, src, dst, target):
    """PivotMDS of the squared distances delta [k, n] (float64), rescaled to the
    given sum of edge lengths; eigenvectors signed by their largest entry."""
    c = delta - delta.mean(0, keepdim=True)
    c -= c.mean(1, keepdim=True)
    c *= -0.5
    lam, vec = torch.linalg.eigh(c @ c.T)
    x = []
    for r in (-1, -2):
        v = vec[:, r]
        v = v * (-1.0 if v[v.abs().argmax()] < 0 else 1.0)
        x.append(v @ c)
    x = torch.stack(x, 1)
    return x * (target / (x[src] - x[dst]).norm(dim=1).sum()), lam[[-1, -2]]


def _sweeps(x, src, dst, length, pivots, dist, s, iters):
    """Jacobi updates of Eq. 4: edges both ways with their lengths, distances
    [k, n], counts s [k, n] (0: no term)."""
    w_e = length ** -2
    for _ in range(iters):
        e = x[src] - x[dst]
        r = e.norm(dim=1, keepdim=True)
        t = x[dst] + torch.where(r > 0, e * length[:, None] / r, 0.0)
        num = torch.zeros_like(x).index_add_(0, src, w_e[:, None] * t)
        den = torch.zeros_like(x[:, 0]).index_add_(0, src, w_e)
        for a in range(len(pivots)):
            d = dist(a)
            w = torch.where(s(a) > 0, s(a) / d.square().clamp(min=1e-300), 0.0)
            xp = x[int(pivots[a])]
            e = x - xp
            r = e.norm(dim=1)
            num += w[:, None] * (xp + e * torch.where(r > 0, d / r, 0.0)[:, None])
            den += w
        x = num / den[:, None]
    return x


def _counts(dip, region, k):
    """s[a, i] = |{j in R(a): 2 d_aj <= d_ai}| for hop distances, 0 where d_ai < 2."""
    top = int(dip.max()) + 1
    out = []
    for a in range(k):
        c = torch.bincount(dip[a][region == a].long(), minlength=top).cumsum(0)
        d = dip[a].long()
        out.append(torch.where(d >= 2, c[d // 2], 0))
    return out


def _bfs_table(n, src, dst, k):
    """Max/min pivots from node 0 and their hop distances, level by level."""
    a, b = torch.cat([src, dst]), torch.cat([dst, src])
    mind = torch.full((n,), 1 << 20, dtype=torch.int32, device=DEV)
    rows, p = [], 0
    for _ in range(k):
        d = torch.full((n,), -1, dtype=torch.int32, device=DEV)
        d[p] = 0
        level = 0
        while True:
            hit = torch.zeros(n, dtype=torch.bool, device=DEV)
            hit[b[d[a] == level]] = True
            hit &= d < 0
            if not bool(hit.any()):
                break
            level += 1
            d[hit] = level
        rows.append(d)
        mind = torch.minimum(mind, d)
        p = int((mind == mind.max()).nonzero()[0])
    return torch.stack(rows)


def exact(case, seed):
    kind = case["kind"]
    if kind == "layout":
        n, src, dst, row, col = _grid(case, seed)
        row, col, src, dst = (torch.from_numpy(np.asarray(t)).long().to(DEV) for t in (row, col, src, dst))
        k = case["k"]
        pivots, mind = [0], None
        for a in range(k):
            d = (row - row[pivots[a]]).abs() + (col - col[pivots[a]]).abs()
            mind = d if a == 0 else torch.minimum(mind, d)
            pivots.append(int((mind == mind.max()).nonzero()[0]))
        pivots = pivots[:k]
        dip = torch.stack([(row - row[p]).abs() + (col - col[p]).abs() for p in pivots])
        region = (dip * k + torch.arange(k, device=DEV)[:, None]).argmin(0)
        x, _ = _mds(dip.double().square(), src, dst, float(len(src)))
        cnt = _counts(dip, region, k)
        a, b = torch.cat([src, dst]), torch.cat([dst, src])
        one = torch.ones(len(a), dtype=torch.float64, device=DEV)
        return {"pos": _sweeps(x, a, b, one, pivots, lambda q: dip[q].double(), lambda q: cnt[q].double(), case["iters"])}
    if kind == "prepare":
        n, src, dst = _edges(case["family"], case["n"], seed)
        if case["family"] == "rgg" and case["n"] > 16384:
            return None  # hundreds of levels for each of the k dependent searches
        src, dst = torch.from_numpy(src).long().to(DEV), torch.from_numpy(dst).long().to(DEV)
        x, lam = _mds(_bfs_table(n, src, dst, case["k"]).double().square(), src, dst, float(len(src)))
        return {"rowptr": None, "colidx": None, "pivots": None, "dip": None, "region": None, "cnt_off": None, "cnt": None,
                "pos": x, "eig": lam}
    if kind == "sweep":
        s = prepare(case, seed)
        a, b = torch.cat([s["src"], s["dst"]]).long(), torch.cat([s["dst"], s["src"]]).long()
        one = torch.ones(len(a), dtype=torch.float64, device=DEV)
        dip = _hops(s["p"].dip)
        cnt = [c.int() for c in _counts(dip, s["p"].region, case["k"])]
        return {"pos": _sweeps(s["x0"].double(), a, b, one, s["p"].pivots.tolist(), lambda q: dip[q].double(),
                               lambda q: cnt[q].double(), case["iters"])}
    if kind == "wlayout":
        s = prepare(case, seed)
        src, dst = s["src"].long(), s["dst"].long()
        length = s["len"].double()
        init, lam = _mds(s["dist"].double().square(), src, dst, float(length.sum()))
        cnt = s["s"].view(torch.int32)
        pos = _sweeps(s["x0"].double(), torch.cat([src, dst]), torch.cat([dst, src]), length.repeat(2), s["piv"].tolist(),
                      lambda q: s["dist"][q].double(), lambda q: cnt[q].double(), case["iters"])
        return {"init": init, "eig": lam, "pos": pos}
    # whole numbers and least float32 path sums, or (stress) distances from a
    # thousand searches of hundreds of levels
    return None
