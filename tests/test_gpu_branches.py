"""Kernel variants that the everyday workloads do not reach, each against the
oracle through the C ABI:

* the grid-wide push bitset BFS (k_msbfs), taken when a graph has more nodes
  than the per-source BFS's shared-memory visited bitmap holds (1,638,400);
* the FP32 sweep with its clamped s table in global memory and the FP64 sweep
  with its counts in global memory, taken when the tables pass 200 KB of
  shared memory (a long path: regions of thousands of hops);
* coincident positions (r = 0, observed by the paper's weakness analysis in
  Section 4): a term whose points coincide adds w x_j only, in every sweep
  form (FP32 full table, FP32 clamped table, FP64, batched).

ssm_last_sweep_config() reports which sweep kernel ran, so each test checks
that it reached the variant it is named for.
"""
import os

import numpy as np
import pytest
import torch

import oracle as O
import paper_1608_08909_gb300 as ssm
from paper_1608_08909_gb300 import inputs as I

pytestmark = pytest.mark.gpu
DEV = "cuda"
THREADS = max(1, min(16, os.cpu_count() or 1))


def _gpu_graph(n, s, d):
    return ssm.ssm_build_graph(n, torch.from_numpy(s).to(DEV), torch.from_numpy(d).to(DEV))


def _norm_err(a, b):
    b = np.asarray(b, np.float64)
    c = b - b.mean(0)
    return np.sqrt(((np.asarray(a, np.float64) - b) ** 2).sum(1)).max() / np.sqrt((c ** 2).sum(1).mean())


def _gpu_pivots(k, prep):
    return ssm.Pivots(k, torch.from_numpy(prep.pivots).to(DEV), torch.from_numpy(prep.dip).to(DEV),
                      torch.from_numpy(prep.region).to(DEV),
                      torch.from_numpy(prep.cnt_off.astype(np.int32)).to(DEV), torch.from_numpy(prep.cnt).to(DEV))


# ------------------------------------------------------------------ push bitset BFS above the bitmap limit

@pytest.mark.parametrize("family,k", [("grid", 3), ("ba", 40)])
def test_pivot_bfs_above_bitmap_limit(family, k):
    """n above 1,638,400: d_ip and the max/min pivots through the cooperative
    kernels (k_msbfs for the distances), bit-exact; the grid has 2,600 BFS
    levels, the BA graph few levels of up to a million nodes."""
    if family == "grid":
        n, s, d = I.grid(1300, 1300)
    else:
        n, s, d = I.ba(1700000, 4, 5)
    assert n > 1638400
    og = O.build_csr(n, s, d)
    g = _gpu_graph(n, s, d)
    piv = ssm.ssm_select_pivots(g, k, 0)
    assert ssm.ssm_last_pivot_config() == {"cluster": 0, "mind_bytes": 4}
    opiv = O.maxmin(og, k, 0)
    assert np.array_equal(piv.cpu().numpy(), opiv)
    dip = ssm.ssm_pivot_bfs(g, piv).cpu().numpy()
    assert np.array_equal(dip, O.pivot_dist_threads(og, opiv, THREADS))


# ------------------------------------------------------------------ tables in global memory

@pytest.fixture(scope="module")
def long_path():
    """A 60000-node path with 6 max/min pivots; its PivotMDS layout is exactly
    collinear and already a fixed point of the sweep, so the sweeps start from
    it with seeded noise added (a relative change well above FP32 rounding)."""
    n, s, d = I.path(60000)
    prep = O.prepare(n, s, d, 6)
    assert prep.dip.max() <= 65534
    x0 = prep.pos0 + np.random.default_rng(12).normal(scale=200.0, size=prep.pos0.shape)
    return n, s, d, prep, x0


def test_sweep_fp32_clamped_table_in_global_memory(long_path):
    n, s, d, prep, start = long_path
    k = len(prep.pivots)
    assert (2 * len(prep.cnt) + k) * 4 + k * 24 > 200 * 1024
    g = _gpu_graph(n, s, d)
    P = _gpu_pivots(k, prep)
    x0 = start.astype(np.float32)
    pos = torch.from_numpy(x0.copy()).to(DEV)
    _, rel = ssm.ssm_iterate(g, P, pos, 1)
    assert ssm.ssm_last_sweep_config()["kernel"] == "f32_clamped_global"
    want, orel = O.sweep_jacobi(prep.g, prep.pivots, prep.dip, prep.w, x0.astype(np.float64))
    assert _norm_err(pos.cpu().numpy(), want) < 1e-5
    assert rel.item() == pytest.approx(orel, rel=1e-4)


def test_sweep_fp64_counts_in_global_memory(long_path):
    n, s, d, prep, start = long_path
    k = len(prep.pivots)
    assert k * 24 + len(prep.cnt) * 8 > 200 * 1024
    g = _gpu_graph(n, s, d)
    P = _gpu_pivots(k, prep)
    pos = torch.from_numpy(start.copy()).to(DEV)
    _, rel = ssm.ssm_iterate(g, P, pos, 5)
    assert ssm.ssm_last_sweep_config()["kernel"] == "f64_counts_global"
    want, orel = O.iterate(prep, start, 5)
    assert np.array_equal(pos.cpu().numpy(), want)
    assert rel.item() == pytest.approx(orel, rel=1e-12)


@pytest.mark.parametrize("scale", [1.0, 1e-130, 1e130, 1e-70])
@pytest.mark.parametrize("name,k", [("path", 7), ("ba", 40), ("star", 5)])
def test_sweep_fp64_ranges_bit_for_bit(name, k, scale):
    """The shared reciprocal square root, its range check (lengths whose squares
    leave 2^+-400 take the IEEE operations), distances below and above the
    table of 1 / d^2, rows on both sides of the long-row limit: the oracle's
    bits."""
    n, s, d = {"path": lambda: I.path(2500), "ba": lambda: I.ba(700, 4, 3),
               "star": lambda: (1000, np.zeros(999, np.int32), np.arange(1, 1000, dtype=np.int32))}[name]()
    prep = O.prepare(n, s, d, k)
    x0 = scale * (prep.pos0 + np.random.default_rng(2).normal(size=(n, 2)))
    x0[::7, 1] = x0[0, 1]  # equal ordinates: a zero difference
    want, _ = O.sweep_jacobi(prep.g, prep.pivots, prep.dip, prep.w, x0)
    pos = torch.from_numpy(x0.copy()).to(DEV)
    ssm.ssm_iterate(_gpu_graph(n, s, d), _gpu_pivots(k, prep), pos, 1)
    assert ssm.ssm_last_sweep_config()["kernel"] == "f64_counts_smem"
    assert np.array_equal(pos.cpu().numpy(), want)


@pytest.mark.parametrize("family,n", [("ba", 9001), ("ba", 9002), ("ba", 9004), ("ba", 9008), ("rgg", 9400), ("path", 8201)])
@pytest.mark.parametrize("shift", [0, 1, 2, 8])
def test_sweep_distance_copy_alignments(family, n, shift):
    """The sweep's tiled copy of d_ip (and the denominators summed with it) from
    rows on any alignment: the same positions as from a table on 16 bytes."""
    n, s, d = {"ba": lambda: I.ba(n, 4, 3), "rgg": lambda: I.rgg(n, 8.0, 7), "path": lambda: I.path(n)}[family]()
    prep = O.prepare(n, s, d, 21)
    g, P = _gpu_graph(n, s, d), _gpu_pivots(21, prep)
    x0 = torch.from_numpy(prep.pos0.astype(np.float32)).to(DEV)
    want, _ = O.sweep_jacobi(prep.g, prep.pivots, prep.dip, prep.w, prep.pos0.astype(np.float32).astype(np.float64))
    room = torch.zeros(21 * n + 16, dtype=torch.uint16, device=DEV)
    moved = room[shift:shift + 21 * n].view(21, n)
    moved.copy_(P.dip)
    a, b = x0.clone(), x0.clone()
    ssm.ssm_iterate(g, P, a, 1)
    P.dip = moved
    ssm.ssm_iterate(g, P, b, 1)
    assert _norm_err(a.cpu().numpy(), want) < 1e-5
    assert torch.equal(a, b)


# ------------------------------------------------------------------ coincident positions

def _coincident_state(prep, rng, count):
    """The PivotMDS start rounded to FP32 with `count` nodes moved onto a pivot
    and `count` nodes moved onto one of their neighbours (exact copies, so
    r = 0 in both precisions)."""
    x = prep.pos0.astype(np.float32).copy()
    g = prep.g
    n = g.n
    nodes = rng.choice(n, 2 * count, replace=False)
    for i in nodes[:count]:
        x[i] = x[prep.pivots[rng.integers(0, len(prep.pivots))]]
    for i in nodes[count:]:
        nb = g.colidx[g.rowptr[i]:g.rowptr[i + 1]]
        x[i] = x[nb[rng.integers(0, len(nb))]]
    return x


@pytest.mark.parametrize("name,k,kernel", [("grid32", 50, "f32_full_table"), ("rgg", 100, "f32_clamped_smem"),
                                           ("ba", 40, "f32_full_table")])
def test_sweep_coincident_positions(name, k, kernel):
    n, s, d = {"grid32": lambda: I.grid(32, 32), "rgg": lambda: I.rgg(6000, 8.0, 7),
               "ba": lambda: I.ba(12000, 4, 3)}[name]()
    prep = O.prepare(n, s, d, k)
    x0 = _coincident_state(prep, np.random.default_rng(3), 40)
    # the state really has coincident pivot and edge terms
    piv_pos = x0[prep.pivots]
    assert any((x0[i] == piv_pos).all(1).any() for i in range(n) if i not in set(prep.pivots.tolist()))
    g = _gpu_graph(n, s, d)
    P = _gpu_pivots(k, prep)
    want, orel = O.sweep_jacobi(prep.g, prep.pivots, prep.dip, prep.w, x0.astype(np.float64))
    assert np.isfinite(want).all()
    # FP32
    pos = torch.from_numpy(x0.copy()).to(DEV)
    _, rel = ssm.ssm_iterate(g, P, pos, 1)
    assert ssm.ssm_last_sweep_config()["kernel"] == kernel
    assert _norm_err(pos.cpu().numpy(), want) < 1e-5
    # FP64: bit for bit
    pos = torch.from_numpy(x0.astype(np.float64)).to(DEV)
    ssm.ssm_iterate(g, P, pos, 1)
    assert np.array_equal(pos.cpu().numpy(), want)
    # batched sweep
    pos = torch.from_numpy(x0.copy()).to(DEV)
    ssm.ssm_batch_iterate([(g, P, pos)], 1)
    assert _norm_err(pos.cpu().numpy(), want) < 1e-5


# ------------------------------------------------------------------ small graphs in one cluster
def _clique(n):
    s, d = np.triu_indices(n, 1)
    return n, s.astype(np.int32), d.astype(np.int32)


CLUSTER = {
    "fewer_nodes_than_ctas": (lambda: I.path(5), 2),
    "one_node_per_cta_and_one_more": (lambda: I.path(17), 17),
    "ragged_blocks": (lambda: I.grid(33, 31), 12),
    "long_rows": (lambda: I.ba(1025, 6, 3), 33),
    "neighbours_beyond_shared_memory": (lambda: _clique(1500), 2),
    "few_partial_sums": (lambda: I.grid(64, 64), 100),
    "largest": (lambda: I.ba(8192, 4, 5), 60),
    "one_too_large": (lambda: I.ba(8193, 4, 5), 60),
}


@pytest.mark.parametrize("name", list(CLUSTER))
def test_sweep_fp32_small_graph_cluster(name):
    """The fifth iteration of a cluster launch against the oracle's step from the
    fourth (two launches that agree on the first four), at the single step's
    bound of 1e-5; a spread-out random start."""
    make, k = CLUSTER[name]
    n, s, d = make()
    prep = O.prepare(n, s, d, k)
    x0 = (np.random.default_rng(n).standard_normal((n, 2)) * np.sqrt(n)).astype(np.float32)
    g, P = _gpu_graph(n, s, d), _gpu_pivots(k, prep)
    four, five = torch.from_numpy(x0.copy()).to(DEV), torch.from_numpy(x0.copy()).to(DEV)
    ssm.ssm_iterate(g, P, four, 4)
    done, rel = ssm.ssm_iterate(g, P, five, 5)
    assert (ssm.ssm_last_sweep_config()["kernel"] == "f32_cluster") == (name != "one_too_large")
    x4 = four.cpu().numpy().astype(np.float64)
    want, orel = O.sweep_jacobi(prep.g, prep.pivots, prep.dip, prep.w, x4)
    assert int(done.item()) == 5
    assert _norm_err(five.cpu().numpy(), want) < 1e-5
    assert rel.item() == pytest.approx(orel, rel=1e-4)


def test_sweep_fp32_cluster_tolerance_and_wrong_hint():
    """tol > 0 stops at the same iteration as single sweeps do; a largest
    distance below the true one is refused."""
    n, s, d = I.grid(32, 32)
    g, P, pos, _ = ssm.prepare(n, s, d, 20)
    one, x = 0, pos.clone()
    while True:
        _, rel = ssm.ssm_iterate(g, P, x, 1)
        one += 1
        if rel.item() < 3e-3:
            break
        assert one < 200
    done, rel = ssm.ssm_iterate(g, P, pos, 200, tol=3e-3)
    assert int(done.item()) == one > 4 and rel.item() < 3e-3
    assert _norm_err(pos.cpu().numpy(), x.cpu().numpy().astype(np.float64)) < one * 1e-5
    P.dmax -= 1
    with pytest.raises(ssm.SSMError) as e:
        ssm.ssm_iterate(g, P, pos, 4)
    assert e.value.code == -1


@pytest.mark.parametrize("n", [2, 7, 8, 15, 16, 17])
def test_sweep_fp32_cluster_of_few_nodes(n):
    """Clusters in which some CTAs own no node, over many iterations: every one
    of them takes part in every exchange, so a run gives the same bits again,
    cut in two, and stopped by the tolerance."""
    s, d = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    g = _gpu_graph(n, s, d)
    piv = torch.arange(n, dtype=torch.int32, device=DEV)
    dip = ssm.ssm_pivot_bfs(g, piv)
    cnt_len, dmax = ssm.ssm_aggregate_size(dip, with_dmax=True)
    P = ssm.Pivots(n, piv, dip, *ssm.ssm_aggregate(dip, cnt_len), dmax)
    x0 = torch.from_numpy((np.random.default_rng(n).standard_normal((n, 2)) * n).astype(np.float32)).to(DEV)

    def run(*cuts, tol=0.0):
        x = x0.clone()
        for iters in cuts:
            done, rel = ssm.ssm_iterate(g, P, x, iters, tol)
        assert ssm.ssm_last_sweep_config()["kernel"] == "f32_cluster"
        return x, int(done.item()), rel.item()

    x, done, _ = run(400)
    assert done == 400 and torch.isfinite(x).all()
    assert torch.equal(run(400)[0], x) and torch.equal(run(150, 250)[0], x)
    y, done, rel = run(400, tol=1e-2)
    assert done == 400 or rel < 1e-2
    assert done < 4 or torch.equal(run(done)[0], y)


def _hubs(n, hubs):
    """Nodes 0 .. hubs - 1 adjacent to every other node."""
    s = np.repeat(np.arange(hubs), n)
    d = np.tile(np.arange(n), hubs)
    keep = s < d
    return n, s[keep].astype(np.int32), d[keep].astype(np.int32)


@pytest.mark.parametrize("name,make,k,cluster", [
    ("row_of_1024", lambda: _hubs(1025, 1), 5, True),      # one warp's
    ("row_of_1025", lambda: _hubs(1026, 1), 5, True),      # segments of 256, the last of one entry
    ("star", lambda: _hubs(8000, 1), 50, True),
    ("hubs_in_some_ctas", lambda: _hubs(8001, 3), 30, True),
    ("64_hubs_a_cta", lambda: _clique(1026), 5, True),     # 65 in two CTAs: a warp each there
    ("rows_partly_kept", lambda: _clique(1300), 20, True),
    ("too_dense", lambda: _clique(1600), 2, False)])
def test_sweep_fp32_cluster_hubs_and_dense_rows(name, make, k, cluster):
    """Rows of more than 1,024 entries, and graphs whose neighbours the cluster
    keeps in part or not at all: one iteration from the fourth against the
    oracle at the single step's bound; the same bits again, and without hints."""
    n, s, d = make()
    prep = O.prepare(n, s, d, k)
    x0 = (np.random.default_rng(n).standard_normal((n, 2)) * np.sqrt(n)).astype(np.float32)
    g, P = _gpu_graph(n, s, d), _gpu_pivots(k, prep)
    P.dmax = int(prep.dip.max())
    four, five = torch.from_numpy(x0.copy()).to(DEV), torch.from_numpy(x0.copy()).to(DEV)
    ssm.ssm_iterate(g, P, four, 4)
    ssm.ssm_iterate(g, P, five, 5)
    assert (ssm.ssm_last_sweep_config()["kernel"] == "f32_cluster") == cluster
    want, _ = O.sweep_jacobi(prep.g, prep.pivots, prep.dip, prep.w, four.cpu().numpy().astype(np.float64))
    assert _norm_err(five.cpu().numpy(), want) < 1e-5
    P.dmax = None
    again = torch.from_numpy(x0.copy()).to(DEV)
    ssm.ssm_iterate(g, P, again, 5)
    assert torch.equal(again, five)


def _hard_quotients(count, seed):
    """(dx, dy) with r = RN(sqrt(RN(RN(dx^2) + RN(dy^2)))) and dx / r within a
    relative 2^-105 of a midpoint between two doubles: r odd, 2^54 dx = M r +- 1
    with M, 54 bits, the inverse of -+r modulo 2^54."""
    rng = np.random.default_rng(seed)
    r, dx = [], []
    while len(r) < count:
        R = int(rng.integers(1 << 52, 1 << 53)) | 1
        for sign in (1, -1):
            M = -sign * pow(R, -1, 1 << 54) % (1 << 54)
            if M >> 53:
                r.append(float(R))
                dx.append(float((M * R + sign) >> 54))
    r, dx = np.array(r), np.array(dx)
    dy = np.sqrt((r - dx) * (r + dx))
    for step in range(1, 40):  # the next dy up and down until r comes out
        off = np.sqrt(dx * dx + dy * dy) - r
        dy = np.where(off > 0, np.nextafter(dy, 0), np.where(off < 0, np.nextafter(dy, np.inf), dy))
    ok = np.sqrt(dx * dx + dy * dy) == r
    return dx[ok], dy[ok]


def _hard_roots():
    """(dx, dy) whose h = RN(RN(dx^2) + RN(dy^2)) has a root next to a midpoint:
    h = H 2^(b - 2) with M^2 = 2^b H - delta for an odd M of 54 bits and a small
    delta, M a root of -delta modulo 2^b."""
    out = []
    for b in (54, 55):
        for delta in list(range(7, 1200, 8)) + list(range(-1, -1200, -8)):
            M = 1
            for bits in range(4, b + 1):  # a root modulo 2^bits
                if (M * M + delta) % (1 << bits):
                    M += 1 << (bits - 2)
            for root in (M, -M, M + (1 << (b - 1)), (1 << (b - 1)) - M):
                root %= 1 << b
                if root >> 53 != 1:
                    continue
                assert (root * root + delta) % (1 << b) == 0
                H = (root * root + delta) >> b
                if H >> 52 != 1:
                    continue
                h = float(H) * 2.0 ** (b - 2 - 104)
                for x in np.sqrt(h * np.linspace(0.3, 0.9, 40)):
                    ys = np.sqrt(h - x * x) + np.arange(-4, 5) * np.spacing(np.sqrt(h - x * x))
                    hit = ys[x * x + ys * ys == h]
                    if len(hit):
                        out.append((x, hit[0]))
                        break
    return np.array(out).T


def test_sweep_fp64_rounds_as_ieee_operations():
    """A leaf of a star whose hub is at the origin moves to (dx / r, dy / r), with
    the square root and the quotients of the shared reciprocal square root:
    the IEEE operations' bits where the exact values lie next to midpoints of
    two doubles, and on ordinary ones."""
    rng = np.random.default_rng(5)
    xy = [_hard_quotients(20000, 1), _hard_quotients(20000, 2)[::-1], _hard_roots(),
          rng.standard_normal((2, 100000)) * 10.0 ** rng.integers(-3, 4, 100000)]
    assert [v.shape[1] if hasattr(v, "shape") else len(v[0]) for v in xy][2] > 100 and len(xy[0][0]) > 15000
    x0 = np.concatenate([np.zeros((1, 2))] + [np.stack(v, 1) for v in xy])
    x0[1:] *= rng.choice([-1.0, 1.0], (len(x0) - 1, 2)) * 2.0 ** rng.integers(-60, 60, (len(x0) - 1, 1))
    n = len(x0)
    g = _gpu_graph(n, np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32))
    piv = torch.zeros(1, dtype=torch.int32, device=DEV)
    dip = ssm.ssm_pivot_bfs(g, piv)
    P = ssm.Pivots(1, piv, dip, *ssm.ssm_aggregate(dip, ssm.ssm_aggregate_size(dip)))
    pos = torch.from_numpy(x0.copy()).to(DEV)
    ssm.ssm_iterate(g, P, pos, 1)
    d = x0[1:]
    want = d / np.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1])[:, None]
    assert np.array_equal(pos.cpu().numpy()[1:], want)


@pytest.mark.parametrize("n,hubs", [(1025, 1), (1026, 1), (9000, 2), (1100, 31), (1100, 32), (1100, 40)])
def test_small_graph_hub_rows(n, hubs):
    """Rows of more than 1,024 entries in the searches of one block's shared
    memory, up to and beyond the 32 of a level that all warps share, single
    graph and batch: the oracle's pivots and distances."""
    n, s, d = _hubs(n, hubs)
    order = np.random.default_rng(n + hubs).permutation(n).astype(np.int32)
    s, d = order[s], order[d]
    k = 20
    og = O.build_csr(n, s, d)
    piv = O.maxmin(og, k, 0)
    dip = O.pivot_dist(og, piv)
    g = _gpu_graph(n, s, d)
    got = ssm.ssm_select_pivots(g, k, 0)
    assert ssm.ssm_last_pivot_config()["cluster"] == 1
    assert np.array_equal(got.cpu().numpy(), piv)
    assert np.array_equal(ssm.ssm_pivot_bfs(g, got).cpu().numpy(), dip)
    b = ssm.ssm_batch_prepare([(n, s, d, k)] * 2)
    assert np.array_equal(b.pivots.cpu().numpy().reshape(2, k), np.stack([piv, piv]))
    assert np.array_equal(b.dip.cpu().numpy().reshape(2, k, n), np.stack([dip, dip]))


@pytest.mark.parametrize("n,deg,cluster", [(1000, 16, True), (1000, 60, True), (1000, 70, True), (3000, 64, True), (8000, 110, False)])
def test_sweep_fp32_cluster_mean_degrees(n, deg, cluster):
    """The limit between rows of one lane per warp and of a warp follows the mean
    degree up to 64; dense graphs of many rows take two kernels: one iteration
    from the fourth against the oracle at the single step's bound."""
    rng = np.random.default_rng(n + deg)
    s = np.concatenate([np.arange(n - 1), rng.integers(0, n, n * deg // 2)]).astype(np.int32)
    d = np.concatenate([np.arange(1, n), rng.integers(0, n, n * deg // 2)]).astype(np.int32)
    prep = O.prepare(n, s, d, 12)
    x0 = (rng.standard_normal((n, 2)) * np.sqrt(n)).astype(np.float32)
    g, P = _gpu_graph(n, s, d), _gpu_pivots(12, prep)
    four, five = torch.from_numpy(x0.copy()).to(DEV), torch.from_numpy(x0.copy()).to(DEV)
    ssm.ssm_iterate(g, P, four, 4)
    ssm.ssm_iterate(g, P, five, 5)
    assert (ssm.ssm_last_sweep_config()["kernel"] == "f32_cluster") == cluster
    want, _ = O.sweep_jacobi(prep.g, prep.pivots, prep.dip, prep.w, four.cpu().numpy().astype(np.float64))
    assert _norm_err(five.cpu().numpy(), want) < 1e-5
