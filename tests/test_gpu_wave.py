"""The wavefront kernels (calls without a configuration) against the oracle
at the sizes where they can go wrong: around a word, a warp and a block of
pending bits, one block and clusters, hubs beyond a block's list, a front too
wide for a cluster, thresholds that saturate or absorb their step, and the
same answers as the queue engine."""
import threading

import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
import paper_2602_10080_gb300 as S
from gpu_util import assert_exact, assert_exact_many, cfg, gpu_batch, gpu_solve, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    S.build()
    S.lib()


def path(n, w):
    return gg.from_edges(n, [(v, v + 1, w(v)) for v in range(n - 1)] + [(v + 1, v, w(v)) for v in range(n - 1)])


def hub_graph(hubs, arcs):
    """0 -> every hub (weight 1); hub h -> `arcs` targets shared by the hubs."""
    n = 1 + hubs + 2 * arcs
    e = [(0, 1 + h, 1 + h % 2) for h in range(hubs)]
    e += [(1 + h, 1 + hubs + (h * 37 + k) % (2 * arcs), 1 + (h * 7 + k * 3) % 50) for h in range(hubs)
          for k in range(arcs)]
    return gg.from_edges(n, e)


def both(g, src):
    """With and without predecessors, against the oracle and the queue engine."""
    G = upload(g)
    d, p = gpu_solve(G, src, pred=True)
    assert_exact(g, src, d, p)
    d2, _ = gpu_solve(G, src, pred=False)
    np.testing.assert_array_equal(d2, d)
    d3, p3 = gpu_solve(G, src, pred=True, config=cfg())
    np.testing.assert_array_equal(d3, d)
    if g.wtype == "u32" and g.m and int(g.w.min()) >= 1:
        np.testing.assert_array_equal(p3, p)
    G.close()


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 1023, 1024, 1025, 8191, 8193, 20000])
def test_paths_around_words_and_blocks(n):
    both(path(n, lambda v: 1 + v * 7919 % 100), n // 2)


@pytest.mark.parametrize("wtype", ["u32", "f32"])
@pytest.mark.parametrize("n,deg", [(300, 3), (5000, 7), (40000, 12)])
def test_random_directed(n, deg, wtype):
    for lo in (0, 1):
        g = gg.random_directed(n, n * deg, lo, 50, seed=n + lo, wtype=wtype)
        both(g, 1)


@pytest.mark.parametrize("hubs,arcs", [(1, 3000), (5, 257), (600, 300)])
def test_hubs_in_a_cluster(hubs, arcs):
    both(hub_graph(hubs, arcs), 0)


def test_more_hubs_than_a_block_lists():
    """One block per query, 200 hubs in one step, the list holds 128."""
    g = hub_graph(200, 257)
    G = upload(g)
    srcs = np.array([0, 1, 200, g.n - 1] * 40, np.int32)
    d, p = gpu_batch(G, srcs, pred=True)
    assert_exact_many(g, srcs, d, p)
    G.close()


@pytest.mark.parametrize("nq", [2, 9, 10, 19, 38, 77, 153])
def test_batches_of_clusters(nq):
    """Every cluster size; repeated sources are independent queries."""
    g = gg.grid(67, 41, 1, 100, seed=nq)
    G = upload(g)
    srcs = (np.arange(nq) * 7919 % (g.n // 2)).astype(np.int32)
    d, p = gpu_batch(G, srcs, pred=True, host=nq % 2 == 1)
    assert_exact_many(g, srcs, d, p)
    G.close()


def test_thresholds_at_the_ends():
    # lengths saturate at 2^32 - 2, and the threshold with them
    both(path(40, lambda v: 0xFFFFFFFF if v % 3 == 0 else 0x70000000), 0)
    # the threshold's step is absorbed by the distances it is added to
    f = gg.from_edges(300, [(v, v + 1, np.float32(1e30 if v < 5 else 1e-6)) for v in range(299)], wtype="f32")
    both(f, 0)
    # no arc, and no arc out of the source
    both(gg.from_edges(700, [(v, v + 1, 5) for v in range(1, 699)]), 0)


def regular(n, deg, seed):
    """`deg` random arcs from every vertex: by its degrees a mesh, by its front not."""
    rng = np.random.default_rng(seed)
    return gg.Graph("regular", n, n * deg, np.arange(n + 1, dtype=np.int32) * deg,
                    rng.integers(0, n, n * deg).astype(np.int32), rng.integers(1, 100, n * deg).astype(np.uint32), "u32")


@pytest.mark.parametrize("n,deg", [(200_000, 4), (130_000, 6)])
def test_front_too_wide_for_a_cluster(n, deg):
    """Sparse graphs begin in one cluster and start over on the grid."""
    both(regular(n, deg, deg), 3)
    both(gg.random_directed(n, n * deg, 1, 100, seed=deg), 3)


@pytest.mark.parametrize("wtype", ["u32", "f32"])
def test_whole_grid(wtype):
    """Above 2^19 arcs: with hubs (slices over the grid) and without."""
    g = gg.rmat(15, 24, seed=8, wtype=wtype)
    both(g, int(gg.giant_sources(g, 1)[0][0]))
    both(gg.erdos_renyi(50_000, 400_000, 1, 1000, seed=3, wtype=wtype), 7)
    if wtype == "u32":
        both(gg.random_directed(60_000, 900_000, 0, 9, seed=2), 5)
        both(gg.grid(1500, 1450, 1, 100, seed=5), 1_000_000)   # thin, but more vertices than a cluster takes


def side_by_side(g, srcs, pred=True):
    G = upload(g)
    srcs = np.asarray(srcs, np.int32)
    for host in (False, True):
        d, p = gpu_batch(G, srcs, pred=pred, host=host)
        assert_exact_many(g, srcs, d, p)
    d2, _ = gpu_batch(G, srcs, pred=False)
    np.testing.assert_array_equal(d2, d)
    G.close()


@pytest.mark.parametrize("nq", [2, 11, 12, 31, 32, 33, 64, 70])
def test_batch_side_by_side(nq):
    """Groups of 32 queries on a graph with hubs, few queries in turn;
    repeated sources, sources without arcs."""
    g = gg.rmat(13, 24, seed=nq)
    srcs = gg.giant_sources(g, nq)[0]
    srcs[nq // 2] = srcs[0]
    srcs[nq - 1] = int(np.flatnonzero(np.diff(g.row_ptr) == 0)[0])
    side_by_side(g, srcs)


@pytest.mark.parametrize("nq", [3, 40])
def test_batch_side_by_side_f32(nq):
    g = gg.rmat(13, 24, seed=5, wtype="f32")
    side_by_side(g, gg.giant_sources(g, nq)[0], pred=nq == 3)
    if nq == 40:   # strict-improvement predecessors
        G = upload(g)
        srcs = gg.giant_sources(g, nq)[0]
        d, p = gpu_batch(G, srcs, pred=True)
        assert_exact_many(g, srcs, d, p)
        G.close()


def test_batch_rows_of_every_length():
    """Rows at the ends of the short list and of the slices, and lengths that
    saturate."""
    arcs = [0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 127, 128, 129, 255, 256, 257, 700]
    n = 4000
    e = [(v, (v * 31 + k * 97 + 1) % n, 1 + (v * k) % 60) for v in range(n) for k in range(arcs[v % len(arcs)])]
    side_by_side(gg.from_edges(n, e), np.arange(40) * 97)
    side_by_side(gg.random_directed(4000, 300_000, 1, 0xFFFFFFFF, seed=3), np.arange(20) * 7)
    side_by_side(gg.erdos_renyi(130_000, 1_300_000, 1, 99, seed=4, wtype="u32"), np.arange(13) * 9999)


def test_levels_on_cluster_and_grid():
    for g in (gg.grid(300, 200, 1, 9, seed=1), gg.rmat(15, 24, seed=8), hub_graph(600, 300)):
        src = int(gg.giant_sources(g, 1)[0][0]) if g.name.startswith("rmat") else 0
        G = upload(g)
        lev = torch.empty(G.n, dtype=torch.int32, device="cuda")
        par = torch.empty(G.n, dtype=torch.int32, device="cuda")
        G.bfs(src, lev, par)
        torch.cuda.synchronize()
        unit = np.ones(g.m, np.uint32)
        ref = oracle.dijkstra_u32(g.row_ptr, g.col, unit, src)
        np.testing.assert_array_equal(lev.cpu().numpy().view(np.uint32), ref)
        np.testing.assert_array_equal(par.cpu().numpy(), oracle.pred_canonical_u32(g.row_ptr, g.col, unit, src, ref))
        G.close()


def test_two_threads_two_graphs():
    """Whole-grid solves of different graphs from two threads and streams."""
    gs = [gg.rmat(14, 40, seed=s) for s in (1, 2)]
    srcs = [gg.giant_sources(g, 6)[0] for g in gs]
    Gs = [upload(g) for g in gs]
    out = {}

    def work(i):
        st = torch.cuda.Stream()
        for k, s in enumerate(srcs[i]):
            d = torch.empty(Gs[i].n, dtype=torch.int32, device="cuda")
            Gs[i].solve(int(s), d, None, None, st)
            out[i, k] = d

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    torch.cuda.synchronize()
    for (i, k), d in out.items():
        assert_exact(gs[i], int(srcs[i][k]), d.cpu().numpy().view(np.uint32))
    [G.close() for G in Gs]


def test_layout_of_another_threshold():
    """The kernels find the arcs of a hub in any layout, and restore the
    graph's own; a layout held by a serving lane stays refused."""
    g = gg.rmat(13, 24, seed=4)
    src = int(gg.giant_sources(g, 1)[0][0])
    G = upload(g)
    own = G.features()["shadows"]
    for split in (32, 300, 0):
        d, p = gpu_solve(G, src, pred=True, config=cfg(split_arcs=split))
        assert_exact(g, src, d, p)
        d, p = gpu_solve(G, src, pred=True)
        assert_exact(g, src, d, p)
        assert G.features()["shadows"] == own
    srv = S.sssp_serve_create()
    try:
        gpu_solve(G, src, config=cfg(split_arcs=64))
        ds = torch.empty(g.n, dtype=torch.int32, device="cuda")
        t = S.sssp_serve_submit(srv, G.handle, src, ds)
        assert S.sssp_serve_wait(srv, t)[0] == S.Q_DONE
        assert_exact(g, src, ds.cpu().numpy().view(np.uint32))
        with pytest.raises(S.SsspError) as ei:
            gpu_solve(G, src)
        assert ei.value.code == S.SSSP_E_BUSY
    finally:
        S.sssp_serve_destroy(srv)
    d, p = gpu_solve(G, src, pred=True)
    assert_exact(g, src, d, p)
    G.close()


def test_noalloc_on_cluster_and_grid():
    """The fixed scratch serves every kernel and size: one cluster, a front
    that outgrows it, the grid with hubs, and the largest vertex count."""
    for g in (regular(200_000, 4, 4), gg.rmat(16, 16, seed=3),
              gg.erdos_renyi(50_000, 400_000, 1, 99, seed=3, wtype="f32"),
              gg.random_directed(S.SSSP_NOALLOC_MAX_VERTICES, 6_000_000, 0, 9, seed=6)):
        src = int(gg.giant_sources(g, 1)[0][0])
        rp = torch.from_numpy(g.row_ptr).cuda()
        arcs = torch.from_numpy(np.stack([g.col.view(np.uint32), g.w_bits], 1).view(np.int32).copy()).cuda()
        d = torch.empty(g.n, dtype=torch.int32, device="cuda")
        p = torch.empty(g.n, dtype=torch.int32, device="cuda")
        for pred in (p, None):
            S.sssp_solve_noalloc(rp, arcs, g.n, g.m, S.SSSP_W_F32 if g.wtype == "f32" else S.SSSP_W_U32, src, d, pred)
            torch.cuda.synchronize()
            assert_exact(g, src, d.cpu().numpy().view(np.uint32), None if pred is None else p.cpu().numpy())


def test_served_bursts_and_concurrent_solves():
    """Express lanes: bursts of queries on a grid-kernel graph (side by side)
    and on a small one (a cluster each), with and without predecessors, host
    and device buffers, cancellations, while another thread solves on the same
    and on other graphs."""
    graphs = [gg.rmat(15, 24, seed=8), gg.rmat(12, 16, seed=2, wtype="f32")]
    Gs = [upload(g) for g in graphs]
    other = gg.rmat(15, 20, seed=9)
    O = upload(other)
    osrc = gg.giant_sources(other, 12)[0]
    got, stop = [], threading.Event()

    def solver():
        k = 0
        while not stop.is_set() or k < 12:
            s = int(osrc[k % 12])
            got.append((s, gpu_solve(O, s, pred=False)[0]))
            gpu_solve(Gs[0], 0, pred=False)
            k += 1

    srv = S.sssp_serve_create()
    th = threading.Thread(target=solver)
    th.start()
    try:
        for rnd in range(2):
            jobs = []
            for gi, g in enumerate(graphs):
                for q, s in enumerate(gg.giant_sources(g, 45, seed=rnd)[0]):
                    host, pred = q % 5 == 4, q % 3 == 0
                    d = np.full(g.n, 7, np.uint32) if host else torch.empty(g.n, dtype=torch.int32, device="cuda")
                    p = None
                    if pred:
                        p = np.empty(g.n, np.int32) if host else torch.empty(g.n, dtype=torch.int32, device="cuda")
                    jobs.append((g, int(s), d, p, S.sssp_serve_submit(srv, Gs[gi].handle, int(s), d, p)))
            cancelled = {j for j in range(0, len(jobs), 11) if S.sssp_serve_cancel(srv, jobs[j][4]) == S.SSSP_OK}
            for j, (g, s, d, p, t) in enumerate(jobs):
                st, code = S.sssp_serve_wait(srv, t, 60000)
                if j in cancelled:
                    assert st == S.Q_ERROR and code == S.SSSP_E_CANCELLED
                    continue
                assert st == S.Q_DONE, S.strerror(code)
                torch.cuda.synchronize()
                db = d if isinstance(d, np.ndarray) else d.cpu().numpy().view(np.uint32)
                pb = p if p is None or isinstance(p, np.ndarray) else p.cpu().numpy()
                assert_exact(g, s, db, pb)
    finally:
        stop.set()
        th.join()
        stats = S.sssp_serve_get_stats(srv)
        S.sssp_serve_destroy(srv)
    assert stats["completed"] + stats["cancelled"] == stats["submitted"] == 180
    for s, d in got[:12]:
        assert_exact(other, s, d)
    [G.close() for G in Gs + [O]]


def test_hops_of_a_warp():
    """Several hops a step: more improved vertices than a warp keeps, breadth
    first by several levels a step, and a batch of one block per query on a mesh
    whose bits just fit."""
    g = gg.grid(700, 3, 1, 3, seed=2)
    both(g, 900)
    star = gg.from_edges(4097, [(0, v, 1) for v in range(1, 4)] +
                         [(v, 4 * v + k, 1 + k % 2) for v in range(1, 1024) for k in range(4)], name="tree")
    both(star, 0)
    for g in (gg.grid(500, 333, 1, 9, seed=1), gg.road(300, 200, seed=3)):
        G = upload(g)
        lev = torch.empty(G.n, dtype=torch.int32, device="cuda")
        par = torch.empty(G.n, dtype=torch.int32, device="cuda")
        G.bfs(77, lev, par)
        torch.cuda.synchronize()
        unit = np.ones(g.m, np.uint32)
        ref = oracle.dijkstra_u32(g.row_ptr, g.col, unit, 77)
        np.testing.assert_array_equal(lev.cpu().numpy().view(np.uint32), ref)
        np.testing.assert_array_equal(par.cpu().numpy(), oracle.pred_canonical_u32(g.row_ptr, g.col, unit, 77, ref))
        G.close()
    g = gg.grid(600, 560, 1, 100, seed=4)   # 2^19 places: two blocks a query
    G = upload(g)
    srcs = (np.arange(160) * 1999).astype(np.int32)
    d, p = gpu_batch(G, srcs, pred=True)
    assert_exact_many(g, srcs[::16], d[::16], p[::16])
    G.close()


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 6000])
def test_layout_around_tiles(n):
    """Split layouts at the edges of the scan's tiles, with hubs at the ends,
    rows above and below the block's limit, and thresholds back and forth."""
    deg = np.arange(n) % 7
    deg[[0, n // 2, n - 1]] = 33, 2049, 700
    if n == 1:
        deg[:] = 0
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    m = int(rp[-1])
    rng = np.random.default_rng(n)
    g = gg.Graph("rows", n, m, rp, rng.integers(0, n, m).astype(np.int32), rng.integers(1, 50, m).astype(np.uint32), "u32")
    G = upload(g)
    for split in (32, 100, 2048, 1 << 20, 33):
        d, p = gpu_solve(G, n // 2, config=cfg(split_arcs=split))
        assert_exact(g, n // 2, d, p)
        assert G.features()["shadows"] == int(sum(-(-int(x) // split) for x in deg if x > split))
        d, p = gpu_solve(G, n // 2)
        assert_exact(g, n // 2, d, p)
    G.close()


def symmetric(n, u, v, w, wtype="u32"):
    key, at = np.unique(np.concatenate([u * n + v, v * n + u]), return_index=True)
    w2 = np.concatenate([w, w])[at]
    # one weight for both directions of a repeated pair: that of the smaller arc
    lo, hi = np.minimum(key // n, key % n), np.maximum(key // n, key % n)
    order = np.lexsort((key, hi, lo))
    first = np.concatenate([[True], (lo[order][1:] != lo[order][:-1]) | (hi[order][1:] != hi[order][:-1])])
    w2[order] = w2[order][np.flatnonzero(first)[np.cumsum(first) - 1]]
    rp = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]).astype(np.int32)
    return gg.Graph("sym", n, len(key), rp, (key % n).astype(np.int32), w2, wtype)


def hubs_and_leaves(n, hubs, arcs, lo, hi, seed, wtype="u32"):
    """A few hubs that reach everything, leaves and self-loops, weights lo..hi."""
    rng = np.random.default_rng(seed)
    u = np.concatenate([rng.integers(0, hubs, arcs), np.arange(n), np.arange(0, n, 97)])
    v = np.concatenate([rng.integers(0, n, arcs), rng.integers(0, n, n), np.arange(0, n, 97)])
    w = rng.integers(lo, hi + 1, len(u))
    w = (w / 64.0).astype(np.float32) if wtype == "f32" else w.astype(np.uint32)
    return symmetric(n, u.astype(np.int64), v.astype(np.int64), w, wtype)


@pytest.mark.parametrize("wtype", ["u32", "f32"])
@pytest.mark.parametrize("lo,hi", [(1, 255), (0, 255), (1, 9), (7, 7), (200, 255)])
def test_core_and_pull(wtype, lo, hi):
    """Symmetric graphs with hubs: heavy arcs left out and pulled, or relaxed
    after all where the core does not settle; no light arcs; sources in the
    core, at its edge, and alone."""
    g = hubs_and_leaves(60_000, 40, 400_000, lo, hi, seed=hi + lo, wtype=wtype)
    G = upload(g)
    deg = np.diff(g.row_ptr)
    for src in (0, int(np.argmax(deg)), int(np.argmin(deg)), 59_999):
        d, p = gpu_solve(G, src, pred=True)
        assert_exact(g, src, d, p)
        d2, _ = gpu_solve(G, src, pred=False)
        np.testing.assert_array_equal(d2, d)
    G.close()


def test_core_needs_symmetry():
    """One arc, one weight or one order that spoils the symmetry, parallel arcs,
    and lengths that saturate: the same answers as ever."""
    g = hubs_and_leaves(50_000, 30, 400_000, 1, 255, seed=1)
    src = 12345
    variants = []
    for k in range(5):
        rp, col, w = g.row_ptr.copy(), g.col.copy(), g.w.copy()
        e = int(rp[40_000])
        if k == 0:
            w[e] = 1 + (int(w[e]) + 7) % 255
        elif k == 1:
            col[e] = (int(col[e]) + 1) % g.n
        elif k == 2:
            hub = int(np.argmax(np.diff(rp)))
            a, b = int(rp[hub]), int(rp[hub + 1])
            col[a:b], w[a:b] = col[a:b][::-1].copy(), w[a:b][::-1].copy()
        elif k == 3:
            col[e + 1], w[e + 1] = col[e], w[e]
        else:
            w[:] = w * 0x1000000 + 0x00FFFFFF
        variants.append(gg.Graph("v%d" % k, g.n, g.m, rp, col, w, "u32"))
    for h in variants:
        G = upload(h)
        d, p = gpu_solve(G, src, pred=True)
        assert_exact(h, src, d, p)
        G.close()


@pytest.mark.parametrize("wtype,lo,hi", [("u32", 1, 255), ("u32", 0, 255), ("u32", 1, 15), ("f32", 1, 255)])
@pytest.mark.parametrize("nq", [12, 33])
def test_batch_core_and_pull(wtype, lo, hi, nq):
    """Side by side on symmetric graphs with hubs: rows with one arc and none,
    a component apart, sources in the core, at its edge and alone."""
    g = hubs_and_leaves(70_000, 60, 300_000, lo, hi, seed=3, wtype=wtype)
    keep = g.n + 100                        # more vertices: some without arcs, some apart
    rp = np.concatenate([g.row_ptr, np.full(100, g.m, np.int32)])
    rp[g.n + 60:] += 2
    rp[g.n + 59] += 1
    col = np.concatenate([g.col, [g.n + 59, g.n + 58]]).astype(np.int32)
    w = np.concatenate([g.w, g.w[:1], g.w[:1]])
    h = gg.Graph("apart", keep, len(col), rp, col, w, wtype)
    G = upload(h)
    deg = np.diff(h.row_ptr)
    srcs = np.concatenate([[np.argmax(deg), g.n + 58, g.n + 59, g.n + 5, 0, 69_999],
                           np.random.default_rng(4).integers(0, g.n, nq - 6)]).astype(np.int32)
    d, p = gpu_batch(G, srcs, pred=True)
    assert_exact_many(h, srcs, d, p)
    d2, _ = gpu_batch(G, srcs, pred=False)
    np.testing.assert_array_equal(d2, d)
    G.close()


@pytest.mark.parametrize("kind", ["leaves", "star", "rmat", "apart", "directed"])
def test_levels_pulled(kind):
    """Wide levels on symmetric graphs with hubs (and on one that is not
    symmetric): rows beyond a warp's, self-loops, leaves, vertices without
    arcs, a component apart; with and without parents."""
    if kind == "star":
        n = 600_000
        leaf = np.arange(1, n)
        g = symmetric(n, np.zeros(n - 1, np.int64), leaf, np.ones(n - 1, np.uint32))
        srcs = (0, 1, n - 1)
    elif kind == "rmat":
        g = gg.rmat(17, 16, seed=5)
        srcs = [int(x) for x in gg.giant_sources(g, 3)[0]] + [int(np.flatnonzero(np.diff(g.row_ptr) == 0)[0])]
    else:
        g = hubs_and_leaves(90_000, 20, 500_000, 1, 99, seed=6)
        if kind == "apart":
            e = np.arange(g.n, g.n + 300_000, 2)
            rp = np.concatenate([g.row_ptr, g.m + 1 + np.arange(300_000)]).astype(np.int32)
            col = np.concatenate([g.col, np.stack([e + 1, e], 1).ravel()]).astype(np.int32)
            g = gg.Graph("apart", g.n + 300_000, len(col), rp, col, np.concatenate([g.w, np.ones(300_000, np.uint32)]), "u32")
        if kind == "directed":
            col = g.col.copy()
            col[::1001] = (col[::1001] + 1) % g.n
            g = gg.Graph("directed", g.n, g.m, g.row_ptr, col, g.w, "u32")
        srcs = (0, int(np.argmax(np.diff(g.row_ptr))), 77_777, g.n - 1)
    G = upload(g)
    unit = np.ones(g.m, np.uint32)
    for src in srcs:
        lev = torch.empty(G.n, dtype=torch.int32, device="cuda")
        par = torch.empty(G.n, dtype=torch.int32, device="cuda")
        G.bfs(src, lev, par)
        torch.cuda.synchronize()
        ref = oracle.dijkstra_u32(g.row_ptr, g.col, unit, src)
        np.testing.assert_array_equal(lev.cpu().numpy().view(np.uint32), ref)
        np.testing.assert_array_equal(par.cpu().numpy(), oracle.pred_canonical_u32(g.row_ptr, g.col, unit, src, ref))
        lev2 = torch.empty(G.n, dtype=torch.int32, device="cuda")
        G.bfs(src, lev2, None)
        torch.cuda.synchronize()
        assert torch.equal(lev, lev2)
    G.close()


@pytest.mark.parametrize("n", [33, 5000, 1_100_000])
@pytest.mark.parametrize("wtype", ["u32", "f32"])
def test_thin_rows_around_four(n, wtype):
    """Meshes whose rows have none to nine arcs, four of them at a fixed place:
    one cluster and the whole grid, one query and a batch, levels."""
    rng = np.random.default_rng(n)
    deg = np.where(rng.random(n) < 0.9, 4, rng.integers(0, 10, n))
    deg[[0, n - 1]] = 5, 9
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    m = int(rp[-1])
    u = np.repeat(np.arange(n), deg)
    col = ((u + rng.choice([-40, -2, -1, 1, 3, 40], m)) % n).astype(np.int32)
    w = rng.integers(1, 60, m)
    g = gg.Graph("mesh", n, m, rp, col, (w / 8.0).astype(np.float32) if wtype == "f32" else w.astype(np.uint32), wtype)
    both(g, n // 2)
    G = upload(g)
    srcs = np.array([0, n - 1, n // 3], np.int32)
    if n <= 5000:
        d, p = gpu_batch(G, srcs, pred=True)
        assert_exact_many(g, srcs, d, p)
    lev = torch.empty(n, dtype=torch.int32, device="cuda")
    G.bfs(0, lev, None)
    torch.cuda.synchronize()
    ref = oracle.dijkstra_u32(rp, col, np.ones(m, np.uint32), 0)
    np.testing.assert_array_equal(lev.cpu().numpy().view(np.uint32), ref)
    G.close()


@pytest.mark.parametrize("slice_us", [1000, 100])
@pytest.mark.parametrize("kind", ["grid", "ring"])
def test_served_meshes(kind, slice_us):
    """Meshes of more than 2^19 arcs: as jobs, and in slices where the server
    asks for short ones; a random graph of equal degrees, whose front is wide."""
    if kind == "grid":
        g = gg.grid(401, 390, 1, 100, seed=2)
    else:
        rng = np.random.default_rng(5)
        n, k = 150_000, 4
        col = np.concatenate([rng.permutation(n) for _ in range(k)]).reshape(k, n).T.ravel().astype(np.int32)
        g = gg.Graph("ring", n, n * k, (np.arange(n + 1) * k).astype(np.int32), col,
                     rng.integers(1, 100, n * k).astype(np.uint32), "u32")
    assert g.m > 1 << 19
    G = upload(g)
    srcs = [0, 77, g.n - 1, g.n // 2, 77]
    srv = S.sssp_serve_create(slice_us=slice_us)
    try:
        d = torch.empty((len(srcs), g.n), dtype=torch.int32, device="cuda")
        p = torch.empty((len(srcs), g.n), dtype=torch.int32, device="cuda")
        tickets = [S.sssp_serve_submit(srv, G.handle, s, d[i], p[i]) for i, s in enumerate(srcs)]
        for t in tickets:
            assert S.sssp_serve_wait(srv, t, 60000)[0] == S.Q_DONE
    finally:
        S.sssp_serve_destroy(srv)
    assert_exact_many(g, np.array(srcs), d.cpu().numpy().view(np.uint32), p.cpu().numpy())
    G.close()


def test_batches_on_large_meshes():
    """A cluster per query on a mesh of more than 2^21 arcs, and one by one
    beyond a cluster's vertices; a random graph of equal degrees starts over."""
    g = gg.grid(760, 740, 1, 50, seed=3)
    assert g.m > 1 << 21
    srcs = np.arange(15) * 37_000
    G = upload(g)
    d, p = gpu_batch(G, srcs, pred=True)
    assert_exact_many(g, srcs, d, p)
    G.close()
    rng = np.random.default_rng(5)
    n, k = 560_000, 4
    col = np.concatenate([rng.permutation(n) for _ in range(k)]).reshape(k, n).T.ravel().astype(np.int32)
    w = rng.integers(1, 100, n * k).astype(np.uint32)
    h = gg.Graph("regular", n, n * k, (np.arange(n + 1) * k).astype(np.int32), col, w, "u32")
    G = upload(h)
    for _ in range(2):
        d, p = gpu_batch(G, srcs, pred=True)
        assert_exact_many(h, srcs, d, p)
    G.close()
    big = gg.grid(1100, 1000, 1, 50, seed=4)
    G = upload(big)
    d, _ = gpu_batch(G, srcs, pred=False)
    assert_exact_many(big, srcs, d, None)
    G.close()
