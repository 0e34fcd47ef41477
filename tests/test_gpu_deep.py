"""Batches and served queries on graphs of many steps: side by side gives up,
a few queries are taken in turn, and many by the queue engine."""
import numpy as np
import pytest
import torch

import graphgen as gg
import paper_2602_10080_gb300 as S
from gpu_util import assert_exact, assert_exact_many, gpu_batch, gpu_solve, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    S.build()
    S.lib()


def by_queues(G):
    return G.stats()["pops_l2"] > 0


def with_chain(hops, wtype="u32"):
    """A power-law graph, from whose last vertex a chain of `hops` arcs leads."""
    g = gg.rmat(13, 24, seed=3, wtype=wtype)
    n = g.n + hops
    rp = np.concatenate([g.row_ptr[:-1], g.m + 1 + np.arange(hops), [g.m + hops]]).astype(np.int32)
    col = np.concatenate([g.col, np.arange(g.n, n)]).astype(np.int32)
    w = np.concatenate([g.w, np.full(hops, 3, g.w.dtype)])
    return gg.Graph("chain", n, g.m + hops, rp, col, w, wtype)


def eight(W, H, seed=1):
    """A W x H grid with eight neighbours a vertex."""
    i = np.arange(W * H).reshape(H, W)
    e = [(i[:, :-1], i[:, 1:]), (i[:-1], i[1:]), (i[:-1, :-1], i[1:, 1:]), (i[:-1, 1:], i[1:, :-1])]
    u = np.concatenate([a.ravel() for a, _ in e] + [b.ravel() for _, b in e])
    v = np.concatenate([b.ravel() for _, b in e] + [a.ravel() for a, _ in e])
    w = np.random.default_rng(seed).integers(1, 100, len(u) // 2).astype(np.uint32)
    o = np.argsort(u, kind="stable")
    rp = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=W * H))]).astype(np.int32)
    return gg.Graph("eight", W * H, len(u), rp, v[o].astype(np.int32), np.concatenate([w, w])[o], "u32")


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("nq", [8, 12, 40])
@pytest.mark.parametrize("hops", [40, 300, *range(762, 769), 2000])
def test_chains_around_the_limit(hops, nq, host):
    """Up to the limit the batch stays side by side; beyond, the first query
    in turn shows how many steps there are and the queues take the others."""
    g = with_chain(hops)
    G = upload(g)
    srcs = gg.giant_sources(g, nq)[0]
    srcs[nq - 1] = g.n - hops - 1
    for _ in range(2):
        d, p = gpu_batch(G, srcs, pred=True, host=host)
        assert_exact_many(g, srcs, d, p)
        if hops <= 300:   # a tail
            assert not by_queues(G)
        d, _ = gpu_batch(G, srcs, pred=False, host=host)
        assert_exact_many(g, srcs, d)
    if hops == 2000:
        d, p = gpu_solve(G, int(srcs[nq - 1]))
        assert_exact(g, int(srcs[nq - 1]), d, p)
        d, p = gpu_batch(G, srcs, pred=True, host=host)
        assert by_queues(G)
        assert_exact_many(g, srcs, d, p)
        d, p = gpu_batch(G, srcs[-3:], pred=True, host=host)
        assert not by_queues(G)
        assert_exact_many(g, srcs[-3:], d, p)
    G.close()


def test_chain_with_real_lengths():
    g = with_chain(1500, "f32")
    G = upload(g)
    srcs = gg.giant_sources(g, 20)[0]
    srcs[3] = g.n - 1501
    for _ in range(2):
        d, _ = gpu_batch(G, srcs, pred=False)
        assert_exact_many(g, srcs, d)
    G.close()


def test_wide_meshes():
    """A grid with eight neighbours: the queues take a batch, from its second
    query on if nothing is known, and the wavefront one query and a few."""
    g = eight(560, 520)
    assert g.m > 1 << 21
    srcs = (np.arange(20) * 14_001).astype(np.int32)
    G = upload(g)
    for nq in (6, 20, 20):
        d, p = gpu_batch(G, srcs[:nq], pred=True)
        assert by_queues(G)
        assert_exact_many(g, srcs[:nq], d, p)
    for nq in (1, 3):
        d, p = gpu_batch(G, srcs[:nq], pred=True)
        assert not by_queues(G)
        assert_exact_many(g, srcs[:nq], d, p)
    G.close()


def test_thin_meshes_too_large_for_a_cluster():
    """In turn up to eight queries, by the queues above."""
    g = gg.grid(1500, 1410, 1, 100, seed=2)
    assert g.n > 1 << 21
    srcs = (np.arange(12) * 171_717).astype(np.int32)
    G = upload(g)
    for nq, queues in ((8, False), (12, True)):
        d, _ = gpu_batch(G, srcs[:nq], pred=False)
        assert by_queues(G) == queues
        assert_exact_many(g, srcs[:nq], d)
    G.close()


@pytest.mark.parametrize("pred", [False, True])
def test_served_on_wide_meshes(pred):
    """Many at once: a job side by side gives up, one shows the steps, slices
    take the others; then a few again, one by one."""
    g = eight(560, 520, seed=4)
    G = upload(g)
    srcs = (np.arange(40) * 7001).astype(np.int32)
    srv = S.sssp_serve_create()
    try:
        for burst in (srcs, srcs[:2], srcs[:30]):
            d = torch.empty((len(burst), g.n), dtype=torch.int32, device="cuda")
            p = torch.empty((len(burst), g.n), dtype=torch.int32, device="cuda") if pred else None
            ts = [S.sssp_serve_submit(srv, G.handle, int(s), d[i], p[i] if pred else None) for i, s in enumerate(burst)]
            for t in ts:
                assert S.sssp_serve_wait(srv, t, 60000)[0] == S.Q_DONE
            torch.cuda.synchronize()
            few = slice(None, None, 7)
            assert_exact_many(g, burst[few], d.cpu().numpy().view(np.uint32)[few],
                              p.cpu().numpy()[few] if pred else None)
    finally:
        S.sssp_serve_destroy(srv)
    G.close()
