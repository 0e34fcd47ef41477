"""The server's slices on graphs that run as jobs by default: a time limit per
query, however long, keeps its lanes in slices."""
import time

import numpy as np
import pytest
import torch

import graphgen as gg
import paper_2602_10080_gb300 as S
from gpu_util import assert_exact, assert_exact_many, upload
from test_zz_no_alloc import _interleave, _spreader_graph

pytestmark = pytest.mark.gpu

LONG_MS = 600_000


@pytest.fixture(scope="module", autouse=True)
def _built():
    S.build()
    S.lib()


def test_a_lane_grows_while_queries_run():
    """More queries than a lane's first eight slots."""
    g = gg.grid(128, 128, 1, 100, seed=1)
    G = upload(g)
    srcs = gg.giant_sources(g, 40, seed=4)[0]
    srv = S.sssp_serve_create(slice_us=150, max_slots=64, query_timeout_ms=LONG_MS)
    try:
        d = torch.empty((40, g.n), dtype=torch.int32, device="cuda")
        ts = []
        for k, s in enumerate(srcs):
            ts.append(S.sssp_serve_submit(srv, G.handle, int(s), d[k], None))
            if k % 10 == 9:
                time.sleep(0.001)
        assert all(S.sssp_serve_wait(srv, t)[0] == S.Q_DONE for t in ts)
        st = S.sssp_serve_get_stats(srv)
    finally:
        S.sssp_serve_destroy(srv)
    assert st["max_resident"] > 8 and st["slices"] > 4, st
    assert_exact_many(g, srcs, d.cpu().numpy().view(np.uint32))
    G.close()


def test_lanes_of_different_graphs_in_slices():
    """Queries of four graphs and both kinds, admitted while others run."""
    gs = [gg.road(384, 384, 0.05, 0.005, 32, 1, 1000, 20, seed=1), gg.grid(128, 128, 1, 100, seed=1),
          gg.rmat(15, 16, lo=1, hi=255, seed=1), gg.erdos_renyi(1 << 14, 1 << 17, seed=5, wtype="f32")]
    Gs = [upload(g) for g in gs]
    srv = S.sssp_serve_create(slice_us=200, query_timeout_ms=LONG_MS)
    out = []
    try:
        for i, (g, G) in enumerate(zip(gs, Gs)):
            for k, s in enumerate(gg.giant_sources(g, 6, seed=2)[0]):
                d = torch.empty(g.n, dtype=torch.int32, device="cuda")
                p = np.empty(g.n, np.int32) if k % 2 == 0 else None
                out.append((g, int(s), d, p, S.sssp_serve_submit(srv, G.handle, int(s), d, p)))
                if len(out) in (1, 4, 10):
                    time.sleep(0.004)
        assert all(S.sssp_serve_wait(srv, o[4])[0] == S.Q_DONE for o in out)
        st = S.sssp_serve_get_stats(srv)
    finally:
        S.sssp_serve_destroy(srv)
    assert st["joined_running"] >= 1 and st["max_resident"] >= 2, st
    torch.cuda.synchronize()
    for g, s, d, p, _ in out:
        assert_exact(g, s, d.cpu().numpy().view(np.uint32), p)
    [G.close() for G in Gs]


def test_the_fixed_scratch_has_no_queue_to_overflow():
    """Two million vertices that wait at once: solved, with and without
    predecessors."""
    g = _spreader_graph()
    rp = torch.from_numpy(g.row_ptr).cuda()
    arcs = _interleave(g)
    d = torch.empty(g.n, dtype=torch.int32, device="cuda")
    p = torch.empty(g.n, dtype=torch.int32, device="cuda")
    for pred in (p, None):
        S.sssp_solve_noalloc(rp, arcs, g.n, g.m, S.SSSP_W_U32, 0, d, pred)
        torch.cuda.synchronize()
        assert_exact(g, 0, d.cpu().numpy().view(np.uint32), None if pred is None else p.cpu().numpy())
