"""Calls side by side from several threads: none changes what another one's
launch depends on, and all stay with the wavefront kernels."""
import threading

import numpy as np
import pytest
import torch

import graphgen as gg
import paper_2602_10080_gb300 as S
from gpu_util import oracle_dist, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    S.build()
    S.lib()


def in_threads(*fns):
    """Runs the functions at once; the first one's exception is raised."""
    errors = []

    def call(f):
        try:
            f()
        except BaseException as e:   # noqa: BLE001 -- handed to the caller
            errors.append(e)

    ts = [threading.Thread(target=call, args=(f,)) for f in fns]
    [t.start() for t in ts]
    [t.join() for t in ts]
    if errors:
        raise errors[0]


def by_wavefront(G):
    st = G.stats()
    return st["pops_l0"] + st["pops_l1"] + st["pops_l2"] + st["refill_tries"] == 0 and st["relax_arcs"] > 0


def test_clusters_of_different_sizes_at_once():
    """Small and large meshes run the same function with little and much shared
    memory, one of them with the fixed scratch."""
    gs = [gg.grid(1000, 900, 1, 100, seed=1), gg.grid(60, 61, 1, 100, seed=2), gg.grid(400, 390, 1, 100, seed=3)]
    Gs = [upload(g) for g in gs]
    refs = [oracle_dist(g, 7) for g in gs]
    rp = torch.from_numpy(gs[2].row_ptr).cuda()
    arcs = torch.from_numpy(np.stack([gs[2].col.view(np.uint32), gs[2].w_bits], 1).view(np.int32).copy()).cuda()

    def solves(i, count):
        st, d = torch.cuda.Stream(), torch.empty(gs[i].n, dtype=torch.int32, device="cuda")
        for _ in range(count):
            Gs[i].solve(7, d, None, None, st)
            assert by_wavefront(Gs[i]), i
        np.testing.assert_array_equal(d.cpu().numpy().view(np.uint32), refs[i])

    def noalloc():
        d = torch.empty(gs[2].n, dtype=torch.int32, device="cuda")
        for _ in range(60):
            S.sssp_solve_noalloc(rp, arcs, gs[2].n, gs[2].m, S.SSSP_W_U32, 7, d)
        np.testing.assert_array_equal(d.cpu().numpy().view(np.uint32), refs[2])

    in_threads(lambda: solves(0, 60), lambda: solves(1, 600), lambda: solves(1, 600), noalloc)
    [G.close() for G in Gs]


def test_a_lane_that_is_never_empty_leaves_the_grid_to_others():
    """One lane of a server always has queries waiting; queries of another
    graph, and of the same one without predecessors, are served in between."""
    a, b = gg.rmat(15, 24, seed=8, wtype="f32"), gg.rmat(15, 20, seed=9)
    A, B = upload(a), upload(b)
    total, served = 400, []
    srv = S.sssp_serve_create()
    started = threading.Event()

    def feed():
        d = torch.empty((4, a.n), dtype=torch.int32, device="cuda")
        p = torch.empty((4, a.n), dtype=torch.int32, device="cuda")
        open_ = [S.sssp_serve_submit(srv, A.handle, 7, d[i], p[i]) for i in range(4)]
        for k in range(total):
            t = open_.pop(0)
            assert S.sssp_serve_wait(srv, t)[0] == S.Q_DONE
            served.append(t)
            open_.append(S.sssp_serve_submit(srv, A.handle, 7, d[k % 4], p[k % 4]))
            if k == 20:
                started.set()
        assert all(S.sssp_serve_wait(srv, t)[0] == S.Q_DONE for t in open_)

    def others():
        started.wait()
        db = torch.empty(b.n, dtype=torch.int32, device="cuda")
        da = torch.empty(a.n, dtype=torch.int32, device="cuda")
        tb, ta = S.sssp_serve_submit(srv, B.handle, 3, db), S.sssp_serve_submit(srv, A.handle, 7, da)
        assert S.sssp_serve_wait(srv, tb)[0] == S.Q_DONE and S.sssp_serve_wait(srv, ta)[0] == S.Q_DONE
        assert len(served) < total // 2, len(served)
        np.testing.assert_array_equal(db.cpu().numpy().view(np.uint32), oracle_dist(b, 3))
        np.testing.assert_array_equal(da.cpu().numpy().view(np.uint32), oracle_dist(a, 7))

    try:
        in_threads(feed, others)
    finally:
        S.sssp_serve_destroy(srv)
    A.close()
    B.close()


def test_tuned_graphs_keep_the_faster_engine():
    """Both engines are timed warm: where the wavefront kernels are several times
    faster, a call without a configuration stays with them after tuning."""
    g = gg.rmat(17, 16, seed=4)
    srcs = gg.giant_sources(g, 40)[0]
    G = upload(g)
    G.autotune(srcs[:1], 150)
    d = torch.empty(40 * g.n, dtype=torch.int32, device="cuda")
    G.solve(int(srcs[0]), d)
    assert by_wavefront(G)
    G.autotune_batch(srcs, 150)
    G.solve_batch(srcs, d)
    assert by_wavefront(G)
    np.testing.assert_array_equal(d.cpu().numpy().view(np.uint32)[:g.n], oracle_dist(g, int(srcs[0])))
    G.close()
