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
