"""Graphs with as many arcs as a row offset can number (2^31 - 1): the last
rows end where a signed index past them would wrap."""
import numpy as np
import pytest
import torch

import paper_2602_10080_gb300 as S

pytestmark = pytest.mark.gpu

N = 1 << 21
M = (1 << 31) - 1
TAIL = 64


@pytest.fixture(scope="module")
def big():
    """Rows of 1024 arcs of weight 100 (the last one of 1023), the last 64 of
    which alone lead to the vertices N - 128 .. N - 65, with weight 7."""
    S.build()
    S.lib()
    rp = (torch.arange(N + 1, dtype=torch.int64, device="cuda") * 1024).clamp(max=M).to(torch.int32)
    arcs = torch.empty((M, 2), dtype=torch.int32, device="cuda")
    step = 1 << 25
    for a in range(0, M, step):
        e = torch.arange(a, min(M, a + step), dtype=torch.int64, device="cuda")
        c = ((e * 2654435761) >> 13) % (N - 64)
        arcs[a:a + len(e), 0] = torch.where(c >= N - 128, c + 64, c).to(torch.int32)
    arcs[:, 1] = 100
    arcs[M - TAIL:, 0] = torch.arange(N - 128, N - 64, dtype=torch.int32, device="cuda")
    arcs[M - TAIL:, 1] = 7
    torch.cuda.synchronize()
    yield rp, arcs


def expected(arcs, src):
    """Dijkstra by distance: all vertices of the next one at once."""
    inf = 1 << 40
    dist = torch.full((N,), inf, dtype=torch.int64, device="cuda")
    dist[src] = 0
    now = -1
    while True:
        open_ = dist[dist > now]
        now = int(open_.min()) if len(open_) else inf
        if now == inf:
            break
        front = (dist == now).nonzero()[:, 0]
        hit = torch.zeros(N, dtype=torch.bool, device="cuda")
        for part in front[front != N - 1].split(1 << 15):
            rows = (part[:, None] * 1024 + torch.arange(1024, device="cuda")[None]).reshape(-1)
            hit[arcs[rows, 0].long()] = True
        if (front == N - 1).any():
            hit[arcs[(N - 1) * 1024:M - TAIL, 0].long()] = True
            dist[N - 128:N - 64] = dist[N - 128:N - 64].clamp(max=now + 7)
        dist = torch.where(hit, dist.clamp(max=now + 100), dist)
    assert int(dist.max()) < inf
    return dist.to(torch.int32)


def check(arcs, src, d, p=None):
    ref = expected(arcs, src)
    assert torch.equal(d, ref)
    if p is not None:
        assert (p[N - 128:N - 64] == N - 1).all() and p[src] == src


def test_noalloc_with_the_most_arcs(big):
    rp, arcs = big
    d = torch.empty(N, dtype=torch.int32, device="cuda")
    p = torch.empty(N, dtype=torch.int32, device="cuda")
    for src in (5, N - 1):
        S.sssp_solve_noalloc(rp, arcs, N, M, S.SSSP_W_U32, src, d, p)
        torch.cuda.synchronize()
        check(arcs, src, d, p)


def test_graph_with_the_most_arcs(big):
    """One query, a batch side by side and levels on a graph handle."""
    rp, arcs = big
    col, w = arcs[:, 0].contiguous(), arcs[:, 1].contiguous()
    torch.cuda.synchronize()   # creation reads them on a stream of its own
    G = S.Graph(rp, col, w, "u32")
    del col, w
    d = torch.empty(N, dtype=torch.int32, device="cuda")
    p = torch.empty(N, dtype=torch.int32, device="cuda")
    G.solve(77, d, p)
    torch.cuda.synchronize()
    check(arcs, 77, d, p)
    srcs = np.arange(9, dtype=np.int32) * 200_000 + 1
    db = torch.empty((9, N), dtype=torch.int32, device="cuda")
    G.solve_batch(torch.from_numpy(srcs).cuda(), db)
    torch.cuda.synchronize()
    for q in (0, 8):
        check(arcs, int(srcs[q]), db[q])
    G.bfs(77, d, p)
    torch.cuda.synchronize()
    dist = expected(arcs, 77)
    far = torch.arange(N, device="cuda")
    far = (far >= N - 128) & (far < N - 64)
    assert int(dist[~far].max()) == 300   # so every length of these is 100 a level
    assert torch.equal(d[~far], dist[~far] // 100)
    assert (d[far] == d[N - 1] + 1).all() and (p[far] == N - 1).all()
    G.close()
