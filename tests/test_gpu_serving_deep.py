"""Served searches of many levels: more than a launch runs (1,024), ended by a call for a query that comes in, resumed
with other lanes beside them; directed graphs; a server closed over a running search."""
import time

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("symmetrize", [True, False])
@pytest.mark.parametrize("max_lanes", [2, 64])
def test_deep_search_beside_short_ones(symmetrize, max_lanes):
    from paper_1208_5542_gb300 import bfs
    depth, fan = 6000, 700
    rng = np.random.default_rng(2)
    # a path, and beside it a random graph with a hub
    src = np.concatenate([np.arange(depth - 1), depth + rng.integers(0, fan, 4 * fan), np.full(fan, depth)])
    dst = np.concatenate([np.arange(1, depth), depth + rng.integers(0, fan, 4 * fan), depth + np.arange(fan)])
    n = depth + fan
    src, dst = src.astype(np.int32), dst.astype(np.int32)
    go = oracle.csr(n, src, dst, symmetrize=symmetrize)
    g = bfs.Graph.from_edges(n, src, dst, symmetrize=symmetrize, p=3)
    srv = bfs.Server(1 << 30, max_lanes)
    gid = srv.add_graph(g)
    queries = [(0, True), (depth // 2, False)]
    tickets = [srv.submit(gid, r, parents=p) for r, p in queries]
    for k in range(12):                                     # come in while the path is being walked
        time.sleep(0.004)
        queries.append((int(depth + rng.integers(0, fan)) if k % 3 else int(rng.integers(0, depth)), k % 2 == 0))
        tickets.append(srv.submit(gid, queries[-1][0], parents=queries[-1][1]))
    for (r, p), t in reversed(list(zip(queries, tickets))):
        got = srv.wait(t, n, parents=p)
        lv, pa = oracle.bfs(go, r)
        assert ((got[0] if p else got).cpu().numpy() == lv).all(), r
        assert not p or (got[1].cpu().numpy() == pa).all(), r
    assert srv.stats()["iterations"] >= depth and srv.stats()["completed"] == len(queries)
    srv.close()
    g.run(0)


def test_close_over_a_running_search():
    from paper_1208_5542_gb300 import bfs
    n = 300_000                                             # some seconds of levels
    i = np.arange(n - 1, dtype=np.int32)
    g = bfs.Graph.from_edges(n, i, i + 1, p=2)
    for wait in (0.0, 0.003, 0.05):
        srv = bfs.Server(1 << 30, 4)
        gid = srv.add_graph(g)
        srv.submit(gid, 0, parents=True)
        srv.submit(gid, n // 2)
        time.sleep(wait)
        t0 = time.perf_counter()
        srv.close()
        assert time.perf_counter() - t0 < 2.0
