"""Batched searches whose levels run from either side, against the oracle: levels, smallest parents and the
entries of the active vertices, with columns around the length at which a warp takes over from a lane."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def graph(kind, n):
    if kind == "kronecker":
        k = (n - 1).bit_length()
        _, src, dst = graphgen.edges(k, 12, seed=11)
        return (src.astype(np.int64) * n >> k).astype(np.int32), (dst.astype(np.int64) * n >> k).astype(np.int32)
    if kind == "uniform":
        return graphgen.random_edges(n, 16 * n, seed=n)
    # every vertex with one column of 30 .. 36 entries into the low ids, hubs beyond a piece there
    rng = np.random.default_rng(n)
    lens = rng.integers(30, 37, n)
    src = np.repeat(np.arange(n), lens).astype(np.int32)
    return src, rng.integers(0, 64, len(src)).astype(np.int32)


@pytest.mark.parametrize("symmetrize", [True, False])
@pytest.mark.parametrize("lanes", [1, 33, 64])
@pytest.mark.parametrize("kind,n,p", [("kronecker", 9001, 3), ("uniform", 6000, 1), ("uniform", 5003, 7), ("short", 3000, 2)])
def test_batch_against_oracle(kind, n, p, lanes, symmetrize):
    from paper_1208_5542_gb300 import bfs
    src, dst = graph(kind, n)
    go = oracle.csr(n, src, dst, symmetrize=symmetrize)
    deg = np.diff(go.row_ptr)
    roots = np.random.default_rng(lanes).choice(src, lanes).astype(np.int32)
    want = [oracle.bfs(go, int(r)) for r in roots]
    g = bfs.Graph.from_edges(n, src, dst, symmetrize=symmetrize, p=p)
    for parents in (False, True):
        lv, pa, st = g.run_batch(roots, parents=parents)
        lv = lv.cpu().numpy()
        for r in range(lanes):
            assert (lv[r] == want[r][0]).all(), r
            if parents:
                assert (pa[r].cpu().numpy() == want[r][1]).all(), r
        active = sum(int(deg[(lv == k).any(axis=0)].sum()) for k in range(lv.max() + 1))
        assert st["edges_scanned"] == active and st["n_levels"] == lv.max() + 1
