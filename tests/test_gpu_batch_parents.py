"""Parents of batched searches whose levels run from the destinations' side, columns of many entries read by a whole
warp in several steps, for few and for all search lanes, on one and on several blocks; against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [1, 32, 33, 64])
@pytest.mark.parametrize("p", [1, 3])
def test_long_columns(p, lanes):
    from paper_1208_5542_gb300 import bfs
    n = 3000
    rng = np.random.default_rng(p)
    # every vertex has 1 .. 700 entries: columns around one and several steps of 128 beyond the first 32
    lens = rng.integers(1, 350, n)
    lens[:64] = [31, 32, 33, 34, 159, 160, 161, 162, 287, 288, 289, 290, 511, 512, 513, 700] * 4
    src = np.repeat(np.arange(n), lens).astype(np.int32)
    dst = rng.integers(0, n, len(src)).astype(np.int32)
    go = oracle.csr(n, src, dst)
    roots = rng.choice(n, lanes).astype(np.int32)
    g = bfs.Graph.from_edges(n, src, dst, p=p)
    lv, pa, _ = g.run_batch(roots, parents=True)
    for r in range(lanes):
        want = oracle.bfs(go, int(roots[r]))
        assert (lv[r].cpu().numpy() == want[0]).all() and (pa[r].cpu().numpy() == want[1]).all(), r
