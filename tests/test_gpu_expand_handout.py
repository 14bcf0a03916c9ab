"""Dense levels without a row window that have more units than four per warp: handed out two at a time, against the
oracle (a fine grid makes the units of a small graph)."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,rows,word_bits", [(0, False, 32), (1, False, 32), (1, False, 64), (2, False, 32),
                                                 (2, True, 32), (2, True, 64)])
@pytest.mark.parametrize("n,p,symmetrize", [(900_001, 33, True), (1_300_000, 40, False)])
def test_many_units_without_a_window(n, p, symmetrize, mode, rows, word_bits):
    import torch
    from paper_1208_5542_gb300 import bfs
    src, dst = graphgen.random_edges(n, 12 * n, seed=p)
    go = oracle.csr(n, src, dst, symmetrize=symmetrize)
    root = int(src[0])
    lv, pa = oracle.bfs(go, root)
    # the widest level: a vertex in nearly every group of every slot, more units than 4 x 152 x 32
    assert np.bincount(lv[lv >= 0]).max() > n // 2 and p * n // (64 * 32) > 4 * 152 * 32 * 0.7
    g = bfs.Graph.from_edges(n, src, dst, symmetrize=symmetrize, p=p, mode=mode, wah_bits=word_bits)
    g.set_row_exchange(rows)
    parent, level, _ = g.run(root)
    assert (level.cpu().numpy() == lv).all() and (parent.cpu().numpy() == pa).all()
    _, _, st = g.run(root, parent, level, stats=True)
    torch.cuda.synchronize()
    assert (level.cpu().numpy() == lv).all() and (parent.cpu().numpy() == pa).all()
    deg = np.diff(go.row_ptr)
    assert sum(v["edges_scanned"] for v in st.levels) == int(deg[lv >= 0].sum())
