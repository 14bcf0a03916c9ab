"""The expansion's dispatch on a GB300 against the oracle: units cut into parts, pieces of long columns at
every piece size, and the three kinds of row window (none, visited bits, visited and next bits)."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def check(n, src, dst, p, mode, rows, root, word_bits=32, symmetrize=True):
    import torch
    from paper_1208_5542_gb300 import bfs
    go = oracle.csr(n, src, dst, symmetrize=symmetrize)
    lv, pa = oracle.bfs(go, root)
    g = bfs.Graph.from_edges(n, src, dst, symmetrize=symmetrize, p=p, mode=mode, wah_bits=word_bits)
    g.set_row_exchange(rows)
    parent, level, _ = g.run(root)
    _, _, st = g.run(root, parent, level, stats=True)
    torch.cuda.synchronize()
    assert (level.cpu().numpy() == lv).all()
    assert (parent.cpu().numpy() == pa).all()
    deg = graphgen.degrees(n, src, dst) if symmetrize else np.bincount(src, minlength=n)
    # every entry of a reached vertex is scanned exactly once, however the units were cut
    assert sum(v["edges_scanned"] for v in st.levels) == int(deg[lv >= 0].sum())


@pytest.mark.parametrize("rows", [False, True])
@pytest.mark.parametrize("length", [31, 32, 33, 63, 64, 65, 511, 512, 513, 1024, 1025, 2048, 2049, 4097])
def test_column_lengths(length, rows):
    """A frontier of a few vertices whose columns have the lengths at which their path changes."""
    n, hubs = 6000, 37
    rng = np.random.default_rng(length)
    src = np.concatenate([np.zeros(hubs, np.int32)] +
                         [np.full(length, 1 + h, np.int32) for h in range(hubs)]).astype(np.int32)
    dst = np.concatenate([np.arange(1, hubs + 1)] +
                         [rng.integers(hubs + 1, n, length) for _ in range(hubs)]).astype(np.int32)
    check(n, src, dst, 1, 2, rows, 0, symmetrize=False)
    check(n, src, dst, 3, 2, rows, 0, symmetrize=False)


@pytest.mark.parametrize("mode,word_bits", [(0, 32), (1, 32), (1, 64), (2, 32), (2, 64)])
@pytest.mark.parametrize("n,p", [(33, 1), (1023, 2), (4096, 1), (4097, 2), (40000, 1), (70001, 3)])
def test_few_units(n, p, mode, word_bits):
    """Dense levels of a small graph: fewer units than warps, cut into parts of up to 32 items."""
    src, dst = graphgen.random_edges(n, 24 * n, seed=n)
    check(n, src, dst, p, mode, False, int(src[0]), word_bits)


@pytest.mark.parametrize("mode,rows", [(0, False), (2, False), (2, True)])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_window_kinds(p, mode, rows):
    """2.1M vertices, ranges that do not start at whole words: no window (p = 1), the visited bits (2), both (3)."""
    n = (1 << 21) + 77
    _, src, dst = graphgen.edges(21, 4, seed=5)
    src = (src.astype(np.int64) * n >> 21).astype(np.int32)
    dst = (dst.astype(np.int64) * n >> 21).astype(np.int32)
    check(n, src, dst, p, mode, rows, int(src[3]))
