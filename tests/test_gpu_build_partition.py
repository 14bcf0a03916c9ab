"""The partitioned graph build (graphs whose counts and entries outgrow L2) on a GB300 against the oracle:
directories, degrees (through the entries a search scans), levels and smallest parents."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

M = 3_000_000          # tuples; every graph's p * n counts are above the direct build's limit (12.6M)


def tuples(kind, n, m):
    rng = np.random.default_rng(n)
    if kind == "kronecker":
        _, src, dst = graphgen.edges(24, 16, seed=3, m=m)
        return (src.astype(np.int64) * n >> 24).astype(np.int32), (dst.astype(np.int64) * n >> 24).astype(np.int32)
    src, dst = graphgen.random_edges(n, m, seed=n)
    if kind == "hub":                       # one column holds a third of the entries, another only self-loops
        src[::3] = n - 1
        src[1:1000:3] = dst[1:1000:3] = n // 2
    return src, dst


@pytest.mark.parametrize("kind,n,p,symmetrize", [
    ("kronecker", 1 << 21, 8, True), ("kronecker", 13_000_003, 1, True), ("kronecker", 4_200_003, 3, False),
    ("uniform", 6_300_673, 2, True),        # a last part of one column beyond whole shared-memory windows
    ("uniform", 400_000, 32, True), ("uniform", 17_000_003, 32, True),   # ... several windows per bucket
    ("uniform", 400_000, 33, True),         # grids above 32 x 32: the direct build
    ("hub", 1_800_001, 7, True)])
def test_partitioned_build(kind, n, p, symmetrize):
    import torch
    from paper_1208_5542_gb300 import bfs
    src, dst = tuples(kind, n, M if symmetrize else 2 * M)
    go = oracle.csr(n, src, dst, symmetrize=symmetrize)
    g = bfs.Graph.from_edges(n, src, dst, symmetrize=symmetrize, p=p)
    assert g.n_entries == len(go.col)
    pairs = [(i, j) for i in range(p) for j in range(p)]
    for i, j in pairs if p <= 8 else pairs[:: p + 2]:
        want = oracle.pack_bits(oracle.directory(go, p, i, j))
        assert (g.directory(i, j).cpu().numpy().view(np.uint32) == want).all(), (i, j)
    deg = np.diff(go.row_ptr)
    for root in (int(src[0]), int(dst[-1])):
        lv, pa = oracle.bfs(go, root)
        parent, level, st = g.run(root, stats=True)
        torch.cuda.synchronize()
        assert (level.cpu().numpy() == lv).all() and (parent.cpu().numpy() == pa).all()
        assert sum(v["edges_scanned"] for v in st.levels) == int(deg[lv >= 0].sum())


@pytest.mark.parametrize("bad", [-1, 6_300_673, 2**31 - 1])
def test_partitioned_build_rejects_ids(bad):
    from paper_1208_5542_gb300 import bfs
    from paper_1208_5542_gb300.native import BfsError
    src, dst = tuples("uniform", 6_300_673, M)
    dst[M // 2] = bad
    with pytest.raises(BfsError, match="INVALID_ARG"):
        bfs.Graph.from_edges(6_300_673, src, dst, p=2)
