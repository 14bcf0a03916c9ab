"""Short slots in small and in large numbers: column streams and row buffers, word for word against the oracle, on
either side of the slot counts at which the one-launch encoder hands over to the passes (152 SMs: 304 slots of more
than 1,024 groups, 1,216 shorter ones)."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [32, 64])
@pytest.mark.parametrize("p,groups", [(17, 1030), (18, 1030), (34, 130), (35, 130), (50, 5)])
def test_streams_around_the_slot_limit(p, groups, w):
    import torch
    from paper_1208_5542_gb300 import bfs
    nb = groups * (w - 1) + p % 9
    n = p * nb - 3
    src, dst = graphgen.random_edges(n, 2 * n, seed=p)
    rng = np.random.default_rng(p)
    src = np.concatenate([src, rng.integers(0, 500, 20_000)]).astype(np.int32)         # a dense stretch
    dst = np.concatenate([dst, rng.integers(max(0, nb - 200), nb + 200, 20_000)]).astype(np.int32)
    go = oracle.csr(n, src, dst)
    root = int(src[-1])
    lv, pa, tr, rows = oracle.dist_bfs(go, p, root, mode=2, w=w, trace=True, rows=True)
    g = bfs.Graph.from_edges(n, src, dst, p=p, mode=2, wah_bits=w)
    parent, level, st = g.run(root, stats=True, trace_capacity=1 << 24, row_trace_capacity=1 << 24)
    torch.cuda.synchronize()
    assert (level.cpu().numpy() == lv).all() and (parent.cpu().numpy() == pa).all()
    dt = np.uint32 if w == 32 else np.uint64
    for got, want in ((st.trace_words[: st.trace_used], tr), (st.row_trace_words[: st.row_trace_used], rows)):
        got = got.cpu().numpy().view(dt)
        want = np.concatenate([np.concatenate(x) for x in want]).astype(dt)
        assert len(got) == len(want) and (got == want).all()
    parent, level, _ = g.run(root)
    assert (level.cpu().numpy() == lv).all() and (parent.cpu().numpy() == pa).all()
    if w == 32:                                     # the adaptive format: every slot's choice and elements
        g.set_exchange_format(True)
        parent, level, st = g.run(root, stats=True, trace_capacity=1 << 24)
        assert (level.cpu().numpy() == lv).all() and (parent.cpu().numpy() == pa).all()
        words, at = st.trace_words.cpu().numpy().view(np.uint32), 0
        formats, counts = st.trace_formats.cpu().numpy(), st.trace_counts.cpu().numpy()
        for k, lvl in enumerate(tr):
            for s, stream in enumerate(lvl):
                fmt, elements = oracle.adaptive_encode(oracle.wah_decode(np.asarray(stream), oracle.range_len(n, p, s % p)))
                assert int(formats[k, s]) == fmt and int(counts[k, s]) == len(elements), (k, s)
                assert (words[at: at + len(elements)] == np.asarray(elements).astype(np.uint32)).all(), (k, s)
                at += len(elements)
