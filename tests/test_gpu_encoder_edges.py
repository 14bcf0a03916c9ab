"""Column streams and row buffers, word for word against the oracle, at the range lengths where the slot
encoder changes its shape: one round of 1,024 and of 4,096 groups, 8 chunks of 1,024 (the last short slot)."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("w", [32, 64])
@pytest.mark.parametrize("groups", [1023, 1024, 1025, 4096, 4097, 8192, 8193])
def test_streams_at_the_encoder_edges(groups, w, adaptive):
    import torch
    from paper_1208_5542_gb300 import bfs
    if adaptive and w == 64:
        pytest.skip("the adaptive format has 32-bit words")
    p, extra = 2, groups % 7                                   # trailing bits, none for some
    nb = groups * (w - 1) + extra
    n = p * nb - 5                                             # a shorter last range
    rng = np.random.default_rng(groups)
    # a dense stretch (literals and 1-fills) in an otherwise sparse graph
    src = np.concatenate([rng.integers(0, n, 6 * n // 10), rng.integers(0, 4000, 120_000)]).astype(np.int32)
    dst = np.concatenate([rng.integers(0, n, 6 * n // 10), rng.integers(nb - 3000, nb + 3000, 120_000)]).astype(np.int32)
    go = oracle.csr(n, src, dst)
    root = int(src[-1])
    res = oracle.dist_bfs(go, p, root, mode=2, w=w, trace=True, rows=True)
    lv, pa, tr, rows = res
    g = bfs.Graph.from_edges(n, src, dst, p=p, mode=2, wah_bits=w)
    g.set_exchange_format(adaptive)
    parent, level, st = g.run(root, stats=True, trace_capacity=1 << 22, row_trace_capacity=1 << 22)
    torch.cuda.synchronize()
    assert (level.cpu().numpy() == lv).all() and (parent.cpu().numpy() == pa).all()
    dt = np.uint32 if w == 32 else np.uint64
    got = st.row_trace_words[: st.row_trace_used].cpu().numpy().view(dt)
    want = np.concatenate([np.concatenate(x) for x in rows]).astype(dt)
    assert len(got) == len(want) and (got == want).all()
    if not adaptive:
        got = st.trace_words[: st.trace_used].cpu().numpy().view(dt)
        want = np.concatenate([np.concatenate(x) for x in tr]).astype(dt)
        assert len(got) == len(want) and (got == want).all()
        return
    # the adaptive choice and elements of every slot, from the slot's bits (the WAH stream decoded)
    at, formats = 0, st.trace_formats.cpu().numpy()
    words, counts = st.trace_words.cpu().numpy().view(np.uint32), st.trace_counts.cpu().numpy()
    for k, lvl in enumerate(tr):
        for s, stream in enumerate(lvl):
            nbits = oracle.range_len(n, p, s % p)
            fmt, elements = oracle.adaptive_encode(oracle.wah_decode(np.asarray(stream), nbits))
            assert int(formats[k, s]) == fmt and int(counts[k, s]) == len(elements)
            assert (words[at: at + len(elements)] == np.asarray(elements).astype(np.uint32)).all()
            at += len(elements)
