"""The codecs at the edges of a cluster round (131,072 elements) and of their word loads, against the oracle."""
import ctypes

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

ROUND = 16 * 1024 * 8      # groups (encode) or words (decode) per round of one cluster


def _bits(rng, nbits, kind):
    if kind == "literals":
        return (rng.random(nbits) < 0.4).astype(np.uint8)
    if kind == "ones":
        return np.ones(nbits, np.uint8)
    out = np.zeros(nbits, np.uint8)             # fills that cross threads, CTAs and rounds, odd bits between them
    pos, val = 0, 1
    while pos < nbits:
        ln = int(rng.choice([1, 31, 62, 8 * 31, 8192 * 31, 3 * 8192 * 31 + 5]))
        out[pos:pos + ln] = val
        pos, val = pos + ln, val ^ 1
    return out


def _dev(bits):
    return torch.from_numpy(oracle.pack_bits(bits).view(np.int32).copy()).cuda()


@pytest.mark.parametrize("kind", ["literals", "ones", "runs"])
@pytest.mark.parametrize("w", [32, 64])
@pytest.mark.parametrize("groups", [8, 8191, 8192, 8193, ROUND - 1, ROUND, ROUND + 1, 2 * ROUND + 9])
def test_wah_rounds(groups, w, kind):
    from paper_1208_5542_gb300 import bfs
    rng = np.random.default_rng(groups + w)
    nbits = groups * (w - 1) + groups % 5
    bits = _bits(rng, nbits, kind)
    want = oracle.wah_encode(bits, w)
    got = bfs.wah_encode(_dev(bits), nbits, w)
    host = got.cpu().numpy().view(np.uint32 if w == 32 else np.uint64)
    assert len(host) == len(want) and (host == want.astype(host.dtype)).all()
    back = bfs.wah_decode(got, nbits, w).cpu().numpy().view(np.uint32)
    assert (back == oracle.pack_bits(bits)).all()


@pytest.mark.parametrize("nbits", [31 * (ROUND - 1) + 7, 31 * (ROUND + 1)])
@pytest.mark.parametrize("kind", ["literals", "runs"])
def test_plwah_and_bbc_rounds(nbits, kind):
    from paper_1208_5542_gb300 import bfs
    bits = _bits(np.random.default_rng(nbits), nbits, kind)
    dev, packed = _dev(bits), oracle.pack_bits(bits)
    for enc, dec, ref, dtype in ((bfs.plwah_encode, bfs.plwah_decode, oracle.plwah_encode, np.uint32),
                                 (bfs.bbc_encode, bfs.bbc_decode, oracle.bbc_encode, np.uint8)):
        got, want = enc(dev, nbits), ref(bits)
        host = got.cpu().numpy().view(dtype)
        assert len(host) == len(want) and (host == np.asarray(want).astype(dtype)).all()
        assert (dec(got, nbits).cpu().numpy().view(np.uint32) == packed).all()


def test_decode_over_its_own_stream():
    """The output overlapping the stream: the same bitmap as decoded apart."""
    from paper_1208_5542_gb300 import native
    bits = _bits(np.random.default_rng(3), 31 * 5000 + 3, "literals")
    words = oracle.wah_encode(bits, 32).astype(np.uint32)
    buf = torch.from_numpy(words.view(np.int32).copy()).cuda()
    rc = native.lib().bfs_wah_decode(ctypes.c_void_p(buf.data_ptr()), len(words), len(bits), 32,
                                     ctypes.c_void_p(buf.data_ptr()), ctypes.c_void_p(0))
    assert rc == 0
    out_words = (len(bits) + 31) // 32
    assert (buf.cpu().numpy().view(np.uint32)[:out_words] == oracle.pack_bits(bits)).all()


@pytest.mark.parametrize("words", [[0xC0000005, 0x80000001], [0x80000001] * 40, [0xFFFFFFFF, 0x7FFFFFFF]])
def test_malformed_streams_write_nothing_past_the_bitmap(words):
    from paper_1208_5542_gb300 import native
    nbits = 31 * 3
    out = torch.full((64,), 7, dtype=torch.int32, device="cuda")
    dev = torch.from_numpy(np.asarray(words, np.uint32).view(np.int32).copy()).cuda()
    rc = native.lib().bfs_wah_decode(ctypes.c_void_p(dev.data_ptr()), len(words), nbits, 32,
                                     ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(0))
    assert native.STATUS[rc] == "BFS_ERR_CORRUPT"
    assert (out[(nbits + 31) // 32:] == 7).all()
