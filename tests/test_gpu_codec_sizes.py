"""The codecs on every cluster size down to one CTA (what a partition of a device may place), against the oracle,
at the edges of the smallest and of a middle round."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

CTA = 1024 * 8             # groups (encode) or words (decode) per CTA and round


@pytest.fixture(params=[1, 2, 4, 8, 16, 0])
def ctas(request):
    from paper_1208_5542_gb300 import native
    assert native.lib().bfs_debug_codec_ctas(request.param) == 0
    yield request.param
    assert native.lib().bfs_debug_codec_ctas(0) == 0


@pytest.mark.parametrize("groups", [5, CTA, CTA + 1, 4 * CTA + 3])
def test_streams_on_every_cluster_size(ctas, groups):
    from paper_1208_5542_gb300 import bfs
    rng = np.random.default_rng(groups)
    bits = np.repeat(rng.random(groups + 1) < 0.5, 31)[:31 * groups + 11].astype(np.uint8)
    bits[rng.random(len(bits)) < 0.02] ^= 1             # literals between 0- and 1-fills
    dev = torch.from_numpy(oracle.pack_bits(bits).view(np.int32).copy()).cuda()
    for enc, dec, ref, dtype in (
            (lambda: bfs.wah_encode(dev, len(bits), 32), lambda w: bfs.wah_decode(w, len(bits), 32),
             oracle.wah_encode(bits, 32), np.uint32),
            (lambda: bfs.wah_encode(dev, len(bits), 64), lambda w: bfs.wah_decode(w, len(bits), 64),
             oracle.wah_encode(bits, 64), np.uint64),
            (lambda: bfs.plwah_encode(dev, len(bits)), lambda w: bfs.plwah_decode(w, len(bits)),
             oracle.plwah_encode(bits), np.uint32),
            (lambda: bfs.bbc_encode(dev, len(bits)), lambda w: bfs.bbc_decode(w, len(bits)),
             oracle.bbc_encode(bits), np.uint8)):
        got = enc()
        host, want = got.cpu().numpy().view(dtype), np.asarray(ref).astype(dtype)
        assert len(host) == len(want) and (host == want).all()
        assert bool((dec(got) == dev).all())


def test_cap_arguments():
    from paper_1208_5542_gb300 import native
    for bad in (-1, 3, 32):
        assert native.STATUS[native.lib().bfs_debug_codec_ctas(bad)] == "BFS_ERR_INVALID_ARG"
