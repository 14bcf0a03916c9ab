"""The codecs on a stream that is not the current one and has other work ahead: the same streams and bitmaps."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code", ["wah32", "wah64", "plwah", "bbc"])
def test_another_stream(code):
    from paper_1208_5542_gb300 import bfs
    bits = (np.random.default_rng(4).random(400_003) < 0.03).astype(np.uint8)
    n = len(bits)
    want = {"wah32": lambda: oracle.wah_encode(bits, 32), "wah64": lambda: oracle.wah_encode(bits, 64),
            "plwah": lambda: oracle.plwah_encode(bits), "bbc": lambda: oracle.bbc_encode(bits)}[code]()
    dtype = {"wah64": np.uint64, "bbc": np.uint8}.get(code, np.uint32)
    extra = (int(code[3:]),) if code.startswith("wah") else ()
    enc = bfs.wah_encode if extra else getattr(bfs, code + "_encode")
    dec = bfs.wah_decode if extra else getattr(bfs, code + "_decode")
    host = torch.from_numpy(oracle.pack_bits(bits).view(np.int32).copy())
    side = torch.cuda.Stream()
    for k in range(3):
        torch.cuda._sleep(20_000_000)                       # some ms of work on both streams
        dev = host.cuda(non_blocking=True) if k else host.cuda().to(torch.int64)    # as given, and copied by the call
        with torch.cuda.stream(side):
            torch.cuda._sleep(20_000_000)
        got = enc(dev, n, *extra, stream=side)
        out = got.cpu().numpy().view(dtype)
        assert len(out) == len(want) and (out == np.asarray(want).astype(dtype)).all()
        with torch.cuda.stream(side):
            torch.cuda._sleep(20_000_000)
        assert (dec(got, n, *extra, stream=side).cpu() == host).all()
