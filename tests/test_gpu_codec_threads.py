"""More host threads inside a decode than the library has mapped flag pairs (256): every call returns, and right.

Run in a child process: threads that wait for one another's pairs would never return."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes, threading
import numpy as np, torch
import oracle
from paper_1208_5542_gb300 import native
rng = np.random.default_rng(1)
bits = (rng.random(31 * 40 + 7) < 0.1).astype(np.uint8)
words = torch.from_numpy(oracle.plwah_encode(bits).astype(np.uint32).view(np.int32).copy()).cuda()
want = torch.from_numpy(oracle.pack_bits(bits).view(np.int32).copy()).cuda()
out = torch.zeros((320, len(want)), dtype=torch.int32, device="cuda")
torch.cuda.synchronize()
lib, rcs, gate = native.lib(), [], threading.Barrier(320)
def work(k):
    gate.wait()
    for _ in range(10):
        rcs.append(lib.bfs_plwah_decode(ctypes.c_void_p(words.data_ptr()), len(words), len(bits),
                                        ctypes.c_void_p(out[k].data_ptr()), ctypes.c_void_p(0)))
threads = [threading.Thread(target=work, args=(k,), daemon=True) for k in range(320)]
for t in threads: t.start()
for t in threads: t.join()
torch.cuda.synchronize()
assert rcs == [0] * 3200 and bool((out == want).all())
print("ok")
"""


def test_more_threads_than_flag_pairs():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=180)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stderr[-2000:]
