"""The workloads whose speed is measured: searches, batches, served queries, graph builds and the codec.

Every case is one call sequence that a program makes through the package's
public entry points (``paper_1208_5542_gb300.bfs``): a breadth-first search on a
resident graph (``Graph.run``), a bit-parallel batch of searches
(``Graph.run_batch``), a burst of queries to the server (``Server``), a graph
loaded and searched once (``Graph.from_edges``), a bitmap coded and decoded
(``wah_encode`` and its relatives).  Graphs are Graph500-style Kronecker tuples
(A = 0.57, B = C = 0.19, D = 0.05, labels scrambled) or uniform Erdos-Renyi
tuples with edge factor 16, made on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_1208_5542_gb300 import bfs

MODES = {"plain": bfs.MODE_PLAIN, "compress": bfs.MODE_COMPRESS, "sieve": bfs.MODE_COMPRESS_SIEVE}
DIRECTIONS = {"top_down": bfs.DIRECTION_TOP_DOWN, "hybrid": bfs.DIRECTION_HYBRID}
SEARCH = {"kind": "search", "graph": "kronecker", "ef": 16, "symmetric": True, "mode": "sieve", "word_bits": 32,
          "rows": True, "adaptive": False, "direction": "top_down", "outputs": "kept"}
CHUNK = 1 << 24                       # tuples generated at a time


def listed():
    s = SEARCH
    return [
        # the smallest call: the library's default options on a graph of the smallest benchmark configuration
        # (scale 12, 2 x 2), outputs allocated by the call
        dict(s, name="search s12", n=1 << 12, p=2, outputs="new"),
        # a small resident graph as the server holds them (scales 16 to 22), default options
        dict(s, name="search s17 ragged", n=150_001, p=5, outputs="new"),
        # a directed graph of no round size, loaded without symmetrisation, with 64-bit words and Alg. 2
        dict(s, name="search directed", graph="uniform", n=1_000_003, p=7, symmetric=False, mode="compress",
             word_bits=64, rows=False),
        # the scale-22 configuration: 8 x 8, Alg. 3 with the fold local to the block-row
        dict(s, name="search s22", n=1 << 22, p=8, rows=False),
        # the same with the library's defaults (the 2D row exchange) and the results read on the host
        dict(s, name="search s22 rows host", n=1 << 22, p=8, outputs="host"),
        # the plain bitmap exchange (Alg. 1) one size below the headline
        dict(s, name="search s24 plain", n=1 << 24, p=16, mode="plain", rows=False),
        # hybrid levels with the level-adaptive exchange
        dict(s, name="search s24 hybrid", n=1 << 24, p=16, rows=False, direction="hybrid", adaptive=True),
        # the headline workload: scale 26 on 16 x 16
        dict(s, name="search s26", n=1 << 26, p=16, rows=False),
        # the 64-root batch of the scale-20 configuration
        dict(s, kind="batch", name="batch s20", n=1 << 20, p=8, lanes=64, parents=False),
        # a burst of queries over three resident graphs; every eighth asks for parents
        dict(s, kind="serve", name="serve burst", n=1 << 18, p=4, queries=96),
        # a graph loaded from tuples on the device and searched once
        dict(s, kind="build", name="build s22", n=1 << 22, p=8, rows=False),
        # one exchanged slice of the headline workload (4M bits) coded and decoded
        {"kind": "codec", "name": "codec wah 4M", "code": "wah32", "nbits": 1 << 22, "density": 0.02},
    ]


def draw(rng):
    kind = rng.choices(["search", "batch", "serve", "build", "codec"], [11, 3, 1, 2, 4])[0]
    if kind == "codec":
        return {"kind": "codec", "code": rng.choice(["wah32", "wah32", "wah64", "plwah", "bbc"]),
                "nbits": int(2 ** rng.uniform(10, 23)) | rng.randint(0, 1),
                "density": round(10 ** rng.uniform(-4, -0.2), 6)}
    top = {"search": 25.5, "batch": 21, "serve": 20, "build": 23}[kind]
    n = int(2 ** rng.uniform(10 if kind == "search" else 14, top))
    if rng.random() < 0.3:
        n = 1 << int(math.log2(n))                      # the benchmark's own sizes are powers of two
    c = dict(SEARCH, kind=kind, n=n, p=rng.choice([1, 2, 3, 4, 7, 8, 8, 16, 16] if n < 1 << 22 else [4, 7, 8, 16]),
             graph=rng.choice(["kronecker", "kronecker", "kronecker", "uniform"]))
    if kind == "batch":
        return dict(c, lanes=rng.choice([1, 5, 17, 32, 63, 64]), parents=rng.random() < 0.3)
    if kind == "serve":
        return dict(c, queries=rng.randint(8, 160))
    c["mode"] = rng.choice(["sieve", "sieve", "sieve", "compress", "plain"])
    c["rows"] = rng.random() < 0.5
    if kind == "build":
        return c
    c["symmetric"] = rng.random() < 0.85
    c["word_bits"] = rng.choice([32, 32, 32, 64])
    c["adaptive"] = c["word_bits"] == 32 and rng.random() < 0.25
    c["direction"] = rng.choice(["top_down", "top_down", "hybrid"]) if c["symmetric"] else "top_down"
    c["outputs"] = rng.choice(["kept", "kept", "new", "host"])
    return c


# -------------------------------------------------------------------- inputs --
def _tuples(case, seed):
    """The directed tuples (int32, on the GPU) of the case's graph."""
    n, m = case["n"], case["ef"] * case["n"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    src = torch.empty(m, dtype=torch.int32, device="cuda")
    dst = torch.empty(m, dtype=torch.int32, device="cuda")
    if case["graph"] == "uniform":
        src.random_(0, n, generator=gen)
        dst.random_(0, n, generator=gen)
        return src, dst
    scale = max(1, (n - 1).bit_length())
    u = torch.empty(min(CHUNK, m), dtype=torch.float32, device="cuda")
    for lo in range(0, m, CHUNK):
        a, b = src[lo:lo + CHUNK], dst[lo:lo + CHUNK]
        a.zero_()
        b.zero_()
        r = u[:len(a)]
        for _ in range(scale):
            r.uniform_(generator=gen)
            row = r >= 0.76                             # quadrants in the order A, B, C, D
            a.mul_(2).add_(row)
            b.mul_(2).add_((r >= 0.95) | ((r >= 0.57) & ~row))
        for x in (a, b):                                # a seeded bijection of [0, 2^scale), cut to [0, n)
            y = x.to(torch.int64)
            for k in range(2):
                y = (y * (2654435761 + 2 * (seed % 65521) + 4 * k + 2)) & ((1 << scale) - 1)
                y ^= y >> ((scale + 1) // 2)
            x.copy_((y * n) >> scale)
    return src, dst


def _graph(case, src, dst):
    g = bfs.Graph.from_edges(case["n"], src, dst, symmetrize=case["symmetric"], p=case["p"],
                             mode=MODES[case["mode"]], wah_bits=case["word_bits"])
    g.set_row_exchange(case["rows"])
    if case["adaptive"]:
        g.set_exchange_format(True)
    if case["direction"] != "top_down":
        g.set_direction(DIRECTIONS[case["direction"]])
    return g


def _roots(src, seed, count):
    """`count` vertices with an entry."""
    at = np.random.default_rng(seed).integers(0, len(src), count)
    return src[torch.from_numpy(at).cuda()].cpu().numpy()


def _bits(case, seed):
    """A frontier slice: set bits whose density varies over the slice (hubs and their neighbourhoods)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = case["nbits"]
    words = (n + 31) // 32
    local = torch.rand((words + 63) // 64, generator=gen, device="cuda") * (2 * case["density"])
    local[torch.rand(len(local), generator=gen, device="cuda") < 0.01] = 1.0     # and runs of ones
    p = local.repeat_interleave(64)[:words]
    out = torch.zeros(words, dtype=torch.int64, device="cuda")
    for b in range(32):
        out |= (torch.rand(words, generator=gen, device="cuda") < p).to(torch.int64) << b
    if n % 32:
        out[-1] &= (1 << (n % 32)) - 1
    return torch.where(out >= 1 << 31, out - (1 << 32), out).to(torch.int32)


class _Burst:
    """A server with its graphs (the server is closed before the graphs it holds)."""

    def __init__(self, graphs):
        self.graphs = graphs
        self.server = bfs.Server(64 << 30)
        self.ids = [self.server.add_graph(g) for g in graphs]

    def __del__(self):
        self.server.close()
        for g in self.graphs:
            g.close()


def _serve_graphs(case):
    """The resident graphs of a served case: the case's own size and two smaller ones."""
    return [dict(case, n=max(1024, case["n"] >> k)) for k in (0, 1, 2)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "codec":
        n, code = case["nbits"], case["code"]
        cap = {"wah64": n // 63 + 1, "bbc": (n + 7) // 8 * 16 // 15 + 16}.get(code, n // 31 + 1)
        unit = {"wah64": torch.int64, "bbc": torch.uint8}.get(code, torch.int32)
        return {"kind": kind, "code": code, "nbits": n, "bits": _bits(case, seed),
                "message": torch.zeros(cap, dtype=unit, device="cuda")}
    if kind == "serve":
        cases = _serve_graphs(case)
        edges = [_tuples(c, seed + k) for k, c in enumerate(cases)]
        burst = _Burst([_graph(c, *e) for c, e in zip(cases, edges)])
        per = [len(range(k, case["queries"], 3)) for k in range(3)]
        roots = [[int(r) for r in _roots(e[0], seed + k, per[k])] for k, e in enumerate(edges)]
        levels = [torch.empty((q, c["n"]), dtype=torch.int32, device="cuda") for q, c in zip(per, cases)]
        return {"kind": kind, "burst": burst, "roots": roots, "levels": levels}
    src, dst = _tuples(case, seed)
    if kind == "batch":
        return {"kind": kind, "graph": _graph(case, src, dst), "roots": _roots(src, seed, case["lanes"]),
                "parents": case["parents"],
                "levels": torch.empty((case["lanes"], case["n"]), dtype=torch.int32, device="cuda")}
    s = {"kind": kind, "root": int(_roots(src, seed, 1)[0]), "parent": None, "level": None}
    if kind == "build":
        return dict(s, src=src, dst=dst, case=dict(case))
    s["graph"] = _graph(case, src, dst)
    if case["outputs"] == "kept":
        s["parent"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
        s["level"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    elif case["outputs"] == "host":
        s["parent"] = torch.empty(case["n"], dtype=torch.int32).pin_memory()
        s["level"] = torch.empty(case["n"], dtype=torch.int32).pin_memory()
    return s


# ---------------------------------------------------------------------- runs --
def run(state):
    kind = state["kind"]
    if kind == "search":
        parent, level, _ = state["graph"].run(state["root"], state["parent"], state["level"])
        return {"level": level, "parent": parent}
    if kind == "batch":
        levels, parents, stats = state["graph"].run_batch(state["roots"], parents=state["parents"],
                                                          levels=state["levels"])
        return {"levels": levels, "parents": parents, "n_levels": stats["n_levels"]}
    if kind == "build":
        g = _graph(state["case"], state["src"], state["dst"])
        parent, level, _ = g.run(state["root"])
        columns = g.nonempty_columns
        g.close()
        return {"level": level, "parent": parent, "nonempty_columns": columns}
    if kind == "serve":
        burst = state["burst"]
        tickets = []
        for k in range(max(len(r) for r in state["roots"])):
            for i, roots in enumerate(state["roots"]):
                if k < len(roots):
                    tickets.append((i, k, burst.server.submit(burst.ids[i], roots[k], parents=k % 8 == 7)))
        parents = []
        for i, k, t in tickets:
            got = burst.server.wait(t, burst.graphs[i].n, out=state["levels"][i][k], parents=k % 8 == 7)
            if k % 8 == 7:
                parents.append(got[1])
        return {"levels": state["levels"], "parents": parents}
    bits, n, code = state["bits"], state["nbits"], state["code"]
    if code in ("wah32", "wah64"):
        words = bfs.wah_encode(bits, n, int(code[3:]))
        back = bfs.wah_decode(words, n, int(code[3:]))
    elif code == "plwah":
        words = bfs.plwah_encode(bits, n)
        back = bfs.plwah_decode(words, n)
    else:
        words = bfs.bbc_encode(bits, n)
        back = bfs.bbc_decode(words, n)
    state["message"][:len(words)] = words               # the buffer that the program sends
    return {"message": state["message"], "count": len(words), "bits": back}


def work(case):
    """Bytes one pass cannot do without: the adjacency once per search, the directories, the results."""
    if case["kind"] == "codec":
        return {"bytes": 4 * (case["nbits"] / 8), "flops": 0}
    n = case["n"]
    entries = case["ef"] * n * (2 if case["symmetric"] else 1)
    search = 4 * entries + 8 * n + case["p"] * n / 8
    if case["kind"] == "batch":
        return {"bytes": 4 * entries + 16 * n + case["lanes"] * 4 * n * (2 if case["parents"] else 1), "flops": 0}
    if case["kind"] == "serve":
        return {"bytes": sum(4 * c["ef"] * c["n"] * 2 + 4 * c["n"] * case["queries"] / 3
                             for c in _serve_graphs(case)), "flops": 0}
    if case["kind"] == "build":
        return {"bytes": search + 8 * case["ef"] * n + 4 * entries, "flops": 0}
    return {"bytes": search, "flops": 0}


# --------------------------------------------------------------------- exact --
def _bfs(n, src, dst, symmetric, root):
    """Levels and smallest parents by level-synchronous search over the tuples, in plain torch."""
    if symmetric:
        src, dst = torch.cat([src, dst]), torch.cat([dst, src])
    src, dst = src.to(torch.int64), dst.to(torch.int64)
    level = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    parent = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    level[root] = 0
    parent[root] = root
    for k in range(n):
        e = (level[src] == k) & (level[dst] < 0)
        if not bool(e.any()):
            break
        best = torch.full((n,), n, dtype=torch.int64, device="cuda")
        best.scatter_reduce_(0, dst[e], src[e], "amin")
        new = best < n
        level[new] = k + 1
        parent[new] = best[new]
    return level.to(torch.int32), parent.to(torch.int32)


def exact(case, seed):
    if case["kind"] == "codec":
        return {"message": None, "count": None, "bits": _bits(case, seed)}
    if case["kind"] not in ("search", "build") or case["n"] > 1 << 22:
        return None
    src, dst = _tuples(case, seed)
    level, parent = _bfs(case["n"], src, dst, case["symmetric"], int(_roots(src, seed, 1)[0]))
    out = {"level": level, "parent": parent}
    return dict(out, nonempty_columns=None) if case["kind"] == "build" else out
