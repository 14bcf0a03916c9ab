// msbfs.cu -- batched multi-source BFS: up to 64 searches at once, bit-parallel.
//
// Every vertex holds three 64-bit lane words (bit r = search r): vis (visited)
// and nxt (next), side by side, and f (frontier).  One level is the boolean
// SpMV of Sec. III-A applied to all 64 lane vectors at once:
//   nxt[v] |= f[u] & ~vis[v]     for every entry u -> v of a nonempty column
// of a block whose source u is active (f[u] != 0); the directory V_{i,j}
// (Eq. 4) sieves the (vertex, block) pairs, exactly as in the single search.
// On an undirected graph the same product can be taken from v's side, v's own
// columns holding its neighbours: a level whose active vertices hold much of
// the graph's entries lets every vertex that some running lane has not visited
// OR its neighbours' frontier words, without an atomic, until no lane is
// missing.  The block-rows are scanned in order, so the first that holds a
// frontier neighbour of a lane holds its smallest: its parent there.
// Then new = nxt & ~vis; vis |= new; f = new; level[r][v] = k + 1 for every new
// bit r; and the next level's active list is the set of v with new != 0.
// Optional parents: parent[r][v] = the smallest u of lane r's previous level
// with an entry u -> v, by a (select, min) reduction per new lane bit.
//
// The whole batch is one CUDA-graph launch: the initialisation, then a
// conditional WHILE node whose body is one level (expand, long-column pieces, or
// the destinations' side; the reduction, whose last CTA decides from the active
// count whether to iterate again).  No host round trip per level.  Kernels read their
// arguments from a device-resident state block, so the graph is built once per
// graph handle and reused by every call.
#include <algorithm>
#include <chrono>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace bfsgb {
namespace {

constexpr int kMT = 256;            // threads of the small kernels
constexpr uint32_t kMsCoop = 32;    // columns of at least this many entries take the whole warp
constexpr uint32_t kMsHub = 512;    // longer columns are cut into pieces
constexpr uint32_t kMsPiece = 512;

// Device-resident arguments and counters of a batch (one per graph).
struct MsState {
    // graph layout (constant)
    const uint32_t* dir;
    const uint32_t* rank;
    int64_t dir_stride;
    const uint32_t* cp;
    const int64_t* cp_base;
    const int64_t* ir_base;
    const int32_t* ir;
    int p;
    int64_t nb, n;
    // lane words and active lists (constant buffers)
    ulonglong2* vn;             // x: vis, y: nxt
    unsigned long long* f[2];
    const uint32_t* deg;        // entries per source vertex
    int symmetric;              // undirected: levels may run from the destinations' side
    int32_t* act[2];
    Item* pieces;
    int64_t piece_cap;
    // per call
    const int32_t* roots;       // device copy of the roots
    int32_t n_roots;
    int32_t max_levels;         // iteration limit (n + 1 at most)
    int32_t* levels;            // [n_roots][n]
    int32_t* parents;           // [n_roots][n] or nullptr
    unsigned long long parent_mask;  // lanes whose parents are computed (with parents != nullptr)
    // per level
    int32_t cur;                // index of the current f / act buffers
    int32_t level;              // k
    unsigned long long act_count[2];
    unsigned long long act_next;     // hand-out cursor over the current active list
    unsigned long long piece_count;
    unsigned long long piece_next;
    unsigned long long edges;        // entries of the active vertices (all levels)
    unsigned long long act_edges;    // the same of the next level
    unsigned long long miss_edges;   // entries of the vertices that a running lane has not visited
    unsigned long long lanes;        // lanes with a frontier vertex at the current level
    int32_t pull;                    // 1: this level runs from the destinations' side
    unsigned int done;               // CTAs of the reduction that have finished
    unsigned long long levels_done;  // levels performed
    // continuous batching (server): lane r's level of v is (iteration + 1) - lane_start[r]
    int32_t lane_start[64];
    unsigned long long alive;        // lanes that reached a new vertex in this iteration
    unsigned long long steps;        // iterations of this launch
    unsigned long long err;          // first failed bounds check: code, then two values
    unsigned long long err_a, err_b;
    unsigned long long running;      // lanes of this launch
    const volatile int* call;        // mapped host word: nonzero asks the iterations to end
    int64_t nnz;                     // entries of the layout
};

// A bounds check failed: keep the first one's code and values (the access is skipped).
__device__ __forceinline__ void ms_fault(MsState* S, unsigned long long code, unsigned long long x,
                                         unsigned long long y) {
    if (atomicCAS(&S->err, 0ull, code) == 0ull) {
        S->err_a = x;
        S->err_b = y;
    }
}

// ------------------------------------------------------------------ init --
__global__ void ms_reset(MsState* S) {
    for (int r = 0; r < 64; ++r) S->lane_start[r] = 0;
    S->alive = 0;
    S->cur = 0;
    S->level = 0;
    S->act_count[0] = 0;
    S->act_count[1] = 0;
    S->act_next = 0;
    S->piece_count = 0;
    S->piece_next = 0;
    S->edges = 0;
    S->act_edges = 0;
    S->miss_edges = 0;
    S->lanes = 0;
    S->pull = 0;
    S->done = 0;
    S->levels_done = 0;
    S->err = 0;
    S->err_a = 0;
    S->err_b = 0;
}

__global__ void ms_clear(MsState* S) {
    const MsState& s = *S;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t v = tid; v < s.n; v += stride) {
        s.vn[v] = make_ulonglong2(0ull, 0ull);
        s.f[0][v] = 0ull;
        s.f[1][v] = 0ull;
    }
    const int64_t total = (int64_t)s.n_roots * s.n;
    for (int64_t x = tid; x < total; x += stride) {
        s.levels[x] = -1;
        if (s.parents) s.parents[x] = -1;
    }
}

__global__ void ms_roots(MsState* S) {
    MsState& s = *S;
    const int r = threadIdx.x;
    if (r >= s.n_roots) return;
    const int32_t v = s.roots[r];
    const unsigned long long bit = 1ull << r;
    const unsigned long long old = atomicOr(&s.vn[v].x, bit);
    atomicOr(s.f[0] + v, bit);
    s.levels[(int64_t)r * s.n + v] = 0;
    if (s.parents) s.parents[(int64_t)r * s.n + v] = v;
    if (old == 0ull) {                       // first lane at this vertex: make it active
        const unsigned long long pos = atomicAdd(&s.act_count[0], 1ull);
        s.act[0][pos] = v;
        atomicAdd(&s.edges, (unsigned long long)s.deg[v]);
    }
    atomicOr(&s.lanes, bit);
}

// ----------------------------------------------------------------- level --
// Visit u -> v given v's words read before (several entries' reads are in
// flight together; a stale nxt only costs an atomic that changes nothing).
struct MsVisit {
    const MsState* s;
    __device__ __forceinline__ bool valid(int32_t v, int32_t u) const {
        if ((uint64_t)(uint32_t)v < (uint64_t)s->n) return true;
        ms_fault(const_cast<MsState*>(s), 2, (uint32_t)v, (uint32_t)u);
        return false;
    }
    __device__ __forceinline__ ulonglong2 probe(int32_t v) const { return __ldcg(s->vn + v); }
    __device__ __forceinline__ void mark(int32_t v, int32_t u, unsigned long long fu, const ulonglong2& w) const {
        const unsigned long long nb = fu & ~w.x;               // vis does not change during the expansion
        if (!nb) return;
        if (nb & ~w.y) atomicOr(&s->vn[v].y, nb);
        if (s->parents) {
            unsigned long long m = nb & s->parent_mask;
            while (m) {
                const int r = __ffsll((long long)m) - 1;
                m &= m - 1;
                atomicMin(reinterpret_cast<unsigned int*>(s->parents + (int64_t)r * s->n + v), (unsigned int)u);
            }
        }
    }
};

constexpr int kMsIlp = 4;           // entries per lane in flight

__device__ __forceinline__ void ms_column(const MsVisit& vis, const int32_t* ir, int32_t u, unsigned long long fu,
                                          int64_t beg, uint32_t len) {
    const int32_t* col = ir + beg;
    for (uint32_t e = lane_id(); e < len; e += 32 * kMsIlp) {
        int32_t v[kMsIlp];
        ulonglong2 w[kMsIlp];
#pragma unroll
        for (int k = 0; k < kMsIlp; ++k) v[k] = e + 32 * k < len ? __ldg(col + e + 32 * k) : -1;
#pragma unroll
        for (int k = 0; k < kMsIlp; ++k)
            if (e + 32 * k < len && !vis.valid(v[k], u)) v[k] = -1;
#pragma unroll
        for (int k = 0; k < kMsIlp; ++k)
            if (v[k] >= 0) w[k] = vis.probe(v[k]);
#pragma unroll
        for (int k = 0; k < kMsIlp; ++k)
            if (v[k] >= 0) vis.mark(v[k], u, fu, w[k]);
    }
}

// One item per lane (u, f[u], column); long columns go to the piece list,
// columns of at least kMsCoop entries take the whole warp, the rest share the
// warp, 32 consecutive entries of the concatenated columns per step: every
// column's first entry sets its bit in the step's head mask, and the owner of
// an entry is the number of heads up to it (the columns are packed in the
// warp's scratch).
struct MsScratch {
    unsigned long long fu[32];
    int64_t off[32];            // column offset minus the entries before it
    int32_t u[32];
};

__device__ __forceinline__ void ms_warp_expand(MsState& s, const MsVisit& vis, int32_t u, unsigned long long fu,
                                               int64_t beg, uint32_t len, MsScratch& ws) {
    if (__any_sync(0xffffffffu, len > kMsHub)) {
        if (len > kMsHub) {
            const uint32_t np = (len + kMsPiece - 1) / kMsPiece;
            const unsigned long long base = atomicAdd(&s.piece_count, (unsigned long long)np);
            for (uint32_t k = 0; k < np && base + k < (unsigned long long)s.piece_cap; ++k) {
                Item it;
                it.u = u;
                it.len = (len - k * kMsPiece < kMsPiece) ? len - k * kMsPiece : kMsPiece;
                it.begin = beg + (int64_t)k * kMsPiece;
                s.pieces[base + k] = it;
            }
            len = 0;
        }
    }
    uint32_t coop = __ballot_sync(0xffffffffu, len >= kMsCoop);
    while (coop) {
        const int src = __ffs(coop) - 1;
        coop &= coop - 1;
        ms_column(vis, s.ir, __shfl_sync(0xffffffffu, u, src), __shfl_sync(0xffffffffu, fu, src),
                  __shfl_sync(0xffffffffu, beg, src), __shfl_sync(0xffffffffu, len, src));
    }
    if (len >= kMsCoop) len = 0;
    const uint32_t nz = __ballot_sync(0xffffffffu, len > 0);
    if (!nz) return;
    const uint32_t incl = warp_incl_sum(len);
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t excl = incl - len;
    const uint32_t below = (1u << lane_id()) - 1u, upto = below | (1u << lane_id());
    __syncwarp();                           // the previous batch's readers are done
    if (len > 0) {
        const int r = __popc(nz & below);
        ws.fu[r] = fu;
        ws.off[r] = beg - (int64_t)excl;
        ws.u[r] = u;
    }
    __syncwarp();
    int before = -1;
    for (uint32_t e0 = 0; e0 < total; e0 += 32 * kMsIlp) {
        int32_t v[kMsIlp];
        int ow[kMsIlp];
        ulonglong2 w[kMsIlp];
#pragma unroll
        for (int k = 0; k < kMsIlp; ++k) {
            const uint32_t rel = excl - (e0 + 32 * k);
            const uint32_t heads = __reduce_or_sync(0xffffffffu, (len > 0 && rel < 32u) ? 1u << rel : 0u);
            const uint32_t e = e0 + 32 * k + lane_id();
            ow[k] = before + __popc(heads & upto);
            before += __popc(heads);
            v[k] = e < total ? __ldg(s.ir + ws.off[ow[k]] + (int64_t)e) : -1;
            if (e < total && !vis.valid(v[k], ws.u[ow[k]])) v[k] = -1;
        }
#pragma unroll
        for (int k = 0; k < kMsIlp; ++k)
            if (v[k] >= 0) w[k] = vis.probe(v[k]);
#pragma unroll
        for (int k = 0; k < kMsIlp; ++k)
            if (v[k] >= 0) vis.mark(v[k], ws.u[ow[k]], ws.fu[ow[k]], w[k]);
    }
}

// Column of local source ul in block b: offset into ir and length (0: empty).
__device__ __forceinline__ void ms_lookup(const MsState& s, int64_t b, int64_t ul, int64_t& beg, uint32_t& len) {
    const uint32_t dw = __ldg(s.dir + b * s.dir_stride + (ul >> 5));
    const uint32_t rk = __ldg(s.rank + b * s.dir_stride + (ul >> 5));
    const uint32_t bit = 1u << (ul & 31);
    beg = 0;
    len = 0;
    if (!(dw & bit)) return;
    const uint32_t* cpb = s.cp + __ldg(s.cp_base + b);
    const uint32_t c = rk + __popc(dw & (bit - 1u));
    const uint32_t c0 = __ldg(cpb + c), c1 = __ldg(cpb + c + 1);
    beg = __ldg(s.ir_base + b) + c0;
    len = c1 - c0;
}

// Expansion.  Unit = (32 active vertices, one block-row i): the vertices whose
// column of block (i, j(u)) is nonempty (directory test) are expanded by one
// warp, the next unit's columns looked up before.  Bound by the scattered
// 16-byte reads of (vis, nxt): four in flight per lane, both words in one
// access.  With ms_pull and the coalesced level writes of ms_reduce a batch of 64
// at scale 20 takes 1.29 ms (4.6 with one read in flight and no other side).  With fewer units than warps
// a unit holds fewer vertices (down to one), so that a short active list, which
// holds the hubs of the early levels, still fills the chip.  Few units are
// dealt out in turn, many handed out by a counter, several at a time.
__global__ void __launch_bounds__(1024) ms_expand(MsState* S) {
    MsState& s = *S;
    if (s.pull) return;
    extern __shared__ MsScratch s_ws[];
    MsScratch& ws = s_ws[threadIdx.x >> 5];
    const MsVisit vis{S};
    const int cur = s.cur, p = s.p;
    const int32_t* act = s.act[cur];
    const int64_t nact = (int64_t)s.act_count[cur];
    const unsigned long long* f = s.f[cur];
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int64_t bw = nact * p / (2 * warps);                       // vertices per unit
    bw = bw < 1 ? 1 : (bw < 32 ? bw : 32);
    const int64_t groups = (nact + bw - 1) / bw, units = groups * p;
    int64_t each = units / (4 * warps);                        // units per hand-out
    each = each < 1 ? 1 : (each < 16 ? each : 16);
    // the column of this lane's vertex in unit x (none past the units or the group)
    auto lookup = [&](int64_t x, int32_t& u, unsigned long long& fu, int64_t& beg, uint32_t& len) {
        fu = 0;
        len = 0;
        beg = 0;
        u = 0;
        if (x >= units) return;
        const int64_t i = x / groups, q = (x - i * groups) * bw + lane_id();   // block-row by block-row
        if ((int64_t)lane_id() >= bw || q >= nact) return;
        u = act[q];
        if ((uint64_t)(uint32_t)u >= (uint64_t)s.n) {
            ms_fault(S, 1, (uint64_t)q, (uint32_t)u);
            u = 0;
            return;
        }
        fu = f[u];
        const int64_t j = (uint32_t)u / (uint32_t)s.nb;        // ids and ranges are below 2^31
        ms_lookup(s, i * p + j, u - j * s.nb, beg, len);
    };
    auto run = [&](int64_t x0, int64_t x1) {
        int32_t u, un;
        unsigned long long fu, fn;
        int64_t beg, bn;
        uint32_t len, ln;
        lookup(x0, u, fu, beg, len);
        for (int64_t x = x0; x < x1; ++x) {
            lookup(x + 1 < x1 ? x + 1 : units, un, fn, bn, ln);
            if (__any_sync(0xffffffffu, len > 0)) ms_warp_expand(s, vis, u, fu, beg, len, ws);
            u = un;
            fu = fn;
            beg = bn;
            len = ln;
        }
    };
    if (units <= 4 * warps) {
        const int64_t w0 = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
        for (int64_t x = w0; x < units; x += warps) run(x, x + 1);
        return;
    }
    for (;;) {
        unsigned long long base = 0;
        if (lane_id() == 0) base = atomicAdd(&s.act_next, (unsigned long long)each);
        base = __shfl_sync(0xffffffffu, base, 0);
        if ((int64_t)base >= units) break;
        run((int64_t)base, (int64_t)base + each < units ? (int64_t)base + each : units);
    }
}

__global__ void __launch_bounds__(kMT) ms_pieces(MsState* S) {
    MsState& s = *S;
    if (s.pull) return;
    const MsVisit vis{S};
    const unsigned long long* f = s.f[s.cur];
    const unsigned long long np = min(s.piece_count, (unsigned long long)s.piece_cap);
    for (;;) {
        unsigned long long pc = 0;
        if (lane_id() == 0) pc = atomicAdd(&s.piece_next, 1ull);
        pc = __shfl_sync(0xffffffffu, pc, 0);
        if (pc >= np) break;
        const Item it = s.pieces[pc];
        if ((uint64_t)(uint32_t)it.u >= (uint64_t)s.n || it.begin < 0 || it.begin + (int64_t)it.len > s.nnz) {
            if (lane_id() == 0) ms_fault(S, 6, pc, (uint64_t)it.begin);
            continue;
        }
        ms_column(vis, s.ir, it.u, f[it.u], it.begin, it.len);
    }
}

// A level from the destinations' side (undirected graphs): every vertex v that
// a running lane has not visited ORs the frontier words of its neighbours --
// its own columns, block-row by block-row -- and stops once no lane is
// missing.  A lane that wants parents takes the smallest neighbour with its
// bit of the first block-row that has one (a column is in any order: it is
// read to its end for such a lane).  A lane of the warp scans its column kMsIlp
// entries at a time; the rest of a column beyond kMsPullLane entries is read
// by the whole warp, which takes the smallest parent of every search lane over
// its entries and keeps it in a register to the column's end (an atomic per entry
// and search lane instead: 17 lanes with parents at scale 20 on 4 x 4 2.26 ms against
// 1.88, 64 lanes 5.25 against 4.47).  Four CTAs per SM, 62 registers; left to itself
// the compiler takes 48 and spills (uniform scale 20 on 8 x 8, 64 lanes: 2.42 ms
// against 2.29).
constexpr uint32_t kMsPullLane = 32;

// Lower the parents of v in the lanes `bits` to u; v belongs to one thread.
__device__ __forceinline__ void ms_parents(const MsState& s, int64_t v, int32_t u, unsigned long long bits) {
    for (; bits; bits &= bits - 1ull) {
        unsigned int* q = reinterpret_cast<unsigned int*>(s.parents + (int64_t)(__ffsll((long long)bits) - 1) * s.n + v);
        if ((unsigned int)u < *q) *q = (unsigned int)u;
    }
}

__global__ void __launch_bounds__(kMT, 4) ms_pull(MsState* S) {
    MsState& s = *S;
    if (!s.pull) return;
    const unsigned long long* f = s.f[s.cur];
    const unsigned long long lanes = s.lanes, pmask = s.parents ? s.parent_mask : 0ull;
    const int p = s.p;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; 32 * g < s.n; g += warps) {
        const int64_t v = 32 * g + lane_id();
        unsigned long long need = v < s.n ? lanes & ~s.vn[v].x : 0ull;
        if (need && s.deg[v] == 0) need = 0;
        if (!__any_sync(0xffffffffu, need != 0ull)) continue;
        const int64_t j = (uint32_t)v / (uint32_t)s.nb, vl = v - j * s.nb;
        unsigned long long got = 0;
        int64_t beg = 0, beg_n = 0;
        uint32_t len = 0, len_n = 0;
        if (need) ms_lookup(s, j, vl, beg, len);
        for (int i = 0; i < p; ++i) {
            len_n = 0;
            if (need && i + 1 < p) ms_lookup(s, (int64_t)(i + 1) * p + j, vl, beg_n, len_n);
            const unsigned long long need0 = need;          // missing before this block-row
            uint32_t e = 0;
            const uint32_t own = len < kMsPullLane ? len : kMsPullLane;
            while (e < own && (need | (need0 & pmask))) {
                int32_t u[kMsIlp];
                unsigned long long w[kMsIlp];
#pragma unroll
                for (int k = 0; k < kMsIlp; ++k) u[k] = e + k < own ? __ldg(s.ir + beg + e + k) : -1;
#pragma unroll
                for (int k = 0; k < kMsIlp; ++k) {
                    w[k] = 0ull;
                    if (u[k] < 0) continue;
                    if ((uint64_t)(uint32_t)u[k] < (uint64_t)s.n) w[k] = __ldg(f + u[k]) & need0;
                    else ms_fault(S, 2, (uint32_t)u[k], (uint64_t)v);
                }
#pragma unroll
                for (int k = 0; k < kMsIlp; ++k) {
                    need &= ~w[k];
                    if (w[k] & pmask) ms_parents(s, v, u[k], w[k] & pmask);
                }
                e += kMsIlp;
            }
            uint32_t more = __ballot_sync(0xffffffffu, len > kMsPullLane && (need | (need0 & pmask)));
            while (more) {                  // the rest of the long columns, one after the other
                const int src = __ffs(more) - 1;
                more &= more - 1;
                const int64_t cb = __shfl_sync(0xffffffffu, beg, src), cv = __shfl_sync(0xffffffffu, v, src);
                const uint32_t cl = __shfl_sync(0xffffffffu, len, src);
                const unsigned long long c0 = __shfl_sync(0xffffffffu, need0, src);
                unsigned long long cn = __shfl_sync(0xffffffffu, need, src);
                uint32_t best[2] = {~0u, ~0u};          // smallest parents of search lanes lane_id(), lane_id() + 32
                for (uint32_t e0 = kMsPullLane; e0 < cl && (cn | (c0 & pmask)); e0 += 32 * kMsIlp) {
                    int32_t u[kMsIlp];
                    unsigned long long h[kMsIlp], w = 0;
#pragma unroll
                    for (int k = 0; k < kMsIlp; ++k) {
                        const uint32_t x = e0 + 32 * k + lane_id();
                        u[k] = x < cl ? __ldg(s.ir + cb + x) : -1;
                    }
#pragma unroll
                    for (int k = 0; k < kMsIlp; ++k) {
                        h[k] = 0ull;
                        if (u[k] < 0) continue;
                        if ((uint64_t)(uint32_t)u[k] < (uint64_t)s.n) h[k] = __ldg(f + u[k]) & c0;
                        else ms_fault(S, 2, (uint32_t)u[k], (uint64_t)cv);
                        w |= h[k];
                    }
                    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)w);
                    const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(w >> 32));
                    const unsigned long long hit = ((unsigned long long)hi << 32) | lo;
                    cn &= ~hit;
                    for (unsigned long long m = hit & pmask; m; m &= m - 1ull) {
                        const int b = __ffsll((long long)m) - 1;
                        uint32_t c = ~0u;
#pragma unroll
                        for (int k = 0; k < kMsIlp; ++k)
                            if ((h[k] >> b) & 1ull) c = min(c, (uint32_t)u[k]);
                        c = __reduce_min_sync(0xffffffffu, c);
                        if ((int)lane_id() == b) best[0] = min(best[0], c);
                        if ((int)lane_id() + 32 == b) best[1] = min(best[1], c);
                    }
                }
                __syncwarp();               // the parents lowered by lane src are seen below
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (best[k] == ~0u) continue;
                    unsigned int* q = reinterpret_cast<unsigned int*>(s.parents) + (int64_t)(lane_id() + 32 * k) * s.n + cv;
                    if (best[k] < *q) *q = best[k];
                }
                __syncwarp();
                if ((int)lane_id() == src) need = cn;
            }
            got |= need0 & ~need;
            if (!__any_sync(0xffffffffu, need != 0ull)) break;
            beg = beg_n;
            len = len_n;
        }
        if (got) s.vn[v].y = got;
    }
}

// The next level runs from the destinations' side when the vertices that miss
// a lane hold no more entries than the active ones -- a visit there is a read,
// from the sources' side a read and often an atomic, and a miss in any of 64
// lanes means that the whole column is read -- or, when lanes want parents (an
// atomic per entry and lane on the sources' side), up to kMsPullParents times as
// many.  With one block-row a column is read to its end for such a lane, and the
// factor only pays for more than 32 of them.  A level with few entries stays on
// the sources' side.  Scale 20, 64 lanes: 1.28 ms (never: 1.82; always on dense
// levels: 1.85).  With parents, on one block: 17 lanes 3.07 ms with the factor, 1.66
// without, uniform with 64 lanes 4.00 and 5.04; on 8 x 8 with 5 lanes, uniform, a
// factor of 8 gives 0.74 ms, 4 gives 0.59.
constexpr unsigned long long kMsPullParents = 4;
constexpr unsigned long long kMsPullShare = 64;

// One level ends: switch to the next one's buffers (one thread, the level's
// counts complete).
__device__ void ms_advance(MsState& s, unsigned long long alive) {
    const int nxt_i = s.cur ^ 1;
    s.act_count[s.cur] = 0;
    s.cur = nxt_i;
    s.level += 1;
    s.levels_done += 1;
    s.act_next = 0;
    s.piece_count = 0;
    s.piece_next = 0;
    const unsigned long long e = __ldcg(&s.act_edges), miss = __ldcg(&s.miss_edges);
    s.edges += e;
    s.act_edges = 0;
    s.miss_edges = 0;
    s.lanes = alive;
    const int parents = s.parents ? __popcll(s.parent_mask & alive) : 0;
    const unsigned long long worth = parents > (s.p == 1 ? 32 : 0) ? kMsPullParents : 1ull;
    s.pull = (s.symmetric && worth * e * kMsPullShare > (unsigned long long)s.nnz && miss <= worth * e) ? 1 : 0;
}

// new = nxt & ~vis; vis |= new; f' = new; level of every new lane, lane by lane
// over the warp's vertices (coalesced stores); next active list, one hand-out
// of places per CTA.  The last CTA to finish (a counter, no waiting) switches
// to the next level and decides whether to iterate again: a batch while a lane
// has a frontier vertex; a server's launch while every running lane has one,
// the host does not call and fewer than kMsSteps levels ran (the host retires
// and admits lanes between launches).
constexpr unsigned long long kMsSteps = 1024;

__global__ void __launch_bounds__(kMT) ms_reduce(MsState* S, cudaGraphConditionalHandle handle, int server) {
    constexpr int NW = kMT / 32;
    __shared__ uint32_t s_cnt[NW];
    __shared__ unsigned long long s_base, s_any[NW], s_deg[NW], s_miss[NW];
    MsState& s = *S;
    const int cur = s.cur, nxt_i = cur ^ 1;
    unsigned long long* fn = s.f[nxt_i];
    int32_t* actn = s.act[nxt_i];
    const int32_t lv = s.level + 1;
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const unsigned long long lanes = s.lanes;
    unsigned long long alive = 0, edges = 0, miss = 0;
    for (int64_t v0 = blockIdx.x * (int64_t)kMT; v0 < s.n; v0 += (int64_t)gridDim.x * kMT) {
        const int64_t v = v0 + threadIdx.x;
        unsigned long long nv = 0;
        if (v < s.n) {
            const ulonglong2 x = s.vn[v];
            nv = x.y & ~x.x;
            if (x.y) s.vn[v] = make_ulonglong2(x.x | nv, 0ull);
            fn[v] = nv;
            const bool missed = (lanes & ~(x.x | nv)) != 0ull;
            const uint32_t d = nv || missed ? s.deg[v] : 0u;
            if (nv) edges += d;
            if (missed) miss += d;
        }
        const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)nv);
        const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(nv >> 32));
        unsigned long long any = ((unsigned long long)hi << 32) | lo;
        alive |= any;
        for (; any; any &= any - 1ull) {
            const int r = __ffsll((long long)any) - 1;
            if ((nv >> r) & 1ull) s.levels[(int64_t)r * s.n + v] = lv - s.lane_start[r];
        }
        const uint32_t ball = __ballot_sync(0xffffffffu, nv != 0ull);
        if (lane == 0) s_cnt[warp] = __popc(ball);
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            if (k < warp) before += s_cnt[k];
            total += s_cnt[k];
        }
        if (threadIdx.x == 0) s_base = total ? atomicAdd(&s.act_count[nxt_i], (unsigned long long)total) : 0ull;
        __syncthreads();
        if (nv) {
            const unsigned long long at = s_base + before + __popc(ball & ((1u << lane) - 1u));
            if (at < (unsigned long long)s.n) actn[at] = (int32_t)v;
            else ms_fault(S, 3, at, (uint64_t)v);
        }
    }
    edges = warp_sum(edges);
    miss = warp_sum(miss);
    if (lane == 0) {
        s_any[warp] = alive;
        s_deg[warp] = edges;
        s_miss[warp] = miss;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int k = 1; k < NW; ++k) {
        alive |= s_any[k];
        edges += s_deg[k];
        miss += s_miss[k];
    }
    if (alive) atomicOr(&s.alive, alive);
    if (edges) atomicAdd(&s.act_edges, edges);
    if (miss) atomicAdd(&s.miss_edges, miss);
    __threadfence();
    if (atomicAdd(&s.done, 1u) != gridDim.x - 1) return;
    __threadfence();
    s.done = 0;
    const unsigned long long cnt = __ldcg(&s.act_count[nxt_i]), any = __ldcg(&s.alive);
    ms_advance(s, any);
    bool go;
    if (server) {
        s.steps += 1;
        go = (s.running & ~any) == 0ull && s.steps < kMsSteps && s.err == 0ull && *s.call == 0;
    } else {
        go = cnt > 0 && s.level < s.max_levels;
    }
    if (go || !server) s.alive = 0;                 // a server's host reads the last iteration's
    cudaGraphSetConditional(handle, go ? 1u : 0u);
}

// Admission, phase A: lanes in `mask` start over -- clear their bits in every
// lane word and their level rows.
__global__ void ms_admit_clear(MsState* S, unsigned long long mask, const int32_t* lanes, int nlanes,
                               unsigned long long running) {
    MsState& s = *S;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const unsigned long long keep = ~mask;
    for (int64_t v = tid; v < s.n; v += stride) {
        if (s.vn[v].x & mask) s.vn[v].x &= keep;
        if (s.f[s.cur][v] & mask) s.f[s.cur][v] &= keep;
        if (s.vn[v].y & mask) s.vn[v].y &= keep;
    }
    const int64_t total = (int64_t)nlanes * s.n;
    for (int64_t x = tid; x < total; x += stride) {
        const int64_t q = x / s.n;
        const int r = lanes[q];
        if (r < 0 || r >= 64) { ms_fault(S, 7, (uint64_t)x, (uint64_t)r); continue; }
        s.levels[(int64_t)r * s.n + (x - q * s.n)] = -1;
        if (s.parents) s.parents[(int64_t)r * s.n + (x - q * s.n)] = -1;
    }
    if (tid == 0) {
        s.alive = 0;
        s.steps = 0;
        s.running = running;
    }
}

// Admission, phase B: lane lanes[q] starts from roots[q] at this iteration,
// computing parents when want_parents[q] != 0.
__global__ void ms_admit_roots(MsState* S, const int32_t* lanes, const int32_t* roots, const int32_t* want_parents,
                               int nlanes) {
    MsState& s = *S;
    const int q = threadIdx.x;
    if (q >= nlanes) return;
    const int r = lanes[q];
    const int32_t v = roots[q];
    if (r < 0 || r >= 64 || (uint64_t)(uint32_t)v >= (uint64_t)s.n) { ms_fault(S, 4, (uint64_t)r, (uint32_t)v); return; }
    const unsigned long long bit = 1ull << r;
    if (want_parents[q]) atomicOr(&s.parent_mask, bit);
    else atomicAnd(&s.parent_mask, ~bit);
    atomicOr(&s.vn[v].x, bit);
    atomicOr(&s.lanes, bit);
    s.pull = 0;                              // a new lane's first level: few entries, many vertices missing
    const unsigned long long old = atomicOr(s.f[s.cur] + v, bit);
    s.levels[(int64_t)r * s.n + v] = 0;
    if (s.parents) s.parents[(int64_t)r * s.n + v] = v;
    s.lane_start[r] = s.level;
    if (old == 0ull) {
        const unsigned long long pos = atomicAdd(&s.act_count[s.cur], 1ull);
        if (pos < (unsigned long long)s.n) s.act[s.cur][pos] = v;
        else ms_fault(S, 5, pos, (uint32_t)v);
    }
}

__global__ void ms_launch(MsState* S, unsigned long long running) {
    S->alive = 0;
    S->steps = 0;
    S->running = running;
}

int ms_sm_count() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
}

}  // namespace

// ---------------------------------------------------------- host side --
struct MsContext {
    DevBuf vn, f0, f1, act0, act1, pieces, state, roots;
    int64_t piece_cap = 0;
    cudaGraph_t graph[2] = {nullptr, nullptr};       // [without parents, with parents]
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    int expand_ctas_per_sm = 4;                       // launch shape, set by the autotuner
    int expand_threads = 256;
    ~MsContext() {
        for (int k = 0; k < 2; ++k) {
            if (exec[k]) cudaGraphExecDestroy(exec[k]);
            if (graph[k]) cudaGraphDestroy(graph[k]);
        }
    }
    void drop_graphs() {
        for (int k = 0; k < 2; ++k) {
            if (exec[k]) cudaGraphExecDestroy(exec[k]);
            if (graph[k]) cudaGraphDestroy(graph[k]);
            exec[k] = nullptr;
            graph[k] = nullptr;
        }
    }
};

void free_msbfs(bfs_graph* g) {
    delete g->ms;
    g->ms = nullptr;
}

namespace {

bfs_status ms_ensure(bfs_graph* g) {
    if (g->ms) return BFS_OK;
    MsContext* c = new (std::nothrow) MsContext();
    if (!c) return set_error(BFS_ERR_OUT_OF_MEMORY, "host allocation");
    const Layout& L = g->L;
    const int64_t n = L.n;
    bfs_status rc = BFS_OK;
    c->piece_cap = L.nnz / kMsPiece + L.nnz / kMsHub + 16;
    if (rc == BFS_OK) rc = c->vn.alloc(16 * n);
    if (rc == BFS_OK) rc = c->f0.alloc(8 * n);
    if (rc == BFS_OK) rc = c->f1.alloc(8 * n);
    if (rc == BFS_OK) rc = c->act0.alloc(4 * n);
    if (rc == BFS_OK) rc = c->act1.alloc(4 * n);
    if (rc == BFS_OK) rc = c->pieces.alloc(sizeof(Item) * c->piece_cap);
    if (rc == BFS_OK) rc = c->state.alloc(sizeof(MsState));
    if (rc == BFS_OK) rc = c->roots.alloc(sizeof(int32_t) * 64);
    if (rc != BFS_OK) { delete c; return rc; }
    MsState h;
    memset(&h, 0, sizeof(h));
    h.dir = L.dir.as<uint32_t>();
    h.rank = L.rank.as<uint32_t>();
    h.dir_stride = L.dir_stride;
    h.cp = L.cp.as<uint32_t>();
    h.cp_base = L.cp_base_d.as<int64_t>();
    h.ir_base = L.ir_base_d.as<int64_t>();
    h.ir = L.ir.as<int32_t>();
    h.p = L.p;
    h.nb = L.nb;
    h.n = n;
    h.nnz = L.nnz;
    h.vn = c->vn.as<ulonglong2>();
    h.deg = L.deg.as<uint32_t>();
    h.symmetric = g->symmetric;
    h.f[0] = c->f0.as<unsigned long long>();
    h.f[1] = c->f1.as<unsigned long long>();
    h.act[0] = c->act0.as<int32_t>();
    h.act[1] = c->act1.as<int32_t>();
    h.pieces = c->pieces.as<Item>();
    h.piece_cap = c->piece_cap;
    h.roots = c->roots.as<int32_t>();
    cudaError_t e = cudaMemcpy(c->state.ptr, &h, sizeof(h), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { delete c; return cuda_error(e, "cudaMemcpy(state)", __FILE__, __LINE__); }
    g->ms = c;
    return BFS_OK;
}

// One level: from the active vertices or the destinations (the kernels of the
// other side return at once), then the reduction.
void launch_ms_level(bfs_graph* g, cudaGraphConditionalHandle handle, int server, cudaStream_t st) {
    MsContext* c = g->ms;
    MsState* S = c->state.as<MsState>();
    const int sms = ms_sm_count();
    const int64_t ctas = (g->L.n + kMT - 1) / kMT;
    const size_t scratch = sizeof(MsScratch) * (size_t)(c->expand_threads / 32);
    ms_expand<<<sms * c->expand_ctas_per_sm, c->expand_threads, scratch, st>>>(S);
    ms_pieces<<<sms * 4, kMT, 0, st>>>(S);
    if (g->symmetric) ms_pull<<<(unsigned)std::min<int64_t>(ctas, (int64_t)sms * 8), kMT, 0, st>>>(S);
    ms_reduce<<<(unsigned)std::min<int64_t>(ctas, (int64_t)sms * 8), kMT, 0, st>>>(S, handle, server);
}

// Build the batch graph: reset, clear, roots, then WHILE(level) { expand,
// pieces, pull, reduce }.
bfs_status ms_build_graph(bfs_graph* g, int with_parents, cudaStream_t st) {
    MsContext* c = g->ms;
    if (c->exec[with_parents]) return BFS_OK;
    MsState* S = c->state.as<MsState>();
    const int sms = ms_sm_count();
    cudaGraph_t graph = nullptr;
    BFS_CUDA_TRY(cudaGraphCreate(&graph, 0));
    cudaGraphConditionalHandle handle;
    BFS_CUDA_TRY(cudaGraphConditionalHandleCreate(&handle, graph, 1, cudaGraphCondAssignDefault));
    // prologue nodes, captured
    cudaStream_t cs = nullptr;
    BFS_CUDA_TRY(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    BFS_CUDA_TRY(cudaStreamBeginCaptureToGraph(cs, graph, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
    ms_reset<<<1, 1, 0, cs>>>(S);
    ms_clear<<<sms * 8, kMT, 0, cs>>>(S);
    ms_roots<<<1, 64, 0, cs>>>(S);
    cudaGraph_t captured = nullptr;
    cudaError_t ce = cudaStreamEndCapture(cs, &captured);
    if (ce != cudaSuccess) {
        cudaStreamDestroy(cs);
        cudaGraphDestroy(graph);
        return cuda_error(ce, "capture of the batch prologue", __FILE__, __LINE__);
    }
    // the conditional loop after the prologue
    size_t nleaf = 0;
    BFS_CUDA_TRY(cudaGraphGetNodes(graph, nullptr, &nleaf));
    std::vector<cudaGraphNode_t> nodes(nleaf);
    BFS_CUDA_TRY(cudaGraphGetNodes(graph, nodes.data(), &nleaf));
    cudaGraphNode_t last = nullptr;
    for (auto nd : nodes) {                      // the prologue is a chain: its sink is the only node without successors
        size_t nout = 0;
        BFS_CUDA_TRY(cudaGraphNodeGetDependentNodes(nd, nullptr, nullptr, &nout));
        if (nout == 0) last = nd;
    }
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = handle;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t cond = nullptr;
    BFS_CUDA_TRY(cudaGraphAddNode(&cond, graph, &last, nullptr, 1, &cp));
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    BFS_CUDA_TRY(cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
    launch_ms_level(g, handle, 0, cs);
    ce = cudaStreamEndCapture(cs, &body);
    cudaStreamDestroy(cs);
    if (ce != cudaSuccess) {
        cudaGraphDestroy(graph);
        return cuda_error(ce, "capture of the batch level body", __FILE__, __LINE__);
    }
    (void)with_parents;
    cudaGraphExec_t exec = nullptr;
    ce = cudaGraphInstantiate(&exec, graph, 0);
    if (ce != cudaSuccess) {
        cudaGraphDestroy(graph);
        return cuda_error(ce, "cudaGraphInstantiate(batch)", __FILE__, __LINE__);
    }
    c->graph[with_parents] = graph;
    c->exec[with_parents] = exec;
    (void)st;
    return BFS_OK;
}

struct MsCall {
    const int32_t* roots;
    int32_t n_roots;
    int32_t max_levels;
    int32_t* levels;
    int32_t* parents;
    unsigned long long parent_mask;
};

bfs_status ms_run(bfs_graph* g, const int32_t* roots_host, int32_t n_roots, int32_t* levels, int32_t* parents,
                  bfs_batch_stats* stats, cudaStream_t st) {
    BFS_TRY(ms_ensure(g));
    MsContext* c = g->ms;
    const int wp = parents ? 1 : 0;
    BFS_TRY(ms_build_graph(g, wp, st));
    // per-call fields of the state block
    BFS_CUDA_TRY(cudaMemcpyAsync(c->roots.ptr, roots_host, sizeof(int32_t) * n_roots, cudaMemcpyHostToDevice, st));
    MsCall call{c->roots.as<int32_t>(), n_roots, (int32_t)std::min<int64_t>(g->L.n + 1, 0x7fffffff), levels, parents,
                parents ? ~0ull : 0ull};
    BFS_CUDA_TRY(cudaMemcpyAsync(reinterpret_cast<char*>(c->state.ptr) + offsetof(MsState, roots), &call,
                                 sizeof(MsCall), cudaMemcpyHostToDevice, st));
    BFS_CUDA_TRY(cudaGraphLaunch(c->exec[wp], st));
    if (stats) {
        MsState h;
        BFS_CUDA_TRY(cudaMemcpyAsync(&h, c->state.ptr, sizeof(h), cudaMemcpyDeviceToHost, st));
        BFS_CUDA_TRY(cudaStreamSynchronize(st));
        stats->n_levels = (int32_t)h.levels_done;
        stats->edges_scanned = (int64_t)h.edges;
    }
    return BFS_OK;
}

}  // namespace
}  // namespace bfsgb

using namespace bfsgb;

extern "C" bfs_status bfs_run_batch(bfs_graph_t g, const int32_t* roots, int32_t n_roots, int32_t* levels,
                                    int32_t* parents, bfs_batch_stats* stats, void* stream) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (!roots || !levels) return set_error(BFS_ERR_INVALID_ARG, "roots and levels are required");
    if (n_roots < 1 || n_roots > 64) return set_error(BFS_ERR_INVALID_ARG, "n_roots %d outside [1, 64]", n_roots);
    if (!is_device_pointer(levels) || (parents && !is_device_pointer(parents)))
        return set_error(BFS_ERR_INVALID_ARG, "levels and parents must be device pointers");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t hroots[64];
    if (is_device_pointer(roots)) {
        BFS_CUDA_TRY(cudaMemcpyAsync(hroots, roots, sizeof(int32_t) * n_roots, cudaMemcpyDeviceToHost, st));
        BFS_CUDA_TRY(cudaStreamSynchronize(st));
    } else {
        memcpy(hroots, roots, sizeof(int32_t) * n_roots);
    }
    for (int r = 0; r < n_roots; ++r)
        if (hroots[r] < 0 || (int64_t)hroots[r] >= g->L.n)
            return set_error(BFS_ERR_INVALID_ARG, "root %d outside [0, %lld)", hroots[r], (long long)g->L.n);
    if (g->autotune && !g->batch_tuned) {       // bfs_options.autotune: tune on the first batch's roots
        g->batch_tuned = true;
        BFS_TRY(bfs_batch_autotune(g, hroots, n_roots, levels, nullptr, nullptr, stream));
    }
    int expect = 0;
    if (!g->busy.compare_exchange_strong(expect, 1)) return set_error(BFS_ERR_BUSY, "another search on this graph is running");
    bfs_status rc = ms_run(g, hroots, n_roots, levels, parents, stats, st);
    if (rc == BFS_OK && !stats) {
        cudaError_t e = cudaStreamSynchronize(st);     // hroots is read by an async copy
        if (e != cudaSuccess) rc = cuda_error(e, "cudaStreamSynchronize", __FILE__, __LINE__);
    }
    g->busy.store(0);
    return rc;
}

extern "C" bfs_status bfs_batch_autotune(bfs_graph_t g, const int32_t* roots, int32_t n_roots, int32_t* levels,
                                         int32_t* best_threads, int32_t* best_ctas_per_sm, void* stream) {
    if (!g || !roots || !levels) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    if (n_roots < 1 || n_roots > 64) return set_error(BFS_ERR_INVALID_ARG, "n_roots %d outside [1, 64]", n_roots);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    BFS_TRY(ms_ensure(g));
    MsContext* c = g->ms;
    static const int threads[] = {128, 256, 512, 1024};
    static const int ctas[] = {1, 2, 4, 8, 16};
    cudaEvent_t e0, e1;
    BFS_CUDA_TRY(cudaEventCreate(&e0));
    BFS_CUDA_TRY(cudaEventCreate(&e1));
    float best = 1e30f;
    int bt = c->expand_threads, bc = c->expand_ctas_per_sm;
    bfs_status rc = BFS_OK;
    for (int t : threads) {
        for (int k : ctas) {
            if (t * k > 2048) continue;                 // threads resident per SM
            c->drop_graphs();
            c->expand_threads = t;
            c->expand_ctas_per_sm = k;
            float ms = 0.f;
            for (int rep = 0; rep < 2 && rc == BFS_OK; ++rep) {
                cudaEventRecord(e0, st);
                rc = bfs_run_batch(g, roots, n_roots, levels, nullptr, nullptr, stream);
                cudaEventRecord(e1, st);
                cudaEventSynchronize(e1);
                cudaEventElapsedTime(&ms, e0, e1);
            }
            if (rc != BFS_OK) break;
            if (ms < best) { best = ms; bt = t; bc = k; }
        }
        if (rc != BFS_OK) break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->drop_graphs();
    c->expand_threads = bt;
    c->expand_ctas_per_sm = bc;
    if (rc != BFS_OK) return rc;
    if (best_threads) *best_threads = bt;
    if (best_ctas_per_sm) *best_ctas_per_sm = bc;
    return BFS_OK;
}


// ===================================================================== server
// Continuous batching over resident graphs.  Every graph keeps up to 64 lanes
// of the bit-parallel search resident on the device; a server thread launches
// iterations (one BFS level of every running lane each) on each graph's own
// stream, so the graphs' work overlaps on the GPU.  A launch repeats iterations on
// the device until a lane's frontier empties, a queued request could take a free
// lane (the host calls) or kMsSteps of them ran.  Then the lanes that ended are
// retired (their level row is copied to a result buffer and the request
// completes) and queued requests are admitted into free lanes (a lane admitted at
// iteration s reports level = iteration + 1 - s).
// Graphs are admitted against an HBM budget by their footprint (layout, lane
// state and level rows); results awaiting collection count against it too, and
// admission of new requests pauses while they would not fit.
#include <condition_variable>
#include <deque>
#include <thread>
#include <unordered_map>

namespace bfsgb {
namespace {

struct ServeGraph {
    bfs_graph* g = nullptr;
    int lanes = 0;
    cudaStream_t stream = nullptr;
    DevBuf levels;                   // [lanes][n]
    DevBuf parents;                  // [lanes][n]: the smallest previous-level neighbour
    DevBuf admit;                    // lanes[64], roots[64], want_parents[64]
    bool lane_parents[64] = {};      // the query running in lane r asked for parents
    int32_t* h_admit = nullptr;      // pinned staging of `admit`
    unsigned long long* h_alive = nullptr;   // pinned copy of the alive mask
    int* h_call = nullptr;           // mapped: asks a launch's iterations to end (MsState::call)
    cudaGraphExec_t step = nullptr;  // WHILE(level): iterations until a lane ends or the host calls
    cudaGraph_t step_graph = nullptr;
    int64_t lane_ticket[64];
    unsigned long long running = 0;
    std::deque<int64_t> pending;
    int64_t footprint = 0;
    int64_t iterations = 0;
    std::atomic<bool> inflight{false};   // a launch is on the stream
    unsigned long long before = 0;   // lanes running in it
};

struct Request {
    int32_t graph = 0;
    int32_t root = 0;
    int state = 0;                   // 0 queued, 1 running, 2 done
    bool parents = false;            // submitted with BFS_QUERY_PARENTS
    std::chrono::steady_clock::time_point t_submit, t_done;
    int32_t* result = nullptr;       // device, once done: the level row (n), then the parent row (n) if asked
};

}  // namespace
}  // namespace bfsgb

struct bfs_server {
    cudaMemPool_t pool = nullptr;    // results; keeps up to kScratchKept bytes between them
    int64_t budget = 0;
    int64_t used = 0;                // resident graphs
    int64_t results_bytes = 0;       // results awaiting collection
    int max_lanes = 64;
    std::vector<bfsgb::ServeGraph*> graphs;
    std::unordered_map<int64_t, bfsgb::Request> req;
    std::mutex mu;
    std::condition_variable cv_work, cv_done;
    std::thread worker;
    bool stop = false;
    bool failed = false;
    char fail_msg[256] = {0};
    int64_t next_ticket = 1;
    int64_t queue_limit = 1 << 20;   // queued requests accepted before BFS_ERR_BUSY
    int64_t submitted = 0, completed = 0, rejected = 0, queued = 0;
    int64_t iterations = 0;
    int peak_lanes = 0;
    std::vector<double> lat_us;
    std::chrono::steady_clock::time_point t0;
    int device = 0;
};

namespace bfsgb {
namespace {

constexpr int64_t kMaxQueued = 1 << 20;      // default queue limit (bfs_server_set_queue_limit)

// A launch runs iterations on the device until a lane's frontier empties (its
// result is to be handed out, its place given to a queued request) or the host
// calls: no host round trip per level, as each used to cost (60-100 us with the
// worker's polling, several times the level on small graphs).
bfs_status build_step_graph(ServeGraph* sg) {
    cudaGraph_t graph = nullptr;
    BFS_CUDA_TRY(cudaGraphCreate(&graph, 0));
    sg->step_graph = graph;                        // released with the server graph
    cudaGraphConditionalHandle handle;
    BFS_CUDA_TRY(cudaGraphConditionalHandleCreate(&handle, graph, 1, cudaGraphCondAssignDefault));
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = handle;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t cond = nullptr;
    BFS_CUDA_TRY(cudaGraphAddNode(&cond, graph, nullptr, nullptr, 0, &cp));
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    BFS_CUDA_TRY(cudaStreamBeginCaptureToGraph(sg->stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
    launch_ms_level(sg->g, handle, 1, sg->stream);
    BFS_CUDA_TRY(cudaStreamEndCapture(sg->stream, &body));
    cudaGraphExec_t exec = nullptr;
    cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
    if (e != cudaSuccess) return cuda_error(e, "cudaGraphInstantiate(step)", __FILE__, __LINE__);
    sg->step = exec;
    return BFS_OK;
}

void release_graph(ServeGraph* sg) {
    if (sg->stream) cudaStreamSynchronize(sg->stream);
    if (sg->step) cudaGraphExecDestroy(sg->step);
    if (sg->step_graph) cudaGraphDestroy(sg->step_graph);
    if (sg->h_admit) cudaFreeHost(sg->h_admit);
    if (sg->h_alive) cudaFreeHost(sg->h_alive);
    if (sg->h_call) cudaFreeHost(sg->h_call);
    if (sg->stream) cudaStreamDestroy(sg->stream);
    sg->levels.release();
    sg->parents.release();
    sg->admit.release();
    if (sg->g) sg->g->busy.store(0);
}

void fail(bfs_server* s, const char* what) {
    std::lock_guard<std::mutex> lk(s->mu);
    s->failed = true;
    snprintf(s->fail_msg, sizeof(s->fail_msg), "%s", what);
    s->cv_done.notify_all();
}

// Retire the lanes whose frontier emptied in the launch that has finished.
bool finish_iteration(bfs_server* s, ServeGraph* sg) {
    if (sg->h_alive[2]) {
        char msg[160];
        snprintf(msg, sizeof(msg), "bounds check %llu failed on the device (%llu, %llu)",
                 (unsigned long long)sg->h_alive[2], (unsigned long long)sg->h_alive[3],
                 (unsigned long long)sg->h_alive[4]);
        fail(s, msg);
        return false;
    }
    const unsigned long long done = sg->before & ~sg->h_alive[0];
    const int64_t n = sg->g->L.n;
    std::vector<std::pair<int64_t, int32_t*>> fin;
    for (int r = 0; r < sg->lanes; ++r) {
        if (!(done & (1ull << r))) continue;
        void* buf = nullptr;
        const int rows = sg->lane_parents[r] ? 2 : 1;
        if (cudaMallocFromPoolAsync(&buf, rows * sizeof(int32_t) * n, s->pool, sg->stream) != cudaSuccess) { fail(s, "result allocation failed"); return false; }
        cudaMemcpyAsync(buf, sg->levels.as<int32_t>() + (int64_t)r * n, sizeof(int32_t) * n,
                        cudaMemcpyDeviceToDevice, sg->stream);
        if (rows == 2)
            cudaMemcpyAsync(static_cast<int32_t*>(buf) + n, sg->parents.as<int32_t>() + (int64_t)r * n,
                            sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, sg->stream);
        fin.push_back({sg->lane_ticket[r], static_cast<int32_t*>(buf)});
        sg->lane_ticket[r] = -1;
    }
    if (!fin.empty() && cudaStreamSynchronize(sg->stream) != cudaSuccess) { fail(s, "result copy failed"); return false; }
    std::lock_guard<std::mutex> lk(s->mu);
    sg->running &= ~done;
    sg->iterations += (int64_t)sg->h_alive[1];
    s->iterations += (int64_t)sg->h_alive[1];
    const auto now = std::chrono::steady_clock::now();
    for (auto& f : fin) {
        Request& q = s->req[f.first];
        q.state = 2;
        q.result = f.second;
        q.t_done = now;
        s->results_bytes += (q.parents ? 2 : 1) * sizeof(int32_t) * n;
        ++s->completed;
        s->lat_us.push_back(std::chrono::duration<double, std::micro>(now - q.t_submit).count());
    }
    if (!fin.empty()) s->cv_done.notify_all();
    return true;
}

// With the server's lock held: a launch in flight ends after its current level
// if a queued request could take a free lane.
void call(ServeGraph* sg) {
    const unsigned long long all = sg->lanes < 64 ? (1ull << sg->lanes) - 1ull : ~0ull;
    if (sg->inflight && !sg->pending.empty() && (sg->running & all) != all) *static_cast<volatile int*>(sg->h_call) = 1;
}

bool launch_iteration(bfs_server* s, ServeGraph* sg) {
    std::unique_lock<std::mutex> lk(s->mu);
    if (s->stop) return false;                       // the call that ends the last launch is not taken back
    // admission into free lanes, while the results would fit in the budget
    int nadm = 0;
    unsigned long long mask = 0;
    for (int r = 0; r < sg->lanes && !sg->pending.empty(); ++r) {
        if (sg->running & (1ull << r)) continue;
        // the result of a lane: its level row (and parent row)
        const int64_t row = (s->req[sg->pending.front()].parents ? 8 : 4) * sg->g->L.n;
        if (s->used + s->results_bytes + row > s->budget) break;     // wait for results to be collected
        const int64_t t = sg->pending.front();
        sg->pending.pop_front();
        --s->queued;
        Request& q = s->req[t];
        q.state = 1;
        sg->lane_ticket[r] = t;
        sg->running |= 1ull << r;
        sg->h_admit[nadm] = r;
        sg->h_admit[64 + nadm] = q.root;
        sg->h_admit[128 + nadm] = q.parents ? 1 : 0;
        sg->lane_parents[r] = q.parents;
        mask |= 1ull << r;
        ++nadm;
    }
    if (!sg->running) return false;
    *static_cast<volatile int*>(sg->h_call) = 0;     // under the lock: a later call stands
    MsState* S = sg->g->ms->state.as<MsState>();
    if (nadm) {
        int32_t* d = sg->admit.as<int32_t>();
        if (cudaMemcpyAsync(d, sg->h_admit, sizeof(int32_t) * 192, cudaMemcpyHostToDevice, sg->stream) != cudaSuccess) {
            lk.unlock(); fail(s, "admission copy failed"); return false;
        }
        ms_admit_clear<<<ms_sm_count() * 4, kMT, 0, sg->stream>>>(S, mask, d, nadm, sg->running);
        ms_admit_roots<<<1, 64, 0, sg->stream>>>(S, d, d + 64, d + 128, nadm);
    } else {
        ms_launch<<<1, 1, 0, sg->stream>>>(S, sg->running);
    }
    if (cudaGraphLaunch(sg->step, sg->stream) != cudaSuccess) {
        lk.unlock(); fail(s, "iteration launch failed"); return false;
    }
    cudaMemcpyAsync(sg->h_alive, reinterpret_cast<char*>(S) + offsetof(MsState, alive),
                    sizeof(unsigned long long) * 5, cudaMemcpyDeviceToHost, sg->stream);   // alive, steps, err, a, b
    sg->before = sg->running;
    sg->inflight = true;
    int lanes_now = 0;
    for (ServeGraph* x : s->graphs) lanes_now += __builtin_popcountll(x->running);
    if (lanes_now > s->peak_lanes) s->peak_lanes = lanes_now;
    return true;
}

// Every graph advances on its own: when its launch has finished (a stream
// query, no waiting on the other graphs) its lanes whose frontier emptied are
// retired, queued requests are admitted into free lanes, and the next launch
// is made.  Returns whether any graph made progress.
bool serve_pass(bfs_server* s) {
    std::vector<ServeGraph*> gs;
    {
        std::lock_guard<std::mutex> lk(s->mu);
        gs = s->graphs;
    }
    bool progressed = false;
    for (ServeGraph* sg : gs) {
        if (sg->inflight) {
            const cudaError_t q = cudaStreamQuery(sg->stream);
            if (q == cudaErrorNotReady) continue;
            sg->inflight = false;
            if (q != cudaSuccess) { fail(s, "iteration failed on the device"); return false; }
            if (!finish_iteration(s, sg)) return false;
            progressed = true;
        }
        if (launch_iteration(s, sg)) progressed = true;
        {
            std::lock_guard<std::mutex> lk(s->mu);
            if (s->failed) return false;
        }
    }
    return progressed;
}

void serve_loop(bfs_server* s) {
    cudaSetDevice(s->device);
    // a sleep takes some 70 us however short it is meant to be: the worker polls
    // that long before it sleeps
    constexpr int kSpins = 64;
    int idle = 0;
    for (;;) {
        {
            std::unique_lock<std::mutex> lk(s->mu);
            if (s->stop || s->failed) break;
            bool work = false;
            for (ServeGraph* sg : s->graphs) work |= sg->inflight.load() || (sg->running != 0) || !sg->pending.empty();
            if (!work) s->cv_work.wait_for(lk, std::chrono::milliseconds(1));
            if (s->stop) break;
        }
        if (serve_pass(s)) {
            idle = 0;
        } else if (++idle < kSpins) {    // iterations in flight and nothing finished yet
            std::this_thread::yield();
        } else {
            std::unique_lock<std::mutex> lk(s->mu);
            if (s->stop || s->failed) break;
            s->cv_work.wait_for(lk, std::chrono::microseconds(20));
        }
    }
    // leave no iteration in flight
    std::vector<ServeGraph*> gs;
    {
        std::lock_guard<std::mutex> lk(s->mu);
        gs = s->graphs;
    }
    for (ServeGraph* sg : gs)
        if (sg->inflight) { cudaStreamSynchronize(sg->stream); sg->inflight = false; }
}

}  // namespace
}  // namespace bfsgb

extern "C" {

bfs_status bfs_server_create(int64_t hbm_budget_bytes, int32_t max_lanes, bfs_server_t* out) {
    if (!out || hbm_budget_bytes <= 0 || max_lanes < 1 || max_lanes > 64)
        return set_error(BFS_ERR_INVALID_ARG, "bad server arguments (budget > 0, 1 <= max_lanes <= 64)");
    bfs_server* s = new (std::nothrow) bfs_server();
    if (!s) return set_error(BFS_ERR_OUT_OF_MEMORY, "host allocation");
    s->budget = hbm_budget_bytes;
    s->max_lanes = max_lanes;
    s->t0 = std::chrono::steady_clock::now();
    cudaGetDevice(&s->device);
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = s->device;
    const cudaError_t pe = cudaMemPoolCreate(&s->pool, &props);
    if (pe != cudaSuccess) {
        delete s;
        return cuda_error(pe, "cudaMemPoolCreate", __FILE__, __LINE__);
    }
    uint64_t keep = kScratchKept;
    cudaMemPoolSetAttribute(s->pool, cudaMemPoolAttrReleaseThreshold, &keep);
    s->worker = std::thread(serve_loop, s);
    *out = s;
    return BFS_OK;
}

bfs_status bfs_server_add_graph(bfs_server_t s, bfs_graph_t g, int32_t* graph_id) {
    if (!s || !g || !graph_id) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    int expect = 0;
    if (!g->busy.compare_exchange_strong(expect, 1)) return set_error(BFS_ERR_BUSY, "graph is in use");
    ServeGraph* sg = new (std::nothrow) ServeGraph();
    if (!sg) { g->busy.store(0); return set_error(BFS_ERR_OUT_OF_MEMORY, "host allocation"); }
    sg->g = g;
    for (auto& t : sg->lane_ticket) t = -1;
    const int64_t n = g->L.n;
    int64_t layout = 0;
    bfs_graph_footprint(g, &layout);
    const int64_t lane_state = 32 * n + 8 * n + (int64_t)sizeof(Item) * (g->L.nnz / kMsPiece + g->L.nnz / kMsHub + 16);
    int lanes = s->max_lanes;
    {
        std::lock_guard<std::mutex> lk(s->mu);
        while (lanes > 0 && s->used + layout + lane_state + 8 * n * (int64_t)lanes > s->budget) lanes /= 2;
    }
    if (lanes == 0) {
        delete sg;
        g->busy.store(0);
        return set_error(BFS_ERR_OUT_OF_MEMORY, "graph does not fit the server's HBM budget");
    }
    sg->lanes = lanes;
    sg->footprint = layout + lane_state + 8 * n * (int64_t)lanes;
    bfs_status rc = ms_ensure(g);
    if (rc == BFS_OK) rc = sg->levels.alloc(sizeof(int32_t) * n * lanes);
    if (rc == BFS_OK) rc = sg->parents.alloc(sizeof(int32_t) * n * lanes);
    if (rc == BFS_OK) rc = sg->admit.alloc(sizeof(int32_t) * 192);
    if (rc == BFS_OK && cudaMallocHost(reinterpret_cast<void**>(&sg->h_admit), sizeof(int32_t) * 192) != cudaSuccess)
        rc = set_error(BFS_ERR_OUT_OF_MEMORY, "pinned host allocation");
    if (rc == BFS_OK && cudaMallocHost(reinterpret_cast<void**>(&sg->h_alive), sizeof(unsigned long long) * 5) != cudaSuccess)
        rc = set_error(BFS_ERR_OUT_OF_MEMORY, "pinned host allocation");
    if (rc == BFS_OK && cudaHostAlloc(reinterpret_cast<void**>(&sg->h_call), sizeof(int),
                                      cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess)
        rc = set_error(BFS_ERR_OUT_OF_MEMORY, "pinned host allocation");
    if (rc == BFS_OK && cudaStreamCreateWithFlags(&sg->stream, cudaStreamNonBlocking) != cudaSuccess)
        rc = set_error(BFS_ERR_CUDA, "stream creation failed");
    if (rc == BFS_OK) {
        MsState* S = g->ms->state.as<MsState>();
        MsCall call{g->ms->roots.as<int32_t>(), lanes, 0x7fffffff, sg->levels.as<int32_t>(), sg->parents.as<int32_t>(),
                    0ull};
        if (cudaMemcpyAsync(reinterpret_cast<char*>(S) + offsetof(MsState, roots), &call, sizeof(call),
                            cudaMemcpyHostToDevice, sg->stream) != cudaSuccess)
            rc = set_error(BFS_ERR_CUDA, "state copy failed");
        if (rc == BFS_OK) {
            *sg->h_call = 0;
            ms_reset<<<1, 1, 0, sg->stream>>>(S);
            ms_clear<<<ms_sm_count() * 8, kMT, 0, sg->stream>>>(S);
            const int* word = sg->h_call;            // unified addressing
            cudaMemcpyAsync(reinterpret_cast<char*>(S) + offsetof(MsState, call), &word, sizeof(word),
                            cudaMemcpyHostToDevice, sg->stream);
            if (cudaStreamSynchronize(sg->stream) != cudaSuccess) rc = set_error(BFS_ERR_CUDA, "lane state initialisation failed");
        }
    }
    if (rc == BFS_OK) rc = build_step_graph(sg);
    if (rc != BFS_OK) {
        release_graph(sg);
        delete sg;
        return rc;
    }
    std::lock_guard<std::mutex> lk(s->mu);
    s->used += sg->footprint;
    s->graphs.push_back(sg);
    *graph_id = (int32_t)s->graphs.size() - 1;
    return BFS_OK;
}

bfs_status bfs_server_submit(bfs_server_t s, int32_t graph_id, int32_t root, int64_t* ticket) {
    return bfs_server_submit_ex(s, graph_id, root, 0, ticket);
}

bfs_status bfs_server_submit_ex(bfs_server_t s, int32_t graph_id, int32_t root, int32_t flags, int64_t* ticket) {
    if (!s || !ticket) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    if (flags & ~BFS_QUERY_PARENTS) return set_error(BFS_ERR_INVALID_ARG, "unknown query flags 0x%x", flags);
    std::lock_guard<std::mutex> lk(s->mu);
    if (s->failed) return set_error(BFS_ERR_CUDA, "server failed: %s", s->fail_msg);
    if (graph_id < 0 || graph_id >= (int32_t)s->graphs.size()) return set_error(BFS_ERR_NOT_FOUND, "unknown graph id %d", graph_id);
    ServeGraph* sg = s->graphs[graph_id];
    if (root < 0 || (int64_t)root >= sg->g->L.n) return set_error(BFS_ERR_INVALID_ARG, "root %d outside [0, %lld)", root, (long long)sg->g->L.n);
    if (s->queued >= s->queue_limit) { ++s->rejected; return set_error(BFS_ERR_BUSY, "server queue is full"); }
    const int64_t t = s->next_ticket++;
    Request q;
    q.graph = graph_id;
    q.root = root;
    q.parents = (flags & BFS_QUERY_PARENTS) != 0;
    q.t_submit = std::chrono::steady_clock::now();
    s->req.emplace(t, q);
    sg->pending.push_back(t);
    call(sg);
    ++s->queued;
    ++s->submitted;
    *ticket = t;
    s->cv_work.notify_one();
    return BFS_OK;
}

bfs_status bfs_server_set_queue_limit(bfs_server_t s, int64_t limit) {
    if (!s || limit < 1 || limit > kMaxQueued)
        return set_error(BFS_ERR_INVALID_ARG, "queue limit outside [1, %lld]", (long long)kMaxQueued);
    std::lock_guard<std::mutex> lk(s->mu);
    s->queue_limit = limit;
    return BFS_OK;
}

bfs_status bfs_server_poll(bfs_server_t s, int64_t ticket, int32_t* done) {
    if (!s || !done) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(s->mu);
    auto it = s->req.find(ticket);
    if (it == s->req.end()) return set_error(BFS_ERR_NOT_FOUND, "unknown ticket %lld", (long long)ticket);
    *done = it->second.state == 2;
    return BFS_OK;
}

bfs_status bfs_server_wait(bfs_server_t s, int64_t ticket, int64_t timeout_us, int32_t* level, int32_t* parent) {
    if (!s) return set_error(BFS_ERR_INVALID_ARG, "NULL server");
    std::unique_lock<std::mutex> lk(s->mu);
    auto it = s->req.find(ticket);
    if (it == s->req.end()) return set_error(BFS_ERR_NOT_FOUND, "unknown ticket %lld", (long long)ticket);
    if (parent && !it->second.parents)
        return set_error(BFS_ERR_INVALID_ARG, "request %lld was submitted without BFS_QUERY_PARENTS", (long long)ticket);
    const auto deadline = std::chrono::steady_clock::now() + std::chrono::microseconds(timeout_us < 0 ? 0 : timeout_us);
    while (s->req[ticket].state != 2 && !s->failed) {
        if (s->cv_done.wait_until(lk, deadline) == std::cv_status::timeout && s->req[ticket].state != 2)
            return set_error(BFS_ERR_TIMEOUT, "request %lld not finished", (long long)ticket);
    }
    if (s->failed) return set_error(BFS_ERR_CUDA, "server failed: %s", s->fail_msg);
    Request q = s->req[ticket];
    s->req.erase(ticket);
    ServeGraph* sg = s->graphs[q.graph];
    const int64_t n = sg->g->L.n;
    s->results_bytes -= (q.parents ? 2 : 1) * sizeof(int32_t) * n;
    bool queued = false;
    for (ServeGraph* x : s->graphs) {
        queued |= !x->pending.empty();
        call(x);                                     // the budget may admit a queued request now
    }
    lk.unlock();
    bfs_status rc = BFS_OK;
    // the result was allocated stream-ordered and completed before the request
    // was marked done: copy it out and free it stream-ordered on the legacy stream
    if (level) {
        cudaError_t e = cudaMemcpyAsync(level, q.result, sizeof(int32_t) * n, cudaMemcpyDefault, 0);
        if (e != cudaSuccess) rc = cuda_error(e, "result copy", __FILE__, __LINE__);
    }
    if (parent && rc == BFS_OK) {
        cudaError_t e = cudaMemcpyAsync(parent, q.result + n, sizeof(int32_t) * n, cudaMemcpyDefault, 0);
        if (e != cudaSuccess) rc = cuda_error(e, "result copy", __FILE__, __LINE__);
    }
    cudaFreeAsync(q.result, 0);
    cudaError_t e = cudaStreamSynchronize(0);
    if (rc == BFS_OK && e != cudaSuccess) rc = cuda_error(e, "result copy", __FILE__, __LINE__);
    if (queued) s->cv_work.notify_one();             // else the worker has nothing to gain from waking
    return rc;
}

bfs_status bfs_server_stats(bfs_server_t s, bfs_server_stats_t* st) {
    if (!s || !st) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(s->mu);
    memset(st, 0, sizeof(*st));
    st->submitted = s->submitted;
    st->completed = s->completed;
    st->rejected = s->rejected;
    st->queued = s->queued;
    st->iterations = s->iterations;
    st->peak_lanes = s->peak_lanes;
    st->graphs = (int32_t)s->graphs.size();
    st->hbm_used_bytes = s->used + s->results_bytes;
    std::vector<double> v = s->lat_us;
    if (!v.empty()) {
        std::sort(v.begin(), v.end());
        auto pct = [&](double q) { return v[std::min(v.size() - 1, (size_t)(q * (double)(v.size() - 1) + 0.5))]; };
        st->p50_us = pct(0.50);
        st->p99_us = pct(0.99);
        st->max_us = v.back();
    }
    return BFS_OK;
}

bfs_status bfs_server_destroy(bfs_server_t s) {
    if (!s) return BFS_OK;
    {
        std::lock_guard<std::mutex> lk(s->mu);
        s->stop = true;
        for (ServeGraph* sg : s->graphs)
            if (sg->h_call) *static_cast<volatile int*>(sg->h_call) = 1;
    }
    s->cv_work.notify_all();
    if (s->worker.joinable()) s->worker.join();
    for (auto& kv : s->req)
        if (kv.second.result) cudaFreeAsync(kv.second.result, 0);
    cudaStreamSynchronize(0);
    cudaMemPoolDestroy(s->pool);
    for (ServeGraph* sg : s->graphs) {
        release_graph(sg);
        delete sg;
    }
    delete s;
    return BFS_OK;
}

}  // extern "C"
