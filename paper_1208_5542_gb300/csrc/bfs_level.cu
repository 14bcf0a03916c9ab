// bfs_level.cu -- one level of the level-synchronous BFS (Alg. 1, 2, 3) on the
// virtual p x p block grid, and the bfs_run entry point.
//
// Per level k (f = frontier of level k, pi = visited, t = next frontier):
//   PLAIN (BIT, Alg. 1):   every block (i,j) reads the raw slice f_j and keeps
//                          the vertices whose column of A_{i,j} is nonempty
//                          (the directory test of its column index).
//   COMPRESS (WAH, Alg. 2): f_j is WAH-encoded once per source range j; every
//                          block-row i decodes stream j and tests its directory.
//   COMPRESS_SIEVE (DIR-WAH, Alg. 3): for every (j, i) the slice f_j is sieved
//                          by V_{i,j} and WAH-encoded; block (i,j) decodes its
//                          stream -- every decoded vertex has a nonempty
//                          column, so only its rank is looked up.
//   expansion:             for every decoded (u, block) item, every entry
//                          u -> v of its column: if v is not in pi, set t[v]
//                          and lower parent[v] to u (the (select, min) semiring).
//   reduce:                t = t & ~pi; pi |= t; level[v] = k + 1 for v in t;
//                          |t| counted on the device; f <- t.
// The exchange itself (Alg. 2, 3) is the identity on one GPU: the receive buffer
// g' is the send buffer in HBM; its sizes are scanned for the statistics and
// packed into the caller's trace when one is requested.
//
// Dense levels of large graphs are expanded row-affine: a block (i,j) only
// ever writes destinations of range i, so a persistent CTA settles on one
// block-row at a time and keeps that row's visited bits pi_i -- and its own
// partial next bits t_i, where both fit -- in shared memory; its warps take
// the row's units.  The partial t_i of every CTA is OR-folded into t when the
// CTA leaves the row (the fold of the 2D partition, done through L2).  All
// other levels hand their units out as one list in the order of the block-rows,
// cut finer when there are few.
//
// Bottom-up levels (the hybrid traversal the paper names in Sec. VIII and IX,
// when enabled): the exchange is the same, its streams are decoded into a
// bitmap, and every unvisited vertex v of range i scans its columns in blocks
// (j, i), j = 0 .. p-1, for a neighbour in the frontier delivered to block
// (i, j); the first range with one gives v the smallest of them as its
// parent.  The device picks each level's direction (level_next), and the
// kernels of the other direction return at once.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "internal.h"
#include "wah.cuh"

namespace bfsgb {

int64_t parallel_encode_chunks(int64_t max_nbits, int wah_bits);
bfs_status launch_wah_encode_parallel(const EncodeArgs& a, int wah_bits, void* sums, void* bases, int64_t cps,
                                      void* flags, unsigned long long* setbits, int grid, cudaStream_t st);
size_t parallel_encode_sum_bytes();
size_t parallel_encode_base_bytes();

namespace {

constexpr int kNT = 256;            // threads of the small kernels
constexpr int kXT = 1024;           // threads of the expansion CTAs
constexpr int kXW = kXT / 32;       // warps of the expansion CTAs
// Columns of at least this many entries take the whole warp (32: scale 26 11.75
// -> 12.16 ms, scale 24 PLAIN 2.76 -> 2.90; 128: the same as 64).
constexpr uint32_t kCoop = 64;
constexpr uint32_t kHub = 2048;     // columns longer than this are cut into pieces of this size
constexpr uint32_t kHubSparse = 512;  // the same on levels with fewer units than warps
// Below this many vertices all visited bits (256 KB) are about as good as in L1
// and no level loads a row window.  A search without it / with it: scale 21
// 0.93 / 0.90 ms, scale 22 1.14 / 0.97, scale 23 2.32 / 1.83, scale 24 PLAIN
// 3.19 / 2.76; from 2^18 on instead: scale 20 0.56 -> 0.58 ms, a directed
// uniform graph of 1M vertices 0.45 -> 0.48.
constexpr int64_t kWindowMinVertices = 1 << 21;
constexpr int64_t kSmemLimit = 227 * 1024;

// Per-level values that the device keeps from level to level, so that one
// level is the same launch sequence every time (and a CUDA graph can repeat it).
struct LevelCtl {
    int64_t frontier;      // vertices of the current frontier
    int64_t visited;       // vertices visited so far
    int32_t level;         // current level k
    int32_t window;        // the expansion loads the row window (dense levels)
    int32_t win_ratio;     // entries of the frontier per vertex of the graph from which on it does
    int32_t dedup;         // read the parent before updating it
    int32_t go;            // 1 while another level follows
    int64_t m_f;           // degree sum of the frontier
    int64_t m_u;           // degree sum of the unvisited vertices
    int32_t bu;            // 1: this level runs bottom-up
    int32_t policy;        // BFS_DIRECTION_*
    int32_t alpha, beta;   // thresholds of the hybrid
    unsigned int done;     // CTAs of reduce_level that have finished
};

struct LevelArgs {
    // layout
    const uint32_t* dir;
    const uint32_t* rank;
    int64_t dir_stride;
    const uint32_t* cp;
    const int64_t* cp_base;
    const int64_t* ir_base;
    const int32_t* ir;
    int p;
    int64_t nb, n;
    // state
    const uint32_t* f;
    const uint32_t* pi;
    uint32_t* t;
    const uint8_t* fsum;                // frontier summary: 1 per 1024 bits of f with a set bit
    const uint32_t* fwords;             // the same per word: bit w of fwords says that word w of f is nonzero
    int32_t* parent;
    // exchange
    const void* xbuf;
    int64_t slot_cap;
    const int64_t* xcount;
    int64_t* chunk_base;
    int64_t chunks_per_slot;
    int64_t* slot_unit_base;            // p*p + 1: WAH units of slot s are [base[s], base[s+1])
    const uint8_t* fmt;                 // per-slot format of the level-adaptive exchange, or nullptr (WAH)
    // work distribution (per level)
    unsigned long long* row_next;       // p
    unsigned long long* row_piece_count;// p
    unsigned long long* row_piece_next; // p
    const int64_t* row_piece_base;      // p
    const int64_t* row_piece_cap;       // p
    Item* pieces;
    unsigned long long* ctr;
    int mode;
    int64_t plain_upb;                  // PLAIN units per block
    int64_t win_words;                  // words of the shared-memory row window (0: none)
    // compressed row exchange (the fold of the 2D partition): per block (i,j)
    // the destinations it reached, t_{i,j}, as a bitmap of range i; the
    // encoder turns t_{i,j} & ~pi_i into the row buffer of slot i*p + j
    uint32_t* tblk;                     // p*p partial bitmaps, dir_stride words each
    const void* rowbuf;                 // row buffers: p*p slots of row_cap words
    int64_t row_cap;
    const int64_t* row_count;           // words in each row buffer
    const int64_t* row_first;           // per (slot, chunk): first word and its first group
    const int64_t* col_first;           // the same for the column slots (bottom-up levels)
    int64_t row_cps;                    // encoder chunks per slot
    int64_t row_bcps;                   // fold chunks per range
    const LevelCtl* ctl;                // this level's values
    // bottom-up levels
    uint32_t* gbits;                    // decoded streams (n bits, OR over the block-rows)
    int range_aligned;                  // 1: ranges start at word boundaries (n_b a multiple of 32)
    int64_t g_words;                    // its uint32 words (a multiple of 4)
    const int64_t* bu_ptr;              // bottom-up rows: offsets (n + 1)
    const int32_t* bu_adj;              // bottom-up rows: neighbour ids
};

__device__ __forceinline__ int64_t range_begin(const LevelArgs& a, int64_t b) {
    const int64_t x = b * a.nb;
    return x < a.n ? x : a.n;
}

// -------------------------------------------------------------- visiting --
// Visit entry u -> v: if v was not visited before this level, lower parent[v]
// to u and set v's next bit.  The parent update is a reduction whose result
// is not used (fire-and-forget at L2).  WIN says what the CTA's row window in
// shared memory holds:
//   kWinNone  nothing: the visited word is read through the read-only path (pi
//             does not change during the expansion) and the next bit is a
//             reduction at L2;
//   kWinPi    the visited bits pi_i of the row; the next bit goes to L2 (or,
//             with the row exchange, to the visiting block's partial);
//   kWinBoth  pi_i and the CTA's partial next bits t_i.
enum Window : int { kWinNone = 0, kWinPi = 1, kWinBoth = 2 };
constexpr uint32_t kNoVertex = 0xffffffffu;

template <int WIN, bool DEDUP, bool ROWX>
struct Visitor {
    const uint32_t* s_pi;
    uint32_t* s_t;
    uint32_t rb;    // first vertex of the row
    uint32_t* tb;   // row exchange: the partial bitmap of the visiting block (i,j), or nullptr
    uint32_t jb;    // row exchange: first vertex of the block's source range j
    // The visited word of v (loads of several entries are issued before
    // their visits, so that their latencies overlap).
    __device__ __forceinline__ uint32_t probe(const LevelArgs& a, uint32_t v) const {
        if (WIN != kWinNone) return s_pi[(v - rb) >> 5];
        return __ldg(a.pi + (v >> 5));
    }
    __device__ __forceinline__ bool fresh(uint32_t v, uint32_t piw) const {
        const uint32_t b = WIN != kWinNone ? v - rb : v;
        return !((piw >> (b & 31u)) & 1u);
    }
    // The parent recorded so far for a fresh v (possibly an older value: the
    // parent only decreases during a level, from -1 = the largest unsigned).
    __device__ __forceinline__ uint32_t seen(const LevelArgs& a, uint32_t v) const {
        return __ldcg(reinterpret_cast<const unsigned int*>(a.parent) + v);
    }
    // The word of v's bit in the visiting block's partial t_{i,j} (row exchange).
    __device__ __forceinline__ uint32_t seen_t(uint32_t v) const { return __ldcg(tb + ((v - rb) >> 5)); }
    // After the visited word piw of v was probed: v <- kNoVertex if v was
    // visited before the level (nothing to do), else piw <- the parent read
    // first (DEDUP) or -1, and tw <- the partial's word read first (DEDUP with
    // the row exchange) or 0.
    __device__ __forceinline__ void stage(const LevelArgs& a, uint32_t& v, uint32_t& piw, uint32_t& tw) const {
        tw = 0u;
        if (v == kNoVertex || !fresh(v, piw)) {
            v = kNoVertex;
            return;
        }
        piw = DEDUP ? seen(a, v) : 0xffffffffu;
        if (DEDUP && ROWX) tw = seen_t(v);
    }
    // Visit of a fresh v from u, given an earlier read pv of its parent: when
    // pv <= u the visit changes nothing (pv != -1 means v already has a
    // visitor in this level, which set the next bit); otherwise lower the
    // parent, and the visitor that read -1 sets the next bit.  The visitor of
    // the first update read -1, so the bit is always set.
    __device__ __forceinline__ void mark(const LevelArgs& a, uint32_t v, uint32_t u, uint32_t pv, uint32_t tw) const {
        if (ROWX) {
            // Row exchange: every block that reaches v records it in its own
            // partial t_{i,j}.  The bit is already there when the word read
            // first has it, or when the parent read first lies in [jb, u]: a
            // visitor of the same source range lowered it and records v in
            // the same partial.  The parent is lowered when pv > u.
            const uint32_t vl = v - rb;
            const bool have = ((tw >> (vl & 31u)) & 1u) || (pv <= u && pv >= jb);
            if (pv > u) atomicMin(reinterpret_cast<unsigned int*>(a.parent) + v, u);
            if (!have) atomicOr(tb + (vl >> 5), 1u << (vl & 31u));
            return;
        }
        if (pv <= u) return;
        atomicMin(reinterpret_cast<unsigned int*>(a.parent) + v, u);
        if (pv != 0xffffffffu) return;
        if (WIN == kWinBoth) {
            const uint32_t vl = v - rb;
            atomicOr(s_t + (vl >> 5), 1u << (vl & 31u));
        } else {
            atomicOr(a.t + (v >> 5), 1u << (v & 31u));
        }
    }
};

// Entries per lane whose loads are in flight together.  The entries are read
// once per search: their loads are marked streaming (evict first), so that
// they do not push the visited, parent and next-bit lines out of L2 (-21% DRAM
// bytes at the growing level of a scale-24 search).
constexpr int kIlp = 4;
constexpr int kPieceIlp = 8;   // the piece kernel: long columns only, more entries in flight

// Scratch of one warp in shared memory: the nonempty words of its unit and the
// short columns of its batch, packed to the front, so that the owner of an
// item or entry is found by counting heads (below) and read in one access.
struct WarpScratch {
    uint4 word[32];        // bits, directory bits at the same vertices, first column, first vertex (local)
    uint32_t wexcl[32];    // items before the word
    uint32_t off[32];      // column offset minus the entries before it
    uint32_t u[32];        // column's source
};

__device__ __forceinline__ uint32_t lanes_below() { return (1u << lane_id()) - 1u; }

// All 32 lanes expand one column: ILP x 32 consecutive entries per step.
template <int WIN, bool DEDUP, bool ROWX, int ILP = kIlp>
__device__ __forceinline__ void warp_column(const LevelArgs& a, const Visitor<WIN, DEDUP, ROWX>& vis, uint32_t u,
                                            const int32_t* col, uint32_t len) {
    for (uint32_t e = lane_id(); e < len; e += 32 * ILP) {
        uint32_t v[ILP], w[ILP], t[ILP];
#pragma unroll
        for (int k = 0; k < ILP; ++k) v[k] = (e + 32 * k < len) ? (uint32_t)__ldcs(col + e + 32 * k) : kNoVertex;
#pragma unroll
        for (int k = 0; k < ILP; ++k) w[k] = (v[k] != kNoVertex) ? vis.probe(a, v[k]) : 0u;
#pragma unroll
        for (int k = 0; k < ILP; ++k) vis.stage(a, v[k], w[k], t[k]);
#pragma unroll
        for (int k = 0; k < ILP; ++k)
            if (v[k] != kNoVertex) vis.mark(a, v[k], u, w[k], t[k]);
    }
}

// How a level's units are shared out, from its number of units, frontier
// vertices and entries (the same for every CTA).  A unit is 32 words of one
// stream (or of one raw slice), which hold up to 992 vertices with columns of
// any length: a level with fewer units than warps would leave most of the chip
// idle, so its units are cut into `parts`, each taking every parts-th group of
// `bw` of the unit's items, and its long columns into shorter pieces.  A part
// decodes and looks up its whole unit again, so the parts stop at half the
// warps: uncut / half / twice the warps takes 314 / 198 / 197 us at scale 12,
// 409 / 331 / 334 at scale 17, 398 / 402 / 436 on a directed uniform graph of 1M,
// 975 / 935 / 962 at scale 22, 1805 / 1803 / 1828 at scale 23.  Pieces of 2048
// on all levels instead of down to 512: 331 -> 393 us at scale 17, 555 -> 631
// at scale 20 (926 against 962 at scale 22, where 512 is a little too short).
struct Split {
    uint32_t parts;        // power of two
    uint32_t bw;           // items per batch of a part (1..32)
    uint32_t hub;          // columns longer than this go to the piece list, in pieces of this size
};

__device__ __forceinline__ Split split_level(int64_t units, int64_t items, int64_t entries) {
    Split s{1u, 32u, kHub};
    const int64_t warps = (int64_t)gridDim.x * kXW;
    // pieces of about a quarter of a warp's share of the entries
    while (s.hub > kHubSparse && (int64_t)s.hub * 4 * warps > entries) s.hub /= 2;
    if (units <= 0 || units >= warps) return s;
    const int64_t avg = items / units > 1 ? items / units : 1;        // items per unit (at most: before the sieve)
    while (2 * (int64_t)s.parts * units < warps && s.parts < 256u && (int64_t)s.parts < avg) s.parts *= 2u;
    const int64_t bw = (avg + s.parts - 1) / s.parts;
    s.bw = bw < 32 ? (uint32_t)bw : 32u;
    return s;
}

// Expand one column per lane (source u, offset c0 of its column in the block's
// entries irb, length; length 0 = none).  Columns longer than the level's hub
// size go to the row's piece list; columns of at least kCoop entries are
// expanded by the whole warp one after the other; the short ones share the warp, 32
// consecutive entries of the concatenated columns per step: every column's
// first entry sets its bit in the step's head mask (one warp-wide OR), and the
// owner of an entry is the number of heads up to it.
template <int WIN, bool DEDUP, bool ROWX>
__device__ __forceinline__ void warp_expand(const LevelArgs& a, const Visitor<WIN, DEDUP, ROWX>& vis, int row,
                                            const Split& sp, const int32_t* irb, uint32_t u, uint32_t c0, uint32_t len,
                                            WarpScratch& ws, unsigned long long& edges, uint32_t& hits) {
    const uint32_t lane = lane_id();
    hits += (len > 0);
    edges += len;
    uint32_t hm = __ballot_sync(0xffffffffu, len > sp.hub);
    while (hm) {                            // the warp queues the column's pieces
        const int src = __ffs(hm) - 1;
        hm &= hm - 1;
        const uint32_t hl = __shfl_sync(0xffffffffu, len, src), hc = __shfl_sync(0xffffffffu, c0, src);
        const uint32_t hu = __shfl_sync(0xffffffffu, u, src);
        const uint32_t np = (hl + sp.hub - 1) / sp.hub;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(a.row_piece_count + row, (unsigned long long)np);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base + np <= (unsigned long long)a.row_piece_cap[row]) {
            Item* dst = a.pieces + a.row_piece_base[row] + base;
            for (uint32_t k = lane; k < np; k += 32) {
                Item it;
                it.u = (int32_t)hu;
                it.len = ((hl - k * sp.hub < sp.hub) ? hl - k * sp.hub : sp.hub);
                it.begin = (irb - a.ir) + (int64_t)hc + (int64_t)k * sp.hub;
                dst[k] = it;
            }
        } else if (lane == 0) {
            atomicOr(a.ctr + C_ERROR, 8ull);        // piece list overflow (cannot happen by the bound)
        }
        if (lane == (uint32_t)src) len = 0;
    }
    uint32_t coop = __ballot_sync(0xffffffffu, len >= kCoop);
    while (coop) {
        const int src = __ffs(coop) - 1;
        coop &= coop - 1;
        warp_column<WIN, DEDUP, ROWX>(a, vis, __shfl_sync(0xffffffffu, u, src),
                                      irb + __shfl_sync(0xffffffffu, c0, src), __shfl_sync(0xffffffffu, len, src));
    }
    if (len >= kCoop) len = 0;
    const uint32_t nz = __ballot_sync(0xffffffffu, len > 0);
    if (!nz) return;
    const uint32_t incl = warp_incl_sum(len);
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t excl = incl - len;
    __syncwarp();                           // the previous batch's readers are done
    if (len > 0) {
        const int r = __popc(nz & lanes_below());
        ws.off[r] = c0 - excl;
        ws.u[r] = u;
    }
    __syncwarp();
    const uint32_t upto = lanes_below() | (1u << lane);
    int before = -1;                        // the last head before the step
    for (uint32_t e0 = 0; e0 < total; e0 += 32 * kIlp) {
        uint32_t v[kIlp], w[kIlp], t[kIlp];
        int ow[kIlp];
#pragma unroll
        for (int k = 0; k < kIlp; ++k) {
            const uint32_t rel = excl - (e0 + 32 * k);
            const uint32_t heads = __reduce_or_sync(0xffffffffu, (len > 0 && rel < 32u) ? 1u << rel : 0u);
            const uint32_t e = e0 + 32 * k + lane;
            ow[k] = before + __popc(heads & upto);
            before += __popc(heads);
            v[k] = (e < total) ? (uint32_t)__ldcs(irb + (uint32_t)(ws.off[ow[k]] + e)) : kNoVertex;
        }
#pragma unroll
        for (int k = 0; k < kIlp; ++k) w[k] = (v[k] != kNoVertex) ? vis.probe(a, v[k]) : 0u;
#pragma unroll
        for (int k = 0; k < kIlp; ++k) vis.stage(a, v[k], w[k], t[k]);
#pragma unroll
        for (int k = 0; k < kIlp; ++k)
            if (v[k] != kNoVertex) vis.mark(a, v[k], ws.u[ow[k]], w[k], t[k]);
    }
}

// Column of source u_local in block b: (offset into ir, length); 0 if empty.
struct BlockView {
    const uint32_t* dir;
    const uint32_t* rank;
    const uint32_t* cp;
    int64_t ir0;
};

__device__ __forceinline__ BlockView block_view(const LevelArgs& a, int64_t b) {
    BlockView bv;
    bv.dir = a.dir + b * a.dir_stride;
    bv.rank = a.rank + b * a.dir_stride;
    bv.cp = a.cp + __ldg(a.cp_base + b);
    bv.ir0 = __ldg(a.ir_base + b);
    return bv;
}

__device__ __forceinline__ void column_of(const LevelArgs& a, const BlockView& bv, int64_t ul, int64_t* begin,
                                          uint32_t* len) {
    const uint32_t dw = __ldg(bv.dir + (ul >> 5));
    const uint32_t rk = __ldg(bv.rank + (ul >> 5));
    const uint32_t bit = 1u << (ul & 31);
    if (!(dw & bit)) {                  // a vertex of the directory's frontier must have a column
        *begin = 0;
        *len = 0;
        atomicOr(a.ctr + C_ERROR, 4ull);
        return;
    }
    const uint32_t c = rk + __popc(dw & (bit - 1u));
    const uint32_t c0 = __ldg(bv.cp + c), c1 = __ldg(bv.cp + c + 1);
    *begin = bv.ir0 + c0;
    *len = c1 - c0;
}

// Bring the L2 lines of a short column's entries on chip ahead of their use
// (long columns are read by the whole warp, coalesced).
__device__ __forceinline__ void prefetch_column(const int32_t* p0, uint32_t len) {
    if (len == 0 || len >= kCoop) return;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p0));
    const int32_t* p1 = p0 + (len - 1);
    if ((reinterpret_cast<uintptr_t>(p0) >> 7) != (reinterpret_cast<uintptr_t>(p1) >> 7))
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p1));
}

// Expand the vertices of one unit: lane l holds the bits x of 32 vertices of
// the source range from local vertex wb on (any alignment), `sieved` says that
// every one has a column (else the directory decides).  The directory bits and
// the first column's number are read once per word, and an item's column is a
// popcount away; the packed nonempty words number the unit's items, which the
// warp takes bw at a time (the part's share of them), the next batch's column
// lookups and prefetches issued before a batch is expanded.
template <int WIN, bool DEDUP, bool ROWX>
__device__ __forceinline__ void warp_words(const LevelArgs& a, const Visitor<WIN, DEDUP, ROWX>& vis, int row,
                                           const BlockView& bv, const Split& sp, uint32_t part, uint32_t jb, uint32_t x,
                                           uint32_t wb, bool sieved, WarpScratch& ws, unsigned long long& edges,
                                           uint32_t& hits) {
    uint32_t g = 0, cb = 0;
    if (x) {
        const uint32_t w = wb >> 5, sh = wb & 31u;
        const uint32_t d0 = __ldg(bv.dir + w), d1 = __ldg(bv.dir + w + 1);   // rows are padded
        g = __funnelshift_r(d0, d1, sh);
        cb = __ldg(bv.rank + w) + __popc(d0 & ((1u << sh) - 1u));
        if (sieved && (x & ~g)) atomicOr(a.ctr + C_ERROR, 4ull);            // a sieved vertex must have a column
        x &= g;
    }
    const uint32_t nz = __ballot_sync(0xffffffffu, x != 0u);
    if (!nz) return;
    const uint32_t cnt = __popc(x);
    const uint32_t incl = warp_incl_sum(cnt);
    const uint32_t items = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t excl = incl - cnt;
    __syncwarp();
    if (x) {
        const int r = __popc(nz & lanes_below());
        ws.word[r] = make_uint4(x, g, cb, wb);
        ws.wexcl[r] = excl;
    }
    __syncwarp();
    const int32_t* irb = a.ir + bv.ir0;
    const uint32_t upto = lanes_below() | (1u << lane_id());
    const uint32_t step = sp.parts * sp.bw;
    auto batch = [&](uint32_t q0, uint32_t& u, uint32_t& c0, uint32_t& len) {
        // heads before the batch, and in it
        const uint32_t rel = excl - q0;
        const uint32_t heads = __reduce_or_sync(0xffffffffu, (x && rel < 32u) ? 1u << rel : 0u);
        const int before = __popc(__ballot_sync(0xffffffffu, x && excl < q0)) - 1;
        const uint32_t q = q0 + lane_id();
        u = 0;
        c0 = 0;
        len = 0;
        if (q < items && lane_id() < sp.bw) {
            const int o = before + __popc(heads & upto);
            const uint4 wd = ws.word[o];
            const uint32_t b = (uint32_t)select32(wd.x, (int)(q - ws.wexcl[o]));
            const uint32_t c = wd.z + __popc(wd.y & ((1u << b) - 1u));
            c0 = __ldg(bv.cp + c);
            len = __ldg(bv.cp + c + 1) - c0;
            u = jb + wd.w + b;
            prefetch_column(irb + c0, len);
        }
    };
    uint32_t q0 = part * sp.bw;
    if (q0 >= items) return;
    uint32_t u, c0, len;
    batch(q0, u, c0, len);
    for (; q0 < items; q0 += step) {
        uint32_t un = 0, cn = 0, ln = 0;
        if (q0 + step < items) batch(q0 + step, un, cn, ln);
        warp_expand<WIN, DEDUP, ROWX>(a, vis, row, sp, irb, u, c0, len, ws, edges, hits);
        u = un;
        c0 = cn;
        len = ln;
    }
}

__device__ __forceinline__ void flush_counts(const LevelArgs& a, unsigned long long edges, unsigned long long hits) {
    edges = warp_sum(edges);
    hits = warp_sum(hits);
    if (lane_id() == 0) {
        if (edges) atomicAdd(a.ctr + C_EDGES, edges);
        if (hits) atomicAdd(a.ctr + C_HITS, hits);
    }
}

// Lane of the last of the 32 lanes whose exclusive count is <= q (the counts
// are nondecreasing over the lanes); every lane must call it.
__device__ __forceinline__ int owner_lane(uint32_t excl, uint64_t q) {
    int lo = 0, hi = 31;
#pragma unroll
    for (int step = 0; step < 5; ++step) {
        const int mid = (lo + hi + 1) >> 1;
        const uint32_t em = __shfl_sync(0xffffffffu, excl, mid);
        if ((uint64_t)em <= q) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ------------------------------------------------------------ row window --
// Leave the current row: fold the CTA's partial next bits into t (OR through
// L2).
__device__ void window_leave(const LevelArgs& a, uint32_t* s_t, int row) {
    const int64_t rb = range_begin(a, row);
    for (int64_t w = threadIdx.x; w < a.win_words; w += kXT) {
        const uint32_t x = s_t[w];
        if (!x) continue;
        const int64_t pos = rb + 32 * w;
        const int64_t gw = pos >> 5;
        const uint32_t sh = (uint32_t)(pos & 31);
        atomicOr(a.t + gw, x << sh);
        if (sh && (x >> (32 - sh))) atomicOr(a.t + gw + 1, x >> (32 - sh));
    }
}

// Enter a row: load pi_i into the window and, with kWinBoth, clear the partial
// next bits.
template <int WIN>
__device__ void window_enter(const LevelArgs& a, uint32_t* s_pi, uint32_t* s_t, int row) {
    const int64_t rb = range_begin(a, row);
    if ((rb & 127) == 0) {                  // 16-byte aligned words: copied four at a time (pi is padded past n)
        const uint4* src = reinterpret_cast<const uint4*>(a.pi + (rb >> 5));
        const int quads = (int)((a.win_words + 3) / 4);
        const int left = (int)((((a.n + 31) >> 5) - (rb >> 5) + 3) / 4);      // quads of pi from rb on
        uint4* dst = reinterpret_cast<uint4*>(s_pi);
        for (int q = threadIdx.x; q < quads; q += kXT)
            dst[q] = q < left ? __ldcg(src + q) : make_uint4(~0u, ~0u, ~0u, ~0u);
    } else {
        for (int64_t w = threadIdx.x; w < a.win_words; w += kXT) {
            const int64_t pos = rb + 32 * w;
            s_pi[w] = (pos < a.n) ? bits32_at_cg(a.pi, (uint64_t)pos) : 0xffffffffu;
        }
    }
    if (WIN == kWinBoth)
        for (int64_t w = threadIdx.x; w < a.win_words; w += kXT) s_t[w] = 0u;
}

// Hand out the units [0, total) of a level without a row window: a warp takes
// `batch` consecutive units at a time.  Few units (up to `deal` per warp) are dealt
// out in turn (no counter to wait for), many by a counter: a guided hand-out of a
// share of what is left (at least `batch`), so that early grabs are large and the
// last ones small.  The units come in the order of the block-rows; the share is one
// of a row's units, so that all warps work on about one row at a time (its
// visited, next and parent lines stay on chip).
// A heavy level (four entries per vertex of the graph) ends on two units at a time:
// with eight, or dealt out up to there, the warps with the last units keep the chip
// waiting (ms a search, scale 24 on 4 x 4 3.35 against 2.88, with the row exchange 3.99 /
// 3.44, PLAIN 2.98 / 2.73, unscrambled 18.5 / 9.7, uniform 20M 4.95 / 4.01; one at a
// time 2.84, 3.39, 2.65 and 3.95, but uniform 25M on 16 x 16 8.36 against 8.00).  The units
// of the others hold too little for that (PLAIN, uniform 2^25 of edge factor 2:
// 4.29 with eight, 4.67 with two).
struct HandOut {
    int64_t batch, deal;
};

__device__ __forceinline__ HandOut hand_out(const LevelArgs& a, int64_t total, int64_t light) {
    if (a.ctl->m_f < 4 * a.n) return HandOut{light, 4 * light};
    return HandOut{total > 4 * (int64_t)gridDim.x * kXW ? 2 : 1, 4};
}

template <typename Work>
__device__ __forceinline__ void flat_units(unsigned long long* counter, int64_t total, HandOut h, int rows,
                                           Work do_units) {
    const int64_t batch = h.batch;
    const int64_t warps = (int64_t)gridDim.x * kXW;
    if (total <= h.deal * warps) {
        const int64_t stride = warps * batch;
        for (int64_t x = ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * batch; x < total; x += stride)
            do_units(x, (x + batch < total) ? x + batch : total);
        return;
    }
    for (;;) {
        int64_t x = 0, b = batch;
        if (lane_id() == 0) {
            const int64_t cur = (int64_t)*reinterpret_cast<volatile unsigned long long*>(counter);
            if (cur < total) {
                const int64_t g = (total - cur) / (warps * rows);
                b = g > batch ? g : batch;
                x = (int64_t)atomicAdd(counter, (unsigned long long)b);
            } else {
                x = total;
            }
        }
        x = __shfl_sync(0xffffffffu, x, 0);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (x >= total) break;
        do_units(x, (x + b < total) ? x + b : total);
    }
}

// Row-affine persistent loop of a level with a row window.  The CTA settles on
// a block-row with units left; its warps take the row's units one at a time
// (warp-granular, no block barrier per unit; the same guided hand-out) until
// the row is drained, then the CTA folds its partial next bits into t, picks
// the next row with units left and loads that row's visited bits.  Every row
// is tried at most once per CTA.  row_begin(r) is the first unit of row r
// among all units of the level.
template <int WIN, typename Begin, typename Units, typename Work>
__device__ __forceinline__ void row_affine(const LevelArgs& a, unsigned long long* counters, int64_t batch,
                                           Begin row_begin, Units units_in_row, Work do_units, uint32_t* s_pi,
                                           uint32_t* s_t, int* s_row) {
    const int p = a.p;
    int tried = 0;
    int from = blockIdx.x % p;
    // warp 0: the next row with units left, 32 rows tested together, or -1
    auto pick = [&]() {
        if (threadIdx.x >= 32) return;
        int row = -1;
        while (tried < p && row < 0) {
            const int q = tried + (int)lane_id();
            int r = from + (int)lane_id();
            while (r >= p) r -= p;
            bool has = false;
            if (q < p)
                has = (int64_t)*reinterpret_cast<volatile unsigned long long*>(counters + r) < units_in_row(r);
            const uint32_t m = __ballot_sync(0xffffffffu, has);
            if (m) {
                row = from + __ffs(m) - 1;
                while (row >= p) row -= p;
            }
            const int skip = m ? __ffs(m) : 32;                      // rows this round leaves behind
            tried += skip;
            from += skip;
            while (from >= p) from -= p;
        }
        if (lane_id() == 0) s_row[0] = row;
    };
    pick();
    __syncthreads();
    int row = s_row[0];
    if (row >= 0) window_enter<WIN>(a, s_pi, s_t, row);
    __syncthreads();
    while (row >= 0) {
        const int64_t nu = units_in_row(row), u0 = row_begin(row);
        for (;;) {
            int64_t x = 0, b = batch;
            if (lane_id() == 0) {
                const int64_t cur = (int64_t)*reinterpret_cast<volatile unsigned long long*>(counters + row);
                if (cur < nu) {
                    const int64_t g = (uint32_t)(nu - cur) / (uint32_t)(gridDim.x * kXW);   // below 2^31 units
                    b = g > batch ? g : batch;
                    x = (int64_t)atomicAdd(counters + row, (unsigned long long)b);
                } else {
                    x = nu;
                }
            }
            x = __shfl_sync(0xffffffffu, x, 0);
            b = __shfl_sync(0xffffffffu, b, 0);
            if (x >= nu) break;
            do_units(u0 + x, u0 + ((x + b < nu) ? x + b : nu));
        }
        __syncthreads();
        if (WIN == kWinBoth) window_leave(a, s_t, row);
        pick();
        __syncthreads();
        row = s_row[0];
        if (row >= 0) window_enter<WIN>(a, s_pi, s_t, row);
        __syncthreads();
    }
}

// ---------------------------------------------------------------- kernels --
// Expansion of the WAH units (COMPRESS, COMPRESS_SIEVE).  Unit = 32 words of
// one stream, decoded by one warp: a warp scan of run lengths from the
// chunk's group base places every word, and warp_words expands the words'
// vertices (the two halves of a 64-bit word's group, and the words of a
// 1-fill, one after the other).
template <typename W, int WIN, bool DEDUP, bool ROWX>
__device__ __forceinline__ void expand_wah_level(const LevelArgs& a, uint32_t* s_pi, uint32_t* s_t, WarpScratch& ws,
                                                 int* s_row) {
    using T = Wah<W>;
    constexpr int GB = T::GB;
    const int p = a.p;
    unsigned long long edges = 0;
    uint32_t hits = 0;
    const bool sieved = a.mode == BFS_MODE_COMPRESS_SIEVE;
    const int64_t units = a.slot_unit_base[(int64_t)p * p];
    const Split sp = split_level(units, a.ctl->frontier * p, a.ctl->m_f);
    const int shift = __ffs((int)sp.parts) - 1;
    // the slot of the previous unit: a grab hands out consecutive units, so the
    // next one is mostly in the same slot or a few slots on
    int last_slot = -1;
    auto do_unit = [&](int64_t g, uint32_t part) {
        // unit -> (slot, chunk): the slot s with base[s] <= g < base[s+1]; the warp
        // searches 32-ary
        int sl = last_slot;
        if (sl >= 0 && a.slot_unit_base[sl + 1] <= g && sl + 2 <= p * p) ++sl;
        if (sl < 0 || a.slot_unit_base[sl] > g || a.slot_unit_base[sl + 1] <= g) {
            int lo = 0, hi = p * p - 1;
            while (lo < hi) {
                const int step = (hi - lo + 32) / 32;
                const int at = lo + step * (int)lane_id();
                const uint32_t m = __ballot_sync(0xffffffffu, at <= hi && a.slot_unit_base[at] <= g);
                lo += step * (31 - __clz(m));              // lane 0 always holds
                hi = lo + step - 1 < hi ? lo + step - 1 : hi;
            }
            sl = lo;
        }
        last_slot = sl;
        const int row = (int)((uint32_t)sl / (uint32_t)p);
        const int64_t s = sl, k = g - a.slot_unit_base[sl];
        const int64_t j = sl - row * p;
        const int64_t stream = sieved ? s : j;
        const uint32_t jb = (uint32_t)range_begin(a, j), jl = (uint32_t)range_begin(a, j + 1) - jb;
        const uint32_t G = jl / (uint32_t)GB;                          // a range is below 2^31 vertices
        const int r = (int)(jl - G * (uint32_t)GB);
        const W* in = static_cast<const W*>(a.xbuf) + stream * a.slot_cap;
        const int64_t count = a.xcount[stream];
        const int64_t xw = k * 32 + lane_id();
        const bool valid = xw < count;
        const W y = valid ? in[xw] : W(0);
        // per lane: the bits of its element's vertices from local vertex wbase
        // on; a 1-fill is a run of `run` vertices instead
        W wbits = W(0);
        uint32_t wbase = 0, run = 0;
        const int fm = a.fmt ? (int)a.fmt[stream] : FMT_WAH;
        if (fm == FMT_WAH) {
            const uint32_t glen = valid ? (uint32_t)word_groups<W>(y) : 0u;   // groups of a slot fit in 32 bits
            const uint32_t gincl = warp_incl_sum(glen);
            const uint32_t gs = (uint32_t)a.chunk_base[stream * a.chunks_per_slot + k] + (gincl - glen);
            if (valid) {
                if (gs < G) {
                    wbase = gs * GB;
                    if (is_fill<W>(y)) run = (y & T::VAL) ? glen * GB : 0u;
                    else wbits = T::from_payload(y);
                } else if (r > 0) {
                    wbase = G * GB;
                    wbits = T::from_active(y, r);                     // the active word
                }
            }
        } else if (valid) {
            const uint32_t e = (uint32_t)y;
            if (fm == FMT_LIST) {                                     // one vertex offset
                wbase = e;
                wbits = W(1);
            } else {                                                  // 32 bits of the raw slice
                wbase = (uint32_t)xw * 32u;
                wbits = (W)e;
            }
        }
        const BlockView bv = block_view(a, s);
        const Visitor<WIN, DEDUP, ROWX> vis{s_pi, s_t, (uint32_t)range_begin(a, row),
                                            ROWX ? a.tblk + s * a.dir_stride : nullptr, jb};
        // one pass per 32 bits of the words, then the words of the 1-fills:
        // lane l takes the vertices 32 l .. 32 l + 31 of every 1024 of a run
        uint32_t fills = __ballot_sync(0xffffffffu, run > 0);
        uint32_t left = 0, at = 0;
        for (int h = 0;; ++h) {
            uint32_t xb, wb;
            if (h < (int)(sizeof(W) / 4)) {
                xb = (uint32_t)(wbits >> (sizeof(W) == 8 && h == 1 ? 32 : 0));
                wb = wbase + 32u * (uint32_t)h;
            } else {
                if (left == 0) {
                    if (!fills) break;
                    const int o = __ffs(fills) - 1;
                    fills &= fills - 1;
                    left = __shfl_sync(0xffffffffu, run, o);
                    at = __shfl_sync(0xffffffffu, wbase, o);
                }
                const uint32_t f0 = 32u * lane_id();
                const uint32_t n1 = left > f0 ? left - f0 : 0u;
                xb = n1 >= 32u ? 0xffffffffu : (1u << n1) - 1u;
                wb = at + f0;
                const uint32_t took = left < 1024u ? left : 1024u;
                left -= took;
                at += took;
            }
            warp_words<WIN, DEDUP, ROWX>(a, vis, row, bv, sp, part, jb, xb, wb, sieved, ws, edges, hits);
        }
    };
    auto do_units = [&](int64_t x, int64_t xe) {
        for (; x < xe; ++x) do_unit(x >> shift, (uint32_t)x & (sp.parts - 1u));
    };
    if (WIN == kWinNone) {
        const int64_t each = (units << shift) / (2 * (int64_t)gridDim.x * kXW);   // few hand-outs per warp
        flat_units(a.row_next, units << shift, hand_out(a, units << shift, each < 1 ? 1 : (each < 8 ? each : 8)), p,
                   do_units);
    } else {
        auto row_begin = [&](int r) -> int64_t { return a.slot_unit_base[(int64_t)r * p] << shift; };
        auto units_in_row = [&](int r) -> int64_t {
            return (a.slot_unit_base[(int64_t)(r + 1) * p] - a.slot_unit_base[(int64_t)r * p]) << shift;
        };
        row_affine<WIN>(a, a.row_next, sp.parts > 1 ? 1 : 2, row_begin, units_in_row, do_units, s_pi, s_t, s_row);
    }
    flush_counts(a, edges, (unsigned long long)hits);
}

// Expansion of the PLAIN units.  Unit = (block (row, j), 32 raw frontier words
// of range j), one warp.  A hand-out tests up to 32 units against the frontier
// summary at once and expands those with a frontier bit.
template <int WIN, bool DEDUP>
__device__ __forceinline__ void expand_plain_level(const LevelArgs& a, uint32_t* s_pi, uint32_t* s_t, WarpScratch& ws,
                                                   int* s_row) {
    const int p = a.p;
    unsigned long long edges = 0;
    uint32_t hits = 0;
    const int64_t per_row = (int64_t)p * a.plain_upb;
    // the units that hold a frontier bit are at most the frontier's vertices, per block-row
    const int64_t live = min(per_row, a.ctl->frontier) * p;
    const Split sp = split_level(live, a.ctl->frontier * p, a.ctl->m_f);
    const int shift = __ffs((int)sp.parts) - 1;
    auto do_units = [&](int64_t x0, int64_t xe) {
        for (int64_t xb = x0; xb < xe; xb += 32) {
            const int64_t xl = xb + lane_id();
            bool has = false;
            if (xl < xe) {
                const uint32_t xu = (uint32_t)(xl >> shift), upb = (uint32_t)a.plain_upb;   // fits in 32 bits
                const uint32_t b = xu / upb;
                const int64_t c = xu - b * upb, j = b % (uint32_t)p;
                const int64_t g0 = range_begin(a, j) + c * 1024, g1 = min(g0 + 1024, range_begin(a, j + 1));
                has = g0 < g1 && (__ldcg(a.fsum + (g0 >> 10)) | __ldcg(a.fsum + ((g1 - 1) >> 10)));
            }
            uint32_t m = __ballot_sync(0xffffffffu, has);
            while (m) {
                const int64_t x = xb + __ffs(m) - 1;
                m &= m - 1;
                const uint32_t xu = (uint32_t)(x >> shift), upb = (uint32_t)a.plain_upb;
                const int64_t b = xu / upb, c = xu - (uint32_t)b * upb;
                const int row = (int)((uint32_t)b / (uint32_t)p);
                const int64_t j = b - (int64_t)row * p;
                const int64_t jb = range_begin(a, j), jl = range_begin(a, j + 1) - jb;
                const int64_t w = c * 32 + lane_id();
                uint32_t bits = 0;
                if (w * 32 < jl) {
                    bits = bits32_at_cg(a.f, (uint64_t)(jb + w * 32));
                    const int64_t left = jl - w * 32;
                    if (left < 32) bits &= (1u << left) - 1u;
                }
                const Visitor<WIN, DEDUP, false> vis{s_pi, s_t, (uint32_t)range_begin(a, row), nullptr, (uint32_t)jb};
                warp_words<WIN, DEDUP, false>(a, vis, row, block_view(a, b), sp, (uint32_t)x & (sp.parts - 1u),
                                              (uint32_t)jb, bits, (uint32_t)(32 * w), false, ws, edges, hits);
            }
        }
    };
    // sparse levels: many units per hand-out (few hold a vertex), as long as every warp
    // gets some; dense ones: few (balance)
    const int64_t total = (per_row << shift) * p;
    const int64_t each = (total + 4 * (int64_t)gridDim.x * kXW - 1) / (4 * (int64_t)gridDim.x * kXW);
    const bool dense = a.ctl->frontier * 64 >= a.n;
    const int64_t batch = dense ? (sp.parts > 1 ? 1 : 2) : (each < 32 ? each : 32);
    if (WIN == kWinNone) {
        flat_units(a.row_next, total, hand_out(a, total, dense ? (each < 8 ? each : 8) : batch), p, do_units);
    } else {
        auto row_begin = [&](int r) -> int64_t { return (per_row << shift) * r; };
        auto units_in_row = [&](int) -> int64_t { return per_row << shift; };
        row_affine<WIN>(a, a.row_next, batch, row_begin, units_in_row, do_units, s_pi, s_t, s_row);
    }
    flush_counts(a, edges, (unsigned long long)hits);
}

// Pieces of long columns, row by row: one warp per piece.
template <int WIN, bool DEDUP, bool ROWX>
__device__ __forceinline__ void expand_pieces_level(const LevelArgs& a, uint32_t* s_pi, uint32_t* s_t, int* s_row) {
    int row = 0;
    auto piece = [&](int64_t at) {
        const Item it = a.pieces[at];
        const uint32_t j = (uint32_t)it.u / (uint32_t)a.nb;               // the piece's source range
        const Visitor<WIN, DEDUP, ROWX> vis{s_pi, s_t, (uint32_t)range_begin(a, row),
                                            ROWX ? a.tblk + ((int64_t)row * a.p + j) * a.dir_stride : nullptr,
                                            (uint32_t)range_begin(a, j)};
        warp_column<WIN, DEDUP, ROWX, kPieceIlp>(a, vis, (uint32_t)it.u, a.ir + it.begin, it.len);
    };
    auto pieces_of = [&](int r) -> int64_t {
        return (int64_t)min(a.row_piece_count[r], (unsigned long long)a.row_piece_cap[r]);
    };
    if (WIN == kWinNone) {
        // the rows in turn: few pieces are dealt out over all warps, the pieces of
        // a long row handed out one by one
        const int64_t warps = (int64_t)gridDim.x * kXW;
        int64_t next = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;   // this warp's next piece among all
        int64_t begin = 0;                                                    // pieces of the rows before
        for (int r0 = 0; r0 < a.p; r0 += 32) {
            const int64_t mine = r0 + (int)lane_id() < a.p ? pieces_of(r0 + (int)lane_id()) : 0;
            uint32_t some = __ballot_sync(0xffffffffu, mine > 0);
            while (some) {
                const int l = __ffs(some) - 1;
                some &= some - 1;
                row = r0 + l;
                const int64_t n = __shfl_sync(0xffffffffu, mine, l), base = a.row_piece_base[row];
                if (n <= 4 * warps) {
                    for (; next < begin + n; next += warps) piece(base + next - begin);
                } else {
                    flat_units(a.row_piece_next + row, n, HandOut{1, 4}, 1, [&](int64_t x, int64_t xe) {
                        for (; x < xe; ++x) piece(base + x);
                    });
                    next += n;
                }
                begin += n;
            }
        }
    } else {
        auto row_begin = [&](int r) -> int64_t {
            row = r;
            return a.row_piece_base[r];
        };
        auto do_units = [&](int64_t x, int64_t xe) {
            for (; x < xe; ++x) piece(x);
        };
        row_affine<WIN>(a, a.row_piece_next, 1, row_begin, pieces_of, do_units, s_pi, s_t, s_row);
    }
}

// What bounds it: at scale 12 a level is one chain of dependent steps (9 units,
// once a warp each: 168 and 176 us for the two levels with entries; cut into
// parts 12); at a growing level the latency of scattered parent reads and L2
// reductions (scale 22: 12 M entries in 58 us and 42 of pieces, 22% issue activity,
// L2 at 18%; scale 24: 286 M in 1.1 ms, L2 at 50%); at the densest level issue slots
// (scale 22: 118 M entries in 435 us, 63% issue activity; 488 with a search for
// every entry's owner in place of head masks), and without the window the
// scattered reads of the visited words (scale 26: 1.5 G entries, 6.8 -> 6.5 ms).
//
// One launch expands a level: WIN is the window the graph's ranges allow, and
// the level's own values pick the body -- with the window on dense levels,
// without it on sparse ones (their visits are too few to pay for loading it),
// where DEDUP says whether the parent is read first.
template <typename W, int WIN, bool ROWX>
__global__ void __launch_bounds__(kXT, 1) expand_wah(LevelArgs a) {
    if (a.ctl->bu) return;                                // a bottom-up level
    extern __shared__ __align__(16) uint32_t s_win[];     // s_pi | s_t
    __shared__ WarpScratch s_ws[kXW];
    __shared__ int s_row[2];
    uint32_t* s_t = s_win + (a.win_words + 3) / 4 * 4;
    WarpScratch& ws = s_ws[threadIdx.x >> 5];
    if (WIN == kWinPi && a.ctl->window && a.ctl->dedup) {
        expand_wah_level<W, WIN, true, ROWX>(a, s_win, s_t, ws, s_row);
    } else if (WIN != kWinNone && a.ctl->window) {
        expand_wah_level<W, WIN, false, ROWX>(a, s_win, s_t, ws, s_row);
    } else if (a.ctl->dedup) {
        expand_wah_level<W, kWinNone, true, ROWX>(a, s_win, s_t, ws, s_row);
    } else {
        expand_wah_level<W, kWinNone, false, ROWX>(a, s_win, s_t, ws, s_row);
    }
}

template <int WIN>
__global__ void __launch_bounds__(kXT, 1) expand_plain(LevelArgs a) {
    if (a.ctl->bu) return;
    extern __shared__ __align__(16) uint32_t s_win[];
    __shared__ WarpScratch s_ws[kXW];
    __shared__ int s_row[2];
    uint32_t* s_t = s_win + (a.win_words + 3) / 4 * 4;
    WarpScratch& ws = s_ws[threadIdx.x >> 5];
    if (WIN == kWinPi && a.ctl->window && a.ctl->dedup) {
        expand_plain_level<WIN, true>(a, s_win, s_t, ws, s_row);
    } else if (WIN != kWinNone && a.ctl->window) {
        expand_plain_level<WIN, false>(a, s_win, s_t, ws, s_row);
    } else if (a.ctl->dedup) {
        expand_plain_level<kWinNone, true>(a, s_win, s_t, ws, s_row);
    } else {
        expand_plain_level<kWinNone, false>(a, s_win, s_t, ws, s_row);
    }
}

template <int WIN, bool ROWX>
__global__ void __launch_bounds__(kXT, 1) expand_pieces(LevelArgs a) {
    if (a.ctl->bu) return;
    extern __shared__ __align__(16) uint32_t s_win[];
    __shared__ int s_row[2];
    uint32_t* s_t = s_win + (a.win_words + 3) / 4 * 4;
    if (WIN == kWinPi && a.ctl->window && a.ctl->dedup) {
        expand_pieces_level<WIN, true, ROWX>(a, s_win, s_t, s_row);
    } else if (WIN != kWinNone && a.ctl->window) {
        expand_pieces_level<WIN, false, ROWX>(a, s_win, s_t, s_row);
    } else if (a.ctl->dedup) {
        expand_pieces_level<kWinNone, true, ROWX>(a, s_win, s_t, s_row);
    } else {
        expand_pieces_level<kWinNone, false, ROWX>(a, s_win, s_t, s_row);
    }
}

// ------------------------------------------------------------------ fold --
// OR the bits of v (bit q at image bit pos + q; at most 63 bits) into a
// shared-memory image of bitmap words.
template <typename W>
__device__ __forceinline__ void img_or(uint32_t* img, uint32_t pos, W v) {
    if (!v) return;
    const uint32_t w = pos >> 5, sh = pos & 31u;
    if constexpr (sizeof(W) == 4) {
        atomicOr(img + w, v << sh);
        if (sh && (v >> (32 - sh))) atomicOr(img + w + 1, v >> (32 - sh));
    } else {
        const unsigned long long x = v;
        const uint32_t w0 = (uint32_t)(x << sh);
        const uint32_t w1 = sh ? (uint32_t)(x >> (32 - sh)) : (uint32_t)(x >> 32);
        const uint32_t w2 = sh ? (uint32_t)(x >> (64 - sh)) : 0u;
        if (w0) atomicOr(img + w, w0);
        if (w1) atomicOr(img + w + 1, w1);
        if (w2) atomicOr(img + w + 2, w2);
    }
}

// Set the image bits [b0, b1), by the whole warp.
__device__ __forceinline__ void img_fill(uint32_t* img, uint32_t b0, uint32_t b1) {
    if (b1 <= b0) return;
    const uint32_t w0 = b0 >> 5, w1 = (b1 - 1) >> 5;
    for (uint32_t w = w0 + lane_id(); w <= w1; w += 32) {
        uint32_t mask = 0xffffffffu;
        if (w == w0) mask &= 0xffffffffu << (b0 & 31u);
        if (w == w1) mask &= 0xffffffffu >> (31u - ((b1 - 1) & 31u));
        atomicOr(img + w, mask);
    }
}

constexpr int kFT = 512;            // threads of the fold CTAs
constexpr int kFoldIlp = 4;         // word tiles whose loads a fold warp issues together

// Chunk-wise OR-decode of exchanged slots.  One CTA per (range b, chunk c of
// kEncChunkGroups groups of the range): its warps take the p slots that carry
// range b in turn, start at the word the encoder recorded for the chunk and
// decode the words covering the chunk's groups (and the active word, in the
// chunk that holds the range's last bits) into a shared-memory image of the
// destination's words; the image is then stored, the words shared with a
// neighbouring chunk or range ORed.  The destination is clear before.
//   ROWS = true: the fold of the compressed row exchange on a top-down level --
//     t_i is the OR over j of the row buffers (i, j), each the WAH stream of
//     t_{i,j} & ~pi_i; nothing else writes t on such a level.
//   ROWS = false: the column slots of a bottom-up level decoded into the one
//     bitmap the bottom-up scan reads -- the OR over the block-rows i of slots
//     (i, j) (COMPRESS_SIEVE) or slot j (COMPRESS); a raw slot of the adaptive
//     format is ORed word by word, vector slots are left to decode_vectors.
// Malformed streams set C_ERROR (16).
template <typename W, bool ROWS>
__global__ void __launch_bounds__(kFT) fold_slots(LevelArgs a) {
    if (ROWS ? a.ctl->bu : !a.ctl->bu) return;
    using T = Wah<W>;
    constexpr int GB = T::GB;
    constexpr int64_t CG = kEncChunkGroups;
    constexpr int64_t CBITS = CG * GB;
    constexpr int IW = (int)(CBITS / 32) + 2;
    constexpr int NW = kFT / 32;
    __shared__ uint32_t img[IW];
    __shared__ int s_err;
    const int p = a.p;
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const int64_t items = (int64_t)p * a.row_bcps;
    const bool sieve = a.mode == BFS_MODE_COMPRESS_SIEVE;
    const int nsrc = (ROWS || sieve) ? p : 1;                      // slots carrying one range
    const void* buf = ROWS ? a.rowbuf : a.xbuf;
    const int64_t cap = ROWS ? a.row_cap : a.slot_cap;
    const int64_t* counts = ROWS ? a.row_count : a.xcount;
    const int64_t* first = ROWS ? a.row_first : a.col_first;
    uint32_t* dst = ROWS ? a.t : a.gbits;
    for (int64_t q = blockIdx.x; q < items; q += gridDim.x) {
        const int b = (int)(q / a.row_bcps);
        const int64_t c = q - (int64_t)b * a.row_bcps;
        const int64_t ib = range_begin(a, b), nbits = range_begin(a, b + 1) - ib;
        const int64_t b0 = c * CBITS;
        if (b0 >= nbits) continue;
        const int64_t b1 = (b0 + CBITS < nbits) ? b0 + CBITS : nbits;
        const int64_t G = nbits / GB;
        const int r = (int)(nbits - G * GB);
        const int64_t nch = (G + CG - 1) / CG;
        const int64_t g_lo = c * CG, g_hi = (g_lo + CG < G) ? g_lo + CG : G;
        const uint32_t al = (uint32_t)((ib + b0) & 31);
        const int nimg = (int)((al + (b1 - b0) + 31) >> 5);
        for (int k = threadIdx.x; k < nimg; k += kFT) img[k] = 0u;
        if (threadIdx.x == 0) s_err = 0;
        __syncthreads();
        for (int x_src = warp; x_src < nsrc; x_src += NW) {
            const int64_t s = ROWS ? (int64_t)b * p + x_src : (sieve ? (int64_t)x_src * p + b : (int64_t)b);
            const int64_t count = counts[s];
            if (!ROWS && a.fmt) {
                const int fm = (int)a.fmt[s];
                if (fm == FMT_LIST) continue;                   // decode_vectors ORs the offsets
                if (fm == FMT_RAW) {                            // the slice's raw words of this chunk
                    const uint32_t* in = static_cast<const uint32_t*>(a.xbuf) + s * a.slot_cap;
                    const int64_t w0 = b0 >> 5, w1 = (b1 + 31) >> 5;
                    for (int64_t w = w0 + lane; w < w1 && w < count; w += 32) {
                        const uint32_t x = in[w];
                        if (x) img_or<uint32_t>(img, al + (uint32_t)(32 * w - b0), x);
                    }
                    continue;
                }
            }
            const W* in = static_cast<const W*>(buf) + s * cap;
            if (c < nch) {
                int64_t x0 = first[2 * (s * a.row_cps + c)];
                int64_t gpos = first[2 * (s * a.row_cps + c) + 1];
                // a run length is at most the slot's G groups: clamped to G + 1,
                // 32 of them sum within 32 bits (a longer fill is malformed and
                // still clipped to the chunk)
                const uint32_t lcap = (uint32_t)(G + 1);
                while (gpos < g_hi) {
                    if (x0 >= count) {                         // the words end before the groups do
                        if (lane == 0) s_err = 1;
                        break;
                    }
                    W y[kFoldIlp];                              // kFoldIlp tiles of 32 words in flight
#pragma unroll
                    for (int k = 0; k < kFoldIlp; ++k) {
                        const int64_t x = x0 + 32 * k + lane;
                        y[k] = (x < count) ? in[x] : W(0);
                    }
#pragma unroll
                    for (int k = 0; k < kFoldIlp; ++k) {
                        if (gpos >= g_hi || x0 >= count) break;   // warp-uniform
                        const int64_t x = x0 + lane;
                        const bool valid = x < count;
                        const bool fill = valid && is_fill<W>(y[k]);
                        uint32_t len = valid ? 1u : 0u, incl;
                        if (__any_sync(0xffffffffu, fill)) {
                            if (fill) {
                                const uint64_t l = word_groups<W>(y[k]);
                                len = l < lcap ? (uint32_t)l : lcap;
                            }
                            incl = warp_incl_sum(len);
                        } else {
                            // literals only: one group each; the lanes past the words are a suffix
                            const uint32_t nvalid = (count - x0 < 32) ? (uint32_t)(count - x0) : 32u;
                            incl = valid ? (uint32_t)lane + 1u : nvalid;
                        }
                        const int64_t gs = gpos + (int64_t)(incl - len);
                        bool one = false;
                        if (valid && gs < g_hi && gs + (int64_t)len > g_lo) {
                            if (!fill) img_or<W>(img, al + (uint32_t)((gs - g_lo) * GB), T::from_payload(y[k]));
                            else one = (y[k] & T::VAL) != W(0);
                        }
                        uint32_t m = __ballot_sync(0xffffffffu, one);
                        while (m) {                             // 1-fills, by the whole warp
                            const int o = __ffs(m) - 1;
                            m &= m - 1;
                            int64_t f0 = __shfl_sync(0xffffffffu, gs, o);
                            int64_t f1 = f0 + (int64_t)__shfl_sync(0xffffffffu, len, o);
                            if (f0 < g_lo) f0 = g_lo;
                            if (f1 > g_hi) f1 = g_hi;
                            img_fill(img, al + (uint32_t)((f0 - g_lo) * GB), al + (uint32_t)((f1 - g_lo) * GB));
                        }
                        x0 += 32;
                        gpos += (int64_t)__shfl_sync(0xffffffffu, incl, 31);
                    }
                }
            }
            // the active word holds the range's last r bits
            if (r > 0 && lane == 0 && G * GB >= b0 && G * GB < b1) {
                const W y = (count > 0) ? in[count - 1] : W(0);
                if (count <= 0 || (y >> r) != W(0)) s_err = 1;
                else img_or<W>(img, al + (uint32_t)(G * GB - b0), T::from_active(y, r));
            }
        }
        __syncthreads();
        const int64_t gw0 = (ib + b0) >> 5;
        // a word inside the chunk (or the bitmap's last, partial word) is this
        // CTA's alone: stored; a word shared with a neighbouring range is ORed.
        // With word-aligned ranges every word of the decoded bitmap is some
        // chunk's alone and is stored even when zero (no clearing pass)
        const bool store_zero = !ROWS && a.range_aligned;
        for (int k = threadIdx.x; k < nimg; k += kFT) {
            const uint32_t x = img[k];
            const int64_t wlo = (gw0 + k) * 32;
            const bool own = wlo >= ib + b0 && (wlo + 32 <= ib + b1 || ib + b1 >= a.n);
            if (own) {
                if (x || store_zero) dst[gw0 + k] = x;
            } else if (x) {
                atomicOr(dst + gw0 + k, x);
            }
        }
        if (threadIdx.x == 0 && s_err) atomicOr(a.ctr + C_ERROR, 16ull);
        __syncthreads();
    }
}

// ----------------------------------------------------- dynamic directory --
// The dynamic cross directory (Sec. V-B): D_{i,j}(u) = 1 while column u of
// block (i,j) still holds an entry into a vertex that is not visited; the
// sieve of exchange k sends f_j (.) D_{i,j}.  A bit matters only at the
// exchange that sends u (u is in one frontier only), and a cleared bit stays
// clear (the visited set only grows), so the bits of the frontier's vertices
// are evaluated from their definition just before the exchange: D starts as a
// copy of V each search, and every (u, i) with f_j(u) = D_{i,j}(u) = 1 whose
// column reaches only visited vertices is cleared.  pi holds the vertices
// visited up to this level, which is the state the synchronous update of
// every earlier visit leaves (the entries into the visited vertices have all
// been counted).  PLAIN-style units: (block (i,j), 32 words of range j), one
// warp; each item (u, i) is decided by its lane (the column's first kDynLane
// entries) and, for the rest of a long column, by the whole warp, stopping at
// the first unvisited destination.
constexpr uint32_t kDynStep = 8;      // entries a lane tests together
constexpr uint32_t kDynLane = 64;     // entries a lane tests before the warp takes over

__global__ void __launch_bounds__(kNT) dyn_sieve(LevelArgs a, uint32_t* __restrict__ ddir,
                                                 const uint8_t* __restrict__ fsum) {
    const int p = a.p;
    const int64_t units = (int64_t)p * p * a.plain_upb;
    const int64_t gw0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t gstride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = (int)lane_id();
    for (int64_t x = gw0; x < units; x += gstride) {
        const int64_t b = x / a.plain_upb, c = x - b * a.plain_upb;
        const int j = (int)(b % p);
        const int64_t jb = range_begin(a, j), jl = range_begin(a, j + 1) - jb;
        if (c * 1024 >= jl) continue;
        const int64_t g0 = jb + c * 1024;               // the unit's first global bit
        if (!fsum[g0 >> 10] && !fsum[(g0 + 1023) >> 10]) continue;   // no frontier bit (warp-uniform)
        const int64_t w = c * 32 + lane;
        uint32_t bits = 0;
        if (w * 32 < jl) {
            bits = bits32_at_cg(a.f, (uint64_t)(jb + w * 32));
            const int64_t left = jl - w * 32;
            if (left < 32) bits &= (1u << left) - 1u;
            if (bits) bits &= ddir[b * a.dir_stride + w];
        }
        const uint32_t cnt = __popc(bits);
        const uint32_t cincl = warp_incl_sum(cnt);
        const uint32_t cexcl = cincl - cnt;
        const uint32_t items = __shfl_sync(0xffffffffu, cincl, 31);
        if (items == 0) continue;
        const BlockView bv = block_view(a, b);
        // the column of item q0 + lane (none past the items); the next round's
        // lookups are issued before this round's scan, so that they overlap
        auto lookup = [&](uint32_t q0, int64_t& ul, int64_t& begin, uint32_t& len) {
            const uint32_t q = q0 + lane;
            const int o = owner_lane(cexcl, q < items ? q : items - 1);
            const uint32_t ob = __shfl_sync(0xffffffffu, bits, o);
            const uint32_t oex = __shfl_sync(0xffffffffu, cexcl, o);
            ul = -1;
            begin = 0;
            len = 0;
            if (q < items) {
                ul = (c * 32 + o) * 32 + select32(ob, (int)(q - oex));
                column_of(a, bv, ul, &begin, &len);
                prefetch_column(a.ir + begin, len);
            }
        };
        int64_t ul, begin;
        uint32_t len;
        lookup(0, ul, begin, len);
        for (uint32_t q0 = 0; q0 < items; q0 += 32) {
            int64_t ul_n = -1, begin_n = 0;
            uint32_t len_n = 0;
            if (q0 + 32 < items) lookup(q0 + 32, ul_n, begin_n, len_n);
            uint32_t e = 0;
            bool alive = ul < 0;
            // the lane scans its column kDynStep entries at a time (their loads
            // in flight together) up to kDynLane entries
            while (!alive && e < len && e < kDynLane) {
                int32_t v[kDynStep];
#pragma unroll
                for (uint32_t k = 0; k < kDynStep; ++k) v[k] = (e + k < len) ? __ldg(a.ir + begin + e + k) : -1;
#pragma unroll
                for (uint32_t k = 0; k < kDynStep; ++k)
                    if (v[k] >= 0 && !((__ldg(a.pi + ((uint32_t)v[k] >> 5)) >> ((uint32_t)v[k] & 31u)) & 1u))
                        alive = true;
                e += kDynStep;
            }
            // the rest of the long columns whose first kDynLane entries are all
            // visited: the whole warp, 32 entries a step, until an unvisited one
            uint32_t m = __ballot_sync(0xffffffffu, !alive && e < len);
            while (m) {
                const int l = __ffs(m) - 1;
                m &= m - 1;
                const int64_t lb = __shfl_sync(0xffffffffu, begin, l);
                const uint32_t ll = __shfl_sync(0xffffffffu, len, l);
                bool found = false;
                for (uint32_t e0 = kDynLane; e0 < ll && !found; e0 += 32) {
                    bool un = false;
                    if (e0 + lane < ll) {
                        const uint32_t v = (uint32_t)__ldg(a.ir + lb + e0 + lane);
                        un = !((__ldg(a.pi + (v >> 5)) >> (v & 31u)) & 1u);
                    }
                    found = __any_sync(0xffffffffu, un);
                }
                if (lane == l) alive = found;
            }
            if (!alive)
                atomicAnd(ddir + b * a.dir_stride + (ul >> 5), ~(1u << ((uint32_t)ul & 31u)));
            ul = ul_n;
            begin = begin_n;
            len = len_n;
        }
    }
}

// ------------------------------------------------------------- bottom-up --
// Zero the decoded bitmap (bottom-up levels only).
__global__ void __launch_bounds__(kNT) clear_gbits(LevelArgs a) {
    if (!a.ctl->bu) return;
    const int64_t quads = a.g_words / 4;
    uint4* q = reinterpret_cast<uint4*>(a.gbits);
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < quads; x += (int64_t)gridDim.x * blockDim.x)
        q[x] = make_uint4(0u, 0u, 0u, 0u);
}

// The exchanged slots that went as vectors of offsets, ORed into the bitmap
// that fold_slots decodes the others to (bottom-up levels of the level-adaptive
// format): offset q of slot (i, j) is bit begin(j) + q, ORed over the block-rows i.
// A block (i, j) only ever tests vertices u of range j with a neighbour in range
// i, whose bit its own slot carries (V_{i,j}(u) = 1): the OR holds exactly that
// bit, and one bitmap serves every block-row.  One warp per 32-element unit of
// the decoder's plan (COMPRESS: the plan of row 0, whose blocks hold the p slots
// once).
__global__ void __launch_bounds__(kNT) decode_vectors(LevelArgs a) {
    if (!a.ctl->bu) return;
    const int p = a.p;
    const bool sieve = a.mode == BFS_MODE_COMPRESS_SIEVE;
    const int nblk = sieve ? p * p : p;
    const int64_t total = a.slot_unit_base[nblk];
    // every warp takes a contiguous share of the units: the slot of the next
    // unit is the current one or a few on (one search per warp)
    const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t u0 = total * gw / nw, u1 = total * (gw + 1) / nw;
    int sl = -1;
    for (int64_t g = u0; g < u1; ++g) {
        if (sl < 0) {
            int lo = 0, hi = nblk - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (a.slot_unit_base[mid] <= g) lo = mid; else hi = mid - 1;
            }
            sl = lo;
        } else {
            while (sl + 1 < nblk && a.slot_unit_base[sl + 1] <= g) ++sl;
        }
        if (a.fmt[sl] != FMT_LIST) continue;
        const int64_t x = (g - a.slot_unit_base[sl]) * 32 + lane_id();
        if (x >= a.xcount[sl]) continue;
        const uint32_t* in = static_cast<const uint32_t*>(a.xbuf) + (int64_t)sl * a.slot_cap;
        const uint32_t v = (uint32_t)range_begin(a, sieve ? sl % p : sl) + in[x];
        atomicOr(a.gbits + (v >> 5), 1u << (v & 31u));
    }
}

// One bottom-up level: every unvisited vertex v of range i scans its columns
// in blocks (j, i) -- its neighbours in range j, the graph being undirected --
// for j = 0, 1, ..., testing each neighbour u against the frontier delivered
// to block (i, j) (the decoded slot, or the raw slice f_j in PLAIN mode).  The
// smallest frontier neighbour of the first range that has one is v's parent:
// the ranges are ordered intervals of ids, so it is the smallest neighbour of
// v on the previous level, and it is the smallest frontier neighbour seen
// once the scan has passed the end of its range.  v's columns are read from
// the bottom-up rows (stored back to back, range by range).  One warp per
// visited word (32 vertices): a row of at most kBuLane entries is scanned by
// its own lane (kBuIlp entries and their frontier words in flight), a longer
// one by the whole warp (kIlp x 32 entries per step); the warp's next bits
// are one store (t is clear and no other kernel writes it this level).
//
// The scattered frontier reads bound it: at scale 24 the first bottom-up level
// is about two thirds of the search.  Entries of a short row in flight: a row
// usually ends after a few, and what was read past its end is lost; 2 / 3 / 4 /
// 6 / 8 give 2.12 / 2.07 / 2.01 / 2.11 / 2.18 ms a search (adaptive format).
//
// A step over a short row tests its entries' ranges whether one hit or not: with
// a shortcut past that (32 registers, 64 warps per SM) the long rows' one-warp
// chains of a sparse level wait on all the others, and a bottom-up search at
// scale 22 takes 4.10 ms instead of 3.31 (40 registers, 48 warps), at scale 24
// 9.36 instead of 7.65.  The words are dealt out to twice the CTAs that fit at once,
// so that an SM that is done early takes another one: 8 / 12 / 16 / 24 CTAs per SM
// give 1.86 / 1.68 / 1.66 / 1.65 ms for a hybrid search at scale 24, 3.31 / 3.15 /
// 3.13 / 3.07 bottom-up at scale 22, 235.9 / 238.5 / 240.2 / 243.3 us hybrid at scale 17.
constexpr int64_t kBuLane = 32;
constexpr int kBuIlp = 4;
constexpr int kBuCtas = 12;         // CTAs per SM (6 are resident)

// The frontier test of an entry u.  A sparse frontier is tested word-wise
// first: `words` has a bit per 32 vertices (64 KB at scale 24, in L1, where
// the bitmap is 2 MB: 940 against 326 G scattered reads a second).  Below
// n / 64 vertices most words are empty and the test ends there (scale 24: 2.17
// ms a search, 2.23 never testing words); a denser frontier would read both.
struct BuFrontier {
    const uint32_t* g;        // the decoded streams, or the raw frontier (PLAIN)
    const uint32_t* words;    // bit (u / 32): the frontier has a vertex in that word; nullptr: a dense frontier
    __device__ __forceinline__ bool maybe(uint32_t u) const {
        return !words || ((__ldg(words + (u >> 10)) >> ((u >> 5) & 31u)) & 1u);
    }
    // whether the frontier delivered to block (i, range of u) holds u
    __device__ __forceinline__ bool test(uint32_t u) const { return (__ldg(g + (u >> 5)) >> (u & 31u)) & 1u; }
};

// STATS: also count the columns and entries read (the stepwise loop asks for them).
template <bool STATS>
__global__ void __launch_bounds__(kNT) expand_bottom_up(LevelArgs a) {
    if (!a.ctl->bu) return;
    const int64_t words = (a.n + 31) >> 5;
    const int64_t gw0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t gstride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t nb = (uint32_t)a.nb;                                // n < 2^31
    const uint32_t NONE = 0xffffffffu;
    const BuFrontier fr{a.mode != BFS_MODE_PLAIN ? a.gbits : a.f, a.ctl->frontier * 64 < a.n ? a.fwords : nullptr};
    unsigned long long edges = 0, cols = 0;
    for (int64_t w = gw0; w < words; w += gstride) {
        const uint32_t piw = __ldg(a.pi + w);
        if (piw == 0xffffffffu) continue;
        const int64_t v = w * 32 + lane_id();
        const bool mine = v < a.n && !((piw >> lane_id()) & 1u);
        int64_t e0 = 0, e1 = 0;
        if (mine) {
            e0 = __ldg(a.bu_ptr + v);
            e1 = __ldg(a.bu_ptr + v + 1);
        }
        uint32_t best = NONE;
        if (mine && e1 - e0 <= kBuLane) {
            uint32_t rend = 0;              // end of the range of the entries so far (STATS), of best's range (else)
            bool stop = false;
            for (int64_t e = e0; e < e1 && !stop; e += kBuIlp) {
                uint32_t u[kBuIlp];
                bool hit[kBuIlp];
#pragma unroll
                for (int k = 0; k < kBuIlp; ++k) u[k] = (e + k < e1) ? (uint32_t)__ldg(a.bu_adj + e + k) : NONE;
#pragma unroll
                for (int k = 0; k < kBuIlp; ++k) hit[k] = u[k] != NONE && fr.maybe(u[k]);
#pragma unroll
                for (int k = 0; k < kBuIlp; ++k)
                    if (hit[k]) hit[k] = fr.test(u[k]);
#pragma unroll
                for (int k = 0; k < kBuIlp; ++k) {
                    if (u[k] == NONE || stop) continue;
                    if (STATS) {
                        if (u[k] >= rend) {                             // a new range
                            if (best != NONE) { stop = true; continue; }
                            rend = (u[k] / nb + 1u) * nb;
                            ++cols;
                        }
                        ++edges;
                    } else if (best != NONE && u[k] >= rend) {
                        stop = true;                                    // past the range of the first hit
                        continue;
                    }
                    if (hit[k]) {
                        if (!STATS && best == NONE) rend = (u[k] / nb + 1u) * nb;
                        best = u[k] < best ? u[k] : best;
                    }
                }
            }
        }
        // long rows, one after the other, by the whole warp
        uint32_t lm = __ballot_sync(0xffffffffu, mine && e1 - e0 > kBuLane);
        while (lm) {
            const int o = __ffs(lm) - 1;
            lm &= lm - 1;
            const int64_t b0 = __shfl_sync(0xffffffffu, e0, o), b1 = __shfl_sync(0xffffffffu, e1, o);
            uint32_t wb = NONE, wend = NONE;                            // best so far and the end of its range
            uint32_t jlast = NONE;                                      // range of the last entry scanned (STATS)
            for (int64_t e = b0; e < b1; e += kIlp * 32) {
                uint32_t u[kIlp];
                bool hit[kIlp];
#pragma unroll
                for (int k = 0; k < kIlp; ++k) {
                    const int64_t x = e + k * 32 + lane_id();
                    u[k] = (x < b1) ? (uint32_t)__ldg(a.bu_adj + x) : NONE;
                }
#pragma unroll
                for (int k = 0; k < kIlp; ++k) hit[k] = u[k] != NONE && fr.maybe(u[k]);
                uint32_t cand = NONE;
                bool past = false;
#pragma unroll
                for (int k = 0; k < kIlp; ++k) {
                    if (hit[k] && u[k] < cand && fr.test(u[k])) cand = u[k];
                    if (STATS) {            // entries (in row order) that open a range
                        const uint32_t j = u[k] != NONE ? u[k] / nb : NONE;
                        uint32_t jp = __shfl_up_sync(0xffffffffu, j, 1);
                        if (lane_id() == 0) jp = jlast;
                        const uint32_t opens = __ballot_sync(0xffffffffu, u[k] != NONE && j != jp);
                        const uint32_t valid = __ballot_sync(0xffffffffu, u[k] != NONE);
                        if (lane_id() == (uint32_t)o) { cols += __popc(opens); edges += __popc(valid); }
                        const uint32_t jl = __shfl_sync(0xffffffffu, j, 31);
                        if (jl != NONE) jlast = jl;
                    }
                }
                if (__any_sync(0xffffffffu, cand != NONE)) {
                    cand = __reduce_min_sync(0xffffffffu, cand);
                    if (cand < wb) {
                        wb = cand;
                        wend = (uint32_t)range_begin(a, cand / nb + 1);
                    }
                }
                if (wb == NONE) continue;
#pragma unroll
                for (int k = 0; k < kIlp; ++k) past |= u[k] != NONE && u[k] >= wend;
                if (__any_sync(0xffffffffu, past)) break;               // the best's range is complete
            }
            if (lane_id() == (uint32_t)o) best = wb;
        }
        const bool found = best != NONE;
        if (found) a.parent[v] = (int32_t)best;
        const uint32_t m = __ballot_sync(0xffffffffu, found);
        if (lane_id() == 0 && m) a.t[w] = m;
    }
    if (STATS) flush_counts(a, edges, cols);
    if (STATS && blockIdx.x == 0 && threadIdx.x == 0) a.ctr[C_BOTTOM_UP] = 1ull;
}

// ---------------------------------------------------------------- reduce --
// The values of the next level, and whether it runs (the frontier is not
// empty, no invariant failed, fewer than max_levels levels).  In a CUDA graph
// the decision drives the conditional WHILE node.
struct NextArgs {
    int64_t n;
    int32_t max_levels;
    cudaGraphConditionalHandle handle;
    int use_handle;                 // the graph-launched loop: also clear the counters for the next level
    volatile uint64_t* h_error;     // pinned host word: the graph-launched loop's error flag once it ends
    unsigned long long* lvl;        // row hand-out counters, nlvl of them
    int nlvl;
};

// One thread; the counters of the level are complete.
__device__ void level_next(LevelCtl* c, unsigned long long* ctr, const NextArgs& nx) {
    const int64_t n = nx.n;
    const int64_t f = (int64_t)__ldcg(ctr + C_NEXT_COUNT);
    const int64_t prev = c->frontier;
    const int64_t mf = (int64_t)__ldcg(ctr + C_NEXT_DEGREE);
    c->m_u -= mf;
    c->m_f = mf;
    // direction of the next level (Beamer et al.): bottom-up once the growing
    // frontier's edges outweigh 1/alpha of the unvisited vertices' edges; back
    // to top-down once the shrinking frontier is below n / beta vertices
    if (c->policy == BFS_DIRECTION_BOTTOM_UP) {
        c->bu = 1;
    } else if (c->policy == BFS_DIRECTION_HYBRID) {
        if (!c->bu) c->bu = (f > prev && mf * (int64_t)c->alpha > c->m_u) ? 1 : 0;
        else c->bu = (f < prev && f * (int64_t)c->beta < n) ? 0 : 1;
    } else {
        c->bu = 0;
    }
    c->frontier = f;
    c->visited += f;
    c->level += 1;
    // the row window pays once a level visits every row's vertices several
    // times: a ratio half or twice as large costs scale 24 PLAIN 4% (2.76 ->
    // 2.87 ms) and moves scales 22 and 23 by less than 2.5% either way
    c->window = (n >= kWindowMinVertices && mf >= (int64_t)c->win_ratio * n) ? 1 : 0;
    // While few vertices are visited, most entries lead to fresh vertices,
    // each reached from many frontier vertices: reading the parent first turns
    // most of those visits into one L2 read instead of two atomics.  With the
    // next bits in the window the bit is a shared-memory atomic: not worth it.
    c->dedup = (c->visited * 16 < n) ? 1 : 0;
    const int go = (f > 0 && __ldcg(ctr + C_ERROR) == 0 && c->level < nx.max_levels) ? 1 : 0;
    c->go = go;
    if (!nx.use_handle) return;
    cudaGraphSetConditional(nx.handle, go ? 1u : 0u);
    if (!go) *nx.h_error = __ldcg(ctr + C_ERROR);
}

// x = t & ~pi; pi |= x; level of the new vertices; |x| and its degree sum; the
// next frontier f = x and t cleared for the next level; frontier summary of x.
// A warp takes WPW words: 32, so that the bitmaps are read and written in whole
// lines, or 4 on small graphs (below kSmallReduce vertices), where the chain of
// a word's level stores and degree loads, one word after the other, is the
// kernel's time (4,096 vertices: 128 words on 4 warps took 9 us).  A search with
// 4 / 32 words a warp: 202 / 212 us at scale 12, 552 / 559 at scale 20, 1021 /
// 971 at scale 22, 12.80 / 11.75 ms at scale 26 (partial lines).
// The last CTA to finish (a counter, no waiting) sets up the next level.
// In the graph-launched loop it also clears the per-level counters and the
// row hand-out counters, in place of memset nodes; the stepwise loop reads them
// first and clears them itself.
constexpr int64_t kSmallReduce = 1 << 20;

template <int WPW>
__global__ void __launch_bounds__(kNT) reduce_level(uint32_t* __restrict__ t, uint32_t* __restrict__ pi,
                                                    uint32_t* __restrict__ f, uint8_t* __restrict__ fsum,
                                                    uint32_t* __restrict__ fwords, int64_t words, int64_t n,
                                                    int32_t* __restrict__ level, LevelCtl* ctl, unsigned long long* ctr,
                                                    const uint32_t* __restrict__ deg, NextArgs nx) {
    constexpr int W = kNT / 32;                         // warps
    __shared__ unsigned long long s_sum[2][W];
    __shared__ uint32_t s_any[W];
    __shared__ int s_last;
    const int32_t next_level = ctl->level + 1;
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const int64_t per_cta = (int64_t)W * WPW;
    unsigned long long cnt = 0, dsum = 0;
    for (int64_t w0 = blockIdx.x * per_cta; w0 < words; w0 += gridDim.x * per_cta) {
        const int64_t wb = w0 + (int64_t)warp * WPW, w = wb + lane;
        uint32_t x = 0;
        if (lane < WPW && w < words) {
            const uint32_t pw = pi[w];
            x = t[w] & ~pw;
            if (x) pi[w] = pw | x;
            f[w] = x;
            t[w] = 0u;
            cnt += __popc(x);
        }
        const uint32_t any = __ballot_sync(0xffffffffu, x != 0u);
        // the levels (and degrees) of the fresh vertices, one word at a time
        // by the whole warp: lane l takes bit l (coalesced stores and loads)
        for (uint32_t m = any; m;) {
            uint32_t d[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {               // four words' degree loads in flight
                const int k = m ? __ffs(m) - 1 : 0;
                const uint32_t xk = m ? __shfl_sync(0xffffffffu, x, k) : 0u;
                m &= m - 1;
                const int64_t v = (wb + k) * 32 + lane;
                const bool fresh = ((xk >> lane) & 1u) && v < n;
                if (fresh) level[v] = next_level;
                d[q] = fresh ? __ldg(deg + v) : 0u;
            }
            dsum += (unsigned long long)d[0] + d[1] + d[2] + d[3];
        }
        if (WPW == 32) {
            if (lane == 0) {
                fsum[wb >> 5] = any ? 1 : 0;
                fwords[wb >> 5] = any;
            }
        } else {                                        // the CTA's words are one byte of the summary
            __syncthreads();                            // the previous round's masks are read
            if (lane == 0) s_any[warp] = any << (WPW * warp & 31);
            __syncthreads();
            if (threadIdx.x == 0) {
                uint32_t all = 0;
                for (int k = 0; k < W; ++k) all |= s_any[k];
                fsum[w0 >> 5] = all ? 1 : 0;
                fwords[w0 >> 5] = all;
            }
        }
    }
    static_assert(WPW == 32 || W * WPW == 32, "a warp or a CTA covers one byte of the frontier summary");
    cnt = warp_sum(cnt);
    dsum = warp_sum(dsum);
    if (lane == 0) {
        s_sum[0][warp] = cnt;
        s_sum[1][warp] = dsum;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < W; ++k) {
            cnt += s_sum[0][k];
            dsum += s_sum[1][k];
        }
        if (cnt) atomicAdd(ctr + C_NEXT_COUNT, cnt);
        if (dsum) atomicAdd(ctr + C_NEXT_DEGREE, dsum);
        __threadfence();
        s_last = atomicAdd(&ctl->done, 1u) == gridDim.x - 1;
        if (s_last) {
            __threadfence();
            ctl->done = 0u;
            level_next(ctl, ctr, nx);
        }
    }
    __syncthreads();
    if (!s_last || !nx.use_handle) return;
    for (int k = threadIdx.x; k < C_NUM; k += kNT)
        if (k < C_ERROR || k >= C_WAH_WORDS) ctr[k] = 0ull;          // the error flag and trace cursors stay
    for (int k = threadIdx.x; k < nx.nlvl; k += kNT) nx.lvl[k] = 0ull;
}

struct InitArgs {
    int32_t* level;
    int32_t* parent;
    int64_t n;
    uint32_t* pi;
    uint32_t* fa;
    uint32_t* fb;
    int64_t words;
    uint8_t* fsum;
    uint32_t* fwords;
    int64_t fsum_len;
    const uint32_t* iso;            // or nullptr
    const uint32_t* deg;
    int64_t entries;
    int32_t root;
    int32_t win_ratio, policy, alpha, beta;
    LevelCtl* ctl;
    unsigned long long* ctr;        // the counters, C_NUM of them
    unsigned long long* lvl;        // row hand-out counters, nlvl of them
    int nlvl;
};

// A search starts from nothing visited but the root -- or, with bottom-up
// levels, from the vertices without entries marked visited (iso): no level
// reaches them, and the bottom-up scans skip them.  One launch sets the
// outputs, bitmaps, counters and the first level's values.
__global__ void __launch_bounds__(kNT) init_search(InitArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t root = a.root;
    for (int64_t v = tid; v < a.n; v += stride) {
        a.level[v] = v == root ? 0 : -1;
        a.parent[v] = v == root ? a.root : -1;
    }
    for (int64_t w = tid; w < a.words; w += stride) {
        const uint32_t r = w == (root >> 5) ? 1u << (root & 31) : 0u;
        a.pi[w] = (a.iso ? a.iso[w] : 0u) | r;
        a.fa[w] = r;
        a.fb[w] = 0u;
    }
    for (int64_t q = tid; q < a.fsum_len; q += stride) {
        const bool r = q == (root >> 10);
        a.fsum[q] = r ? 1 : 0;
        a.fwords[q] = r ? 1u << ((root >> 5) & 31) : 0u;
    }
    for (int64_t q = tid; q < C_NUM; q += stride) a.ctr[q] = 0ull;
    for (int64_t q = tid; q < a.nlvl; q += stride) a.lvl[q] = 0ull;
    if (tid != 0) return;
    LevelCtl* c = a.ctl;
    c->frontier = 1;
    c->visited = 1;
    c->level = 0;
    c->done = 0u;
    c->window = 0;
    c->win_ratio = a.win_ratio;
    c->dedup = (16 < a.n) ? 1 : 0;
    c->go = 1;
    c->policy = a.policy;
    c->alpha = a.alpha;
    c->beta = a.beta;
    c->bu = (a.policy == BFS_DIRECTION_BOTTOM_UP) ? 1 : 0;
    c->m_f = (int64_t)a.deg[root];
    c->m_u = a.entries - c->m_f;
}

// Pack the streams of this exchange into a trace (the receive buffer g'):
// ctr[cursor] is the trace's fill, kept from level to level.
__global__ void __launch_bounds__(kNT) trace_offsets(const int64_t* __restrict__ counts, int nslots, int u32_per_word,
                                                     int64_t* __restrict__ slot_off, int64_t* __restrict__ trace_counts,
                                                     unsigned long long* ctr, int cursor, int64_t capacity,
                                                     const uint8_t* fmt, uint8_t* trace_fmt) {
    __shared__ unsigned long long red[kNT / 32 + 1];
    const unsigned long long used = ctr[cursor];
    unsigned long long carry = 0;
    for (int s0 = 0; s0 < nslots; s0 += kNT) {
        const int s = s0 + threadIdx.x;
        const unsigned long long c = (s < nslots) ? (unsigned long long)counts[s] * u32_per_word : 0ull;
        unsigned long long tot;
        const unsigned long long ex = block_excl_scan<kNT>(c, 0ull, OpSum(), red, &tot);
        if (s < nslots) {
            slot_off[s] = (int64_t)(used + carry + ex);
            trace_counts[s] = counts[s];
            if (trace_fmt) trace_fmt[s] = fmt ? fmt[s] : (uint8_t)FMT_WAH;
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        if (used + carry > (unsigned long long)capacity) {
            ctr[C_ERROR] |= 2ull;                 // trace overflow
            ctr[cursor] = (unsigned long long)capacity + 1;
        } else {
            ctr[cursor] = used + carry;
        }
    }
}

__global__ void trace_copy(const uint32_t* __restrict__ xbuf, int64_t slot_cap_u32, const int64_t* __restrict__ counts,
                           int nslots, int u32_per_word, const int64_t* __restrict__ slot_off,
                           uint32_t* __restrict__ trace, int64_t capacity) {
    for (int s = blockIdx.y; s < nslots; s += gridDim.y) {
        const int64_t c = counts[s] * u32_per_word;
        const int64_t off = slot_off[s];
        if (off + c > capacity) continue;
        for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < c; x += (int64_t)gridDim.x * blockDim.x)
            trace[off + x] = xbuf[(int64_t)s * slot_cap_u32 + x];
    }
}

// The output checks of bfs_check_search: root level 0 and its own parent;
// an unreached vertex -1 / -1; a reached one a parent in [0, n) one level
// closer to the root.  out[0] counts failures, out[1] keeps the smallest
// failing vertex, out[2] counts the reached vertices.
__global__ void __launch_bounds__(kNT) verify_search(const int32_t* __restrict__ parent,
                                                     const int32_t* __restrict__ level, int64_t n, int32_t root,
                                                     unsigned long long* out) {
    unsigned long long bad = 0, reached = 0, first = ~0ull;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t lv = level[v], pv = parent[v];
        bool ok;
        if (v == root) ok = lv == 0 && pv == root;
        else if (lv < 0) ok = lv == -1 && pv == -1;
        else ok = lv > 0 && pv >= 0 && (int64_t)pv < n && level[pv] == lv - 1;
        reached += lv >= 0;
        if (!ok) {
            ++bad;
            if ((unsigned long long)v < first) first = (unsigned long long)v;
        }
    }
    bad = warp_sum(bad);
    reached = warp_sum(reached);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, first, d);
        first = y < first ? y : first;
    }
    if (lane_id() == 0) {
        if (bad) atomicAdd(out, bad);
        if (first != ~0ull) atomicMin(out + 1, first);
        if (reached) atomicAdd(out + 2, reached);
    }
}

__global__ void visited_count(const LevelCtl* c, unsigned long long* out) { out[3] = (unsigned long long)c->visited; }

int sm_count() {
    static int cached = 0;
    if (!cached) {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        cached = v > 0 ? v : 1;
    }
    return cached;
}

// Dynamic shared memory of the expansion kernels: the row window.  Its kind
// is the largest that fits beside the warps' scratch: pi_i and the partial t_i,
// else pi_i alone (all the row exchange needs), else none.
size_t window_bytes(int64_t win_words, int kind) {
    return (size_t)((win_words + 3) / 4 * 16) * (kind == kWinBoth ? 2 : (kind == kWinPi ? 1 : 0));
}

constexpr size_t kWindowRoom = (size_t)kSmemLimit - sizeof(WarpScratch) * kXW - 2048;

int window_kind(int64_t win_words, bool rowx) {
    if (!rowx && window_bytes(win_words, kWinBoth) <= kWindowRoom) return kWinBoth;
    return window_bytes(win_words, kWinPi) <= kWindowRoom ? kWinPi : kWinNone;
}

// The limit is the function's, shared by every graph: always the whole room.
template <typename K>
bfs_status allow_smem(K kernel) {
    BFS_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWindowRoom));
    return BFS_OK;
}

template <int WIN, bool ROWX>
bfs_status allow_window() {
    BFS_TRY(allow_smem(expand_wah<uint32_t, WIN, ROWX>));
    BFS_TRY(allow_smem(expand_wah<unsigned long long, WIN, ROWX>));
    BFS_TRY(allow_smem(expand_pieces<WIN, ROWX>));
    if (!ROWX) BFS_TRY(allow_smem(expand_plain<WIN>));
    return BFS_OK;
}

// The expansion of a level's units, then of its long columns' pieces.
template <int WIN, bool ROWX>
void launch_expand(const LevelArgs& a, int wbits, int grid, size_t dyn, cudaStream_t s) {
    if (a.mode == BFS_MODE_PLAIN) expand_plain<WIN><<<grid, kXT, dyn, s>>>(a);
    else if (wbits == 32) expand_wah<uint32_t, WIN, ROWX><<<grid, kXT, dyn, s>>>(a);
    else expand_wah<unsigned long long, WIN, ROWX><<<grid, kXT, dyn, s>>>(a);
    expand_pieces<WIN, ROWX><<<grid, kXT, dyn, s>>>(a);
}

}  // namespace

// ------------------------------------------------------------- workspace --
bfs_status ensure_workspace_once(bfs_graph* g);

// All of the search workspace or none of it: a failed allocation releases the rest.
bfs_status ensure_workspace(bfs_graph* g, cudaStream_t st) {
    (void)st;
    if (g->W.bm_words) return BFS_OK;
    const bfs_status rc = ensure_workspace_once(g);
    if (rc != BFS_OK) free_workspace(g);
    return rc;
}

bfs_status ensure_workspace_once(bfs_graph* g) {
    Workspace& W = g->W;
    const Layout& L = g->L;
    const int p = L.p;
    const int64_t p2 = (int64_t)p * p;
    W.bm_words = ((L.n + 31) / 32 + 4 + 3) / 4 * 4;
    W.fsum_len = ((W.bm_words + 31) / 32 + 64 + 3) / 4 * 4;   // whole 32-bit words
    const int64_t cap32 = L.nb / 31 + 2, cap64 = L.nb / 63 + 2;
    W.slot_cap = cap32;
    W.chunks_per_slot = (cap32 + 31) / 32;
    const int64_t xbytes = p2 * std::max<int64_t>(4 * cap32, 8 * cap64);
    W.enc_cps = parallel_encode_chunks(L.nb, 32);                       // 31-bit groups: the most chunks
    // pieces: per row, sum over the columns longer than h of ceil(len/h) <= 2 nnz_row/h, most for the smallest h
    std::vector<int64_t> meta(2 * (size_t)p);
    int64_t total = 0;
    for (int i = 0; i < p; ++i) {
        int64_t nnz_row = 0;
        for (int j = 0; j < p; ++j) nnz_row += L.nnz_b[(int64_t)i * p + j];
        const int64_t cap = 2 * (nnz_row / kHubSparse) + 4;
        meta[i] = total;
        meta[p + i] = cap;
        total += cap;
    }
    W.piece_cap = total;
    const size_t chunks = (size_t)(p2 * W.enc_cps);
    BFS_TRY(alloc_parts(W.whole, {{&W.pi, (size_t)(4 * W.bm_words)},
                                  {&W.fa, (size_t)(4 * W.bm_words)},
                                  {&W.fb, (size_t)(4 * W.bm_words)},
                                  {&W.fsum, (size_t)W.fsum_len},
                                  {&W.fwords, sizeof(uint32_t) * (size_t)W.fsum_len},
                                  {&W.xbuf, (size_t)xbytes},
                                  {&W.xcount, sizeof(int64_t) * p2},
                                  {&W.chunk_base, sizeof(int64_t) * p2 * W.chunks_per_slot},
                                  {&W.units, sizeof(int64_t) * (p2 + 1)},      // slot unit bases
                                  {&W.xfmt, (size_t)p2},
                                  {&W.enc_sums, parallel_encode_sum_bytes() * chunks},
                                  {&W.enc_bases, parallel_encode_base_bytes() * chunks},
                                  {&W.enc_flags, chunks},
                                  {&W.enc_done, sizeof(unsigned int)},
                                  {&W.ctl, sizeof(LevelCtl)},
                                  {&W.counters, sizeof(unsigned long long) * C_NUM},
                                  {&W.pieces, sizeof(Item) * total},
                                  // per-level scratch: row_next[p], row_piece_count[p], row_piece_next[p]
                                  {&W.level_scratch, sizeof(unsigned long long) * (3 * p + 1)},
                                  {&W.row_meta, sizeof(int64_t) * 2 * p}}));   // row piece bases and caps
    BFS_CUDA_TRY(cudaMemset(W.enc_done.ptr, 0, sizeof(unsigned int)));
    BFS_CUDA_TRY(cudaMemcpy(W.row_meta.ptr, meta.data(), sizeof(int64_t) * 2 * p, cudaMemcpyHostToDevice));
    if (!W.h_counters) {
        void* h = nullptr;
        BFS_CUDA_TRY(cudaMallocHost(&h, sizeof(uint64_t) * C_NUM));
        W.h_counters = static_cast<uint64_t*>(h);
    }
    if (!W.events) {
        for (auto& e : W.ev) BFS_CUDA_TRY(cudaEventCreate(&e));
        W.events = true;
    }
    // the row window of the expansion
    W.win_words = (L.nb + 31) / 32;
    const int both = window_kind(W.win_words, false), rows = window_kind(W.win_words, true);
    if (both == kWinBoth) BFS_TRY((allow_window<kWinBoth, false>()));
    if (both == kWinPi) BFS_TRY((allow_window<kWinPi, false>()));
    if (rows == kWinPi) BFS_TRY((allow_window<kWinPi, true>()));
    return BFS_OK;
}

void free_workspace(bfs_graph* g) {
    Workspace& W = g->W;
    W.pi.release(); W.fa.release(); W.fb.release(); W.fsum.release(); W.fwords.release(); W.xbuf.release();
    W.xcount.release(); W.chunk_base.release(); W.units.release(); W.counters.release(); W.pieces.release();
    W.level_scratch.release(); W.row_meta.release();
    W.tblk.release(); W.rowbuf.release(); W.rowcount.release(); W.rowfirst.release(); W.rowlive.release();
    W.tblk_dirty = false;
    W.enc_sums.release(); W.enc_bases.release(); W.enc_flags.release(); W.enc_done.release(); W.ctl.release();
    W.gbits.release();
    W.colfirst.release();
    W.xfmt.release();
    W.ddir.release();
    for (auto& c : W.sgraph) {
        if (c.exec) cudaGraphExecDestroy(c.exec);
        if (c.graph) cudaGraphDestroy(c.graph);
        c = SearchGraph();
    }
    W.sgraph_next = 0;
    W.tmp_parent.release(); W.tmp_level.release();
    if (W.h_counters) cudaFreeHost(W.h_counters);
    W.h_counters = nullptr;
    if (W.events) for (auto& e : W.ev) cudaEventDestroy(e);
    W.events = false;
    W.whole.release();
    W.bm_words = 0;
}

namespace {

struct BusyGuard {
    bfs_graph* g;
    bool ok;
    explicit BusyGuard(bfs_graph* gg) : g(gg) {
        int expect = 0;
        ok = g->busy.compare_exchange_strong(expect, 1);
    }
    ~BusyGuard() { if (ok) g->busy.store(0); }
};

float elapsed(cudaEvent_t a, cudaEvent_t b) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) { cudaGetLastError(); return 0.f; }
    return ms;
}

// Run the output checks on device outputs; with ctl, the reached count must
// also equal the vertices the search visited.
bfs_status check_outputs(int64_t n, int32_t root, const int32_t* parent, const int32_t* level, const LevelCtl* ctl,
                         cudaStream_t st) {
    DevBuf out;
    BFS_TRY(out.alloc(4 * sizeof(unsigned long long)));
    unsigned long long init[4] = {0ull, ~0ull, 0ull, 0ull};
    BFS_CUDA_TRY(cudaMemcpyAsync(out.ptr, init, sizeof(init), cudaMemcpyHostToDevice, st));
    verify_search<<<(int)std::min<int64_t>((n + kNT - 1) / kNT, (int64_t)sm_count() * 8), kNT, 0, st>>>(
        parent, level, n, root, out.as<unsigned long long>());
    if (ctl) visited_count<<<1, 1, 0, st>>>(ctl, out.as<unsigned long long>());
    BFS_CUDA_TRY(cudaGetLastError());
    unsigned long long h[4];
    BFS_CUDA_TRY(cudaMemcpyAsync(h, out.ptr, sizeof(h), cudaMemcpyDeviceToHost, st));
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    if (h[0])
        return set_error(BFS_ERR_CORRUPT, "%llu vertices fail the level/parent checks (first: vertex %llu)", h[0], h[1]);
    if (ctl && h[2] != h[3])
        return set_error(BFS_ERR_CORRUPT, "%llu vertices reached but %llu visited by the search", h[2], h[3]);
    return BFS_OK;
}

bfs_status run_search(bfs_graph* g, int32_t root, int32_t* parent, int32_t* level, bfs_run_stats* stats,
                      cudaStream_t st) {
    Layout& L = g->L;
    Workspace& W = g->W;
    BFS_TRY(ensure_workspace(g, st));
    const int mode = g->mode;
    const int wbits = g->wah_bits;
    const int p = L.p;
    const int64_t p2 = (int64_t)p * p;
    const int64_t slot_cap = (wbits == 32) ? L.nb / 31 + 2 : L.nb / 63 + 2;
    const int nslots = (mode == BFS_MODE_COMPRESS_SIEVE) ? (int)p2 : (mode == BFS_MODE_COMPRESS ? p : 0);
    const bool timing = stats && stats->timing;
    const bool tracing = stats && stats->trace_words && stats->trace_counts && nslots > 0;
    unsigned long long* ctr = W.counters.as<unsigned long long>();
    const int xgrid = sm_count();                  // persistent: one 1024-thread CTA per SM
    // the compressed row exchange of the fold belongs to DIR-WAH (COMPRESS_SIEVE)
    const bool rowx = g->row_exchange && mode == BFS_MODE_COMPRESS_SIEVE;
    if (rowx && !W.tblk.ptr) {
        // allocated once (all or none): captured level loops keep the addresses
        const int64_t cap32 = L.nb / 31 + 2, cap64 = L.nb / 63 + 2;
        W.row_cap = cap32;
        bfs_status rc = W.rowbuf.alloc((size_t)p2 * std::max<int64_t>(4 * cap32, 8 * cap64));
        if (rc == BFS_OK) rc = W.rowcount.alloc(sizeof(int64_t) * (size_t)p2);
        if (rc == BFS_OK) rc = W.rowfirst.alloc(sizeof(int64_t) * 2 * (size_t)(p2 * W.enc_cps));
        if (rc == BFS_OK) rc = W.rowlive.alloc((size_t)p2);
        if (rc == BFS_OK) rc = W.tblk.alloc(sizeof(uint32_t) * (size_t)(p2 * L.dir_stride));
        if (rc != BFS_OK) {
            W.tblk.release(); W.rowbuf.release(); W.rowcount.release(); W.rowfirst.release(); W.rowlive.release();
            return rc;
        }
        BFS_CUDA_TRY(cudaMemsetAsync(W.tblk.ptr, 0, W.tblk.bytes, st));
        W.tblk_dirty = false;
    }
    if (rowx && W.tblk_dirty) {          // an earlier search stopped between marking and encoding
        BFS_CUDA_TRY(cudaMemsetAsync(W.tblk.ptr, 0, W.tblk.bytes, st));
        W.tblk_dirty = false;
    }
    const int64_t row_cap = (wbits == 32) ? L.nb / 31 + 2 : L.nb / 63 + 2;
    const bool adaptive = g->adaptive && mode != BFS_MODE_PLAIN;
    if (adaptive && wbits != 32)
        return set_error(BFS_ERR_INVALID_ARG, "the level-adaptive exchange format needs 32-bit WAH words");
    const bool row_tracing = stats && rowx && stats->row_trace_words && stats->row_trace_counts;
    // the dynamic cross directory belongs to the sieve (COMPRESS_SIEVE)
    const bool dynamic = g->dynamic_dir && mode == BFS_MODE_COMPRESS_SIEVE;
    if (dynamic && !W.ddir.ptr) {
        // allocated once: captured level loops keep the address
        BFS_TRY(W.ddir.alloc(sizeof(uint32_t) * (size_t)(p2 * L.dir_stride)));
    }
    const int win = window_kind(W.win_words, rowx);
    const size_t dyn = window_bytes(W.win_words, win);
    // bottom-up levels: degrees (direction choice) and the decoded streams
    const bool bu_kernels = g->direction != BFS_DIRECTION_TOP_DOWN;
    if (bu_kernels) BFS_TRY(ensure_bottom_up(g, st));
    const int64_t g_words = (W.bm_words + 3) / 4 * 4;
    if (bu_kernels && (!W.gbits.ptr || !W.colfirst.ptr)) {
        // allocated once (both or neither): captured level loops keep the addresses
        bfs_status rc = W.gbits.alloc(sizeof(uint32_t) * (size_t)g_words);
        if (rc == BFS_OK) rc = W.colfirst.alloc(sizeof(int64_t) * 2 * (size_t)(p2 * W.enc_cps));
        if (rc != BFS_OK) { W.gbits.release(); W.colfirst.release(); return rc; }
    }
    DevBuf slot_off;
    if (tracing || row_tracing) BFS_TRY(slot_off.alloc(sizeof(int64_t) * (size_t)std::max<int64_t>(nslots, p2)));
    if (stats) { stats->n_levels = 0; stats->trace_used = 0; stats->row_trace_used = 0; }

    LevelCtl* ctl = W.ctl.as<LevelCtl>();
    const uint32_t* deg = L.deg.as<uint32_t>();
    unsigned long long* lvl = W.level_scratch.as<unsigned long long>();
    const InitArgs init{level, parent, L.n, W.pi.as<uint32_t>(), W.fa.as<uint32_t>(), W.fb.as<uint32_t>(), W.bm_words,
                        W.fsum.as<uint8_t>(), W.fwords.as<uint32_t>(), W.fsum_len,
                        bu_kernels ? L.iso.as<uint32_t>() : nullptr, deg, L.nnz, root, rowx ? 4 : 2, g->direction,
                        g->alpha, g->beta, ctl, ctr, lvl, 3 * p + 1};
    init_search<<<(unsigned)std::min<int64_t>((L.n + kNT - 1) / kNT, sm_count() * 4), kNT, 0, st>>>(init);
    BFS_CUDA_TRY(cudaGetLastError());

    LevelArgs a;
    memset(&a, 0, sizeof(a));
    a.dir = L.dir.as<uint32_t>();
    a.rank = L.rank.as<uint32_t>();
    a.dir_stride = L.dir_stride;
    a.cp = L.cp.as<uint32_t>();
    a.cp_base = L.cp_base_d.as<int64_t>();
    a.ir_base = L.ir_base_d.as<int64_t>();
    a.ir = L.ir.as<int32_t>();
    a.p = p;
    a.nb = L.nb;
    a.n = L.n;
    a.pi = W.pi.as<uint32_t>();
    a.parent = parent;
    a.xbuf = W.xbuf.ptr;
    a.slot_cap = slot_cap;
    a.xcount = W.xcount.as<int64_t>();
    a.chunk_base = W.chunk_base.as<int64_t>();
    a.chunks_per_slot = W.chunks_per_slot;
    a.slot_unit_base = W.units.as<int64_t>();
    a.row_next = lvl;
    a.row_piece_count = lvl + p;
    a.row_piece_next = lvl + 2 * p;
    a.row_piece_base = W.row_meta.as<int64_t>();
    a.row_piece_cap = W.row_meta.as<int64_t>() + p;
    a.pieces = W.pieces.as<Item>();
    a.ctr = ctr;
    a.mode = mode;
    a.plain_upb = (L.nb + 1023) / 1024;               // 32 raw words per PLAIN unit
    a.win_words = W.win_words;
    a.tblk = W.tblk.as<uint32_t>();
    a.rowbuf = W.rowbuf.ptr;
    a.row_cap = row_cap;
    a.row_count = W.rowcount.as<int64_t>();
    a.row_first = W.rowfirst.as<int64_t>();
    a.row_cps = W.enc_cps;
    a.row_bcps = (L.nb + (int64_t)kEncChunkGroups * (wbits - 1) - 1) / ((int64_t)kEncChunkGroups * (wbits - 1));
    a.gbits = W.gbits.as<uint32_t>();
    a.range_aligned = (L.nb % 32 == 0) ? 1 : 0;
    a.g_words = g_words;
    a.bu_ptr = L.bu_ptr.as<int64_t>();
    a.bu_adj = L.bu_adj.as<int32_t>();

    EncodeArgs ea;
    memset(&ea, 0, sizeof(ea));
    ea.dir = (mode == BFS_MODE_COMPRESS_SIEVE) ? (dynamic ? W.ddir.as<uint32_t>() : L.dir.as<uint32_t>()) : nullptr;
    ea.dir_stride = L.dir_stride;
    ea.p = p;
    ea.nb = L.nb;
    ea.n = L.n;
    ea.sieve = (mode == BFS_MODE_COMPRESS_SIEVE);
    ea.nslots = nslots;
    ea.fsum = W.fsum.as<uint8_t>();
    ea.out = W.xbuf.ptr;
    ea.slot_cap = slot_cap;
    ea.counts = W.xcount.as<int64_t>();
    ea.unit_base = W.chunk_base.as<int64_t>();      // the decoder's unit bases, written by the encoder
    ea.unit_stride = W.chunks_per_slot;
    ea.wah_words = ctr + C_WAH_WORDS;
    ea.plan_base = W.units.as<int64_t>();            // the unit plan, laid out by the encoder's scan
    ea.plan_units = ctr + C_UNITS;
    ea.plan_done = W.enc_done.as<unsigned int>();
    ea.frontier_words = W.bm_words;
    if (rowx) ea.slot_bits = W.rowlive.as<uint8_t>();    // the row encoder skips blocks that expanded nothing
    ea.adaptive = adaptive ? 1 : 0;
    ea.fmt = W.xfmt.as<uint8_t>();
    if (bu_kernels) ea.chunk_first = W.colfirst.as<int64_t>();   // the bottom-up decode starts chunk by chunk
    a.col_first = W.colfirst.as<int64_t>();
    a.fmt = adaptive ? W.xfmt.as<uint8_t>() : nullptr;

    // the row encoder: slot s = i*p + j is the partial t_{i,j} (the directory
    // operand, consumed and cleared) sieved by not(pi_i) (the frontier operand
    // at range i, complemented)
    EncodeArgs ra;
    memset(&ra, 0, sizeof(ra));
    ra.frontier = W.pi.as<uint32_t>();
    ra.frontier_words = W.bm_words;
    ra.invert_frontier = 1;
    ra.dir = W.tblk.as<uint32_t>();
    ra.dir_clear = W.tblk.as<uint32_t>();
    ra.dir_stride = L.dir_stride;
    ra.p = p;
    ra.nb = L.nb;
    ra.n = L.n;
    ra.sieve = 1;
    ra.row_slots = 1;
    ra.nslots = (int)p2;
    ra.out = W.rowbuf.ptr;
    ra.slot_cap = row_cap;
    ra.counts = W.rowcount.as<int64_t>();
    ra.wah_words = ctr + C_ROW_WORDS;
    ra.chunk_first = W.rowfirst.as<int64_t>();
    ra.slot_live = W.rowlive.as<uint8_t>();      // t_{i,j} = 0 when stream (i,j) carried no vertex

    uint32_t* f = W.fa.as<uint32_t>();       // frontier of the level (reduce_level writes the next one here)
    uint32_t* t = W.fb.as<uint32_t>();       // next bits (cleared by reduce_level)
    a.f = f;
    a.t = t;
    a.fsum = W.fsum.as<uint8_t>();
    a.fwords = W.fwords.as<uint32_t>();
    a.ctl = ctl;
    ea.frontier = f;
    ra.skip = &ctl->bu;                      // bottom-up levels have no row exchange
    const int32_t max_levels = (int32_t)std::min<int64_t>(L.n + 1, INT32_MAX);

    if (dynamic)                     // the search's directories start as V
        BFS_CUDA_TRY(cudaMemcpyAsync(W.ddir.ptr, L.dir.ptr, W.ddir.bytes, cudaMemcpyDeviceToDevice, st));

    // One level: the same launch sequence every time.  `host` adds the
    // statistics, the trace and the phase events (and k is known on the host).
    auto level_body = [&](cudaStream_t s, bool host, int32_t k, cudaGraphConditionalHandle handle) -> bfs_status {
        // per-level counters (the error flag and the trace cursor persist): the
        // stepwise loop clears them here, the graph-launched loop's reduce_level
        // at the end of the level before (and the search's setup for the first)
        if (host) {
            BFS_CUDA_TRY(cudaMemsetAsync(ctr, 0, sizeof(unsigned long long) * C_ERROR, s));
            BFS_CUDA_TRY(cudaMemsetAsync(ctr + C_WAH_WORDS, 0, sizeof(unsigned long long) * (C_NUM - C_WAH_WORDS), s));
            BFS_CUDA_TRY(cudaMemsetAsync(lvl, 0, sizeof(unsigned long long) * (3 * p + 1), s));
        }
        if (host && timing) cudaEventRecord(W.ev[7], s);
        if (dynamic) {                  // the frontier's bits of the dynamic directory
            dyn_sieve<<<sm_count() * 8, kNT, 0, s>>>(a, W.ddir.as<uint32_t>(), W.fsum.as<uint8_t>());
            BFS_CUDA_TRY(cudaGetLastError());
        }
        if (host && timing) cudaEventRecord(W.ev[0], s);
        if (mode == BFS_MODE_PLAIN) {
            if (host && timing) { cudaEventRecord(W.ev[1], s); cudaEventRecord(W.ev[2], s); }
        } else {
            // the exchanged-vertex and chunk counts are statistics: only the stepwise loop asks for them
            EncodeArgs eh = ea;
            eh.live_chunks = host ? ctr + C_ENC_CHUNKS : nullptr;
            BFS_TRY(launch_wah_encode_parallel(eh, wbits, W.enc_sums.ptr, W.enc_bases.ptr, W.enc_cps,
                                               W.enc_flags.ptr, host ? ctr + C_EXCHANGED : nullptr, sm_count() * 6, s));
            if (bu_kernels) {           // a bottom-up level reads the streams as bitmaps
                if (!a.range_aligned) clear_gbits<<<sm_count() * 4, kNT, 0, s>>>(a);   // shared boundary words
                const int64_t fitems = (int64_t)p * a.row_bcps;
                const int fgrid = (int)std::min<int64_t>(std::max<int64_t>(fitems, 1), (int64_t)sm_count() * 4);
                if (wbits == 32) fold_slots<uint32_t, false><<<fgrid, kFT, 0, s>>>(a);
                else fold_slots<unsigned long long, false><<<fgrid, kFT, 0, s>>>(a);
                if (adaptive) decode_vectors<<<sm_count() * 8, kNT, 0, s>>>(a);
                BFS_CUDA_TRY(cudaGetLastError());
            }
            if (host && timing) cudaEventRecord(W.ev[1], s);
            if (host && tracing && k < stats->capacity_levels) {
                const int u32pw = wbits / 32;
                trace_offsets<<<1, kNT, 0, s>>>(W.xcount.as<int64_t>(), nslots, u32pw, slot_off.as<int64_t>(),
                                                stats->trace_counts + (int64_t)k * nslots, ctr, C_TRACE_USED,
                                                stats->trace_capacity, a.fmt,
                                                stats->trace_formats ? stats->trace_formats + (int64_t)k * nslots
                                                                     : nullptr);
                dim3 tg(8, std::min(nslots, 65535));
                trace_copy<<<tg, kNT, 0, s>>>(W.xbuf.as<uint32_t>(), slot_cap * u32pw, W.xcount.as<int64_t>(), nslots,
                                              u32pw, slot_off.as<int64_t>(), stats->trace_words, stats->trace_capacity);
                BFS_CUDA_TRY(cudaGetLastError());
            }
            if (host && timing) cudaEventRecord(W.ev[2], s);
        }
        if (rowx) {
            if (win == kWinPi) launch_expand<kWinPi, true>(a, wbits, xgrid, dyn, s);
            else launch_expand<kWinNone, true>(a, wbits, xgrid, 0, s);
        } else {
            if (win == kWinBoth) launch_expand<kWinBoth, false>(a, wbits, xgrid, dyn, s);
            else if (win == kWinPi) launch_expand<kWinPi, false>(a, wbits, xgrid, dyn, s);
            else launch_expand<kWinNone, false>(a, wbits, xgrid, 0, s);
        }
        BFS_CUDA_TRY(cudaGetLastError());
        if (bu_kernels) {
            const int64_t ctas = ((L.n + 31) / 32 + kNT / 32 - 1) / (kNT / 32);      // a warp per visited word
            const unsigned bgrid = (unsigned)std::min<int64_t>(ctas, (int64_t)sm_count() * kBuCtas);
            if (host) expand_bottom_up<true><<<bgrid, kNT, 0, s>>>(a);
            else expand_bottom_up<false><<<bgrid, kNT, 0, s>>>(a);
            BFS_CUDA_TRY(cudaGetLastError());
        }
        if (host && timing) cudaEventRecord(W.ev[3], s);
        if (rowx) {
            // the row exchange: every block's partial, sieved by not(pi_i), WAH-encoded
            // into its row buffer; the fold OR-decodes the buffers of each block-row into t
            EncodeArgs rh = ra;
            rh.live_chunks = host ? ctr + C_ROW_CHUNKS : nullptr;
            BFS_TRY(launch_wah_encode_parallel(rh, wbits, W.enc_sums.ptr, W.enc_bases.ptr, W.enc_cps, W.enc_flags.ptr,
                                               nullptr, sm_count() * 6, s));
            if (host && timing) cudaEventRecord(W.ev[5], s);
            if (host && row_tracing && k < stats->capacity_levels) {
                const int u32pw = wbits / 32;
                trace_offsets<<<1, kNT, 0, s>>>(W.rowcount.as<int64_t>(), (int)p2, u32pw, slot_off.as<int64_t>(),
                                                stats->row_trace_counts + (int64_t)k * p2, ctr, C_ROW_TRACE_USED,
                                                stats->row_trace_capacity, nullptr, nullptr);
                dim3 tg(8, (unsigned)std::min<int64_t>(p2, 65535));
                trace_copy<<<tg, kNT, 0, s>>>(static_cast<const uint32_t*>(W.rowbuf.ptr), row_cap * u32pw,
                                              W.rowcount.as<int64_t>(), (int)p2, u32pw, slot_off.as<int64_t>(),
                                              stats->row_trace_words, stats->row_trace_capacity);
                BFS_CUDA_TRY(cudaGetLastError());
            }
            const int64_t fitems = (int64_t)p * a.row_bcps;
            const int fgrid = (int)std::min<int64_t>(std::max<int64_t>(fitems, 1), (int64_t)sm_count() * 4);
            if (wbits == 32) fold_slots<uint32_t, true><<<fgrid, kFT, 0, s>>>(a);
            else fold_slots<unsigned long long, true><<<fgrid, kFT, 0, s>>>(a);
            BFS_CUDA_TRY(cudaGetLastError());
            if (host && timing) cudaEventRecord(W.ev[6], s);
        } else if (host && timing) {
            cudaEventRecord(W.ev[5], s);
            cudaEventRecord(W.ev[6], s);
        }
        const NextArgs nx{L.n, max_levels, handle, host ? 0 : 1, W.h_counters + C_ERROR, lvl, 3 * p + 1};
        if (L.n < kSmallReduce)
            reduce_level<4><<<(unsigned)((W.bm_words + 31) / 32), kNT, 0, s>>>(
                t, W.pi.as<uint32_t>(), f, W.fsum.as<uint8_t>(), W.fwords.as<uint32_t>(), W.bm_words, L.n, level, ctl,
                ctr, deg, nx);
        else
            reduce_level<32><<<std::min<int64_t>((W.bm_words + 255) / 256, sm_count() * 16), kNT, 0, s>>>(
                t, W.pi.as<uint32_t>(), f, W.fsum.as<uint8_t>(), W.fwords.as<uint32_t>(), W.bm_words, L.n, level, ctl,
                ctr, deg, nx);
        BFS_CUDA_TRY(cudaGetLastError());
        if (host && timing) cudaEventRecord(W.ev[4], s);
        return BFS_OK;
    };

    if (!stats) {
        // The whole level loop as one CUDA-graph launch: a conditional WHILE
        // node repeats the level while level_next says so.  No host round
        // trip per level; the graph is built once per configuration and output
        // buffers and reused.
        SearchGraph* sg = nullptr;
        for (auto& c : W.sgraph)
            if (c.exec && c.mode == mode && c.wbits == wbits && c.rowx == (int)rowx &&
                c.bottom_up == (int)bu_kernels && c.adaptive == (int)adaptive && c.dynamic == (int)dynamic &&
                c.parent == parent &&
                c.level == level)
                sg = &c;
        if (!sg) {
            SearchGraph& c = W.sgraph[W.sgraph_next];
            W.sgraph_next = (W.sgraph_next + 1) % (int)(sizeof(W.sgraph) / sizeof(W.sgraph[0]));
            if (c.exec) { cudaGraphExecDestroy(c.exec); c.exec = nullptr; }
            if (c.graph) { cudaGraphDestroy(c.graph); c.graph = nullptr; }
            cudaGraph_t graph = nullptr;
            BFS_CUDA_TRY(cudaGraphCreate(&graph, 0));
            cudaGraphConditionalHandle handle;
            BFS_CUDA_TRY(cudaGraphConditionalHandleCreate(&handle, graph, 1, cudaGraphCondAssignDefault));
            cudaGraphNodeParams cp = {};
            cp.type = cudaGraphNodeTypeConditional;
            cp.conditional.handle = handle;
            cp.conditional.type = cudaGraphCondTypeWhile;
            cp.conditional.size = 1;
            cudaGraphNode_t cond = nullptr;
            cudaError_t ce = cudaGraphAddNode(&cond, graph, nullptr, nullptr, 0, &cp);
            if (ce != cudaSuccess) { cudaGraphDestroy(graph); return cuda_error(ce, "conditional node", __FILE__, __LINE__); }
            cudaGraph_t body = cp.conditional.phGraph_out[0];
            cudaStream_t cs = nullptr;
            BFS_CUDA_TRY(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
            ce = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
            bfs_status bs = BFS_OK;
            if (ce == cudaSuccess) bs = level_body(cs, false, 0, handle);
            cudaError_t ce2 = cudaStreamEndCapture(cs, &body);
            cudaStreamDestroy(cs);
            if (ce != cudaSuccess || ce2 != cudaSuccess || bs != BFS_OK) {
                cudaGraphDestroy(graph);
                if (bs != BFS_OK) return bs;
                return cuda_error(ce != cudaSuccess ? ce : ce2, "capture of the level body", __FILE__, __LINE__);
            }
            cudaGraphExec_t exec = nullptr;
            ce = cudaGraphInstantiate(&exec, graph, 0);
            if (ce != cudaSuccess) { cudaGraphDestroy(graph); return cuda_error(ce, "cudaGraphInstantiate(search)", __FILE__, __LINE__); }
            c.graph = graph;
            c.exec = exec;
            c.mode = mode;
            c.wbits = wbits;
            c.rowx = rowx ? 1 : 0;
            c.bottom_up = bu_kernels ? 1 : 0;
            c.adaptive = adaptive ? 1 : 0;
            c.dynamic = dynamic ? 1 : 0;
            c.parent = parent;
            c.level = level;
            sg = &c;
        }
        W.h_counters[C_ERROR] = 0;
        BFS_CUDA_TRY(cudaGraphLaunch(sg->exec, st));
        BFS_CUDA_TRY(cudaStreamSynchronize(st));
        const volatile uint64_t* h = W.h_counters;
        if (h[C_ERROR] & 2ull) return set_error(BFS_ERR_INVALID_ARG, "trace capacity exceeded");
        if (h[C_ERROR])
            return set_error(BFS_ERR_CORRUPT, "device invariant check failed (code %llu)",
                             (unsigned long long)h[C_ERROR]);
        if (g->debug_checks) return check_outputs(L.n, root, parent, level, ctl, st);
        return BFS_OK;
    }

    int64_t frontier = 1;
    int64_t raw_bytes = 0;
    for (int j = 0; j < p; ++j) raw_bytes += 4 * ((L.range_len(j) + 31) / 32);
    raw_bytes *= p;
    for (int32_t k = 0;; ++k) {
        BFS_TRY(level_body(st, true, k, cudaGraphConditionalHandle{}));
        BFS_CUDA_TRY(cudaMemcpyAsync(W.h_counters, ctr, sizeof(uint64_t) * C_NUM, cudaMemcpyDeviceToHost, st));
        BFS_CUDA_TRY(cudaStreamSynchronize(st));
        const uint64_t* h = W.h_counters;
        if (h[C_ERROR] & 2ull) return set_error(BFS_ERR_INVALID_ARG, "trace capacity exceeded");
        if (h[C_ERROR])
            return set_error(BFS_ERR_CORRUPT, "device invariant check failed (code %llu) at level %d",
                             (unsigned long long)h[C_ERROR], k);
        if (stats->levels && k < stats->capacity_levels) {
            bfs_level_stats& ls = stats->levels[k];
            memset(&ls, 0, sizeof(ls));
            ls.frontier_vertices = frontier;
            ls.exchanged_vertices = (mode == BFS_MODE_COMPRESS_SIEVE) ? (int64_t)h[C_EXCHANGED] : p * frontier;
            ls.column_hits = (int64_t)h[C_HITS];
            ls.raw_bytes = raw_bytes;
            ls.wah_bytes = (mode == BFS_MODE_PLAIN) ? 0 : (int64_t)h[C_WAH_WORDS] * (wbits / 8);
            ls.edges_scanned = (int64_t)h[C_EDGES];
            ls.row_wah_bytes = (int64_t)h[C_ROW_WORDS] * (wbits / 8);
            ls.bottom_up = h[C_BOTTOM_UP] ? 1 : 0;
            ls.compress_chunks = (int64_t)h[C_ENC_CHUNKS];
            ls.row_compress_chunks = (int64_t)h[C_ROW_CHUNKS];
            if (timing) {
                ls.ms_compress_sieve = elapsed(W.ev[0], W.ev[1]);
                ls.ms_communication = elapsed(W.ev[1], W.ev[2]);
                ls.ms_traversing = elapsed(W.ev[2], W.ev[3]);
                ls.ms_row_compress = elapsed(W.ev[3], W.ev[5]);
                ls.ms_row_fold = elapsed(W.ev[5], W.ev[6]);
                ls.ms_reducing = elapsed(W.ev[6], W.ev[4]);
                ls.ms_directory_update = dynamic ? elapsed(W.ev[7], W.ev[0]) : 0.0f;
            }
        }
        stats->n_levels = k + 1;
        if (tracing) stats->trace_used = (int64_t)h[C_TRACE_USED];
        if (row_tracing) stats->row_trace_used = (int64_t)h[C_ROW_TRACE_USED];
        frontier = (int64_t)h[C_NEXT_COUNT];
        if (frontier == 0 || k + 1 >= max_levels) break;
    }
    if (g->debug_checks) return check_outputs(L.n, root, parent, level, ctl, st);
    return BFS_OK;
}

}  // namespace
}  // namespace bfsgb

using namespace bfsgb;

extern "C" bfs_status bfs_check_search(bfs_graph_t g, int32_t root, const int32_t* parent, const int32_t* level,
                                       void* stream) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (root < 0 || (int64_t)root >= g->L.n) return set_error(BFS_ERR_INVALID_ARG, "root %d outside [0, %lld)", root, (long long)g->L.n);
    if (!is_device_pointer(parent) || !is_device_pointer(level))
        return set_error(BFS_ERR_INVALID_ARG, "parent and level must be device pointers");
    return check_outputs(g->L.n, root, parent, level, nullptr, static_cast<cudaStream_t>(stream));
}

extern "C" bfs_status bfs_run(bfs_graph_t g, int32_t root, int32_t* parent, int32_t* level, bfs_run_stats* stats,
                              void* stream) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (!parent || !level) return set_error(BFS_ERR_INVALID_ARG, "parent and level are required");
    if (root < 0 || (int64_t)root >= g->L.n) return set_error(BFS_ERR_INVALID_ARG, "root %d outside [0, %lld)", root, (long long)g->L.n);
    if (stats && stats->capacity_levels < 0) return set_error(BFS_ERR_INVALID_ARG, "negative capacity_levels");
    BusyGuard guard(g);
    if (!guard.ok) return set_error(BFS_ERR_BUSY, "another search on this graph is running");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool dev_p = is_device_pointer(parent), dev_l = is_device_pointer(level);
    if (dev_p != dev_l) return set_error(BFS_ERR_INVALID_ARG, "parent and level must both be host or both be device pointers");
    if (dev_p) {
        const bfs_status rs = run_search(g, root, parent, level, stats, st);
        if (rs != BFS_OK) g->W.tblk_dirty = true;     // the row partials may hold a level's marks
        return rs;
    }
    Workspace& W = g->W;
    if (!W.tmp_parent.ptr || !W.tmp_level.ptr) {
        bfs_status rc = W.tmp_parent.alloc(sizeof(int32_t) * g->L.n);
        if (rc == BFS_OK) rc = W.tmp_level.alloc(sizeof(int32_t) * g->L.n);
        if (rc != BFS_OK) { W.tmp_parent.release(); W.tmp_level.release(); return rc; }
    }
    {
        const bfs_status rs = run_search(g, root, W.tmp_parent.as<int32_t>(), W.tmp_level.as<int32_t>(), stats, st);
        if (rs != BFS_OK) { W.tblk_dirty = true; return rs; }
    }
    BFS_CUDA_TRY(cudaMemcpyAsync(parent, W.tmp_parent.ptr, sizeof(int32_t) * g->L.n, cudaMemcpyDeviceToHost, st));
    BFS_CUDA_TRY(cudaMemcpyAsync(level, W.tmp_level.ptr, sizeof(int32_t) * g->L.n, cudaMemcpyDeviceToHost, st));
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    return BFS_OK;
}
