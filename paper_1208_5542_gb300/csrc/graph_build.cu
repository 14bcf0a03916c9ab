// graph_build.cu -- the blocked layout of the adjacency (Eq. 1-4) built on the
// device, and the graph-management entry points of the C ABI.
//
// Layout (one-time per graph, amortised over every search as the paper
// assumes for its cross directory, Sec. V-B): the directed entries u -> v are
// counted per (block-row i = range of v, source u); a per-block segmented scan
// of those counts gives the block-local column offsets; set counts give the
// directory V_{i,j} (Eq. 4); a scan of directory popcounts gives the rank of
// every nonempty column; the entries are then scattered column by column.
#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <cstdarg>
#include <cstring>
#include <new>
#include <utility>

#include "cluster.cuh"
#include "common.cuh"
#include "internal.h"

namespace bfsgb {

// ------------------------------------------------------------------ errors --
namespace {
thread_local bfs_status t_last_status = BFS_OK;
thread_local char t_last_msg[512] = "no error";
}

bfs_status set_error(bfs_status s, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(t_last_msg, sizeof(t_last_msg), fmt, ap);
    va_end(ap);
    t_last_status = s;
    return s;
}

bfs_status cuda_error(cudaError_t e, const char* what, const char* file, int line) {
    bfs_status s = (e == cudaErrorMemoryAllocation) ? BFS_ERR_OUT_OF_MEMORY : BFS_ERR_CUDA;
    return set_error(s, "%s failed: %s (%s:%d)", what, cudaGetErrorString(e), file, line);
}

bool is_device_pointer(const void* p) {
    if (!p) return false;
    cudaPointerAttributes attr;
    cudaError_t e = cudaPointerGetAttributes(&attr, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged;
}

// Allocation-failure injection (bfs_debug_fail_allocation): the armed
// allocation fails as if the device were out of memory.  0 = disarmed.
std::atomic<int64_t> g_fail_countdown{0};

bfs_status DevBuf::alloc(size_t nbytes) {
    release();
    if (nbytes == 0) nbytes = 16;
    int64_t k = g_fail_countdown.load();
    while (k > 0 && !g_fail_countdown.compare_exchange_weak(k, k - 1)) {
    }
    if (k == 1) return set_error(BFS_ERR_OUT_OF_MEMORY, "cudaMalloc(%zu bytes): injected failure", nbytes);
    cudaError_t e = cudaMalloc(&ptr, nbytes);
    if (e != cudaSuccess) {
        ptr = nullptr;
        cudaGetLastError();
        return set_error(BFS_ERR_OUT_OF_MEMORY, "cudaMalloc(%zu bytes): %s", nbytes, cudaGetErrorString(e));
    }
    bytes = nbytes;
    return BFS_OK;
}

void DevBuf::release() {
    if (ptr && !part) cudaFree(ptr);
    ptr = nullptr;
    bytes = 0;
    part = false;
}

bfs_status alloc_parts(DevBuf& whole, std::initializer_list<PartSize> parts) {
    auto padded = [](size_t n) { return (n + 255) / 256 * 256 + 256; };     // parts start 256-byte aligned
    size_t total = 0;
    for (const PartSize& p : parts) total += padded(p.bytes);
    BFS_TRY(whole.alloc(total));
    char* at = whole.as<char>();
    for (const PartSize& p : parts) {
        p.buf->release();
        p.buf->ptr = at;
        p.buf->bytes = p.bytes;
        p.buf->part = true;
        at += padded(p.bytes);
    }
    return BFS_OK;
}

// ---------------------------------------------------------- call scratch --
namespace {
constexpr int kMaxDevices = 64;
std::mutex t_pool_mu;
cudaMemPool_t t_pool[kMaxDevices] = {};

std::mutex t_flag_mu;
std::condition_variable t_flag_free;
unsigned long long* t_flags = nullptr;             // kHostFlags pairs, mapped and portable
uint64_t t_flag_used[kHostFlags / 64] = {};

thread_local int t_codec_ctas = kCC;
}

int codec_ctas_cap() { return t_codec_ctas; }

bfs_status Scratch::alloc(size_t nbytes, cudaStream_t st) {
    int64_t k = g_fail_countdown.load();
    while (k > 0 && !g_fail_countdown.compare_exchange_weak(k, k - 1)) {
    }
    if (k == 1) return set_error(BFS_ERR_OUT_OF_MEMORY, "scratch of %zu bytes: injected failure", nbytes);
    int dev = 0;
    BFS_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return set_error(BFS_ERR_INVALID_ARG, "device ordinal %d out of range", dev);
    {
        std::lock_guard<std::mutex> lk(t_pool_mu);
        if (!t_pool[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.handleTypes = cudaMemHandleTypeNone;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t pool = nullptr;
            BFS_CUDA_TRY(cudaMemPoolCreate(&pool, &props));
            uint64_t keep = kScratchKept;
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
            t_pool[dev] = pool;
        }
    }
    stream = st;
    cudaError_t e = cudaMallocFromPoolAsync(&ptr, nbytes ? nbytes : 16, t_pool[dev], st);
    if (e != cudaSuccess) {
        ptr = nullptr;
        cudaGetLastError();
        return set_error(BFS_ERR_OUT_OF_MEMORY, "scratch of %zu bytes: %s", nbytes, cudaGetErrorString(e));
    }
    return BFS_OK;
}

bfs_status HostFlag::take(cudaStream_t st) {
    stream = st;
    std::unique_lock<std::mutex> lk(t_flag_mu);
    if (!t_flags) {
        void* p = nullptr;
        BFS_CUDA_TRY(cudaHostAlloc(&p, sizeof(unsigned long long) * 2 * kHostFlags,
                                   cudaHostAllocMapped | cudaHostAllocPortable));
        t_flags = static_cast<unsigned long long*>(p);
    }
    for (;;) {
        for (int w = 0; w < kHostFlags / 64; ++w)
            if (~t_flag_used[w]) {
                const int b = __builtin_ctzll(~t_flag_used[w]);
                t_flag_used[w] |= 1ull << b;
                slot = 64 * w + b;
                t_flags[2 * slot] = t_flags[2 * slot + 1] = 0ull;
                return BFS_OK;
            }
        t_flag_free.wait(lk);
    }
}

bfs_status HostFlag::wait() {
    BFS_CUDA_TRY(cudaStreamSynchronize(stream));
    waited = true;
    return BFS_OK;
}

HostFlag::~HostFlag() {
    if (slot < 0) return;
    if (!waited) cudaStreamSynchronize(stream);
    std::lock_guard<std::mutex> lk(t_flag_mu);
    t_flag_used[slot / 64] &= ~(1ull << (slot % 64));
    t_flag_free.notify_one();
}

volatile unsigned long long* HostFlag::device(int word) const { return t_flags + 2 * slot + word; }   // unified addressing
unsigned long long HostFlag::value(int word) const {
    return *static_cast<volatile unsigned long long*>(t_flags + 2 * slot + word);
}

// ------------------------------------------------------------ build kernels --
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int64_t kScanTile = (int64_t)kScanThreads * kScanItems;
// Graphs whose column counts take at most this are built in tuple order: the
// counts stay in L2 (scale 20 on 8 x 8, 32 MiB of counts: 1.66 ms against 1.95
// partitioned; scale 21, 64 MiB: 3.37 against 2.87; scale 22 on one block, 16
// MiB: 4.1 against 4.6; scale 22 on 8 x 8, 128 MiB: 8.3 against 4.6).
constexpr int64_t kDirectBytes = 48ll << 20;

// Count entries per (block-row of the destination, source) and flag bad ids.
__global__ void count_entries(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int64_t m,
                              int symmetrize, int64_t n, int64_t nb, int64_t row_stride,
                              uint32_t* __restrict__ cnt, unsigned long long* err) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = src[e], b = dst[e];
        if (a < 0 || a >= n || b < 0 || b >= n) {
            atomicOr(err, 1ull);
            continue;
        }
        atomicAdd(cnt + (int64_t)(b / nb) * row_stride + a, 1u);
        if (symmetrize) atomicAdd(cnt + (int64_t)(a / nb) * row_stride + b, 1u);
    }
}

// Directory words: bit q of word w of block b = (count of column 32w+q > 0).
// One warp per word; also writes the word's popcount into rank (scanned later).
__global__ void directory_words(const uint32_t* __restrict__ cnt, int64_t nblocks, int64_t nb,
                                int64_t words_per_block, int64_t dir_stride,
                                uint32_t* __restrict__ dir, uint32_t* __restrict__ rank) {
    const int64_t warps = nblocks * words_per_block;
    const int64_t gw0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t gstride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t gw = gw0; gw < warps; gw += gstride) {
        const int64_t b = gw / words_per_block, w = gw % words_per_block;
        const int64_t x = w * 32 + lane_id();
        const uint32_t c = (x < nb) ? cnt[b * nb + x] : 0u;
        const uint32_t bits = __ballot_sync(0xffffffffu, c != 0u);
        if (lane_id() == 0) {
            dir[b * dir_stride + w] = bits;
            rank[b * dir_stride + w] = __popc(bits);
        }
    }
}

// Segmented scan, phase A: sums of tiles of kScanTile elements; segments of
// length seg_len (uniform), tiles never cross a segment boundary.
__global__ void __launch_bounds__(kScanThreads)
scan_tile_sums(const uint32_t* __restrict__ a, int64_t nseg, int64_t seg_len, int64_t seg_stride,
               int64_t tiles_per_seg, unsigned long long* __restrict__ tile_sum) {
    __shared__ unsigned long long sm[kScanThreads / 32 + 1];
    const int64_t tile = blockIdx.x;
    const int64_t s = tile / tiles_per_seg, t = tile % tiles_per_seg;
    if (s >= nseg) return;
    const int64_t base = s * seg_stride + t * kScanTile;
    const int64_t lim = seg_len - t * kScanTile;
    unsigned long long acc = 0;
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t x = (int64_t)k * kScanThreads + threadIdx.x;
        if (x < lim) acc += a[base + x];
    }
    unsigned long long tot;
    block_incl_sum<kScanThreads>(acc, sm, &tot);
    if (threadIdx.x == 0) tile_sum[tile] = tot;
}

// Phase B: per segment, exclusive scan of its tile sums; segment totals.
__global__ void __launch_bounds__(kScanThreads)
scan_tile_offsets(unsigned long long* __restrict__ tile_sum, int64_t nseg, int64_t tiles_per_seg,
                  unsigned long long* __restrict__ seg_total) {
    __shared__ unsigned long long sm[kScanThreads / 32 + 1];
    const int64_t s = blockIdx.x;
    if (s >= nseg) return;
    unsigned long long carry = 0;
    for (int64_t t0 = 0; t0 < tiles_per_seg; t0 += kScanThreads) {
        const int64_t t = t0 + threadIdx.x;
        const unsigned long long v = (t < tiles_per_seg) ? tile_sum[s * tiles_per_seg + t] : 0ull;
        unsigned long long tot;
        const unsigned long long incl = block_incl_sum<kScanThreads>(v, sm, &tot);
        if (t < tiles_per_seg) tile_sum[s * tiles_per_seg + t] = carry + incl - v;
        carry += tot;
    }
    if (threadIdx.x == 0) seg_total[s] = carry;
}

// Phase C: exclusive scan inside each tile plus the tile offset, in place.
// Elements are loaded blocked (thread t owns elements t*kScanItems ...).
__global__ void __launch_bounds__(kScanThreads)
scan_tiles_apply(uint32_t* __restrict__ a, int64_t nseg, int64_t seg_len, int64_t seg_stride,
                 int64_t tiles_per_seg, const unsigned long long* __restrict__ tile_off) {
    __shared__ unsigned long long sm[kScanThreads / 32 + 1];
    const int64_t tile = blockIdx.x;
    const int64_t s = tile / tiles_per_seg, t = tile % tiles_per_seg;
    if (s >= nseg) return;
    const int64_t base = s * seg_stride + t * kScanTile;
    const int64_t lim = seg_len - t * kScanTile;
    uint32_t v[kScanItems];
    unsigned long long acc = 0;
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t x = (int64_t)threadIdx.x * kScanItems + k;
        v[k] = (x < lim) ? a[base + x] : 0u;
        acc += v[k];
    }
    unsigned long long tot;
    const unsigned long long incl = block_incl_sum<kScanThreads>(acc, sm, &tot);
    unsigned long long run = tile_off[tile] + incl - acc;
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t x = (int64_t)threadIdx.x * kScanItems + k;
        if (x < lim) a[base + x] = (uint32_t)run;
        run += v[k];
    }
}

// Column pointers: for every nonempty column (u_local) of block b, cp of its
// rank = the block-local offset of the column; plus the closing entry.
__global__ void column_pointers(const uint32_t* __restrict__ off, const uint32_t* __restrict__ dir,
                                const uint32_t* __restrict__ rank, int64_t nblocks, int64_t nb,
                                int64_t dir_stride, const int64_t* __restrict__ cp_base,
                                const unsigned long long* __restrict__ nnz_b,
                                const unsigned long long* __restrict__ nnzc_b, uint32_t* __restrict__ cp) {
    const int64_t total = nblocks * nb;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total;
         x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = x / nb, ul = x % nb;
        const uint32_t dw = dir[b * dir_stride + (ul >> 5)];
        const uint32_t bit = 1u << (ul & 31);
        if (dw & bit) {
            const uint32_t c = rank[b * dir_stride + (ul >> 5)] + __popc(dw & (bit - 1u));
            cp[cp_base[b] + c] = off[b * nb + ul];
        }
        if (ul == 0) cp[cp_base[b] + (int64_t)nnzc_b[b]] = (uint32_t)nnz_b[b];
    }
}

// Scatter every entry into its column (order inside a column is arbitrary).
__global__ void scatter_entries(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int64_t m,
                                int symmetrize, int64_t nb, int p, int64_t row_stride,
                                uint32_t* __restrict__ off, const int64_t* __restrict__ ir_base,
                                int32_t* __restrict__ ir) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = src[e], b = dst[e];
        {
            const int64_t i = b / nb, j = a / nb;
            const uint32_t pos = atomicAdd(off + i * row_stride + a, 1u);
            ir[ir_base[i * p + j] + pos] = b;
        }
        if (symmetrize) {
            const int64_t i = a / nb, j = b / nb;
            const uint32_t pos = atomicAdd(off + i * row_stride + b, 1u);
            ir[ir_base[i * p + j] + pos] = a;
        }
    }
}

// ------------------------------------------------------ partitioned build --
// Counting and scattering the entries in tuple order costs an L2 reduction and
// an atomic with its result per entry on random counts, and a random 4-byte
// store: at 134M entries 1.3 + 5.6 ms, most of it 32-byte sectors moved to and
// from DRAM for 4 bytes each (with the counts in L2 still 1.1 + 2.2 ms: the
// rate of L2 atomics).  Larger graphs therefore partition the entries by their
// block and a part of its source range first (0.7 ms); a bucket's columns are
// then counted, and its entries placed, by one CTA through counts in shared
// memory, and the bucket's stores fall into one stretch of the entries.  A
// partitioned entry is its column's count index, relative to the first
// block-row of its group, and its destination.
//
// Three kinds of graph are built in tuple order whatever their size:
//   - with few entries per count: the partitioned build reads and writes every
//     count where the direct one touches the entries' own.  Uniform 2^25 vertices
//     on 8 x 8, entries per count 1/16: 6.87 ms against 7.48, 1/8: 9.15 against
//     8.44; on 32 x 32, 1/16: 25.9 against 26.9, 1/8: 35.1 against 32.5;
//   - whose tuples come in an order in which neighbours share their columns'
//     sectors (a mesh in its natural order, a sorted directed graph): the counts
//     they touch are on chip anyway.  A 3000 x 3000 grid on 8 x 8 2.30 ms against
//     3.46, a sorted directed scale-24 graph on 16 x 16 10.1 against 15.7;
//   - whose partition buffer does not fit in memory beside the counts and the
//     entries.
constexpr int kPartThreads = 512;
constexpr int kPartTuples = 8;                                  // per thread and tile
constexpr int kPartTile = kPartThreads * kPartTuples;           // tuples per tile: up to twice the entries
constexpr int kGroupBuckets = 1024;                             // buckets of one partition pass
constexpr int kAllBuckets = 16384;                              // buckets of all passes
constexpr int kColThreads = 1024;
constexpr int kColWindow = 32768;                               // columns counted together in shared memory
constexpr int kMaxPartGrid = 32;                                // grids up to 32 x 32 (1024 blocks) are partitioned
constexpr int kCountsPerEntry = 8;                              // more counts per entry than this: direct
constexpr int kColCtas = 152;
constexpr int64_t kMinShare = 32768;                            // entries of a part of a split bucket, at least

struct PartArgs {
    const int32_t* src;
    const int32_t* dst;
    int64_t m;
    int symmetrize, p;
    int parts, shift;        // parts of a block's source range, 2^shift sources each
    uint32_t n, nb;
};

// Bucket of the entry u -> v, u in range ru, v in range rv.
__device__ __forceinline__ uint32_t bucket_of(const PartArgs& a, uint32_t u, uint32_t ru, uint32_t rv) {
    return (rv * (uint32_t)a.p + ru) * (uint32_t)a.parts + ((u - ru * a.nb) >> a.shift);
}

// What order the tuples come in, from kOrderWarps pieces of 32 of them spread
// over the whole list: said[1] counts the entries whose column lies in the same 16
// counts as the one of the tuple before it, said[2] the pieces that start in the
// same 16 counts as the piece before them (a column with many of all entries).
constexpr int kOrderWarps = 4096;

__global__ void __launch_bounds__(kPartThreads) tuple_order(PartArgs a, unsigned long long* said) {
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (w >= kOrderWarps) return;
    const int64_t step = a.m / kOrderWarps;
    const uint32_t u = (uint32_t)a.src[w * step + lane_id()] >> 4, v = (uint32_t)a.dst[w * step + lane_id()] >> 4;
    const uint32_t pu = __shfl_up_sync(0xffffffffu, u, 1), pv = __shfl_up_sync(0xffffffffu, v, 1);
    const uint32_t near = warp_sum(lane_id() ? (uint32_t)(pu == u) + (uint32_t)(a.symmetrize && pv == v) : 0u);
    if (lane_id() != 0) return;
    atomicAdd(said + 1, (unsigned long long)near);
    if (w > 0 && ((uint32_t)a.src[(w - 1) * step] >> 4 == u || (a.symmetrize && (uint32_t)a.dst[(w - 1) * step] >> 4 == v)))
        atomicAdd(said + 2, 1ull);
}

// Entries per bucket; flags ids outside [0, n).
__global__ void __launch_bounds__(kPartThreads) bucket_counts(PartArgs a, int buckets, unsigned long long* counts,
                                                              unsigned long long* err) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem);
    for (int b = threadIdx.x; b < buckets; b += kPartThreads) s_cnt[b] = 0;
    __syncthreads();
    bool bad = false;
    // a CTA's tuples are below 2^31 for any grid of a CTA or more per SM
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < a.m; e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t u = (uint32_t)a.src[e], v = (uint32_t)a.dst[e];
        if (u >= a.n || v >= a.n) {
            bad = true;
            continue;
        }
        const uint32_t ru = u / a.nb, rv = v / a.nb;
        atomicAdd(s_cnt + bucket_of(a, u, ru, rv), 1u);
        if (a.symmetrize) atomicAdd(s_cnt + bucket_of(a, v, rv, ru), 1u);
    }
    if (bad) atomicOr(err, 1ull);
    __syncthreads();
    for (int b = threadIdx.x; b < buckets; b += kPartThreads)
        if (s_cnt[b]) atomicAdd(counts + b, (unsigned long long)s_cnt[b]);
}

// The entries of block-rows [r0, r1) into their buckets (b0: the first of
// them): a tile's entries are ranked per bucket in shared memory, every bucket
// takes its space with one atomic, and the tile is written out bucket by
// bucket from a sorted copy.
__global__ void __launch_bounds__(kPartThreads) partition_entries(PartArgs a, int r0, int r1, uint32_t b0,
                                                                  unsigned long long* __restrict__ cursor,
                                                                  uint2* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint2* s_pair = reinterpret_cast<uint2*>(smem);                                   // 2 * kPartTile
    unsigned long long* s_base = reinterpret_cast<unsigned long long*>(s_pair + 2 * kPartTile);
    uint32_t* s_off = reinterpret_cast<uint32_t*>(s_base + kGroupBuckets);            // counts, then offsets
    uint16_t* s_bkt = reinterpret_cast<uint16_t*>(s_off + kGroupBuckets);             // 2 * kPartTile
    __shared__ uint32_t s_scan[kPartThreads / 32 + 1];
    const uint32_t stride = (uint32_t)a.p * a.nb;
    const int64_t ntiles = (a.m + kPartTile - 1) / kPartTile;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        s_off[2 * threadIdx.x] = 0;
        s_off[2 * threadIdx.x + 1] = 0;
        __syncthreads();
        uint32_t u[kPartTuples], v[kPartTuples], bk[2 * kPartTuples], rk[2 * kPartTuples];
#pragma unroll
        for (int k = 0; k < kPartTuples; ++k) {
            const int64_t e = t * kPartTile + k * kPartThreads + threadIdx.x;
            u[k] = e < a.m ? (uint32_t)a.src[e] : 0u;
            v[k] = e < a.m ? (uint32_t)a.dst[e] : 0u;
        }
#pragma unroll
        for (int k = 0; k < kPartTuples; ++k) {
            const bool in = t * kPartTile + k * kPartThreads + threadIdx.x < a.m;
            const uint32_t ru = u[k] / a.nb, rv = v[k] / a.nb;
            bk[2 * k] = (in && (int)rv >= r0 && (int)rv < r1) ? bucket_of(a, u[k], ru, rv) - b0 : ~0u;
            bk[2 * k + 1] = (in && a.symmetrize && (int)ru >= r0 && (int)ru < r1) ? bucket_of(a, v[k], rv, ru) - b0 : ~0u;
            rk[2 * k] = bk[2 * k] != ~0u ? atomicAdd(s_off + bk[2 * k], 1u) : 0u;
            rk[2 * k + 1] = bk[2 * k + 1] != ~0u ? atomicAdd(s_off + bk[2 * k + 1], 1u) : 0u;
        }
        __syncthreads();
        // space for every bucket's entries, and their places in the sorted copy
        const uint32_t c0 = s_off[2 * threadIdx.x], c1 = s_off[2 * threadIdx.x + 1];
        uint32_t total;
        const uint32_t excl = block_excl_scan<kPartThreads>(c0 + c1, 0u, OpSum(), s_scan, &total);
        s_off[2 * threadIdx.x] = excl;
        s_off[2 * threadIdx.x + 1] = excl + c0;
        if (c0) s_base[2 * threadIdx.x] = atomicAdd(cursor + 2 * threadIdx.x, (unsigned long long)c0) - excl;
        if (c1) s_base[2 * threadIdx.x + 1] = atomicAdd(cursor + 2 * threadIdx.x + 1, (unsigned long long)c1) - (excl + c0);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPartTuples; ++k) {
            // the column's count index: block-row (relative to the group's first) x p*nb + source
            if (bk[2 * k] != ~0u) {
                const uint32_t at = s_off[bk[2 * k]] + rk[2 * k];
                s_pair[at] = make_uint2((v[k] / a.nb - (uint32_t)r0) * stride + u[k], v[k]);
                s_bkt[at] = (uint16_t)bk[2 * k];
            }
            if (bk[2 * k + 1] != ~0u) {
                const uint32_t at = s_off[bk[2 * k + 1]] + rk[2 * k + 1];
                s_pair[at] = make_uint2((u[k] / a.nb - (uint32_t)r0) * stride + v[k], u[k]);
                s_bkt[at] = (uint16_t)bk[2 * k + 1];
            }
        }
        __syncthreads();
        for (uint32_t q = threadIdx.x; q < total; q += kPartThreads) out[s_base[s_bkt[q]] + q] = s_pair[q];
        __syncthreads();
    }
}

constexpr size_t kPartSmem = sizeof(uint2) * 2 * kPartTile + (sizeof(uint32_t) + sizeof(unsigned long long)) * kGroupBuckets +
                             sizeof(uint16_t) * 2 * kPartTile;
static_assert(kGroupBuckets == 2 * kPartThreads, "a thread scans two buckets");

// Work of a CTA: a bucket of a group, or a share of a large one's entries.
struct ColUnit {
    int64_t e0, e1;         // entries
    int32_t bucket;
    int32_t share;          // -1: the whole bucket; else its row of `before`
};

// One CTA per unit, taken in turn from *next, kColWindow of its bucket's columns
// at a time (a bucket with more columns reads its entries again, from L2).
//   COUNT: the entries of every column, written to cnt (the group's counts).
//          The shares of a split bucket add theirs to cnt (zero before) and
//          keep what was there: the place of their entries in the column.
//   else:  every entry into its column (order inside a column is arbitrary);
//          off holds the columns' offsets in their blocks, ir_base the blocks'.
// A bucket with many times the entries of the others would leave the chip to
// one CTA (a Kronecker graph whose labels are not scrambled: 6% of scale 22's
// entries on 8 x 8 in one of 1024 buckets: COUNT and fill took 1.6 + 5.9 ms, the
// build 11.4; with the shares of split_buckets 5.7).
template <bool COUNT>
__global__ void __launch_bounds__(kColThreads) bucket_columns(PartArgs a, const uint2* __restrict__ pairs,
                                                              const ColUnit* __restrict__ units, int nunits, int* next,
                                                              uint32_t* __restrict__ cnt,
                                                              uint32_t* __restrict__ before, int64_t before_cols,
                                                              const int64_t* __restrict__ ir_base,
                                                              int32_t* __restrict__ ir) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_unit;
    uint32_t* s_col = reinterpret_cast<uint32_t*>(smem);
    constexpr int K = 4;
    for (;;) {
        if (threadIdx.x == 0) s_unit = atomicAdd(next, 1);
        __syncthreads();
        const int x0 = s_unit;
        __syncthreads();
        if (x0 >= nunits) return;
        const ColUnit un = units[x0];
        const uint32_t block = (uint32_t)un.bucket / (uint32_t)a.parts, part = (uint32_t)un.bucket % (uint32_t)a.parts;
        const uint32_t first = part << a.shift;
        const uint32_t cols = first < a.nb ? min(1u << a.shift, a.nb - first) : 0u;
        for (uint32_t w0 = 0; w0 < cols; w0 += kColWindow) {
            const uint32_t wn = min((uint32_t)kColWindow, cols - w0);
            const uint32_t c0 = block * a.nb + first + w0;         // count index of the window's first column
            uint32_t* g = cnt + c0;
            uint32_t* bf = un.share >= 0 ? before + un.share * before_cols + w0 : nullptr;
            for (uint32_t c = threadIdx.x; c < wn; c += kColThreads) s_col[c] = COUNT ? 0u : g[c] + (bf ? bf[c] : 0u);
            __syncthreads();
            int32_t* out = COUNT ? nullptr : ir + ir_base[block];
            for (int64_t e = un.e0 + threadIdx.x; e < un.e1; e += K * kColThreads) {
                uint2 x[K];
#pragma unroll
                for (int k = 0; k < K; ++k) x[k] = e + k * kColThreads < un.e1 ? pairs[e + k * kColThreads] : make_uint2(~0u, 0u);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    if (e + k * kColThreads >= un.e1 || x[k].x - c0 >= wn) continue;
                    const uint32_t pos = atomicAdd(s_col + (x[k].x - c0), 1u);
                    if (!COUNT) out[pos] = (int32_t)x[k].y;
                }
            }
            __syncthreads();
            if (COUNT)
                for (uint32_t c = threadIdx.x; c < wn; c += kColThreads) {
                    if (!bf) g[c] = s_col[c];
                    else bf[c] = s_col[c] ? atomicAdd(g + c, s_col[c]) : 0u;
                }
            __syncthreads();
        }
    }
}

// The units of buckets with `held` entries each, laid out from entry 0 on.  A
// bucket of more than a CTA's mean is cut into shares of half of it (the largest
// units first, then).  Returns the number of shares.
int split_buckets(const uint64_t* held, int buckets, std::vector<ColUnit>& units) {
    int64_t total = 0;
    for (int b = 0; b < buckets; ++b) total += (int64_t)held[b];
    const int64_t share = std::max(kMinShare, total / (2 * kColCtas));
    int shares = 0;
    int64_t at = 0;
    units.clear();
    for (int b = 0; b < buckets; ++b) {
        const int64_t end = at + (int64_t)held[b];
        if (end - at <= 2 * share) units.push_back({at, end, b, -1});
        else
            for (int64_t e = at; e < end; e += share) units.push_back({e, std::min(e + share, end), b, shares++});
        at = end;
    }
    if (shares)
        std::stable_sort(units.begin(), units.end(),
                         [](const ColUnit& x, const ColUnit& y) { return x.e1 - x.e0 > y.e1 - y.e0; });
    return shares;
}

// The parts of a block's source range: as many as give kColWindow columns
// each, on all blocks at most kAllBuckets and in a block-row at most kGroupBuckets.
void choose_parts(PartArgs& a) {
    const int64_t nblocks = (int64_t)a.p * a.p;
    a.shift = 31;
    while (a.shift > 0 && (1ll << (a.shift - 1)) >= (int64_t)a.nb) --a.shift;
    a.parts = 1;
    while (a.shift > 0 && (1ll << a.shift) > kColWindow) {
        const int64_t more = ((int64_t)a.nb + (1ll << (a.shift - 1)) - 1) >> (a.shift - 1);
        if (nblocks * more > kAllBuckets || a.p * more > kGroupBuckets) break;
        a.parts = (int)more;
        --a.shift;
    }
}

// Degree of every vertex u: its entries in the blocks of `rows` block-rows (the
// rows of the counts, read in order), added to deg, saturated at 2^32 - 1.
__global__ void vertex_degrees(const uint32_t* __restrict__ cnt, int rows, int64_t row_stride, int64_t n,
                               uint32_t* __restrict__ deg) {
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
        uint64_t d = deg[u];
        for (int i = 0; i < rows; i += 8) {                             // eight rows' counts in flight
            uint32_t c[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) c[k] = i + k < rows ? __ldg(cnt + (i + k) * row_stride + u) : 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k) d += c[k];
        }
        deg[u] = d > 0xffffffffull ? 0xffffffffu : (uint32_t)d;
    }
}

// Bitmap of the vertices without entries: no search reaches them from
// another vertex, and a bottom-up level need not scan them.
__global__ void isolated_bits(const uint32_t* __restrict__ deg, int64_t n, int64_t words, uint32_t* __restrict__ iso) {
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < words; w += (int64_t)gridDim.x * blockDim.x) {
        uint32_t x = 0;
        for (int b = 0; b < 32; ++b) {
            const int64_t v = w * 32 + b;
            if (v < n && deg[v] == 0) x |= 1u << b;
        }
        iso[w] = x;
    }
}

// Bottom-up layout, step 1: exclusive scan of the degrees in tiles of 1024,
// in 64 bits, with every tile's total.
__global__ void __launch_bounds__(1024) degree_tile_scan(const uint32_t* __restrict__ deg, int64_t n,
                                                         int64_t* __restrict__ ptr, int64_t* __restrict__ tile_sum) {
    __shared__ int64_t warp_tot[32];
    const int64_t x = blockIdx.x * 1024LL + threadIdx.x;
    const int64_t d = x < n ? (int64_t)deg[x] : 0;
    int64_t incl = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane_id() >= o) incl += y;
    }
    if (lane_id() == 31) warp_tot[threadIdx.x >> 5] = incl;
    __syncthreads();
    if (threadIdx.x < 32) {
        int64_t t = warp_tot[threadIdx.x], ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if ((int)threadIdx.x >= o) ti += y;
        }
        warp_tot[threadIdx.x] = ti - t;
        if (threadIdx.x == 31) tile_sum[blockIdx.x] = ti;
    }
    __syncthreads();
    if (x <= n) ptr[x] = incl - d + warp_tot[threadIdx.x >> 5];      // ptr[n]: the entries before n in its tile
}

// Step 2: add the tiles' scanned totals; ptr[n] = the total.
__global__ void degree_tile_add(int64_t* __restrict__ ptr, int64_t n, const int64_t* __restrict__ tile_base) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x <= n; x += (int64_t)gridDim.x * blockDim.x)
        ptr[x] += tile_base[x >> 10];
}

// Step 3: the columns of every vertex v (range i) in blocks (0,i), (1,i), ...
// copied back to back from bu_ptr[v]: its neighbours grouped by range j in
// ascending order (in any order inside a range).
__global__ void bottom_up_rows(const uint32_t* __restrict__ dir, const uint32_t* __restrict__ rank,
                               int64_t dir_stride, const uint32_t* __restrict__ cp,
                               const int64_t* __restrict__ cp_base, const int64_t* __restrict__ ir_base,
                               const int32_t* __restrict__ ir, int p, int64_t nb, int64_t n,
                               const int64_t* __restrict__ ptr, int32_t* __restrict__ adj) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = v / nb, vl = v - i * nb;
        const uint32_t bit = 1u << (vl & 31);
        int64_t pos = ptr[v];
        for (int j = 0; j < p; ++j) {
            const int64_t b = (int64_t)j * p + i;
            const uint32_t dw = dir[b * dir_stride + (vl >> 5)];
            if (!(dw & bit)) continue;
            const int64_t c = cp_base[b] + rank[b * dir_stride + (vl >> 5)] + __popc(dw & (bit - 1u));
            const int32_t* col = ir + ir_base[b];
            const uint32_t c0 = cp[c], c1 = cp[c + 1];
            for (uint32_t e = c0; e < c1; ++e) adj[pos++] = col[e];
        }
    }
}

// CSR -> per-entry source ids.
__global__ void expand_rows(const int64_t* __restrict__ row_ptr, int64_t n, int32_t* __restrict__ src) {
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * blockDim.x)
        for (int64_t e = row_ptr[u]; e < row_ptr[u + 1]; ++e) src[e] = (int32_t)u;
}

__global__ void check_csr(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int64_t n,
                          int64_t nnz, unsigned long long* err) {
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n;
         u += (int64_t)gridDim.x * blockDim.x) {
        if (row_ptr[u] > row_ptr[u + 1] || row_ptr[u] < 0 || row_ptr[u + 1] > nnz) atomicOr(err, 1ull);
    }
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x)
        if (col[e] < 0 || col[e] >= n) atomicOr(err, 1ull);
}

int grid_for(int64_t work, int threads) {
    int64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 152 * 64) g = 152 * 64;
    return (int)g;
}

// In-place segmented exclusive scan of `a` (nseg segments of seg_len
// elements, segment s at s*seg_stride); seg_total[s] receives the totals.
bfs_status segmented_scan(uint32_t* a, int64_t nseg, int64_t seg_len, int64_t seg_stride,
                          std::vector<uint64_t>& totals, cudaStream_t st) {
    const int64_t tiles_per_seg = seg_len > 0 ? (seg_len + kScanTile - 1) / kScanTile : 1;
    Scratch tile_sum, seg_total;
    BFS_TRY(tile_sum.alloc(sizeof(unsigned long long) * nseg * tiles_per_seg, st));
    BFS_TRY(seg_total.alloc(sizeof(unsigned long long) * nseg, st));
    const int64_t ntiles = nseg * tiles_per_seg;
    if (ntiles > 0x7fffffffLL) return set_error(BFS_ERR_INVALID_ARG, "graph too large for the layout scan");
    scan_tile_sums<<<(unsigned)ntiles, kScanThreads, 0, st>>>(a, nseg, seg_len, seg_stride, tiles_per_seg,
                                                              tile_sum.as<unsigned long long>());
    BFS_CUDA_TRY(cudaGetLastError());
    scan_tile_offsets<<<(unsigned)nseg, kScanThreads, 0, st>>>(tile_sum.as<unsigned long long>(), nseg,
                                                               tiles_per_seg, seg_total.as<unsigned long long>());
    BFS_CUDA_TRY(cudaGetLastError());
    totals.assign(nseg, 0);
    BFS_CUDA_TRY(cudaMemcpyAsync(totals.data(), seg_total.ptr, sizeof(uint64_t) * nseg, cudaMemcpyDeviceToHost, st));
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    for (int64_t s = 0; s < nseg; ++s)
        if (totals[s] > 0xffffffffull)
            return set_error(BFS_ERR_INVALID_ARG, "a block holds 2^32 or more entries; use a larger grid");
    scan_tiles_apply<<<(unsigned)ntiles, kScanThreads, 0, st>>>(a, nseg, seg_len, seg_stride, tiles_per_seg,
                                                                tile_sum.as<unsigned long long>());
    BFS_CUDA_TRY(cudaGetLastError());
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    return BFS_OK;
}

}  // namespace

bfs_status build_layout(bfs_graph* g, int64_t n, int64_t m, const int32_t* d_src, const int32_t* d_dst,
                        int symmetrize, cudaStream_t st) {
    Layout& L = g->L;
    const int p = L.p;
    L.n = n;
    L.nb = (n + p - 1) / p;
    L.nnz = symmetrize ? 2 * m : m;
    const int64_t nb = L.nb;
    const int64_t nblocks = (int64_t)p * p;
    const int64_t row_stride = (int64_t)p * nb;
    const int64_t words_per_block = (nb + 31) / 32;
    L.dir_stride = ((words_per_block + 3 + 3) / 4) * 4;   // >= 3 words of padding, 16-byte rows

    bool partitioned = p <= kMaxPartGrid && 4 * nblocks * nb > kDirectBytes && L.nnz * kCountsPerEntry >= nblocks * nb;
    PartArgs pa{d_src, d_dst, m, symmetrize, p, 1, 31, (uint32_t)n, (uint32_t)nb};
    if (partitioned) choose_parts(pa);
    const int buckets = (int)nblocks * pa.parts, per_row = p * pa.parts;
    DevBuf cnt;
    Scratch said, cursor;
    BFS_TRY(cnt.alloc(sizeof(uint32_t) * nblocks * nb));
    BFS_TRY(said.alloc(3 * sizeof(unsigned long long), st));
    BFS_CUDA_TRY(cudaMemsetAsync(said.ptr, 0, 3 * sizeof(unsigned long long), st));
    unsigned long long h_said[3] = {0, 0, 0};                          // bad ids; the tuples' order (tuple_order)
    auto hear = [&]() -> bfs_status {
        BFS_CUDA_TRY(cudaGetLastError());
        BFS_CUDA_TRY(cudaMemcpyAsync(h_said, said.ptr, sizeof(h_said), cudaMemcpyDeviceToHost, st));
        BFS_CUDA_TRY(cudaStreamSynchronize(st));
        if (h_said[0]) return set_error(BFS_ERR_INVALID_ARG, "an edge names a vertex outside [0, %lld)", (long long)n);
        return BFS_OK;
    };
    if (partitioned && m >= 32 * (int64_t)kOrderWarps) {
        tuple_order<<<kOrderWarps * 32 / kPartThreads, kPartThreads, 0, st>>>(pa, said.as<unsigned long long>());
        BFS_TRY(hear());
        // in order, and no column that draws the atomics of many: built in tuple order
        const uint64_t seen = (uint64_t)kOrderWarps * 31 * (symmetrize ? 2 : 1);
        partitioned = !(h_said[1] >= seen / 4 * 3 && h_said[2] < kOrderWarps / 32);
    }
    std::vector<uint64_t> held(partitioned ? buckets : 0);             // entries per bucket
    if (partitioned) {
        const size_t cursor_bytes = sizeof(unsigned long long) * std::max(buckets, kGroupBuckets);
        BFS_TRY(cursor.alloc(cursor_bytes, st));
        BFS_CUDA_TRY(cudaMemsetAsync(cursor.ptr, 0, cursor_bytes, st));
        const size_t smem = sizeof(uint32_t) * (size_t)buckets;
        BFS_CUDA_TRY(cudaFuncSetAttribute(bucket_counts, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(sizeof(uint32_t) * kAllBuckets)));
        bucket_counts<<<152 * 3, kPartThreads, smem, st>>>(pa, buckets, cursor.as<unsigned long long>(),
                                                           said.as<unsigned long long>());
        BFS_CUDA_TRY(cudaMemcpyAsync(held.data(), cursor.ptr, sizeof(uint64_t) * buckets, cudaMemcpyDeviceToHost, st));
        BFS_TRY(hear());
    }

    BFS_TRY(alloc_parts(L.small, {{&L.dir, sizeof(uint32_t) * nblocks * L.dir_stride},
                                  {&L.rank, sizeof(uint32_t) * nblocks * L.dir_stride},
                                  {&L.deg, sizeof(uint32_t) * n},
                                  {&L.cp_base_d, sizeof(int64_t) * nblocks},
                                  {&L.ir_base_d, sizeof(int64_t) * nblocks}}));
    BFS_TRY(L.ir.alloc(sizeof(int32_t) * (L.nnz > 0 ? L.nnz : 1)));
    BFS_CUDA_TRY(cudaMemsetAsync(L.dir.ptr, 0, L.dir.bytes, st));
    BFS_CUDA_TRY(cudaMemsetAsync(L.rank.ptr, 0, L.rank.bytes, st));
    BFS_CUDA_TRY(cudaMemsetAsync(L.deg.ptr, 0, L.deg.bytes, st));

    // block-rows [r0, r1) counted: their degrees, directory and popcounts; then
    // the counts become block-local column offsets (an exclusive scan per block)
    std::vector<uint64_t> nnzc_b, nnz_b;
    auto counted = [&](int r0, int r1) -> bfs_status {
        uint32_t* c = cnt.as<uint32_t>() + r0 * row_stride;
        const int64_t blocks = (int64_t)(r1 - r0) * p, b0 = (int64_t)r0 * p;
        vertex_degrees<<<grid_for(n, 256), 256, 0, st>>>(c, r1 - r0, row_stride, n, L.deg.as<uint32_t>());
        directory_words<<<grid_for(blocks * words_per_block * 32, 256), 256, 0, st>>>(
            c, blocks, nb, words_per_block, L.dir_stride, L.dir.as<uint32_t>() + b0 * L.dir_stride,
            L.rank.as<uint32_t>() + b0 * L.dir_stride);
        BFS_CUDA_TRY(cudaGetLastError());
        std::vector<uint64_t> totals;
        BFS_TRY(segmented_scan(c, blocks, nb, nb, totals, st));
        nnz_b.insert(nnz_b.end(), totals.begin(), totals.end());
        return BFS_OK;
    };

    auto partitioned_columns = [&]() -> bfs_status {
        // groups of block-rows: at most kGroupBuckets buckets, and an eighth of all
        // entries, at least 1 GiB of them (a block-row that holds more is a group of
        // its own: with p = 1 the buffer takes twice the entries' own memory); every
        // group reads all tuples once
        struct Group { int r0, r1; int64_t entries; };
        std::vector<Group> groups;
        const int64_t room = std::max<int64_t>(L.nnz / 8, (1ll << 30) / (int64_t)sizeof(uint2));
        int64_t most = 1;
        for (int r = 0; r < p; ++r) {
            int64_t row = 0;
            for (int k = 0; k < per_row; ++k) row += (int64_t)held[(size_t)r * per_row + k];
            if (groups.empty() || groups.back().entries + row > room ||
                (r + 1 - groups.back().r0) * per_row > kGroupBuckets ||
                (int64_t)(r + 1 - groups.back().r0) * row_stride > 0xffffffffll)
                groups.push_back({r, r + 1, row});
            else
                groups.back() = {groups.back().r0, r + 1, groups.back().entries + row};
            most = std::max(most, groups.back().entries);
        }
        DevBuf pairs;                                                   // released on return: the column offsets come next
        Scratch d_base, d_units, d_next;
        constexpr size_t kMaxUnits = kGroupBuckets + 3 * kColCtas;      // 2 kColCtas shares and one more per split bucket
        BFS_TRY(pairs.alloc(sizeof(uint2) * (size_t)most));
        BFS_TRY(d_base.alloc(sizeof(int64_t) * (size_t)nblocks, st));
        BFS_TRY(d_units.alloc(sizeof(ColUnit) * kMaxUnits, st));
        BFS_TRY(d_next.alloc(2 * sizeof(int), st));
        std::vector<int64_t> base((size_t)nblocks, 0);                  // first entry of every block
        for (int64_t b = 0, at = 0; b < nblocks; ++b) {
            base[b] = at;
            for (int k = 0; k < pa.parts; ++k) at += (int64_t)held[(size_t)b * pa.parts + k];
        }
        BFS_CUDA_TRY(cudaMemcpyAsync(d_base.ptr, base.data(), sizeof(int64_t) * nblocks, cudaMemcpyHostToDevice, st));
        const int col_smem = (int)sizeof(uint32_t) * (int)std::min<int64_t>(kColWindow, nb);
        const int64_t bucket_cols = std::min<int64_t>(1ll << pa.shift, nb);
        BFS_CUDA_TRY(cudaFuncSetAttribute(partition_entries, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPartSmem));
        for (auto k : {bucket_columns<true>, bucket_columns<false>})
            BFS_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)sizeof(uint32_t) * kColWindow));
        std::vector<ColUnit> units;
        for (const Group& g : groups) {
            const int b0 = g.r0 * per_row, nbk = (g.r1 - g.r0) * per_row;
            std::vector<int64_t> at((size_t)nbk, 0);
            for (int k = 0; k + 1 < nbk; ++k) at[k + 1] = at[k] + (int64_t)held[(size_t)b0 + k];
            const int shares = split_buckets(held.data() + b0, nbk, units);
            if (units.size() > kMaxUnits) return set_error(BFS_ERR_CUDA, "layout build: %zu units", units.size());
            uint32_t* c = cnt.as<uint32_t>() + g.r0 * row_stride;
            Scratch before;                                             // per share and column: the entries of the shares before
            if (shares) {
                BFS_TRY(before.alloc(sizeof(uint32_t) * (size_t)(shares * bucket_cols), st));
                BFS_CUDA_TRY(cudaMemsetAsync(c, 0, sizeof(uint32_t) * (size_t)((g.r1 - g.r0) * row_stride), st));
            }
            BFS_CUDA_TRY(cudaMemcpyAsync(cursor.ptr, at.data(), sizeof(int64_t) * nbk, cudaMemcpyHostToDevice, st));
            BFS_CUDA_TRY(cudaMemcpyAsync(d_units.ptr, units.data(), sizeof(ColUnit) * units.size(), cudaMemcpyHostToDevice, st));
            BFS_CUDA_TRY(cudaMemsetAsync(d_next.ptr, 0, 2 * sizeof(int), st));
            partition_entries<<<152 * 2, kPartThreads, kPartSmem, st>>>(pa, g.r0, g.r1, (uint32_t)b0,
                                                                        cursor.as<unsigned long long>(), pairs.as<uint2>());
            bucket_columns<true><<<kColCtas, kColThreads, col_smem, st>>>(
                pa, pairs.as<uint2>(), d_units.as<ColUnit>(), (int)units.size(), d_next.as<int>(), c,
                before.as<uint32_t>(), bucket_cols, nullptr, nullptr);
            BFS_CUDA_TRY(cudaGetLastError());
            BFS_TRY(counted(g.r0, g.r1));                                // synchronises: the host arrays are free to go
            bucket_columns<false><<<kColCtas, kColThreads, col_smem, st>>>(
                pa, pairs.as<uint2>(), d_units.as<ColUnit>(), (int)units.size(), d_next.as<int>() + 1, c,
                before.as<uint32_t>(), bucket_cols, d_base.as<int64_t>() + (int64_t)g.r0 * p, L.ir.as<int32_t>());
            BFS_CUDA_TRY(cudaGetLastError());
        }
        return BFS_OK;
    };
    if (partitioned) {
        const bfs_status rc = partitioned_columns();
        if (rc == BFS_ERR_OUT_OF_MEMORY) {                               // the direct build needs none of it
            partitioned = false;
            nnz_b.clear();
            BFS_CUDA_TRY(cudaMemsetAsync(L.deg.ptr, 0, L.deg.bytes, st));
        } else if (rc != BFS_OK) {
            return rc;
        }
    }
    if (!partitioned) {
        BFS_CUDA_TRY(cudaMemsetAsync(cnt.ptr, 0, cnt.bytes, st));
        count_entries<<<grid_for(m, 256), 256, 0, st>>>(d_src, d_dst, m, symmetrize, n, nb, row_stride,
                                                        cnt.as<uint32_t>(), said.as<unsigned long long>());
        BFS_TRY(hear());
        BFS_TRY(counted(0, p));
    }

    // rank = exclusive scan of popcounts per block; nnzc_b = totals
    BFS_TRY(segmented_scan(L.rank.as<uint32_t>(), nblocks, L.dir_stride, L.dir_stride, nnzc_b, st));

    L.cp_base.assign(nblocks, 0);
    L.ir_base.assign(nblocks, 0);
    L.nnzc.assign(nblocks, 0);
    L.nnz_b.assign(nblocks, 0);
    int64_t cpt = 0, irt = 0;
    for (int64_t b = 0; b < nblocks; ++b) {
        L.cp_base[b] = cpt;
        L.ir_base[b] = irt;
        L.nnzc[b] = (int64_t)nnzc_b[b];
        L.nnz_b[b] = (int64_t)nnz_b[b];
        cpt += (int64_t)nnzc_b[b] + 1;
        irt += (int64_t)nnz_b[b];
    }
    L.nnzc_total = cpt - nblocks;
    if (irt != L.nnz) return set_error(BFS_ERR_CUDA, "layout build lost entries (%lld of %lld)", (long long)irt, (long long)L.nnz);

    BFS_TRY(L.cp.alloc(sizeof(uint32_t) * (cpt > 0 ? cpt : 1)));
    Scratch d_nnz_b, d_nnzc_b;
    BFS_TRY(d_nnz_b.alloc(sizeof(uint64_t) * nblocks, st));
    BFS_TRY(d_nnzc_b.alloc(sizeof(uint64_t) * nblocks, st));
    BFS_CUDA_TRY(cudaMemcpyAsync(L.cp_base_d.ptr, L.cp_base.data(), sizeof(int64_t) * nblocks, cudaMemcpyHostToDevice, st));
    BFS_CUDA_TRY(cudaMemcpyAsync(L.ir_base_d.ptr, L.ir_base.data(), sizeof(int64_t) * nblocks, cudaMemcpyHostToDevice, st));
    BFS_CUDA_TRY(cudaMemcpyAsync(d_nnz_b.ptr, nnz_b.data(), sizeof(uint64_t) * nblocks, cudaMemcpyHostToDevice, st));
    BFS_CUDA_TRY(cudaMemcpyAsync(d_nnzc_b.ptr, nnzc_b.data(), sizeof(uint64_t) * nblocks, cudaMemcpyHostToDevice, st));

    column_pointers<<<grid_for(nblocks * nb, 256), 256, 0, st>>>(
        cnt.as<uint32_t>(), L.dir.as<uint32_t>(), L.rank.as<uint32_t>(), nblocks, nb, L.dir_stride,
        L.cp_base_d.as<int64_t>(), d_nnz_b.as<unsigned long long>(), d_nnzc_b.as<unsigned long long>(),
        L.cp.as<uint32_t>());
    BFS_CUDA_TRY(cudaGetLastError());
    if (!partitioned)
        scatter_entries<<<grid_for(m, 256), 256, 0, st>>>(d_src, d_dst, m, symmetrize, nb, p, row_stride,
                                                          cnt.as<uint32_t>(), L.ir_base_d.as<int64_t>(), L.ir.as<int32_t>());
    BFS_CUDA_TRY(cudaGetLastError());
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    return BFS_OK;
}

bfs_status ensure_bottom_up(bfs_graph* g, cudaStream_t st) {
    Layout& L = g->L;
    if (L.bu_ptr.ptr) return BFS_OK;
    const DevBuf& deg = L.deg;
    DevBuf iso;
    const int64_t iso_words = ((L.n + 31) / 32 + 4 + 3) / 4 * 4;        // the search bitmaps' padded size
    BFS_TRY(iso.alloc(sizeof(uint32_t) * iso_words));
    isolated_bits<<<grid_for(iso_words, 256), 256, 0, st>>>(deg.as<uint32_t>(), L.n, iso_words, iso.as<uint32_t>());
    BFS_CUDA_TRY(cudaGetLastError());
    // the bottom-up rows: offsets = scan of the degrees, then the columns
    const int64_t tiles = (L.n + 1 + 1023) / 1024;
    DevBuf ptr, adj, tsum;
    BFS_TRY(ptr.alloc(sizeof(int64_t) * (L.n + 1)));
    BFS_TRY(adj.alloc(sizeof(int32_t) * (L.nnz > 0 ? L.nnz : 1)));
    BFS_TRY(tsum.alloc(sizeof(int64_t) * tiles));
    degree_tile_scan<<<tiles, 1024, 0, st>>>(deg.as<uint32_t>(), L.n, ptr.as<int64_t>(), tsum.as<int64_t>());
    BFS_CUDA_TRY(cudaGetLastError());
    std::vector<int64_t> h(tiles);
    BFS_CUDA_TRY(cudaMemcpyAsync(h.data(), tsum.ptr, sizeof(int64_t) * tiles, cudaMemcpyDeviceToHost, st));
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    int64_t run = 0;
    for (int64_t t = 0; t < tiles; ++t) {
        const int64_t x = h[t];
        h[t] = run;
        run += x;
    }
    if (run != L.nnz)
        return set_error(BFS_ERR_CUDA, "bottom-up rows: degrees sum to %lld, not %lld entries", (long long)run,
                         (long long)L.nnz);
    BFS_CUDA_TRY(cudaMemcpyAsync(tsum.ptr, h.data(), sizeof(int64_t) * tiles, cudaMemcpyHostToDevice, st));
    degree_tile_add<<<grid_for(L.n + 1, 256), 256, 0, st>>>(ptr.as<int64_t>(), L.n, tsum.as<int64_t>());
    BFS_CUDA_TRY(cudaGetLastError());
    bottom_up_rows<<<grid_for(L.n, 256), 256, 0, st>>>(L.dir.as<uint32_t>(), L.rank.as<uint32_t>(), L.dir_stride,
                                                       L.cp.as<uint32_t>(), L.cp_base_d.as<int64_t>(),
                                                       L.ir_base_d.as<int64_t>(), L.ir.as<int32_t>(), L.p, L.nb,
                                                       L.n, ptr.as<int64_t>(), adj.as<int32_t>());
    BFS_CUDA_TRY(cudaGetLastError());
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    std::swap(L.iso.ptr, iso.ptr);
    std::swap(L.iso.bytes, iso.bytes);
    std::swap(L.bu_ptr.ptr, ptr.ptr);
    std::swap(L.bu_ptr.bytes, ptr.bytes);
    std::swap(L.bu_adj.ptr, adj.ptr);
    std::swap(L.bu_adj.bytes, adj.bytes);
    return BFS_OK;
}

// --------------------------------------------------------- entry helpers --
namespace {

bfs_status check_options(const bfs_options* o, int64_t n) {
    if (!o) return BFS_OK;
    if (o->grid_r != o->grid_c) return set_error(BFS_ERR_INVALID_ARG, "grid must be square (grid_r == grid_c)");
    if (o->grid_r < 1 || o->grid_r > 1024 || o->grid_r > n)
        return set_error(BFS_ERR_INVALID_ARG, "grid size %d outside [1, min(n, 1024)]", o->grid_r);
    if (o->mode < 0 || o->mode > 2) return set_error(BFS_ERR_INVALID_ARG, "unknown mode %d", o->mode);
    if (o->wah_word_bits != 32 && o->wah_word_bits != 64)
        return set_error(BFS_ERR_INVALID_ARG, "wah_word_bits must be 32 or 64");
    return BFS_OK;
}

cudaStream_t as_stream(void* s) { return static_cast<cudaStream_t>(s); }

bfs_status create_common(int64_t n, int64_t m, const int32_t* src, const int32_t* dst, int symmetrize,
                         const bfs_options* opt, void* stream, bfs_graph_t* out, bool src_is_device_scratch) {
    bfs_options o;
    bfs_options_default(&o);
    if (opt) o = *opt;
    BFS_TRY(check_options(&o, n));
    cudaStream_t st = as_stream(stream);
    bfs_graph* g = new (std::nothrow) bfs_graph();
    if (!g) return set_error(BFS_ERR_OUT_OF_MEMORY, "host allocation of the graph handle");
    g->L.p = o.grid_r;
    g->mode = o.mode;
    g->wah_bits = o.wah_word_bits;
    g->debug_checks = o.debug_checks ? 1 : 0;
    g->autotune = o.autotune ? 1 : 0;
    g->row_exchange = o.row_exchange ? 1 : 0;
    g->symmetric = symmetrize ? 1 : 0;
    cudaGetDevice(&g->device);

    DevBuf dsrc, ddst;
    const int32_t* s_ptr = src;
    const int32_t* d_ptr = dst;
    bfs_status rc = BFS_OK;
    if (!src_is_device_scratch) {
        if (m > 0 && !is_device_pointer(src)) {
            rc = dsrc.alloc(sizeof(int32_t) * m);
            if (rc == BFS_OK && cudaMemcpyAsync(dsrc.ptr, src, sizeof(int32_t) * m, cudaMemcpyHostToDevice, st) != cudaSuccess)
                rc = set_error(BFS_ERR_CUDA, "copy of src to the device failed");
            s_ptr = dsrc.as<int32_t>();
        }
        if (rc == BFS_OK && m > 0 && !is_device_pointer(dst)) {
            rc = ddst.alloc(sizeof(int32_t) * m);
            if (rc == BFS_OK && cudaMemcpyAsync(ddst.ptr, dst, sizeof(int32_t) * m, cudaMemcpyHostToDevice, st) != cudaSuccess)
                rc = set_error(BFS_ERR_CUDA, "copy of dst to the device failed");
            d_ptr = ddst.as<int32_t>();
        }
    }
    if (rc == BFS_OK) rc = build_layout(g, n, m, s_ptr, d_ptr, symmetrize, st);
    if (rc == BFS_OK) rc = ensure_workspace(g, st);
    if (rc != BFS_OK) {
        cudaStreamSynchronize(st);
        free_workspace(g);
        delete g;
        return rc;
    }
    *out = g;
    return BFS_OK;
}

}  // namespace
}  // namespace bfsgb

using namespace bfsgb;

extern "C" {

void bfs_options_default(bfs_options* opt) {
    if (!opt) return;
    opt->grid_r = 1;
    opt->grid_c = 1;
    opt->mode = BFS_MODE_COMPRESS_SIEVE;
    opt->wah_word_bits = 32;
    opt->autotune = 0;
    opt->debug_checks = 0;
    opt->row_exchange = 1;
}

const char* bfs_status_string(bfs_status s) {
    switch (s) {
        case BFS_OK: return "BFS_OK";
        case BFS_ERR_INVALID_ARG: return "BFS_ERR_INVALID_ARG";
        case BFS_ERR_OUT_OF_MEMORY: return "BFS_ERR_OUT_OF_MEMORY";
        case BFS_ERR_CUDA: return "BFS_ERR_CUDA";
        case BFS_ERR_TIMEOUT: return "BFS_ERR_TIMEOUT";
        case BFS_ERR_CORRUPT: return "BFS_ERR_CORRUPT";
        case BFS_ERR_BUSY: return "BFS_ERR_BUSY";
        case BFS_ERR_NOT_FOUND: return "BFS_ERR_NOT_FOUND";
    }
    return "BFS_ERR_UNKNOWN";
}

bfs_status bfs_debug_codec_ctas(int32_t ctas) {
    if (ctas < 0 || ctas > kCC || (ctas & (ctas - 1)))
        return set_error(BFS_ERR_INVALID_ARG, "codec CTAs %d not 0 or a power of two up to %d", ctas, kCC);
    t_codec_ctas = ctas ? ctas : kCC;
    return BFS_OK;
}

bfs_status bfs_debug_fail_allocation(int64_t k) {
    if (k < 0) return set_error(BFS_ERR_INVALID_ARG, "k must be >= 0");
    g_fail_countdown.store(k);
    return BFS_OK;
}

bfs_status bfs_last_error(char* buf, int64_t len) {
    if (buf && len > 0) {
        strncpy(buf, t_last_msg, (size_t)len - 1);
        buf[len - 1] = '\0';
    }
    return t_last_status;
}

bfs_status bfs_graph_create_edges(int64_t n, int64_t m, const int32_t* src, const int32_t* dst, int32_t symmetrize,
                                  const bfs_options* opt, void* stream, bfs_graph_t* out) {
    if (!out) return set_error(BFS_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (n < 1 || n > 0x7fffffffLL) return set_error(BFS_ERR_INVALID_ARG, "n_vertices %lld outside [1, 2^31-1]", (long long)n);
    if (m < 0 || (m > 0 && (!src || !dst))) return set_error(BFS_ERR_INVALID_ARG, "bad edge arrays");
    if ((symmetrize ? 2 * m : m) > (int64_t)0x7fffffff * 16)
        return set_error(BFS_ERR_INVALID_ARG, "too many entries");
    return create_common(n, m, src, dst, symmetrize ? 1 : 0, opt, stream, out, false);
}

bfs_status bfs_graph_create_csr(int64_t n, const int64_t* row_ptr, const int32_t* col, const bfs_options* opt,
                                void* stream, bfs_graph_t* out) {
    if (!out) return set_error(BFS_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (n < 1 || n > 0x7fffffffLL) return set_error(BFS_ERR_INVALID_ARG, "n_vertices %lld outside [1, 2^31-1]", (long long)n);
    if (!row_ptr) return set_error(BFS_ERR_INVALID_ARG, "row_ptr is NULL");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool rp_dev = is_device_pointer(row_ptr);
    int64_t first = 0, nnz = 0;
    BFS_CUDA_TRY(cudaMemcpyAsync(&first, row_ptr, sizeof(int64_t), rp_dev ? cudaMemcpyDeviceToHost : cudaMemcpyHostToHost, st));
    BFS_CUDA_TRY(cudaMemcpyAsync(&nnz, row_ptr + n, sizeof(int64_t), rp_dev ? cudaMemcpyDeviceToHost : cudaMemcpyHostToHost, st));
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    if (first != 0 || nnz < 0) return set_error(BFS_ERR_INVALID_ARG, "row_ptr[0] must be 0 and row_ptr[n] >= 0");
    if (nnz > 0 && !col) return set_error(BFS_ERR_INVALID_ARG, "col is NULL");
    DevBuf drp, dcol, dsrc, err;
    const int64_t* rp = row_ptr;
    const int32_t* cl = col;
    if (!rp_dev) {
        BFS_TRY(drp.alloc(sizeof(int64_t) * (n + 1)));
        BFS_CUDA_TRY(cudaMemcpyAsync(drp.ptr, row_ptr, sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, st));
        rp = drp.as<int64_t>();
    }
    if (nnz > 0 && !is_device_pointer(col)) {
        BFS_TRY(dcol.alloc(sizeof(int32_t) * nnz));
        BFS_CUDA_TRY(cudaMemcpyAsync(dcol.ptr, col, sizeof(int32_t) * nnz, cudaMemcpyHostToDevice, st));
        cl = dcol.as<int32_t>();
    }
    BFS_TRY(err.alloc(sizeof(unsigned long long)));
    BFS_CUDA_TRY(cudaMemsetAsync(err.ptr, 0, err.bytes, st));
    check_csr<<<grid_for(n > nnz ? n : nnz, 256), 256, 0, st>>>(rp, cl, n, nnz, err.as<unsigned long long>());
    BFS_CUDA_TRY(cudaGetLastError());
    unsigned long long h_err = 0;
    BFS_CUDA_TRY(cudaMemcpyAsync(&h_err, err.ptr, sizeof(h_err), cudaMemcpyDeviceToHost, st));
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    if (h_err) return set_error(BFS_ERR_INVALID_ARG, "row_ptr is not nondecreasing or col names a vertex outside [0, n)");
    BFS_TRY(dsrc.alloc(sizeof(int32_t) * (nnz > 0 ? nnz : 1)));
    expand_rows<<<grid_for(n, 256), 256, 0, st>>>(rp, n, dsrc.as<int32_t>());
    BFS_CUDA_TRY(cudaGetLastError());
    return create_common(n, nnz, dsrc.as<int32_t>(), cl, 0, opt, stream, out, true);
}

bfs_status bfs_graph_destroy(bfs_graph_t g) {
    if (!g) return BFS_OK;
    if (g->busy.load()) return set_error(BFS_ERR_BUSY, "graph is in use");
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(g->device);
    cudaDeviceSynchronize();
    free_msbfs(g);
    free_workspace(g);
    delete g;
    cudaSetDevice(cur);
    return BFS_OK;
}

bfs_status bfs_graph_footprint(bfs_graph_t g, int64_t* bytes) {
    if (!g || !bytes) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    const Layout& L = g->L;
    const Workspace& W = g->W;
    int64_t b = (int64_t)(L.dir.bytes + L.rank.bytes + L.cp.bytes + L.ir.bytes + L.cp_base_d.bytes + L.ir_base_d.bytes +
                          L.deg.bytes + L.iso.bytes + L.bu_ptr.bytes + L.bu_adj.bytes);
    b += (int64_t)(W.pi.bytes + W.fa.bytes + W.fb.bytes + W.fsum.bytes + W.fwords.bytes + W.xbuf.bytes + W.xcount.bytes +
                   W.chunk_base.bytes + W.units.bytes + W.counters.bytes + W.tmp_parent.bytes + W.tmp_level.bytes +
                   W.pieces.bytes + W.level_scratch.bytes + W.row_meta.bytes + W.tblk.bytes + W.rowbuf.bytes +
                   W.rowcount.bytes + W.rowfirst.bytes + W.rowlive.bytes + W.xfmt.bytes + W.enc_sums.bytes + W.enc_bases.bytes + W.enc_flags.bytes +
                   W.enc_done.bytes + W.gbits.bytes + W.colfirst.bytes + W.ddir.bytes);
    *bytes = b;
    return BFS_OK;
}

bfs_status bfs_graph_info(bfs_graph_t g, bfs_graph_info_t* info) {
    if (!g || !info) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    memset(info, 0, sizeof(*info));
    info->n_vertices = g->L.n;
    info->n_entries = g->L.nnz;
    info->p = g->L.p;
    info->mode = g->mode;
    info->wah_word_bits = g->wah_bits;
    info->range_size = g->L.nb;
    info->row_exchange = g->row_exchange;
    info->exchange_format = g->adaptive ? BFS_FORMAT_ADAPTIVE : BFS_FORMAT_WAH;
    info->direction = g->direction;
    info->dynamic_directory = g->dynamic_dir;
    info->nonempty_columns = g->L.nnzc_total;
    return BFS_OK;
}

bfs_status bfs_graph_set_mode(bfs_graph_t g, int32_t mode, int32_t wah_word_bits) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (mode < 0 || mode > 2) return set_error(BFS_ERR_INVALID_ARG, "unknown mode %d", mode);
    if (wah_word_bits != 32 && wah_word_bits != 64) return set_error(BFS_ERR_INVALID_ARG, "wah_word_bits must be 32 or 64");
    if (g->busy.load()) return set_error(BFS_ERR_BUSY, "graph is in use");
    std::lock_guard<std::mutex> lk(g->mu);
    g->mode = mode;
    g->wah_bits = wah_word_bits;
    return BFS_OK;
}

bfs_status bfs_graph_set_row_exchange(bfs_graph_t g, int32_t enabled) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (g->busy.load()) return set_error(BFS_ERR_BUSY, "graph is in use");
    std::lock_guard<std::mutex> lk(g->mu);
    g->row_exchange = enabled ? 1 : 0;
    return BFS_OK;
}

bfs_status bfs_graph_set_exchange_format(bfs_graph_t g, int32_t format) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (format != BFS_FORMAT_WAH && format != BFS_FORMAT_ADAPTIVE)
        return set_error(BFS_ERR_INVALID_ARG, "unknown exchange format %d", format);
    if (g->busy.load()) return set_error(BFS_ERR_BUSY, "graph is in use");
    std::lock_guard<std::mutex> lk(g->mu);
    g->adaptive = format == BFS_FORMAT_ADAPTIVE ? 1 : 0;
    return BFS_OK;
}

bfs_status bfs_graph_set_dynamic_directory(bfs_graph_t g, int32_t enabled) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (enabled != 0 && enabled != 1) return set_error(BFS_ERR_INVALID_ARG, "enabled must be 0 or 1");
    if (g->busy.load()) return set_error(BFS_ERR_BUSY, "graph is in use");
    std::lock_guard<std::mutex> lk(g->mu);
    g->dynamic_dir = enabled;
    return BFS_OK;
}

bfs_status bfs_graph_set_direction(bfs_graph_t g, int32_t policy, int32_t alpha, int32_t beta) {
    if (!g) return set_error(BFS_ERR_INVALID_ARG, "graph is NULL");
    if (policy < BFS_DIRECTION_TOP_DOWN || policy > BFS_DIRECTION_BOTTOM_UP)
        return set_error(BFS_ERR_INVALID_ARG, "unknown direction policy %d", policy);
    if (alpha < 1 || alpha > 1000000 || beta < 1 || beta > 1000000)
        return set_error(BFS_ERR_INVALID_ARG, "alpha and beta must lie in [1, 1000000]");
    if (policy != BFS_DIRECTION_TOP_DOWN && !g->symmetric)
        return set_error(BFS_ERR_INVALID_ARG, "bottom-up levels need an undirected graph (created with symmetrize = 1)");
    if (g->busy.load()) return set_error(BFS_ERR_BUSY, "graph is in use");
    std::lock_guard<std::mutex> lk(g->mu);
    if (policy != BFS_DIRECTION_TOP_DOWN) {
        int cur = 0;
        cudaGetDevice(&cur);
        cudaSetDevice(g->device);
        const bfs_status rc = ensure_bottom_up(g, nullptr);
        cudaSetDevice(cur);
        BFS_TRY(rc);
    }
    g->direction = policy;
    g->alpha = alpha;
    g->beta = beta;
    return BFS_OK;
}

bfs_status bfs_graph_directory(bfs_graph_t g, int32_t i, int32_t j, uint32_t* out_words, void* stream) {
    if (!g || !out_words) return set_error(BFS_ERR_INVALID_ARG, "NULL argument");
    const int p = g->L.p;
    if (i < 0 || i >= p || j < 0 || j >= p) return set_error(BFS_ERR_INVALID_ARG, "block (%d,%d) outside the %dx%d grid", i, j, p, p);
    const int64_t words = (g->L.range_len(j) + 31) / 32;
    if (words == 0) return BFS_OK;
    const uint32_t* src = g->L.dir.as<uint32_t>() + ((int64_t)i * p + j) * g->L.dir_stride;
    BFS_CUDA_TRY(cudaMemcpyAsync(out_words, src, sizeof(uint32_t) * words, cudaMemcpyDeviceToDevice,
                                 static_cast<cudaStream_t>(stream)));
    return BFS_OK;
}

}  // extern "C"
