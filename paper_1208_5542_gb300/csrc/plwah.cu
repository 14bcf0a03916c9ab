// plwah.cu -- position-list word-aligned hybrid (PLWAH) code of one bitmap:
// the alternative bitmap code Sec. IV names beside WAH (Deliege and
// Pedersen).  32-bit words over 31-bit groups, as the 32-bit WAH code; a fill
// word keeps 25 bits of run length and uses bits 29..25 for the position
// (1 = first bit of the group, 0 = none) of the one odd bit of the group right
// after its run, which is then not written.
//
// PLWAH of a bitmap is its WAH stream with every literal that follows a fill
// word and differs from the fill value in one bit folded into that fill word
// (runs stay below 2^25 groups under the size limit of the entry points), so
// both directions are word-parallel transcodings around the WAH kernels: one
// cluster walks the stream in rounds, a scan places the output words.
#include <cstring>

#include "cluster.cuh"
#include "common.cuh"
#include "internal.h"

namespace bfsgb {
namespace {

constexpr uint32_t kTop = 0x80000000u, kVal = 0x40000000u, kOnes = 0x7fffffffu;
constexpr uint32_t kCount25 = (1u << 25) - 1u;
constexpr int64_t kPlwahMaxBits = 31LL * ((1LL << 25) - 1);   // every run below 2^25 groups

// The odd bit of a literal against fill value v: its place (1..31), or 0 if
// the literal differs from the fill pattern in more or fewer than one bit.
__device__ __forceinline__ uint32_t odd_place(uint32_t lit, uint32_t v) {
    const uint32_t diff = lit ^ (v ? kOnes : 0u);
    return (diff && !(diff & (diff - 1u))) ? (uint32_t)__clz(diff) : 0u;   // bit 30 (first) -> 1
}

// WAH (32-bit words, runs < 2^25 groups) -> PLWAH.  A literal word k is
// folded when word k-1 is a fill and the literal is one bit off its value;
// the active word (the last word when nbits mod 31 != 0) is copied.
__global__ void __launch_bounds__(kCT) plwah_from_wah(const uint32_t* __restrict__ wah, const int64_t* __restrict__ nw_p,
                                                      int64_t nbits, uint32_t* __restrict__ out,
                                                      int64_t* __restrict__ out_count) {
    __shared__ ClusterScan<int64_t> s_scan;
    const int64_t nw = *nw_p;
    const int64_t body = nw - ((nbits % 31) != 0 ? 1 : 0);           // words before the active word
    auto is_fill = [&](uint32_t w) { return (w & kTop) != 0u; };
    int64_t carry = 0;
    int turn = 0;
    const int64_t round = cluster_round();
    for (int64_t base = 0; base < nw; base += round, ++turn) {
        const int64_t k0 = base + cluster_thread() * kCK;
        uint32_t word[kCK], emit = 0;
        uint32_t before = (k0 > 0 && k0 <= body) ? wah[k0 - 1] : 0u;   // no fill before the first word
        uint32_t w = k0 < nw ? wah[k0] : 0u;
#pragma unroll
        for (int i = 0; i < kCK; ++i) {
            const int64_t k = k0 + i;
            const uint32_t next = k + 1 < nw ? wah[k + 1] : 0u;
            word[i] = w;
            if (k < body) {
                const bool folded = !is_fill(w) && is_fill(before) && odd_place(w, before & kVal) != 0u;
                if (!folded) emit |= 1u << i;
                if (is_fill(w)) {
                    const uint32_t q = (k + 1 < body && !is_fill(next)) ? odd_place(next, w & kVal) : 0u;
                    word[i] = kTop | (w & kVal) | (q << 25) | (w & kCount25);
                }
            } else if (k < nw) {
                emit |= 1u << i;                                       // the active word
            }
            before = w;
            w = next;
        }
        int64_t total;
        int64_t pos = carry + cluster_excl_scan((int64_t)__popc(emit), (int64_t)0, OpSum(), s_scan, turn, &total);
#pragma unroll
        for (int i = 0; i < kCK; ++i)
            if ((emit >> i) & 1u) out[pos++] = word[i];
        carry += total;
    }
    if (cluster_thread() == 0) *out_count = carry;
    cluster_done();
}

// PLWAH -> WAH: a fill word with a position becomes the fill and the literal
// it stands for.  A fill of length 0 is flagged (the WAH decoder checks the
// rest of the structure).
__global__ void __launch_bounds__(kCT) wah_from_plwah(const uint32_t* __restrict__ pl, int64_t nw, int64_t nbits,
                                                      uint32_t* __restrict__ out, volatile unsigned long long* out_count,
                                                      volatile unsigned long long* err) {
    __shared__ ClusterScan<int64_t> s_scan;
    const int64_t body = nw - ((nbits % 31) != 0 ? 1 : 0);
    int64_t carry = 0;
    bool bad = false;
    int turn = 0;
    const int64_t round = cluster_round();
    for (int64_t base = 0; base < nw; base += round, ++turn) {
        const int64_t k0 = base + cluster_thread() * kCK;
        uint32_t w[kCK], c = 0;
#pragma unroll
        for (int i = 0; i < kCK; ++i) {
            const int64_t k = k0 + i;
            w[i] = k < nw ? pl[k] : 0u;
            if (k < nw) ++c;
            if (k < body && (w[i] & kTop)) {
                if ((w[i] & kCount25) == 0u) bad = true;
                if ((w[i] >> 25) & 31u) ++c;
            }
        }
        int64_t total;
        int64_t pos = carry + cluster_excl_scan((int64_t)c, (int64_t)0, OpSum(), s_scan, turn, &total);
#pragma unroll
        for (int i = 0; i < kCK; ++i) {
            const int64_t k = k0 + i;
            if (k >= nw) break;
            if (k < body && (w[i] & kTop)) {
                const uint32_t q = (w[i] >> 25) & 31u;
                out[pos++] = kTop | (w[i] & kVal) | (w[i] & kCount25);
                if (q) out[pos++] = ((w[i] & kVal) ? kOnes : 0u) ^ (1u << (31 - q));
            } else {
                out[pos++] = w[i];
            }
        }
        carry += total;
    }
    if (cluster_thread() == 0) *out_count = (unsigned long long)carry;
    if (bad) *err = 1ull;
    cluster_done();
}

}  // namespace
}  // namespace bfsgb

using namespace bfsgb;

extern "C" {

bfs_status bfs_plwah_encode(const uint32_t* bits, int64_t nbits, uint32_t* words, int64_t capacity_words,
                            int64_t* nwords, void* stream) {
    if (nbits < 0 || nbits > kPlwahMaxBits)
        return set_error(BFS_ERR_INVALID_ARG, "nbits %lld outside [0, %lld]", (long long)nbits, (long long)kPlwahMaxBits);
    if (!nwords || (nbits > 0 && (!bits || !words))) return set_error(BFS_ERR_INVALID_ARG, "bad encode arguments");
    const int64_t bound = nbits / 31 + 1;
    if (capacity_words < bound)
        return set_error(BFS_ERR_INVALID_ARG, "capacity %lld below the bound %lld", (long long)capacity_words,
                         (long long)bound);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (nbits == 0) {
        BFS_CUDA_TRY(cudaMemsetAsync(nwords, 0, sizeof(int64_t), st));
        return BFS_OK;
    }
    // one scratch block: the count, then the WAH words
    Scratch tmp;
    BFS_TRY(tmp.alloc(sizeof(int64_t) + sizeof(uint32_t) * (size_t)(bound + 1), st));
    int64_t* cnt = tmp.as<int64_t>();
    uint32_t* wah = reinterpret_cast<uint32_t*>(cnt + 1);
    BFS_TRY(launch_wah_encode(bits, nbits, 32, wah, cnt, st));
    BFS_CUDA_TRY(launch_cluster<plwah_from_wah>(st, wah, cnt, nbits, words, nwords));
    BFS_CUDA_TRY(cudaStreamSynchronize(st));
    return BFS_OK;
}

bfs_status bfs_plwah_decode(const uint32_t* words, int64_t nwords, int64_t nbits, uint32_t* bits, void* stream) {
    if (nbits < 0 || nbits > kPlwahMaxBits)
        return set_error(BFS_ERR_INVALID_ARG, "nbits %lld outside [0, %lld]", (long long)nbits, (long long)kPlwahMaxBits);
    if (nwords < 0 || (nwords > 0 && !words) || (nbits > 0 && !bits))
        return set_error(BFS_ERR_INVALID_ARG, "bad decode arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    Scratch wah;
    BFS_TRY(wah.alloc(sizeof(uint32_t) * (size_t)(2 * nwords + 1), st));
    int64_t h_cnt = 0;
    if (nwords > 0) {
        HostFlag said;                                // error, count; given back before the WAH decode takes its own
        BFS_TRY(said.take(st));
        BFS_CUDA_TRY(launch_cluster<wah_from_plwah>(st, words, nwords, nbits, wah.as<uint32_t>(),
                                    said.device(1), said.device(0)));
        BFS_TRY(said.wait());
        h_cnt = (int64_t)said.value(1);
        if (said.value(0)) return set_error(BFS_ERR_CORRUPT, "malformed PLWAH stream (a fill of length 0)");
    }
    const bfs_status rc = bfs_wah_decode(wah.ptr, h_cnt, nbits, 32, bits, stream);
    if (rc == BFS_ERR_CORRUPT) return set_error(BFS_ERR_CORRUPT, "malformed PLWAH stream");
    return rc;
}

}  // extern "C"
