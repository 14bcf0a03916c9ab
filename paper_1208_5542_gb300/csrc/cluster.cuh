// cluster.cuh -- scans over one thread-block cluster, for the codecs that turn
// one bitmap or stream into another.
//
// A codec call is one sequential run of words; what bounds it is the scan that
// places them, not bytes or arithmetic.  One CTA per call (256 threads, a
// scan per 1024 groups) took 0.3-0.5 ms for a 4M-bit slice on one of 152 SMs.
// A cluster of 16 CTAs scans 131,072 elements per round through distributed
// shared memory with one hardware barrier, needs no scratch in device memory
// (a call can be captured, and calls on several streams share nothing), and
// is scheduled as a whole.  An encode and a decode of such a slice through the
// API, host work and synchronisation included: 1.02 -> 0.13 ms.  16 CTAs are
// more than the portable 8, and a partition of the device may not have their
// SMs side by side: a kernel takes the largest size that the device can place,
// down to one CTA, which runs anywhere (the round shrinks with it).
#pragma once

#include <atomic>
#include <cooperative_groups.h>
#include <cstdint>

#include "common.cuh"

namespace bfsgb {

constexpr int kCC = 16;             // the most CTAs of a codec cluster (non-portable size: see launch_cluster)
constexpr int kCT = 1024;           // threads per CTA
constexpr int kCK = 8;              // elements per thread and round
constexpr int kCDevices = 64;       // devices whose cluster size is remembered

// Elements per round of the running cluster.
__device__ __forceinline__ int64_t cluster_round() {
    return (int64_t)cooperative_groups::this_cluster().num_blocks() * kCT * kCK;
}

// Shared memory of a cluster scan; the two slots of `part` alternate, so that
// one cluster barrier per scan is enough (a slot is written again only after
// the next barrier, which every reader has passed).
template <typename T>
struct ClusterScan {
    T warp[kCT / 32 + 1];
    T part[2];
    T before, all;
};

// Exclusive scan of one value per thread over the cluster's threads in rank
// order with an associative op and its identity; *total gets the reduction of
// all.  Contains CTA and cluster barriers: every thread of the cluster calls
// it, `turn` counting the calls on this scratch.
template <typename T, typename Op>
__device__ __forceinline__ T cluster_excl_scan(T x, T identity, Op op, ClusterScan<T>& s, int turn, T* total) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    T cta;
    const T excl = block_excl_scan<kCT>(x, identity, op, s.warp, &cta);
    if (threadIdx.x == 0) s.part[turn & 1] = cta;
    cl.sync();
    if (threadIdx.x < 32) {
        const int l = (int)threadIdx.x;
        const T v = l < (int)cl.num_blocks() ? *cl.map_shared_rank(&s.part[turn & 1], l) : identity;
        T incl = v;
#pragma unroll
        for (int d = 1; d < kCC; d <<= 1) {
            const T y = __shfl_up_sync(0xffffffffu, incl, d);
            if (l >= d) incl = op(y, incl);
        }
        T ex = __shfl_up_sync(0xffffffffu, incl, 1);
        if (l == 0) ex = identity;
        if (l == (int)cl.block_rank()) s.before = ex;
        if (l == kCC - 1) s.all = incl;
    }
    __syncthreads();
    *total = s.all;
    return op(s.before, excl);
}

// Keeps every CTA's shared memory alive until its peers have read it; the last
// thing a cluster kernel does.
__device__ __forceinline__ void cluster_done() { cooperative_groups::this_cluster().sync(); }

__device__ __forceinline__ int64_t cluster_thread() {
    return (int64_t)cooperative_groups::this_cluster().block_rank() * kCT + threadIdx.x;
}

// The calling thread's cap on the CTAs of a codec cluster (bfs_debug_codec_ctas;
// kCC unless a test lowered it).
int codec_ctas_cap();

struct ClusterConfig {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    ClusterConfig(int ctas, cudaStream_t st) {
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(kCT);
        cfg.stream = st;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = ctas;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};

// The largest power of two of CTAs, at most kCC, of which the current device
// can place a cluster of this kernel (asked once per kernel and device).
// More than 8 need the kernel's consent.
template <typename... P>
cudaError_t cluster_ctas(void (*kernel)(P...), std::atomic<int>* known, int* ctas) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < kCDevices && (*ctas = known[dev].load()) > 0) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) cudaGetLastError();            // the portable sizes are left
    for (*ctas = kCC; *ctas > 1; *ctas /= 2) {
        int fit = 0;
        ClusterConfig c(*ctas, nullptr);
        if (cudaOccupancyMaxActiveClusters(&fit, kernel, &c.cfg) == cudaSuccess && fit > 0) break;
        cudaGetLastError();
    }
    if (dev < kCDevices) known[dev].store(*ctas);
    return cudaSuccess;
}

template <typename... P, typename... A>
cudaError_t launch_sized(void (*kernel)(P...), int ctas, cudaStream_t st, A... args) {
    ClusterConfig c(ctas, st);
    return cudaLaunchKernelEx(&c.cfg, kernel, static_cast<P>(args)...);
}

// Launch one cluster.
template <auto Kernel, typename... A>
cudaError_t launch_cluster(cudaStream_t st, A... args) {
    static std::atomic<int> known[kCDevices];
    int ctas = 1;
    const cudaError_t e = cluster_ctas(Kernel, known, &ctas);
    if (e != cudaSuccess) return e;
    const int cap = codec_ctas_cap();
    return launch_sized(Kernel, ctas < cap ? ctas : cap, st, args...);
}

}  // namespace bfsgb
