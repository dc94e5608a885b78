// Cut evaluation that allocates no device memory (bipart_cut_noalloc in include/bipart.h).
//
// Who needs it: callers that cannot call cudaMalloc at the point where they want a cut -- for
// example a host application that hands all of HBM to its own memory pool up front, so any
// allocation by a library fails or breaks the pool's accounting, or a latency-critical loop that
// cannot afford the device-wide synchronisation an allocation may imply.  They pass the
// hypergraph, the partition and the output slot in device memory they already own; the only
// scratch is the fixed-size array below, which is part of this library's device image.
//
// Scratch: g_cut_scratch holds, per call, a small header (completion counter, error flag, list length),
// the per-block partial sums and the list of the hyperedges that take a block each.  It is sized
// for at most kCutNoAllocMaxHedges hyperedges (16 MiB plus 15 KiB on every GPU that loads the
// library, held until the process exits).  Every call uses the same array: calls that overlap
// on the GPU (different streams, or different host threads on the same device) race on it and
// must be serialised by the caller.
//
// What bounds it: chains of a pin load and a part gather per hyperedge.  One thread a hyperedge of up to
// 32 pins keeps four chains in flight; up to 512 pins take a warp with four loads a lane, larger ones a
// block of 512 threads with eight (a warp walking 10,000 pins one load at a time was the whole run).
// lambda goes straight into the partial sums.  1M-node netlist, 8.3M pins, k = 8: 60 us, 175 us with a warp per large hyperedge.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"

namespace bp {
namespace {

constexpr int kCutNoAllocMaxHedges = 1 << 22;  // 4,194,304 hyperedges
constexpr int kCutNoAllocMaxParts = 64;
constexpr int kNaBlock = 256;
constexpr int kNaBigBlock = 512;
constexpr int kNaMaxBlocks = 1216;       // 8 blocks of 256 threads on each of 152 SMs
constexpr int kNaBigBlocks = 608;
constexpr int kNaThreadDeg = 32, kNaWarpDeg = 512;
// layout in 8-byte words: [0] counter, [1] error flag, [2] list length, [64 .. 64+kNaPartials) partials of
// both kernels, then kCutNoAllocMaxHedges int32 list entries
constexpr int kNaPartials = kNaMaxBlocks + kNaBigBlocks;
constexpr size_t kNaHeaderWords = 64;
constexpr size_t kNaWords = kNaHeaderWords + kNaPartials + kCutNoAllocMaxHedges / 2;

static __device__ __align__(256) unsigned long long g_cut_scratch[kNaWords];

constexpr int kMaxDevices = 64;
std::mutex g_na_mu;
unsigned long long *g_na_ptr[kMaxDevices] = {};

__device__ __forceinline__ int *na_list(unsigned long long *scratch) {
    return reinterpret_cast<int *>(scratch + kNaHeaderWords + kNaPartials);
}

// Part mask of the pins a + t, a + t + nt, ... below b, kU of them in flight; a pin outside [0, N) or a
// part outside [0, k) sets `bad` instead of being used.
template <int kU>
__device__ __forceinline__ unsigned long long na_mask(const int *__restrict__ pins, const int *__restrict__ parts,
                                                      int N, int k, int a, int b, int t, int nt, bool &bad) {
    unsigned long long m = 0;
    for (int64_t i0 = (int64_t)a + t; i0 < b; i0 += (int64_t)kU * nt) {
        int v[kU], p[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) v[u] = i0 + (int64_t)u * nt < b ? __ldg(pins + i0 + (int64_t)u * nt) : -2;
#pragma unroll
        for (int u = 0; u < kU; ++u) p[u] = v[u] >= 0 && v[u] < N ? __ldg(parts + v[u]) : -1;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (v[u] == -2 && i0 + (int64_t)u * nt >= b) continue;  // past the end
            if (p[u] < 0 || p[u] >= k) bad = true;
            else m |= 1ull << p[u];
        }
    }
    return m;
}

__device__ __forceinline__ unsigned long long warp_or(unsigned long long m) {
    return (unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)(m >> 32)) << 32 |
           __reduce_or_sync(0xffffffffu, (unsigned)m);
}

__device__ __forceinline__ unsigned long long na_cost(unsigned long long m, int w) {
    const int l = __popcll(m);
    return l > 1 ? (unsigned long long)w * (unsigned long long)(l - 1) : 0ull;
}

// Hyperedges of up to kNaWarpDeg pins: w_e (lambda_e - 1) summed per block, lambda_e = number of distinct
// parts among the pins of e; larger ones are listed for k_na_big.  A weight below 1 raises the error flag.
__global__ void __launch_bounds__(kNaBlock)
k_na_small(int N, int E, const int *__restrict__ hoff, const int *__restrict__ pins,
           const int *__restrict__ hw, const int *__restrict__ parts, int k,
           unsigned long long *__restrict__ scratch) {
    __shared__ unsigned long long red[33];
    const int lane = threadIdx.x & 31;
    const int warps = gridDim.x * (blockDim.x >> 5);
    bool bad = false;
    unsigned long long sum = 0;
    for (int e0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; e0 < E; e0 += warps * 32) {
        const int e = e0 + lane;
        int a = 0, d = 0, w = 1;
        if (e < E) {
            a = __ldg(hoff + e);
            d = __ldg(hoff + e + 1) - a;
            if (hw) w = __ldg(hw + e);
            if (w < 1) bad = true;
        }
        if (d <= kNaThreadDeg) sum += na_cost(na_mask<4>(pins, parts, N, k, a, a + d, 0, 1, bad), w);
        if (d > kNaWarpDeg) na_list(scratch)[atomicAdd(reinterpret_cast<unsigned *>(scratch + 2), 1u)] = e;
        unsigned mid = __ballot_sync(0xffffffffu, d > kNaThreadDeg && d <= kNaWarpDeg);
        while (mid) {
            const int src = __ffs(mid) - 1;
            mid &= mid - 1;
            const int ab = __shfl_sync(0xffffffffu, a, src), db = __shfl_sync(0xffffffffu, d, src);
            const unsigned long long m = warp_or(na_mask<4>(pins, parts, N, k, ab, ab + db, lane, 32, bad));
            if (lane == src) sum += na_cost(m, w);
        }
    }
    if (bad) atomicOr(&scratch[1], 1ull);
    sum = block_sum(sum, red);
    if (threadIdx.x == 0) scratch[kNaHeaderWords + blockIdx.x] = sum;
}

// The listed hyperedges, a block each; then the last block to finish adds all partial sums and writes the
// caller's output (-1 when a pin, a part or a weight was out of range).
__global__ void __launch_bounds__(kNaBigBlock)
k_na_big(int N, int small_blocks, const int *__restrict__ hoff, const int *__restrict__ pins,
         const int *__restrict__ hw, const int *__restrict__ parts, int k,
         unsigned long long *__restrict__ scratch, long long *__restrict__ out) {
    __shared__ unsigned long long red[33];
    __shared__ unsigned long long s_mask;
    __shared__ bool last;
    unsigned long long *partials = scratch + kNaHeaderWords;
    const int n = (int)*reinterpret_cast<const unsigned *>(scratch + 2);
    bool bad = false;
    unsigned long long sum = 0;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        const int e = na_list(scratch)[i];
        const int a = __ldg(hoff + e), b = __ldg(hoff + e + 1);
        if (threadIdx.x == 0) s_mask = 0;
        __syncthreads();
        const unsigned long long m = warp_or(na_mask<8>(pins, parts, N, k, a, b, (int)threadIdx.x, kNaBigBlock, bad));
        if ((threadIdx.x & 31) == 0 && m) atomicOr(&s_mask, m);
        __syncthreads();
        if (threadIdx.x == 0) sum += na_cost(s_mask, hw ? __ldg(hw + e) : 1);
    }
    if (bad) atomicOr(&scratch[1], 1ull);
    __syncthreads();
    if (threadIdx.x == 0) {
        partials[kNaMaxBlocks + blockIdx.x] = sum;
        __threadfence();
        last = atomicAdd(&scratch[0], 1ull) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    unsigned long long t = 0;
    for (int b = threadIdx.x; b < small_blocks; b += blockDim.x) t += __ldcg(partials + b);
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) t += __ldcg(partials + kNaMaxBlocks + b);
    t = block_sum(t, red);
    if (threadIdx.x == 0) *out = __ldcg(scratch + 1) != 0 ? -1ll : (long long)t;
}

}  // namespace
}  // namespace bp

using namespace bp;

// The first call on a device looks up the scratch array's device address with that device
// current (cudaGetSymbolAddress); later calls on the device reuse it.  Make that first call
// before any stream capture begins.
extern "C" int bipart_cut_noalloc(int32_t num_nodes, int32_t num_hedges,
                                  const int32_t *d_hedge_offsets, const int32_t *d_hedge_pins,
                                  const int32_t *d_hedge_weights, const int32_t *d_parts,
                                  int32_t k, int64_t *d_cut, void *stream) {
    if (num_nodes < 0 || num_hedges < 0) {
        set_error("bipart_cut_noalloc: negative size");
        return BIPART_ERR_INVALID_ARG;
    }
    if (num_hedges > kCutNoAllocMaxHedges) {
        set_error("bipart_cut_noalloc: " + std::to_string(num_hedges) +
                  " hyperedges exceed the fixed scratch limit of " +
                  std::to_string(kCutNoAllocMaxHedges));
        return BIPART_ERR_INVALID_ARG;
    }
    if (k < 1 || k > kCutNoAllocMaxParts) {
        set_error("bipart_cut_noalloc: k must be in [1, 64]");
        return BIPART_ERR_INVALID_ARG;
    }
    if (!d_cut || (num_hedges > 0 && (!d_hedge_offsets || !d_hedge_pins || !d_parts))) {
        set_error("bipart_cut_noalloc: NULL argument");
        return BIPART_ERR_INVALID_ARG;
    }
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        set_error(std::string("bipart_cut_noalloc: no usable device: ") + cudaGetErrorString(err));
        return BIPART_ERR_CUDA;
    }
    unsigned long long *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_na_mu);
        if (!g_na_ptr[dev]) {
            void *p = nullptr;
            err = cudaGetSymbolAddress(&p, g_cut_scratch);
            if (err != cudaSuccess || !p) {
                set_error(std::string("bipart_cut_noalloc: cudaGetSymbolAddress failed: ") +
                          cudaGetErrorString(err));
                return BIPART_ERR_CUDA;
            }
            g_na_ptr[dev] = static_cast<unsigned long long *>(p);
        }
        scratch = g_na_ptr[dev];
    }
    cudaStream_t s = (cudaStream_t)stream;
    // counter, error flag and list length start at zero; the rest is written before it is read
    err = cudaMemsetAsync(scratch, 0, 3 * sizeof(unsigned long long), s);
    if (err != cudaSuccess) {
        set_error(std::string("bipart_cut_noalloc: ") + cudaGetErrorString(err));
        return BIPART_ERR_CUDA;
    }
    const int small = std::min((num_hedges + kNaBlock - 1) / kNaBlock, kNaMaxBlocks);
    if (num_hedges > 0) {
        k_na_small<<<small, kNaBlock, 0, s>>>(num_nodes, num_hedges, d_hedge_offsets, d_hedge_pins,
                                              d_hedge_weights, d_parts, k, scratch);
        note_launch();
    }
    // few of the hyperedges are listed as a rule; 608 blocks cost a small call more than it takes (1,322
    // hyperedges: 14.8 us with them)
    const int big = std::max(1, std::min((num_hedges + 63) / 64, kNaBigBlocks));
    k_na_big<<<big, kNaBigBlock, 0, s>>>(num_nodes, small, d_hedge_offsets, d_hedge_pins, d_hedge_weights,
                                         d_parts, k, scratch, reinterpret_cast<long long *>(d_cut));
    note_launch();
    err = cudaGetLastError();
    if (err != cudaSuccess) {
        set_error(std::string("bipart_cut_noalloc: launch failed: ") + cudaGetErrorString(err));
        return BIPART_ERR_CUDA;
    }
    return BIPART_OK;
}
