// Pieces shared by the FP32 passes (fft.cu), the fixed-point passes (fft_fix.cu) and the residue products (rns.cu).
#pragma once

#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

#include "rsdft_internal.h"

namespace rsdft {

// x / d for x < 2^16 from the multiply-high divisor of d (mag = 0 means d = 1).
__device__ __forceinline__ int qdiv(int x, unsigned mag) { return mag ? (int)__umulhi((unsigned)x, mag) : x; }

// xy planes live in shared memory with an odd row stride RS = Nx | 1 (complex
// values): the lines of both transform directions are then read by consecutive
// threads without bank conflicts (successive rows start two banks apart).
__device__ __forceinline__ int plane_rs(int Nx) { return Nx | 1; }
// shared-memory index of plane element i = y Nx + x
__device__ __forceinline__ int pidx(int i, int Nx, int RS, unsigned nxmag) { return i + qdiv(i, nxmag) * (RS - Nx); }

// Global -> shared copy of a plane or slab with several loads in flight per thread:
// each batch issues its loads (src(i)) before any of its stores (dst(i, v)); the
// plain loop would leave one load per thread in flight, and the passes stalled on
// load latency well below the HBM rate.
template <typename V, typename SrcF, typename DstF>
__device__ __forceinline__ void stage_in(int tot, SrcF src, DstF dst) {
    constexpr int U = sizeof(V) == 8 ? 8 : 4;
    for (int i0 = threadIdx.x; i0 < tot; i0 += U * blockDim.x) {
        V r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i < tot) r[u] = src(i);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i < tot) dst(i, r[u]);
        }
    }
}

constexpr size_t MAX_DYN_SMEM = 227 * 1024;   // largest dynamic shared memory of one CTA

// The attribute belongs to a function on a device, for the whole process, so it is raised once for each to the
// largest size, `most` (occupancy follows each launch's own dynamic size); lowering it
// per launch would race with launches of other contexts on other threads.
template <typename K> static rsdft_status set_smem(rsdft_ctx *ctx, K kernel, size_t bytes, size_t most = MAX_DYN_SMEM) {
    if (bytes <= 48 * 1024) return RSDFT_OK;
    if (bytes > most) return fail(ctx, RSDFT_E_INVALID, "plane needs %zu B of shared memory", bytes);
    int dev = 0;
    RS_CUDA(ctx, cudaGetDevice(&dev));
    static std::mutex mu;
    static std::vector<std::pair<int, const void *>> done;
    std::lock_guard<std::mutex> g(mu);
    const std::pair<int, const void *> key(dev, reinterpret_cast<const void *>(kernel));
    if (std::find(done.begin(), done.end(), key) == done.end()) {
        RS_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
        done.push_back(key);
    }
    return RSDFT_OK;
}

// Threads of a pass of `ctas` blocks, `smem` bytes and `points` points each.  With blocks for more than
// three on an SM: 256 where three share it (fewer for small planes), else enough to fill it alone or in pairs.  With fewer
// blocks the chain of a block is what counts, and more threads shorten it: one band on 24^3, 8 atoms, FP64 H psi 68 -> 62
// us, FP32 41 -> 35, TPA 48 -> 41; on 64^3, 64 atoms 155 -> 139, 72 -> 62, 89 -> 78; 16 bands on 24^3 78 -> 72, 42 -> 39.  From
// three blocks an SM on (24 bands on 24^3) both sides are the same or fewer threads the faster.
inline int pass_threads(size_t smem, int points, long long ctas, int sms, int least) {
    if (smem <= 75 * 1024) {
        if (ctas > 3LL * sms) return std::max(least, std::min(256, cdiv(points, 256) * 32));
        return std::max(least, std::min(ctas <= sms ? 512 : (ctas <= 2LL * sms ? 384 : 256), cdiv(points, 64) * 32));
    }
    return smem <= 113 * 1024 ? 384 : 768;
}

}  // namespace rsdft
