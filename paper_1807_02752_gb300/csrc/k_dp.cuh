// Block-wide helpers of the per-frame DP kernels (k_dp.cu, k_vpx.cu).
#pragma once

#include "ld_internal.cuh"

namespace ld {
namespace {

constexpr int kMaxChunks = (LD_MAX_H + 31) / 32 + 2;
constexpr int kSent = 0x3fffffff;  // larger than any DP energy (checked when the handle is created)

template <typename T>
__device__ __forceinline__ T *carve(unsigned char *&p, size_t count)
{
    const size_t off = ((size_t)p + 15) & ~(size_t)15;
    T *r = reinterpret_cast<T *>(off);
    p = reinterpret_cast<unsigned char *>(off + sizeof(T) * count);
    return r;
}

// Lexicographic (value, index) minimum over the block; every thread receives the index.
__device__ int block_argmin(int val, int idx, int *scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int d = 16; d > 0; d >>= 1) {
        const int ov = __shfl_down_sync(0xffffffffu, val, d);
        const int oi = __shfl_down_sync(0xffffffffu, idx, d);
        if (ov < val || (ov == val && oi < idx)) {
            val = ov;
            idx = oi;
        }
    }
    if (lane == 0) {
        scratch[2 * warp] = val;
        scratch[2 * warp + 1] = idx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int bv = scratch[0], bi = scratch[1];
        for (int w = 1; w < nw; ++w)
            if (scratch[2 * w] < bv || (scratch[2 * w] == bv && scratch[2 * w + 1] < bi)) {
                bv = scratch[2 * w];
                bi = scratch[2 * w + 1];
            }
        scratch[0] = bi;
    }
    __syncthreads();
    const int r = scratch[0];
    __syncthreads();
    return r;
}

// Ascending list of j < n with flag[j]; returns the count.  chunk: >= n/32 + 2 ints.
__device__ int block_compact(const uint8_t *flag, int n, int16_t *list, int *chunk)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nch = (n + 31) >> 5;
    for (int c = warp; c < nch; c += nw) {
        const int j = (c << 5) + lane;
        const unsigned m = __ballot_sync(0xffffffffu, j < n && flag[j]);
        if (lane == 0)
            chunk[c] = __popc(m);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int c = 0; c < nch; ++c) {
            const int t = chunk[c];
            chunk[c] = s;
            s += t;
        }
        chunk[nch] = s;
    }
    __syncthreads();
    for (int c = warp; c < nch; c += nw) {
        const int j = (c << 5) + lane;
        const bool b = j < n && flag[j];
        const unsigned m = __ballot_sync(0xffffffffu, b);
        if (b)
            list[chunk[c] + __popc(m & ((1u << lane) - 1u))] = (int16_t)j;
    }
    __syncthreads();
    const int cnt = chunk[nch];
    __syncthreads();
    return cnt;
}


// Shared-memory accesses through 32-bit shared addresses (keeps the hot DP loop on the shared-memory path
// whatever pointers the compiler can prove).
__device__ __forceinline__ uint32_t sa(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void atoms_add(uint32_t a, int v) { asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(a), "r"(v)); }

}  // namespace
}  // namespace ld
