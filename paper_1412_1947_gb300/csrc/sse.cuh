// What the SSE passes of the float32 and the tensor-core path share: the fixed order of the
// float64 sums (so that both give the same bits), row tiles in shared memory and a minimum of three.
#pragma once

#include "pscl_internal.cuh"

namespace pscl {
namespace {

constexpr int kSseThreads = 256;

// min(a, b, c) in one instruction (sm_100 and later)
__device__ __forceinline__ float min3f(float a, float b, float c)
{
    float m;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
    return m;
}

// 16-byte words between rows of d floats in shared memory: an odd number, so that 8
// consecutive rows fall in different banks.
__host__ __device__ constexpr int tile_ld4(int d) { return ((d + 3) / 4) | 1; }

// n rows of d floats from src into shared memory at a stride of ld4 16-byte words, zeros past
// d and in the rows up to n_pad.
__device__ __forceinline__ void tile_load(float4 *dst, const float *__restrict__ src, int n, int n_pad, int d, int ld4)
{
    const int d4 = (d + 3) / 4;
    const bool vec = d % 4 == 0 && ((uintptr_t)src & 15u) == 0;
    for (int e = threadIdx.x; e < n_pad * d4; e += kSseThreads) {
        const int r = e / d4, q = e - r * d4;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (r < n) {
            const float *p = src + (int64_t)r * d + 4 * q;
            if (vec) {
                v = __ldg(reinterpret_cast<const float4 *>(p));
            } else {
                v.x = __ldg(p);
                if (4 * q + 1 < d) v.y = __ldg(p + 1);
                if (4 * q + 2 < d) v.z = __ldg(p + 2);
                if (4 * q + 3 < d) v.w = __ldg(p + 3);
            }
        }
        dst[r * ld4 + q] = v;
    }
}

// The sum of a value over the block in a fixed tree (thread 0 gets it).
__device__ __forceinline__ double block_tree_sum(double part)
{
    for (int o = 16; o; o >>= 1) part = __dadd_rn(part, __shfl_down_sync(0xffffffffu, part, o));
    __shared__ double ws[kSseThreads / 32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = part;
    __syncthreads();
    double b = 0.0;
    if (threadIdx.x == 0) {
        b = ws[0];
        for (int w = 1; w < kSseThreads / 32; w++) b = __dadd_rn(b, ws[w]);
    }
    return b;
}

// The blocks' sums, added by the last block to finish: thread t those of blocks t, t + 256,
// ... in that order, then the same tree.  (One thread adding 1216 blocks' sums in order was a
// chain of as many float64 additions, 40-60 us behind every SSE pass.)
// Without a ticket the blocks (kClusterSse at most) are one cluster and hand their sums to its
// first through shared memory, in the same order: one launch, where the ticket takes a clearing
// before it (1000 x 16: 10.2 -> 7.9 us a call).  A block may write to another's shared memory only
// once that one has started: every thread of such a kernel passes sse_enter first, and the wait
// for all of the cluster's arrivals there comes just before the write, behind the scoring.
constexpr int kClusterSse = 8;

__device__ __forceinline__ void sse_enter(const uint32_t *ticket)
{
    if (!ticket) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
}

__device__ __forceinline__ void sse_reduce(double part, double *blk_sse, double *sse, uint32_t *ticket)
{
    const double b = block_tree_sum(part);
    if (!ticket) {
        __shared__ double all[kClusterSse];
        asm volatile("barrier.cluster.wait;" ::: "memory");
        if (threadIdx.x == 0) {
            uint32_t at = (uint32_t)__cvta_generic_to_shared(&all[blockIdx.x]);
            asm volatile("mapa.shared::cluster.u32 %0, %0, 0;" : "+r"(at));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(b) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
        if (blockIdx.x != 0) return;
        const double tot = block_tree_sum(threadIdx.x < gridDim.x ? __dadd_rn(0.0, all[threadIdx.x]) : 0.0);
        if (threadIdx.x == 0) *sse = tot;
        return;
    }
    if (threadIdx.x == 0) blk_sse[blockIdx.x] = b;
    __shared__ bool is_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    double tot = 0.0;
    for (unsigned q = threadIdx.x; q < gridDim.x; q += kSseThreads) tot = __dadd_rn(tot, __ldcg(&blk_sse[q]));
    __syncthreads();
    tot = block_tree_sum(tot);
    if (threadIdx.x == 0) {
        *sse = tot;
        *ticket = 0;
    }
}

}  // namespace
}  // namespace pscl
