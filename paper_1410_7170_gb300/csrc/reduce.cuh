// Deterministic grid reductions: warp shuffles, one shared-memory stage per block,
// per-block partials in global scratch, and the last block to finish (found with an
// atomic counter after a memory fence) sums the partials in block order and runs a
// finalisation functor on thread 0. The summation order depends only on the launch
// shape, so repeated runs give bit-identical results.
#pragma once
#include "ff.cuh"
#include "internal.h"

namespace ovl {

template <int NV, int LANES = 32>
__device__ __forceinline__ void warp_sum(double v[NV]) {   // of the first LANES lanes, a power of two
#pragma unroll
    for (int k = 0; k < NV; k++)
#pragma unroll
        for (int off = LANES / 2; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
}

// The end of a reducing kernel is a chain of latencies: the block's sum, a fence, the arrival, the
// partials, their sum, the scalars. A dependent FP64 instruction takes 64 clocks or more, so sums are
// trees; arrivals order memory as acquire and release, which is cheaper than the sequentially
// consistent __threadfence(); a finalisation's inputs (fin.before()) are loaded with the partials. The
// whole sign at 8^4 in FP64 5.33 -> 5.06 ms, at 16^4 in float-float 12.15 -> 11.60 ms; the recursively
// preconditioned solve at 16^4 (FP32 iterations of 36 us) 118.1 -> 112.6 ms.

// Counts an arrival: what the block's threads wrote before the last barrier is visible to those that
// see a later count, and what was written before earlier arrivals to this block after its next barrier.
__device__ __forceinline__ unsigned arrive(unsigned *counter) {
    unsigned t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
    return t;
}

constexpr int kBlockWarps = kBlock / 32;
static_assert(kBlockWarps == 8, "the trees below");

// Block-wide sum of per-thread FP64 values, blockDim.x <= kBlock, valid in thread 0: the first warp adds the warps'
// values lane by lane and then its lanes, 12 FP64 instructions of one warp instead of 5 of every warp
// and 5 more (each occupies the SM's FP64 unit for 16 clocks).
template <int NV>
__device__ __forceinline__ void block_sum(const double vd[NV], double v[NV]) {
    __shared__ double sm[NV][kBlock];
    const int nw = (blockDim.x + 31) >> 5;
    __syncthreads();   // protect sm from a previous use in the same kernel
#pragma unroll
    for (int k = 0; k < NV; k++) sm[k][threadIdx.x] = vd[k];
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int k = 0; k < NV; k++) {
            double a[kBlockWarps];
#pragma unroll
            for (int w = 0; w < kBlockWarps; w++) a[w] = w < nw ? sm[k][32 * w + threadIdx.x] : 0.0;
            v[k] = ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
        }
        warp_sum<NV>(v);
    }
}
template <int NV>
__device__ __forceinline__ void block_sum(double v[NV]) { block_sum<NV>(v, v); }

// Block-wide sum of per-thread FP32 values, blockDim.x <= kBlock: the warp stage in FP32 (shuffles), the sum
// over warps in FP64 by the first warp; the FP64 result is valid in thread 0. GB300 runs
// FP64 at 1/64 of its FP32 rate, so FP64 work stays at one warp per block.
template <int NV>
__device__ __forceinline__ void block_sum(const float vf[NV], double v[NV]) {
    __shared__ double sm[NV][kBlockWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    float t[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) {
        t[k] = vf[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t[k] += __shfl_down_sync(0xffffffffu, t[k], off);
    }
    __syncthreads();   // protect sm from a previous use in the same kernel
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; k++) sm[k][warp] = (double)t[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] = lane < nw ? sm[k][lane & (kBlockWarps - 1)] : 0.0;
        warp_sum<NV, kBlockWarps>(v);
    }
}
// A sum of many FP32 terms without the growth of its rounding error: the running sum and the errors of
// its additions (TwoSum), which are exact. Where one wave of blocks takes the whole lattice a thread
// adds thousands of terms and a row of the grid has few warps; with plain FP32 sums in threads and
// warps the relative error of a squared norm at 32^4 had grown tenfold against one site per thread, with
// these it is that of the terms. Six FP32 additions for one, in kernels that wait for memory, and about
// 100 clocks more for the shuffles at their ends.
struct fsum {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float x) {
        const ff t = ff_two_sum(s, x);
        s = t.hi;
        e = __fadd_rn(e, t.lo);
    }
    __device__ __forceinline__ void add(const fsum &x) {
        const ff t = ff_two_sum(s, x.s);
        s = t.hi;
        e = __fadd_rn(__fadd_rn(e, x.e), t.lo);
    }
};
// Block-wide sum of per-thread sums of this kind, blockDim.x <= kBlock: the warp stage in FP32 with its
// errors, the sum over warps in FP64 by the first warp.
template <int NV>
__device__ __forceinline__ void block_sum(const fsum vf[NV], double v[NV]) {
    __shared__ double sm[NV][kBlockWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    fsum t[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) {
        t[k] = vf[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            fsum o;
            o.s = __shfl_down_sync(0xffffffffu, t[k].s, off);
            o.e = __shfl_down_sync(0xffffffffu, t[k].e, off);
            t[k].add(o);
        }
    }
    __syncthreads();   // protect sm from a previous use in the same kernel
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; k++) sm[k][warp] = (double)t[k].s + (double)t[k].e;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] = lane < nw ? sm[k][lane & (kBlockWarps - 1)] : 0.0;
        warp_sum<NV, kBlockWarps>(v);
    }
}
// Block-wide sum of per-thread float-float values, blockDim.x <= kBlock: the warp stage in float-float (both
// words shuffled), the sum over warps in FP64 by the first warp.
template <int NV>
__device__ __forceinline__ void block_sum(const ff vf[NV], double v[NV]) {
    __shared__ double sm[NV][kBlockWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    ff t[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) {
        t[k] = vf[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            t[k] += ff(__shfl_down_sync(0xffffffffu, t[k].hi, off), __shfl_down_sync(0xffffffffu, t[k].lo, off));
    }
    __syncthreads();   // protect sm from a previous use in the same kernel
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; k++) sm[k][warp] = t[k].to_double();
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] = lane < nw ? sm[k][lane & (kBlockWarps - 1)] : 0.0;
        warp_sum<NV, kBlockWarps>(v);
    }
}
// Reduce v[NV] (per-thread FP64, FP32, fsum or float-float partial sums) over the grid; the last block calls
// fin(total, fin.before()) on thread 0 and resets the counter. Must be reached by every thread of
// every block.
template <int NV, typename T, typename Fin>
__device__ __forceinline__ void grid_reduce(const T vt[NV], RedScratch rs, Fin fin) {
    __shared__ int is_last;
    double v[NV];
    block_sum<NV>(vt, v);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; k++) rs.partials[k * kMaxRedBlocks + blockIdx.x] = v[k];
        is_last = arrive(rs.counter) == gridDim.x - 1;
    }
    __syncthreads();
    if (is_last) {
        decltype(fin.before()) in;
        if (threadIdx.x == 0) in = fin.before();
        double s[NV];
#pragma unroll
        for (int k = 0; k < NV; k++) {
            s[k] = 0.0;
            for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
                s[k] += __ldcg(rs.partials + k * kMaxRedBlocks + b);
        }
        block_sum<NV>(s);
        if (threadIdx.x == 0) {
            fin(s, in);
            *rs.counter = 0u;
        }
    }
}

// As grid_reduce, but the last block runs fin(total, lane, fin.before(lane)) on all 32 lanes of its first
// warp (for finalisations that are parallel over a small index, e.g. one lane per shift).
template <int NV, typename T, typename Fin>
__device__ __forceinline__ void grid_reduce_warp(const T vt[NV], RedScratch rs, Fin fin) {
    __shared__ int is_last;
    __shared__ double tot[NV];
    double v[NV];
    block_sum<NV>(vt, v);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; k++) rs.partials[k * kMaxRedBlocks + blockIdx.x] = v[k];
        is_last = arrive(rs.counter) == gridDim.x - 1;
    }
    __syncthreads();
    if (is_last) {
        decltype(fin.before(0)) in;
        if (threadIdx.x < 32) in = fin.before((int)threadIdx.x);
        double s[NV];
#pragma unroll
        for (int k = 0; k < NV; k++) {
            s[k] = 0.0;
            for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
                s[k] += __ldcg(rs.partials + k * kMaxRedBlocks + b);
        }
        block_sum<NV>(s);
        if (threadIdx.x == 0)
#pragma unroll
            for (int k = 0; k < NV; k++) tot[k] = s[k];
        __syncthreads();
        if (threadIdx.x < 32) {
            double t2[NV];
#pragma unroll
            for (int k = 0; k < NV; k++) t2[k] = tot[k];
            fin(t2, (int)threadIdx.x, in);
            if (threadIdx.x == 0) *rs.counter = 0u;
        }
    }
}

// Last-block detection without values: returns true in every thread of the block that
// arrives last (all blocks' global writes before are visible to it) and
// resets the counter. Must be reached by every thread of every block.
__device__ __forceinline__ bool grid_last_block(unsigned *counter) {
    __shared__ int is_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        is_last = arrive(counter) == gridDim.x - 1;
        if (is_last) *counter = 0u;
    }
    __syncthreads();
    return is_last;
}

}  // namespace ovl
