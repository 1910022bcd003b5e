// Deterministic FP64 reductions for the row-parallel kernels.
//
// Each block reduces its per-thread partial sums in a fixed tree (warp shuffles, then
// the per-warp sums in order) and stores one partial per block and chain.  The last
// block to finish -- found with a fence and an atomic ticket, no waiting -- adds the
// per-block partials in a fixed order, one warp per chain, and publishes the totals.
// For a fixed grid the summation order never changes, so results are bit-reproducible.
#pragma once

#include "ftlm_internal.cuh"

namespace ftlm {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;  // use lane 0's value: lanes may differ in the last bit
}

// Per-thread accumulator of dot-product terms a * b.  For FP32 operands every
// product is split exactly into p + e (p = fl(a b), e = fma(a, b, -p)) and added
// to a two-float sum (hi, lo) with the error-free TwoSum of Knuth, so the running
// sum keeps about 48 significant bits without touching the FP64 pipe, which is
// narrow on GB300; value() hands the sum to the FP64 block and grid reductions.
// FP64 operands accumulate in FP64 directly.
template <typename V> struct DotAcc;

template <> struct DotAcc<float> {
    float hi = 0.f, lo = 0.f;
    // The _rn intrinsics are never contracted into FMAs: TwoSum needs the rounded
    // product p, not a fused hi + a * b.
    __device__ __forceinline__ void add(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        const float e = fmaf(a, b, -p);
        const float s = __fadd_rn(hi, p);
        const float bv = __fsub_rn(s, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bv)), __fsub_rn(p, bv));
        hi = s;
        lo = __fadd_rn(lo, __fadd_rn(err, e));
    }
    // Adds another accumulator: TwoSum of the high parts, low parts summed.  The
    // TwoSum error is exact, so a.merge(b) and b.merge(a) give the same bits.
    __device__ __forceinline__ void merge(const DotAcc &o)
    {
        const float s = __fadd_rn(hi, o.hi);
        const float bv = __fsub_rn(s, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bv)), __fsub_rn(o.hi, bv));
        hi = s;
        lo = __fadd_rn(__fadd_rn(lo, o.lo), err);
    }
    __device__ __forceinline__ DotAcc shfl_xor(int o) const
    {
        DotAcc r;
        r.hi = __shfl_xor_sync(0xffffffffu, hi, o);
        r.lo = __shfl_xor_sync(0xffffffffu, lo, o);
        return r;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

template <> struct DotAcc<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double a, double b) { v = fma(a, b, v); }
    __device__ __forceinline__ void merge(const DotAcc &o) { v += o.v; }
    __device__ __forceinline__ DotAcc shfl_xor(int o) const
    {
        DotAcc r;
        r.v = __shfl_xor_sync(0xffffffffu, v, o);
        return r;
    }
    __device__ __forceinline__ double value() const { return v; }
};

// Warp sums of B accumulators (B = 1, 2, 4, 8 or 16) by a transposed butterfly: at
// each of the first log2(B) levels a lane keeps one half of its partial sums, sends
// the other half to its partner and merges what it receives (B - 1 merges and
// shuffles in all, instead of 5 B), then a plain butterfly over the remaining
// lanes.  Lane l ends with the sum of accumulator warp_multi_index<B>(l): the bit
// reversal of its low log2(B) bits, so lanes 0 .. B-1 hold the B sums.  The tree
// is fixed: reproducible.
template <typename V, int B>
__device__ __forceinline__ DotAcc<V> warp_sum_multi(DotAcc<V> (&a)[B])
{
    static_assert(B == 1 || B == 2 || B == 4 || B == 8 || B == 16, "B must be a power of two <= 16");
    const unsigned lane = threadIdx.x & 31u;
#pragma unroll
    for (int lvl = 0; (B >> lvl) > 1; ++lvl) {
        const int h = (B >> lvl) / 2;
        const bool upper = (lane >> lvl) & 1u;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            DotAcc<V> keep = upper ? a[i + h] : a[i];
            const DotAcc<V> send = upper ? a[i] : a[i + h];
            keep.merge(send.shfl_xor(1 << lvl));
            a[i] = keep;
        }
    }
    DotAcc<V> t = a[0];
#pragma unroll
    for (int o = B; o < 32; o <<= 1) t.merge(t.shfl_xor(o));
    return t;
}

template <int B> __device__ __forceinline__ int warp_multi_index(unsigned lane)
{
    int r = 0;
#pragma unroll
    for (int lvl = 0; (B >> lvl) > 1; ++lvl) r += ((lane >> lvl) & 1u) ? (B >> (lvl + 1)) : 0;
    return r;
}

// Block sums of B accumulators, in FP64: one transposed warp tree for all of them, then
// thread r < B adds accumulator r's warp sums in warp order and returns the total
// (other threads: 0).  Two barriers, whatever B: one tree per accumulator, each with
// two barriers, cost 8 times the latency and the FP64 instructions at B = 8.
template <typename V, int B, int THREADS>
__device__ __forceinline__ double block_sums(const DotAcc<V> (&a)[B])
{
    constexpr int kWarps = THREADS / 32;
    __shared__ double s_w[kWarps][B];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    DotAcc<double> p[B];
#pragma unroll
    for (int r = 0; r < B; ++r) p[r].v = a[r].value();
    const DotAcc<double> t = warp_sum_multi<double, B>(p);
    if (lane < B) s_w[wid][warp_multi_index<B>(lane)] = t.v;
    __syncthreads();
    double v = 0.0;
    if (threadIdx.x < B) {
#pragma unroll
        for (int i = 0; i < kWarps; ++i) v += s_w[i][threadIdx.x];
    }
    __syncthreads();
    return v;
}

// Stores this block's B sums (thread r < B holds the r-th) in its slot of partials;
// returns true (in every thread) in the last block of the grid to arrive.
template <int B>
__device__ __forceinline__ bool publish_sums(double v, double *partials, unsigned int *counter)
{
    __shared__ bool s_last;
    if (threadIdx.x < B) {
        partials[(size_t)blockIdx.x * B + threadIdx.x] = v;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    return s_last;
}

// Fixed-order totals of partials[0 .. n-1][B], one warp per accumulator, all warps at
// once; done(r, total) runs in lane 0 of the warp that added accumulator r.
template <int B, int THREADS, typename Done>
__device__ __forceinline__ void totals(const double *partials, uint32_t n, Done &&done)
{
    const uint32_t lane = threadIdx.x & 31u;
    for (int r = threadIdx.x >> 5; r < B; r += THREADS / 32) {
        double v = 0.0;
#pragma unroll 4
        for (uint32_t g = lane; g < n; g += 32) v += __ldcg(partials + (size_t)g * B + r);
        v = warp_sum(v);
        if (lane == 0) done(r, v);
    }
}

}  // namespace ftlm
