// Lanczos epilogue of the H.v launches (step a4 fused into step a3), shared by the
// spin-1/2 kernel (hv.cu) and the general-spin kernel (spin.cu).
//
// Paige's ordering, per chain r of a block of B interleaved vectors.  The stored
// vector u_j is un-normalized, q_j = u_j / s_j.  With x = u_j and the in-place
// buffer holding u_{j-1}:
//   y[t] = (H u_j)[t] / s_j - (beta_{j-1} / s_{j-1}) u_{j-1}[t]     (overwrites u_{j-1})
//   alpha partial += q_j[t] y[t]                                    (FP64-class)
// Per-thread partial dot products use DotAcc (exact products, two-float
// compensated sums for FP32 vectors).  Two ways to finish alpha_j:
//  - static tile order (a warp takes every nwarps-th tile of rows): the block sum
//    is an FP64 tree and the last block to finish adds the per-block partials in
//    a fixed order and stores alpha_j (epi_end);
//  - dynamic tile order (CR and FP32 general-spin launches: tiles handed out by a
//    counter, so that all warps work on one frontier of rows and the gathers of the rows
//    in flight share L2): each tile's sums go through a fixed warp tree and are added as
//    whole numbers of two words (AlphaSums), whose sum does not depend on the order; a
//    launch of one warp (CR) or the last CTA (general spin) turns it into alpha_j.  A
//    slot per tile, added in tile order by a second launch, cost 15 to 41 us per step and
//    2 B bytes per row.
// Either way the result is fixed for a given sector and grid: alpha_j is reproducible.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ftlm_internal.cuh"
#include "reduce.cuh"
#include "two_word.cuh"
#include "vec.cuh"

namespace ftlm {

struct EpiDev {
    ChainState *st;
    double *partials;
    unsigned int *counter;  // [0] block ticket; [1], [2], [3] dynamic tile order
    double *alpha_out;
    unsigned long long *fixed;  // sums of the dynamic tile order, two words per chain
    double scale, unscale;      // 2^alpha_shift and 2^-alpha_shift: the first word of a sum
                                // counts 2^-alpha_shift
    uint64_t slot;              // bytes between the blocks of chains of a launch (blockIdx.y)
    int alpha_stride;
    int has_prev;
};

// The epilogue and the vectors of this CTA's block of chains.
template <int B> __device__ __forceinline__ EpiDev epi_block(EpiDev ep)
{
    if (blockIdx.y) {
        const uint64_t o = blockIdx.y * ep.slot;
        ep.st = reinterpret_cast<ChainState *>(reinterpret_cast<char *>(ep.st) + o);
        ep.partials = reinterpret_cast<double *>(reinterpret_cast<char *>(ep.partials) + o);
        ep.counter = reinterpret_cast<unsigned int *>(reinterpret_cast<char *>(ep.counter) + o);
        ep.fixed = reinterpret_cast<unsigned long long *>(reinterpret_cast<char *>(ep.fixed) + o);
        ep.alpha_out += (size_t)blockIdx.y * B * ep.alpha_stride;
    }
    return ep;
}
template <typename T> __device__ __forceinline__ T *block_ptr(T *p, uint64_t slot)
{
    using C = typename std::conditional<std::is_const<T>::value, const char, char>::type;
    return reinterpret_cast<T *>(reinterpret_cast<C *>(p) + blockIdx.y * slot);
}

inline EpiDev epi_of(const LanczosHv *epi)
{
    EpiDev ep{};
    if (epi) {
        ep.st = epi->st;
        ep.partials = epi->partials;
        ep.counter = epi->counter;
        ep.alpha_out = epi->alpha_out;
        ep.fixed = epi->fixed;
        // |alpha_j| <= ||H|| < 2^e, and ||y|| <= 2 ||H||: the tiles' sums together stay
        // below 2^50 units in magnitude, whatever their number (two_word.cuh for their rests)
        // (a bound out of range, at either end, does not put alpha there)
        const double nb = epi->norm_bound;
        const int shift = !std::isfinite(nb) ? 49 - 1025 : nb > 0.0 ? std::min(1000, 48 - std::ilogb(nb)) : 1000;
        ep.scale = std::ldexp(1.0, shift);
        ep.unscale = std::ldexp(1.0, -shift);
        ep.alpha_stride = epi->alpha_stride;
        ep.slot = epi->slot;
        ep.has_prev = epi->j > 1;
    }
    return ep;
}

// Per-chain scalars 1/s_j and beta_{j-1}/s_{j-1} into shared memory.  Returns true
// (in every thread) when every chain of the block has stopped: the launch then has
// nothing to do, and the test is uniform over the grid.
template <typename V, int B>
__device__ __forceinline__ bool epi_begin(const EpiDev &ep, V *s_inv_s, V *s_c_prev)
{
    bool all_stopped = true;
#pragma unroll
    for (int r = 0; r < B; ++r) all_stopped &= ep.st[r].stopped != 0;
    if (all_stopped) return true;
    if (threadIdx.x < B) {
        const ChainState &st = ep.st[threadIdx.x];
        s_inv_s[threadIdx.x] = (V)(1.0 / st.s_cur);
        s_c_prev[threadIdx.x] = ep.has_prev ? (V)(st.beta_prev / st.s_prev) : (V)0;
    }
    return false;
}

// Output row t: y = diag * x[t] + acc (plain H.v) or the epilogue above.
template <typename V, int B, bool LANCZOS>
__device__ __forceinline__ void epi_row(const EpiDev &ep, const V *s_inv_s, const V *s_c_prev,
                                        const V *__restrict__ x, V *y, uint32_t t, V diag, const V (&acc)[B],
                                        DotAcc<V> (&apart)[B])
{
    V xt[B], out[B];
    ld_vec<B>(x + (size_t)t * B, xt, false);
    if (LANCZOS) {
        V up[B];
        if (ep.has_prev) ld_vec<B>(y + (size_t)t * B, up, true);
#pragma unroll
        for (int r = 0; r < B; ++r) {
            const V inv_s = s_inv_s[r];
            const V hv = fma(diag, xt[r], acc[r]);
            out[r] = ep.has_prev ? fma(-s_c_prev[r], up[r], hv * inv_s) : hv * inv_s;
            apart[r].add(xt[r] * inv_s, out[r]);
        }
    } else {
#pragma unroll
        for (int r = 0; r < B; ++r) out[r] = fma(diag, xt[r], acc[r]);
    }
    st_vec<B>(y + (size_t)t * B, out);
}

// Output row t of walk A of a split H.v (CR): the Lanczos output of the bonds of
// walk A, y = (H_A u_j)[t] / s_j - (beta_{j-1} / s_{j-1}) u_{j-1}[t], with no alpha
// partial (walk B adds the rest of the row and finishes alpha).
template <typename V, int B>
__device__ __forceinline__ void epi_row_walk_a(const EpiDev &ep, const V *s_inv_s, const V *s_c_prev,
                                               const V *__restrict__ x, V *y, uint32_t t, V diag,
                                               const V (&acc)[B])
{
    V xt[B], out[B], up[B];
    ld_vec<B>(x + (size_t)t * B, xt, false);
    if (ep.has_prev) ld_vec<B>(y + (size_t)t * B, up, true);
#pragma unroll
    for (int r = 0; r < B; ++r) {
        const V hv = fma(diag, xt[r], acc[r]);
        out[r] = ep.has_prev ? fma(-s_c_prev[r], up[r], hv * s_inv_s[r]) : hv * s_inv_s[r];
    }
    st_vec<B>(y + (size_t)t * B, out);
}

// Block sums of the alpha partials, publication, and the last block's fixed-order
// grid sum into alpha_j (chains that have stopped keep their value).
template <typename V, int B, int THREADS>
__device__ __forceinline__ void epi_end(const EpiDev &ep, DotAcc<V> (&apart)[B])
{
    const double part = block_sums<V, B, THREADS>(apart);
    if (publish_sums<B>(part, ep.partials, ep.counter)) {
        totals<B, THREADS>(ep.partials, gridDim.x, [&](int r, double v) {
            if (ep.st[r].stopped) return;
            ep.st[r].alpha = v;
            ep.alpha_out[(size_t)r * ep.alpha_stride] = v;
        });
        if (threadIdx.x == 0) *ep.counter = 0;
    }
}

// Dynamic tile order: a warp's first tile is its index, later ones come from the
// counter ep.counter[1], which is zero when a launch starts: alpha_kernel zeroes it at
// the end of a step, and walk A's last warp to run out of tiles (ep.counter[2] counts
// them) for the walk B that follows.  A warp
// claims its next tile when it starts a tile (claim_tile, lane 0) and reads the
// claim when it finishes (claimed_tile), so the atomic's round trip is hidden.
__device__ __forceinline__ uint32_t claim_tile(const EpiDev &ep)
{
    return (threadIdx.x & 31u) == 0 ? atomicAdd(ep.counter + 1, 1u) : 0u;
}

__device__ __forceinline__ uint32_t claimed_tile(uint32_t claim, uint32_t nwarps)
{
    return __shfl_sync(0xffffffffu, claim, 0) + nwarps;
}

// Sums of per-tile values as whole numbers of two words (two_word.cuh), one pair per warp
// and chain in shared memory: the first word counts 2^-alpha_shift, the second 2^-(alpha_shift +
// 40).  Every value is taken to 2^-(alpha_shift + 40), about 2^-90 ||H||, and whole
// numbers add in any order to the same sum, so the warps may take their tiles in any
// order.  A warp's second word stays below 2^40, so those of all warps of a launch add up
// within 64 bits.  bad: bit r is set when a value of chain r was not finite.
template <int B, int THREADS> struct AlphaSums {
    long long v[THREADS / 32][2 * B];
    unsigned int bad;
};

// Before the launch's first barrier, by every thread.
template <int B, int THREADS> __device__ __forceinline__ void tiles_begin(AlphaSums<B, THREADS> &s)
{
    for (int i = threadIdx.x; i < THREADS / 32 * 2 * B; i += THREADS) s.v[i / (2 * B)][i % (2 * B)] = 0;
    if (threadIdx.x == 0) s.bad = 0;
}

// Adds the warp's alpha partial sums of one tile, through a fixed warp tree.  Called by
// the whole warp.
template <typename V, int B, int THREADS>
__device__ __forceinline__ void add_tile(const EpiDev &ep, AlphaSums<B, THREADS> &s, DotAcc<V> (&a)[B])
{
    const DotAcc<V> t = warp_sum_multi<V, B>(a);
    const unsigned lane = threadIdx.x & 31u;
    if (lane < B) {
        const int r = warp_multi_index<B>(lane);
        if (!two_word_add(s.v[threadIdx.x >> 5] + 2 * r, t.value(), ep.scale)) atomicOr(&s.bad, 1u << r);
    }
}

// End of a launch with the dynamic tile order, called by every thread: the CTA's
// sums, one atomic addition per chain and word.  alpha_kernel (hv.cu) turns them into
// alpha_j and zeroes the sums and the tile counter for the next step.
template <int B, int THREADS>
__device__ __forceinline__ void tiles_done(const EpiDev &ep, AlphaSums<B, THREADS> &s)
{
    __syncthreads();
    if (threadIdx.x < 2 * B) {
        long long v = 0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) v += s.v[w][threadIdx.x];
        atomicAdd(&ep.fixed[threadIdx.x], (unsigned long long)v);
        if (threadIdx.x == 0 && s.bad) atomicOr(ep.counter + 3, s.bad);
    }
}

// The same with alpha_j formed by the last CTA to arrive, from one pair of words per CTA and
// chain in ep.partials (2 B words per CTA of the grid).
template <int B, int THREADS>
__device__ __forceinline__ void tiles_end(const EpiDev &ep, AlphaSums<B, THREADS> &s)
{
    constexpr uint32_t W = 2 * B;
    static_assert(THREADS % W == 0, "a slice of the CTAs per W threads");
    __shared__ bool s_last;
    unsigned long long *part = reinterpret_cast<unsigned long long *>(ep.partials);
    __syncthreads();
    if (threadIdx.x < W) {
        long long v = 0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) v += s.v[w][threadIdx.x];
        part[(size_t)blockIdx.x * W + threadIdx.x] = (unsigned long long)v;
        if (threadIdx.x == 0 && s.bad) atomicOr(ep.counter + 3, s.bad);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ep.counter, 1u) == gridDim.x - 1;
    if (threadIdx.x < W) s.v[0][threadIdx.x] = 0;
    __syncthreads();
    if (!s_last) return;
    unsigned long long v = 0;
    for (uint32_t g = threadIdx.x / W; g < gridDim.x; g += THREADS / W) v += __ldcg(part + (size_t)g * W + threadIdx.x % W);
    atomicAdd(reinterpret_cast<unsigned long long *>(&s.v[0][threadIdx.x % W]), v);
    __syncthreads();
    if (threadIdx.x < B) {
        const int r = threadIdx.x;
        const bool bad = (__ldcg(ep.counter + 3) >> r) & 1u;
        const double a = two_word_value(s.v[0][2 * r], s.v[0][2 * r + 1], ep.unscale);
        if (!ep.st[r].stopped) {
            ep.st[r].alpha = bad ? NAN : a;
            ep.alpha_out[(size_t)r * ep.alpha_stride] = bad ? NAN : a;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) ep.counter[0] = ep.counter[1] = ep.counter[3] = 0;
}

// End of a launch that takes its tiles in dynamic order and leaves no sums (walk A).
__device__ __forceinline__ void tiles_done(const EpiDev &ep, uint32_t nwarps)
{
    if ((threadIdx.x & 31u) == 0) {
        __threadfence();
        if (atomicAdd(ep.counter + 2, 1u) == nwarps - 1) {
            ep.counter[1] = 0;
            ep.counter[2] = 0;
        }
    }
}

}  // namespace ftlm
