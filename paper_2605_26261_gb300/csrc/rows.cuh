// Row work of the H.v gather (Eq. 12-14 at s = 1/2) shared by the single-launch
// kernel (hv.cu) and the batched kernel (batch.cu): the inverse map of a row, the
// rank of every exchanged label (CR digit blocks or CLT), and the chunked,
// predicated gathers of B interleaved vectors.  NC = true gathers through the
// read-only path (x is not written during the launch); the batched kernel, which
// rewrites its vectors between passes, uses coherent loads.
#pragma once

#include "ftlm_internal.cuh"
#include "vec.cuh"

namespace ftlm {

// J/2 of a bond slot in the vector type.
template <typename V> __device__ __forceinline__ V slot_jh(const uint4 &e);
template <> __device__ __forceinline__ float slot_jh<float>(const uint4 &e) { return __uint_as_float(e.z); }
template <> __device__ __forceinline__ double slot_jh<double>(const uint4 &e)
{
    return __hiloint2double((int)e.w, (int)e.z);
}


// Bond data of one chunk, read once and applied to every row of the thread.
template <typename V, int C>
struct Chunk {
    static_assert(kBondChunk % C == 0, "bond ranges are padded to whole chunks of kBondChunk");
    uint32_t mlo[C], mhi[C];
    V jh[C];
};

template <typename V, int C>
__device__ __forceinline__ void load_chunk(const uint4 *s_bond, int b0, Chunk<V, C> &c)
{
#pragma unroll
    for (int q = 0; q < C; ++q) {
        const uint4 e = s_bond[b0 + q];  // same address in every lane: a broadcast
        c.mlo[q] = e.x;
        c.mhi[q] = e.y;
        c.jh[q] = slot_jh<V>(e);
    }
}

// Gather the chunk's antiparallel terms of RT rows (predicated loads, all issued
// before the first use) and accumulate them into acc[row][vector].
template <typename V, int RT, int B, int C, bool NC = true>
__device__ __forceinline__ void gather_accumulate(const V *__restrict__ x, const Chunk<V, C> &c,
                                                  const bool (&aa)[RT][C], const uint32_t (&kk)[RT][C],
                                                  V (&acc)[RT][B], V (&dsum)[RT])
{
    V xv[RT][C][B];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int q = 0; q < C; ++q) {
            if (aa[i][q]) {
                if constexpr (NC) ld_vec<B>(x + (size_t)kk[i][q] * B, xv[i][q], false);
                else ld_vec_coherent<B>(x + (size_t)kk[i][q] * B, xv[i][q]);
            } else {
#pragma unroll
                for (int r = 0; r < B; ++r) xv[i][q][r] = (V)0;
            }
        }
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int q = 0; q < C; ++q)
            if (aa[i][q]) {
#pragma unroll
                for (int r = 0; r < B; ++r) acc[i][r] = fma(c.jh[q], xv[i][q][r], acc[i][r]);
                dsum[i] += c.jh[q];
            }
}

// Inverse map t -> (h, l) through the digit-block tables: the coarse index bounds
// h to [hs[t >> kHsShift], hs[(t >> kHsShift) + 1]]; a binary search of thi finds
// the last h with thi[h] <= t; the low pattern is entry t - thi[h] of popcount
// group K - popcount(h).
__device__ __forceinline__ void unrank_hl(const SectorTables &s, uint32_t t, uint32_t &h, uint32_t &l,
                                          uint32_t &r_hi, uint32_t &r_lo)
{
    const uint32_t kc = t >> kHsShift;
    uint32_t lo = __ldg(s.hs + kc), hi = __ldg(s.hs + kc + 1) + 1;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(s.thi + mid) <= t) lo = mid;
        else hi = mid;
    }
    h = lo;
    r_hi = __ldg(s.thi + h);
    r_lo = t - r_hi;
    l = __ldg(s.ulo + __ldg(s.uoff + (s.K - __popc(h))) + r_lo);
}

// Row sums of RT output rows (CR): sum over antiparallel bonds of (J_b/2) x[k_b]
// in acc, sum of their J_b/2 in dsum.
template <typename V, typename Lbl, int RT, int B, int C, bool NC = true>
__device__ __forceinline__ void rows_cr(const SectorTables &s, const BondList &bl, const uint4 *s_bond,
                                        const uint16_t *s_tlo, const V *__restrict__ x,
                                        const uint32_t (&t)[RT], V (&acc)[RT][B], V (&dsum)[RT])
{
    uint32_t h[RT], l[RT], r_hi[RT], r_lo[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) unrank_hl(s, t[i], h[i], l[i], r_hi[i], r_lo[i]);
    Chunk<V, C> c;
    bool aa[RT][C];
    uint32_t kk[RT][C];
    const int e_lo = bl.n_lo, e_hi = bl.n_lo + bl.n_hi;
    for (int b0 = 0; b0 < e_lo; b0 += C) {  // both sites in the low block
        load_chunk(s_bond, b0, c);
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const uint32_t m = c.mlo[q], xm = l[i] & m;
                aa[i][q] = (xm != 0u) & (xm != m);
                kk[i][q] = r_hi[i] + s_tlo[l[i] ^ m];
            }
        gather_accumulate<V, RT, B, C, NC>(x, c, aa, kk, acc, dsum);
    }
    for (int b0 = e_lo; b0 < e_hi; b0 += C) {  // both sites in the high block
        load_chunk(s_bond, b0, c);
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const uint32_t m = c.mhi[q], xm = h[i] & m;
                aa[i][q] = (xm != 0u) & (xm != m);
                kk[i][q] = __ldg(s.thi + (h[i] ^ m)) + r_lo[i];
            }
        gather_accumulate<V, RT, B, C, NC>(x, c, aa, kk, acc, dsum);
    }
    for (int b0 = e_hi; b0 < bl.nb; b0 += C) {  // any bond
        load_chunk(s_bond, b0, c);
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const Lbl n = ((Lbl)h[i] << s.L) | l[i];
#pragma unroll
            for (int q = 0; q < C; ++q) {
                Lbl m = c.mlo[q];
                if constexpr (sizeof(Lbl) == 8) m |= (Lbl)c.mhi[q] << 32;
                const Lbl xm = n & m, nn = n ^ m;
                aa[i][q] = (xm != 0) & (xm != m);
                kk[i][q] = __ldg(s.thi + (uint32_t)(nn >> s.L)) + s_tlo[(uint32_t)nn & s.lomask];
            }
        }
        gather_accumulate<V, RT, B, C, NC>(x, c, aa, kk, acc, dsum);
    }
}

// Row sums of RT output rows (CLT, Algorithm 2 per exchanged label).
template <typename V, int RT, int B, int C, bool NC = true>
__device__ __forceinline__ void rows_clt(const SectorTables &s, const BondList &bl, const uint4 *s_bond,
                                         const V *__restrict__ x, const uint32_t (&t)[RT], V (&acc)[RT][B],
                                         V (&dsum)[RT])
{
    uint32_t n[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) n[i] = __ldcs(s.basis + t[i]);
    Chunk<V, C> c;
    bool aa[RT][C];
    uint32_t kk[RT][C];
    for (int b0 = 0; b0 < bl.nb; b0 += C) {
        load_chunk(s_bond, b0, c);
        uint2 e2[RT][C];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const uint32_t m = c.mlo[q], xm = n[i] & m;
                aa[i][q] = (xm != 0u) & (xm != m);
                e2[i][q] = aa[i][q] ? __ldg(s.clt + ((n[i] ^ m) >> 5)) : make_uint2(0u, 0u);
            }
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const uint32_t nn = n[i] ^ c.mlo[q];
                kk[i][q] = e2[i][q].y + __popc(e2[i][q].x & ((1u << (nn & 31u)) - 1u));
            }
        gather_accumulate<V, RT, B, C, NC>(x, c, aa, kk, acc, dsum);
    }
}

// ---- rows of doubles ---------------------------------------------------------
// GB300's FP64 pipe takes two lanes per cycle, so a warp-wide FMA holds it for 16
// cycles whether all lanes or one are active, and about half of a row's bonds are
// parallel.  A row of doubles is therefore summed over a list of its antiparallel
// bonds of its own: a bit mask per lane (integer work), from which every lane takes its
// next bond, so that a pass over B chains costs as many FMAs as the warp's longest
// list has entries (about 60 % of the bonds) instead of one per bond.  The diagonal is
// summed as a whole number (J/2 in units of junscale, exact to 2^-62 sum |J|) instead
// of one FP64 addition per bond and row.  The bonds come in the order of their lower
// site, highest first: those above the bits that differ inside a warp are antiparallel
// in all lanes or in none, so the lanes take them together and gather contiguous rows.
// Measured on GB300 against one FMA and one addition per bond and row: plain H.v of
// blocks of 4, N = 23 random cluster, 46 bonds, 1.14 M rows: 527 -> 284 us; Lanczos H.v of
// blocks of 4, 4 x 6 J1-J2, 96 bonds, 2.7 M rows: 2.46 -> 1.22 ms.
template <typename Lbl> struct BondLists {
    Lbl m[kMaxBondSlots];        // both site bits
    double j[kMaxBondSlots];     // J / 2
    long long f[kMaxBondSlots];  // J / 2 in units of bl.junscale
};

template <typename Lbl>
__device__ __forceinline__ void stage_lists(const BondList &bl, BondLists<Lbl> &s)
{
    for (int i = threadIdx.x; i < bl.n64; i += blockDim.x) {
        const uint4 e = bl.slots_f64[i];
        Lbl m = (Lbl)e.x;
        if constexpr (sizeof(Lbl) == 8) m |= (Lbl)e.y << 32;
        s.m[i] = m;
        s.j[i] = slot_jh<double>(e);
        s.f[i] = bl.whole_f64[i];
    }
}

// Row t: acc[r] += sum over antiparallel bonds of (J/2) x[k], dsum = their sum of J/2; U
// gathers in flight per lane.
template <typename Lbl, bool CLT, int B, int U, bool NC = true>
__device__ __forceinline__ void row_f64(const SectorTables &s, const BondList &bl, const BondLists<Lbl> &s_b,
                                        const uint16_t *s_tlo, const double *__restrict__ x, uint32_t t,
                                        double (&acc)[B], double &dsum)
{
    Lbl n;
    if constexpr (CLT) {
        n = (Lbl)__ldcs(s.basis + t);
    } else {
        uint32_t h, l, r_hi, r_lo;
        unrank_hl(s, t, h, l, r_hi, r_lo);
        n = ((Lbl)h << s.L) | l;
    }
    long long fsum = 0;
    for (int b0 = 0; b0 < bl.n64; b0 += 64) {
        const int nb = min(64, bl.n64 - b0);
        uint64_t todo = 0;
#pragma unroll 4
        for (int b = 0; b < nb; ++b) {
            const Lbl m = s_b.m[b0 + b], xm = n & m;
            const bool anti = (xm != 0) & (xm != m);
            todo |= (uint64_t)anti << b;
            fsum += anti ? s_b.f[b0 + b] : 0ll;
        }
        while (todo) {
            double xv[U][B], j[U];
            bool on[U];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                on[q] = todo != 0;
                const int b = b0 + (on[q] ? __ffsll((long long)todo) - 1 : 0);
                todo &= todo - 1;
                if (on[q]) {
                    j[q] = s_b.j[b];
                    const Lbl nn = n ^ s_b.m[b];
                    uint32_t k;
                    if constexpr (CLT) {
                        const uint2 e = __ldg(s.clt + (nn >> 5));
                        k = e.y + __popc(e.x & ((1u << (nn & 31u)) - 1u));
                    } else {
                        k = __ldg(s.thi + (uint32_t)(nn >> s.L)) + s_tlo[(uint32_t)nn & s.lomask];
                    }
                    if constexpr (NC) ld_vec<B>(x + (size_t)k * B, xv[q], false);
                    else ld_vec_coherent<B>(x + (size_t)k * B, xv[q]);
                } else {  // a value on either path keeps the load here, ahead of its use
                    j[q] = 0.0;
#pragma unroll
                    for (int r = 0; r < B; ++r) xv[q][r] = 0.0;
                }
            }
#pragma unroll
            for (int q = 0; q < U; ++q)
                if (on[q]) {
#pragma unroll
                    for (int r = 0; r < B; ++r) acc[r] = fma(j[q], xv[q][r], acc[r]);
                }
        }
    }
    dsum = (double)fsum * bl.junscale;
}

// Gathers in flight per lane.
template <int B> __host__ __device__ constexpr int f64_gathers() { return B >= 16 ? 1 : (B >= 8 ? 2 : (B >= 4 ? 4 : 8)); }

// ---- one row per thread, for the kernels that stage the bonds themselves -----------
// The bonds of a sector in shared memory in the form its rows take them.
template <typename V, typename Lbl> struct RowBonds {
    uint4 e[kMaxBondSlots];
    __device__ __forceinline__ void stage(const BondList &bl)
    {
        for (int i = threadIdx.x; i < bl.nb; i += blockDim.x) e[i] = bl.slots_f32[i];
    }
};
template <typename Lbl> struct RowBonds<double, Lbl> {
    BondLists<Lbl> l;
    __device__ __forceinline__ void stage(const BondList &bl) { stage_lists<Lbl>(bl, l); }
};
template <typename V, typename Lbl, bool CLT, int B, int C, bool NC>
__device__ __forceinline__ void row_sums(const SectorTables &s, const BondList &bl, const RowBonds<V, Lbl> &s_b,
                                         const uint16_t *s_tlo, const V *__restrict__ x, uint32_t t, V (&acc)[B],
                                         V &dsum)
{
#pragma unroll
    for (int r = 0; r < B; ++r) acc[r] = (V)0;
    if constexpr (sizeof(V) == 8) {
        row_f64<Lbl, CLT, B, f64_gathers<B>(), NC>(s, bl, s_b.l, s_tlo, x, t, acc, dsum);
    } else {
        const uint32_t tt[1] = {t};
        V a[1][B], d[1] = {(V)0};
#pragma unroll
        for (int r = 0; r < B; ++r) a[0][r] = (V)0;
        if constexpr (CLT) rows_clt<V, 1, B, C, NC>(s, bl, s_b.e, x, tt, a, d);
        else rows_cr<V, Lbl, 1, B, C, NC>(s, bl, s_b.e, s_tlo, x, tt, a, d);
#pragma unroll
        for (int r = 0; r < B; ++r) acc[r] = a[0][r];
        dsum = d[0];
    }
}

// One warp owns a tile of 32 RT consecutive rows; lane l handles rows
// tile_base + l + 32 i (i < RT).  The launches hand the tiles out in row order --
// round-robin over the warps (plain H.v, CLT) or from a counter (CR Lanczos) --
// so the whole grid works on one contiguous window of rows at a time.

}  // namespace ftlm
