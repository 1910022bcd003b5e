// Row work of the general-spin H.v (Eq. 12-14 for any s), shared by the
// single-sector kernel (spin.cu) and the multi-sector path (msv.cu): the inverse
// map of a row to its base-d digits, and the per-row sums of the two ladder terms
// of every bond, class by class (both sites in the low digit block, both in the
// high block, one in each), each class with its own digit-block rank arithmetic
// (gathers of a chunk of bonds issued together, predicated).
#pragma once

#include "ftlm_internal.cuh"
#include "vec.cuh"

namespace ftlm {

constexpr int kSpinMaxSites = 16;           // 4-bit digit fields in 64 bits
constexpr int kSpinMaxTwoS = 7;             // d <= 8
constexpr int kSpinMaxBonds = kSpinMaxSites * (kSpinMaxSites - 1) / 2;  // bonds are distinct pairs
constexpr uint64_t kSpinMaxLow = 1u << 14;  // tlo entries (shared memory)
constexpr uint64_t kSpinMaxHigh = 1u << 27; // thi entries

__device__ __forceinline__ uint32_t div_d(const SpinDev &p, uint32_t n)
{
    return (uint32_t)(((uint64_t)n * p.magic) >> p.shift);
}

struct SpinRow {
    uint32_t lo, hi;      // low and high labels of the row
    uint32_t thi_h, r_lo; // the row's two halves of its rank
    uint64_t dig;         // digit k in bits 4k .. 4k+3
};

__device__ __forceinline__ void spin_unrank(const SectorTables &s, const SpinDev &p, uint32_t t, SpinRow &w)
{
    const uint32_t kc = t >> kHsShift;
    uint32_t lo = __ldg(s.hs + kc), hi = __ldg(s.hs + kc + 1) + 1;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(s.thi + mid) <= t) lo = mid;
        else hi = mid;
    }
    w.hi = lo;
    w.thi_h = __ldg(s.thi + lo);
    w.r_lo = t - w.thi_h;
    uint64_t dig = 0;
    uint32_t n = w.hi, sum = 0;
    for (int k = s.L; k < s.N; ++k) {
        const uint32_t q = div_d(p, n), a = n - q * p.d;
        dig |= (uint64_t)a << (4 * k);
        sum += a;
        n = q;
    }
    w.lo = __ldg(s.ulo + __ldg(s.uoff + (p.A - sum)) + w.r_lo);
    n = w.lo;
    for (int k = 0; k < s.L; ++k) {
        const uint32_t q = div_d(p, n), a = n - q * p.d;
        dig |= (uint64_t)a << (4 * k);
        n = q;
    }
    w.dig = dig;
}

template <typename V> __device__ __forceinline__ const V *spin_J(const SpinDev &p);
template <> __device__ __forceinline__ const float *spin_J<float>(const SpinDev &p) { return p.jf; }
template <> __device__ __forceinline__ const double *spin_J<double>(const SpinDev &p) { return p.jd; }
template <typename V> __device__ __forceinline__ const V *spin_up(const SpinDev &p);
template <> __device__ __forceinline__ const float *spin_up<float>(const SpinDev &p) { return p.upf; }
template <> __device__ __forceinline__ const double *spin_up<double>(const SpinDev &p) { return p.upd; }

// Per-bond factors of a row, indexed by the digit pair d a_i + a_j (d <= 8):
// [0, 64) the s_i^+ s_j^- factor of Eq. 13 and [64, 128) the s_i^- s_j^+ factor of
// Eq. 14, both with the 1/2 of Eq. 12 and zero where the source digit leaves
// 0 .. 2s; [128, 192) m_i m_j (exact: products of half-integers).  The compact
// index keeps the d^2 entries of a table in distinct shared-memory banks for
// d <= 5, so the lanes of a warp read them without bank conflicts.
constexpr int kSpinCoef = 3 * 64;

template <typename V> __device__ __forceinline__ void spin_stage_coef(const SpinDev &p, V *s_cf)
{
    const V *up = spin_up<V>(p);
    const uint32_t two_s = p.two_s, d = p.d;
    const V sv = (V)(0.5 * p.two_s);
    for (uint32_t idx = threadIdx.x; idx < (uint32_t)kSpinCoef; idx += blockDim.x) {
        const uint32_t tab = idx >> 6, rem = idx & 63u, ai = rem / d, aj = rem % d;
        V v = (V)0;
        if (rem < d * d) {
            if (tab == 0u && ai >= 1u && aj < two_s) v = (V)0.5 * up[ai - 1] * up[aj];
            else if (tab == 1u && ai < two_s && aj >= 1u) v = (V)0.5 * up[ai] * up[aj - 1];
            else if (tab == 2u) v = ((V)ai - sv) * ((V)aj - sv);
        }
        s_cf[idx] = v;
    }
}

// The two ladder terms of C bonds: s_i^+ s_j^- from row k0 (source digits a_i - 1, a_j + 1,
// Eq. 13) and s_i^- s_j^+ from row k1 (a_i + 1, a_j - 1, Eq. 14), and their diagonal.  A term
// whose factor is zero does not exist.  All gathers are issued before the first sum.
template <typename V, int B, int C>
__device__ __forceinline__ void spin_terms(const V *(&cf)[C], V (&J)[C], uint32_t (&k0)[C], uint32_t (&k1)[C],
                                           const V *__restrict__ x, V (&acc)[B], V &diag)
{
    V c[2 * C], xv[2 * C][B];
#pragma unroll
    for (int q = 0; q < C; ++q) {
        const V f0 = cf[q][0], f1 = cf[q][64];
        diag = fma(J[q], cf[q][128], diag);
        c[2 * q] = J[q] * f0;
        c[2 * q + 1] = J[q] * f1;
        const bool use[2] = {f0 != (V)0, f1 != (V)0};
        const uint32_t k[2] = {use[0] ? k0[q] : 0u, use[1] ? k1[q] : 0u};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (use[h]) {
                ld_vec<B>(x + (size_t)k[h] * B, xv[2 * q + h], false);
            } else {
#pragma unroll
                for (int r = 0; r < B; ++r) xv[2 * q + h][r] = (V)0;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 2 * C; ++q)
#pragma unroll
        for (int r = 0; r < B; ++r) acc[r] = fma(c[q], xv[q][r], acc[r]);
}

// The bonds [b, end), each described by bond(b, factors, J, k0, k1): C at a time, the
// rest one by one.
template <typename V, int B, int C, typename Bond>
__device__ __forceinline__ void spin_bonds(uint32_t b, uint32_t end, Bond &&bond, const V *__restrict__ x,
                                           V (&acc)[B], V &diag)
{
    if (C > 1)
        for (; b + C <= end; b += C) {
            const V *cf[C];
            V J[C];
            uint32_t k0[C], k1[C];
#pragma unroll
            for (int q = 0; q < C; ++q) bond(b + q, cf[q], J[q], k0[q], k1[q]);
            spin_terms<V, B, C>(cf, J, k0, k1, x, acc, diag);
        }
    for (; b < end; ++b) {
        const V *cf[1];
        V J[1];
        uint32_t k0[1], k1[1];
        bond(b, cf[0], J[0], k0[0], k1[0]);
        spin_terms<V, B, 1>(cf, J, k0, k1, x, acc, diag);
    }
}

// The bonds [b_beg, b_end) of one class of row w: the two ladder terms of each,
// with the rank arithmetic of the class (CLS 0: both sites in the low block, only
// the low half of the rank moves; 1: both in the high block; 2: site i low, site j
// high).  Adds J m_i m_j to diag and the terms to acc; the clamps keep the table
// addresses of a term that does not exist in range.
template <typename V, int B, int C, int CLS>
__device__ __forceinline__ void spin_class(const SectorTables &s, const SpinDev &p, const uint16_t *s_tlo,
                                           const uint4 *s_bond, const V *s_J, const V *s_cf,
                                           const V *__restrict__ x, const SpinRow &w, uint32_t b_beg, uint32_t b_end,
                                           V (&acc)[B], V &diag)
{
    auto bond = [&](uint32_t b, const V *&cf, V &J, uint32_t &k0, uint32_t &k1) {
        const uint4 e = s_bond[b];
        const uint32_t i = e.x & 255u, j = (e.x >> 8) & 255u, pi = e.y, pj = e.z;
        const uint32_t ai = (uint32_t)(w.dig >> (4 * i)) & 15u, aj = (uint32_t)(w.dig >> (4 * j)) & 15u;
        if constexpr (CLS == 0) {
            k0 = w.thi_h + s_tlo[min(w.lo - pi + pj, s.lomask)];
            k1 = w.thi_h + s_tlo[min(w.lo + pi - pj, s.lomask)];
        } else if constexpr (CLS == 1) {
            k0 = __ldg(s.thi + min(w.hi - pi + pj, s.H - 1u)) + w.r_lo;
            k1 = __ldg(s.thi + min(w.hi + pi - pj, s.H - 1u)) + w.r_lo;
        } else {
            k0 = __ldg(s.thi + min(w.hi + pj, s.H - 1u)) + s_tlo[min(w.lo - pi, s.lomask)];
            k1 = __ldg(s.thi + min(w.hi - pj, s.H - 1u)) + s_tlo[min(w.lo + pi, s.lomask)];
        }
        cf = s_cf + (ai * p.d + aj);
        J = s_J[b];
    };
    spin_bonds<V, B, C>(b_beg, b_end, bond, x, acc, diag);
}

// ---- tiles of 32 rows with one high label ------------------------------------
// Rows of one high label are consecutive (D / H of them on average: 1255 for the spin-2
// icosahedron, 911 for spin 1), so nearly every tile of a warp has one.  Then a
// high-high bond is the same two moves in every lane: its existing terms are listed once
// per tile, one lane per bond, as {first source row, factor}, and a row only gathers and
// accumulates.  A cross bond has its digit of the high site and both high ranks
// listed.  The terms and their order are those of spin_class, so a row's sums have the
// same bits on either path.  Spin-2 icosahedron, us per Lanczos H.v launch without and with
// the lists: blocks of 8 floats 2118 and 1949, vectors 1223 and 1066, blocks of 4
// doubles 14130 and 12640.
template <typename V> struct SpinList {
    uint4 *cross;    // cross bonds: {4 i | a_j << 8, d^i, thi of h + d^j, thi of h - d^j}
    V *c;            // high-high terms: J times the term's factor
    uint32_t *base;  // and thi of the source's high label
    float *mm;       // m_i m_j of the high-high bonds (quarters: exact)
};

template <typename V> __host__ __device__ constexpr uint32_t spin_list_bytes(uint32_t n_hh, uint32_t n_cross)
{
    return (16u * n_cross + n_hh * (2u * (uint32_t)sizeof(V) + 12u) + 15u) & ~15u;
}

// The most a basis can have.  Its d^L > 2^14 / d (L < N) and d^(N-L) <= 2^27 leave N - L <= 10
// for d >= 5, 9 for d = 4 and 8 for d = 3, so at most 45 bonds are high-high; L (N - L) <= 64.
constexpr uint32_t kSpinMaxHH = 45, kSpinMaxCross = 64;

// Entries of the staged tlo, up to the 16-byte boundary where the lists begin.
__host__ __device__ __forceinline__ uint32_t spin_tlo_entries(const SectorTables &s) { return (s.lomask + 8u) & ~7u; }

// The calling warp's lists, in order behind each other from a 16-byte boundary.
template <typename V>
__device__ __forceinline__ SpinList<V> spin_list(const SpinDev &p, void *lists)
{
    const uint32_t n_cross = p.nb - p.n_ll - p.n_hh;
    char *at = static_cast<char *>(lists) + (threadIdx.x >> 5) * spin_list_bytes<V>(p.n_hh, n_cross);
    SpinList<V> l;
    l.cross = reinterpret_cast<uint4 *>(at);
    l.c = reinterpret_cast<V *>(at + 16u * n_cross);
    l.base = reinterpret_cast<uint32_t *>(l.c + 2u * p.n_hh);
    l.mm = reinterpret_cast<float *>(l.base + 2u * p.n_hh);
    return l;
}

// The lists of the warp's high label (the row w of any lane); returns the number of
// high-high terms.
template <typename V>
__device__ __forceinline__ uint32_t spin_list_fill(const SectorTables &s, const SpinDev &p, const uint4 *s_bond,
                                                   const V *s_J, const V *s_cf, const SpinRow &w,
                                                   const SpinList<V> &ls)
{
    const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u, e_hh = p.n_ll + p.n_hh;
    uint32_t n = 0;
    __syncwarp();  // the lists of the warp's previous tile have been read
    for (uint32_t q0 = 0; q0 < p.n_hh; q0 += 32u) {
        const uint32_t q = q0 + lane;
        bool u0 = false, u1 = false;
        V c0 = (V)0, c1 = (V)0;
        uint32_t b0 = 0, b1 = 0;
        if (q < p.n_hh) {
            const uint4 e = s_bond[p.n_ll + q];
            const uint32_t ai = (uint32_t)(w.dig >> (4 * (e.x & 255u))) & 15u;
            const uint32_t aj = (uint32_t)(w.dig >> (4 * ((e.x >> 8) & 255u))) & 15u;
            const uint32_t ij = ai * p.d + aj;
            const V J = s_J[p.n_ll + q], f0 = s_cf[ij], f1 = s_cf[64 + ij];
            u0 = f0 != (V)0;
            u1 = f1 != (V)0;
            c0 = J * f0;
            c1 = J * f1;
            b0 = __ldg(s.thi + min(w.hi - e.y + e.z, s.H - 1u));
            b1 = __ldg(s.thi + min(w.hi + e.y - e.z, s.H - 1u));
            ls.mm[q] = (float)s_cf[128 + ij];
        }
        const uint32_t m0 = __ballot_sync(~0u, u0), m1 = __ballot_sync(~0u, u1);
        uint32_t pos = n + __popc(m0 & below) + __popc(m1 & below);
        if (u0) {
            ls.base[pos] = b0;
            ls.c[pos] = c0;
            ++pos;
        }
        if (u1) {
            ls.base[pos] = b1;
            ls.c[pos] = c1;
        }
        n += __popc(m0) + __popc(m1);
    }
    for (uint32_t q = lane; q < p.nb - e_hh; q += 32u) {
        const uint4 e = s_bond[e_hh + q];
        const uint32_t aj = (uint32_t)(w.dig >> (4 * ((e.x >> 8) & 255u))) & 15u;
        ls.cross[q] = make_uint4(4u * (e.x & 255u) | (aj << 8), e.y, __ldg(s.thi + min(w.hi + e.z, s.H - 1u)),
                                 __ldg(s.thi + min(w.hi - e.z, s.H - 1u)));
    }
    __syncwarp();
    return n;
}

// High-high bonds of row w: n listed terms, U gathers together (their addresses need no rank
// work, so more of them fit in the registers than of the other bonds).
template <typename V, int B, int U>
__device__ __forceinline__ void spin_list_hh(const SpinDev &p, const V *s_J, const SpinList<V> &ls, uint32_t n,
                                             const V *__restrict__ x, const SpinRow &w, V (&acc)[B], V &diag)
{
    for (uint32_t b = 0; b < p.n_hh; ++b) diag = fma(s_J[p.n_ll + b], (V)ls.mm[b], diag);
    uint32_t q0 = 0;
    for (; q0 + U <= n; q0 += U) {
        V xv[U][B];
#pragma unroll
        for (int q = 0; q < U; ++q) ld_vec<B>(x + (size_t)(ls.base[q0 + q] + w.r_lo) * B, xv[q], false);
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const V c = ls.c[q0 + q];
#pragma unroll
            for (int r = 0; r < B; ++r) acc[r] = fma(c, xv[q][r], acc[r]);
        }
    }
    for (; q0 < n; ++q0) {
        V xv[B];
        ld_vec<B>(x + (size_t)(ls.base[q0] + w.r_lo) * B, xv, false);
        const V c = ls.c[q0];
#pragma unroll
        for (int r = 0; r < B; ++r) acc[r] = fma(c, xv[r], acc[r]);
    }
}

// Cross bonds of row w.
template <typename V, int B, int C>
__device__ __forceinline__ void spin_list_cross(const SectorTables &s, const SpinDev &p, const uint16_t *s_tlo,
                                                const V *s_J, const V *s_cf, const SpinList<V> &ls,
                                                const V *__restrict__ x, const SpinRow &w, V (&acc)[B], V &diag)
{
    const uint32_t e_hh = p.n_ll + p.n_hh;
    auto bond = [&](uint32_t b, const V *&cf, V &J, uint32_t &k0, uint32_t &k1) {
        const uint4 e = ls.cross[b];
        cf = s_cf + (((uint32_t)(w.dig >> (e.x & 255u)) & 15u) * p.d + (e.x >> 8));
        J = s_J[e_hh + b];
        k0 = e.z + s_tlo[min(w.lo - e.y, s.lomask)];
        k1 = e.w + s_tlo[min(w.lo + e.y, s.lomask)];
    };
    spin_bonds<V, B, C>(0u, p.nb - e_hh, bond, x, acc, diag);
}

// Row t: acc[r] = sum of the ladder terms of vector r, diag = sum_b J_b m_i m_j.  The 32
// lanes of the warp call it together, on increasing rows; ls is the warp's own, unused
// unless lists is set.
template <typename V, int B, int C>
__device__ __forceinline__ void spin_row(const SectorTables &s, const SpinDev &p, const uint16_t *s_tlo,
                                         const uint4 *s_bond, const V *s_J, const V *s_cf, const SpinList<V> &ls,
                                         bool lists, const V *__restrict__ x, uint32_t t, V (&acc)[B], V &diag)
{
    SpinRow w;
    spin_unrank(s, p, t, w);
    diag = (V)0;
#pragma unroll
    for (int r = 0; r < B; ++r) acc[r] = (V)0;
    const uint32_t e_ll = p.n_ll, e_hh = p.n_ll + p.n_hh;
    spin_class<V, B, C, 0>(s, p, s_tlo, s_bond, s_J, s_cf, x, w, 0u, e_ll, acc, diag);
    if (lists && __shfl_sync(~0u, w.hi, 0) == __shfl_sync(~0u, w.hi, 31)) {
        const uint32_t n = spin_list_fill<V>(s, p, s_bond, s_J, s_cf, w, ls);
        spin_list_hh<V, B, (B >= 16 ? 2 : 8)>(p, s_J, ls, n, x, w, acc, diag);
        spin_list_cross<V, B, C>(s, p, s_tlo, s_J, s_cf, ls, x, w, acc, diag);
    } else {
        spin_class<V, B, C, 1>(s, p, s_tlo, s_bond, s_J, s_cf, x, w, e_ll, e_hh, acc, diag);
        spin_class<V, B, C, 2>(s, p, s_tlo, s_bond, s_J, s_cf, x, w, e_hh, p.nb, acc, diag);
    }
}

}  // namespace ftlm
