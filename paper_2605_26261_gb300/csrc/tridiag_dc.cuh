// Symmetric tridiagonal eigenproblem in FP64 by divide and conquer, one CTA per
// problem: every eigenvalue and the first component of every eigenvector (the Ritz
// step, a5).
//
// Method.  Cuppen's rank-one tearing (Cuppen 1981) down to 1 x 1 blocks: with
// rho = |e| at a cut, T = diag(T_1', T_2') + rho v v^T, so a merge of two solved blocks
// is the eigenproblem of D + rho z z^T, z = (last row of Q_1, first row of Q_2).
// Components with a negligible z and pairs of close d are deflated (Dongarra &
// Sorensen 1987); the roots of 1/rho + sum_j z_j^2 / (d_j - x) are found one per
// thread by rational interpolation of the two half sums (Bunch, Nielsen & Sorensen
// 1978; Li 1994) inside a shrinking bracket, as offsets from the nearer pole, and the
// eigenvectors are those of the z recomputed from the roots, which makes them
// orthogonal to working accuracy (Gu & Eisenstat 1995).  Only the first and last row
// of the eigenvector matrix are carried: the last one feeds the z of the next merge,
// the first one squared is the weight.  A sign of e only flips signs of eigenvector
// components, so |e| is used.
//
// Bound: FP64 instructions (two lanes per cycle and SM).  Per root of a merge of n
// poles four passes over the poles remain: a float estimate (not on the FP64 pipe)
// leaves two double steps, then z and the rows take one pass each, about 37 FP64
// instructions per pole and root; the merges of all levels cost twice the last one.
// Measured on GB300, rows of Lanczos coefficients, against implicit QR with one thread
// per problem (a chain of about m^2 dependent rotations), n problems of m rows: m = 100,
// n = 8 / 690 / 4096: 21.2 / 21.3 / 21.3 ms -> 0.56 / 1.7 / 9.0 ms; m = 20, n = 8: 0.97
// -> 0.15 ms; m = 300, n = 8: 180 -> 5.1 ms; only for tens of thousands of problems at
// once is QR as fast.  Without the float estimate (doubles from the middle of the gap)
// 1.6 ms at m = 100, n = 8; with the half-sum steps alone 0.96 ms, 10 to 18 double steps for
// one or two roots of the last merge.
//
// Every step is a phase executed by all threads between two barriers, written as a
// function of (thread, thread count), so that the same code runs on the host, one
// thread after another, where its results can be compared with LAPACK.
#pragma once

#include <cmath>
#include <cstdint>

namespace ftlm {
namespace dc {

constexpr int kMaxIter = 100;  // secular iterations per root (a few are needed)

// Shared-memory arrays of one problem, `m` entries each.  d, f, l: eigenvalues, first
// and last eigenvector components of the solved blocks; ds .. ls: the same in sorted
// order, then the merged block's new values; z: the merge vector, then the recomputed
// one; tau: root offsets; e: the couplings.  dh + dl: d as the sum of two floats, zh: z
// as a float.  org: pole a root is measured from; cnt: entries that stay of the block
// that starts at an index; keep, pair: flags of the deflation.
struct Work {
    double *d, *f, *l, *z, *ds, *fs, *ls, *zs, *tau, *e;
    float *dh, *dl, *zh;
    int *org, *cnt, *keep, *pair;
    int m;
};
constexpr size_t kBytesPerRow = 10 * sizeof(double) + 3 * sizeof(float) + 4 * sizeof(int);

__host__ __device__ inline Work carve(void *p, int m)
{
    Work w;
    double *q = static_cast<double *>(p);
    double **const arr[10] = {&w.d, &w.f, &w.l, &w.z, &w.ds, &w.fs, &w.ls, &w.zs, &w.tau, &w.e};
    for (int i = 0; i < 10; ++i) *arr[i] = q + (size_t)i * m;
    w.dh = reinterpret_cast<float *>(q + (size_t)10 * m);
    w.dl = w.dh + m;
    w.zh = w.dl + m;
    w.org = reinterpret_cast<int *>(w.zh + m);
    w.cnt = w.org + m;
    w.keep = w.cnt + m;
    w.pair = w.keep + m;
    w.m = m;
    return w;
}

// 1 / x within one unit in the last place for 2^-1021 <= |x| <= 2^1021 (NaN for subnormal x and zero):
// the Newton-Raphson iteration r (2 - x r) for the reciprocal, two steps from the PTX ISA's
// rcp.approx.ftz.f64, whose error of about 2^-20 they square twice.  No branch and four FP64
// instructions; with 1.0 / x the Ritz step of 8 / 690 chains of m = 100 takes 0.60 / 2.50 ms
// instead of 0.56 / 1.66.
__host__ __device__ __forceinline__ double recip(double x)
{
#ifdef __CUDA_ARCH__
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
#else
    return 1.0 / x;
#endif
}

__host__ __device__ __forceinline__ float recip(float x)
{
#ifdef __CUDA_ARCH__
    return __fdividef(1.f, x);
#else
    return 1.f / x;
#endif
}

// Order-preserving integer image of a double (comparisons off the FP64 pipe).
__host__ __device__ __forceinline__ long long order_key(double x)
{
#ifdef __CUDA_ARCH__
    const long long b = __double_as_longlong(x);
#else
    long long b;
    memcpy(&b, &x, 8);
#endif
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// The block of width 2 s that index i belongs to: [lo, hi), cut at mid; a merge
// happens when mid < hi.
struct Span {
    int lo, mid, hi;
};
__host__ __device__ __forceinline__ Span span_of(int i, int s, int m)
{
    Span p;
    p.lo = i / (2 * s) * (2 * s);
    p.mid = p.lo + s < m ? p.lo + s : m;
    p.hi = p.lo + 2 * s < m ? p.lo + 2 * s : m;
    return p;
}

// Couplings below this are taken as zero (the largest coefficient is about one): they move
// no eigenvalue by more.  In a block of this scale s the distances between poles and roots
// are at least s 2^-110, so every reciprocal, and the square of one, stays in range.
constexpr double kNoCoupling = 0x1p-400;

// Phase 0: leaves of the tearing (w.d and w.e hold the matrix on entry, e[k] couples
// k and k + 1 and is replaced by its absolute value).
__host__ __device__ inline void leaf_abs(const Work &w, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        const double e = i + 1 < w.m ? fabs(w.e[i]) : 0.0;
        w.e[i] = e >= kNoCoupling ? e : 0.0;
    }
}
__host__ __device__ inline void leaf_tear(const Work &w, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        w.d[i] -= (i > 0 ? w.e[i - 1] : 0.0) + w.e[i];
        w.f[i] = 1.0;
        w.l[i] = 1.0;
    }
}

// Phase 1: every entry of a merged block to its place in ascending order of d, with
// its z (normalized: |z| = 1) and its rows of blkdiag(Q_1, Q_2).
__host__ __device__ inline void sort_block(const Work &w, int s, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        const Span p = span_of(i, s, w.m);
        const long long k = order_key(w.d[i]);
        int r = p.lo;
#pragma unroll 4
        for (int j = p.lo; j < p.hi; ++j) {
            const long long q = order_key(w.d[j]);
            r += (q < k) | ((q == k) & (j < i));
        }
        const bool left = i < p.mid;
        const bool merge = p.mid < p.hi;
        w.ds[r] = w.d[i];
        w.zs[r] = (left ? w.l[i] : w.f[i]) * 0.70710678118654752440;
        w.fs[r] = (left || !merge) ? w.f[i] : 0.0;
        w.ls[r] = (left && merge) ? 0.0 : w.l[i];
    }
}

// Deflation tolerance of a merged block.
__host__ __device__ __forceinline__ double deflation_tol(const Work &w, const Span &p)
{
    return 4.0 * 0x1p-52 * (fmax(fabs(w.ds[p.lo]), fabs(w.ds[p.hi - 1])) + 2.0 * w.e[p.mid - 1]);
}

// Phase 2a: entries whose z is not negligible.
__host__ __device__ inline void mark_small(const Work &w, int s, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        const Span p = span_of(i, s, w.m);
        w.keep[i] = p.mid < p.hi && 2.0 * w.e[p.mid - 1] * fabs(w.zs[i]) > deflation_tol(w, p);
        w.pair[i] = 0;
    }
}

// Whether two neighbouring entries of the merged block are so close that a rotation
// makes one of their z negligible.
__host__ __device__ __forceinline__ bool close_pair(double gap, double z0, double z1, double tol)
{
    return fabs(gap * z0 * z1) <= tol * fma(z0, z0, z1 * z1);
}

// Phase 2b: does a block have a close pair among the entries that stay?
__host__ __device__ inline void mark_pairs(const Work &w, int s, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        if (!w.keep[i]) continue;
        const Span p = span_of(i, s, w.m);
        int j = i - 1;
        while (j >= p.lo && !w.keep[j]) --j;
        if (j >= p.lo && close_pair(w.ds[i] - w.ds[j], w.zs[j], w.zs[i], deflation_tol(w, p))) w.pair[p.lo] = 1;
    }
}

// Phase 2c: entries that stay are packed at the front of the block in d, z, f, l
// (ascending d), deflated ones at its back.  A block without a close pair is packed by
// all its threads; one with a close pair by its first thread, one entry after another
// (a rotated pair may be close to the next entry).
__host__ __device__ inline void deflate(const Work &w, int s, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        const Span p = span_of(i, s, w.m);
        if (!w.pair[p.lo]) {
            int before = 0;
#pragma unroll 4
            for (int j = p.lo; j < i; ++j) before += w.keep[j];
            const int to = w.keep[i] ? p.lo + before : p.hi - 1 - (i - p.lo - before);
            w.d[to] = w.ds[i];
            w.z[to] = w.zs[i];
            w.f[to] = w.fs[i];
            w.l[to] = w.ls[i];
            if (i == p.hi - 1) w.cnt[p.lo] = before + w.keep[i];
            continue;
        }
        if (i != p.lo) continue;
        const double rho = 2.0 * w.e[p.mid - 1];
        const double tol = deflation_tol(w, p);
        int k = p.lo, back = p.hi;
        // (cd, cz, cf, cl): the last entry that stays, not yet written
        bool have = false;
        double cd = 0.0, cz = 0.0, cf = 0.0, cl = 0.0;
        for (int j = p.lo; j < p.hi; ++j) {
            double d = w.ds[j], z = w.zs[j], f = w.fs[j], l = w.ls[j];
            if (!(rho * fabs(z) > tol)) {
                --back;
                w.d[back] = d;
                w.f[back] = f;
                w.l[back] = l;
                continue;
            }
            if (have) {
                if (close_pair(d - cd, cz, z, tol)) {
                    // a rotation moves the pair's z to this entry and deflates the other
                    const double q2 = fma(cz, cz, z * z);
                    const double ir = rsqrt(q2), c = z * ir, sn = cz * ir;
                    const double dn = fma(c * c, d, sn * sn * cd), dp = fma(sn * sn, d, c * c * cd);
                    --back;
                    w.d[back] = dp;
                    w.f[back] = c * cf - sn * f;
                    w.l[back] = c * cl - sn * l;
                    f = sn * cf + c * f;
                    l = sn * cl + c * l;
                    d = dn;
                    z = q2 * ir;
                } else {
                    w.d[k] = cd;
                    w.z[k] = cz;
                    w.f[k] = cf;
                    w.l[k] = cl;
                    ++k;
                }
            }
            have = true;
            cd = d;
            cz = z;
            cf = f;
            cl = l;
        }
        if (have) {
            w.d[k] = cd;
            w.z[k] = cz;
            w.f[k] = cf;
            w.l[k] = cl;
            ++k;
        }
        w.cnt[p.lo] = k - p.lo;
    }
}

// The half sums of the secular function at x = d[o] + tau and their derivatives:
// psi over the poles lo .. cut, phi over cut + 1 .. hi - 1.
template <typename F> struct Halves {
    F psi, dpsi, phi, dphi;
};
template <typename F> __host__ __device__ __forceinline__ void add_term(F z, F q, F &s, F &ds)
{
    s = fma(z, q, s);
    ds = fma(q, q, ds);
}
// The poles of a warp's blocks in three ranges, so that its lanes, whose cuts differ by
// a few poles, run the same loops: below every cut psi, above every cut phi, between
// them both with the other one's term selected away.  lo0, hi0: smallest and largest
// cut of the warp, counted from the start of the lane's block.
struct Cuts {
    int lo0, hi0;
};
__host__ __device__ __forceinline__ Cuts warp_cuts(int rel)
{
#ifdef __CUDA_ARCH__
    const unsigned on = __activemask();
    return {__reduce_min_sync(on, rel), __reduce_max_sync(on, rel)};
#else
    return {rel, rel};
#endif
}
template <typename F, typename Delta>
__host__ __device__ __forceinline__ Halves<F> half_sums(const F *z, int lo, int cut, int hi, Cuts c, Delta &&inv)
{
    Halves<F> h{(F)0, (F)0, (F)0, (F)0};
    const int e0 = lo + c.lo0 + 1, e1 = lo + c.hi0 + 1 < hi ? lo + c.hi0 + 1 : hi;
    int j = lo;
#pragma unroll 4
    for (; j < e0; ++j) add_term(z[j], z[j] * inv(j), h.psi, h.dpsi);
#pragma unroll 4
    for (; j < e1; ++j) {
        const F q = z[j] * inv(j), p = j <= cut ? q : (F)0, r = j <= cut ? (F)0 : q;
        add_term(z[j], p, h.psi, h.dpsi);
        add_term(z[j], r, h.phi, h.dphi);
    }
#pragma unroll 4
    for (; j < hi; ++j) add_term(z[j], z[j] * inv(j), h.phi, h.dphi);
    return h;
}
__host__ __device__ __forceinline__ Halves<double> secular(const Work &w, int lo, int cut, int hi, Cuts c, int o,
                                                           double tau)
{
    const double *d = w.d, dorg = w.d[o];
    return half_sums<double>(w.z, lo, cut, hi, c, [=](int j) { return recip((d[j] - dorg) - tau); });
}
// The same in floats (differences of the two-float images keep their relative accuracy).
__host__ __device__ __forceinline__ Halves<float> secular(const Work &w, int lo, int cut, int hi, Cuts c, int o,
                                                          float tau)
{
    const float *dh = w.dh, *dl = w.dl, oh = w.dh[o], ol = w.dl[o];
    return half_sums<float>(w.zh, lo, cut, hi, c,
                            [=](int j) { return recip(((dh[j] - oh) + (dl[j] - ol)) - tau); });
}

// Step from x of the rational model c + S/(d_a - x) + R/(d_b - x) with the value w = f(x)
// (da = d_a - x, db = d_b - x): the root eta of c eta^2 - A eta + da db w = 0 between
// the two poles (last: to the right of both).
template <typename F>
__host__ __device__ __forceinline__ F model_root(F c, F S, F R, F da, F db, F w, bool last)
{
    const F A = fma(c, da + db, S + R);
    const F B = da * db * w;
    const F disc = sqrt(fmax((F)0, fma(A, A, (F)-4 * c * B)));
    const F sd = last ? -disc : disc;
    const bool minus = last ? A >= (F)0 : A <= (F)0;  // the quotient without cancellation
    return (minus ? A - sd : (F)2 * B) * recip(minus ? (F)2 * c : A + sd);
}
// The weights that match both half sums and their derivatives (Bunch, Nielsen & Sorensen).
template <typename F>
__host__ __device__ __forceinline__ F rational_step(const Halves<F> &h, F da, F db, F w, bool last)
{
    return model_root<F>(w - da * h.dpsi - db * h.dphi, da * da * h.dpsi, db * db * h.dphi, da, db, w, last);
}
// The near pole's own weight z^2 (near_z: z of pole a if near_a, else of b), the other one
// matching the rest of the derivative (Li 1994).  The step above attributes far poles' part
// of the derivative to a near pole of tiny z and then only halves the distance; this one
// is exact there.  Ghosts of Lanczos coefficients have such roots in the last merges.
template <typename F>
__host__ __device__ __forceinline__ F fixed_step(const Halves<F> &h, F da, F db, F w, bool last, bool near_a, F near_z)
{
    const F dn = near_a ? da : db, df = near_a ? db : da;
    const F q = near_z * recip(dn), rest = fmax((F)0, h.dpsi + h.dphi - q * q);
    const F zz = near_z * near_z, rr = df * df * rest;
    return model_root<F>(w - near_z * q - df * rest, near_a ? zz : rr, near_a ? rr : zz, da, db, w, last);
}

// A point inside a bracket: one that reaches the pole is cut by a factor, not by its
// middle.
template <typename F> __host__ __device__ __forceinline__ F cut(F lb, F ub)
{
    return lb == (F)0 ? (F)0.0625 * ub : (ub == (F)0 ? (F)0.0625 * lb : (F)0.5 * (lb + ub));
}

// A float estimate of the root between poles a and b (last: above b) and the pole to
// measure it from.  Nothing depends on its quality but the number of double steps
// that follow: three digits or more in a few steps.
__host__ __device__ inline float root_estimate(const Work &w, int lo, int hi, int a, int b, bool last, Cuts c,
                                               float rho, int &o)
{
    const float irho = 1.f / rho;
    float x, lb = 0.f, ub = 0.f;  // bracket, as offsets from pole o
    if (last) {
        o = b;
        x = 0.5f * rho;
        ub = rho * 1.01f;
    } else {
        const float half = 0.5f * ((w.dh[b] - w.dh[a]) + (w.dl[b] - w.dl[a]));
        const Halves<float> h = secular(w, lo, a, hi, c, a, half);
        const float v = irho + h.psi + h.phi;
        // f rises from -inf at d[a] to +inf at d[b]: the sign at the middle tells the
        // nearer pole
        o = v >= 0.f ? a : b;
        lb = v >= 0.f ? 0.f : -half;
        ub = v >= 0.f ? half : 0.f;
        x = (v >= 0.f ? half : -half) + rational_step(h, -half, half, v, false);
    }
    const float x0 = 0.5f * (lb + ub);
    for (int it = 0; it < 16; ++it) {
        const float da = ((w.dh[a] - w.dh[o]) + (w.dl[a] - w.dl[o])) - x;
        const float db = ((w.dh[b] - w.dh[o]) + (w.dl[b] - w.dl[o])) - x;
        const Halves<float> h = secular(w, lo, a, hi, c, o, x);
        const float v = irho + h.psi + h.phi;
        if (it < 4) {
            const float eta = rational_step(h, da, db, v, last);
            x += eta;
            if (!(fabs(eta) > 1e-4f * fabs(x))) break;
            if (it == 3 && !(x > lb && x < ub)) x = x0;
        } else {  // one of the slow roots: inside the bracket from here on
            if (v < 0.f) lb = x;
            else ub = x;
            float y = x + fixed_step(h, da, db, v, last, o == a, w.zh[o]);
            if (!(y > lb && y < ub)) y = cut(lb, ub);
            const bool done = fabs(y - x) <= 1e-4f * fabs(y);
            x = y;
            if (done) break;
        }
    }
    return x;
}

// Root `i` of the block with poles lo .. hi-1: its pole `o` and offset tau.  Returns
// false when the iteration limit was reached.
__host__ __device__ inline bool secular_root(const Work &w, int lo, int hi, int i, double rho, int &o, double &tau)
{
    const int n = hi - lo;
    if (n == 1) {
        o = lo;
        tau = rho * w.z[lo] * w.z[lo];
        return true;
    }
    const double irho = 1.0 / rho;
    const bool last = i == hi - 1;
    const int a = last ? i - 1 : i, b = a + 1;  // poles of the model; psi ends at a
    const Cuts c = warp_cuts(a - lo);
    double x = root_estimate(w, lo, hi, a, b, last, c, (float)rho, o);
    double dorg = w.d[o];
    // bracket, as offsets from d[o]
    double lb = o == a ? 0.0 : (last ? 0.0 : w.d[a] - dorg);
    double ub = last ? rho * (1.0 + 0x1p-30) : (o == a ? w.d[b] - dorg : 0.0);  // |z| <= 1 up to rounding
    if (!(x > lb && x < ub)) x = 0.5 * (lb + ub);
    double prev = INFINITY;
    for (int it = 0; it < kMaxIter; ++it) {
        const Halves<double> h = secular(w, lo, a, hi, c, o, x);
        const double v = irho + h.psi + h.phi;
        tau = x;
        if (v != v) return false;
        if (v < 0.0) lb = x;
        else ub = x;
        // rounding level of f at x (Gu & Eisenstat's stopping rule)
        const bool small = fabs(v) <= 0x1p-52 * n * (irho + fabs(h.psi) + fabs(h.phi));
        const double da = (w.d[a] - dorg) - x, db = (w.d[b] - dorg) - x;
        // after a step that left more than a tenth of f, one with the near pole's own weight
        const bool slow = !(fabs(v) <= 0.1 * prev);
        prev = fabs(v);
        const double eta = slow && it > 0 ? fixed_step(h, da, db, v, last, o == a, w.z[o])
                                          : rational_step(h, da, db, v, last);
        double y = x + eta;
        if (!(y > lb && y < ub)) {
            y = cut(lb, ub);
            if (small || !(y > lb && y < ub)) return true;  // converged, or the bracket has closed
        } else if (!last && 4.0 * fabs(o == a ? db - eta : da - eta) < fabs(y)) {
            // the root is next to the other pole: measured from there its offset keeps
            // its relative accuracy
            o = o == a ? b : a;
            const double shift = w.d[o] - dorg;
            dorg = w.d[o];
            lb -= shift;
            ub -= shift;
            y -= shift;
            if (!(y > lb && y < ub)) y = cut(lb, ub);
            x = y;
            continue;
        } else if (small || fabs(eta) <= 0x1p-30 * fmin(fabs(da), fabs(db))) {
            // the steps converge quadratically: the next one would be below rounding
            tau = y;
            return true;
        }
        if (y == x) return true;
        x = y;
    }
    return false;
}

// Phase 3a: float images of the poles and of z.
__host__ __device__ inline void float_images(const Work &w, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        const float h = (float)w.d[i];
        w.dh[i] = h;
        w.dl[i] = (float)(w.d[i] - (double)h);
        w.zh[i] = (float)w.z[i];
    }
}

// Phase 3: the roots.  Returns false if one did not converge.
__host__ __device__ inline bool roots(const Work &w, int s, int t, int T)
{
    bool ok = true;
    for (int i = t; i < w.m; i += T) {
        const Span p = span_of(i, s, w.m);
        const int hi = p.lo + w.cnt[p.lo];
        if (i >= hi) continue;
        int o;
        double tau;
        ok &= secular_root(w, p.lo, hi, i, 2.0 * w.e[p.mid - 1], o, tau);
        w.org[i] = o;
        w.tau[i] = tau;
    }
    return ok;
}

// Phase 4: the z whose secular equation has exactly these roots,
// z_j^2 ~ prod_i (x_i - d_j) / prod_{i != j} (d_i - d_j), each root paired with a pole
// next to it so that the partial products stay near one.
__host__ __device__ inline void refit(const Work &w, int s, int t, int T)
{
    for (int j = t; j < w.m; j += T) {
        const Span p = span_of(j, s, w.m);
        const int hi = p.lo + w.cnt[p.lo];
        if (j >= hi) continue;
        const double dj = w.d[j];
        double q = (w.d[w.org[hi - 1]] - dj) + w.tau[hi - 1];
#pragma unroll 4
        for (int i = p.lo; i < hi - 1; ++i)
            q *= ((w.d[w.org[i]] - dj) + w.tau[i]) * recip(w.d[i + (i >= j)] - dj);
        w.zs[j] = copysign(sqrt(fabs(q)), w.z[j]);
    }
}

// Phase 5: first and last row of the merged block's eigenvectors, and its eigenvalues,
// into ds, fs, ls.
__host__ __device__ inline void rows(const Work &w, int s, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        const Span p = span_of(i, s, w.m);
        const int hi = p.lo + w.cnt[p.lo];
        if (i >= hi) {
            w.ds[i] = w.d[i];
            w.fs[i] = w.f[i];
            w.ls[i] = w.l[i];
            continue;
        }
        const double dorg = w.d[w.org[i]], tau = w.tau[i];
        double nn = 0.0, fn = 0.0, ln = 0.0;
#pragma unroll 4
        for (int j = p.lo; j < hi; ++j) {
            const double u = w.zs[j] * recip((w.d[j] - dorg) - tau);
            nn = fma(u, u, nn);
            fn = fma(u, w.f[j], fn);
            ln = fma(u, w.l[j], ln);
        }
        const double ir = rsqrt(nn);
        w.ds[i] = dorg + tau;
        w.fs[i] = fn * ir;
        w.ls[i] = ln * ir;
    }
}
__host__ __device__ inline void commit(const Work &w, int t, int T)
{
    for (int i = t; i < w.m; i += T) {
        w.d[i] = w.ds[i];
        w.f[i] = w.fs[i];
        w.l[i] = w.ls[i];
    }
}

}  // namespace dc
}  // namespace ftlm
