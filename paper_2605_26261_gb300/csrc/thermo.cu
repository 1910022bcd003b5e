// FTLM thermodynamic sums (step a6, Eq. 6-9), FP64 on the device.
//
// Every (sector image, chain, Ritz pair) contributes weight (D/R) w_k at energy
// E = theta_k - h S^z (Zeeman term -h S^z) and magnetization S^z; sectors with
// S^z > 0 also stand for -S^z when mirroring is on (identical spectra, Sec. 2).
// With E0 the lowest energy:
//   Z = sum b,  b = (D/R) w e^{-beta (E - E0)}       (Eq. 7, shifted by E0)
//   <E - E0> = sum b (E - E0) / Z,  Var(H) = sum b (E - E0 - <E - E0>)^2 / Z
//   <S^z> = sum b S^z / Z,  <(S^z)^2> = sum b (S^z)^2 / Z,
//   Var(S^z) = sum b (S^z - <S^z>)^2 / Z
// and C = beta^2 Var(H) (Eq. 8 moments, central form), chi = g^2 beta <(S^z)^2>
// at h = 0 (Eq. 9) and g^2 beta Var(S^z) otherwise.  The shift keeps e^{-beta E}
// finite at T = 0.01 and cancels in every ratio; the central second moment avoids
// the cancellation of <H^2> - <H>^2 at high T.
//
// Per sector: with t_s its lowest Ritz value, p = w e^{-beta (theta - t_s)} is the same
// for the sector and its mirror image, which differ by the factor
// G = (D/R) e^{-beta (t_s - h S^z - E0)}.  A first pass over the pairs forms
// a0 = sum p and a1 = sum p (theta - t_s), a second one the sector's own central moment
// a2 = sum p (theta - t_s - a1/a0)^2; every observable is a sum over sectors and images
// of a0, a1, a2 (the variance as the sum of the variances inside and between them, all
// terms positive).
//
// Bound: the FP64 pipe (two lanes per cycle and SM), an exponential being about 20 of
// its instructions.  One exponential per pair and temperature instead of four (two
// images, two passes), kept in shared memory for the second pass where it fits, and a
// cluster of CTAs per temperature, whose partial sums meet in distributed shared
// memory, so that 200 temperatures spread evenly over 152 SMs.  Measured on GB300, 200
// temperatures, against one CTA per temperature and an exponential per image and pass:
// 11 sectors x 16 chains x 100 pairs 1.13 -> 0.35 ms, 13 x 24 x 100 1.99 -> 0.62 ms, 13 x 64
// x 150 7.9 -> 2.6 ms.  Every sum has a fixed order, so results are reproducible.
#include <algorithm>
#include <cmath>

#include <cooperative_groups.h>

#include "ftlm_internal.cuh"
#include "reduce.cuh"
#include "tridiag_dc.cuh"

namespace ftlm {

namespace {

constexpr int kThermoThreads = 256;
// Shared memory for the weights of a CTA's pairs: two CTAs per SM with clusters of 4,
// one with clusters of 8.
constexpr uint64_t kThermoSmall = 2048;
constexpr size_t kThermoStore4 = 88 << 10, kThermoStore8 = 192 << 10;

struct ThermoArgs {
    int ns, R, M, mirror;
    double g, h;
    const double *theta[FTLM_MAX_SECTORS];
    const double *weight[FTLM_MAX_SECTORS];
    const int *meff[FTLM_MAX_SECTORS];
    double wscale[FTLM_MAX_SECTORS];  // D / R
    double sz[FTLM_MAX_SECTORS];      // S^z
};

constexpr int kThermoWarps = kThermoThreads / 32;

// Sums of the warps of a CTA for every sector, read by the other CTAs of the cluster.
struct SectorSums {
    double v[FTLM_MAX_SECTORS][kThermoWarps][2];
};

// Cluster-wide totals of sector s by one warp, a lane per warp of the cluster: the first
// in lane 0, the second in lane 1.
template <int C>
__device__ __forceinline__ double cluster_totals(cooperative_groups::cluster_group &cl, SectorSums &sums, int s)
{
    DotAcc<double> t[2];
    for (int k = (int)(threadIdx.x & 31u); k < C * kThermoWarps; k += 32) {
        const SectorSums *r = cl.map_shared_rank(&sums, k / kThermoWarps);
        t[0].v += r->v[s][k % kThermoWarps][0];
        t[1].v += r->v[s][k % kThermoWarps][1];
    }
    return warp_sum_multi<double, 2>(t).v;
}

// Warp sums of two accumulators, to slot [s][warp] of the CTA's sums.
__device__ __forceinline__ void warp_pair(SectorSums &sums, int s, double x, double y)
{
    DotAcc<double> a[2];
    a[0].v = x;
    a[1].v = y;
    const DotAcc<double> t = warp_sum_multi<double, 2>(a);
    const unsigned lane = threadIdx.x & 31u;
    if (lane < 2) sums.v[s][threadIdx.x >> 5][warp_multi_index<2>(lane)] = t.v;
}

// One cluster of C CTAs per temperature.  STORE: the weights p of a thread's pairs stay
// in shared memory between the passes.
template <int C, bool STORE>
__global__ void __launch_bounds__(kThermoThreads)
thermo_kernel(const ThermoArgs a, const double *__restrict__ T, double *E, double *C_out, double *chi, double *mag,
              double *Zs, double *E0s)
{
    extern __shared__ double s_p[];
    __shared__ SectorSums sums;
    __shared__ long long s_min[FTLM_MAX_SECTORS];  // order_key of t_s over this CTA's pairs
    __shared__ int s_any[FTLM_MAX_SECTORS];
    __shared__ double s_t[FTLM_MAX_SECTORS], s_mu[FTLM_MAX_SECTORS], s_a[FTLM_MAX_SECTORS][2],
        s_a2[FTLM_MAX_SECTORS], s_G[FTLM_MAX_SECTORS][2];
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const unsigned lane = threadIdx.x & 31u;
    // unsigned: with up to 2^31 - 1 pairs the index of a thread's last step passes 2^31
    const unsigned M = (unsigned)a.M, per_sector = (unsigned)a.R * M;
    const unsigned first = cl.block_rank() * kThermoThreads + threadIdx.x;  // pairs first, first + 256 C, ...
    constexpr unsigned kStep = kThermoThreads * C;
    const double beta = 1.0 / T[blockIdx.x / C];
    const long long inf_key = dc::order_key(INFINITY);

    for (int s = threadIdx.x; s < a.ns; s += kThermoThreads) {
        s_min[s] = inf_key;
        s_any[s] = 0;
    }
    __syncthreads();
    for (int s = 0; s < a.ns; ++s) {
        long long m = inf_key;
        int any = 0;
        for (unsigned i = first; i < per_sector; i += kStep) {
            const unsigned r = i / M;
            if ((int)(i - r * M) >= __ldg(a.meff[s] + r)) continue;
            m = min(m, dc::order_key(__ldg(a.theta[s] + i)));
            any = 1;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(0xffffffffu, m, o));
        any = __any_sync(0xffffffffu, any);
        if (lane == 0 && any) {
            atomicMin(&s_min[s], m);
            s_any[s] = 1;
        }
    }
    cl.sync();
    for (int s = threadIdx.x; s < a.ns; s += kThermoThreads) {
        long long m = inf_key;
        int any = 0;
        for (int c = 0; c < C; ++c) {
            m = min(m, cl.map_shared_rank(s_min, c)[s]);
            any |= cl.map_shared_rank(s_any, c)[s];
        }
        // order_key is its own inverse on its sign bit; a sector whose values are all NaN
        // keeps a finite reference, and its weights become NaN below
        const double t = __longlong_as_double(m ^ ((m >> 63) & 0x7fffffffffffffffll));
        s_t[s] = any ? (m < inf_key ? t : 0.0) : INFINITY;
    }
    __syncthreads();

    int slot = (int)threadIdx.x;
    for (int s = 0; s < a.ns; ++s) {
        const double t = s_t[s];
        double x0 = 0.0, x1 = 0.0;
        for (unsigned i = first; i < per_sector; i += kStep) {
            const unsigned r = i / M;
            double p = 0.0;
            if ((int)(i - r * M) < __ldg(a.meff[s] + r)) {
                const double x = __ldg(a.theta[s] + i) - t;
                p = __ldg(a.weight[s] + i) * exp(-beta * x);
                x0 += p;
                x1 = fma(p, x, x1);
            }
            if (STORE) {
                s_p[slot] = p;
                slot += kThermoThreads;
            }
        }
        warp_pair(sums, s, x0, x1);
    }
    cl.sync();
    for (int s = (int)threadIdx.x >> 5; s < a.ns; s += kThermoWarps) {
        const double v = cluster_totals<C>(cl, sums, s);
        if (lane < 2) s_a[s][lane] = v;
        __syncwarp();
        if (lane == 0) s_mu[s] = s_a[s][0] != 0.0 ? s_a[s][1] / s_a[s][0] : 0.0;
    }
    cl.sync();  // every CTA has read the sums before they are written again

    slot = (int)threadIdx.x;
    for (int s = 0; s < a.ns; ++s) {
        const double t = s_t[s], mu = s_mu[s];
        double x2 = 0.0;
        for (unsigned i = first; i < per_sector; i += kStep) {
            const unsigned r = i / M;
            if ((int)(i - r * M) < __ldg(a.meff[s] + r)) {
                const double x = __ldg(a.theta[s] + i) - t;
                const double p = STORE ? s_p[slot] : __ldg(a.weight[s] + i) * exp(-beta * x);
                const double d = x - mu;
                x2 = fma(p * d, d, x2);
            }
            if (STORE) slot += kThermoThreads;
        }
        warp_pair(sums, s, x2, 0.0);
    }
    cl.sync();
    // the observables in warp 0 of the cluster's first CTA, sectors over its lanes
    if (cl.block_rank() == 0) {
        for (int s = (int)threadIdx.x >> 5; s < a.ns; s += kThermoWarps) {
            const double v = cluster_totals<C>(cl, sums, s);
            if (lane == 0) s_a2[s] = v;
        }
        __syncthreads();
    }
    if (cl.block_rank() == 0 && threadIdx.x < 32) {
        double e0 = INFINITY;
        for (int s = (int)lane; s < a.ns; s += 32) {
            const double hz = a.h * a.sz[s];
            e0 = fmin(e0, s_t[s] - hz);
            if (a.mirror && a.sz[s] > 0.0) e0 = fmin(e0, s_t[s] + hz);
        }
        for (int o = 16; o > 0; o >>= 1) e0 = fmin(e0, __shfl_xor_sync(0xffffffffu, e0, o));
        const double E0 = __shfl_sync(0xffffffffu, e0, 0);
        auto images = [&](auto &&f) {  // (sector, image, S^z, energy of t_s above E0)
            for (int s = (int)lane; s < a.ns; s += 32) {
                if (s_t[s] == INFINITY) continue;  // no pairs
                const int n = (a.mirror && a.sz[s] > 0.0) ? 2 : 1;
                for (int im = 0; im < n; ++im) {
                    const double mz = im ? -a.sz[s] : a.sz[s];
                    f(s, im, mz, s_t[s] - a.h * mz - E0);
                }
            }
        };
        DotAcc<double> m[4];  // Z, <E - E0> Z, <S^z> Z, <(S^z)^2> Z
        images([&](int s, int im, double mz, double off) {
            // without a field the images of a sector have one weight
            const double G = (im && a.h == 0.0) ? s_G[s][0] : a.wscale[s] * exp(-beta * off);
            s_G[s][im] = G;
            const double b = G * s_a[s][0];
            m[0].v += b;
            m[1].v += G * fma(off, s_a[s][0], s_a[s][1]);
            m[2].v += b * mz;
            m[3].v += b * mz * mz;
        });
        const double t4 = warp_sum_multi<double, 4>(m).v;  // accumulator 0, 2, 1, 3 in lanes 0 .. 3
        const double Z = __shfl_sync(0xffffffffu, t4, 0), rZ = 1.0 / Z;
        const double e1 = __shfl_sync(0xffffffffu, t4, 2) * rZ;
        const double M1 = __shfl_sync(0xffffffffu, t4, 1) * rZ;
        const double M2 = __shfl_sync(0xffffffffu, t4, 3) * rZ;
        DotAcc<double> c[2];
        images([&](int s, int im, double mz, double off) {
            const double dc = s_mu[s] + off - e1, dm = mz - M1, G = s_G[s][im];
            c[0].v += G * fma(s_a[s][0] * dc, dc, s_a2[s]);
            c[1].v += G * s_a[s][0] * dm * dm;
        });
        const double t2 = warp_sum_multi<double, 2>(c).v;
        const double S2 = __shfl_sync(0xffffffffu, t2, 0), V2 = __shfl_sync(0xffffffffu, t2, 1);
        if (lane == 0) {
            const int t = blockIdx.x / C;
            if (E) E[t] = E0 + e1;
            if (C_out) C_out[t] = beta * beta * (S2 * rZ);
            if (chi) chi[t] = a.g * a.g * beta * (a.h == 0.0 ? M2 : V2 * rZ);
            if (mag) mag[t] = M1;
            if (Zs) Zs[t] = Z;
            if (E0s) E0s[t] = E0;
        }
    }
    cl.sync();  // the other CTAs' sums stay in place until they have been read
}

template <int C, bool STORE>
ftlm_status launch_thermo_c(const ThermoArgs &a, int nT, size_t smem, const double *T, double *E, double *Co,
                            double *chi, double *mag, double *Z, double *E0, cudaStream_t stream)
{
    auto kern = thermo_kernel<C, STORE>;
    if (smem) {
        int occ = 1;
        FTLM_CUDA(kernel_occupancy((const void *)kern, kThermoThreads, kThermoStore8, true, &occ));
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)nT * C);
    cfg.blockDim = dim3(kThermoThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = C;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    FTLM_CUDA(cudaLaunchKernelEx(&cfg, kern, a, T, E, Co, chi, mag, Z, E0));
    note_launch();
    return FTLM_OK;
}

// One CTA for a few pairs, else clusters of 4 CTAs; of 8 when only then the weights of the pairs fit in shared memory
// (twice the exponentials else).
ftlm_status launch_thermo(const ThermoArgs &a, int nT, const double *T, double *E, double *Co, double *chi,
                          double *mag, double *Z, double *E0, cudaStream_t stream)
{
    auto store = [&](int c) {
        const uint64_t rounds = ((uint64_t)a.R * a.M + (uint64_t)kThermoThreads * c - 1) / ((uint64_t)kThermoThreads * c);
        return rounds * a.ns * kThermoThreads * sizeof(double);
    };
    if ((uint64_t)a.ns * a.R * a.M <= kThermoSmall)
        return launch_thermo_c<1, true>(a, nT, store(1), T, E, Co, chi, mag, Z, E0, stream);
    if (store(4) <= kThermoStore4)
        return launch_thermo_c<4, true>(a, nT, store(4), T, E, Co, chi, mag, Z, E0, stream);
    if (store(8) <= kThermoStore8)
        return launch_thermo_c<8, true>(a, nT, store(8), T, E, Co, chi, mag, Z, E0, stream);
    return launch_thermo_c<4, false>(a, nT, 0, T, E, Co, chi, mag, Z, E0, stream);
}

}  // namespace

}  // namespace ftlm

using namespace ftlm;

extern "C" ftlm_status ftlm_thermo(int n_sectors, const int *two_sz, const uint64_t *dims, int R, int M,
                                   const double *const *theta, const double *const *weight,
                                   const int *const *m_eff, int mirror_neg, double g, double h, int nT,
                                   const double *T_dev, double *E_dev, double *C_dev, double *chi_dev,
                                   double *mag_dev, void *stream)
{
    if (n_sectors < 1 || n_sectors > FTLM_MAX_SECTORS) return fail(FTLM_EINVAL, "n_sectors out of range");
    if (R < 1 || M < 1 || M > FTLM_MAX_LANCZOS) return fail(FTLM_EINVAL, "R or M out of range");
    if ((int64_t)n_sectors * R * M > (1ll << 31) - 1) return fail(FTLM_EUNSUPPORTED, "too many Ritz pairs");
    if (nT < 0) return fail(FTLM_EINVAL, "nT < 0");
    if (!two_sz || !dims || !theta || !weight || !m_eff) return fail(FTLM_EINVAL, "NULL host array");
    if (nT > 0 && (!T_dev || !E_dev || !C_dev || !chi_dev)) return fail(FTLM_EINVAL, "NULL device output");
    ThermoArgs a{};
    a.ns = n_sectors;
    a.R = R;
    a.M = M;
    a.mirror = mirror_neg != 0;
    a.g = g;
    a.h = h;
    for (int s = 0; s < n_sectors; ++s) {
        if (!theta[s] || !weight[s] || !m_eff[s]) return fail(FTLM_EINVAL, "NULL sector pointer");
        if (dims[s] == 0) return fail(FTLM_EINVAL, "zero sector dimension");
        a.theta[s] = theta[s];
        a.weight[s] = weight[s];
        a.meff[s] = m_eff[s];
        a.wscale[s] = (double)dims[s] / R;
        a.sz[s] = two_sz[s] / 2.0;
    }
    if (nT == 0) return FTLM_OK;
    return launch_thermo(a, nT, T_dev, E_dev, C_dev, chi_dev, mag_dev, nullptr, nullptr, (cudaStream_t)stream);
}

extern "C" ftlm_status ftlm_partition(int n_sectors, const int *two_sz, const uint64_t *dims, int R, int M,
                                      const double *const *theta, const double *const *weight,
                                      const int *const *m_eff, int mirror_neg, double h, int nT, const double *T_dev,
                                      double *Z_dev, double *E0_dev, void *stream)
{
    if (n_sectors < 1 || n_sectors > FTLM_MAX_SECTORS) return fail(FTLM_EINVAL, "n_sectors out of range");
    if (R < 1 || M < 1 || M > FTLM_MAX_LANCZOS) return fail(FTLM_EINVAL, "R or M out of range");
    if ((int64_t)n_sectors * R * M > (1ll << 31) - 1) return fail(FTLM_EUNSUPPORTED, "too many Ritz pairs");
    if (nT < 0) return fail(FTLM_EINVAL, "nT < 0");
    if (!two_sz || !dims || !theta || !weight || !m_eff) return fail(FTLM_EINVAL, "NULL host array");
    if (nT > 0 && (!T_dev || !Z_dev)) return fail(FTLM_EINVAL, "NULL device output");
    ThermoArgs a{};
    a.ns = n_sectors;
    a.R = R;
    a.M = M;
    a.mirror = mirror_neg != 0;
    a.g = 0.0;
    a.h = h;
    for (int s = 0; s < n_sectors; ++s) {
        if (!theta[s] || !weight[s] || !m_eff[s]) return fail(FTLM_EINVAL, "NULL sector pointer");
        if (dims[s] == 0) return fail(FTLM_EINVAL, "zero sector dimension");
        a.theta[s] = theta[s];
        a.weight[s] = weight[s];
        a.meff[s] = m_eff[s];
        a.wscale[s] = (double)dims[s] / R;
        a.sz[s] = two_sz[s] / 2.0;
    }
    if (nT == 0) return FTLM_OK;
    return launch_thermo(a, nT, T_dev, nullptr, nullptr, nullptr, nullptr, Z_dev, E0_dev, (cudaStream_t)stream);
}
