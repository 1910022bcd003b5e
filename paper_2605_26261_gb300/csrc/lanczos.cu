// Lanczos chains (steps a2, a4, a5): start vectors, the vector update, the Ritz
// step, and the launch sequence of ftlm_lanczos / ftlm_lanczos_from.
//
// Recurrence (Sec. 2, FTLM paragraph; Paige's ordering, no reorthogonalization):
//     y = H q_j - beta_{j-1} q_{j-1};  alpha_j = <q_j, y>;  w = y - alpha_j q_j;
//     beta_j = ||w||;  q_{j+1} = w / beta_j.
// Only two vectors per chain are stored.  The H.v launch (hv.cu) reads u_j and
// overwrites u_{j-1} with y; the update launch below overwrites y with w in place
// and publishes beta_j.  The division by beta_j is folded into the next H.v (the
// stored vectors stay un-normalized, q_j = u_j / s_j), so every step streams each
// vector exactly once per launch.  All scalars stay on the device; the host only
// queues 2 launches per step (3 for CR sectors, whose H.v launch leaves the sums of
// alpha_j for a launch of one warp, 4 where it runs as two walks), and a chain that
// breaks down (beta_j <= tau) turns the rest of its launches into no-ops.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include <cuda.h>

#include "epi.cuh"
#include "ftlm_internal.cuh"
#include "reduce.cuh"
#include "vec.cuh"
#include "rng.cuh"
#include "tridiag.cuh"
#include "tridiag_dc.cuh"

namespace ftlm {

namespace {

// The blocks of chains of a launch (blockIdx.y): bytes between their vectors, states,
// partials and counters; block k holds the chains that follow block k - 1's.
struct BlockSlots {
    uint64_t bytes;
};

// Keys of the start vectors: chain r of block k is keyed chain0 + k B + r.
struct KeySpec {
    uint64_t seed;
    int key_n, K, chain0;
};

// Start vectors of a block of B chains (generated, or copied from src rows of
// length D), interleaved, and s_1 = ||u|| of each chain's stored (dtype-rounded)
// entries.
template <typename V, int B>
__global__ void __launch_bounds__(kRowThreads)
start_kernel(uint32_t D, const KeySpec keys, int dist, const double *__restrict__ src, V *__restrict__ u,
             ChainState *st, double *partials, unsigned int *counter, const BlockSlots slots)
{
    u = block_ptr(u, slots.bytes);
    st = block_ptr(st, slots.bytes);
    partials = block_ptr(partials, slots.bytes);
    counter = block_ptr(counter, slots.bytes);
    if (src) src += (size_t)blockIdx.y * B * D;
    __shared__ uint64_t s_key[B];
    if (threadIdx.x < B)
        s_key[threadIdx.x] =
            chain_key(keys.seed, keys.key_n, keys.K, (uint32_t)keys.chain0 + blockIdx.y * B + threadIdx.x);
    __syncthreads();
    DotAcc<V> acc[B];
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < D; t += stride) {
        V out[B];
#pragma unroll
        for (int r = 0; r < B; ++r) {
            out[r] = src ? (V)src[(size_t)r * D + t] : start_entry<V>(s_key[r], t, dist);
            acc[r].add(out[r], out[r]);
        }
        st_vec<B>(u + (size_t)t * B, out);
    }
    const double v = block_sums<V, B, kRowThreads>(acc);
    if (publish_sums<B>(v, partials, counter)) {
        totals<B, kRowThreads>(partials, gridDim.x, [&](int r, double sum) {
            const double nrm = sqrt(sum);
            ChainState &c = st[r];
            c.s_cur = nrm;
            c.s_prev = 1.0;
            c.beta_prev = 0.0;
            c.alpha = 0.0;
            c.m_eff = 0;
            c.stopped = (nrm > 0.0 && isfinite(nrm)) ? 0 : 1;
        });
        if (threadIdx.x == 0) *counter = 0;
    }
}

// w = y - alpha_j q_j per chain (in place over y), beta_j = ||w||, breakdown test.
// Columns of chains that have ended are set to zero.  The block is processed in
// units of U = max(B, 16 bytes) values; entry e of a unit belongs to chain e % B.
template <typename V, int B>
__global__ void __launch_bounds__(kRowThreads)
update_kernel(uint32_t D, V *__restrict__ y, const V *__restrict__ u, ChainState *st, double *partials,
              unsigned int *counter, int j, int m_max, double tau, double *beta_out, int beta_stride,
              const BlockSlots slots)
{
    y = block_ptr(y, slots.bytes);
    u = block_ptr(u, slots.bytes);
    st = block_ptr(st, slots.bytes);
    partials = block_ptr(partials, slots.bytes);
    counter = block_ptr(counter, slots.bytes);
    beta_out += (size_t)blockIdx.y * B * beta_stride;
    // the per-chain scalars once per CTA: a division in every thread is 10 FP64
    // instructions per chain on a pipe of two lanes per cycle (40 us per launch at B = 8,
    // whatever D)
    __shared__ V s_a[B];
    __shared__ int s_zero[B];
    if (threadIdx.x < B) {
        const ChainState &c = st[threadIdx.x];
        s_zero[threadIdx.x] = c.stopped;
        s_a[threadIdx.x] = c.stopped ? (V)0 : (V)(c.alpha / c.s_cur);
    }
    __syncthreads();
    V a[B];
    bool zero[B];
    bool all_stopped = true;
#pragma unroll
    for (int r = 0; r < B; ++r) {
        zero[r] = s_zero[r] != 0;
        all_stopped &= zero[r];
        a[r] = s_a[r];
    }
    if (all_stopped) return;
    constexpr int W = 16 / (int)sizeof(V);
    constexpr int U = B > W ? B : W;
    DotAcc<V> acc[B];
    const uint64_t total = (uint64_t)D * B, units = total / U;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < units; i += stride) {
        V yv[U], uv[U], w[U];
        ld_vec<U>(y + i * U, yv, true);
        ld_vec<U>(u + i * U, uv, true);
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int r = e % B;
            w[e] = zero[r] ? (V)0 : fma(-a[r], uv[e], yv[e]);
            acc[r].add(w[e], w[e]);
        }
        st_vec<U>(y + i * U, w);
    }
    for (uint64_t e = units * U + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < total; e += stride) {
        // only reached with B = 1 (and D not a multiple of U)
        const V w = zero[0] ? (V)0 : fma(-a[0], u[e], y[e]);
        y[e] = w;
        acc[0].add(w, w);
    }
    const double v = block_sums<V, B, kRowThreads>(acc);
    if (publish_sums<B>(v, partials, counter)) {
        totals<B, kRowThreads>(partials, gridDim.x, [&](int r, double sum) {
            ChainState &c = st[r];
            if (c.stopped) return;
            const double bt = sqrt(sum);
            if (j < m_max) {
                if (bt <= tau) {
                    c.stopped = 1;
                    c.m_eff = j;
                } else {
                    beta_out[(size_t)r * beta_stride + (j - 1)] = bt;
                    c.s_prev = c.s_cur;
                    c.s_cur = bt;
                    c.beta_prev = bt;
                }
            } else {
                c.m_eff = m_max;
            }
        });
        if (threadIdx.x == 0) *counter = 0;
    }
}

__global__ void copy_meff_kernel(const ChainState *st, int B, int *dst, const BlockSlots slots)
{
    if (threadIdx.x < B) dst[blockIdx.y * B + threadIdx.x] = block_ptr(st, slots.bytes)[threadIdx.x].m_eff;
}

constexpr int kRitzThreads = 128;

// Tridiagonal problems of this translation unit that did not converge (read and
// cleared by ftlm_ritz_status); one copy per device.
__device__ unsigned long long g_ritz_unconverged;

// Coefficient row and outputs of chain c of a Ritz launch.  rows == nullptr: chain c
// reads row c of alpha/beta/mv and writes row c of theta/weight; else rows[c] names
// its coefficient row and its outputs (and m_eff is copied out).
struct RitzIo {
    size_t row;
    double *theta, *weight;
    int m;
};
__device__ __forceinline__ RitzIo ritz_io(int c, int M, const int *mv, double *theta, double *weight,
                                          const RitzRow *rows, bool writer)
{
    RitzIo io;
    if (rows) {
        const RitzRow r = rows[c];
        io.row = r.row;
        io.theta = r.theta;
        io.weight = r.weight;
    } else {
        io.row = (size_t)c;
        io.theta = theta + io.row * M;
        io.weight = weight + io.row * M;
    }
    const int m = mv[io.row];
    if (rows && writer) rows[c].m_eff[0] = m;
    io.m = m < 0 ? 0 : (m > M ? M : m);
    return io;
}

// The Ritz step by divide and conquer (tridiag_dc.cuh), one CTA per chain; a chain's
// results depend on its coefficients only, not on the launch.  A chain with a
// non-finite coefficient or an unconverged root gets NaN Ritz values and weights.
//
// Bound: FP64 instructions on one SM per chain (two lanes per cycle).  One thread per
// root of the merge; the whole problem lives in shared memory (dc::kBytesPerRow, 108).
__global__ void __launch_bounds__(kRitzThreads)
ritz_dc_kernel(int M, const double *__restrict__ alpha, const double *__restrict__ beta, const int *__restrict__ mv,
               double *theta, double *weight, const RitzRow *rows)
{
    extern __shared__ double sh[];
    __shared__ unsigned long long s_max;  // largest |coefficient|, as bits (NaN above inf above all)
    const int t = threadIdx.x, T = blockDim.x;
    const RitzIo io = ritz_io(blockIdx.x, M, mv, theta, weight, rows, t == 0);
    const int m = io.m;
    const double *a = alpha + io.row * M, *b = beta + io.row * M;
    bool ok = true;
    dc::Work w = dc::carve(sh, m);
    double back = 1.0;  // scale of the eigenvalues
    if (m == 1) {
        if (t == 0) {
            w.d[0] = a[0];
            w.f[0] = 1.0;
        }
        __syncthreads();
    } else if (m > 1) {
        if (t == 0) s_max = 0;
        __syncthreads();
        unsigned long long mx = 0;
        for (int i = t; i < m; i += T) {
            w.d[i] = a[i];
            w.e[i] = i + 1 < m ? b[i] : 0.0;
            mx = max(mx, (unsigned long long)__double_as_longlong(fabs(w.d[i])));
            mx = max(mx, (unsigned long long)__double_as_longlong(fabs(w.e[i])));
        }
        atomicMax(&s_max, mx);
        __syncthreads();
        mx = s_max;
        ok = mx < 0x7ff0000000000000ull;
        if (ok) {  // uniform over the CTA
            // an exact power of two brings the coefficients near one
            const int ex = mx ? max(-1000, ilogb(__longlong_as_double((long long)mx))) : 0;
            const double sc = ldexp(1.0, -ex);
            back = ldexp(1.0, ex);
            for (int i = t; i < m; i += T) {
                w.d[i] *= sc;
                w.e[i] *= sc;
            }
            dc::leaf_abs(w, t, T);
            __syncthreads();
            dc::leaf_tear(w, t, T);
            __syncthreads();
            for (int s = 1; s < m; s *= 2) {
                dc::sort_block(w, s, t, T);
                __syncthreads();
                dc::mark_small(w, s, t, T);
                __syncthreads();
                dc::mark_pairs(w, s, t, T);
                __syncthreads();
                dc::deflate(w, s, t, T);
                __syncthreads();
                dc::float_images(w, t, T);
                __syncthreads();
                ok &= dc::roots(w, s, t, T);
                __syncthreads();
                dc::refit(w, s, t, T);
                __syncthreads();
                dc::rows(w, s, t, T);
                __syncthreads();
                dc::commit(w, t, T);
                __syncthreads();
            }
        }
        ok = __syncthreads_and(ok);
        if (!ok && t == 0) atomicAdd(&g_ritz_unconverged, 1ull);
    }
    for (int k = t; k < M; k += T) {
        if (k >= m || !ok) {
            io.theta[k] = k < m ? NAN : 0.0;
            io.weight[k] = k < m ? NAN : 0.0;
        }
    }
    if (!ok) return;
    for (int i = t; i < m; i += T) {  // ascending order
        const long long key = dc::order_key(w.d[i]);
        int r = 0;
        for (int j = 0; j < m; ++j) {
            const long long q = dc::order_key(w.d[j]);
            r += (q < key) | ((q == key) & (j < i));
        }
        io.theta[r] = w.d[i] * back;
        io.weight[r] = w.f[i] * w.f[i];
    }
}

// The same by implicit QR with a sweep limit (ftlm_ritz_set_max_sweeps): one thread
// per chain, T chains per CTA.  A chain whose iteration does not converge within
// max_sweeps gets NaN Ritz values and weights.
__global__ void ritz_kernel(int n, int M, const double *__restrict__ alpha, const double *__restrict__ beta,
                            const int *__restrict__ mv, double *theta, double *weight, const RitzRow *rows,
                            int max_sweeps)
{
    extern __shared__ double sh[];
    const int T = blockDim.x, i = threadIdx.x;
    const int c = blockIdx.x * T + i;
    if (c >= n) return;
    Strided d{sh + i, T}, e{sh + (size_t)M * T + i, T}, z{sh + (size_t)2 * M * T + i, T};
    const RitzIo io = ritz_io(c, M, mv, theta, weight, rows, true);
    const size_t row = io.row;
    double *th = io.theta, *wt = io.weight;
    const int m = io.m;
    for (int k = 0; k < m; ++k) {
        d[k] = alpha[row * M + k];
        e[k] = k + 1 < m ? beta[row * M + k] : 0.0;
        z[k] = k == 0 ? 1.0 : 0.0;
    }
    bool ok = true;
    if (m > 1) {
        ok = tridiag_qr(d, e, z, m, max_sweeps);
        if (ok) sort_ascending(d, z, m);
        else atomicAdd(&g_ritz_unconverged, 1ull);
    }
    for (int k = 0; k < M; ++k) {
        th[k] = k < m ? (ok ? d[k] : NAN) : 0.0;
        wt[k] = k < m ? (ok ? z[k] * z[k] : NAN) : 0.0;
    }
}

}  // namespace

std::atomic<int> g_ritz_max_sweeps{0};
int ritz_max_sweeps() { return g_ritz_max_sweeps.load(std::memory_order_relaxed); }

namespace {

ftlm_status ritz_launch(int n, int M, const double *alpha, const double *beta, const int *mv, double *theta,
                        double *weight, const RitzRow *rows, cudaStream_t stream)
{
    if (n == 0) return FTLM_OK;
    int occ = 1;
    const int max_sweeps = ritz_max_sweeps();
    if (max_sweeps <= 0) {
        // one thread per row up to kRitzThreads; the choice changes no result
        const int T = std::min(kRitzThreads, (M + 31) / 32 * 32);
        FTLM_CUDA(kernel_occupancy((const void *)ritz_dc_kernel, kRitzThreads, dc::kBytesPerRow * FTLM_MAX_LANCZOS,
                                   true, &occ));
        ritz_dc_kernel<<<n, T, dc::kBytesPerRow * M, stream>>>(M, alpha, beta, mv, theta, weight, rows);
        note_launch();
        FTLM_CUDA(cudaGetLastError());
        return FTLM_OK;
    }
    constexpr size_t kSmemMax = 96 * 1024;
    FTLM_CUDA(kernel_occupancy((const void *)ritz_kernel, 32, kSmemMax, true, &occ));
    const size_t per_chain = 3 * (size_t)M * sizeof(double);
    int T = (int)(kSmemMax / per_chain);
    T = T < 1 ? 1 : (T > 32 ? 32 : T);
    if (T > n) T = n;
    const int grid = (n + T - 1) / T;
    ritz_kernel<<<grid, T, per_chain * T, stream>>>(n, M, alpha, beta, mv, theta, weight, rows, max_sweeps);
    note_launch();
    FTLM_CUDA(cudaGetLastError());
    return FTLM_OK;
}

}  // namespace

ftlm_status launch_ritz(int n, int M, const double *alpha, const double *beta, const int *mv,
                        double *theta, double *weight, cudaStream_t stream)
{
    return ritz_launch(n, M, alpha, beta, mv, theta, weight, nullptr, stream);
}

ftlm_status launch_ritz_rows(int n, int M, const double *alpha, const double *beta, const int *mv,
                             const RitzRow *rows, cudaStream_t stream)
{
    return ritz_launch(n, M, alpha, beta, mv, nullptr, nullptr, rows, stream);
}

namespace {

// ---- workspace and block plan -------------------------------------------
uint64_t align256(uint64_t v) { return (v + 255) & ~255ull; }

// Widest block of chains: the width set by ftlm_lanczos_set_block, else FTLM_BLOCK
// (1, 4, 8 or 16), else 8 vectors (FP32) or 4 (FP64).
std::atomic<int> g_block_width{0};

int max_block(ftlm_dtype dtype)
{
    static const int over = [] {
        const char *e = getenv("FTLM_BLOCK");
        const int v = e ? atoi(e) : 0;
        return valid_block(v) ? v : 0;
    }();
    const int set = g_block_width.load(std::memory_order_relaxed);
    if (set) return set;
    return over ? over : (dtype == FTLM_F32 ? 8 : 4);
}

// Split R chains into blocks: the widest allowed width in {16, 8, 4} that fits the
// chains left, then single chains for fewer than 4.  bmax = 0: max_block(dtype).
std::vector<int> block_plan(int R, ftlm_dtype dtype, int bmax)
{
    if (!bmax) bmax = max_block(dtype);
    std::vector<int> plan;
    int left = R;
    for (int w : {16, 8, 4}) {
        if (w > bmax) continue;
        while (left >= w) {
            plan.push_back(w);
            left -= w;
        }
    }
    while (left-- > 0) plan.push_back(1);
    return plan;
}

// Blocks of one width that run side by side in the same launches (block k in grid row
// y = k) while their slots fit kSideBySideBytes.  A small sector's launch is bound by
// its dependent chain of latencies, not by the work of one block, and holds a part of
// the SMs only: the N = 16 ring in FP64, R = 20 (five blocks of 4, 12 870 rows), takes
// 29 us per step for all five against 5 x 28 us one after another.  At 24 MiB the rows of
// one block of 8 floats number 0.19 million or more, enough for every SM.  A block's
// grid and sums are those of a launch of its own, so its results do not change.
constexpr uint64_t kSideBySideBytes = 24ull << 20;

// Workspace: `slots` block slots (two vector blocks, partials, states and counters, and
// the alpha sums of CR H.v launches), then the coefficients of every chain.
struct Layout {
    int bw;     // widest block
    int slots;  // blocks side by side
    uint64_t slot, vec1, partials, state, sums;  // bytes of a slot and offsets in it (vectors first)
    uint64_t alpha, beta, meff, total;
};

Layout layout(const ftlm_basis *b, int R, int M, ftlm_dtype dtype, int bmax = 0)
{
    Layout l;
    l.bw = 1;
    int same = 1, most = 1, last = 0;
    for (int w : block_plan(R, dtype, bmax)) {
        l.bw = w > l.bw ? w : l.bw;
        same = w == last ? same + 1 : 1;
        last = w;
        most = std::max(most, same);
    }
    const uint64_t vb = align256(b->D * (uint64_t)l.bw * (dtype == FTLM_F32 ? 4ull : 8ull));
    l.vec1 = vb;
    l.partials = 2 * vb;
    l.state = l.partials + align256((uint64_t)max_row_grid(b) * l.bw * sizeof(double));
    l.sums = l.state + align256(l.bw * sizeof(ChainState) + 64);
    l.slot = l.sums + (b->two_s == 1 && b->mode == FTLM_RANK_CR ? align256(kAlphaFixedBytes) : 0);
    const uint64_t rows = 2 * align256((uint64_t)R * M * sizeof(double)) + align256((uint64_t)R * sizeof(int));
    const uint64_t room = kSideBySideBytes > rows ? kSideBySideBytes - rows : 0;
    l.slots = (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)most, room / l.slot));
    l.alpha = l.slots * l.slot;
    l.beta = l.alpha + align256((uint64_t)R * M * sizeof(double));
    l.meff = l.beta + align256((uint64_t)R * M * sizeof(double));
    l.total = l.meff + align256((uint64_t)R * sizeof(int));
    return l;
}

// n blocks of B chains side by side: start vectors, then min(M, D) fused H.v + update
// launches.
template <typename V, int B>
ftlm_status run_blocks(const ftlm_basis *b, int M, int r0, int n, int chain0, uint64_t seed, int dist,
                       const double *src, ftlm_dtype dtype, char *ws, const Layout &lay, cudaStream_t stream)
{
    int occ_start = 1, occ_upd = 1;
    FTLM_CUDA(kernel_occupancy((const void *)start_kernel<V, B>, kRowThreads, 0, false, &occ_start));
    FTLM_CUDA(kernel_occupancy((const void *)update_kernel<V, B>, kRowThreads, 0, false, &occ_upd));
    V *vec[2] = {(V *)ws, (V *)(ws + lay.vec1)};
    double *partials = (double *)(ws + lay.partials);
    ChainState *st = (ChainState *)(ws + lay.state);
    unsigned int *counter = (unsigned int *)(st + lay.bw);
    double *alpha_ws = (double *)(ws + lay.alpha);
    double *beta_ws = (double *)(ws + lay.beta);
    int *meff_ws = (int *)(ws + lay.meff);
    const uint32_t D = (uint32_t)b->D;
    const int m_max = (uint64_t)M < b->D ? M : (int)b->D;
    const double tau = dtype == FTLM_F32 ? b->tau32 : b->tau64;
    constexpr int W = 16 / (int)sizeof(V);
    constexpr int U = B > W ? B : W;
    const dim3 g_start(row_grid(b, D, occ_start), n);
    const dim3 g_upd(row_grid(b, ((uint64_t)D * B + U - 1) / U, occ_upd), n);
    const BlockSlots slots{lay.slot};

    // states and counters, and the alpha sums behind them
    const uint64_t zero = lay.slot > lay.sums ? lay.slot - lay.state : lay.bw * sizeof(ChainState) + 64;
    FTLM_CUDA(cudaMemset2DAsync(st, lay.slot, 0, zero, n, stream));
    start_kernel<V, B><<<g_start, kRowThreads, 0, stream>>>(
        D, KeySpec{seed, b->key_n, b->K, chain0 + r0}, dist, src ? src + (size_t)r0 * D : nullptr, vec[0], st,
        partials, counter, slots);
    note_launch();
    FTLM_CUDA(cudaGetLastError());
    int cur = 0;
    for (int j = 1; j <= m_max; ++j) {
        LanczosHv epi{st, partials, counter, alpha_ws + (size_t)r0 * M + (j - 1), M, j,
                      (unsigned long long *)(ws + lay.sums), b->tau64 * (0x1p53 / 100.0), n, lay.slot};
        ftlm_status s = launch_hv(b, dtype, B, vec[cur], vec[1 - cur], &epi, stream);
        if (s != FTLM_OK) return s;
        void *tok = profile_begin(kProfUpdate, stream);
        update_kernel<V, B><<<g_upd, kRowThreads, 0, stream>>>(D, vec[1 - cur], vec[cur], st, partials, counter, j,
                                                               m_max, tau, beta_ws + (size_t)r0 * M, M, slots);
        note_launch();
        profile_end(tok, stream);
        FTLM_CUDA(cudaGetLastError());
        cur = 1 - cur;
    }
    copy_meff_kernel<<<dim3(1, n), 32, 0, stream>>>(st, B, meff_ws + r0, slots);
    note_launch();
    FTLM_CUDA(cudaGetLastError());
    return FTLM_OK;
}

template <typename V>
ftlm_status run_chains(const ftlm_basis *b, int R, int M, int chain0, uint64_t seed, int dist, const double *src,
                       ftlm_dtype dtype, int bmax, char *ws, const Layout &lay, double *theta, double *weight,
                       int *m_eff, double *alpha_dev, double *beta_dev, cudaStream_t stream)
{
    double *alpha_ws = (double *)(ws + lay.alpha);
    double *beta_ws = (double *)(ws + lay.beta);
    int *meff_ws = (int *)(ws + lay.meff);
    FTLM_CUDA(cudaMemsetAsync(alpha_ws, 0, (size_t)R * M * sizeof(double), stream));
    FTLM_CUDA(cudaMemsetAsync(beta_ws, 0, (size_t)R * M * sizeof(double), stream));
    const std::vector<int> plan = block_plan(R, dtype, bmax);
    int r0 = 0;
    for (size_t k = 0; k < plan.size();) {
        const int B = plan[k];
        int n = 1;  // blocks of this width that run side by side
        const int most = hv_splits(b, dtype, B) ? 1 : lay.slots;
        while (n < most && k + n < plan.size() && plan[k + n] == B) ++n;
        ftlm_status s;
        switch (B) {
        case 16: s = run_blocks<V, 16>(b, M, r0, n, chain0, seed, dist, src, dtype, ws, lay, stream); break;
        case 8: s = run_blocks<V, 8>(b, M, r0, n, chain0, seed, dist, src, dtype, ws, lay, stream); break;
        case 4: s = run_blocks<V, 4>(b, M, r0, n, chain0, seed, dist, src, dtype, ws, lay, stream); break;
        default: s = run_blocks<V, 1>(b, M, r0, n, chain0, seed, dist, src, dtype, ws, lay, stream); break;
        }
        if (s != FTLM_OK) return s;
        r0 += n * B;
        k += n;
    }
    ftlm_status s = launch_ritz(R, M, alpha_ws, beta_ws, meff_ws, theta, weight, stream);
    if (s != FTLM_OK) return s;
    FTLM_CUDA(cudaMemcpyAsync(m_eff, meff_ws, (size_t)R * sizeof(int), cudaMemcpyDeviceToDevice, stream));
    if (alpha_dev)
        FTLM_CUDA(cudaMemcpyAsync(alpha_dev, alpha_ws, (size_t)R * M * sizeof(double), cudaMemcpyDeviceToDevice, stream));
    if (beta_dev)
        FTLM_CUDA(cudaMemcpyAsync(beta_dev, beta_ws, (size_t)R * M * sizeof(double), cudaMemcpyDeviceToDevice, stream));
    return FTLM_OK;
}

}  // namespace

ftlm_status lanczos_run(const ftlm_basis *b, int R, int M, int chain0, uint64_t seed, int dist, const double *src,
                        ftlm_dtype dtype, void *work, uint64_t work_bytes, double *theta, double *weight,
                        int *m_eff, double *alpha_dev, double *beta_dev, cudaStream_t stream, int bmax)
{
    if (!b) return fail(FTLM_EINVAL, "NULL basis");
    if (R < 1) return fail(FTLM_EINVAL, "R < 1");
    if (bmax && !valid_block(bmax)) return fail(FTLM_EINVAL, "block width must be 1, 4, 8 or 16");
    if (!bmax) bmax = max_block(dtype);
    if (M < 1 || M > FTLM_MAX_LANCZOS) return fail(FTLM_EINVAL, "M out of range");
    if (dtype != FTLM_F32 && dtype != FTLM_F64) return fail(FTLM_EINVAL, "bad dtype");
    if (dist != FTLM_VEC_GAUSS && dist != FTLM_VEC_RADEMACHER) return fail(FTLM_EINVAL, "bad distribution");
    if (!theta || !weight || !m_eff) return fail(FTLM_EINVAL, "NULL output");
    if (!work || ((uintptr_t)work & 255u)) return fail(FTLM_EINVAL, "workspace NULL or not 256-byte aligned");
    const Layout lay = layout(b, R, M, dtype, bmax);
    if (work_bytes < lay.total) return fail(FTLM_ENOMEM, "workspace smaller than ftlm_lanczos_workspace_bytes()");
    return dtype == FTLM_F32
               ? run_chains<float>(b, R, M, chain0, seed, dist, src, dtype, bmax, (char *)work, lay, theta, weight,
                                   m_eff, alpha_dev, beta_dev, stream)
               : run_chains<double>(b, R, M, chain0, seed, dist, src, dtype, bmax, (char *)work, lay, theta, weight,
                                    m_eff, alpha_dev, beta_dev, stream);
}

uint64_t lanczos_workspace(const ftlm_basis *b, int R, int M, ftlm_dtype dtype, int bmax)
{
    return layout(b, R, M, dtype, bmax).total;
}

namespace {

// Scratch of ftlm_lanczos_noalloc, for callers that cannot allocate device memory.
// Host code sees only a host-side stand-in for this symbol; its device address is
// looked up once per device with cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[FTLM_NOALLOC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
// Per device: the context the address was looked up in (cuCtxGetId, never reused
// within a process) and the address.  A device reset gives the device a new
// primary context, and the module with the array is loaded again at a new
// address; the id comparison makes the next call look it up again.
struct NoallocSlot {
    unsigned long long ctx_id;
    void *ptr;
};
NoallocSlot g_noalloc[kMaxDevices] = {};

// Id of the current context, from the driver through the runtime's entry-point
// query (no link-time dependency on the driver library); false if unavailable.
bool current_context_id(unsigned long long *id)
{
    using GetCurrent = CUresult (*)(CUcontext *);
    using GetId = CUresult (*)(CUcontext, unsigned long long *);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrent>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
    });
    CUcontext ctx = nullptr;
    if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx) return false;
    return get_id(ctx, id) == CUDA_SUCCESS;
}

// Device address of g_noalloc_scratch on the current device: looked up with
// cudaGetSymbolAddress on the first call in a context, cached for later calls.
// (Before any runtime call on this thread no context may be current yet; then the
// address is looked up, which binds the primary context, and cached from the
// next call on.)
ftlm_status noalloc_scratch(void **out)
{
    int dev = 0;
    FTLM_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(FTLM_EUNSUPPORTED, "device index beyond 64");
    unsigned long long ctx = 0;
    const bool have_id = current_context_id(&ctx);
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    NoallocSlot &slot = g_noalloc[dev];
    if (!slot.ptr || !have_id || slot.ctx_id != ctx) {
        void *p = nullptr;
        FTLM_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        slot.ptr = p;
        slot.ctx_id = have_id ? ctx : 0;
    }
    *out = slot.ptr;
    return FTLM_OK;
}

}  // namespace

}  // namespace ftlm

using namespace ftlm;

extern "C" ftlm_status ftlm_lanczos_noalloc(const ftlm_basis *b, int R, int M, uint64_t seed,
                                            ftlm_vec_dist dist, ftlm_dtype dtype, double *theta_dev,
                                            double *weight_dev, int *m_eff_dev, double *alpha_dev,
                                            double *beta_dev, void *stream)
{
    if (!b) return fail(FTLM_EINVAL, "NULL basis");
    if (R < 1 || M < 1 || M > FTLM_MAX_LANCZOS) return fail(FTLM_EINVAL, "R or M out of range");
    if (dtype != FTLM_F32 && dtype != FTLM_F64) return fail(FTLM_EINVAL, "bad dtype");
    const uint64_t need = layout(b, R, M, dtype).total;
    if (need > FTLM_NOALLOC_SCRATCH_BYTES)
        return fail(FTLM_EUNSUPPORTED, "workspace of " + std::to_string(need) +
                                           " bytes exceeds the static scratch of FTLM_NOALLOC_SCRATCH_BYTES (" +
                                           std::to_string(FTLM_NOALLOC_SCRATCH_BYTES) + " bytes)");
    void *scratch = nullptr;
    ftlm_status s = noalloc_scratch(&scratch);
    if (s != FTLM_OK) return s;
    return lanczos_run(b, R, M, 0, seed, dist, nullptr, dtype, scratch, FTLM_NOALLOC_SCRATCH_BYTES, theta_dev,
                       weight_dev, m_eff_dev, alpha_dev, beta_dev, (cudaStream_t)stream);
}

extern "C" ftlm_status ftlm_lanczos_set_block(int width)
{
    if (width != 0 && !valid_block(width)) return fail(FTLM_EINVAL, "block width must be 0, 1, 4, 8 or 16");
    g_block_width.store(width, std::memory_order_relaxed);
    return FTLM_OK;
}

extern "C" ftlm_status ftlm_lanczos_workspace_bytes(const ftlm_basis *b, int R, int M, ftlm_dtype dtype,
                                                    uint64_t *bytes)
{
    if (!b || !bytes) return fail(FTLM_EINVAL, "NULL argument");
    if (R < 1 || M < 1 || M > FTLM_MAX_LANCZOS) return fail(FTLM_EINVAL, "R or M out of range");
    if (dtype != FTLM_F32 && dtype != FTLM_F64) return fail(FTLM_EINVAL, "bad dtype");
    *bytes = layout(b, R, M, dtype).total;
    return FTLM_OK;
}

extern "C" ftlm_status ftlm_lanczos(const ftlm_basis *b, int R, int M, uint64_t seed, ftlm_vec_dist dist,
                                    ftlm_dtype dtype, void *work_dev, uint64_t work_bytes, double *theta_dev,
                                    double *weight_dev, int *m_eff_dev, double *alpha_dev, double *beta_dev,
                                    void *stream)
{
    return lanczos_run(b, R, M, 0, seed, dist, nullptr, dtype, work_dev, work_bytes, theta_dev, weight_dev, m_eff_dev,
                       alpha_dev, beta_dev, (cudaStream_t)stream);
}

extern "C" ftlm_status ftlm_lanczos_from(const ftlm_basis *b, int R, int M, const double *start_dev,
                                         ftlm_dtype dtype, void *work_dev, uint64_t work_bytes,
                                         double *theta_dev, double *weight_dev, int *m_eff_dev,
                                         double *alpha_dev, double *beta_dev, void *stream)
{
    if (!start_dev) return fail(FTLM_EINVAL, "start_dev is NULL");
    return lanczos_run(b, R, M, 0, 0, FTLM_VEC_GAUSS, start_dev, dtype, work_dev, work_bytes, theta_dev, weight_dev,
                       m_eff_dev, alpha_dev, beta_dev, (cudaStream_t)stream);
}

namespace ftlm {
ftlm_status ritz_unconverged_take(cudaStream_t stream, uint64_t *count)
{
    unsigned long long v = 0, zero = 0;
    FTLM_CUDA(cudaMemcpyFromSymbolAsync(&v, g_ritz_unconverged, sizeof(v), 0, cudaMemcpyDeviceToHost, stream));
    FTLM_CUDA(cudaMemcpyToSymbolAsync(g_ritz_unconverged, &zero, sizeof(zero), 0, cudaMemcpyHostToDevice, stream));
    FTLM_CUDA(cudaStreamSynchronize(stream));
    *count = v;
    return FTLM_OK;
}
}  // namespace ftlm

extern "C" ftlm_status ftlm_ritz_status(void *stream, uint64_t *unconverged)
{
    uint64_t a = 0, b = 0;
    ftlm_status s = ritz_unconverged_take((cudaStream_t)stream, &a);
    if (s == FTLM_OK) s = ghost_unconverged_take((cudaStream_t)stream, &b);
    if (s != FTLM_OK) return s;
    if (unconverged) *unconverged = a + b;
    if (a + b) return fail(FTLM_ENOCONV, std::to_string(a + b) + " tridiagonal eigenproblem(s) did not converge");
    return FTLM_OK;
}

extern "C" ftlm_status ftlm_ritz_set_max_sweeps(int sweeps)
{
    if (sweeps < 0) return fail(FTLM_EINVAL, "sweeps < 0");
    g_ritz_max_sweeps.store(sweeps, std::memory_order_relaxed);
    return FTLM_OK;
}

extern "C" ftlm_status ftlm_ritz(int n, int M, const double *alpha_dev, const double *beta_dev,
                                 const int *m_dev, double *theta_dev, double *weight_dev, void *stream)
{
    if (n < 0 || M < 1 || M > FTLM_MAX_LANCZOS) return fail(FTLM_EINVAL, "n or M out of range");
    if (n > 0 && (!alpha_dev || !beta_dev || !m_dev || !theta_dev || !weight_dev))
        return fail(FTLM_EINVAL, "NULL device pointer");
    return launch_ritz(n, M, alpha_dev, beta_dev, m_dev, theta_dev, weight_dev, (cudaStream_t)stream);
}
