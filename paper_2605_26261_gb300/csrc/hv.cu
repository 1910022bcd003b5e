// H.v gather (step a3), Eq. 12 with the ladder coefficients of Eq. 13-14 at
// s = 1/2, and the Lanczos epilogue fused into the same launch (step a4).
//
// One thread owns one output row t (the row-wise gather of Sec. 2): it recovers
// its label n_t, and for every bond whose two spins are antiparallel in n_t it
// exchanges them, ranks the resulting source label k and gathers (J_b/2) x[k].
// The diagonal sum_b J_b m_i m_j equals sum_b J_b/4 - sum_{b antiparallel} J_b/2,
// so it is accumulated alongside the gathers.  Each thread writes one y[t]; there
// are no atomics.
//
// Bonds are warp-uniform (staged once per CTA in shared memory and read as
// broadcasts), and the 32 rows of a warp are 32 consecutive sector indices, i.e.
// 32 consecutive labels in increasing order that differ only in their lowest bits.  For a bond
// on high sites the exchange therefore shifts all 32 ranks by the same amount and
// the warp's gather is one contiguous 128-byte line; bonds on low sites land within
// a few lines of the warp's own rows.  The grid is persistent (a multiple of the
// SM count) and walks the rows in order, so at any moment every bond's gather
// stream sits in a narrow window of x and the windows stay L2-resident.  CLT
// launches and plain H.v deal 32-row tiles to warps round-robin; CR Lanczos
// launches hand them out from a counter, which keeps the warps on one frontier
// of rows (they drift apart under the round-robin order, and the union of the
// gather windows outgrows L2: 20 % fewer DRAM bytes, 25 % less time on the N = 30
// icosahedral sector).  Their alpha sums are then added per tile as whole
// numbers (epi.cuh).
//
// Two rank strategies:
//   CLT  label n_t = basis[t]; rank(n') = C_b + popc(M_b & (2^j - 1)) with
//        b = n' >> 5, j = n' & 31 (Eq. 19-20, Algorithm 2); {M_b, C_b} is one
//        8-byte entry.
//   CR   rank(n) = thi[n >> L] + tlo[n & (2^L-1)] (Algorithm 1 with the L low
//        digits and the N-L high digits each collapsed into one table lookup);
//        the row label is recovered by the inverse map (binary search of thi,
//        then ulo).  tlo (2^L x 16 bit) is staged in shared memory; thi is read
//        through L1 and is warp-uniform for almost every row.  A bond with both
//        sites in one block changes only that block's lookup: the other half of
//        the rank is the row's own.
//
// Block H.v (B vectors, interleaved: element (t, r) at t * B + r).  The row's rank
// work is done once and every antiparallel bond gathers B contiguous values
// (32 bytes, one DRAM sector, for B = 8 in FP32), so the index arithmetic and the
// table lookups are shared by the B vectors -- the batched scheme of Sec. 3.4.
//
// The Lanczos epilogue (Paige's ordering) runs in the same launch (epi.cuh).
#include <algorithm>
#include <cstdlib>

#include "epi.cuh"
#include "ftlm_internal.cuh"
#include "reduce.cuh"
#include "vec.cuh"
#include "rows.cuh"

namespace ftlm {

namespace {

// Resident CTAs per SM the compiler must allow for (register budget).  Single
// vectors with up to 2 rows per thread keep a small register footprint (6 CTAs of
// 256 threads, the shared-memory limit of the CR kernel); 4 rows per thread and
// blocks of 4-8 vectors get at least 3 CTAs per SM (fewer starve the loads), 2 with
// 8-bond chunks of 8-wide blocks (their 16 gathers per row in flight carry it);
// 16-wide blocks keep all their registers (a cap spills).  FP64 rows (row_f64): 3 CTAs
// up to blocks of 4, 2 for blocks of 8 and 1 for wider ones.
// Build option FTLM_B8_MIN_CTAS: the FP32 cut for 8-wide blocks with chunks of 4.
#ifndef FTLM_B8_MIN_CTAS
#define FTLM_B8_MIN_CTAS 3
#endif

template <typename V, int RT, int B, int C> __host__ __device__ constexpr int min_ctas()
{
    if (sizeof(V) == 8)
        return B >= 16 ? 1 : (B >= 8 ? 2 : 3);
    return B >= 16 ? 1
                   : (B >= 8 && C >= 8 ? 2
                                       : (B >= 8 && C <= 2 ? 4 : (B >= 8 ? FTLM_B8_MIN_CTAS : (B >= 4 || RT >= 4 ? 3 : 6))));
}

// EPI: kPlain (y = H x) or kLanczos (fused Lanczos epilogue with alpha).
enum { kPlain = 0, kLanczos = 1 };

template <typename V, typename Lbl, bool CLT, int EPI, int RT, int B, int C>
__global__ void __launch_bounds__(kRowThreads, min_ctas<V, RT, B, C>())
hv_kernel(const SectorTables s, const BondList bl, const V *__restrict__ x0, V *y0, const EpiDev ep0)
{
    constexpr bool LANCZOS = EPI != kPlain;
    const EpiDev ep = LANCZOS ? epi_block<B>(ep0) : ep0;
    const V *__restrict__ x = LANCZOS ? block_ptr(x0, ep0.slot) : x0;
    V *y = LANCZOS ? block_ptr(y0, ep0.slot) : y0;
    // CR Lanczos launches take their tiles in dynamic order (their gathers gain the
    // most from a narrow frontier of rows) and add their alpha sums per tile
    constexpr bool TILES = LANCZOS && !CLT;
    extern __shared__ uint16_t s_tlo[];
    __shared__ RowBonds<V, Lbl> s_bond;
    __shared__ V s_inv_s[B], s_c_prev[B];  // per-chain scalars of the epilogue
    __shared__ AlphaSums<TILES ? B : 1, kRowThreads> s_asum;
    if (LANCZOS && epi_begin<V, B>(ep, s_inv_s, s_c_prev)) return;
    if constexpr (TILES) tiles_begin(s_asum);
    s_bond.stage(bl);
    if (!CLT)
        for (uint32_t i = threadIdx.x; i <= s.lomask; i += blockDim.x) s_tlo[i] = __ldg(s.tlo + i);
    __syncthreads();
    const V jsum4 = (V)bl.jsum4;
    DotAcc<V> apart[B];
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t tile_rows = 32u * RT;
    const uint32_t ntiles = (uint32_t)(((uint64_t)s.D + tile_rows - 1) / tile_rows);
    // the rows of one tile: rank work, gathers and the epilogue of the mode
    auto do_tile = [&](uint32_t tile) {
        uint32_t t[RT];
        bool ok[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const uint32_t tt = tile * tile_rows + 32u * i + lane;
            ok[i] = tt < s.D;
            t[i] = ok[i] ? tt : s.D - 1;  // rows past the end recompute the last row, unstored
        }
        V acc[RT][B], dsum[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            dsum[i] = (V)0;
#pragma unroll
            for (int r = 0; r < B; ++r) acc[i][r] = (V)0;
        }
        if constexpr (sizeof(V) == 8) {
            static_assert(RT == 1 || sizeof(V) == 4, "one row of doubles per thread");
            row_f64<Lbl, CLT, B, C>(s, bl, s_bond.l, s_tlo, x, t[0], acc[0], dsum[0]);
        } else if constexpr (CLT) {
            rows_clt<V, RT, B, C>(s, bl, s_bond.e, x, t, acc, dsum);
        } else {
            rows_cr<V, Lbl, RT, B, C>(s, bl, s_bond.e, s_tlo, x, t, acc, dsum);
        }
        if constexpr (TILES) {
            DotAcc<V> tacc[B];
#pragma unroll
            for (int i = 0; i < RT; ++i)
                if (ok[i]) epi_row<V, B, true>(ep, s_inv_s, s_c_prev, x, y, t[i], jsum4 - dsum[i], acc[i], tacc);
            add_tile<V, B>(ep, s_asum, tacc);
        } else {
#pragma unroll
            for (int i = 0; i < RT; ++i)
                if (ok[i]) epi_row<V, B, LANCZOS>(ep, s_inv_s, s_c_prev, x, y, t[i], jsum4 - dsum[i], acc[i], apart);
        }
    };
    for (uint32_t tile = warp; tile < ntiles;) {
        // claim the next tile now; its atomic completes while this tile's rows run
        const uint32_t claim = TILES ? claim_tile(ep) : 0u;
        do_tile(tile);
        tile = TILES ? claimed_tile(claim, nwarps) : tile + nwarps;
    }
    if constexpr (TILES) tiles_done(ep, s_asum);
    else if constexpr (LANCZOS) epi_end<V, B, kRowThreads>(ep, apart);
}

// alpha_j of a dynamically ordered launch from its sums (epi.cuh); one warp.
template <int B> __global__ void __launch_bounds__(32) alpha_kernel(const EpiDev ep0)
{
    const EpiDev ep = epi_block<B>(ep0);
    const int r = threadIdx.x;
    if (r < B) {
        const long long hi = (long long)ep.fixed[2 * r], lo = (long long)ep.fixed[2 * r + 1];
        const bool bad = (ep.counter[3] >> r) & 1u;
        const double v = two_word_value(hi, lo, ep.unscale);
        ep.fixed[2 * r] = 0;
        ep.fixed[2 * r + 1] = 0;
        if (!ep.st[r].stopped) {
            ep.st[r].alpha = bad ? NAN : v;
            ep.alpha_out[(size_t)r * ep.alpha_stride] = bad ? NAN : v;
        }
    }
    __syncwarp();
    if (r == 0) {
        ep.counter[1] = 0;
        ep.counter[3] = 0;
    }
}

// Rows per thread (RT) for single vectors.  Measured on GB300 (icosidodecahedron,
// FP32): CR is fastest with 2 rows per thread (its rank tables are L1/shared-memory
// resident and the bond chunk is reused across rows), CLT with 1 (its two dependent
// gathers per bond already fill the load queues).  Blocks of vectors use 1.
// FTLM_HV_ROWS = 1, 2 or 4 overrides the single-vector choice.
int rows_per_thread(bool clt)
{
    static const int over = [] {
        const char *e = getenv("FTLM_HV_ROWS");
        const int v = e ? atoi(e) : 0;
        return (v == 1 || v == 2 || v == 4) ? v : 0;
    }();
    return over ? over : (clt ? 1 : 2);
}

// Cap on resident CTAs per SM used for the H.v grid (FTLM_HV_CTAS, default: no cap).
// Fewer CTAs shrink the window of rows in flight and with it the L2 working set of
// the gather streams.
int hv_cta_cap()
{
    static const int cap = [] {
        const char *e = getenv("FTLM_HV_CTAS");
        const int v = e ? atoi(e) : 0;
        return v > 0 ? v : kMaxBlocksPerSm;
    }();
    return cap;
}

// Split Lanczos H.v (see HiWalk, LoWalk): used when the basis asks for it, or
// under FTLM_HV_AUTO for blocks of FP32 vectors of at least kSplitMinBytes32
// (kSplitMinBytes32Rows for rows of 32 bytes or more) of sectors with at least
// kSplitMinHiBonds high-high bonds.  Measured on GB300 (H.v
// step, one walk -> split), N = 30 icosidodecahedral sectors (26 of 60 bonds
// high-high), FP32 blocks of 8 with both walks in 128-thread CTAs: S^z = 0 / -5 /
// -6 / -7 (5, 0.96, 0.46, 0.19 GB) 16.7 -> 14.0, 3.18 -> 2.78, 1.54 -> 1.40, 0.669
// -> 0.661 ms; with walk A in blocks and 256-thread CTAs: FP32 blocks of 4 / 1 at
// S^z = 0 (2.5, 0.6 GB) 9.72 -> 9.22, 5.54 -> 6.15 ms.  N = 34 ring (19 of 34 bonds high-high), FP32 blocks of 8, S^z = 0
// (75 GB): 177.1 -> 157.6 ms (179.0 -> 183.1 with 256-thread CTAs).  N = 26 ladder
// and ring (11 high-high bonds), S^z = 0, blocks of 8 (0.33 GB): 1.34 -> 1.41, 1.20
// -> 1.24 ms.  The split moves two row streams per step instead of one but no
// long-jump gather misses L2; with few high-high bonds per row, or on small blocks,
// the second pass costs more than the misses it saves.  FP64 rows are bound by the FP64
// pipe and the walks issue an FMA per bond and row, so there one walk over the lists of
// antiparallel bonds wins everywhere: icosidodecahedron S^z = 0 (1.2, 5, 10, 20 GB of blocks
// of 1, 4, 8, 16) 15.3, 45.2, 84.5, 165 against 26.9, 69.7, 115, 220 ms split; N = 32 ring
// 41.7, 114, 208, 399 against 68.5, 166, 260, 499.
constexpr uint64_t kSplitMinBytes32Rows = 256ull << 20;
constexpr uint64_t kSplitMinBytes32 = 768ull << 20;
constexpr int kSplitMinHiBonds = 16;
constexpr int kDefaultWalkRh = 8;

bool split_walks(const ftlm_basis *b, int B, size_t vsize, HiWalk *w)
{
    if (b->hv_schedule == FTLM_HV_ONE_WALK || !b->lo_tiles) return false;
    const uint64_t bytes = b->D * (uint64_t)B * vsize;
    const uint64_t min_bytes = B * vsize >= 32 ? kSplitMinBytes32Rows : kSplitMinBytes32;
    if (b->hv_schedule == FTLM_HV_AUTO && (vsize == 8 || bytes < min_bytes || b->n_hi_bonds < kSplitMinHiBonds))
        return false;
    return build_hi_walk(b, b->walk_rh ? b->walk_rh : kDefaultWalkRh, w);
}

// One hv_kernel launch over every row.
template <typename V, typename Lbl, bool CLT, int EPI, int RT, int B, int C>
ftlm_status launch_rows(const ftlm_basis *b, const BondList &bl, const V *x, V *y, const EpiDev &ep, int blocks,
                        int max_ctas, cudaStream_t stream)
{
    const size_t smem = CLT ? 0 : ((size_t)1 << b->L) * sizeof(uint16_t);
    auto kern = hv_kernel<V, Lbl, CLT, EPI, RT, B, C>;
    int occ = 1;  // resident blocks per SM for this instantiation
    const size_t smem_max = CLT ? 0 : ((size_t)1 << kLoBitsMax) * sizeof(uint16_t);
    // A plain H.v has no block sums, so its blocks may be smaller: with the CLT (no table
    // to stage per block) a sector too small for one block of kRowThreads rows on every
    // SM is cut into smaller ones.
    int threads = kRowThreads;
    if (CLT && EPI == kPlain)
        while (threads > 64 && b->D < (uint64_t)threads * RT * b->num_sms) threads /= 2;
    FTLM_CUDA(kernel_occupancy((const void *)kern, threads, smem_max, false, &occ));
    const uint64_t need = (b->D + (uint64_t)threads * RT - 1) / ((uint64_t)threads * RT);
    const uint64_t cap = (uint64_t)b->num_sms * std::max(1, std::min({occ, hv_cta_cap(), max_ctas}));
    const int grid = (int)std::max<uint64_t>(1, std::min(need, cap));
    kern<<<dim3(grid, blocks), threads, smem, stream>>>(b->tables(), bl, x, y, ep);
    note_launch();
    return FTLM_OK;
}

template <typename V, typename Lbl, bool CLT, bool LANCZOS, int RT, int B, int C>
ftlm_status launch(const ftlm_basis *b, const V *x, V *y, const EpiDev &ep, int blocks, cudaStream_t stream,
                   int max_ctas = kMaxBlocksPerSm)
{
    void *tok = profile_begin(kProfHv, stream, B * blocks);
    ftlm_status st = FTLM_OK;
    if constexpr (LANCZOS && !CLT) {
        // CR Lanczos step: one walk over the rows, or the split (walk A, then walk B
        // over the high-high bonds in the transposed order)
        HiWalk w;
        if (blocks == 1 && split_walks(b, B, sizeof(V), &w)) {
            const ftlm_dtype dt = sizeof(V) == 4 ? FTLM_F32 : FTLM_F64;
            LoWalk la;
            st = build_lo_walk(b, &la) ? launch_walk_a(b, la, dt, B, x, y, ep, stream)
                                       : fail(FTLM_EUNSUPPORTED, "split H.v without a walk A tile table");
            if (st == FTLM_OK) st = launch_walk_b(b, w, dt, B, x, y, ep, stream);
        } else {
            st = launch_rows<V, Lbl, false, kLanczos, RT, B, C>(b, b->bonds_cr, x, y, ep, blocks, max_ctas, stream);
        }
        if (st == FTLM_OK) {
            alpha_kernel<B><<<dim3(1, blocks), 32, 0, stream>>>(ep);
            note_launch();
        }
    } else {
        st = launch_rows<V, Lbl, CLT, LANCZOS ? kLanczos : kPlain, RT, B, C>(b, CLT ? b->bonds_clt : b->bonds_cr, x,
                                                                           y, ep, blocks, max_ctas, stream);
    }
    profile_end(tok, stream);
    if (st != FTLM_OK) return st;
    FTLM_CUDA(cudaGetLastError());
    return FTLM_OK;
}

// Bonds per chunk for 8-wide blocks (FTLM_HV_CHUNK = 2, 4 or 8 overrides the choice): a
// larger chunk keeps more gathers in flight per row, a smaller one leaves registers for
// more resident warps.  4, but 8 in lookup-table Lanczos launches with few rows, which
// the resident warps do not fill anyway.  us per launch with 4 and 8, S^z = 0 or 1/2:
// N = 16 16.6 and 15.7, 18 20.6 and 20.3, 19 26.8 and 24.2, 20 (0.18 M rows) 33.2 and 32.3, 21
// (0.35 M) 43.2 and 43.3; with combinatorial ranks 19 32.1 and 34.2.
//
// Blocks side by side have a grid each.  A block's grid fixes the order of its sums, so it is
// that of chunks of 8 (two CTAs per SM) for every sector of few rows, whichever chunk the
// launch takes; the chunk changes no result.  Chunks of 8 there while all CTAs fit in two per
// SM, and from the rows where a block alone fills those twice; between the two chunks of
// 4.  ms per run of 100 steps, two blocks, chunks of 4 and 8 (and 4 with the grid of three
// CTAs per SM that a block alone does not have): 320 rows per SM 4.46 and 5.23 (4.45), 608
// 6.29 and 6.39 (6.67), 829 7.43 and 7.10 (7.81), 1105 9.08 and 8.53 (8.31), 1215 8.76 and 8.56
// (8.65); three blocks 608 8.05 and 8.62 (9.05), 829 9.30 and 9.70 (10.28), 1105 13.8 and 13.3
// (13.1), 1215 13.8 and 13.5 (13.7).
constexpr uint64_t kChunk8Rows = 1280, kChunk8RowsBlocks = 2 * kRowThreads,
                   kChunk8RowsFull = 4 * kRowThreads;  // rows per SM

int chunk8(bool wide)
{
    static const int c = [] {
        const char *e = getenv("FTLM_HV_CHUNK");
        const int v = e ? atoi(e) : 0;
        return (v == 8 || v == 4 || v == 2) ? v : 0;
    }();
    return c ? c : (wide ? 8 : 4);
}

template <typename V, typename Lbl, bool CLT, bool LANCZOS>
ftlm_status launch_b(const ftlm_basis *b, int B, const void *x, void *y, const EpiDev &ep, int blocks,
                     cudaStream_t stream)
{
    const V *xv = (const V *)x;
    V *yv = (V *)y;
    if constexpr (sizeof(V) == 8) {
        switch (B) {
        case 4: return launch<V, Lbl, CLT, LANCZOS, 1, 4, f64_gathers<4>()>(b, xv, yv, ep, blocks, stream);
        case 8: return launch<V, Lbl, CLT, LANCZOS, 1, 8, f64_gathers<8>()>(b, xv, yv, ep, blocks, stream);
        case 16: return launch<V, Lbl, CLT, LANCZOS, 1, 16, f64_gathers<16>()>(b, xv, yv, ep, blocks, stream);
        default: return launch<V, Lbl, CLT, LANCZOS, 1, 1, f64_gathers<1>()>(b, xv, yv, ep, blocks, stream);
        }
    } else {
    switch (B) {
    case 4: return launch<V, Lbl, CLT, LANCZOS, 1, 4, 8>(b, xv, yv, ep, blocks, stream);
    case 8: {
        const bool few = CLT && LANCZOS && b->D <= kChunk8Rows * b->num_sms;
        const int ctas = few ? min_ctas<V, 1, 8, 8>() : kMaxBlocksPerSm;
        const bool wide = blocks == 1 || b->D * blocks <= kChunk8RowsBlocks * b->num_sms ||
                          b->D >= kChunk8RowsFull * b->num_sms;
        switch (chunk8(few && wide)) {
        case 8: return launch<V, Lbl, CLT, LANCZOS, 1, 8, 8>(b, xv, yv, ep, blocks, stream, ctas);
        case 2: return launch<V, Lbl, CLT, LANCZOS, 1, 8, 2>(b, xv, yv, ep, blocks, stream, ctas);
        default: return launch<V, Lbl, CLT, LANCZOS, 1, 8, 4>(b, xv, yv, ep, blocks, stream, ctas);
        }
    }
    case 16: return launch<V, Lbl, CLT, LANCZOS, 1, 16, 4>(b, xv, yv, ep, blocks, stream);
    default: break;
    }
    switch (rows_per_thread(CLT)) {
    case 1: return launch<V, Lbl, CLT, LANCZOS, 1, 1, 8>(b, xv, yv, ep, blocks, stream);
    case 4: return launch<V, Lbl, CLT, LANCZOS, 4, 1, 8>(b, xv, yv, ep, blocks, stream);
    default: return launch<V, Lbl, CLT, LANCZOS, 2, 1, 8>(b, xv, yv, ep, blocks, stream);
    }
    }
}

template <typename V, bool LANCZOS>
ftlm_status launch_mode(const ftlm_basis *b, int B, const void *x, void *y, const EpiDev &ep, int blocks,
                        cudaStream_t stream)
{
    if (b->mode == FTLM_RANK_CLT) return launch_b<V, uint32_t, true, LANCZOS>(b, B, x, y, ep, blocks, stream);
    if (b->N <= 32) return launch_b<V, uint32_t, false, LANCZOS>(b, B, x, y, ep, blocks, stream);
    return launch_b<V, uint64_t, false, LANCZOS>(b, B, x, y, ep, blocks, stream);
}

template <typename V>
ftlm_status launch_typed(const ftlm_basis *b, int B, const void *x, void *y, const LanczosHv *epi,
                         cudaStream_t stream)
{
    const EpiDev ep = epi_of(epi);
    if (epi) return launch_mode<V, true>(b, B, x, y, ep, epi->blocks, stream);
    return launch_mode<V, false>(b, B, x, y, ep, 1, stream);
}

}  // namespace

bool valid_block(int B) { return B == 1 || B == 4 || B == 8 || B == 16; }

bool hv_splits(const ftlm_basis *b, ftlm_dtype dtype, int B)
{
    HiWalk w;
    return b->two_s == 1 && b->mode == FTLM_RANK_CR && split_walks(b, B, dtype == FTLM_F32 ? 4 : 8, &w);
}

ftlm_status launch_hv(const ftlm_basis *b, ftlm_dtype dtype, int B, const void *x, void *y,
                      const LanczosHv *epi, cudaStream_t stream)
{
    if (b->two_s > 1) return launch_hv_spin(b, dtype, B, x, y, epi, stream);
    return dtype == FTLM_F32 ? launch_typed<float>(b, B, x, y, epi, stream)
                             : launch_typed<double>(b, B, x, y, epi, stream);
}

}  // namespace ftlm

namespace {
ftlm_status check_hv_args(const ftlm_basis *b, ftlm_dtype dtype, int B, const void *x_dev, void *y_dev)
{
    if (!b) return ftlm::fail(FTLM_EINVAL, "NULL basis");
    if (dtype != FTLM_F32 && dtype != FTLM_F64) return ftlm::fail(FTLM_EINVAL, "bad dtype");
    if (!x_dev || !y_dev) return ftlm::fail(FTLM_EINVAL, "NULL vector");
    if (x_dev == y_dev) return ftlm::fail(FTLM_EINVAL, "x and y must not overlap");
    // rows of 32 bytes or more move as 32-byte transactions
    const unsigned row = (unsigned)B * (dtype == FTLM_F32 ? 4u : 8u);
    const uintptr_t mask = row >= 32 ? 31u : 15u;
    if (((uintptr_t)x_dev | (uintptr_t)y_dev) & mask)
        return ftlm::fail(FTLM_EINVAL, row >= 32 ? "vectors must be 32-byte aligned for rows of 32 bytes or more"
                                                 : "vectors must be 16-byte aligned");
    return FTLM_OK;
}
}  // namespace

extern "C" ftlm_status ftlm_basis_hv_schedule(const ftlm_basis *b, int B, ftlm_dtype dtype, ftlm_hv_schedule *used)
{
    if (!b || !used) return ftlm::fail(FTLM_EINVAL, "NULL argument");
    if (!ftlm::valid_block(B)) return ftlm::fail(FTLM_EINVAL, "block width must be 1, 4, 8 or 16");
    if (dtype != FTLM_F32 && dtype != FTLM_F64) return ftlm::fail(FTLM_EINVAL, "bad dtype");
    *used = ftlm::hv_splits(b, dtype, B) ? FTLM_HV_SPLIT : FTLM_HV_ONE_WALK;
    return FTLM_OK;
}

extern "C" ftlm_status ftlm_hv(const ftlm_basis *b, ftlm_dtype dtype, const void *x_dev, void *y_dev,
                               void *stream)
{
    ftlm_status s = check_hv_args(b, dtype, 1, x_dev, y_dev);
    if (s != FTLM_OK) return s;
    return ftlm::launch_hv(b, dtype, 1, x_dev, y_dev, nullptr, (cudaStream_t)stream);
}

extern "C" ftlm_status ftlm_hv_block(const ftlm_basis *b, ftlm_dtype dtype, int B, const void *x_dev,
                                     void *y_dev, void *stream)
{
    if (!ftlm::valid_block(B)) return ftlm::fail(FTLM_EINVAL, "block width must be 1, 4, 8 or 16");
    ftlm_status s = check_hv_args(b, dtype, B, x_dev, y_dev);
    if (s != FTLM_OK) return s;
    return ftlm::launch_hv(b, dtype, B, x_dev, y_dev, nullptr, (cudaStream_t)stream);
}
