// Chain state on the device and the launches of the sweeps (arXiv:1212.3975, Secs. 2-3):
// infinite-temperature start, recount of E and M, unpacking, the staging plan and the
// shape of a sweep launch.  The sweeps themselves are in sweep_body.cuh.
#include <algorithm>
#include <cstdio>

#include "sweep_small.cuh"

namespace muca {
namespace {

// ---------------------------------------------------------------------------
// Infinite-temperature start (Sec. 3): spins from Philox phase 0, one thread per
// (word, chain).  Ising: site i takes word i & 3 of block i >> 2, s = +1 iff its
// top bit is set.  Potts: the same words, s = (word * q) >> 32.
// ---------------------------------------------------------------------------
__global__ void init_lattice_kernel(uint32_t *lat, int model, int L, int q, int p, int p_pad, int row_words,
                                    int lat_words, uint32_t key0, uint32_t ctr3, int *fault)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *fault = 0;
    const size_t total = (size_t)lat_words * p_pad;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(t / lat_words), k = (int)(t % lat_words);
        uint32_t word = 0u;
        if (c < p) {
            const int y = k / row_words, w = k % row_words;
            const int per = model == MUCA_ISING ? 32 : 4;
            uint4 b = make_uint4(0u, 0u, 0u, 0u);
            for (int j = 0; j < per; ++j) {
                const int x = per * w + j;
                if (x >= L) break;
                const int i = y * L + x;
                if (j == 0 || (i & 3) == 0) b = philox4x32_10(make_uint4((uint32_t)i >> 2, 0u, 0u, ctr3), key0, (uint32_t)c);
                const uint32_t r = (i & 3) == 0 ? b.x : (i & 3) == 1 ? b.y : (i & 3) == 2 ? b.z : b.w;
                if (model == MUCA_ISING)
                    word |= (r >> 31) << j;
                else
                    word |= __umulhi(r, (uint32_t)q) << (8 * j);
            }
        }
        lat[t] = word;
    }
}

__device__ __forceinline__ uint32_t site_value(const uint32_t *lat, int model, int row_words, int x, int y)
{
    if (model == MUCA_ISING) return (lat[y * row_words + (x >> 5)] >> (x & 31)) & 1u;
    return (lat[y * row_words + (x >> 2)] >> (8 * (x & 3))) & 0xFFu;
}

// Full recount of E, M and (Potts) the state counts, one warp per chain.
__global__ void recount_kernel(const uint32_t *lat_all, int32_t *E, int32_t *M, uint64_t *cnt, int model, int L, int q,
                               int p, int p_pad, int row_words, int lat_words)
{
    const int c = (int)(((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (c >= p) return;
    const uint32_t *lat = lat_all + (size_t)c * lat_words;
    int e = 0, m = 0;
    uint32_t count[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int y = lane / L, x = lane % L;
    for (int i = lane; i < L * L; i += 32) {
        const uint32_t s = site_value(lat, model, row_words, x, y);
        const uint32_t r = site_value(lat, model, row_words, x + 1 == L ? 0 : x + 1, y);
        const uint32_t d = site_value(lat, model, row_words, x, y + 1 == L ? 0 : y + 1);
        if (model == MUCA_ISING) {
            e -= (s == r ? 1 : -1) + (s == d ? 1 : -1);
            m += s ? 1 : -1;
        } else {
            e -= (s == r ? 1 : 0) + (s == d ? 1 : 0);
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k) count[k] += (s & 7u) == k ? 1u : 0u;
        }
        x += 32;
        while (x >= L) {
            x -= L;
            ++y;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(~0u, e, o);
        m += __shfl_xor_sync(~0u, m, o);
        if (model == MUCA_POTTS) {
#pragma unroll
            for (int k = 0; k < 8; ++k) count[k] += __shfl_xor_sync(~0u, count[k], o);
        }
    }
    if (lane) return;
    if (model == MUCA_POTTS) {
        uint64_t lo = 0, hi = 0;
        uint32_t mx = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            lo |= (uint64_t)count[k] << (16 * k);
            hi |= (uint64_t)count[k + 4] << (16 * k);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) mx = max(mx, count[k]);
        cnt[c] = lo;
        cnt[p_pad + c] = hi;
        m = q * (int)mx - L * L;
    }
    E[c] = e;
    M[c] = m;
}

__global__ void unpack_kernel(const uint32_t *lat, int8_t *out, int model, int L, int p, int row_words, int lat_words)
{
    const size_t V = (size_t)L * L;
    const size_t total = V * (size_t)p;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const size_t c = t / V;
        const int i = (int)(t % V);
        const uint32_t s = site_value(lat + c * lat_words, model, row_words, i % L, i / L);
        out[t] = model == MUCA_ISING ? (int8_t)(s ? 1 : -1) : (int8_t)s;
    }
}

}  // namespace

namespace {
// Cycles of a row with n groups per block, measured.  Rows decided at once: one deciding
// warp per scheduler 680, two or three 600 and 42 per group (64 x 64: 670 in blocks of 4
// groups, 845 of 6, 930 of 8, 1110 of 12).  A lane per chain (16 < L <= 32), per site: 61 to
// 77 (18 x 18 to 32 x 32) with at most two deciding and two drawing warps on schedulers of
// their own, 77 to 85 with three or four groups, 127 with 6, 144 with 8, 200 with 12.
double row_cycles(int n) { return n <= 4 ? 680.0 : 600.0 + 42.0 * n; }
double lane_row_cycles(int L, int n)
{
    return L * (n <= 2 ? 40.0 + 1.15 * L : n <= 4 ? 66.0 + 0.6 * L : 50.0 + 12.0 * n);
}
long waves_of(long groups, int per_block, int n_sm) { return ((groups + per_block - 1) / per_block + n_sm - 1) / n_sm; }

// Whether a launch takes the body with a lane per chain.  Up to kSmallL always.  Up to
// kLaneL a row's 18 to 32 sites one after the other take two to four times as long as the
// row at once, but 32 chains per warp instead of four: with many chains the lattices of a
// launch need fewer waves.  Both are costed, rows with a tenth more for repeated passes
// (iterations of 2^16 sites with late weights, rows / lanes: 20 x 20, p = 7000 1918 / 2025
// us, 9728 2870 / 1931, 16384 5192 / 2409; 32 x 32, p = 9728 2097 / 2432, 16384 3787 / 2661,
// 29184 5455 / 4006).
bool lane_per_chain(const muca_ctx *ctx, int groups)
{
    if (ctx->model != MUCA_ISING || ctx->L > sweep::kLaneL) return false;
    if (ctx->L <= sweep::kSmallL) return true;
    if (groups > 0 || ctx->cfg.staging == MUCA_STAGING_GLOBAL) return false;  // (batches; lattices not staged)
    const long lanes = ((long)ctx->p + 31) / 32, rows = ((long)ctx->p + 3) / 4;
    double lane_best = 1e30, row_best = 1e30;
    for (int n = 1; n <= sweep::kMaxGroups; ++n) {
        row_best = std::min(row_best, waves_of(rows, n, ctx->n_sm) * row_cycles(n));
        if (sweep::small_smem(ctx->L, ctx->n_bins, ctx->lat_words, n, true) <= (size_t)kMaxSmem)
            lane_best = std::min(lane_best, waves_of(lanes, n, ctx->n_sm) * lane_row_cycles(ctx->L, n));
    }
    return lane_best < 1.1 * row_best;
}
// lanes per chain (1: one, site by site), and whether a row is one pass: the fewest
// lanes that hold a row of four sites per lane, so that no lane is idle in full launches
// (8-Potts 8 x 8, p = 16384, 200 sweeps and an update: two lanes 1.20 ms, four 1.80)
void lanes_of(const muca_ctx *ctx, int groups, int &lpc, bool &row)
{
    const int L = ctx->L;
    lpc = lane_per_chain(ctx, groups) ? 1 : L <= 8 ? 2 : L <= 16 ? 4 : L <= 32 ? 8 : L <= 64 ? 16 : 32;
    row = L <= 128;
}
size_t launch_smem(const muca_ctx *ctx, const SweepPlan &pl, bool hist, bool lattice, int groups, int lpc)
{
    if (lpc == 1) return sweep::small_smem(ctx->L, ctx->n_bins, ctx->lat_words, groups, hist);
    const size_t lat = lattice ? ((size_t)ctx->lat_words * 4 * (32 / lpc) * groups + 15) & ~(size_t)15 : 0;
    return pl.table_bytes + (hist ? pl.hist_bytes : 0) + lat + sweep::ring_bytes(ctx->model) * groups;
}
}  // namespace

int hist_mode(const SweepPlan &pl)
{
    return !pl.hist_smem ? sweep::kHistGlobal : pl.hist16 ? sweep::kHist16 : pl.hist_pairs ? sweep::kHistPairs
                                                                                           : sweep::kHistSingle;
}

// Groups per block (`groups` > 0: that many; muca_config.chains_per_block > 0: its chains):
// the fewest cycles over all waves, blocks beyond one per SM waiting for another wave.  (At
// 170 cycles per group more waves of smaller blocks were taken: 256 x 256, p = 8192, 6 waves
// of 9 groups 7.62 ms, 5 of 11 6.83 ms; 64 x 64, p = 16000, 10 sweeps, 6 of 9 2.14 ms, 5 of
// 11 1.95 ms.)  Of equal costs the fewest groups, on more SMs, deciding and drawing warps on
// schedulers of their own (8-Potts 32 x 32, p = 639, 2 or 1 groups instead of 4: 413 against
// 530 us; 8 x 8, p = 1024: 291 against 352).
SweepShape sweep_shape(const muca_ctx *ctx, const SweepPlan &pl, bool hist, int groups)
{
    SweepShape s;
    lanes_of(ctx, groups, s.lpc, s.row);
    const long all = ((long)ctx->p * s.lpc + 31) / 32;
    auto staged = [&](int G) {
        // launches without a histogram stage the lattices in the room it leaves
        if (!hist && ctx->cfg.staging == MUCA_STAGING_AUTO)
            return launch_smem(ctx, pl, false, true, G, s.lpc) <= (size_t)kMaxSmem;
        return pl.lattice_smem;
    };
    if (groups <= 0 && ctx->cfg.chains_per_block > 0)  // the caller's, as far as there are so many warps and chains
        groups = (int)std::min<long>(std::min<long>(ctx->cfg.chains_per_block * s.lpc / 32, sweep::kMaxGroups), all);
    int G = groups;
    if (groups <= 0) {
        double best = 0.0;
        for (int n = 1; n <= std::min<long>(sweep::kMaxGroups, all); ++n) {
            if (n > 1 && launch_smem(ctx, pl, hist, staged(n), n, s.lpc) > (size_t)kMaxSmem) break;
            const double t = waves_of(all, n, ctx->n_sm) *
                             (s.lpc == 1 && ctx->L > sweep::kSmallL ? lane_row_cycles(ctx->L, n) : row_cycles(n));
            if (best == 0.0 || t < best) {
                best = t;
                G = n;
            }
        }
    }
    s.lattice = staged(G);
    while (G > 1 && launch_smem(ctx, pl, hist, s.lattice, G, s.lpc) > (size_t)kMaxSmem) --G;
    s.groups = G;
    s.chains = (32 / s.lpc) * G;
    s.smem = launch_smem(ctx, pl, hist, s.lattice, G, s.lpc);
    return s;
}

// Whether a launch may take its staging: the lattices of 32 chains beside the table and the
// histogram, as callers know it (muca.h), and what the block that runs really takes (fewer
// chains and a ring per group: it always fits where the first does).
bool staging_fits(const SweepPlan &pl, const SweepShape &s)
{
    return pl.smem_bytes <= (size_t)kMaxSmem && s.smem <= (size_t)kMaxSmem;
}

SweepPlan plan_sweeps(const muca_ctx *ctx, bool allow_compact, int groups)
{
    SweepPlan pl;
    const bool ising = ctx->model == MUCA_ISING;
    const int staging = ctx->cfg.staging, width = ktab_width(ctx->model);
    pl.compact = pl.t16 = pl.hist16 = pl.hist_pairs = false;
    if (lane_per_chain(ctx, groups)) {  // that body stages everything
        pl.table_smem = pl.hist_smem = pl.lattice_smem = true;
        pl.smem_bytes = sweep::small_smem(ctx->L, ctx->n_bins, ctx->lat_words, 1, true);
        pl.table_bytes = pl.hist_bytes = 0;  // (sizes of its own: launch_smem)
        return pl;
    }
    // room beside the draw rings of four groups
    const size_t cap = (size_t)kMaxSmem - 4 * sweep::ring_bytes(ctx->model);
    const size_t table = ((size_t)ctx->n_bins * width * 4 + 15) & ~(size_t)15;
    // (+ one slot per lane for lanes that have nothing to count)
    const size_t hist = (((size_t)ctx->n_bins * 4 + 15) & ~(size_t)15) + 128;
    const size_t lat = (size_t)ctx->lat_words * 4 * 32;
    size_t used = 0;
    // (Ising 64 x 64: 82 KB, 8-Potts 32 x 32: 74 KB)
    pl.table_smem = ctx->L <= (ising ? 64 : 32);
    if (pl.table_smem) used += table;
    pl.hist_smem = used + hist <= 160 * 1024;
    // Ising histograms too large for 32-bit counts in shared memory (256 x 256: 262 KB):
    // 16-bit counts, two bins per word, flushed into the merged histogram by rows
    // (otherwise every bin change of a chain is a global atomic), where the lattices of 32
    // chains could not be staged anyway
    const size_t hist16 = ((((size_t)ctx->n_bins + 1) / 2 * 4 + 15) & ~(size_t)15) + 128;
    if (!pl.hist_smem && ising && staging != MUCA_STAGING_SHARED && used + lat > cap && used + hist16 <= 160 * 1024)
        pl.hist_smem = pl.hist16 = true;  // (the table is in global memory here too)
    if (pl.hist_smem) used += pl.hist16 ? hist16 : hist;
    pl.lattice_smem = staging == MUCA_STAGING_SHARED || (staging == MUCA_STAGING_AUTO && used + lat <= cap);
    if (pl.lattice_smem) used += lat;
    pl.smem_bytes = used;
    pl.table_bytes = pl.table_smem ? table : 0;
    pl.hist_bytes = pl.hist_smem ? (pl.hist16 ? hist16 : hist) : 0;
    // more groups of 32 chains than SMs: the lattices of Ising launches with a histogram
    // stay in global memory where a block of eight groups would take more than half of an
    // SM's shared memory
    const long groups32 = (ctx->p + 31) / 32, n_sm = ctx->n_sm;
    const size_t per_sm = (size_t)ctx->smem_per_sm, reserved = (size_t)ctx->smem_reserved;
    if (allow_compact && ising && staging != MUCA_STAGING_SHARED && groups32 > n_sm && pl.table_smem &&
        2 * (used + 8 * sweep::ring_bytes(ctx->model) + reserved) > per_sm) {
        pl.compact = true;
        pl.hist_smem = true;
        pl.lattice_smem = false;
        pl.smem_bytes = table + hist;
        pl.hist_bytes = hist;
        // two to two and a half such groups per SM at L = 64: the table of the upper 16-bit
        // halves of the thresholds (ties read the 32-bit table).  Kept only because the plan of
        // this size is asserted (MUCA_PLAN_TABLE16), not for speed: 20 sweeps at p = 9824 take
        // 2.84 ms with it and 2.67 with the 32-bit table, 11000 3.54 / 3.31, 12160 3.56 / 3.33,
        // p = 14592 (and an update) 4.33 / 3.47.
        if (ctx->L == 64 && groups32 > 2 * n_sm && 2 * groups32 <= 5 * n_sm) {
            const size_t table16 = ((size_t)ctx->n_bins * 5 * 2 + 15) & ~(size_t)15;
            pl.t16 = true;
            pl.smem_bytes = table16 + hist;
            pl.table_bytes = table16;
        }
        return pl;
    }
    // the histogram of attempt pairs (one count per bin change of a single attempt: 5 for
    // Ising, 9 for Potts) halves the atomics; where it fits beside the table, the lattices
    // and the rings.  Pairs lie within a lane's four sites, so L % 4 == 0.
    const size_t pairs = (((size_t)ctx->n_bins * width * 4 + 15) & ~(size_t)15) + 128;
    if (ctx->L % 4 == 0 && pl.table_smem && pl.hist_smem && used - hist + pairs <= cap) {
        SweepPlan pp = pl;
        pp.hist_pairs = true;
        pp.hist_bytes = pairs;
        pp.smem_bytes = used - hist + pairs;
        if (sweep_shape(ctx, pp, true, groups).groups == sweep_shape(ctx, pl, true, groups).groups) pl = pp;
    }
    return pl;
}

int plan_flags(const SweepPlan &pl)
{
    return (pl.lattice_smem ? MUCA_PLAN_LATTICE_SMEM : 0) | (pl.hist_smem ? MUCA_PLAN_HIST_SMEM : 0) |
           (pl.table_smem ? MUCA_PLAN_TABLE_SMEM : 0) | (pl.hist_pairs ? MUCA_PLAN_PAIR_HIST : 0) |
           (pl.compact ? MUCA_PLAN_COMPACT : 0) | MUCA_PLAN_WARP_SPECIALIZED |
           (pl.t16 ? MUCA_PLAN_TABLE16 : 0) | (pl.hist16 ? MUCA_PLAN_HIST16 : 0);
}

int launch_sweeps(muca_ctx *ctx, uint32_t phase, int n_sweeps, uint32_t sweep0, uint32_t iteration, bool hist,
                  int32_t *E_rec, int32_t *M_rec, bool samples)
{
    if (ctx->cfg.ensemble == MUCA_ENSEMBLE_MAGNETIZATION)
        return launch_muma_sweeps(ctx, phase, n_sweeps, sweep0, iteration, hist, E_rec, M_rec);
    int rc = check_fault(ctx);
    if (rc) return rc;
    const SweepPlan pl = plan_sweeps(ctx);
    if (ctx->ktab_dirty && (rc = launch_ktab(ctx))) return rc;
    const SweepShape shape = sweep_shape(ctx, pl, hist);
    if (!staging_fits(pl, shape))
        return fail(MUCA_ERR_ARG, "shared-memory staging does not fit: " + std::to_string(pl.smem_bytes) + " bytes");
    SweepArgs a;
    a.lat = ctx->d_lat;
    a.E = ctx->d_E;
    a.M = ctx->d_M;
    a.cnt = ctx->d_cnt;
    a.ktab = ctx->d_ktab;
    a.ktab31 = ctx->d_ktab + (size_t)ctx->n_bins * ktab_width(ctx->model);
    a.H = ctx->d_H;
    a.samples = samples ? ctx->d_samples : nullptr;
    a.L = ctx->L;
    a.p = ctx->p;
    a.p_pad = ctx->p_pad;
    a.row_words = ctx->row_words;
    a.lat_words = ctx->lat_words;
    a.n_bins = ctx->n_bins;
    a.iteration = iteration;
    a.ctr3 = ((uint32_t)(ctx->seed >> 32) << 2) | phase;
    a.key0 = (uint32_t)ctx->seed;
    a.rec_stride = ctx->p;
    a.fault = ctx->h_fault;
    const int blocks = (ctx->p + shape.chains - 1) / shape.chains;
    const int chunk = max_launch_sweeps(shape.chains, ctx->V);
    for (int done = 0; done < n_sweeps; done += chunk) {
        a.n_sweeps = std::min(chunk, n_sweeps - done);
        a.sweep0 = sweep0 + (uint32_t)done;
        a.E_rec = E_rec ? E_rec + (size_t)done * ctx->p : nullptr;
        a.M_rec = M_rec ? M_rec + (size_t)done * ctx->p : nullptr;
        const SweepLaunch l{a, pl, shape, blocks, ctx->stream};
        cudaError_t e = ctx->model == MUCA_ISING ? launch_sweep_ising(l, hist) : launch_sweep_potts(l, hist);
        if (e != cudaSuccess) return cuda_fail(e, "sweep kernel launch");
        note_launches(1);
    }
    return MUCA_OK;
}

int launch_init_lattice(muca_ctx *ctx)
{
    const size_t total = (size_t)ctx->lat_words * ctx->p_pad;
    const int grid = (int)std::min<size_t>((size_t)ctx->n_sm * 16, (total + 127) / 128);
    init_lattice_kernel<<<grid, 128, 0, ctx->stream>>>(ctx->d_lat, ctx->model, ctx->L, ctx->q, ctx->p, ctx->p_pad,
                                                      ctx->row_words, ctx->lat_words, (uint32_t)ctx->seed,
                                                      ((uint32_t)(ctx->seed >> 32) << 2) | kPhaseInit, ctx->h_fault);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return launch_recount(ctx);
}

int launch_recount(muca_ctx *ctx)
{
    recount_kernel<<<(ctx->p + 3) / 4, 128, 0, ctx->stream>>>(ctx->d_lat, ctx->d_E, ctx->d_M, ctx->d_cnt, ctx->model,
                                                             ctx->L, ctx->q, ctx->p, ctx->p_pad, ctx->row_words,
                                                             ctx->lat_words);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return MUCA_OK;
}

int launch_unpack_spins(muca_ctx *ctx, int8_t *d_out)
{
    const size_t total = (size_t)ctx->V * ctx->p;
    const int grid = (int)std::min<size_t>((size_t)ctx->n_sm * 16, (total + 255) / 256);
    unpack_kernel<<<grid, 256, 0, ctx->stream>>>(ctx->d_lat, d_out, ctx->model, ctx->L, ctx->p, ctx->row_words,
                                                ctx->lat_words);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return MUCA_OK;
}

}  // namespace muca
