// Internal declarations of libmuca (not part of the C ABI).
//
// Device data layout (chain-major, so that the lanes that share a chain read its rows
// from consecutive bytes):
//   Ising: one bit per site, bit j of word w of row y holds site x = 32 w + j
//          (1 = spin +1); row_words = ceil(L / 32).
//   Potts: one byte per site, byte j of word w of row y holds site x = 4 w + j;
//          row_words = ceil(L / 4).
//   word k = y * row_words + w of chain c lives at lat[c * lat_words + k]; bits and bytes
//   past a row's last site are zero.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>
#include <string>

#include "muca.h"

namespace muca {

constexpr uint32_t kAlways = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of the 4 x 32-bit
// S-P network, multipliers 0xD2511F53 / 0xCD9E8D57, Weyl key bumps 0x9E3779B9 /
// 0xBB67AE85 between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 ctr, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        if (round > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t lo0 = 0xD2511F53u * ctr.x;
        const uint32_t hi0 = __umulhi(0xD2511F53u, ctr.x);
        const uint32_t lo1 = 0xCD9E8D57u * ctr.z;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, ctr.z);
        ctr = make_uint4(hi1 ^ ctr.y ^ k0, lo1, hi0 ^ ctr.w ^ k1, lo0);
    }
    return ctr;
}

// counter word 3: (seed >> 32) << 2 | phase
enum Phase : uint32_t { kPhaseInit = 0, kPhaseIterate = 1, kPhaseThermalize = 2, kPhaseProduce = 3 };

__host__ __device__ inline int n_bins_of(int model, int L)
{
    return model == MUCA_ISING ? L * L + 1 : 2 * L * L + 1;
}
__host__ __device__ inline int n_de_of(int model) { return model == MUCA_ISING ? 4 : 8; }

// Arguments of one sweep launch (plain values and device pointers).
struct SweepArgs {
    uint32_t *lat;        // [p_pad][lat_words]
    int32_t *E;           // [p_pad] running energy
    int32_t *M;           // [p_pad] running magnetisation (Ising) / record scratch
    uint64_t *cnt;        // Potts packed state counts [2][p_pad]
    const uint32_t *ktab; // kernel table: Ising [n_bins][5] by unequal neighbours, Potts [n_bins][9] by dE+4
    const uint32_t *ktab31; // the same, entries >> 1
    uint64_t *H;          // merged histogram [n_bins] (uint64, atomically added)
    int32_t *E_rec;       // [n_sweeps][rec_stride] or null
    int32_t *M_rec;
    uint64_t *samples;    // [3][n_bins] production sums (n, sum|M|, sum M^2) or null
    int L, p, p_pad, row_words, lat_words, n_bins;
    int n_sweeps;
    uint32_t sweep0;      // counter word 1 of the first sweep
    uint32_t iteration;   // counter word 2
    uint32_t ctr3;        // counter word 3 = (seed_hi << 2) | phase
    uint32_t key0;        // low 32 bits of the seed
    int rec_stride;       // records row stride (= p)
    int *fault;           // set where a pass did not settle (muca_ctx::h_fault)
};

// staging of the sweep launches of a context
struct SweepPlan {
    bool table_smem, hist_smem;
    bool lattice_smem;      // of launches with a histogram (the others take what room it leaves)
    bool hist_pairs;        // shared histogram of attempt pairs
    bool compact;           // many chains: lattices in global memory, histogram of single attempts
    bool t16;               // compact with a table of 16-bit threshold halves
    bool hist16;            // histogram of 16-bit counts, two bins per word, flushed by rows
    size_t smem_bytes;      // staging of the plan for 32 chains (table, histogram, lattices)
    size_t table_bytes, hist_bytes;
};

// Shape of a sweep launch: lanes per chain, whether a row is one pass, groups (warps of
// 32 / lpc chains) per block, lattices staged, shared memory.
struct SweepShape {
    int lpc;
    bool row;
    int groups, chains;  // per block
    bool lattice;
    size_t smem;
};

// Sweeps of one launch at most, `chains` chains per block: a block's 32-bit histogram
// counts (every chain in one bin), the sums of them that its flush makes and the draw
// positions stay below 2^31.
inline int max_launch_sweeps(int chains, int V)
{
    const uint64_t per_sweep = (uint64_t)(chains > 32 ? chains : 32) * (uint64_t)(V + 3), n = (1ull << 31) / per_sweep;
    return n < 1 ? 1 : n > (1u << 30) ? 1 << 30 : (int)n;
}
// Launches that n_sweeps sweeps take: `split` or as many as `most` sweeps per launch need
// (launch s of them makes the sweeps from n s / launches to n (s + 1) / launches).
inline int sweep_launches(int n_sweeps, int split, int most)
{
    const int need = n_sweeps / most + (n_sweeps % most != 0);
    const int n = split > need ? split : need;
    return n < 1 ? 1 : n < n_sweeps ? n : n_sweeps;
}

// Device view of one lattice of a batch (pointers into its context).
struct BatchJob {
    int model, L, p, p_pad, row_words, lat_words, n_bins, n_de, V;
    int accumulated, width;
    uint32_t key0, ctr3_iter;   // seed low word; counter word 3 of weight iterations
    uint32_t *lat;
    int32_t *E, *M;
    uint64_t *cnt;
    double *lnw, *P, *wscratch;
    uint8_t *acc;
    uint32_t *thr, *ktab;
    uint64_t *H;
    muca_iter_stats *stats;
    uint32_t *iteration;        // device counter of weight iterations (counter word 2)
    int hist, lattice;          // staging of the sweep body (sweep_body.cuh)
    int lpc, row;               // lanes per chain; a row is one pass
    int *active;                // 0: the lattice is frozen (converged) and every batch kernel skips it
    int *fault;                 // muca_ctx::h_fault
    int *conv;                  // iteration at which the lattice converged, -1 before
    uint32_t ctr3_therm;        // counter word 3 of thermalisation sweeps
    uint32_t *therm;            // device counter of thermalisation sweeps (counter word 1)
};

}  // namespace muca

// Host-side context (opaque to callers).
struct muca_ctx {
    int model, L, q, p, V, n_bins, n_de;
    uint64_t seed;
    muca_config cfg;
    cudaStream_t stream;
    int device;
    int n_sm;                 // streaming multiprocessors of the device (queried at init)
    int smem_per_sm;          // shared memory per SM and reserved per block (bytes, queried)
    int smem_reserved;
    int row_words, lat_words, p_pad;
    // device state
    uint32_t *d_lat;
    int32_t *d_E, *d_M;
    uint64_t *d_cnt;
    double *d_lnw, *d_P, *d_lnw_prod, *d_wscratch;
    uint8_t *d_acc;
    uint32_t *d_thr;
    uint32_t *d_ktab;         // thresholds re-indexed for the sweep kernels
    int ktab_dirty;
    uint64_t *d_H;
    uint64_t *d_samples;      // [3][n_bins]
    muca_iter_stats *d_stats;
    muca_iter_stats *h_stats; // pinned
    int *h_fault;             // pinned, behind h_stats: set by a sweep whose pass did not settle
    // production series scratch (used when the caller passes host or null buffers)
    int32_t *d_series;        // [2][series_cap]
    size_t series_cap;        // records per array
    // reweighting scratch: per-bin table inputs, and outputs/betas of one call
    void *d_rw;
    size_t rw_bytes;
    double *d_rwout;
    size_t rwout_cap;         // doubles
    void *d_rwtile;           // per-call tile scratch of the reweighting (grown on demand)
    size_t rwtile_bytes;
    // counters and flags
    uint32_t iteration;
    uint32_t sweeps_therm, sweeps_prod;
    int have_hist;
    int samples_active;
    uint64_t lnw_version, samples_lnw_version;
    // metric log: host clock at the start of the last iteration's sweeps, its attempts
    double it_t0, it_attempts;
};

namespace muca {

// error plumbing (thread-local message)
int fail(int code, const std::string &msg);
int cuda_fail(cudaError_t e, const char *what);
void note_launches(uint64_t n);
// MUCA_ERR_TIMEOUT if a sweep of the context gave up on a pass (the chains are then not
// those of the method until a reset); asked before sweeps and after every wait for them
int check_fault(const muca_ctx *ctx);

// NVTX range around an entry point (visible in profilers; free without one attached)
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};
#define MUCA_RANGE(name) ::muca::NvtxRange muca_range_(name)

// Test hook: with the environment variable MUCA_TEST_FAIL_ALLOC=k the k-th allocation
// of the process (device or pinned host memory, counting from 1) fails as if no memory
// were left, so that the clean-up of every allocation path can be tested without a GPU
// fault.
bool alloc_should_fail();

#define MUCA_CUDA_TRY(call)                                           \
    do {                                                              \
        cudaError_t e_ = (call);                                      \
        if (e_ != cudaSuccess) return ::muca::cuda_fail(e_, #call);   \
    } while (0)

// launches (defined in the kernel translation units)
int launch_init_lattice(muca_ctx *ctx);
int launch_recount(muca_ctx *ctx);
int launch_sweeps(muca_ctx *ctx, uint32_t phase, int n_sweeps, uint32_t sweep0,
                  uint32_t iteration, bool hist, int32_t *E_rec, int32_t *M_rec,
                  bool samples);
int launch_unpack_spins(muca_ctx *ctx, int8_t *d_out);
int launch_thresholds(muca_ctx *ctx);
int launch_update(muca_ctx *ctx);
int launch_reweight(muca_ctx *ctx, const double *d_betas, int n_beta, int precision,
                    double *const out[4] /* e, C, absm, chi: device [n_beta] each */);
constexpr int kMaxSmem = 227 * 1024;
// groups per block: 0 for as many as suit p (a batch's blocks have a fixed number)
SweepPlan plan_sweeps(const muca_ctx *ctx, bool allow_compact = true, int groups = 0);
SweepShape sweep_shape(const muca_ctx *ctx, const SweepPlan &pl, bool hist, int groups = 0);
bool staging_fits(const SweepPlan &pl, const SweepShape &s);
int hist_mode(const SweepPlan &pl);
int plan_flags(const SweepPlan &pl);  // MUCA_PLAN_* bit mask
constexpr int kBatchGroups = 4;       // groups of chains per work unit of a batch
// sweeps of one launch of a batch that holds this lattice, at most
int batch_max_sweeps(const muca_ctx *ctx);
cudaError_t launch_batch_update(const BatchJob *d_jobs, int n_jobs, int max_bins, int max_thr, cudaStream_t st);
int launch_ktab(muca_ctx *ctx);
// kernel table: Ising [n_bins][5] by unequal neighbours, Potts [n_bins][9] by dE + 4
__host__ __device__ constexpr int ktab_width(int model) { return model == MUCA_ISING ? 5 : 9; }
// Scratch of the tiled reweighting kernels (reweight_kernels.cu): a per-bin part (five
// FP64 arrays, a float copy of ln Omega, the sampled range) and a per-call part for
// n_beta betas (tile parameters, shifts, item offsets, partial sums), 256-byte aligned
// pieces.
constexpr int kRwTile = 8;          // betas per tile
constexpr int kRwMaxChunks = 32;    // bin chunks per tile at most
constexpr size_t kRwTileParamsBytes = 72;
constexpr size_t rw_align256(size_t b) { return (b + 255) & ~(size_t)255; }
// per-bin part: five FP64 arrays (the second, bin energies, is the BF16 path's; the tiled
// kernels keep the sampled range of every 64 bins there), five float arrays (ln Omega and
// mean |M| as float pairs, the within-bin variance), a free piece of 8 bytes per 256 bins
// (callers know the size of the whole), and the completion counter of the setup kernel
// (zero between calls: zeroed with the scratch, reset by its last user)
constexpr size_t rw_bin_part_bytes(size_t nb)
{
    return rw_align256(5 * nb * 8) + 5 * rw_align256(nb * 4) + rw_align256(8 * ((nb + 255) / 256)) + 256;
}
// per-call part: tile parameters, shifts (FP64, and the float constants of every beta),
// every beta's reference bin (mean |M| in FP64 and as a float pair),
// item offsets, the tiles' completion counters (each zeroed by its setup block), the
// tile of every item, partial sums
constexpr size_t rw_tile_part_bytes(size_t n_beta)
{
    return rw_align256(kRwTileParamsBytes * ((n_beta + kRwTile - 1) / kRwTile)) + rw_align256(8 * n_beta) +
           rw_align256(16 * n_beta) + rw_align256(8 * n_beta) + rw_align256(8 * n_beta) +
           rw_align256(4 * ((n_beta + kRwTile - 1) / kRwTile + 1)) +
           rw_align256(4 * ((n_beta + kRwTile - 1) / kRwTile + 1)) +
           rw_align256(4 * ((n_beta + kRwTile - 1) / kRwTile) * kRwMaxChunks) +
           8 * ((n_beta + kRwTile - 1) / kRwTile) * kRwMaxChunks * kRwTile * 6;
}
// allocation-free reweighting (reweight_noalloc.cu): the bins and betas per pass it
// serves, its fixed scratch and the launch on caller buffers
constexpr int kNoallocMaxBins = 16385;       // Ising L <= 128, 8-Potts L <= 90
constexpr int kNoallocBetasPerPass = 512;
constexpr size_t kNoallocScratchBytes = rw_bin_part_bytes(kNoallocMaxBins) + rw_tile_part_bytes(kNoallocBetasPerPass);
cudaError_t launch_reweight_buffers(double *scratch, const uint64_t *samples, const double *lnw, int model, int L,
                                    int q, const double *d_betas, int n_beta, int precision, double *d_out, int n_sm,
                                    cudaStream_t st);
// multimagnetic Ising ensemble (muma.cu)
int launch_muma_thresholds(muca_ctx *ctx);
int launch_muma_sweeps(muca_ctx *ctx, uint32_t phase, int n_sweeps, uint32_t sweep0, uint32_t iteration, bool hist,
                       int32_t *E_rec, int32_t *M_rec);
// one sweep launch of either model (sweep_ising.cu, sweep_potts.cu)
struct SweepLaunch {
    const SweepArgs &args;
    const SweepPlan &plan;
    const SweepShape &shape;
    int blocks;
    cudaStream_t stream;
};
cudaError_t launch_sweep_ising(const SweepLaunch &l, bool hist);
cudaError_t launch_sweep_potts(const SweepLaunch &l, bool hist);

}  // namespace muca
