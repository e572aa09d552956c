// Multimagnetic Ising ensemble (Sec. 4, Fig. 6): the weights live on the
// magnetisation M at a fixed inverse temperature beta, so a chain samples
// W(M) exp(-beta E) and the histograms are over the V+1 bins (M + V)/2.
//
// Threshold table: per M bin 10 columns, column 5 (s == +1) + n for the flipped spin s
// and its n unequal neighbours; then E' - E = 8 - 4n and the bin moves by -s.  The
// sweep kernel is one thread per chain over the bit-packed lattice, in typewriter
// order, with the Ising random streams (group i >> 2, word i & 3) and the integer
// acceptance test (A = 2^32-1 or u < A); the histogram is incremented after every
// attempt.
#include <cmath>

#include "muca_internal.cuh"

namespace muca {
namespace {

__global__ void muma_thresholds_kernel(const double *lnw, uint32_t *thr, int n_bins, double beta)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_bins * 10) return;
    const int b = t / 10, col = t % 10;
    const int s = col >= 5 ? 1 : -1, n = col % 5;
    const int bp = b - s;
    uint32_t A = 0u;
    if (bp >= 0 && bp < n_bins) {
        const double d = __dsub_rn(__dsub_rn(lnw[bp], lnw[b]), __dmul_rn(beta, (double)(8 - 4 * n)));
        if (d >= 0.0) {
            A = kAlways;
        } else {
            const double x = floor(ldexp(exp(d), 32));
            A = x >= 4294967295.0 ? kAlways : (uint32_t)x;
        }
    }
    thr[t] = A;
}

struct MumaArgs {
    uint32_t *lat;
    int32_t *E, *M;
    const uint32_t *thr;
    uint64_t *H;
    int32_t *E_rec, *M_rec;
    int L, p, p_pad, row_words, n_bins, n_sweeps, rec_stride;
    uint32_t sweep0, iteration, ctr3, key0;
};

// One thread per chain, one lattice word at a time: the word being decided and the words
// above and below it stay in registers, so a site reads nothing of the lattice.  With five
// bit loads per site the lanes of a warp, whose lattices lie L x row_words words apart, cost
// up to 32 cache lines per load.  Time of a chain's attempt at p = 4096 with bit loads, with
// bit loads of lattices interleaved word by word, and with words in registers: 64 x 64 557,
// 348 and 205 ns; 32 x 32 508, 284 and 171; 8 x 8 297, 275 and 172.  Bound by the chain's
// serial step: the table load that depends on M, the test, and a quarter of a Philox block.
template <bool HIST, bool SMEM_HIST>
__global__ void __launch_bounds__(128) muma_sweep_kernel(MumaArgs a)
{
    extern __shared__ uint32_t s_hist[];
    if (HIST && SMEM_HIST) {
        for (int i = threadIdx.x; i < a.n_bins; i += blockDim.x) s_hist[i] = 0u;
        __syncthreads();
    }
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < a.p) {
        const int L = a.L, V = L * L, RW = a.row_words;
        uint32_t *lat = a.lat + (size_t)c * (size_t)(L * RW);
        int E = a.E[c], M = a.M[c];
        for (int sw = 0; sw < a.n_sweeps; ++sw) {
            const uint32_t sweep = a.sweep0 + (uint32_t)sw;
            uint4 blk = make_uint4(0u, 0u, 0u, 0u);
            int i = 0;  // site
            for (int y = 0; y < L; ++y) {
                uint32_t *const row = lat + y * RW;
                const uint32_t *const up = lat + (y == 0 ? L - 1 : y - 1) * RW;
                const uint32_t *const down = lat + (y == L - 1 ? 0 : y + 1) * RW;
                // left neighbour of the next site (of site 0 the row's last one, old); site 0, new
                uint32_t left = (row[RW - 1] >> ((L - 1) & 31)) & 1u, first = 0u;
                for (int w = 0; w < RW; ++w) {
                    const int n = min(32, L - 32 * w);
                    uint32_t R = row[w];
                    const uint32_t U = up[w], D = down[w], next = w + 1 < RW ? row[w + 1] & 1u : 0u;
                    for (int j = 0; j < n; ++j, ++i) {
                        if ((i & 3) == 0)
                            blk = philox4x32_10(make_uint4((uint32_t)i >> 2, sweep, a.iteration, a.ctr3), a.key0,
                                                (uint32_t)c);
                        const uint32_t u = (i & 3) == 0 ? blk.x : (i & 3) == 1 ? blk.y : (i & 3) == 2 ? blk.z : blk.w;
                        const uint32_t me = (R >> j) & 1u;
                        const uint32_t right = j + 1 < n ? (R >> (j + 1)) & 1u : w + 1 < RW ? next : w == 0 ? R & 1u : first;
                        const int unequal = (int)((right ^ me) + (left ^ me) + (((U >> j) & 1u) ^ me) + (((D >> j) & 1u) ^ me));
                        const int b = (M + V) >> 1;
                        const uint32_t A = a.thr[b * 10 + (me ? 5 : 0) + unequal];
                        if (A == kAlways || u < A) {
                            R ^= 1u << j;
                            E += 8 - 4 * unequal;
                            M -= me ? 2 : -2;
                        }
                        left = (R >> j) & 1u;
                        if (HIST) {
                            const int bn = (M + V) >> 1;
                            if (SMEM_HIST)
                                atomicAdd(&s_hist[bn], 1u);
                            else
                                atomicAdd(reinterpret_cast<unsigned long long *>(&a.H[bn]), 1ull);
                        }
                    }
                    row[w] = R;
                    if (w == 0) first = R & 1u;
                }
            }
            if (a.E_rec) a.E_rec[(size_t)sw * a.rec_stride + c] = E;
            if (a.M_rec) a.M_rec[(size_t)sw * a.rec_stride + c] = M;
        }
        a.E[c] = E;
        a.M[c] = M;
    }
    if (HIST && SMEM_HIST) {
        __syncthreads();
        for (int i = threadIdx.x; i < a.n_bins; i += blockDim.x) {
            const uint32_t v = s_hist[i];
            if (v) atomicAdd(reinterpret_cast<unsigned long long *>(&a.H[i]), (unsigned long long)v);
        }
    }
}

}  // namespace

int launch_muma_thresholds(muca_ctx *ctx)
{
    const int n = ctx->n_bins * 10;
    muma_thresholds_kernel<<<(n + 255) / 256, 256, 0, ctx->stream>>>(ctx->d_lnw, ctx->d_thr, ctx->n_bins,
                                                                    ctx->cfg.beta);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return MUCA_OK;
}

int launch_muma_sweeps(muca_ctx *ctx, uint32_t phase, int n_sweeps, uint32_t sweep0, uint32_t iteration, bool hist,
                       int32_t *E_rec, int32_t *M_rec)
{
    MumaArgs a;
    a.lat = ctx->d_lat;
    a.E = ctx->d_E;
    a.M = ctx->d_M;
    a.thr = ctx->d_thr;
    a.H = ctx->d_H;
    a.E_rec = E_rec;
    a.M_rec = M_rec;
    a.L = ctx->L;
    a.p = ctx->p;
    a.p_pad = ctx->p_pad;
    a.row_words = ctx->row_words;
    a.n_bins = ctx->n_bins;
    a.n_sweeps = n_sweeps;
    a.rec_stride = ctx->p;
    a.sweep0 = sweep0;
    a.iteration = iteration;
    a.ctr3 = ((uint32_t)(ctx->seed >> 32) << 2) | phase;
    a.key0 = (uint32_t)ctx->seed;
    const int blocks = (ctx->p + 127) / 128;
    const size_t smem = (size_t)ctx->n_bins * sizeof(uint32_t);
    // block histograms are uint32: 128 chains x n_sweeps x V entries per launch
    const bool smem_hist = smem <= 48 * 1024 && 128.0 * n_sweeps * ctx->V < 4.0e9;
    if (!hist)
        muma_sweep_kernel<false, false><<<blocks, 128, 0, ctx->stream>>>(a);
    else if (smem_hist)
        muma_sweep_kernel<true, true><<<blocks, 128, smem, ctx->stream>>>(a);
    else
        muma_sweep_kernel<true, false><<<blocks, 128, 0, ctx->stream>>>(a);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    return MUCA_OK;
}

}  // namespace muca
