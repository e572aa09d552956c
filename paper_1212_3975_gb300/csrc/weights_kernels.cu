// Weight side of the parallel multicanonical method (arXiv:1212.3975, Secs. 2-3), on
// the device: the master-process step of the paper (histogram in, new weights out)
// runs as one FP64 kernel whose result every sweep block reads from global memory,
// so no host round trip and no broadcast is needed.
//
// FP64 operations use explicit round-to-nearest intrinsics (and this file is built
// with -fmad=false) so that every sum and product is rounded in the order the
// recursion is written; only exp/log come from the CUDA math library.
#include <algorithm>

#include "muca_internal.cuh"

namespace muca {
namespace {

__device__ __forceinline__ int bin_delta(int model, int col)
{
    if (model == MUCA_ISING) return col < 2 ? col - 2 : col - 1;  // -2 -1 1 2
    return col < 4 ? col - 4 : col - 3;                            // -4..-1 1..4
}

// Acceptance thresholds (Eq. 1 as an integer test): d = lnW[b'] - lnW[b];
// A = 2^32-1 if d >= 0, else min(floor(2^32 exp(d)), 2^32-1); 0 if b' is out of range
// or inaccessible (never entered).
__global__ void thresholds_kernel(const double *lnw, const uint8_t *acc, uint32_t *thr, int model, int n_bins,
                                  int n_de)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_bins * n_de) return;
    const int b = t / n_de, col = t % n_de;
    const int bp = b + bin_delta(model, col);
    uint32_t A = 0u;
    if (acc[b] && bp >= 0 && bp < n_bins && acc[bp]) {
        const double d = __dsub_rn(lnw[bp], lnw[b]);
        if (d >= 0.0) {
            A = kAlways;
        } else {
            const double x = floor(ldexp(exp(d), 32));
            A = x >= 4294967295.0 ? kAlways : (uint32_t)x;
        }
    }
    thr[t] = A;
}

// Kernel layout of the thresholds for the sweep bodies: one row per
// bin, one column per local configuration so that the column offset follows from the
// neighbours without a branch.  Ising: column = number of unequal neighbours n
// (dE = 8 - 4n, so n = 2 is dE = 0 and always accepts); Potts: column = dE + 4.
__global__ void ktab_kernel(const uint32_t *thr, uint32_t *ktab, int model, int n_bins)
{
    const int width = ktab_width(model);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_bins * width) return;
    const int b = t / width, k = t % width;
    uint32_t v;
    if (model == MUCA_ISING) {
        // API columns by ascending dE: -8, -4, 4, 8 (n = 4, 3, 1, 0)
        v = k == 2 ? kAlways : thr[b * 4 + (k >= 3 ? 4 - k : 3 - k)];
    } else {
        const int dE = k - 4;
        v = dE == 0 ? kAlways : thr[b * 8 + (dE < 0 ? dE + 4 : dE + 3)];
    }
    ktab[t] = v;
    ktab[n_bins * width + t] = v >> 1;  // (as the sweep bodies compare them)
}

// The update runs as two kernels.  The recursion's differences (two logarithms and two
// divisions in FP64 per bin, at two FP64 operations per clock and SM: 0.15 ms for 4097
// bins on one SM) take a grid of blocks; what follows is one block per lattice
// (kUpdateThreads):
//   1. convergence statistics of H over accessible bins (Sec. 3);
//   2. prefix sums of the differences over accessible bins in ascending order, rounded
//      as the sequential sum (prefix_piece);
//   3. boundary correction beyond [lo, hi] with the slope of the innermost
//      `width` bins (Sec. 3);
//   4. ln W -= max over accessible bins; inaccessible bins = 0.
constexpr int kPiece = 4096;         // bins of the prefix staged at a time
constexpr int kPrefixThreads = 256;  // threads of the prefix, four bins each at a time

__device__ __forceinline__ void prefix_barrier()
{
    asm volatile("bar.sync 1, %0;" ::"n"(kPrefixThreads) : "memory");
}

// Sequential FP64 sum cur += x[i] of n values in shared memory, in place, by the block's
// first kPrefixThreads threads, four values each at a time; returns the last sum.  The
// result is that of adding one value after the other, bit for bit: while the sum stays in
// one binade it is a multiple k of one unit u in the last place, and adding x rounds to
// k + (x / u rounded to the nearest integer), so a run of additions is a prefix sum of
// integers.  Where that does not hold (a sum that leaves the binade or changes sign, an
// x / u halfway between integers, an x above the binade, a sum of zero) the one addition is
// done in FP64.  A chain of FP64 additions takes 117 cycles per value on this GPU (two FP64
// operations per clock and SM): 0.23 ms for the 4097 bins of a 64 x 64 Ising lattice.  One
// warp took 50 rounds of 128 values at 1750 cycles each for 64 x 64
// (18 of them for sums that leave their binade); with eight warps and
// rounds of 1024 values the whole update kernel takes 40 us instead of 68 (90 x 90: 64
// instead of 105).
__device__ __forceinline__ double prefix_piece(double *x, int n, double cur, int tid)
{
    constexpr unsigned long long one = 1ull << 52, frac = one - 1ull;
    constexpr int NW = kPrefixThreads / 32, span = 4 * kPrefixThreads;
    __shared__ long long s_tot[NW];
    __shared__ int s_stop[NW];
    const int lane = tid & 31, warp = tid >> 5;
    int late = -1;  // a sum still to be stored (thread 0)
    double late_sum = 0.0;
    for (int i = 0; i < n;) {
        const unsigned long long cb = (unsigned long long)__double_as_longlong(cur);
        const int ce = (int)(cb >> 52) & 0x7FF;
        const long long mag = (long long)((cb & frac) | one), k = cb >> 63 ? -mag : mag;
        const bool zero = cb == 0ull, regular = ce > 0 && ce < 0x7FF;
        long long v[4];   // the thread's inclusive sums of rounded integers
        int good = 4;     // values of the thread before the first that needs FP64
        long long sum = 0;
        const int j0 = i + 4 * tid;
#pragma unroll
        for (int t = 3; t >= 0; --t) v[t] = __double_as_longlong(j0 + t < n ? x[j0 + t] : 0.0);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const unsigned long long b = (unsigned long long)v[t];
            const int e = (int)(b >> 52) & 0x7FF, sh = ce - max(e, 1);
            const unsigned long long mt = ((b & frac) | (e ? one : 0ull)) << 1;
            // x / u with one more bit, and whether that is all of it
            const int s = min(max(sh, 0), 63);
            const unsigned long long r2 = mt >> s;
            const bool tie = (r2 & 1ull) && (r2 << s) == mt;
            const long long r = (long long)((r2 + 1ull) >> 1);
            const bool ok = j0 + t < n && (zero ? (b << 1) == 0ull : regular && e != 0x7FF && sh >= 0 && !tie);
            if (!ok) good = min(good, t);
            if (!zero) sum += b >> 63 ? -r : r;
            v[t] = sum;
        }
        long long incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(~0u, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_tot[warp] = incl;
        prefix_barrier();
        if (late >= 0 && tid == 0) x[late] = late_sum;
        long long below = k + incl - sum;
#pragma unroll
        for (int w = 0; w < NW - 1; ++w)
            if (w < warp) below += s_tot[w];
#pragma unroll
        for (int t = 3; t >= 0; --t) {
            v[t] += below;
            const unsigned long long q = (unsigned long long)(v[t] < 0 ? -v[t] : v[t]);
            if (!zero && !(q > one && q < one << 1 && (v[t] < 0) == (k < 0))) good = min(good, t);
        }
        const int stop = __reduce_min_sync(~0u, good < 4 ? 4 * tid + good : span);
        if (lane == 0) s_stop[warp] = stop;
        prefix_barrier();
        int done = s_stop[0];  // (values past n stop it)
#pragma unroll
        for (int w = 1; w < NW; ++w) done = min(done, s_stop[w]);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (4 * tid + t < done) {
                const unsigned long long q = (unsigned long long)(v[t] < 0 ? -v[t] : v[t]);
                const unsigned long long bits = zero ? 0ull : (q & frac) | (unsigned long long)ce << 52 | (cb & (1ull << 63));
                x[j0 + t] = __longlong_as_double((long long)bits);
            }
        }
        prefix_barrier();
        if (done > 0) cur = x[i + done - 1];
        i += done;
        late = -1;
        if (done < span && i < n) {
            // (stored when every thread has read it)
            cur = __dadd_rn(cur, x[i]);
            late = i;
            late_sum = cur;
            ++i;
        }
    }
    prefix_barrier();
    if (late >= 0 && tid == 0) x[late] = late_sum;
    return cur;
}

// The same by one thread, one addition after the other: a round of prefix_piece takes some
// 1900 cycles, and a small lattice's sums leave their binade every few bins (8 x 8: 6 to 19
// rounds for 65 bins).
constexpr int kSequentialBins = 256;
__device__ __forceinline__ void prefix_sequential(double *x, int n)
{
    double cur = 0.0;
    for (int i = 0; i < n; i += 8) {
        double v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) v[t] = i + t < n ? x[i + t] : 0.0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            cur = __dadd_rn(cur, v[t]);
            if (i + t < n) x[i + t] = cur;
        }
    }
}

// Threads per block where every thread evaluates FP64 logarithms, divisions or an
// exponential: small, so that the bins spread over all SMs' FP64 pipes.
constexpr int kBinThreads = 64;

// Recursion (Sec. 2) of bin u: scratch[v] = difference to bin v from the accessible bin u
// before it (accumulated form), or ln W after the simple recursion.
__device__ __forceinline__ void update_bin(const double *lnw, double *P, double *scratch, const uint64_t *H,
                                           const uint8_t *acc, int n_bins, int accumulated, int u)
{
    if (!acc[u]) return;
    if (accumulated) {
        int v = u + 1;
        while (v < n_bins && !acc[v]) ++v;
        if (v >= n_bins) return;
        double d = __dsub_rn(lnw[v], lnw[u]);
        const uint64_t hu_i = H[u], hv_i = H[v];
        if (hu_i > 0 && hv_i > 0) {
            const double hu = (double)hu_i, hv = (double)hv_i;
            const double g0 = __ddiv_rn(__dmul_rn(hu, hv), __dadd_rn(hu, hv));
            const double pu = __dadd_rn(P[u], g0);
            P[u] = pu;
            const double g = __ddiv_rn(g0, pu);
            d = __dsub_rn(d, __dmul_rn(g, __dsub_rn(log(hv), log(hu))));
        }
        scratch[v] = d;
    } else {
        double v = lnw[u];
        if (H[u] > 0) v = __dsub_rn(v, log((double)H[u]));
        scratch[u] = v;
    }
}

// Order of doubles as integers (NaN lowest): the FP64 maximum of a block is 32 comparisons
// in a row at some 100 cycles each.
__device__ __forceinline__ long long order_key(double x)
{
    const long long b = __double_as_longlong(x);
    return x != x ? (long long)(1ull << 63) : b < 0 ? b ^ 0x7FFFFFFFFFFFFFFFll : b;
}
__device__ __forceinline__ double order_value(long long k)
{
    return __longlong_as_double(k < 0 ? k ^ 0x7FFFFFFFFFFFFFFFll : k);
}

// blockDim.x = kUpdateThreads
constexpr int kUpdateThreads = 1024;
__device__ __forceinline__ void update_body(double *lnw, const double *scratch, const uint64_t *H, const uint8_t *acc,
                                            int n_bins, int accumulated, int width_cfg, muca_iter_stats *stats)
{
    constexpr int NW = kUpdateThreads / 32;
    static_assert(NW == 32, "a warp reduces the warps' values");
    __shared__ unsigned long long s_total[NW], s_min[NW], s_max[NW];
    __shared__ int s_ns[NW], s_K[NW], s_lo[NW], s_hi[NW], s_first[NW];
    __shared__ long long s_top[NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // 1. statistics
    unsigned long long tot = 0, mn = ~0ull, mx = 0;
    int ns = 0, K = 0, lo = n_bins, hi = -1, first = n_bins;
    for (int b = tid; b < n_bins; b += kUpdateThreads) {
        if (!acc[b]) continue;
        const unsigned long long h = H[b];
        tot += h;
        mn = min(mn, h);
        mx = max(mx, h);
        K += 1;
        first = min(first, b);
        if (h) {
            ns += 1;
            lo = min(lo, b);
            hi = max(hi, b);
        }
    }
    auto reduce_counts = [&] {
        for (int o = 16; o > 0; o >>= 1) {
            tot += __shfl_xor_sync(~0u, tot, o);
            mn = min(mn, __shfl_xor_sync(~0u, mn, o));
            mx = max(mx, __shfl_xor_sync(~0u, mx, o));
        }
        ns = __reduce_add_sync(~0u, ns);
        K = __reduce_add_sync(~0u, K);
    };
    reduce_counts();
    lo = __reduce_min_sync(~0u, lo);
    hi = __reduce_max_sync(~0u, hi);
    first = __reduce_min_sync(~0u, first);
    if (lane == 0) {
        s_total[warp] = tot; s_min[warp] = mn; s_max[warp] = mx; s_ns[warp] = ns; s_K[warp] = K;
        s_lo[warp] = lo; s_hi[warp] = hi; s_first[warp] = first;
    }
    __syncthreads();
    lo = __reduce_min_sync(~0u, s_lo[lane]);
    hi = __reduce_max_sync(~0u, s_hi[lane]);
    first = __reduce_min_sync(~0u, s_first[lane]);
    const int slo = hi >= 0 ? lo : -1, shi = hi >= 0 ? hi : -1;
    if (warp == NW - 1) {
        // (beside the prefix: five FP64 divisions and comparisons in a row)
        tot = s_total[lane]; mn = s_min[lane]; mx = s_max[lane]; ns = s_ns[lane]; K = s_K[lane];
        reduce_counts();
        if (lane == 0) {
            const double mean = (double)tot / (double)(unsigned long long)K;
            muca_iter_stats st;
            st.covered = (ns == K);
            st.flat = st.covered && ((double)mn >= 0.5 * mean) && ((double)mx <= 2.0 * mean);
            st.lo = slo;
            st.hi = shi;
            st.n_sampled = (int64_t)ns;
            st.min_over_mean = mean > 0 ? (double)mn / mean : 0.0;
            st.max_over_mean = mean > 0 ? (double)mx / mean : 0.0;
            st.total = tot;
            *stats = st;
        }
    }

    // 2. prefix in ascending order
    if (accumulated) {
        __shared__ double s_d[kPiece];
        double cur = 0.0;  // (threads of the prefix)
        for (int b0 = 0; b0 < n_bins; b0 += kPiece) {
            const int n = min(kPiece, n_bins - b0);
            // (an inaccessible bin adds nothing; the first accessible one has no difference)
            for (int i = tid; i < n; i += kUpdateThreads)
                s_d[i] = acc[b0 + i] && b0 + i != first ? scratch[b0 + i] : 0.0;
            __syncthreads();
            if (n_bins <= kSequentialBins) {
                if (tid == 0) prefix_sequential(s_d, n);
            } else if (tid < kPrefixThreads) {
                cur = prefix_piece(s_d, n, cur, tid);
            }
            __syncthreads();
            for (int i = tid; i < n; i += kUpdateThreads)
                if (acc[b0 + i]) lnw[b0 + i] = s_d[i];
            __syncthreads();
        }
    } else {
        for (int b = tid; b < n_bins; b += kUpdateThreads)
            if (acc[b]) lnw[b] = scratch[b];
        __syncthreads();
    }

    // 3. boundary correction
    const bool bounds = slo >= 0 && shi > slo;
    double vlo = 0.0, vhi = 0.0;
    __shared__ double s_slope[2];
    if (bounds) {
        const int width = min(width_cfg, shi - slo);
        if (lane == 0 && warp < 2) {
            // (warp 0 the lower, warp 1 the upper end)
            int b = warp == 0 ? slo + width : shi - width;
            while (!acc[b]) b += warp == 0 ? 1 : -1;
            s_slope[warp] = warp == 0 ? __ddiv_rn(__dsub_rn(lnw[b], lnw[slo]), (double)(b - slo))
                                      : __ddiv_rn(__dsub_rn(lnw[shi], lnw[b]), (double)(shi - b));
        }
        vlo = lnw[slo];
        vhi = lnw[shi];
        __syncthreads();
    }
    const double sl_lo = s_slope[0], sl_hi = s_slope[1];

    // 4. normalisation: max over accessible bins is 0
    long long key = (long long)(1ull << 63);
    for (int b = tid; b < n_bins; b += kUpdateThreads) {
        if (!acc[b]) continue;
        double x;
        if (bounds && b < slo) x = lnw[b] = __dadd_rn(vlo, __dmul_rn(sl_lo, (double)(b - slo)));
        else if (bounds && b > shi) x = lnw[b] = __dadd_rn(vhi, __dmul_rn(sl_hi, (double)(b - shi)));
        else x = lnw[b];
        key = max(key, order_key(x));
    }
    for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(~0u, key, o));
    if (lane == 0) s_top[warp] = key;
    __syncthreads();
    key = s_top[lane];
    for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(~0u, key, o));
    const double top = order_value(key);
    // (each bin was last written by its own thread)
    for (int b = tid; b < n_bins; b += kUpdateThreads) lnw[b] = acc[b] ? __dsub_rn(lnw[b], top) : 0.0;
}

__global__ void update_bins_kernel(const double *lnw, double *P, double *scratch, const uint64_t *H, const uint8_t *acc,
                                   int n_bins, int accumulated)
{
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < n_bins) update_bin(lnw, P, scratch, H, acc, n_bins, accumulated, u);
}

__global__ void __launch_bounds__(kUpdateThreads) update_kernel(double *lnw, const double *scratch, const uint64_t *H,
                                                      const uint8_t *acc, int n_bins, int accumulated, int width_cfg,
                                                      muca_iter_stats *stats)
{
    update_body(lnw, scratch, H, acc, n_bins, accumulated, width_cfg, stats);
}

// bins of every lattice of a batch (blockIdx.y = lattice), then one block per lattice
__global__ void update_bins_batch_kernel(const BatchJob *jobs)
{
    const BatchJob &j = jobs[blockIdx.y];
    if (!*j.active) return;  // converged lattice: frozen
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < j.n_bins) update_bin(j.lnw, j.P, j.wscratch, j.H, j.acc, j.n_bins, j.accumulated, u);
}

__global__ void __launch_bounds__(kUpdateThreads) update_batch_kernel(const BatchJob *jobs)
{
    const BatchJob &j = jobs[blockIdx.x];
    if (!*j.active) return;
    update_body(j.lnw, j.wscratch, j.H, j.acc, j.n_bins, j.accumulated, j.width, j.stats);
}

// thresholds of every lattice of a batch: blockIdx.y = lattice
__global__ void thresholds_batch_kernel(const BatchJob *jobs)
{
    const BatchJob &j = jobs[blockIdx.y];
    if (!*j.active) return;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < j.n_bins * j.n_de; t += gridDim.x * blockDim.x) {
        const int b = t / j.n_de, col = t % j.n_de;
        const int bp = b + bin_delta(j.model, col);
        uint32_t A = 0u;
        if (j.acc[b] && bp >= 0 && bp < j.n_bins && j.acc[bp]) {
            const double d = __dsub_rn(j.lnw[bp], j.lnw[b]);
            if (d >= 0.0) {
                A = kAlways;
            } else {
                const double x = floor(ldexp(exp(d), 32));
                A = x >= 4294967295.0 ? kAlways : (uint32_t)x;
            }
        }
        j.thr[t] = A;
    }
}

}  // namespace

cudaError_t launch_batch_update(const BatchJob *d_jobs, int n_jobs, int max_bins, int max_thr, cudaStream_t st)
{
    update_bins_batch_kernel<<<dim3((max_bins + kBinThreads - 1) / kBinThreads, n_jobs), kBinThreads, 0, st>>>(d_jobs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    update_batch_kernel<<<n_jobs, kUpdateThreads, 0, st>>>(d_jobs);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    dim3 grid((max_thr + kBinThreads - 1) / kBinThreads, n_jobs);
    thresholds_batch_kernel<<<grid, kBinThreads, 0, st>>>(d_jobs);
    e = cudaGetLastError();
    if (e == cudaSuccess) note_launches(3);
    return e;
}

int launch_thresholds(muca_ctx *ctx)
{
    if (ctx->cfg.ensemble == MUCA_ENSEMBLE_MAGNETIZATION) return launch_muma_thresholds(ctx);
    const int n = ctx->n_bins * ctx->n_de;
    thresholds_kernel<<<(n + kBinThreads - 1) / kBinThreads, kBinThreads, 0, ctx->stream>>>(
        ctx->d_lnw, ctx->d_acc, ctx->d_thr, ctx->model, ctx->n_bins, ctx->n_de);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    ctx->ktab_dirty = 1;
    return MUCA_OK;
}

int launch_update(muca_ctx *ctx)
{
    const int width = ctx->cfg.correction_width > 0 ? ctx->cfg.correction_width : ctx->L;
    const int accumulated = ctx->cfg.recursion == MUCA_RECURSION_ACCUMULATED;
    update_bins_kernel<<<(ctx->n_bins + kBinThreads - 1) / kBinThreads, kBinThreads, 0, ctx->stream>>>(
        ctx->d_lnw, ctx->d_P, ctx->d_wscratch, ctx->d_H, ctx->d_acc, ctx->n_bins, accumulated);
    MUCA_CUDA_TRY(cudaGetLastError());
    update_kernel<<<1, kUpdateThreads, 0, ctx->stream>>>(ctx->d_lnw, ctx->d_wscratch, ctx->d_H, ctx->d_acc, ctx->n_bins,
                                                         accumulated, width, ctx->d_stats);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(2);
    return launch_thresholds(ctx);
}

int launch_ktab(muca_ctx *ctx)
{
    const int width = ktab_width(ctx->model);
    const int n = ctx->n_bins * width;
    ktab_kernel<<<(n + 255) / 256, 256, 0, ctx->stream>>>(ctx->d_thr, ctx->d_ktab, ctx->model, ctx->n_bins);
    MUCA_CUDA_TRY(cudaGetLastError());
    note_launches(1);
    ctx->ktab_dirty = 0;
    return MUCA_OK;
}

}  // namespace muca
