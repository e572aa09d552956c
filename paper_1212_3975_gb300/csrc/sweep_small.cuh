// Ising sweep body with one lane per chain, site by site: small lattices (L <= 16), and with
// many chains every lattice of one word per row (L <= 32).
//
// A pass of sweep_body.cuh takes a chain of some 600 cycles however few its sites, so on
// rows of up to 16 sites deciding one site after the other is faster (three iterations of
// 200 sweeps of 8 x 8 at p = 8, updates included: 2.05 ms with the earlier site-by-site
// kernel, 2.60 with passes of a row, 1.43 with this body).  The dependent step is kept
// short as follows: the table row of the next attempt is one of two candidates (this
// attempt rejected or accepted), and both candidates' thresholds are loaded before this
// attempt is decided, so a decision waits for one load and one select.  What a row needs at
// its start (draws, the neighbours of its first sites) is made during the row before: 61
// cycles per site of 8 x 8 instead of 76, of which some 28 are instructions to issue.
//
// Longer rows (16 < L <= 32) take 61 to 77 cycles per site; 32 chains per warp make up for it
// where a launch fills the GPU several times (lane_per_chain has the rule): 32 x 32,
// p = 16384, 64 sweeps 2.66 ms against 3.79 of rows at once, 20 x 20 2.41 against 5.19.
//
// A block has G groups of 32 chains: warps 0..G-1 decide, up to four more draw the random
// numbers into a ring per group (16 sites per hand-off).  Every lane has a histogram of its
// own, count of bin b at word 32 b + lane: the chains of a warp share a few bins, and
// atomics on one address wait on each other, and the table loads on them.  (L > 16: one
// histogram per block, with a count per lane or per two lanes.)
#pragma once
#include "sweep_body.cuh"

namespace muca {
namespace sweep {

constexpr int kSmallL = 16;   // always in this body up to here
constexpr int kLaneL = 32;    // with many chains up to here (one word per row)

// Draws of a chain, hand-offs of 16 sites.  Rows of up to 16 sites: three hand-offs, then
// the first again so that no row wraps.  Longer rows: four (the row being loaded spans up to
// three while the next is drawn), addressed modulo 64.  4 mod 32 words from chain to chain
// (vector loads of a warp hit every bank).
struct SmallRing {
    static constexpr int kPhase = 16, kSites = 3 * kPhase, kWrap = 4 * kPhase, kStride = kWrap + 4;
    static constexpr size_t kBytes = 32 * kStride * 4;
};

// Counts per bin of a block's histogram, L > kSmallL: one per lane, or per two lanes where
// one per lane would leave no room for twelve groups.  (28 x 28, p = 9728, 83 sweeps: eight
// counts per bin 3059 us, 16 2237, 32 2203; p = 58368 16 6520, 32 7929.)
__host__ __device__ constexpr int lane_counts(int L) { return L <= 22 ? 32 : 16; }

// shared memory of a launch: table, histograms (one per lane and group up to kSmallL; beyond,
// lane_counts counts per bin for the block, and a word per lane for padding chains),
// lattices, rings
__host__ __device__ constexpr size_t small_smem(int L, int n_bins, int lat_words, int groups, bool hist)
{
    const size_t h = !hist ? 0 : L <= kSmallL ? (size_t)n_bins * 128 * groups : (size_t)n_bins * 4 * lane_counts(L) + 128;
    return (size_t)n_bins * 32 + h + ((size_t)lat_words * 128 + SmallRing::kBytes) * groups;
}

// Table offsets 4 n and row changes 64 - 32 n of four sites, one per byte, for the
// previous attempt rejected (0) / accepted (1); n = unequal neighbours.  A byte product
// with 1 in the site's byte adds either to a row address.
struct Quad {
    uint32_t K0, K1, D0, D1;
};
__device__ __forceinline__ Quad quad_of(uint32_t lo, uint32_t hi, uint32_t q, int g)
{
    // (bits 0..3 to bit 2 or 3 of the four bytes)
    const uint32_t pre = ((((lo >> (4 * g)) & 0xFu) * 0x00810204u) & 0x04040404u) +
                         ((((hi >> (4 * g)) & 0xFu) * 0x01020408u) & 0x08080808u),
                   l = (((q >> (4 * g)) & 0xFu) * 0x00810204u) & 0x04040404u;
    Quad r;
    r.K0 = pre + l;
    r.K1 = pre + 0x04040404u - l;
    r.D0 = (0xC0C0C0C0u - 8u * r.K0) ^ 0x80808080u;  // (per byte 192 - 32 n >= 64: no borrow)
    r.D1 = (0xC0C0C0C0u - 8u * r.K1) ^ 0x80808080u;
    return r;
}

// L as a template parameter: the sites of a row are one unrolled block without branches.
template <int L, bool HIST>
__device__ __forceinline__ void small_body(const SweepArgs &a, const int cblk, const int G, uint32_t *smem)
{
    using Rg = SmallRing;
    static_assert(L >= 4 && L <= kLaneL && L % 2 == 0, "small lattices");
    constexpr int V = L * L, lat_words = L;
    constexpr bool LONG = L > kSmallL;
    __syncthreads();  // (persistent kernel: smem may still be read by the previous unit)
    const int tid = threadIdx.x, nt = block_threads(G), lane = tid & 31, warp = tid >> 5;
    const int n_bins = a.n_bins, lw = 32 * G, c0 = cblk * lw;
    uint32_t *const s_tab = smem;
    constexpr int C = lane_counts(L);                     // (LONG)
    uint32_t *const s_hist = s_tab + 8 * n_bins;          // [G][n_bins][32], LONG: [n_bins][C], [32]
    const int n_hist = !HIST ? 0 : LONG ? C * n_bins + 32 : 32 * n_bins * G;
    uint32_t *const s_lat = s_hist + n_hist;              // [lat_words][lw]
    uint32_t *const s_ring = s_lat + lat_words * lw;
    // (many loads in flight per thread: a block may have two warps only.  One 16 x 16 sweep of
    // 8 chains took 45 us with a load at a time here and a warp per bin at the end, 24 now; of
    // 8 x 8 18 and 12)
#pragma unroll 16
    for (int i = tid; i < 8 * n_bins; i += nt) s_tab[i] = (i & 7) < 5 ? a.ktab[5 * (i >> 3) + (i & 7)] : 0u;
    for (int i = tid; i < n_hist / 4; i += nt) reinterpret_cast<uint4 *>(s_hist)[i] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 8
    for (int i = tid; i < lat_words * lw; i += nt) {
        const int k = i % lat_words, c = i / lat_words;
        s_lat[k * lw + c] = c0 + c < a.p ? a.lat[(size_t)c0 * lat_words + i] : 0u;
    }
    __syncthreads();

    const int phases = (int)(((long long)a.n_sweeps * V + Rg::kPhase - 1) / Rg::kPhase);
    auto ring_of = [&](int grp) { return s_ring + grp * (int)(Rg::kBytes / 4) + lane * Rg::kStride; };

    if (warp >= G) {
        // ---------------- draws: a chain per lane, four sites per Philox block ------------------
        const uint32_t quads = (uint32_t)V >> 2, key0 = a.key0, iter = a.iteration, ctr3 = a.ctr3;
        uint32_t qd0 = 0u, ctr0 = a.sweep0;
        int slot = 0;
        for (int t = 0; t < phases; ++t) {
            uint32_t qd = qd0, ctr1 = ctr0;
            for (int grp = warp - G; grp < G; grp += draw_warps(G)) {
                const uint32_t key1 = (uint32_t)(c0 + 32 * grp + lane);
                // padding chains draw 2^32-1, which never accepts; the others at most
                // 2^32-2, so that u < A decides
                const bool active = key1 < (uint32_t)a.p;
                uint32_t *const ring = ring_of(grp) + slot * Rg::kPhase;
                qd = qd0;
                ctr1 = ctr0;
#pragma unroll
                for (int pass = 0; pass < 4; ++pass) {
                    uint4 b = philox4x32_10(make_uint4(qd, ctr1, iter, ctr3), key0, key1);
                    b.x = active ? min(b.x, 0xFFFFFFFEu) : 0xFFFFFFFFu;
                    b.y = active ? min(b.y, 0xFFFFFFFEu) : 0xFFFFFFFFu;
                    b.z = active ? min(b.z, 0xFFFFFFFEu) : 0xFFFFFFFFu;
                    b.w = active ? min(b.w, 0xFFFFFFFEu) : 0xFFFFFFFFu;
                    *reinterpret_cast<uint4 *>(ring + 4 * pass) = b;
                    if (!LONG && slot == 0) *reinterpret_cast<uint4 *>(ring + 4 * pass + Rg::kSites) = b;
                    if (++qd == quads) {
                        qd = 0u;
                        ++ctr1;
                    }
                }
                bar_sync(1 + grp, 64);
            }
            qd0 = qd;
            ctr0 = ctr1;
            slot = slot == (LONG ? 3 : 2) ? 0 : slot + 1;
        }
    } else {
        // ---------------- the chains ------------------------------------------------------------
        const int grp = warp, c = c0 + 32 * grp + lane;
        const bool active = c < a.p;
        const uint32_t lat_s = (uint32_t)__cvta_generic_to_shared(s_lat + 32 * grp + lane), ls = 4u * (uint32_t)lw;
        auto row_of = [&](int y) { return lds32(lat_s + (uint32_t)y * ls); };
        const uint32_t tab0 = (uint32_t)__cvta_generic_to_shared(s_tab);
        const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring_of(grp));
        const bool record = !HIST && (a.E_rec || a.M_rec || a.samples);
        // (count of the row at P: word 32 (P - tab0) / 32 + lane, LONG: C (P - tab0) / 32 + lane % C;
        // padding chains stay in one bin, and count it in the words behind)
        constexpr uint32_t HS = LONG ? (uint32_t)C / 8u : 4u;
        uint32_t hist0 = (uint32_t)__cvta_generic_to_shared(s_hist + (LONG ? lane % C : 32 * n_bins * grp + lane)) - HS * tab0;
        if (LONG && !active) hist0 = (uint32_t)__cvta_generic_to_shared(s_hist + C * n_bins + lane) - HS * (tab0 + 32u * (V >> 1));

        // P0 / P1: table row before the site if the previous attempt was rejected / accepted
        // (ap: which); Q0 / Q1: the row after it if the site accepts, A0 / A1: the thresholds
        uint32_t P0 = tab0 + 32u * (uint32_t)(active ? (a.E[c] + 2 * V) >> 2 : V >> 1), P1 = P0;
        bool ap = false;
        uint32_t R = row_of(0), U = row_of(L - 1), D = row_of(1);
        // unequal neighbours of a row's first site (its left one is site L - 1, old)
        auto first_site = [&](uint32_t r, uint32_t u, uint32_t d) {
            const uint32_t s = 0u - (r & 1u);  // (all bits: the spin)
            return ((s ^ u) & 1u) + ((s ^ d) & 1u) + ((s ^ (r >> 1)) & 1u) + ((s ^ (r >> (L - 1))) & 1u);
        };
        const uint32_t n = first_site(R, U, D);
        uint32_t Q0 = P0 + 64u - 32u * n, Q1 = Q0;
        uint32_t A0 = lds32(P0 + 4u * n), A1 = A0;
        const int rows = a.n_sweeps * L;
        int y = 0, sw = 0, pos = 0, lin = L, next_sync = Rg::kPhase;
        int ups = 0;
        // draws of the row; each block of four (two) makes room for the next row's
        uint32_t u[L];
        constexpr int W = L % 4 == 0 ? 4 : 2;
        auto load_draws = [&](int j) {
            const uint32_t us = ring_s + 4u * (uint32_t)(LONG ? (pos + j) & (Rg::kWrap - 1) : pos + j);
            if constexpr (W == 4)
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(u[j]), "=r"(u[j + 1]), "=r"(u[j + 2]), "=r"(u[j + 3])
                             : "r"(us));
            else
                asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(u[j]), "=r"(u[j + 1]) : "r"(us));
        };
        auto next_draws = [&] {
            pos = LONG ? (pos + L) & (Rg::kWrap - 1) : pos + L >= Rg::kSites ? pos + L - Rg::kSites : pos + L;
            lin += L;
        };
        bar_sync(1 + grp, 64);
        if (LONG) {  // (two hand-offs: at least 324 sites are drawn)
            bar_sync(1 + grp, 64);
            next_sync += Rg::kPhase;
        }
#pragma unroll
        for (int j = 0; j < L; j += W) load_draws(j);
        next_draws();
        Quad qd;  // of the four sites around the next one
        {
            const uint32_t ua = R ^ U, ub = R ^ D, tr = R ^ (R >> 1);
            qd = quad_of(ua ^ ub ^ tr, (ua & ub) | (tr & (ua ^ ub)), R ^ (R << 1), 0);
        }
        for (int it = 0; it < rows; ++it) {
            // the next row's draws are handed off (past the last row: old ones, not used)
#pragma unroll
            for (int k = 0; k < (LONG ? 2 : 1); ++k)
                if (lin > next_sync) {
                    if (next_sync < phases * Rg::kPhase) bar_sync(1 + grp, 64);
                    next_sync += Rg::kPhase;
                }
            const int y1 = y + 1 == L ? 0 : y + 1;
            const uint32_t R1 = row_of(y1), D1w = row_of(y1 + 1 == L ? 0 : y1 + 1);
            const uint32_t ua = R ^ U, ub = R ^ D, tr = R ^ (R >> 1), q = R ^ (R << 1);
            const uint32_t lo = ua ^ ub ^ tr, hi = (ua & ub) | (tr & (ua ^ ub));
            uint32_t Rw = R, last = 0u;  // last: unequal neighbours of the last site but its left one
            uint32_t n1 = 0u;                // unequal neighbours of the next row's first site
            Quad qn;                         // the next row's first quad
#pragma unroll
            for (int j = 0; j < L; ++j) {
                // (what the next row needs of this one's first sites, as soon as these are
                // decided: the row's end does not wait for it)
                if (j == 1) n1 = first_site(R1, Rw, D1w);
                if (L >= 6 && j == L - 2) {
                    const uint32_t va = R1 ^ Rw, vb = R1 ^ D1w, tr1 = R1 ^ (R1 >> 1);
                    qn = quad_of(va ^ vb ^ tr1, (va & vb) | (tr1 & (va ^ vb)), R1 ^ (R1 << 1), 0);
                }
                // the next site's table offset and row change, for this attempt rejected / accepted
                const uint32_t Pc = ap ? P1 : P0, Pa = ap ? Q1 : Q0;
                uint32_t B0, B1;
                if (j + 1 == L) {
                    B0 = lds32(Pc + 4u * n1);
                    B1 = lds32(Pa + 4u * n1);
                    Q0 = Pc + 64u - 32u * n1;
                    Q1 = Pa + 64u - 32u * n1;
                } else if (j + 2 == L) {
                    const uint32_t l = (q >> (L - 1)) & 1u, k0 = last + l, k1 = last + 1u - l;
                    B0 = lds32(Pc + 4u * k0);
                    B1 = lds32(Pa + 4u * k1);
                    Q0 = Pc + 64u - 32u * k0;
                    Q1 = Pa + 64u - 32u * k1;
                } else {
                    if ((j & 3) == 3) qd = quad_of(lo, hi, q, (j + 1) >> 2);
                    const int k = 1 << (8 * ((j + 1) & 3));
                    B0 = lds32((uint32_t)__dp4a((int)qd.K0, k, (int)Pc));
                    B1 = lds32((uint32_t)__dp4a((int)qd.K1, k, (int)Pa));
                    Q0 = (uint32_t)__dp4a((int)qd.D0, k, (int)Pc);
                    Q1 = (uint32_t)__dp4a((int)qd.D1, k, (int)Pa);
                }
                const bool acc = u[j] < (ap ? A1 : A0);
                if (HIST) red_shared(hist0 + HS * (acc ? Pa : Pc), 1u);
                Rw ^= acc ? 1u << j : 0u;
                if (j == 0)  // the row's last site sees the updated site 0 to its right
                    last = ((ua >> (L - 1)) & 1u) + ((ub >> (L - 1)) & 1u) + (((R >> (L - 1)) ^ Rw) & 1u);
                P0 = Pc;
                P1 = Pa;
                A0 = B0;
                A1 = B1;
                ap = acc;
                if (j % W == W - 1) load_draws(j - (W - 1));
            }
            next_draws();
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(lat_s + (uint32_t)y * ls), "r"(Rw) : "memory");
            ups += __popc(Rw);
            if (y1 == 0) {
                if (record && active) {
                    const int b = (int)(((ap ? P1 : P0) - tab0) >> 5), M = 2 * ups - V;
                    if (a.E_rec) a.E_rec[(size_t)sw * a.rec_stride + c] = 4 * b - 2 * V;
                    if (a.M_rec) a.M_rec[(size_t)sw * a.rec_stride + c] = M;
                    if (a.samples) {
                        const unsigned long long am = (unsigned long long)(M < 0 ? -M : M);
                        unsigned long long *sp = reinterpret_cast<unsigned long long *>(a.samples);
                        atomicAdd(&sp[b], 1ull);
                        atomicAdd(&sp[n_bins + b], am);
                        atomicAdd(&sp[2 * n_bins + b], am * am);
                    }
                }
                ++sw;
                if (it + 1 < rows) ups = 0;
            }
            // (R1 and D1w were read before this row was stored: at L >= 4 they are other rows)
            if (L < 6) {
                const uint32_t va = R1 ^ Rw, vb = R1 ^ D1w, tr1 = R1 ^ (R1 >> 1);
                qn = quad_of(va ^ vb ^ tr1, (va & vb) | (tr1 & (va ^ vb)), R1 ^ (R1 << 1), 0);
            }
            qd = qn;
            U = Rw;
            R = R1;
            D = D1w;
            y = y1;
        }
        if (active) {
            a.E[c] = 4 * (int)(((ap ? P1 : P0) - tab0) >> 5) - 2 * V;
            a.M[c] = 2 * ups - V;
        }
    }
    __syncthreads();
    for (int i = tid; i < lat_words * lw; i += nt) {
        const int k = i % lat_words, c = i / lat_words;
        if (c0 + c < a.p) a.lat[(size_t)c0 * lat_words + i] = s_lat[k * lw + c];
    }
    if (HIST && LONG) {
        for (int b = tid; b < n_bins; b += nt) {
            uint32_t x = 0u;
#pragma unroll
            for (int i = 0; i < C; ++i) x += s_hist[C * b + (i + b) % C];
            if (x) atomicAdd(reinterpret_cast<unsigned long long *>(a.H + b), (unsigned long long)x);
        }
    } else if (HIST) {
        // a thread per bin: counts of the block's chains (padding chains left out); all of a
        // launch's are below 2^31 (max_launch_sweeps)
        for (int b = tid; b < n_bins; b += nt) {
            uint32_t x = 0u;
            for (int g = 0; g < G; ++g) {
                const int n = a.p - c0 - 32 * g;  // chains of the group, or more
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int k = (i + b) & 31;
                    const uint32_t v = s_hist[32 * (n_bins * g + b) + k];
                    x += k < n ? v : 0u;
                }
            }
            if (x) atomicAdd(reinterpret_cast<unsigned long long *>(a.H + b), (unsigned long long)x);
        }
    }
}

}  // namespace sweep
}  // namespace muca
