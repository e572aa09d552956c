// Sweep body of both models, all lattice sizes: up to 128 consecutive sites of a row are
// decided at once and then checked.
//
// Within one chain every attempt depends on the previous one twice: through the left
// neighbour's spin and through the global energy, which names the row of the threshold
// table.  Deciding site by site costs a chain a dependent table load per site (36 to 60
// cycles on this GPU).  Instead:
//
//   predict  the draw of every site is compared with the thresholds of the pass's FIRST
//            bin, for the left neighbour kept and changed.  That leaves one bit of
//            dependence from site to site, which a parallel prefix resolves.
//   verify   the predicted decisions give every site its neighbours and, by prefix sums
//            of the bin changes, its own bin; each draw is compared with the threshold of
//            exactly that bin and neighbourhood.  If every decision agrees, the
//            prediction is the chain's trajectory: site by site, each decision is the
//            exact test of Eq. 1 given the decisions before it.
//   repair   otherwise the verified thresholds replace the predicted ones and the pass is
//            resolved again.  Each repetition extends the agreeing prefix by at least one
//            site (the first disagreeing site had the right history, so its test was
//            exact), so this ends; thresholds of neighbouring bins differ by little, and
//            most passes need no repair.  (A launch that repeats more than 4 LPC + 2 times
//            per pass, which passes of 4 LPC sites cannot need, gives up and says so in
//            a.fault.)
//
// Every decision is the exact integer test, so trajectories, histograms and records are
// those of the site-by-site form, bit for bit.  Any predicted decisions give a real
// configuration, so predicted bins never leave the table.
//
// A lane holds four consecutive sites, one per byte; a chain takes LPC lanes (4 LPC sites
// per pass), a warp (a group) 32 / LPC chains.  A lane composes the one-bit maps of its
// sites for both values of the incoming bit; two ballots and a prefix over the ballots'
// bits carry the decisions from lane to lane, and bytes in shared memory the bin changes.
// A pass is a chain of dependent steps whatever its sites, so a row in one pass (ROW,
// L <= 4 LPC) is what shortens a sweep.  A block has G groups: warps 0..G-1 decide, up to
// four more draw the random numbers (Philox) into a ring per group, 16 LPC sites per
// hand-off (one named barrier per group).
//
// Tests are made on integers, not predicates: the table holds thresholds and the lanes
// hold draws shifted right by one, so that the sign of draw - threshold is the test, and
// signs are combined with logic instructions (5 cycles a step, a predicate takes 13).  A
// difference of zero leaves the test open (once in 2^31): the 32-bit table decides it.
#pragma once
#include <type_traits>

#include "muca_internal.cuh"

namespace muca {
namespace sweep {

constexpr int kMaxGroups = 12;  // groups per block at most
constexpr int kFlushBarrier = 15;
static_assert(kMaxGroups < kFlushBarrier, "named barrier ids");
// warps that draw: one per scheduler at most (a scheduler's 20 high products per Philox
// block take 84 cycles; a pass of a deciding warp some 500)
__host__ __device__ constexpr int draw_warps(int groups) { return groups < 4 ? groups : 4; }
__host__ __device__ constexpr int block_threads(int groups) { return 32 * (groups + draw_warps(groups)); }

// Threshold table (31-bit entries): in global memory, in shared memory, or in shared memory
// as the upper 16 bits of each threshold.
enum Table { kTabGlobal = 0, kTabShared = 1, kTabShared16 = 2 };
// Block histogram: in global memory, one 32-bit count per attempt, one per pair of
// consecutive attempts (C[b][d + D]: the first ends in bin b, the second in b + d; D the
// largest bin change), or 16-bit counts, two bins per word, flushed before any overflows.
enum Hist { kHistNone = -1, kHistGlobal = 0, kHistSingle = 1, kHistPairs = 2, kHist16 = 3 };

// Draws of a chain: three hand-offs, then the first pass of the first again so that no
// pass wraps; for Potts also a byte per site (proposal offsets, two words of slack).
template <int LPC>
struct Ring {
    static constexpr int kChains = 32 / LPC, kPhase = 16 * LPC, kSites = 3 * kPhase;
    static constexpr int kStride = kSites + 4 * LPC, kByteStride = kStride + 8;
};
// shared memory of a group: its ring, and a byte per lane for the sums over lanes
__host__ __device__ constexpr size_t ring_bytes(int model) { return 6656 + (model == MUCA_POTTS ? 1664 + 8 * 16 : 0) + 32; }

__device__ __forceinline__ void bar_sync(int id, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
// the same where `take` is true (uniform): no branch
__device__ __forceinline__ void bar_sync_if(bool take, int id, int n)
{
    asm volatile("{.reg .pred p; setp.ne.u32 p, %2, 0; @p bar.sync %0, %1;}" ::"r"(id), "r"(n), "r"((uint32_t)take)
                 : "memory");
}
__device__ __forceinline__ void red_shared(uint32_t saddr, uint32_t v)
{
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(saddr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds32(uint32_t saddr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(saddr));
    return v;
}

// one threshold at byte address `ad` of the table
template <int TAB>
__device__ __forceinline__ uint32_t table_load(const char *ktab, uint32_t ad)
{
    uint32_t v;
    if (TAB == kTabGlobal) {
        asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(ktab + ad));
    } else if (TAB == kTabShared) {
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(ad));
    } else {
        uint16_t h;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(ad));
        v = h;
    }
    return v;
}

// 0xFF in byte i where the i-th argument is negative
__device__ __forceinline__ uint32_t sign_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    uint32_t x, y;
    asm("prmt.b32 %0, %1, %2, 0x00FB;" : "=r"(x) : "r"(a), "r"(b));
    asm("prmt.b32 %0, %1, %2, 0xFB00;" : "=r"(y) : "r"(c), "r"(d));
    return __byte_perm(x, y, 0x7610);
}
// bits of t where m, of f elsewhere
__device__ __forceinline__ uint32_t select(uint32_t m, uint32_t t, uint32_t f) { return (m & t) | (~m & f); }

// bits 0..3 of x to bit 0 of the four bytes, and back
__device__ __forceinline__ uint32_t spread4(uint32_t x) { return ((x & 0xFu) * 0x00204081u) & 0x01010101u; }
__device__ __forceinline__ uint32_t pack4(uint32_t x) { return (x * 0x10204080u) >> 28; }
// 0x01 in every byte of x (bytes below 128) that is not zero
__device__ __forceinline__ uint32_t nz_bytes(uint32_t x) { return ((x + 0x7F7F7F7Fu) >> 7) & 0x01010101u; }

// proposal offset floor(7 w / 2^32) in 0..6, exactly: 7 w = 8 w - w
__device__ __forceinline__ uint32_t offset7(uint32_t x) { return (x >> 29) - ((x << 3) < x ? 1u : 0u); }

// State counts of a word of four Potts spins, one 4-bit field per state.
__device__ __forceinline__ uint32_t count_fields(uint32_t w)
{
    uint32_t x = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) x += 1u << ((w >> (8 * i) & 7u) * 4u);
    return x;
}
// Counters of a lane: 16-bit fields of states (0,4), (2,6), (1,5), (3,7).
struct StateCounts {
    uint32_t f[4] = {0u, 0u, 0u, 0u};
    uint32_t e = 0u, o = 0u;  // bytes: even and odd states since the last flush
    __device__ __forceinline__ void add(uint32_t word)
    {
        const uint32_t x = count_fields(word);
        e += x & 0x0F0F0F0Fu;
        o += (x >> 4) & 0x0F0F0F0Fu;
    }
    __device__ __forceinline__ void flush()  // at most 63 words after the last one
    {
        f[0] += e & 0x00FF00FFu;
        f[1] += (e >> 8) & 0x00FF00FFu;
        f[2] += o & 0x00FF00FFu;
        f[3] += (o >> 8) & 0x00FF00FFu;
        e = o = 0u;
    }
    template <int LPC>
    __device__ __forceinline__ void reduce(uint32_t padding)  // `padding` sites counted as state 0
    {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int x = 1; x < LPC; x <<= 1) f[k] += __shfl_xor_sync(~0u, f[k], x);
        f[0] -= padding;
    }
    __device__ __forceinline__ uint32_t max_count() const
    {
        uint32_t n = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) n = max(n, max(f[k] & 0xFFFFu, f[k] >> 16));
        return n;
    }
    // counts of states 0..3 / 4..7, 16 bits each
    __device__ __forceinline__ uint64_t low() const
    {
        return (uint64_t)(f[0] & 0xFFFFu) | (uint64_t)(f[2] & 0xFFFFu) << 16 | (uint64_t)(f[1] & 0xFFFFu) << 32 |
               (uint64_t)(f[3] & 0xFFFFu) << 48;
    }
    __device__ __forceinline__ uint64_t high() const
    {
        return (uint64_t)(f[0] >> 16) | (uint64_t)(f[2] >> 16) << 16 | (uint64_t)(f[1] >> 16) << 32 |
               (uint64_t)(f[3] >> 16) << 48;
    }
};

// ROW: a row is one pass (L <= 4 LPC): the last site's right neighbour, site 0, is decided
// in the same pass, and the next pass's upper neighbours are this pass's new spins.
// Otherwise LPC = 32 and a row is several passes of 128 sites.
// AL: L is a multiple of four (every lane's sites are whole, draws are aligned).
// HMODE: histogram mode, kHistNone for launches without one.  Both, as everything else
// that a branch would decide in every pass, are template parameters: with one deciding
// warp per scheduler a uniform branch costs a pass some 20 cycles (64 x 64, p = 1024: 566
// against 375 ns per pass with the modes as run-time flags).
// PEEL: the first attempt of a pass is code of its own, in whose gaps the next pass is
// prepared, and a repetition does without that.  Shorter passes while latency bounds them,
// more code than the instruction caches like where a scheduler has three deciding warps.
// TWO: a row is two passes (128 < L <= 256): every lane keeps the spins of both in
// registers (a pass's row below is the spins of the pass two on, its decisions the row
// above of the pass two on), so that a pass reads four sites per lane of the lattice where
// rows of any length read five quads (256 x 256, p = 8192, 4 sweeps: 7.6 ms against 8.8).
template <int MODEL, int LPC, bool ROW, bool AL, int TAB, int HMODE, bool PEEL, bool TWO>
__device__ __forceinline__ void sweep_body(const SweepArgs &a, const int cblk, const int G, const bool stage_lattice,
                                           uint32_t *smem)
{
    using Rg = Ring<LPC>;
    constexpr bool POTTS = MODEL == MUCA_POTTS;
    constexpr uint32_t NC = POTTS ? 9u : 5u;                  // table columns
    constexpr uint32_t COLB = TAB == kTabShared16 ? 2u : 4u;  // bytes per table entry
    constexpr uint32_t ROWB = NC * COLB;                      // bytes per bin
    constexpr uint32_t EB = POTTS ? 4u : 2u;                  // largest bin change
    constexpr uint32_t BB = 4u * EB;                          // bias of a lane's bin offsets
    constexpr uint32_t m = 0x01010101u;
    constexpr bool HIST = HMODE != kHistNone;
    static_assert(ROW || LPC == 32, "long rows take whole warps");
    static_assert(ROW || !PEEL, "rows of one pass");
    static_assert(!ROW || !TWO, "one pass or two");
    static_assert(AL || HMODE != kHistPairs, "pairs lie within a lane's four sites");
    __syncthreads();  // (persistent kernel: smem may still be read by the previous unit)
    const int tid = threadIdx.x, nt = block_threads(G), lane = tid & 31, warp = tid >> 5;
    const int n_bins = a.n_bins, n_tab = n_bins * (int)NC;
    const int tab_words = TAB == kTabShared ? n_tab : TAB == kTabShared16 ? (n_tab + 1) >> 1 : 0;
    const int n_hist = HMODE == kHistSingle ? n_bins : HMODE == kHistPairs ? n_tab : HMODE == kHist16 ? (n_bins + 1) >> 1 : 0;
    const int lw = Rg::kChains * G, lat_words = a.lat_words;  // chains of the block, words of a chain
    uint32_t *const s_tab = smem;
    uint32_t *const s_hist = s_tab + ((tab_words + 3) & ~3);
    // (the histogram is followed by a slot per lane for lanes that have nothing to count)
    uint32_t *const s_lat = s_hist + (n_hist ? ((n_hist + 3) & ~3) + 32 : 0);
    uint32_t *const s_ring = s_lat + (stage_lattice ? (lat_words * lw + 3) & ~3 : 0);
    const int c0 = cblk * lw, n_own = max(0, min(lw, a.p - c0));  // first chain, chains of the block

    if (TAB == kTabShared)
        for (int i = tid; i < n_tab; i += nt) s_tab[i] = a.ktab[i] >> 1;
    if (TAB == kTabShared16)
        for (int i = tid; i < n_tab; i += nt) reinterpret_cast<uint16_t *>(s_tab)[i] = (uint16_t)(a.ktab[i] >> 16);
    for (int i = tid; i < n_hist; i += nt) s_hist[i] = 0u;
    if (stage_lattice)
        for (int i = tid; i < lat_words * lw; i += nt)
            s_lat[i] = i < lat_words * n_own ? a.lat[(size_t)c0 * lat_words + i] : 0u;
    __syncthreads();

    const int ch = lane / LPC, cl = lane % LPC;  // chain of the group, lane of the chain
    const int L = a.L, V = L * L;
    const int VS = AL ? V : (V + 3) & ~3;  // draws of a sweep (whole lanes of the drawing warps)
    const int phases = (int)(((long long)a.n_sweeps * VS + Rg::kPhase - 1) / Rg::kPhase);
    // a group's ring: draws, and (Potts) proposal offsets, a byte per site
    auto ring_of = [&](int grp) { return s_ring + grp * (int)(ring_bytes(MODEL) / 4) + ch * Rg::kStride; };
    auto offs_of = [&](int grp) {
        return reinterpret_cast<uint8_t *>(s_ring + grp * (int)(ring_bytes(MODEL) / 4) + Rg::kChains * Rg::kStride) +
               ch * Rg::kByteStride;
    };

    if (warp >= G) {
        // ---------------- draws of four sites per lane and pass, in site order ------------------
        // (of groups warp - G, warp - G + draw_warps, ..., a hand-off of each in turn: the groups
        // of a drawing warp settle at different points of their hand-offs)
        const uint32_t quads = (uint32_t)VS >> 2, key0 = a.key0, iter = a.iteration, ctr3 = a.ctr3;
        uint32_t qd0 = (uint32_t)cl, ctr0 = a.sweep0;
        while (qd0 >= quads) {
            qd0 -= quads;
            ++ctr0;
        }
        int slot = 0;
        for (int t = 0; t < phases; ++t) {
            uint32_t qd = qd0, ctr1 = ctr0;
            for (int grp = warp - G; grp < G; grp += draw_warps(G)) {
                const uint32_t key1 = (uint32_t)(c0 + grp * Rg::kChains + ch);
                uint32_t *const ring = ring_of(grp);
                uint8_t *const offs = offs_of(grp);
                const int d0 = slot * Rg::kPhase + 4 * cl;
                qd = qd0;
                ctr1 = ctr0;
#pragma unroll 2
                for (int pass = 0; pass < 4; ++pass) {
                    uint4 b;
                    uint32_t off = 0u;
                    if (POTTS) {
                        const uint4 b0 = philox4x32_10(make_uint4(2u * qd, ctr1, iter, ctr3), key0, key1);
                        const uint4 b1 = philox4x32_10(make_uint4(2u * qd + 1u, ctr1, iter, ctr3), key0, key1);
                        b = make_uint4(b0.x, b0.z, b1.x, b1.z);
                        off = offset7(b0.y) | (offset7(b0.w) << 8) | (offset7(b1.y) << 16) | (offset7(b1.w) << 24);
                    } else {
                        b = philox4x32_10(make_uint4(qd, ctr1, iter, ctr3), key0, key1);
                    }
                    // clamped so that u < A decides (A = 2^32-1 always accepts)
                    b.x = min(b.x, 0xFFFFFFFEu);
                    b.y = min(b.y, 0xFFFFFFFEu);
                    b.z = min(b.z, 0xFFFFFFFEu);
                    b.w = min(b.w, 0xFFFFFFFEu);
                    const int d = d0 + 4 * LPC * pass;
                    *reinterpret_cast<uint4 *>(ring + d) = b;
                    if (POTTS) *reinterpret_cast<uint32_t *>(offs + d) = off;
                    if (pass == 0 && slot == 0) {
                        *reinterpret_cast<uint4 *>(ring + d + Rg::kSites) = b;
                        if (POTTS) *reinterpret_cast<uint32_t *>(offs + d + Rg::kSites) = off;
                    }
                    qd += (uint32_t)LPC;
                    while (qd >= quads) {
                        qd -= quads;
                        ++ctr1;
                    }
                }
                bar_sync(1 + grp, 64);
            }
            qd0 = qd;
            ctr0 = ctr1;
            slot = slot == 2 ? 0 : slot + 1;
        }
    } else {
        // ---------------- the chains ------------------------------------------------------------
        // (padding chains read chain p - 1's spins and never accept; they store nothing)
        const int grp = warp;
        const int c = c0 + grp * Rg::kChains + ch;
        const bool active = c < a.p;
        uint8_t *const lat = reinterpret_cast<uint8_t *>(
            stage_lattice ? s_lat + (size_t)(grp * Rg::kChains + ch) * lat_words
                        : a.lat + (size_t)(active ? c : a.p - 1) * lat_words);
        const uint32_t rowb = 4u * (uint32_t)a.row_words;  // bytes per lattice row
        const int nl = (L + 3) >> 2, jb = AL ? 3 : (L - 1) & 3;  // lanes' worth of sites per row, last site's byte
        const int nq = ROW ? 1 : (nl + LPC - 1) / LPC;     // passes per row
        const char *const tab_g = reinterpret_cast<const char *>(a.ktab31);
        const uint32_t tab0 = TAB == kTabGlobal ? 0u : (uint32_t)__cvta_generic_to_shared(s_tab);
        const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring_of(grp));
        const uint32_t offs_s = (uint32_t)__cvta_generic_to_shared(offs_of(grp));
        const uint32_t hist_s = (uint32_t)__cvta_generic_to_shared(s_hist);
        const uint32_t dummy = hist_s + 4u * (uint32_t)(((n_hist + 3) & ~3) + lane);
        const uint32_t starts = LPC == 2 ? 0x55555555u : LPC == 4 ? 0x11111111u : LPC == 8 ? 0x01010101u : LPC == 16 ? 0x00010001u : 1u;
        const uint32_t prevbit = cl == 0 ? 0u : 1u << (lane - 1);
        const int prevshift = (32 - lane) & 31;  // ... to bit 31
        // sums over the lanes of a chain: each lane's as a byte in shared memory, read back as
        // words and summed up to the lane by byte products (a shuffle scan takes twice as long)
        const uint32_t sums_s = (uint32_t)__cvta_generic_to_shared(s_ring) +
                                (uint32_t)((grp + 1) * (int)ring_bytes(MODEL) - 32 + LPC * ch);
        constexpr int NW = LPC < 4 ? 1 : LPC / 4;  // words of the lanes' bytes
        uint32_t lower[NW];  // 1 in the bytes of the lanes below this one
#pragma unroll
        for (int k = 0; k < NW; ++k)
            lower[k] = cl >= 4 * k + 4 ? m : cl <= 4 * k ? 0u : m & ((1u << (8 * (cl - 4 * k))) - 1u);
        const uint32_t lane_bias = BB + 4u * EB * (uint32_t)cl;

        // sites of a lane (its quad qi of the row), one bit per byte; none of a padding chain
        auto valid_of = [&](int qi) {
            return !active || qi >= nl ? 0u : qi < nl - 1 ? m : m & (0xFFFFFFFFu >> (8 * (3 - jb)));
        };
        // spins of quad qi of row y: raw memory contents, and bytes
        auto raw_load = [&](int y, int qi) -> uint32_t {
            const int k = min(qi, nl - 1);
            const uint8_t *const r = lat + (size_t)y * rowb;
            return POTTS ? *reinterpret_cast<const volatile uint32_t *>(r + 4 * k)
                         : (uint32_t) * reinterpret_cast<const volatile uint8_t *>(r + (k >> 1));
        };
        auto spins = [&](uint32_t raw, int qi, uint32_t vb) -> uint32_t {
            return POTTS ? raw & (vb * 255u) : spread4(raw >> (4 * (qi & 1))) & vb;
        };

        int y = 0, q = 0, qi = cl;  // (long rows) row, pass of the row; quad of the row
        uint32_t vb = valid_of(qi), vm = vb * 255u;
        // (ROW) this lane's spins of the rows being decided and three rows on: byte offsets
        // (TWO: of the row two on; the second pass's share is own1 bytes further)
        uint8_t *const own = lat + (POTTS ? 4 * min(cl, nl - 1) : min(cl, nl - 1) >> 1);
        const uint32_t allb = rowb * (uint32_t)L;
        uint32_t o0 = 0u, o3 = TWO ? 2u * rowb : L > 3 ? 3u * rowb : 0u;
        const uint32_t own1 = (uint32_t)(POTTS ? 4 * (min(LPC + cl, nl - 1) - cl) : (min(LPC + cl, nl - 1) >> 1) - (cl >> 1));
        const uint32_t vb2 = valid_of(LPC + cl);  // (TWO) sites of the second pass
        // neighbouring quads: shuffle sources and byte selectors (a row's ends wrap)
        const int base = ch * LPC;
        const int rsrc = ROW ? base + (cl >= nl - 1 ? 0 : cl + 1) : lane + 1;
        const int lsrc = ROW ? base + (cl == 0 ? nl - 1 : cl - 1) : lane - 1;
        auto rsel_of = [&](int qi) { return qi == nl - 1 && jb < 3 ? (jb == 0 ? 0x3214u : jb == 1 ? 0x3241u : 0x3421u) : 0x4321u; };
        auto lsel_of = [&](int qi) { return qi == 0 ? 0x2104u + (uint32_t)jb : 0x2107u; };
        // the row's last site in this lane's bytes (ROW)
        const uint32_t lastm = ROW && active && cl == nl - 1 ? 1u << (8 * jb) : 0u;
        const uint32_t wjb = COLB << (8 * jb);
        const uint32_t basebit = 1u << base;

        constexpr int SH = TAB == kTabShared16 ? 16 : 1;
        uint32_t u[4], offn = 0u;  // draws >> SH, as the table's entries
        auto load_draws = [&](int pos) {
            const uint32_t s = ring_s + 4u * (uint32_t)(pos + 4 * cl);
            if (AL || (pos & 3) == 0) {
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3])
                             : "r"(s));
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) u[i] = lds32(s + 4u * i);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) u[i] >>= SH;
        };
        auto load_offsets = [&](int pos) {
            const uint32_t o = offs_s + (uint32_t)((pos & ~3) + 4 * cl);
            offn = lds32(o);
            if (!AL) offn = __funnelshift_r(offn, lds32(o + 4u), 8 * (pos & 3));
        };
        // Potts: contribution of neighbours x to the columns dE + 4 of spins R, proposals S
        auto zs = [&](uint32_t x, uint32_t R, uint32_t S) { return nz_bytes(x ^ S) - nz_bytes(x ^ R); };

        // ---- rows in the pipeline: R is being decided; R1, D1 the next pass's spins and the row
        // below it (ROW: the row below is the pass after, loaded as raw2 one pass ahead)
        const int bin0 = active ? (POTTS ? a.E[c] + 2 * V : (a.E[c] + 2 * V) >> 2) : V >> 1;
        int bin = bin0;
        uint32_t R = spins(raw_load(0, qi), qi, vb), SN = 0u;
        uint32_t R1 = 0u, SN1 = 0u, raw2 = 0u;
        uint32_t R2 = 0u, W1 = 0u;  // (TWO) the spins of the pass after the next, the new spins of the pass before
        if (ROW) {
            R1 = spins(raw_load(1, qi), qi, vb);
            raw2 = raw_load(2, qi);
        }
        if (TWO) {
            R1 = spins(raw_load(0, LPC + cl), cl, vb2);
            R2 = spins(raw_load(1, cl), cl, vb);
            raw2 = raw_load(1, LPC + cl);
            W1 = spins(raw_load(L - 1, LPC + cl), cl, vb2);
        }

        // columns of the pass's sites with the left neighbour kept (n0) / changed (n1); dalt:
        // their change at the row's last site if site 0 is changed (ROW)
        uint32_t n0, n1, dalt = 0u;
        uint32_t A0[4], A1[4], B0 = 0u, B1 = 0u;
        auto load_candidates = [&](uint32_t row) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                A0[i] = table_load<TAB>(tab_g, __dp4a(n0, COLB << (8 * i), row));
                A1[i] = table_load<TAB>(tab_g, __dp4a(n1, COLB << (8 * i), row));
            }
            if (ROW) {
                B0 = table_load<TAB>(tab_g, __dp4a(n0 + dalt, wjb, row));
                B1 = table_load<TAB>(tab_g, __dp4a(n1 + dalt, wjb, row));
            }
        };
        // the part of the columns that does not depend on the pass before: spins X, proposals S,
        // row below D, the quads to the right (RN, proposals SNr) and left (LP, SNl)
        auto columns = [&](uint32_t X, uint32_t S, uint32_t D, uint32_t RN, uint32_t LP, uint32_t SNr, uint32_t SNl,
                           uint32_t rsel, uint32_t lsel, uint32_t &k0, uint32_t &k1, uint32_t &da) {
            const uint32_t rt = __byte_perm(X, RN, AL ? 0x4321u : rsel), lf = __byte_perm(X, LP, AL ? 0x2107u : lsel);
            if (POTTS) {
                const uint32_t zr = zs(rt, X, S), b = 4u * m + zs(D, X, S) + zr;
                k0 = b + zs(lf, X, S);
                k1 = b + zs(__byte_perm(S, SNl, AL ? 0x2107u : lsel), X, S);
                if (ROW) {
                    const uint32_t r2 = __byte_perm(X, SNr, AL ? 0x4321u : rsel);  // site 0 changed
                    da = (nz_bytes(r2 ^ S) & lastm) - (nz_bytes(r2 ^ X) & lastm) - (nz_bytes(rt ^ S) & lastm) +
                         (nz_bytes(rt ^ X) & lastm);
                }
            } else {
                const uint32_t tr = X ^ rt, b = (X ^ D) + tr, l = X ^ lf;
                k0 = b + l;
                k1 = b + (l ^ m);
                if (ROW) da = lastm - 2u * (tr & lastm);
            }
        };
        auto upper = [&](uint32_t U, uint32_t X, uint32_t S) { return POTTS ? zs(U, X, S) : U ^ X; };

        // ---- the first pass
        int pos = 0, sw = 0;
        // draws handed off and not yet in a pass; hand-offs taken
        int ahead = Rg::kPhase - (ROW ? L : min(4 * LPC, L)), taken = 1;
        bar_sync(1 + grp, 64);
        load_draws(0);
        if (POTTS) load_offsets(0);
        uint32_t first = 0u;  // (long rows) the row's first quad, new
        {
            if (POTTS) SN = (R + m + offn) & (7u * m);
            uint32_t RN, LP, SNr = 0u, SNl = 0u;
            RN = __shfl_sync(~0u, R, rsrc & 31);
            LP = __shfl_sync(~0u, R, lsrc & 31);
            if (POTTS) {
                SNr = __shfl_sync(~0u, SN, rsrc & 31);
                SNl = __shfl_sync(~0u, SN, lsrc & 31);
            }
            if (!ROW) {
                const uint32_t rr = spins(raw_load(0, 32), 32, POTTS ? m : m), ll = spins(raw_load(0, nl - 1), nl - 1, m);
                if (lane == 31) RN = rr;
                if (lane == 0) LP = ll;
            }
            const uint32_t D = ROW ? R1 : spins(raw_load(1, qi), qi, vb), U = spins(raw_load(L - 1, qi), qi, vb);
            columns(R, SN, D, RN, LP, SNr, SNl, rsel_of(qi), lsel_of(qi), n0, n1, dalt);
            const uint32_t t = upper(U, R, SN);
            n0 += t;
            n1 += t;
        }
        load_candidates(tab0 + ROWB * (uint32_t)bin);
        const int passes = a.n_sweeps * L * nq;
        const bool record = !HIST && (a.E_rec || a.M_rec || a.samples);
        int ups = 0;          // Ising records: spins up in the sweep so far
        StateCounts counts;   // Potts records: states in the sweep so far
        int rows = 0;
        const int flush_rows = HMODE == kHist16 ? max(1, 65535 / (lw * L)) : 0;
        const uint32_t rselw = ROW ? rsel_of(cl) : 0u, lselw = ROW ? lsel_of(cl) : 0u;

        // repetitions that a launch may need at most (max_launch_sweeps keeps this an int).
        // Beyond, no site is decided any more: a pass then agrees with itself and the launch
        // ends.  (One allowance per launch and no exit of its own from the loop: a count per
        // pass with a break took 3661 instead of 2967 us at 64 x 64, p = 14592.)
        int left = passes * (4 * LPC + 2);
        for (int it = 0; it < passes; ++it) {
            const bool lastq = ROW || q == nq - 1;
            // ---- the next pass: what does not depend on this one's decisions
            int y1 = y, q1 = q + 1;
            if (!ROW && lastq) {
                q1 = 0;
                if (!TWO) y1 = y + 1 == L ? 0 : y + 1;
            }
            const bool last_row = ROW || TWO ? o0 + rowb == allb : y == L - 1;
            const int qi1 = ROW ? cl : q1 * LPC + cl;
            // its draws
            const int len = ROW ? L : min(4 * LPC, L - 4 * LPC * q), len1 = ROW ? L : min(4 * LPC, L - 4 * LPC * q1);
            const int skip = !AL && lastq && last_row ? VS - V : 0;
            int pos1 = pos + len + skip;
            pos1 = pos1 >= Rg::kSites ? pos1 - Rg::kSites : pos1;
            uint32_t D1 = 0u, vb1 = vb, rsel1 = rselw, lsel1 = lselw, U1 = 0u, rr = 0u, ll = 0u;
            auto next_pass = [&] {
                ahead -= skip + len1;
                if (PEEL) {
                    bar_sync_if(ahead < 0 && taken < phases, 1 + grp, 64);
                    taken -= ahead >> 31;
                    ahead += (ahead >> 31) & Rg::kPhase;
                } else if (ahead < 0) {
                    if (taken < phases) bar_sync(1 + grp, 64);
                    ++taken;
                    ahead += Rg::kPhase;
                }
                if (POTTS) load_offsets(pos1);
                if (ROW) return;
                if (TWO) {
                    vb1 = q1 ? vb2 : active ? m : 0u;
                    D1 = spins(raw2, cl, vb1);
                    U1 = W1;
                    rsel1 = rsel_of(qi1);
                    lsel1 = lsel_of(qi1);
                    return;
                }
                vb1 = valid_of(qi1);
                R1 = spins(raw_load(y1, qi1), qi1, vb1);
                D1 = spins(raw_load(y1 + 1 == L ? 0 : y1 + 1, qi1), qi1, vb1);
                U1 = spins(raw_load(y1 == 0 ? L - 1 : y1 - 1, qi1), qi1, vb1);
                // the quad behind the pass (old), and the row's last one (old)
                rr = spins(raw_load(y1, (q1 + 1) * LPC), 0, m);
                ll = spins(raw_load(y1, nl - 1), nl - 1, m);
                rsel1 = rsel_of(qi1);
                lsel1 = lsel_of(qi1);
            };

            if (!PEEL) next_pass();

            // ---- predict
            // (ROW) all ones in the lane of the row's last site if site 0 is changed: site 0's
            // test is exact (its bin is the pass's first; an open one is found below), and the
            // last site's right neighbour is fixed by it
            uint32_t flip = 0u;
            if (ROW) {
                const bool f = (__ballot_sync(~0u, (int)(u[0] - A0[0]) < 0) & basebit) != 0u && lastm;
                flip = f ? ~0u : 0u;
                n0 += dalt & flip;
                n1 += dalt & flip;
                if (!AL) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        A0[i] = f && i == jb ? B0 : A0[i];
                        A1[i] = f && i == jb ? B1 : A1[i];
                    }
                }
            }
            uint32_t dm, lm, N, X, Q, e, Rw, k0, k1, da, SNr = 0u, SNl = 0u, RN1, LP1, T[4], df[4], bad, open, nib = 0u;
            int bin1, binw;
            auto attempt = [&](auto first_try) {
                // the lane's four sites for either incoming bit (signs: 0 kept, 1 changed), then
                // the incoming bits
                uint32_t d0, d1, b0, b1;
                {
                    uint32_t f0[4], f1[4];
                    f0[0] = u[0] - A0[0];
                    f1[0] = u[0] - A1[0];
#pragma unroll
                    for (int i = 1; i < 4; ++i) {
                        const uint32_t p = u[i] - A0[i], r = u[i] - A1[i];
                        f0[i] = select(f0[i - 1], r, p);
                        f1[i] = select(f1[i - 1], r, p);
                    }
                    b0 = __ballot_sync(~0u, (int)f0[3] < 0);
                    b1 = __ballot_sync(~0u, (int)f1[3] < 0);
                    if (ROW && AL) {
                        // (the last lane's outgoing bits are not used, so that only its own last
                        // decision waits for site 0's)
                        const uint32_t p = u[3] - B0, r = u[3] - B1;
                        f0[3] = select(flip, select(f0[2], r, p), f0[3]);
                        f1[3] = select(flip, select(f1[2], r, p), f1[3]);
                    }
                    d0 = sign_bytes(f0[0], f0[1], f0[2], f0[3]);
                    d1 = sign_bytes(f1[0], f1[1], f1[2], f1[3]);
                }
                if constexpr (decltype(first_try)::value) {
                    // (the next pass's spins, neighbours and columns fill the gaps of this chain)
                    if (PEEL) next_pass();
                    if (POTTS) SN1 = (R1 + m + offn) & (7u * m);
                    // (TWO, first pass: to lane 31's right is the second pass, to lane 0's left its
                    // last quad)
                    RN1 = __shfl_sync(~0u, TWO && lane == 0 && q1 == 0 ? R2 : R1, rsrc & 31);
                    LP1 = __shfl_sync(~0u, R1, lsrc & 31);
                    if (POTTS) {
                        SNl = __shfl_sync(~0u, SN1, lsrc & 31);
                        if (ROW) SNr = __shfl_sync(~0u, SN1, rsrc & 31);
                    }
                    if (ROW) {
                        D1 = spins(raw2, cl, vb);
                        columns(R1, SN1, D1, RN1, LP1, SNr, SNl, rsel1, lsel1, k0, k1, da);
                    } else {
                        if (TWO) ll = __shfl_sync(~0u, R2, nl - 1 - LPC);
                        else RN1 = lane == 31 ? rr : RN1;
                        LP1 = lane == 0 && q1 == 0 ? ll : LP1;
                    }
                }
                b1 = (b1 & ~starts) | (b0 & starts);  // (a chain's first lane has no incoming change)
#pragma unroll
                for (int s = 1; s < LPC; s <<= 1) {
                    const uint32_t l0 = b0 << s, l1 = b1 << s;
                    const uint32_t x = (l0 & b1) | (~l0 & b0), z = (l1 & b1) | (~l1 & b0);
                    b0 = x;
                    b1 = z;
                }
                // (all ones where the lane before ends with a change)
                const uint32_t cin = (uint32_t)((int)((b0 & prevbit) << prevshift) >> 31);
                dm = select(cin, d1, d0) & vm;
                // columns of the sites as they were met, bin changes plus EB
                lm = __byte_perm(dm, cin, 0x2104);
                N = select(lm, n1, n0);
                e = select(dm, POTTS ? N : 4u * m - N, EB * m);
                // sums over the lane's sites and the chain's lanes: bins before (X) and after (Q)
                // every attempt are binw + byte
                const uint32_t s = e * m;
                uint32_t below = 0u, tot = 0u;
                {
                    asm volatile("st.shared.u8 [%0], %1;" ::"r"(sums_s + (uint32_t)cl), "r"(s >> 24) : "memory");
                    __syncwarp();
                    uint32_t w[NW];
                    if constexpr (LPC == 2) {
                        uint16_t h;
                        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(sums_s) : "memory");
                        w[0] = h;
                    } else if constexpr (LPC == 4) {
                        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[0]) : "r"(sums_s) : "memory");
                    } else if constexpr (LPC == 8) {
                        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(sums_s) : "memory");
                    } else {
#pragma unroll
                        for (int k = 0; k < LPC / 4; k += 4)
                            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                         : "=r"(w[k]), "=r"(w[k + 1]), "=r"(w[k + 2]), "=r"(w[k + 3])
                                         : "r"(sums_s + 4u * k)
                                         : "memory");
                    }
#pragma unroll
                    for (int k = 0; k < NW; ++k) below = __dp4a(w[k], lower[k], below);
#pragma unroll
                    for (int k = 0; k < NW; ++k) tot = __dp4a(w[k], m, tot);
                }
                bin1 = bin + (int)tot - (int)(4u * EB * LPC);
                binw = bin + (int)below - (int)lane_bias;
                X = s * 256u + (POTTS ? 0x04080C10u : 0x02040608u);
                Q = s + (POTTS ? 0x0004080Cu : 0x00020406u);
                const uint32_t rw = tab0 + ROWB * (uint32_t)binw;
                // verify
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint32_t ad = __dp4a(N, COLB << (8 * i), __dp4a(X, ROWB << (8 * i), rw));
                    T[i] = table_load<TAB>(tab_g, ad);
                }
                Rw = POTTS ? select(dm, SN, R) : R ^ (dm & m);
                if (!POTTS && !PEEL) {
                    nib = pack4(Rw);
                    nib |= __shfl_down_sync(~0u, nib, 1) << 4;
                }
                if (!ROW) {
                    // the row's first quad, and the quad before the next pass
                    const uint32_t fw = __shfl_sync(~0u, Rw, 0), pv = __shfl_sync(~0u, Rw, 31);
                    columns(R1, SN1, D1, qi1 == nl - 1 ? (TWO || q == 0 ? fw : first) : RN1, lane == 0 && q1 > 0 ? pv : LP1, 0u,
                            SNl, rsel1, lsel1, k0, k1, da);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) df[i] = u[i] - T[i];
                open = min(min(df[0], df[1]), min(df[2], df[3]));  // zero: a test is open
                bad = (sign_bytes(df[0], df[1], df[2], df[3]) ^ dm) & vm;
            };
            if constexpr (PEEL) attempt(std::true_type{});
            for (;;) {
                if constexpr (!PEEL) attempt(std::true_type{});
                if (!__any_sync(~0u, bad != 0u || open == 0u)) break;
                if (__any_sync(~0u, open == 0u)) {
                    // draws that equal their entries: the 32-bit tests decide
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (df[i] == 0u && vb & (1u << (8 * i))) {
                            const uint32_t b = (uint32_t)binw + ((X >> (8 * i)) & 0xFFu);
                            const uint32_t A = __ldg(a.ktab + NC * b + ((N >> (8 * i)) & 0xFFu));
                            T[i] = lds32(ring_s + 4u * (uint32_t)(pos + 4 * cl + i)) < A ? 0x80000000u : 0u;
                            df[i] = u[i] - T[i];
                        }
                    }
                    bad = (sign_bytes(df[0], df[1], df[2], df[3]) ^ dm) & vm;
                    if (ROW) {
                        // site 0 (its neighbours and bin are exact): what the last site saw of it
                        const bool f = (__ballot_sync(~0u, (int)df[0] < 0) & basebit) != 0u && lastm;
                        const uint32_t flip1 = f ? ~0u : 0u;
                        n0 += (dalt & flip1) - (dalt & flip);
                        n1 += (dalt & flip1) - (dalt & flip);
                        bad |= flip1 ^ flip;
                        flip = flip1;
                    }
                    if (!__any_sync(~0u, bad != 0u)) break;
                }
                if (--left < 0) {
                    if (lane == 0) *reinterpret_cast<volatile int *>(a.fault) = 1;
                    vm = 0u;
                }
                // repair: the verified thresholds, for the left neighbours as met
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool l = (lm >> (8 * i)) & 1u;
                    A1[i] = l ? T[i] : A1[i];
                    A0[i] = l ? A0[i] : T[i];
                    if (ROW && AL && i == 3) {
                        B1 = l ? T[i] : B1;
                        B0 = l ? B0 : T[i];
                    }
                }
                if constexpr (PEEL) attempt(std::false_type{});
            }

            // ---- the next pass's candidates and draws (their latency is hidden by what follows)
            {
                const uint32_t t = upper(ROW ? Rw : U1, R1, SN1);
                n0 = k0 + t;
                n1 = k1 + t;
                dalt = ROW ? da : 0u;
                load_candidates(tab0 + ROWB * (uint32_t)bin1);
                load_draws(pos1);
                if (!POTTS && PEEL) {
                    nib = pack4(Rw);
                    nib |= __shfl_down_sync(~0u, nib, 1) << 4;
                }
            }
            // ---- commit
            {
                uint8_t *const r = ROW ? own + o0 : TWO ? own + (o0 + (q ? own1 : 0u)) : lat + (size_t)y * rowb + (POTTS ? 4 * qi : qi >> 1);
                if (POTTS) {
                    if (vb) *reinterpret_cast<volatile uint32_t *>(r) = Rw;
                } else {
                    if (vb && !(cl & 1)) *reinterpret_cast<volatile uint8_t *>(r) = (uint8_t)nib;
                }
            }
            __syncwarp();  // other lanes read these spins
            if (!ROW && !TWO && q == 0) first = __shfl_sync(~0u, Rw, 0);
            if (HIST) {
                constexpr bool part = !AL;  // (a row's last lane has fewer than four sites)
                if (HMODE == kHistPairs) {
                    const uint32_t h0 = vb ? hist_s + 4u * NC * (uint32_t)binw : dummy - 4u * (NC * BB + EB);
#pragma unroll
                    for (int i = 1; i < 4; i += 2) {
                        uint32_t ad = __dp4a(e, 4u << (8 * i), __dp4a(Q, (4u * NC) << (8 * (i - 1)), h0));
                        if (part && !(vb & (1u << (8 * i)))) ad = dummy;
                        red_shared(ad, 1u);
                    }
                } else if (HMODE == kHistSingle) {
                    const uint32_t h0 = vb ? hist_s + 4u * (uint32_t)binw : dummy - 4u * BB;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t ad = __dp4a(Q, 4u << (8 * i), h0);
                        if (part && !(vb & (1u << (8 * i)))) ad = dummy;
                        red_shared(ad, 1u);
                    }
                } else if (HMODE == kHist16) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t b = (uint32_t)binw + ((Q >> (8 * i)) & 0xFFu);
                        red_shared(vb & (1u << (8 * i)) ? hist_s + 4u * (b >> 1) : dummy, 1u << ((b & 1u) << 4));
                    }
                } else {
                    // runs of equal bins among the lane's four
                    uint32_t run = 0u, prev = 0u;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t b = (uint32_t)binw + ((Q >> (8 * i)) & 0xFFu);
                        if (vb & (1u << (8 * i))) {
                            if (run && b != prev) {
                                atomicAdd(reinterpret_cast<unsigned long long *>(a.H + prev), (unsigned long long)run);
                                run = 0u;
                            }
                            prev = b;
                            ++run;
                        }
                    }
                    if (run) atomicAdd(reinterpret_cast<unsigned long long *>(a.H + prev), (unsigned long long)run);
                }
            }
            bin = bin1;
            if (record) {
                if (POTTS) {
                    counts.add(Rw);
                    if ((it & 31) == 31) counts.flush();
                } else {
                    ups = (int)__dp4a(Rw, m, (uint32_t)ups);
                }
            }
            if (lastq) {
                if (record && last_row) {
                    int M;
                    if (POTTS) {
                        counts.flush();
                        counts.template reduce<LPC>((uint32_t)(4 * LPC * nq - L) * (uint32_t)L);
                        M = 8 * (int)counts.max_count() - V;
                        counts = StateCounts();
                    } else {
#pragma unroll
                        for (int x = 1; x < LPC; x <<= 1) ups += __shfl_xor_sync(~0u, ups, x);
                        M = 2 * ups - V;
                        ups = 0;
                    }
                    if (active && cl == 0) {
                        const int E = POTTS ? bin - 2 * V : 4 * bin - 2 * V;
                        if (a.E_rec) a.E_rec[(size_t)sw * a.rec_stride + c] = E;
                        if (a.M_rec) a.M_rec[(size_t)sw * a.rec_stride + c] = M;
                        if (a.samples) {
                            const unsigned long long am = (unsigned long long)(M < 0 ? -M : M);
                            unsigned long long *sp = reinterpret_cast<unsigned long long *>(a.samples);
                            atomicAdd(&sp[bin], 1ull);
                            atomicAdd(&sp[n_bins + bin], am);
                            atomicAdd(&sp[2 * n_bins + bin], am * am);
                        }
                    }
                    ++sw;
                }
                if (HMODE == kHist16 && ++rows == flush_rows && it + 1 < passes) {
                    // every decider warp has run the same rows: no count has reached 2^16
                    rows = 0;
                    bar_sync(kFlushBarrier, 32 * G);
                    for (int i = tid; i < n_hist; i += 32 * G) {
                        const uint32_t x = s_hist[i];
                        if (x) {
                            s_hist[i] = 0u;
                            unsigned long long *Hg = reinterpret_cast<unsigned long long *>(a.H) + 2 * i;
                            if (x & 0xFFFFu) atomicAdd(Hg, (unsigned long long)(x & 0xFFFFu));
                            if (x >> 16) atomicAdd(Hg + 1, (unsigned long long)(x >> 16));
                        }
                    }
                    bar_sync(kFlushBarrier, 32 * G);
                }
            }
            R = R1;
            SN = SN1;
            if (ROW) {
                R1 = D1;
                // (now that this row is final: the row below the pass after next)
                raw2 = POTTS ? *reinterpret_cast<const volatile uint32_t *>(own + o3)
                             : (uint32_t) * reinterpret_cast<const volatile uint8_t *>(own + o3);
                o0 = last_row ? 0u : o0 + rowb;
                o3 = o3 + rowb == allb ? 0u : o3 + rowb;
            }
            if (TWO) {
                R1 = R2;
                R2 = D1;
                W1 = Rw;
                // (final by now: the row below the pass after next)
                const uint8_t *const r = own + (o3 + (q ? own1 : 0u));
                raw2 = POTTS ? *reinterpret_cast<const volatile uint32_t *>(r)
                             : (uint32_t) * reinterpret_cast<const volatile uint8_t *>(r);
                if (lastq) {
                    o0 = last_row ? 0u : o0 + rowb;
                    o3 = o3 + rowb == allb ? 0u : o3 + rowb;
                }
            }
            if (!ROW) {
                vb = vb1;
                vm = vb * 255u;
            }
            qi = qi1;
            y = y1;
            q = q1;
            pos = pos1;
        }
        // magnetisation (and state counts) of the final lattice, a share of the words per lane
        const uint32_t *const words = reinterpret_cast<const uint32_t *>(lat);
        if (POTTS) {
            StateCounts n;
            int k = cl, i = 0;
            for (; k < lat_words; k += LPC) {
                n.add(words[k]);
                if ((++i & 31) == 0) n.flush();
            }
            n.flush();
            n.template reduce<LPC>((uint32_t)(4 * lat_words - V));
            if (active && cl == 0) {
                a.E[c] = bin - 2 * V;
                a.M[c] = 8 * (int)n.max_count() - V;
                a.cnt[c] = n.low();
                a.cnt[a.p_pad + c] = n.high();
            }
        } else {
            int n = 0;
            for (int k = cl; k < lat_words; k += LPC) n += __popc(words[k]);
#pragma unroll
            for (int x = 1; x < LPC; x <<= 1) n += __shfl_xor_sync(~0u, n, x);
            if (active && cl == 0) {
                a.E[c] = 4 * bin - 2 * V;
                a.M[c] = 2 * n - V;
            }
        }
    }
    __syncthreads();
    if (stage_lattice)
        for (int i = tid; i < lat_words * n_own; i += nt) a.lat[(size_t)c0 * lat_words + i] = s_lat[i];
    unsigned long long *const H = reinterpret_cast<unsigned long long *>(a.H);
    if (HMODE == kHistPairs) {
        // first attempts of the pairs in bin b, then second attempts (from bin b - d)
        for (int b = tid; b < n_bins; b += nt) {
            uint32_t s = 0u;
#pragma unroll
            for (int d = -(int)EB; d <= (int)EB; ++d) {
                s += s_hist[(int)NC * b + (int)EB + d];
                if (b - d >= 0 && b - d < n_bins) s += s_hist[(int)NC * (b - d) + (int)EB + d];
            }
            if (s) atomicAdd(H + b, (unsigned long long)s);
        }
    } else if (HMODE == kHist16) {
        for (int i = tid; i < n_hist; i += nt) {
            const uint32_t x = s_hist[i];
            if (x & 0xFFFFu) atomicAdd(H + 2 * i, (unsigned long long)(x & 0xFFFFu));
            if (x >> 16) atomicAdd(H + 2 * i + 1, (unsigned long long)(x >> 16));
        }
    } else {
        for (int i = tid; i < n_hist; i += nt) {
            const uint32_t x = s_hist[i];
            if (x) atomicAdd(H + i, (unsigned long long)x);
        }
    }
}

}  // namespace sweep
}  // namespace muca
