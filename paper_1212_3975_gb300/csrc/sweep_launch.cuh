// Launch of a sweep body as a kernel of its own: one block per `chains` chains.
#pragma once
#include "sweep_small.cuh"

namespace muca {
namespace sweep {

// Blocks of at most this many groups take the body with the first attempt peeled.  20
// sweeps and an update, peeled / not: Ising 64 x 64, 4 groups 489 / 498 us, 6 groups
// 607 / 609, 8 groups 662 / 664, 12 groups (p = 14592) 3331 / 2968; 8-Potts 32 x 32, 4
// groups 336 / 355, 6 groups 424 / 432, 8 groups 489 / 493.  First iterations, whose
// passes repeat often (64 x 64, p = 1024): 4.13 / 4.24 ms.
constexpr int kPeelGroups = 6;

template <int MODEL, int LPC, bool ROW, bool AL, int TAB, int HMODE, bool PEEL, bool TWO>
__global__ void __launch_bounds__(block_threads(kMaxGroups), 1) sweep_kernel(SweepArgs a, int groups, bool stage_lattice)
{
    extern __shared__ __align__(16) uint32_t smem[];
    sweep_body<MODEL, LPC, ROW, AL, TAB, HMODE, PEEL, TWO>(a, blockIdx.x, groups, stage_lattice, smem);
}

template <int MODEL, int LPC, bool ROW, bool AL, int TAB, int HMODE, bool PEEL, bool TWO>
cudaError_t launch_as(const SweepLaunch &l)
{
    auto kern = sweep_kernel<MODEL, LPC, ROW, AL, TAB, HMODE, PEEL, TWO>;
    if (l.shape.smem > 48 * 1024) {  // (one limit for all: another thread may launch the kernel too)
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return e;
    }
    kern<<<l.blocks, block_threads(l.shape.groups), l.shape.smem, l.stream>>>(l.args, l.shape.groups, l.shape.lattice);
    return cudaGetLastError();
}

template <int MODEL, int LPC, bool ROW, bool AL, int TAB, int HMODE>
cudaError_t launch(const SweepLaunch &l)
{
    if constexpr (ROW && TAB != kTabShared16)
        if (l.shape.groups <= kPeelGroups) return launch_as<MODEL, LPC, ROW, AL, TAB, HMODE, true, false>(l);
    if constexpr (!ROW)
        if (l.args.L <= 8 * LPC) return launch_as<MODEL, LPC, ROW, AL, TAB, HMODE, false, true>(l);
    return launch_as<MODEL, LPC, ROW, AL, TAB, HMODE, false, false>(l);
}

template <int L, bool HIST>
__global__ void __launch_bounds__(block_threads(kMaxGroups), 1) small_kernel(SweepArgs a, int groups)
{
    extern __shared__ __align__(16) uint32_t smem[];
    small_body<L, HIST>(a, blockIdx.x, groups, smem);
}

template <int L, bool HIST>
cudaError_t launch_small_as(const SweepLaunch &l)
{
    auto kern = small_kernel<L, HIST>;
    if (l.shape.smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return e;
    }
    kern<<<l.blocks, block_threads(l.shape.groups), l.shape.smem, l.stream>>>(l.args, l.shape.groups);
    return cudaGetLastError();
}

template <bool HIST>
cudaError_t launch_small(const SweepLaunch &l)
{
    switch (l.args.L) {
    case 4: return launch_small_as<4, HIST>(l);
    case 6: return launch_small_as<6, HIST>(l);
    case 8: return launch_small_as<8, HIST>(l);
    case 10: return launch_small_as<10, HIST>(l);
    case 12: return launch_small_as<12, HIST>(l);
    case 14: return launch_small_as<14, HIST>(l);
    case 16: return launch_small_as<16, HIST>(l);
    case 18: return launch_small_as<18, HIST>(l);
    case 20: return launch_small_as<20, HIST>(l);
    case 22: return launch_small_as<22, HIST>(l);
    case 24: return launch_small_as<24, HIST>(l);
    case 26: return launch_small_as<26, HIST>(l);
    case 28: return launch_small_as<28, HIST>(l);
    case 30: return launch_small_as<30, HIST>(l);
    case 32: return launch_small_as<32, HIST>(l);
    default: return cudaErrorInvalidConfiguration;
    }
}

// The histogram modes that the plan has for a shape: tables in shared memory leave room
// for one of single attempts at least (pairs with aligned rows); rows of one pass have at
// most 128 x 128 sites, whose 32-bit histogram fits; long rows have any but pairs.
template <int MODEL, int LPC, bool ROW, bool AL, int TAB>
cudaError_t launch_hist(const SweepLaunch &l, bool hist)
{
    if (!hist) return launch<MODEL, LPC, ROW, AL, TAB, kHistNone>(l);
    switch (hist_mode(l.plan)) {
    case kHistSingle: return launch<MODEL, LPC, ROW, AL, TAB, kHistSingle>(l);
    case kHistPairs:
        if constexpr (AL && TAB == kTabShared) return launch<MODEL, LPC, ROW, AL, TAB, kHistPairs>(l);
        break;
    case kHist16:
        if constexpr (!ROW && MODEL == MUCA_ISING) return launch<MODEL, LPC, ROW, AL, TAB, kHist16>(l);
        break;
    default:
        if constexpr (!ROW) return launch<MODEL, LPC, ROW, AL, TAB, kHistGlobal>(l);
    }
    return cudaErrorInvalidConfiguration;  // not planned
}

// (the table is in shared memory up to L = 64 for Ising and L = 32 for Potts: plan_sweeps)
template <int MODEL, bool AL>
cudaError_t launch_shape(const SweepLaunch &l, bool hist)
{
    const bool ts = l.plan.table_smem;
    switch (l.shape.lpc) {
    case 1:
        if constexpr (MODEL == MUCA_ISING) return hist ? launch_small<true>(l) : launch_small<false>(l);
        return cudaErrorInvalidConfiguration;
    case 2:
        if constexpr (MODEL == MUCA_POTTS) return ts ? launch_hist<MODEL, 2, true, AL, kTabShared>(l, hist) : cudaErrorInvalidConfiguration;
        return cudaErrorInvalidConfiguration;
    case 4:
        if constexpr (MODEL == MUCA_POTTS) return ts ? launch_hist<MODEL, 4, true, AL, kTabShared>(l, hist) : cudaErrorInvalidConfiguration;
        return cudaErrorInvalidConfiguration;
    case 8: return ts ? launch_hist<MODEL, 8, true, AL, kTabShared>(l, hist) : cudaErrorInvalidConfiguration;
    case 16:
        if constexpr (MODEL == MUCA_ISING) {
            if constexpr (AL)
                if (l.plan.t16)
                    return hist ? launch<MODEL, 16, true, true, kTabShared16, kHistSingle>(l)
                                : launch<MODEL, 16, true, true, kTabShared16, kHistNone>(l);
            return ts ? launch_hist<MODEL, 16, true, AL, kTabShared>(l, hist) : cudaErrorInvalidConfiguration;
        } else {
            return ts ? cudaErrorInvalidConfiguration : launch_hist<MODEL, 16, true, AL, kTabGlobal>(l, hist);
        }
    default:
        if (ts) return cudaErrorInvalidConfiguration;
        return l.shape.row ? launch_hist<MODEL, 32, true, AL, kTabGlobal>(l, hist)
                           : launch_hist<MODEL, 32, false, AL, kTabGlobal>(l, hist);
    }
}

template <int MODEL>
cudaError_t launch_model(const SweepLaunch &l, bool hist)
{
    return l.args.L % 4 == 0 ? launch_shape<MODEL, true>(l, hist) : launch_shape<MODEL, false>(l, hist);
}

}  // namespace sweep
}  // namespace muca
