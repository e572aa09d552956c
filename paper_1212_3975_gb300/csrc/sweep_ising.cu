// Standalone launches of the Ising sweep bodies (sweep_body.cuh).
#include "sweep_launch.cuh"

namespace muca {
cudaError_t launch_sweep_ising(const SweepLaunch &l, bool hist)
{
    return sweep::launch_model<MUCA_ISING>(l, hist);
}
}  // namespace muca
