// Standalone launches of the 8-Potts sweep bodies (sweep_body.cuh).
#include "sweep_launch.cuh"

namespace muca {
cudaError_t launch_sweep_potts(const SweepLaunch &l, bool hist)
{
    return sweep::launch_model<MUCA_POTTS>(l, hist);
}
}  // namespace muca
