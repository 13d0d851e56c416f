// Mixed instantiations: float storage and arithmetic, with the fifth
// difference of the detector (Eq. eq28), whose cancellation decides the
// hybrid switch, formed as exact nested float differences.
#include "weno_launch.cuh"

namespace wis {

cudaError_t sweep_mixed(int dim, int dir, int variant, const SweepArgs& a, cudaStream_t s)
{
    return launch_sweep_t<float, true>(dim, dir, variant, a, s);
}

cudaError_t run1d_prepare_mixed(int* max_cluster) { return run1d_prepare<float, true>(max_cluster); }
cudaError_t run1d_mixed(const Run1DArgs& r, int ctas, cudaStream_t s) { return launch_run1d<float, true>(r, ctas, s); }

}  // namespace wis
