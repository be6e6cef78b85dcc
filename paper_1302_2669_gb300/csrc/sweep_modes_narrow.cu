// The kernels of sweep_modes.cu for planes of 4 and 8 chains.
#include "sweep_modes.cuh"

namespace surfmcmc {

cudaError_t launch_sweep_modes_narrow(const SweepParams& p, int lam, cudaStream_t s) {
    return launch_modes_narrow_planes<false>(p, lam, s);
}

}  // namespace surfmcmc
