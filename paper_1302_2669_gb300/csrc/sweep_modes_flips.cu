// The kernels of sweep_modes.cu for independent bit and phase flips.
#include "sweep_modes.cuh"

namespace surfmcmc {

cudaError_t launch_sweep_modes_flips(const SweepParams& p, int lam, cudaStream_t s) {
    return p.G >= 16 ? launch_modes_wide_planes<true>(p, lam, s) : cudaErrorNotSupported;
}

}  // namespace surfmcmc
