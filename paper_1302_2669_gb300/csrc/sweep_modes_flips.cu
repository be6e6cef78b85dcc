// The kernels of sweep_modes.cu for independent bit and phase flips.
#include "sweep_modes.cuh"

namespace surfmcmc {

cudaError_t launch_sweep_modes_flips(const SweepParams& p, int lam, cudaStream_t s) {
    if (p.G == 16) return launch_modes_16<true>(p, lam, s);
    return p.G == 32 ? launch_modes_32<true>(p, lam, s) : cudaErrorNotSupported;
}

}  // namespace surfmcmc
