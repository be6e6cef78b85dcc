// The kernels of sweep_modes.cu for planes of 16 chains.
#include "sweep_modes.cuh"

namespace surfmcmc {

cudaError_t launch_sweep_modes_16(const SweepParams& p, int lam, cudaStream_t s) {
    return launch_modes_16<false>(p, lam, s);
}

}  // namespace surfmcmc
