// Sweep kernels with the digit-plane modes known at compile time (the four
// head patterns, see head_pattern), for depolarizing noise and 2 to 32 lanes
// per bundle, here on planes of 32 chains (16: sweep_modes_16.cu; 4 and 8:
// sweep_modes_narrow.cu; independent flips: sweep_modes_flips.cu).
#include "sweep_modes.cuh"

namespace surfmcmc {

cudaError_t launch_sweep_modes(const SweepParams& p, int lam, cudaStream_t s) {
    if (p.noise == 1) return launch_sweep_modes_flips(p, lam, s);
    if (p.G == 16) return launch_sweep_modes_16(p, lam, s);
    return p.G == 32 ? launch_modes_32<false>(p, lam, s) : launch_sweep_modes_narrow(p, lam, s);
}

}  // namespace surfmcmc
