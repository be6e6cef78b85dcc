// Sweep kernels with the digit-plane modes known at compile time (the three
// head patterns, see head_pattern), for depolarizing noise and 4, 8, 16 or 32
// lanes per bundle (independent flips: sweep_modes_flips.cu).
#include "sweep_modes.cuh"

namespace surfmcmc {

cudaError_t launch_sweep_modes(const SweepParams& p, int lam, cudaStream_t s) {
    if (p.noise == 1) return launch_sweep_modes_flips(p, lam, s);
    return p.G >= 16 ? launch_modes_wide_planes<false>(p, lam, s) : launch_sweep_modes_narrow(p, lam, s);
}

}  // namespace surfmcmc
