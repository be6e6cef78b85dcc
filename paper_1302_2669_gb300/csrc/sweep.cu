// Sweep kernel instantiations for depolarizing noise, the shared-memory and
// work-unit sizes, and the launch entry points (independent bit and phase
// flips are instantiated in sweep_flips.cu).
#include "sweep_kernel.cuh"

namespace surfmcmc {

size_t sweep_smem_bytes(int nq, int nc, int lam) {
    const int B = 32 / lam;
    return (size_t)8 * nc * 4 +
           (size_t)kWarps * ((size_t)B * (kHeadFixedWords + bundle_stride(nq, lam)) + warp_aux_words(B)) * 4;
}

long long sweep_units(long long n_bundles, int lam) { return (n_bundles + (long long)kWarps * (32 / lam) - 1) /
                                                               ((long long)kWarps * (32 / lam)); }

cudaError_t launch_sweep(const SweepParams& p, int lam, cudaStream_t s) {
    if (p.scan) return launch_sweep_scan(p, s);
    if (p.wide) return launch_sweep_wide(p, s);
    // kernels with the launch's digit-plane modes compiled in, where they exist
    const cudaError_t e = launch_sweep_modes(p, lam, s);
    if (e != cudaErrorNotSupported) return e;
    return p.noise == 1 ? launch_sweep_flips(p, lam, s) : launch_noise<false>(p, lam, s);
}

}  // namespace surfmcmc
