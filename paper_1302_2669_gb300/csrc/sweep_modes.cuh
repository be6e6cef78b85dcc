// Launchers of the sweep kernels with a compiled-in head pattern.  The
// 32-chain kernels take every chain of a bundle as valid, so they serve
// launches whose chain count per syndrome is a multiple of 32.  Launches
// without such a kernel (cudaErrorNotSupported, nothing launched) use those of
// sweep.cu, which read the modes from their parameters.
#pragma once
#include "sweep_kernel.cuh"

namespace surfmcmc {

// Whether a launch of 32-chain planes at 16 lanes fills less than half of the
// device's resident blocks.  Such a launch runs at the latency of its units,
// which is 2 to 6 % shorter with the bundle's map kept (L = 4 .. 13); fuller
// ones run faster without it (16,384 syndromes of 64 chains at L = 13, 1,000
// sweeps: 113.1 against 115.0 ms; at L = 17, 300 sweeps: 60.3 against 61.9) but
// for some sizes with a short last wave (10,000 syndromes at L = 13, 600 sweeps:
// 45.8 against 44.2).
static inline bool few_units(const SweepParams& p) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return true;
    return 2 * p.total_units < (long long)sms * sweep_blocks_per_sm(32, 16);
}

template <int G, bool IND, int HM>
static cudaError_t launch_hm(const SweepParams& p, int lam, cudaStream_t s) {
    switch (lam) {
        case 2: return launch_t<G, 2, IND, false, HM>(p, s);
        case 4: return launch_t<G, 4, IND, false, HM>(p, s);
        case 8: return launch_t<G, 8, IND, false, HM>(p, s);
        case 16:
            if constexpr (G == 32)
                if (!few_units(p)) return launch_t<G, 16, IND, false, HM, false>(p, s);
            return launch_t<G, 16, IND, false, HM>(p, s);
        case 32: return launch_t<G, 32, IND, false, HM>(p, s);
        default: return cudaErrorNotSupported;
    }
}

template <int G, bool IND>
static cudaError_t launch_g_hm(const SweepParams& p, int lam, cudaStream_t s) {
    switch (head_pattern(p)) {
        case 1: return launch_hm<G, IND, 1>(p, lam, s);
        case 2: return launch_hm<G, IND, 2>(p, lam, s);
        case 3: return launch_hm<G, IND, 3>(p, lam, s);
        case 4: return launch_hm<G, IND, 4>(p, lam, s);
        default: return cudaErrorNotSupported;
    }
}

template <bool IND>
static cudaError_t launch_modes_32(const SweepParams& p, int lam, cudaStream_t s) {
    return p.accepts || p.C % 32 ? cudaErrorNotSupported : launch_g_hm<32, IND>(p, lam, s);
}

template <bool IND>
static cudaError_t launch_modes_16(const SweepParams& p, int lam, cudaStream_t s) {
    return p.accepts ? cudaErrorNotSupported : launch_g_hm<16, IND>(p, lam, s);
}

template <bool IND>
static cudaError_t launch_modes_narrow_planes(const SweepParams& p, int lam, cudaStream_t s) {
    if (p.accepts) return cudaErrorNotSupported;
    return p.G == 8 ? launch_g_hm<8, IND>(p, lam, s) : launch_g_hm<4, IND>(p, lam, s);
}

}  // namespace surfmcmc
