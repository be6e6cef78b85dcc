// Random scan (Sec. IV as written): each step of a chain draws one generator
// and applies it when Delta n <= 0 or u < T[Delta n].
//
// A chain is serial and each touches other generators, so nothing is
// bit-sliced here: a lane runs one chain on its own copy of the frame, one
// 32-bit word per grid row and plane, kept at [row][lane] in shared memory.
// Every access of a warp then falls on 32 different banks, no other lane's
// words are written (no atomics, no synchronisation in a sweep), and the four
// qubits of a generator are one bit of the row above, two of its own row and
// one of the row below: three words of each plane.  Their eight bits index a
// table of (threshold, Delta n) for the generator's shape, built per block
// from the energies and T, which replaces the per-qubit energy arithmetic.
//
// Bound: instruction issue and the serial chain of a step (words -> table ->
// words).  The Philox blocks of four steps are drawn together ahead of them;
// the rounds that only see the syndrome, chain and sweep are computed once
// per sweep (three of the eight products of rounds 0-2 remain), and the words
// not used fall away in the last two.
//
// Measured (GB300, L = 9, 4,096 syndromes x 16 chains, 200 sweeps): 24.5 ms on
// the bit-sliced frames this replaced (8 loads and 4 atomics per step on
// random banks, the energy of each qubit by selects), 10.1 ms here (10.9 before
// the planar code took its two middle bits together).
#include <algorithm>

#include "sweep_kernel.cuh"

namespace surfmcmc {

namespace {

constexpr int kScanWarps = 2;         // bundles per block: 2048 bundles spread evenly over 152 SMs
constexpr int kShapes = 3;            // all four qubits; without the first / the second of a pair
constexpr int kMoves = 2 * kShapes * 256;

// Grid rows kept per plane, with a row of padding above and below (the
// planar code's missing neighbours).
__host__ __device__ __forceinline__ int scan_rows(int code, int L) { return (code ? 2 * L : 2 * L - 1) + 2; }

__host__ __device__ inline size_t scan_smem_bytes(int code, int L) {
    return (size_t)kMoves * 8 + (size_t)geo_nstab(code, L) * 4 + (size_t)kScanWarps * 2 * scan_rows(code, L) * 128;
}

// Grid row (with the padding) and bit of qubit q in that row's word.  Planar:
// even rows hold columns 2 bit, odd rows columns 2 bit - 1, so that a
// sigma_x generator's left and right neighbours are bits j and j + 1 there as
// well (bits 0 and L of an odd row stand for the missing ones).
__device__ __forceinline__ void scan_place(int code, int L, int q, int& row, int& bit) {
    if (code) {
        row = q / L + 1;
        bit = q - (row - 1) * L;
    } else {
        const int pair = q / (2 * L - 1), k = q - pair * (2 * L - 1);
        row = 2 * pair + (k >= L) + 1;
        bit = k >= L ? k - L + 1 : k;
    }
}

// Generator g of the syndrome order, packed: bl (bits 0-4) and br (25-29) the
// bits of its left and right qubit, bit 5 set when the upper and lower qubit
// have bit br (else bl), the rows M, U, D of its own, the upper and the lower
// qubits at bits 7, 13 and 19 (so that row * 128 bytes is a mask away), the
// shape at bits 30-31.
__device__ __forceinline__ uint32_t scan_generator(int code, int L, int g, int n_x) {
    const int type = g >= n_x, h = type ? g - n_x : g;
    int M, U, D, bl, br, bu, shape = 0;
    if (code) {
        const int i = h / L, j = h - i * L, r = 2 * i + type, rows = 2 * L;
        M = r + 1;
        U = (r + rows - 1) % rows + 1;
        D = (r + 1) % rows + 1;
        bl = type ? j : (j + L - 1) % L;
        br = type ? (j + 1) % L : j;
        bu = j;
    } else if (type == 0) {
        const int i = h / L, j = h - i * L;
        M = 2 * i + 2;
        U = M - 1;
        D = M + 1;
        bl = j;
        br = j + 1;
        bu = j;
        shape = j == 0 ? 1 : j == L - 1 ? 2 : 0;
    } else {
        const int i = h / (L - 1), j = h - i * (L - 1);
        M = 2 * i + 1;
        U = M - 1;
        D = M + 1;
        bl = j;
        br = j + 1;
        bu = j + 1;
        shape = i == 0 ? 1 : i == L - 1 ? 2 : 0;
    }
    return (uint32_t)bl | (uint32_t)(bu == br && bu != bl) << 5 | (uint32_t)M << 7 | (uint32_t)U << 13 |
           (uint32_t)D << 19 | (uint32_t)br << 25 | (uint32_t)shape << 30;
}

// Move table entry: Delta n of flipping the generator's plane for the bits
// idx = own l, r, u, d (bits 0-3) and other l, r, u, d (bits 4-7), and the
// threshold its uniform is compared with: (T, 2 Delta n + 1) accepts always.
__device__ __forceinline__ uint2 scan_move(const SweepParams& p, int type, int shape, int idx) {
    int dn = 0;
    for (int k = 0; k < 4; ++k) {
        // sigma_x: the left (shape 1) or right qubit is missing, sigma_z: the upper or lower
        if (shape == 1 && k == 2 * type) continue;
        if (shape == 2 && k == 2 * type + 1) continue;
        const int o = (idx >> k) & 1, t = (idx >> (4 + k)) & 1;
        const int a = type == 0 ? o + 2 * t : t + 2 * o, b = type == 0 ? (o ^ 1) + 2 * t : t + 2 * (o ^ 1);
        dn += p.energy[b] - p.energy[a];
    }
    const bool always = dn <= 0 || p.T[dn] >= 4294967296ull;
    return make_uint2(always ? 0u : (uint32_t)p.T[dn], (uint32_t)(2 * dn) | (always ? 1u : 0u));
}

// v >> (s mod 32)
__device__ __forceinline__ uint32_t shr(uint32_t v, uint32_t s) { return v >> (s & 31u); }

// Words 0 and 1 of Philox4x32-10 for the counters (id, chain, t, step) of one
// sweep: the rounds' parts that do not depend on the step.
struct ScanPhilox {
    uint32_t z1, x2, z3, w2, h2, y3;

    __device__ __forceinline__ ScanPhilox(uint32_t id, uint32_t chain, uint32_t t, const RoundKeys& rk) {
        z1 = __umulhi(kPhiloxMa, id) ^ rk.k[1];                                      // ^ step
        const uint32_t x1 = __umulhi(kPhiloxMb, t) ^ chain ^ rk.k[0], y1 = kPhiloxMb * t, w1 = kPhiloxMa * id;
        x2 = y1 ^ rk.k[2];                                                           // ^ hi(Mb z1)
        const uint32_t z2 = __umulhi(kPhiloxMa, x1) ^ w1 ^ rk.k[3];
        w2 = kPhiloxMa * x1;
        h2 = __umulhi(kPhiloxMb, z2) ^ rk.k[4];                                      // ^ y2: x3
        y3 = kPhiloxMb * z2;
        z3 = w2 ^ rk.k[5];                                                           // ^ hi(Ma x2)
    }
    __device__ __forceinline__ uint2 draw(uint32_t step, const RoundKeys& rk) const {
        const uint32_t z = z1 ^ step;
        const uint32_t x = __umulhi(kPhiloxMb, z) ^ x2, y2 = kPhiloxMb * z;          // state after round 1
        const uint4 r = philox_rounds<3>(make_uint4(h2 ^ y2, y3, __umulhi(kPhiloxMa, x) ^ z3, kPhiloxMa * x), rk);
        return make_uint2(r.x, r.y);
    }
};

template <int G, bool TORIC>
__global__ void __launch_bounds__(32 * kScanWarps) scan_kernel(const __grid_constant__ SweepParams p) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long unit = blockIdx.x;
    int gi = 0;
    auto units = [&](int g) { return (p.grp[g].n_bundles + kScanWarps - 1) / kScanWarps; };
    while (gi + 1 < p.n_groups && unit >= units(gi)) unit -= units(gi++);
    const GroupDesc& gd = p.grp[gi];
    const int L = gd.L, nq = gd.nq, W = gd.W, ns = geo_nstab(p.code, L);
    const int n_x = p.code ? L * L : L * (L - 1);   // sigma_x generators come first
    const int rows = scan_rows(p.code, L);

    uint2* moves = reinterpret_cast<uint2*>(smem);
    uint32_t* gens = smem + 2 * kMoves;
    uint32_t* X = gens + ns + (size_t)warp * 2 * rows * 32;     // [row][lane]
    uint32_t* Z = X + rows * 32;
    for (int i = threadIdx.x; i < kMoves; i += blockDim.x)
        moves[i] = scan_move(p, i / (kShapes * 256), (i / 256) % kShapes, i & 255);
    for (int g = threadIdx.x; g < ns; g += blockDim.x) gens[g] = scan_generator(p.code, L, g, n_x);

    const BundleMap<G> bm(p, gd, unit * kScanWarps + warp);
    const bool mine = (bm.valid >> lane) & 1u;
    const size_t ci = (size_t)bm.syn_of(lane) * p.C + bm.chain_of(lane);   // (bits outside valid: not used)

    // Start state: 32 qubits' words at a time, transposed to the lanes' rows.
    for (int i = 0; i < 2 * rows; ++i) X[i * 32 + lane] = 0u;
    {
        const StartState<G> start(p, gd, bm);
        for (int q0 = 0; q0 < nq; q0 += 32) {
            uint32_t xw = 0, zw = 0;
            if (q0 + lane < nq) start.word(q0 + lane, xw, zw);
            const int k = nq - q0 < 32 ? nq - q0 : 32;
            for (int i = 0; i < k; ++i) {
                int row, bit;
                scan_place(p.code, L, q0 + i, row, bit);
                const uint32_t x = __shfl_sync(0xffffffffu, xw, i), z = __shfl_sync(0xffffffffu, zw, i);
                X[row * 32 + lane] |= ((x >> lane) & 1u) << bit;
                Z[row * 32 + lane] |= ((z >> lane) & 1u) << bit;
            }
        }
    }
    __syncthreads();

    auto qubit = [&](int q, uint32_t& x, uint32_t& z) {
        int row, bit;
        scan_place(p.code, L, q, row, bit);
        x = (X[row * 32 + lane] >> bit) & 1u;
        z = (Z[row * 32 + lane] >> bit) & 1u;
    };
    int n = 0;
    for (int q = 0; q < nq; ++q) {
        uint32_t x, z;
        qubit(q, x, z);
        n += p.energy[x + 2 * z];
    }

    uint64_t sum = 0, n_acc = 0;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(X) + 4u * lane, plane = 128u * (uint32_t)rows;
    const uint32_t my_sid = bm.sid[G == 32 ? 0 : lane / G], chain = (uint32_t)bm.chain_of(lane);
    constexpr int U = 4;    // steps drawn together; n_stab is a multiple of 4 for either code
    for (uint32_t t = gd.t_begin; t < gd.t_end; ++t) {
        const ScanPhilox ph(my_sid, chain, t, p.rk);
        uint32_t sweep_sum = 0, accepted = 0;   // n <= 8 n_q < 2^14, n_stab < 2^11
        for (int s0 = 0; s0 < ns; s0 += U) {
            uint32_t e[U], u[U], tbl[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint2 r = ph.draw((uint32_t)(s0 + k), p.rk);
                const int g = (int)__umulhi(r.x, (uint32_t)ns);
                e[k] = gens[g];
                u[k] = r.y;
                // table of the generator's type and shape; the type's plane in bit 31
                tbl[k] = (g >= n_x ? 0x80000000u + kShapes * 256u : 0u) + (e[k] >> 30) * 256u;
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint32_t own = base + ((int)tbl[k] < 0 ? plane : 0u), oth = base + ((int)tbl[k] < 0 ? 0u : plane);
                const uint32_t rm = e[k] & 0x1F80u, ru = (e[k] >> 6) & 0x1F80u, rd = (e[k] >> 12) & 0x1F80u;
                const uint32_t bl = e[k], br = e[k] >> 25;   // (shifts take the low 5 bits)
                const uint32_t bu = TORIC ? (e[k] & 32u ? br : bl) : bl + ((e[k] >> 5) & 1u);
                auto ld = [](uint32_t a) {
                    uint32_t v;
                    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
                    return v;
                };
                auto st = [](uint32_t a, uint32_t v) {
                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
                };
                const uint32_t om = ld(own + rm), ou = ld(own + ru), od = ld(own + rd);
                const uint32_t tm = ld(oth + rm), tu = ld(oth + ru), td = ld(oth + rd);
                // own l, r, u, d in bits 0-3, other l, r, u, d in bits 4-7; the
                // planar code's r is the bit after l
                uint32_t o, x;
                if (TORIC) {
                    o = (shr(om, bl) & 1u) + 2u * (shr(om, br) & 1u);
                    x = (shr(tm, bl) & 1u) + 2u * (shr(tm, br) & 1u);
                } else {
                    o = shr(om, bl) & 3u;
                    x = shr(tm, bl) & 3u;
                }
                o += 4u * (shr(ou, bu) & 1u);
                x += 4u * (shr(tu, bu) & 1u);
                o += 8u * (shr(od, bu) & 1u);
                x += 8u * (shr(td, bu) & 1u);
                const uint32_t idx = o + 16u * x;
                const uint2 mv = moves[(tbl[k] & 0x7FFFFFFFu) + idx];
                if (u[k] < mv.x || (mv.y & 1u)) {
                    const uint32_t up = 1u << (bu & 31u);
                    st(own + rm, om ^ (TORIC ? 1u << (bl & 31u) ^ 1u << (br & 31u) : 3u << (bl & 31u)));
                    st(own + ru, ou ^ up);
                    st(own + rd, od ^ up);
                    n += (int)mv.y >> 1;
                    ++accepted;
                }
                sweep_sum += (uint32_t)n;
            }
        }
        if (t >= gd.burn_in) sum += sweep_sum;
        n_acc += accepted;
    }

    if (mine) {
        if (p.chain_sum) p.chain_sum[ci] = (p.init_sum ? p.init_sum[ci] : 0ull) + sum;
        if (p.accepts) p.accepts[ci] += n_acc;   // one lane per chain
        if (p.chain_n) p.chain_n[ci] = n;
        if (p.chain_frames) {
            uint32_t* f = p.chain_frames + gd.frames_off - (size_t)gd.item_base * p.C * 2 * W + ci * 2 * W;
            for (int wi = 0; wi < W; ++wi) {
                uint32_t xw = 0, zw = 0;
                for (int i = 0; i < 32 && 32 * wi + i < nq; ++i) {
                    uint32_t x, z;
                    qubit(32 * wi + i, x, z);
                    xw |= x << i;
                    zw |= z << i;
                }
                f[wi] = xw;
                f[W + wi] = zw;
            }
        }
    }
    if (p.state_out && bm.active) {
        uint32_t* st = p.state_out + gd.state_off + (size_t)bm.bid * 2 * nq;
        for (int q = 0; q < nq; ++q) {
            uint32_t x, z;
            qubit(q, x, z);
            const uint32_t xw = __ballot_sync(0xffffffffu, x), zw = __ballot_sync(0xffffffffu, z);
            if (lane == (q & 31)) {
                st[q] = xw;
                st[nq + q] = zw;
            }
        }
    }
}

template <int G, bool TORIC>
cudaError_t launch_scan_t(const SweepParams& p, cudaStream_t s) {
    long long blocks = 0;
    size_t smem = 0;
    for (int g = 0; g < p.n_groups; ++g) {
        blocks += (p.grp[g].n_bundles + kScanWarps - 1) / kScanWarps;
        smem = std::max(smem, scan_smem_bytes(p.code, p.grp[g].L));
    }
    if (blocks == 0) return cudaSuccess;
    static SmemLimit limit;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && smem > 48 * 1024) e = limit.ensure(scan_kernel<G, TORIC>, dev, smem);
    if (e != cudaSuccess) return e;
    scan_kernel<G, TORIC><<<(unsigned)blocks, 32 * kScanWarps, smem, s>>>(p);
    return cudaGetLastError();
}

template <int G>
cudaError_t launch_scan_g(const SweepParams& p, cudaStream_t s) {
    return p.code ? launch_scan_t<G, true>(p, s) : launch_scan_t<G, false>(p, s);
}

}  // namespace

cudaError_t launch_sweep_scan(const SweepParams& p, cudaStream_t s) {
    switch (p.G) {
        case 4: return launch_scan_g<4>(p, s);
        case 8: return launch_scan_g<8>(p, s);
        case 16: return launch_scan_g<16>(p, s);
        case 32: return launch_scan_g<32>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace surfmcmc
