// The colour sweep for batches too small to fill the device: one block per
// 32-chain bundle, with the random part of every proposal taken off the
// chains' serial path.
//
// What bounds a small batch is latency: a sweep is four dependent colour
// phases, and on the throughput kernel (sweep_kernel.cuh) a phase of one
// warp's bundle is ceil(generators / lanes) proposals one after the other,
// each a chain of shared-memory loads, classification, Philox rounds and
// digit comparisons, then the straggler queue.  Nothing of the Philox and
// comparison part depends on the chains' state, so here
//   * the block is 2 to 12 sets of warps, set s taking the phases s, s +
//     sets, ...; a thread owns one generator of its phase;
//   * while the other sets run their phases a thread computes, for its next
//     proposal, the accept masks of all four uphill steps: bit b of lt[d-1]
//     is u_b < T[d] for chain b (digit planes as in the throughput kernel,
//     drawn until no chain's comparison is open for any d);
//   * the state-dependent rest of a phase is one barrier, 8 loads, ~20
//     logic operations, 4 stores.
// The phases stay strictly in order (named barriers from set to set), so the
// results are the throughput kernel's bit for bit.  A proposal costs more
// instructions here (every d is compared, not the one that applies), which
// is why full batches keep the throughput kernel.
//
// After 8 planes a fifth of the proposals have an open comparison for some
// chain and some d.  In sets of more than one warp those are pooled in
// shared memory and finished packed, by one warp in three instead of all.
//
// n is sampled on the way in: same-colour generators cover every qubit
// once (but L boundary qubits of the planar code, which extra threads load
// without proposing), so the words a phase loads are the state after the
// phase before; a thread adds its unoccupied words to a bit-sliced counter
// after its stores, off the serial path.
//
// Measured (GB300, 4 x 4 chains): a 60-sweep decode with 1, 2 and 4 bundles per
// multiprocessor takes 144, 231, 394 us at L = 13 against 524-531 on the
// throughput kernel's best split, and 322, 638, 1212 against 1270 at L = 25; at
// 8 per multiprocessor the throughput kernel is as fast or faster at every
// size, hence the limit in wide_batch (plan.cuh).
#include <algorithm>

#include "sweep_kernel.cuh"

namespace surfmcmc {

namespace {

constexpr int kWideMaxThreads = 1024;
// Sets of a block, at most: their barriers have ids 1 .. 12, or with pooled
// stragglers (two per set) 1 .. 14.
constexpr int kWideMaxSets = 12, kWideMaxPoolSets = 7;
constexpr int kWidePlanes = 12;                       // bit planes of a thread's counter
constexpr int kWideFlushPlanes = kWidePlanes + 5;     // summed over a warp

// Phase slots: the colour's generators and, for the planar code, the L
// qubits it does not touch, four to a slot.
__host__ __device__ __forceinline__ int wide_slots(int code, int L) {
    return geo_nc(code, L) + (code ? 0 : (L + 3) / 4);
}
__host__ __device__ __forceinline__ int wide_set_threads(int code, int L) {
    return (wide_slots(code, L) + 31) / 32 * 32;
}
// Sets of a block of at most `budget` threads (at least two).
__host__ __device__ __forceinline__ int wide_sets(int code, int L, int budget) {
    const int ts = wide_set_threads(code, L), ns = budget / ts, most = ts > 32 ? kWideMaxPoolSets : kWideMaxSets;
    return ns < 2 ? 2 : ns > most ? most : ns;
}
static_assert(2 * ((465 + 8 + 31) / 32 * 32) <= kWideMaxThreads, "two sets hold the largest code");

// k-th qubit (k < L) that no generator of planar colour col touches: on the
// first and last row (sigma_x) or column (sigma_z) every other qubit.
__device__ __forceinline__ int untouched_qubit(int L, int col, int k) {
    const int par = col & 1, f0 = 1 - par, f1 = (par + 1 + L) & 1, c0 = (L - f0 + 1) / 2;
    const bool first = k < c0;
    const int j = first ? f0 + 2 * k : f1 + 2 * (k - c0);
    if (col < 2) return first ? j : (L - 1) * (2 * L - 1) + j;
    return j * (2 * L - 1) + (first ? 0 : L - 1);
}

// Batches with kept fixed Philox parts (16 planes; all 32 with G = 4), and
// those every proposal draws (8 planes; 16 and 32 with G = 8 and 4).
template <int G>
constexpr int wide_fixed() { return G == 32 ? 4 : G == 16 ? 2 : 1; }
template <int G>
constexpr int wide_head() { return G == 32 ? 2 : 1; }

// Shared memory of a block, in words: fixed Philox parts, per set the accept
// masks and the straggler pool (with more than one warp), the support table,
// the frames, the final counts and the pools' counters.
__host__ __device__ inline size_t wide_smem_words(int nq, int set_threads, int sets, int fixed_blocks) {
    return 4 * (size_t)fixed_blocks + (set_threads > 32 ? 8 * (size_t)set_threads * sets : 0) + 8 * (size_t)set_threads +
           2 * (size_t)(nq + 2) + 32 + 2 * kWideMaxPoolSets + (set_threads > 32 ? (size_t)set_threads * sets : 0);
}

// Digits 4q .. 4q+3 of the comparison u < T[d]: lt gains the chains decided
// as less, eq keeps the undecided ones.  The digits are taken from the least
// significant, one operation each for "less" and "equal".
__device__ __forceinline__ void compare_digits(const uint32_t c[4], const uint32_t r[4], uint32_t& lt, uint32_t& eq) {
    uint32_t l = c[3] & ~r[3], e = ~(c[3] ^ r[3]);
#pragma unroll
    for (int i = 2; i >= 0; --i) {
        l = (c[i] & ~r[i]) | (~(c[i] ^ r[i]) & l);
        e &= ~(c[i] ^ r[i]);
    }
    lt |= eq & l;
    eq &= e;
}

// The same for d = 1..4 (index d - 1); thresholds without nonzero digits in
// the quad reject at any 1 digit.
__device__ __forceinline__ void compare_quad(const SweepParams& p, int q, const uint32_t r[4], uint32_t lt[4],
                                             uint32_t eq[4]) {
    const uint32_t mode = (p.qmodes >> (2 * q)) & 3u;
    if (mode >= 2) {
#pragma unroll
        for (int d = 0; d < 4; ++d) compare_digits(p.tb[d] + 4 * q, r, lt[d], eq[d]);
    } else {
        const uint32_t zero = ~(r[0] | r[1] | r[2] | r[3]);
        if (mode == 1) compare_digits(p.tb[0] + 4 * q, r, lt[0], eq[0]);
        else eq[0] &= zero;
        eq[1] &= zero;
        eq[2] &= zero;
        eq[3] &= zero;
    }
}

// Accept masks lt[d-1] of one proposal for every uphill step d = 1..4 from
// the batches [BT0, BT1) whose fixed Philox parts are kept; eq[d-1]: the
// chains still undecided.
template <int G, int BT0, int BT1>
__device__ __forceinline__ void accept_masks(const SweepParams& p, const uint4* fixed, uint32_t t, uint32_t colm,
                                             uint32_t lt[4], uint32_t eq[4]) {
    using PB = PlaneBatch<G>;
    constexpr int SLOTS = PB::SLOTS, PPB = PB::PPB;
    const PhiloxVarying pv = philox_varying(t, colm, p.rk);
#pragma unroll
    for (int bt = BT0; bt < BT1; ++bt) {
        uint4 b[SLOTS];
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) {
            const uint4 f = fixed[bt * SLOTS + s];
            b[s] = philox10_split(f.x, f.y, f.z, pv, p.rk);
        }
        PB pb;
        pb.merge(b);
#pragma unroll
        for (int qd = 0; qd < PPB / 4; ++qd) compare_quad(p, (bt * PPB) / 4 + qd, pb.pl + 4 * qd, lt, eq);
    }
}

// The rest of an undecided proposal's comparisons.
template <int G>
__device__ __forceinline__ void accept_masks_rest(const SweepParams& p, const uint4* fixed, const BundleMap<G>& bm,
                                                  uint32_t t, uint32_t colm, uint32_t lt[4], uint32_t eq[4]) {
    using PB = PlaneBatch<G>;
    constexpr int PPB = PB::PPB, HEAD = wide_head<G>(), FIXED = wide_fixed<G>();
    if constexpr (HEAD < FIXED) accept_masks<G, HEAD, FIXED>(p, fixed, t, colm, lt, eq);
    if constexpr (FIXED * PPB < 32) {
#pragma unroll 1
        for (int bt = FIXED; bt * PPB < 32 && (eq[0] | eq[1] | eq[2] | eq[3]); ++bt) {
            PB pb;
            pb.make(p, bm.sid, bm.w, t, colm, (uint32_t)bt);
#pragma unroll
            for (int qd = 0; qd < PPB / 4; ++qd) compare_quad(p, (bt * PPB) / 4 + qd, pb.pl + 4 * qd, lt, eq);
        }
    }
}

// Named barrier `id` over `threads` threads: waiting at it, or arriving only.
__device__ __forceinline__ void bar_wait(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ uint32_t lds(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Adds the bit-sliced number (n0, n1, n2) to the counter.
__device__ __forceinline__ void count_add(uint32_t v[kWidePlanes], uint32_t n0, uint32_t n1, uint32_t n2) {
    uint32_t c = v[0] & n0;
    v[0] ^= n0;
    csa(c, v[1], v[1], n1, c);
    csa(c, v[2], v[2], n2, c);
#pragma unroll
    for (int k = 3; k < kWidePlanes; ++k) {
        if (k >= 5 && !c) break;
        const uint32_t o = v[k] & c;
        v[k] ^= c;
        c = o;
    }
}

// Sum of four one-bit numbers as three planes.
__device__ __forceinline__ void sum4(uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t& n0, uint32_t& n1,
                                     uint32_t& n2) {
    uint32_t h, l;
    csa(h, l, a, b, c);
    n0 = l ^ d;
    const uint32_t k = l & d;
    n1 = h ^ k;
    n2 = h & k;
}

// The counter of chain `lane`, summed over the warp's lanes; clears it.
__device__ __forceinline__ uint32_t count_flush(uint32_t v[kWidePlanes], int lane) {
    uint32_t s[kWideFlushPlanes];
#pragma unroll
    for (int k = 0; k < kWideFlushPlanes; ++k) s[k] = k < kWidePlanes ? v[k] : 0u;
#pragma unroll
    for (int k = 0; k < kWidePlanes; ++k) v[k] = 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        uint32_t c = 0;
#pragma unroll
        for (int k = 0; k < kWideFlushPlanes; ++k) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, s[k], off);
            csa(c, s[k], s[k], o, c);
        }
    }
    uint32_t n = 0;
#pragma unroll
    for (int k = 0; k < kWideFlushPlanes; ++k) n |= ((s[k] >> lane) & 1u) << k;
    return n;
}

// Word of qubit q in a plane: even qubits first, then odd ones.  Same-colour
// generators of a row are two qubits apart, so their words lie on 32
// different banks instead of 16 (a burst of 512 requests of L = 9 .. 25: 6.08
// -> 5.87 ms, one syndrome at L = 13: 324 -> 320 us).
__device__ __forceinline__ int word_of(int q, int nq) { return (q >> 1) + (q & 1 ? (nq + 1) >> 1 : 0); }

template <int G, bool IND>
__global__ void __launch_bounds__(kWideMaxThreads, 1) wide_kernel(const __grid_constant__ SweepParams p) {
    constexpr int SLOTS = PlaneBatch<G>::SLOTS, FIXED = wide_fixed<G>();
    extern __shared__ __align__(16) uint32_t smem[];
    long long bid = blockIdx.x;
    int gi = 0;
    while (gi + 1 < p.n_groups && bid >= p.grp[gi].n_bundles) bid -= p.grp[gi++].n_bundles;
    const GroupDesc& gd = p.grp[gi];
    const int L = gd.L, nq = gd.nq, nc = gd.nc, W = gd.W;
    const int TS = wide_set_threads(p.code, L), NS = wide_sets(p.code, L, p.wide);
    const int tid = threadIdx.x, lane = tid & 31, nt = blockDim.x;

    // stragglers of a phase are pooled over the set's warps (see below)
    const bool pooled = TS > 32;
    const int set = tid / TS, m = tid - set * TS;
    uint4* fixed = reinterpret_cast<uint4*>(smem);                    // head blocks' fixed Philox parts
    uint4* masks = fixed + FIXED * SLOTS;                             // [NS][TS] accept masks (pooled)
    uint4* pool_eq = masks + (pooled ? NS * TS : 0);                  // [NS][TS] undecided chains per d
    ushort4* tab = reinterpret_cast<ushort4*>(pool_eq + (pooled ? NS * TS : 0));  // [4][TS] word indices
    uint32_t* X = reinterpret_cast<uint32_t*>(tab + 4 * TS);
    uint32_t* Z = X + nq + 2;
    uint32_t* left = Z + nq + 2;                                      // [32] unoccupied at the end, per chain
    uint32_t* pool_n = left + 32;                                     // [2][sets] pool sizes
    uint32_t* pool_m = pool_n + 2 * kWideMaxPoolSets;                 // [NS][TS] the pooled generators

    const BundleMap<G> bm(p, gd, bid);
    const uint32_t valid = bm.valid;
    auto ci_of = [&](int b) -> size_t { return (size_t)bm.syn_of(b) * p.C + bm.chain_of(b); };

    if (tid < 2 * kWideMaxPoolSets) pool_n[tid] = 0u;
    if (tid < FIXED * SLOTS) {
        const int bt = tid / SLOTS, s = tid % SLOTS;
        uint32_t id = bm.sid[0];
#pragma unroll
        for (int i = 1; i < SLOTS; ++i)
            if (i == s) id = bm.sid[i];
        const PhiloxFixed f = philox_fixed(id, G == 32 ? (bm.w << 8) | (uint32_t)bt : (uint32_t)bt, p.rk);
        fixed[tid] = make_uint4(f.M, f.N, f.A, 0u);
    }
    for (int idx = tid; idx < 4 * TS; idx += nt) {
        const int col = idx / TS, m = idx - col * TS;
        const int dummy = col < 2 ? nq : nq + 1;
        int q[4] = {dummy, dummy, dummy, dummy};
        if (m < nc) {
            if (p.code) toric_colour_support(L, col, m, q);
            else colour_support(L, col, m, q);
        } else if (!p.code) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (4 * (m - nc) + k < L) q[k] = untouched_qubit(L, col, 4 * (m - nc) + k);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (q[k] < nq) q[k] = word_of(q[k], nq);      // (the dummies stay behind the planes)
        tab[idx] = make_ushort4((unsigned short)q[0], (unsigned short)q[1], (unsigned short)q[2],
                                (unsigned short)q[3]);
    }
    {
        const StartState<G> start(p, gd, bm);
        for (int q = tid; q < nq; q += nt) {
            uint32_t xw, zw;
            start.word(q, xw, zw);
            X[word_of(q, nq)] = xw;
            Z[word_of(q, nq)] = zw;
        }
    }
    // samples: the states after the phases of sweeps first .. t_end - 1
    const uint32_t first = gd.burn_in > gd.t_begin ? gd.burn_in : gd.t_begin;
    const uint64_t n_samples = gd.t_end > first ? 4ull * (gd.t_end - first) : 0ull;
    if (tid < 32) {
        if (tid == 0) {
            X[nq] = 0u; Z[nq] = 0xFFFFFFFFu;          // dummy of sigma_x generators
            X[nq + 1] = 0xFFFFFFFFu; Z[nq + 1] = 0u;  // dummy of sigma_z generators
        }
        left[tid] = 0u;
        if (p.chain_sum && ((valid >> tid) & 1u)) {
            // every position counted as occupied; the counters below take the
            // unoccupied ones off
            const size_t ci = ci_of(tid);
            p.chain_sum[ci] = (p.init_sum ? p.init_sum[ci] : 0ull) + n_samples * (uint64_t)((IND ? 2 : 1) * nq);
        }
    }
    __syncthreads();

    uint32_t v[kWidePlanes];
#pragma unroll
    for (int k = 0; k < kWidePlanes; ++k) v[k] = 0;
    auto credit = [&]() {
        const uint32_t n = count_flush(v, lane);
        if (p.chain_sum && ((valid >> lane) & 1u))
            atomicAdd(reinterpret_cast<unsigned long long*>(p.chain_sum + ci_of(lane)), 0ull - (unsigned long long)n);
    };
    if (set < NS && (uint64_t)gd.t_begin + (uint32_t)(set >> 2) < gd.t_end) {
        constexpr uint32_t kPer = IND ? 8 : 4;                        // counts per phase and thread
        constexpr uint32_t kFlushEvery = ((1u << kWidePlanes) - 1u) / kPer;
        const uint32_t flips = m < nc ? valid : 0u;
        uint32_t t = gd.t_begin + (uint32_t)(set >> 2), since = 0;
        int col = set & 3, turn = 0;
        const uint32_t x_addr = (uint32_t)__cvta_generic_to_shared(X), z_step = 4u * (uint32_t)(nq + 2);
        while (true) {
            // state-independent part of this thread's proposal
            const uint32_t colm = ((uint32_t)col << 24) | (uint32_t)m;
            // shared-memory addresses of the support's words: the plane the
            // generator flips, and the other
            const ushort4 sp = tab[col * TS + m];
            uint32_t ow[4] = {x_addr + 4u * sp.x, x_addr + 4u * sp.y, x_addr + 4u * sp.z, x_addr + 4u * sp.w}, ot[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                ot[k] = ow[k] + (col < 2 ? z_step : 0u);
                ow[k] += col < 2 ? 0u : z_step;
            }
            const bool begin = t == gd.t_begin && col == 0;
            const bool end = t + 1 == gd.t_end && col == 3;
            uint32_t lt[4], eq[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                lt[d] = p.accept_all ? ~0u : 0u;
                eq[d] = valid;
            }
            if (!(p.accept_all || p.reject_all)) {
                accept_masks<G, 0, wide_head<G>()>(p, fixed, t, colm, lt, eq);
                const bool open = m < nc && (eq[0] | eq[1] | eq[2] | eq[3]) != 0u;
                if (!pooled) {
                    if (open) accept_masks_rest<G>(p, fixed, bm, t, colm, lt, eq);
                } else {
                    // about a fifth of the proposals have an open comparison:
                    // the set's threads finish them packed into few warps
                    masks[tid] = make_uint4(lt[0], lt[1], lt[2], lt[3]);
                    if (open) {
                        const uint32_t i = atomicAdd(&pool_n[kWideMaxPoolSets * turn + set], 1u);
                        pool_eq[set * TS + i] = make_uint4(eq[0], eq[1], eq[2], eq[3]);
                        pool_m[set * TS + i] = (uint32_t)m;
                    }
                    __syncwarp();
                    bar_wait(1 + NS + set, TS);
                    if (m < (int)pool_n[kWideMaxPoolSets * turn + set]) {
                        const uint32_t pm = pool_m[tid];
                        const uint4 e = pool_eq[tid], l = masks[set * TS + pm];
                        uint32_t le[4] = {l.x, l.y, l.z, l.w}, qe[4] = {e.x, e.y, e.z, e.w};
                        accept_masks_rest<G>(p, fixed, bm, t, ((uint32_t)col << 24) | pm, le, qe);
                        masks[set * TS + pm] = make_uint4(le[0], le[1], le[2], le[3]);
                    }
                    turn ^= 1;
                    if (m == 0) pool_n[kWideMaxPoolSets * turn + set] = 0u;   // the next phase's
                }
            }
            // keep the masks and addresses ahead of the wait (the compiler would
            // move them to their use, onto the serial path)
            asm volatile("" : "+r"(lt[0]), "+r"(lt[1]), "+r"(lt[2]), "+r"(lt[3]));
            asm volatile("" : "+r"(ow[0]), "+r"(ow[1]), "+r"(ow[2]), "+r"(ow[3]), "+r"(ot[0]), "+r"(ot[1]),
                         "+r"(ot[2]), "+r"(ot[3]));
            __syncwarp();
            if (!begin) bar_wait(1 + set, 2 * TS);    // the phase before (and the set's pool) is done
            else if (pooled) bar_wait(1 + NS + set, TS);
            if (pooled && !(p.accept_all || p.reject_all)) {
                const uint4 l = masks[tid];
                lt[0] = l.x; lt[1] = l.y; lt[2] = l.z; lt[3] = l.w;
            }
            const uint32_t o0 = lds(ow[0]), o1 = lds(ow[1]), o2 = lds(ow[2]), o3 = lds(ow[3]);
            const uint32_t t0 = lds(ot[0]), t1 = lds(ot[1]), t2 = lds(ot[2]), t3 = lds(ot[3]);
            // movable qubits, W their number, D the movable errors removed (see run_unit)
            const uint32_t m0 = IND ? (sp.x < nq ? ~0u : 0u) : ~t0;
            const uint32_t m1 = IND ? (sp.y < nq ? ~0u : 0u) : ~t1;
            const uint32_t m2 = IND ? (sp.z < nq ? ~0u : 0u) : ~t2;
            const uint32_t m3 = IND ? (sp.w < nq ? ~0u : 0u) : ~t3;
            uint32_t w0, w1, w2;
            sum4(m0, m1, m2, m3, w0, w1, w2);
            const uint32_t d0 = m0 & o0, d1 = m1 & o1, d2 = m2 & o2, d3 = m3 & o3;
            const uint32_t ds = d0 ^ d1 ^ d2, dc = (d0 & d1) | (d2 & (d0 ^ d1));
            const uint32_t Z0 = ~(ds | dc | d3), D1 = ~dc & (ds ^ d3);
            const uint32_t Wge1 = w0 | w1 | w2, Wge3 = w2 | (w1 & w0);
            const uint32_t up = (Z0 & Wge1) | (D1 & Wge3);
            // Delta n - 1 = ~w0 + 2 E1 selects the uphill chains' accept mask
            const uint32_t E1 = Z0 & Wge3;
            const uint32_t lo = (w0 & lt[0]) | (~w0 & lt[1]), hi = (w0 & lt[2]) | (~w0 & lt[3]);
            const uint32_t acc = flips & (~up | ((E1 & hi) | (~E1 & lo)));
            sts(ow[0], o0 ^ acc);
            sts(ow[1], o1 ^ acc);
            sts(ow[2], o2 ^ acc);
            sts(ow[3], o3 ^ acc);
            __syncwarp();
            if (!end) bar_arrive(1 + (set + 1 == NS ? 0 : set + 1), 2 * TS);
            // the state before this phase is a sample if the phase before is one
            if (t > first || (t == first && col > 0)) {
                uint32_t n0, n1, n2;
                if (IND) {
                    sum4(m0 & ~o0, m1 & ~o1, m2 & ~o2, m3 & ~o3, n0, n1, n2);
                    count_add(v, n0, n1, n2);
                    sum4(m0 & ~t0, m1 & ~t1, m2 & ~t2, m3 & ~t3, n0, n1, n2);
                    count_add(v, n0, n1, n2);
                } else {
                    sum4(~(o0 | t0), ~(o1 | t1), ~(o2 | t2), ~(o3 | t3), n0, n1, n2);
                    count_add(v, n0, n1, n2);
                }
                if (++since == kFlushEvery) {
                    credit();
                    since = 0;
                }
            }
            col += NS;
            const uint32_t ahead = (uint32_t)col >> 2;
            col &= 3;
            if (gd.t_end - t <= ahead) break;
            t += ahead;
        }
        if (since) credit();
    }
    __syncthreads();

    // the state after the last phase: its sample, n, and what the caller asked for
    if (n_samples || p.chain_n) {
        for (int q = tid; q < nq; q += nt) {
            if (IND) {
                count_add(v, ~X[q], 0u, 0u);
                count_add(v, ~Z[q], 0u, 0u);
            } else {
                count_add(v, ~(X[q] | Z[q]), 0u, 0u);
            }
        }
        const uint32_t n = count_flush(v, lane);
        if (n) atomicAdd(&left[lane], n);
        __syncthreads();
        if (tid < 32 && ((valid >> tid) & 1u)) {
            const size_t ci = ci_of(tid);
            const uint32_t un = left[tid];
            if (n_samples && p.chain_sum)
                atomicAdd(reinterpret_cast<unsigned long long*>(p.chain_sum + ci), 0ull - (unsigned long long)un);
            if (p.chain_n) p.chain_n[ci] = (IND ? 2 : 1) * nq - (int)un;
        }
    }
    if (p.state_out) {
        uint32_t* st = p.state_out + gd.state_off + (size_t)bid * 2 * nq;
        for (int q = tid; q < nq; q += nt) {
            st[q] = X[word_of(q, nq)];
            st[nq + q] = Z[word_of(q, nq)];
        }
    }
    if (p.chain_frames) {
        uint32_t* cfg = p.chain_frames + gd.frames_off - (size_t)gd.item_base * p.C * 2 * W;
        for (int i = tid; i < 32 * W; i += nt) {
            const int b = i / W, wi = i - b * W;
            if (!((valid >> b) & 1u)) continue;
            uint32_t xw = 0, zw = 0;
            for (int k = 0; k < 32 && 32 * wi + k < nq; ++k) {
                xw |= ((X[word_of(32 * wi + k, nq)] >> b) & 1u) << k;
                zw |= ((Z[word_of(32 * wi + k, nq)] >> b) & 1u) << k;
            }
            uint32_t* f = cfg + ci_of(b) * 2 * W;
            f[wi] = xw;
            f[W + wi] = zw;
        }
    }
}

template <int G, bool IND>
cudaError_t launch_wide_t(const SweepParams& p, cudaStream_t s) {
    long long blocks = 0;
    int threads = 0;
    size_t words = 0;
    for (int g = 0; g < p.n_groups; ++g) {
        const int L = p.grp[g].L, ts = wide_set_threads(p.code, L), ns = wide_sets(p.code, L, p.wide);
        blocks += p.grp[g].n_bundles;
        threads = std::max(threads, ns * ts);
        words = std::max(words, wide_smem_words(p.grp[g].nq, ts, ns, wide_fixed<G>() * PlaneBatch<G>::SLOTS));
    }
    if (blocks == 0) return cudaSuccess;
    static SmemLimit limit;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && 4 * words > 48 * 1024) e = limit.ensure(wide_kernel<G, IND>, dev, 4 * words);
    if (e != cudaSuccess) return e;
    wide_kernel<G, IND><<<(unsigned)blocks, threads, 4 * words, s>>>(p);
    return cudaGetLastError();
}

template <int G>
cudaError_t launch_wide_g(const SweepParams& p, cudaStream_t s) {
    return p.noise == 1 ? launch_wide_t<G, true>(p, s) : launch_wide_t<G, false>(p, s);
}

}  // namespace

cudaError_t launch_sweep_wide(const SweepParams& p, cudaStream_t s) {
    switch (p.G) {
        case 4: return launch_wide_g<4>(p, s);
        case 8: return launch_wide_g<8>(p, s);
        case 16: return launch_wide_g<16>(p, s);
        case 32: return launch_wide_g<32>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace surfmcmc
