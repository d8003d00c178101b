// copies.cuh -- what the bit-sliced resident sweep kernels (bitsweep.cu,
// stream.cu) do with a copy after its sweeps: write its energy and magnetisation,
// decide its exchanges in parallel tempering.
#pragma once
#include <climits>
#include <cstdint>

#include "check.cuh"
#include "device.cuh"
#include "internal.h"

namespace gbmc {

// Whether the configurations at temperatures k and k + 1 of instance `inst`, with
// energies Ea and Eb, are exchanged in round `round`.
__device__ __forceinline__ bool pt_accept(const PtExchange& X, uint32_t inst, uint32_t k, int32_t Ea, int32_t Eb,
                                          uint32_t round) {
    if (Eb >= Ea) return true;
    const uint32_t m = (uint32_t)(Ea - Eb) >> 2;
    const long long thr = X.tab[(uint64_t)k * (X.M + 1) + (m <= X.M ? m : X.M)];
    const uint4 w = philox4x32_10(make_uint4(k >> 2, round, 0u, (4u << 28) | (X.inst_base + inst)), (uint32_t)X.seed,
                                  (uint32_t)(X.seed >> 32));
    return (long long)word_of(w, k & 3u) <= thr;
}

// Energy and magnetisation of one copy after the last sweep (or of every
// sweep when a series is asked for): lane 0 writes them and, for annealing
// runs, adds them to the population's histogram, range and exact sums.
__device__ __forceinline__ void record_copy(const SweepJob& J, uint64_t slot, uint32_t inst, uint32_t s, bool sweep,
                                            bool last, int E, int M) {
    const uint64_t ncopies = (uint64_t)J.n_inst * J.R;
    if (J.Eser && sweep) J.Eser[(uint64_t)s * ncopies + slot] = E;
    if (J.Mser && sweep) J.Mser[(uint64_t)s * ncopies + slot] = M;
    if (!last) return;
    if (J.E) J.E[slot] = E;
    if (J.M) J.M[slot] = M;
    if (J.hist) {
        atomicAdd(&J.hist[(uint64_t)inst * J.nbins + GBMC_IDX((uint32_t)((E - J.e_lo) >> 2), J.nbins)], 1u);
        atomicMin(&J.emin[inst], E);
        atomicMax(&J.emax[inst], E);
        unsigned long long* su = J.sums + (uint64_t)inst * 4;
        const long long el = E, ml = M;
        atomicAdd(&su[0], (unsigned long long)el);
        atomicAdd(&su[1], (unsigned long long)(el * el));
        atomicAdd(&su[2], (unsigned long long)(ml < 0 ? -ml : ml));
        atomicAdd(&su[3], (unsigned long long)(ml * ml));
    }
}

// Sites of a copy held on chip, at most: as many as bytes of shared memory.
constexpr uint32_t kCopySites = 1u << 18;

// The same for the copies of a warp (has: this lane holds one), called by all 32
// lanes: the population's range and sums are reduced over the warp first when
// its copies belong to one instance, one set of atomics per warp. (Atomics on one
// address are worked off one after the other, about 2.7 ns per copy for the six
// of record_copy: annealing 10^5 copies of 2D L = 10 spent 270 of 325 us per
// three-sweep launch on them.)
__device__ __forceinline__ void record_copies(const SweepJob& J, bool has, uint64_t slot, uint32_t inst, uint32_t s,
                                              bool sweep, bool last, int E, int M) {
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    if (!(last && J.hist)) {
        if (has) record_copy(J, slot, inst, s, sweep, last, E, M);
        return;
    }
    const uint32_t mask = __ballot_sync(kAll, has);
    if (!mask) return;
    const uint32_t leader = (uint32_t)__ffs(mask) - 1u;
    const uint32_t inst0 = __shfl_sync(kAll, inst, leader);
    if (!__all_sync(kAll, !has || inst == inst0)) {
        if (has) record_copy(J, slot, inst, s, sweep, last, E, M);
        return;
    }
    if (has) {
        const uint64_t ncopies = (uint64_t)J.n_inst * J.R;
        if (J.Eser && sweep) J.Eser[(uint64_t)s * ncopies + slot] = E;
        if (J.Mser && sweep) J.Mser[(uint64_t)s * ncopies + slot] = M;
        if (J.E) J.E[slot] = E;
        if (J.M) J.M[slot] = M;
        atomicAdd(&J.hist[(uint64_t)inst * J.nbins + GBMC_IDX((uint32_t)((E - J.e_lo) >> 2), J.nbins)], 1u);
    }
    const int mn = __reduce_min_sync(kAll, has ? E : INT_MAX), mx = __reduce_max_sync(kAll, has ? E : INT_MIN);
    // copies held on chip have fewer than kCopySites sites: |E| < 2^20, squares below
    // 2^40 summed as two 20-bit halves
    const int e = has ? E : 0, m = has ? (M < 0 ? -M : M) : 0;
    const uint64_t e2 = (uint64_t)((long long)e * e), m2 = (uint64_t)((long long)m * m);
    const int se = __reduce_add_sync(kAll, e), sm = __reduce_add_sync(kAll, m);
    const uint64_t se2 = (uint64_t)__reduce_add_sync(kAll, (uint32_t)(e2 & 0xFFFFFu)) +
                         ((uint64_t)__reduce_add_sync(kAll, (uint32_t)(e2 >> 20)) << 20);
    const uint64_t sm2 = (uint64_t)__reduce_add_sync(kAll, (uint32_t)(m2 & 0xFFFFFu)) +
                         ((uint64_t)__reduce_add_sync(kAll, (uint32_t)(m2 >> 20)) << 20);
    if ((threadIdx.x & 31u) == leader) {
        atomicMin(&J.emin[inst0], mn);
        atomicMax(&J.emax[inst0], mx);
        unsigned long long* su = J.sums + (uint64_t)inst0 * 4;
        atomicAdd(&su[0], (unsigned long long)(long long)se);
        atomicAdd(&su[1], (unsigned long long)se2);
        atomicAdd(&su[2], (unsigned long long)sm);
        atomicAdd(&su[3], (unsigned long long)sm2);
    }
}

}  // namespace gbmc
