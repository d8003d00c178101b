// pa.cu -- population-annealing resampling (Sec. 5.4, step 2; Eq. (13)).
//
// Per population (one instance of one lattice, R replicas), from the energies
// left by the previous sweep launch and its histogram/min/max accumulators:
//   k_pa_weights : integer weight W_j = floor(2^s exp(-dbeta (E_j - Emin))) from
//                  the host-computed table; inclusive sums within 2048-replica
//                  chunks, chunk totals.
//   k_pa_reduce  : ln Q_i = -dbeta Emin + ln sum_E h(E) exp(-dbeta (E-Emin)) - ln R
//                  over the histogram (fixed-order fp64 tree), ln Z += ln Q;
//                  exclusive scan of the chunk totals -> the cumulative weights
//                  C_j = cpre[chunk] + cloc[j] in replica order; reset of the
//                  accumulators for the next sweep.
//   k_pa_draws   : R multinomial draws x_k = floor(U64_k C_R / 2^64) (Philox,
//                  purpose 2), parent = least j with C_j > x_k (two-level
//                  bisection), counts[parent] += 1 (integer atomics: the result
//                  does not depend on their order).
//   k_pa_count_scan, k_pa_place : exclusive scan of the counts; parent j fills
//                  slots [S_j, S_j + n_j): children contiguous, parents in order.
// The sweep kernel then gathers slot c from parent[c] while loading.
//
// Nearest-integer law (variable populations, P.nprev / P.nnext set): the
// draws are replaced by k_pa_nearest -- replica j gets floor(tau_j) copies
// plus one with probability frac(tau_j), tau_j = R0 W_j / C, decided in
// integers -- every phase only looks at the R_{i-1} live replicas, ln Q uses
// R_{i-1}, and the placement writes R_i (at most the capacity P.R).
//
// The phases run in one launch: small and medium populations each in a cluster of blocks
// (k_pa_resample_clusters), larger ones over the whole grid (k_pa_resample_fused); the
// separate kernels are for captured runs and on request.
#include <climits>
#include <cstring>

#include <cooperative_groups.h>

#include "../../include/gbmc.h"
#include "check.cuh"
#include "device.cuh"
#include "internal.h"

namespace gbmc {

namespace cg = cooperative_groups;

constexpr int kScanThreads = 512;
constexpr int kPerThread = kScanChunk / kScanThreads;  // 4

// Replicas of population `inst` before this step's resampling: R_{i-1}.
__device__ __forceinline__ uint32_t live_prev(const PaLattice& P, uint32_t inst) {
    return P.nprev ? __ldcg(P.nprev + inst) : P.R;
}

// 64-bit uniform of resampling draw (or replica) k of population `inst`;
// r > 0: the extra pieces of a large Poisson mean.
__device__ __forceinline__ unsigned long long resample_u64(const PaLattice& P, uint32_t inst, uint32_t k,
                                                           uint32_t r = 0u) {
    const uint4 w = philox4x32_10(
        make_uint4(k >> 1, P.step, r, c3_word(kPurposeResample, 0u, P.inst_base + inst)),
        (uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    return (k & 1u) ? (((unsigned long long)w.w << 32) | w.z) : (((unsigned long long)w.y << 32) | w.x);
}

// Draws 2 p and 2 p + 1.
__device__ __forceinline__ void resample_u64_pair(const PaLattice& P, uint32_t inst, uint32_t p,
                                                  unsigned long long (&U)[2]) {
    const uint4 w = philox4x32_10(make_uint4(p, P.step, 0u, c3_word(kPurposeResample, 0u, P.inst_base + inst)),
                                  (uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    U[0] = ((unsigned long long)w.y << 32) | w.x;
    U[1] = ((unsigned long long)w.w << 32) | w.z;
}

// ---- the five phases, as block-level device functions ----

// Integer weights of one chunk and their inclusive sums within the chunk.
__device__ __forceinline__ void phase_weights(const PaLattice& P, uint32_t inst, uint32_t chunk,
                                              unsigned long long* sh) {
    const uint64_t base = (uint64_t)inst * P.R;
    const uint32_t live = live_prev(P, inst);
    const uint32_t j0 = chunk * kScanChunk + threadIdx.x * kPerThread;
    const int32_t emin = P.emin[inst];
    unsigned long long w[kPerThread];
    unsigned long long run = 0;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const uint32_t j = j0 + i;
        unsigned long long v = 0;
        if (j < live) v = P.wint[GBMC_IDX((uint32_t)(P.E[base + j] - emin) >> 2, P.nbins)];
        run += v;
        w[i] = run;
    }
    unsigned long long total;
    const unsigned long long incl = block_inclusive_scan<unsigned long long>(run, sh, &total);
    const unsigned long long excl = incl - run;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const uint32_t j = j0 + i;
        if (j < P.R) P.cloc[base + j] = excl + w[i];
    }
    if (threadIdx.x == 0) P.ctot[(uint64_t)inst * P.nchunks + chunk] = total;
}

// This thread's share of sum_E h(E) exp(-dbeta (E - Emin)); clears the histogram.
__device__ __forceinline__ double hist_weight(const PaLattice& P, uint32_t inst, int32_t emin, int32_t emax) {
    uint32_t* h = P.hist + (uint64_t)inst * P.nbins;
    double acc = 0.0;
    if (emin <= emax) {  // an empty population (variable sizes) has no range
        const uint32_t bmin = (uint32_t)(emin - P.e_lo) >> 2, bmax = (uint32_t)(emax - P.e_lo) >> 2;
        for (uint32_t b = bmin + threadIdx.x; b <= bmax; b += blockDim.x) {
            const uint32_t hb = h[b];
            if (hb) acc += (double)hb * P.wexp[GBMC_IDX(b - bmin, P.nbins)];
            h[b] = 0u;
        }
    }
    return acc;
}

__device__ __forceinline__ void reset_accumulators(const PaLattice& P, uint32_t inst) {
    P.emin[inst] = INT_MAX;
    P.emax[inst] = INT_MIN;
    unsigned long long* sums = P.sums + (uint64_t)inst * 4;
    sums[0] = sums[1] = sums[2] = sums[3] = 0ull;
}

// ln Q of one population (fixed-order fp64 tree), ln Z += ln Q, exclusive
// scan of its chunk totals, reset of the accumulators for the next sweep.
__device__ __forceinline__ void phase_reduce(const PaLattice& P, uint32_t inst, double* lnZ, double* lnQ_out,
                                             double* sd, unsigned long long* su) {
    const int32_t emin = P.emin[inst], emax = P.emax[inst];
    double acc = warp_sum(hist_weight(P, inst, emin, emax));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (lane == 0) sd[warp] = acc;
    __syncthreads();
    if (warp == 0) {
        double v = lane < nwarps ? sd[lane] : 0.0;
        v = warp_sum(v);
        if (lane == 0) {
            const double log_R = P.nprev ? log((double)live_prev(P, inst)) : P.log_R;
            const double lnQ = -P.dbeta * (double)emin + log(v) - log_R;
            lnQ_out[inst] = lnQ;
            lnZ[inst] += lnQ;
        }
    }
    const unsigned long long* ct = P.ctot + (uint64_t)inst * P.nchunks;
    unsigned long long* cp = P.cpre + (uint64_t)inst * (P.nchunks + 1);
    unsigned long long carry = 0;
    for (uint32_t c0 = 0; c0 < P.nchunks; c0 += blockDim.x) {
        const uint32_t c = c0 + threadIdx.x;
        const unsigned long long v = c < P.nchunks ? __ldcg(ct + c) : 0ull;
        unsigned long long tot;
        const unsigned long long incl = block_inclusive_scan<unsigned long long>(v, su, &tot);
        if (c < P.nchunks) cp[c] = carry + incl - v;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        cp[P.nchunks] = carry;
        reset_accumulators(P, inst);
    }
    __syncthreads();
}

// Multinomial draw g (global over the lattice's populations).
__device__ __forceinline__ void phase_draw(const PaLattice& P, uint64_t g) {
    const uint32_t inst = (uint32_t)(g / P.R), k = (uint32_t)(g - (uint64_t)inst * P.R);
    const unsigned long long U = resample_u64(P, inst, k);
    const unsigned long long* cp = P.cpre + (uint64_t)inst * (P.nchunks + 1);
    // data written by other CTAs earlier in a fused launch: read through L2 (__ldcg)
    const unsigned long long x = __umul64hi(U, __ldcg(cp + P.nchunks));
    // least chunk c with cp[c+1] > x
    uint32_t lo = 0, hi = P.nchunks - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldcg(cp + mid + 1) > x) hi = mid;
        else lo = mid + 1;
    }
    const uint32_t c = lo;
    const unsigned long long xr = x - __ldcg(cp + c);  // least j of the chunk with cloc[j] > xr
    const uint64_t base = (uint64_t)inst * P.R;
    uint32_t a = c * kScanChunk, b = min(P.R, (c + 1) * kScanChunk) - 1;
    while (a < b) {
        const uint32_t mid = (a + b) >> 1;
        if (__ldcg(P.cloc + base + mid) > xr) b = mid;
        else a = mid + 1;
    }
    atomicAdd(&P.counts[base + GBMC_IDX(a, P.R)], 1u);
}

// Nearest-integer copies of replica g (global over the lattice's populations):
// n_j = floor(R0 W_j / C) + [floor(U64_j C / 2^64) < (R0 W_j mod C)], C = sum W.
// R0 W_j <= capacity 2^s <= 2^63 and C <= R_{i-1} 2^s <= 2^63 by the choice of s.
__device__ __forceinline__ uint32_t nearest_copies(const PaLattice& P, uint32_t inst, uint32_t j,
                                                   unsigned long long W, unsigned long long C) {
    const unsigned long long num = (unsigned long long)P.R0 * W;
    const unsigned long long n0 = num / C, rem = num - n0 * C;
    const unsigned long long x = __umul64hi(resample_u64(P, inst, j), C);
    return (uint32_t)n0 + (x < rem ? 1u : 0u);
}

__device__ __forceinline__ void phase_nearest(const PaLattice& P, uint64_t g) {
    const uint32_t inst = (uint32_t)(g / P.R), j = (uint32_t)(g - (uint64_t)inst * P.R);
    if (j >= live_prev(P, inst)) return;
    const uint64_t base = (uint64_t)inst * P.R;
    // W_j from the inclusive in-chunk sums (E_min was already reset by ln Q's phase)
    const unsigned long long W = __ldcg(P.cloc + base + j) - ((j % kScanChunk) ? __ldcg(P.cloc + base + j - 1) : 0ull);
    const unsigned long long C = __ldcg(P.cpre + (uint64_t)inst * (P.nchunks + 1) + P.nchunks);
    P.counts[base + j] = nearest_copies(P, inst, j, W, C);
}

// a / n rounded to nearest for a small integer n, y = 1 / n rounded to nearest, 2^-900 <= |a|,
// in three operations of fp64 (whose rate is 1/64 of fp32's) instead of a division's ten or more.
// q = a y is within 1.5 units in the last place of a / n, so e = a - n q is exact, a / n =
// q + e / n, and e y differs from e / n by less than 2^-52 units; but a / n is no tie of the
// rounding (n odd: n times a 54-bit odd number does not fit 53 bits; powers of two divide
// out) and lies at least 1 / (2 n) units from one.
__device__ __forceinline__ double div_small(double a, double n, double y) {
    const double q = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-n, q, a), y, q);
}
constexpr double kDivSmallest = 0x1p-900;

// n and 1 / n, up to the counts that a mean of 500 reaches (a few sigma of 22 above it).
struct Inverses {
    static constexpr uint32_t kMost = 767;
    double2 v[kMost + 1];
    constexpr Inverses() : v() {
        for (uint32_t n = 1; n <= kMost; ++n) {
            v[n].x = (double)n;
            v[n].y = 1.0 / (double)n;
        }
    }
};
__constant__ constexpr Inverses kInverses;

// e^{-x}, x >= 0, in a fixed sequence of correctly rounded fp64 operations
// (so host and device agree bit for bit): Cody and Waite's reduction x = k ln2
// + r, |r| <= ln2/2, with ln2 = head + tail (the head's last 11 mantissa bits
// zero, so k * head is exact), e^{-r} by Horner's rule on its Taylor series to
// degree 20 (s <- 1 - (r/n) s, n = 20..1), then exact scaling by 2^-k; 0 for
// x > 700.
__device__ __forceinline__ double exp_neg_ieee(double x) {
    if (x > 700.0) return 0.0;
    const double k = floor(__dadd_rn(__ddiv_rn(x, 0.6931471805599453094172321), 0.5));
    const double r = __dsub_rn(__dsub_rn(x, __dmul_rn(k, 0.693147180559890330187045037746429443359375)),
                               __dmul_rn(k, 5.4979230187083711552420206887059365096458314e-14));
    double s = 1.0;
    if (fabs(r) >= kDivSmallest) {
#pragma unroll
        for (int n = 20; n >= 1; --n) s = __dsub_rn(1.0, __dmul_rn(div_small(r, (double)n, 1.0 / n), s));
    } else {  // a step this small rounds away: s = 1 either way, in the sequence's own words
#pragma unroll 1
        for (int n = 20; n >= 1; --n) s = __dsub_rn(1.0, __dmul_rn(__ddiv_rn(r, (double)n), s));
    }
    return ldexp(s, -(int)k);
}

// Poisson(tau) copies by inversion from the 64-bit uniform U: the least n with
// u < F(n), u = the top 53 bits of U as a fraction, F built term by term; a
// term that no longer changes F past the mode ends the search (tau <= 500
// here, so e^{-tau} is a normal number).
__device__ __forceinline__ uint32_t poisson_count(double tau, unsigned long long U) {
    if (tau > 700.0) return 0xFFFFFFFFu;
    const double u = __dmul_rn(__ull2double_rn(U >> 11), 1.1102230246251565404236316680908203125e-16);
    double p = exp_neg_ieee(tau), F = p;
    uint32_t n = 0;
    // None of the values compared is negative: they compare as their bits do, and n > tau as
    // n > floor(tau), both off the fp64 unit. A replica with a mean in the hundreds makes this
    // loop the kernel's longest chain; its five fp64 operations replace some 17 (17 populations of 4170
    // with such replicas: 420 -> 215 us a step).
    const uint32_t mode = (uint32_t)floor(tau);
    const long long ub = __double_as_longlong(u);
    const bool small = tau >= kDivSmallest;
    while (ub >= __double_as_longlong(F) && n < 100000u) {
        n += 1;
        double q;
        if (small && n <= Inverses::kMost) {
            const double2 d = kInverses.v[n];
            q = div_small(tau, d.x, d.y);
        } else {
            q = __ddiv_rn(tau, (double)n);
        }
        p = __dmul_rn(p, q);
        const double Fn = __dadd_rn(F, p);
        if (__double_as_longlong(Fn) == __double_as_longlong(F) && n > mode) break;
        F = Fn;
    }
    return n;
}

// Poisson copies of replica j: Poisson(tau_j), tau_j = R0 W_j / C in fp64; a
// mean above 500 as the sum of m = ceil(tau / 500) Poisson(tau / m) pieces,
// piece p from the replica's resampling word with counter field r = p.
__device__ __forceinline__ uint32_t poisson_copies(const PaLattice& P, uint32_t inst, uint32_t j,
                                                   unsigned long long W, unsigned long long C) {
    const double tau = __ddiv_rn(__ull2double_rn((unsigned long long)P.R0 * W), __ull2double_rn(C));
    if (tau <= 500.0) return poisson_count(tau, resample_u64(P, inst, j));
    uint32_t n = 0;
    const uint32_t m = (uint32_t)ceil(__ddiv_rn(tau, 500.0));
    const double part = __ddiv_rn(tau, (double)m);
    for (uint32_t p = 0; p < m; ++p) n += poisson_count(part, resample_u64(P, inst, j, p));
    return n;
}

__device__ __forceinline__ void phase_poisson(const PaLattice& P, uint64_t g) {
    const uint32_t inst = (uint32_t)(g / P.R), j = (uint32_t)(g - (uint64_t)inst * P.R);
    if (j >= live_prev(P, inst)) return;
    const uint64_t base = (uint64_t)inst * P.R;
    const unsigned long long W = __ldcg(P.cloc + base + j) - ((j % kScanChunk) ? __ldcg(P.cloc + base + j - 1) : 0ull);
    const unsigned long long C = __ldcg(P.cpre + (uint64_t)inst * (P.nchunks + 1) + P.nchunks);
    P.counts[base + j] = poisson_copies(P, inst, j, W, C);
}

// Exclusive scan of the counts within one chunk, chunk total.
__device__ __forceinline__ void phase_count_scan(const PaLattice& P, uint32_t inst, uint32_t chunk, uint32_t* sh) {
    const uint64_t base = (uint64_t)inst * P.R;
    const uint32_t live = live_prev(P, inst);
    const uint32_t j0 = chunk * kScanChunk + threadIdx.x * kPerThread;
    uint32_t v[kPerThread];
    uint32_t run = 0;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const uint32_t j = j0 + i;
        v[i] = run;  // exclusive within the thread
        if (j < live) run += __ldcg(P.counts + base + j);
    }
    uint32_t total;
    const uint32_t incl = block_inclusive_scan<uint32_t>(run, sh, &total);
    const uint32_t excl = incl - run;
#pragma unroll
    for (int i = 0; i < kPerThread; ++i) {
        const uint32_t j = j0 + i;
        if (j < live) P.sloc[base + j] = excl + v[i];
    }
    if (threadIdx.x == 0) P.ntot[(uint64_t)inst * P.nchunks + chunk] = total;
}

// R_i of a variable population.
__device__ __forceinline__ void record_population(const PaLattice& P, uint32_t inst, uint64_t total) {
    if (total > P.R || total == 0) {  // outgrown its capacity, or died out
        atomicExch(P.overflow, 1u);
        if (total > P.R) total = P.R;
    }
    P.nnext[inst] = (uint32_t)total;
}

// Parent j fills the slots [S, S + n); whole warps call it (n = 0: nothing to place). A
// parent with many children -- a large step leaves a few replicas most of the
// population -- has them written by all lanes: one thread's loop over them took 40 of
// 53 us per step for 2D L = 96.
__device__ __forceinline__ void place_children(const PaLattice& P, uint64_t base, uint64_t S, uint32_t n, uint32_t j) {
    constexpr uint32_t kAll = 0xFFFFFFFFu, kFew = 4u;
    if (n && S + n > P.R) {
        atomicExch(P.overflow, 1u);
        n = S < P.R ? (uint32_t)(P.R - S) : 0u;
    }
    uint32_t* to = P.parent + base;
    if (n <= kFew)
        for (uint32_t m = 0; m < n; ++m) to[GBMC_IDX(S + m, P.R)] = j;
    for (uint32_t many = __ballot_sync(kAll, n > kFew); many; many &= many - 1u) {
        const int src = __ffs(many) - 1;
        const uint32_t nn = __shfl_sync(kAll, n, src), jj = __shfl_sync(kAll, j, src);
        const uint64_t SS = __shfl_sync(kAll, (unsigned long long)S, src);
        for (uint32_t m = threadIdx.x & 31u; m < nn; m += 32u) to[GBMC_IDX(SS + m, P.R)] = jj;
    }
}

// Parent j fills slots [S_j, S_j + n_j); counts are cleared for the next step.
// Variable populations: slots at or beyond the capacity are not written (the
// overflow flag is raised instead) and the last chunk's CTA records R_i.
__device__ __forceinline__ void phase_place(const PaLattice& P, uint32_t inst, uint32_t chunk, uint32_t* prefix) {
    const uint64_t base = (uint64_t)inst * P.R;
    const uint32_t live = live_prev(P, inst);
    if (threadIdx.x < 32) {
        uint32_t acc = 0;
        for (uint32_t c = threadIdx.x; c < chunk; c += 32) acc += __ldcg(P.ntot + (uint64_t)inst * P.nchunks + c);
        acc = warp_sum(acc);
        if (threadIdx.x == 0) *prefix = acc;
    }
    __syncthreads();
    const uint32_t pre = *prefix;
    if (P.nnext && threadIdx.x == 0 && chunk + 1 == P.nchunks) {
        record_population(P, inst, (uint64_t)pre + __ldcg(P.ntot + (uint64_t)inst * P.nchunks + chunk));
    }
    for (uint32_t i = threadIdx.x; i < kScanChunk; i += blockDim.x) {  // whole warps
        const uint32_t j = chunk * kScanChunk + i;
        const uint32_t n = j < live ? __ldcg(P.counts + base + j) : 0u;
        place_children(P, base, n ? (uint64_t)pre + __ldcg(P.sloc + base + j) : 0u, n, j);
        if (n) P.counts[base + j] = 0u;
    }
    __syncthreads();
}

// ---- separate kernels (one per phase) ----

__global__ void __launch_bounds__(kScanThreads) k_pa_weights(const __grid_constant__ PaLattice P) {
    __shared__ unsigned long long sh[32];
    phase_weights(P, blockIdx.y, blockIdx.x, sh);
}

cudaError_t launch_pa_weights(const PaLattice& P, cudaStream_t s) {
    dim3 grid(P.nchunks, P.n_inst);
    k_pa_weights<<<grid, kScanThreads, 0, s>>>(P);
    count_launch();
    return cudaGetLastError();
}

// One CTA per population.
__global__ void __launch_bounds__(1024) k_pa_reduce(const __grid_constant__ PaLattice P, double* lnZ,
                                                    double* lnQ_out) {
    __shared__ double sd[32];
    __shared__ unsigned long long su[32];
    phase_reduce(P, blockIdx.x, lnZ, lnQ_out, sd, su);
}

cudaError_t launch_pa_reduce(const PaLattice& P, double* lnZ, int /*first_step*/, cudaStream_t s) {
    // lnQ of the step is kept next to lnZ: lnZ[n_inst .. 2 n_inst)
    k_pa_reduce<<<P.n_inst, 1024, 0, s>>>(P, lnZ, lnZ + P.n_inst);
    count_launch();
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_pa_draws(const __grid_constant__ PaLattice P) {
    const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (g >= (uint64_t)P.n_inst * P.R) return;
    phase_draw(P, g);
}

cudaError_t launch_pa_draws(const PaLattice& P, cudaStream_t s) {
    const uint64_t total = (uint64_t)P.n_inst * P.R;
    k_pa_draws<<<(uint32_t)((total + 255) / 256), 256, 0, s>>>(P);
    count_launch();
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_pa_nearest(const __grid_constant__ PaLattice P) {
    const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (g >= (uint64_t)P.n_inst * P.R) return;
    if (P.nearest == 2) phase_poisson(P, g);
    else phase_nearest(P, g);
}

cudaError_t launch_pa_nearest(const PaLattice& P, cudaStream_t s) {
    const uint64_t total = (uint64_t)P.n_inst * P.R;
    k_pa_nearest<<<(uint32_t)((total + 255) / 256), 256, 0, s>>>(P);
    count_launch();
    return cudaGetLastError();
}

__global__ void __launch_bounds__(kScanThreads) k_pa_count_scan(const __grid_constant__ PaLattice P) {
    __shared__ uint32_t sh[32];
    phase_count_scan(P, blockIdx.y, blockIdx.x, sh);
}

__global__ void __launch_bounds__(kScanThreads) k_pa_place(const __grid_constant__ PaLattice P) {
    __shared__ uint32_t prefix;
    phase_place(P, blockIdx.y, blockIdx.x, &prefix);
}

cudaError_t launch_pa_place(const PaLattice& P, cudaStream_t s) {
    dim3 grid(P.nchunks, P.n_inst);
    k_pa_count_scan<<<grid, kScanThreads, 0, s>>>(P);
    count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_pa_place<<<grid, kScanThreads, 0, s>>>(P);
    count_launch();
    return cudaGetLastError();
}

// ---- fused resampling: one cooperative launch, phases separated by grid barriers ----

// Grid barrier on a monotone arrival counter. Every wait is bounded: after
// `budget` cycles the waiting thread raises *err and gives up, the kernel
// returns, and the host reports GBMC_ERR_TIMEOUT at its next check; nothing
// spins forever. Returns false once *err is set.
__device__ bool grid_barrier(const GridBarrier& B, uint32_t& target) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        target += gridDim.x + B.phantom;
        __threadfence();
        atomicAdd(B.counter, 1u);
        const long long t0 = clock64();
        int ok = 1;
        while (atomicAdd(B.counter, 0u) < target) {
            if (atomicAdd(B.err, 0u) != 0u || clock64() - t0 > B.budget) {
                atomicExch(B.err, 1u);
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

__global__ void __launch_bounds__(kScanThreads) k_pa_resample_fused(const __grid_constant__ PaLattice P, double* lnZ,
                                                                     const __grid_constant__ GridBarrier B) {
    __shared__ unsigned long long sh64[32];
    __shared__ double sd[32];
    __shared__ uint32_t sh32[32];
    __shared__ uint32_t prefix;
    uint32_t target = 0;
    const uint32_t nch = P.n_inst * P.nchunks;
    for (uint32_t c = blockIdx.x; c < nch; c += gridDim.x) phase_weights(P, c / P.nchunks, c % P.nchunks, sh64);
    if (!grid_barrier(B, target)) return;
    for (uint32_t inst = blockIdx.x; inst < P.n_inst; inst += gridDim.x)
        phase_reduce(P, inst, lnZ, lnZ + P.n_inst, sd, sh64);
    if (!grid_barrier(B, target)) return;
    const uint64_t total = (uint64_t)P.n_inst * P.R;
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < total; g += (uint64_t)gridDim.x * blockDim.x) {
        if (P.nearest == 2) phase_poisson(P, g);
        else if (P.nearest) phase_nearest(P, g);
        else phase_draw(P, g);
    }
    if (!grid_barrier(B, target)) return;
    for (uint32_t c = blockIdx.x; c < nch; c += gridDim.x) phase_count_scan(P, c / P.nchunks, c % P.nchunks, sh32);
    if (!grid_barrier(B, target)) return;
    for (uint32_t c = blockIdx.x; c < nch; c += gridDim.x) phase_place(P, c / P.nchunks, c % P.nchunks, &prefix);
}

cudaError_t launch_pa_resample_fused(const PaLattice& P, double* lnZ, const GridBarrier& B, int n_sms,
                                     cudaStream_t s) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pa_resample_fused, kScanThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const uint64_t work = (uint64_t)P.n_inst * P.nchunks;
    uint64_t grid = (uint64_t)n_sms * (uint64_t)per_sm;
    if (grid > work * 4) grid = work * 4;  // draws use more CTAs than chunks
    if (grid < 1) grid = 1;
    e = cudaMemsetAsync(B.counter, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    PaLattice Pc = P;
    double* lz = lnZ;
    GridBarrier Bc = B;
    void* args[] = {&Pc, &lz, &Bc};
    e = cudaLaunchCooperativeKernel((const void*)k_pa_resample_fused, dim3((uint32_t)grid), dim3(kScanThreads), args,
                                    0, s);
    count_launch();
    return e;
}

// ---- small and medium populations: one cluster of blocks per population ----
//
// The weights, draws, counts and placement of one population in the shared memory of
// C - 1 worker blocks, each with a contiguous slice of the replicas; what they exchange
// are the slices' totals, and the waits between the phases are the cluster's hardware
// barrier. Every worker goes through all draws and keeps those that fall into its slice:
// a generator call costs less than a search in another block's memory (five reads and
// an atomic there: 14 us for 20 000 draws over 15 workers, going through all 8 us). The last
// block of the cluster works out ln Q meanwhile (its fp64 sum and logarithm take as long as
// the draws) and clears the accumulators. The populations of all lattices stepping go
// in one launch. Same integers, and the same fp64 sum for ln Q, as k_pa_resample_fused.
//
// Bound: latency -- a few thousand replicas' chains of dependent loads.
// With the launch's own 5 us: 10 us for 500 copies, 14 us for 5000, 15 us for 8 x 5000, where
// the grid-wide kernel with its five barriers over L2 takes 21, 27 and 29 us.

constexpr uint32_t kMaxWorkers = 15;

struct ResampleClusters {
    PaLattice jobs[kMaxJobs];
    double* lnZ[kMaxJobs];
    uint32_t first[kMaxJobs + 1];  // job j's clusters: [first[j], first[j + 1])
    uint32_t slice;                // replicas a worker can hold (even)
};

// ln Q, ln Z and the reset of the accumulators, around the workers' three waits.
__device__ __forceinline__ void cluster_lnq(const PaLattice& P, uint32_t inst, double* lnZ, double* sd) {
    const int32_t emin = P.emin[inst], emax = P.emax[inst];
    const uint32_t live = live_prev(P, inst);
    cg::cluster_group cluster = cg::this_cluster();
    cluster.barrier_arrive();
    const double acc = hist_weight(P, inst, emin, emax);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    // a warp without a bin holds zeros
    const bool any = emin <= emax && (uint32_t)(emax - emin) >> 2 >= (threadIdx.x & ~31u);
    const double w = any ? warp_sum(acc) : 0.0;
    if (lane == 0) sd[warp] = w;
    __syncthreads();
    cluster.barrier_wait();  // all blocks have started
    cluster.barrier_arrive();
    if (warp == 0) {
        const double v = warp_sum(lane < nwarps ? sd[lane] : 0.0);
        if (lane == 0) {
            const double log_R = P.nprev ? log((double)live) : P.log_R;
            const double lnQ = -P.dbeta * (double)emin + log(v) - log_R;
            lnZ[P.n_inst + inst] = lnQ;
            lnZ[inst] += lnQ;
        }
        __syncwarp();
    }
    cluster.barrier_wait();  // every worker has read E_min
    cluster.barrier_arrive();
    if (threadIdx.x == 0) reset_accumulators(P, inst);
    __syncwarp();
    cluster.barrier_wait();  // the counts' totals
}

__global__ void __launch_bounds__(kScanThreads, 2) k_pa_resample_clusters(const __grid_constant__ ResampleClusters A) {
    extern __shared__ __align__(16) unsigned long long dyn[];
    __shared__ unsigned long long tot[kMaxWorkers], pre[kMaxWorkers + 1];
    __shared__ uint32_t ntot[kMaxWorkers];
    __shared__ unsigned long long sh64[32];
    __shared__ uint32_t sh32[32];
    __shared__ double sd[32];
    chain_begin();
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), K = cluster.num_blocks() - 1u, cid = blockIdx.x / (K + 1u);
    uint32_t job = 0;
    while (cid >= A.first[job + 1]) ++job;
    const PaLattice& P = A.jobs[job];
    const uint32_t inst = cid - A.first[job];
    if (rank == K) {
        cluster_lnq(P, inst, A.lnZ[job], sd);
        return;
    }
    cluster.barrier_arrive();
    unsigned long long* cum = dyn;                                   // [slice] inclusive sums of the slice
    uint32_t* cnt = reinterpret_cast<uint32_t*>(dyn + A.slice);      // [slice]
    unsigned long long* mine = dyn + A.slice + A.slice / 2u + 64u * (threadIdx.x / 32u);  // [64] per warp: draws kept

    // the slice [j0, j0 + n), `per` consecutive replicas per thread
    const uint64_t base = (uint64_t)inst * P.R;
    const uint32_t live = live_prev(P, inst);
    const uint32_t width = (live + K - 1u) / K;
    const uint32_t j0 = min(live, rank * width), n = min(live - j0, width);
    const uint32_t per = (width + kScanThreads - 1u) / kScanThreads;
    const uint32_t i0 = min(n, threadIdx.x * per), i1 = min(n, i0 + per);
    {
        const int32_t emin = P.emin[inst];
        unsigned long long run = 0;
        const int32_t* E = P.E + base + j0;
        for (uint32_t i = i0; i < i1; i += 4u) {  // four replicas' loads in flight
            uint32_t bin[4];
            unsigned long long w[4];
#pragma unroll
            for (uint32_t k = 0; k < 4u; ++k) bin[k] = (uint32_t)(E[GBMC_IDX(min(i + k, i1 - 1u), n)] - emin) >> 2;
#pragma unroll
            for (uint32_t k = 0; k < 4u; ++k) w[k] = P.wint[GBMC_IDX(bin[k], P.nbins)];
#pragma unroll
            for (uint32_t k = 0; k < 4u; ++k)
                if (i + k < i1) {
                    run += w[k];
                    cum[GBMC_IDX(i + k, A.slice)] = run;
                    cnt[i + k] = 0u;
                }
        }
        unsigned long long total;
        const unsigned long long excl = block_inclusive_scan<unsigned long long>(run, sh64, &total) - run;
        for (uint32_t i = i0; i < i1; ++i) cum[i] += excl;
        cluster.barrier_wait();  // all blocks have started: their shared memory may be written
        if (threadIdx.x < K) *cluster.map_shared_rank(&tot[rank], threadIdx.x) = total;
    }
    cluster.sync();

    if (threadIdx.x < 32u) {
        const unsigned long long v = threadIdx.x < K ? tot[threadIdx.x] : 0ull;
        const unsigned long long incl = warp_inclusive_scan(v);
        if (threadIdx.x < K) pre[threadIdx.x + 1u] = incl;
        if (threadIdx.x == 0) pre[0] = 0ull;
    }
    __syncthreads();
    const unsigned long long C = pre[K];
    if (!P.nearest) {
        // draws 2 p and 2 p + 1 share a generator call; a warp gathers those of its slice
        // and looks them up 32 at a time
        const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
        const unsigned long long lo = pre[rank], span = pre[rank + 1u] - lo;
        const uint32_t top = n ? 1u << (31 - __clz(n)) : 0u;
        uint32_t kept = 0;
        auto look_up = [&](uint32_t first, uint32_t count) {
            __syncwarp();
            if (lane < count) {
                const unsigned long long xr = mine[GBMC_IDX(first + lane, 64u)];
                uint32_t pos = 0;  // the sums that do not exceed x
                for (uint32_t step = top; step; step >>= 1)
                    if (pos + step <= n && cum[pos + step - 1u] <= xr) pos += step;
                atomicAdd(cnt + GBMC_IDX(pos, n), 1u);
            }
            __syncwarp();
        };
        for (uint32_t p0 = threadIdx.x - lane; 2u * p0 < live; p0 += kScanThreads) {
            unsigned long long U[2];
            resample_u64_pair(P, inst, p0 + lane, U);
#pragma unroll
            for (uint32_t e = 0; e < 2u; ++e) {
                const unsigned long long xr = __umul64hi(U[e], C) - lo;
                const bool hit = 2u * (p0 + lane) + e < live && xr < span;
                const uint32_t hits = __ballot_sync(~0u, hit);
                if (hit) mine[GBMC_IDX(kept + __popc(hits & below), 64u)] = xr;
                kept += __popc(hits);
                if (kept >= 32u) {
                    kept -= 32u;
                    look_up(kept, 32u);
                }
            }
        }
        look_up(0u, kept);
        __syncthreads();
    } else {
        for (uint32_t i = threadIdx.x; i < n; i += kScanThreads) {
            const unsigned long long W = cum[i] - (i ? cum[i - 1u] : 0ull);
            cnt[GBMC_IDX(i, A.slice)] = P.nearest == 2 ? poisson_copies(P, inst, j0 + i, W, C) : nearest_copies(P, inst, j0 + i, W, C);
        }
        __syncthreads();
    }

    uint32_t run = 0, total;
    for (uint32_t i = i0; i < i1; ++i) run += cnt[i];
    uint32_t S32 = block_inclusive_scan<uint32_t>(run, sh32, &total) - run;
    if (threadIdx.x < K) *cluster.map_shared_rank(&ntot[rank], threadIdx.x) = total;
    cluster.sync();
    uint32_t before = 0;
    for (uint32_t c = 0; c < rank; ++c) before += ntot[c];
    if (P.nnext && threadIdx.x == 0 && rank + 1u == K) record_population(P, inst, (uint64_t)before + total);
    for (uint32_t k = 0; k < per; ++k) {  // whole warps
        const uint32_t i = i0 + k, c = i < i1 ? cnt[i] : 0u;
        place_children(P, base, (uint64_t)before + S32, c, j0 + i);
        S32 += c;
    }
}

// The populations that clusters resample faster than the grid-wide kernel, whose blocks are all
// of the chip's (us, clusters : grid). One population: multinomial 20 000 copies 22 : 29, 40 000
// 33 : 30. Nearest integer 80 000 24 : 28. Poisson, bound by fp64 in a cluster's few
// multiprocessors, 5000 27 : 49, 10 000 44 : 52, 20 000 77 : 54. Many populations: some 34
// clusters run at a time, 5 us for the smallest, where the grid-wide kernel has a block per
// population: multinomial, 100 copies, 96, 128, 256, 1024 populations 20 : 26, 25 : 26, 45 : 26,
// 155 : 48; 2000 copies, 128, 200, 256 34 : 39, 48 : 45, 59 : 50; 5000 copies, 256 90 : 99. Nearest
// integer, 1000 copies, 96, 128 25 : 27, 31 : 27; 5000 copies, 200, 256 52 : 53, 65 : 61. Poisson,
// 100 copies, 128, 256 47 : 54, 84 : 55; 2000 copies, 128, 200 137 : 138, 201 : 188.
bool resample_in_clusters(const PaLattice& P) {
    return P.R <= (P.nearest == 2 ? 8192u : P.nearest ? 65536u : 24576u) && P.n_inst <= 100u + P.R / 40u;
}

cudaError_t launch_pa_resample_clusters(const PaLattice* jobs, double* const* lnZ, uint32_t njobs, cudaStream_t s) {
    static_assert(sizeof(ResampleClusters) <= 4000, "kernel parameters");
    ResampleClusters A;
    std::memset(&A, 0, sizeof(A));
    uint32_t R = 1;
    for (uint32_t j = 0; j < njobs; ++j) {
        A.jobs[j] = jobs[j];
        A.lnZ[j] = lnZ[j];
        A.first[j + 1] = A.first[j] + jobs[j].n_inst;
        R = jobs[j].R > R ? jobs[j].R : R;
    }
    for (uint32_t j = njobs; j < (uint32_t)kMaxJobs; ++j) A.first[j + 1] = A.first[j];
    // Blocks per cluster: 8; 16 for larger populations while there are few of them, as only a
    // few clusters of 16 find room at once (multinomial, us for 16 : 8 : 4 blocks: one population
    // of 5000 14 : 15 : 18, of 20 000 22 : 26 : 44; 32 of 5000 32 : 18 : 20).
    uint32_t blocks = R > 2048u && A.first[njobs] <= 4u ? 16u : 8u;
    cudaError_t e = cudaSuccess;
    for (;; blocks = 8u) {
        const uint32_t K = blocks - 1u;
        A.slice = ((R + K - 1u) / K + 1u) & ~1u;
        const size_t bytes = (size_t)A.slice * 12u + kScanThreads / 32 * 64 * 8;
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(kScanThreads);
        cfg.gridDim = dim3(blocks * A.first[njobs]);
        cfg.dynamicSmemBytes = bytes;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = blocks;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaFuncSetAttribute(k_pa_resample_clusters, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        if (blocks > 8u) {  // beyond the portable size: where the device can place it
            e = cudaFuncSetAttribute(k_pa_resample_clusters, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            int clusters = 0;
            if (e != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&clusters, k_pa_resample_clusters, &cfg) != cudaSuccess || clusters < 1) {
                cudaGetLastError();
                continue;
            }
        }
        return launch_chained_as(k_pa_resample_clusters, cfg.gridDim, kScanThreads, bytes, blocks, s, A);
    }
}

// Record of one step for every population of a lattice, after its sweeps.
__global__ void k_pa_record(const __grid_constant__ PaLattice P, const double* lnZ) {
    chain_begin();
    const uint32_t inst = blockIdx.x * blockDim.x + threadIdx.x;
    if (inst >= P.n_inst) return;
    gbmc_pa_stats* st = reinterpret_cast<gbmc_pa_stats*>(P.stats) + inst;
    const unsigned long long* su = P.sums + (uint64_t)inst * 4;
    st->beta = P.beta;
    st->dbeta = P.dbeta;
    st->lnQ = P.step == 0 ? 0.0 : lnZ[P.n_inst + inst];
    st->lnZ = lnZ[inst];
    st->sumE = (int64_t)su[0];
    st->sumE2 = (int64_t)su[1];
    st->sumAbsM = (int64_t)su[2];
    st->sumM2 = (int64_t)su[3];
    st->Emin = P.emin[inst];
    st->Emax = P.emax[inst];
    st->step = P.step;
    st->n_replicas = P.nnext ? P.nnext[inst] : P.R;
    st->overlap = P.overlap;
    st->proposal_kind = P.kind;
    st->pad = 0;
}

cudaError_t launch_pa_record(const PaLattice& P, const double* lnZ, double, cudaStream_t s) {
    return launch_chained(k_pa_record, dim3((P.n_inst + 127) / 128), 128, s, P, lnZ);
}

// Reset of the accumulators before the first measurement (step 0).
__global__ void k_pa_reset(const __grid_constant__ PaLattice P) {
    const uint32_t inst = blockIdx.x;
    uint32_t* h = P.hist + (uint64_t)inst * P.nbins;
    for (uint32_t b = threadIdx.x; b < P.nbins; b += blockDim.x) h[b] = 0u;
    if (threadIdx.x == 0) {
        P.emin[inst] = INT_MAX;
        P.emax[inst] = INT_MIN;
        unsigned long long* sums = P.sums + (uint64_t)inst * 4;
        sums[0] = sums[1] = sums[2] = sums[3] = 0ull;
        if (P.nnext) P.nnext[inst] = P.R0;  // R_0
    }
}

cudaError_t launch_pa_reset(const PaLattice& P, cudaStream_t s) {
    k_pa_reset<<<P.n_inst, 256, 0, s>>>(P);
    count_launch();
    return cudaGetLastError();
}

}  // namespace gbmc
