// schedule.cu -- adaptive annealing steps (Sec. 5.4 cites adaptive
// temperature steps without fixing them). Reading: the step dbeta is chosen so
// that the current population's energy histogram h(E) and its reweighting to
// beta + dbeta, P1(E) ~ h(E) exp(-dbeta E), overlap by a target,
//   alpha(dbeta) = sum_E min(h(E)/R, P1(E)),
// by bisection (50 halvings of [0, dmax]); or an MLP proposes dbeta from the
// population's energy moments and is accepted when its realised overlap lies
// in a band, the bisection being the fallback.
//
// One cluster of thread blocks per lattice. An overlap is computed by one block, its
// sums always in the same order; the blocks of the cluster evaluate the next levels of
// the bisection's tree at once -- 15 of the 16 blocks the midpoints that the next
// four halvings can come to -- and then every block walks down the tree by the
// computed overlaps, so the result is the sequential one's to the last bit. Most of
// the comparisons with the target are far from a tie: they are decided by overlap_fast,
// within 1e-12 of overlap_eval at a quarter of its cost, and only the last rounds (and the
// overlap reported) take the latter. The population's moments, which only the report
// needs when no step is proposed, are worked out by a second cluster meanwhile.
//
// Bound: fp64, 1/64 of fp32's rate on this chip (a warp holds its scheduler for 64 cycles
// with each operation): overlap_eval has an exponential and a division per occupied bin,
// 5 us for 2D L = 64, R = 4000. One block, one evaluation after the other: 333 us per
// step; the cluster with overlap_eval alone 95 us; as it is 56 us.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "check.cuh"
#include "device.cuh"
#include "internal.h"

namespace gbmc {

namespace cg = cooperative_groups;

namespace {

// Bins of the population's range kept in shared memory (40 bytes each); a wider
// range is read again from the histogram.
constexpr uint32_t kSchedBins = 4096;
constexpr uint32_t kSchedThreads = 256;
struct SchedBins {
    double h[kSchedBins], p0[kSchedBins];
    double w[kSchedBins];               // overlap_eval's weights
    float2 hf[kSchedBins], pf[kSchedBins];  // h and p0 as pairs of floats
    float2 coarse[kSchedBins / 32], fine[32];  // overlap_fast's exponentials
};
// Error bound of overlap_fast against overlap_eval, u = 2^-24: a product is within 5 u^2, an
// addition of positive terms within 3 u^2 (Joldes, Muller, Popescu 2017), and on the way from a
// bin to a sum lie at most 15 additions of the thread's own, 5 in the warp and 7 over the warps: 81
// u^2. A weight is within 12 u^2 (two products, three conversions), their sum W 93, 1 / W 102, p1
// 119, the overlap 200 u^2 = 7.1e-13; the exponentials' arguments add less than 2e-14 where a
// bin's weight matters. (Measured: 5e-15.)
constexpr double kFastError = 1e-12;
static_assert(kSchedBins / kSchedThreads <= 16 && kSchedThreads <= 256, "overlap_fast's error bound");

__device__ __forceinline__ float bfr(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Sum over the block; every thread receives the result. sh: 33 doubles.
__device__ double block_sum_d(double v, double* sh) {
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double s = lane < nw ? sh[lane] : 0.0;
        s = warp_sum(s);
        if (lane == 0) sh[32] = s;
    }
    __syncthreads();
    const double r = sh[32];
    __syncthreads();
    return r;
}

// The overlap at step d; whole block (256 threads, thread t the bins t, t + 256, ..).
__device__ double overlap_eval(const uint32_t* h, const SchedBins* S, uint32_t bmin, uint32_t bmax, double R, double d,
                               double* sh) {
    double w = 0.0;
    if (S) {
        SchedBins* Sw = const_cast<SchedBins*>(S);
        for (uint32_t i = threadIdx.x; i <= bmax - bmin; i += blockDim.x) {
            const double hb = S->h[i];
            if (hb != 0.0) {
                const double x = hb * exp(-d * 4.0 * (double)i);
                Sw->w[i] = x;
                w += x;
            }
        }
    } else {
        for (uint32_t b = bmin + threadIdx.x; b <= bmax; b += blockDim.x) {
            const uint32_t hb = h[b];
            if (hb) w += (double)hb * exp(-d * 4.0 * (double)(b - bmin));
        }
    }
    const double W = block_sum_d(w, sh);
    double a = 0.0;
    if (S) {
        for (uint32_t i = threadIdx.x; i <= bmax - bmin; i += blockDim.x) {
            if (S->h[i] != 0.0) {
                const double p0 = S->p0[i], p1 = S->w[i] / W;
                a += p0 < p1 ? p0 : p1;
            }
        }
    } else {
        for (uint32_t b = bmin + threadIdx.x; b <= bmax; b += blockDim.x) {
            const uint32_t hb = h[b];
            if (hb) {
                const double p0 = (double)hb / R;
                const double p1 = (double)hb * exp(-d * 4.0 * (double)(b - bmin)) / W;
                a += p0 < p1 ? p0 : p1;
            }
        }
    }
    return block_sum_d(a, sh);
}

// Pairs of floats: the unevaluated sum x + y, |y| <= ulp(x) / 2.
__device__ __forceinline__ float2 pair_of(double v) {
    const float x = (float)v;
    return make_float2(x, (float)(v - (double)x));
}
__device__ __forceinline__ float2 pair_norm(float x, float y) {
    const float s = __fadd_rn(x, y);
    return make_float2(s, __fsub_rn(y, __fsub_rn(s, x)));
}
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
    const float s = __fadd_rn(a.x, b.x), z = __fsub_rn(s, a.x);
    const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, z)), __fsub_rn(b.x, z));
    return pair_norm(s, __fadd_rn(e, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    return pair_norm(p, __fadd_rn(__fmaf_rn(a.x, b.x, -p), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x))));
}
// 1 / a: a float's reciprocal and one Newton step
__device__ __forceinline__ float2 pair_inv(float2 a) {
    const float y = __fdiv_rn(1.0f, a.x);
    return pair_norm(y, __fmul_rn(y, __fmaf_rn(-a.y, y, __fmaf_rn(-a.x, y, 1.0f))));
}
__device__ __forceinline__ float2 pair_warp_sum(float2 v) {
#pragma unroll
    for (int o = 16; o; o >>= 1)
        v = pair_add(v, make_float2(__shfl_xor_sync(~0u, v.x, o), __shfl_xor_sync(~0u, v.y, o)));
    return v;
}

// The same within kFastError, without fp64 but for the exponentials: exp(-4 d i) is the
// product of two tabulated factors, the rest is in pairs of floats (48 bits; a product is
// 7 instructions at 64 times fp64's rate). Whole block; every thread receives the
// result. sf: 16 entries.
__device__ double overlap_fast(SchedBins* S, uint32_t n, double d, float2* sf) {
    const uint32_t t = threadIdx.x, warp = t >> 5;
    constexpr uint32_t kWarps = kSchedThreads / 32;
    for (uint32_t i = t; i < 32u + (n + 31u) / 32u; i += kSchedThreads) {
        if (i < 32u) S->fine[i] = pair_of(exp(-d * 4.0 * (double)i));
        else S->coarse[i - 32u] = pair_of(exp(-d * 4.0 * (double)(32u * (i - 32u))));
    }
    __syncthreads();
    // a thread's bins as in overlap_eval; the weights are worked out again in the second
    // pass, for less than keeping them would take
    auto weight = [&](uint32_t i) { return pair_mul(S->hf[i], pair_mul(S->coarse[GBMC_IDX(i >> 5, kSchedBins / 32u)], S->fine[i & 31u])); };
    float2 w = make_float2(0.0f, 0.0f);
    for (uint32_t i = t; i < n; i += kSchedThreads) w = pair_add(w, weight(i));
    w = pair_warp_sum(w);
    if ((t & 31u) == 0u) sf[warp] = w;
    __syncthreads();
    float2 W = sf[0];
#pragma unroll
    for (uint32_t k = 1; k < kWarps; ++k) W = pair_add(W, sf[k]);
    const float2 inv = pair_inv(W);
    float2 a = make_float2(0.0f, 0.0f);
    for (uint32_t i = t; i < n; i += kSchedThreads) {
        const float2 p0 = S->pf[i], p1 = pair_mul(weight(i), inv);
        const bool first = p0.x < p1.x || (p0.x == p1.x && p0.y < p1.y);
        a = pair_add(a, first ? p0 : p1);
    }
    a = pair_warp_sum(a);
    if ((t & 31u) == 0u) sf[kWarps + warp] = a;
    __syncthreads();
    a = sf[kWarps];
#pragma unroll
    for (uint32_t k = 1; k < kWarps; ++k) a = pair_add(a, sf[kWarps + k]);
    return (double)a.x + (double)a.y;
}

// One evaluated node of the bisection's tree.
struct SchedNode {
    double alpha, mid;
};

// The bisection's state, kept by warp 0 of each block for the others.
struct SchedWalk {
    double lo, hi, alo;
    double mid;  // this block's node of the coming round
    int it;
    bool exact, alo_exact, clamped;
};

// The midpoint of node v of the tree under [l, u]: the bits below v's leading one say
// which half each earlier level kept (1: the upper).
__device__ double node_mid(double l, double u, uint32_t v) {
    for (int k = 30 - __clz(v); k >= 0; --k) {
        const double mid = 0.5 * (l + u);
        if ((v >> k) & 1u) l = mid;
        else u = mid;
    }
    return 0.5 * (l + u);
}

}  // namespace

// Block r of a lattice's cluster; where nothing is proposed, a second cluster's block 0
// reports the moments.
__global__ void __launch_bounds__(kSchedThreads) k_schedule(const __grid_constant__ SchedLaunch S) {
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ double sh[33];
    __shared__ float2 sf[2 * kSchedThreads / 32];
    __shared__ SchedNode node_mine[2];  // this block's evaluation, read by the others (by round parity)
    __shared__ double alpha_prop;
    __shared__ SchedWalk walk;
    __shared__ float xin[kMlpIn], h1[kMlpHidden], h2[kMlpHidden];
    __shared__ double ys;
    chain_begin();
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), n_blocks = cluster.num_blocks();
    const uint32_t job = (blockIdx.x / n_blocks) % (uint32_t)S.njobs;
    const bool propose = S.mode == 2 && S.mlp;
    const bool reporter = blockIdx.x / n_blocks >= (uint32_t)S.njobs;
    if (reporter && rank != 0) return;
    const SchedJob& J = S.jobs[job];
    SchedOut& out = S.out[job];
    const int32_t emin = *J.emin, emax = *J.emax;
    const uint32_t bmin = (uint32_t)(emin - J.e_lo) >> 2, bmax = (uint32_t)(emax - J.e_lo) >> 2;
    const double R = (double)J.R;
    // moments of E - Emin and the features: where a step is proposed every block needs them
    if (reporter || propose) {
        double s1 = 0.0;
        for (uint32_t b = bmin + threadIdx.x; b <= bmax; b += blockDim.x)
            s1 += (double)J.hist[GBMC_IDX(b, J.nbins)] * 4.0 * (double)(b - bmin);
        const double m1 = block_sum_d(s1, sh) / R;
        double s2 = 0.0, s3 = 0.0;
        for (uint32_t b = bmin + threadIdx.x; b <= bmax; b += blockDim.x) {
            const double hb = (double)J.hist[b];
            const double dx = 4.0 * (double)(b - bmin) - m1;
            s2 += hb * dx * dx;
            s3 += hb * dx * dx * dx;
        }
        const double var = block_sum_d(s2, sh) / R;
        const double m3 = block_sum_d(s3, sh) / R;
        if (threadIdx.x == 0) {
            double skew = var > 0.0 ? m3 / (var * sqrt(var)) : 0.0;
            skew = skew < -10.0 ? -10.0 : (skew > 10.0 ? 10.0 : skew);
            xin[0] = (float)(((double)emin + m1) / (double)J.N);
            xin[1] = (float)log(var / (double)J.N + 1e-6);
            xin[2] = (float)skew;
            xin[3] = (float)J.beta;
            xin[4] = (float)log((double)J.L);
            xin[5] = (float)log(R);
            ys = var;
            if (rank == 0) {
                out.var = var;
                for (int i = 0; i < kMlpIn; ++i) out.feat[i] = xin[i];
            }
        }
        __syncthreads();
        if (reporter) return;
    }
    SchedBins* bins = bmax - bmin < kSchedBins ? reinterpret_cast<SchedBins*>(raw) : nullptr;
    if (bins)  // each thread reads back only its own bins
        for (uint32_t b = bmin + threadIdx.x; b <= bmax; b += blockDim.x) {
            const double hb = (double)J.hist[GBMC_IDX(b, J.nbins)], p0 = hb / R;
            bins->h[GBMC_IDX(b - bmin, kSchedBins)] = hb;
            bins->p0[b - bmin] = p0;
            bins->hf[b - bmin] = pair_of(hb);
            bins->pf[b - bmin] = pair_of(p0);
        }

    int kind = 1, evals = 0;
    double dbeta = 0.0, alpha = 1.0, proposal = 0.0, alpha_p = 0.0;
    if (propose) {
        const float* p = S.mlp;
        if (threadIdx.x < kMlpHidden) {
            const int j = threadIdx.x;
            float a = bfr(p[kOffB1 + j]);
            for (int i = 0; i < kMlpIn; ++i) a += bfr(p[kOffW1 + j * kMlpIn + i]) * xin[i];
            h1[j] = tanhf(a);
        }
        __syncthreads();
        if (threadIdx.x < kMlpHidden) {
            const int j = threadIdx.x;
            float a = bfr(p[kOffB2 + j]);
            for (int k = 0; k < kMlpHidden; ++k) a += bfr(p[kOffW2 + j * kMlpHidden + k]) * h1[k];
            h2[j] = tanhf(a);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            float y = bfr(p[kOffB3]);
            for (int j = 0; j < kMlpHidden; ++j) y += bfr(p[kOffW3 + j]) * h2[j];
            // output y = log(dbeta sigma_E)
            const double var = ys;
            const double sigma = sqrt(var > 1e-12 ? var : 1e-12);
            const double d = exp((double)y) / sigma;
            ys = d > J.dmax ? J.dmax : d;
        }
        __syncthreads();
        proposal = ys;
    }
    if (propose) {  // its overlap, by the last block
        if (rank == n_blocks - 1u) {
            const double a = overlap_eval(J.hist, bins, bmin, bmax, R, proposal, sh);
            if (threadIdx.x == 0) alpha_prop = a;
        }
        cluster.sync();
        alpha_p = *cluster.map_shared_rank(&alpha_prop, n_blocks - 1u);
        ++evals;
        if (S.lo <= alpha_p && alpha_p <= S.hi) {
            kind = 2;
            dbeta = proposal;
            alpha = alpha_p;
        }
    }
    if (kind == 1) {
        // 50 halvings of [0, dmax], `levels` of them per round: block v (1 .. 2^levels - 1)
        // takes node v of the tree of midpoints; block 0 the largest step, in the first
        // round
        uint32_t levels = 1;
        while ((2u << levels) <= n_blocks) ++levels;
        if (threadIdx.x == 0)
            walk = SchedWalk{0.0, J.dmax, 1.0, rank ? node_mid(0.0, J.dmax, rank) : J.dmax, 0, !bins, true, false};
        __syncthreads();
        for (uint32_t round = 0; walk.it < 50 && !walk.clamped; ++round) {
            const uint32_t m = min(levels, (uint32_t)(50 - walk.it)), nodes = (1u << m) - 1u;
            const bool exact = walk.exact;
            if (rank ? rank <= nodes : !round) {
                const double mid = walk.mid;
                double a = 1.0;
                if (!exact) a = overlap_fast(bins, bmax - bmin + 1u, mid, sf);
                if (exact || (rank == 0 && a > S.target - kFastError))
                    a = overlap_eval(J.hist, bins, bmin, bmax, R, mid, sh);
                if (threadIdx.x == 0) node_mine[round & 1u] = SchedNode{a, mid};
            }
            cluster.sync();
            if (threadIdx.x < 32u) {
                // down the tree; a fast overlap too near the target ends the walk, and the
                // halvings from there on take the exact one
                const uint32_t lane = threadIdx.x;
                SchedNode n = {0.0, 0.0};
                if (lane <= nodes && (lane || !round)) n = *cluster.map_shared_rank(&node_mine[round & 1u], lane);
                const uint32_t above = __ballot_sync(~0u, n.alpha >= S.target);
                const uint32_t tie = exact ? 0u : __ballot_sync(~0u, fabs(n.alpha - S.target) <= kFastError);
                uint32_t v = 1, lo_v = 0, hi_v = 0, taken = 0;
                for (; taken < m && !((tie >> v) & 1u); ++taken) {
                    const uint32_t up = (above >> v) & 1u;
                    (up ? lo_v : hi_v) = v;
                    v = 2u * v + up;
                }
                SchedWalk k = walk;
                const double lo = __shfl_sync(~0u, n.mid, lo_v), alo = __shfl_sync(~0u, n.alpha, lo_v);
                const double hi = __shfl_sync(~0u, n.mid, hi_v), amax = __shfl_sync(~0u, n.alpha, 0);
                __syncwarp();
                if (!round && (above & 1u)) {
                    k.clamped = true;
                    k.lo = J.dmax;
                    k.alo = amax;
                } else {
                    if (lo_v) {
                        k.lo = lo;
                        k.alo = alo;
                        k.alo_exact = exact;
                    }
                    if (hi_v) k.hi = hi;
                    k.it += (int)taken;
                    k.exact = exact || taken < m;
                    if (rank) k.mid = node_mid(k.lo, k.hi, rank);
                }
                if (lane == 0) walk = k;
            }
            __syncthreads();
        }
        evals += walk.clamped ? 1 : 51;
        dbeta = walk.lo;
        alpha = walk.alo;
        if (!walk.alo_exact && rank == 0) alpha = overlap_eval(J.hist, bins, bmin, bmax, R, dbeta, sh);
    }
    const int clamped = dbeta == J.dmax;
    cluster.sync();  // no block leaves while others read its shared memory
    if (rank == 0 && threadIdx.x == 0) {
        out.dbeta = dbeta;
        out.alpha = alpha;
        out.proposal = proposal;
        out.alpha_proposal = alpha_p;
        out.kind = kind;
        out.clamped = clamped;
        out.evals = evals;
        out.emin = emin;
        out.emax = emax;
        out.pad = 0;
    }
}

cudaError_t launch_schedule(const SchedLaunch& S, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_schedule, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SchedBins));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_schedule, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kSchedThreads);
    cfg.dynamicSmemBytes = sizeof(SchedBins);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // 16 blocks where the device can place such a cluster, else the portable 8
    for (uint32_t n : {16u, 8u}) {
        cfg.gridDim = dim3(n * (uint32_t)S.njobs * (S.mode == 2 && S.mlp ? 1u : 2u));
        attr[0].val.clusterDim.x = n;
        int clusters = 0;
        if (n > 8u && (cudaOccupancyMaxActiveClusters(&clusters, k_schedule, &cfg) != cudaSuccess || clusters < 1)) {
            cudaGetLastError();
            continue;
        }
        return launch_chained_as(k_schedule, cfg.gridDim, kSchedThreads, sizeof(SchedBins), n, s, S);
    }
    return cudaErrorInvalidConfiguration;
}

}  // namespace gbmc
