// lattice.cu -- initial configurations (Sec. 3.1 step 1), bimodal couplings
// (Sec. 6) and the observables E (Eq. (7)) and M of int8 lattices.
#include "device.cuh"
#include "internal.h"

namespace gbmc {

// One thread per group of 4 consecutive sites of one copy: the INIT word of
// q = site>>2 gives all four spins (s = +1 iff the word's top bit is 0).
__global__ void k_init_spins(uint32_t* spins4, uint32_t N4, uint32_t L, uint32_t R, uint64_t ncopies,
                             uint32_t inst_base, uint32_t k0, uint32_t k1, int random_start) {
    const uint64_t total = ncopies * (uint64_t)N4;
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < total;
         g += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t copy = g / N4;
        const uint32_t q = (uint32_t)(g - copy * N4);
        uint32_t packed = 0x01010101u;
        if (random_start) {
            const uint32_t inst = (uint32_t)(copy / R), r = (uint32_t)(copy - (uint64_t)inst * R);
            const uint4 w = philox4x32_10(make_uint4(q, 0u, r, c3_word(kPurposeInit, 0u, inst_base + inst)), k0, k1);
            packed = ((w.x >> 31) ? 0xFFu : 0x01u) | (((w.y >> 31) ? 0xFFu : 0x01u) << 8) |
                     (((w.z >> 31) ? 0xFFu : 0x01u) << 16) | (((w.w >> 31) ? 0xFFu : 0x01u) << 24);
        }
        spins4[g] = packed;
    }
}

cudaError_t launch_init_spins(int8_t* spins, int dim, uint32_t L, uint32_t n_inst, uint32_t R,
                              uint32_t inst_base, uint64_t seed, int random_start, cudaStream_t s) {
    uint64_t N = L;
    for (int d = 1; d < dim; ++d) N *= L;
    const uint64_t ncopies = (uint64_t)n_inst * R;
    const uint64_t total = ncopies * (N / 4);
    const uint32_t threads = 256;
    const uint64_t blocks = (total + threads - 1) / threads;
    const uint32_t grid = (uint32_t)(blocks < 152ull * 64 ? blocks : 152ull * 64);
    k_init_spins<<<grid, threads, 0, s>>>(reinterpret_cast<uint32_t*>(spins), (uint32_t)(N / 4), L, R,
                                          ncopies, inst_base, (uint32_t)seed, (uint32_t)(seed >> 32),
                                          random_start);
    count_launch();
    return cudaGetLastError();
}

// Couplings: bond b = 3*site + mu, word b&3 of q = b>>2 (t = r = 0). Stored as
// three byte planes per instance, [inst][mu][site], byte 1 where J = -1.
__global__ void k_couplings(uint8_t* jbits, uint32_t N, uint32_t n_inst, uint32_t inst_base,
                            uint32_t k0, uint32_t k1) {
    const uint64_t total = (uint64_t)n_inst * N;
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < total;
         g += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t inst = (uint32_t)(g / N), site = (uint32_t)(g - (uint64_t)inst * N);
        const uint32_t c3 = c3_word(kPurposeCoupling, 0u, inst_base + inst);
#pragma unroll
        for (uint32_t mu = 0; mu < 3; ++mu) {
            const uint64_t b = 3ull * site + mu;
            const uint4 w = philox4x32_10(make_uint4((uint32_t)(b >> 2), 0u, 0u, c3), k0, k1);
            const uint32_t u = word_of(w, (uint32_t)(b & 3));
            jbits[((uint64_t)inst * 3 + mu) * N + site] = (uint8_t)(u >> 31);
        }
    }
}

cudaError_t launch_couplings(uint8_t* jbits, uint32_t L, uint32_t n_inst, uint32_t inst_base,
                             uint64_t seed, cudaStream_t s) {
    const uint32_t N = L * L * L;
    const uint64_t total = (uint64_t)n_inst * N;
    const uint32_t threads = 256;
    uint64_t blocks = (total + threads - 1) / threads;
    if (blocks > 152ull * 32) blocks = 152ull * 32;
    k_couplings<<<(uint32_t)blocks, threads, 0, s>>>(jbits, N, n_inst, inst_base, (uint32_t)seed,
                                                      (uint32_t)(seed >> 32));
    count_launch();
    return cudaGetLastError();
}

// jsplit[((inst*2 + c)*6 + d)*(N/2) + row*(L/2) + j] = 4 if the bond in
// direction d of the colour-c site (row, j) has J = -1. Directions: the x
// neighbour with the same plane index j, the other x neighbour, y-1, y+1,
// z-1, z+1. The site is x = 2j + o with o = (y+z+c)&1: for o = 0 the same-j
// neighbour is x+1 and the other x-1; for o = 1 the reverse.
__global__ void k_split_bonds(const uint8_t* jbits, uint8_t* jsplit, uint32_t L, uint32_t n_inst) {
    const uint32_t N = L * L * L, H = N / 2;
    const uint64_t total = (uint64_t)n_inst * N;  // (inst, c, row, j)
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < total;
         g += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t inst = (uint32_t)(g / N);
        const uint32_t rem = (uint32_t)(g - (uint64_t)inst * N);
        const uint32_t c = rem / H, k = rem - c * H;
        const uint32_t row = k / (L / 2), j = k - row * (L / 2);
        const uint32_t y = row % L, z = row / L;
        const uint32_t o = (y + z + c) & 1u;
        const uint32_t x = 2 * j + o;
        const uint8_t* Jx = jbits + (uint64_t)inst * 3 * N;
        const uint8_t* Jy = Jx + N;
        const uint8_t* Jz = Jx + 2 * N;
        const uint32_t site = row * L + x;
        const uint32_t xm = row * L + (x == 0 ? L - 1 : x - 1);
        const uint32_t ym = (z * L + (y == 0 ? L - 1 : y - 1)) * L + x;
        const uint32_t zm = ((z == 0 ? L - 1 : z - 1) * L + y) * L + x;
        const uint8_t fwd_x = Jx[site], bwd_x = Jx[xm];
        uint8_t b[6];
        b[0] = o ? bwd_x : fwd_x;
        b[1] = o ? fwd_x : bwd_x;
        b[2] = Jy[ym];
        b[3] = Jy[site];
        b[4] = Jz[zm];
        b[5] = Jz[site];
        uint8_t* dst = jsplit + ((uint64_t)inst * 2 + c) * 6 * H + k;
#pragma unroll
        for (int d = 0; d < 6; ++d) dst[(uint64_t)d * H] = b[d] ? 4 : 0;
    }
}

cudaError_t launch_split_bonds(const uint8_t* jbits, uint8_t* jsplit, uint32_t L, uint32_t n_inst,
                               cudaStream_t s) {
    k_split_bonds<<<152 * 8, 256, 0, s>>>(jbits, jsplit, L, n_inst);
    count_launch();
    return cudaGetLastError();
}

__global__ void k_jbits_to_int8(const uint8_t* jbits, int8_t* out, uint32_t N, uint32_t n_inst) {
    const uint64_t total = (uint64_t)n_inst * N * 3;
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < total;
         g += (uint64_t)gridDim.x * blockDim.x) {
        // out layout [inst][site][mu]
        const uint64_t inst = g / (3ull * N);
        const uint64_t rem = g - inst * 3ull * N;
        const uint64_t site = rem / 3, mu = rem % 3;
        out[g] = jbits[(inst * 3 + mu) * N + site] ? -1 : 1;
    }
}

cudaError_t launch_jbits_to_int8(const uint8_t* jbits, int8_t* out, uint32_t N, uint32_t n_inst,
                                 cudaStream_t s) {
    k_jbits_to_int8<<<152 * 8, 256, 0, s>>>(jbits, out, N, n_inst);
    count_launch();
    return cudaGetLastError();
}

// ---- observables ----
//
// E = -sum_i sum_mu J_{i,mu} s_i s_{i+mu} (forward bonds) = 2 U - dim N, U the
// unsatisfied bonds, and M = sum_i s_i = N - 2 D, D the down spins: both counted
// four sites to a 32-bit word (bit 1 of a byte: down; bit 1 of own ^ neighbour ^
// (J = -1): unsatisfied). A copy is one run of N bytes, so the neighbours of the
// word at byte i start at byte i + 1, i + L (wrapping within the copy, in 3D
// within its slab) and i + L^2; rows need not start on a word (L % 4 = 2). The
// shift by one byte pairs the last site of a row with the next row's first one;
// that bond is put right per row. L % 16 == 0: 16 sites per thread, no such bonds.
//
// Bound: reading the spins once (the neighbours come from L1 and L2). T threads
// serve a copy; copies too few to fill the device are spread over several blocks
// each, whose shares are added to outputs zeroed first. One lattice of L = 4096: 92 us
// (one site at a time, three divisions each) -> 12 us with both launches; L = 1000
// 90 -> 10 us.

__device__ __forceinline__ uint32_t unsat4(uint32_t own, uint32_t nb, uint32_t j) {
    return (((own ^ nb) >> 1) ^ j) & 0x01010101u;
}

// U and D of the sites [16 c, 16 c + 16) (L % 16 == 0).
template <int DIM, bool EA>
__device__ __forceinline__ void obs_chunk(const int8_t* s, const uint8_t* jb, uint32_t L, uint32_t N, uint32_t c,
                                          int& U, int& D) {
    const uint32_t W = L >> 4, row = c / W, g = c - row * W;
    const uint32_t A = DIM == 3 ? L * L : N, yi = DIM == 3 ? row % L : row;
    const uint4 own = reinterpret_cast<const uint4*>(s)[c];
    const uint32_t nxt = *reinterpret_cast<const uint32_t*>(s + (uint64_t)row * L + (g + 1u == W ? 0u : 16u * (g + 1u)));
    const uint32_t yd = yi + 1u == L ? 16u * c + L - A : 16u * c + L;
    const uint4 dn = *reinterpret_cast<const uint4*>(s + yd);
    uint4 fr = make_uint4(0u, 0u, 0u, 0u), jx = fr, jy = fr, jz = fr;
    if constexpr (DIM == 3) {
        const uint32_t zd = 16u * c + A >= N ? 16u * c + A - N : 16u * c + A;
        fr = *reinterpret_cast<const uint4*>(s + zd);
    }
    if constexpr (EA) {
        jx = reinterpret_cast<const uint4*>(jb)[c];
        jy = reinterpret_cast<const uint4*>(jb + N)[c];
        jz = reinterpret_cast<const uint4*>(jb + 2ull * N)[c];
    }
    const uint32_t o[5] = {own.x, own.y, own.z, own.w, nxt}, d[4] = {dn.x, dn.y, dn.z, dn.w};
    const uint32_t f[4] = {fr.x, fr.y, fr.z, fr.w}, x[4] = {jx.x, jx.y, jx.z, jx.w};
    const uint32_t y[4] = {jy.x, jy.y, jy.z, jy.w}, z[4] = {jz.x, jz.y, jz.z, jz.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t u = unsat4(o[k], __funnelshift_r(o[k], o[k + 1], 8), x[k]) + unsat4(o[k], d[k], y[k]);
        if constexpr (DIM == 3) u += unsat4(o[k], f[k], z[k]);
        U += (int)((u * 0x01010101u) >> 24);
        D += __popc(o[k] & 0x02020202u);
    }
}

// The same for the word of sites 4 c .. 4 c + 3, any even L; the bond of a row's
// last site is taken to the next byte (obs_row puts it right).
template <int DIM, bool EA>
__device__ __forceinline__ void obs_word(const int8_t* s, const uint8_t* jb, uint32_t L, uint32_t N, uint32_t c,
                                         int& U, int& D) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(s);
    const uint32_t NW = N >> 2, AW = DIM == 3 ? (L * L) >> 2 : NW, own = w[c];
    const uint32_t nxt = w[c + 1u == NW ? 0u : c + 1u];
    // byte 4 c + L, wrapping within the slab (2D: the copy)
    const uint32_t slab = DIM == 3 ? c / AW * AW : 0u;
    uint32_t p = c - slab + (L >> 2);
    if (p >= AW) p -= AW;
    uint32_t dn = w[slab + p];
    if (L & 2u) dn = __funnelshift_r(dn, w[slab + (p + 1u == AW ? 0u : p + 1u)], 16);
    const uint32_t* j = reinterpret_cast<const uint32_t*>(jb);
    uint32_t u = unsat4(own, __funnelshift_r(own, nxt, 8), EA ? j[c] : 0u) + unsat4(own, dn, EA ? j[NW + c] : 0u);
    if constexpr (DIM == 3) u += unsat4(own, w[c + AW >= NW ? c + AW - NW : c + AW], EA ? j[2u * NW + c] : 0u);
    U += (int)((u * 0x01010101u) >> 24);
    D += __popc(own & 0x02020202u);
}

__device__ __forceinline__ void obs_row(const int8_t* s, uint32_t L, uint32_t N, uint32_t row, const uint8_t* jb,
                                        int& U) {
    const uint32_t e = row * L + L - 1u, n = e + 1u == N ? 0u : e + 1u;
    const int last = s[e], j = jb && jb[e] ? 1 : 0;
    U += ((last != s[row * L]) ^ j) - ((last != s[n]) ^ j);
}

// T threads (a power of two) per copy, blockDim.x / T copies per block; with
// gridDim.x > 1 (T = blockDim.x) block x takes the x-th share of its copy.
template <int DIM, bool EA, bool WIDE>
__global__ void __launch_bounds__(256) k_observables(const int8_t* spins, const uint8_t* jbits, uint32_t L, uint32_t N,
                                                     uint32_t R, uint32_t T, uint64_t copy0, uint64_t ncopies,
                                                     int32_t* E, int32_t* M) {
    chain_begin();
    const uint64_t copy = copy0 + (uint64_t)blockIdx.y * (blockDim.x / T) + threadIdx.x / T;
    const uint32_t t = blockIdx.x * T + threadIdx.x % T, n = gridDim.x * T;
    int U = 0, D = 0;
    if (copy < ncopies) {
        const int8_t* s = spins + copy * N;
        uint32_t inst, r;
        split_copy(copy, R, inst, r);
        const uint8_t* jb = EA ? jbits + (uint64_t)inst * 3 * N : nullptr;
        if constexpr (WIDE) {
            for (uint32_t c = t; c < (N >> 4); c += n) obs_chunk<DIM, EA>(s, jb, L, N, c, U, D);
        } else {
            for (uint32_t c = t; c < (N >> 2); c += n) obs_word<DIM, EA>(s, jb, L, N, c, U, D);
            for (uint32_t row = t; row < N / L; row += n) obs_row(s, L, N, row, jb, U);
        }
    }
    for (uint32_t o = min(T, 32u) >> 1; o > 0; o >>= 1) {
        U += __shfl_xor_sync(0xffffffffu, U, o);
        D += __shfl_xor_sync(0xffffffffu, D, o);
    }
    if (T > 32u) {  // one copy per T / 32 warps
        __shared__ int su[8], sd[8];
        const uint32_t warp = threadIdx.x >> 5, per = T >> 5;
        if ((threadIdx.x & 31u) == 0u) {
            su[warp] = U;
            sd[warp] = D;
        }
        __syncthreads();
        if (threadIdx.x % T == 0u)
            for (uint32_t k = 1; k < per; ++k) {
                U += su[warp + k];
                D += sd[warp + k];
            }
    }
    if (threadIdx.x % T == 0u && copy < ncopies) {
        // block 0 brings the constant terms (partial sums may wrap, the totals fit)
        const uint32_t N0 = blockIdx.x == 0 ? N : 0u;
        const int e = (int)(2u * (uint32_t)U - (uint32_t)DIM * N0), m = (int)(N0 - 2u * (uint32_t)D);
        if (gridDim.x == 1) {
            if (E) E[copy] = e;
            if (M) M[copy] = m;
        } else {
            if (E) atomicAdd(&E[copy], e);
            if (M) atomicAdd(&M[copy], m);
        }
    }
}

__global__ void k_zero2(int32_t* a, int32_t* b, uint64_t n) {
    chain_begin();
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (a) a[i] = 0;
    if (b) b[i] = 0;
}

cudaError_t launch_zero2(int32_t* a, int32_t* b, uint64_t n, cudaStream_t s) {
    return launch_chained(k_zero2, dim3((uint32_t)((n + 255u) / 256u)), 256, s, a, b, n);
}

cudaError_t launch_observables(const int8_t* spins, const uint8_t* jbits, int dim, uint32_t L,
                               uint32_t n_inst, uint32_t R, int32_t* E, int32_t* M, cudaStream_t s, bool zeroed) {
    const uint32_t N = L * L * (dim == 3 ? L : 1);
    const uint64_t copies = (uint64_t)n_inst * R;
    const bool wide = L % 16 == 0;
    const uint32_t items = wide ? N >> 4 : N >> 2;
    // about four items per thread while that fills the device, whole blocks and
    // up to 8 blocks per SM over all copies beyond 256 threads
    uint32_t T = 8;
    while (T < 256u && 4u * T < items) T <<= 1;
    uint32_t bx = 1;
    if (T == 256u) {
        const uint64_t most = copies < 152ull * 8ull ? 152ull * 8ull / copies : 1ull;
        bx = (items + 4u * 256u - 1u) / (4u * 256u);
        if (bx > most) bx = (uint32_t)most;
    }
    if (bx > 1 && !zeroed) {
        cudaError_t e = launch_zero2(E, M, copies, s);
        if (e != cudaSuccess) return e;
    }
    const uint32_t per = 256u / T;
    // blockIdx.y is limited to 65535: larger copy counts take several launches
    for (uint64_t c0 = 0; c0 < copies; c0 += 65535ull * per) {
        const uint64_t left = (copies - c0 + per - 1u) / per;
        const dim3 grid(bx, (uint32_t)(left < 65535ull ? left : 65535ull));
        cudaError_t e;
#define GBMC_OBS(D, A) \
    e = launch_chained(wide ? k_observables<D, A, true> : k_observables<D, A, false>, grid, 256, s, spins, jbits, L, N, R, T, \
                       c0, copies, E, M)
        if (dim == 2) GBMC_OBS(2, false);
        else if (jbits) GBMC_OBS(3, true);
        else GBMC_OBS(3, false);
#undef GBMC_OBS
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace gbmc
