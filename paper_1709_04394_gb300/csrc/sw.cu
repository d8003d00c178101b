// sw.cu -- Swendsen-Wang cluster updates of the Ising ferromagnet (Sec. 3.3):
// bond activation, connected components, cluster flips.
//
//  k_sw_bonds : one thread per 4 sites. Forward bond b = dim i + mu is active
//               iff s_i = s_j and its Philox word (purpose 6, counter
//               (b >> 2, t, replica, c3), word b & 3) is <= T_bond =
//               ceil((1 - exp(-2 beta)) 2^32) - 1; bit mu of bonds[i]. Also
//               resets parent[i] = i.
//  k_sw_union : one thread per site unites i with the far end of each of its
//               active bonds in a lock-free union-find (atomicMin hooks the
//               larger root under the smaller one; a hook that lost a race
//               retries from the value it found, so no link is dropped). Every
//               component ends as one tree rooted at its smallest site.
//  k_sw_flip  : one thread per site finds its root r (with path halving) and
//               flips iff the top bit of r's Philox word (purpose 7, counter
//               (r >> 2, t, replica, c3), word r & 3) is 1; optionally writes r.
// Parent pointers only ever decrease, so every find walks a strictly
// decreasing chain and ends; the hook loops are additionally capped (error flag).
//
// Tiled labelling of 3D lattices (L % 16 == 0: 16 x 8 x 8 tiles), the tile
// decomposition of Sec. 3.3 with the consolidation done by atomics:
//  k_sw_local      : one CTA per tile computes the tile's bond flags (the same
//                    Philox words as k_sw_bonds), labels the tile's components
//                    in shared memory with the same lock-free union-find, and
//                    writes parent[i] = the smallest site of i's component
//                    within the tile (global index: increasing with the local one);
//  k_sw_cross      : one thread per bond that leaves a tile recomputes its
//                    flag and, if active, unites its ends in the global forest;
//  k_sw_flip_tiled : one CTA per tile copies the tile's parent pointers to
//                    shared memory and follows each site's chain there to the
//                    last node inside the tile; only those end nodes look up
//                    their root in the global forest and draw the root's coin,
//                    which every site of the tile then reads from shared memory.
// Each component again ends rooted at its smallest site (a hook always puts
// the larger root under the smaller), so the labels and coins do not depend
// on the order of the unions.
//
// 2D lattices from L = 32 take 32 x 32 tiles (the last ones cut by the lattice's edge;
// L is even) with a scanline labelling,
// the tile labels kept apart from the global forest:
//  k_sw_scan2    : one block per tile, its warps four rows each, lane x = column x,
//                  the rows in order. Row r's x bonds cut it into runs; a run's
//                  label is the smallest of its start and of the labels its y
//                  bonds reach in row r - 1, and a run that reaches two components
//                  above hooks the larger label under the smaller in the tile's
//                  label forest (shared memory); then the warps' seams are united.
//                  At the end every site's label is resolved to its component's
//                  smallest site: lab[i] = that site's tile-local index, and
//                  parent[g] = g for each such tile root g, the only nodes of the
//                  global forest. Bound by the chain of a warp's rows (shuffles and
//                  label lookups, about 2000 cycles each): L = 1024 36 us with one
//                  warp for a tile's 32 rows, 16 us with 8 rows each, 13 us with 4;
//  k_sw_cross    : unites the tile roots of the two ends of each active
//                  tile-crossing bond in the global forest, one bond of a warp's
//                  between the same two roots for all;
//  k_sw_flip_lab : one CTA per tile finds the global root of each tile root
//                  whose component touches the tile border (the others are
//                  roots of whole clusters) and draws each tile root's coin
//                  once; every site takes its tile root's.
//
// The kernels of an update, E and M's, and the next update's follow each other chained (each is
// in place when the one before it ends): L = 1024, 10 updates with E and M 451 -> 373
// us.
//
// Small lattices take none of this but one launch for all updates of a call, a block per
// copy, labels and spins in shared memory (k_sw_resident).
#include <algorithm>
#include <cmath>

#include "bits.cuh"
#include "check.cuh"
#include "device.cuh"
#include "internal.h"

namespace gbmc {

constexpr uint32_t kPurposeSwBond = 6u, kPurposeSwFlip = 7u;
constexpr uint32_t kSwHookCap = 1u << 24;

__device__ __forceinline__ uint32_t sw_forward(uint32_t i, uint32_t mu, uint32_t L, uint32_t dim) {
    const uint32_t x = i % L, y = (i / L) % L;
    if (mu == 0) return i - x + (x + 1 == L ? 0 : x + 1);
    if (mu == 1) return i + (y + 1 == L ? 0 - (L - 1) * L : L);
    const uint32_t LL = L * L, z = i / LL;
    return i + (z + 1 == L ? 0 - (L - 1) * LL : LL);
}

// Forest reads: global forests through L2 (other CTAs hook concurrently),
// shared-memory forests through volatile loads.
template <bool GLOBAL>
__device__ __forceinline__ uint32_t sw_ld(uint32_t* p) {
    if constexpr (GLOBAL) return __ldcg(p);
    else return *reinterpret_cast<volatile uint32_t*>(p);
}

template <bool GLOBAL>
__device__ __forceinline__ uint32_t sw_find(uint32_t* par, uint32_t x) {
    uint32_t cur = sw_ld<GLOBAL>(par + x);
    if (cur == x) return x;
    uint32_t prev = x, next;
    while (cur > (next = sw_ld<GLOBAL>(par + cur))) {
        par[prev] = next;  // path halving: pointers only move to smaller indices
        prev = cur;
        cur = next;
    }
    return cur;
}

// The active flags (bit mu) of the forward bonds of sites i0 .. i0 + 3
// (i0 % 4 == 0): DIM Philox calls cover bonds DIM i0 .. DIM (i0 + 4) - 1; bond
// 4 c + k of them belongs to site i0 + (4 c + k) / DIM.
template <uint32_t DIM>
__device__ __forceinline__ void sw_bond_flags(const SwLaunch& P, const int8_t* s, uint32_t i0, uint32_t r,
                                              uint32_t c3, uint32_t flags[4]) {
    flags[0] = flags[1] = flags[2] = flags[3] = 0u;
#pragma unroll
    for (uint32_t c = 0; c < DIM; ++c) {
        const uint32_t q = (DIM * i0) / 4 + c;
        const uint4 w = philox4x32_10(make_uint4(q, P.t, r, c3), (uint32_t)P.seed, (uint32_t)(P.seed >> 32));
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t n = (4 * c + k) / DIM, mu = (4 * c + k) % DIM, i = i0 + n;
            const uint32_t u = k == 0 ? w.x : k == 1 ? w.y : k == 2 ? w.z : w.w;
            const uint32_t j = sw_forward(i, mu, P.L, DIM);
            if (s[i] == s[j] && (long long)u <= P.T_bond) flags[n] |= 1u << mu;
        }
    }
}

// The same flags for sites i0 .. i0 + 3 = x0 .. x0 + 3 of row y, layer z
// (x0 % 4 == 0, so the four lie in one row): the spins come as 32-bit words
// (own, right-shifted by one site, row below, layer in front) and bit 1 of
// byte n of own ^ neighbour says whether site n differs from it (+-1 bytes).
template <uint32_t DIM>
__device__ __forceinline__ void sw_bond_flags_row(const SwLaunch& P, const int8_t* s, uint32_t i0, uint32_t x0,
                                                  uint32_t y, uint32_t z, uint32_t r, uint32_t c3,
                                                  uint32_t flags[4]) {
    const uint32_t L = P.L;
    const uint32_t own = *reinterpret_cast<const uint32_t*>(s + i0);
    const uint32_t nxt = (uint32_t)(uint8_t)s[i0 - x0 + (x0 + 4 == L ? 0 : x0 + 4)];
    uint32_t dif[DIM];
    dif[0] = own ^ ((own >> 8) | (nxt << 24));
    dif[1] = own ^ *reinterpret_cast<const uint32_t*>(s + (y + 1 == L ? i0 - (L - 1) * L : i0 + L));
    if constexpr (DIM == 3) {
        const uint32_t LL = L * L;
        dif[2] = own ^ *reinterpret_cast<const uint32_t*>(s + (z + 1 == L ? i0 - (L - 1) * LL : i0 + LL));
    }
    flags[0] = flags[1] = flags[2] = flags[3] = 0u;
    // the same words as philox4x32_10((q, t, r, c3)): t, r and c3 hoisted, wide products
    const PhiloxFixed pf = philox_fix(P.t, r, c3, (uint32_t)P.seed, (uint32_t)(P.seed >> 32));
#pragma unroll
    for (uint32_t c = 0; c < DIM; ++c) {
        const uint4 w = philox_q_wide(pf, (DIM * i0) / 4 + c);
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t n = (4 * c + k) / DIM, mu = (4 * c + k) % DIM;
            const uint32_t u = k == 0 ? w.x : k == 1 ? w.y : k == 2 ? w.z : w.w;
            if (!((dif[mu] >> (8 * n + 1)) & 1u) && (long long)u <= P.T_bond) flags[n] |= 1u << mu;
        }
    }
}

// Whether forward bond mu of site i, to site j, is active: the same Philox
// word as in sw_bond_flags (bond b = dim i + mu, call b >> 2, word b & 3).
__device__ __forceinline__ bool sw_bond_active(const SwLaunch& P, const int8_t* s, uint32_t i, uint32_t j,
                                               uint32_t mu, uint32_t r, uint32_t c3) {
    const uint32_t b = P.dim * i + mu;
    if (s[i] != s[j]) return false;
    const uint4 w = philox4x32_10(make_uint4(b >> 2, P.t, r, c3), (uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    const uint32_t u = (b & 3u) == 0 ? w.x : (b & 3u) == 1 ? w.y : (b & 3u) == 2 ? w.z : w.w;
    return (long long)u <= P.T_bond;
}

// Lock-free union of a and b in forest par (global or shared memory).
template <bool GLOBAL>
__device__ __forceinline__ void sw_unite(uint32_t* par, uint32_t a, uint32_t b, unsigned int* err) {
    uint32_t ra = sw_find<GLOBAL>(par, a), rb = sw_find<GLOBAL>(par, b);
    uint32_t n = 0;
    while (ra != rb) {
        if (ra > rb) {
            const uint32_t tmp = ra;
            ra = rb;
            rb = tmp;
        }
        const uint32_t old = atomicMin(par + rb, ra);  // hook the larger root under the smaller
        if (old == rb) break;
        rb = sw_find<GLOBAL>(par, old);  // rb had been hooked meanwhile: merge with its new root
        ra = sw_find<GLOBAL>(par, ra);
        if (++n == kSwHookCap) {
            atomicExch(err, 1u);
            break;
        }
    }
}

template <uint32_t DIM>
__global__ void __launch_bounds__(256) k_sw_bonds(const __grid_constant__ SwLaunch P) {
    chain_begin();
    const uint64_t copy = P.copy0 + blockIdx.y;
    const uint32_t i0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (i0 >= P.N) return;
    const int8_t* s = P.spins + copy * P.N;
    uint8_t* bonds = P.bonds + copy * P.N;
    uint32_t* par = P.parent + copy * P.N;
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    const uint32_t c3 = c3_word(kPurposeSwBond, 0u, P.inst_base + inst);
    uint32_t flags[4];
    sw_bond_flags<DIM>(P, s, i0, r, c3, flags);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        bonds[i0 + k] = (uint8_t)flags[k];
        par[i0 + k] = i0 + k;
    }
}

struct SwTile {
    uint32_t tx, ty, tz;  // tile edge lengths
};

__device__ __forceinline__ SwTile sw_tile(uint32_t dim) {
    return dim == 2 ? SwTile{32u, 32u, 1u} : SwTile{16u, 8u, 8u};
}

template <uint32_t DIM>
__global__ void __launch_bounds__(256) k_sw_local(const __grid_constant__ SwLaunch P) {
    chain_begin();
    __shared__ uint32_t lp[1024];
    const uint64_t copy = P.copy0 + blockIdx.y;
    const int8_t* s = P.spins + copy * P.N;
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    const uint32_t c3 = c3_word(kPurposeSwBond, 0u, P.inst_base + inst);
    const SwTile T = sw_tile(DIM);
    const uint32_t ntx = P.L / T.tx, nty = P.L / T.ty;
    const uint32_t bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, bz = blockIdx.x / (ntx * nty);
    // thread t: local sites l = 4t .. 4t+3 (consecutive x in one tile row)
    const uint32_t l0 = 4 * threadIdx.x;
    const uint32_t lx = l0 % T.tx, ly = (l0 / T.tx) % T.ty, lz = l0 / (T.tx * T.ty);
    const uint32_t i0 = ((bz * T.tz + lz) * P.L + by * T.ty + ly) * P.L + bx * T.tx + lx;
    uint32_t flags[4];
    sw_bond_flags_row<DIM>(P, s, i0, bx * T.tx + lx, by * T.ty + ly, bz * T.tz + lz, r, c3, flags);
    // runs along x: a site starts a run at x == 0 or where the bond from its
    // left neighbour is inactive. Each site's first parent is the start of its
    // run (a tile row spans TPR lanes of one warp: its run starts form one
    // 32-bit mask), so only the bonds along y (and z) go through the union-find.
    constexpr uint32_t TPR = (DIM == 2 ? 32u : 16u) / 4u;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t left = __shfl_up_sync(0xffffffffu, flags[3] & 1u, 1);  // bond into this thread's first site
    uint32_t starts = (lx == 0 || !left) ? 1u : 0u;
#pragma unroll
    for (int k = 1; k < 4; ++k) starts |= (flags[k - 1] & 1u) ? 0u : 1u << k;
    starts <<= 4 * (lane % TPR);
#pragma unroll
    for (uint32_t o = 1; o < TPR; o <<= 1) starts |= __shfl_xor_sync(0xffffffffu, starts, o);
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k)  // bit 0 (x == 0) is always set
        lp[l0 + k] = l0 - lx + 31u - __clz(starts & ((2u << (lx + k)) - 1u));
    __syncthreads();
    // bonds along y and z inside the tile: unite in shared memory
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t l = l0 + k;
        if ((flags[k] & 2u) && ly + 1 < T.ty) sw_unite<false>(lp, l, l + T.tx, P.err);
        if ((flags[k] & 4u) && lz + 1 < T.tz) sw_unite<false>(lp, l, l + T.tx * T.ty, P.err);
    }
    __syncthreads();
    uint32_t g[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t root = sw_find<false>(lp, l0 + k);
        const uint32_t rx = root % T.tx, ry = (root / T.tx) % T.ty, rz = root / (T.tx * T.ty);
        g[k] = ((bz * T.tz + rz) * P.L + by * T.ty + ry) * P.L + bx * T.tx + rx;
    }
    // i0 % 4 == 0, N % 4 == 0 and the forest is a cudaMalloc block: 16-byte aligned
    *reinterpret_cast<uint4*>(P.parent + copy * P.N + i0) = make_uint4(g[0], g[1], g[2], g[3]);
}

// Appends the items with has = true of the warp's lanes to the warp's queue q
// (lane order), advancing n; all 32 lanes call it together.
__device__ __forceinline__ void sw_warp_push(uint32_t* q, uint32_t& n, bool has, uint32_t item) {
    const uint32_t b = __ballot_sync(0xffffffffu, has);
    if (has) q[n + __popc(b & ((1u << (threadIdx.x & 31u)) - 1u))] = item;
    n += __popc(b);
}

// ---- 2D scanline tiles ----

constexpr uint32_t kSwRows = 4, kSwWarps = 32u / kSwRows;  // rows per warp, warps per tile of k_sw_scan2

// Global index of the 32 x 32 tile-local site k (k = 32 row + column) of the
// tile holding site i.
__device__ __forceinline__ uint32_t sw_tile_root(uint32_t k, uint32_t i, uint32_t L) {
    const uint32_t y = i / L, x = i - y * L;
    return ((y & ~31u) + (k >> 5)) * L + (x & ~31u) + (k & 31u);
}

__global__ void __launch_bounds__(32 * kSwWarps) k_sw_scan2(const __grid_constant__ SwLaunch P) {
    chain_begin();
    __shared__ uint32_t f[1024];   // the tile's label forest (local indices)
    __shared__ uint16_t rl[1024];  // each site's run label
    constexpr uint32_t kAll = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31u, r0 = (threadIdx.x >> 5) * kSwRows;
    const uint32_t L = P.L, ntx = (L + 31u) >> 5;
    const uint64_t copy = P.copy0 + blockIdx.y;
    const int8_t* s = P.spins + copy * P.N;
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    const uint32_t bx = blockIdx.x % ntx, by = blockIdx.x / ntx, X = bx * 32u + lane, Y = by * 32u + r0;
    const bool more = r0 + kSwRows < 32u;  // the bonds below the last strip leave the tile (k_sw_cross)
    int sp[kSwRows + 1];  // 0 beyond the lattice's edge: no bond joins it
#pragma unroll
    for (uint32_t k = 0; k <= kSwRows; ++k)
        sp[k] = (k < kSwRows || more) && X < L && Y + k < L ? s[GBMC_IDX((uint64_t)(Y + k) * L + X, P.N)] : 0;
    // bond words: the forward bonds b = 2 i + mu of sites i = 2 q, 2 q + 1 are
    // the four words of Philox call q (t, replica and c3 hoisted). All the strip's bonds
    // first: masks over the row of the bonds to the right and of those below
    const PhiloxFixed pf = philox_fix(P.t, r, c3_word(kPurposeSwBond, 0u, P.inst_base + inst), (uint32_t)P.seed,
                                      (uint32_t)(P.seed >> 32));
    const long long Tb = P.T_bond;
    uint32_t right[kSwRows], below[kSwRows];
#pragma unroll
    for (uint32_t k = 0; k < kSwRows; k += 2u) {
        // lane l: the call of sites 2 (l & 15), +1 of row k + l / 16
        const uint4 c = philox_q_wide(pf, ((Y + k + (lane >> 4)) * L + bx * 32u + 2u * (lane & 15u)) >> 1);
#pragma unroll
        for (uint32_t e = 0; e < 2u; ++e) {
            const uint32_t src = (e << 4) | (lane >> 1);
            const uint32_t a0 = __shfl_sync(kAll, c.x, src), a1 = __shfl_sync(kAll, c.y, src);
            const uint32_t a2 = __shfl_sync(kAll, c.z, src), a3 = __shfl_sync(kAll, c.w, src);
            const uint32_t w0 = (lane & 1u) ? a2 : a0;  // bond along x: word (2 i) & 3
            const uint32_t w1 = (lane & 1u) ? a3 : a1;  // bond along y: word (2 i + 1) & 3
            const int sr = __shfl_down_sync(kAll, sp[k + e], 1);
            // the bond from lane 31 leaves the tile
            right[k + e] = __ballot_sync(kAll, lane < 31u && sp[k + e] == sr && (long long)w0 <= Tb);
            below[k + e] = __ballot_sync(kAll, sp[k + e] == sp[k + e + 1u] && (long long)w1 <= Tb);
        }
    }
    uint32_t lab_prev = 0u;
#pragma unroll
    for (uint32_t k = 0; k < kSwRows; ++k) {
        const bool yb = k > 0u && ((below[k ? k - 1u : 0u] >> lane) & 1u);
        const uint32_t R = ~(right[k] << 1);  // run starts
        const uint32_t own = (r0 + k) * 32u + lane;
        f[own] = own;
        const uint32_t la = yb ? sw_find<false>(f, lab_prev) : 0u;  // the component above, if reached
        // the run's label: segmented minimum over the run (lane x - d is in x's
        // run when no run starts at x - d + 1 .. x), then read at the run's end
        uint32_t v = yb ? la : own;
#pragma unroll
        for (uint32_t d = 1; d < 32u; d <<= 1) {
            const uint32_t t = __shfl_up_sync(kAll, v, d);
            if (lane >= d && ((R >> (lane - d + 1u)) & ((1u << d) - 1u)) == 0u) v = t < v ? t : v;
        }
        const uint32_t nxt = R & ~((2u << lane) - 1u);  // run starts right of this lane
        const uint32_t m = __shfl_sync(kAll, v, nxt ? (uint32_t)__ffs(nxt) - 2u : 31u);
        if (yb && la != m) sw_unite<false>(f, la, m, P.err);  // a second component above joins the run
        rl[own] = (uint16_t)m;
        lab_prev = m;
        __syncwarp();
    }
    // the strips' seams: a bond between the same two runs as the lane before is that lane's
    __syncthreads();
    if (more) {
        const uint32_t under = rl[(r0 + kSwRows) * 32u + lane], up = below[kSwRows - 1u];
        const uint32_t pu = __shfl_up_sync(kAll, under, 1), pl = __shfl_up_sync(kAll, lab_prev, 1);
        const bool same = lane > 0u && ((up >> (lane - 1u)) & 1u) && pu == under && pl == lab_prev;
        if (((up >> lane) & 1u) && !same) sw_unite<false>(f, lab_prev, under, P.err);
    }
    __syncthreads();
    // every site's label resolved to its component's smallest site: lab = its
    // tile-local index; each tile root a node of the global forest
    uint32_t* par = P.parent + copy * P.N;
    uint16_t* lab = P.lab + copy * P.N;
#pragma unroll
    for (uint32_t k = 0; k < kSwRows; ++k) {
        const uint32_t own = (r0 + k) * 32u + lane, i = (Y + k) * L + X;
        if (X >= L || Y + k >= L) continue;
        const uint32_t root = sw_find<false>(f, rl[own]);
        lab[GBMC_IDX(i, P.N)] = (uint16_t)root;
        if (root == own) par[GBMC_IDX(i, P.N)] = i;
    }
}

// The bonds that leave their tile: first those of the sites at a tile's last column
// (bond along x), then those at a tile's last row (along y), then in 3D at its last
// layer (along z). A 2D lattice's last tiles may end with it.
__host__ __device__ __forceinline__ uint32_t sw_cross_count(uint32_t N, uint32_t L, uint32_t dim) {
    return dim == 2 ? 2u * L * ((L + 31u) / 32u) : N / 16 + N / 8 + N / 8;
}

__global__ void __launch_bounds__(256) k_sw_cross(const __grid_constant__ SwLaunch P) {
    chain_begin();
    const uint64_t copy = P.copy0 + blockIdx.y;
    uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = e < sw_cross_count(P.N, P.L, P.dim);
    if (!in) e = 0u;
    const SwTile T = sw_tile(P.dim);
    const uint32_t L = P.L, LL = L * L;
    uint32_t i, j, mu;
    const uint32_t rows = P.N / L, nx = rows * ((L + T.tx - 1u) / T.tx), ny = rows * ((L + T.ty - 1u) / T.ty);
    if (e < nx) {  // (tile column, row): neighbouring lanes down the same tile edge
        const uint32_t c = e / rows, row = e - c * rows, x = min(c * T.tx + T.tx, L) - 1u;
        i = row * L + x;
        j = x + 1 == L ? i - x : i + 1;
        mu = 0;
    } else if ((e -= nx) < ny) {  // (z, tile row k, x)
        const uint32_t nk = (L + T.ty - 1u) / T.ty, rest = e / L, x = e - rest * L, z = rest / nk;
        const uint32_t y = min((rest - z * nk) * T.ty + T.ty, L) - 1u;
        i = (z * L + y) * L + x;
        j = y + 1 == L ? i - (L - 1) * L : i + L;
        mu = 1;
    } else {  // (tile layer k, y, x) -> z = tz k + tz - 1
        e -= ny;
        const uint32_t k = e / LL, z = k * T.tz + T.tz - 1;
        i = z * LL + (e - k * LL);
        j = z + 1 == L ? i - (L - 1) * LL : i + LL;
        mu = 2;
    }
    const int8_t* s = P.spins + copy * P.N;
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    uint32_t* par = P.parent + copy * P.N;
    // a node of the global forest for each end: its tile root (2D), or what its parent
    // pointer holds (3D), read beside the spins
    uint32_t a, b;
    if (P.lab) {
        const uint16_t* lab = P.lab + copy * P.N;
        a = sw_tile_root(lab[GBMC_IDX(i, P.N)], i, L);
        b = sw_tile_root(lab[GBMC_IDX(j, P.N)], j, L);
    } else {
        a = __ldcg(par + GBMC_IDX(i, P.N));
        b = __ldcg(par + GBMC_IDX(j, P.N));
    }
    const bool active = in && sw_bond_active(P, s, i, j, mu, r, c3_word(kPurposeSwBond, 0u, P.inst_base + inst));
    const uint32_t mask = __ballot_sync(0xffffffffu, active);
    if (!active) return;
    // of the warp's bonds between the same two nodes (most of a large cluster's are) one unites
    const uint32_t same = __match_any_sync(mask, ((uint64_t)min(a, b) << 32) | max(a, b));
    if ((threadIdx.x & 31u) + 1u == (uint32_t)__ffs(same)) sw_unite<true>(par, a, b, P.err);
}

__global__ void __launch_bounds__(256) k_sw_union(const __grid_constant__ SwLaunch P) {
    chain_begin();
    const uint64_t copy = P.copy0 + blockIdx.y;
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    const uint8_t f = P.bonds[copy * P.N + i];
    if (!f) return;
    uint32_t* par = P.parent + copy * P.N;
    for (uint32_t mu = 0; mu < P.dim; ++mu)
        if ((f >> mu) & 1u) sw_unite<true>(par, i, sw_forward(i, mu, P.L, P.dim), P.err);
}

__global__ void __launch_bounds__(256) k_sw_flip(const __grid_constant__ SwLaunch P) {
    chain_begin();
    const uint64_t copy = P.copy0 + blockIdx.y;
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    uint32_t* par = P.parent + copy * P.N;
    const uint32_t root = sw_find<true>(par, i);
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    const uint4 w = philox4x32_10(make_uint4(root >> 2, P.t, r, c3_word(kPurposeSwFlip, 0u, P.inst_base + inst)),
                                  (uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    const uint32_t word = (root & 3u) == 0 ? w.x : (root & 3u) == 1 ? w.y : (root & 3u) == 2 ? w.z : w.w;
    if (word >> 31) P.spins[copy * P.N + i] = (int8_t)(-P.spins[copy * P.N + i]);
    if (P.labels) P.labels[copy * P.N + i] = (int32_t)root;
}

__device__ __forceinline__ uint32_t sw_coin(const PhiloxFixed& pf, uint32_t root) {
    const uint4 w = philox_q_wide(pf, root >> 2);
    const uint32_t word = (root & 3u) == 0 ? w.x : (root & 3u) == 1 ? w.y : (root & 3u) == 2 ? w.z : w.w;
    return word >> 31;
}

__global__ void __launch_bounds__(256) k_sw_flip_tiled(const __grid_constant__ SwLaunch P) {
    chain_begin();
    __shared__ uint32_t tpar[1024];   // the tile's parent pointers (global site indices)
    __shared__ uint32_t troot[1024];  // root of each end node
    __shared__ uint8_t tcoin[1024];   // its coin (1: the cluster flips)
    __shared__ uint32_t tqueue[8][128];  // per warp: its end nodes (local indices)
    const uint64_t copy = P.copy0 + blockIdx.y;
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    const SwTile T = sw_tile(P.dim);
    const uint32_t L = P.L, ntx = L / T.tx, nty = L / T.ty;
    const uint32_t bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % nty, bz = blockIdx.x / (ntx * nty);
    const uint32_t l0 = 4 * threadIdx.x;
    const uint32_t lx = l0 % T.tx, ly = (l0 / T.tx) % T.ty, lz = l0 / (T.tx * T.ty);
    const uint32_t i0 = ((bz * T.tz + lz) * L + by * T.ty + ly) * L + bx * T.tx + lx;
    uint32_t* par = P.parent + copy * P.N;
    const uint4 p4 = __ldcg(reinterpret_cast<const uint4*>(par + i0));
    tpar[l0] = p4.x;
    tpar[l0 + 1] = p4.y;
    tpar[l0 + 2] = p4.z;
    tpar[l0 + 3] = p4.w;
    __syncthreads();
    // each site's chain inside the tile (pointers strictly decrease until a
    // root, so at most 1024 steps) ends at node `end`: a root, or a node whose
    // parent lies in another tile
    uint32_t end[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t cl = l0 + k, cg = i0 + k;
        for (uint32_t n = 0; n < 1024; ++n) {
            const uint32_t p = tpar[cl];
            if (p == cg) break;
            uint32_t px, py, pz;
            if (P.lshift) {  // L = 2^lshift
                px = p & (L - 1);
                py = (p >> P.lshift) & (L - 1);
                pz = p >> (2 * P.lshift);
            } else {
                const uint32_t row = p / L;
                px = p - row * L;
                py = row % L;
                pz = row / L;
            }
            if (px / T.tx != bx || py / T.ty != by || pz / T.tz != bz) break;
            cl = ((pz - bz * T.tz) * T.ty + (py - by * T.ty)) * T.tx + (px - bx * T.tx);
            cg = p;
        }
        end[k] = cl;
    }
    // end nodes: the root in the global forest and its coin, through a per-warp
    // queue so that every lane works on one end node at a time
    const PhiloxFixed pf = philox_fix(P.t, r, c3_word(kPurposeSwFlip, 0u, P.inst_base + inst), (uint32_t)P.seed,
                                      (uint32_t)(P.seed >> 32));
    uint32_t* q = tqueue[threadIdx.x >> 5];
    uint32_t n = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) sw_warp_push(q, n, end[k] == l0 + k, l0 + k);
    __syncwarp();
    for (uint32_t i = threadIdx.x & 31u; i < n; i += 32u) {
        const uint32_t l = q[i];
        const uint32_t ex = l % T.tx, ey = (l / T.tx) % T.ty, ez = l / (T.tx * T.ty);
        const uint32_t gl = ((bz * T.tz + ez) * L + by * T.ty + ey) * L + bx * T.tx + ex;  // its global index
        const uint32_t p = tpar[l];
        const uint32_t root = p == gl ? p : sw_find<true>(par, p);
        troot[l] = root;
        tcoin[l] = (uint8_t)sw_coin(pf, root);
    }
    __syncthreads();
    // i0 % 4 == 0 and the spin buffer is 16-byte aligned: one word per thread
    uint32_t* sw = reinterpret_cast<uint32_t*>(P.spins + copy * P.N + i0);
    uint32_t w = *sw;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!tcoin[end[k]]) continue;
        const uint32_t b = (uint32_t)(uint8_t)(-(int8_t)(w >> (8 * k)));
        w = (w & ~(0xFFu << (8 * k))) | (b << (8 * k));
    }
    *sw = w;
    if (P.labels) {
#pragma unroll
        for (int k = 0; k < 4; ++k) P.labels[copy * P.N + i0 + k] = (int32_t)troot[end[k]];
    }
}

// QUADS (L % 4 = 0): a thread has four sites of a row, loaded and stored together (1 us of 10 at
// L = 1024); else four rows' sites of a column.
template <bool QUADS>
__global__ void __launch_bounds__(256) k_sw_flip_lab(const __grid_constant__ SwLaunch P) {
    chain_begin();
    __shared__ uint32_t troot[1024];     // global root of each tile root (by local index)
    __shared__ uint8_t tcoin[1024];      // its coin (1: the cluster flips)
    __shared__ uint32_t tqueue[8][128];  // per warp: its tile roots (local indices)
    __shared__ uint32_t tedge[32];       // the tile roots whose component touches the tile border
    const uint64_t copy = P.copy0 + blockIdx.y;
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    const uint32_t L = P.L, ntx = (L + 31u) >> 5;
    const uint32_t bx = blockIdx.x % ntx, by = blockIdx.x / ntx;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t lx = QUADS ? 4u * (threadIdx.x & 7u) : lane, ly = QUADS ? threadIdx.x >> 3 : 4u * (threadIdx.x >> 5);
    auto x = [&](uint32_t j) { return lx + (QUADS ? j : 0u); };  // of site j within the tile
    auto y = [&](uint32_t j) { return ly + (QUADS ? 0u : j); };
    const uint32_t X = bx * 32u + lx, Y = by * 32u + ly, i0 = Y * L + X, step = QUADS ? 1u : L;
    const uint16_t* lab = P.lab + copy * P.N;
    int8_t* s = P.spins + copy * P.N;
    bool on[4];
    uint32_t k[4], quad = 0u;
    int8_t sp[4];
    if constexpr (QUADS) {
        const bool in = X < L && Y < L;
        // i0 % 4 == 0, the label buffer is a cudaMalloc block and the spin buffer 16-byte
        // aligned: one word each
        const uint2 lv = in ? *reinterpret_cast<const uint2*>(lab + GBMC_IDX(i0, P.N)) : make_uint2(0u, 0u);
        if (in) quad = *reinterpret_cast<const uint32_t*>(s + i0);
        k[0] = lv.x & 0xFFFFu, k[1] = lv.x >> 16, k[2] = lv.y & 0xFFFFu, k[3] = lv.y >> 16;
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
            on[j] = in;
            if (!in) k[j] = 0xFFFFFFFFu;
        }
    } else {
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
            on[j] = X < L && Y + j < L;
            k[j] = on[j] ? lab[GBMC_IDX(i0 + j * L, P.N)] : 0xFFFFFFFFu;
            sp[j] = on[j] ? s[i0 + j * L] : (int8_t)0;
        }
    }
    // the tile roots whose component has a site on the tile border: only
    // they can have been united with other tiles' components
    if (threadIdx.x < 32u) tedge[threadIdx.x] = 0u;
    __syncthreads();
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j)
        if (on[j] && (x(j) == 0u || x(j) == 31u || bx * 32u + x(j) + 1u == L || y(j) == 0u || y(j) == 31u ||
                      by * 32u + y(j) + 1u == L))
            atomicOr(&tedge[k[j] >> 5], 1u << (k[j] & 31u));
    __syncthreads();
    // the tile roots: their global root and coin, through a per-warp queue so
    // that every lane works on one at a time
    const PhiloxFixed pf = philox_fix(P.t, r, c3_word(kPurposeSwFlip, 0u, P.inst_base + inst), (uint32_t)P.seed,
                                      (uint32_t)(P.seed >> 32));
    uint32_t* par = P.parent + copy * P.N;
    uint32_t* q = tqueue[threadIdx.x >> 5];
    uint32_t n = 0;
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
        const uint32_t l = 32u * y(j) + x(j);
        sw_warp_push(q, n, k[j] == l, l);
    }
    __syncwarp();
    for (uint32_t a = lane; a < n; a += 32u) {
        const uint32_t l = q[a];
        const uint32_t g = (by * 32u + (l >> 5)) * L + bx * 32u + (l & 31u);
        // a component away from the tile border is a whole cluster, rooted at g
        const uint32_t root = ((tedge[l >> 5] >> (l & 31u)) & 1u) ? sw_find<true>(par, g) : g;
        troot[l] = root;
        tcoin[l] = (uint8_t)sw_coin(pf, root);
    }
    __syncthreads();
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
        if (!on[j]) continue;
        if (tcoin[GBMC_IDX(k[j], 1024u)]) {
            if constexpr (QUADS) {
                const uint32_t b = (uint32_t)(uint8_t)(-(int8_t)(quad >> (8 * j)));
                quad = (quad & ~(0xFFu << (8 * j))) | (b << (8 * j));
            } else {
                s[i0 + j * L] = (int8_t)(-sp[j]);
            }
        }
        if (P.labels) P.labels[copy * P.N + i0 + j * step] = (int32_t)troot[k[j]];
    }
    if (QUADS && on[0]) *reinterpret_cast<uint32_t*>(s + i0) = quad;
}

// ---- lattices that fit in one block's shared memory ----

// Shared memory of k_sw_resident: every site's label, then bit masks over the sites: spins
// (1: down; the first four again behind the last), bonds to the right within a row, around a
// row's end, along y and z, coins.
__host__ __device__ __forceinline__ uint32_t sw_mask_words(uint32_t N) { return N / 32u + 2u; }
__host__ __device__ __forceinline__ uint32_t sw_resident_words(uint32_t N, uint32_t dim) {
    return N + (3u + dim) * sw_mask_words(N);
}

// All updates of a call, one block per copy. A thread takes four consecutive sites (one
// Philox call covers their coins, DIM their bonds); eight lanes' nibbles make a mask word.
// Labels start at the first site of each run of bonds along x. Then in rounds: each
// bond whose ends' labels differ lowers the larger label's own label to the smaller one,
// and all labels follow theirs to the end of the chain, until no bond's ends differ. A link
// that a second bond's overwrites is found again in the next round, as its bond's ends still
// differ; every round hooks all labels but the smallest among their neighbours.
template <uint32_t DIM>
__global__ void __launch_bounds__(1024, 1) k_sw_resident(const __grid_constant__ SwLaunch P, uint32_t n_updates,
                                                        uint64_t copies, int32_t* E_series, int32_t* M_series) {
    extern __shared__ __align__(16) uint32_t f[];  // the labels
    __shared__ int red[2];                         // unsatisfied bonds, down spins
    constexpr uint32_t kAll = 0xffffffffu;
    const uint32_t N = P.N, L = P.L, LL = L * L, Q = N / 4u, W = sw_mask_words(N);
    uint32_t* const spin = f + N;
    uint32_t* const right = spin + W;
    uint32_t* const around = right + W;
    uint32_t* const along = around + W;               // [DIM - 1][W]
    uint32_t* const coin = along + (DIM - 1u) * W;
    const uint64_t copy = P.copy0 + blockIdx.x;
    int8_t* s = P.spins + copy * N;
    uint32_t inst, r;
    split_copy(copy, P.R, inst, r);
    const uint32_t k0 = (uint32_t)P.seed, k1 = (uint32_t)(P.seed >> 32);
    const uint32_t lane = threadIdx.x & 31u;
    // quotients by L: exact, as the numerators times L stay below 2^32
    const uint32_t inv = 0xFFFFFFFFu / L + 1u;
    auto nibble_of = [&](const uint32_t* m, uint32_t q) { return (m[GBMC_IDX(q >> 3, W)] >> (4u * (q & 7u))) & 15u; };
    // the nibbles of eight lanes to a word of m, nq quads in all (whole warps; q: the lane's)
    auto store = [&](uint32_t* m, uint32_t q, uint32_t nq, uint32_t nibble) {
        uint32_t v = q < nq ? nibble << (4u * (lane & 7u)) : 0u;
#pragma unroll
        for (uint32_t o = 1; o < 8u; o <<= 1) v |= __shfl_xor_sync(kAll, v, o);
        if ((lane & 7u) == 0u && q < nq) m[GBMC_IDX(q >> 3, W)] = v;
    };
    const uint32_t T = blockDim.x, Qr = (Q + 1u + 31u) & ~31u;  // whole warps over the quads and one more
    for (uint32_t q = threadIdx.x; q < Qr; q += T) {
        const uint32_t w = q <= Q ? *reinterpret_cast<const uint32_t*>(s + 4u * (q < Q ? q : 0u)) : 0u;
        const uint32_t neg = (w >> 7) & 0x01010101u;  // -1 bytes
        store(spin, q, Q + 1u, (neg * 0x01020408u) >> 24);
    }
    if (threadIdx.x < 2u) red[threadIdx.x] = 0;
    __syncthreads();
    const bool series = E_series || M_series;
    const uint32_t Tb = (uint32_t)P.T_bond;
    for (uint32_t u = 0; u <= n_updates; ++u) {
        const bool update = u < n_updates, measure = u > 0u && series;
        if (!update && !measure) break;
        // bonds, and E and M of the update before
        const PhiloxFixed pb = philox_fix(P.t + u, r, c3_word(kPurposeSwBond, 0u, P.inst_base + inst), k0, k1);
        int unsat = 0, down = 0;
        for (uint32_t q = threadIdx.x; q < Qr; q += T) {
            uint32_t act[DIM], ends = 0u;
#pragma unroll
            for (uint32_t mu = 0; mu < DIM; ++mu) act[mu] = 0u;
            if (q < Q) {
                const uint32_t i0 = 4u * q, row = __umulhi(i0, inv), x = i0 - row * L;
                auto window = [&](uint32_t p) {  // four bits of the spins from site p (cyclic)
                    p = p >= N ? p - N : p;
                    return __funnelshift_r(spin[GBMC_IDX(p >> 5, W)], spin[GBMC_IDX((p >> 5) + 1u, W)], p & 31u);
                };
                const uint32_t at = window(i0), own = at & 15u;
                uint32_t dif[DIM];
                dif[0] = own ^ ((at >> 1) & 15u);
                const uint32_t e = L - 1u - x;  // the row's end, if among the four
                if (e < 4u) {
                    ends = 1u << e;
                    const uint32_t first = row * L;
                    dif[0] = (dif[0] & ~ends) | ((((own >> e) ^ (spin[first >> 5] >> (first & 31u))) & 1u) << e);
                }
                uint32_t below = window(i0 + L);
                if constexpr (DIM == 3) {
                    // sites of a layer's last row go around to its first: the whole quad, or
                    // (L % 4 = 2) the part of it before or after a row's end
                    const uint32_t y = row - __umulhi(row, inv) * L, head = e < 3u ? (2u << e) - 1u : 15u;
                    const uint32_t last = (y + 1u == L ? head : 0u) | (y + 2u == L ? ~head & 15u : 0u);
                    if (last) below = (below & ~last) | (window(i0 + L + N - LL) & last);
                    dif[2] = own ^ (window(i0 + LL) & 15u);
                }
                dif[1] = own ^ (below & 15u);
                down += __popc(own);
#pragma unroll
                for (uint32_t mu = 0; mu < DIM; ++mu) unsat += __popc(dif[mu]);
                if (update && P.T_bond >= 0) {
#pragma unroll
                    for (uint32_t c = 0; c < DIM; ++c) {
                        const uint4 w = philox_q_wide(pb, DIM * q + c);
#pragma unroll
                        for (uint32_t k = 0; k < 4u; ++k) {
                            const uint32_t n = (4u * c + k) / DIM, mu = (4u * c + k) % DIM;
                            const uint32_t v = k == 0u ? w.x : k == 1u ? w.y : k == 2u ? w.z : w.w;
                            if (v <= Tb) act[mu] |= 1u << n;
                        }
                    }
#pragma unroll
                    for (uint32_t mu = 0; mu < DIM; ++mu) act[mu] &= ~dif[mu];
                }
            }
            if (update) {
                store(right, q, Q, act[0] & ~ends);
                store(around, q, Q, act[0] & ends);
#pragma unroll
                for (uint32_t mu = 1; mu < DIM; ++mu) store(along + (mu - 1u) * W, q, Q, act[mu]);
            }
        }
        if (measure) {
            unsat = __reduce_add_sync(kAll, unsat);
            down = __reduce_add_sync(kAll, down);
            if (lane == 0u) {
                atomicAdd(red, unsat);
                atomicAdd(red + 1, down);
            }
        }
        __syncthreads();
        if (measure && threadIdx.x == 0u) {
            const uint64_t to = GBMC_IDX((uint64_t)(u - 1u) * copies + copy, n_updates * copies);
            if (E_series) E_series[to] = 2 * red[0] - (int)(DIM * N);
            if (M_series) M_series[to] = (int)N - 2 * red[1];
            red[0] = red[1] = 0;  // next added to after two barriers
        }
        if (!update) break;
        for (uint32_t q = threadIdx.x; q < Q; q += T) {
            const uint32_t i0 = 4u * q;
            uint32_t w = i0 >> 5, start = 0u;
            uint32_t open = ~right[w] & ((1u << (i0 & 31u)) - 1u);  // sites below i0 not bonded to the next
            while (!open && w) open = ~right[--w];
            if (open) start = 32u * w + 32u - (uint32_t)__clz(open);
            const uint32_t joined = right[i0 >> 5] >> (i0 & 31u);
            uint4 v;
            v.x = start;
            v.y = (joined & 1u) ? v.x : i0 + 1u;
            v.z = (joined & 2u) ? v.y : i0 + 2u;
            v.w = (joined & 4u) ? v.z : i0 + 3u;
            *reinterpret_cast<uint4*>(f + GBMC_IDX(i0, N - 3u)) = v;
        }
        __syncthreads();
        for (;;) {
            bool differ = false;
            for (uint32_t q = threadIdx.x; q < Qr; q += T) {
                const uint32_t i0 = 4u * q;
                uint32_t on[DIM], any = 0u;
                const uint32_t qm = min(q, Q);  // (the masks end there)
                on[0] = nibble_of(around, qm);
#pragma unroll
                for (uint32_t mu = 1; mu < DIM; ++mu) on[mu] = nibble_of(along + (mu - 1u) * W, qm);
#pragma unroll
                for (uint32_t mu = 0; mu < DIM; ++mu) {
                    if (q >= Q) on[mu] = 0u;
                    any |= on[mu];
                }
                if (!__any_sync(kAll, any != 0u)) continue;  // whole warps
                uint32_t done[DIM];  // bonds whose ends have one label: out of the rounds to come
#pragma unroll
                for (uint32_t mu = 0; mu < DIM; ++mu) done[mu] = 0u;
                if (any) {
                    const uint32_t row = __umulhi(i0, inv), x = i0 - row * L;
                    const uint32_t y = DIM == 3 ? row - __umulhi(row, inv) * L : 0u;
                    const uint4 v = *reinterpret_cast<const uint4*>(f + i0);
                    const uint32_t own[4] = {v.x, v.y, v.z, v.w};
                    // one direction's bonds together: their far ends' labels, then the larger
                    // labels' own, then the links (most of a large cluster's are made already)
                    volatile uint32_t* vf = f;
                    auto join = [&](uint32_t mu, const uint32_t (&far)[4]) {
                        uint32_t lo[4], hi[4], now[4];
#pragma unroll
                        for (uint32_t n = 0; n < 4u; ++n) {
                            const uint32_t b = (on[mu] >> n) & 1u ? vf[GBMC_IDX(far[n], N)] : own[n];
                            lo[n] = min(own[n], b);
                            hi[n] = max(own[n], b);
                        }
#pragma unroll
                        for (uint32_t n = 0; n < 4u; ++n) now[n] = vf[GBMC_IDX(hi[n], N)];
#pragma unroll
                        for (uint32_t n = 0; n < 4u; ++n) {
                            if (lo[n] == hi[n]) done[mu] |= on[mu] & (1u << n);
                            else differ = true;
                            if (lo[n] < now[n] && lo[n] != hi[n]) atomicMin(f + hi[n], lo[n]);
                        }
                    };
                    uint32_t far[4];
#pragma unroll
                    for (uint32_t n = 0; n < 4u; ++n) {
                        uint32_t j = i0 + n + L;
                        if constexpr (DIM == 2) j -= j >= N ? N : 0u;
                        else if ((x + n >= L ? (y + 1u == L ? 0u : y + 1u) : y) + 1u == L) j -= LL;
                        far[n] = j;
                    }
                    if (on[1]) join(1u, far);
                    if constexpr (DIM == 3) {
#pragma unroll
                        for (uint32_t n = 0; n < 4u; ++n) far[n] = i0 + n + LL >= N ? i0 + n + LL - N : i0 + n + LL;
                        if (on[2]) join(2u, far);
                    }
                    if (on[0]) {
#pragma unroll
                        for (uint32_t n = 0; n < 4u; ++n) far[n] = row * L;  // (the one bond's row begins there)
                        join(0u, far);
                    }
                }
#pragma unroll
                for (uint32_t mu = 0; mu < DIM; ++mu)
                    if (__any_sync(kAll, done[mu] != 0u))
                        store(mu ? along + (mu - 1u) * W : around, q, Q, on[mu] & ~done[mu]);
            }
            if (!__syncthreads_or(differ)) break;
            for (uint32_t q = threadIdx.x; q < Q; q += T) {
                volatile uint32_t* l = f + 4u * q;
                uint32_t a0 = l[0], a1 = l[1], a2 = l[2], a3 = l[3];
                for (;;) {  // every label follows its own, and is itself what others follow
                    volatile uint32_t* vf = f;
                    const uint32_t b0 = vf[GBMC_IDX(a0, N)], b1 = vf[GBMC_IDX(a1, N)], b2 = vf[GBMC_IDX(a2, N)],
                                   b3 = vf[GBMC_IDX(a3, N)];
                    if (b0 == a0 && b1 == a1 && b2 == a2 && b3 == a3) break;
                    l[0] = a0 = b0, l[1] = a1 = b1, l[2] = a2 = b2, l[3] = a3 = b3;
                }
            }
            __syncthreads();
        }
        const PhiloxFixed pf = philox_fix(P.t + u, r, c3_word(kPurposeSwFlip, 0u, P.inst_base + inst), k0, k1);
        for (uint32_t q = threadIdx.x; q < Qr; q += T) {
            uint32_t up = 0u;
            if (q < Q) {
                const uint4 v = *reinterpret_cast<const uint4*>(f + 4u * q);
                if (v.x == 4u * q || v.y == 4u * q + 1u || v.z == 4u * q + 2u || v.w == 4u * q + 3u) {
                    const uint4 w = philox_q_wide(pf, q);
                    up = (w.x >> 31) | (w.y >> 31) << 1 | (w.z >> 31) << 2 | (w.w >> 31) << 3;
                }
            }
            store(coin, q, Q, up);
        }
        __syncthreads();
        const bool named = P.labels && u + 1u == n_updates;
        for (uint32_t q = threadIdx.x; q < Qr; q += T) {
            uint32_t now = 0u;
            if (q <= Q) {
                const uint32_t from = q < Q ? q : 0u;  // (the first quad again behind the last)
                const uint4 v = *reinterpret_cast<const uint4*>(f + 4u * from);
                auto up = [&](uint32_t root) { return (coin[GBMC_IDX(root >> 5, W)] >> (root & 31u)) & 1u; };
                now = up(v.x) | up(v.y) << 1 | up(v.z) << 2 | up(v.w) << 3;
                if (named && q < Q) {
                    int32_t* to = P.labels + copy * N + 4u * q;
                    to[0] = (int32_t)v.x, to[1] = (int32_t)v.y, to[2] = (int32_t)v.z, to[3] = (int32_t)v.w;
                }
            }
            store(right, q, Q + 1u, now);
        }
        __syncthreads();
        for (uint32_t w = threadIdx.x; w < W; w += T)
            if (w < (Q + 8u) / 8u) spin[w] ^= right[w];
        __syncthreads();
    }
    for (uint32_t q = threadIdx.x; q < Q; q += T) {
        const uint32_t b = (nibble_of(spin, q) * 0x00204081u) & 0x01010101u;  // bit n to byte n
        *reinterpret_cast<uint32_t*>(s + 4u * q) = (b * 0xFEu) | 0x01010101u;
    }
}

// One copy takes 5 us and 3.1 (2D) or 3.7 ns per site and update, one block after the other
// on a multiprocessor; three kernels over the lattice and one for E and M take 19 to 30
// us and, per site, 13 ps (2D, whole tiles) or 22 (3D) in tiles, 90 or 60 without. Measured, us
// per update, the kernels -> resident: 2D L = 16 20 -> 6, L = 64 17 -> 16 (152 copies 32 -> 17), L =
// 90 19 -> 27 (152 copies 40 -> 29), L = 128 20 -> 52; 3D L = 8 22 -> 8, L = 16 22 -> 19 (256 copies
// 51 -> 39), L = 20 30 -> 33 (152 copies 102 -> 35), L = 24 30 -> 53 (152 copies 154 -> 57).
bool sw_resident(uint32_t dim, uint32_t L, uint32_t N, uint64_t copies, bool series, int sm_count) {
    const uint32_t bytes = sw_resident_words(N, dim) * 4u;
    if (L < 4u || bytes > 224u * 1024u) return false;  // a quad holds at most one row's end
    const double held = std::min(std::floor(1024.0 / std::min(1024u, (N / 4u + 31u) & ~31u)),
                                 std::floor(228.0 * 1024.0 / (bytes + 1024.0)));
    const double each = (double)N * (dim == 2 ? 0.0031 : 0.0037), c = (double)copies;
    const double chip = std::ceil(c / sm_count) * each + 5.0 * std::ceil(c / (sm_count * held));
    const bool tiled = sw_tiled(dim, L);
    const double area = dim == 2 && tiled ? 1024.0 * ((L + 31u) / 32u) * ((L + 31u) / 32u) : (double)N;
    const double grid = (tiled ? (dim == 2 ? 19.0 : 23.0) : 26.0 + N * 4e-4) - (series ? 0.0 : 6.0) +
                        c * area * (tiled ? (dim == 2 ? 1.3e-5 : 2.2e-5) : dim == 2 ? 9e-5 : 6e-5);
    return chip < grid;
}

cudaError_t launch_sw_resident(const SwLaunch& P0, uint64_t copies, uint32_t n_updates, int32_t* E_series,
                               int32_t* M_series, cudaStream_t s) {
    if (P0.N % 4 != 0) return cudaErrorInvalidValue;
    const size_t smem = sw_resident_words(P0.N, P0.dim) * 4u;
    auto kern = P0.dim == 2 ? k_sw_resident<2> : k_sw_resident<3>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const uint32_t threads = std::min(1024u, (P0.N / 4u + 31u) & ~31u);
    // a launch is kept to some ten milliseconds
    const uint32_t most = std::max(1u, (1u << 24) / P0.N);
    for (uint64_t u = 0; u < n_updates; u += most) {  // (64 bits: u does not wrap past the last launch)
        SwLaunch P = P0;
        P.t = P0.t + (uint32_t)u;
        const uint32_t n = (uint32_t)std::min<uint64_t>(most, n_updates - u);
        if (u + n < n_updates) P.labels = nullptr;
        for (uint64_t c0 = 0; c0 < copies; c0 += 0x40000000u) {
            P.copy0 = c0;
            const uint32_t nc = (uint32_t)std::min<uint64_t>(copies - c0, 0x40000000u);
            kern<<<nc, threads, smem, s>>>(P, n, copies, E_series ? E_series + u * copies : nullptr,
                                           M_series ? M_series + u * copies : nullptr);
            count_launch();
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_sw_update(const SwLaunch& P0, uint64_t copies, cudaStream_t s) {
    if (P0.N % 4 != 0) return cudaErrorInvalidValue;
    for (uint64_t c0 = 0; c0 < copies; c0 += 65535) {
        SwLaunch P = P0;
        P.copy0 = c0;
        const uint32_t nc = (uint32_t)((copies - c0) < 65535 ? (copies - c0) : 65535);
        const uint32_t quads = P.N / 4;
        const bool tiled = sw_tiled(P.dim, P.L);
        cudaError_t e;
        if (tiled && P.dim == 2) {
            if (!P.lab) return cudaErrorInvalidValue;
            const uint32_t edge = (P.L + 31u) / 32u, tiles = edge * edge;
            e = launch_chained(k_sw_scan2, dim3(tiles, nc), 32 * kSwWarps, s, P);
            if (e != cudaSuccess) return e;
            e = launch_chained(k_sw_cross, dim3((sw_cross_count(P.N, P.L, P.dim) + 255) / 256, nc), 256, s, P);
            if (e != cudaSuccess) return e;
            if (P.L % 4 == 0) e = launch_chained(k_sw_flip_lab<true>, dim3(tiles, nc), 256, s, P);
            else e = launch_chained(k_sw_flip_lab<false>, dim3(tiles, nc), 256, s, P);
            if (e != cudaSuccess) return e;
            continue;
        }
        P.lab = nullptr;
        if (tiled) {
            e = launch_chained(k_sw_local<3>, dim3(P.N / 1024, nc), 256, s, P);
            if (e != cudaSuccess) return e;
            e = launch_chained(k_sw_cross, dim3((sw_cross_count(P.N, P.L, P.dim) + 255) / 256, nc), 256, s, P);
            if (e != cudaSuccess) return e;
            e = launch_chained(k_sw_flip_tiled, dim3(P.N / 1024, nc), 256, s, P);
            if (e != cudaSuccess) return e;
            continue;
        } else {
            if (P.dim == 2) e = launch_chained(k_sw_bonds<2>, dim3((quads + 255) / 256, nc), 256, s, P);
            else e = launch_chained(k_sw_bonds<3>, dim3((quads + 255) / 256, nc), 256, s, P);
            if (e != cudaSuccess) return e;
            e = launch_chained(k_sw_union, dim3((P.N + 255) / 256, nc), 256, s, P);
            if (e != cudaSuccess) return e;
        }
        e = launch_chained(k_sw_flip, dim3((P.N + 255) / 256, nc), 256, s, P);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace gbmc
