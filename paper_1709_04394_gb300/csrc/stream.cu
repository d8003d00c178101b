// stream.cu -- checkerboard Metropolis sweeps (Sec. 3.1, Eq. (8)) of copies held
// bit-sliced on chip for every even L, several copies per thread.
//
// A colour plane is one cyclic stream of its H = N / 2 sites in colour-rank
// order (bit k & 31 of word k >> 5; s = L / 2 ranks per row, A = s L per slab of
// a 3D lattice), whatever L is. The neighbours of the 32 sites of a word are
// then windows of the other plane's stream at offsets -s, +s (y), -A, +A (z) and
// single-bit shifts (x), with the row and slab ends taken from windows at
// +-(s - 1) and +-(A - s) under per-word masks (k_stream_tables). Reads run up
// to 31 bits past the end of the stream, so each plane keeps its first bits
// again behind its last one (stream_extend).
//
// A thread updates the same word of C copies (C = 4, 2 or 1) of one instance
// together. Window positions, masks and +-J bond words are worked out once for
// the C copies, their words lie side by side in shared memory (one 128-bit load
// for C = 4), and the Philox calls of the copies run in lockstep: they share
// the counter q, hence the products of round 0 and of round 1's second word
// (2 of 18 wide multiplies per call) and every round's key.
//
// Bound: the integer pipes together. Measured on sm_103a with independent
// instructions and eight warps per scheduler, a three-input xor or a compare
// takes 2.1 cycles of a scheduler, a wide 32 x 32 -> 64-bit multiply 4.3, and a mix
// of both 2.1 per logic instruction + 2.2 per multiply: the two do not overlap. A
// Philox call (4 sites) is 18 xors, 16.5 to 18 multiplies and 8 (2D) or 12 (3D)
// threshold compares, 92 to 95 cycles in 2D and 100 to 104 in 3D; the kernel runs at 107 to 109 (2D).
// Replacing the carry compares by predicates, or moving them to the float adder,
// left that unchanged. Site updates per ns before (byte planes; per-site loop where
// L % 8 != 0) and after, theta = 10 sweeps per load: 2D L = 24 610 -> 1392, L = 96
// 843 -> 1366, L = 10 286 -> 1110; 3D +-J L = 4 240 -> 1306, L = 10 248 -> 1272, L = 12
// 240 -> 1215, L = 32 540 -> 1319. (L = 16, 32, 64 in 2D and L = 8, 16 in 3D stay on
// bitsweep.cu, whose fixed sizes need no windows: 1475 / 1512 and 1323 / 1337 there
// against 1437 / 1486 and 1317 / 1328 here.)
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <utility>

#include <cooperative_groups.h>

#include "bits.cuh"
#include "check.cuh"
#include "copies.cuh"
#include "device.cuh"
#include "internal.h"

namespace gbmc {

namespace cg = cooperative_groups;

namespace {

constexpr uint32_t kStreamThreads = 128;      // threads per block with one-warp teams
constexpr size_t kStreamSmem = 227 * 1024;   // shared memory of an SM
static_assert(kStreamSmem < kCopySites, "record_copies: a copy that runs have is one that would fit as bytes");
constexpr uint32_t kStreamTeamWords = 3072;  // a one-warp team's share of shared memory, at most
// temperatures of the copies of a launch (kRounds: exchanged, too, round after round)
enum { kOneTemp = 0, kPerCopy = 1, kRounds = 2 };
// largest block, and blocks per SM the registers have to leave room for: 64 registers
// a thread for C = 1 and 2 (128 for S = 4 and for C = 1 in rounds), 96 for C = 4
constexpr uint32_t stream_max_threads(int C, int S, int PT = kOneTemp) {
    return C == 4 ? 128u : C == 2 || S > 1 || PT == kRounds ? 512u : 1024u;
}
constexpr uint32_t stream_min_blocks(int C) { return C == 4 ? 5u : C == 2 ? 2u : 1u; }

// Philox calls of one copy in lockstep: with fewer copies per thread more calls of
// the same copy keep as many independent chains in flight. Measured (site updates
// per ns, 2D L = 96 / 3D +-J L = 10, large populations): C = 1: 1, 4, 8 calls 1143 /
// 919, 1209 / 946, 1209 / 957; C = 2: 1, 2, 4 calls 1282 / 1097, 1230 / 1136, 1333 /
// 1163; C = 4: 1 call (loop unrolled twice), 2 calls 1309 / 1270, 1296 / 1223.
constexpr int stream_calls(int C) { return C == 4 ? 1 : 8 / C; }

// C words (one per copy) loaded and stored together.
template <int C>
struct alignas(4 * C) Words {
    uint32_t v[C];
};

struct StreamShape {
    uint32_t L, s, A, H, PW, PWX;
    uint32_t mh, h;  // valid bits of the last word: mask and count (1..32)
};

template <int DIM>
__device__ __forceinline__ StreamShape stream_shape(uint32_t L, uint32_t N) {
    StreamShape g;
    g.L = L;
    g.s = L >> 1;
    g.A = DIM == 3 ? g.s * L : 0u;
    g.H = N >> 1;
    g.PW = (g.H + 31u) >> 5;
    g.PWX = g.PW + 1u;
    g.h = ((g.H - 1u) & 31u) + 1u;
    g.mh = 0xFFFFFFFFu >> (32u - g.h);
    return g;
}

// 32 bits of a stream from bit p: the two words that hold them.
template <int C>
struct Window {
    Words<C> a, b;
    uint32_t sh;
    __device__ __forceinline__ void load(const Words<C>* pl, uint32_t p, uint32_t n_words) {
        const uint32_t i = p >> 5;
        a = pl[GBMC_IDX(i, n_words)];
        b = pl[GBMC_IDX(i + 1u, n_words)];
        sh = p & 31u;
    }
    // the window from bit p (at<0>) or p + 1 (at<1>: shift 1..32, 32 gives the upper word)
    template <int PLUS>
    __device__ __forceinline__ uint32_t at(int c) const {
        return PLUS ? __funnelshift_rc(a.v[c], b.v[c], sh + 1u) : __funnelshift_r(a.v[c], b.v[c], sh);
    }
};

__device__ __forceinline__ uint32_t sel(uint32_t m, uint32_t a, uint32_t b) { return (a & m) | (b & ~m); }

// What the update of word w reads besides spins: masks for colour 0 (odd, edge) and
// colour 1, and the windows' positions. EAGER: worked out by set() and kept (a
// thread with one word for the whole launch); else where they are used.
template <int DIM, bool EAGER>
struct Place {
    uint32_t w;
    const uint32_t* mask;
    uint32_t kept[EAGER ? (DIM == 3 ? 11 : 5) : 1];
    __device__ __forceinline__ uint32_t mask_word(const StreamShape& g, uint32_t k) const {
        return __ldg(mask + k * g.PW + w);
    }
    __device__ __forceinline__ uint32_t position(const StreamShape& g, int k) const {
        const uint32_t k0 = w << 5;
        auto wrap = [&](uint32_t p) { return p >= g.H ? p - g.H : p; };
        switch (k) {
            case 0: return k0 >= g.s ? k0 - g.s : k0 + g.H - g.s;                  // from k - s
            case 1: return wrap(k0 + g.s - 1u);                                    // from k + s - 1
            case 2: return wrap(k0 + g.A - g.s);                                   // 3D, y = 0: row L - 1 of the slab
            case 3: return k0 + g.s >= g.A ? k0 + g.s - g.A : k0 + g.s + g.H - g.A;  // y = L - 1: row 0
            case 4: return k0 >= g.A ? k0 - g.A : k0 + g.H - g.A;                  // z - 1
            default: return wrap(k0 + g.A);                                        // z + 1
        }
    }
    __device__ __forceinline__ void set(const StreamShape& g, uint32_t word, const uint32_t* m) {
        w = word;
        mask = m;
        if constexpr (EAGER) {
#pragma unroll
            for (int k = 0; k < 3; ++k) kept[k] = mask_word(g, k);
#pragma unroll
            for (int k = 0; k < (DIM == 3 ? 6 : 2); ++k) kept[3 + k] = position(g, k);
            if constexpr (DIM == 3) {
                kept[9] = mask_word(g, 3u);
                kept[10] = mask_word(g, 4u);
            }
        }
    }
    __device__ __forceinline__ uint32_t odd(const StreamShape& g, uint32_t colour) const {
        const uint32_t o = EAGER ? kept[0] : mask_word(g, 0u);
        return colour ? ~o : o;
    }
    __device__ __forceinline__ uint32_t edge(const StreamShape& g, uint32_t colour) const {
        if constexpr (EAGER) return colour ? kept[2] : kept[1];
        return mask_word(g, 1u + colour);
    }
    template <int K>
    __device__ __forceinline__ uint32_t at(const StreamShape& g) const {
        if constexpr (EAGER) return kept[3 + K];
        return position(g, K);
    }
    __device__ __forceinline__ uint32_t first_row(const StreamShape& g) const {
        if constexpr (EAGER && DIM == 3) return kept[9];
        return mask_word(g, 3u);
    }
    __device__ __forceinline__ uint32_t last_row(const StreamShape& g) const {
        if constexpr (EAGER && DIM == 3) return kept[10];
        return mask_word(g, 4u);
    }
};

// Unsatisfied-bond masks of word w of colour c: d[k][copy], k in the order
// (same-j x neighbour, other x neighbour, y - 1, y + 1, z - 1, z + 1), j the bond
// words in that order, and the other plane's word w (same).
template <int DIM, int C, bool EAGER>
__device__ __forceinline__ void stream_unsat(const StreamShape& g, const Words<C>* oth, const Words<C>& own,
                                             const Place<DIM, EAGER>& at, uint32_t colour,
                                             const uint32_t (&j)[2 * DIM],
                                             uint32_t d[2 * DIM][C], Words<C>& same) {
    const uint32_t w = at.w;
    const uint32_t odd = at.odd(g, colour), edge = at.edge(g, colour);
    Window<C> up, dn;
    up.load(oth, at.template at<0>(g), g.PWX);
    dn.load(oth, at.template at<1>(g), g.PWX);
    same = oth[GBMC_IDX(w, g.PWX)];
    {
        const Words<C> prv = oth[w ? w - 1u : 0u];  // bit 0 of word 0 starts a row: its edge window is taken
        const Words<C> nxt = oth[GBMC_IDX(w + 1u, g.PWX)];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            // the x neighbour not sharing j: j + 1 for odd x, j - 1 for even x; at
            // the row's end the first (k - (s - 1)), resp. last (k + s - 1) site of the row
            const uint32_t to_next = sel(edge, up.template at<1>(c), __funnelshift_r(same.v[c], nxt.v[c], 1));
            const uint32_t to_prev = sel(edge, dn.template at<0>(c), __funnelshift_l(prv.v[c], same.v[c], 1));
            d[0][c] = own.v[c] ^ same.v[c] ^ j[0];
            d[1][c] = own.v[c] ^ sel(odd, to_next, to_prev) ^ j[1];
        }
    }
    if constexpr (DIM == 2) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            d[2][c] = own.v[c] ^ up.template at<0>(c) ^ j[2];
            d[3][c] = own.v[c] ^ dn.template at<1>(c) ^ j[3];
        }
    } else {
        const uint32_t y0 = at.first_row(g), yl = at.last_row(g);
        Window<C> a, b;
        a.load(oth, at.template at<2>(g), g.PWX);  // y = 0: row L - 1 of the slab
        b.load(oth, at.template at<3>(g), g.PWX);  // y = L - 1: row 0
#pragma unroll
        for (int c = 0; c < C; ++c) {
            d[2][c] = own.v[c] ^ sel(y0, a.template at<0>(c), up.template at<0>(c)) ^ j[2];
            d[3][c] = own.v[c] ^ sel(yl, b.template at<0>(c), dn.template at<1>(c)) ^ j[3];
        }
        a.load(oth, at.template at<4>(g), g.PWX);
        b.load(oth, at.template at<5>(g), g.PWX);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            d[4][c] = own.v[c] ^ a.template at<0>(c) ^ j[4];
            d[5][c] = own.v[c] ^ b.template at<0>(c) ^ j[5];
        }
    }
}

// Philox constants of one copy: round 1 before the q-dependent words.
struct CopyKey {
    uint32_t b1, u1, v1;
};

// Thread teams: one warp each, or the whole block for copies too large for a warp's share.
__device__ __forceinline__ void team_sync(bool warp) {
    if (warp) __syncwarp();
    else __syncthreads();
}

// First bits of each plane again behind its last one.
template <int C>
__device__ __forceinline__ void stream_extend(uint32_t* plane, uint32_t n, const StreamShape& g, uint32_t tl,
                                              uint32_t T) {
    for (uint32_t i = tl; i < n * C; i += T) {
        uint32_t* p = plane + (i / C) * g.PWX * C + i % C;
        const uint32_t tail = p[(g.PW - 1u) * C] & g.mh;
        const uint64_t e = tail | ((uint64_t)(g.PW == 1u ? tail : p[0]) << g.h);
        p[(g.PW - 1u) * C] = (uint32_t)e;
        p[g.PW * C] = (uint32_t)(e >> 32);
    }
}

// A team of T threads (a warp, or the block) sweeps G groups of C copies;
// item i of its n_groups * PW words is word i % PW of group i / PW. S = 4 or 2 (C = 1
// only): so many threads per word, each the sites of a byte or half of it (two or four
// Philox calls), for launches too small to give every scheduler two warps.
//
// PT = kRounds: X.rounds rounds of parallel tempering. The copies of an instance are
// divided over the blocks of one cluster and stay there; after a round's sweeps every
// block receives all their energies, works out all exchanges for itself and takes its
// copies' new thresholds. Against a sweep and an exchange launch per round: 3D +-J L = 8,
// 128 x 32 copies, 10 sweeps per round 34 -> 27 us per round, 1 x 32 copies 28
// -> 10.
template <int DIM, bool EA, int C, int S, int PT>
__global__ void __launch_bounds__(stream_max_threads(C, S, PT), stream_min_blocks(C))
    k_sweep_stream(const __grid_constant__ SweepLaunch P, const __grid_constant__ PtExchange X, uint32_t smem_words) {
    extern __shared__ __align__(16) uint32_t smw[];
    int jid = 0;
    while (jid + 1 < P.njobs && blockIdx.x >= P.cta_begin[jid + 1]) ++jid;
    const SweepJob& J = P.jobs[jid];
    const uint32_t T = J.team, G = J.rpc;
    const bool warp = T == 32u;
    const uint32_t tib = warp ? threadIdx.x >> 5 : 0u, tl = warp ? threadIdx.x & 31u : threadIdx.x;
    const uint32_t ng = J.ctas_per_inst;  // groups per instance
    const uint32_t n_all = J.n_inst * ng;
    uint64_t first = ((uint64_t)(blockIdx.x - P.cta_begin[jid]) * (blockDim.x / T) + tib) * G;
    if (first >= n_all && PT != kRounds) return;  // the whole team; teams share no barrier
    uint32_t n = min(G, n_all - (uint32_t)first);
    uint32_t rank = 0, n_blocks = 1;
    if constexpr (PT == kRounds) {  // the last blocks of a cluster may have no copies
        rank = cg::this_cluster().block_rank();
        n_blocks = cg::this_cluster().num_blocks();
        const uint32_t lo = min(ng, (rank * (blockDim.x / T) + tib) * G);
        first = (uint64_t)(blockIdx.x / n_blocks) * ng + lo;
        n = min(G, ng - lo);
    }
    const StreamShape g = stream_shape<DIM>(J.L, J.N);
    // shared memory of the team: planes [colour][group][word][copy], then per
    // group [instance, first replica, active copies] and per copy [U, D], the
    // replica it is read from and (tempering) its thresholds
    uint32_t* const sm = smw + tib * smem_words;
    const uint32_t plane = G * g.PWX * C;
    uint32_t* const meta = sm + 2u * plane;
    int* const acc = reinterpret_cast<int*>(meta + 3u * G);
    uint32_t* const sfrom = meta + 3u * G + 2u * G * C;
    uint32_t* const sthr = sfrom + G * C;
    // rounds of tempering: the instance's maps, accepted swaps and (by round parity) energies
    uint32_t* const srep = smw + (blockDim.x / T) * smem_words;
    uint32_t* const stmp = srep + J.R;
    uint32_t* const sacc = stmp + J.R;
    int* const sE = reinterpret_cast<int*>(sacc + J.R);
    if constexpr (PT == kRounds) {
        const uint64_t base = (uint64_t)(blockIdx.x / n_blocks) * J.R;
        for (uint32_t k = threadIdx.x; k < J.R; k += blockDim.x) {
            srep[k] = X.rep_of[base + k];
            stmp[k] = X.temp_of[base + k];
            sacc[k] = 0u;
        }
        cg::this_cluster().barrier_arrive();
    }
    uint32_t any = 0;
    for (uint32_t gi = tl; gi < n; gi += T) {
        const uint32_t grp = (uint32_t)first + gi, inst = grp / ng, r0 = (grp - inst * ng) * C;
        // variable populations: only the first nlive[inst] slots hold replicas
        const uint32_t live = J.nlive ? J.nlive[inst] : J.R;
        const uint32_t na = r0 < live ? min((uint32_t)C, live - r0) : 0u;
        meta[3u * gi] = inst;
        meta[3u * gi + 1u] = r0;
        meta[3u * gi + 2u] = na;
        any |= na;
        for (uint32_t c = 0; c < C; ++c) {
            acc[2u * (gi * C + c)] = acc[2u * (gi * C + c) + 1u] = 0;
            if (c < na) sfrom[gi * C + c] = J.parent ? J.parent[(uint64_t)inst * J.R + r0 + c] : r0 + c;
            if (PT && c < na) {
                const uint32_t* th = J.thr_temp + 3ull * J.temp_of[(uint64_t)inst * J.R + r0 + c];
                for (uint32_t k = 0; k < 3; ++k) sthr[3u * (gi * C + c) + k] = th[k];
            } else if (PT) {
                for (uint32_t k = 0; k < 3; ++k) sthr[3u * (gi * C + c) + k] = 0u;
            }
        }
    }
    if constexpr (PT == kRounds) {
        cg::this_cluster().barrier_wait();  // all have started, and read the maps
    } else if (warp ? !__any_sync(0xFFFFFFFFu, any != 0u) : !__syncthreads_or(any != 0u)) {
        return;
    }
    team_sync(warp);

    const uint32_t* mask = J.smask;
    const uint8_t* odd_b = reinterpret_cast<const uint8_t*>(mask);
    // ---- load: 16 sites in row-major order are 8 pairs (even x, odd x) = byte ch
    // of the streams of even-x and of odd-x sites; a site of the even-x stream
    // has colour 0 where its row's colour-0 sites have even x (odd mask bit 0) ----
    const uint32_t nch = (J.N + 15u) >> 4;
    const bool wide = (J.N & 15u) == 0u;
    // four chunks per thread in flight
    for (uint32_t i0 = tl; i0 < n * C * nch; i0 += 4u * T) {
        uint4 v[4];
        uint32_t at[4], chunk[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t i = i0 + k * T, cp = i / nch, ch = i - cp * nch, gi = cp / C, c = cp % C;
            at[k] = 0xFFFFFFFFu;
            if (i >= n * C * nch || c >= meta[3u * gi + 2u]) continue;
            const uint64_t from = (uint64_t)meta[3u * gi] * J.R + sfrom[cp];
            const int8_t* src = J.src + GBMC_IDX(from, (uint64_t)J.n_inst * J.R) * J.N + 16u * ch;
            if (wide) {
                v[k] = *reinterpret_cast<const uint4*>(src);
            } else {  // copies start on 4-byte boundaries (N % 4 == 0), the last chunk is short
                const uint32_t* s4 = reinterpret_cast<const uint32_t*>(src);
                const uint32_t left = J.N - 16u * ch;
                v[k].x = s4[0];
                v[k].y = left > 4u ? s4[1] : 0u;
                v[k].z = left > 8u ? s4[2] : 0u;
                v[k].w = left > 12u ? s4[3] : 0u;
            }
            at[k] = ((GBMC_IDX(gi * g.PWX + (ch >> 2), G * g.PWX)) * C + c) * 4u + (ch & 3u);
            chunk[k] = ch;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (at[k] == 0xFFFFFFFFu) continue;
            uint32_t e0, o0, e1, o1;
            pack8(v[k].x, v[k].y, e0, o0);
            pack8(v[k].z, v[k].w, e1, o1);
            const uint32_t ev = e0 | (e1 << 4), od = o0 | (o1 << 4), m = odd_b[chunk[k]];
            uint8_t* p0 = reinterpret_cast<uint8_t*>(sm) + at[k];
            p0[0] = (uint8_t)sel(m, od, ev);
            p0[4u * plane] = (uint8_t)sel(m, ev, od);
        }
    }
    team_sync(warp);
    stream_extend<C>(sm, n, g, tl, T);
    stream_extend<C>(sm + plane, n, g, tl, T);
    team_sync(warp);

    const uint32_t k0 = (uint32_t)J.seed, k1 = (uint32_t)(J.seed >> 32);
    const bool want_final = J.E || J.M || J.hist;
    const uint32_t items = n * g.PW, nsw = J.nsweeps;
    static_assert(S == 1 || ((S == 2 || S == 4) && C == 1), "");
    constexpr int NQ = S > 1 ? 8 / S : stream_calls(C);
    constexpr uint32_t kBits = 32u / S;  // sites of a thread, and their mask in the word
    auto my_bits = [](uint32_t part) { return S > 1 ? (0xFFFFFFFFu >> (32u - kBits)) << (kBits * part) : 0xFFFFFFFFu; };
    const uint32_t NB = 2u * DIM * g.PW;  // bond words per instance and colour
    // item is -> group, copies and place; worked out once where a thread has one
    // item at most (small populations, where the chain of a half-sweep is what counts)
    uint32_t gi = 0, part = 0, inst = 0, r0 = 0;
    constexpr bool kEager = S > 1 || (C == 1 && PT == kRounds);
    Place<DIM, kEager> at;
    uint32_t jkept[PT == kRounds && EA ? 2 : 1][2 * DIM];  // bond words of both colours
    auto bonds = [&](uint32_t colour, uint32_t in, uint32_t (&j)[2 * DIM]) {
#pragma unroll
        for (int k = 0; k < 2 * DIM; ++k) {
            if constexpr (!EA) j[k] = 0u;
            else if constexpr (PT == kRounds) j[k] = colour ? jkept[1][k] : jkept[0][k];
            else j[k] = __ldg(J.sbond + ((uint64_t)in * 2u + colour) * NB + k * g.PW + at.w);
        }
    };
    auto locate = [&](uint32_t is) {
        const uint32_t i = is / S;
        part = is % S;
        gi = G == 1u ? 0u : i / g.PW;
        inst = meta[3u * gi];
        r0 = meta[3u * gi + 1u];
        at.set(g, i - gi * g.PW, mask);
        if constexpr (PT == kRounds && EA) {
#pragma unroll
            for (int k = 0; k < 2 * 2 * DIM; ++k)
                jkept[k / (2 * DIM)][k % (2 * DIM)] =
                    __ldg(J.sbond + ((uint64_t)inst * 2u + k / (2 * DIM)) * NB + (k % (2 * DIM)) * g.PW + at.w);
        }
    };
    const bool once = kEager && items * S <= T;
    if (once && tl < items * S) locate(tl);
    // adds an item's unsatisfied bonds (of colour-0 sites, d) and down spins to its
    // copies' sums: at once, or in registers first where all items are one group's
    int U[C], D[C];
    auto tally = [&](const uint32_t (&d)[2 * DIM][C], const Words<C>& p0, const Words<C>& p1, uint32_t mine) {
        const uint32_t valid = at.w + 1u == g.PW ? g.mh & mine : mine;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            int u = 0;
#pragma unroll
            for (int k = 0; k < 2 * DIM; ++k) u += __popc(d[k][c] & valid);
            const int dn = __popc(p0.v[c] & valid) + __popc(p1.v[c] & valid);
            if (G == 1u) {
                U[c] += u;
                D[c] += dn;
            } else {
                atomicAdd(acc + 2u * (gi * C + c), u);
                atomicAdd(acc + 2u * (gi * C + c) + 1u, dn);
            }
        }
    };
    auto flush = [&]() {  // whole warps
        if (G != 1u) return;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int u = __reduce_add_sync(0xFFFFFFFFu, U[c]), dn = __reduce_add_sync(0xFFFFFFFFu, D[c]);
            if ((threadIdx.x & 31u) == 0u) {
                atomicAdd(acc + 2 * c, u);
                atomicAdd(acc + 2 * c + 1, dn);
            }
        }
    };
    auto record = [&](uint32_t s, bool sweep, bool last) {
        for (uint32_t i0 = 0; i0 < n * C; i0 += T) {  // whole warps (record_copies)
            const uint32_t i = i0 + tl, gr = i < n * C ? i / C : 0u, c = i % C, ins = meta[3u * gr];
            const bool has = i < n * C && c < meta[3u * gr + 2u];
            // every bond has one colour-0 end: E = 2 (unsatisfied bonds of the colour-0 sites) - DIM N
            record_copies(J, has, (uint64_t)ins * J.R + meta[3u * gr + 1u] + c, ins, s, sweep, last,
                          has ? 2 * acc[2u * i] - DIM * (int)J.N : 0, has ? (int)J.N - 2 * acc[2u * i + 1u] : 0);
            if (i < n * C) acc[2u * i] = acc[2u * i + 1u] = 0;
        }
    };
    // Exchanges of a round of tempering, from the copies' sums
    auto exchange = [&](uint32_t round) {
        cg::cluster_group cluster = cg::this_cluster();
        int* E = sE + (round & 1u) * J.R;
        const uint32_t in = blockIdx.x / n_blocks;
        for (uint32_t i = tl; i < n * C; i += T) {
            const uint32_t gr = i / C, c = i % C, slot = meta[3u * gr + 1u] + c;
            if (c < meta[3u * gr + 2u]) {
                const int e = 2 * acc[2u * i] - DIM * (int)J.N;
                for (uint32_t b = 0; b < n_blocks; ++b) *cluster.map_shared_rank(E + slot, b) = e;
                if (round + 1u == X.rounds) {
                    J.E[(uint64_t)in * J.R + slot] = e;
                    J.M[(uint64_t)in * J.R + slot] = (int)J.N - 2 * acc[2u * i + 1u];
                }
            }
            acc[2u * i] = acc[2u * i + 1u] = 0;
        }
        cluster.sync();
        for (uint32_t k = 2u * threadIdx.x + ((X.round + round) & 1u); k + 1u < J.R; k += 2u * blockDim.x) {
            const uint32_t a = srep[k], b = srep[k + 1u];
            if (pt_accept(X, in, k, E[a], E[b], X.round + round)) {
                srep[k] = b;
                srep[k + 1u] = a;
                stmp[b] = k;
                stmp[a] = k + 1u;
                sacc[k] += 1u;
            }
        }
        __syncthreads();
        for (uint32_t i = tl; i < n * C; i += T) {
            const uint32_t gr = i / C, c = i % C;
            if (c >= meta[3u * gr + 2u]) continue;
            const uint32_t* th = J.thr_temp + 3ull * stmp[meta[3u * gr + 1u] + c];
            for (uint32_t k = 0; k < 3u; ++k) sthr[3u * i + k] = th[k];
        }
    };
#pragma unroll
    for (int c = 0; c < C; ++c) U[c] = D[c] = 0;
    const bool series = PT != kRounds && (J.Eser || J.Mser);
    for (uint32_t round = 0; round < (PT == kRounds ? X.rounds : 1u); ++round)
    for (uint32_t s = 0; s <= nsw; ++s) {
        if (s == nsw && nsw != 0) break;  // s == nsw: measurement-only pass when nothing is swept
        const bool sweep = s < nsw;
        for (uint32_t colour = 0; sweep && colour < 2; ++colour) {
            // a series' E and M after sweep s - 1 come from the words this update reads
            // (one copy per thread; with more the tallies cost more registers than the
            // pass of their own below costs time)
            const bool measure = C == 1 && series && colour == 0u && s > 0u;
            for (uint32_t is = tl; is < items * S; is += T) {
                if (!once) locate(is);
                const uint32_t w = at.w;
                Words<C>* own = reinterpret_cast<Words<C>*>(sm + colour * plane + gi * g.PWX * C);
                const Words<C>* oth = reinterpret_cast<const Words<C>*>(sm + (colour ^ 1u) * plane + gi * g.PWX * C);
                Words<C> nw = own[GBMC_IDX(w, g.PWX)];
                uint32_t ge[C], ea[C], eb[C];  // dE <= 0; dE = 4; dE = 8 (3D)
                {
                    uint32_t d[2 * DIM][C], j[2 * DIM];
                    Words<C> same;
                    bonds(colour, inst, j);
                    stream_unsat<DIM, C>(g, oth, nw, at, colour, j, d, same);
                    if (measure) tally(d, nw, same, my_bits(part));
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        if constexpr (DIM == 2) {
                            const uint32_t s1 = d[0][c] ^ d[1][c], c1 = d[0][c] & d[1][c];
                            const uint32_t s2 = d[2][c] ^ d[3][c], c2 = d[2][c] & d[3][c];
                            ge[c] = c1 | c2 | (s1 & s2);      // two or more unsatisfied bonds
                            ea[c] = (s1 ^ s2) & ~ge[c];       // one
                            eb[c] = 0u;
                        } else {
                            const uint32_t s1 = d[0][c] ^ d[1][c] ^ d[2][c], c1 = maj3(d[0][c], d[1][c], d[2][c]);
                            const uint32_t s2 = d[3][c] ^ d[4][c] ^ d[5][c], c2 = maj3(d[3][c], d[4][c], d[5][c]);
                            const uint32_t a0 = s1 ^ s2, t = s1 & s2;
                            const uint32_t a1 = c1 ^ c2 ^ t, a2 = maj3(c1, c2, t);
                            ge[c] = a2 | (a1 & a0);           // three or more
                            ea[c] = a1 & ~(a0 | a2);          // two
                            eb[c] = a0 & ~(a1 | a2);          // one
                        }
                    }
                }
                CopyKey ck[C];
                uint32_t T4[C], T8[C], T12[C];
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    uint32_t hi, lo, uh, ul;
                    mulhilo_wide(kPhiloxM1, r0 + c, hi, lo);
                    mulhilo_wide(kPhiloxM0, hi ^ (PT == kRounds ? J.t0 + round * nsw + s : J.t0 + s) ^ k0, uh, ul);
                    ck[c].b1 = lo ^ (k0 + kPhiloxW0);
                    ck[c].u1 = uh ^ (k1 + kPhiloxW1);
                    ck[c].v1 = ul;
                    T4[c] = PT ? sthr[3u * (gi * C + c)] : J.thr[0];
                    T8[c] = PT ? sthr[3u * (gi * C + c) + 1u] : J.thr[1];
                    T12[c] = PT ? sthr[3u * (gi * C + c) + 2u] : J.thr[2];
                }
                const uint32_t x0 = c3_word(kPurposeMetro, colour, J.inst_base + inst) ^ k1;
                uint32_t r4[C], r8[C], r12[C];
#pragma unroll
                for (int c = 0; c < C; ++c) r4[c] = r8[c] = r12[c] = 0u;
#pragma unroll 2
                for (uint32_t k = 0; k < 8u / S; k += NQ) {
                    const uint32_t q = 8u * w + (8u / S) * part + k;  // part: 0 where S = 1
                    uint4 v[NQ][C];
#pragma unroll
                    for (int m = 0; m < NQ; ++m) {
                        uint32_t x, y, h1, l1;  // the same for every copy
                        mulhilo_wide(kPhiloxM0, q + m, x, y);
                        mulhilo_wide(kPhiloxM1, x ^ x0, h1, l1);
#pragma unroll
                        for (int c = 0; c < C; ++c) v[m][c] = make_uint4(h1 ^ ck[c].b1, l1, ck[c].u1 ^ y, ck[c].v1);
                    }
                    uint32_t ka = k0 + 2u * kPhiloxW0, kb = k1 + 2u * kPhiloxW1;
#pragma unroll
                    for (int round = 2; round < 10; ++round) {
#pragma unroll
                        for (int m = 0; m < NQ; ++m)
#pragma unroll
                            for (int c = 0; c < C; ++c) {
                                uint4& u = v[m][c];
                                uint32_t hi0, lo0, hi1, lo1;
                                mulhilo_wide(kPhiloxM0, u.x, hi0, lo0);
                                mulhilo_wide(kPhiloxM1, u.z, hi1, lo1);
                                u = make_uint4(hi1 ^ u.y ^ ka, lo1, hi0 ^ u.w ^ kb, lo0);
                            }
                        ka += kPhiloxW0;
                        kb += kPhiloxW1;
                    }
#pragma unroll
                    for (int m = 0; m < NQ; ++m)
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const uint4 u = v[m][c];
                            if constexpr (DIM == 2) {
                                accept_bits(r4[c], r8[c], T4[c], T8[c], u.x);
                                accept_bits(r4[c], r8[c], T4[c], T8[c], u.y);
                                accept_bits(r4[c], r8[c], T4[c], T8[c], u.z);
                                accept_bits(r4[c], r8[c], T4[c], T8[c], u.w);
                            } else {
                                accept_bits3(r4[c], r8[c], r12[c], T4[c], T8[c], T12[c], u.x);
                                accept_bits3(r4[c], r8[c], r12[c], T4[c], T8[c], T12[c], u.y);
                                accept_bits3(r4[c], r8[c], r12[c], T4[c], T8[c], T12[c], u.z);
                                accept_bits3(r4[c], r8[c], r12[c], T4[c], T8[c], T12[c], u.w);
                            }
                        }
                }
                if constexpr (S > 1) {
                    const uint32_t sh = kBits * part, gb = ge[0] >> sh, ab = ea[0] >> sh, bb = eb[0] >> sh;
                    const uint32_t a4 = __brev(r4[0]) >> (32u - kBits), a8 = __brev(r8[0]) >> (32u - kBits),
                                   a12 = __brev(r12[0]) >> (32u - kBits);
                    const uint32_t f = DIM == 2 ? gb | (ab & a4) | (~(gb | ab) & a8)
                                                : gb | (ab & a4) | (bb & a8) | (~(gb | ab | bb) & a12);
                    using Part = std::conditional_t<S == 4, uint8_t, uint16_t>;
                    Part* ob = reinterpret_cast<Part*>(own) + part;
                    const Part nb = (Part)((nw.v[0] >> sh) ^ f);
                    ob[S * w] = nb;  // the other parts of the word belong to the neighbouring threads
                    if (g.h == 32u && w == 0u) ob[S * g.PW] = nb;
                } else {
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        uint32_t f;
                        if constexpr (DIM == 2)
                            f = ge[c] | (ea[c] & __brev(r4[c])) | (~(ge[c] | ea[c]) & __brev(r8[c]));
                        else
                            f = ge[c] | (ea[c] & __brev(r4[c])) | (eb[c] & __brev(r8[c])) |
                                (~(ge[c] | ea[c] | eb[c]) & __brev(r12[c]));
                        nw.v[c] ^= f;
                    }
                    own[w] = nw;
                    if (g.h == 32u && w == 0u) own[g.PW] = nw;  // whole words: the extension is word 0 again
                }
            }
            if (measure) flush();
            team_sync(warp);
            if (g.h != 32u) {
                stream_extend<C>(sm + colour * plane, n, g, tl, T);
                team_sync(warp);
            }
            if (measure) {
                record(s - 1u, true, false);  // the sums' next use is a half-sweep, and its sync, away
#pragma unroll
                for (int c = 0; c < C; ++c) U[c] = D[c] = 0;
            }
        }
        const bool last = sweep ? s + 1u == nsw : true;
        if ((last && want_final) || (series && sweep && (last || C > 1))) {
            // (a word's four threads of S = 4 count a byte each)
            constexpr uint32_t kParts = PT == kRounds ? S : 1;
            for (uint32_t is = tl; is < items * kParts; is += T) {
                if constexpr (PT == kRounds) {
                    if (!once) locate(is);
                } else {
                    gi = G == 1u ? 0u : is / g.PW;
                    inst = meta[3u * gi];
                    at.set(g, is - gi * g.PW, mask);
                }
                const Words<C>* p0 = reinterpret_cast<const Words<C>*>(sm + gi * g.PWX * C);
                const Words<C>* p1 = reinterpret_cast<const Words<C>*>(sm + plane + gi * g.PWX * C);
                const Words<C> w0 = p0[at.w];
                uint32_t d[2 * DIM][C], j[2 * DIM];
                Words<C> w1;
                bonds(0u, inst, j);
                stream_unsat<DIM, C>(g, p1, w0, at, 0u, j, d, w1);
                tally(d, w0, w1, kParts > 1u ? my_bits(part) : 0xFFFFFFFFu);
            }
            flush();
            team_sync(warp);
            if constexpr (PT == kRounds) exchange(round);
            else record(s, sweep, last);
#pragma unroll
            for (int c = 0; c < C; ++c) U[c] = D[c] = 0;
            team_sync(warp);
        }
    }

    if constexpr (PT == kRounds) {
        if (rank == 0) {
            const uint64_t in = blockIdx.x / n_blocks;
            for (uint32_t k = threadIdx.x; k < J.R; k += blockDim.x) {
                X.rep_of[in * J.R + k] = srep[k];
                X.temp_of[in * J.R + k] = stmp[k];
                if (k + 1u < J.R) X.accepted[in * (J.R - 1u) + k] += sacc[k];
            }
        }
    }

    // ---- store ----
    if (nsw > 0 || J.dst != J.src || J.parent) {
        for (uint32_t i = tl; i < n * C * nch; i += T) {
            const uint32_t cp = i / nch, ch = i - cp * nch, gi = cp / C, c = cp % C;
            if (c >= meta[3u * gi + 2u]) continue;
            const uint8_t* p0 =
                reinterpret_cast<const uint8_t*>(sm + (GBMC_IDX(gi * g.PWX + (ch >> 2), G * g.PWX)) * C + c) + (ch & 3u);
            const uint32_t a = p0[0], b = p0[4u * plane], m = odd_b[ch];
            const uint32_t ev = sel(m, b, a), od = sel(m, a, b);
            const uint2 lo = unpack8(ev & 15u, od & 15u), hi = unpack8(ev >> 4, od >> 4);
            const uint64_t slot = (uint64_t)meta[3u * gi] * J.R + meta[3u * gi + 1u] + c;
            int8_t* dst = J.dst + slot * J.N + 16u * ch;
            if (wide) {
                *reinterpret_cast<uint4*>(dst) = make_uint4(lo.x, lo.y, hi.x, hi.y);
            } else {
                uint32_t* d4 = reinterpret_cast<uint32_t*>(dst);
                const uint32_t left = J.N - 16u * ch;
                d4[0] = lo.x;
                if (left > 4u) d4[1] = lo.y;
                if (left > 8u) d4[2] = hi.x;
                if (left > 12u) d4[3] = hi.y;
            }
        }
    }
}

// ---- few copies: the acceptance bits drawn ahead of the sweeps ----
//
// A copy alone on a multiprocessor sweeps as fast as the chain of a half-sweep allows, and
// most of that chain are the ten rounds of Philox, which do not depend on the spins. One
// block per copy: its first warps (a thread per word) update, the other kDrawers warps draw
// acceptance words ahead of them into a ring in shared memory, 32 words a batch,
// whatever half-sweeps these belong to. A batch's flag says that its words are there;
// `taken` counts the half-sweeps whose words have been read. Drawers wait for room in the ring
// `naps` times at most (the caller's budget of cycles), and an updater's batch comes once its
// drawer has stopped waiting: a wait that runs out raises *err and ends all others. Test aid:
// with `phantom` the flags are that many batches behind, and the drawers see to it at the end that
// nobody waits for what will not come. (Bounds in the updaters' own loop cost the chain: by the
// clock 2D L = 16 1148 -> 1171 us, L = 64 966 -> 1041; theirs is a count far above any budget.)
//
// Bound: the chain of a half-sweep (words and masks loaded, some 25 dependent
// instructions, word stored, barrier); from some 64 words per plane the drawers' integer pipes.
// Measured, 400 sweeps with E and M, threads drawing their own words -> ahead: 2D L = 8, 9 copies
// 442 -> 237 us, L = 32, 40 copies 437 -> 267, L = 64 510 -> 394, L = 90 834 -> 526; 3D L = 4 510 ->
// 281, L = 16 590 -> 439.

constexpr uint32_t kDrawers = 12, kAheadThreads = 512;
constexpr uint32_t kAheadWords = 32u * (kAheadThreads / 32u - kDrawers);  // words per plane, at most
constexpr uint32_t kAheadPolls = 1u << 26;
constexpr uint32_t kNapCycles = 512u;  // a look at `taken` and a sleep of 200 ns, about

// items, a power of two, several half-sweeps: 1024 for all sizes taken (as a constant in the
// kernel 1 to 6 % slower)
__host__ __device__ __forceinline__ uint32_t ahead_ring(uint32_t PW) {
    uint32_t n = 1024u;
    while (n < 8u * PW) n <<= 1;
    return n;
}

template <int DIM, bool EA>
__global__ void __launch_bounds__(kAheadThreads, 1)
    k_sweep_ahead(const __grid_constant__ SweepLaunch P, unsigned int* err, uint32_t naps, uint32_t phantom) {
    extern __shared__ __align__(16) uint32_t smw[];
    __shared__ uint32_t taken, dead;  // dead: a wait ran out, nothing waits any more
    __shared__ int acc[2][2];
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    const SweepJob& J = P.jobs[0];
    const StreamShape g = stream_shape<DIM>(J.L, J.N);
    const uint32_t slot = blockIdx.x, inst = slot / J.R, r = slot - inst * J.R;
    const uint32_t tid = threadIdx.x, T = blockDim.x, lane = tid & 31u, Wc = (g.PW + 31u) / 32u;
    const uint32_t ring = ahead_ring(g.PW), k0 = (uint32_t)J.seed, k1 = (uint32_t)(J.seed >> 32);
    uint2* const m48 = reinterpret_cast<uint2*>(smw + 2u * g.PWX);  // [ring] acceptance bits of dE = 4, 8
    uint32_t* const m12 = reinterpret_cast<uint32_t*>(m48 + ring);  // (3D: 12)
    uint32_t* const flag = m12 + (DIM == 3 ? ring : 0u);
    volatile uint32_t *const vtaken = &taken, *const vdead = &dead;
    auto give_up = [&]() {
        *vdead = 1u;
        atomicExch(err, 1u);
    };

    const uint8_t* odd_b = reinterpret_cast<const uint8_t*>(J.smask);
    const uint32_t nch = (J.N + 15u) >> 4;
    const bool wide = (J.N & 15u) == 0u;
    for (uint32_t ch = tid; ch < nch; ch += T) {
        const int8_t* src = J.src + (uint64_t)slot * J.N + 16u * ch;
        uint4 v;
        if (wide) {
            v = *reinterpret_cast<const uint4*>(src);
        } else {  // copies start on 4-byte boundaries, the last chunk is short
            const uint32_t* s4 = reinterpret_cast<const uint32_t*>(src);
            const uint32_t left = J.N - 16u * ch;
            v.x = s4[0];
            v.y = left > 4u ? s4[1] : 0u;
            v.z = left > 8u ? s4[2] : 0u;
            v.w = left > 12u ? s4[3] : 0u;
        }
        uint32_t e0, o0, e1, o1;
        pack8(v.x, v.y, e0, o0);
        pack8(v.z, v.w, e1, o1);
        const uint32_t ev = e0 | (e1 << 4), od = o0 | (o1 << 4), m = odd_b[ch];
        uint8_t* p0 = reinterpret_cast<uint8_t*>(smw) + GBMC_IDX(ch, 4u * g.PWX);
        p0[0] = (uint8_t)sel(m, od, ev);
        p0[4u * g.PWX] = (uint8_t)sel(m, ev, od);
    }
    for (uint32_t i = tid; i < ring / 32u; i += T) flag[i] = 0u;
    if (tid == 0u) taken = dead = 0u;
    if (tid < 4u) acc[tid >> 1][tid & 1u] = 0;
    __syncthreads();
    stream_extend<1>(smw, 1u, g, tid, T);
    stream_extend<1>(smw + g.PWX, 1u, g, tid, T);
    __syncthreads();

    const uint32_t n_half = 2u * J.nsweeps;
    // one updating warp has its scheduler (every fourth warp's) for itself: 2D L = 16, 2000 sweeps
    // with E and M 1268 -> 1147 us
    const uint32_t warp = tid / 32u, warps = T / 32u;
    const bool spared = Wc == 1u && warp != 0u && (warp & 3u) == 0u;
    if (tid >= 32u * Wc && !spared) {
        const uint64_t items = (uint64_t)n_half * g.PW;
        const uint32_t drawers = Wc == 1u ? warps - (warps + 3u) / 4u : warps - Wc;
        for (uint64_t b = Wc == 1u ? warp - warp / 4u - 1u : warp - Wc; 32u * b < items; b += drawers) {
            const uint64_t i = 32u * b + lane, last = 32u * b + 31u;  // (the last batch may end past the items)
            // (asleep between looks: drawers far ahead would take the updaters' issue slots)
            for (uint32_t n = 0; last >= (uint64_t)*vtaken * g.PW + ring && !*vdead; ++n) {
                __nanosleep(200);
                if (n == naps) give_up();
            }
            const uint32_t h = (uint32_t)(i / g.PW), w = (uint32_t)(i - (uint64_t)h * g.PW);
            const PhiloxFixed pf = philox_fix(J.t0 + (h >> 1), r, c3_word(kPurposeMetro, h & 1u, J.inst_base + inst), k0, k1);
            uint32_t r4 = 0u, r8 = 0u, r12 = 0u;
#pragma unroll
            for (uint32_t k = 0; k < 8u; ++k) {
                const uint4 v = philox_q_wide(pf, 8u * w + k);
                if constexpr (DIM == 2) {
                    accept_bits(r4, r8, J.thr[0], J.thr[1], v.x);
                    accept_bits(r4, r8, J.thr[0], J.thr[1], v.y);
                    accept_bits(r4, r8, J.thr[0], J.thr[1], v.z);
                    accept_bits(r4, r8, J.thr[0], J.thr[1], v.w);
                } else {
                    accept_bits3(r4, r8, r12, J.thr[0], J.thr[1], J.thr[2], v.x);
                    accept_bits3(r4, r8, r12, J.thr[0], J.thr[1], J.thr[2], v.y);
                    accept_bits3(r4, r8, r12, J.thr[0], J.thr[1], J.thr[2], v.z);
                    accept_bits3(r4, r8, r12, J.thr[0], J.thr[1], J.thr[2], v.w);
                }
            }
            const uint32_t at = (uint32_t)GBMC_IDX((uint32_t)i & (ring - 1u), ring);
            m48[at] = make_uint2(__brev(r4), __brev(r8));
            if constexpr (DIM == 3) m12[at] = __brev(r12);
            __threadfence_block();
            __syncwarp();
            if (lane == 0u) *(volatile uint32_t*)(flag + GBMC_IDX((uint32_t)b & (ring / 32u - 1u), ring / 32u)) = (uint32_t)b + 1u - phantom;
        }
        if (phantom && lane == 0u)  // no more batches: what the updaters still wait for will not come
            for (uint32_t n = 0; *vtaken <= n_half && !*vdead; ++n) {
                __nanosleep(200);
                if (n == naps) give_up();
            }
        __syncwarp();
    } else if (!spared) {
        const uint32_t w = min(tid, g.PW - 1u);
        const bool has = tid < g.PW;
        Place<DIM, true> at;
        at.set(g, w, J.smask);
        uint32_t jb[2][2 * DIM];
#pragma unroll
        for (int k = 0; k < 4 * DIM; ++k)
            jb[k / (2 * DIM)][k % (2 * DIM)] =
                EA ? __ldg(J.sbond + (((uint64_t)inst * 2u + k / (2 * DIM)) * 2u * DIM + k % (2 * DIM)) * g.PW + w) : 0u;
        auto sync = [&]() {
            if (Wc == 1u) __syncwarp();
            else asm volatile("bar.sync 1, %0;" ::"r"(32u * Wc) : "memory");
        };
        uint32_t a4 = 0u, a8 = 0u, a12 = 0u;
        uint64_t known = 0;  // items below are known to be there, to this thread
        auto fetch = [&](uint32_t h) {  // this word's acceptance bits of half-sweep h
            const uint64_t i = (uint64_t)h * g.PW + w;
            if (i >= known) {
                const uint32_t b = (uint32_t)(i >> 5);
                volatile uint32_t* f = flag + GBMC_IDX(b & (ring / 32u - 1u), ring / 32u);
                for (uint32_t n = 0; *f != b + 1u && !*vdead; ++n)
                    if (n == kAheadPolls) give_up();
                __threadfence_block();
                known = (uint64_t)(b + 1u) << 5;
            }
            const uint32_t k = (uint32_t)GBMC_IDX((uint32_t)i & (ring - 1u), ring);
            const uint2 m = m48[k];
            a4 = m.x;
            a8 = m.y;
            if constexpr (DIM == 3) a12 = m12[k];
        };
        const bool series = J.Eser || J.Mser;
        const uint64_t ncopies = (uint64_t)J.n_inst * J.R;
        auto write = [&](uint32_t s, int U, int D) {  // every bond has one colour-0 end
            if (J.Eser) J.Eser[GBMC_IDX(s * ncopies + slot, J.nsweeps * ncopies)] = 2 * U - DIM * (int)J.N;
            if (J.Mser) J.Mser[GBMC_IDX(s * ncopies + slot, J.nsweeps * ncopies)] = (int)J.N - 2 * D;
        };
        if (n_half) fetch(0u);
        auto half = [&](auto colour, uint32_t h) {
            constexpr uint32_t c = decltype(colour)::value;
            const bool update = h < n_half, measure = c == 0u && series && h > 0u;
            uint32_t* const own = smw + c * g.PWX;
            const Words<1>* oth = reinterpret_cast<const Words<1>*>(smw + (c ^ 1u) * g.PWX);
            Words<1> nw = {{own[GBMC_IDX(w, g.PWX)]}}, same;
            uint32_t d[2 * DIM][1], j[2 * DIM];
#pragma unroll
            for (int k = 0; k < 2 * DIM; ++k) j[k] = EA ? jb[c][k] : 0u;
            stream_unsat<DIM, 1>(g, oth, nw, at, c, j, d, same);
            if (measure) {
                const uint32_t valid = !has ? 0u : w + 1u == g.PW ? g.mh : kAll;
                int u = 0;
#pragma unroll
                for (int k = 0; k < 2 * DIM; ++k) u += __popc(d[k][0] & valid);
                // both in one sum: a warp's down spins stay below 2^16
                const int sum = __reduce_add_sync(kAll, u << 16 | (__popc(nw.v[0] & valid) + __popc(same.v[0] & valid)));
                if (lane == 0u) {
                    if (Wc == 1u) {
                        write((h >> 1) - 1u, sum >> 16, sum & 0xFFFF);
                    } else {
                        atomicAdd(&acc[(h >> 1) & 1u][0], sum >> 16);
                        atomicAdd(&acc[(h >> 1) & 1u][1], sum & 0xFFFF);
                    }
                }
            }
            if (update) {
                uint32_t f;
                if constexpr (DIM == 2) {
                    const uint32_t s1 = d[0][0] ^ d[1][0], c1 = d[0][0] & d[1][0];
                    const uint32_t s2 = d[2][0] ^ d[3][0], c2 = d[2][0] & d[3][0];
                    const uint32_t ge = c1 | c2 | (s1 & s2), ea = (s1 ^ s2) & ~ge;
                    f = ge | (ea & a4) | (~(ge | ea) & a8);
                } else {
                    const uint32_t s1 = d[0][0] ^ d[1][0] ^ d[2][0], c1 = maj3(d[0][0], d[1][0], d[2][0]);
                    const uint32_t s2 = d[3][0] ^ d[4][0] ^ d[5][0], c2 = maj3(d[3][0], d[4][0], d[5][0]);
                    const uint32_t a0 = s1 ^ s2, t = s1 & s2, a1 = c1 ^ c2 ^ t, a2 = maj3(c1, c2, t);
                    const uint32_t ge = a2 | (a1 & a0), ea = a1 & ~(a0 | a2), eb = a0 & ~(a1 | a2);
                    f = ge | (ea & a4) | (eb & a8) | (~(ge | ea | eb) & a12);
                }
                nw.v[0] ^= f;
                if (g.h == 32u || Wc > 1u) {
                    if (has) own[w] = nw.v[0];
                    if (g.h == 32u && tid == 0u) own[g.PW] = nw.v[0];  // the extension is word 0 again
                } else {  // the extension follows the last word's h bits
                    const uint32_t first = __shfl_sync(kAll, nw.v[0], 0);
                    const bool end = has && w + 1u == g.PW;
                    const uint32_t tail = nw.v[0] & g.mh;
                    const uint64_t e = tail | ((uint64_t)(g.PW == 1u ? tail : first) << g.h);
                    if (has) own[w] = end ? (uint32_t)e : nw.v[0];
                    if (end) own[g.PW] = (uint32_t)(e >> 32);
                }
                if (h + 1u < n_half) fetch(h + 1u);
            }
            sync();
            if (tid == 0u) *vtaken = h + 2u;  // half-sweeps whose acceptance bits have been read
            if (update && g.h != 32u && Wc > 1u) {
                stream_extend<1>(own, 1u, g, tid, 32u * Wc);
                sync();
            }
            if (measure && Wc > 1u && tid == 0u) {
                int* a = acc[(h >> 1) & 1u];
                write((h >> 1) - 1u, a[0], a[1]);
                a[0] = a[1] = 0;  // next added to two sweeps later
            }
        };
        for (uint32_t h = 0; h < n_half; h += 2u) {
            half(std::integral_constant<uint32_t, 0>{}, h);
            half(std::integral_constant<uint32_t, 1>{}, h + 1u);
        }
        if (series) half(std::integral_constant<uint32_t, 0>{}, n_half);
    }
    __syncthreads();
    for (uint32_t ch = tid; ch < nch; ch += T) {
        const uint8_t* p0 = reinterpret_cast<const uint8_t*>(smw) + GBMC_IDX(ch, 4u * g.PWX);
        const uint32_t a = p0[0], b = p0[4u * g.PWX], m = odd_b[ch];
        const uint32_t ev = sel(m, b, a), od = sel(m, a, b);
        const uint2 lo = unpack8(ev & 15u, od & 15u), hi = unpack8(ev >> 4, od >> 4);
        int8_t* dst = J.dst + (uint64_t)slot * J.N + 16u * ch;
        if (wide) {
            *reinterpret_cast<uint4*>(dst) = make_uint4(lo.x, lo.y, hi.x, hi.y);
        } else {
            uint32_t* d4 = reinterpret_cast<uint32_t*>(dst);
            const uint32_t left = J.N - 16u * ch;
            d4[0] = lo.x;
            if (left > 4u) d4[1] = lo.y;
            if (left > 8u) d4[2] = hi.x;
            if (left > 12u) d4[3] = hi.y;
        }
    }
}

// Per-word masks of a lattice class, [5][PW]: the sites whose colour-0 row starts
// at odd x; the row ends whose x neighbour wraps around, for colour 0 and for
// colour 1; the sites with y = 0; those with y = L - 1. Bits past the stream's
// end are 0. With +-J bonds, per instance [2][6][PW] bond words: bit 1 where the
// bond from the colour-c site to its k-th neighbour (order of stream_unsat) has
// J = -1 (jbits: [inst][mu][site] bytes, 1 where the forward bond has J = -1).
__global__ void k_stream_tables(const uint8_t* jbits, uint32_t* smask, uint32_t* sbond, uint32_t dim, uint32_t L,
                                uint32_t N, uint32_t n_inst) {
    const uint32_t s = L >> 1, H = N >> 1, PW = (H + 31u) >> 5;
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i < 5u * PW) {
        const uint32_t t = (uint32_t)i / PW, w = (uint32_t)i % PW;
        uint32_t word = 0;
        for (uint32_t b = 0; b < 32u && 32u * w + b < H; ++b) {
            const uint32_t k = 32u * w + b, row = k / s, j = k - row * s;
            const uint32_t y = row % L, z = dim == 3 ? row / L : 0u;  // 2D: row < L
            const uint32_t o = (y + z) & 1u;
            bool on;
            switch (t) {
                case 0: on = o; break;
                case 1: on = o ? j == s - 1u : j == 0u; break;
                case 2: on = o ? j == 0u : j == s - 1u; break;
                case 3: on = y == 0u; break;
                default: on = y == L - 1u; break;
            }
            word |= (on ? 1u : 0u) << b;
        }
        smask[i] = word;
    }
    if (sbond && i < 12ull * n_inst * PW) {
        const uint32_t w = (uint32_t)(i % PW), k = (uint32_t)(i / PW % 6u), c = (uint32_t)(i / (6u * PW) % 2u);
        const uint8_t* jx = jbits + i / (12ull * PW) * 3u * N;
        const uint8_t *jy = jx + N, *jz = jx + 2u * N;
        uint32_t word = 0;
        for (uint32_t b = 0; b < 32u && 32u * w + b < H; ++b) {
            const uint32_t kk = 32u * w + b, row = kk / s, y = row % L, z = row / L;
            const uint32_t o = (y + z + c) & 1u, x = 2u * (kk - row * s) + o, site = row * L + x;
            const uint32_t xm = row * L + (x ? x - 1u : L - 1u);
            uint32_t bond;
            switch (k) {
                case 0: bond = o ? jx[xm] : jx[site]; break;
                case 1: bond = o ? jx[site] : jx[xm]; break;
                case 2: bond = jy[(z * L + (y ? y - 1u : L - 1u)) * L + x]; break;
                case 3: bond = jy[site]; break;
                case 4: bond = jz[((z ? z - 1u : L - 1u) * L + y) * L + x]; break;
                default: bond = jz[site]; break;
            }
            word |= (bond ? 1u : 0u) << b;
        }
        sbond[i] = word;
    }
}

// Words of a team's shared memory for G groups of C copies.
uint32_t stream_smem_words(uint32_t N, uint32_t G, uint32_t C, bool pt) {
    const uint32_t PWX = (N / 2u + 31u) / 32u + 1u;
    return (2u * G * PWX * C + 3u * G + 3u * G * C + (pt ? 3u * G * C : 0u) + 3u) & ~3u;
}

// How a launch spreads its jobs: C copies per thread, and per job teams of T
// threads (32: four one-warp teams per block; else the block) with G groups of C
// copies each. The estimate is in cycles of a scheduler per half-sweep: a pass of
// a warp over its words issues for `pass` cycles (the multiply and logic pipes)
// but takes `lat` by itself, so a scheduler with w warps at work spends
// max(pass, lat / w) per pass. Where one job's teams are all held at once the fullest
// scheduler's count; else the average and 0.6 of the longest team, for what the last
// teams leave idle (several jobs' teams are chosen by the whole of their own: the last
// job's are what is left at the end). Estimate : measured, thousand cycles per half-sweep,
// C = 1, 2, 4 (* taken): 2D L = 24, 40, 96 together 64 : 56, 60* : 49, 62 : 57; 3D L = 10, 8 x
// 5000 copies 41 : 41, 37 : 36, 33* : 34; L = 12, 4 x 1000 copies 8.7* : 9.0, 9.6 : 9.1, 9.0 : 8.3.
static_assert(StreamPlan{}.threads == kStreamThreads, "");

// measured: 2D L = 64 and 3D L = 10 with large populations (pass), populations with one to
// seven warps per scheduler (lat, stream_wave)
double stream_pass(int C, int split, int dim) {
    return dim == 2 ? (C == 4 ? 3430.0 : C == 2 ? 1810.0 : split == 1 ? 1030.0 : split == 2 ? 620.0 : 430.0)
                    : (C == 4 ? 3730.0 : C == 2 ? 2150.0 : split == 1 ? 1240.0 : split == 2 ? 750.0 : 560.0);
}
double stream_lat(int C, int split, int dim) {
    return (C == 4 ? 9000.0 : (C == 2 ? 4200.0 : split == 1 ? 2100.0 : split == 2 ? 1300.0 : 900.0) * (dim == 3 ? 1.15 : 1.0));
}
// A pass with w warps on every scheduler, in teams of T: two copies per thread leave gaps where
// the warps are few, and a block's teams wait for their slowest warp.
double stream_wave(int C, int split, int dim, double w, uint32_t T) {
    const double lat = stream_lat(C, split, dim);
    return std::max(w * stream_pass(C, split, dim), lat) + (w > 1.0 && C <= 2 ? (C == 2 ? 0.8 : 0.2) * lat / w : 0.0) +
           (T == 32u ? 0.0 : 12.0 * (T / 32u));
}

StreamPlan stream_plan(const SweepLaunch& P, int C, int split, bool pt, int sm_count) {
    const double pass = stream_pass(C, split, P.dim), lat = stream_lat(C, split, P.dim);
    const double by_regs = C == 4 ? 5.0 : 8.0;  // warps per scheduler the registers allow
    const double schedulers = 4.0 * sm_count;
    StreamPlan S;
    S.C = C;
    S.split = split;
    double total = 0.0, longest = 0.0;
    // the jobs' warps share the schedulers: those of the other jobs, from the round before
    double shares[kMaxJobs] = {}, others = 0.0;
    for (int round = 0; round < (P.njobs > 1 ? 2 : 1); ++round) {
        total = longest = 0.0;
        for (int j = 0; j < P.njobs; ++j) {
            const SweepJob& J = P.jobs[j];
            const uint32_t PW = (J.N / 2u + 31u) / 32u * (uint32_t)split;  // items of a copy
            const double groups = (double)J.n_inst * ((J.R + C - 1u) / C);
            double best = 1e300, best_sum = 0.0, best_len = 0.0, best_share = 0.0;
            others = 0.0;
            for (int k = 0; k < P.njobs; ++k) others += k == j ? 0.0 : shares[k];
            auto consider = [&](uint32_t T, uint32_t G) {
                const double p = (double)((G * PW + T - 1u) / T);
                const double share = std::ceil(groups / G) * (T / 32u) / schedulers;
                const uint32_t warps = T == 32u ? kStreamThreads / 32u : T / 32u;
                const size_t smem = (size_t)stream_smem_words(J.N, G, C, pt) * 4u * (T == 32u ? warps : 1u);
                const double fit = std::floor((double)kStreamSmem / smem) * warps / 4.0;
                const double cap = std::min(by_regs, fit), w = std::max(1.0, std::min(share + others, cap));
                const double step = std::max(pass, lat / w) + (T == 32u ? 0.0 : 60.0), len = p * step;
                double sum = p * share * step, cost = sum + (P.njobs > 1 ? 1.0 : 0.6) * len;
                if (P.njobs == 1 && share <= cap) {  // all teams at once; a block's warps share its SM
                    const double fullest = T == 32u ? share : std::ceil(groups / sm_count) * (T / 32u) / 4.0;
                    cost = sum = p * stream_wave(C, split, P.dim, std::ceil(fullest), T);
                }
                if (cost < best * 0.98) {
                    best = cost;
                    best_sum = sum;
                    best_len = std::min(cost - sum, 0.6 * len);
                    best_share = share;
                    S.T[j] = T;
                    S.G[j] = G;
                }
            };
            // one-warp teams; a single lattice with too few copies to give every scheduler
            // work takes whole blocks
            for (uint32_t G = 1; G <= 32u && stream_smem_words(J.N, G, C, pt) <= kStreamTeamWords; ++G) consider(32u, G);
            if (P.njobs == 1)
                for (uint32_t T = 64u; T <= stream_max_threads(C, split) && T < PW + 32u; T += 32u) consider(T, 1u);
            // Copies too large for that take whole blocks; beside other lattices' teams so may
            // all from 24 500 sites, where four copies pass a one-warp team's share (annealing
            // 200 copies of 2D L = 160 with 2000 of L = 24, 10 steps: 2480 us without, 1150 with;
            // 1000 of L = 180 with 5000 of L = 40: 4700 and 3780)
            if (best == 1e300 || (P.njobs > 1 && stream_smem_words(J.N, 1u, 4u, pt) > kStreamTeamWords))
                consider(kStreamThreads, 1u);
            shares[j] = best_share;
            total += best_sum;
            longest = std::max(longest, best_len);
        }
    }
    if (P.njobs == 1 && S.T[0] != 32u) S.threads = S.T[0];
    S.cost = total + longest;
    return S;
}

template <int DIM, bool EA, int C, int SP, int PT>
cudaError_t launch_stream(const SweepLaunch& P0, const StreamPlan& S, cudaStream_t st) {
    SweepLaunch P = P0;
    uint64_t total = 0;
    size_t smem = 0;
    uint32_t warp_words = 0;
    for (int j = 0; j < P.njobs; ++j) {
        SweepJob& J = P.jobs[j];
        J.ctas_per_inst = (J.R + C - 1u) / C;  // groups per instance
        J.team = S.T[j];
        J.rpc = S.G[j];
        const uint64_t groups = (uint64_t)J.n_inst * J.ctas_per_inst;
        if (groups > 0x7FFFFFFFull) return cudaErrorInvalidValue;
        if (J.team == 32u) warp_words = std::max(warp_words, stream_smem_words(J.N, J.rpc, C, PT));
        else smem = std::max(smem, (size_t)stream_smem_words(J.N, 1u, C, PT) * 4u);
        const uint64_t teams = (groups + J.rpc - 1u) / J.rpc, per_block = S.threads / J.team;
        P.cta_begin[j] = (uint32_t)total;
        total += (teams + per_block - 1u) / per_block;
        if (total > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    }
    smem = std::max(smem, (size_t)warp_words * 4u * (S.threads / 32u));
    P.cta_begin[P.njobs] = (uint32_t)total;
    P.total = (uint32_t)total;
    if (total == 0) return cudaSuccess;
    auto kern = k_sweep_stream<DIM, EA, C, SP, PT>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<(uint32_t)total, S.threads, smem, st>>>(P, PtExchange{}, warp_words);
    count_launch();
    return cudaGetLastError();
}

template <int DIM, bool EA>
cudaError_t launch_stream_c(const SweepLaunch& P, const StreamPlan& S, bool pt, cudaStream_t st) {
    if (S.C == 4) return pt ? launch_stream<DIM, EA, 4, 1, kPerCopy>(P, S, st) : launch_stream<DIM, EA, 4, 1, kOneTemp>(P, S, st);
    if (S.C == 2) return pt ? launch_stream<DIM, EA, 2, 1, kPerCopy>(P, S, st) : launch_stream<DIM, EA, 2, 1, kOneTemp>(P, S, st);
    if (S.split == 2)
        return pt ? launch_stream<DIM, EA, 1, 2, kPerCopy>(P, S, st) : launch_stream<DIM, EA, 1, 2, kOneTemp>(P, S, st);
    if (S.split == 4)
        return pt ? launch_stream<DIM, EA, 1, 4, kPerCopy>(P, S, st) : launch_stream<DIM, EA, 1, 4, kOneTemp>(P, S, st);
    return pt ? launch_stream<DIM, EA, 1, 1, kPerCopy>(P, S, st) : launch_stream<DIM, EA, 1, 1, kOneTemp>(P, S, st);
}

// How the copies of every instance are divided for rounds of tempering (one copy per thread:
// two measured 20 % slower for want of work in flight). In cycles per
// round, by the same pass and latency as above: a block keeps its place to the
// end, so the blocks count in whole waves.
size_t rounds_smem(const SweepJob& J, const RoundsPlan& p) {
    return (size_t)(p.threads / p.T * stream_smem_words(J.N, p.G, 1u, true) + 5u * J.R) * 4u;
}

// A plan's cycles per round, its blocks on so many multiprocessors, and how often these fill up.
struct RoundsCost {
    double cycles, waves;
};
RoundsCost rounds_cost(const SweepJob& J, int dim, const RoundsPlan& p, double sms) {
    const uint32_t PW = (J.N / 2u + 31u) / 32u;
    // (with places and bond words kept: less than a sweep launch's pass)
    const double pass = (p.split == 4 ? 420.0 : 980.0) * (dim == 3 ? 1.15 : 1.0), lat = stream_lat(1, p.split, 2);
    const double passes = std::ceil(p.G * PW * p.split / (double)p.T), warps = p.threads / 32.0;
    const double held = std::min({std::floor((double)stream_max_threads(1, p.split, kRounds) / p.threads),  // by registers
                                  std::floor((double)kStreamSmem / (rounds_smem(J, p) + 1024.0)), 16.0});
    const double blocks = (double)J.n_inst * p.B, wave = held * sms, full = std::floor(blocks / wave);
    auto half = [&](double per_sm) {  // a half-sweep with so many blocks on an SM
        const double w = std::ceil(per_sm * warps / 4.0);
        return passes * (std::max(lat, w * pass) + (w > 1.0 ? 200.0 : 0.0) + 2.0 * per_sm * warps) +
               (p.T > 32u ? 300.0 : 0.0);
    };
    const double rest = std::ceil((blocks - full * wave) / sms);
    const double t = full * half(held) + (rest > 0.0 ? half(rest) : 0.0);
    const double waves = full + (rest > 0.0 ? 1.0 : 0.0);
    return {(2.0 * J.nsweeps + 0.4) * t + waves * (p.B > 1u ? 2500.0 : 1500.0), waves};
}

RoundsPlan rounds_plan(const SweepJob& J, int dim, int sm_count) {
    RoundsPlan best;
    const uint32_t PW = (J.N / 2u + 31u) / 32u;
    const uint32_t ng = J.R;
    for (const int split : {4, 1}) {
        const uint32_t most = stream_max_threads(1, split, kRounds);
        auto consider = [&](uint32_t B, uint32_t G, uint32_t T, uint32_t threads) {
            RoundsPlan p;
            p.split = split, p.B = B, p.G = G, p.T = T, p.threads = threads;
            if (rounds_smem(J, p) > 200u * 1024u) return;
            p.cost = rounds_cost(J, dim, p, sm_count).cycles;
            if (p.cost < best.cost) best = p;
        };
        for (uint32_t B = 1; B <= 8u && B <= ng; B *= 2u) {
            // one-warp teams, with up to eight passes over their words
            for (uint32_t G = 1; G <= ng && G * PW * split <= 256u; ++G) {
                const uint32_t teams = (ng + G - 1u) / G, warps = (teams + B - 1u) / B;
                if (warps * 32u <= most) consider(B, G, 32u, warps * 32u);
            }
            const uint32_t G = (ng + B - 1u) / B, items = G * PW * (uint32_t)split, passes = (items + most - 1u) / most;
            const uint32_t threads = ((items + passes - 1u) / passes + 31u) & ~31u;
            if (threads > 32u) consider(B, G, threads, threads);
        }
    }
    return best;
}

template <int DIM, bool EA, int SP>
cudaError_t launch_rounds(const SweepLaunch& P0, const PtExchange& X, const RoundsPlan& R, cudaStream_t st) {
    SweepLaunch P = P0;
    SweepJob& J = P.jobs[0];
    J.ctas_per_inst = J.R;
    J.team = R.T;
    J.rpc = R.G;
    P.cta_begin[0] = 0;
    P.cta_begin[1] = P.total = J.n_inst * R.B;
    auto kern = k_sweep_stream<DIM, EA, 1, SP, kRounds>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P.total);
    cfg.blockDim = dim3(R.threads);
    cfg.dynamicSmemBytes = rounds_smem(J, R);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = R.B;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cfg.dynamicSmemBytes > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaLaunchKernelEx(&cfg, kern, P, X, stream_smem_words(J.N, R.G, 1u, true));
    count_launch();
    return e;
}

template <int DIM, bool EA>
cudaError_t launch_rounds_c(const SweepLaunch& P, const PtExchange& X, const RoundsPlan& R, cudaStream_t st) {
    return R.split == 4 ? launch_rounds<DIM, EA, 4>(P, X, R, st) : launch_rounds<DIM, EA, 1>(P, X, R, st);
}

}  // namespace

// Plain sweeps of at most one copy per multiprocessor.
bool sweeps_ahead(const SweepLaunch& P, int sm_count) {
    if (P.njobs != 1) return false;
    const SweepJob& J = P.jobs[0];
    const uint64_t copies = (uint64_t)J.n_inst * J.R;
    return J.smask && (!P.ea || J.sbond) && (J.N / 2u + 31u) / 32u <= kAheadWords && copies <= (uint64_t)sm_count &&
           J.nsweeps >= 2u && J.nsweeps <= 0x3FFFFFFFu && !J.parent && !J.hist && !J.temp_of && !J.nlive && !J.E && !J.M &&
           J.src == J.dst;
}

cudaError_t launch_sweep_ahead(const SweepLaunch& P, unsigned int* err, long long budget, uint32_t phantom,
                               cudaStream_t s) {
    const SweepJob& J = P.jobs[0];
    const uint32_t PW = (J.N / 2u + 31u) / 32u, ring = ahead_ring(PW), Wc = (PW + 31u) / 32u;
    const size_t smem = 4ull * (2u * (PW + 1u) + (P.dim == 3 ? 3u : 2u) * ring + ring / 32u);
    auto kern = P.dim == 2 ? k_sweep_ahead<2, false> : P.ea ? k_sweep_ahead<3, true> : k_sweep_ahead<3, false>;
    const uint32_t naps = (uint32_t)std::min<long long>(budget / kNapCycles, 0x7FFFFFFF);
    kern<<<J.n_inst * J.R, 32u * (Wc == 1u ? 12u : Wc + kDrawers), smem, s>>>(P, err, naps, phantom);
    count_launch();
    return cudaGetLastError();
}

// A round by itself is a sweep launch, whose copies are loaded and stored, and an
// exchange launch, 20 000 to 27 000 cycles beside the half-sweeps (3D L = 8, 250 x 40 copies,
// one sweep per round: 15.4 us, 4.8 of them sweeping; L = 12, 60 x 14: 16.4, 2). What speaks for it is that its blocks
// change places between rounds: 256 x 40 copies of L = 12, 10 sweeps per round, 207 us
// each against 248 in one launch of rounds; 100 x 36 53 against 38. A launch of rounds loads
// the maps and the copies once, so it has to have rounds enough: 2000 x 4 copies of 3D L = 8, one
// sweep per round, 1, 2 and 20 rounds per call 20.7, 13.6 and 8.0 us per round in one launch, 12.6
// apart; 200 x 8 14.6, 9.9, 5.6 and 10.4.
TemperingCost tempering_cost(const SweepLaunch& P, int sm_count) {
    const SweepJob& J = P.jobs[0];
    if (!J.smask || (P.ea && !J.sbond) || J.nsweeps == 0u || J.R < 2u || J.R > 1024u) return {};
    double alone = std::min(stream_plan(P, 1, 4, true, sm_count).cost, stream_plan(P, 1, 2, true, sm_count).cost);
    for (int C = 4; C >= 1; C >>= 1)
        if (C == 1 || stream_smem_words(J.N, 1u, (uint32_t)C, true) * 4u <= 36u * 1024u)
            alone = std::min(alone, stream_plan(P, C, 1, true, sm_count).cost);
    if (bits_supported(P.dim, (int)J.L)) {  // those sweeps are bitsweep.cu's, faster where they fill the chip
        const double copies = (double)J.n_inst * J.R, per = std::max(1.0, J.N / 2048.0);  // warps' words per lane
        const double warps = std::ceil(copies * (J.N / 64.0) / 32.0 / per / (4.0 * sm_count));
        alone = std::min(alone, per * std::max(warps * (P.dim == 3 ? 950.0 : 840.0), 2100.0));
    }
    const RoundsPlan p = rounds_plan(J, P.dim, sm_count);
    if (!(p.cost < 2.0 * J.nsweeps * alone + 24000.0)) return {};
    // A cluster's blocks lie within one group of the device's multiprocessors, of which some are
    // left over: 16 clusters of eight blocks that fill a multiprocessor each run as two waves
    const double sms = J.n_inst == 1u || p.B == 1u ? 1.0 : p.B == 8u ? 0.74 : p.B == 4u ? 0.9 : 0.97;
    const RoundsCost c = rounds_cost(J, P.dim, p, std::floor(sms * sm_count));
    const double copies = (double)J.n_inst * J.R, kb = J.N / 1024.0, blocks = (double)J.n_inst * p.B;
    TemperingCost t;
    t.plan = p;
    t.round = c.cycles;
    t.launch = 12000.0 + 830.0 * blocks / sm_count +
               std::max(c.waves * std::ceil((double)J.R / p.B), copies / sm_count) * (100.0 + 110.0 * kb);
    t.apart = 2.0 * J.nsweeps * alone + 22800.0 + 0.35 * copies * kb;
    return t;
}

cudaError_t launch_tempering_rounds(const SweepLaunch& P, const PtExchange& X, const RoundsPlan& R, cudaStream_t s) {
    if (P.dim == 2 && !P.ea) return launch_rounds_c<2, false>(P, X, R, s);
    if (P.dim == 3 && !P.ea) return launch_rounds_c<3, false>(P, X, R, s);
    if (P.dim == 3 && P.ea) return launch_rounds_c<3, true>(P, X, R, s);
    return cudaErrorInvalidValue;
}

size_t stream_mask_words(uint32_t N) { return 5ull * ((N / 2u + 31u) / 32u); }
size_t stream_bond_words(uint32_t N) { return 12ull * ((N / 2u + 31u) / 32u); }

cudaError_t launch_stream_tables(const uint8_t* jbits, uint32_t* smask, uint32_t* sbond, int dim, uint32_t L,
                                 uint32_t n_inst, cudaStream_t s) {
    const uint32_t N = L * L * (dim == 3 ? L : 1u);
    uint64_t n = stream_mask_words(N);
    if (sbond && stream_bond_words(N) * n_inst > n) n = stream_bond_words(N) * n_inst;
    k_stream_tables<<<(uint32_t)((n + 127u) / 128u), 128, 0, s>>>(jbits, smask, sbond, (uint32_t)dim, L, N, n_inst);
    count_launch();
    return cudaGetLastError();
}

// Largest copies first: their blocks are dispatched first, shortening the tail.
static void largest_first(SweepLaunch& P) {
    for (int a = 1; a < P.njobs; ++a)
        for (int b = a; b > 0 && P.jobs[b].N > P.jobs[b - 1].N; --b) std::swap(P.jobs[b], P.jobs[b - 1]);
}

StreamPlan stream_plan(const SweepLaunch& P0, bool pt, int sm_count) {
    SweepLaunch P = P0;
    largest_first(P);
    StreamPlan S = stream_plan(P, 1, 4, pt, sm_count);
    const StreamPlan halves = stream_plan(P, 1, 2, pt, sm_count);
    if (halves.cost < S.cost) S = halves;
    for (int C = 4; C >= 1; C >>= 1) {
        // a group's planes at most 36 KB, so that an SM holds six blocks
        if (C > 1 && stream_smem_words(P.jobs[0].N, 1u, (uint32_t)C, pt) * 4u > 36u * 1024u) continue;
        const StreamPlan t = stream_plan(P, C, 1, pt, sm_count);
        if (t.cost < S.cost) S = t;
    }
    return S;
}

cudaError_t launch_sweep_stream(const SweepLaunch& P0, int sm_count, cudaStream_t s) {
    SweepLaunch P = P0;
    largest_first(P);
    bool pt = false;
    for (int j = 0; j < P.njobs; ++j) {
        if (!P.jobs[j].smask || (P.ea && !P.jobs[j].sbond)) return cudaErrorInvalidValue;
        pt = pt || P.jobs[j].temp_of != nullptr;
    }
    // the plan depends only on these numbers; a run's launches repeat the last ones
    struct Key {
        uint32_t head[4], job[kMaxJobs][3];
    };
    static thread_local Key last = {};
    static thread_local StreamPlan S;
    Key key = {};
    key.head[0] = (uint32_t)P.njobs, key.head[1] = (uint32_t)sm_count, key.head[2] = pt, key.head[3] = (uint32_t)P.dim;
    for (int j = 0; j < P.njobs; ++j)
        key.job[j][0] = P.jobs[j].N, key.job[j][1] = P.jobs[j].R, key.job[j][2] = P.jobs[j].n_inst;
    if (std::memcmp(&key, &last, sizeof(key)) != 0) {
        S = stream_plan(P, pt, sm_count);
        last = key;
    }
    if (P.dim == 2 && !P.ea) return launch_stream_c<2, false>(P, S, pt, s);
    if (P.dim == 3 && !P.ea) return launch_stream_c<3, false>(P, S, pt, s);
    if (P.dim == 3 && P.ea) return launch_stream_c<3, true>(P, S, pt, s);
    return cudaErrorInvalidValue;
}

}  // namespace gbmc
