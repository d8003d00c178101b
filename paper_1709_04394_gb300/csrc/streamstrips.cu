// streamstrips.cu -- checkerboard Metropolis sweeps (Sec. 3.1, Eq. (8)) of large
// lattices, one bit per spin, every half-sweep of a call in one cooperative
// launch: any even L (2D ferromagnets from L = 64, 3D lattices), few copies, with
// E and M after every sweep when asked for.
//
// The configuration is two colour planes in global memory, each the cyclic bit
// stream of stream.cu (H = N / 2 sites in colour-rank order), every 32-bit word
// beside a tag: the number of half-sweeps it has seen plus one, 0 at the start.
// Word and tag are written and read as one 64-bit access, so a thread simply reads
// the words its update needs until their tags say that they are the previous
// half-sweep's: the data carry their own synchronisation, there is no barrier, no
// fence and no flag. A word can only be overwritten two half-sweeps later, which
// its owner does after seeing the tags of its neighbours' next values -- computed
// from the old word --, so no reader misses it. All CTAs are resident at once
// (cooperative launch) and every wait is for an earlier half-sweep, so some thread
// can always go on; waits are bounded all the same. The words at the ends of a
// CTA's run, which other CTAs wait for, are updated first.
//
// Small lattices leave a thread less than a word: S = 4 threads then share one
// word, each the eight sites of one byte of it (two Philox calls).
//
// E and M after sweep t are taken in the next half-sweep, which reads every bond's
// two ends anyway (colour 0 before its update, colour 1 as its neighbours), and
// after the last sweep in one more pass: no launch of their own.
//
// Where a run is longer than its ends (2D, four threads per word) the CTA keeps it in
// shared memory, and only the ends are written to and read from global memory.
//
// Bound: for small lattices the chain of a half-sweep -- words loaded from L2,
// update, words stored --, for larger ones the integer pipes (stream.cu).
#include "bits.cuh"
#include "check.cuh"
#include "device.cuh"
#include "internal.h"

namespace gbmc {

namespace {

constexpr uint32_t kStripMaxThreads = 1024;  // one word per thread; four threads per word: at most 512

struct PlaneShape {
    uint32_t L, s, A, H, PW, h, mh;
};

__host__ __device__ __forceinline__ PlaneShape plane_shape(uint32_t dim, uint32_t L, uint32_t N) {
    PlaneShape g;
    g.L = L;
    g.s = L >> 1;
    g.A = dim == 3 ? g.s * L : 0u;
    g.H = N >> 1;
    g.PW = (g.H + 31u) >> 5;
    g.h = ((g.H - 1u) & 31u) + 1u;
    g.mh = 0xFFFFFFFFu >> (32u - g.h);
    return g;
}

__device__ __forceinline__ uint32_t pick(uint32_t m, uint32_t a, uint32_t b) { return (a & m) | (b & ~m); }

// Row masks of word w of colour c in a 2D lattice (s >= 32: at most two rows to a
// word): odd = the sites of odd x, edge = those whose other x neighbour wraps
// (first site of an even-x row, last site of an odd-x row).
__device__ __forceinline__ void row_masks(const PlaneShape& g, uint32_t w, uint32_t colour, uint32_t& odd,
                                          uint32_t& edge) {
    const uint32_t k0 = w << 5, r = k0 / g.s, j = k0 - r * g.s, b = g.s - j;  // b sites of row r left, b >= 1
    const uint32_t low = b >= 32u ? 0xFFFFFFFFu : (1u << b) - 1u;
    const bool o = ((r + colour) & 1u) != 0u;
    odd = o ? low : ~low;
    const uint32_t first = j == 0u ? 1u : 0u, last = b <= 32u ? 1u << (b - 1u) : 0u;
    // the next row has the other parity: its first site is bit b (o set: even x there)
    edge = o ? last | (b < 32u ? 1u << b : 0u) : first;
}

// A plane's words, the least tag seen, and the 32 bits of its stream from bit p < H
// on, across its end. HELD: the CTA's own run, words first .. first + count - 1, is in
// shared memory.
__device__ __forceinline__ uint64_t shared_word(const uint64_t* p) {
    uint64_t x;
    asm volatile("ld.relaxed.cta.shared.u64 %0, [%1];" : "=l"(x) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
    return x;
}
template <bool HELD>
struct Plane {
    const uint64_t *w, *run;
    uint32_t first, count, words, tag;
    __device__ __forceinline__ uint32_t word(uint32_t i) {
        uint64_t x;
        if (HELD && i - first < count) x = shared_word(run + (i - first));
        else asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(w + GBMC_IDX(i, words)) : "memory");
        tag = min(tag, (uint32_t)(x >> 32));
        return (uint32_t)x;
    }
    __device__ __forceinline__ void window(const PlaneShape& g, uint32_t p, uint32_t& v0, uint32_t& v1) {
        // v0: bits p .. p + 31, v1: bits p + 1 .. p + 32
        const uint32_t i = p >> 5, sh = p & 31u;
        uint32_t a = word(i), b = word(i + 1u == g.PW ? 0u : i + 1u);
        if (g.h != 32u && i + 2u >= g.PW) {
            // the stream's last word holds h bits, its first bits follow
            const uint32_t w0 = i + 1u == g.PW ? b : word(0u);
            const uint32_t w1 = g.PW > 1u ? word(1u) : w0;
            if (i + 1u == g.PW) {
                const uint64_t e = (uint64_t)w0 << g.h;
                a |= (uint32_t)e;
                b = (uint32_t)(e >> 32) | w1 << g.h;
            } else {
                b |= w0 << g.h;
            }
        }
        v0 = __funnelshift_r(a, b, sh);
        v1 = __funnelshift_rc(a, b, sh + 1u);
    }
};

template <int DIM, bool EA, int S, bool HELD>
__global__ void __launch_bounds__(S == 4 ? 512 : kStripMaxThreads, 1) k_stream_strips(const __grid_constant__ StreamStrips P) {
    __shared__ int acc[2][2];  // by sweep parity: unsatisfied bonds and down spins of this CTA's words
    const uint32_t tid = threadIdx.x, T = blockDim.x;
    const PlaneShape g = plane_shape(DIM, P.L, P.N);
    const uint32_t copy = P.copy0 + blockIdx.x / P.Gc, cta = blockIdx.x % P.Gc;
    const uint32_t w0 = (uint32_t)((uint64_t)cta * g.PW / P.Gc), w1 = (uint32_t)((uint64_t)(cta + 1u) * g.PW / P.Gc);
    const uint32_t n_words = w1 - w0;
    const uint32_t inst = copy / P.R, r = copy - inst * P.R, instance = P.inst_base + inst;
    const uint32_t k0 = (uint32_t)P.seed, k1 = (uint32_t)(P.seed >> 32);
    uint64_t* const planes = P.P + (uint64_t)copy * 2u * g.PW;
    // HELD: the run's words of both planes, read by this CTA's threads without the way to L2
    extern __shared__ __align__(16) uint64_t runs[];
    if constexpr (HELD) {
        for (uint32_t i = tid; i < 2u * n_words; i += T)
            runs[i] = planes[GBMC_IDX((uint64_t)(i / n_words) * g.PW + w0 + i % n_words, 2u * g.PW)];
        __syncthreads();
    }
    // words near an end of the run come first: n_edge of them on either side
    const uint32_t n_edge = min(P.edge, (n_words + 1u) / 2u), n_first = min(2u * n_edge, n_words);
    const uint32_t items = n_words * S;
    const bool series = P.Eser || P.Mser;
    if (series) {
        if (tid < 4u) acc[tid >> 1][tid & 1u] = 0;
        __syncthreads();
    }
    bool dead = false;  // a wait ran out: nothing more is updated

    const uint32_t n_half = P.n_half + (series ? 1u : 0u);  // the last one only measures
    for (uint32_t h = 0; h < n_half; ++h) {
        const uint32_t c = h & 1u;
        const bool update = h < P.n_half, measure = series && c == 0u && h > 0u;
        uint64_t* const own = planes + c * g.PW;
        const PhiloxFixed pf = philox_fix(P.t0 + (h >> 1), r, c3_word(kPurposeMetro, c, instance), k0, k1);
        int U = 0, D = 0;
        for (uint32_t i0 = 0; i0 < items; i0 += T) {  // whole warps take every step
            const uint32_t i = i0 + tid;
            const bool has = i < items && !dead;
            const uint32_t x = i < items ? i / S : 0u, part = i % S;
            const uint32_t w = w0 + (x < n_first ? (x < n_edge ? x : n_words - n_first + x) : x - n_first + n_edge);
            const uint32_t b0 = w << 5;
            uint32_t odd, edge, y0 = 0u, yl = 0u;
            if constexpr (DIM == 2) {
                row_masks(g, w, c, odd, edge);
            } else {
                odd = __ldg(P.mask + GBMC_IDX(w, g.PW)) ^ (c ? 0xFFFFFFFFu : 0u);
                edge = __ldg(P.mask + (1u + c) * g.PW + w);
                y0 = __ldg(P.mask + 3u * g.PW + w);
                yl = __ldg(P.mask + 4u * g.PW + w);
            }
            // acceptance bits. The random words do not depend on the spins: with a whole
            // word per thread in 3D they are drawn before the neighbours' words are
            // looked at (8 copies of L = 96: 512 -> 424 us per 50 sweeps), elsewhere after
            // (L = 2000 254 against 281 us, 3D L = 48 238 against 252)
            constexpr bool kDrawFirst = DIM == 3 && S == 1;
            uint32_t r4 = 0, r8 = 0, r12 = 0;
            constexpr uint32_t NC = 8u / S;  // Philox calls of this thread
            auto draw = [&]() {
#pragma unroll
                for (uint32_t k = 0; k < NC; ++k) {
                    const uint4 v = philox_q_wide(pf, 8u * w + NC * part + k);
                    if constexpr (DIM == 2) {
                        accept_bits(r4, r8, P.T4, P.T8, v.x);
                        accept_bits(r4, r8, P.T4, P.T8, v.y);
                        accept_bits(r4, r8, P.T4, P.T8, v.z);
                        accept_bits(r4, r8, P.T4, P.T8, v.w);
                    } else {
                        accept_bits3(r4, r8, r12, P.T4, P.T8, P.T12, v.x);
                        accept_bits3(r4, r8, r12, P.T4, P.T8, P.T12, v.y);
                        accept_bits3(r4, r8, r12, P.T4, P.T8, P.T12, v.z);
                        accept_bits3(r4, r8, r12, P.T4, P.T8, P.T12, v.w);
                    }
                }
            };
            // the words the update reads; ready once their tags show the other plane's
            // half-sweep h - 1 (tag h) and this word's own h - 2
            uint32_t s0, same, prv, nxt, up, up1, dn1, dn, ya = 0u, yb = 0u, za = 0u, zb = 0u, tag_me, tag_oth;
            auto look = [&]() {
                Plane<HELD> me{own, runs + c * n_words, w0, n_words, g.PW, 0xFFFFFFFFu};
                Plane<HELD> oth{planes + (c ^ 1u) * g.PW, runs + (c ^ 1u) * n_words, w0, n_words, g.PW, 0xFFFFFFFFu};
                s0 = me.word(w);
                same = oth.word(w);
                prv = oth.word(w ? w - 1u : 0u);
                nxt = oth.word(w + 1u == g.PW ? 0u : w + 1u);
                oth.window(g, b0 >= g.s ? b0 - g.s : b0 + g.H - g.s, up, up1);  // from k - s
                uint32_t p = b0 + g.s - 1u;
                if (p >= g.H) p -= g.H;
                oth.window(g, p, dn1, dn);  // from k + s - 1
                if constexpr (DIM == 3) {
                    uint32_t unused;
                    p = b0 + g.A - g.s;
                    if (p >= g.H) p -= g.H;
                    oth.window(g, p, ya, unused);  // y = 0: row L - 1 of the slab
                    // y = L - 1: row 0
                    oth.window(g, b0 + g.s >= g.A ? b0 + g.s - g.A : b0 + g.s + g.H - g.A, yb, unused);
                    oth.window(g, b0 >= g.A ? b0 - g.A : b0 + g.H - g.A, za, unused);
                    p = b0 + g.A;
                    if (p >= g.H) p -= g.H;
                    oth.window(g, p, zb, unused);
                }
                tag_me = me.tag;
                tag_oth = oth.tag;
            };
            if (kDrawFirst && update) draw();
            look();
            uint32_t spins = 0;
            long long start = 0;
            while (has && !dead && !(tag_oth >= h + P.phantom && tag_me + 1u >= h)) {
                if ((++spins & 31u) == 0u) {
                    if (start == 0) start = clock64();
                    if (*reinterpret_cast<volatile unsigned int*>(P.err) != 0u || clock64() - start > P.budget) {
                        atomicExch(P.err, 1u);
                        dead = true;
                    }
                }
                look();
            }
            __syncwarp();
            if (S == 4) dead = __any_sync(0xFFFFFFFFu, dead) != 0;
            const bool live = has && !dead;
            const uint32_t to_next = pick(edge, up1, __funnelshift_r(same, nxt, 1));
            const uint32_t to_prev = pick(edge, dn1, __funnelshift_l(prv, same, 1));
            uint32_t d[6];
            d[0] = s0 ^ same;
            d[1] = s0 ^ pick(odd, to_next, to_prev);
            if constexpr (DIM == 2) {
                d[2] = s0 ^ up;
                d[3] = s0 ^ dn;
                d[4] = d[5] = 0u;
            } else {
                d[2] = s0 ^ pick(y0, ya, up);
                d[3] = s0 ^ pick(yl, yb, dn);
                d[4] = s0 ^ za;
                d[5] = s0 ^ zb;
            }
            if constexpr (EA) {
                const uint32_t* bond = P.bond + ((uint64_t)inst * 2u + c) * 6u * g.PW + w;
#pragma unroll
                for (int k = 0; k < 6; ++k) d[k] ^= __ldg(bond + (uint64_t)k * g.PW);
            }
            const uint32_t valid = w + 1u == g.PW ? g.mh : 0xFFFFFFFFu;
            if (measure && live) {
                const uint32_t m = S == 4 ? valid & (0xFFu << (8u * part)) : valid;  // this thread's sites
#pragma unroll
                for (int k = 0; k < 2 * DIM; ++k) U += __popc(d[k] & m);
                D += __popc(s0 & m) + __popc(same & m);
            }
            if (!update) continue;
            if (!kDrawFirst) draw();
            uint32_t ge, ea, eb = 0u;  // dE <= 0; dE = 4; dE = 8 (3D)
            if constexpr (DIM == 2) {
                const uint32_t s1 = d[0] ^ d[1], c1 = d[0] & d[1], s2 = d[2] ^ d[3], c2 = d[2] & d[3];
                ge = c1 | c2 | (s1 & s2);
                ea = (s1 ^ s2) & ~ge;
            } else {
                const uint32_t s1 = d[0] ^ d[1] ^ d[2], c1 = maj3(d[0], d[1], d[2]);
                const uint32_t s2 = d[3] ^ d[4] ^ d[5], c2 = maj3(d[3], d[4], d[5]);
                const uint32_t a0 = s1 ^ s2, t = s1 & s2, a1 = c1 ^ c2 ^ t, a2 = maj3(c1, c2, t);
                ge = a2 | (a1 & a0);
                ea = a1 & ~(a0 | a2);
                eb = a0 & ~(a1 | a2);
            }
            // the first site's bit is the highest of the 4 NC accumulated
            constexpr uint32_t down = 32u - 4u * NC;
            const uint32_t sh = 4u * NC * part;
            r4 = __brev(r4) >> down << sh;
            r8 = __brev(r8) >> down << sh;
            const uint32_t f = DIM == 2 ? ge | (ea & r4) | (~(ge | ea) & r8)
                                        : ge | (ea & r4) | (eb & r8) | (~(ge | ea | eb) & (__brev(r12) >> down << sh));
            uint32_t v = (s0 ^ f) & valid;
            if constexpr (S == 4) {  // the word's four bytes, from its four threads
                v &= 0xFFu << sh;
                v |= __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                v |= __shfl_xor_sync(0xFFFFFFFFu, v, 2);
            }
            if (live && part == 0u) {
                const uint64_t out = (uint64_t)(h + 1u) << 32 | v;
                if (HELD)
                    asm volatile("st.relaxed.cta.shared.u64 [%0], %1;" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(runs + GBMC_IDX(c * n_words + (w - w0), 2u * n_words))),
                                 "l"(out)
                                 : "memory");
                // other CTAs read the run's ends, the caller what is there at the end
                if (!HELD || x < n_first || h + 2u >= P.n_half)
                    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(own + GBMC_IDX(w, g.PW)), "l"(out)
                                 : "memory");
            }
        }
        if (measure) {
            U = __reduce_add_sync(0xFFFFFFFFu, U);
            D = __reduce_add_sync(0xFFFFFFFFu, D);
            int* const a = acc[(h >> 1) & 1u];
            if ((tid & 31u) == 0u) {
                atomicAdd(a, U);
                atomicAdd(a + 1, D);
            }
            if (__syncthreads_or(dead)) return;
            if (tid == 0) {  // E = 2 U - DIM N, M = N - 2 D: the constants are there already
                const uint64_t at = GBMC_IDX((uint64_t)((h >> 1) - 1u) * P.ncopies + copy, P.n_half / 2u * P.ncopies);
                if (P.Eser) atomicAdd(P.Eser + at, 2 * a[0]);
                if (P.Mser) atomicAdd(P.Mser + at, -2 * a[1]);
                a[0] = a[1] = 0;  // next added to two sweeps later, a block barrier in between
            }
        } else if (!series && dead) {
            return;
        }
    }
}

// int8 row-major <-> the planes above, one thread per 16 consecutive sites (= byte
// ch of the streams of even-x and of odd-x sites; the colour-0 one is the even-x
// one in rows whose colour-0 sites have even x). Copies start on 4-byte boundaries.
template <int DIM, bool PACK>
__global__ void __launch_bounds__(256) k_stream_convert(int8_t* spins, uint64_t* P, const uint32_t* mask, uint32_t L,
                                                        uint32_t N, uint64_t copies) {
    chain_begin();
    const PlaneShape g = plane_shape(DIM, L, N);
    const uint32_t nch = (N + 15u) >> 4;
    const bool wide = (N & 15u) == 0u;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < copies * nch;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t copy = i / nch;
        const uint32_t ch = (uint32_t)(i - copy * nch), left = N - 16u * ch;
        uint32_t m;
        if constexpr (DIM == 2) {
            uint32_t odd, edge;
            row_masks(g, ch >> 2, 0u, odd, edge);
            m = (odd >> (8u * (ch & 3u))) & 0xFFu;
        } else {
            m = reinterpret_cast<const uint8_t*>(mask)[ch];
        }
        uint64_t* const w0 = P + GBMC_IDX(copy * 2u * g.PW + (ch >> 2), copies * 2u * g.PW - g.PW);
        uint64_t* const w1 = w0 + g.PW;
        uint8_t* p0 = reinterpret_cast<uint8_t*>(w0) + (ch & 3u);
        uint8_t* p1 = reinterpret_cast<uint8_t*>(w1) + (ch & 3u);
        int8_t* site = spins + GBMC_IDX(copy * N + 16ull * ch, copies * N);
        uint32_t* s4 = reinterpret_cast<uint32_t*>(site);
        if constexpr (PACK) {
            uint4 v;
            if (wide) {
                v = *reinterpret_cast<const uint4*>(site);
            } else {
                v.x = s4[0];
                v.y = left > 4u ? s4[1] : 0u;
                v.z = left > 8u ? s4[2] : 0u;
                v.w = left > 12u ? s4[3] : 0u;
            }
            uint32_t e0, o0, e1, o1;
            pack8(v.x, v.y, e0, o0);
            pack8(v.z, v.w, e1, o1);
            const uint32_t ev = e0 | (e1 << 4), od = o0 | (o1 << 4);
            *p0 = (uint8_t)pick(m, od, ev);
            *p1 = (uint8_t)pick(m, ev, od);
            if ((ch & 3u) == 0u) {  // tags
                reinterpret_cast<uint32_t*>(w0)[1] = 0u;
                reinterpret_cast<uint32_t*>(w1)[1] = 0u;
            }
            for (uint32_t k = (ch & 3u) + 1u; left <= 16u && k < 4u; ++k) {  // nothing behind the last site
                reinterpret_cast<uint8_t*>(w0)[k] = 0;
                reinterpret_cast<uint8_t*>(w1)[k] = 0;
            }
        } else {
            const uint32_t a = *p0, b = *p1, ev = pick(m, b, a), od = pick(m, a, b);
            const uint2 lo = unpack8(ev & 15u, od & 15u), hi = unpack8(ev >> 4, od >> 4);
            if (wide) {
                *reinterpret_cast<uint4*>(site) = make_uint4(lo.x, lo.y, hi.x, hi.y);
            } else {
                s4[0] = lo.x;
                if (left > 4u) s4[1] = lo.y;
                if (left > 8u) s4[2] = hi.x;
                if (left > 12u) s4[3] = hi.y;
            }
        }
    }
}

// The bit-packed layout's words (the same streams) <-> the words beside tags.
template <bool PACK>
__global__ void __launch_bounds__(256) k_stream_words(uint32_t* words, uint64_t* P, uint64_t n) {
    chain_begin();
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        if constexpr (PACK) P[i] = words[i];  // tag 0
        else words[i] = (uint32_t)P[i];
    }
}

// Series entries start from their constant terms.
__global__ void k_series_init(int32_t* E, int32_t* M, int32_t e, int32_t m, uint64_t n) {
    chain_begin();
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        if (E) E[i] = e;
        if (M) M[i] = m;
    }
}

template <int DIM, bool EA, int S, bool HELD>
cudaError_t launch_strips(StreamStrips P, uint64_t copies, int sm_count, uint32_t T, cudaStream_t s) {
    auto kern = k_stream_strips<DIM, EA, S, HELD>;
    int per_sm = 0;
    const size_t smem = HELD ? 16ull * ((stream_plane_words(P.N) / 2u + P.Gc - 1u) / P.Gc) : 0u;
    cudaError_t e = cudaSuccess;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (int)T, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
    const uint64_t batch = (uint64_t)sm_count / P.Gc;  // copies per launch, one CTA per SM
    for (uint64_t c0 = 0; c0 < copies; c0 += batch) {
        const uint64_t n = copies - c0 < batch ? copies - c0 : batch;
        P.copy0 = (uint32_t)c0;
        void* args[] = {&P};
        e = cudaLaunchCooperativeKernel((const void*)kern, dim3((uint32_t)(n * P.Gc)), dim3(T), args, smem, s);
        count_launch();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

size_t stream_plane_words(uint32_t N) { return 2ull * ((N / 2u + 31u) / 32u); }

cudaError_t launch_stream_convert(int8_t* spins, uint64_t* P, const uint32_t* mask, int dim, uint32_t L, uint64_t copies,
                                  bool pack, cudaStream_t s) {
    const uint32_t N = L * L * (dim == 3 ? L : 1u);
    const uint64_t chunks = copies * ((N + 15u) >> 4);
    uint64_t blocks = (chunks + 255u) / 256u;
    if (blocks > 152ull * 32ull) blocks = 152ull * 32ull;
    auto kern = dim == 2 ? (pack ? k_stream_convert<2, true> : k_stream_convert<2, false>)
                         : (pack ? k_stream_convert<3, true> : k_stream_convert<3, false>);
    return launch_chained(kern, dim3((uint32_t)blocks), 256, s, spins, P, mask, L, N, copies);
}

cudaError_t launch_stream_words(uint32_t* words, uint64_t* P, uint64_t n, bool pack, cudaStream_t s) {
    uint64_t blocks = (n + 255u) / 256u;
    if (blocks > 152ull * 32ull) blocks = 152ull * 32ull;
    auto kern = pack ? k_stream_words<true> : k_stream_words<false>;
    return launch_chained(kern, dim3((uint32_t)blocks), 256, s, words, P, n);
}

cudaError_t launch_stream_strips(const StreamStrips& P0, int dim, uint64_t copies, int sm_count, cudaStream_t s) {
    StreamStrips P = P0;
    const PlaneShape g = plane_shape((uint32_t)dim, P.L, P.N);
    // one CTA per SM over all copies (copies beyond that in further launches), eight
    // words or more each
    uint64_t per_copy = copies < (uint64_t)sm_count ? (uint64_t)sm_count / copies : 1u;
    if (per_copy * 8u > g.PW) per_copy = g.PW / 8u;
    if (per_copy < 1u) per_copy = 1u;
    P.Gc = (uint32_t)per_copy;
    P.ncopies = copies;
    const uint32_t words = (g.PW + P.Gc - 1u) / P.Gc;
    // words within D bits of a run's ends are read by other CTAs
    P.edge = P.Gc == 1u ? 0u : ((dim == 3 ? g.A : g.s) + 31u) / 32u + 2u;
    // four threads per word while they make at most four warps per scheduler
    // (2100 cycles for a word per thread, 420 per warp and quarter)
    const bool split = words <= 128u;
    // runs with more words inside than at their ends are held in shared memory, so that only
    // the ends wait for L2 (L = 1000, 100 sweeps: 416 -> 331 us; with a word per thread the
    // choice for every word costs more than it brings: L = 1600 456 -> 466, L = 3000 459 -> 505)
    const bool held = dim == 2 && split && 4u * P.edge <= words;
    const uint32_t items = split ? 4u * words : words;
    const uint32_t iters = (items + kStripMaxThreads - 1u) / kStripMaxThreads;
    const uint32_t T = ((items + iters - 1u) / iters + 31u) / 32u * 32u;
    if (P.Eser || P.Mser) {
        const uint64_t n = (uint64_t)(P.n_half / 2u) * copies;
        const uint64_t blocks = (n + 255u) / 256u;
        k_series_init<<<(uint32_t)(blocks < 1024u ? blocks : 1024u), 256, 0, s>>>(P.Eser, P.Mser, -dim * (int32_t)P.N,
                                                                                 (int32_t)P.N, n);
        count_launch();
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
#define GBMC_STRIPS(D_, A_)                                                                  \
    (split ? launch_strips<D_, A_, 4, false>(P, copies, sm_count, T, s)                      \
           : launch_strips<D_, A_, 1, false>(P, copies, sm_count, T, s))
    if (held) return launch_strips<2, false, 4, true>(P, copies, sm_count, T, s);
    if (dim == 2) return GBMC_STRIPS(2, false);
    return P.bond ? GBMC_STRIPS(3, true) : GBMC_STRIPS(3, false);
#undef GBMC_STRIPS
}

}  // namespace gbmc
