// Wide frame decoder: a frame pair's states spread over many lanes, its
// survivors in shared memory.
//
// Streams of few frames leave most of the chip idle in the kernels of
// vd_stream.cuh, where one lane carries all 64 states of a pair (K=7): a
// call then takes the latency of one warp, whatever its length.  Here L lanes share a
// pair (NR = 2^(K-1) / L registers each, 8 in the compiled forms), so a
// stage is a short dependent chain instead of some 260 issue slots, the
// survivor records (the same as StreamCfg's embedded forms: 3-bit fields
// every three stages for K=7, 2-bit fields every two for K=9) stay in shared
// memory, and the traceback starts from there without a trip to global
// memory.  Same frames, ties, metrics and bits as forward_pair: Eq. BM, Eq.
// PM, Eq. SP0, Algorithms 1 and 2, the frames of Sec. III.
//
// Registers and phases are those of vd_stream.cuh: register R (lane = its top
// log2 L bits) holds at stage tau the metric of state ROTR^tau(R), so the
// butterfly partners of stage tau differ in bit tau mod (K-1).  Where that
// is a lane bit the partner's metric comes by one shuffle, and the lane that
// holds the even (odd) register computes the butterfly's first (second) right
// state.  Both codes satisfy the corollary of Thm. 2 (complement outputs), so
// either lane adds A[a] to its own metric and the complement to the other's;
// only the mark of the odd candidate differs, and no per-state select is needed.
//
// What bounds it: one warp's latency.  A K=7 stage is 21 ALU and 21 FMA-pipe
// instructions of 47 (both pipes take a warp instruction every other cycle, so
// 42 cycles) around a chain of add (4 cycles) and fused add+max (6), after a
// shuffle (24) in half of the phases; measured 80 cycles a stage alone on a
// scheduler, 54 with two warps, 15 a stage for the traceback.  L = 8 for K=7:
// with 16 lanes four of six phases would shuffle and the branch metrics,
// which do not shrink with L, would weigh double; with 4 lanes the survivors
// of a warp's 16 frames would fill a quarter of the SM's shared memory.  L = 32 for K=9:
// its record is four times as large, and one pair per warp lets five warps share an
// SM.  Every branch in the loop over chunks is taken by all lanes or none: a
// store kept to some lanes made the shuffles resynchronise the warp and cost
// 15 cycles a stage.  Measured (us per vd_decode call, against one lane (K=7) or four (K=9) per
// pair): K=7, 100,003 bits 22 against 101; K=9, 12,000 bits 44 against 351.
//
// Branch metrics: the received values are staged in shared memory as one byte
// w = l + 128 each, frame 0 and frame 1 of the pair side by side per stage.
// A lane's part of the output pattern is a sign per (phase, output), folded
// into one multiply-add: u = SC (w - 1) or SC (255 - w), the scaled l + 127
// of Eq. BM with the lane's sign.
//
// Normalisation: every chunk of K-1 stages subtracts the minimum over lane
// 0's registers only.  These are the states whose last r = log2 L inputs are
// zero; any state shares its older inputs with one of them, and the two
// metrics come from a common ancestor r stages back, so no state is more than
// X = 2 B r below that minimum: it is brought to X, and every metric stays in
// [0, X + 254 DMAX + 2 U B].  A frame that starts from the reset state sets
// state 0 to HT and the others to 0 when its first stage arrives (its metrics
// are all equal before); if fewer than K-1 stages of that chunk remain, the
// chunk's normalisation leaves that frame alone, and its metrics stay
// within HT + 2 (2 U - 1) B.
#pragma once
#include <cooperative_groups.h>

#include "vd_stream.cuh"

namespace vd {

struct WideParams {
    const int8_t *llr;      // depunctured received LLRs, [T][beta], int8
    int64_t n_info, T, f, v;
    int64_t n_win, n_pairs;
    uint32_t flags;         // bit0: terminated, bit1: start state unknown
    int32_t wpad;           // padded frame length (a multiple of K-1), the same for every pair
    int32_t rec0;           // first record kept (the first of a chunk): no frame decodes a stage before it
    uint32_t *out;          // packed decoded bits, LSB-first
    int32_t *pm_out;        // optional [n_win][2^(K-1)] canonical final metrics
};

template <int K, int BETA, uint64_t GENS, int L>
struct WideCfg {
    using C = Code<K, BETA, GENS>;
    static constexpr int NB = C::NB, NS = C::NS, U = NB;
    static constexpr int NR = NS / L, LR = ilog2(NR), LB = NB - LR;   // registers per lane, register / lane bits
    static constexpr int ES = NB % 3 == 0 ? 3 : 2;        // stages per record
    static constexpr int SC = 1 << ES;
    static constexpr int FW = ES == 3 ? 4 : 2, RPW = 16 / FW, NWE = NR / RPW;
    static constexpr int ROW = NS / RPW;                  // words of one pair's record: register R in word R / RPW
    static constexpr int LW = BETA <= 2 ? 1 : 2;          // staged words per stage of a pair
    static constexpr int X = 2 * C::B * LB;               // see above
    static constexpr int TOP_STEADY = X + 254 * C::DMAX + 2 * U * C::B;
    static constexpr int TOP_RESET = C::HT + 2 * (2 * U - 1) * C::B;
    static_assert(NR % RPW == 0 && NWE >= 1 && U % ES == 0 && NB <= 8, "record layout");
    static_assert(SC * TOP_STEADY + SC - 1 <= 65535 && SC * TOP_RESET + SC - 1 <= 65535, "metric range");
    static_assert(C::lv() == (1u << BETA) - 1u && C::mv() == (1u << BETA) - 1u, "complement branch outputs");
    // output b at phase ph as a parity of lane bits: the part of alpha that the lane bits contribute
    __host__ __device__ static constexpr uint32_t lane_mask(int ph, int b) {
        uint32_t m = 0;
        for (int i = 0; i < LB; ++i)
            m |= ((C::alpha(C::rotr(1u << (LR + i), ph) >> 1) >> b) & 1u) << i;
        return m;
    }
    // shared memory of one warp: staged values, then records; the packed
    // groups of decoded bits (a byte per K-1 stages and frame) reuse the staged values
    __host__ __device__ static constexpr size_t pair_bytes(int wpad, int rec0) {
        return ((size_t)wpad * LW + (size_t)(wpad / ES - rec0) * ROW) * 4u;
    }
};

// Received bytes of a pair's two frames into its staged words: w = l + 128
// per byte, 128 (l = 0) outside a frame.  A step of 12 bytes per frame (6
// stages of beta = 2, 4 of beta = 3) is three aligned words shifted into
// place and three or four stores; the L lanes take the steps in turn.
template <int BETA, int LW, int L>
__device__ __forceinline__ void wide_stage_pair(const int8_t *base0, const int8_t *base1, int w0, int w1, int wpad,
                                                uint32_t *dst, int lane) {
    constexpr int SPS = 12 / BETA;   // stages per step
    const int hi0 = w0 * BETA, hi1 = w1 * BETA;
    const int off0 = (wpad - w0) * BETA, off1 = (wpad - w1) * BETA;
    constexpr int D = 4;             // steps in flight
    for (int k0 = lane; k0 * SPS < wpad; k0 += D * L) {
        ChunkRaw<3> r0[D], r1[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            r0[i].fast = r1[i].fast = false;
            if ((k0 + i * L) * SPS < wpad) {
                fetch_chunk<3>(base0, 12 * (k0 + i * L) - off0, hi0, r0[i]);
                fetch_chunk<3>(base1, 12 * (k0 + i * L) - off1, hi1, r1[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const int k = k0 + i * L;
            if (k * SPS < wpad) {
                uint32_t a[3] = {0u, 0u, 0u}, b[3] = {0u, 0u, 0u};
                const int v0 = 12 * k - off0, v1 = 12 * k - off1;
                if (v0 > -12 && v0 < hi0) finish_chunk<3>(base0, v0, hi0, r0[i], a);   // else wholly outside
                if (v1 > -12 && v1 < hi1) finish_chunk<3>(base1, v1, hi1, r1[i], b);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    a[j] ^= 0x80808080u;
                    b[j] ^= 0x80808080u;
                }
                if constexpr (BETA == 2) {
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        *reinterpret_cast<uint2 *>(dst + 6 * k + 2 * j) =
                            make_uint2(prmt(a[j], b[j], 0x5410u), prmt(a[j], b[j], 0x7632u));
                } else {
                    static_assert(BETA == 2 || BETA == 3, "staged layouts");
                    // stage i of the step: bytes 3 i .. 3 i + 2, byte 3 zero
                    auto three = [](const uint32_t (&x)[3], int q) {
                        const uint32_t y = q == 0 ? x[0] : q == 3 ? x[2] >> 8 : funnel_r(x[q - 1], x[q], 32u - 8u * q);
                        return y & 0x00FFFFFFu;
                    };
                    uint4 *d = reinterpret_cast<uint4 *>(dst + 8 * k);
                    d[0] = make_uint4(three(a, 0), three(b, 0), three(a, 1), three(b, 1));
                    d[1] = make_uint4(three(a, 2), three(b, 2), three(a, 3), three(b, 3));
                }
            }
        }
    }
}

// The forward procedure over nchunks chunks of U = K-1 stages: P[] in and out.
template <int K, int BETA, uint64_t GENS, int L, int PPW>
struct WideForward {
    using Cfg = WideCfg<K, BETA, GENS, L>;
    using C = typename Cfg::C;
    static constexpr int NB = Cfg::NB, NR = Cfg::NR, LR = Cfg::LR, LB = Cfg::LB, U = Cfg::U, ES = Cfg::ES;
    static constexpr int SC = Cfg::SC, LW = Cfg::LW, NWE = Cfg::NWE, RPW = Cfg::RPW, FW = Cfg::FW;
    static constexpr uint32_t H = 0x00010001u;
    static constexpr uint32_t FM = ((1u << ES) - 1u) * H;
    static constexpr uint32_t SEED = (uint32_t)(SC * Cfg::X) * H;

    // stg: this pair's staged words; rec: this lane's words of record rec0
    // (rows of PPW pairs), rec0 the first of a chunk; reset: stage at which frame h
    // starts from the reset state (-1: none).
    // MODE: keep the records from rec0 on, none of them, or all of them.
    enum Mode { FROM_REC0, NONE, ALL };
    template <Mode MODE = FROM_REC0>
    __device__ __forceinline__ static void run(uint32_t (&P)[NR], const uint32_t *stg, int nchunks, uint32_t *rec,
                                               int rec0, int reset0, int reset1, int lane) {
        const uint32_t one = threadIdx.y + 1u;   // 1, unknown to the compiler: keeps multiply-adds on the FMA pipe
        const uint32_t m1 = 0u - one, fwmul = one << FW;
        // per parity mask over the lane bits: u = w mul + add (only the masks in use cost registers)
        uint32_t mul[1 << LB], add[1 << LB];
#pragma unroll
        for (int m = 0; m < (1 << LB); ++m) {
            const bool neg = __popc((uint32_t)lane & (uint32_t)m) & 1;
            mul[m] = neg ? 0u - (uint32_t)SC : (uint32_t)SC;
            add[m] = neg ? (uint32_t)(255 * SC) * H : 0u - (uint32_t)SC * H;
        }
        uint32_t xm[LB];
#pragma unroll
        for (int i = 0; i < LB; ++i) xm[i] = (((uint32_t)lane >> i) & 1u) * H;

        // staged words of the chunk: the words of stages S - S % 4 .. S are replaced
        // by the next chunk's as soon as stage S has read the last of them
        uint32_t w[U * LW];
        constexpr int VL = (U * LW) % 4 == 0 ? 4 : 2;   // words per load
        const uint32_t *wp = stg;
        auto load = [&](int i) {
            if constexpr (VL == 4) {
                const uint4 x = *reinterpret_cast<const uint4 *>(wp + i);
                w[i] = x.x; w[i + 1] = x.y; w[i + 2] = x.z; w[i + 3] = x.w;
            } else {
                const uint2 x = *reinterpret_cast<const uint2 *>(wp + i);
                w[i] = x.x; w[i + 1] = x.y;
            }
        };
#pragma unroll
        for (int i = 0; i < U * LW; i += VL) load(i);
        uint32_t sub = SEED;
        uint32_t keepn = 0xFFFFFFFFu;   // halves that the next normalisation may shift
        // One chunk.  RESET: a frame of the warp may start in it; STORE: its
        // records are kept.  Straight-line code otherwise: a branch per stage
        // would keep the compiler from overlapping the branch metrics of the
        // next stages with the dependent chain of this one.
        auto chunk = [&](auto Reset, auto Store, int c) {
            constexpr bool RESET = decltype(Reset)::value, STORE = decltype(Store)::value;
            if (c + 1 < nchunks) wp += U * LW;   // the last chunk loads its own words again
            const uint32_t tn = sub_s16x2(SEED, sub) & keepn;
            keepn = 0xFFFFFFFFu;
            static_for<U>([&](auto Sc) {
                constexpr int S = decltype(Sc)::value;
                constexpr int PH = S, KS = S % ES;
                constexpr uint32_t OFF = H << KS;
                [[maybe_unused]] const int tau = c * U + S;
                if (RESET && (tau == reset0 || tau == reset1)) {
                    const uint32_t hm = (tau == reset0 ? 0xFFFFu : 0u) | (tau == reset1 ? 0xFFFF0000u : 0u);
#pragma unroll
                    for (int r = 0; r < NR; ++r)
                        P[r] = (P[r] & ~hm) | ((r == 0 && lane == 0) ? ((uint32_t)(SC * C::HT) * H) & hm : 0u);
                    if (S == 0) {
                        // this stage's folded normalisation must not shift the new start
                        if (tn & hm) {
#pragma unroll
                            for (int r = 0; r < NR; ++r) P[r] = sub_s16x2(P[r], tn & hm);
                        }
                    } else {
                        keepn &= ~hm;
                    }
                }
                // ---- branch metrics (Eq. BM): scaled, biased by B, both frames
                uint32_t u[BETA];
#pragma unroll
                for (int b = 0; b < BETA; ++b) {
                    const uint32_t x = LW == 1 ? prmt(w[S], 0u, 0x4040u | (uint32_t)b | ((uint32_t)(b + 2) << 8))
                                               : prmt(w[S * LW], w[S * LW + LW - 1],
                                                      0x3030u | (uint32_t)b | ((uint32_t)(b + 4) << 8));
                    const uint32_t m = Cfg::lane_mask(PH, b);
                    u[b] = imad(x, mul[m], add[m]);
                }
                if constexpr (((S + 1) * LW) % VL == 0) load((S + 1) * LW - VL);
                // In a phase whose butterfly bit is a lane bit, the lane that holds the
                // odd register carries the odd candidate's mark in all its metrics:
                // added to one u, it reaches every pattern sum.
                constexpr bool CROSS = PH >= LR;
                constexpr int lb = CROSS ? PH - LR : 0;
                const uint32_t own = CROSS ? xm[lb] << KS : 0u;
                if constexpr (CROSS) u[BETA - 1] += own;
                constexpr int HALF = 1 << (BETA - 1), FULL = (1 << BETA) - 1;
                uint32_t E[1 << BETA];
                E[0] = u[BETA - 1];
#pragma unroll
                for (int b = 0; b < BETA - 1; ++b) {
#pragma unroll
                    for (int x = 0; x < (1 << b); ++x) {
                        E[x | (1 << b)] = (E[x] + (uint32_t)(254 * SC) * H) - u[b];
                        E[x] = E[x] + u[b];
                    }
                }
                // complement patterns: 2 B minus the pattern's metric
                constexpr uint32_t CC = (uint32_t)(2 * C::B * SC) * H;
                const uint32_t cc = CROSS ? CC + 2u * own : CC;
#pragma unroll
                for (int x = 0; x < HALF; ++x) E[x ^ FULL] = imad(E[x], m1, cc);
                uint32_t O[1 << BETA];   // the other candidate's: marked where E is not
#pragma unroll
                for (int x = 0; x <= FULL; ++x) {
                    if constexpr (CROSS) O[x] = imad(E[x], m1, CC + OFF);   // complement of pattern x
                    else O[x] = imad(E[x], one, OFF);
                }
                if constexpr (S == 0) {
#pragma unroll
                    for (int x = 0; x <= FULL; ++x) {
                        E[x] = add_u16x2(E[x], tn);
                        O[x] = add_u16x2(O[x], tn);
                    }
                }
                // ---- add-compare-select (Eq. PM), decisions in the low bits (Eq. SP0)
                if constexpr (!CROSS) {
#pragma unroll
                    for (int ra = 0; ra < NR; ++ra) {
                        if (ra & (1 << PH)) continue;
                        const int rb = ra | (1 << PH);
                        const uint32_t a = C::alpha(C::rotr((uint32_t)ra, PH) >> 1);
                        const uint32_t Pa = P[ra], Pb = P[rb];
                        const uint32_t cb0 = add_u16x2(Pb, O[a ^ FULL]), cb1 = add_u16x2(Pb, O[a]);
                        P[ra] = addmax_u16x2(Pa, E[a], cb0);
                        P[rb] = addmax_u16x2(Pa, E[a ^ FULL], cb1);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const uint32_t a = C::alpha(C::rotr((uint32_t)r, PH) >> 1);
                        const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, P[r], 1 << lb);
                        P[r] = addmax_u16x2(P[r], E[a], add_u16x2(o, O[a]));
                    }
                }
                if constexpr (KS == ES - 1) {
                    if constexpr (STORE) {
                        uint32_t rw[NWE];
#pragma unroll
                        for (int m = 0; m < NWE; ++m) {
                            const int r0 = RPW * m;
                            if constexpr (RPW == 4) {
                                const uint32_t x = prmt(P[r0], P[r0 + 2], 0x6240u);
                                const uint32_t y = prmt(P[r0 + 1], P[r0 + 3], 0x6240u);
                                rw[m] = (x & 0x07070707u) | (imad(y, fwmul, 0u) & ~0x07070707u);
                            } else {
                                const uint32_t x0 = prmt(P[r0], P[r0 + 4], 0x6240u);
                                const uint32_t x1 = imad(prmt(P[r0 + 1], P[r0 + 5], 0x6240u), fwmul, 0u);
                                const uint32_t x2 = imad(prmt(P[r0 + 2], P[r0 + 6], 0x6240u), one << 4, 0u);
                                const uint32_t x3 = imad(prmt(P[r0 + 3], P[r0 + 7], 0x6240u), one << 6, 0u);
                                const uint32_t a = (x0 & 0x03030303u) | (x1 & ~0x03030303u);
                                const uint32_t b = (x2 & 0x30303030u) | (x3 & ~0x30303030u);
                                rw[m] = (a & 0x0F0F0F0Fu) | (b & ~0x0F0F0F0Fu);
                            }
                        }
                        uint32_t *d = rec + (S / ES) * (PPW * Cfg::ROW);
                        if constexpr (NWE == 1) *d = rw[0];
                        else if constexpr (NWE == 2) *reinterpret_cast<uint2 *>(d) = make_uint2(rw[0], rw[1]);
                        else
#pragma unroll
                            for (int i = 0; i < NWE; ++i) d[i] = rw[i];
                    }
#pragma unroll
                    for (int r = 0; r < NR; ++r) P[r] &= ~FM;
                }
            });
            // the minimum over lane 0's registers, for the next chunk's first stage
            sub = __shfl_sync(0xFFFFFFFFu, min_tree<NR>(P), 0, L);
            if constexpr (STORE) rec += (U / ES) * (PPW * Cfg::ROW);
        };
        const int c0 = rec0 / (U / ES);
        // chunks [ra, rz] hold every frame start of the warp
        const int rhi = reset0 > reset1 ? reset0 : reset1;
        const int rlo = reset0 < 0 ? reset1 : (reset1 < 0 || reset0 < reset1) ? reset0 : reset1;
        const int ra = (int)(__reduce_min_sync(0xFFFFFFFFu, rlo < 0 ? 0x7FFFFFFFu : (unsigned)rlo) / U);
        const int rz = __reduce_max_sync(0xFFFFFFFFu, rhi) / U;
        for (int c = 0; c < nchunks; ++c) {
            const bool store = MODE == ALL || (MODE == FROM_REC0 && c >= c0);
            if (c >= ra && c <= rz) {
                if (store) chunk(std::true_type{}, std::true_type{}, c);
                else chunk(std::true_type{}, std::false_type{}, c);
            } else if (store) {
                chunk(std::false_type{}, std::true_type{}, c);
            } else {
                chunk(std::false_type{}, std::false_type{}, c);
            }
        }
    }

    // The best state of frame h over the group's L lanes (the lowest index
    // among equals; states with a bit of `unreach` left out) and the smallest metric.
    __device__ __forceinline__ static uint32_t best_state(const uint32_t (&P)[NR], int h, int lane, uint32_t unreach,
                                                          uint32_t &mn) {
        uint32_t best = 0;
        mn = 0xFFFFu;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const uint32_t m = h ? (P[r] >> 16) : (P[r] & 0xFFFFu);
            const uint32_t Rg = ((uint32_t)lane << LR) | (uint32_t)r;
            const uint32_t key = (Rg & unreach) ? 0u : ((m << 16) | (0xFFFFu - Rg));
            best = best > key ? best : key;
            mn = mn < m ? mn : m;
        }
#pragma unroll
        for (int m = 1; m < L; m <<= 1) {
            const uint32_t x = __shfl_xor_sync(0xFFFFFFFFu, best, m);
            const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, mn, m);
            best = best > x ? best : x;
            mn = mn < y ? mn : y;
        }
        return 0xFFFFu - (best & 0xFFFFu);
    }

    // Traceback over one group of K-1 stages of frame h; rp: the pair's last record of the group.
    __device__ __forceinline__ static void back(uint32_t &Rc, const uint32_t *&rp, int h) {
        static_for<NB / ES>([&](auto jc) {
            constexpr int j = decltype(jc)::value;
            constexpr int ph0 = NB - ES * (j + 1);   // phase of the record's first stage
            constexpr uint32_t m = ((1u << ES) - 1u) << ph0;
            const uint32_t word = rp[Rc / RPW];
            rp -= PPW * Cfg::ROW;
            const uint32_t sh = (uint32_t)FW * (Rc & (uint32_t)(RPW - 1)) + 16u * (uint32_t)h;
            Rc = (Rc & ~m) | (__funnelshift_r(word, word, sh - (uint32_t)ph0) & m);
        });
    }

    // Subtracts each frame's smallest metric from all its metrics.
    __device__ __forceinline__ static void canonical(uint32_t (&P)[NR]) {
        uint32_t mn = min_tree<NR>(P);
#pragma unroll
        for (int m = 1; m < L; m <<= 1) mn = min_u16x2(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, m));
#pragma unroll
        for (int r = 0; r < NR; ++r) P[r] -= mn;   // no half is below its minimum: no borrow
    }
};

// One warp per block: PPW frame pairs (2q, 2q+1), L lanes each.
template <int K, int BETA, uint64_t GENS, int L, int PPW>
__global__ void __launch_bounds__(32, 8) wide_kernel(const WideParams p) {
    using Cfg = WideCfg<K, BETA, GENS, L>;
    using Fw = WideForward<K, BETA, GENS, L, PPW>;
    constexpr int NB = Cfg::NB, NS = Cfg::NS, NR = Cfg::NR, LR = Cfg::LR, ES = Cfg::ES, SC = Cfg::SC;
    constexpr int LW = Cfg::LW, ROW = Cfg::ROW;
    extern __shared__ __align__(16) uint32_t vd_wide_smem[];
    const int wlane = (int)threadIdx.x;
    const int group = wlane / L, lane = wlane % L;
    // with one pair per warp every group of lanes decodes that pair: no lane
    // takes a branch of its own, and equal words are stored to equal places
    const int ga = PPW == 1 ? 0 : group;
    const int64_t q = (int64_t)blockIdx.x * PPW + ga;
    const bool active = q < p.n_pairs && (PPW > 1 || group == 0);
    const int wpad = p.wpad, stg_words = wpad * LW;
    uint32_t *stg = vd_wide_smem + (size_t)ga * stg_words;
    uint32_t *recs = vd_wide_smem + (size_t)PPW * stg_words + (size_t)ga * ROW;
    constexpr int row = PPW * ROW;

    int tau0[2], tauo[2], taue[2], reset[2];
    int W[2];
    bool known[2], term[2], valid[2];
    int64_t o0[2];
    const int8_t *base[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t s = 2 * q + h;
        const FrameTask ft = frame_task(p.llr, p.out, nullptr, s, p.n_win, p.n_info, p.T, p.f, p.v, p.flags);
        valid[h] = ft.valid != 0;
        known[h] = ft.known != 0;
        term[h] = ft.term != 0;
        W[h] = valid[h] ? (int)(ft.b - ft.a) : 0;
        tau0[h] = wpad - W[h];
        tauo[h] = valid[h] ? tau0[h] + (int)(ft.o - ft.a) : wpad;
        taue[h] = valid[h] ? tau0[h] + (int)(ft.e - ft.a) : wpad;
        reset[h] = known[h] ? tau0[h] : -1;
        o0[h] = ft.o;
        base[h] = p.llr + ft.a * BETA;
    }
    if (PPW > 1 || group == 0) wide_stage_pair<BETA, LW, L>(base[0], base[1], W[0], W[1], wpad, stg, lane);
    __syncwarp();

    uint32_t P[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) P[r] = Fw::SEED;
    Fw::run(P, stg, wpad / NB, recs + lane * Cfg::NWE, p.rec0, reset[0], reset[1], lane);

    // ---- traceback start (Algorithm 2): the best state, the lowest index among equals
    uint32_t R[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // states a reset frame of fewer than K-1 stages cannot reach are left out
        const uint32_t unreach = (known[h] && W[h] < NB) ? ((1u << (NB - W[h])) - 1u) : 0u;
        uint32_t mn;
        const uint32_t best = Fw::best_state(P, h, lane, unreach, mn);
        R[h] = term[h] ? 0u : best;
        if (p.pm_out && valid[h] && active) {
            int32_t *dst = p.pm_out + (2 * q + h) * NS + ((int64_t)lane << LR);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const uint32_t m = h ? (P[r] >> 16) : (P[r] & 0xFFFFu);
                dst[r] = ((int32_t)m - (int32_t)mn) / SC;
            }
        }
    }
    __syncwarp();

    // ---- traceback (Algorithm 2): lanes 0 and 1 of a group follow its two
    // frames (the others repeat them).  A register index at the top of a group
    // of K-1 stages is the group's decoded bits, stage by stage from bit 0.
    const int h = lane & 1;
    uint32_t Rc = h ? R[1] : R[0];
    uint8_t *grp = reinterpret_cast<uint8_t *>(stg);   // frame h, group g at byte 2 g + h
    const int g0 = p.rec0 / (NB / ES);
    const uint32_t *rp = recs + (wpad / ES - 1 - p.rec0) * row;   // the last record
    for (int g = wpad / NB - 1; g >= g0; --g) {
        if ((PPW > 1 || group == 0) && lane < 2) grp[2 * g + h] = (uint8_t)Rc;
        Fw::back(Rc, rp, h);
    }
    __syncwarp();

    // ---- decoded words: frames write whole words (f is a multiple of 32)
    if (active) {
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int nbits = taue[hh] - tauo[hh];
            uint32_t *dst = p.out + (o0[hh] >> 5);
            for (int w = lane; 32 * w < nbits; w += L) {
                const int t = tauo[hh] + 32 * w;
                const int g = t / NB, skip = t - g * NB;
                uint64_t acc = 0;
                constexpr int NG = (31 + NB - 1) / NB + 1;   // groups that 32 stages can touch
#pragma unroll
                for (int i = 0; i < NG; ++i)
                    if ((g + i) * NB < wpad) acc |= (uint64_t)grp[2 * (g + i) + hh] << (NB * i);
                acc >>= skip;
                const int left = nbits - 32 * w;
                dst[w] = (uint32_t)acc & (left >= 32 ? 0xFFFFFFFFu : ((1u << left) - 1u));
            }
        }
    }
}

// ------------------------------------------------------------- split frames
//
// A frame is a serial chain of W stages; where there are few frames and each is
// long (a packet decoded full length) that chain is all the time there is.
// Here a cluster of blocks decodes one frame in segments, all at once, and the
// result is exact:
//   * a segment of S chunks starts M chunks early from all-equal metrics.
//     After the warm-up its metrics differ from the true ones by a constant if
//     every survivor of the warm-up has one ancestor, which is nearly always so;
//   * a segment's metrics at its start (less their minimum) are compared
//     with the end of the segment before.  Equal metrics give equal decisions,
//     so when all agree, every segment is exact, from the first one (which
//     starts where the frame does) on.  Segments that disagree run again from
//     the metrics at the end of the segment before, until none disagrees: at
//     most as many rounds as segments, since each round settles one more;
//   * each segment is traced back from its best end state at first; then the
//     segments whose successor's traceback arrives in another state are traced again from
//     that state, as far as the two paths differ, until none changes.
// Segments go through the registers in pairs, as frames do in wide_kernel.
//
// What bounds it: the warm-up and the segment, (16 + S) (K-1) stages of 80
// (K=7) or 100 (K=9) cycles, and some five barriers of the cluster.  Four warps a block, one
// per scheduler (a second one on a scheduler costs 28 cycles a stage); clusters of 1 to 8
// blocks, as wide as keeps S at half the warm-up.  A frame of more than 8 (K=7: 256, K=9: 64 segments)
// times the chunks that fit a block, 136,704 or 49,152 stages, is left to the other forms.  Measured (us per vd_decode
// call, this form / wide / one lane per pair): K=7 full length, terminated, 3 dB, 4,096
// bits 14.7 / 209 / 1172, 30,000 bits 18.7 / - / 8452; K=9, 4,096 bits 20.8 / - /
// 2148; at 0 dB, where some segments run twice, 28.9 and 33.0.
struct SplitParams {
    const int8_t *llr;
    int64_t n_info, T, f, v;
    int64_t n_win;
    uint32_t flags;
    int32_t S, M;           // chunks of a segment, and of its warm-up
    uint32_t *out;
    int32_t *pm_out;
};

// Words of shared memory of a block of `warps` warps.
template <int K, int BETA, uint64_t GENS, int L>
struct SplitSmem {
    using Cfg = WideCfg<K, BETA, GENS, L>;
    static constexpr int PPW = 32 / L;
    int stg, rec, ve, gl, total;   // words per pair / per warp / per pair / in all / in all
    __host__ __device__ constexpr SplitSmem(int warps, int S, int M)
        : stg((S + M) * Cfg::U * Cfg::LW), rec(S * (Cfg::U / Cfg::ES) * PPW * Cfg::ROW), ve(Cfg::NS),
          gl((warps * PPW * 2 * S + 3) / 4),
          total(warps * (PPW * (stg + ve) + rec) + gl + (warps * PPW * 2 + 3) / 4 + 4) {}
};

template <int K, int BETA, uint64_t GENS, int L, int MAXT>
__global__ void __launch_bounds__(MAXT) split_kernel(const SplitParams p) {
    constexpr int PPW = 32 / L;
    using Cfg = WideCfg<K, BETA, GENS, L>;
    using Fw = WideForward<K, BETA, GENS, L, PPW>;
    constexpr int NB = Cfg::NB, NS = Cfg::NS, NR = Cfg::NR, LR = Cfg::LR, ES = Cfg::ES, SC = Cfg::SC, U = Cfg::U;
    constexpr int ROW = Cfg::ROW;
    extern __shared__ __align__(16) uint32_t vd_wide_smem[];
    auto cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
    const int warps = (int)blockDim.x / 32, warp = (int)threadIdx.x / 32, wlane = (int)threadIdx.x % 32;
    const int group = wlane / L, lane = wlane % L;
    const SplitSmem<K, BETA, GENS, L> sm(warps, p.S, p.M);
    const int pairs = warps * PPW, pair = warp * PPW + group;   // of this block
    const int gp = rank * pairs + pair;                         // the frame's pair: segments 2 gp, 2 gp + 1
    const int nseg = 2 * ranks * pairs;
    uint32_t *stg = vd_wide_smem + pair * sm.stg;
    uint32_t *recs = vd_wide_smem + pairs * sm.stg + warp * sm.rec + group * ROW;
    uint32_t *ve = vd_wide_smem + pairs * sm.stg + warps * sm.rec;   // metrics at the segments' ends, by state
    uint8_t *gl = reinterpret_cast<uint8_t *>(ve + pairs * NS);      // register index at the top of every chunk
    uint8_t *xs = gl + 4 * sm.gl;                                    // state each segment's traceback arrives in
    uint32_t *flag = ve + pairs * NS + sm.gl + (pairs * 2 + 3) / 4;
    auto sync = [&] {
        if (ranks == 1) __syncthreads();
        else cluster.sync();
    };
    // whether any thread of the cluster says yes; a barrier for all of them
    int round = 0;
    auto any_of = [&](bool yes) {
        const int mine = __syncthreads_or(yes);
        if (ranks == 1) return mine != 0;
        uint32_t *f = flag + (round++ & 1);
        if (threadIdx.x == 0) *f = (uint32_t)mine;
        cluster.sync();
        uint32_t all = 0;
        for (int k = 0; k < ranks; ++k) all |= *cluster.map_shared_rank(f, k);
        return all != 0;
    };

    const FrameTask ft = frame_task(p.llr, p.out, nullptr, (int64_t)(blockIdx.x / ranks), p.n_win, p.n_info, p.T, p.f,
                                    p.v, p.flags);
    const int W = (int)(ft.b - ft.a);
    const int wpad = (p.S + p.M) * U, seg = p.S * U;
    int w[2], reset[2];
    const int8_t *base[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // segment i ends (nseg - 1 - i) segments before the frame's end; its window begins
        // S + M chunks earlier or with the frame
        const int y = W - (nseg - 1 - (2 * gp + h)) * seg;
        const int x = y > wpad ? y - wpad : 0;
        w[h] = y > 0 ? y - x : 0;
        base[h] = ft.llr + (ft.a + x) * BETA;
        reset[h] = (ft.known && x == 0 && y > 0) ? wpad - w[h] : -1;
    }
    wide_stage_pair<BETA, Cfg::LW, L>(base[0], base[1], w[0], w[1], wpad, stg, lane);
    __syncwarp();

    // ---- forward: warm-up, then the segment, until its start is the end of the one before
    uint32_t P[NR], V[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) P[r] = Fw::SEED;
    Fw::template run<Fw::NONE>(P, stg, p.M, nullptr, 0, reset[0], reset[1], lane);
    Fw::canonical(P);
    const int first = p.M * U;
    const int rs0 = reset[0] >= first ? reset[0] - first : -1, rs1 = reset[1] >= first ? reset[1] - first : -1;
    bool run = true;
    while (true) {
        if (run) {
#pragma unroll
            for (int r = 0; r < NR; ++r) V[r] = P[r];
            Fw::template run<Fw::ALL>(P, stg + first * Cfg::LW, p.S, recs + lane * Cfg::NWE, 0, rs0, rs1, lane);
            Fw::canonical(P);
#pragma unroll
            for (int r = 0; r < NR; ++r) ve[pair * NS + ((lane << LR) | r)] = P[r];
        }
        sync();
        const uint32_t *own = ve + pair * NS;
        const uint32_t *prev = pair > 0 ? own - NS
                               : rank > 0 ? cluster.map_shared_rank(ve, rank - 1) + (pairs - 1) * NS : nullptr;
        uint32_t N[NR];
        bool bad = false;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int st = (lane << LR) | r;
            N[r] = (prev ? prev[st] >> 16 : V[r] & 0xFFFFu) | (own[st] << 16);
            bad |= N[r] != V[r];
        }
        run = __any_sync(0xFFFFFFFFu, bad);
        if (!any_of(run)) break;
        if (run) {
#pragma unroll
            for (int r = 0; r < NR; ++r) P[r] = N[r];
        }
    }

    // ---- traceback: lanes 0 and 1 of a group take its two segments
    const int h = lane & 1;
    const int si = 2 * gp + h;
    uint32_t R0 = 0;
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        uint32_t mn;
        const uint32_t unreach = (ft.known && W < NB) ? ((1u << (NB - W)) - 1u) : 0u;
        const uint32_t best = Fw::best_state(P, hh, lane, 2 * gp + hh == nseg - 1 ? unreach : 0u, mn);
        if (h == hh) R0 = (ft.term && 2 * gp + hh == nseg - 1) ? 0u : best;
        if (p.pm_out && 2 * gp + hh == nseg - 1) {   // canonical final metrics
            int32_t *dst = p.pm_out + (int64_t)(blockIdx.x / ranks) * NS + (lane << LR);
#pragma unroll
            for (int r = 0; r < NR; ++r) dst[r] = (int32_t)((hh ? (P[r] >> 16) : (P[r] & 0xFFFFu)) - mn) / SC;
        }
    }
    const bool tracer = lane < 2;
    const uint32_t *last = recs + (p.S * (U / ES) - 1) * (PPW * ROW);
    uint8_t *mygl = gl + (2 * pair + h) * p.S;
    if (tracer) {
        uint32_t Rc = R0;
        const uint32_t *rp = last;
        for (int g = p.S - 1; g >= 0; --g) {
            mygl[g] = (uint8_t)Rc;
            Fw::back(Rc, rp, h);
        }
        xs[2 * pair + h] = (uint8_t)Rc;
    }
    while (true) {
        sync();
        uint32_t Rc = R0;
        if (tracer && si < nseg - 1)
            Rc = 2 * pair + h + 1 < 2 * pairs ? xs[2 * pair + h + 1] : *cluster.map_shared_rank(xs, rank + 1);
        const bool change = tracer && Rc != R0;
        if (!any_of(change)) break;
        if (change) {
            R0 = Rc;
            const uint32_t *rp = last;
            int g = p.S - 1;
            for (; g >= 0 && mygl[g] != (uint8_t)Rc; --g) {   // from there on the path is the old one
                mygl[g] = (uint8_t)Rc;
                Fw::back(Rc, rp, h);
            }
            if (g < 0) xs[2 * pair + h] = (uint8_t)Rc;
        }
    }

    // ---- decoded words, in turn over the cluster's threads
    const int per = 2 * pairs * p.S;                   // chunks per block
    const int pad = nseg * seg - W;                    // stages before the frame's first one
    const int o = (int)(ft.o - ft.a) + pad, nbits = (int)(ft.e - ft.o);
    uint32_t *dst = ft.out + (ft.o >> 5);
    for (int wd = rank * (int)blockDim.x + (int)threadIdx.x; 32 * wd < nbits; wd += ranks * (int)blockDim.x) {
        const int t = o + 32 * wd, g = t / NB;
        uint64_t acc = 0;
        constexpr int NG = (31 + NB - 1) / NB + 1;   // chunks that 32 stages can touch
#pragma unroll
        for (int i = 0; i < NG; ++i)
            if (g + i < ranks * per) acc |= (uint64_t)cluster.map_shared_rank(gl, (g + i) / per)[(g + i) % per] << (NB * i);
        acc >>= t - g * NB;
        const int left = nbits - 32 * wd;
        dst[wd] = (uint32_t)acc & (left >= 32 ? 0xFFFFFFFFu : ((1u << left) - 1u));
    }
    if (ranks > 1) cluster.sync();   // no block leaves while another may read its shared memory
}

}  // namespace vd
