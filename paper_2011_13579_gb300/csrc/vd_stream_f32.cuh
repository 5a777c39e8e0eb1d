// Frame-pair decoder with fp16 received LLRs and fp32 path metrics (the
// precision study of Sec. IX-B: the channel values in half precision, the
// accumulated metrics in single precision).  Same frame plan, register
// rotation, lane split, survivor layout and traceback as the integer decoder;
// the two frames of a pair live in the two halves of 64-bit register pairs.
//
// Decisions: d = (c_odd >= c_even), read from the sign of c_odd - c_even
// computed from the same rounded candidates the maximum uses (an exact tie
// gives +0, so the odd predecessor wins it, as in Algorithm 1).  The metric of
// state 0 is subtracted from every metric every chunk, which
// keeps magnitudes (and so rounding) small; the reset start gives every state
// but 0 the metric -1e30, which no finite path metric approaches.
#pragma once
#include <cuda_fp16.h>

#include "vd_stream.cuh"

namespace vd {

template <int K, int BETA, uint64_t GENS, int L>
struct StreamCfgF32 {
    using C = Code<K, BETA, GENS>;
    static constexpr int NB = C::NB;
    static constexpr int NS = C::NS;
    static constexpr int NR = NS / L;
    static constexpr int LR = ilog2(NR);
    static constexpr int U = chunk_stages(K, 2 * BETA);   // 2 bytes per LLR
    static constexpr int UW = U * BETA / 2;               // 32-bit words per chunk per frame
    static constexpr int NW = NR / 16;                    // survivor words per lane per stage
    static_assert(NR == 16 || NR == 32, "half a decision word or a word per frame and lane");
    static_assert(C::lv() == (1u << BETA) - 1u && C::mv() == (1u << BETA) - 1u, "complement branch outputs");
    // output b at phase ph: the lane bits whose parity flips it
    __host__ __device__ static constexpr uint32_t lane_mask(int ph, int b) {
        uint32_t m = 0;
        for (int i = 0; i < NB - LR; ++i)
            m |= ((C::alpha(C::rotr(1u << (LR + i), ph) >> 1) >> b) & 1u) << i;
        return m;
    }
};

// Two floats in a register pair, frame 0 in the low word: the packed fp32
// operations round each half as the scalar ones do and take one issue slot.
using f32x2 = uint64_t;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void unpack2(f32x2 x, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 max2(f32x2 a, f32x2 b) {
    float a0, a1, b0, b1;
    unpack2(a, a0, a1);
    unpack2(b, b0, b1);
    return pack2(fmaxf(a0, b0), fmaxf(a1, b1));
}
__device__ __forceinline__ float half_at(uint32_t word, int hi) {
    const unsigned short bits = (unsigned short)(hi ? (word >> 16) : (word & 0xFFFFu));
    return __half2float(__ushort_as_half(bits));
}

template <int K, int BETA, uint64_t GENS, int L>
__device__ __forceinline__ bool forward_pair_f32(const FrameTask (&ft)[2], uint32_t *surv, int wpad_cap,
                                                 int wlane, int lane, unsigned gmask, int grp_base,
                                                 int *status, TbState &tb) {
    using Cfg = StreamCfgF32<K, BETA, GENS, L>;
    using C = typename Cfg::C;
    constexpr int NB = Cfg::NB, NR = Cfg::NR, LR = Cfg::LR, U = Cfg::U, UW = Cfg::UW, NW = Cfg::NW;
    constexpr float NEG = -1e30f;

    int64_t fa[2], fb[2], W[2];
    bool valid[2], known[2], term[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        fa[h] = ft[h].a;
        fb[h] = ft[h].b;
        valid[h] = ft[h].valid != 0;
        known[h] = ft[h].known != 0;
        term[h] = ft[h].term != 0;
        W[h] = valid[h] ? fb[h] - fa[h] : 0;
    }
    const int64_t Wmax = W[0] > W[1] ? W[0] : W[1];
    const int Wpad = (int)(((Wmax + U - 1) / U) * U);
    tb.t0 = -1;
    tb.tau_store = 0;
    if (Wpad > wpad_cap) {
        if (lane == 0) atomicOr(status, 1);
        return false;
    }
    int tau0[2], tauo[2], taue[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        tau0[h] = Wpad - (int)W[h];
        tauo[h] = valid[h] ? tau0[h] + (int)(ft[h].o - fa[h]) : Wpad;
        taue[h] = valid[h] ? tau0[h] + (int)(ft[h].e - fa[h]) : Wpad;
    }
    const int tau_store = tauo[0] < tauo[1] ? tauo[0] : tauo[1];
    const int reset0 = known[0] ? tau0[0] : -1;
    const int reset1 = known[1] ? tau0[1] : -1;

    const uint32_t one = threadIdx.y + 1u;                // 1, unknown to the compiler: multiply-adds stay on the FMA pipe
    const uint32_t minv = 0u - (one << 16) - one;         // 65535 (-65537) = 1 mod 2^32
    f32x2 P[NR];   // register r of both frames
#pragma unroll
    for (int r = 0; r < NR; ++r) P[r] = pack2(0.0f, 0.0f);

    // fp16 LLR bytes relative to each frame's first stage, fetched half a chunk ahead
    const int8_t *fbase0 = ft[0].llr + fa[0] * BETA * 2, *fbase1 = ft[1].llr + fa[1] * BETA * 2;
    const int32_t hi0 = valid[0] ? (int32_t)W[0] * BETA * 2 : 0, hi1 = valid[1] ? (int32_t)W[1] * BETA * 2 : 0;
    int32_t vb0 = -tau0[0] * BETA * 2, vb1 = -tau0[1] * BETA * 2;
    constexpr int HS = U / 2, HW = UW / 2;
    static_assert(U % 2 == 0 && (HS * BETA) % 2 == 0, "half a chunk is a whole number of words");

    // signs of the lane's part of each branch output, as +-1 in both halves, by
    // parity of the lane bits (only the masks in use cost registers)
    constexpr int LB = NB - LR;
    f32x2 sgn[1 << LB];
#pragma unroll
    for (int m = 0; m < (1 << LB); ++m) {
        const float x = (__popc((uint32_t)lane & (uint32_t)m) & 1) ? -1.0f : 1.0f;
        sgn[m] = pack2(x, x);
    }

    const int nchunks = Wpad / U;
    ChunkRaw<HW> nx0, nx1;
    if (nchunks > 0) {
        fetch_chunk<HW>(fbase0, vb0, hi0, nx0);
        fetch_chunk<HW>(fbase1, vb1, hi1, nx1);
    }
    for (int c = 0; c < nchunks; ++c) {
        uint32_t cw0[HW], cw1[HW];
        static_for<U>([&](auto Sc) {
            constexpr int S = decltype(Sc)::value;
            constexpr int PH = S % NB;
            const int tau = c * U + S;
            if constexpr (S % HS == 0) {
                const ChunkRaw<HW> cur0 = nx0, cur1 = nx1;
                const int32_t cb0 = vb0, cb1 = vb1;
                vb0 += HS * BETA * 2;
                vb1 += HS * BETA * 2;
                if (S == 0 || c + 1 < nchunks) {
                    fetch_chunk<HW>(fbase0, vb0, hi0, nx0);
                    fetch_chunk<HW>(fbase1, vb1, hi1, nx1);
                }
                finish_chunk<HW>(fbase0, cb0, hi0, cur0, cw0);
                finish_chunk<HW>(fbase1, cb1, hi1, cur1, cw1);
            }
            if (tau == reset0 || tau == reset1) {
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    float p0, p1;
                    unpack2(P[r], p0, p1);
                    const float start = (r == 0 && lane == 0) ? 0.0f : NEG;
                    P[r] = pack2(tau == reset0 ? start : p0, tau == reset1 ? start : p1);
                }
            }
            // ---- branch metrics (Eq. BM) of output patterns x < 2^(BETA-1); the complement's are the negatives
            f32x2 A[1 << (BETA - 1)];
            {
                f32x2 l[BETA];
#pragma unroll
                for (int b = 0; b < BETA; ++b) {
                    const int j = (S % HS) * BETA + b;
                    l[b] = pack2(half_at(cw0[j >> 1], j & 1), half_at(cw1[j >> 1], j & 1));
                    if (Cfg::lane_mask(PH, b) != 0u) l[b] = mul2(l[b], sgn[Cfg::lane_mask(PH, b)]);
                }
                // sums in the order of the output bits: ((+-l_0) +- l_1) +- l_2
                A[0] = l[0];
                if constexpr (BETA > 1) {
                    f32x2 T[1 << BETA];
                    T[0] = l[0];
                    T[1] = mul2(l[0], pack2(-1.0f, -1.0f));
#pragma unroll
                    for (int b = 1; b < BETA; ++b) {
#pragma unroll
                        for (int x = 0; x < (1 << b); ++x) {
                            T[x | (1 << b)] = sub2(T[x], l[b]);
                            T[x] = add2(T[x], l[b]);
                        }
                    }
#pragma unroll
                    for (int x = 0; x < (1 << (BETA - 1)); ++x) A[x] = T[x];
                }
            }
            constexpr uint32_t FULL = (1u << BETA) - 1u;
            auto plus = [&](f32x2 p, uint32_t a) { return a <= FULL / 2 ? add2(p, A[a]) : sub2(p, A[a ^ FULL]); };
            auto minus = [&](f32x2 p, uint32_t a) { return a <= FULL / 2 ? sub2(p, A[a]) : add2(p, A[a ^ FULL]); };
            // ---- add-compare-select (Eq. PM) and decisions (Eq. SP0): the sign of
            // c_odd - c_even (clear: odd wins or ties) of register r goes to bits r % 16
            // and 16 + r % 16 of word r / 16.  A byte permute fills each half with its frame's
            // sign; even registers take their bit by a select (ALU), odd ones add 2^r times the
            // permuted word (FMA pipe), 65535 times their bits in all, which a product undoes.
            uint32_t accs[NW], accm[NW];
#pragma unroll
            for (int i = 0; i < NW; ++i) accs[i] = accm[i] = 0u;
            auto decide = [&](int r, f32x2 x) {
                const uint32_t t = prmt((uint32_t)x, (uint32_t)(x >> 32), 0xFFBBu);
                if (r & 1) accm[r / 16] = imad(t, one << (r % 16), accm[r / 16]);
                else accs[r / 16] |= t & (0x00010001u << (r % 16));
            };
            if constexpr (PH < LR) {
#pragma unroll
                for (int ra = 0; ra < NR; ++ra) {
                    if (ra & (1 << PH)) continue;
                    const int rb = ra | (1 << PH);
                    const uint32_t a = C::alpha(C::rotr((uint32_t)ra, PH) >> 1);
                    const f32x2 ca0 = plus(P[ra], a), cb0 = minus(P[rb], a);
                    const f32x2 ca1 = minus(P[ra], a), cb1 = plus(P[rb], a);
                    P[ra] = max2(ca0, cb0);
                    P[rb] = max2(ca1, cb1);
                    decide(ra, sub2(cb0, ca0));
                    decide(rb, sub2(cb1, ca1));
                }
            } else {
                // the partner is in another lane: own + A[a] against other - A[a];
                // own is the even candidate on the lane of the even register
                constexpr int lb = PH >= LR ? PH - LR : 0;
                const f32x2 s = sgn[1 << lb], ns = mul2(s, pack2(-1.0f, -1.0f));   // +1: this lane holds the even register
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const uint32_t a = C::alpha(C::rotr((uint32_t)r, PH) >> 1);
                    float p0, p1;
                    unpack2(P[r], p0, p1);
                    const f32x2 oth = pack2(__shfl_xor_sync(gmask, p0, 1 << lb), __shfl_xor_sync(gmask, p1, 1 << lb));
                    const f32x2 co = plus(P[r], a), cp = minus(oth, a);
                    P[r] = max2(co, cp);
                    decide(r, fma2(s, cp, mul2(ns, co)));   // odd - even, one rounding
                }
            }
            uint32_t wd[NW];
#pragma unroll
            for (int i = 0; i < NW; ++i) wd[i] = ~imad(accm[i], minv, accs[i]);
            if (tau >= tau_store) {
                uint32_t *dst = surv + ((size_t)tau * 32 + wlane) * NW;
                // a lane with 32 registers has a word per frame
                if constexpr (NW == 1) *dst = wd[0];
                else *reinterpret_cast<uint2 *>(dst) = make_uint2(prmt(wd[0], wd[NW - 1], 0x5410u), prmt(wd[0], wd[NW - 1], 0x7632u));
            }
        });
        // normalisation: subtract state 0's metric (register 0 of lane 0) per frame
        float ref0, ref1;
        unpack2(P[0], ref0, ref1);
        if constexpr (L > 1) {
            ref0 = __shfl_sync(gmask, ref0, grp_base);
            ref1 = __shfl_sync(gmask, ref1, grp_base);
        }
        const f32x2 ref = pack2(ref0, ref1);
#pragma unroll
        for (int r = 0; r < NR; ++r) P[r] = sub2(P[r], ref);
    }

    // traceback start: after Wpad stages register R holds state R again
    uint32_t R[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float best = -INFINITY;
        uint32_t bR = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            float p0, p1;
            unpack2(P[r], p0, p1);
            const float x = h ? p1 : p0;
            if (x > best) { best = x; bR = ((uint32_t)lane << LR) | (uint32_t)r; }
        }
        if constexpr (L > 1) {
#pragma unroll
            for (int m = 1; m < L; m <<= 1) {
                const float ob = __shfl_xor_sync(gmask, best, m);
                const uint32_t oR = __shfl_xor_sync(gmask, bR, m);
                if (ob > best || (ob == best && oR < bR)) { best = ob; bR = oR; }
            }
        }
        R[h] = term[h] ? 0u : bR;
    }
    tb.set_out(0, ft[0].out);
    tb.set_out(1, ft[1].out);
    tb.set_surv(surv + (size_t)wlane * NW);
    tb.R[0] = R[0];
    tb.R[1] = R[1];
    tb.set_oacc(0, 0u);
    tb.set_oacc(1, 0u);
    tb.onb[0] = tb.onb[1] = 0;
    tb.t0 = Wpad - 1;
    tb.tau_store = tau_store;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        tb.tauo[h] = tauo[h];
        tb.taue[h] = taue[h];
        tb.toff[h] = (int32_t)(fa[h] - tau0[h]);
    }
    return true;
}

template <int K, int BETA, uint64_t GENS, int L, int NT>
__global__ void __launch_bounds__(NT, StreamCfgF32<K, BETA, GENS, L>::NR == 16 ? 4 : 3) stream_kernel_f32(const StreamParams p) {
    using Cfg = StreamCfgF32<K, BETA, GENS, L>;
    using Tb = Traceback<K, L, false, Cfg::NR, Cfg::NW>;
    __shared__ TbState tbs[NT];
    __shared__ __align__(16) uint32_t stg[NT / 32][Tb::STAGE_WORDS];
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t q = gtid / L;
    const int lane = (int)(gtid % L);
    if (q >= p.n_pairs) return;
    const int wlane = (int)(threadIdx.x & 31u);
    const unsigned gmask = (L == 32) ? 0xFFFFFFFFu : (((1u << L) - 1u) << (wlane & ~(L - 1)));
    const int grp_base = wlane & ~(L - 1);
    FrameTask ft[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t s = 2 * q + h;
        ft[h] = frame_task(p.llr, p.out, nullptr, s, p.n_win, p.n_info, p.T, p.f, p.v, p.flags);
    }
    uint32_t *surv = p.surv + (size_t)(gtid >> 5) * (size_t)p.wpad_max * 32u *
                                  (size_t)StreamCfgF32<K, BETA, GENS, L>::NW;
    TbState tb;
    forward_pair_f32<K, BETA, GENS, L>(ft, surv, p.wpad_max, wlane, lane, gmask, grp_base, p.status, tb);
    TbState &st = tbs[threadIdx.x];
    st = tb;
    uint32_t *my_stg = stg[threadIdx.x >> 5];
    if (Tb::active(st)) {
        Tb::begin(st, my_stg, wlane);
        Tb::drain(st, my_stg, wlane, lane, gmask, grp_base);
    }
}

}  // namespace vd
