// Input pre-pass helper: expands transmitted (kept) LLR values to beta int8
// LLRs per stage, inserting 0 at the positions a puncturing pattern erases,
// sign-extending 4-bit values and mapping hard decisions to +-1.  The kept
// values are stage-major with b ascending.
//
// What bounds it: memory, once a thread's work is small.  The pattern of erased
// positions repeats over a cycle of output words (the least common multiple of a
// puncturing period's bytes and 4), so each output word is four kept values in
// a row, read as one unaligned field, and a byte permute that puts them, or zero,
// in their places: a table gives both per word of the cycle.  A warp writes 128
// contiguous bytes at a time.  Measured (GB300, us, against a thread per puncturing period with byte
// loads): 43,690 punctured packets (175 MB in, 216 MB out) 245 -> 107; 3 M stages of 4-bit values 18.4 -> 7.1.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/vd.h"

namespace vd {

constexpr int kPrepWords = 24;   // words of a cycle: at most 21 (period 7 of 3 outputs, 5 or 7 of 4 bytes a period less)

// The cycle of one code: `words` output words hold `kept` kept values; word w
// begins with the cycle's kept value first[w] (or a later one) and is the byte
// permute sel[w] of that value and the three after it (nibble 4: zero).
struct PrepTable {
    int32_t words, kept;
    uint8_t first[kPrepWords];
    uint16_t sel[kPrepWords];
};

inline PrepTable prep_table(int beta, int period, const uint8_t (&punct)[4][8]) {
    PrepTable t = {};
    const int bytes = beta * period;
    int cycle = bytes;
    while (cycle % 4) cycle += bytes;
    t.words = cycle / 4;
    int k = 0;
    for (int w = 0; w < t.words; ++w) {
        t.first[w] = (uint8_t)k;
        for (int i = 0; i < 4; ++i) {
            const int j = (4 * w + i) % bytes;
            const bool on = punct[j % beta][j / beta] != 0;
            t.sel[w] |= (uint16_t)((on ? k - t.first[w] : 4) << (4 * i));
            if (on) ++k;
        }
    }
    t.kept = k;
    return t;
}

// Expands output words [0, n) of a piece that begins a cycle: out_bytes bytes at dst (4-byte aligned)
// from the kept values k0 .. kept_end of src.  Threads tid, tid + nthr, .. of the
// caller share the work.  A piece is short enough for 32-bit offsets, which is most of
// what a word costs: an earlier form with 64-bit ones took 85 instructions a word.
// Only aligned 32-bit words that hold part of a kept value before kept_end are read.
template <int BITS>
__device__ __forceinline__ void prep_piece(const uint8_t *src, int64_t k0, int64_t kept_end, uint32_t out_bytes,
                                           const PrepTable &t, int8_t *dst, uint32_t tid, uint32_t nthr) {
    const uint64_t bit0 = (uint64_t)k0 * BITS;
    const uint8_t *a = src + (bit0 >> 3);
    const uint32_t mis = (uint32_t)(reinterpret_cast<uintptr_t>(a) & 3u);
    const uint32_t *in = reinterpret_cast<const uint32_t *>(a - mis);
    const uint32_t b0 = 8u * mis + (uint32_t)(bit0 & 7u);                  // first kept value, in bits from `in`
    const uint64_t left = (uint64_t)(kept_end - k0) * BITS + b0;
    const uint32_t n_in = left > 0x7FFFFFE0ull ? 0x3FFFFFFu : (uint32_t)((left + 31u) >> 5);   // words that may be read
    const uint32_t n_full = out_bytes / 4, n_words = (out_bytes + 3) / 4;
    const uint32_t words = (uint32_t)t.words, kept = (uint32_t)t.kept;
    const uint32_t c0 = tid / words, dc = nthr / words, dw = nthr - dc * words, dk = dc * kept;
    uint32_t w = tid - c0 * words, k = c0 * kept;
    uint32_t *out = reinterpret_cast<uint32_t *>(dst);
    constexpr int N = 4;             // words in flight
    for (uint32_t i0 = tid; i0 < n_words; i0 += N * nthr) {
        uint32_t lo[N], hi[N], sh[N], sel[N];
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const uint32_t bit = b0 + (k + t.first[w]) * BITS;
            const uint32_t j = bit >> 5;
            sh[n] = bit & 31u;
            sel[n] = t.sel[w];
            // a word past the last one reads nothing that is used
            lo[n] = j < n_in ? __ldg(in + j) : 0u;
            hi[n] = j + 1u < n_in && sh[n] + 4u * BITS > 32u ? __ldg(in + j + 1) : 0u;
            k += dk;
            w += dw;
            if (w >= words) {
                w -= words;
                k += kept;
            }
        }
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const uint32_t i = i0 + n * nthr;
            uint32_t x = __funnelshift_r(lo[n], hi[n], sh[n]);
            if constexpr (BITS == 4) {
                x &= 0xFFFFu;
                x = (x | (x << 8)) & 0x00FF00FFu;
                x = (x | (x << 4)) & 0x0F0F0F0Fu;
                x |= (x & 0x08080808u) * 0x1Eu;                             // sign: 0x08 -> 0xF8
            } else if constexpr (BITS == 1) {
                // bit 0 -> 1, bit 1 -> -1
                x = 0x01010101u + (((x & 0xFu) * 0x00204081u) & 0x01010101u) * 0xFEu;
            }
            uint32_t y;
            asm("prmt.b32 %0, %1, %2, %3;" : "=r"(y) : "r"(x), "r"(0u), "r"(sel[n]));
            if (i < n_full) {
                out[i] = y;
            } else if (i < n_words) {
                for (uint32_t b = 0; 4 * i + b < out_bytes; ++b) dst[4 * i + b] = (int8_t)(y >> (8 * b));
            }
        }
    }
}

__device__ __forceinline__ void prep_piece(const uint8_t *src, int64_t k0, int64_t kept_end, int llr_type,
                                           uint32_t out_bytes, const PrepTable &t, int8_t *dst, uint32_t tid,
                                           uint32_t nthr) {
    if (llr_type == VD_LLR_HARD) prep_piece<1>(src, k0, kept_end, out_bytes, t, dst, tid, nthr);
    else if (llr_type == VD_LLR_S4) prep_piece<4>(src, k0, kept_end, out_bytes, t, dst, tid, nthr);
    else prep_piece<8>(src, k0, kept_end, out_bytes, t, dst, tid, nthr);
}

// Output words of a piece of about `target` words: whole cycles.
__host__ __device__ inline int64_t prep_piece_words(const PrepTable &t, int64_t target) {
    return (target + t.words - 1) / t.words * t.words;
}

}  // namespace vd
