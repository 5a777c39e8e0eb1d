// vd_transmit: the transmitter and channel of the paper's verification
// system (Sec. IX-B) on the GPU, so that a decoder (or the serving loop) can
// be fed without host-generated LLRs: information bits -> convolutional
// encoder (Sec. II-A) -> puncturing -> BPSK -> AWGN -> quantiser.
//
// One thread makes eight consecutive kept values (two Philox blocks).  For
// kept value k the stage t and output b come from the puncturing pattern
// (k-th kept position in stage-major, b-ascending order); the encoder output
// is the parity of g_b and the register of inputs t-K+1 .. t, read straight
// from the packed information bits (zero before the start and in the tail).
// The noise is the k-th standard normal of the stream: Philox4x64-10 (Salmon
// et al., SC 2011) with key (seed, stream_id) on counter block k / 4, turned
// into four normals by the Box-Muller transform in double precision.
//
// What bounds it: instruction issue (74% of the cycles; 174 instructions a value,
// the 64-bit integer products of Philox first).  In double precision
// alone the transform bound it (the fp64 units give two lanes per clock and SM): 732 us for
// 8.4 M int8 values, on GB300.  The transform is therefore taken in single precision with an
// error bound, which settles the quantised value unless a rounding border
// lies within the bound; a pair with such a value (1 in 10^4 for int8, 1 in 300 for half
// precision) comes from the double-precision transform instead.  The bytes are those of
// the double-precision transform.  Measured, 8.4 M int8 values (2^22 bits, K=7): 732 us; with logf,
// log1pf and sincospif and eight values at a time in double precision 77; with the
// polynomials below and two at a time 56.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "../../include/vd.h"
#include "vd_code.h"

namespace {

struct TxParams {
    const uint32_t *bits;   // packed information bits, LSB-first
    int64_t n_info, n_kept, n_words;
    int K, beta, period, kept_per_period;
    uint32_t gens[4];
    uint8_t pos_phase[32], pos_b[32];   // r-th kept position of a period: (phase, output)
    double sigma, inv_var2;             // sigma and 2 / sigma^2
    float sigma_f, inv_var2_f;
    uint64_t kpp_magic;                 // 2^64 / kept_per_period, rounded up: k / kept_per_period = high word of k kpp_magic
    int aligned;                        // out on a 16-byte boundary
    uint64_t seed, stream_id;
    void *out;
};

// hi:lo of a * m: four 32 x 32 -> 64-bit multiply-adds (no partial sum overflows).
__device__ __forceinline__ void mul_wide64(uint64_t a, uint64_t m, uint64_t &hi, uint64_t &lo) {
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), m0 = (uint32_t)m, m1 = (uint32_t)(m >> 32);
    const uint64_t p00 = (uint64_t)a0 * m0;
    const uint64_t p01 = (uint64_t)a0 * m1 + (p00 >> 32);
    const uint64_t p10 = (uint64_t)a1 * m0 + (uint32_t)p01;
    hi = (uint64_t)a1 * m1 + (p01 >> 32) + (p10 >> 32);
    lo = (p10 << 32) | (uint32_t)p00;
}

__device__ __forceinline__ void philox4x64(uint64_t (&c)[4], uint64_t k0, uint64_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint64_t lo0, hi0, lo1, hi1;
        mul_wide64(c[0], 0xD2E7470EE14C6C93ull, hi0, lo0);
        mul_wide64(c[2], 0xCA5A826395121157ull, hi1, lo1);
        const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
        k0 += 0x9E3779B97F4A7C15ull;
        k1 += 0xBB67AE8584CAA73Bull;
    }
}

__device__ __forceinline__ double unit53(uint64_t x) { return (double)((x >> 11) + 1ull) * 0x1.0p-53; }

// Bits [lo, lo + 32) of the information stream (zero outside [0, n_info)).
__device__ __forceinline__ uint32_t info_window(const TxParams &p, int64_t lo) {
    uint32_t v = 0;
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        const int64_t base = (lo >> 5) + w;          // word holding bits base*32 ..
        uint32_t x = (base >= 0 && base < p.n_words) ? p.bits[base] : 0u;
        const int64_t first = base * 32;
        if (first + 32 > p.n_info) {                 // clear bits at or past n_info
            const int64_t keep = p.n_info - first;
            x = keep <= 0 ? 0u : (x & (0xFFFFFFFFu >> (32 - (int)keep)));
        }
        const int64_t sh = first - lo;               // position of bit `first` in the window
        if (sh >= 0 && sh < 32) v |= x << sh;
        else if (sh < 0 && sh > -32) v |= x >> (-sh);
    }
    return v;
}

// The quantised value of a sample as the bits it has in the output.
template <int TYPE>
__device__ __forceinline__ uint32_t quantise(double y, double inv_var2) {
    if constexpr (TYPE == VD_LLR_S8) return (uint32_t)(int)fmin(fmax(rint(32.0 * y), -127.0), 127.0) & 0xFFu;
    else if constexpr (TYPE == VD_LLR_S4) return (uint32_t)(int)fmin(fmax(rint(2.0 * y), -7.0), 7.0) & 0xFu;
    else if constexpr (TYPE == VD_LLR_F16) return (uint32_t)__half_as_ushort(__double2half(y * inv_var2));
    else return y < 0.0 ? 1u : 0u;
}

// Double precision for a pair of values that single precision leaves open (two 16-bit fields).
template <int TYPE>
__device__ __noinline__ uint32_t exact_pair(uint64_t wu, uint64_t wv, uint32_t cbits, double sigma, double inv_var2) {
    const double u = unit53(wu), v = unit53(wv);
    const double rad = sqrt(-2.0 * log(u)), ang = 2.0 * 3.14159265358979323846 * v;
    const double y0 = ((cbits & 1u) ? -1.0 : 1.0) + sigma * (rad * cos(ang));
    const double y1 = ((cbits & 2u) ? -1.0 : 1.0) + sigma * (rad * sin(ang));
    return quantise<TYPE>(y0, inv_var2) | quantise<TYPE>(y1, inv_var2) << 16;
}

// ln(U 2^-53) for U in 1 .. 2^53.  U 2^-53 = (1 + f) 2^e with 1 + f in [2/3, 4/3), f
// from an exact integer difference; ln(1 + f) = f q(f), q the polynomial of degree 10
// that interpolates ln(1 + f) / f at the Chebyshev nodes of [-1/3, 1/3].  Within 1.7e-7 of
// itself (checked against 64 bits over all binades and both ends).
__device__ __forceinline__ float ln_u53(uint64_t U) {
    const int lz = __clzll((long long)U);
    const uint64_t M = U << (lz - 10);                       // in [2^53, 2^54)
    const bool up = M >= (1ull << 55) / 3ull;                // 1 + f = M 2^-54, else M 2^-53
    const float f = __ll2float_rn((long long)(M - (up ? 1ull << 54 : 1ull << 53))) * (up ? 0x1.0p-54f : 0x1.0p-53f);
    float q = 0.11900901794433594f;
    q = fmaf(q, f, -0.13038060069084167f);
    q = fmaf(q, f, 0.10781308263540268f);
    q = fmaf(q, f, -0.12143635004758835f);
    q = fmaf(q, f, 0.14302155375480652f);
    q = fmaf(q, f, -0.16684426367282867f);
    q = fmaf(q, f, 0.1999966949224472f);
    q = fmaf(q, f, -0.24999643862247467f);
    q = fmaf(q, f, 0.3333333432674408f);
    q = fmaf(q, f, -0.5f);
    q = fmaf(q, f, 1.0f);
    return fmaf((float)(10 - lz + (up ? 1 : 0)), 0.693147180559945f, f * q);
}

// A Box-Muller pair in single precision; u = U 2^-53 and v = V 2^-53 enter as
// integers, so that the angle's offset from the nearest quarter turn is exact before it is rounded
// to 24 bits.  Errors: rad 2.1e-7 of itself (half of the logarithm's 1.7e-7, 2^-23 of the
// square root), the cosine and sine (Taylor polynomials on an eighth of a
// turn) 8.7e-8 and 4.7e-8 for the angle: rad times either is off by less than 3.5e-7 rad.
__device__ __forceinline__ void pair_f32(uint64_t wu, uint64_t wv, float &rad, float &c, float &s) {
    const float x = -2.0f * ln_u53((wu >> 11) + 1ull);
    asm("sqrt.approx.f32 %0, %1;" : "=f"(rad) : "f"(x));
    const uint64_t V = (wv >> 11) + 1ull;
    const uint64_t quad = (V + (1ull << 50)) >> 51;
    const float r = __ll2float_rn((long long)(V - (quad << 51))) * 0x1.0p-52f;   // half turns, at most 1/4
    const float t = r * r;
    float sn = 0.0821458866f;                      // pi^9 / 9!
    sn = fmaf(sn, t, -0.599264529f);
    sn = fmaf(sn, t, 2.55016404f);
    sn = fmaf(sn, t, -5.16771278f);
    sn = fmaf(sn, t, 3.14159265f);
    sn *= r;
    float cs = -0.0258068913f;                     // -pi^10 / 10!
    cs = fmaf(cs, t, 0.235330630f);
    cs = fmaf(cs, t, -1.33526277f);
    cs = fmaf(cs, t, 4.05871213f);
    cs = fmaf(cs, t, -4.93480220f);
    cs = fmaf(cs, t, 1.0f);
    const bool odd = quad & 1ull;
    const float p = odd ? sn : cs, q = odd ? cs : sn;
    c = (quad + 1ull) & 2ull ? -p : p;   // quarter turns 1, 2: negative cosine
    s = quad & 2ull ? -q : q;            // quarter turns 2, 3: negative sine
}

template <int TYPE>
__global__ void __launch_bounds__(256) transmit_kernel(const __grid_constant__ TxParams p) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t k0 = 8 * j;
    if (k0 >= p.n_kept) return;
    // encoder outputs of the thread's kept values: at most eight stages, one window of input bits
    int64_t g = p.kept_per_period == 1 ? k0 : (int64_t)__umul64hi((uint64_t)k0, p.kpp_magic);
    int r = (int)(k0 - g * p.kept_per_period);
    const int64_t t0 = g * p.period + p.pos_phase[r];
    const uint32_t win = info_window(p, t0 - (p.K - 1));
    // output b of all stages of the window at once: bit dt of o[b] is stage t0 + dt
    uint32_t o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        if (b < p.beta) {
#pragma unroll
            for (int i = 0; i < 9; ++i) o[b] ^= (p.gens[b] >> i & 1u) ? win >> i : 0u;
        }
    }
    uint32_t cbits = 0;
    int dt = 0 - p.pos_phase[r];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int b = p.pos_b[r];
        const uint32_t x = b == 0 ? o[0] : b == 1 ? o[1] : b == 2 ? o[2] : o[3];
        cbits |= ((x >> (dt + p.pos_phase[r])) & 1u) << i;
        if (++r == p.kept_per_period) {
            r = 0;
            dt += p.period;
        }
    }
    uint64_t w[2][4] = {{(uint64_t)(2 * j), 0ull, 0ull, 0ull}, {(uint64_t)(2 * j + 1), 0ull, 0ull, 0ull}};
    philox4x64(w[0], p.seed, p.stream_id);
    philox4x64(w[1], p.seed, p.stream_id);
    uint32_t q[8];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint64_t wu = w[m >> 1][2 * (m & 1)], wv = w[m >> 1][2 * (m & 1) + 1];
        float rad, cs[2];
        pair_f32(wu, wv, rad, cs[0], cs[1]);
        // y = +-1 + sigma z: the pair's 3.5e-7 sigma rad, the roundings of sigma, of
        // sigma rad and of the sum (6e-8 each of theirs), with half as much again to spare
        const float srad = p.sigma_f * rad, ey = 8e-7f * srad + 1.5e-7f;
        bool open = false;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int i = 2 * m + k;
            const float y = fmaf(srad, cs[k], ((cbits >> i) & 1u) ? -1.0f : 1.0f);
            if constexpr (TYPE == VD_LLR_S8 || TYPE == VD_LLR_S4) {
                // scaled by a power of two and clipped; adding 1.5 2^23 rounds to the nearest
                // integer, ties to even, and leaves it in the low bits.  Open: within the bound of
                // a half-integer, unless well past the clip.
                constexpr float SCALE = TYPE == VD_LLR_S8 ? 32.0f : 2.0f, TOP = TYPE == VD_LLR_S8 ? 127.0f : 7.0f;
                const float t = SCALE * y, et = SCALE * ey;
                const float tc = fminf(fmaxf(t, -TOP), TOP);
                const float big = tc + 12582912.0f;
                q[i] = __float_as_uint(big) & (TYPE == VD_LLR_S8 ? 0xFFu : 0xFu);
                open |= fabsf(tc - (big - 12582912.0f)) > 0.5f - et && fabsf(t) < TOP + 1.0f + et;
            } else if constexpr (TYPE == VD_LLR_F16) {
                const float x = y * p.inv_var2_f, ex = ey * p.inv_var2_f + 3e-7f * fabsf(x);
                q[i] = __half_as_ushort(__float2half_rn(x - ex));
                open |= q[i] != (uint32_t)__half_as_ushort(__float2half_rn(x + ex));
            } else {
                q[i] = y < 0.0f ? 1u : 0u;
                open |= fabsf(y) <= ey;
            }
        }
        if (open) {
            const uint32_t e = exact_pair<TYPE>(wu, wv, cbits >> (2 * m), p.sigma, p.inv_var2);
            q[2 * m] = e & 0xFFFFu;
            q[2 * m + 1] = e >> 16;
        }
    }
    const int n = p.n_kept - k0 < 8 ? (int)(p.n_kept - k0) : 8;   // values of this thread
    if constexpr (TYPE == VD_LLR_S8) {
        int8_t *o = static_cast<int8_t *>(p.out) + k0;
        if (n == 8 && p.aligned) {
            *reinterpret_cast<uint2 *>(o) = make_uint2(q[0] | q[1] << 8 | q[2] << 16 | q[3] << 24,
                                                       q[4] | q[5] << 8 | q[6] << 16 | q[7] << 24);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < n) o[i] = (int8_t)q[i];
        }
    } else if constexpr (TYPE == VD_LLR_F16) {
        uint16_t *o = static_cast<uint16_t *>(p.out) + k0;
        if (n == 8 && p.aligned) {
            *reinterpret_cast<uint4 *>(o) =
                make_uint4(q[0] | q[1] << 16, q[2] | q[3] << 16, q[4] | q[5] << 16, q[6] | q[7] << 16);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < n) o[i] = (uint16_t)q[i];
        }
    } else {
        // values past the last one are zero bits (4-bit: two per byte, hard: eight)
        constexpr int BITS = TYPE == VD_LLR_S4 ? 4 : 1;
        uint32_t packed = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < n) packed |= q[i] << (BITS * i);
        uint8_t *o = static_cast<uint8_t *>(p.out) + BITS * j;
        if (BITS == 4 && n == 8 && p.aligned) {
            *reinterpret_cast<uint32_t *>(o) = packed;
        } else {
#pragma unroll
            for (int i = 0; i < BITS; ++i)
                if (BITS * n > 8 * i) o[i] = (uint8_t)(packed >> (8 * i));
        }
    }
}

vd_status fail(vd_status st, const char *msg) {
    vd_internal_set_error(msg);
    return st;
}

}  // namespace

extern "C" int64_t vd_transmit_bytes(const vd_code *c, int64_t n_info, uint32_t flags, int llr_type) {
    if (!c || n_info < 0) return -1;
    const int64_t T = n_info + ((flags & VD_TERMINATED) ? c->K - 1 : 0);
    const int64_t kept = vd_num_kept(c, T);
    switch (llr_type) {
    case VD_LLR_S8: return kept;
    case VD_LLR_S4: return (kept + 1) / 2;
    case VD_LLR_F16: return 2 * kept;
    case VD_LLR_HARD: return (kept + 7) / 8;
    default: return -1;
    }
}

extern "C" vd_status vd_transmit(const vd_code *c, const uint32_t *d_bits, int64_t n_info, uint32_t flags,
                                 double sigma, uint64_t seed, uint64_t stream_id, int llr_type, void *d_out,
                                 void *stream) {
    if (!c) return fail(VD_EINVAL, "vd_transmit: code is NULL");
    if (n_info < 0 || n_info > ((int64_t)1 << 40)) return fail(VD_EINVAL, "vd_transmit: bad n_info");
    if (flags & ~(uint32_t)VD_TERMINATED) return fail(VD_EINVAL, "vd_transmit: flags other than VD_TERMINATED");
    if (!(sigma >= 0.0) || sigma > 1e6) return fail(VD_EINVAL, "vd_transmit: sigma must be in [0, 1e6]");
    if (llr_type == VD_LLR_F16 && sigma == 0.0)
        return fail(VD_EINVAL, "vd_transmit: fp16 LLRs (2 y / sigma^2) need sigma > 0");
    if (llr_type != VD_LLR_S8 && llr_type != VD_LLR_S4 && llr_type != VD_LLR_F16 && llr_type != VD_LLR_HARD)
        return fail(VD_EINVAL, "vd_transmit: unknown llr_type");
    const int64_t T = n_info + ((flags & VD_TERMINATED) ? c->K - 1 : 0);
    TxParams p;
    memset(&p, 0, sizeof p);
    p.n_kept = vd_num_kept(c, T);
    if (p.n_kept == 0) return VD_OK;
    if (!d_out || (n_info > 0 && !d_bits)) return fail(VD_EINVAL, "vd_transmit: NULL device pointer");
    p.bits = d_bits;
    p.n_info = n_info;
    p.n_words = (n_info + 31) / 32;
    p.K = c->K;
    p.beta = c->beta;
    p.period = c->period;
    p.kept_per_period = c->kept_per_period;
    for (int b = 0; b < c->beta; ++b) p.gens[b] = c->gens[b];
    int r = 0;
    for (int ph = 0; ph < c->period; ++ph)
        for (int b = 0; b < c->beta; ++b)
            if (c->punct[b][ph]) {
                p.pos_phase[r] = (uint8_t)ph;
                p.pos_b[r] = (uint8_t)b;
                ++r;
            }
    p.sigma = sigma;
    p.inv_var2 = sigma > 0.0 ? 2.0 / (sigma * sigma) : 0.0;
    p.sigma_f = (float)p.sigma;
    p.inv_var2_f = (float)p.inv_var2;
    // k < 2^43, so the rounded-up reciprocal's excess (at most 32 of 2^64) never reaches the quotient
    if (p.kept_per_period > 1) p.kpp_magic = ~0ull / (uint64_t)p.kept_per_period + 1ull;
    p.aligned = ((uintptr_t)d_out & 15u) == 0;
    p.seed = seed;
    p.stream_id = stream_id;
    p.out = d_out;
    const int64_t threads = (p.n_kept + 7) / 8;
    const int tb = 256;
    const int64_t blocks = (threads + tb - 1) / tb;
    if (blocks > 0x7FFFFFFF) return fail(VD_EINVAL, "vd_transmit: stream too long");
    const cudaStream_t cs = (cudaStream_t)stream;
    switch (llr_type) {
    case VD_LLR_S8: transmit_kernel<VD_LLR_S8><<<(unsigned)blocks, tb, 0, cs>>>(p); break;
    case VD_LLR_S4: transmit_kernel<VD_LLR_S4><<<(unsigned)blocks, tb, 0, cs>>>(p); break;
    case VD_LLR_F16: transmit_kernel<VD_LLR_F16><<<(unsigned)blocks, tb, 0, cs>>>(p); break;
    default: transmit_kernel<VD_LLR_HARD><<<(unsigned)blocks, tb, 0, cs>>>(p); break;
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(VD_ECUDA, cudaGetErrorString(e));
    return VD_OK;
}
