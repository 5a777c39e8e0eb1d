// Wide kernel instantiations (vd_wide.cuh): K=7 with 8 lanes per frame pair, K=9 with 32.
#include <atomic>

#include "vd_launch.h"
#include "vd_wide.cuh"

namespace vd {

namespace {

template <int K> struct WideOf;
template <> struct WideOf<7> { static constexpr int BETA = 2, L = 8; static constexpr uint64_t GENS = GENS_K7; };
template <> struct WideOf<9> { static constexpr int BETA = 3, L = 32; static constexpr uint64_t GENS = GENS_K9; };

template <int K>
bool plan(const WideParams &in, WideParams *out, int64_t *blocks, size_t *smem, bool *full) {
    using Cfg = WideCfg<K, WideOf<K>::BETA, WideOf<K>::GENS, WideOf<K>::L>;
    WideParams p = in;
    const int64_t span = p.f + 2 * p.v, wmax = p.T < span ? p.T : span;
    if (wmax > (1 << 20)) return false;
    p.wpad = (int32_t)((wmax + Cfg::U - 1) / Cfg::U * Cfg::U);
    const int64_t kept = p.T < p.f + p.v ? p.T : p.f + p.v;   // stages from a frame's first decoded one to its end
    p.rec0 = (int32_t)((p.wpad - kept) / Cfg::U * (Cfg::U / Cfg::ES));
    const size_t pair = Cfg::pair_bytes(p.wpad, p.rec0);
    if (pair > kWideSmemMax) return false;
    constexpr int G = 32 / WideOf<K>::L;
    const int ppw = pair * G <= kWideSmemMax ? G : 1;   // frames too long for that: one pair per warp
    *blocks = (p.n_pairs + ppw - 1) / ppw;
    *smem = pair * (size_t)ppw;
    *full = ppw == G;
    *out = p;
    return true;
}

template <int K, int PPW>
cudaError_t launch(const WideParams &p, int64_t blocks, size_t smem, cudaStream_t st) {
    auto kern = wide_kernel<K, WideOf<K>::BETA, WideOf<K>::GENS, WideOf<K>::L, PPW>;
    // more than 48 KB of shared memory needs the kernel's opt-in, once per device
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? (1ull << dev) : 0ull;
    if (!bit || !(done.load(std::memory_order_acquire) & bit)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmemMax);
        if (e != cudaSuccess) return e;
        if (bit) done.fetch_or(bit, std::memory_order_acq_rel);
    }
    kern<<<(unsigned)blocks, 32, smem, st>>>(p);
    return cudaGetLastError();
}

}  // namespace

bool wide_plan(int K, const WideParams &in, WideParams *out, int64_t *blocks, size_t *smem, bool *full) {
    return K == 7 ? plan<7>(in, out, blocks, smem, full) : K == 9 ? plan<9>(in, out, blocks, smem, full) : false;
}

cudaError_t launch_wide(int K, const WideParams &p, int64_t blocks, size_t smem, bool full, cudaStream_t st) {
    if (K == 9) return launch<9, 1>(p, blocks, smem, st);
    if (K != 7) return cudaErrorInvalidValue;
    return full ? launch<7, 4>(p, blocks, smem, st) : launch<7, 1>(p, blocks, smem, st);
}

}  // namespace vd
