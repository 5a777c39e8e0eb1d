// Wide kernel instantiations (vd_wide.cuh): K=7 with 8 lanes per frame pair, K=9 with 32.
#include <atomic>

#include "vd_variants.cuh"
#include "vd_wide.cuh"

namespace vd {

namespace {

template <int K> constexpr int kLanes = K == 7 ? 8 : 32;
template <int K> using CfgOf = WideCfg<K, CodeOf<K>::BETA, CodeOf<K>::GENS, kLanes<K>>;

template <int K>
bool plan(const WideParams &in, WideParams *out, int64_t *blocks, size_t *smem, bool *full) {
    using Cfg = CfgOf<K>;
    WideParams p = in;
    const int64_t span = p.f + 2 * p.v, wmax = p.T < span ? p.T : span;
    if (wmax > (1 << 20)) return false;
    p.wpad = (int32_t)((wmax + Cfg::U - 1) / Cfg::U * Cfg::U);
    const int64_t kept = p.T < p.f + p.v ? p.T : p.f + p.v;   // stages from a frame's first decoded one to its end
    p.rec0 = (int32_t)((p.wpad - kept) / Cfg::U * (Cfg::U / Cfg::ES));
    const size_t pair = Cfg::pair_bytes(p.wpad, p.rec0);
    if (pair > kWideSmemMax) return false;
    constexpr int G = 32 / kLanes<K>;
    const int ppw = pair * G <= kWideSmemMax ? G : 1;   // frames too long for that: one pair per warp
    *blocks = (p.n_pairs + ppw - 1) / ppw;
    *smem = pair * (size_t)ppw;
    *full = ppw == G;
    *out = p;
    return true;
}

template <int K, int PPW>
cudaError_t launch(const WideParams &p, int64_t blocks, size_t smem, cudaStream_t st) {
    auto kern = wide_kernel<K, CodeOf<K>::BETA, CodeOf<K>::GENS, kLanes<K>, PPW>;
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = opt_in_smem(kern, kWideSmemMax, done);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)blocks, 32, smem, st>>>(p);
    return cudaGetLastError();
}

constexpr int kSplitWarps = 4;

template <int K>
bool split(const WideParams &in, int n_sm, SplitParams *out, int *ranks, size_t *smem) {
    using Cfg = CfgOf<K>;
    const int64_t span = in.f + 2 * in.v, wmax = in.T < span ? in.T : span;
    if (wmax > (1 << 20)) return false;
    const int nc = (int)((wmax + Cfg::U - 1) / Cfg::U);
    // Blocks per SM up to which segments pay for their warm-up (times of both
    // forms grow with the frame; us, split / wide): K=7, f = 256 (340 stages): 235
    // frames 16.7 / 20.8, 391 22.7 / 20.8; f = 512 (596): 391 20.7 / 35; K=9, f = 512
    // (640): 196 31 / 43, 391 33 / 43.
    const int64_t per_sm = wmax < 170 ? 1 : wmax / 170 < 3 ? wmax / 170 : 3;
    bool have = false;
    for (int r = 1; r <= 8; r *= 2) {
        if (in.n_win * r > per_sm * n_sm) break;
        const int nseg = r * kSplitWarps * 2 * (32 / kLanes<K>);
        const int S = (nc + nseg - 1) / nseg;
        const size_t bytes = (size_t)SplitSmem<K, CodeOf<K>::BETA, CodeOf<K>::GENS, kLanes<K>>(kSplitWarps, S, kSplitWarmup).total * 4u;
        if (bytes > kWideSmemMax) continue;
        have = true;
        out->S = S;
        *ranks = r;
        *smem = bytes;
        if (2 * S <= kSplitWarmup) break;   // a wider cluster would mostly run warm-ups
    }
    if (!have) return false;
    if (nc < out->S + kSplitWarmup + kSplitGain) return false;   // no chain shorter than the frame's
    out->llr = in.llr;
    out->n_info = in.n_info;
    out->T = in.T;
    out->f = in.f;
    out->v = in.v;
    out->n_win = in.n_win;
    out->flags = in.flags;
    out->M = kSplitWarmup;
    out->out = in.out;
    out->pm_out = in.pm_out;
    return true;
}

template <int K>
cudaError_t launch_s(const SplitParams &p, int ranks, size_t smem, cudaStream_t st) {
    auto kern = split_kernel<K, CodeOf<K>::BETA, CodeOf<K>::GENS, kLanes<K>, 32 * kSplitWarps>;
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = opt_in_smem(kern, kWideSmemMax, done);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.n_win * ranks));
    cfg.blockDim = dim3(32 * kSplitWarps);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ranks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace

int wide_lanes(int K) { return K == 7 ? kLanes<7> : kLanes<9>; }

bool split_plan(int K, const WideParams &in, int n_sm, SplitParams *out, int *ranks, size_t *smem) {
    return K == 7 ? split<7>(in, n_sm, out, ranks, smem) : K == 9 ? split<9>(in, n_sm, out, ranks, smem) : false;
}

cudaError_t launch_split(int K, const SplitParams &p, int ranks, size_t smem, cudaStream_t st) {
    return K == 7 ? launch_s<7>(p, ranks, smem, st) : K == 9 ? launch_s<9>(p, ranks, smem, st) : cudaErrorInvalidValue;
}

bool wide_plan(int K, const WideParams &in, WideParams *out, int64_t *blocks, size_t *smem, bool *full) {
    return K == 7 ? plan<7>(in, out, blocks, smem, full) : K == 9 ? plan<9>(in, out, blocks, smem, full) : false;
}

cudaError_t launch_wide(int K, const WideParams &p, int64_t blocks, size_t smem, bool full, cudaStream_t st) {
    if (K == 9) return launch<9, 1>(p, blocks, smem, st);
    if (K != 7) return cudaErrorInvalidValue;
    return full ? launch<7, 4>(p, blocks, smem, st) : launch<7, 1>(p, blocks, smem, st);
}

}  // namespace vd
