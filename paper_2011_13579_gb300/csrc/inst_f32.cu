// fp16-LLR / fp32-metric stream kernel instantiations: a frame pair over 4
// lanes (K=7), 16 or 8 (K=9).  The caller's names of these forms
// (vd_tune.lanes) are 2 and 8.
#include "vd_variants.cuh"
#include "vd_stream_f32.cuh"

namespace vd {

namespace {

template <int K, int L>
cudaError_t launch(const StreamParams &p, int64_t blocks, cudaStream_t st) {
    stream_kernel_f32<K, CodeOf<K>::BETA, CodeOf<K>::GENS, L, kThreads><<<(unsigned)blocks, kThreads, 0, st>>>(p);
    return cudaGetLastError();
}

template <int K, int L>
F32Geom geom() {
    using Cfg = StreamCfgF32<K, CodeOf<K>::BETA, CodeOf<K>::GENS, L>;
    F32Geom g;
    g.geom.U = Cfg::U;
    g.geom.NW = Cfg::NW;
    g.threads_per_pair = L;
    return g;
}

}  // namespace

// K=9: 16 lanes per pair while all pairs are resident at once (four blocks
// of 128 threads an SM), 8 beyond.  Sixteen lanes halve the chain of a stage, eight take 45
// instructions per frame and stage instead of 62.  Measured (us, 16 / 8 lanes): 2^20 bits
// 283 / 429, 2^22 (1.7 times the residents) 537 / 490, 2^24 1772 / 1657.  K=7 (4 / 2 lanes):
// 132 / 201, 166 / 214, 436 / 502.
F32Geom geom_f32(int K, int64_t n_pairs, int n_sm) {
    if (K == 7) return geom<7, 4>();
    return n_pairs * 16 <= (int64_t)n_sm * 4 * kThreads ? geom<9, 16>() : geom<9, 8>();
}

cudaError_t launch_stream_f32(int K, int threads_per_pair, const StreamParams &p, int64_t blocks, cudaStream_t st) {
    if (K == 7 && threads_per_pair == 4) return launch<7, 4>(p, blocks, st);
    if (K == 9 && threads_per_pair == 8) return launch<9, 8>(p, blocks, st);
    if (K == 9 && threads_per_pair == 16) return launch<9, 16>(p, blocks, st);
    return cudaErrorInvalidValue;
}

}  // namespace vd
