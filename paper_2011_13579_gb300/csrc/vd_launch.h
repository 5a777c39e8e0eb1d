// Launchers for the kernel instantiations compiled in separate translation units.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "vd_batch.cuh"
#include "vd_wide.cuh"

namespace vd {

// Codes with compiled kernels.  Generators are packed 16 bits each.
constexpr uint64_t pack_gens(uint32_t g0, uint32_t g1, uint32_t g2 = 0, uint32_t g3 = 0) {
    return (uint64_t)g0 | ((uint64_t)g1 << 16) | ((uint64_t)g2 << 32) | ((uint64_t)g3 << 48);
}
constexpr uint64_t GENS_K7 = pack_gens(0171, 0133);
constexpr uint64_t GENS_K9 = pack_gens(0557, 0663, 0711);

enum CodeKind { KIND_NONE = 0, KIND_K7_R2 = 1, KIND_K9_R3 = 2 };

constexpr int kThreads = 128;

// Geometry of one instantiation, for scratch sizing on the host.
struct KernelGeom {
    int U;       // stages per chunk
    int NW;      // survivor scratch words per thread per stage (StreamCfg::SW)
};

// Returns cudaErrorInvalidValue if (kind, lanes, radix4) has no instantiation.
// deep: the traceback ring for launches of which every block is resident at once (StreamSmem).
cudaError_t launch_stream_k7(int lanes, bool radix4, const StreamParams &p, int64_t blocks, bool deep,
                             cudaStream_t st);
cudaError_t launch_stream_k9(int lanes, bool radix4, const StreamParams &p, int64_t blocks, bool deep,
                             cudaStream_t st);
cudaError_t launch_batch_k7(int lanes, bool radix4, const BatchParams &p, int64_t blocks,
                            cudaStream_t st);
cudaError_t launch_batch_k9(int lanes, bool radix4, const BatchParams &p, int64_t blocks,
                            cudaStream_t st);
cudaError_t batch_occupancy_k7(int lanes, bool radix4, int *blocks_per_sm);
cudaError_t batch_occupancy_k9(int lanes, bool radix4, int *blocks_per_sm);
// Persistent stream decode (K = 7 or 9): p.counter must be zero at launch.
cudaError_t launch_stream_persistent(int K, int lanes, bool radix4, const StreamParams &p, int64_t blocks,
                                     cudaStream_t st);
cudaError_t stream_persistent_occupancy(int K, int lanes, bool radix4, int *blocks_per_sm);
// The same for the kernel with one lane group per frame pair (launch_stream_k7 / _k9).
cudaError_t stream_wave_occupancy(int K, int lanes, bool radix4, bool deep, int *blocks_per_sm);

// Wide form (vd_wide.cuh), for streams of few frames: wide_plan fills the
// padded length, the records kept and the pairs per warp, and says how many
// blocks of one warp and how much shared memory each takes; false if a
// frame pair's survivors do not fit.
constexpr size_t kWideSmemMax = 226u * 1024u;
int wide_lanes(int K);   // lanes per pair of the wide and the split form
bool wide_plan(int K, const WideParams &in, WideParams *out, int64_t *blocks, size_t *smem, bool *full);
cudaError_t launch_wide(int K, const WideParams &p, int64_t blocks, size_t smem, bool full, cudaStream_t st);

// Split form (vd_wide.cuh): one frame per cluster of `ranks` blocks; false
// if frames are too many, too short to gain, or too long for a cluster's shared memory.
// kSplitWarmup: chunks of K-1 stages (96 stages for K=7, 128 for K=9, 14 to 16 constraint lengths): at
// 2 dB and above hardly a segment runs twice.  kSplitGain: what the checks and barriers cost, in chunks.
constexpr int kSplitWarmup = 16, kSplitGain = 8;
bool split_plan(int K, const WideParams &in, int n_sm, SplitParams *out, int *ranks, size_t *smem);
cudaError_t launch_split(int K, const SplitParams &p, int ranks, size_t smem, cudaStream_t st);

// fp16 input: kernel shape for a stream of n_pairs frame pairs, and its launch.
struct F32Geom {
    KernelGeom geom;
    int threads_per_pair;
};
F32Geom geom_f32(int K, int64_t n_pairs, int n_sm);
cudaError_t launch_stream_f32(int K, int threads_per_pair, const StreamParams &p, int64_t blocks, cudaStream_t st);
bool geom_k7(int lanes, bool radix4, KernelGeom *g);
bool geom_k9(int lanes, bool radix4, KernelGeom *g);

}  // namespace vd
