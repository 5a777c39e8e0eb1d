// Segmented stream decode: branch metrics, radix-2 / radix-4 add-compare-select
// with packed survivors, and traceback from the overlap, fused in one kernel.
//
// Paper: arXiv 2011.13579.  Eq. BM (branch metric), Eq. PM / Eq. SP0 (ACS and
// survivor), Algorithms 1 and 2 (forward and backward procedures), Sec. III
// (frames of f stages with overlap), Thm. 1 (butterfly state indices),
// Thm. 2 and its corollary (all four branch outputs of a butterfly follow
// from its main output), Sec. VIII-A / Eq. radix4:PM, radix4:SP0 (two stages
// per step, traceback two stages per step).
//
// Mapping (one group of L lanes per PAIR of frames):
//   * the two frames of a pair are the two 16-bit halves of every register;
//   * register R (K-1 bits; the top log2(L) bits select the lane) holds, at
//     stage tau, the metric of state ROTR^tau(R).  With this rotation the two
//     left states 2g, 2g+1 of every butterfly sit in registers that differ
//     only in bit (tau mod (K-1)), and its two right states g, g+2^(K-2) land
//     in the same two registers: the ACS is in place.  When that bit is a
//     lane bit the partner comes from the other lane by one shuffle;
//   * the main output alpha of butterfly g is linear in the bits of g, so the
//     part contributed by the lane bits is folded into the LLR signs of that
//     lane and the rest is a compile-time constant per register;
//   * frames of a pair are right-aligned on a common padded length Wpad (a
//     multiple of the unroll period U), so they end together; the shorter
//     frame is preceded by stages of zero LLRs, which keep all-equal metrics
//     all-equal, and a frame that starts from the reset state gets its head
//     start on state 0 when its first stage arrives;
//   * decisions are embedded in the metrics (see StreamCfg::ES and
//     forward_pair) and go to a global scratch buffer: each group of ES stages leaves one
//     record of FW-bit fields per register, word r / RPW at bits FW (r % RPW) +
//     16h (h = 0, 1 the frame), whose highest bit is the register's decision at the record's last
//     stage, the next the decision at the stage before of the register it came
//     from, and so on along the same survivor.  K=7 radix 2: three stages, 4-bit
//     fields; K=9 and radix 4: two stages, 2-bit fields;
//   * radix-4: stages are taken in pairs (t-1, t).  The metrics are two
//     radix-2 steps (grouping the four candidates of a right state by their
//     middle state, as Eq. radix4:PM allows, gives exactly the same integers
//     and ties), and the survivor of right state j is the 2-bit pair
//     (d_m, d_i): the decision of j at stage t and the decision of the
//     middle state it selects at stage t-1 - exactly the 2-bit field of the
//     stage-pair records;
//   * traceback (Algorithm 2) walks groups of K-1 stages whose survivor words
//     are staged in shared memory; a group's decoded bits are the register
//     index at the group's start.  The persistent kernels (vd_batch.cuh) run
//     one pair's traceback, two groups every second group of stages, during
//     the next pair's forward pass.
#pragma once
#include <utility>
#include "vd_device.cuh"

namespace vd {

struct StreamParams {
    const int8_t *llr;      // depunctured received LLRs, [T][beta], int8
    int64_t n_info, T, f, v;
    int64_t n_win, n_pairs;
    uint32_t flags;         // bit0: terminated, bit1: start state unknown
    int32_t wpad_max;       // padded frame length the scratch of one warp holds
    uint32_t *out;          // packed decoded bits, LSB-first
    uint32_t *surv;         // survivor scratch: wpad_max x 32 x SW words per warp
    int32_t *pm_out;        // optional [n_win][2^(K-1)] canonical final metrics
    int *status;            // device status word (bit 0: a frame pair exceeded the scratch)
    int *counter;           // persistent form: task counter, zero at launch
    int64_t n_tasks;        // persistent form: tasks of 32/L frame pairs
};

// One frame as the decoder core sees it: stage indices are relative to the
// first stage of its stream (or packet), whose LLRs start at llr and whose
// decoded bits start at bit 0 of out.
struct FrameTask {
    const int8_t *llr;      // [T][beta] int8 of the frame's stream
    uint32_t *out;          // packed output of the frame's stream
    int32_t *pm;            // NULL, or 2^(K-1) canonical final metrics of this frame
    int64_t a, b, o, e;     // trellis stages [a, b), decoded stages [o, e)
    int valid, known, term; // real frame / starts from state 0 / ends at a terminated end
};

__host__ __device__ __forceinline__ FrameTask frame_task(const int8_t *llr, uint32_t *out, int32_t *pm,
                                                        int64_t s, int64_t n_win, int64_t n_info,
                                                        int64_t T, int64_t f, int64_t v,
                                                        uint32_t flags) {
    FrameTask t;
    t.llr = llr;
    t.out = out;
    t.valid = s < n_win;
    const Frame w = frame_of(t.valid ? s : 0, n_info, T, f, v, flags);
    t.a = w.a; t.b = w.b; t.o = w.o; t.e = w.e;
    t.known = t.valid && w.known_start;
    t.term = t.valid && w.term_end;
    t.pm = t.valid ? pm : nullptr;
    return t;
}

__host__ __device__ constexpr int ilog2(int x) { return x <= 1 ? 0 : 1 + ilog2(x / 2); }

// Unroll period: an even multiple of K-1 (rotation period) whose chunk of LLR
// bytes is a whole number of 32-bit words.
__host__ __device__ constexpr int chunk_stages(int K, int beta) {
    int u = K - 1;
    while ((u * beta) % 4 || (u % 2)) u += K - 1;
    return u;
}

template <int K, int BETA, uint64_t GENS, int L, bool RADIX4>
struct StreamCfg {
    using C = Code<K, BETA, GENS>;
    static constexpr int NB = C::NB;
    static constexpr int NS = C::NS;
    static constexpr int NR = NS / L;                 // registers per lane
    static constexpr int LR = ilog2(NR);              // local register bits
    static constexpr int U = chunk_stages(K, BETA);   // stages per chunk
    static constexpr int UW = U * BETA / 4;           // LLR words per chunk per frame
    // Embedded decisions: metrics are kept as 2^ES m + j, the ES low bits j of
    // each half carrying the decisions of the current record of ES stages;
    // see forward_pair.  ES = 3 (scale 8) for radix 2 where the range allows, else ES = 2
    // (scale 4).  Radix-4 takes stage-pair records: a field's two bits are the
    // radix-4 survivor of Eq. radix4:SP0 (the decision at the pair's second stage
    // and that of the middle state it selects), the candidates grouped by
    // middle state as two exact radix-2 steps (R10).
    //
    // Range.  Every branch metric carries + B, so it lies in [0, 2B] and no
    // metric falls within a chunk (a common per-stage offset changes no
    // decision, Eq. PM).  Every chunk of U = K-1 stages starts by shifting the
    // smallest metric of some states to X = 2 B NRECENT: the states whose last
    // NRECENT inputs are zero (all of them for NRECENT = 0).  Any state shares its older
    // inputs with one of them, and both metrics come from one ancestor NRECENT stages back (before a
    // frame's first stages have filled the register, from starts that are equal or
    // higher on the few), so no metric falls below zero.  Bounds on m (per half):
    //   * steady state: all metrics lie within 254 DMAX of each other (Code),
    //     so after the shift m is in [0, X + 254 DMAX], and a chunk adds at most 2 U B;
    //   * a frame that starts from the reset state puts state 0 HT above the others
    //     when its first stage arrives; for NRECENT > 0 the others go to 0.  If t < K-1 stages of
    //     that chunk follow, its metrics then reach at most HT + 2 t B (NRECENT = 0: from the
    //     level of the others, at least the smallest metric); that chunk's shift leaves
    //     the frame alone (NRECENT = 0: it moves the smallest metric to 0), and the next chunk adds 2 U B.
    // The largest 2^ES m + 2^ES - 1 must stay within 16 unsigned bits.  With several
    // lanes NRECENT is as large as that allows: the smallest metric of two registers instead
    // of a lane's all and a reduction over the lanes (K=9, four lanes: 672 -> 634 us for 2^24 bits
    // together with the lane signs below; then 621 with a copy of the chunk for frame starts).  With one
    // lane the smallest of all 64 costs 5 instructions a stage that the chip has room for, and
    // was measured 1% faster than the copies and masks of the other way (654 against 660 us for six
    // streams of 2^24 bits).
    static constexpr int TOP_RESET = C::HT + 2 * (2 * U - 1) * C::B;
    __host__ __device__ static constexpr int top_steady(int recent) {
        return 2 * C::B * recent + 254 * C::DMAX + 2 * U * C::B;
    }
    __host__ __device__ static constexpr bool fits(int es, int top) { return (top << es) + (1 << es) - 1 <= 65535; }
    static constexpr bool ES3_OK = !RADIX4 && NB % 3 == 0 && NR % 4 == 0 && fits(3, TOP_RESET) && fits(3, top_steady(0));
    static constexpr int ES = ES3_OK ? 3 : 2;
    static constexpr int LB = NB - LR;                // lane bits of a register index
    __host__ __device__ static constexpr int recent() {
        int r = 0;
        while (L > 1 && r < NB - 1 && fits(ES, top_steady(r + 1))) ++r;
        return r;
    }
    static constexpr int NRECENT = recent();
    static constexpr int NMIN = 1 << (NB - NRECENT);  // those states: registers 0 .. NMIN - 1 of lane 0
    static constexpr int X = 2 * C::B * NRECENT;
    static constexpr int SC = 1 << ES;                // metric scale
    static constexpr int FW = ES == 3 ? 4 : 2;        // record field width (bits)
    static constexpr int RPW = 16 / FW;               // registers per record word (per half)
    static constexpr int NW = NR / RPW;               // record words per lane
    static constexpr int SW = (NW + ES - 1) / ES;     // scratch words per lane per stage
    // output b at phase ph: the lane bits whose parity flips it (the lanes' part of alpha)
    __host__ __device__ static constexpr uint32_t lane_mask(int ph, int b) {
        uint32_t m = 0;
        for (int i = 0; i < LB; ++i)
            m |= ((C::alpha(C::rotr(1u << (LR + i), ph) >> 1) >> b) & 1u) << i;
        return m;
    }
    static_assert(NS % L == 0 && L <= 32 && (L & (L - 1)) == 0, "L must be a power of two");
    static_assert(U == NB && U % ES == 0, "a chunk is one rotation of the registers and holds whole records");
    static_assert(NRECENT >= LB && NMIN <= NR, "the states of the shift sit in lane 0");
    static_assert(NR % RPW == 0 && NW * 32 <= 32 * ES * SW, "a record fits the scratch of its ES stages");
    static_assert(fits(ES, TOP_RESET) && fits(ES, top_steady(NRECENT)), "metric range");
    static_assert(C::lv() == (1u << BETA) - 1u && C::mv() == (1u << BETA) - 1u, "complement branch outputs");
};

template <typename Fn, int... S>
__device__ __forceinline__ void static_for_impl(Fn &&fn, std::integer_sequence<int, S...>) {
    (fn(std::integral_constant<int, S>{}), ...);
}
// Calls fn(integral_constant<int, i>) for i = 0 .. N-1: loop indices are compile-time.
template <int N, typename Fn>
__device__ __forceinline__ void static_for(Fn &&fn) {
    static_for_impl(fn, std::make_integer_sequence<int, N>{});
}

// LLR chunk loading in two steps so the loads of chunk c+1 are in flight while
// chunk c is decoded: fetch() issues the aligned 32-bit loads of bytes
// [vb, vb + 4*UW) relative to the frame's first byte `base`, finish()
// re-aligns them with funnel shifts.  A chunk that is not wholly inside the
// frame's bytes [0, hi) (the first chunk of a padded frame) is assembled byte
// by byte in finish() with zeros outside the range.  Offsets are 32-bit: a
// frame spans far fewer than 2^31 bytes.
template <int UW>
struct ChunkRaw {
    uint32_t raw[UW + 1];
    uint32_t sh;
    bool fast;
};

template <int UW>
__device__ __forceinline__ void fetch_chunk(const int8_t *base, int32_t vb, int32_t hi, ChunkRaw<UW> &c) {
    c.fast = vb >= 0 && vb + 4 * UW <= hi;
    if (c.fast) {
        const uintptr_t addr = reinterpret_cast<uintptr_t>(base) + (uintptr_t)(uint32_t)vb;
        const uint32_t mis = (uint32_t)(addr & 3u);
        const uint32_t *p = reinterpret_cast<const uint32_t *>(addr - mis);
#pragma unroll
        for (int i = 0; i < UW; ++i) c.raw[i] = __ldg(p + i);
        // the extra word holds the last bytes of the chunk when it is misaligned;
        // it contains at least one byte inside the stream, so it is readable
        c.raw[UW] = mis ? __ldg(p + UW) : 0u;
        c.sh = 8u * mis;
    }
}

template <int UW>
__device__ __forceinline__ void finish_chunk(const int8_t *base, int32_t vb, int32_t hi,
                                             const ChunkRaw<UW> &c, uint32_t (&w)[UW]) {
    if (c.fast) {
#pragma unroll
        for (int i = 0; i < UW; ++i) w[i] = funnel_r(c.raw[i], c.raw[i + 1], c.sh);
    } else {
#pragma unroll
        for (int i = 0; i < UW; ++i) {
            uint32_t x = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int32_t pos = vb + 4 * i + k;
                if (pos >= 0 && pos < hi) x |= (uint32_t)(uint8_t)base[pos] << (8 * k);
            }
            w[i] = x;
        }
    }
}

// Selects element idx of a small register array without local memory.
template <int N>
__device__ __forceinline__ uint32_t pick(const uint32_t *a, uint32_t idx) {
    uint32_t r = a[0];
#pragma unroll
    for (int i = 1; i < N; ++i) r = (idx == (uint32_t)i) ? a[i] : r;
    return r;
}

// Per-half minimum of N packed registers: a tree of three-input minima.
template <int N>
__device__ __forceinline__ uint32_t min_tree(const uint32_t (&v)[N]) {
    if constexpr (N == 1) {
        return v[0];
    } else if constexpr (N == 2) {
        return min_u16x2(v[0], v[1]);
    } else {
        constexpr int M = (N + 2) / 3;
        uint32_t w[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (3 * i + 2 < N) w[i] = __vimin3_u16x2(v[3 * i], v[3 * i + 1], v[3 * i + 2]);
            else if (3 * i + 1 < N) w[i] = min_u16x2(v[3 * i], v[3 * i + 1]);
            else w[i] = v[3 * i];
        }
        return min_tree<M>(w);
    }
}

// ------------------------------------------------------------ traceback
//
// Backward procedure (Algorithm 2) for one pair of frames, resumable: it walks
// groups of K-1 stages (so the phase of every stage in a group is a
// compile-time constant) from Wpad-1 down to the frames' first decoded
// stages.  A persistent warp calls step() after every second chunk of the NEXT frame
// pair's forward pass, so the traceback's dependent chain and its memory
// latency hide behind forward work.  The survivor records of the groups walked next (two, or
// 2 D: see D below) are copied into a per-warp shared-memory staging area by cp.async
// while earlier groups are walked; the per-lane state lives in shared memory
// between steps.  One lane per pair follows both frames.  With several lanes and embedded
// decisions, lanes 0 and 1 of a group (and those that repeat them) follow one frame each and read
// any lane's records from the staging.  In the fp32 form (a decision word per stage and
// frame: bit (r & 31) of word (r >> 5) for register r, or bit r and 16 + r of one word for lanes of 16 registers)
// every lane follows both frames and the lane that owns the current register supplies its bit by a shuffle.

// All fields are 32-bit words (pointers and the 64-bit bit accumulator are
// split in two): 23 words, an odd stride, so the per-thread records in shared
// memory are read and written without bank conflicts.
struct TbState {
    uint32_t out_w[2][2];    // packed output of each frame's stream (pointer words)
    uint32_t surv_w[2];      // this lane's survivor records (pointer words)
    uint32_t oacc_w[2][2];   // decoded bits not yet stored: bit i = stage (lowest emitted + i)
    uint32_t R[2];           // current register of each frame (traceback state)
    int32_t onb[2];          // number of bits in oacc
    int32_t t0;              // first stage of the next group; finished when t0 < tau_store
    int32_t tau_store;
    int32_t tauo[2], taue[2];
    int32_t toff[2];         // stage in the frame's stream = tau + toff
    int32_t slot;            // pair of slots walked next (deep staging only)

    __device__ __forceinline__ static uint64_t join(uint32_t lo, uint32_t hi) {
        return ((uint64_t)hi << 32) | lo;
    }
    __device__ __forceinline__ uint32_t *out(int h) const {
        return reinterpret_cast<uint32_t *>(join(out_w[h][0], out_w[h][1]));
    }
    __device__ __forceinline__ void set_out(int h, uint32_t *p) {
        const uint64_t x = reinterpret_cast<uint64_t>(p);
        out_w[h][0] = (uint32_t)x;
        out_w[h][1] = (uint32_t)(x >> 32);
    }
    __device__ __forceinline__ const uint32_t *surv() const {
        return reinterpret_cast<const uint32_t *>(join(surv_w[0], surv_w[1]));
    }
    __device__ __forceinline__ void set_surv(const uint32_t *p) {
        const uint64_t x = reinterpret_cast<uint64_t>(p);
        surv_w[0] = (uint32_t)x;
        surv_w[1] = (uint32_t)(x >> 32);
    }
    __device__ __forceinline__ uint64_t oacc(int h) const { return join(oacc_w[h][0], oacc_w[h][1]); }
    __device__ __forceinline__ void set_oacc(int h, uint64_t v) {
        oacc_w[h][0] = (uint32_t)v;
        oacc_w[h][1] = (uint32_t)(v >> 32);
    }
};
static_assert(sizeof(TbState) == 23 * 4 && alignof(TbState) == 4, "odd-word traceback record");

__device__ __forceinline__ void cp_async_bytes16(void *smem, const void *gmem) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_bytes8(void *smem, const void *gmem) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_bytes4(void *smem, const void *gmem) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// D: pairs of groups in flight.  The persistent kernels walk a pair between two
// chunks of forward work and need one; the kernels that trace back with
// nothing else to do keep several, so that a step waits for a copy issued D steps before.
template <int K, int L, bool RADIX4, int NR, int NW, int ES = 0, int D = 1>
struct Traceback {
    static constexpr int NB = K - 1;
    static constexpr int G = NB;                 // stages per group
    static constexpr int LR = ilog2(NR);
    static constexpr int WPF = NR >= 32 ? NR / 32 : 1;
    static constexpr bool EMB = ES != 0;
    static constexpr int FW = ES == 3 ? 4 : 2;   // record field width (bits)
    static constexpr int RPW = 16 / FW;          // registers per record word (per half)
    // survivor records: one per stage (NW words per lane), or with embedded
    // decisions one per ES stages (NR / RPW words per lane, FW-bit fields)
    static constexpr int REC = EMB ? G / ES : G; // records per group
    static constexpr int RW = EMB ? NR / RPW : NW;   // words per record and lane
    static constexpr int SLOT_WORDS = REC * 32 * RW;
    static constexpr int STAGE_WORDS = 2 * SLOT_WORDS * D;   // per warp
    static_assert(!EMB || (G % ES == 0 && (!RADIX4 || ES == 2)), "embedded decisions: whole records per group");

    // Copies the records of stages t0, t0-1, .., t0-G+1 (those >= tau_store)
    // to a slot (the caller commits the copies as one group).
    __device__ static void issue_slot(const TbState &s, int t0, uint32_t *slot, int wlane) {
#pragma unroll
        for (int g = 0; g < REC; ++g) {
            const int t = t0 - (EMB ? ES * g : g);   // EMB: the last stage of a record
            if (t >= s.tau_store) {
                uint32_t *dst = slot + (g * 32 + wlane) * RW;
                // this lane's words of scratch row t / ES (EMB) or t
                const uint32_t *src = s.surv() + (size_t)(EMB ? (t / ES) : t) * 32 * RW;
                if constexpr (RW == 1) {
                    cp_async_bytes4(dst, src);
                } else if constexpr (RW == 2) {
                    cp_async_bytes8(dst, src);
                } else {
#pragma unroll
                    for (int i = 0; i < RW; i += 4) cp_async_bytes16(dst + i, src + i);
                }
            }
        }
    }

    // Copies the groups of top stages t0 and t0 - G to slots 0 and 1 as one group of copies.
    __device__ static void issue_pair(const TbState &s, int t0, uint32_t *stg, int wlane) {
        issue_slot(s, t0, stg, wlane);
        issue_slot(s, t0 - G, stg + SLOT_WORDS, wlane);
        cp_async_commit();
    }

    __device__ static bool active(const TbState &s) { return s.t0 >= s.tau_store; }

    // The staging of the pair that is walked next.
    __device__ static uint32_t *current(const TbState &s, uint32_t *stg) {
        if constexpr (D == 1) return stg;
        else return stg + s.slot * (2 * SLOT_WORDS);
    }

    // Starts the copies of the first D pairs of groups.
    __device__ static void begin(TbState &s, uint32_t *stg, int wlane) {
        s.slot = 0;
#pragma unroll
        for (int d = 0; d < D; ++d) issue_pair(s, s.t0 - 2 * G * d, stg + d * (2 * SLOT_WORDS), wlane);
    }

    // With embedded decisions and several lanes per pair, lanes 0 and 1 (and
    // those that repeat them) follow one frame each; otherwise every lane follows both.
    static constexpr bool SPLIT = EMB && L > 1;
    static constexpr int NF = SPLIT ? 1 : 2;
    __device__ __forceinline__ static int frame(int i, int lane) { return SPLIT ? (lane & 1) : i; }

    // A step walks the two staged groups: open() before the first group's
    // first record, walk<j>() per record of each group, close() after the
    // second group's last record.
    static constexpr int STEPS = EMB ? G / ES : G;   // walk<> calls per group
    struct Live {
        uint32_t R[2];           // traceback registers (SPLIT: one)
        const uint32_t *slot;    // staging slot of the group
        bool act;
    };

    // Branch-free: an inactive walk (act false) reads in-bounds staging words
    // and changes nothing that close() keeps, so the embedded-decision walk
    // runs unconditionally (measured 3% faster than a branch around it).
    __device__ static void open(const TbState &s, const uint32_t *stg, Live &v, int lane, unsigned gmask) {
        v.act = active(s);
        cp_async_wait<D - 1>();
        if constexpr (SPLIT) __syncwarp(gmask);   // the group's lanes read one another's copies
        v.slot = stg;   // of the current pair
#pragma unroll
        for (int i = 0; i < NF; ++i) v.R[i] = s.R[frame(i, lane)] & (uint32_t)((1 << NB) - 1);
    }

    template <int j>
    __device__ static void walk(Live &v, int wlane, int lane, unsigned gmask, int grp_base) {
        if (!EMB && !v.act) return;
        auto words = [&](int g, uint32_t (&wd)[RW]) {
            const uint32_t *p = v.slot + (g * 32 + wlane) * RW;
            if constexpr (RW == 1) {
                wd[0] = p[0];
            } else if constexpr (RW == 2) {
                const uint2 x = *reinterpret_cast<const uint2 *>(p);
                wd[0] = x.x; wd[1] = x.y;
            } else {
#pragma unroll
                for (int i = 0; i < RW; i += 4) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(p + i);
                    wd[i] = x.x; wd[i + 1] = x.y; wd[i + 2] = x.z; wd[i + 3] = x.w;
                }
            }
        };
        // The survivor word of register R in frame h, rotated right so that
        // R's decision bit lands at bit position ph.
        auto rotated = [&](const uint32_t (&wd)[RW], int h, uint32_t R, int ph) -> uint32_t {
            uint32_t word, bit;
            if constexpr (NR >= 32) {
                word = pick<WPF>(&wd[h * WPF], (R >> 5) & (uint32_t)(WPF - 1));
                bit = R;
            } else {
                word = wd[0];
                bit = (R & (uint32_t)(NR - 1)) + 16u * (uint32_t)h;
            }
            return __funnelshift_r(word, word, bit - (uint32_t)ph);
        };
        auto owner = [&](uint32_t x, uint32_t R) -> uint32_t {
            if constexpr (L > 1) return __shfl_sync(gmask, x, grp_base + (int)(R >> LR));
            else return x;
        };
        if constexpr (EMB) {
            // record of stages (t-ES+1 .. t): register R's field holds the
            // decision of R at stage t (bit ES-1), the decision at stage t-1
            // of the register it came from (bit ES-2), and so on.  The phases
            // of the record's stages are adjacent (a group starts at phase 0
            // and holds whole records), so one rotation puts every bit in
            // place and one select replaces those bits of R.
            constexpr int phh = ((NB - 1 - ES * j) % NB + NB) % NB;   // phase of stage t
            constexpr int ph0 = phh - (ES - 1);
            static_assert(ph0 >= 0, "a record's phases do not wrap");
            constexpr uint32_t m = ((1u << ES) - 1u) << ph0;
            // the pair's record: register R in word R / RPW, the group's lanes one after another
            const uint32_t *rec = v.slot + (j * 32 + grp_base) * RW;
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const uint32_t R = v.R[i];
                const uint32_t word = rec[R / RPW];   // the word holding R
                const uint32_t sh = (uint32_t)FW * (R & (uint32_t)(RPW - 1)) + 16u * (uint32_t)frame(i, lane);
                const uint32_t t = __funnelshift_r(word, word, sh - (uint32_t)ph0);
                v.R[i] = (R & ~m) | (t & m);
            }
        } else {
            constexpr int ph = ((NB - 1 - j) % NB + NB) % NB;   // group starts at -1 mod (K-1)
            uint32_t wd[RW];
            words(j, wd);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t t = owner(rotated(wd, h, v.R[h], ph), v.R[h]);
                v.R[h] = (v.R[h] & ~(1u << ph)) | (t & (1u << ph));
            }
        }
    }

    // Emits the two groups' decoded bits, refills both slots with the two
    // groups after them and advances.  RB: the registers after group A (the
    // start of group B).
    __device__ static void close(TbState &s, uint32_t *stg, const Live &v, const uint32_t (&RB)[2], int wlane,
                                 int lane, unsigned gmask) {
        if (!v.act) return;   // the same for all lanes of a group
        const int t0 = s.t0;
        const int tl = t0 - (2 * G - 1);   // lowest stage of group B
        // Each bit position of R is replaced once per group, so a group's
        // decoded bits (the input bit of each stage's state) are the bits of
        // R at the start of the group: group A's from s.R, group B's from RB;
        // stage tl + i is bit i of (R_A << G) | R_B.
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            const int h = frame(i, lane);
            const int lo = tl > s.tauo[h] ? tl : s.tauo[h];
            const int hi = (t0 + 1) < s.taue[h] ? (t0 + 1) : s.taue[h];
            if (hi > lo) {
                const int m = hi - lo;
                const uint32_t X = ((s.R[h] & (uint32_t)((1 << NB) - 1)) << G) | RB[i];
                const uint64_t bits = (uint64_t)((X >> (lo - tl)) & ((1u << m) - 1u));
                uint64_t acc = (s.oacc(h) << m) | bits;
                int nb = s.onb[h] + m;
                const int a = lo + s.toff[h];              // stream stage of bit 0
                const int wb = (a + nb - 1) & ~31;         // first stage of the top word
                if (a <= wb) {
                    if (SPLIT ? lane < 2 : lane == (L > 1 ? h : 0)) s.out(h)[wb >> 5] = (uint32_t)(acc >> (wb - a));
                    nb = wb - a;
                    acc &= (1ull << nb) - 1ull;
                }
                s.set_oacc(h, acc);
                s.onb[h] = nb;
            }
        }
#pragma unroll
        for (int i = 0; i < NF; ++i) s.R[frame(i, lane)] = v.R[i];
        if constexpr (SPLIT) __syncwarp(gmask);   // every lane has read the slots
        // refill both slots with the two groups D pairs on, then advance
        issue_pair(s, t0 - 2 * G * D, stg, wlane);
        s.t0 = t0 - 2 * G;
        if constexpr (D > 1) s.slot = s.slot + 1 == D ? 0 : s.slot + 1;
    }

    // The traceback work that belongs after stage S of chunk c of a forward
    // pass (chunks of U stages, a whole number of groups): one step (two
    // groups) after the last stage of every second group, so the state
    // bookkeeping, the wait and the commit are paid once per two groups.
    // (Spreading the records over the stages was measured 2% slower: the
    // forward stages schedule better as whole blocks.)
    template <int S, int U>
    __device__ static void sub(TbState &s, uint32_t *stg, Live &, int wlane, int lane, unsigned gmask,
                               int grp_base, int c) {
        static_assert(U % G == 0, "chunks hold whole groups");
        if constexpr (S % G == G - 1) {
            if ((c * (U / G) + S / G) & 1) step(s, stg, wlane, lane, gmask, grp_base);
        }
    }

    // Walks the two staged groups (those that remain) and refills both slots.
    __device__ static void step(TbState &s, uint32_t *ring, int wlane, int lane, unsigned gmask,
                                int grp_base) {
        uint32_t *stg = current(s, ring);
        Live v;
        v.R[0] = v.R[1] = 0u;
        open(s, stg, v, lane, gmask);
        static_for<STEPS>([&](auto jc) { walk<decltype(jc)::value>(v, wlane, lane, gmask, grp_base); });
        const uint32_t RB[2] = {v.R[0], v.R[1]};
        const bool act = v.act;
        v.slot = stg + SLOT_WORDS;
        v.act = act && s.t0 - G >= s.tau_store;
        static_for<STEPS>([&](auto jc) { walk<decltype(jc)::value>(v, wlane, lane, gmask, grp_base); });
        v.act = act;
        close(s, stg, v, RB, wlane, lane, gmask);
    }

    // Walks every remaining group and waits for all copies.
    __device__ static void drain(TbState &s, uint32_t *stg, int wlane, int lane, unsigned gmask,
                                 int grp_base) {
        while (active(s)) step(s, stg, wlane, lane, gmask, grp_base);
        cp_async_wait<0>();
    }
};

// Forward procedure (Algorithm 1) and survivor storage for one pair of frames.
// Called by one group of L lanes; surv is the frame pair's survivor buffer in
// this warp's scratch (wpad_cap stages x 32 lanes x SW words); wlane is the
// lane in the warp.  hook(integral_constant<int, S>, c) runs after stage S of
// every chunk c of U stages (the persistent kernels walk a previous pair's
// traceback there, two groups of K-1 stages every second group).  On return tb
// holds the traceback start of this pair; returns false (tb inactive) if the
// pair does not fit the scratch, which host plans never produce.
template <int K, int BETA, uint64_t GENS, int L, bool RADIX4, typename Hook>
__device__ __forceinline__ bool forward_pair(const FrameTask (&ft)[2], uint32_t *surv, int wpad_cap,
                                             int wlane, int lane, unsigned gmask, int grp_base,
                                             int *status, TbState &tb, Hook &&hook) {
    using Cfg = StreamCfg<K, BETA, GENS, L, RADIX4>;
    using C = typename Cfg::C;
    constexpr int NB = Cfg::NB, NR = Cfg::NR, LR = Cfg::LR, LB = Cfg::LB, U = Cfg::U, UW = Cfg::UW, NW = Cfg::NW;
    constexpr int ES = Cfg::ES, SC = Cfg::SC, RPW = Cfg::RPW, FW = Cfg::FW;
    constexpr uint32_t H = 0x00010001u;
    constexpr uint32_t SEED = (uint32_t)(SC * Cfg::X) * H;   // all-equal start and target of the chunks' shift

    // ---------------------------------------------------------- frame plan
    int64_t fa[2], fb[2], fo[2], fe[2];
    bool known[2], term[2], valid[2];
    int64_t W[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        fa[h] = ft[h].a; fb[h] = ft[h].b; fo[h] = ft[h].o; fe[h] = ft[h].e;
        valid[h] = ft[h].valid != 0;
        known[h] = ft[h].known != 0;
        term[h] = ft[h].term != 0;
        W[h] = valid[h] ? (fb[h] - fa[h]) : 0;
    }
    const int64_t Wmax = W[0] > W[1] ? W[0] : W[1];
    const int Wpad = (int)(((Wmax + U - 1) / U) * U);
    tb.t0 = -1;
    tb.tau_store = 0;
    tb.slot = 0;
    tb.R[0] = tb.R[1] = 0;
    if (Wpad > wpad_cap) {   // never happens for plans built by the host; refuse, do not overrun
        if (lane == 0) atomicOr(status, 1);
        return false;
    }
    int tau0[2], tauo[2], taue[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        tau0[h] = Wpad - (int)W[h];
        tauo[h] = valid[h] ? tau0[h] + (int)(fo[h] - fa[h]) : Wpad;
        taue[h] = valid[h] ? tau0[h] + (int)(fe[h] - fa[h]) : Wpad;
    }
    const int tau_store = tauo[0] < tauo[1] ? tauo[0] : tauo[1];
    const int reset_at0 = known[0] ? tau0[0] : -1;
    const int reset_at1 = known[1] ? tau0[1] : -1;

    // the traceback's fixed parameters are written now (tb may live in
    // shared memory), so they hold no registers during the forward pass
    tb.set_out(0, ft[0].out);
    tb.set_out(1, ft[1].out);
    tb.set_surv(surv + (size_t)wlane * NW);
    tb.set_oacc(0, 0u);
    tb.set_oacc(1, 0u);
    tb.onb[0] = tb.onb[1] = 0;
    tb.tau_store = tau_store;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        tb.tauo[h] = tauo[h];
        tb.taue[h] = taue[h];
        tb.toff[h] = (int32_t)(fa[h] - tau0[h]);
    }

    // ------------------------------------------------------------ metrics
    uint32_t P[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) P[r] = SEED;   // all-equal: unknown start

    // LLR bytes relative to each frame's first stage; stage tau of the pair is
    // frame stage tau - tau0
    const int8_t *fbase0 = ft[0].llr + fa[0] * BETA, *fbase1 = ft[1].llr + fa[1] * BETA;
    const int32_t hi0 = valid[0] ? (int32_t)W[0] * BETA : 0, hi1 = valid[1] ? (int32_t)W[1] * BETA : 0;
    int32_t vb0 = -tau0[0] * BETA, vb1 = -tau0[1] * BETA;   // offset of the chunk being fetched

    // the record of stages (tau - ES + 1 .. tau) is row tau / ES of the scratch:
    // NW words per lane, lane-major
    auto store_rec = [&](int tau, const uint32_t (&v)[NW]) {
        uint32_t *dst = surv + ((size_t)(tau / ES) * 32 + (size_t)wlane) * NW;
        if constexpr (NW == 1) {
            *dst = v[0];
        } else if constexpr (NW == 2) {
            *reinterpret_cast<uint2 *>(dst) = make_uint2(v[0], v[1]);
        } else {
#pragma unroll
            for (int i = 0; i < NW; i += 4)
                *reinterpret_cast<uint4 *>(dst + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        }
    };

    // runtime +1 / -1 for the FMA-pipe multiply-adds (blocks are one-dimensional)
    const uint32_t one = threadIdx.y + 1u;
    const uint32_t m1 = 0u - one;
    const uint32_t fwmul = one << FW;   // 2^FW: shifts a record word by one field
    const uint32_t mul16 = one << 4, mul64 = one << 6;   // 2-bit fields: shifts by two and three fields

    // A lane's part of the branch outputs is a sign per (phase, output): with
    // x = l + 127, u = SC x or SC (254 - x) = x mul + add is the scaled
    // l + 127 with that sign (one pair of registers per parity mask in use).
    uint32_t mul[1 << LB], add[1 << LB], xm[LB > 0 ? LB : 1];
#pragma unroll
    for (int m = 0; m < (1 << LB); ++m) {
        const bool neg = __popc((uint32_t)lane & (uint32_t)m) & 1;
        mul[m] = neg ? 0u - (uint32_t)SC : (uint32_t)SC;
        add[m] = neg ? (uint32_t)(254 * SC) * H : 0u;
    }
    xm[0] = 0u;
#pragma unroll
    for (int i = 0; i < LB; ++i) xm[i] = (((uint32_t)lane >> i) & 1u) * H;

    const int nchunks = Wpad / U;
    uint32_t pmin = SEED;            // per half: smallest metric of the states of the shift
    uint32_t keepn = 0xFFFFFFFFu;    // halves that the next chunk's shift moves
    ChunkRaw<UW> nx0, nx1;
    if (nchunks > 0) {
        fetch_chunk<UW>(fbase0, vb0, hi0, nx0);
        fetch_chunk<UW>(fbase1, vb1, hi1, nx1);
    }
    // One chunk; RESET: a frame may start in it from the reset state.  The copy
    // without that test is straight-line code but for the traceback of the hook: a
    // branch per stage keeps the compiler from overlapping the stages' branch
    // metrics with their dependent chains.
    constexpr bool HEADSTART_COPY = Cfg::NRECENT > 0;
    auto chunk = [&](auto Reset, int c) {
        constexpr bool RESET = decltype(Reset)::value;
        uint32_t cw0[UW], cw1[UW];
        {
            const ChunkRaw<UW> cur0 = nx0, cur1 = nx1;
            const int32_t cb0 = vb0, cb1 = vb1;
            vb0 += U * BETA;
            vb1 += U * BETA;
            if (c + 1 < nchunks) {
                fetch_chunk<UW>(fbase0, vb0, hi0, nx0);
                fetch_chunk<UW>(fbase1, vb1, hi1, nx1);
            }
            finish_chunk<UW>(fbase0, cb0, hi0, cur0, cw0);
            finish_chunk<UW>(fbase1, cb1, hi1, cur1, cw1);
        }
        // the shift of a chunk is folded into the branch metrics of its first
        // stage (adding tn to every candidate shifts every new metric by tn)
        const uint32_t tn = sub_s16x2(SEED, pmin) & keepn;
        keepn = 0xFFFFFFFFu;

        static_for<U>([&](auto Sc) {
            constexpr int S = decltype(Sc)::value;
            constexpr int PH = S;
            constexpr int KS = S % ES;               // stage within the record
            constexpr uint32_t OFF = H << KS;        // the odd candidates' mark
            constexpr uint32_t FM = ((1u << ES) - 1u) * H;
            constexpr bool CROSS = PH >= LR;         // the butterfly's partner is in another lane
            constexpr int lb = CROSS ? PH - LR : 0;
            const int tau = c * U + S;

            if constexpr (!HEADSTART_COPY) {
                if (__builtin_expect(tau == reset_at0 || tau == reset_at1, 0)) {
                    const uint32_t hm = (tau == reset_at0 ? 0xFFFFu : 0u) | (tau == reset_at1 ? 0xFFFF0000u : 0u);
                    if (lane == 0) P[0] = add_u16x2(P[0], ((uint32_t)(SC * C::HT) * H) & hm);
                }
            }

            // ---- branch metrics of this stage (Eq. BM), both frames at once,
            // scaled and biased: u_b = SC (l_b + 127) in [0, 254 SC], and the metric
            // of pattern x is sum_b (x_b ? 254 SC - u_b : u_b).  Every half of every
            // intermediate is non-negative and below 2^16, so plain 32-bit
            // arithmetic is exact per half.  Where the partner is in another lane, the
            // lane of the odd register carries the odd candidate's mark in all its own
            // metrics: added to one u, it reaches every sum.
            uint32_t u[BETA];
#pragma unroll
            for (int b = 0; b < BETA; ++b) {
                const int j = S * BETA + b;
                const uint32_t k = (uint32_t)(j & 3);
                const uint32_t sel = k | ((k + 8u) << 4) | ((k + 4u) << 8) | ((k + 12u) << 12);
                const uint32_t x = add_u16x2(prmt(cw0[j >> 2], cw1[j >> 2], sel), 127u * H);   // sign-extended pair + 127
                const uint32_t m = Cfg::lane_mask(PH, b);
                u[b] = L == 1 ? x : imad(x, mul[m], add[m]);
            }
            const uint32_t own = CROSS ? xm[lb] << KS : 0u;
            if constexpr (CROSS) u[BETA - 1] += own;
            constexpr int HALF = 1 << (BETA - 1), FULL = (1 << BETA) - 1;
            uint32_t E[1 << BETA];
            E[0] = u[BETA - 1];
#pragma unroll
            for (int b = 0; b < BETA - 1; ++b) {
#pragma unroll
                for (int x = 0; x < (1 << b); ++x) {
                    E[x | (1 << b)] = (E[x] + (uint32_t)(254 * (L == 1 ? 1 : SC)) * H) - u[b];
                    E[x] = E[x] + u[b];
                }
            }
            if constexpr (L == 1) {
#pragma unroll
                for (int x = 0; x < HALF; ++x) E[x] <<= ES;
            }
            // complement patterns (corollary of Thm. 2): 2 B minus the pattern's metric
            constexpr uint32_t CC = (uint32_t)(2 * C::B * SC) * H;
            const uint32_t cc = CROSS ? CC + 2u * own : CC;
#pragma unroll
            for (int x = 0; x < HALF; ++x) E[x ^ FULL] = CROSS ? imad(E[x], m1, cc) : CC - E[x];
            uint32_t O[1 << BETA];   // the candidates marked where E's are not (CROSS: of the complement of x)
#pragma unroll
            for (int x = 0; x <= FULL; ++x) {
                if constexpr (CROSS) O[x] = imad(E[x], m1, CC + OFF);
                else O[x] = x < HALF ? E[x] + OFF : (CC + OFF) - E[x ^ FULL];
            }
            if constexpr (S == 0) {
#pragma unroll
                for (int x = 0; x <= FULL; ++x) {
                    E[x] = add_u16x2(E[x], tn);
                    O[x] = add_u16x2(O[x], tn);
                }
            }
            // A frame that starts from the reset state: until its first stage its
            // half of every metric is X + S B (all-equal start, zero-LLR stages,
            // shifts to X).  Its start sets state 0 (register 0 of lane 0 at every stage) to HT and
            // the others to 0: that level goes out through this stage's branch metrics.
            if (RESET && HEADSTART_COPY && (tau == reset_at0 || tau == reset_at1)) {
                const uint32_t hm = (tau == reset_at0 ? 0xFFFFu : 0u) | (tau == reset_at1 ? 0xFFFF0000u : 0u);
                const uint32_t down = ((0u - (uint32_t)(SC * (Cfg::X + S * C::B))) & 0xFFFFu) * H & hm;
#pragma unroll
                for (int x = 0; x <= FULL; ++x) {
                    E[x] = add_u16x2(E[x], down);
                    O[x] = add_u16x2(O[x], down);
                }
                if (lane == 0) P[0] = add_u16x2(P[0], ((uint32_t)(SC * C::HT) * H) & hm);
                if constexpr (S > 0) keepn &= ~hm;
            }

            // ---- add-compare-select with embedded decisions.  A metric half is
            // 2^ES m + j: m the path metric (Eq. PM) and j < 2^ES the decisions (Eq. SP0)
            // of the current record of ES stages along the state's
            // survivor.  Odd candidates carry + 2^k at the record's stage
            // k, so the max itself records "the odd predecessor wins or
            // ties" in bit k: with j_even, j_odd < 2^k a tie leaves the
            // odd candidate larger by 2^k + j_odd - j_even > 0, and a
            // metric difference of one (2^ES in these units) outweighs
            // 2^k + j_odd - j_even <= 2^(k+1) - 1 <= 2^ES - 1.  The
            // winner's own bits below k (its decisions at the record's
            // earlier stages) travel with it.  After the record's last
            // stage the fields are stored and cleared: no per-state
            // decision arithmetic.
            if constexpr (!CROSS) {
#pragma unroll
                for (int ra = 0; ra < NR; ++ra) {
                    if (ra & (1 << PH)) continue;
                    const int rb = ra | (1 << PH);
                    const uint32_t a = C::alpha(C::rotr((uint32_t)ra, PH) >> 1);
                    const uint32_t Pa = P[ra], Pb = P[rb];
                    const uint32_t cb0 = add_u16x2(Pb, O[a ^ FULL]);    // odd -> j0
                    const uint32_t cb1 = add_u16x2(Pb, O[a]);           // odd -> j1
                    P[ra] = addmax_u16x2(Pa, E[a], cb0);                // even -> j0
                    P[rb] = addmax_u16x2(Pa, E[a ^ FULL], cb1);         // even -> j1
                }
            } else {
                // the lane of the even (odd) register computes j0 (j1): either way its
                // own branch carries pattern a and the other lane's the complement
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const uint32_t a = C::alpha(C::rotr((uint32_t)r, PH) >> 1);
                    const uint32_t oth = __shfl_xor_sync(gmask, P[r], 1 << lb);
                    P[r] = addmax_u16x2(P[r], E[a], add_u16x2(oth, O[a]));
                }
            }
            if constexpr (KS == ES - 1) {
                // record word m: register RPW m + i at bits FW i (frame 0)
                // and 16 + FW i (frame 1).  Two forms, alternating by word
                // so that the ALU and FMA pipes stay balanced (measured:
                // either form alone is slower):
                //  * byte permutes: the low byte of each half holds a
                //    register's field (and metric bits above it, which
                //    the traceback masks off); prmt(P[a], P[b], 0x6240)
                //    puts a's low bytes at bits 0 and 16 and b's at 8 and
                //    24, a multiply-add shifts a second such word by one
                //    field and a select merges them; the fields are then
                //    cleared by selects (ALU);
                //  * extracted fields: d = P & FM (ALU), cleared by a
                //    multiply-add P - d and gathered by multiply-adds
                //    acc = 16 acc + d (FMA pipe).
                auto merge = [](uint32_t a, uint32_t b, uint32_t keep_a) { return (a & keep_a) | (b & ~keep_a); };
                if constexpr (S == U - 1) {
                    // the smallest metric of the states of the shift (fields masked off)
                    uint32_t q[Cfg::NMIN];
#pragma unroll
                    for (int r = 0; r < Cfg::NMIN; ++r) q[r] = P[r];
                    pmin = min_tree<Cfg::NMIN>(q) & ~FM;
                    if constexpr (L > 1) pmin = __shfl_sync(gmask, pmin, grp_base);
                }
                uint32_t rec[NW];
#pragma unroll
                for (int m = 0; m < NW; ++m) {
                    const int r0 = RPW * m;
                    if constexpr (RPW == 4) {
                        if (m & 1) {
                            uint32_t acc = 0;
#pragma unroll
                            for (int i = RPW - 1; i >= 0; --i) {
                                const int r = r0 + i;
                                const uint32_t d = P[r] & FM;
                                P[r] = imad(d, m1, P[r]);
                                acc = (i == RPW - 1) ? d : imad(acc, fwmul, d);
                            }
                            rec[m] = acc;
                        } else {
                            const uint32_t x = prmt(P[r0], P[r0 + 2], 0x6240u);
                            const uint32_t y = prmt(P[r0 + 1], P[r0 + 3], 0x6240u);
                            rec[m] = merge(x, imad(y, fwmul, 0u), 0x07070707u);
#pragma unroll
                            for (int i = 0; i < RPW; ++i) P[r0 + i] &= ~FM;
                        }
                    } else if (K >= 9 && (m & 1)) {
                        // 2-bit fields, extracted (K=9 only: the two forms
                        // alternating were measured 4.5% faster for the K=9
                        // stream kernel and 1.6% slower for K=7 radix-4,
                        // whose records are rarer per instruction)
                        static_assert(RPW == 8, "2-bit or 4-bit record fields");
                        uint32_t acc = 0;
#pragma unroll
                        for (int i = RPW - 1; i >= 0; --i) {
                            const int r = r0 + i;
                            const uint32_t d = P[r] & FM;
                            P[r] = imad(d, m1, P[r]);
                            acc = (i == RPW - 1) ? d : imad(acc, fwmul, d);
                        }
                        rec[m] = acc;
                    } else {
                        // 2-bit fields: registers r0 + i, r0 + i + 4 shifted by 2 i bits
                        static_assert(RPW == 8, "2-bit or 4-bit record fields");
                        const uint32_t x0 = prmt(P[r0], P[r0 + 4], 0x6240u);
                        const uint32_t x1 = imad(prmt(P[r0 + 1], P[r0 + 5], 0x6240u), fwmul, 0u);
                        const uint32_t x2 = imad(prmt(P[r0 + 2], P[r0 + 6], 0x6240u), mul16, 0u);
                        const uint32_t x3 = imad(prmt(P[r0 + 3], P[r0 + 7], 0x6240u), mul64, 0u);
                        rec[m] = merge(merge(x0, x1, 0x03030303u), merge(x2, x3, 0x30303030u), 0x0F0F0F0Fu);
#pragma unroll
                        for (int i = 0; i < RPW; ++i) P[r0 + i] &= ~FM;
                    }
                }
                if (tau >= tau_store) store_rec(tau, rec);
            }
            hook(Sc, c);
        });
    };
    // The condition is the same for all lanes of a group, and so is the copy that they take: both
    // copies shuffle over gmask, which is defined only if the group's lanes run the same one.
    // (Groups of a warp may differ; no vote over them, since no set of lanes is known to be
    // together here: their chunk counts differ.)
    const int rc0 = reset_at0 >= 0 ? reset_at0 / U : -1, rc1 = reset_at1 >= 0 ? reset_at1 / U : -1;
    for (int c = 0; c < nchunks; ++c) {
        if (HEADSTART_COPY && (c == rc0 || c == rc1)) chunk(std::true_type{}, c);
        else chunk(std::false_type{}, c);
    }

    // ------------------------------------------------- traceback start state
    // After Wpad stages (a multiple of K-1) register R holds state R again.
    // A frame that starts from the reset state and has fewer than K-1
    // stages can only be in a state whose low K-1-W bits are zero (the
    // others are -infinity for Algorithm 1 with a known start); the finite
    // head start does not keep every such state below them, so they are
    // left out of the argmax explicitly.
    uint32_t R[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t unreach = (known[h] && W[h] < NB) ? ((1u << (NB - (int)W[h])) - 1u) : 0u;
        uint32_t best = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const uint32_t v = h ? (P[r] >> 16) : (P[r] & 0xFFFFu);
            const uint32_t Rg = ((uint32_t)lane << LR) | (uint32_t)r;
            const uint32_t key = (v << 16) | (0xFFFFu - Rg);
            best = best > key ? best : key;
        }
        if (__builtin_expect(unreach != 0u, 0)) {
            best = 0;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const uint32_t v = h ? (P[r] >> 16) : (P[r] & 0xFFFFu);
                const uint32_t Rg = ((uint32_t)lane << LR) | (uint32_t)r;
                const uint32_t key = (Rg & unreach) ? 0u : ((v << 16) | (0xFFFFu - Rg));
                best = best > key ? best : key;
            }
        }
        if constexpr (L > 1) {
#pragma unroll
            for (int m = 1; m < L; m <<= 1) {
                const uint32_t o = __shfl_xor_sync(gmask, best, m);
                best = best > o ? best : o;
            }
        }
        R[h] = term[h] ? 0u : (0xFFFFu - (best & 0xFFFFu));
    }

    // optional canonical final metrics (lambda - min lambda), for parity checks
    if (ft[0].pm || ft[1].pm) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t mn = 0xFFFFu;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const uint32_t v = h ? (P[r] >> 16) : (P[r] & 0xFFFFu);
                mn = mn < v ? mn : v;
            }
            if constexpr (L > 1) {
#pragma unroll
                for (int m = 1; m < L; m <<= 1) {
                    const uint32_t o = __shfl_xor_sync(gmask, mn, m);
                    mn = mn < o ? mn : o;
                }
            }
            if (ft[h].pm) {
                int32_t *dst = ft[h].pm + ((int64_t)lane << LR);
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const uint32_t v = h ? (P[r] >> 16) : (P[r] & 0xFFFFu);
                    dst[r] = ((int32_t)v - (int32_t)mn) / Cfg::SC;
                }
            }
        }
    }

    tb.R[0] = R[0];
    tb.R[1] = R[1];
    tb.t0 = Wpad - 1;
    return true;
}

// Shared memory of the one-wave kernel (dynamic): per warp the staging of its
// traceback, then a traceback record per thread.  Its traceback has the SM
// to itself, so its time is the latency of the copies over the pairs in flight (DEEP): two
// where a pair of groups takes 6 KB a warp or more (three would leave the loads of received
// values 28 KB of L1), three otherwise.  Where a pair takes 8 KB a warp (K=7 radix 2 with one
// lane, K=9 with four) that leaves two blocks an SM.  Launches of more blocks than those hold at
// once take the shallow form there: one pair in flight, and registers for three blocks (us, deep /
// shallow: K=7 with one lane, 22 M bits 243 / 213, 26 M 244 / 216; K=9 with four, 10 M bits 538 / 441, 14.5 M
// 606 / 476).
template <int K, int BETA, uint64_t GENS, int L, bool RADIX4, int NT, bool DEEP>
struct StreamSmem {
    using Cfg = StreamCfg<K, BETA, GENS, L, RADIX4>;
    static constexpr size_t PAIR_BYTES = Traceback<K, L, RADIX4, Cfg::NR, Cfg::NW, Cfg::ES>::STAGE_WORDS * 4u;
    static constexpr int D = !DEEP ? 1 : PAIR_BYTES >= 6144 ? 2 : 3;
    static constexpr bool HAS_SHALLOW = PAIR_BYTES >= 8192;
    using Tb = Traceback<K, L, RADIX4, Cfg::NR, Cfg::NW, Cfg::ES, D>;
    static constexpr size_t STG_BYTES = (size_t)(NT / 32) * Tb::STAGE_WORDS * 4u;
    static constexpr size_t BYTES = STG_BYTES + (size_t)NT * sizeof(TbState);
    static_assert(STG_BYTES % 16 == 0, "records follow the staging at a 16-byte boundary");
};

// Segmented decode of one stream: frame pair q = (2q, 2q+1) per group of L lanes.
template <int K, int BETA, uint64_t GENS, int L, bool RADIX4, int NT, bool DEEP>
__global__ void __launch_bounds__(NT, DEEP ? 0 : 3) stream_kernel(const StreamParams p) {
    constexpr int NS = 1 << (K - 1);
    using Cfg = StreamCfg<K, BETA, GENS, L, RADIX4>;
    using Sm = StreamSmem<K, BETA, GENS, L, RADIX4, NT, DEEP>;
    using Tb = typename Sm::Tb;
    extern __shared__ __align__(16) uint4 vd_dyn_smem[];
    auto stg = reinterpret_cast<uint32_t (*)[Tb::STAGE_WORDS]>(vd_dyn_smem);
    TbState *tbs = reinterpret_cast<TbState *>(reinterpret_cast<unsigned char *>(vd_dyn_smem) + Sm::STG_BYTES);
    const int64_t gtid = (int64_t)blockIdx.x * NT + threadIdx.x;
    const int64_t q = gtid / L;
    const int lane = (int)(gtid % L);
    if (q >= p.n_pairs) return;   // whole lane groups leave together
    const int wlane = (int)(threadIdx.x & 31u);
    const unsigned gmask = (L == 32) ? 0xFFFFFFFFu : (((1u << L) - 1u) << (wlane & ~(L - 1)));
    const int grp_base = wlane & ~(L - 1);
    FrameTask ft[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t s = 2 * q + h;
        ft[h] = frame_task(p.llr, p.out, p.pm_out ? p.pm_out + s * NS : nullptr, s, p.n_win,
                           p.n_info, p.T, p.f, p.v, p.flags);
    }
    uint32_t *surv = p.surv + (size_t)(gtid >> 5) * (size_t)p.wpad_max * 32u * (size_t)Cfg::SW;
    TbState &st = tbs[threadIdx.x];
    forward_pair<K, BETA, GENS, L, RADIX4>(ft, surv, p.wpad_max, wlane, lane, gmask, grp_base, p.status,
                                           st, [](auto, int) {});
    uint32_t *my_stg = stg[threadIdx.x >> 5];
    if (Tb::active(st)) {
        Tb::begin(st, my_stg, wlane);
        Tb::drain(st, my_stg, wlane, lane, gmask, grp_base);
    }
}

}  // namespace vd
