// Dispatch rules: which kernel a call takes and how its work is cut.  Plain C++ without a CUDA header, so that the rules can
// be asked without a device; what depends on one (multiprocessors, clusters that it can place) comes in as arguments.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace fq {

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

inline int log2_ceil(int v) {
    int r = 0;
    while ((1 << r) < v) ++r;
    return r;
}

constexpr int kMaxCluster = 8;         // CTAs of a cluster, at most (the portable limit)
constexpr int kTileN = 128;            // output channels per MMA

// `held(ctas)` below: clusters of 2, 4 or 8 CTAs, one per SM, that the device can hold at a time (0: such a launch is refused).

// ---- short batches in one launch (linear_fused.cu) -------------------------------------------------------------------
constexpr int kFusedMaxTokens = 64;
constexpr int kFusedRun = 16;          // channels per thread and round

struct FusedPlan {
    int lanes = 0, rounds = 0, ctas_shift = 0, unit = 0, units = 0, slice = 0, grid = 0;   // lanes = 0: not for this shape
    uint32_t off_part = 0, off_codes = 0, off_g = 0;
    size_t smem = 0;
};

// At most 64 tokens, in one wave of CTAs.  One launch minus two, us per call (bf16, 4 / 8 bits, weights from memory): in a chain
// of graph nodes, of calls made eagerly (bound by the host, which one launch saves), and in a graph behind a kernel that triggers
// nothing, where the launch's start does not hide:
//                                  chain          eager          behind another kernel
//   K x N = 1024 x 1024   M = 8    -0.2 / +0.2    -1.1 / -1.1    +1.4 / +1.5
//                         M = 16   -0.8 / -0.2    -1.0 / -0.6    +0.7 / +1.1
//                         M = 24   -0.9 / -1.2    -1.3 / -1.6    -0.3 / -0.1
//                         M = 50   -0.2 / -0.4    -0.3 / -0.7    -0.2 / +0.3
//   2048 x 1024           M = 24   -1.2 / -2.3    -1.6 / -2.5    -1.2 / -1.6
//                         M = 50   -0.3 / -0.3    -0.9 / -1.1    -0.4 / +0.5
//   4096 x 1024           M = 24   -1.2 / -1.6    -1.8 / -2.3    -1.4 / -0.6
//   1024 x 4096 (128 CTAs) M = 17  -0.1 / -0.4    -0.3 / -0.5    -0.3 / +0.1;   x 4736 (148) +0.2 / -0.1, -0.4 / -0.7, +1.1 / +1.2
//   512 x 1024 (32)       M = 50   -0.1 / -0.2    -0.5 / -0.7    +0.2 / +0.8;   x 2048 (64) +0.3 / +0.4, +0.3 / +0.2, +0.2 / +0.8
//   1024 x 1280 (80)      M = 50   +0.4 / +0.2    +0.6 / +0.2    -0.1 / +0.4;   x 2304 (144) +1.1 / +0.9, +0.6 / +0.5, +1.5 / +2.0
//   256 x 1024            M = 50   +0.3 / +0.5    -0.2 / -0.4    +0.4 / +1.2
// So at most 128 CTAs, and of more than 32 tokens (whose transform every channel tile repeats over twice the CTAs) 64 CTAs, 12
// channel tiles and no rows below 384 channels.  With at most 8 tokens the largest grids are behind in a chain, too (8 bits, M = 1
// 4.5 / 4.0): 96 CTAs.  CTAs of two rounds share an SM with nobody and clusters of eight do not fill the chip, so that 128 of them
// would take two waves (K = 4096, N = 2048: 10.3 / 6.3): 96 as well.  Two launches where the device cannot place the clusters.
template <typename Held>
FusedPlan plan_fused(int64_t M, int64_t N, int64_t K, int block, int bits, bool mult, int sms, Held held) {
    FusedPlan f;
    if (M < 1 || M > kFusedMaxTokens || K % 128 != 0) return f;
    const int lanes = M <= 32 ? 16 : 8, round = lanes * kFusedRun;
    const int unit = block > 128 ? block : 128;
    if (K % unit != 0 || block > round || K > (int64_t)kMaxCluster * 2 * round) return f;
    const int units = (int)(K / unit), bt = (int)((M + 15) / 16 * 16);
    int shift = 0;
    auto slice = [&](int s) { return (units + (1 << s) - 1) / (1 << s) * unit; };
    while (shift < 3 && slice(shift) > round) ++shift;
    if (slice(shift) > 2 * round) return f;
    const int64_t grid = ((N + kTileN - 1) / kTileN) << shift;
    const bool two_rounds = slice(shift) > round;
    if (grid > sms || grid > (two_rounds || M <= 8 ? 96 : (M <= 32 ? 128 : 64))) return f;
    if (M > 32 && !two_rounds && (K < 384 || N > 12 * kTileN)) return f;
    if (shift > 0 && held(1 << shift) < 1) return f;
    f.ctas_shift = shift; f.unit = unit; f.units = units; f.slice = slice(shift); f.grid = (int)grid;
    f.rounds = f.slice > round ? 2 : 1;
    const size_t w_bytes = (size_t)kTileN * f.slice * bits / 8;
    const size_t part_bytes = (size_t)(1 << shift) * (1 << log2_ceil((int)((M + (1 << shift) - 1) >> shift))) * kTileN * 4;
    // the partial sums take the packed 4-bit weights' place (read by then in the whole cluster: the maxima were exchanged
    // behind the expansion); 8-bit weights are still being multiplied when another CTA's sums arrive
    const size_t head = bits == 4 ? (w_bytes > part_bytes ? w_bytes : part_bytes) : w_bytes + part_bytes;
    f.off_part = bits == 4 ? 0u : (uint32_t)w_bytes;
    f.off_codes = (uint32_t)align_up(head, 1024);
    f.off_g = (uint32_t)align_up(f.off_codes + (size_t)bt * f.slice, 1024);
    f.smem = f.off_g + (mult ? (size_t)f.slice / kFusedRun * (kFusedRun + 4) * 4 : 0) + 1024;
    // At most two CTAs per SM, whatever launches they belong to: a CTA holds up to half of tensor memory, and one that waited
    // for columns while its cluster waited for it must not be another cluster's reason to wait (launches of two streams).
    if (f.smem < 77 * 1024) f.smem = 77 * 1024;
    f.lanes = lanes;
    return f;
}

// ---- composite rotation and quantizer in one launch (composite.cu) ---------------------------------------------------
constexpr int kCompositeWarps = 8;
constexpr int kCompositeColumns = 16;  // columns of the matrices per step

struct CompositePlan {
    int tok = 0;                       // tokens per cluster: 16, or 8 where 16 rows do not fit; 0: rows too long, two launches
    int ctas_shift = 0, items = 0;     // log2 of the CTAs per cluster; work items (of 64 outputs, or a smaller block) per tile
    int u_pitch = 0, span = 0;
    uint32_t off_u = 0, off_b = 0, off_p = 0, off_s = 0;
    int64_t grid = 0;
    size_t smem = 0;
};

// As many CTAs per tile of tokens as leave half the warps an item each and make one wave: every CTA begins by staging the
// tokens' rows, so a second wave costs more than longer CTAs (block 64: M = 816, K = 2048 19.7 us with clusters of four in two
// waves, 15.4 with pairs in one; M = 1184, K = 1024 21.0 and 9.6).  Two CTAs share an SM where shared memory allows it
// (816 x 1024, block 32: 7.8 us so, 10.4 with pairs).  More CTAs where the rotated channels would not fit otherwise.
template <typename Held>
CompositePlan plan_composite(int64_t rows, int64_t K, int elem_bytes, int beta, int sms, Held held) {
    CompositePlan f;
    const int out = beta < 64 ? beta : 64;
    f.items = (int)K / out;
    for (int tok = 16; tok >= (beta >= 32 ? 8 : 16); tok /= 2) {
        const int64_t tiles = (rows + tok - 1) / tok;
        auto fits = [&](int shift) {
            const int width = ((f.items + (1 << shift) - 1) >> shift) * out;
            f.u_pitch = width + 4;
            f.span = width + (beta > out ? 2 * beta : 0);
            size_t at = align_up((size_t)K * elem_bytes * tok, 16);
            f.off_u = (uint32_t)at; at += align_up((size_t)f.u_pitch * 4 * tok, 16);
            f.off_b = (uint32_t)at; at += (size_t)kCompositeWarps * 2 * out * kCompositeColumns * 4;
            f.off_p = (uint32_t)at; at += (size_t)kCompositeWarps * kCompositeColumns * (tok + 4) * 4;
            f.off_s = (uint32_t)at; at += (size_t)f.span * 8;
            f.smem = at;
            return f.smem <= 224 * 1024;
        };
        auto placed = [&](int shift) { return shift == 0 ? (int64_t)sms : (int64_t)held(1 << shift) << shift; };   // CTAs at a time, one per SM
        auto one_wave = [&](int shift) {
            return fits(shift) && (tiles << shift) <= placed(shift) * (2 * (f.smem + 3072) <= 228 * 1024 ? 2 : 1);
        };
        int shift = 3;
        while (shift > 0 && (f.items >> shift < 4 || !one_wave(shift)) && fits(shift - 1)) --shift;
        if (!fits(shift) || f.items >> shift < 1 || (tiles << shift) > 0x7fffffffll || placed(shift) < 1) continue;
        f.tok = tok; f.ctas_shift = shift; f.grid = tiles << shift;
        return f;
    }
    return f;
}

// ---- streamed prologue (act_quant_ring.cu) instead of the register one -------------------------------------------------
constexpr int kRingThreads = 512;
constexpr int kRingMaxSlots = 128;

struct RingPlan {
    int e = 0;                         // channels per thread; 0: the register kernel
    int gw = 0, ngroups = 0, depth = 0;   // warps per row group, groups per CTA, ring slots per group
    size_t half = 0, slot = 0;         // bytes of a row in shared memory, and of a slot (two rows for gated sites)
    size_t g_bytes = 0, stage_bytes = 0;  // the multiplier's stage, the codes' stage
};

// bytes_out: one byte per code; mult: a per-channel multiplier, after: behind the rotation.
inline RingPlan plan_ring(int64_t rows, int64_t K, int elem_bytes, bool gated, bool bytes_out, bool mult, bool after, int block, int sms) {
    RingPlan f;
    const size_t row_bytes = (size_t)K * elem_bytes;
    // shape gate: whole 128-byte lines, at most 256 of them per box, blocks of 32..256 channels
    if (K < 1024 || row_bytes % 128 != 0 || row_bytes / 128 > 256 || rows > 0x7fffffffll || block < 32)
        return RingPlan();
    // Gated sites: from two rows per SM on, or long rows.  Prologue alone, GELU, 8-bit codes, operands from memory, here /
    // register kernel: M = 816, K = 2048 4.6 / 5.7 us, K = 8192 14.0 / 16.0, K = 16384 25.9 / 37.7 (66 before the paired
    // gate arithmetic); M = 148, K = 8192 4.1 / 3.9, K = 16384 7.0 / 8.5.
    if (gated && (elem_bytes != 2 || after || (rows < 2 * (int64_t)sms && K <= 8192)))
        return RingPlan();

    // Channels per thread: 64 where at least two rows per group fit (the fold-after variant with shuffle stages would spill)
    f.half = (row_bytes + 1023) / 1024 * 1024;
    f.slot = gated ? 2 * f.half : f.half;
    f.g_bytes = mult ? ((size_t)K * 4 + 1023) / 1024 * 1024 : 0;
    auto fits = [&](int channels) {
        f.e = channels;
        f.gw = 1;
        while ((int64_t)f.gw * 32 * f.e < K) f.gw <<= 1;
        f.ngroups = (kRingThreads / 32) / f.gw;
        if (f.ngroups < 1 || (f.gw > 1 && f.ngroups > 15)) return false;             // one named barrier per group
        f.stage_bytes = bytes_out && f.e == 64 ? (size_t)kRingThreads * f.e : 0;
        const size_t budget = 227 * 1024 - 2048 - 1024 - f.stage_bytes;
        if (f.g_bytes + 2 * f.slot * f.ngroups > budget) return false;
        f.depth = (int)((budget - f.g_bytes) / (f.slot * f.ngroups));
        if (f.depth > 4) f.depth = 4;
        return f.ngroups * f.depth <= kRingMaxSlots;
    };
    const bool may64 = !gated && K >= 2048 && K % 64 == 0 && !(after && block >= 128);
    if (!(may64 && fits(64)) && !fits(32)) return RingPlan();
    // Short batches are latency-bound and go to the register kernel, which spreads a row over more threads and leaves its SMs'
    // shared memory to the GEMM behind it, whose CTAs set up and fetch weights beside it.  The line is drawn by what whole
    // calls take, in channels per SM; it lies higher where a row leaves lanes of its group idle (with a multiplier such lanes'
    // warps still read it).  Streamed minus register, us per fq_linear call (N = 2048, 8 bits; rows and channels, in brackets
    // thousands of channels per SM), in a chain of calls / each behind a kernel that triggers nothing, where the streamed
    // kernel's longer start does not hide:
    //   bf16, all lanes  816 x 2048 (11) +0.43 / +1.28;  1156 x 2048 (16) +0.71 / +0.84, with a multiplier +0.35 / +0.40;  1300 x
    //                    2048 (18) -0.69 / +0.60, -0.49 / +0.13;  614 x 4096 (17) +0.54 / +0.62;  758 x 4096 (21) -0.46 / +0.48,
    //                    -0.36 / +0.25;  307 x 8192 (17) +0.12 / +0.46;  379 x 8192 (21) -1.01 / +0.19;  975 x 4096 (27) -0.73 /
    //                    -0.59;  1638 x 1536 (17) +0.76 / +1.56;  1734 x 1536 (18) -0.05 / +1.19;  81 x 16384 (9) -0.43 / -0.18,
    //                    with a multiplier -0.49 / -1.29
    //   seven eighths    825 x 3584 (20) -0.05 / +0.97;  1238 x 3584 (30) -0.41 / +0.21, 619 x 7168 (30) -1.60 / 0.00
    //   three quarters   1445 x 3072 (30) +0.57 / +0.70;  1927 x 3072 (40) -0.27 / +0.50;  2890 x 3072 (60) -0.57 / -0.04, with a
    //                    multiplier -0.02 / -0.34;  963 x 6144 (40) -0.88 / -0.08, with one -0.75 / +0.09
    //   less             1734 x 2560 (30) +1.25 / +1.24;  3468 x 2560 (60) +0.50 / +0.40;  4625 x 2560 (80) -0.84 / -0.34;  with a
    //                    multiplier 6359 x 2560 (110) +1.23 / -0.17, 9250 x 2560 (160) -0.66 / -1.81, 3179 x 5120 (110) +0.07 / +0.03
    //   ... past 8192    201 x 11008 (15) -0.22 / -0.02, with a multiplier -0.28 / -0.62;  1170 x 10240 with one -2.10 / -2.05
    //   binary32         614 x 2048 (8.5) -0.29 / +0.32, with a multiplier -0.32 / -0.08;  153 x 8192 -0.70 / -0.45;  1156 x 1536
    //                    (12) +0.22 / +0.68 (4 bits);  2167 x 1024 (15) -0.98 / +0.32;  1445 x 1536 (15) -0.33 / +0.91;  770 x 3072
    //                    (16) -0.85 / +0.81;  with a multiplier 3121 x 2560 (54) -0.02 / +0.18, 4682 x 2560 (81) -0.95 / -1.06
    // (Prologues alone in a chain of themselves, by which the line was drawn once, have the streamed one ahead from 9 on:
    // 816 x 2048 3.28 / 3.46 us; behind a kernel that triggers nothing it is 3.97 / 3.46.)
    if (!gated) {
        const int64_t width = (int64_t)f.gw * 32 * f.e;          // channels that the group's lanes could hold
        int64_t line;
        if (elem_bytes == 4) line = K < 2048 ? 13000 : (width == K ? 8000 : (mult && 4 * K < 3 * width ? 60000 : 15000));
        else if (K > 8192) line = width == K ? 8000 : 15000;
        else if (width == K || K < 2048) line = 18000;
        else if (8 * K >= 7 * width) line = 27000;
        else if (4 * K >= 3 * width) line = 45000;
        else line = mult ? 130000 : 80000;
        if (rows * K < line * sms) return RingPlan();
    }
    return f;
}

// ---- stacked tiles of the integer GEMM (gemm_tcgen05.cu) -----------------------------------------------------------------
// Short batches on 4-bit matrices of too few channels leave SMs idle, and a split of K over CTAs pays for the exchange of sums.
// A stacked tile splits K inside one MMA tile: its 128 rows are 64 channels at two slices of K, its columns the tokens at those
// two slices; every row is multiplied with all columns, and only its own slice's count.  Twice the CTAs, each with half the
// k-blocks, and the sums meet in the CTA.  Chains of calls, stacked / the best of the others, us:
//   M <= 32   24 x 3072 x 2048 (M x K x N) 6.5 / 7.2;  32 x 3072 x 6144 6.6 / 7.4;  32 x 4096 x 2048 7.0 / 8.2;  16 x 4096 x 8192
//             7.5 / 8.5;  32 x 4096 x 8192 8.0 / 8.3;  32 x 5120 x 4096 7.6 / 9.2;  32 x 6144 x 6144 8.5 / 10.5;  16 x 6144 x 8704
//             10.1 / 11.6;  16 x 8192 x 8192 11.5 / 13.6;  32 x 8192 x 9472 12.2 / 12.8;  16 x 16384 x 8192 16.0 / 17.4
//   behind    fewer channels, where clusters split K: 32 x 5120 x 2048 7.5 / 6.9, 32 x 8192 x 4096 9.7 / 8.9;  a short K: 32 x 2048
//             x 8192 6.7 / 6.6;  a launch on all SMs, which leaves none to the next one: 16 x 4096 x 9472 8.9 / 8.1
//   M <= 48   3072 x 4096 7.1 / 7.7, 4096 x 6144 8.1 / 9.0, 6144 x 6144 9.5 / 11.2;  behind 4096 x 2048 7.8 / 7.4, 6144 x 4096 9.3 / 8.8
//   M <= 64   3072 x 4096 7.5 / 8.0, 4096 x 4096 8.2 / 9.1, 4096 x 6144 8.6 / 9.1;  behind 5120 x 4096 9.1 / 8.8, 6144 x 6144 10.7 / 10.0
// (Four slices of 32 channels, 8-bit weights, whose operands pass through shared memory twice then, and longer batches are behind.)
// (One tile of tokens and at most 64 x SMs channels: a CTA has one tile.)
constexpr int kStackSlices = 2;
inline bool stacked_applies(int64_t M, int64_t N, int64_t K, int bits, int sms) {
    if (bits != 4 || M < 1 || M > 64 || K % 256 != 0 || K < 3072) return false;
    if (M <= 32) {
        const int64_t least = K <= 4096 ? 2048 : (2 * K / 3 < 5120 ? 2 * K / 3 : 5120);
        return N >= least && N <= 64ll * (K >= 8192 ? sms : sms - 12);
    }
    return K <= (M <= 48 ? 6144 : 4096) && 4 * N >= 3 * K && N <= 7168 && N <= 64ll * (sms - 12);
}

// ---- integer GEMM (gemm_tcgen05.cu) ------------------------------------------------------------------------------------
constexpr int kBlockK = 128;           // int8 elements (= bytes) of K per pipeline stage
constexpr int kAccStages = 2;
constexpr int kUnpackSets = 2;         // sets of four unpack warps, one TMEM lane quadrant each
constexpr int kMaxStages = 16;         // ring slots, at most: activations, packed weights, unpacked weights
constexpr int kMaxStagesP = 16;
constexpr int kMaxStagesW = 8;
constexpr int kColsW = kBlockK / 4;    // TMEM columns of one unpacked k-block (128 int8 per lane)
constexpr int kEpiWarps = 8, kEpiWarpsMany = 16;         // epilogue warps (see epi_warps)
constexpr int kEpiBuffers = 2;                          // output buffers per epilogue warp (bulk stores in flight; four measured no faster)
constexpr int kEpiStageBytes = kEpiBuffers * 16 * 64;   // per epilogue warp: buffers of 16 tokens x 32 channels of bf16
constexpr int kMaxSplit = 16;          // K slices per tile, at most
constexpr int kMaxSplitTiles = 1024;   // tiles of a launch that splits K (one counter each, ahead of the partial sums)
constexpr size_t kCounterBytes = kMaxSplitTiles * sizeof(uint32_t);

struct GemmPlan {
    int bt = 0;       // tokens per tile
    int ctas = 1;     // 2: CTA pairs on 256-channel tiles (cta_group::2)
    int split = 1;    // >1: every tile is that many work units, each on a slice of K
    bool cluster = false; // the slices of a tile are the CTAs of a cluster (no scratch)
    int epi = kEpiWarps;  // epilogue warps
    int stack = 1;        // 2: a stacked tile, 64 channels at two slices of K (see stacked_applies); bt counts its columns
    size_t scratch = 0;   // bytes of scratch the split needs: the tile counters, then the int32 partial tiles
};
inline GemmPlan cluster_plan(int bt, int ctas, int split) {
    GemmPlan plan;
    plan.bt = bt; plan.ctas = ctas; plan.split = split; plan.cluster = true;
    return plan;
}

// Atoms (of 128 channels) per pipeline stage.  4-bit weights, single CTAs: two for token tiles of at most 128, four for the
// shortest (the accumulators of longer tiles leave no room for wider TMEM slots); whole atoms, slices of whole stages.
inline int atoms_per_stage(int bits, int ctas, int bt, int64_t K, int split) {
    const int64_t kb = (K + kBlockK - 1) / kBlockK;
    if (bits != 4 || ctas != 1 || bt > 128 || K % kBlockK != 0) return 1;
    if (bt <= 64 && kb >= 4 * split && (split == 1 || kb % (4 * split) == 0)) return 4;
    return split == 1 || kb % (2 * split) == 0 ? 2 : 1;
}
// Shared memory of the pipeline rings; `sums`: bytes taken by the sums of a cluster split.
// Bytes of an epilogue warp's output buffers (8-bit launches that split K have one: the ring is worth more).
inline int epi_stage_bytes(int bits, bool split) { return bits == 8 && split ? kEpiStageBytes / kEpiBuffers : kEpiStageBytes; }
inline size_t ring_budget(int epi, int bits, bool split, size_t sums) {
    return 227 * 1024 - 1024 /*alignment slack*/ - 1024 /*static*/ - (size_t)epi * epi_stage_bytes(bits, split) - sums;
}
inline size_t stage_bytes(int bits, int ctas, int bt, int atoms) {
    return ((size_t)(bt / ctas) * kBlockK + (size_t)kTileN * kBlockK * bits / 8) * atoms;
}
// Epilogue warps.  The last tile of a launch has nothing to hide its epilogue behind, a chain of TMEM load, arithmetic and store per
// 16 tokens, some 500 cycles each; twice the warps halve it.  They also take registers that the next call's prologue could start on
// (608 threads x 96 instead of 352 x 128), issue slots from the main loop, and 16 KB from the ring.  Unsplit 8-bit launches, sixteen /
// eight, chains of calls, M x K x N, us (at 4 bits the unpack warps leave no registers for them; with K split a CTA finishes its
// share only: 64 x 8192 x 8192 17.0 / 16.5, 400 x 16384 x 2048 29.0 / 25.9, 816 x 16384 x 2048 35.7 / 35.2):
//   single CTAs, one round: 512 x 4096 x 4096 (128-token tiles) 14.8 / 15.2, 400 x 4096 x 4096 (112) 14.4 / 14.8; with fewer tokens ahead on
//     short rows only (256 x 1024 x 4096 7.5 / 7.7; 816 x 4096 x 2048 (96) 14.9 / 14.8, 269 x 3072 x 3968 (80) 12.0 / 11.5, 128 x 4096 x
//     9472 (64) 13.5 / 12.4); more rounds: 783 x 1408 x 6368 (160) 13.95 / 14.6, 300 x 256 x 16384 (160) 9.4 / 10.2, 100 x 1024 x 30000
//     (112) 11.5 / 11.6, 600 x 1536 x 8192 (160) 14.2 / 14.3; 1200 x 2048 x 4104 (160) 18.1 / 17.0, 100 x 2048 x 30000 (112) 17.3 / 16.7,
//     64 x 1024 x 20000 9.7 / 9.3
//   pairs, one round: 1000 x 4096 x 4104 20.1 / 21.5, 208 x 2048 x 16384 13.7 / 14.7
//     more: ahead on short rows, whose every tile is mostly epilogue (16384 x 1024 x 4096 80 / 103, 816 x 1024 x 16384 19.5 / 22.1), and
//     up to 2048 channels or two rounds (16384 x 2048 x 2048 72.6 / 75.9, 2000 x 4096 x 4104 31.6 / 32.2) unless the ring loses a stage
//     by them (816 x 2048 x 32768 49.3 / 46.5, 7312 x 8960 x 792 106 / 104); else no faster (4096 x 4096 x 4096 59 / 59)
inline int epi_warps(int bits, int ctas, int bt, int64_t K, int64_t rounds, int split) {
    if (bits == 4 || split > 1) return kEpiWarps;
    if (rounds == 1 ? (ctas == 2 || bt >= 112 || K <= 1024) : (ctas == 2 ? K <= 1024 : bt >= 112 && K <= 1536)) return kEpiWarpsMany;
    const size_t stage = stage_bytes(bits, ctas, bt, 1);
    return ctas == 2 && (rounds == 2 || (rounds > 2 && K <= 2048)) &&
                   ring_budget(kEpiWarps, bits, false, 0) / stage == ring_budget(kEpiWarpsMany, bits, false, 0) / stage
               ? kEpiWarpsMany : kEpiWarps;
}
inline size_t cluster_sums_bytes(int bt, int split) { return (size_t)(split - 1) * ((bt / 16 + split - 1) / split) * 16 * kTileN * sizeof(int32_t); }

inline size_t stacked_sums_bytes(int tok) { return (size_t)((tok / 16 + 1) / 2) * 16 * kTileN * sizeof(int32_t); }
// Bytes of the ring's memory that a CTA of a cluster split stages the sums in which it sends: the n-th chunk that a warp sends lies at
// [n][warp], and a warp sends every (warps / 4)-th chunk of 16 tokens but those that its own slice finishes.
constexpr int kSumBytes = 16 * 32 * 4;                   // a warp's sums of one token chunk
inline size_t staged_sums_bytes(int warps, int bt, int split) {
    const int sets = warps / 4;
    int top = 0;
    for (int slice = 0; slice < split; ++slice)
        for (int set = 0; set < sets; ++set) {
            int sent = 0;
            for (int c = set; c < bt / 16; c += sets) sent += (c & (split - 1)) != slice;
            if (sent > 0 && (sent - 1) * warps + 4 * (set + 1) > top) top = (sent - 1) * warps + 4 * (set + 1);
        }
    return (size_t)top * kSumBytes;
}

// The rings of a plan: slots of activations (and int8 weights, in lockstep), of packed and of unpacked 4-bit weights.
struct GemmRings {
    bool fits = false;
    int atoms = 1, stages = 0, stages_p = 0, stages_w = 0, tmem_cols = 0;
    bool slot_first = false;           // the unpack sets wait for the TMEM slot ahead of the packed stage (see the kernel)
    size_t smem = 0;
};
inline GemmRings gemm_rings(const GemmPlan& plan, int bits, int64_t K) {
    GemmRings f;
    const int bt = plan.bt;
    const bool split = plan.split > 1 || plan.stack > 1;
    f.atoms = atoms_per_stage(bits, plan.ctas, bt, K / plan.stack, plan.split);
    const size_t sums = plan.cluster ? cluster_sums_bytes(bt, plan.split) : (plan.stack > 1 ? stacked_sums_bytes(bt / plan.stack) : 0), budget = ring_budget(plan.epi, bits, split, sums);
    const size_t epi_bytes = (size_t)plan.epi * epi_stage_bytes(bits, split) + sums;
    const size_t a_bytes = (size_t)(bt / plan.ctas) * kBlockK * f.atoms, w_bytes = (size_t)kTileN * kBlockK, pk_bytes = w_bytes / 2 * f.atoms;
    // 4-bit weights: every TMEM column the accumulators leave free becomes unpacked-weight ring
    f.stages_w = bits == 4 ? (512 - kAccStages * bt) / (kColsW * f.atoms) : 0;
    if (f.stages_w > kMaxStagesW) f.stages_w = kMaxStagesW;
    for (f.tmem_cols = 32; f.tmem_cols < kAccStages * bt + f.stages_w * kColsW * f.atoms;) f.tmem_cols <<= 1;
    if (bits == 4) {
        // Both TMA rings need the same look-ahead in k-blocks (their latencies are the same): split the budget evenly, then
        // give the remainder to the cheaper packed ring.
        f.stages = (int)(budget / (a_bytes + pk_bytes));
        if (f.stages > kMaxStages) f.stages = kMaxStages;
        if (f.stages < 2) return f;
        f.stages_p = (int)((budget - f.stages * a_bytes) / pk_bytes);
        if (f.stages_p > kMaxStagesP) f.stages_p = kMaxStagesP;
        if (f.stages_w > f.stages) f.stages_w = f.stages;       // the unpack warps wait on the activation ring's barriers
        // (a ring one shorter is slower, one TMEM slot less no faster: 128 x 4096 x 4096 10.5, 11.3 and 10.4 us, 256 x 2048 x
        // 4096 9.95, 10.1 and 9.9)
        f.slot_first = f.stages_p % kUnpackSets != 0 && f.stages_p < f.stages_w + kUnpackSets;
        if (f.slot_first && f.stages_w > f.stages_p) return f;
        f.smem = f.stages * a_bytes + f.stages_p * pk_bytes + epi_bytes + 1024;
    } else {
        f.stages = (int)(budget / (a_bytes + w_bytes));
        if (f.stages > kMaxStages) f.stages = kMaxStages;
        if (f.stages < 2) return f;
        f.smem = (a_bytes + w_bytes) * f.stages + epi_bytes + 1024;
    }
    // (mostly there is room for every chunk of the tile: no need to count those that are sent)
    const size_t ring = f.smem - epi_bytes - 1024;
    if (plan.cluster && (size_t)(bt / 16 + 3) * 4 * kSumBytes > ring && staged_sums_bytes(plan.epi, bt, plan.split) > ring) return f;
    // One CTA of this kind per SM, and none of the short-batch kernel beside it: a cluster whose CTA waited for tensor memory
    // must not be what another cluster on that SM waits for (launches of two streams).
    if (plan.cluster && f.smem < 152 * 1024) f.smem = 152 * 1024;
    f.fits = true;
    return f;
}

// Token tile, CTA grouping and K split.  Upper bound of the tile from TMEM: two accumulator stages,
// plus the unpacked-weight ring for 4-bit weights (2*bt + 3*32 <= 512 columns).  M is split evenly
// over m_tiles so that ragged M wastes little.  Candidates are ranked by a cost model fitted to
// measured launches (cycles): rounds of work units over the SMs, each unit costing
//     k_blocks * per_kblock(bt) + 16*bt + 1000          (the tail: epilogue and tile hand-over)
//   4-bit weights:          per_kblock = 330 + bt       (issue floor, then the MMAs' 2*bt); 235 + bt for tiles of at
//                                        most 128 tokens, whose stages hold two or four k-blocks
//   8-bit, one CTA:         per_kblock = max(350 + 0.8*bt, 230 + 2*bt)   (issue floor, then shared memory:
//                                        both operands pass through it)
//   8-bit, CTA pair:        per_kblock = max(545, 2.62*bt)   (each CTA stages half of the token tile)
//   4-bit, CTA pair:        0.95 of a single CTA's, for launches of 1.6e11 multiplications and K >= 2048.  Each CTA stages
//                           half of the token tile, so shared memory is read half as often: no faster while the clock is
//                           at its highest, but less power, hence a higher clock under the power cap.  Chains of calls,
//                           pairs / single CTAs, the clock still high and after 0.2 s of load: 16384 x 8192 x 8192
//                           (M x K x N) 773 / 804 us and 905 / 922, 16384 x 4096 x 4096 222 / 226 and 262 / 268,
//                           4096 x 8192 x 8192 199 / 200 and 235 / 238, 12000 x 2048 x 8192 158 / 163 and 189 / 194; below
//                           the line 7000 x 4096 x 4096 103 / 100 and 117 / 119, 4096 x 4096 x 4096 67.2 / 64.9 and 73.0 /
//                           73.3; a short K: 16384 x 1024 x 4096 96 / 97 and 105 / 104.
// (A plan takes the host 0.1 to 3 us; asking for the clusters of every candidate first took up to 30.)
// K split: problems with fewer tiles than SMs and a long K (short batches, few output channels).
//   By clusters of 2, 4 or 8 CTAs (one wave; at least four k-blocks of ring beside the sums and two output buffers per warp -- with
//   one, as 8-bit splits have, pairs of long tiles come in that are behind: 644 x 3584 x 1280 (M x K x N) 13.8 / 12.4 us,
//   203 x 11264 x 3008 20.0 / 19.4 --, 4-bit tiles of at most 128 tokens): the tail shrinks to 16*bt/split, the exchange costs 2800 + 40 per CTA of the launch at 4 bits, 3300 + 18 at 8
//   (the more SMs a launch takes, the less of the next one starts beside it), and 500 per extra slice.  Measured, chains of
//   calls, split against the best unsplit tile: 64 x 16384 x 2048 (M x K x N) 12.8 / 22.1 us at 4 bits and 14.1 / 31.3 at 8;
//   16 x 16384 x 4096 12.8 / 21.6 and 16.2 / 30.1; 64 x 4096 x 1024 7.5 / 8.9 and 7.5 / 10.8; 64 x 4096 x 4096 8.75 / 11.0
//   at 8 bits; 128 x 4096 x 1024 9.2 / 9.7 and 7.9 / 11.3; 256 x 4096 x 1024 9.9 / 9.7 and 9.9 / 11.5; CTA pairs,
//   816 x 16384 x 2048 34.9 / 39.3.
//   Through scratch, where the device cannot hold the clusters, their sums leave too little ring, or 4-bit tiles have more than
//   128 tokens (CTA pairs on 8-bit weights, too; on a whole B200 rows of 20480 channels and more): 12500 + 40*bt + 1500 per extra slice.
template <typename Held>
GemmPlan plan_gemm(int64_t M, int64_t N, int64_t K, int bits, int sms, size_t scratch_avail, bool clusters, Held held) {
    const int bt_max = bits == 4 ? 208 : 256;
    const int64_t kb = (K + kBlockK - 1) / kBlockK;
    GemmPlan best;
    double best_cost = 0.0;
    int64_t best_rounds = 0;
    int capacity[kMaxCluster + 1] = {};                  // by CTAs per cluster, asked for once per plan; 0: not yet, else + 1
    auto holds = [&](int ctas) {
        if (capacity[ctas] == 0) capacity[ctas] = held(ctas) + 1;
        return capacity[ctas] - 1;
    };
    const bool pairs = N > kTileN && (bits == 8 || (K >= 2048 && (double)M * (double)N * (double)K >= 1.6e11));
    for (int c = 1; c <= (pairs ? 2 : 1); ++c) {
        if (c == 2 && clusters && holds(2) < 1) break;
        const int64_t n_units = (N + kTileN * c - 1) / (kTileN * c);
        for (int mt = (int)((M + bt_max - 1) / bt_max); mt <= (int)((M + 63) / 64); ++mt) {
            const int b = (int)(((M + mt - 1) / mt + 15) / 16 * 16);
            if (b > bt_max) continue;
            const int64_t units = n_units * ((M + b - 1) / b);
            const double w8_single = 350.0 + 0.8 * b > 230.0 + 2.0 * b ? 350.0 + 0.8 * b : 230.0 + 2.0 * b;
            // 4-bit, tiles of at most 128 tokens: stages of several atoms (see the kernel) cost less per 128 channels
            const double w4 = c == 2 ? 0.95 * (330.0 + b) : (b <= 128 && K % kBlockK == 0 ? 235.0 + b : 330.0 + b);
            const double per_kb = bits == 4 ? w4 : (c == 1 ? w8_single : (2.62 * b > 545.0 ? 2.62 * b : 545.0));
            const int slots = sms / c;
            auto offer = [&](int sp, bool cluster, size_t scratch, double unit_cost) {
                const int64_t rounds = (units * sp + slots - 1) / slots;
                const double cost = (double)rounds * unit_cost;
                // ties: the earlier candidate (larger tile, no split)
                if (best.bt == 0 || (cost < best_cost * 0.98 && (!cluster || gemm_rings(cluster_plan(b, c, sp), bits, K).fits))) {
                    best.bt = b; best.ctas = c; best.split = sp; best.cluster = cluster; best.scratch = scratch;
                    best_rounds = rounds;
                    best_cost = cost;
                }
            };
            offer(1, false, 0, (double)kb * per_kb + 16.0 * b + 1000.0);
            if (bits == 4 && c == 2) continue;           // (long launches have tiles enough: no kernel for a split of these)
            if (units * 2 > slots && units * c * 2 > 4 * (int64_t)sms) continue;       // too many tiles for any split
            for (int sp = 2; sp <= kMaxSplit; sp *= 2) {
                if (kb % sp != 0 || kb / sp < 2) break;
                const double slice = (double)(kb / sp) * per_kb + 1000.0;
                const int atoms = atoms_per_stage(bits, c, b, K, sp);
                const double ctas = (double)(units * sp * c);
                if (clusters && (bits == 8 || b <= 128) && sp * c <= kMaxCluster && units * sp <= slots &&
                    ring_budget(kEpiWarps, bits, false, cluster_sums_bytes(b, sp)) * atoms >= 4 * stage_bytes(bits, c, b, atoms) && units <= holds(sp * c))
                    offer(sp, true, 0, slice + 16.0 * b / sp + (bits == 4 ? 2800.0 + 40.0 * ctas : 3300.0 + 18.0 * ctas) + 500.0 * (sp - 1));
                if ((c == 1 || bits == 8) && units * c <= kMaxSplitTiles && units * c * sp <= 4 * (int64_t)sms) {
                    const size_t scratch = kCounterBytes + (size_t)units * c * sp * kTileN * b * sizeof(int32_t);
                    if (scratch <= scratch_avail) offer(sp, false, scratch, slice + 16.0 * b + 12500.0 + 40.0 * b + 1500.0 * (sp - 1));
                }
            }
        }
    }
    if (best.bt != 0) best.epi = epi_warps(bits, best.ctas, best.bt, K, best_rounds, best.split);
    return best;
}

// ---- integer product of short batches: the weight-streaming kernel (linear_wonly.cu) instead of the tcgen05 one ----------
// (Rows of whole 128-byte lines only.)  Chains of calls, operands from memory, stream / the other kernel, M x K x N, us.
// One round of row groups over the SMs (N <= 32 x SMs): ahead (16 x 4096 x 4096 7.0 / 9.7), up to 64 Mi weights.  8-bit weights:
// 16 x 8192 x 4096 10.4 / 10.3 in a chain, and 0.55 us ahead between unrelated calls; 16 x 4096 x 8192, two rounds, 14.0 / 11.5.
//   Long rows: behind a split of K into four or more slices by clusters -- where the plan has one: 16 x 16384 x 4096 15.2 / 12.6 at 4 bits
//   and 18.5 / 16.9 at 8, 16 x 10240 x 2048 10.0 / 9.4 and 10.9 / 10.9, 16 x 10752 x 2048 at 8 bits 11.4 / 11.0.  Ahead of everything
//   else, which is what widths with fewer factors of two get: 16 x 10496 x 4096 (two slices) 12.1 / 16.7 and 13.6 / 15.1, 16 x 16256 x
//   4096 (none) at 8 bits 18.1 / 32.0.  At 4 bits the slices have to be whole stages of two atoms (16 x 10752 x 4096 11.9 / 12.5),
//   and up to 12 tokens the rows 12288 channels (12 x 10240 x 2048 9.2 / 9.5, 12 x 12288 x 4096 11.75 / 11.3).  At most 8 tokens: on 8 bits
//   and eight slices only (8 x 10240 x 1024 10.0 / 9.2, 8 x 16384 x 1024 14.2 / 11.3; four: 8 x 16384 x 2048 14.3 / 14.2).
// Two rounds, at most 8 tokens on 4 bits, up to 128 Mi weights: ahead of plain tiles (8 x 4096 x 8192 9.7 / 10.1; 16 x 4096 x 8192
//   13.5 / 10.1: every row group ends with a rendezvous and a reduction), behind stacked ones with 5 tokens and more
//   (8 x 4096 x 8192 8.5 / 7.4, 5 x 9216 x 8704 13.7 / 13.1).  With fewer the streamed calls are shorter, and ahead (1 x 4096 x
//   8192 7.05 / 7.7, 2 x 6144 x 8192 10.2 / 10.5, 1 x 12288 x 9472 15.2 / 15.4) but for long rows (1 x 7168 x 7168 11.0 / 10.4,
//   4 x 8192 x 8192 12.3 / 11.8, 1 x 16384 x 5120 16.8 / 14.7) and where a stacked tile has few stages (4 x 3072 x 5120 6.3 / 5.95, 3 x 4096 x
//   7168 7.55 / 7.1).
inline bool stacked_beats_stream(int64_t M, int64_t N, int64_t K) {
    if (M > 4) return true;
    if (K >= 7168) return N <= (K >= 8192 ? 8192 : 7168);
    return K == 3072 ? N <= 6144 : (M >= 3 && K >= 3840 && K <= 4096 && N <= 7168);
}
// `held`: as for plan_gemm.
template <typename Held>
bool plan_stream(int64_t M, int64_t N, int64_t K, int bits, int sms, Held held) {
    if (K % (bits == 4 ? 256 : 128) != 0 || M < 1 || M > 16) return false;
    const int64_t rounds = (N + 32ll * sms - 1) / (32ll * sms);
    if (rounds > (bits == 4 && M <= 8 ? 2 : 1) || N * K > (bits == 4 && M <= 8 ? 1ll << 27 : 1ll << 26)) return false;
    if (rounds == 2) return !(stacked_applies(M, N, K, bits, sms) && stacked_beats_stream(M, N, K));
    // (no plan is made where its answer would change nothing: it is the host's time)
    const bool ask = K >= 10240 && (bits == 8 ? (M > 8 || N <= 1024) : (M > 8 && K % 1024 == 0 && (M > 12 || K >= 12288)));
    if (!ask) return true;
    const GemmPlan plan = plan_gemm(M, N, K, bits, sms, 0, true, held);
    return !(plan.cluster && plan.split >= (M > 8 ? 4 : 8));
}

// The plan of a call: a stacked tile where they are the faster ones, else plan_gemm's.
template <typename Held>
GemmPlan plan_call(int64_t M, int64_t N, int64_t K, int bits, int sms, size_t scratch_avail, Held held) {
    if (!stacked_applies(M, N, K, bits, sms)) return plan_gemm(M, N, K, bits, sms, scratch_avail, true, held);
    GemmPlan plan;
    plan.bt = kStackSlices * (int)((M + 15) / 16 * 16);
    plan.stack = kStackSlices;
    return plan;
}

}  // namespace fq
