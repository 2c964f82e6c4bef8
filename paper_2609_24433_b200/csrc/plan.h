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

// At most 64 tokens, in one wave of CTAs.  In a chain of calls (graph replays, weights from memory; one launch against two):
// 1024 x 1024: M = 8 3.8 / 4.2 us, M = 32 5.0 / 6.0, M = 50 5.8 / 6.8; K = 2048, N = 1024: M = 32 5.3 / 7.1, M = 50 6.7 / 8.1;
// K = 4096, N = 1024: M = 16 5.4 / 6.3, M = 32 6.4 / 9.0; the largest grids are even (1024 x 4096: M = 32 6.1 / 6.2), and
// behind with few tokens (8 bits, M = 1 4.5 / 4.0): 96 CTAs at most there.  An eager call costs the host 5.4 us instead of 7.7.
// CTAs of two rounds share an SM with nobody and clusters of eight do not fill the chip, so that 128 of them would take two
// waves (K = 4096, N = 2048: 10.3 / 6.3): 96 at most.  Two launches where the device cannot place the clusters.
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
    if (grid > (slice(shift) > round || M <= 8 ? 96 : sms)) return f;
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

}  // namespace fq
