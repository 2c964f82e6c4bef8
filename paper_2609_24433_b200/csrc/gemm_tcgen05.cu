// Integer GEMM of Eq. 8 on the 5th-generation tensor cores (sm_100a):
//   acc[j][t] = sum_c qW[j][c] * qA[t][c]   tcgen05.mma kind::i8, int32 accumulators in TMEM
//   y[t][j]   = delta_t * s^W_j * acc + b_j fused epilogue straight out of TMEM
//
// Orientation.  The 128 rows of an MMA tile are OUTPUT CHANNELS (weight rows),
// the MMA's N dimension (16..256, any multiple of 16) is a tile of TOKENS.  A
// TMEM lane therefore owns one output channel: its scale and bias are per-thread
// scalars in the epilogue, a warp stores 32 consecutive channels of one token
// (coalesced), and ragged token counts (M = 50, 816, ...) are absorbed by the
// free N dimension instead of padding a fixed 128-row tile.
//
// Operands.  Activations (the MMA's B operand) arrive as int8 by TMA, K-major with
// 128-byte rows in the 128B-swizzled shared memory layout.  8-bit weights (the A
// operand) arrive the same way.  4-bit weights stay packed in HBM and in their TMA
// stage; four unpack warps expand each row's 64 packed bytes to 128 int8 holding
// 16*code (nibble moved to the high half of the byte: no sign extension needed) and
// write them with tcgen05.st straight into TENSOR MEMORY, from where the MMA takes
// its A operand -- the unpacked weights never touch shared memory, which is the
// bandwidth that bounds this kernel.  The accumulator is then an exact multiple of
// 2^acc_shift that the epilogue folds into the scale.
//
// Roles (warp specialised, persistent over tiles):
//   warp 0       TMA producer          warp 1  MMA issuer + TMEM allocator
//   4-bit weights: warps 2-9 epilogue (two warps per TMEM lane quadrant, alternating 16-token chunks),
//                warps 10-17 nibble unpack (two sets of four, alternating k-blocks), warp 18 TMA producer
//                of packed weights
//   8-bit weights: warps 2-9 epilogue, warp 10 TMA producer of int8 weights; or warps 2-17 (four per quadrant) and warp 18 (see epi_warps())
// Every role runs its loop with the whole warp converged and elects one lane (elect.sync) for
// the issue itself; a k-block of the MMA warp is one block of PTX that also tests the next
// k-block's barriers (see issue_kblock_*).  With 4-bit weights three rings are decoupled:
// activations (TMA -> MMA), packed weights (TMA -> unpack, deep and cheap: 8 KB a stage) and
// unpacked weights (unpack -> MMA, 32 TMEM columns a stage); one tcgen05.commit per k-block
// frees both the activation stage and the k-block's TMEM slot.
// Variants: CTAS = 2 runs CTA pairs (cta_group::2, 256 channels per MMA, each CTA staging half
// of the token tile); SPLIT lets CTAs share a tile along K and exchange int32 partial sums,
// through the cluster's shared memory or through global scratch, or stacks two slices of K in one tile.
// bf16 outputs leave through a per-warp 1 KB shared-memory transposer so that global
// stores are 16-byte vectors of 8 consecutive channels; fp32/raw outputs store directly.
// Every mbarrier wait is bounded by wall-clock time; on expiry the CTA records a
// code in the watchdog word, stops issuing work, and still frees its TMEM.
#include <cuda_bf16.h>

#include <string.h>

#include <mutex>
#include <type_traits>

#include "fq_common.cuh"
#include "ptx_sm100.cuh"
#include "act_common.cuh"
#include "tc_sm100.cuh"

namespace fq {

__device__ uint32_t g_watchdog_word = 0;

uint32_t* watchdog_device_ptr() {
    // the symbol's address differs per device: looked up once for each
    static std::mutex mutex;
    static uint32_t* addr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    const bool cached = dev >= 0 && dev < 64;
    std::lock_guard<std::mutex> lock(mutex);
    if (cached && addr[dev] != nullptr) return addr[dev];
    uint32_t* p = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_watchdog_word) != cudaSuccess) return nullptr;
    if (cached) addr[dev] = p;
    return p;
}

// Self-test of the bounded-wait machinery: one warp waits, with the ordinary wait routine and a caller-chosen
// limit, on a barrier that nobody ever arrives at.  The wait must give up, record its code in the watchdog word
// and let the kernel end normally.
__global__ void watchdog_selftest_kernel(uint32_t* watchdog, uint64_t limit_ns) {
    __shared__ uint64_t s_bar;
    __shared__ int s_abort;
    if (threadIdx.x == 0) {
        s_abort = 0;
        mbar_init(smem_u32(&s_bar), 1);
        fence_mbarrier_init();
    }
    __syncthreads();
    mbar_wait_all(smem_u32(&s_bar), 0u, &s_abort, watchdog, 0x400u, false, limit_ns);
}

cudaError_t launch_watchdog_selftest(uint64_t limit_ns, cudaStream_t stream) {
    uint32_t* wd = watchdog_device_ptr();
    if (!wd) return cudaErrorUnknown;
    watchdog_selftest_kernel<<<1, 32, 0, stream>>>(wd, limit_ns);
    return cudaGetLastError();
}

cudaError_t read_and_clear_watchdog(uint32_t* word) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return e;
    e = cudaMemcpyFromSymbol(word, g_watchdog_word, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    const uint32_t zero = 0;
    return cudaMemcpyToSymbol(g_watchdog_word, &zero, sizeof(uint32_t));
}

namespace {

// Activation producer, MMA issuer, epilogue, nibble unpack, weight producer.
constexpr int gemm_threads(int bits, int epi) { return 32 * (2 + epi) + (bits == 4 ? kUnpackSets * 128 : 0) + 32; }
// 8-bit weights, eight epilogue warps: at most 128 registers per thread (140 to 147 without), so that the next call's prologue finds room
// beside it: 64 x 2048 x 20000 14.1 -> 12.8 us, 128 x 4096 x 9472 13.2 -> 12.4.
constexpr int gemm_bounds(int bits, int epi) { return bits == 8 && epi == kEpiWarps ? 512 : gemm_threads(bits, epi); }
constexpr int kFirstUnpackWarp = 2 + kEpiWarps;
constexpr int kStackRows = kTileN / kStackSlices;        // channels of a stacked tile
enum : int { kUnsplit = 0, kSplitScratch = 1, kSplitCluster = 2, kStacked = 3 };

struct Params {
    int64_t M, N, K;
    int bt;              // columns per tile (MMA N): tokens, times the K slices of a stacked tile; multiple of 16, <= 256
    int tok;             // tokens per tile
    int stages;          // activation ring (and int8 weight ring, in lockstep, for 8-bit weights)
    int stages_p;        // packed-weight ring (4-bit weights)
    int stages_w;        // unpacked-weight ring (4-bit weights)
    int m_tiles, n_tiles;
    int band;            // token tiles per band of the tile order (see tile_coords); m_tiles = one band = channel-major order
    int tmem_cols;
    int acc_shift;
    const float* w_scale;
    const float* bias;
    GemmOut out;
    uint32_t* watchdog;
    // index arithmetic done once on the host (integer divisions cost the short launches ~0.3 us)
    int cluster_shift;   // log2 of the CTAs per cluster (1 for CTA pairs)
    int unit_step;       // CTAs (or pairs) in the grid
    int units_q, units_rem;   // work units per CTA: units_q, one more for the first units_rem CTAs
    int kb_per;          // k-blocks of one work unit (all of K, or K / split)
    int split, split_shift;   // K split: a tile is `split` (power of two) work units, each on a slice of K
    int32_t* partials;   // [tile][slice][bt tokens][128 channels] int32 raw sums of the slices (K split)
    uint32_t* counters;  // [tile] slices finished so far; zeroed by the host before the launch (K split)
    int delta_vec;       // a_delta is 16-byte aligned: the epilogue may read four steps per load
    int slot_first;      // 1: the unpack sets wait for the TMEM slot ahead of the packed stage (see there)
    uint32_t zero;       // 0, as a run-time value (see the unpack warps' release of a packed stage)
};

// ---- CTA-pair (cta_group::2) helpers -----------------------------------------------------
// Arrive on the barrier at the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ void mbar_arrive_cta(uint32_t bar, uint32_t rank) {
    asm volatile(
        "{\n\t.reg .b32 ra;\n\t"
        "mapa.shared::cluster.u32 ra, %0, %1;\n\t"
        "mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}"
        ::"r"(bar), "r"(rank)
        : "memory");
}
// Pair variant of the tiled load: issued by both CTAs into their own shared memory, but the
// bytes are counted on the barrier of the pair's even CTA (address with the peer bit cleared).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar & 0xFEFFFFFFu)
        : "memory");
}
// One k-block of work for the issuing warp, as ONE block of PTX so that the two barrier tests for
// the NEXT k-block are in flight while this k-block's four MMAs and its commits are issued (their
// results are read only at the end; separate asm statements would stall on each test's ~100-cycle
// latency).  Must be called by a converged warp: every lane executes the tests, and the lane that
// elect.sync picks inside the block issues the MMAs and commits (measured: 160 cycles per k-block
// with the election inside the block, 400 with a predicate derived from the lane index).
//   a[4]      A operand of the four K=32 steps: TMEM addresses (TS) or shared-memory descriptors (SS)
//   bar_stage barrier that frees the k-block's shared-memory (and TMEM weight) stage
//   bar_acc   barrier "accumulator complete", or 0 when this is not the tile's last k-block
//   mask      (CTA pairs) cluster ranks of the pair, whose barriers the commits arrive at
// Returns 1 if both tested phases were complete (0 when `peek` is 0).
#define FQ_ISSUE_HEAD                                                   \
    "{\n\t"                                                             \
    ".reg .pred pl, pacc, pt, pk, pa, pw, pc;\n\t"                       \
    "elect.sync _|pl, 0xffffffff;\n\t"                                  \
    "setp.ne.b32 pacc, %12, 0;\n\t"                                     \
    "setp.eq.b32 pt, %1, %1;\n\t"                                       \
    "setp.ne.b32 pk, %15, 0;\n\t"                                       \
    "setp.ne.b32 pa, %1, %1;\n\t"                                       \
    "setp.ne.b32 pw, %1, %1;\n\t"                                       \
    "@pk mbarrier.test_wait.parity.shared::cta.b64 pa, [%16], %17;\n\t" \
    "@pk mbarrier.test_wait.parity.shared::cta.b64 pw, [%18], %19;\n\t"
#define FQ_ISSUE_MMAS(CG, L, R)                                                          \
    "@pl tcgen05.mma.cta_group::" CG ".kind::i8 [%2], " L "%3" R ", %7, %11, pacc;\n\t"   \
    "@pl tcgen05.mma.cta_group::" CG ".kind::i8 [%2], " L "%4" R ", %8, %11, pt;\n\t"     \
    "@pl tcgen05.mma.cta_group::" CG ".kind::i8 [%2], " L "%5" R ", %9, %11, pt;\n\t"     \
    "@pl tcgen05.mma.cta_group::" CG ".kind::i8 [%2], " L "%6" R ", %10, %11, pt;\n\t"
#define FQ_ISSUE_COMMITS_1                                                                          \
    "@pl tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%13];\n\t"          \
    "setp.ne.and.b32 pc, %14, 0, pl;\n\t"                                                           \
    "@pc tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%14];\n\t"
#define FQ_ISSUE_COMMITS_2                                                                                          \
    "@pl tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%13], %20;\n\t"  \
    "setp.ne.and.b32 pc, %14, 0, pl;\n\t"                                                                           \
    "@pc tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%14], %20;\n\t"
#define FQ_ISSUE_TAIL            \
    "and.pred pa, pa, pw;\n\t"   \
    "selp.b32 %0, 1, 0, pa;\n\t" \
    "}"
#define FQ_ISSUE_OPERANDS(ACON)                                                                                      \
    : "=r"(ready)                                                                                                    \
    : "r"(issue), "r"(d_tmem), ACON(a[0]), ACON(a[1]), ACON(a[2]), ACON(a[3]), "l"(b[0]), "l"(b[1]), "l"(b[2]),      \
      "l"(b[3]), "r"(idesc), "r"(accumulate), "r"(bar_stage), "r"(bar_acc), "r"(peek), "r"(peek_bar_a),              \
      "r"(peek_par_a), "r"(peek_bar_w), "r"(peek_par_w), "h"(mask)                                                   \
    : "memory"
#define FQ_CON_R(x) "r"(x)
#define FQ_CON_L(x) "l"(x)

template <int CTAS>
__device__ __forceinline__ uint32_t issue_kblock_ts(uint32_t issue, uint32_t d_tmem, const uint32_t* a, const uint64_t* b,
                                                    uint32_t idesc, uint32_t accumulate, uint32_t bar_stage,
                                                    uint32_t bar_acc, uint32_t peek, uint32_t peek_bar_a,
                                                    uint32_t peek_par_a, uint32_t peek_bar_w, uint32_t peek_par_w, uint16_t mask) {
    uint32_t ready;
    if (CTAS == 1)
        asm volatile(FQ_ISSUE_HEAD FQ_ISSUE_MMAS("1", "[", "]") FQ_ISSUE_COMMITS_1 FQ_ISSUE_TAIL FQ_ISSUE_OPERANDS(FQ_CON_R));
    else
        asm volatile(FQ_ISSUE_HEAD FQ_ISSUE_MMAS("2", "[", "]") FQ_ISSUE_COMMITS_2 FQ_ISSUE_TAIL FQ_ISSUE_OPERANDS(FQ_CON_R));
    return ready;
}
template <int CTAS>
__device__ __forceinline__ uint32_t issue_kblock_ss(uint32_t issue, uint32_t d_tmem, const uint64_t* a, const uint64_t* b,
                                                    uint32_t idesc, uint32_t accumulate, uint32_t bar_stage,
                                                    uint32_t bar_acc, uint32_t peek, uint32_t peek_bar_a,
                                                    uint32_t peek_par_a, uint32_t peek_bar_w, uint32_t peek_par_w, uint16_t mask) {
    uint32_t ready;
    if (CTAS == 1)
        asm volatile(FQ_ISSUE_HEAD FQ_ISSUE_MMAS("1", "", "") FQ_ISSUE_COMMITS_1 FQ_ISSUE_TAIL FQ_ISSUE_OPERANDS(FQ_CON_L));
    else
        asm volatile(FQ_ISSUE_HEAD FQ_ISSUE_MMAS("2", "", "") FQ_ISSUE_COMMITS_2 FQ_ISSUE_TAIL FQ_ISSUE_OPERANDS(FQ_CON_L));
    return ready;
}
// 16 TMEM lanes x 16 columns in the layout of a warp-level MMA accumulator: thread T holds, for column groups n = 0, 1,
//   r[4n + 0], r[4n + 1] = lane T/4,     columns 8n + 2(T%4), 8n + 2(T%4) + 1
//   r[4n + 2], r[4n + 3] = lane T/4 + 8, the same two columns.
// With channels on the lanes and tokens on the columns, a register pair is one channel at two adjacent tokens --
// the fragment that stmatrix stores transposed, i.e. token-major.
__device__ __forceinline__ void tmem_ld_16x256b_x2(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
// Four 8x8 matrices of 16-bit elements, each thread's register i a fragment (row T/4, columns 2(T%4), 2(T%4)+1) of
// matrix i, stored TRANSPOSED: the 16 bytes at the address given by thread 8i + r receive column r of matrix i.
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                 ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
                 : "memory");
}
// Tiled bulk STORE shared -> global (a store, never a multicast load); rows and columns beyond the tensor's extent
// are clipped by the copy engine.  Completion is tracked per issuing thread in bulk groups.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int c0, int c1, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(src)
                 : "memory");
}
// One channel at two adjacent tokens: y = acc * (delta_t * s_j) + b_j, rounded to bf16, token 2k in the low half.
__device__ __forceinline__ uint32_t scale_pair_bf16(uint32_t a0, uint32_t a1, float2 d, float2 sw2, float2 bj2) {
    const float2 a2 = make_float2((float)(int)a0, (float)(int)a1);
    const float2 v2 = f2_fma(a2, f2_mul(d, sw2), bj2);
    uint32_t w;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(v2.y), "f"(v2.x));
    return w;
}

enum : uint32_t {
    kWdProducer = 1u, kWdMmaFull = 2u, kWdMmaAcc = 4u, kWdEpilogue = 8u, kWdUnpackFull = 16u,
    kWdUnpackEmpty = 32u, kWdDrain = 64u, kWdPartials = 128u
};

// CTAS = 2: two CTAs of a cluster work as a pair on a 256-channel x bt-token tile (cta_group::2):
// each loads its own 128 weight rows and HALF of the token tile, the even CTA issues the MMAs for
// both, and every MMA reads the token halves out of both CTAs' shared memory.  This halves the
// activation bytes each SM pulls from L2, which is what bounds the single-CTA kernel.
// ATOMS (4-bit weights, single CTAs, token tiles of at most 128): a pipeline stage holds ATOMS k-blocks of 128
// channels (two 128-byte swizzle atoms side by side).  The kernel is bound by instruction issue, and the waits,
// arrivals, fences and ring arithmetic of every role are paid per stage: twice the channels per stage take a
// third off the instructions per channel.  (Longer token tiles have no TMEM left for slots twice as wide.)
// SPLIT: kSplitScratch exchanges the K slices' sums through global scratch, any CTA taking any slice; kSplitCluster gives the
// slices of a tile to the CTAs of a cluster, one tile per cluster and launch, and exchanges through distributed shared memory.
template <int BITS, int CTAS, int SPLIT, int ATOMS, int EPI>
__global__ void __launch_bounds__(gemm_bounds(BITS, EPI), 1)
gemm_tcgen05_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_w,
                    const __grid_constant__ CUtensorMap map_y, const Params p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t s_full_tma[kMaxStages];     // activations (+ int8 weights) landed
    __shared__ uint64_t s_empty[kMaxStages];        // ... consumed by the MMAs (one commit per k-block; for 4-bit
                                                    // weights it also frees that k-block's TMEM weight slot)
    __shared__ uint64_t s_full_p[kMaxStagesP];      // packed weights landed
    __shared__ uint64_t s_empty_p[kMaxStagesP];     // ... read by the unpack warps
    __shared__ uint64_t s_full_w8[kMaxStagesW];     // unpacked weights written
    __shared__ uint64_t s_acc_full[kAccStages];
    __shared__ uint64_t s_acc_empty[kAccStages];
    __shared__ uint64_t s_sums;                     // cluster split: the other slices' sums are here
    __shared__ uint64_t s_epi_sync;                 // K split: rendezvous of the eight epilogue warps (bounded, unlike bar.sync)
    __shared__ int s_last[2];                       // K split: this CTA counted the last slice of its tile (alternating slots)
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile int* abort_flag = &s_abort;
    if (threadIdx.x == 32) {
        // the three copy descriptors are kernel parameters: fetching them now takes their first-use latency (a few
        // hundred nanoseconds each) off the path between the end of the kernel ahead and this kernel's first copy
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_w)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_y)) : "memory");
    }
    const uint32_t pair_base = CTAS == 2 ? cluster_ctarank() & ~1u : 0u;      // cluster rank of the pair's even CTA
    const uint32_t cta_rank = CTAS == 2 ? cluster_ctarank() & 1u : 0u;
    const bool leader = cta_rank == 0;
    constexpr bool kCluster = SPLIT == kSplitCluster;
    constexpr bool kStack = SPLIT == kStacked;
    constexpr int kEpiSets = EPI / 4;               // epilogue warps per TMEM lane quadrant: each takes every kEpiSets-th chunk
    // K split: a tile is `split` work units, unit = tile * split + slice, slice s
    // covering k-blocks [s * k_blocks, (s + 1) * k_blocks).  Any CTA takes any unit; the CTA that
    // finishes a tile's last slice adds up the slices' partial sums and runs the epilogue.
    const int split = SPLIT != kUnsplit && !kStack ? p.split : 1;   // compile-time 1 in the common instantiation
    const int split_shift = SPLIT != kUnsplit && !kStack ? p.split_shift : 0;
    const int bt_cta = p.bt / CTAS;                 // token rows this CTA loads

    // carve dynamic shared memory: [A8 stages][W8 stages][packed stages][epilogue transposers], 1024-byte aligned
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_atom = (uint32_t)bt_cta * kBlockK;        // one 128-channel atom of the token tile
    const uint32_t a_bytes = a_atom * ATOMS;
    const uint32_t w_bytes = kTileN * kBlockK;
    const uint32_t pk_atom = kTileN * kBlockK / 2;
    const uint32_t pk_bytes = pk_atom * ATOMS;
    constexpr int kSlotCols = kColsW * ATOMS;                   // TMEM columns of one unpacked stage
    const uint32_t smem_a = base;
    const uint32_t smem_w = smem_a + (uint32_t)p.stages * a_bytes;
    const uint32_t smem_p = smem_w + (BITS == 4 ? 0u : (uint32_t)p.stages * w_bytes);
    const uint32_t smem_e = smem_p + (BITS == 4 ? (uint32_t)p.stages_p * pk_bytes : 0u);
    constexpr int kEpiBytes = BITS == 8 && SPLIT != kUnsplit ? kEpiStageBytes / kEpiBuffers : kEpiStageBytes;
    const uint32_t smem_sums = smem_e + (uint32_t)(EPI * kEpiBytes);    // cluster split: the other slices' sums
    uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));   // generic pointer to `base`

    if (threadIdx.x == 0) {
        // (One thread on purpose: spreading these initialisations over the lanes of a warp, one ring
        // slot per lane, shortened the set-up by 0.3 us but made the 8-bit main loop 10 % slower.)
        s_abort = 0;
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&s_full_tma[s]), BITS == 8 ? 2 : 1);   // 8-bit: activation and weight producers
            mbar_init(smem_u32(&s_empty[s]), 1);
        }
        if (BITS == 4) {
            for (int s = 0; s < p.stages_p; ++s) {
                mbar_init(smem_u32(&s_full_p[s]), 1);
                mbar_init(smem_u32(&s_empty_p[s]), 4);
            }
            for (int s = 0; s < p.stages_w; ++s) mbar_init(smem_u32(&s_full_w8[s]), 4 * CTAS);
        }
        for (int a = 0; a < kAccStages; ++a) {
            mbar_init(smem_u32(&s_acc_full[a]), 1);
            mbar_init(smem_u32(&s_acc_empty[a]), EPI * CTAS);
        }
        mbar_init(smem_u32(&s_epi_sync), EPI);
        mbar_init(smem_u32(&s_sums), 1);
        fence_mbarrier_init();
        fence_proxy_async_smem();
    }
    if (warp == 1) tmem_alloc<CTAS>(smem_u32(&s_tmem_base), (uint32_t)p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    if (CTAS == 2) cluster_sync_all();              // the peer's barriers exist before anyone signals them
    // Tile order.  Consecutive tile numbers -- the tiles the SMs work on at the same time -- cover a compact block of
    // the output: the token tiles are cut into bands of p.band, a band is walked channel tile by channel tile with
    // its token tiles fastest.  What one wave of CTAs pulls through L2 is then band activation tiles plus SMs/band
    // weight tiles instead of every activation tile of the batch (long batches: the int8 activations alone exceed
    // L2, and in channel-major order every wave streamed all of them from HBM again).
    auto m_of = [&](int tile) {
        if (p.band >= p.m_tiles) return tile % p.m_tiles;
        const int b = tile / (p.band * p.n_tiles);
        const int r = tile - b * (p.band * p.n_tiles);
        const int rows = max(1, min(p.band, p.m_tiles - b * p.band));   // (a producer also maps the unit past its last one)
        return b * p.band + r % rows;
    };
    if (kCluster) {
        // what the other slices will send: the chunks of 16 tokens that this one finishes
        const int unit = (int)blockIdx.x >> p.cluster_shift, tile = unit >> split_shift, slice = unit & (split - 1);
        if (threadIdx.x == 0) {
            const int64_t left = p.M - (int64_t)m_of(tile) * p.bt;
            const int chunks = min(p.bt / 16, (int)min((left + 15) / 16, (int64_t)16));
            mbar_arrive_expect_tx(smem_u32(&s_sums), (uint32_t)((split - 1) * ((chunks - slice + split - 1) >> split_shift) * 4 * kSumBytes));
        }
        __syncwarp();                               // (the arrival is the converged warp's)
        cluster_arrive();                           // "this CTA exists": awaited before the first copy to another
    }
    tc_fence_after();
    const uint32_t tmem_base = s_tmem_base;
    // Everything above is on-chip setup; from here on global memory is touched (activations written
    // by the kernel before this one, outputs that it may still be reading).
    // Only the warps that touch what the kernel ahead writes (or may still read) wait for it: the activation
    // producer, and the epilogue warps (per-token steps, K-split scratch, the output).  A weight handle is
    // complete before any call that uses it is enqueued, so the weight producer streams tiles in, the unpack
    // warps fill their TMEM slots, and the MMA warp parks on its barriers while the prologue still runs.
    if (warp == 0 || (warp >= 2 && warp < 2 + EPI)) griddep_wait();
    griddep_launch_dependents();

    // work units: (super-tile of 128*CTAS channels) x (token tile) [x K slice]; one unit per CTA or
    // CTA pair at a time
    const int num_units = (p.m_tiles * p.n_tiles) << split_shift;
    const int unit0 = (int)blockIdx.x >> p.cluster_shift;
    const int unit_step = p.unit_step;
    const int my_units = p.units_q + (unit0 < p.units_rem ? 1 : 0);
    const int k_blocks = p.kb_per;
    auto tile_of = [&](int unit) { return unit >> split_shift; };
    auto n_of = [&](int tile) {
        if (p.band >= p.m_tiles) return tile / p.m_tiles;
        const int b = tile / (p.band * p.n_tiles);
        const int r = tile - b * (p.band * p.n_tiles);
        return r / max(1, min(p.band, p.m_tiles - b * p.band));
    };
    auto kb0_of = [&](int unit) { return (unit & (split - 1)) * k_blocks; };   // first k-block of the unit's slice

    // Steps of the 16 tokens of this warp's next chunk: lanes 16 (n & 1) ... of the first register; requested ahead of the sums,
    // so that their trip through L2 is over when those are complete.  (Not in unsplit launches on 4-bit weights, whose epilogue
    // takes its issue slots from the nibble unpack: with the exchange between lanes binary32 outputs took 2048 x 4096 x 4096 42.0 us
    // instead of 40.6, 6819 x 5120 x 2176 82.1 instead of 80.2.)
    constexpr bool kStepsAhead = BITS == 8 || SPLIT != kUnsplit;
    constexpr int kStepRegs = (16 / kEpiSets + 1) / 2;          // tiles have at most sixteen chunks
    [[maybe_unused]] float steps[kStepRegs] = {};
    auto next_steps = [&](int n) {
        if ((n & 1) != 0) {
#pragma unroll
            for (int i = 0; i + 1 < kStepRegs; ++i) steps[i] = steps[i + 1];
        }
    };
    [[maybe_unused]] float2 tail = make_float2(0.0f, 0.0f);   // (cluster split: scale and bias of this lane's channel)
    [[maybe_unused]] bool ok = true, waited = false;   // (ok: of the epilogue warps; the other roles have their own)
    // ---- output of 16 tokens from tc on (this warp's n-th chunk), lane = channel j of this warp's 32 (jq ..): r = integer sums
    auto emit = [&](uint32_t* r, int n, int64_t tc, int64_t jq, float sw, float bj, uint8_t* xpose) {
        const int64_t j = jq + lane;
        const bool j_ok = j < p.N;
        if (p.out.acc != nullptr) {
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (tc + i < p.M && j_ok) p.out.acc[(tc + i) * p.N + j] = ((int)r[i]) >> p.acc_shift;
            return;
        }
        float d[16];
        if constexpr (kStepsAhead) {
#pragma unroll
            for (int i = 0; i < 16; ++i) d[i] = __shfl_sync(0xffffffffu, steps[0], 16 * (n & 1) + i);
            next_steps(n);
        } else if (tc + 16 <= p.M && p.delta_vec) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 q = ld_global_f4(p.out.a_delta + tc + 4 * i);
                d[4 * i + 0] = q.x; d[4 * i + 1] = q.y; d[4 * i + 2] = q.z; d[4 * i + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) d[i] = tc + i < p.M ? ld_global_f32(p.out.a_delta + tc + i) : 0.0f;
        }
        tmem_ld_wait();                          // (the sums may still be on their way)
        if (p.out.yt == FQ_BF16) {
            // Transpose 32 channels x 16 tokens through shared memory, then 16-byte stores.  Tokens
            // go in pairs: packed multiply, packed FMA and one two-way bf16 conversion per pair, the
            // pair's word (token 2k low, token 2k+1 high) stored at [pair k][channel].  A lane then
            // reads 8 channels of one pair (32 bytes), splits the two tokens with byte permutes and
            // writes 8 consecutive channels of each token.
            uint32_t* xw = reinterpret_cast<uint32_t*>(xpose);
            const float2 sw2 = make_float2(sw, sw), bj2 = make_float2(bj, bj);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float2 a2 = make_float2((float)(int)r[2 * k], (float)(int)r[2 * k + 1]);
                const float2 v2 = f2_fma(a2, f2_mul(make_float2(d[2 * k], d[2 * k + 1]), sw2), bj2);
                uint32_t w;
                asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(v2.y), "f"(v2.x));
                xw[k * 32 + lane] = w;
            }
            __syncwarp();
            __nv_bfloat16* y = static_cast<__nv_bfloat16*>(p.out.y);
            {
                const int k = lane >> 2;
                const int64_t jj = jq + (lane & 3) * 8;
                const uint4 q0 = *reinterpret_cast<const uint4*>(xw + k * 32 + (lane & 3) * 8);
                const uint4 q1 = *reinterpret_cast<const uint4*>(xw + k * 32 + (lane & 3) * 8 + 4);
                uint4 lo, hi;     // token 2k and token 2k + 1, channels jj .. jj + 7
                lo.x = __byte_perm(q0.x, q0.y, 0x5410); hi.x = __byte_perm(q0.x, q0.y, 0x7632);
                lo.y = __byte_perm(q0.z, q0.w, 0x5410); hi.y = __byte_perm(q0.z, q0.w, 0x7632);
                lo.z = __byte_perm(q1.x, q1.y, 0x5410); hi.z = __byte_perm(q1.x, q1.y, 0x7632);
                lo.w = __byte_perm(q1.z, q1.w, 0x5410); hi.w = __byte_perm(q1.z, q1.w, 0x7632);
                if (jj < p.N) {
                    if (tc + 2 * k < p.M) *reinterpret_cast<uint4*>(y + (tc + 2 * k) * p.out.ldy + jj) = lo;
                    if (tc + 2 * k + 1 < p.M) *reinterpret_cast<uint4*>(y + (tc + 2 * k + 1) * p.out.ldy + jj) = hi;
                }
            }
            __syncwarp();
        } else {
            float* y = static_cast<float*>(p.out.y) + tc * p.out.ldy + j;
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (tc + i < p.M && j_ok) y[i * p.out.ldy] = fmaf((float)(int)r[i], d[i] * sw, bj);
        }
    };
    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        // The whole warp runs the loop and waits; one lane issues.  (A lone lane looping while its
        // warp-mates are parked at the final __syncthreads was measured 2-3x slower per barrier
        // hand-off: every dependent wait/branch of the lone lane pays for the divergent warp.)
        {
            const uint32_t tx = a_bytes;
            const int total_kb = my_units * k_blocks;
            bool ok = true;
            int stage = 0, kb = 0, unit = unit0;
            uint32_t phase = 0;
            int t0 = m_of(tile_of(unit)) * p.tok + (int)cta_rank * bt_cta;
            int kb0 = kb0_of(unit);
            bool peek = false;
            for (int n = 0; n < total_kb; ++n) {
                ok = mbar_wait_all_lazy(smem_u32(&s_empty[stage]), phase ^ 1u, abort_flag, p.watchdog, kWdProducer, peek);
                if (!ok) break;
                {   // look at the next stage now: the test's latency hides behind the copy issued below
                    const int s1 = stage + 1 == p.stages ? 0 : stage + 1;
                    const uint32_t ph1 = s1 == 0 ? phase ^ 1u : phase;
                    peek = n + 1 < total_kb && mbar_test_wait(smem_u32(&s_empty[s1]), ph1 ^ 1u);
                }
                if (elect_one()) {
                    const uint32_t bar = smem_u32(&s_full_tma[stage]);
                    if (CTAS == 1) {
                        mbar_arrive_expect_tx(bar, tx);
                        if constexpr (kStack) tma_load_4d(smem_a + stage * a_bytes, &map_a, 0, t0, 0, (kb0 + kb) * ATOMS, bar);
                        else {
#pragma unroll
                            for (int h = 0; h < ATOMS; ++h)     // channels past K arrive as zeros
                                tma_load_2d(smem_a + stage * a_bytes + h * a_atom, &map_a, ((kb0 + kb) * ATOMS + h) * kBlockK, t0, bar);
                        }
                    } else {
                        // the pair's bytes are all counted on the even CTA's barrier, which it arms for both
                        if (leader) mbar_arrive_expect_tx(bar, tx * CTAS);
                        tma_load_2d_pair(smem_a + stage * a_bytes, &map_a, (kb0 + kb) * kBlockK, t0, bar);
                    }
                }
                if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                if (++kb == k_blocks) {
                    kb = 0;
                    unit += unit_step;
                    t0 = m_of(tile_of(unit)) * p.tok + (int)cta_rank * bt_cta;
                    kb0 = kb0_of(unit);
                }
            }
            if (!ok && lane == 0) drain_after_abort();
        }
    } else if (warp == 1) {
        // -------------------------------------------------------------- MMA issuer
        // All lanes of the warp run the loop and the waits (converged); lane 0 of the pair's even
        // CTA issues the MMAs and commits.
        if (leader) {
            const uint32_t idesc = instr_desc_i8(kTileN * CTAS, p.bt);
            const uint16_t pair_mask = (uint16_t)(3u << pair_base);   // cluster ranks that a pair's commits arrive at
            int stage = 0, wstage = 0;
            uint32_t phase = 0, wphase = 0;
            int acc_stage = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            // The barriers of the NEXT k-block are tested (without blocking) inside the block of PTX
            // that issues the current one: a barrier test has ~100 cycles of latency, and two of them
            // in series per k-block would otherwise sit on the issuing warp's critical path.
            bool ready = false;
            int left = my_units * k_blocks;   // k-blocks still to issue
            for (int unit = unit0; unit < num_units && ok; unit += unit_step) {
                ok = mbar_wait_all(smem_u32(&s_acc_empty[acc_stage]), acc_phase ^ 1u, abort_flag, p.watchdog, kWdMmaAcc);
                if (!ok) break;
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc_stage * p.bt);
                for (int kb = 0; kb < k_blocks; ++kb) {
                    if (!__all_sync(0xffffffffu, ready)) {
                        ok = mbar_wait_all(smem_u32(&s_full_tma[stage]), phase, abort_flag, p.watchdog, kWdMmaFull);
                        if (ok && BITS == 4)
                            ok = mbar_wait_all(smem_u32(&s_full_w8[wstage]), wphase, abort_flag, p.watchdog, kWdMmaFull);
                        if (!ok) break;
                    }
                    --left;
                    tc_fence_after();
                    const int s1 = stage + 1 == p.stages ? 0 : stage + 1;
                    const uint32_t ph1 = s1 == 0 ? phase ^ 1u : phase;
                    const int w1 = wstage + 1 == p.stages_w ? 0 : wstage + 1;
                    const uint32_t wph1 = w1 == 0 ? wphase ^ 1u : wphase;
                    const uint32_t peek_bar_a = smem_u32(&s_full_tma[s1]);
                    const uint32_t peek_bar_w = BITS == 4 ? smem_u32(&s_full_w8[w1]) : peek_bar_a;
                    const uint32_t peek_par_w = BITS == 4 ? wph1 : ph1;
                    const uint32_t bar_acc = kb == k_blocks - 1 ? smem_u32(&s_acc_full[acc_stage]) : 0u;
                    uint32_t accumulate = kb != 0 ? 1u : 0u;
                    if (BITS == 4 && ATOMS > 1) {        // all atoms of the stage but the last: four MMAs each, no commit yet
#pragma unroll
                        for (int h = 0; h < ATOMS - 1; ++h) {
                            const uint64_t adesc0 = smem_desc_sw128(smem_a + stage * a_bytes + h * a_atom);
                            const uint64_t bd0[4] = {adesc0, adesc0 + 2, adesc0 + 4, adesc0 + 6};
                            const uint32_t w0 = tmem_base + (uint32_t)(kAccStages * p.bt + wstage * kSlotCols + h * kColsW);
                            const uint32_t at0[4] = {w0, w0 + 8, w0 + 16, w0 + 24};
                            issue_mmas_ts(d_tmem, at0, bd0, idesc, accumulate);
                            accumulate = 1u;
                        }
                    }
                    const uint64_t adesc = smem_desc_sw128(smem_a + stage * a_bytes + (ATOMS - 1) * a_atom);
                    // step 32 bytes along K inside the swizzle atom: +2 in 16-byte address units
                    const uint64_t bd[4] = {adesc, adesc + 2, adesc + 4, adesc + 6};
                    uint32_t r;
                    if (BITS == 4) {
                        // 32 int8 of K = 8 TMEM columns per MMA
                        const uint32_t w_tmem = tmem_base + (uint32_t)(kAccStages * p.bt + wstage * kSlotCols + (ATOMS - 1) * kColsW);
                        const uint32_t at[4] = {w_tmem, w_tmem + 8, w_tmem + 16, w_tmem + 24};
                        r = issue_kblock_ts<CTAS>(0u, d_tmem, at, bd, idesc, accumulate,
                                                  smem_u32(&s_empty[stage]), bar_acc, left > 0 ? 1u : 0u, peek_bar_a, ph1,
                                                  peek_bar_w, peek_par_w, pair_mask);
                    } else {
                        const uint64_t wdesc = smem_desc_sw128(smem_w + stage * w_bytes);
                        const uint64_t ad[4] = {wdesc, wdesc + 2, wdesc + 4, wdesc + 6};
                        r = issue_kblock_ss<CTAS>(0u, d_tmem, ad, bd, idesc, kb != 0 ? 1u : 0u,
                                                  smem_u32(&s_empty[stage]), bar_acc, left > 0 ? 1u : 0u, peek_bar_a, ph1,
                                                  peek_bar_w, peek_par_w, pair_mask);
                    }
                    ready = r != 0;
                    stage = s1;
                    phase = ph1;
                    if (BITS == 4) { wstage = w1; wphase = wph1; }
                }
                if (!ok) break;
                if (++acc_stage == kAccStages) { acc_stage = 0; acc_phase ^= 1u; }
            }
        }
    } else if (warp < 2 + EPI) {
        // ---------------------------------------------------------------- epilogue
        const int quad = warp & 3;                       // TMEM lanes [32*quad, 32*quad + 32)
        const int half = (warp - 2) >> 2;                // which of the alternating 16-token chunks
        uint8_t* xpose = gen_base + (smem_e - base) + (warp - 2) * kEpiBytes;
        const bool staged = p.out.acc == nullptr && p.out.yt == FQ_BF16;
        const float unshift = 1.0f / (float)(1 << p.acc_shift);   // exact power of two
        auto constants = [&](int64_t j) {                // of channel j: scale and bias
            const bool j_ok = j < p.N && p.out.acc == nullptr;
            // ((float)acc * 2^-shift is exact: the shift is folded into the scale)
            return j_ok ? make_float2(__ldg(p.w_scale + j) * unshift, __ldg(p.bias + j)) : make_float2(0.0f, 0.0f);
        };
        int acc_stage = 0;
        uint32_t acc_phase = 0;
        [[maybe_unused]] uint32_t epi_phase = 0;
        [[maybe_unused]] int epi_use = 0;
        [[maybe_unused]] int store_use = 0;             // bulk stores issued by this warp so far (buffer = parity)
        for (int unit = unit0; unit < num_units && ok; unit += unit_step) {
            const int tile = tile_of(unit);
            // first channel of this warp
            const int64_t jq = kStack ? (int64_t)n_of(tile) * kStackRows + (quad & 1) * 32
                                      : (int64_t)n_of(tile) * (kTileN * CTAS) + (int64_t)cta_rank * kTileN + quad * 32;
            const int64_t t0 = (int64_t)m_of(tile) * p.tok;
            const float2 cj = constants(jq + lane);
            const float sw = cj.x, bj = cj.y;
            if (kStepsAhead && (SPLIT != kUnsplit || !staged)) {   // the steps of this warp's chunks
                const int sh = kStack ? 1 : (kCluster ? split_shift : 0);
                const int off = kStack ? quad >> 1 : (kCluster ? unit & (split - 1) : 0);
#pragma unroll
                for (int i = 0; i < kStepRegs; ++i) {
                    const int t = (((half + (2 * i + (lane >> 4)) * kEpiSets) << sh) + off) * 16 + (lane & 15);
                    steps[i] = p.out.acc == nullptr && t < p.tok && t0 + t < p.M ? ld_global_f32(p.out.a_delta + t0 + t) : 0.0f;
                }
            }
            // bf16 outputs of an unsplit launch: the four channels of this thread's accumulator fragments
            [[maybe_unused]] float2 sw4[4], bj4[4], nd0, nd1;
            auto request_steps = [&](int c) {                // ... and the steps of its four tokens
                const int64_t ta = t0 + c + 2 * (lane & 3), tb = ta + 8;
                nd0.x = ta < p.M ? ld_global_f32(p.out.a_delta + ta) : 0.0f;
                nd0.y = ta + 1 < p.M ? ld_global_f32(p.out.a_delta + ta + 1) : 0.0f;
                nd1.x = tb < p.M ? ld_global_f32(p.out.a_delta + tb) : 0.0f;
                nd1.y = tb + 1 < p.M ? ld_global_f32(p.out.a_delta + tb + 1) : 0.0f;
            };
            auto request_constants = [&]() {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 ci = constants(jq + (lane >> 2) + 8 * i);
                    sw4[i] = make_float2(ci.x, ci.x);
                    bj4[i] = make_float2(ci.y, ci.y);
                }
                request_steps(half * 16);
            };
            // Ahead of the sums for the last tile, whose epilogue hides behind nothing: their trip through L2 is over when the
            // sums are complete.  (Not for the others, beside whose epilogue the next tile is multiplied: 816 x 2048 x 32768 47.8 us
            // instead of 48.1; the pairs of 4-bit weights have no registers for it.)
            const bool ahead = !(BITS == 4 && CTAS == 2) && unit + unit_step >= num_units;
            if (SPLIT == kUnsplit && staged && ahead) request_constants();
            // a tile takes at least ~0.2 us per k-block: sleep through a quarter of that before the first look,
            // so that idle warps do not spend issue slots polling while a long tile is being accumulated
            if (k_blocks * ATOMS >= 32) __nanosleep(k_blocks * ATOMS >= 400 ? 20000u : (unsigned)(k_blocks * ATOMS) * 50u);
            ok = mbar_wait_warp_relaxed(smem_u32(&s_acc_full[acc_stage]), acc_phase, abort_flag, p.watchdog, kWdEpilogue);
            if (!ok) break;
            if (kCluster) {
                // Token chunk c (16 tokens) is finished by slice c % split of the cluster: the others send it their sums, a
                // bulk copy of [16 tokens][32 channels] per warp and chunk, counted on the finisher's barrier.  (CTA pairs: each
                // CTA has 128 channels of its own, and exchanges with the CTA of the same parity.)  The copies' sources are the
                // ring's memory: everything in it has been multiplied.
                // Four-byte stores into the other CTAs went out at 17 bytes per cycle, and the cluster barrier behind them, whose
                // arrivals wait for them, took 2750 cycles: 816 x 16384 x 2048 (8 bits) 35.8 us, so 34.6.
                cluster_wait();                  // the cluster's CTAs exist, their barriers are armed
                waited = true;
                tc_fence_after();
                const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16);
                const int slice = unit & (split - 1), per = (p.bt / 16 + split - 1) >> split_shift;
                for (int c = half, sent = 0; c < p.bt / 16; c += kEpiSets) {
                    const int owner = c & (split - 1);
                    if (t0 + c * 16 >= p.M) break;
                    if (owner == slice) continue;
                    uint32_t r[16];
                    tmem_ld16(taddr + (uint32_t)(c * 16), r);
                    tmem_ld_wait();
                    const uint32_t from = base + (uint32_t)((sent * EPI + warp - 2) * kSumBytes);
#pragma unroll
                    for (int i = 0; i < 16; ++i) sts32(from + (uint32_t)(i * 32 + lane) * 4u, r[i]);
                    fence_proxy_async_smem();
                    __syncwarp();
                    const int sender = slice - (slice > owner ? 1 : 0);
                    const uint32_t to = (uint32_t)owner * CTAS + cta_rank;
                    if (lane == 0)
                        bulk_copy_cluster(cluster_address(smem_sums + (uint32_t)(((sender * per + (c >> split_shift)) * 4 + quad) * kSumBytes), to),
                                          from, (uint32_t)kSumBytes, cluster_address(smem_u32(&s_sums), to));
                    __syncwarp();
                    ++sent;
                }
                tc_fence_before();
                tail = cj;
                break;                           // one tile per cluster
            }
            if constexpr (kStack) {
                // Half g of the tile's lanes holds K slice g of the tile's 64 channels, and only that slice's columns count.  Token
                // chunk c is finished by half c % 2: the other half's warps hand it their sums through shared memory,
                // [finisher][chunk / 2][token][channel].
                tc_fence_after();
                const int g = quad >> 1, chunks = p.tok / 16, per = (chunks + 1) / 2;
                const uint32_t mine = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc_stage * p.bt + g * p.tok);
                int32_t* sums = reinterpret_cast<int32_t*>(gen_base + (smem_sums - base)) + (quad & 1) * 32 + lane;
                for (int c = half; c < chunks; c += kEpiSets) {
                    if (t0 + c * 16 >= p.M) break;
                    if ((c & 1) == g) continue;
                    uint32_t r[16];
                    tmem_ld16(mine + (uint32_t)(c * 16), r);
                    tmem_ld_wait();
                    int32_t* q = sums + (((c & 1) * per + c / 2) * 16) * kStackRows;
#pragma unroll
                    for (int i = 0; i < 16; ++i) q[i * kStackRows] = (int)r[i];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_epi_sync));
                ok = mbar_wait_all(smem_u32(&s_epi_sync), epi_phase, abort_flag, p.watchdog, kWdPartials);
                if (!ok) break;
                for (int i = half, n = 0; i < per; i += kEpiSets, ++n) {
                    const int c = 2 * i + g;
                    if (c >= chunks || t0 + c * 16 >= p.M) break;
                    uint32_t r[16];
                    tmem_ld16(mine + (uint32_t)(c * 16), r);
                    tmem_ld_wait();
                    const int32_t* q = sums + ((g * per + i) * 16) * kStackRows;
#pragma unroll
                    for (int t = 0; t < 16; ++t) r[t] += (uint32_t)q[t * kStackRows];
                    emit(r, n, t0 + c * 16, jq, sw, bj, xpose);
                }
                tc_fence_before();
                break;                           // one tile per CTA (see stacked_applies())
            }
            // K split.  Every slice writes its raw int32 sums to its own block of scratch
            // ([tile][slice][bt tokens][128 channels]: a warp's 32 channels of one token are one 128-byte
            // line, coalesced both ways) and then counts itself in; the CTA that counts last adds the other
            // slices to its own accumulator (still in TMEM) and runs the epilogue.  Nobody waits for anybody.
            const int32_t* part = nullptr;
            const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc_stage * p.bt);
            const int slice = unit & (split - 1);
            if (SPLIT == kSplitScratch && split > 1) {
                tc_fence_after();
                // (in a CTA pair each CTA exchanges and counts its own 128 channels of the tile)
                const int ctile = tile * CTAS + (int)cta_rank;
                int32_t* tile_part = p.partials + (size_t)ctile * (size_t)split * kTileN * (size_t)p.bt + (size_t)(quad * 32 + lane);
                int32_t* mine = tile_part + (size_t)slice * kTileN * (size_t)p.bt;
                for (int c = half * 16; c < p.bt; c += 16 * kEpiSets) {
                    if (t0 + c >= p.M) break;
                    uint32_t r[16];
                    tmem_ld16(taddr + (uint32_t)c, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) __stcg(mine + (size_t)(c + i) * kTileN, (int)r[i]);
                }
                __threadfence();                 // this slice's sums are visible before it is counted
                // rendezvous 1: every epilogue warp has written and fenced its part
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_epi_sync));
                ok = mbar_wait_all(smem_u32(&s_epi_sync), epi_phase, abort_flag, p.watchdog, kWdPartials);
                epi_phase ^= 1u;
                if (!ok) break;
                int* last_slot = &s_last[epi_use & 1];
                if (warp == 2 && lane == 0) {
                    const uint32_t done = atomicAdd(p.counters + ctile, 1u);
                    *last_slot = done == (uint32_t)(split - 1) ? 1 : 0;
                }
                // rendezvous 2: the outcome is written (its slot is reused two tiles later, after both
                // rendezvous of the next tile)
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_epi_sync));
                ok = mbar_wait_all(smem_u32(&s_epi_sync), epi_phase, abort_flag, p.watchdog, kWdPartials);
                epi_phase ^= 1u;
                if (!ok) break;
                const bool last = *reinterpret_cast<volatile int*>(last_slot) != 0;
                ++epi_use;
                if (!last) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if (CTAS == 1) mbar_arrive(smem_u32(&s_acc_empty[acc_stage]));
                        else mbar_arrive_cta(smem_u32(&s_acc_empty[acc_stage]), pair_base);
                    }
                    if (++acc_stage == kAccStages) { acc_stage = 0; acc_phase ^= 1u; }
                    continue;
                }
                __threadfence();                 // the other slices' sums, written through L2
                part = tile_part;
            }
            tc_fence_after();
            if (SPLIT == kUnsplit && staged) {
                // bf16 outputs.  The accumulators are read as MMA-style fragments (a thread: four channels, two adjacent
                // tokens of each 8-token group), scaled in packed pairs, stored token-major into a 1 KB buffer of
                // [16 tokens][32 channels] with two transposing matrix stores, and leave as one tiled bulk store; two
                // buffers alternate so that a chunk is written while the previous one is on its way out.
                // address of "matrix lane>>3, row lane&7" inside a buffer: token (lane>>4)*8 + (lane&7), 16-byte
                // chunk ((lane>>3)&1) [+2 for channels 16..31], chunk index XORed with (token>>1)&3 (64-byte swizzle)
                const uint32_t tok = (uint32_t)((lane >> 4) * 8 + (lane & 7));
                const uint32_t ch = (uint32_t)((lane >> 3) & 1);
                const uint32_t off_a = tok * 64u + ((ch ^ ((tok >> 1) & 3u)) << 4);
                const uint32_t off_b = tok * 64u + (((ch + 2u) ^ ((tok >> 1) & 3u)) << 4);
                const uint32_t buf0 = smem_e + (uint32_t)(warp - 2) * kEpiBytes;
                const bool any_channel = jq < p.N;        // warp-uniform
                if (!ahead) request_constants();
                // The accumulators and steps of a chunk are requested as soon as the chunk before it has been handed to the copy
                // engine.
                uint32_t na[8], nb[8];
                auto request = [&](int c) {
                    tmem_ld_16x256b_x2(taddr + (uint32_t)c, na);                    // channels 0..15 of the quadrant
                    tmem_ld_16x256b_x2(taddr + (16u << 16) + (uint32_t)c, nb);      // channels 16..31
                };
                if (half * 16 < p.bt && t0 + half * 16 < p.M) request(half * 16);
                for (int c = half * 16; c < p.bt; c += 16 * kEpiSets) {
                    const int64_t tc = t0 + c;
                    if (tc >= p.M) break;                // tokens beyond M: nothing to store (warp-uniform)
                    tmem_ld_wait();
                    uint32_t ra[8], rb[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) { ra[i] = na[i]; rb[i] = nb[i]; }
                    const float2 d0 = nd0, d1 = nd1;
                    const uint32_t buf = buf0 + (uint32_t)(store_use % kEpiBuffers) * 1024u;
                    if (store_use >= kEpiBuffers) {      // the store that last used this buffer has read it
                        if (lane == 0) bulk_wait_read<kEpiBuffers - 1>();
                        __syncwarp();
                    }
                    const uint32_t wa0 = scale_pair_bf16(ra[0], ra[1], d0, sw4[0], bj4[0]);
                    const uint32_t wa1 = scale_pair_bf16(ra[2], ra[3], d0, sw4[1], bj4[1]);
                    const uint32_t wa2 = scale_pair_bf16(ra[4], ra[5], d1, sw4[0], bj4[0]);
                    const uint32_t wa3 = scale_pair_bf16(ra[6], ra[7], d1, sw4[1], bj4[1]);
                    stmatrix_x4_trans(buf + off_a, wa0, wa1, wa2, wa3);
                    const uint32_t wb0 = scale_pair_bf16(rb[0], rb[1], d0, sw4[2], bj4[2]);
                    const uint32_t wb1 = scale_pair_bf16(rb[2], rb[3], d0, sw4[3], bj4[3]);
                    const uint32_t wb2 = scale_pair_bf16(rb[4], rb[5], d1, sw4[2], bj4[2]);
                    const uint32_t wb3 = scale_pair_bf16(rb[6], rb[7], d1, sw4[3], bj4[3]);
                    stmatrix_x4_trans(buf + off_b, wb0, wb1, wb2, wb3);
                    fence_proxy_async_smem();            // the buffer, written through the generic proxy, is read by the copy engine
                    __syncwarp();
                    if (lane == 0 && any_channel) {
                        tma_store_2d(&map_y, (int)jq * 2, (int)tc, buf);   // the output map counts bytes along a row
                        bulk_commit();
                    }
                    ++store_use;
                    // (requested only now: with the next chunk's TMEM loads in flight during the arithmetic above, the
                    // main loop beside this epilogue ran slower -- gate/up 46.5 against 44.9 us)
                    if (c + 16 * kEpiSets < p.bt && tc + 16 * kEpiSets < p.M) {
                        request(c + 16 * kEpiSets);
                        request_steps(c + 16 * kEpiSets);
                    }
                }
                tmem_ld_wait();                          // (nothing outstanding unless the loop broke early)
            } else {
            // K split: the other slices' sums of a chunk are requested one chunk ahead of their use, so that their
            // trip through L2 overlaps the arithmetic and stores of the chunk before.
            [[maybe_unused]] int32_t pv_next[16];
            auto fetch_partials = [&](int c) {
#pragma unroll
                for (int i = 0; i < 16; ++i) pv_next[i] = 0;
                for (int rk = 0; rk < split; ++rk) {
                    if (rk == slice) continue;
                    const int32_t* src = part + ((size_t)rk * (size_t)p.bt + (size_t)c) * kTileN;
#pragma unroll
                    for (int i = 0; i < 16; ++i) pv_next[i] += __ldcg(src + (size_t)i * kTileN);
                }
            };
            if (split > 1 && half * 16 < p.bt && t0 + half * 16 < p.M) fetch_partials(half * 16);
            for (int c = half * 16, n = 0; c < p.bt; c += 16 * kEpiSets, ++n) {
                const int64_t tc = t0 + c;
                if (tc >= p.M) break;                    // tokens beyond M: nothing to store (warp-uniform)
                uint32_t r[16];
                tmem_ld16(taddr + (uint32_t)c, r);
                if (split > 1) {
                    int32_t pv[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) pv[i] = pv_next[i];
                    if (c + 16 * kEpiSets < p.bt && tc + 16 * kEpiSets < p.M) fetch_partials(c + 16 * kEpiSets);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) r[i] += (uint32_t)pv[i];
                }
                emit(r, n, tc, jq, sw, bj, xpose);
            }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (CTAS == 1) mbar_arrive(smem_u32(&s_acc_empty[acc_stage]));
                else mbar_arrive_cta(smem_u32(&s_acc_empty[acc_stage]), pair_base);   // the even CTA issues the MMAs
            }
            if (++acc_stage == kAccStages) { acc_stage = 0; acc_phase ^= 1u; }
        }
        // this warp's stores have read their buffers before the CTA gives up its shared memory (the writes themselves
        // are complete when the grid is: no need to wait for them here, which would add their latency to the tail)
        if (SPLIT == kUnsplit && staged && lane == 0) bulk_wait_read<0>();
    } else if (BITS == 8) {
        // ------------------------------------------------- TMA producer, int8 weights
        // (converged warp, one issuing lane: see the activation producer)
        {
            const int total_kb = my_units * k_blocks;
            bool ok = true;
            int stage = 0, kb = 0, unit = unit0;
            uint32_t phase = 0;
            int n0 = n_of(tile_of(unit)) * (kTileN * CTAS) + (int)cta_rank * kTileN;
            int kb0 = kb0_of(unit);
            bool peek = false;
            for (int n = 0; n < total_kb; ++n) {
                ok = mbar_wait_all_lazy(smem_u32(&s_empty[stage]), phase ^ 1u, abort_flag, p.watchdog, kWdProducer, peek);
                if (!ok) break;
                {
                    const int s1 = stage + 1 == p.stages ? 0 : stage + 1;
                    const uint32_t ph1 = s1 == 0 ? phase ^ 1u : phase;
                    peek = n + 1 < total_kb && mbar_test_wait(smem_u32(&s_empty[s1]), ph1 ^ 1u);
                }
                if (elect_one()) {
                    const uint32_t bar = smem_u32(&s_full_tma[stage]);
                    if (CTAS == 1) {
                        mbar_arrive_expect_tx(bar, w_bytes);
                        tma_load_2d(smem_w + stage * w_bytes, &map_w, (kb0 + kb) * kBlockK, n0, bar);
                    } else {
                        if (leader) mbar_arrive_expect_tx(bar, w_bytes * CTAS);
                        tma_load_2d_pair(smem_w + stage * w_bytes, &map_w, (kb0 + kb) * kBlockK, n0, bar);
                    }
                }
                if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                if (++kb == k_blocks) {
                    kb = 0;
                    unit += unit_step;
                    n0 = n_of(tile_of(unit)) * (kTileN * CTAS) + (int)cta_rank * kTileN;
                    kb0 = kb0_of(unit);
                }
            }
            if (!ok && lane == 0) drain_after_abort();
        }
    } else if (warp < kFirstUnpackWarp + 4 * kUnpackSets) {
        // ------------------------------------------------------------ nibble unpack
        // A thread owns one weight row (= one TMEM lane of its warp's quadrant).  The packed tile is
        // 128 rows x 64 bytes with the 64-byte TMA swizzle: 16-byte chunk c of row r sits at
        // chunk c ^ ((r >> 1) & 3), which makes the row-per-thread reads bank-conflict free.
        const int row = (warp & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const int swz = (row >> 1) & 3;
        uint32_t row_off[4];                             // this lane's four 16-byte chunks inside a packed stage
#pragma unroll
        for (int c = 0; c < 4; ++c) row_off[c] = (uint32_t)(row * 64 + ((c ^ swz) << 4));
        // Set `uset` takes the k-blocks whose running index n is congruent to it modulo kUnpackSets,
        // so two k-blocks are in flight per quadrant and one set's store latency hides behind the other.
        const int uset = (warp - kFirstUnpackWarp) >> 2;
        const int total_kb = my_units * k_blocks;
        bool ok = true;
        int ps = uset, ws = uset;                        // ring slots of k-block n, kept incrementally
        uint32_t pph = 0;
        while (ps >= p.stages_p) { ps -= p.stages_p; pph ^= 1u; }
        while (ws >= p.stages_w) ws -= p.stages_w;
        // TMEM slot ws is free once the MMAs of k-block m = n - stages_w have retired, which is the
        // same event that frees that k-block's activation stage: barrier s_empty[m % stages], use
        // number m / stages (stages_w <= stages, so the barrier cannot run a phase ahead of this wait).
        int m = uset - p.stages_w, es = 0;
        uint32_t eph = 0;
        if (m >= 0) es = m;
        while (es >= p.stages) { es -= p.stages; eph ^= 1u; }
        for (int n = uset; n < total_kb && ok; n += kUnpackSets) {
            {
                bool slot_free = false;
                if (p.slot_first && m >= 0) {
                    // A parity wait cannot tell use k of a packed stage from use k - 2.  On a ring of odd length a stage's uses
                    // alternate between the two sets, and a set that has finished k-block n - 2 only knows that k-block
                    // n - 2 - stages_w was multiplied, hence that it had landed.  Where the stage's previous use, k-block
                    // n - stages_p, is later than that, its copy may still be in flight (copies land in any order), and the
                    // wait below would return at once: stale weights, a stage given back twice, copies still under way when
                    // the CTA ends (a launch failure with 64-token tiles on a ring of three).  With the TMEM slot free,
                    // k-block n - stages_w was multiplied, and stages_w <= stages_p.
                    ok = mbar_wait_all(smem_u32(&s_empty[es]), eph, abort_flag, p.watchdog, kWdUnpackEmpty);
                    if (!ok) break;
                    slot_free = true;
                }
                ok = mbar_wait_all(smem_u32(&s_full_p[ps]), pph, abort_flag, p.watchdog, kWdUnpackFull);
                if (!ok) break;
                const uint32_t src = smem_p + (uint32_t)ps * pk_bytes;     // shared-space address of the stage
                const uint32_t w_tmem = tmem_base + lane_addr + (uint32_t)(kAccStages * p.bt + ws * kSlotCols);
#pragma unroll
                for (int h = 0; h < ATOMS; ++h) {
                    uint4 pk[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) pk[c] = lds128(src + h * pk_atom + row_off[c]);
                    if (h == 0 && !slot_free) {
                        // is the TMEM slot free?  (tested now, needed only after the expansion below)
                        slot_free = m < 0 || mbar_test_wait(smem_u32(&s_empty[es]), eph);
                    }
                    uint32_t o[32];                          // 128 codes -> 128 int8 = 32 TMEM columns
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t w[4] = {pk[c].x, pk[c].y, pk[c].z, pk[c].w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t lo = (w[q] << 4) & 0xF0F0F0F0u;   // even channels, 16*code
                            const uint32_t hi = w[q] & 0xF0F0F0F0u;          // odd channels
                            o[8 * c + 2 * q + 0] = lo;   // same (even, odd) channel order as the int8 activations
                            o[8 * c + 2 * q + 1] = hi;
                        }
                    }
                    if (h == ATOMS - 1) {
                        // The packed stage goes back to its producer behind the expansion that consumed what was loaded
                        // from it, and the barrier's address is formed from one expanded word of each load and a run-time
                        // zero: neither the compiler nor the load/store unit may let the arrival overtake the loads (the
                        // ring is always full, a freed stage is overwritten at once; the weight-streaming kernel, which
                        // released its stages right behind the loads, returned wrong sums once in a thousand launches).
                        const uint32_t dep = (o[0] ^ o[9] ^ o[18] ^ o[27]) & p.zero;
                        __syncwarp();
                        if (elect_one()) mbar_arrive(smem_u32(&s_empty_p[ps]) + dep);
                    }
                    if (h == 0) {
                        ok = mbar_wait_all(smem_u32(&s_empty[es]), eph, abort_flag, p.watchdog, kWdUnpackEmpty, slot_free);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    tmem_st32(w_tmem + h * kColsW, o);
                }
                if (!ok) break;
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (elect_one()) {
                    if (CTAS == 1) mbar_arrive(smem_u32(&s_full_w8[ws]));
                    else mbar_arrive_cta(smem_u32(&s_full_w8[ws]), pair_base);
                }
                // (every ring has at least kUnpackSets slots: one subtraction brings an index back into range)
                ps += kUnpackSets;
                if (ps >= p.stages_p) { ps -= p.stages_p; pph ^= 1u; }
                ws += kUnpackSets;
                if (ws >= p.stages_w) ws -= p.stages_w;
                m += kUnpackSets;
                if (m >= kUnpackSets) es += kUnpackSets;
                else if (m >= 0) es = m;
                if (es >= p.stages) { es -= p.stages; eph ^= 1u; }
            }
        }
    } else if (BITS == 4) {
        // ------------------------------------------------- TMA producer, packed weights
        {
            const int total_kb = my_units * k_blocks;
            bool ok = true;
            int ps = 0, kb = 0, unit = unit0;
            uint32_t pph = 0;
            int n0 = n_of(tile_of(unit)) * (kStack ? kStackRows : kTileN * CTAS) + (int)cta_rank * kTileN;
            int kb0 = kb0_of(unit);
            bool peek = false;
            for (int n = 0; n < total_kb; ++n) {
                ok = mbar_wait_all_lazy(smem_u32(&s_empty_p[ps]), pph ^ 1u, abort_flag, p.watchdog, kWdProducer, peek);
                if (!ok) break;
                {
                    const int s1 = ps + 1 == p.stages_p ? 0 : ps + 1;
                    const uint32_t ph1 = s1 == 0 ? pph ^ 1u : pph;
                    peek = n + 1 < total_kb && mbar_test_wait(smem_u32(&s_empty_p[s1]), ph1 ^ 1u);
                }
                if (elect_one()) {
                    const uint32_t bar = smem_u32(&s_full_p[ps]);
                    mbar_arrive_expect_tx(bar, pk_bytes);
                    if constexpr (kStack) tma_load_4d(smem_p + ps * pk_bytes, &map_w, 0, n0, 0, (kb0 + kb) * ATOMS, bar);
                    else {
#pragma unroll
                        for (int h = 0; h < ATOMS; ++h)
                            tma_load_2d(smem_p + ps * pk_bytes + h * pk_atom, &map_w, ((kb0 + kb) * ATOMS + h) * (kBlockK / 2), n0, bar);
                    }
                }
                if (++ps == p.stages_p) { ps = 0; pph ^= 1u; }
                if (++kb == k_blocks) {
                    kb = 0;
                    unit += unit_step;
                    n0 = n_of(tile_of(unit)) * (kStack ? kStackRows : kTileN * CTAS) + (int)cta_rank * kTileN;
                    kb0 = kb0_of(unit);
                }
            }
            if (!ok && lane == 0) drain_after_abort();
        }
    }

    if (kCluster) {
        __syncwarp();
        if (!waited) cluster_wait();
        const bool finishes = warp >= 2 && warp < 2 + EPI && ok && unit0 < num_units;
        if (finishes) ok = mbar_wait_all(smem_u32(&s_sums), 0u, abort_flag, p.watchdog, kWdPartials);
        __syncwarp();
        // "this CTA has its sums": no copy is under way when everybody has said so.  (Pairs say it at the end, behind their last read
        // of tensor memory.)
        if (CTAS == 1) cluster_arrive_relaxed();
        if (finishes && ok) {
            const int quad = warp & 3, half = (warp - 2) >> 2, slice = unit0 & (split - 1);
            const int tile = tile_of(unit0);
            const int64_t jq = (int64_t)n_of(tile) * (kTileN * CTAS) + (int64_t)cta_rank * kTileN + quad * 32;
            const int64_t t0 = (int64_t)m_of(tile) * p.bt;
            const int per = (p.bt / 16 + split - 1) >> split_shift;
            const int32_t* sums = reinterpret_cast<const int32_t*>(gen_base + (smem_sums - base)) + lane;
            uint8_t* xpose = gen_base + (smem_e - base) + (warp - 2) * kEpiBytes;
            tc_fence_after();
            for (int i = half, n = 0; i < per; i += kEpiSets, ++n) {
                const int c = (i << split_shift) + slice;
                const int64_t tc = t0 + c * 16;
                if (c * 16 >= p.bt || tc >= p.M) break;
                uint32_t r[16];
                tmem_ld16(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(c * 16), r);
                tmem_ld_wait();
                for (int k = 0; k < split - 1; ++k) {
                    const int32_t* q = sums + (size_t)((k * per + i) * 4 + quad) * (kSumBytes / 4);
#pragma unroll
                    for (int t = 0; t < 16; ++t) r[t] += (uint32_t)q[t * 32];
                }
                emit(r, n, tc, jq, tail.x, tail.y, xpose);
            }
        }
    }

    // ------------------------------------------------------------------ teardown
    tc_fence_before();
    __syncthreads();
    // Nobody leaves while its own copies may still be under way.  Pairs free their tensor memory together, with both CTAs present and
    // neither reading it any more, and neither leaves while the other may still signal it.
    if (CTAS == 2) cluster_sync_all();
    else if (kCluster) cluster_wait();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc<CTAS>(tmem_base, (uint32_t)p.tmem_cols);
    }
}

// ---- host side ---------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static const EncodeTiledFn fn = [] {             // (looked up once, by one of the threads that come first; the others wait)
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        const bool ok = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) == cudaSuccess &&
                        q == cudaDriverEntryPointSuccess;
        return ok ? reinterpret_cast<EncodeTiledFn>(sym) : nullptr;
    }();
    return fn;
}

// 2-D byte tensor [rows, row_bytes] (row pitch = pitch_bytes, 0 = row_bytes), box [box_rows, box_bytes].
bool encode_2d(CUtensorMap* map, const void* ptr, uint64_t row_bytes, uint64_t rows, uint32_t box_bytes,
               uint32_t box_rows, CUtensorMapSwizzle swizzle, uint64_t pitch_bytes = 0) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {row_bytes, rows};
    const cuuint64_t strides[1] = {pitch_bytes ? pitch_bytes : row_bytes};
    const cuuint32_t box[2] = {box_bytes, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool encode_tiled(CUtensorMap* map, CUtensorMapDataType dt, uint32_t rank, const void* ptr, const uint64_t* dims,
                  const uint64_t* strides_bytes, const uint32_t* box, CUtensorMapSwizzle swizzle) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t d[5], st[5];
    cuuint32_t b[5], es[5];
    for (uint32_t i = 0; i < rank; ++i) { d[i] = dims[i]; b[i] = box[i]; es[i] = 1; }
    for (uint32_t i = 0; i + 1 < rank; ++i) st[i] = strides_bytes[i];
    return fn(map, dt, rank, const_cast<void*>(ptr), d, st, b, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {
// Rows of whole atoms as [atom][K slice][row][byte]: a stacked tile's stage is one copy.
bool encode_stacked(CUtensorMap* map, const void* ptr, uint64_t row_bytes, uint64_t rows, uint32_t atom_bytes, uint32_t box_rows, uint32_t atoms,
                    CUtensorMapSwizzle swizzle) {
    const uint64_t slice_bytes = row_bytes / kStackSlices;
    const uint64_t dims[4] = {atom_bytes, rows, kStackSlices, slice_bytes / atom_bytes}, strides[3] = {row_bytes, slice_bytes, atom_bytes};
    const uint32_t box[4] = {atom_bytes, box_rows, kStackSlices, atoms};
    return encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, ptr, dims, strides, box, swizzle);
}
}  // namespace

fq_status build_weight_tmap(Weights& W) {
    W.tmap_valid = false;
    if (W.N == 0) return FQ_OK;
    const bool ok = W.bits == 4
                        ? encode_2d(&W.tmap, W.codes, (uint64_t)W.K / 2, (uint64_t)W.N, kBlockK / 2, kTileN,
                                    CU_TENSOR_MAP_SWIZZLE_64B)
                        : encode_2d(&W.tmap, W.codes, (uint64_t)W.K, (uint64_t)W.N, kBlockK, kTileN,
                                    CU_TENSOR_MAP_SWIZZLE_128B);
    if (!ok) return FQ_ERR_CUDA;
    W.tmap_valid = true;
    build_stream_tmap(W);       // optional second view (short batches); shapes it does not fit go without
    return FQ_OK;
}

namespace {

template <int BITS, int CTAS, int SPLIT, int ATOMS = 1, int EPI = kEpiWarps>
fq_status launch_variant(const CUtensorMap& map_a, const CUtensorMap& map_w, const CUtensorMap& map_y, const Params& p,
                         int grid, size_t smem, int cluster, cudaStream_t stream, bool* refused) {
    auto kern = gemm_tcgen05_kernel<BITS, CTAS, SPLIT, ATOMS, EPI>;
    if (ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem) != cudaSuccess) return FQ_ERR_CUDA;
    const cudaError_t e = launch_pdl(kern, (unsigned)grid, (unsigned)gemm_threads(BITS, EPI), smem, stream,
                                     (unsigned)cluster, map_a, map_w, map_y, p);
    *refused = cluster > 1 && cluster_refused(e);
    return e == cudaSuccess ? FQ_OK : FQ_ERR_CUDA;
}

}  // namespace

int cluster_capacity(int ctas) {
    static std::mutex mutex;
    static int known[64][3];                         // 0: not asked yet, else capacity + 1
    const int defaults[3] = {74, 36, 14}, i = ctas == 2 ? 0 : (ctas == 4 ? 1 : 2);
    int dev = 0;
    if (device_cc_major() != 10 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        (void)cudaGetLastError();
        return defaults[i];
    }
    std::lock_guard<std::mutex> lock(mutex);
    if (known[dev][i] == 0) {
        const auto kern = gemm_tcgen05_kernel<8, 1, kSplitCluster, 1, kEpiWarps>;
        const size_t smem = 224 * 1024;              // one CTA per SM
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)ctas, 1, 1);
        cfg.blockDim = dim3((unsigned)gemm_threads(8, kEpiWarps), 1, 1);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)ctas; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        if (ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        known[dev][i] = n + 1;
    }
    return known[dev][i] - 1;
}

// A launch that splits K counts the finished slices of every tile in counters at the head of the scratch.
// They are cleared here, by a memset node enqueued AHEAD of the call's first kernel (between the prologue
// and the GEMM it would break the programmatic overlap of the two): each call starts from zero whatever an
// earlier call -- even one that gave up on an expired wait -- left there, and nothing in the weight handle
// changes at run time.
fq_status gemm_prepare(int64_t M, const Weights& W, void* scratch, size_t scratch_bytes, cudaStream_t stream) {
    if (M <= 0 || W.N == 0 || scratch == nullptr || gemm_stream_applies(M, W)) return FQ_OK;
    const GemmPlan plan = plan_call(M, W.N, W.K, W.bits, device_sm_count(), scratch_bytes, cluster_capacity);
    if (plan.split <= 1 || plan.cluster) return FQ_OK;
    return cudaMemsetAsync(scratch, 0, kCounterBytes, stream) == cudaSuccess ? FQ_OK : FQ_ERR_CUDA;
}

fq_status launch_gemm(const int8_t* a8, int64_t M, const Weights& W, int acc_shift, const GemmOut& out, void* scratch,
                      size_t scratch_bytes, cudaStream_t stream) {
    if (M == 0 || W.N == 0) return FQ_OK;
    if (gemm_stream_applies(M, W))
        return launch_gemm_stream(a8, M, W, acc_shift, out, stream) == cudaSuccess ? FQ_OK : FQ_ERR_CUDA;
    return launch_gemm_tcgen05(a8, M, W, acc_shift, out, scratch, scratch_bytes, stream);
}

size_t gemm_scratch_bytes(int64_t M, int64_t N, int64_t K, int bits) {
    if (M <= 0 || N <= 0 || K <= 0) return 0;
    // (asked for whether or not this device holds the clusters that would do without: a caller sizes its workspace once)
    return plan_gemm(M, N, K, bits, device_sm_count(), (size_t)-1, false, cluster_capacity).scratch;
}

namespace {

int no_clusters(int) { return 0; }

// *refused: the device did not take the launch's clusters, nothing was enqueued.
fq_status launch_planned(const int8_t* a8, int64_t M, const Weights& W, int acc_shift, const GemmOut& out, void* scratch,
                         size_t scratch_bytes, int (*held)(int), cudaStream_t stream, bool* refused) {
    Params p{};
    p.M = M; p.N = W.N; p.K = W.K;
    const int sms = device_sm_count();
    const GemmPlan plan = plan_call(M, W.N, W.K, W.bits, sms, scratch ? scratch_bytes : 0, held);
    const int bt = plan.bt, tok = bt / plan.stack, ctas = plan.ctas, split = plan.split;
    p.split = split;
    p.counters = static_cast<uint32_t*>(scratch);            // cleared by gemm_prepare()
    p.partials = reinterpret_cast<int32_t*>(static_cast<uint8_t*>(scratch) + kCounterBytes);
    p.delta_vec = (reinterpret_cast<uintptr_t>(out.a_delta) & 15u) == 0 ? 1 : 0;
    p.bt = bt;
    p.tok = tok;
    p.m_tiles = (int)((M + tok - 1) / tok);
    const int n_step = plan.stack > 1 ? kStackRows : kTileN * ctas;
    p.n_tiles = (int)((W.N + n_step - 1) / n_step);
    // Bands of 8 token tiles once the batch is long enough for the order to matter: a wave of 148 CTAs (74 pairs)
    // then covers 8 token tiles x 18 (9) channel tiles, close to the square that minimises the bytes it shares.
    p.band = p.m_tiles >= 16 ? 8 : p.m_tiles;
    p.acc_shift = acc_shift;
    p.w_scale = W.w_scale;
    p.bias = W.bias;
    p.out = out;
    p.watchdog = watchdog_device_ptr();
    if (!p.watchdog) return FQ_ERR_CUDA;
    const GemmRings rings = gemm_rings(plan, W.bits, W.K);
    if (!rings.fits) return FQ_ERR_UNSUPPORTED;      // (no tile comes here)
    const int atoms = rings.atoms;
    p.stages = rings.stages; p.stages_p = rings.stages_p; p.stages_w = rings.stages_w;
    p.slot_first = rings.slot_first ? 1 : 0;
    p.tmem_cols = rings.tmem_cols;
    const size_t smem = rings.smem;

    // each CTA of a pair loads its own half of the token tile
    CUtensorMap map_a;
    CUtensorMap map_stacked;
    if (plan.stack > 1) {
        if (!encode_stacked(&map_stacked, W.codes, (uint64_t)W.K / 2, (uint64_t)W.N, kBlockK / 2, kStackRows, (uint32_t)atoms, CU_TENSOR_MAP_SWIZZLE_64B) ||
            !encode_stacked(&map_a, a8, (uint64_t)W.K, (uint64_t)M, kBlockK, (uint32_t)tok, (uint32_t)atoms, CU_TENSOR_MAP_SWIZZLE_128B))
            return FQ_ERR_CUDA;
    } else if (!encode_2d(&map_a, a8, (uint64_t)W.K, (uint64_t)M, kBlockK, (uint32_t)(bt / ctas), CU_TENSOR_MAP_SWIZZLE_128B)) {
        return FQ_ERR_CUDA;
    }
    const CUtensorMap& map_w = plan.stack > 1 ? map_stacked : W.tmap;

    // bf16 outputs of an unsplit launch leave through tiled bulk stores of [16 tokens x 32 channels] (64-byte rows,
    // 64-byte swizzle in shared memory); the copy engine clips what lies beyond M tokens or N channels
    CUtensorMap map_y;
    memset(&map_y, 0, sizeof(map_y));
    if (out.acc == nullptr && out.yt == FQ_BF16 && split == 1 && plan.stack == 1 &&
        !encode_2d(&map_y, out.y, (uint64_t)W.N * 2, (uint64_t)M, 64, 16, CU_TENSOR_MAP_SWIZZLE_64B, (uint64_t)out.ldy * 2))
        return FQ_ERR_CUDA;

    const int num_units = p.m_tiles * p.n_tiles * split;       // a K split makes `split` units of every tile
    const int max_units = sms / ctas;
    const int clusters = num_units < max_units ? num_units : max_units;
    const int grid = clusters * ctas;
    p.cluster_shift = ctas == 2 ? 1 : 0;
    p.unit_step = clusters;
    p.units_q = num_units / clusters;
    p.units_rem = num_units % clusters;
    p.kb_per = (int)(((W.K / plan.stack + kBlockK - 1) / kBlockK + atoms - 1) / atoms) / split;      // stages per unit; the planner only picks splits that divide it
    p.split_shift = split == 1 ? 0 : (split == 2 ? 1 : (split == 4 ? 2 : (split == 8 ? 3 : 4)));

    const int cluster = plan.cluster ? split * ctas : ctas;
    auto go = [&](auto bits, auto pair, auto atoms_c) -> fq_status {
        constexpr int B = decltype(bits)::value, C = decltype(pair)::value, A = decltype(atoms_c)::value;
        if constexpr (B == 4 && A > 1)
            if (plan.stack > 1) return launch_variant<B, C, kStacked, A>(map_a, map_w, map_y, p, grid, smem, cluster, stream, refused);
        if constexpr (B == 8)
            if (plan.epi == kEpiWarpsMany) return launch_variant<B, C, kUnsplit, A, kEpiWarpsMany>(map_a, map_w, map_y, p, grid, smem, cluster, stream, refused);
        if (split == 1) return launch_variant<B, C, kUnsplit, A>(map_a, map_w, map_y, p, grid, smem, cluster, stream, refused);
        if (plan.cluster) return launch_variant<B, C, kSplitCluster, A>(map_a, map_w, map_y, p, grid, smem, cluster, stream, refused);
        return launch_variant<B, C, kSplitScratch, A>(map_a, map_w, map_y, p, grid, smem, cluster, stream, refused);
    };
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    using I4 = std::integral_constant<int, 4>;
    using I8 = std::integral_constant<int, 8>;
    if (W.bits == 4 && ctas == 2) return launch_variant<4, 2, kUnsplit>(map_a, map_w, map_y, p, grid, smem, cluster, stream, refused);
    if (W.bits == 4) return atoms == 4 ? go(I4(), I1(), I4()) : (atoms == 2 ? go(I4(), I1(), I2()) : go(I4(), I1(), I1()));
    return ctas == 2 ? go(I8(), I2(), I1()) : go(I8(), I1(), I1());
}

}  // namespace

fq_status launch_gemm_tcgen05(const int8_t* a8, int64_t M, const Weights& W, int acc_shift, const GemmOut& out,
                              void* scratch, size_t scratch_bytes, cudaStream_t stream) {
    if (M == 0 || W.N == 0) return FQ_OK;
    if (!W.tmap_valid) return FQ_ERR_CUDA;
    bool refused = false;
    const fq_status st = launch_planned(a8, M, W, acc_shift, out, scratch, scratch_bytes, cluster_capacity, stream, &refused);
    // (without scratch: gemm_prepare() cleared the counters of the plan that was refused, if any)
    if (refused && gemm_stream_applies(M, W, no_clusters))
        return launch_gemm_stream(a8, M, W, acc_shift, out, stream) == cudaSuccess ? FQ_OK : FQ_ERR_CUDA;
    return refused ? launch_planned(a8, M, W, acc_shift, out, nullptr, 0, no_clusters, stream, &refused) : st;
}

}  // namespace fq
