// Streaming variant of the runtime prologue (Alg. 1 runtime half lines 1-2, Eq. 5) for longer
// batches: same arithmetic, bit for bit, as transform_quantize_kernel, but tokens reach the
// SM through a TMA-fed shared-memory ring so that many rows are in flight per SM regardless
// of register pressure, and the floating-point work is issued as packed f32x2 instructions.
//
//   - One persistent CTA of 512 threads per SM, split into row groups of `gw` warps; a
//     group owns one token at a time, a thread owns E = 64 (or 32) consecutive channels.
//   - A token row is fetched as a 3-D tiled TMA box {128 bytes, K*e/128, 1} with the 128-byte
//     swizzle, which makes the per-thread 64..256-byte reads bank-conflict free.  The per-
//     channel multiplier is staged once in shared memory with the same swizzle.
//   - Each group runs `depth` slots: the group barrier that exchanges the per-warp maxima also
//     proves that every warp has finished reading the slot, so the group's leader refills it
//     right there -- no separate "empty" barrier.
//   - Register layout: float2 v[p] = (channel p, channel p + E/2).  Butterflies with stride
//     below E/2 then act on both halves at once (fadd2 / ffma2 by -1: each lane of a packed
//     instruction is one IEEE binary32 operation, so the rounding is that of the scalar
//     network); the stride-E/2 stage works inside the pairs; strides E..block/2 go across
//     lanes (one shuffle per value, one packed FMA per pair).
//   - A thread's 64 one-byte codes are a run of 64 bytes, so a warp-wide 16-byte store would touch 32 sectors and fill half
//     of each.  They go through 2 KB of shared memory per warp instead and leave as one bulk store of 32 runs (64-byte
//     swizzle: the 16-byte pieces of 8 lanes lie in different banks).  16384 x 8192, 8-bit codes, blocks of 64, 128 and 256
//     channels: 79.6, 83.6 and 93.3 us with direct stores, 59.6 (the copy rate), 70.3 and 81.0 now.  Runs of 32 and 16 bytes
//     (4-bit codes, 32 channels per thread) gain nothing (57.0 and 59.0 us; gated 1-5 % slower) and are stored directly.
//     640 threads at 96 registers: 58.9, 68.4 and 81.2 us, and slower for short rows.
#include <cuda_bf16.h>
#include <float.h>
#include <string.h>

#include "fq_common.cuh"
#include "ptx_sm100.cuh"
#include "act_common.cuh"

namespace fq {
namespace {

constexpr int kThreads = kRingThreads;
// Threads of a CTA.  (1024 threads of 32 channels -- twice the warps at 64 registers -- measured
// slower than 512 threads of 64 channels for 4-bit output: 0.65 against 0.75 of the copy rate at K = 8192, block 128;
// the extra cross-lane butterfly stage costs more than the occupancy returns.)
constexpr int kMaxSlots = kRingMaxSlots;

// 128-byte swizzle of a byte offset inside a 1024-byte aligned region.
__device__ __forceinline__ uint32_t swz128(uint32_t off) { return off ^ (((off >> 7) & 7u) << 4); }

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}
// The same box as far as L2 only.
__device__ __forceinline__ void prefetch_row(const CUtensorMap* map, int line, int row) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(line), "r"(row)
                 : "memory");
}
// Tiled bulk STORE shared -> global; what lies beyond the tensor's extent is clipped by the copy engine.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, int c0, int c1, int c2, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void sts128(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// Group barrier that also ANDs a predicate over the group (ids 1..15, count a multiple of 32).
__device__ __forceinline__ bool group_barrier_and(int id, int count, bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 q, %3, 0;\n\t"
        "bar.red.and.pred p, %1, %2, q;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(id), "r"(count), "r"((uint32_t)pred)
        : "memory");
    return r != 0;
}
// max(m, |x|, |y|) in one instruction (3-input max of sm_100).
__device__ __forceinline__ float max3_abs(float m, float x, float y) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(fabsf(x)), "f"(fabsf(y)));
    return r;
}
// A thread's slice is 64, 128 or 256 contiguous bytes of a swizzled, 1024-byte aligned region.
// Inside one 128-byte line the swizzled address of 16-byte piece i is (address of piece 0) ^ (i << 4),
// so one address per line (line0, line1 = swizzled starts of the slice's lines) is all a thread keeps.
// Addresses are 32-bit shared-window addresses and the loads explicit ld.shared: through generic
// pointers the same reads cost 64-bit address arithmetic (about one extra instruction per element).
__device__ __forceinline__ uint32_t piece(uint32_t line0, uint32_t line1, int i) {
    return (i < 8 ? line0 : line1) ^ (uint32_t)((i & 7) << 4);
}
// (Not volatile, so that the compiler may batch and hoist them; the caller pins their addresses
// behind the barrier wait that makes the data valid, see `pin_after_wait`.)
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
// An empty volatile statement that "rewrites" an address: loads through that address cannot be
// moved above it, and it cannot be moved above the (volatile) barrier wait before it.
__device__ __forceinline__ void pin_after_wait(uint32_t& addr) { asm volatile("" : "+r"(addr) : : "memory"); }
// Volatile variant for the multiplier: kept in program order, interleaved with the multiplies that
// consume it (hoisting all of them too would not fit the register file).
__device__ __forceinline__ float4 lds128f_ordered(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ float4 lds128f(uint32_t addr) {
    float4 v;
    asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}

struct RingParams {
    int64_t rows;
    int K;
    float cnorm, qmax, clip_ratio;
    const float* mult;
    int mult_after;    // 1: multiply by cnorm before the butterflies and by mult after them (fold-after sites)
    uint8_t* codes;
    float* delta;
    int gw;            // warps per row group (power of two)
    int depth;         // ring slots per group
    uint32_t slot_bytes;
    uint32_t stage_off; // where the codes of the warps wait for their bulk store
    uint32_t g_bytes;  // bytes of the multiplier stage (0 if no multiplier)
    uint32_t up_bytes; // gated sites: the row's up half starts so many bytes into its slot, and at this line of the row
    int up_line;
    int gate_kind;
    int mult_ready;    // the multiplier may be read before the kernel ahead has finished
    uint32_t* watchdog;
};

// GATED: a row is [gate | up], 2K bf16 channels in one slot; the transform's input is act(gate) * up, formed as the row is
// read from shared memory.
template <typename XT, int FMT, bool CLAMP, int E, int BLOCK, bool AFTER, bool GATED>
__global__ void __launch_bounds__(kThreads, 1)
transform_quantize_ring_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_c,
                               const RingParams p) {
    constexpr int H = E / 2;                       // channels per half: v[i] = (channel i, channel i + H)
    constexpr bool kStaged = FMT != 0 && E == 64;  // the codes leave through bulk stores
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t s_full[kMaxSlots];
    __shared__ float s_part[2][32];
    __shared__ int s_abort;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ngroups = (kThreads / 32) / p.gw;
    const int group = warp / p.gw;
    const int wg = warp - group * p.gw;
    const int col0 = (wg * 32 + lane) * E;
    const bool col_ok = col0 < p.K;
    const bool leader = wg == 0 && lane == 0;
    volatile int* abort_flag = &s_abort;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t slots_off = (p.g_bytes + 1023u) & ~1023u;

    if (tid == 0) {
        s_abort = 0;
        for (int s = 0; s < ngroups * p.depth; ++s) mbar_init(smem_u32(&s_full[s]), 1);
        fence_mbarrier_init();
        fence_proxy_async_smem();
    }
    __syncthreads();                 // barriers initialised before any copy is issued
    auto stage_multiplier = [&]() {
        if (p.mult == nullptr) return;
        // Stage the multiplier in the order the registers hold a slice: inside every thread slice (E floats)
        // the entries are interleaved as (g[q], g[q + H]) pairs, so that one 16-byte read yields two ready
        // operands of the packed multiply (no register moves to pair them up), and the 16-byte pieces are
        // XOR-swizzled by the slice index, so that the slice-per-thread reads are bank-conflict free.
        for (int i = tid * 4; i < p.K; i += kThreads * 4) {
            const float4 g4 = ld_global_f4(p.mult + i);
            const float gv[4] = {g4.x, g4.y, g4.z, g4.w};
            const uint32_t slice = (uint32_t)i / E;
            const uint32_t key = (slice & 7u) << 4;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t q = ((uint32_t)i % E) + k;                       // position inside the slice
                const uint32_t off = q < H ? q * 8u : (q - H) * 8u + 4u;         // pair q (low half) or q - H (high half)
                *reinterpret_cast<float*>(gen + ((slice * (E * 4u) + off) ^ key)) = gv[k];
            }
        }
    };
    if (p.mult_ready) stage_multiplier();
    // The group's first row comes as far as L2 while the kernel ahead still runs.  (All rows of the ring: no better for short
    // batches and slower for long ones, 2368 x 8192 13.6 us against 11.1; none: 11.5, and 816 x 2048 3.1 against 2.95.)
    if (leader && group * (int)gridDim.x + (int)blockIdx.x < (int)p.rows) {
        prefetch_row(&map_x, 0, group * (int)gridDim.x + (int)blockIdx.x);
        if (GATED) prefetch_row(&map_x, p.up_line, group * (int)gridDim.x + (int)blockIdx.x);
    }
    griddep_wait();                  // the kernel before this one may still be writing x (or reading codes)
    griddep_launch_dependents();

    const int first = group * (int)gridDim.x + (int)blockIdx.x;   // rows < 2^31 (checked by the launcher)
    const int step = (int)gridDim.x * ngroups;
    const int rows = (int)p.rows;
    const uint32_t tx = (uint32_t)p.K * (uint32_t)sizeof(XT) * (GATED ? 2u : 1u);
    const uint32_t slot0 = base + slots_off + (uint32_t)(group * p.depth) * p.slot_bytes;
    uint64_t* full0 = &s_full[group * p.depth];

    // The first rows are requested before the multiplier is staged, so that their flight time
    // overlaps the staging loop.
    int issued = 0;          // rows requested by this group's leader
    if (leader) {
        for (int d = 0; d < p.depth; ++d) {
            const int r = first + d * step;
            if (r < rows) {
                mbar_arrive_expect_tx(smem_u32(&full0[d]), tx);
                tma_load_3d(slot0 + d * p.slot_bytes, &map_x, 0, 0, r, smem_u32(&full0[d]));
                if (GATED) tma_load_3d(slot0 + d * p.slot_bytes + p.up_bytes, &map_x, 0, p.up_line, r, smem_u32(&full0[d]));
                ++issued;
            }
        }
    }
    if (!p.mult_ready) stage_multiplier();
    __syncthreads();

    // swizzled starts of the (up to two) 128-byte lines of this thread's slices
    const uint32_t xs0 = swz128((uint32_t)col0 * (uint32_t)sizeof(XT));
    const uint32_t xs1 = swz128((uint32_t)col0 * (uint32_t)sizeof(XT) + 128u);
    const uint32_t gkey = (uint32_t)((col0 / E) & 7) << 4;
    const uint32_t g0 = base + (((uint32_t)col0 * 4u) ^ gkey);
    const uint32_t g1 = base + (((uint32_t)col0 * 4u + 128u) ^ gkey);
    const bool warp_ok = __all_sync(0xffffffffu, col_ok);   // the usual case: no lane of the warp is past K
    const float2 neg1 = make_float2(-1.0f, -1.0f);

    const uint32_t stage = base + p.stage_off + (uint32_t)(warp * 32 * E);
    const uint32_t stage_line = stage + (uint32_t)(lane * E);
    const uint32_t stage_key = (uint32_t)((lane >> 1) & 3);

    int n = 0, d = 0;
    uint32_t ph = 0;
    for (int row = first; row < rows; row += step, ++n) {
        bool ok = mbar_wait_all(smem_u32(&full0[d]), ph, abort_flag, p.watchdog, 0x100u);   // every lane polls: cheaper than one lane + broadcast

        float2 v[H];
        const uint32_t slot = base + slots_off + (uint32_t)(group * p.depth + d) * p.slot_bytes;
        uint32_t x0 = slot + xs0, x1 = slot + xs1;
        pin_after_wait(x0);
        pin_after_wait(x1);
        auto load_row = [&]() {
            auto widen = [](const uint4& lo, const uint4& hi, float2* out) {      // 8 pairs (channel of lo, channel of hi)
                const uint32_t wl[4] = {lo.x, lo.y, lo.z, lo.w}, wh[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    out[2 * j + 0] = make_float2(__uint_as_float(wl[j] << 16), __uint_as_float(wh[j] << 16));
                    out[2 * j + 1] = make_float2(__uint_as_float(wl[j] & 0xffff0000u), __uint_as_float(wh[j] & 0xffff0000u));
                }
            };
            if (GATED) {
#pragma unroll
                for (int i = 0; i < H / 8; ++i) {
                    float2 u[8];
                    widen(lds128(piece(x0, x1, i)), lds128(piece(x0, x1, i + H / 8)), v + 8 * i);
                    widen(lds128(piece(x0 + p.up_bytes, x1 + p.up_bytes, i)), lds128(piece(x0 + p.up_bytes, x1 + p.up_bytes, i + H / 8)), u);
                    gate_product<8>(v + 8 * i, u, p.gate_kind);
                }
            } else if (sizeof(XT) == 2) {
                // bf16: 8 channels per 16-byte piece; pieces [0, H/8) are the low half, the rest the high half
#pragma unroll
                for (int i = 0; i < H / 8; ++i) {
                    widen(lds128(piece(x0, x1, i)), lds128(piece(x0, x1, i + H / 8)), v + 8 * i);
                }
            } else {
#pragma unroll
                for (int i = 0; i < H / 4; ++i) {
                    const float4 lo = lds128f(piece(x0, x1, i));
                    const float4 hi = lds128f(piece(x0, x1, i + H / 4));
                    v[4 * i + 0] = make_float2(lo.x, hi.x);
                    v[4 * i + 1] = make_float2(lo.y, hi.y);
                    v[4 * i + 2] = make_float2(lo.z, hi.z);
                    v[4 * i + 3] = make_float2(lo.w, hi.w);
                }
            }
            if (!AFTER && p.mult != nullptr) {
#pragma unroll
                for (int i = 0; i < H / 2; ++i) {           // one piece = the multipliers of pairs 2i and 2i + 1
                    const float4 q = lds128f_ordered(piece(g0, g1, i));
                    v[2 * i + 0] = f2_mul(v[2 * i + 0], make_float2(q.x, q.y));
                    v[2 * i + 1] = f2_mul(v[2 * i + 1], make_float2(q.z, q.w));
                }
            } else {
                const float2 c2 = make_float2(p.cnorm, p.cnorm);
#pragma unroll
                for (int i = 0; i < H; ++i) v[i] = f2_mul(v[i], c2);
            }
        };
        // Warp-uniform fast path: with a per-lane `col_ok` the zero fill below is compiled into
        // predicated instructions that every row pays for (half an instruction per element).
        if (warp_ok) {
            load_row();
        } else if (col_ok) {
            load_row();
        } else {
#pragma unroll
            for (int i = 0; i < H; ++i) v[i] = make_float2(0.0f, 0.0f);
        }

        // strides 1 .. H/2: both halves at once
#pragma unroll
        for (int h = 1; h < H; h <<= 1) {
            if (h < BLOCK) {
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    if ((i & h) == 0) {
                        const float2 a = v[i], b = v[i + h];
                        v[i] = f2_add(a, b);
                        v[i + h] = f2_fma(b, neg1, a);       // a - b, exact product
                    }
                }
            }
        }
        // stride H: inside each pair
        if (H < BLOCK) {
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const float a = v[i].x, b = v[i].y;
                v[i] = make_float2(__fadd_rn(a, b), __fsub_rn(a, b));
            }
        }
        // strides E .. BLOCK/2: partner lane = lane ^ (h / E); upper lane keeps partner - own
#pragma unroll
        for (int h = E; h < BLOCK; h <<= 1) {
            const int lm = h / E;
            const float s = (lane & lm) ? -1.0f : 1.0f;
            const float2 s2 = make_float2(s, s);
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const float2 q = make_float2(__shfl_xor_sync(0xffffffffu, v[i].x, lm),
                                             __shfl_xor_sync(0xffffffffu, v[i].y, lm));
                v[i] = f2_fma(v[i], s2, q);
            }
        }

        // fold-after sites: the diagonal sits behind the rotation (z = D^o R x)
        if (AFTER && col_ok) {
#pragma unroll
            for (int i = 0; i < H / 2; ++i) {
                const float4 q = lds128f_ordered(piece(g0, g1, i));
                v[2 * i + 0] = f2_mul(v[2 * i + 0], make_float2(q.x, q.y));
                v[2 * i + 1] = f2_mul(v[2 * i + 1], make_float2(q.z, q.w));
            }
        }

        float m = 0.0f;
#pragma unroll
        for (int i = 0; i < H; ++i) m = max3_abs(m, v[i].x, v[i].y);
        m = warp_max_nonneg(m);
        if (p.gw > 1) {
            if (lane == 0) s_part[n & 1][warp] = m;
            ok = group_barrier_and(1 + group, p.gw * 32, ok);
            m = (lane < p.gw) ? s_part[n & 1][group * p.gw + lane] : 0.0f;
            m = warp_max_nonneg(m);
        }
        if (!ok) break;

        // every warp of the group has read the slot: refill it with the row `depth` steps ahead
        if (leader) {
            const int nr = row + p.depth * step;
            if (nr < rows) {
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(smem_u32(&full0[d]), tx);
                tma_load_3d(slot0 + d * p.slot_bytes, &map_x, 0, 0, nr, smem_u32(&full0[d]));
                if (GATED) tma_load_3d(slot0 + d * p.slot_bytes + p.up_bytes, &map_x, 0, p.up_line, nr, smem_u32(&full0[d]));
                ++issued;
            }
        }

        float dl = __fdiv_rn(__fmul_rn(p.clip_ratio, m), p.qmax);
        float inv;
        if (dl >= FLT_MIN) {
            inv = __fdiv_rn(1.0f, dl);
        } else {
            dl = 0.0f;
            inv = 0.0f;
        }
        // codes: channel i from .x, channel i + H from .y
        constexpr int kPer = FMT == 0 ? 8 : 4;               // codes per 32-bit word
        constexpr int kWords = H / kPer;                     // words per half
        const float2 inv2 = make_float2(inv, inv);
        uint32_t wlo[kWords], whi[kWords];
#pragma unroll
        for (int j = 0; j < kWords; ++j) {
            uint32_t bl[kPer], bh[kPer];
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                float2 t = f2_mul(v[code_index<FMT>(j, i)], inv2);
                if (CLAMP) {
                    t.x = fminf(fmaxf(t.x, -p.qmax), p.qmax);
                    t.y = fminf(fmaxf(t.y, -p.qmax), p.qmax);
                }
                // t * 1 + magic as an explicit packed FMA (exact product, so it rounds like the add).  A
                // packed multiply feeding a packed ADD was observed to be fused into one packed FMA by the
                // assembler, which rounds exact ties differently.
                t = f2_fma(t, make_float2(1.0f, 1.0f), make_float2(12582912.0f, 12582912.0f));
                bl[i] = __float_as_uint(t.x);
                bh[i] = __float_as_uint(t.y);
            }
            wlo[j] = pack_word<FMT>(bl);
            whi[j] = pack_word<FMT>(bh);
        }
        // low-half words then high-half words are consecutive channels: one contiguous store run
        uint32_t w[2 * kWords];
#pragma unroll
        for (int j = 0; j < kWords; ++j) { w[j] = wlo[j]; w[kWords + j] = whi[j]; }
        if (kStaged) {
            if (lane == 0) bulk_wait_read<0>();          // the row before this one has left the buffer
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 2 * kWords / 4; ++j)
                sts128(stage_line + (((uint32_t)j ^ stage_key) << 4), make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]));
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && wg * 32 * E < p.K) {
                tma_store_3d(&map_c, 0, wg * 32, row, stage);
                bulk_commit();
                if (wg == 0) p.delta[row] = dl;
            }
        } else if (col_ok) {
            const int64_t pitch = FMT == 0 ? p.K / 2 : p.K;
            uint4* dst = reinterpret_cast<uint4*>(p.codes + (int64_t)row * pitch + (FMT == 0 ? col0 / 2 : col0));
#pragma unroll
            for (int j = 0; j < 2 * kWords / 4; ++j) dst[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            if (wg == 0 && lane == 0) p.delta[row] = dl;
        }
        if (++d == p.depth) { d = 0; ph ^= 1u; }
    }

    if (kStaged && lane == 0) bulk_wait_read<0>();       // (the last codes leave shared memory before the CTA does)

    // Winding down after an expired wait: let the copies this group still has in flight land.
    if (leader && *abort_flag) {
        for (int k = n; k < issued; ++k) {
            const int dk = k % p.depth;
            const uint32_t phk = (uint32_t)((k / p.depth) & 1);
            const uint64_t t0 = global_timer_ns();
            while (!mbar_try_wait(smem_u32(&full0[dk]), phk)) {
                if (global_timer_ns() - t0 > kWaitLimitNs) { atomicOr(p.watchdog, 0x200u); break; }
            }
        }
    }
}

template <typename XT, int FMT, int E, int BLOCK, bool GATED = false>
cudaError_t launch_ring(const CUtensorMap& map, const CUtensorMap& map_c, const RingParams& p, int grid, size_t smem,
                        cudaStream_t stream) {
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
        if (e != cudaSuccess) return e;
        return launch_pdl(kern, (unsigned)grid, (unsigned)kThreads, smem, stream, 1u, map, map_c, p);
    };
    // (the fold-after variant is its own instantiation: as a run-time branch it cost the default path registers, and spills,
    // in the 64-channels-per-thread kernels; it has no gated form, nor one for 64 channels with shuffle stages)
    if constexpr (!GATED && (E == 32 || BLOCK <= 64)) {
        if (p.mult_after) {
            if (p.clip_ratio < 1.0f) return go(transform_quantize_ring_kernel<XT, FMT, true, E, BLOCK, true, false>);
            return go(transform_quantize_ring_kernel<XT, FMT, false, E, BLOCK, true, false>);
        }
    }
    if (p.mult_after) return cudaErrorNotSupported;
    if (p.clip_ratio < 1.0f) return go(transform_quantize_ring_kernel<XT, FMT, true, E, BLOCK, false, GATED>);
    return go(transform_quantize_ring_kernel<XT, FMT, false, E, BLOCK, false, GATED>);
}

template <typename XT, int FMT, int E, bool GATED = false>
cudaError_t launch_ring_block(int block, const CUtensorMap& map, const CUtensorMap& map_c, const RingParams& p, int grid,
                              size_t smem, cudaStream_t stream) {
    switch (block) {
        case 32: return launch_ring<XT, FMT, E, 32, GATED>(map, map_c, p, grid, smem, stream);
        case 64: return launch_ring<XT, FMT, E, 64, GATED>(map, map_c, p, grid, smem, stream);
        case 128: return launch_ring<XT, FMT, E, 128, GATED>(map, map_c, p, grid, smem, stream);
        case 256: return launch_ring<XT, FMT, E, 256, GATED>(map, map_c, p, grid, smem, stream);
        default: return cudaErrorNotSupported;
    }
}

template <typename XT, int FMT>
cudaError_t launch_ring_e(int e, int block, const CUtensorMap& map, const CUtensorMap& map_c, const RingParams& p, int grid,
                          size_t smem, cudaStream_t stream) {
    return e == 64 ? launch_ring_block<XT, FMT, 64>(block, map, map_c, p, grid, smem, stream)
                   : launch_ring_block<XT, FMT, 32>(block, map, map_c, p, grid, smem, stream);
}

}  // namespace

cudaError_t launch_transform_quantize_ring(const void* x, fq_dtype xt, int64_t rows, int64_t K, int64_t ldx,
                                           const float* mult, float cnorm, bool mult_after_rotation, int block,
                                           int qmax, float clip_ratio, StoreFmt fmt, void* codes, float* delta,
                                           cudaStream_t stream, int gate_kind, bool mult_ready) {
    const bool gated = gate_kind >= 0;
    const size_t esz = xt == FQ_BF16 ? 2 : 4;
    const size_t row_bytes = (size_t)K * esz;
    const RingPlan f = plan_ring(rows, K, (int)esz, gated, fmt != StoreFmt::Nibble, mult != nullptr, mult != nullptr && mult_after_rotation,
                                 block, device_sm_count());
    if (f.e == 0) return cudaErrorNotSupported;
    const int e = f.e, gw = f.gw, ngroups = f.ngroups, depth = f.depth, sms = device_sm_count();
    const size_t half = f.half, slot = f.slot, g_bytes = f.g_bytes, stage_bytes = f.stage_bytes;

    CUtensorMap map;
    const uint64_t dims[3] = {128 / esz, row_bytes / 128 * (gated ? 2 : 1), (uint64_t)rows};
    const uint64_t strides[2] = {128, (uint64_t)ldx * esz};
    const uint32_t box[3] = {(uint32_t)(128 / esz), (uint32_t)(row_bytes / 128), 1};
    if (!encode_tiled(&map, xt == FQ_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, x,
                      dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorNotSupported;

    CUtensorMap map_c;
    memset(&map_c, 0, sizeof(map_c));
    if (stage_bytes) {
        const uint64_t cdims[3] = {(uint64_t)e, (uint64_t)(K / e), (uint64_t)rows};
        const uint64_t cstrides[2] = {(uint64_t)e, (uint64_t)K};
        const uint32_t cbox[3] = {(uint32_t)e, 32, 1};
        if (!encode_tiled(&map_c, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, codes, cdims, cstrides, cbox, CU_TENSOR_MAP_SWIZZLE_64B))
            return cudaErrorNotSupported;
    }

    RingParams p{};
    p.rows = rows; p.K = (int)K; p.cnorm = cnorm; p.qmax = (float)qmax; p.clip_ratio = clip_ratio;
    p.mult = mult; p.mult_after = (mult != nullptr && mult_after_rotation) ? 1 : 0; p.codes = static_cast<uint8_t*>(codes); p.delta = delta; p.gw = gw; p.depth = depth;
    p.up_bytes = (uint32_t)half; p.up_line = (int)(row_bytes / 128); p.gate_kind = gate_kind;
    p.mult_ready = mult_ready ? 1 : 0;
    p.slot_bytes = (uint32_t)slot; p.g_bytes = (uint32_t)g_bytes;
    p.watchdog = watchdog_device_ptr();
    if (!p.watchdog) return cudaErrorUnknown;
    p.stage_off = (uint32_t)(g_bytes + slot * ngroups * depth);
    const size_t smem = p.stage_off + stage_bytes + 1024;
    // Rows are dealt to the CTAs first and to a CTA's row groups second (row r -> CTA r % grid),
    // so that a short batch spreads over all SMs instead of filling every group of a few CTAs.
    const int grid = (int)(rows < sms ? rows : sms);
    if (gated) {
        if (fmt == StoreFmt::Nibble) return launch_ring_block<__nv_bfloat16, 0, 32, true>(block, map, map_c, p, grid, smem, stream);
        if (fmt == StoreFmt::Int8) return launch_ring_block<__nv_bfloat16, 1, 32, true>(block, map, map_c, p, grid, smem, stream);
        return launch_ring_block<__nv_bfloat16, 2, 32, true>(block, map, map_c, p, grid, smem, stream);
    }
    if (xt == FQ_BF16)
    {
        if (fmt == StoreFmt::Nibble) return launch_ring_e<__nv_bfloat16, 0>(e, block, map, map_c, p, grid, smem, stream);
        if (fmt == StoreFmt::Int8) return launch_ring_e<__nv_bfloat16, 1>(e, block, map, map_c, p, grid, smem, stream);
        return launch_ring_e<__nv_bfloat16, 2>(e, block, map, map_c, p, grid, smem, stream);
    }
    if (fmt == StoreFmt::Nibble) return launch_ring_e<float, 0>(e, block, map, map_c, p, grid, smem, stream);
    if (fmt == StoreFmt::Int8) return launch_ring_e<float, 1>(e, block, map, map_c, p, grid, smem, stream);
    return launch_ring_e<float, 2>(e, block, map, map_c, p, grid, smem, stream);
}

}  // namespace fq
