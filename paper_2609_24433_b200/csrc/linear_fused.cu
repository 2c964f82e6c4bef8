// The whole runtime path of a short batch (at most 64 tokens) in ONE launch: transform, quantization, integer GEMM and
// epilogue (Alg. 1 runtime half; Eq. 5 and 8).
//
// A call of two dependent kernels on 50 tokens took 7.9 us in a chain of calls, whatever its size: the hand-over between
// the kernels, the codes' way through L2 and the second kernel's pipeline fill are most of it.  Here a cluster of C
// CTAs computes 128 output channels of all tokens, split along K:
//   - a CTA transforms the tokens' channels of its own K slice (at most 512), so no codes are exchanged -- only the
//     slices' maxima, one float per token and CTA, through distributed shared memory;
//   - its codes go straight into the swizzled shared-memory operand of its MMAs; its weights arrived by TMA, and 4-bit
//     ones were expanded into tensor memory, before the kernel ahead in the stream had finished;
//   - the int32 partial sums meet in distributed shared memory, every CTA finishing its share of the tokens.
// The transform is repeated by every cluster, and what is left is a chain of latencies: at M = 50, K = N = 1024, clock marks
// behind the wait for the kernel ahead count some 600 cycles for the load, 1200 for the butterflies, 1300 for the
// exchange of maxima, 1000 for the codes, 700 for the MMAs and 1700 for the sums' exchange and the outputs.  So slices are as
// narrow as clusters of eight allow, and a thread holds sixteen channels (32: 6.8 instead of 5.8 us per call); thirty-two (T = 2
// rounds) only where rows are too long for that.
//
// Arithmetic: that of the prologue and GEMM kernels, operation by operation, so codes, steps, sums and outputs are
// theirs bit for bit.  Codes and steps also go to the caller's workspace, as the two-kernel path leaves them.
#include <cuda_bf16.h>
#include <float.h>

#include "fq_common.cuh"
#include "ptx_sm100.cuh"
#include "act_common.cuh"
#include "tc_sm100.cuh"

namespace fq {
namespace {

constexpr int kThreads = 512;
constexpr int kMaxTokens = kFusedMaxTokens;
constexpr int E = kFusedRun, H = E / 2;       // channels per thread and round: v[p] = (channel p, channel p + H)
constexpr int kTile = kTileN;          // output channels per MMA

enum : uint32_t { kWdFusedWeights = 0x2000u, kWdFusedMma = 0x4000u };

struct FusedParams {
    const void* x;
    int64_t ldx, ldy;
    int M, N, K;
    int bt;                    // tokens, rounded up to the MMA's multiple of 16
    int ctas_shift;            // log2 of the CTAs per cluster
    int unit, units;           // K is dealt to the CTAs in units (of a block, at least 128 channels)
    int tok_shift;             // log2 of the tokens a CTA finishes
    int tmem_cols, w_col;      // tensor memory: columns, first column of the expanded weights
    uint32_t off_part, off_codes, off_g;     // shared memory: partial sums, codes, multiplier (weights first)
    const float* mult;         // per-channel multiplier or null
    int mult_after;
    float cnorm, qmax, clip_ratio, unshift;
    int block;
    const float* w_scale;
    const float* bias;
    void* y;
    fq_dtype yt;
    int8_t* ws_codes;          // [M][K] and [M], or null
    float* ws_delta;
    uint32_t* watchdog;
};

// Sixteen channels of one token, halves paired so that butterflies below stride 8 act on both with one packed instruction.
template <typename XT>
struct Row;
template <>
struct Row<__nv_bfloat16> {
    uint4 lo, hi;
    __device__ __forceinline__ void load(const __nv_bfloat16* p, bool ok) {
        lo = ld_global_v4(p, ok);
        hi = ld_global_v4(p + 8, ok);
    }
    __device__ __forceinline__ void widen(float2* v) const {
        const uint32_t wl[4] = {lo.x, lo.y, lo.z, lo.w}, wh[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[2 * j + 0] = make_float2(__uint_as_float(wl[j] << 16), __uint_as_float(wh[j] << 16));
            v[2 * j + 1] = make_float2(__uint_as_float(wl[j] & 0xffff0000u), __uint_as_float(wh[j] & 0xffff0000u));
        }
    }
};
template <>
struct Row<float> {
    float4 q[4];
    __device__ __forceinline__ void load(const float* p, bool ok) {
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = ld_global_f4(p + 4 * i, ok);
    }
    __device__ __forceinline__ void widen(float2* v) const {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            v[4 * i + 0] = make_float2(q[i].x, q[i + 2].x);
            v[4 * i + 1] = make_float2(q[i].y, q[i + 2].y);
            v[4 * i + 2] = make_float2(q[i].z, q[i + 2].z);
            v[4 * i + 3] = make_float2(q[i].w, q[i + 2].w);
        }
    }
};

// LG lanes share a token: 16 (256 channels a round, 32 tokens) or 8 (128 channels, 64 tokens); T rounds.
template <typename XT, int BITS, int LG, int T>
__global__ void __launch_bounds__(kThreads, T == 1 ? 2 : 1)
linear_fused_kernel(const __grid_constant__ CUtensorMap map_w, const FusedParams p) {
    constexpr int kRoundCh = LG * E;
    constexpr int FMT = BITS == 4 ? 2 : 1;                 // int8 codes, 4-bit ones in the order the weights unpack to
    constexpr int kWAtom = kTile * 128 * BITS / 8;         // weight bytes of 128 rows x 128 channels
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t s_bar_w, s_bar_mma;
    __shared__ float s_max[kMaxCluster][kMaxTokens];
    __shared__ float s_delta[kMaxTokens];
    __shared__ float s_scale[kTile], s_bias[kTile];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
    const int C = 1 << p.ctas_shift;
    const uint32_t rank = C > 1 ? cluster_ctarank() : 0u;
    const int tile = (int)blockIdx.x >> p.ctas_shift;
    const int j0 = tile * kTile;                           // first output channel of the cluster
    const int k0 = (((int)rank * p.units) >> p.ctas_shift) * p.unit;
    const int ks = ((((int)rank + 1) * p.units) >> p.ctas_shift) * p.unit - k0;
    const int atoms = ks >> 7;

    if (tid == 0) {
        s_abort = 0;
        mbar_init(smem_u32(&s_bar_w), 1);
        mbar_init(smem_u32(&s_bar_mma), 1);
        fence_mbarrier_init();
        fence_proxy_async_smem();
        // a handle is complete before any call that uses it: the weights need not wait for the kernel ahead
        const uint32_t bar = smem_u32(&s_bar_w);
        mbar_arrive_expect_tx(bar, (uint32_t)(atoms * kWAtom));
        for (int a = 0; a < atoms; ++a)                    // rows past N arrive as zeros
            tma_load_2d(base + (uint32_t)(a * kWAtom), &map_w, (k0 + a * 128) * BITS / 8, j0, bar);
    }
    if (warp == 1) tmem_alloc<1>(smem_u32(&s_tmem), (uint32_t)p.tmem_cols);
    if (tid >= kThreads - kTile) {                         // what the epilogue needs of the handle, ahead of everything
        const int o = tid - (kThreads - kTile), j = j0 + o;
        const bool ok = j < p.N;
        s_scale[o] = ok ? __ldg(p.w_scale + j) * p.unshift : 0.0f;
        s_bias[o] = ok ? __ldg(p.bias + j) : 0.0f;
    }
    if (p.mult != nullptr) {
        // the slice's multipliers as (g[q], g[q + H]) pairs per run of E channels, runs 16 bytes apart modulo 128
        for (int i = tid; i < ks; i += kThreads) {
            const int q = i % E;
            reinterpret_cast<float*>(gen + p.off_g)[i / E * (E + 4) + (q < H ? 2 * q : 2 * (q - H) + 1)] = __ldg(p.mult + k0 + i);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    if (C > 1) cluster_arrive();                           // "this CTA exists": awaited before the first remote store
    griddep_launch_dependents();

    if (tid / LG < p.M && tid % LG * E < ks)               // tokens that lie in memory come as far as L2 meanwhile
        prefetch_l2(static_cast<const XT*>(p.x) + (int64_t)(tid / LG) * p.ldx + k0 + tid % LG * E);
    if (BITS == 4) {
        mbar_wait_all(smem_u32(&s_bar_w), 0u, &s_abort, p.watchdog, kWdFusedWeights);
        // a thread owns one weight row (TMEM lane) of every fourth atom: 64 packed bytes, 64-byte TMA swizzle, to
        // 128 int8 holding 16 * code in the order of the activations' codes
        const int row = (warp & 3) * 32 + lane;
        const uint32_t swz = (uint32_t)(row >> 1) & 3u;
        for (int it = warp >> 2; it < atoms; it += 4) {
            const uint32_t src = base + (uint32_t)(it * kWAtom + row * 64);
            uint32_t o[32];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 q = lds128(src + (((uint32_t)c ^ swz) << 4));
                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    o[8 * c + 2 * i + 0] = (w[i] << 4) & 0xF0F0F0F0u;
                    o[8 * c + 2 * i + 1] = w[i] & 0xF0F0F0F0u;
                }
            }
            tmem_st32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(p.w_col + it * 32), o);
        }
        tmem_st_wait();
    }
    griddep_wait();                                        // the kernel ahead wrote x, and may still read y or the workspace

    // ---- transform: T rounds of kRoundCh channels, LG lanes per token
    const int token = tid / LG, gl = tid % LG;
    const bool tok_ok = token < p.M;
    const bool busy = warp * (32 / LG) < p.M;              // (warp-uniform) some lane of this warp has a token
    float2 v[T][H];
    float m = 0.0f;
    const float4* gp = reinterpret_cast<const float4*>(gen + p.off_g);
    if (busy) {
        const XT* xp = static_cast<const XT*>(p.x) + (int64_t)token * p.ldx + k0 + gl * E;
        Row<XT> raw[T];
#pragma unroll
        for (int r = 0; r < T; ++r) raw[r].load(xp + r * kRoundCh, tok_ok && r * kRoundCh + gl * E < ks);
#pragma unroll
        for (int r = 0; r < T; ++r) raw[r].widen(v[r]);
        auto by_channel = [&](int r) {
            const int run = (r * kRoundCh + gl * E) / E;
            if (run * E >= ks) return;                         // (zeros stay zeros)
#pragma unroll
            for (int i = 0; i < H / 2; ++i) {
                const float4 q = gp[run * (E + 4) / 4 + i];
                v[r][2 * i + 0] = f2_mul(v[r][2 * i + 0], make_float2(q.x, q.y));
                v[r][2 * i + 1] = f2_mul(v[r][2 * i + 1], make_float2(q.z, q.w));
            }
        };
        const float2 neg1 = make_float2(-1.0f, -1.0f), c2 = make_float2(p.cnorm, p.cnorm);
#pragma unroll
        for (int r = 0; r < T; ++r) {
            if (p.mult != nullptr && !p.mult_after) {
                by_channel(r);
            } else {
#pragma unroll
                for (int i = 0; i < H; ++i) v[r][i] = f2_mul(v[r][i], c2);
            }
#pragma unroll
            for (int h = 1; h < H; h <<= 1) {
                if (h < p.block) {
#pragma unroll
                    for (int i = 0; i < H; ++i) {
                        if ((i & h) == 0) {
                            const float2 a = v[r][i], b = v[r][i + h];
                            v[r][i] = f2_add(a, b);
                            v[r][i + h] = f2_fma(b, neg1, a);          // a - b, exact product
                        }
                    }
                }
            }
            if (H < p.block) {
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    const float a = v[r][i].x, b = v[r][i].y;
                    v[r][i] = make_float2(__fadd_rn(a, b), __fsub_rn(a, b));
                }
            }
            for (int h = E; h < p.block; h <<= 1) {            // partner lane = lane ^ (h / E); upper lane keeps partner - own
                const int lm = h / E;
                const float sg = (lane & lm) ? -1.0f : 1.0f;
                const float2 s2 = make_float2(sg, sg);
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    const float2 q = make_float2(__shfl_xor_sync(0xffffffffu, v[r][i].x, lm), __shfl_xor_sync(0xffffffffu, v[r][i].y, lm));
                    v[r][i] = f2_fma(v[r][i], s2, q);
                }
            }
            if (p.mult != nullptr && p.mult_after) by_channel(r);
#pragma unroll
            for (int i = 0; i < H; ++i)
                asm("max.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(fabsf(v[r][i].x)), "f"(fabsf(v[r][i].y)));
        }
#pragma unroll
        for (int lm = 1; lm < LG; lm <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, lm));
    }
    if (C > 1) {
        cluster_wait();
        if (busy && gl < C) st_cluster(cluster_address(smem_u32(&s_max[rank][token]), (uint32_t)gl), __float_as_uint(m));
        __syncwarp();
        cluster_arrive();
        cluster_wait();
#pragma unroll
        for (int c = 0; c < kMaxCluster; ++c)
            if (c < C) m = fmaxf(m, s_max[c][token]);
    }

    // ---- Eq. 5, codes into the MMA's operand: [atom][token][128 bytes], 128-byte swizzle
    if (busy) {
        float d = __fdiv_rn(__fmul_rn(p.clip_ratio, m), p.qmax);
        float inv;
        if (d >= FLT_MIN) {
            inv = __fdiv_rn(1.0f, d);
        } else {
            d = 0.0f;
            inv = 0.0f;
        }
        const bool keeps = p.ws_codes != nullptr && tile == 0;
        if (gl == 0) {
            s_delta[token] = d;
            if (keeps && rank == 0 && tok_ok) p.ws_delta[token] = d;
        }
        const float2 inv2 = make_float2(inv, inv);
        const bool clamp = p.clip_ratio < 1.0f;
#pragma unroll
        for (int r = 0; r < T; ++r) {
            const int c = r * kRoundCh + gl * E;
            if (tok_ok && c < ks) {
                constexpr int kWords = H / 4;
                uint32_t w[2 * kWords];
#pragma unroll
                for (int j = 0; j < kWords; ++j) {
                    uint32_t bl[4], bh[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float2 t = f2_mul(v[r][code_index<FMT>(j, i)], inv2);
                        if (clamp) {
                            t.x = fminf(fmaxf(t.x, -p.qmax), p.qmax);
                            t.y = fminf(fmaxf(t.y, -p.qmax), p.qmax);
                        }
                        t = f2_fma(t, make_float2(1.0f, 1.0f), make_float2(12582912.0f, 12582912.0f));   // exact product: rounds like the add
                        bl[i] = __float_as_uint(t.x);
                        bh[i] = __float_as_uint(t.y);
                    }
                    w[j] = pack_word<FMT>(bl);
                    w[kWords + j] = pack_word<FMT>(bh);
                }
                const uint32_t row = p.off_codes + (uint32_t)((c >> 7) * p.bt + token) * 128u;
                const uint32_t chunk = (uint32_t)(c & 127) >> 4, key = (uint32_t)token & 7u;
#pragma unroll
                for (int j = 0; j < E / 16; ++j) {
                    const uint4 q = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
                    *reinterpret_cast<uint4*>(gen + row + (((chunk + j) ^ key) << 4)) = q;
                    if (keeps) *reinterpret_cast<uint4*>(p.ws_codes + (int64_t)token * p.K + k0 + c + 16 * j) = q;
                }
            }
        }
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();

    // ---- acc[channel][token] of this slice
    if (warp == 0) {
        bool ok = true;
        if (BITS == 8) ok = mbar_wait_all(smem_u32(&s_bar_w), 0u, &s_abort, p.watchdog, kWdFusedWeights);
        tc_fence_after();
        if (ok && elect_one()) {
            const uint32_t idesc = instr_desc_i8(kTile, p.bt);
            for (int a = 0; a < atoms; ++a) {
                const uint64_t bd = smem_desc_sw128(base + p.off_codes + (uint32_t)(a * p.bt) * 128u);
                const uint64_t ad = smem_desc_sw128(base + (uint32_t)(a * kWAtom));
                const uint32_t at = tmem + (uint32_t)(p.w_col + a * 32);
#pragma unroll
                for (int s = 0; s < 4; ++s) {              // 32 bytes along K: +2 in a descriptor, 8 TMEM columns
                    if (BITS == 4) mma_i8_ts(tmem, at + 8 * s, bd + 2 * s, idesc, (a | s) != 0);
                    else mma_i8_ss(tmem, ad + 2 * s, bd + 2 * s, idesc, (a | s) != 0);
                }
            }
            mma_commit(smem_u32(&s_bar_mma));
        }
        __syncwarp();
    }
    mbar_wait_all(smem_u32(&s_bar_mma), 0u, &s_abort, p.watchdog, kWdFusedMma);
    tc_fence_after();

    // ---- partial sums to the CTA that finishes the token: [slice][token][128 channels]
    if (const int t0 = (warp >> 2) * 16; t0 < p.M) {       // a warp: 32 channels, 16 tokens
        uint32_t a[16];
        if (atoms > 0) {
            tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)t0, a);
            tmem_ld_wait();
        } else {                                           // fewer units than CTAs: no channels here, nothing multiplied
#pragma unroll
            for (int i = 0; i < 16; ++i) a[i] = 0u;
        }
        const uint32_t dst = base + p.off_part + (uint32_t)((warp & 3) * 32 + lane) * 4u;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int t = t0 + i;
            if (t < p.M) {
                const uint32_t at = dst + (uint32_t)(((int)rank << p.tok_shift) + (t & ((1 << p.tok_shift) - 1))) * (kTile * 4u);
                st_cluster(cluster_address(at, (uint32_t)(t >> p.tok_shift)), a[i]);
            }
        }
    }
    tc_fence_before();
    __syncwarp();
    if (C > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }

    // ---- Eq. 8: two channels of a token per thread
    const int first = (int)rank << p.tok_shift, mine = min(1 << p.tok_shift, p.M - first);
    const int jj = (tid & 63) * 2;
    const int32_t* part = reinterpret_cast<const int32_t*>(gen + p.off_part) + jj;
    if (j0 + jj < p.N && !*reinterpret_cast<volatile int*>(&s_abort)) {
        const float sw0 = s_scale[jj], sw1 = s_scale[jj + 1], b0 = s_bias[jj], b1 = s_bias[jj + 1];
        for (int tt = tid >> 6; tt < mine; tt += kThreads / 64) {
            int2 q[kMaxCluster];
#pragma unroll
            for (int c = 0; c < kMaxCluster; ++c)
                if (c < C) q[c] = *reinterpret_cast<const int2*>(part + ((c << p.tok_shift) + tt) * kTile);
            int2 sum = q[0];
#pragma unroll
            for (int c = 1; c < kMaxCluster; ++c)
                if (c < C) {
                    sum.x += q[c].x;
                    sum.y += q[c].y;
                }
            const float dt = s_delta[first + tt];
            const float y0 = fmaf((float)sum.x, dt * sw0, b0), y1 = fmaf((float)sum.y, dt * sw1, b1);
            const int64_t at = (int64_t)(first + tt) * p.ldy + j0 + jj;
            if (p.yt == FQ_F32) *reinterpret_cast<float2*>(static_cast<float*>(p.y) + at) = make_float2(y0, y1);
            else *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(p.y) + at) = __floats2bfloat162_rn(y0, y1);
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc<1>(tmem, (uint32_t)p.tmem_cols);
    }
    if (s_abort && tid == 0) drain_after_abort();
}

template <typename XT, int BITS, int LG, int T>
cudaError_t launch_variant(const CUtensorMap& map, const FusedParams& p, const FusedPlan& f, cudaStream_t stream) {
    auto kern = linear_fused_kernel<XT, BITS, LG, T>;
    const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), f.smem);
    if (e != cudaSuccess) return e;
    const cudaError_t launched = launch_pdl(kern, (unsigned)f.grid, (unsigned)kThreads, f.smem, stream, 1u << f.ctas_shift, map, p);
    return f.ctas_shift > 0 && cluster_refused(launched) ? cudaErrorNotSupported : launched;
}
template <typename XT, int BITS>
cudaError_t launch_bits(const CUtensorMap& map, const FusedParams& p, const FusedPlan& f, cudaStream_t stream) {
    if (f.lanes == 16) return f.rounds == 1 ? launch_variant<XT, BITS, 16, 1>(map, p, f, stream) : launch_variant<XT, BITS, 16, 2>(map, p, f, stream);
    return f.rounds == 1 ? launch_variant<XT, BITS, 8, 1>(map, p, f, stream) : launch_variant<XT, BITS, 8, 2>(map, p, f, stream);
}

}  // namespace

cudaError_t launch_linear_fused(const void* x, fq_dtype xt, int64_t M, int64_t ldx, const Weights& W, float cnorm, int qmax,
                                float clip_ratio, void* y, fq_dtype yt, int64_t ldy, int8_t* ws_codes, float* ws_delta,
                                cudaStream_t stream) {
    if (!W.tmap_valid) return cudaErrorNotSupported;
    // a multiplier that is block^-1/2 in every channel is passed as "none": same products, no vector to stage
    const float* mult = W.mult_const ? nullptr : W.mult_g;
    const FusedPlan f = plan_fused(M, W.N, W.K, W.block, W.bits, mult != nullptr, device_sm_count(), cluster_capacity);
    if (f.lanes == 0) return cudaErrorNotSupported;
    FusedParams p{};
    p.x = x; p.ldx = ldx; p.ldy = ldy;
    p.M = (int)M; p.N = (int)W.N; p.K = (int)W.K;
    p.bt = (int)((M + 15) / 16 * 16);
    p.ctas_shift = f.ctas_shift; p.unit = f.unit; p.units = f.units;
    p.tok_shift = log2_ceil((int)((M + (1 << f.ctas_shift) - 1) >> f.ctas_shift));
    p.w_col = (p.bt + 31) / 32 * 32;
    const int cols = p.w_col + (W.bits == 4 ? f.slice / 4 : 0);
    p.tmem_cols = 1 << log2_ceil(cols < 32 ? 32 : cols);
    if (p.tmem_cols > 256) return cudaErrorNotSupported;
    p.off_part = f.off_part; p.off_codes = f.off_codes; p.off_g = f.off_g;
    p.mult = mult; p.mult_after = mult != nullptr && W.fold_after ? 1 : 0;
    p.cnorm = cnorm; p.qmax = (float)qmax; p.clip_ratio = clip_ratio; p.unshift = W.bits == 4 ? 1.0f / 16.0f : 1.0f;
    p.block = W.block;
    p.w_scale = W.w_scale; p.bias = W.bias; p.y = y; p.yt = yt;
    p.ws_codes = ws_codes; p.ws_delta = ws_delta;
    p.watchdog = watchdog_device_ptr();
    if (!p.watchdog) return cudaErrorUnknown;
    if (xt == FQ_BF16)
        return W.bits == 4 ? launch_bits<__nv_bfloat16, 4>(W.tmap, p, f, stream) : launch_bits<__nv_bfloat16, 8>(W.tmap, p, f, stream);
    return W.bits == 4 ? launch_bits<float, 4>(W.tmap, p, f, stream) : launch_bits<float, 8>(W.tmap, p, f, stream);
}

}  // namespace fq
