// Stored composite rotation (optional transform of the action expert): a channel permutation followed
// by one stored dense matrix per block of `beta` channels,
//   R = blockdiag(B_0 .. B_{K/beta-1}) Pi,      u[t][b*beta + i] = sum_j B_b[i][j] * v[t][perm[b*beta + j]],
//   v = x (.) d  (d = 1/s at run time, s when folding weights).
// This kernel produces u in binary32 (one multiply for the diagonal, then one fused multiply-add per
// term in ascending j, starting from 0 -- the order the results are defined in); the per-token step and
// the codes of Eq. 5 are then taken by the ordinary prologue kernel run with the identity rotation.
// The contraction is 2*beta flops per element against 6 for the butterflies; it is dense but tiny per
// block (beta x beta) and the sums must keep their order: CUDA cores.  Two forms:
//   composite_quantize_kernel  the whole runtime prologue of a site in one launch (rows of up to some 4096 channels)
//   composite_rotate_kernel    the rotated rows in binary32, one CTA per (block, tile of tokens), the block's matrix staged
//                              through shared memory in transposed chunks; the ordinary prologue kernel then quantizes
//                              (weight folding, and rows too long for the other one)
#include <cuda_bf16.h>
#include <float.h>

#include "fq_common.cuh"
#include "ptx_sm100.cuh"
#include "act_common.cuh"
#include "tc_sm100.cuh"

namespace fq {
namespace {

constexpr int kThreads = 256;
constexpr int kChunkJ = 32;          // columns of B staged at a time

template <typename XT>
__device__ __forceinline__ float load_as_float(const XT* p);
template <>
__device__ __forceinline__ float load_as_float<float>(const float* p) { return ld_global_f32(p); }
template <>
__device__ __forceinline__ float load_as_float<__nv_bfloat16>(const __nv_bfloat16* p) {
    return __uint_as_float(ld_global_u16(p) << 16);
}

// BETA in {16, 32, 64, 128, 256}.  Thread (group = tid / BETA, i = tid % BETA) computes output i of
// R = 8 tokens (one shared-memory read of the matrix entry and two 16-byte reads of the inputs feed eight
// multiply-adds); a CTA covers (256 / BETA) * 8 tokens of one block.
template <typename XT, int BETA>
__global__ void __launch_bounds__(kThreads)
composite_rotate_kernel(const XT* __restrict__ x, int64_t rows, int K, int64_t ldx, const float* __restrict__ diag,
                        const int32_t* __restrict__ perm, const float* __restrict__ blocks, float* __restrict__ u) {
    constexpr int G = kThreads / BETA;
    constexpr int R = 8;
    constexpr int TOK = G * R;
    __shared__ __align__(16) float s_p[BETA][TOK];   // permuted, scaled inputs of the tile, token-minor
    __shared__ float s_b[kChunkJ][BETA + 1];         // B_b[.][j0 .. j0+31], transposed: s_b[jj][i]
    griddep_wait();
    griddep_launch_dependents();
    const int tid = threadIdx.x;
    const int b = blockIdx.x;
    const int64_t tile0 = (int64_t)blockIdx.y * TOK;
    // gather: p[tok][j] = x[tok][perm[b*BETA + j]] * d[perm[...]]   (an index outside [0, K) is clamped)
    for (int o = tid; o < TOK * BETA; o += kThreads) {
        const int tok = o / BETA, j = o % BETA;
        int src = (int)ld_global_u32(perm + b * BETA + j);
        src = src < 0 ? 0 : (src >= K ? K - 1 : src);
        float v = 0.0f;
        if (tile0 + tok < rows) {
            v = load_as_float<XT>(x + (tile0 + tok) * ldx + src);
            if (diag != nullptr) v = __fmul_rn(v, ld_global_f32(diag + src));
        }
        s_p[j][tok] = v;
    }
    const int grp = tid / BETA, i = tid % BETA;
    float acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0f;
    const float* B = blocks + (size_t)b * BETA * BETA;
    for (int j0 = 0; j0 < BETA; j0 += kChunkJ) {
        __syncthreads();                             // s_p written (first pass) / previous chunk consumed
        constexpr int CJ = BETA < kChunkJ ? BETA : kChunkJ;
        for (int o = tid; o < BETA * CJ; o += kThreads) {
            const int row = o / CJ, jj = o % CJ;     // consecutive threads: consecutive columns of one row
            s_b[jj][row] = ld_global_f32(B + (size_t)row * BETA + j0 + jj);
        }
        __syncthreads();
#pragma unroll 8
        for (int jj = 0; jj < CJ; ++jj) {
            const float bv = s_b[jj][i];
            const float4 pa = *reinterpret_cast<const float4*>(&s_p[j0 + jj][grp * R]);
            const float4 pb = *reinterpret_cast<const float4*>(&s_p[j0 + jj][grp * R + 4]);
            acc[0] = __fmaf_rn(bv, pa.x, acc[0]); acc[1] = __fmaf_rn(bv, pa.y, acc[1]);
            acc[2] = __fmaf_rn(bv, pa.z, acc[2]); acc[3] = __fmaf_rn(bv, pa.w, acc[3]);
            acc[4] = __fmaf_rn(bv, pb.x, acc[4]); acc[5] = __fmaf_rn(bv, pb.y, acc[5]);
            acc[6] = __fmaf_rn(bv, pb.z, acc[6]); acc[7] = __fmaf_rn(bv, pb.w, acc[7]);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t t = tile0 + grp * R + r;
        if (t < rows) u[t * K + b * BETA + i] = acc[r];
    }
}

// Rotation and quantization of TOK tokens (16, or 8 where 16 rows do not fit) by a cluster of C CTAs, each computing a share
// of the output channels.
//   - Every CTA stages the tokens' whole rows in shared memory: a permuted channel costs a 32-byte sector when it is fetched
//     from L2 two or four bytes at a time, which bounded the separate rotation (21.8 us at M = 816, K = 2048, block 64).
//   - A warp takes 64 outputs (or a whole smaller block) at a time, sixteen columns after sixteen: it gathers the columns'
//     inputs token-minor, and its lanes accumulate four outputs of TPL tokens each, two tokens per packed multiply-add, from
//     matrix columns that cp.async brings a step ahead.  Ascending j from 0: the defined order.
//   - The rotated channels stay in shared memory until the cluster has exchanged the tokens' maxima; only codes and steps
//     leave the SM.
// M = 816, K = 2048, block 64: 15.4 us in a chain of calls, 19.7 while the clusters made two waves (31 us for rotation and
// quantizer as two kernels, cold caches); matrix rows read by each lane straight from L2 instead of through cp.async took 52 us.
struct CompositeParams {
    const void* x;
    int64_t ldx, rows;
    int K;
    int ctas_shift;           // log2 of the CTAs per cluster
    int items;                // K / outputs per item
    int vec;                  // x and its rows are 16-byte aligned
    uint32_t off_u, off_b, off_p, off_s;      // shared memory: rows of x, rotated channels, matrix columns, inputs, sources
    int u_pitch;              // floats
    int span;                 // channels of the blocks that a CTA's items touch, at most
    int bits;
    const float* diag;
    const int32_t* perm;
    const float* blocks;
    float clip_ratio, qmax;
    uint8_t* codes;
    float* delta;
};
constexpr int kCol = kCompositeColumns;                // columns per step
constexpr int kWarps = kThreads / 32;
static_assert(kWarps == kCompositeWarps, "the plan sizes shared memory for these warps");

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename XT, int BETA, int TOK>
__global__ void __launch_bounds__(kThreads, 1)
composite_quantize_kernel(const CompositeParams p) {
    constexpr int OUT = BETA < 64 ? BETA : 64;         // outputs per item
    constexpr int COLS = OUT / 4;                      // lanes across the outputs: outputs cg, cg + COLS, ...
    constexpr int TPL = TOK / (32 / COLS);             // tokens per lane
    constexpr int PITCH = TOK + 4;                     // gathered inputs: rows 16 bytes apart modulo 128, conflict-free
    constexpr int STEPS = BETA / kCol;
    extern __shared__ __align__(16) uint8_t s_raw[];
    __shared__ float s_wmax[kWarps][TOK], s_max[8][TOK];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = 1 << p.ctas_shift;
    const uint32_t rank = C > 1 ? cluster_ctarank() : 0u;
    const int64_t t0 = (int64_t)(blockIdx.x >> p.ctas_shift) * TOK;
    const XT* s_x = reinterpret_cast<const XT*>(s_raw);
    float* s_u = reinterpret_cast<float*>(s_raw + p.off_u);
    float* s_b = reinterpret_cast<float*>(s_raw + p.off_b) + warp * 2 * OUT * kCol;
    float* s_p = reinterpret_cast<float*>(s_raw + p.off_p) + warp * kCol * PITCH;
    int* s_src = reinterpret_cast<int*>(s_raw + p.off_s);
    float* s_dg = reinterpret_cast<float*>(s_src + p.span);
    if (C > 1) cluster_arrive();                       // "this CTA exists": awaited before the first remote store
    griddep_launch_dependents();
    griddep_wait();

    const int item0 = ((int)rank * p.items) >> p.ctas_shift, item1 = (((int)rank + 1) * p.items) >> p.ctas_shift;
    const int c0 = item0 * OUT / BETA * BETA;          // first channel of the first block
    const XT* xr = static_cast<const XT*>(p.x) + t0 * p.ldx;
    const int mine = p.rows - t0 < TOK ? (int)(p.rows - t0) : TOK;
    if (p.vec) {
        constexpr int V = 16 / sizeof(XT);
        for (int r = 0; r < mine; ++r)
            for (int c = tid * V; c < p.K; c += kThreads * V) cp_async16(smem_u32(s_x + r * p.K + c), xr + r * p.ldx + c);
    } else {
        for (int r = 0; r < mine; ++r)
            for (int c = tid; c < p.K; c += kThreads) {
                if (sizeof(XT) == 2) reinterpret_cast<uint16_t*>(s_raw)[r * p.K + c] = (uint16_t)ld_global_u16(xr + r * p.ldx + c);
                else reinterpret_cast<uint32_t*>(s_raw)[r * p.K + c] = ld_global_u32(xr + r * p.ldx + c);
            }
    }
    cp_commit();
    // step (item, columns) of this warp: 16 columns of the item's matrix rows, 64 bytes a row, 16-byte chunks XORed by the row
    auto fetch = [&](int item, int step, int buf) {
        if (item < item1) {
            const float* B = p.blocks + ((size_t)(item / (BETA / OUT)) * BETA + item % (BETA / OUT) * OUT) * BETA + step * kCol;
#pragma unroll
            for (int o = lane; o < OUT * 4; o += 32) {
                const int row = o >> 2, ch = o & 3;
                cp_async16(smem_u32(s_b + buf * OUT * kCol + row * kCol + ((ch ^ ((row >> 1) & 3)) << 2)), B + (size_t)row * BETA + ch * 4);
            }
        }
        cp_commit();
    };
    fetch(item0 + warp, 0, 0);
    for (int i = tid; i < p.span && c0 + i < p.K; i += kThreads) {
        int src = (int)ld_global_u32(p.perm + c0 + i); // (an index outside [0, K) is clamped)
        src = src < 0 ? 0 : (src >= p.K ? p.K - 1 : src);
        s_src[i] = src;
        s_dg[i] = p.diag != nullptr ? ld_global_f32(p.diag + src) : 1.0f;
    }
    cp_wait<1>();                                      // the rows of x (the first matrix columns may still be on their way)
    __syncthreads();

    const int cg = lane % COLS, tg = lane / COLS;
    float m[TPL];
#pragma unroll
    for (int i = 0; i < TPL; ++i) m[i] = 0.0f;
    int buf = 0;
    for (int item = item0 + warp; item < item1; item += kWarps) {
        const int first = item / (BETA / OUT) * BETA - c0;            // the block's first channel in s_src
        float2 acc[4][TPL / 2];
#pragma unroll
        for (int o = 0; o < 4; ++o)
#pragma unroll
            for (int i = 0; i < TPL / 2; ++i) acc[o][i] = make_float2(0.0f, 0.0f);
#pragma unroll 1
        for (int step = 0; step < STEPS; ++step, buf ^= 1) {
            const bool last = step == STEPS - 1;
            fetch(last ? item + kWarps : item, last ? 0 : step + 1, buf ^ 1);
            {   // inputs of the columns: lane = (column, half of the tokens)
                const int j = lane & (kCol - 1), h = lane / kCol * (TOK / 2);
                const int src = s_src[first + step * kCol + j];
                const float dg = s_dg[first + step * kCol + j];
                float v[TOK / 2];
#pragma unroll
                for (int t = 0; t < TOK / 2; ++t) {
                    if (sizeof(XT) == 2) v[t] = __uint_as_float((uint32_t)reinterpret_cast<const unsigned short*>(s_x)[(h + t) * p.K + src] << 16);
                    else v[t] = reinterpret_cast<const float*>(s_x)[(h + t) * p.K + src];
                    v[t] = __fmul_rn(v[t], dg);
                }
#pragma unroll
                for (int t = 0; t < TOK / 2; t += 4)
                    *reinterpret_cast<float4*>(s_p + j * PITCH + h + t) = make_float4(v[t], v[t + 1], v[t + 2], v[t + 3]);
            }
            cp_wait<1>();                              // this step's matrix columns
            __syncwarp();
            const float* bs = s_b + buf * OUT * kCol;
#pragma unroll
            for (int q = 0; q < kCol / 4; ++q) {
                float4 w[4];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const int row = cg + COLS * o;
                    w[o] = *reinterpret_cast<const float4*>(bs + row * kCol + ((q ^ ((row >> 1) & 3)) << 2));
                }
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    float2 pv[TPL / 2];
                    const float* src = s_p + (4 * q + jj) * PITCH + tg * TPL;
                    if constexpr (TPL >= 4) {
#pragma unroll
                        for (int i = 0; i < TPL / 4; ++i) {
                            const float4 t = *reinterpret_cast<const float4*>(src + 4 * i);
                            pv[2 * i] = make_float2(t.x, t.y);
                            pv[2 * i + 1] = make_float2(t.z, t.w);
                        }
                    } else {
                        pv[0] = *reinterpret_cast<const float2*>(src);
                    }
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        const float c = jj == 0 ? w[o].x : (jj == 1 ? w[o].y : (jj == 2 ? w[o].z : w[o].w));
#pragma unroll
                        for (int i = 0; i < TPL / 2; ++i) acc[o][i] = f2_fma(make_float2(c, c), pv[i], acc[o][i]);
                    }
                }
            }
            __syncwarp();                              // inputs and columns are free again
        }
        float* u = s_u + (item - item0) * OUT + cg;
#pragma unroll
        for (int i = 0; i < TPL; ++i)
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const float v = i % 2 ? acc[o][i / 2].y : acc[o][i / 2].x;
                m[i] = fmaxf(m[i], fabsf(v));
                u[(tg * TPL + i) * p.u_pitch + COLS * o] = v;
            }
    }
    cp_wait<0>();
#pragma unroll
    for (int i = 0; i < TPL; ++i) {
#pragma unroll
        for (int lm = 1; lm < COLS; lm <<= 1) m[i] = fmaxf(m[i], __shfl_xor_sync(0xffffffffu, m[i], lm));
        if (cg == 0) s_wmax[warp][tg * TPL + i] = m[i];
    }
    __syncthreads();
    float mt = 0.0f;
    if (tid < TOK * C)                                 // token tid % TOK, for CTA tid / TOK
#pragma unroll
        for (int w = 0; w < kWarps; ++w) mt = fmaxf(mt, s_wmax[w][tid % TOK]);
    if (C > 1) {
        cluster_wait();
        if (tid < TOK * C) st_cluster(cluster_address(smem_u32(&s_max[rank][tid % TOK]), (uint32_t)(tid / TOK)), __float_as_uint(mt));
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    } else {
        if (tid < TOK) s_max[0][tid] = mt;
        __syncthreads();
    }

    // Eq. 5: the threads of a token take eight channels each at a time
    constexpr int TPT = kThreads / TOK;
    const int t = tid / TPT;
    if (t >= mine) return;
    mt = 0.0f;
    for (int c = 0; c < C; ++c) mt = fmaxf(mt, s_max[c][t]);
    float d = __fdiv_rn(__fmul_rn(p.clip_ratio, mt), p.qmax);
    float inv;
    if (d >= FLT_MIN) {
        inv = __fdiv_rn(1.0f, d);
    } else {
        d = 0.0f;
        inv = 0.0f;
    }
    if (rank == 0 && tid % TPT == 0) p.delta[t0 + t] = d;
    const int width = (item1 - item0) * OUT;
    const float* ut = s_u + t * p.u_pitch;
    uint8_t* dst = p.codes + ((t0 + t) * (int64_t)p.K + item0 * OUT) * p.bits / 8;
    for (int c = tid % TPT * 8; c < width; c += TPT * 8) {
        const float4 a = *reinterpret_cast<const float4*>(ut + c), e = *reinterpret_cast<const float4*>(ut + c + 4);
        const float v[8] = {a.x, a.y, a.z, a.w, e.x, e.y, e.z, e.w};
        uint32_t q[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            q[i] = __float_as_uint(__fadd_rn(fminf(fmaxf(__fmul_rn(v[i], inv), -p.qmax), p.qmax), 12582912.0f));
        if (p.bits == 4) *reinterpret_cast<uint32_t*>(dst + c / 2) = pack_word<0>(q);
        else *reinterpret_cast<uint2*>(dst + c) = make_uint2(pack_word<1>(q), pack_word<1>(q + 4));
    }
}

// *p is complete but for the sizes.
template <typename XT, int BETA, int TOK>
cudaError_t launch_quantize_tok(const CompositeParams& p, const CompositePlan& f, cudaStream_t stream) {
    auto kern = composite_quantize_kernel<XT, BETA, TOK>;
    const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), f.smem);
    if (e != cudaSuccess) return e;
    const cudaError_t launched = launch_pdl(kern, (unsigned)f.grid, (unsigned)kThreads, f.smem, stream, 1u << f.ctas_shift, p);
    return f.ctas_shift > 0 && cluster_refused(launched) ? cudaErrorNotSupported : launched;
}
template <typename XT, int BETA>
cudaError_t launch_quantize(CompositeParams p, cudaStream_t stream) {
    const CompositePlan f = plan_composite(p.rows, p.K, (int)sizeof(XT), BETA, device_sm_count(), cluster_capacity);
    if (f.tok == 0) return cudaErrorNotSupported;
    p.items = f.items; p.ctas_shift = f.ctas_shift; p.u_pitch = f.u_pitch; p.span = f.span;
    p.off_u = f.off_u; p.off_b = f.off_b; p.off_p = f.off_p; p.off_s = f.off_s;
    if constexpr (BETA >= 32) {
        if (f.tok == 8) return launch_quantize_tok<XT, BETA, 8>(p, f, stream);
    }
    return launch_quantize_tok<XT, BETA, 16>(p, f, stream);
}
template <typename XT>
cudaError_t launch_quantize_beta(int beta, const CompositeParams& p, cudaStream_t stream) {
    switch (beta) {
        case 16: return launch_quantize<XT, 16>(p, stream);
        case 32: return launch_quantize<XT, 32>(p, stream);
        case 64: return launch_quantize<XT, 64>(p, stream);
        case 128: return launch_quantize<XT, 128>(p, stream);
        case 256: return launch_quantize<XT, 256>(p, stream);
        default: return cudaErrorNotSupported;
    }
}

template <typename XT, int BETA>
cudaError_t launch_beta(const XT* x, int64_t rows, int K, int64_t ldx, const float* diag, const int32_t* perm,
                        const float* blocks, float* u, cudaStream_t stream) {
    constexpr int TOK = (kThreads / BETA) * 8;
    const int64_t tiles = (rows + TOK - 1) / TOK;
    if (tiles > 65535) return cudaErrorInvalidConfiguration;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(K / BETA), (unsigned)tiles, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, composite_rotate_kernel<XT, BETA>, x, rows, K, ldx, diag, perm, blocks, u);
}

template <typename XT>
cudaError_t launch_xt(const XT* x, int64_t rows, int K, int64_t ldx, const float* diag, const int32_t* perm,
                      const float* blocks, int beta, float* u, cudaStream_t stream) {
    switch (beta) {
        case 16: return launch_beta<XT, 16>(x, rows, K, ldx, diag, perm, blocks, u, stream);
        case 32: return launch_beta<XT, 32>(x, rows, K, ldx, diag, perm, blocks, u, stream);
        case 64: return launch_beta<XT, 64>(x, rows, K, ldx, diag, perm, blocks, u, stream);
        case 128: return launch_beta<XT, 128>(x, rows, K, ldx, diag, perm, blocks, u, stream);
        case 256: return launch_beta<XT, 256>(x, rows, K, ldx, diag, perm, blocks, u, stream);
        default: return cudaErrorNotSupported;
    }
}

__global__ void perm_check_kernel(const int32_t* __restrict__ perm, int K, int* __restrict__ bad) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < K && (perm[c] < 0 || perm[c] >= K)) *bad = 1;
}

}  // namespace

cudaError_t launch_composite_rotate(const void* x, fq_dtype xt, int64_t rows, int64_t K, int64_t ldx, const float* diag,
                                    const int32_t* perm, const float* blocks, int beta, float* u, cudaStream_t stream) {
    if (rows == 0) return cudaSuccess;
    if (xt == FQ_F32)
        return launch_xt(static_cast<const float*>(x), rows, (int)K, ldx, diag, perm, blocks, beta, u, stream);
    return launch_xt(static_cast<const __nv_bfloat16*>(x), rows, (int)K, ldx, diag, perm, blocks, beta, u, stream);
}

cudaError_t launch_perm_check(const int32_t* perm, int64_t K, int* bad_flag, cudaStream_t stream) {
    perm_check_kernel<<<(unsigned)((K + 255) / 256), 256, 0, stream>>>(perm, (int)K, bad_flag);
    return cudaGetLastError();
}

// The runtime prologue in one launch, or cudaErrorNotSupported where the rows of eight tokens do not fit shared memory.
cudaError_t launch_composite_quantize(const void* x, fq_dtype xt, int64_t rows, int64_t K, int64_t ldx, const float* diag,
                                      const int32_t* perm, const float* blocks, int beta, int bits, float clip_ratio,
                                      void* codes, float* delta, cudaStream_t stream) {
    if (reinterpret_cast<uintptr_t>(blocks) & 15u) return cudaErrorNotSupported;
    CompositeParams p{};
    p.x = x; p.ldx = ldx; p.rows = rows; p.K = (int)K; p.bits = bits;
    p.vec = (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && (size_t)ldx * (xt == FQ_BF16 ? 2 : 4) % 16 == 0 ? 1 : 0;
    p.diag = diag; p.perm = perm; p.blocks = blocks;
    p.clip_ratio = clip_ratio; p.qmax = bits == 4 ? 7.0f : 127.0f;
    p.codes = static_cast<uint8_t*>(codes); p.delta = delta;
    return xt == FQ_BF16 ? launch_quantize_beta<__nv_bfloat16>(beta, p, stream) : launch_quantize_beta<float>(beta, p, stream);
}

}  // namespace fq
