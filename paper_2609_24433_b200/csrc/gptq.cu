// GPTQ rounding in transformed coordinates (offline; section "Rounding and native execution", Eq. 7):
//   min_Q ||(W~ - Q) Z||_F^2,  G = Z Z^T, H = G + lambda I,  H^-1 = U^T U (U upper triangular),
// channels rounded one after the other, each rounding error spread along the row of U over the channels
// still to come.  Everything here decides integer codes, so all arithmetic is binary32 in a fixed order
// (fused multiply-add chains in ascending index): results do not depend on how the work is split over
// threads, only on these definitions.
//   transform_rows    z = (I (x) H_beta)(x (.) mult): the prologue's transform without its quantizer
//   gram              G[a][b] = sum_t z[t][a] z[t][b], t ascending
//   damp              lambda = damp * (sum_a G[a][a]) / K (sum in ascending a); dead channels (G[a][a] = 0) get 1
//   factor            columns j = K-1 .. 0 of the upper factor M of H = M M^T, and U = M^-1 row by row behind it
//   rev_chol_col, tri_inverse    the same two for rows too long for the factor kernel's shared memory
//                     (M stored transposed there: Mt[k][i] = M[i][k])
//   sweep             per weight row, channels i = 0 .. K-1: code, error, update of the channels j > i
#include <cuda_bf16.h>
#include <float.h>

#include "fq_common.cuh"
#include "ptx_sm100.cuh"

namespace fq {
namespace {

template <typename XT>
__device__ __forceinline__ float ld_f32(const XT* p);
template <>
__device__ __forceinline__ float ld_f32<float>(const float* p) { return __ldg(p); }
template <>
__device__ __forceinline__ float ld_f32<__nv_bfloat16>(const __nv_bfloat16* p) {
    return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p)) << 16);
}

// One CTA per row; the row lives in shared memory (K floats) while the butterflies run.
template <typename XT>
__global__ void __launch_bounds__(256)
transform_rows_kernel(const XT* __restrict__ x, int K, int64_t ldx, const float* __restrict__ mult, float cnorm,
                      int block, float* __restrict__ z) {
    extern __shared__ float s_v[];
    const int64_t r = blockIdx.x;
    for (int c = threadIdx.x; c < K; c += blockDim.x)
        s_v[c] = __fmul_rn(ld_f32<XT>(x + r * ldx + c), mult ? __ldg(mult + c) : cnorm);
    for (int h = 1; h < block; h <<= 1) {
        __syncthreads();
        for (int p = threadIdx.x; p < K / 2; p += blockDim.x) {
            const int i = ((p / h) * 2 * h) + (p % h);        // the pair (i, i + h), i & h == 0
            const float a = s_v[i], b = s_v[i + h];
            s_v[i] = __fadd_rn(a, b);
            s_v[i + h] = __fsub_rn(a, b);
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < K; c += blockDim.x) z[r * K + c] = s_v[c];
}

// G[a][b] for the tiles on and above the diagonal (nothing below it is ever read): 64 x 64 outputs per CTA of 128
// threads, 8 x 4 per thread, tokens staged 32 at a time through two cp.async buffers.  Every output is one chain of
// fused multiply-adds over ascending t, so the 32 accumulators of a thread are its instruction parallelism.  Bound by
// the FMA pipe: K = 2048, Mc = 4096 takes 0.45 ms (8.7 G multiply-adds above the diagonal); one output per thread over
// the full square took 5.1 ms, bound by its two shared-memory reads per multiply-add.
constexpr int kGramTile = 64, kGramTok = 32;
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__global__ void __launch_bounds__(128)
gram_kernel(const float* __restrict__ z, int64_t Mc, int K, float* __restrict__ G) {
    __shared__ __align__(16) float s_a[2][kGramTok][kGramTile], s_b[2][kGramTok][kGramTile];
    // the CTA's tile on or above the diagonal: row of tiles ty holds the tiles tx >= ty
    const int tiles = (K + kGramTile - 1) / kGramTile;
    int ty = 0, left = blockIdx.x;
    while (left >= tiles - ty) { left -= tiles - ty; ++ty; }
    const int a0 = ty * kGramTile, b0 = (ty + left) * kGramTile;
    const int ra = (threadIdx.x >> 4) * 8, rb = (threadIdx.x & 15) * 4;
    auto stage = [&](int buf, int64_t t0) {          // tokens past Mc and channels past K arrive as zeros
#pragma unroll
        for (int q = 0; q < kGramTok * kGramTile / 4 / 128; ++q) {
            const int o = q * 128 + threadIdx.x, t = o / (kGramTile / 4), c = o % (kGramTile / 4) * 4;
            const bool row = t0 + t < Mc;
            const float* zr = z + (row ? t0 + t : 0) * K;
            const bool oka = row && a0 + c < K, okb = row && b0 + c < K;
            cp_async16(smem_u32(&s_a[buf][t][c]), zr + (oka ? a0 + c : 0), oka);
            cp_async16(smem_u32(&s_b[buf][t][c]), zr + (okb ? b0 + c : 0), okb);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    auto multiply = [&](int buf, int k) {
        const float4 p = *reinterpret_cast<const float4*>(&s_a[buf][k][ra]);
        const float4 q = *reinterpret_cast<const float4*>(&s_a[buf][k][ra + 4]);
        const float4 r = *reinterpret_cast<const float4*>(&s_b[buf][k][rb]);
        const float av[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w}, bv[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = __fmaf_rn(av[i], bv[j], acc[i][j]);
    };
    stage(0, 0);
    int buf = 0;
    for (int64_t t0 = 0; t0 < Mc; t0 += kGramTok, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                             // this buffer has landed for everyone, the other one has been read
        if (t0 + kGramTok < Mc) stage(buf ^ 1, t0 + kGramTok);
        if (Mc - t0 >= kGramTok) {
#pragma unroll 8
            for (int k = 0; k < kGramTok; ++k) multiply(buf, k);
        } else {
            for (int k = 0; k < (int)(Mc - t0); ++k) multiply(buf, k);
        }
    }
    if (b0 + rb < K)
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (a0 + ra + i < K)
                *reinterpret_cast<float4*>(G + (int64_t)(a0 + ra + i) * K + b0 + rb) =
                    make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
}

// The diagonal is gathered by all threads first: the sum over ascending channels is one thread's chain.
__global__ void __launch_bounds__(1024)
damp_kernel(float* __restrict__ H, int K, float damp, uint8_t* __restrict__ dead) {
    extern __shared__ float s_diag[];
    __shared__ float s_lambda;
    for (int a = threadIdx.x; a < K; a += blockDim.x) s_diag[a] = H[(int64_t)a * K + a];
    __syncthreads();
    if (threadIdx.x == 0) {
        float sum = 0.0f;
#pragma unroll 16
        for (int a = 0; a < K; ++a) sum = __fadd_rn(sum, s_diag[a]);
        s_lambda = __fmul_rn(damp, __fdiv_rn(sum, (float)K));
    }
    __syncthreads();
    for (int a = threadIdx.x; a < K; a += blockDim.x) {
        float d = s_diag[a];
        const bool is_dead = d == 0.0f;
        dead[a] = is_dead ? 1 : 0;
        if (is_dead) d = 1.0f;
        H[(int64_t)a * K + a] = __fadd_rn(d, s_lambda);
    }
}

// ---- factor and inverse in one cooperative kernel (K up to what shared memory holds: 2176 channels on 148 SMs) --------
// Every entry of M and of U is a chain over ascending k, NEWEST column first: M[i][j] starts with the term of column
// j + 1, which was finished one step ago.  So nothing of a chain can be summed ahead of time, and the factorisation
// takes at least sum_j (K - 1 - j) dependent multiply-adds: 2.1 M at K = 2048, 4.3 ms at four cycles each.  What this
// kernel does is come close to that: the operands of the chains are in shared memory, the inverse runs beside
// the factorisation, one row behind, and the CTAs meet once per eight columns.
//   - Rows i of M are dealt to the CTAs cyclically (i = cta + G m: equal lengths everywhere), one lane of warp 0 each,
//     the finished part of a row in shared memory.
//   - The rows of the eight columns in work (the window) are kept by EVERY CTA, computed redundantly by eight more
//     lanes of the same warp: within a block of eight columns nothing has to come from another CTA.  At the end of a
//     block each CTA publishes its rows' eight new entries, the grid meets, and the next window is read through L2.
//   - Warp 1 owns columns c = cta + G m of U.  U[i][c] needs row i of M, which the window holds when column i is done:
//     it works on row j + 1 while warp 0 works on column j.
// Lanes read their rows four entries at a time; the rows' bases are spread over the banks (4 words apart mod 32).
// K = 2048: 6.95 ms for both (44 ms for 2048 launches of a column kernel and 110 ms for the inverse before).
constexpr int kWin = 8;                    // columns per block = rows of the window
constexpr int kWinSlots = kWin + 1;        // + the row the inverse still reads while the next window is being loaded
constexpr int kFactorThreads = 256;
constexpr int kFactorMaxRows = 32 - kWin;  // own rows per CTA: the lanes the window leaves
constexpr int kUPad = 16;                  // zeros behind a column of U: its chains run in whole chunks

// Start of a region of shared memory for lane `l` at or behind `at` words, in the lane's bank group.
__host__ __device__ inline int bank_base(int at, int l) { return (at + 31) / 32 * 32 + 4 * (l & 7); }
// Words of shared memory: the window's slots, then the rows of M and the columns of U of the CTA that has most.
__host__ __device__ inline int window_stride(int K) { return bank_base(K + kUPad, 1); }      // = 4 mod 32
inline size_t factor_smem_words(int K, int G) {
    int at = kWinSlots * window_stride(K);
    for (int m = 0; m * G < K; ++m) at = bank_base(at, m) + K - m * G / 32 * 32;               // row i keeps k >= i
    for (int m = 0; m * G < K; ++m) {
        const int c = m * G + G - 1 < K ? m * G + G - 1 : K - 1;
        at = bank_base(at, m) + c + 1 + kUPad;
    }
    return (size_t)at;
}

struct FactorParams {
    float* H;             // [K][K]: H above the diagonal on entry; finished columns of M replace it row by row
    float* U;             // [K][K]: entries on and above the diagonal
    int K;
    uint32_t* arrivals;   // grid barrier: CTAs counted in so far, zeroed by the host
    int* bad;             // bit 0: not positive definite, bit 1: the grid barrier gave up
};

// acc -+ sum_k a[k] b[k] over `n` entries, n a multiple of 8, both 16-byte aligned; two chunks of 16 alternate, the
// loads of one in flight while the other is summed.  NEG: subtract the products (fma(-a, b, acc)).
template <bool NEG>
__device__ __forceinline__ float chain(const float* a, const float* b, int n, float acc) {
    const float4 *pa = reinterpret_cast<const float4*>(a), *pb = reinterpret_cast<const float4*>(b);
    struct Chunk { float4 x[4], y[4]; };
    auto step = [&](const float4& x, const float4& y) {
        acc = __fmaf_rn(NEG ? -x.x : x.x, y.x, acc);
        acc = __fmaf_rn(NEG ? -x.y : x.y, y.y, acc);
        acc = __fmaf_rn(NEG ? -x.z : x.z, y.z, acc);
        acc = __fmaf_rn(NEG ? -x.w : x.w, y.w, acc);
    };
    auto load = [&](Chunk& c) {
#pragma unroll
        for (int q = 0; q < 4; ++q) { c.x[q] = pa[q]; c.y[q] = pb[q]; }
        pa += 4; pb += 4;
    };
    auto sum = [&](const Chunk& c) {
#pragma unroll
        for (int q = 0; q < 4; ++q) step(c.x[q], c.y[q]);
    };
    if (n & 8) {
        const float4 x0 = pa[0], x1 = pa[1], y0 = pb[0], y1 = pb[1];
        step(x0, y0); step(x1, y1);
        pa += 2; pb += 2;
    }
    n >>= 4;
    if (n == 0) return acc;
    Chunk c0, c1;
    load(c0);
    for (; n > 2; n -= 2) {
        load(c1);
        sum(c0);
        load(c0);
        sum(c1);
    }
    if (n == 2) {
        load(c1);
        sum(c0);
        sum(c1);
    } else {
        sum(c0);
    }
    return acc;
}

// The up to seven entries k0 <= k < k1 ahead of a multiple of 8: all loads first, then the chain.
template <bool NEG>
__device__ __forceinline__ float chain_head(const float* a, const float* b, int k0, int k1, float acc) {
    float x[kWin - 1], y[kWin - 1];
#pragma unroll
    for (int q = 0; q < kWin - 1; ++q) {
        x[q] = k0 + q < k1 ? a[k0 + q] : 0.0f;
        y[q] = k0 + q < k1 ? b[k0 + q] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < kWin - 1; ++q)
        if (k0 + q < k1) acc = __fmaf_rn(NEG ? -x[q] : x[q], y[q], acc);
    return acc;
}

__global__ void __launch_bounds__(kFactorThreads, 1)
gptq_factor_kernel(const FactorParams p) {
    extern __shared__ __align__(128) float s_mem[];
    __shared__ float s_hw[kWin][kWin];                   // H of the window's rows at the block's columns
    __shared__ float s_ho[kFactorMaxRows][kWin];         // ... of this CTA's rows
    __shared__ int s_row[kFactorMaxRows], s_col[32];     // s_mem index of entry k = 0 of a row of M / a column of U
    __shared__ int s_abort;
    const int K = p.K, G = (int)gridDim.x, cta = (int)blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wstride = window_stride(K);
    const int own = cta < K ? (K - 1 - cta) / G + 1 : 0; // rows of M, and columns of U, of this CTA

    for (int o = tid; o < kWinSlots * wstride; o += kFactorThreads) s_mem[o] = 0.0f;    // (the slots' tails stay zero)
    if (tid == 0) {
        s_abort = 0;
        int at = kWinSlots * wstride;
        for (int m = 0; m < own; ++m) {
            const int first = (cta + m * G) / 32 * 32;
            s_row[m] = bank_base(at, m) - first;
            at = s_row[m] + K;
        }
        for (int m = 0; m < own; ++m) {
            s_col[m] = bank_base(at, m);
            at = s_col[m] + cta + m * G + 1 + kUPad;
        }
    }
    __syncthreads();
    for (int m = 0; m < own; ++m)
        if (tid < kUPad) s_mem[s_col[m] + cta + m * G + 1 + tid] = 0.0f;

    auto slot = [&](int row) { return s_mem + (row % kWinSlots) * wstride; };
    // U[i][c] for this lane's column c, row i of M in its slot
    auto inverse_row = [&](int i) {
        if (lane >= own) return;
        const int c = cta + lane * G;
        if (c < i) return;
        const float* m = slot(i);
        float* u = s_mem + s_col[lane];
        const float d = m[i];
        float v;
        if (c == i) {
            v = __fdiv_rn(1.0f, d);
        } else {
            float acc = 0.0f;
            const int a = (i + 8) & ~7;                  // first multiple of 8 behind i; entries past c are zeros
            acc = chain_head<false>(m, u, i + 1, a, acc);
            if (a <= c) acc = chain<false>(m + a, u + a, (c - a) / 8 * 8 + 8, acc);
            v = __fdiv_rn(-acc, d);
        }
        u[i] = v;
        p.U[(int64_t)i * K + c] = v;
    };

    uint32_t target = 0;
    for (int j0 = K - kWin; j0 >= 0; j0 -= kWin) {
        // the window's rows behind the block (published by their owners before the last meeting), and H at the block
        const int n4 = (K - j0 - kWin) / 4;
        for (int o = tid; o < kWin * n4; o += kFactorThreads) {
            const int r = o / n4, k = j0 + kWin + (o - r * n4) * 4;
            *reinterpret_cast<float4*>(slot(j0 + r) + k) = __ldcg(reinterpret_cast<const float4*>(p.H + (int64_t)(j0 + r) * K + k));
        }
        for (int o = tid; o < kWin * kWin; o += kFactorThreads)
            s_hw[o / kWin][o % kWin] = __ldcg(p.H + (int64_t)(j0 + o / kWin) * K + j0 + o % kWin);
        for (int o = tid; o < own * kWin; o += kFactorThreads) {
            const int i = cta + o / kWin * G;
            if (i < j0) s_ho[o / kWin][o % kWin] = __ldcg(p.H + (int64_t)i * K + j0 + o % kWin);
        }
        __syncthreads();
        if (warp < 2) {
#pragma unroll 1
            for (int jj = kWin - 1; jj >= 0; --jj) {
                const int j = j0 + jj;
                if (warp == 0) {
                    const float* mj = slot(j);
                    const int m = lane - kWin;
                    const bool in_window = lane < kWin;
                    const bool active = in_window ? lane <= jj : (m < own && cta + m * G < j0);
                    float* mi = active && !in_window ? s_mem + s_row[m] : slot(j0 + (in_window ? lane : 0));
                    // No branch around the chain: lanes without a row work on the window's first and keep nothing.  (As
                    // `if (active)` the lanes' chains were executed in two parts: 11.6 instead of 6.95 ms for the kernel.)
                    __syncwarp();
                    float acc = in_window ? s_hw[lane][jj] : s_ho[active ? m : 0][jj];
                    acc = chain_head<true>(mi, mj, j + 1, j0 + kWin, acc);
                    acc = chain<true>(mi + j0 + kWin, mj + j0 + kWin, K - j0 - kWin, acc);
                    float dd = __shfl_sync(0xffffffffu, acc, jj);
                    if (!(dd > 0.0f)) {
                        if (lane == 0) atomicOr(p.bad, 1);
                        dd = 1.0f;
                    }
                    const float d = __fsqrt_rn(dd);
                    if (active) mi[j] = lane == jj ? d : __fdiv_rn(acc, d);
                } else if (j + 1 < K) {
                    inverse_row(j + 1);
                }
                asm volatile("bar.sync 1, 64;" ::: "memory");
            }
        }
        if (j0 == 0) break;
        if (warp == 0 && lane < own && cta + lane * G < j0) {
            const float4* src = reinterpret_cast<const float4*>(s_mem + s_row[lane] + j0);
            float4* dst = reinterpret_cast<float4*>(p.H + (int64_t)(cta + lane * G) * K + j0);
            __stcg(dst, src[0]);
            __stcg(dst + 1, src[1]);
            __threadfence();
        }
        target += (uint32_t)G;
        if (warp == 0) {
            __syncwarp();
            if (lane == 0) {
                atomicAdd(p.arrivals, 1u);
                const uint64_t t0 = global_timer_ns();
                uint32_t seen;
                for (;;) {
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(p.arrivals) : "memory");
                    if (seen >= target) break;
                    if (global_timer_ns() - t0 > kWaitLimitNs) { s_abort = 1; atomicOr(p.bad, 2); break; }
                }
            }
        }
        __syncthreads();
        if (s_abort) return;
    }
    if (warp == 1) inverse_row(0);
}

// Column j of M (H = M M^T, M upper triangular), stored as row j of Mt.  Every CTA first copies the
// finished entries M[j][k], k > j, into shared memory (all threads load, so the strided reads overlap),
// then recomputes the diagonal entry from them (one chain of at most K terms) instead of waiting for
// another CTA to publish it; the off-diagonal chains read the same copy.
__global__ void __launch_bounds__(256)
rev_chol_col_kernel(const float* __restrict__ H, float* __restrict__ Mt, int K, int j, int* __restrict__ bad) {
    extern __shared__ float s_mj[];                  // K floats: s_mj[k - j - 1] = M[j][k]
    __shared__ float s_d;
    const int n = K - 1 - j;
    for (int o = threadIdx.x; o < n; o += blockDim.x) s_mj[o] = Mt[(int64_t)(j + 1 + o) * K + j];
    __syncthreads();
    if (threadIdx.x == 0) {
        float acc = H[(int64_t)j * K + j];
        for (int o = 0; o < n; ++o) acc = __fmaf_rn(-s_mj[o], s_mj[o], acc);
        if (!(acc > 0.0f)) { *bad = 1; acc = 1.0f; }
        s_d = __fsqrt_rn(acc);
    }
    __syncthreads();
    const float d = s_d;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == j) Mt[(int64_t)j * K + j] = d;
    if (i < j) {
        // sixteen loads in flight ahead of the (sequential) chain: the loop is bound by their latency otherwise
        float acc = H[(int64_t)i * K + j];
        const float* col = Mt + (int64_t)(j + 1) * K + i;
        int o = 0;
        if (n >= 32) {
            float cur[32], nxt[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) cur[q] = col[(int64_t)q * K];
            for (; o + 64 <= n; o += 32) {           // the next batch is requested before this one is consumed
#pragma unroll
                for (int q = 0; q < 32; ++q) nxt[q] = col[(int64_t)(o + 32 + q) * K];
#pragma unroll
                for (int q = 0; q < 32; ++q) acc = __fmaf_rn(-cur[q], s_mj[o + q], acc);
#pragma unroll
                for (int q = 0; q < 32; ++q) cur[q] = nxt[q];
            }
#pragma unroll
            for (int q = 0; q < 32; ++q) acc = __fmaf_rn(-cur[q], s_mj[o + q], acc);
            o += 32;
        }
        for (; o < n; ++o) acc = __fmaf_rn(-col[(int64_t)o * K], s_mj[o], acc);
        Mt[(int64_t)j * K + i] = __fdiv_rn(acc, d);
    }
}

// U = M^-1: column c from row c upwards; U row-major [K][K], zeros below the diagonal.
__global__ void __launch_bounds__(128)
tri_inverse_kernel(const float* __restrict__ Mt, float* __restrict__ U, int K) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= K) return;
    for (int i = K - 1; i > c; --i) U[(int64_t)i * K + c] = 0.0f;
    U[(int64_t)c * K + c] = __fdiv_rn(1.0f, Mt[(int64_t)c * K + c]);
    for (int i = c - 1; i >= 0; --i) {
        float acc = 0.0f;
        int k = i + 1;
        for (; k + 8 <= c + 1; k += 8) {             // eight pairs of loads in flight ahead of the chain
            float m[8], u[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) { m[q] = Mt[(int64_t)(k + q) * K + i]; u[q] = U[(int64_t)(k + q) * K + c]; }
#pragma unroll
            for (int q = 0; q < 8; ++q) acc = __fmaf_rn(m[q], u[q], acc);
        }
        for (; k <= c; ++k) acc = __fmaf_rn(Mt[(int64_t)k * K + i], U[(int64_t)k * K + c], acc);
        U[(int64_t)i * K + c] = __fdiv_rn(-acc, Mt[(int64_t)i * K + i]);
    }
}

// The sweep is independent per weight row: a CTA keeps ROWS rows in shared memory and walks the channels in blocks of 32.
// Within a block a warp has a row and a lane a channel: 32 steps of code, error and update of the lanes behind, the
// error's division being the step's latency.  The channels behind the block then take all 32 errors at once, each in
// one chain over ascending i -- the same operations in the same order as channel by channel -- four columns and up to
// four rows per thread, so that U is read 16 bytes per 16 multiply-adds and the CTA meets twice per block instead of
// twice per channel.  K = 2048, N = 2560: 0.98 ms (3.9 ms channel by channel).
template <int BITS, int ROWS>
__global__ void __launch_bounds__(256)
gptq_sweep_kernel(const float* __restrict__ Wt, int64_t N, int K, const float* __restrict__ U,
                  const uint8_t* __restrict__ dead, const float* __restrict__ w_scale, uint8_t* __restrict__ codes) {
    constexpr int kPer = ROWS < 4 ? ROWS : 4;        // rows per thread in the update
    constexpr int kColThreads = 256 / (ROWS / kPer);
    extern __shared__ __align__(16) float s_w[];     // [ROWS][K]
    __shared__ __align__(16) float s_e[32][ROWS];    // the block's errors, negated
    __shared__ float s_u[32][33];                    // U at the block's rows and columns
    __shared__ uint8_t s_dead[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * ROWS;
    for (int o = tid * 4; o < ROWS * K; o += 256 * 4) {
        const int r = o / K, c = o - r * K;
        *reinterpret_cast<float4*>(s_w + o) = r0 + r < N ? *reinterpret_cast<const float4*>(Wt + (r0 + r) * K + c)
                                                         : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    const float qmax = BITS == 4 ? 7.0f : 127.0f;
    const int64_t row = r0 + warp;
    const bool has_row = warp < ROWS && row < N;
    float s = 0.0f, inv = 0.0f;
    if (has_row) {
        s = w_scale[row];
        inv = s >= FLT_MIN ? __fdiv_rn(1.0f, s) : 0.0f;
    }
    auto fetch_u = [&](int i0, float* u) {           // this thread's four entries of the block's square of U
#pragma unroll
        for (int q = 0; q < 4; ++q) u[q] = __ldg(U + (int64_t)(i0 + q * 8 + warp) * K + i0 + lane);
    };
    float u_next[4];
    fetch_u(0, u_next);
    for (int i0 = 0; i0 < K; i0 += 32) {
#pragma unroll
        for (int q = 0; q < 4; ++q) s_u[q * 8 + warp][lane] = u_next[q];
        if (tid < 32) s_dead[tid] = dead[i0 + tid];
        __syncthreads();
        if (i0 + 32 < K) fetch_u(i0 + 32, u_next);
        if (warp < ROWS) {
            float w = s_w[warp * K + i0 + lane];
            int code = 0;
#pragma unroll 4
            for (int q = 0; q < 32; ++q) {
                float wi = __shfl_sync(0xffffffffu, w, q);
                if (s_dead[q]) wi = 0.0f;
                float t = rintf(__fmul_rn(wi, inv));
                t = fminf(fmaxf(t, -qmax), qmax);
                const float e = -__fdiv_rn(__fsub_rn(wi, __fmul_rn(t, s)), s_u[q][q]);
                if (lane == q) {
                    code = (int)t;
                    s_e[q][warp] = e;
                }
                if (lane > q) w = __fmaf_rn(e, s_u[q][lane], w);
            }
            const int odd = __shfl_down_sync(0xffffffffu, code, 1);
            if (has_row) {
                if (BITS == 8) codes[row * (int64_t)K + i0 + lane] = (uint8_t)(int8_t)code;
                else if ((lane & 1) == 0) codes[row * (int64_t)(K / 2) + (i0 + lane) / 2] = (uint8_t)((code & 15) | ((odd & 15) << 4));
            }
        }
        __syncthreads();
        const int rg = tid / kColThreads * kPer;
        for (int j = i0 + 32 + tid % kColThreads * 4; j < K; j += kColThreads * 4) {
            float4 w[kPer];
#pragma unroll
            for (int r = 0; r < kPer; ++r) w[r] = *reinterpret_cast<const float4*>(s_w + (rg + r) * K + j);
            const float* up = U + (int64_t)i0 * K + j;
#pragma unroll 8
            for (int q = 0; q < 32; ++q) {
                const float4 u = __ldg(reinterpret_cast<const float4*>(up + (int64_t)q * K));
#pragma unroll
                for (int r = 0; r < kPer; ++r) {
                    const float e = s_e[q][rg + r];
                    w[r].x = __fmaf_rn(e, u.x, w[r].x);
                    w[r].y = __fmaf_rn(e, u.y, w[r].y);
                    w[r].z = __fmaf_rn(e, u.z, w[r].z);
                    w[r].w = __fmaf_rn(e, u.w, w[r].w);
                }
            }
#pragma unroll
            for (int r = 0; r < kPer; ++r) *reinterpret_cast<float4*>(s_w + (rg + r) * K + j) = w[r];
        }
        // (the next block's first meeting separates this update from its readers; s_e is rewritten behind it)
    }
}

}  // namespace

cudaError_t launch_transform_rows(const void* x, fq_dtype xt, int64_t rows, int64_t K, int64_t ldx, const float* mult,
                                  float cnorm, int block, float* z, cudaStream_t stream) {
    if (rows == 0) return cudaSuccess;
    const size_t smem = sizeof(float) * (size_t)K;
    auto run = [&](auto kern, auto* p) -> cudaError_t {
        const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
        if (e != cudaSuccess) return e;
        kern<<<(unsigned)rows, 256, smem, stream>>>(p, (int)K, ldx, mult, cnorm, block, z);
        return cudaGetLastError();
    };
    return xt == FQ_F32 ? run(transform_rows_kernel<float>, static_cast<const float*>(x))
                        : run(transform_rows_kernel<__nv_bfloat16>, static_cast<const __nv_bfloat16*>(x));
}

// Whether factor and inverse of this width run in the cooperative kernel: at most 24 rows per CTA, one CTA per SM
// (which its shared memory makes sure of), and everything within 227 KB.  On 148 SMs: K <= 2176.
bool gptq_factor_fits(int64_t K) {
    const int sms = device_sm_count();
    return K <= (int64_t)sms * kFactorMaxRows && sizeof(float) * factor_smem_words((int)K, sms) + 4096 <= 227 * 1024;
}

// H (K x K) from Z, damped; U = upper factor of H^-1.  flags: two device ints, zeroed by the caller; flags[0] has bit 0
// set if H is not positive definite in binary32 and bit 1 if the grid barrier gave up, flags[1] counts arrivals.
// H is scratch; Mt (K x K) only where gptq_factor_fits() says no, null otherwise.
cudaError_t launch_gptq_factor(const float* z, int64_t Mc, int64_t K, float damp, float* H, float* Mt, float* U,
                               uint8_t* dead, int* flags, cudaStream_t stream) {
    const int64_t tiles = (K + kGramTile - 1) / kGramTile;
    gram_kernel<<<(unsigned)(tiles * (tiles + 1) / 2), 128, 0, stream>>>(z, Mc, (int)K, H);
    const size_t row_smem = sizeof(float) * (size_t)K;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(damp_kernel), row_smem);
    if (e != cudaSuccess) return e;
    damp_kernel<<<1, 1024, row_smem, stream>>>(H, (int)K, damp, dead);
    if (gptq_factor_fits(K)) {
        const int sms = device_sm_count();
        const size_t smem = sizeof(float) * factor_smem_words((int)K, sms);
        e = ensure_dynamic_smem(reinterpret_cast<const void*>(gptq_factor_kernel), smem);
        if (e != cudaSuccess) return e;
        FactorParams p{H, U, (int)K, reinterpret_cast<uint32_t*>(flags + 1), flags};
        void* args[] = {&p};
        return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(gptq_factor_kernel), dim3((unsigned)sms),
                                           dim3(kFactorThreads), args, smem, stream);
    }
    e = cudaMemsetAsync(Mt, 0, sizeof(float) * (size_t)K * (size_t)K, stream);
    if (e != cudaSuccess) return e;
    e = ensure_dynamic_smem(reinterpret_cast<const void*>(rev_chol_col_kernel), row_smem);
    if (e != cudaSuccess) return e;
    for (int j = (int)K - 1; j >= 0; --j)
        rev_chol_col_kernel<<<(unsigned)(j / 256 + 1), 256, row_smem, stream>>>(H, Mt, (int)K, j, flags);
    tri_inverse_kernel<<<(unsigned)((K + 127) / 128), 128, 0, stream>>>(Mt, U, (int)K);
    return cudaGetLastError();
}

namespace {
template <int BITS, int ROWS>
cudaError_t launch_sweep_variant(const float* Wt, int64_t N, int64_t K, const float* U, const uint8_t* dead,
                                 const float* w_scale, uint8_t* codes, cudaStream_t stream) {
    const size_t smem = sizeof(float) * (size_t)ROWS * (size_t)K;
    const unsigned grid = (unsigned)((N + ROWS - 1) / ROWS);
    auto kern = gptq_sweep_kernel<BITS, ROWS>;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, 256, smem, stream>>>(Wt, N, (int)K, U, dead, w_scale, codes);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_gptq_sweep(const float* Wt, int64_t N, int64_t K, const float* U, const uint8_t* dead,
                              const float* w_scale, int bits, uint8_t* codes, cudaStream_t stream) {
    if (N == 0) return cudaSuccess;
    // rows of K floats per CTA: eight up to K = 4096 (three such CTAs share an SM at K = 2048), four up to 8192, two beyond
    // (128 KB each)
    if (K <= 4096)
        return bits == 4 ? launch_sweep_variant<4, 8>(Wt, N, K, U, dead, w_scale, codes, stream)
                         : launch_sweep_variant<8, 8>(Wt, N, K, U, dead, w_scale, codes, stream);
    if (K <= 8192)
        return bits == 4 ? launch_sweep_variant<4, 4>(Wt, N, K, U, dead, w_scale, codes, stream)
                         : launch_sweep_variant<8, 4>(Wt, N, K, U, dead, w_scale, codes, stream);
    return bits == 4 ? launch_sweep_variant<4, 2>(Wt, N, K, U, dead, w_scale, codes, stream)
                     : launch_sweep_variant<8, 2>(Wt, N, K, U, dead, w_scale, codes, stream);
}

}  // namespace fq
