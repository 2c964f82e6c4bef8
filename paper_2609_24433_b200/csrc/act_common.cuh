// Device helpers shared by the two prologue kernels.
#pragma once

#include <stdint.h>

namespace fq {

// Round-to-nearest-even code extraction: bits(t + 1.5*2^23) = 0x4B400000 + rint(t) for |t| < 2^22.
constexpr uint32_t kMagicBits = 0x4B400000u;

// Pack 8 four-bit (or 4 eight-bit) two's-complement codes from the raw bit patterns
// b[i] = kMagicBits + code_i (element 0 in the lowest field) with one shift-add per code:
// the Horner sum of the raw patterns equals the Horner sum of the codes plus a constant;
// adding half the field range to every field removes the borrows between fields, and
// flipping each field's top bit afterwards turns offset binary into two's complement.
template <int FMT>
__device__ __forceinline__ uint32_t pack_word(const uint32_t* b) {
    if (FMT == 0) {
        uint32_t w = b[7];
#pragma unroll
        for (int i = 6; i >= 0; --i) w = (w << 4) + b[i];
        return (w + (0x88888888u - kMagicBits * 0x11111111u)) ^ 0x88888888u;
    } else {
        // 8-bit codes: the low byte of every raw pattern already is the two's-complement code
        // (0x4B400000 + code has the code's low 8 bits in its lowest byte), so three byte permutes
        // gather the four bytes.
        uint32_t lo, hi, w;
        asm("prmt.b32 %0, %1, %2, 0x0040;" : "=r"(lo) : "r"(b[0]), "r"(b[1]));
        asm("prmt.b32 %0, %1, %2, 0x0040;" : "=r"(hi) : "r"(b[2]), "r"(b[3]));
        asm("prmt.b32 %0, %1, %2, 0x5410;" : "=r"(w) : "r"(lo), "r"(hi));
        return w;
    }
}

// Warp maximum of a non-negative float (an absolute-value maximum): non-negative IEEE values order
// like their bit patterns, so one integer warp reduction replaces five shuffle + max steps.
__device__ __forceinline__ float warp_max_nonneg(float m) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
}

// Channel (within a thread's run) that field i of 32-bit word j holds, per store format.
template <int FMT>
__device__ __forceinline__ constexpr int code_index(int j, int i) {
    return FMT == 0 ? 8 * j + i : (FMT == 1 ? 4 * j + i : 8 * (j / 2) + 2 * i + (j & 1));
}

// Packed binary32 arithmetic (two independent IEEE operations per instruction).  Written as PTX
// with an explicit rounding modifier: such instructions are never contracted into fused
// multiply-adds by the optimizer, which the bit-exact contract of the prologue depends on.
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) {
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(*reinterpret_cast<uint64_t*>(&d))
        : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)));
    return d;
}
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) {
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(*reinterpret_cast<uint64_t*>(&d))
        : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)));
    return d;
}
__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) {
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(*reinterpret_cast<uint64_t*>(&d))
        : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)),
          "l"(*reinterpret_cast<const uint64_t*>(&c)));
    return d;
}


// ---- gate non-linearity of a gated MLP ---------------------------------------------------------------------------
// act(x) = x * sigmoid(k), k = x (SiLU, kind 0) or k = 2 sqrt(2/pi) (x + 0.044715 x^3) (GELU, tanh form, kind 1), in
// fixed binary32 arithmetic.  exp(-k): argument clamped to [-87, 88], n = rint(a log2e), two-step reduction by ln2,
// degree-6 Taylor polynomial in Horner form, times 2^n from its exponent bits; then one IEEE division.  The product
// act(gate) * up feeds a quantizer, so every operation and its order are part of the definition.
__device__ __forceinline__ float exp_fixed(float a) {
    a = fminf(fmaxf(a, -87.0f), 88.0f);
    const float n = rintf(__fmul_rn(a, 1.44269504f));
    float r = __fmaf_rn(n, -0.693145752f, a);
    r = __fmaf_rn(n, -1.42860677e-06f, r);
    float p = 1.38888892e-03f;
    p = __fmaf_rn(p, r, 8.33333377e-03f);
    p = __fmaf_rn(p, r, 4.16666679e-02f);
    p = __fmaf_rn(p, r, 1.66666672e-01f);
    p = __fmaf_rn(p, r, 0.5f);
    p = __fmaf_rn(p, r, 1.0f);
    p = __fmaf_rn(p, r, 1.0f);
    return __fmul_rn(p, __int_as_float(((int)n + 127) << 23));
}
__device__ __forceinline__ float gate_act(float x, int kind) {
    float k = x;
    if (kind == 1) {
        const float x3 = __fmul_rn(__fmul_rn(x, x), x);
        k = __fmul_rn(1.59576917f, __fmaf_rn(0.044715f, x3, x));
    }
    return __fdiv_rn(x, __fadd_rn(1.0f, exp_fixed(-k)));
}
__device__ __forceinline__ float2 f2_const(float c) { return make_float2(c, c); }
__device__ __forceinline__ float rcp_approx(float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return r;
}
// k of gate_act for two values
__device__ __forceinline__ float2 gate_k(float2 x, int kind) {
    if (kind == 0) return x;
    const float2 x3 = f2_mul(f2_mul(x, x), x);
    return f2_mul(f2_const(1.59576917f), f2_fma(f2_const(0.044715f), x3, x));
}
// gate_act of two values, k clamped to [-88, 87] if it was outside.  The same roundings as gate_act, two at a time and
// without its slow parts:
//   - the reduction runs on -r (every rounding is symmetric in sign), so no operand has to be negated;
//   - rint by adding and subtracting 1.5 * 2^23, whose sum also carries n in its low bits: 2^n enters by one shift-add
//     on p's exponent (p is in (0.7, 1.42), and below 1 where n = 127: no overflow, and exact like the multiply);
//   - the quotient by an approximate reciprocal, one Newton step and one correction with the exact remainder (Markstein's
//     method: IBM J. Res. Dev. 34(1), 1990), all on a quarter of the denominator, whose reciprocal is never denormal.
// Equal to gate_act for every binary32 |x| < 8e37, both kinds (all of them were compared; the sign of a zero may differ,
// which no code depends on); four times a larger x could overflow.
__device__ __forceinline__ float2 gate_act_pair(float2 x, float2 k) {
    const float2 m = f2_mul(k, f2_const(-1.44269504f));
    const float2 t = f2_fma(m, f2_const(1.0f), f2_const(12582912.0f));
    const float2 n = f2_add(t, f2_const(-12582912.0f));
    float2 r = f2_fma(n, f2_const(0.693145752f), k);             // -r of exp_fixed
    r = f2_fma(n, f2_const(1.42860677e-06f), r);
    float2 p = f2_fma(f2_const(1.38888892e-03f), r, f2_const(-8.33333377e-03f));
    p = f2_fma(p, r, f2_const(4.16666679e-02f));
    p = f2_fma(p, r, f2_const(-1.66666672e-01f));
    p = f2_fma(p, r, f2_const(0.5f));
    p = f2_fma(p, r, f2_const(-1.0f));
    p = f2_fma(p, r, f2_const(1.0f));
    const float2 e = make_float2(__uint_as_float(__float_as_uint(p.x) + (__float_as_uint(t.x) << 23)),
                                 __uint_as_float(__float_as_uint(p.y) + (__float_as_uint(t.y) << 23)));
    const float2 nd = f2_fma(e, f2_const(-0.25f), f2_const(-0.25f));    // -(1 + e) / 4: the rounding of 1 + e
    float2 y = make_float2(rcp_approx(-nd.x), rcp_approx(-nd.y));
    y = f2_fma(y, f2_fma(nd, y, f2_const(1.0f)), y);
    const float2 q = f2_mul(x, y);
    return f2_mul(f2_fma(f2_fma(nd, q, x), y, q), f2_const(0.25f));
}
// g[i] = gate_act(g[i]) * u[i] for N pairs; the clamp of k is looked for once for all of them.
template <int N>
__device__ __forceinline__ void gate_product(float2* g, const float2* u, int kind) {
    float2 k[N];
    float kmax = 0.0f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        k[i] = gate_k(g[i], kind);
        asm("max.f32 %0, %0, %1, %2;" : "+f"(kmax) : "f"(fabsf(k[i].x)), "f"(fabsf(k[i].y)));
    }
    if (kmax > 87.0f) {
        float xmax = 0.0f;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            asm("max.f32 %0, %0, %1, %2;" : "+f"(xmax) : "f"(fabsf(g[i].x)), "f"(fabsf(g[i].y)));
            k[i] = make_float2(fminf(fmaxf(k[i].x, -88.0f), 87.0f), fminf(fmaxf(k[i].y, -88.0f), 87.0f));
        }
        if (xmax >= 8e37f) {
#pragma unroll 1
            for (int i = 0; i < N; ++i) {
                // (selected by comparison: an index that varies would put the arrays into local memory)
                float2 x = make_float2(0.0f, 0.0f), w = x;
#pragma unroll
                for (int j = 0; j < N; ++j)
                    if (j == i) { x = g[j]; w = u[j]; }
                x = make_float2(__fmul_rn(gate_act(x.x, kind), w.x), __fmul_rn(gate_act(x.y, kind), w.y));
#pragma unroll
                for (int j = 0; j < N; ++j)
                    if (j == i) g[j] = x;
            }
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) g[i] = f2_mul(gate_act_pair(g[i], k[i]), u[i]);
}

}  // namespace fq
