// lbm_df64.cuh -- double-binary32 ("df64") arithmetic on the FP32 pipe, and
// the Peng-Robinson chemical potentials of Eqs. (9)-(12) with the interface
// term of Eq. (5) evaluated in it.
//
// GB300 executes binary64 at about 1/64 of the binary32 rate, so the
// thermodynamics that must keep binary64 accuracy (the mixture parameters of
// Eqs. (10)-(11), the logarithmic fugacity terms of Eq. (12) and the
// chemical-potential differences that make the force of Eq. (5)) are carried
// as unevaluated sums hi + lo of two binary32 numbers.  The building blocks
// are the classical error-free transformations:
//   TwoSum      s + e = a + b exactly              (Knuth, TAOCP 2, 4.2.2)
//   FastTwoSum  s + e = a + b exactly if |a| >= |b| (Dekker 1971)
//   TwoProd     p + e = a * b exactly, e = fma(a, b, -p)
// The relative error of every derived quantity is about 2^-44 (binary64: 2^-53,
// binary32: 2^-24); the tests compare ln f_i, mu_i and the force with the binary64
// oracle at that level.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace lbmfug {
namespace df {

struct F2 {
    float hi, lo;
};

// binary32 split of a binary64 constant (host or device, constant-folded)
__host__ __device__ constexpr float hi_of(double x) { return (float)x; }
__host__ __device__ constexpr float lo_of(double x) { return (float)(x - (double)(float)x); }

// The intrinsics below are never contracted into a fused multiply-add, which
// the error-free transformations rely on.
__device__ __forceinline__ F2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
    return {s, e};
}

// TwoSum of two non-negative numbers: FastTwoSum of the larger and the
// smaller, which is exact, so (s, e) equals two_sum's.  The operands are
// ordered by their bit patterns, which order non-negative binary32 numbers as
// their values and put a NaN above every number, so a NaN propagates.  Three
// additions on the FMA pipe and two integer min/max on the ALU pipe, against
// six additions.
__device__ __forceinline__ F2 two_sum_pos(float a, float b)
{
    const int ia = __float_as_int(a), ib = __float_as_int(b);
    const float big = __int_as_float(max(ia, ib)), small = __int_as_float(min(ia, ib));
    const float s = __fadd_rn(big, small);
    return {s, __fsub_rn(small, __fsub_rn(s, big))};
}

__device__ __forceinline__ F2 fast_two_sum(float a, float b)  // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    const float e = __fsub_rn(b, __fsub_rn(s, a));
    return {s, e};
}

__device__ __forceinline__ F2 two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, fmaf(a, b, -p)};
}

// a + b.  Absolute error about 2^-48 (|a| + |b|) (the "sloppy" double-word
// sum); the callers need absolute, not relative, accuracy of sums.
__device__ __forceinline__ F2 add(F2 a, F2 b)
{
    const F2 s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}

__device__ __forceinline__ F2 neg(F2 a) { return {-a.hi, -a.lo}; }

// a * b, relative error about 2^-46
__device__ __forceinline__ F2 mul(F2 a, F2 b)
{
    const F2 p = two_prod(a.hi, b.hi);
    return fast_two_sum(p.hi, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, p.lo)));
}

// binary32 reciprocal to about 1 ulp (the hardware approximation); callers
// refine or scale it so that its error stays below 2^-44 of the result
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ---- packed FP32x2 operations --------------------------------------------------
// One instruction does the binary32 operation on both lanes, each rounded as
// the scalar operation rounds it.  They are written in PTX with an explicit
// rounding mode, so that no compiler pass fuses a product into a following
// sum: the error-free transformations built on them need the same guarantee
// that __fmul_rn and __fadd_rn give the scalar routines.
__device__ __forceinline__ float2 vbc(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 vmul(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mov.b64 rc, {%6, %7};\n\tfma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return vfma(b, vbc(-1.0f), a); }

}  // namespace df
}  // namespace lbmfug
