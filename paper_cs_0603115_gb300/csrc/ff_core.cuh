// ff_core.cuh -- device-side error-free transformations and float-float
// operators (Da Graca & Defour, Section 4.1), written with explicit
// round-to-nearest binary32 intrinsics so that the compiler can neither
// contract a multiply and an add into an FMA nor reassociate anything.  The
// only fused multiply-add is the explicit one of Mul12.
//
// A float-float value is a float2 {x = hi, y = lo}: the unevaluated sum
// hi + lo (the format of Section 4).
#pragma once
#include <cuda_runtime.h>

namespace ffk {

// Waits until the kernels before this one in the stream have ended and their
// writes are visible (nothing to wait for unless the launch allowed overlap), and
// returns 0.  First in every kernel; the addresses of all reads are formed with
// the result, so that no read of read-only data is moved above the wait.
__device__ __forceinline__ unsigned prior_kernel_done()
{
    unsigned zero;
    asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(zero)::"memory");
    return zero;
}

// Add12 theorem (Knuth): s = a (+) b, r = (a + b) - s exactly; branch free.
__device__ __forceinline__ float2 add12(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    const float r = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
    return make_float2(s, r);
}

// Mul12 theorem: p = a (x) b, e = a*b - p exactly.  The paper derives the
// error with Dekker's Split; one correctly rounded FMA gives the same pair
// (the pair is unique wherever neither part under- or overflows).
__device__ __forceinline__ float2 mul12(float a, float b)
{
    const float p = __fmul_rn(a, b);
    const float e = __fmaf_rn(a, b, -p);
    return make_float2(p, e);
}

// Add22 theorem.  The paper's one test |ah| >= |bh| chooses which high part
// is subtracted from r first; here it selects operands instead of branching
// (the paper prefers extra work to tests on GPUs, Section 4), so that
//   s = (((P (-) r) (+) Q) (+) L1) (+) L2
// is, operation for operation, the paper's line for the taken branch.
__device__ __forceinline__ float2 add22(float2 a, float2 b)
{
    const float r = __fadd_rn(a.x, b.x);
    const bool c = fabsf(a.x) >= fabsf(b.x);
    const float P = c ? a.x : b.x;
    const float Q = c ? b.x : a.x;
    const float L1 = c ? b.y : a.y;
    const float L2 = c ? a.y : b.y;
    const float s = __fadd_rn(__fadd_rn(__fadd_rn(__fsub_rn(P, r), Q), L1), L2);
    return add12(r, s);
}

// Mul22 theorem: (t1, t2) = Mul12(ah, bh); t3 = ((ah bl) + (al bh)) + t2;
// result Add12(t1, t3).  al * bl is dropped, as in the paper.
__device__ __forceinline__ float2 mul22(float2 a, float2 b)
{
    const float2 t = mul12(a.x, b.x);
    const float t3 = __fadd_rn(__fadd_rn(__fmul_rn(a.x, b.y), __fmul_rn(a.y, b.x)), t.y);
    return add12(t.x, t3);
}

// Fast2Sum (Dekker): s = a (+) b, t = (a + b) - s exactly when the exponent
// of a is at least that of b.
__device__ __forceinline__ float2 fast2sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    return make_float2(s, __fsub_rn(b, z));
}

// ---------------------------------------------------------------------------
// Mul22 and Add22 with Fast2Sum in place of their closing Add12: 9 + 13 = 22
// instructions per accumulated term instead of 12 + 16 = 28, for the kernels
// bound by FP32 issue.  Sums of such terms have the bits of sums of mul22 / add22
// under these conditions:
//
// mul22_fast: |t3| <= |t1| (or t1 = t3 = 0).  Both forms then give
//   RN(t1 + t3) and its exact error.  A pair whose sum rounds to its high
//   part (RN(hi + lo) == hi, "normalised") has |lo| <= ulp(hi) / 2, so two
//   normalised operands give |t3| <~ 3 2^-24 |t1|; where a high product
//   underflows the low products are zero too.
// add22_fast: both operands normalised.  With |ah| >= |bh|, ulps ua >= ub:
//   either ah (+) bh is inexact, then |r| >= 2^23 ulp(r) and every part of s
//   is at most ulp(r); or it is exact, r a multiple of ub: |r| >= ua >= |al +
//   bl|, or r = +-ua / 2 (ah a power of two, bh just below it, ub = ua / 2)
//   and |s| <= 3 ua / 4, the same exponent; or r = 0.  The exponent of r is
//   never below that of s, which is Fast2Sum's condition.
// A closing sum that is exact leaves a normalised result, so accumulating
// mul22_fast terms from (0, 0) (or from any Add22 result) stays inside the
// conditions.  Signs of zeros: the closings differ where their second operand is
// -0 (Add12 leaves lo = +0, Fast2Sum -0).  mul22_fast meets that when products
// underflow: (-2^-100, -2^-130) times (2^-100, 2^-130) gives t3 = -0 and (-0, -0) for
// mul22's (-0, +0).  So its result is only ever an addend, not to be stored itself.
// A sum from (+0, +0) never holds -0 and does not see the sign of a zero added to
// it: P, the sum's own high part when both are zero, is not -0, so neither P - r
// nor anything added to that is; s, never -0, closes alike both ways.
// (add22_from_zero_fast adds +0, with the same effect.)
// Infinities and NaN: any step with a non-finite operand gives (NaN, NaN) in
// both forms.  The one difference is a step that overflows to hi = +-inf: lo
// is NaN with Add12 and -+inf with Fast2Sum; a further add22 / add22_fast
// makes both (NaN, NaN), and ff_overflow_lo() restores the NaN of a last one.
// ---------------------------------------------------------------------------

// The pair's sum rounds to its high part (false for a NaN).
__device__ __forceinline__ bool normalised(float2 v) { return __fadd_rn(v.x, v.y) == v.x; }

__device__ __forceinline__ float2 mul22_fast(float2 a, float2 b)
{
    const float2 t = mul12(a.x, b.x);
    const float t3 = __fadd_rn(__fadd_rn(__fmul_rn(a.x, b.y), __fmul_rn(a.y, b.x)), t.y);
    return fast2sum(t.x, t3);
}

// mul22_fast for operands that nothing has checked: `bad` is set when the
// condition fails (one comparison, for kernels that use each operand pair
// once); the caller then repeats the sum with mul22 / add22.
__device__ __forceinline__ float2 mul22_fast_checked(float2 a, float2 b, bool& bad)
{
    const float2 t = mul12(a.x, b.x);
    const float t3 = __fadd_rn(__fadd_rn(__fmul_rn(a.x, b.y), __fmul_rn(a.y, b.x)), t.y);
    bad |= fabsf(t3) > fabsf(t.x);
    return fast2sum(t.x, t3);
}

__device__ __forceinline__ float2 add22_fast(float2 a, float2 b)
{
    const float r = __fadd_rn(a.x, b.x);
    const bool c = fabsf(a.x) >= fabsf(b.x);
    const float P = c ? a.x : b.x;
    const float Q = c ? b.x : a.x;
    const float L1 = c ? b.y : a.y;
    const float L2 = c ? a.y : b.y;
    const float s = __fadd_rn(__fadd_rn(__fadd_rn(__fsub_rn(P, r), Q), L1), L2);
    return fast2sum(r, s);
}

// The low part that Add12 leaves beside an overflowed high part.
__device__ __forceinline__ float2 ff_overflow_lo(float2 v)
{
    return make_float2(v.x, fabsf(v.x) == __int_as_float(0x7f800000) ? __int_as_float(0x7fc00000) : v.y);
}

// Div22: Dekker's div2 with the paper's Add12 as the final renormalisation.
//   ch = ah / bh; (uh, ul) = Mul12(ch, bh);
//   cl = ((((ah - uh) - ul) + al) - ch bl) / bh;  result Add12(ch, cl)
__device__ __forceinline__ float2 div22(float2 a, float2 b)
{
    const float ch = __fdiv_rn(a.x, b.x);
    const float2 u = mul12(ch, b.x);
    const float num = __fsub_rn(__fadd_rn(__fsub_rn(__fsub_rn(a.x, u.x), u.y), a.y),
                                __fmul_rn(ch, b.y));
    const float cl = __fdiv_rn(num, b.x);
    return add12(ch, cl);
}

// Sqrt22: Dekker's sqrt2 with the paper's Add12 as the final step.
//   c = sqrt(ah); (u, uu) = Mul12(c, c);
//   cc = ((((ah - u) - uu) + al) * 0.5) / c;  result Add12(c, cc)
// ah == 0 returns (ah, 0) (keeping the sign of zero).  A negative ah makes
// every step NaN, so the result is (NaN, NaN) without a test.
__device__ __forceinline__ float2 sqrt22(float2 a)
{
    const float c = __fsqrt_rn(a.x);
    const float2 u = mul12(c, c);
    const float rem = __fadd_rn(__fsub_rn(__fsub_rn(a.x, u.x), u.y), a.y);
    const float cc = __fdiv_rn(__fmul_rn(rem, 0.5f), c);
    const float2 r = add12(c, cc);
    const bool z = (a.x == 0.0f);
    return make_float2(z ? a.x : r.x, z ? 0.0f : r.y);
}

// Accurate float-float addition (Joldes, Muller and Popescu 2017,
// Algorithm 6): the two TwoSums of the high and the low parts, then two
// Fast2Sum renormalisations.  Relative error <= 3u^2 / (1 - 4u) (u = 2^-24)
// even under cancellation, where Add22 only bounds the error by 2^-24 |al + bl|.
__device__ __forceinline__ float2 add22_accurate(float2 x, float2 y)
{
    const float2 s = add12(x.x, y.x);
    const float2 t = add12(x.y, y.y);
    const float c = __fadd_rn(s.y, t.x);
    const float2 v = fast2sum(s.x, c);
    const float w = __fadd_rn(t.y, v.y);
    return fast2sum(v.x, w);
}

}  // namespace ffk
