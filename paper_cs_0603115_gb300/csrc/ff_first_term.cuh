// ff_first_term.cuh -- the first accumulation step of a float-float sum that
// starts from (0, 0), as the weight gradient forms it: every output element
// is Add22((0, 0), term_0), then Add22 of the later terms.  (The GEMM kernel
// keeps the plain first step: peeling it off the slice loop measured 0.3-1%
// slower, its loop being tuned for instruction fetch.)
#pragma once
#include <cuda_runtime.h>

#include "ff_core.cuh"

namespace ffk {

// Add22((+0, +0), t) bit for bit for a finite normalised t (every mul22 result is
// one, or not finite, and so is every mul22_fast result of normalised operands): the Add22 theorem's
// steps reduce to r = th (+) 0, s = tl (+) 0 and a closing sum that returns (r,
// s): th - r = +0 (the tie branch when th = +-0, which forces tl = +-0), the
// zero operand's low part adds nothing.  "(+) 0" does what the full sequence
// does to a negative zero (it becomes +0).  For an infinite th the full step
// gives (NaN, NaN): any later Add22 does the same to what this one leaves, and
// a single-term sum ends with from_zero_infinite().
__device__ __forceinline__ float2 add22_from_zero_fast(float2 t)
{
    return make_float2(__fadd_rn(t.x, 0.0f), __fadd_rn(t.y, 0.0f));
}

__device__ __forceinline__ float2 from_zero_infinite(float2 v)
{
    const float nan = __int_as_float(0x7fc00000);
    return fabsf(v.x) == __int_as_float(0x7f800000) ? make_float2(nan, nan) : v;
}

}  // namespace ffk
