// TF32 rounding for a tensor core that truncates: its operands are FP32 words of
// which it drops the low 13 mantissa bits.
#pragma once

#include <cuda_runtime.h>

namespace mwi {

constexpr unsigned kTf32Half = 0x1000u;  // half a unit in the last place of TF32

// The word whose truncation is v rounded to the nearest TF32 value, ties away
// from zero: half a unit more in magnitude.  All 32 bits are kept, tf32_unbias
// gives v back exactly.  Infinities and NaNs stay as they are, and so does the
// last half unit below FLT_MAX, which would overflow.  One comparison (false for
// a NaN) and one addition.
__device__ __forceinline__ float tf32_bias(float v) {
    const float most = __uint_as_float(0x7f800000u - kTf32Half);
    return fabsf(v) < most ? __uint_as_float(__float_as_uint(v) + kTf32Half) : v;
}
__device__ __forceinline__ float tf32_unbias(float v) {
    const float inf = __uint_as_float(0x7f800000u);
    return fabsf(v) < inf ? __uint_as_float(__float_as_uint(v) - kTf32Half) : v;
}

// v rounded to the nearest TF32 value, ties away from zero
__device__ __forceinline__ float tf32_round(float v) {
    unsigned r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
    return __uint_as_float(r);
}

}  // namespace mwi
