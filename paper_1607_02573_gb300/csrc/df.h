// Double-float arithmetic: a real number carried as an unevaluated sum hi + lo
// of two FP32 values (about 48 significant bits), built from the error-free
// transformations TwoSum (Knuth, TAOCP vol. 2, 4.2.2) and TwoProduct via a
// fused multiply-add (Dekker 1971; Ogita, Rump and Oishi 2005).  On GB300 the
// FP64 units run at 1/64 of the FP32 rate, so FP64-accurate vector work of
// the outer Krylov solver is done in this form on the FP32 pipes.
//
// The expressions rely on IEEE FP32 semantics without reassociation (no fast
// math); contraction into FMA is harmless where it occurs.
#pragma once

#include <cuda_runtime.h>

namespace mwi {

struct dfl {
    float h, l;
};

// s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// s + e = a + b exactly, given |a| >= |b| (or a = 0)
__device__ __forceinline__ void quick_two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    e = b - (s - a);
}

__device__ __forceinline__ dfl df_norm(dfl a) {
    dfl r;
    quick_two_sum(a.h, a.l, r.h, r.l);
    return r;
}

// acc += (ah + al) * (bh + bl), the product to about 2^-46 relative; acc is
// left unnormalised (lo accumulates), df_norm it before storing
__device__ __forceinline__ void df_mac(dfl& acc, float ah, float al, float bh, float bl) {
    const float p = ah * bh;
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    e = fmaf(al, bh, e);
    float s, t;
    two_sum(acc.h, p, s, t);
    acc.h = s;
    acc.l += t + e;
}

// acc += a * (bh + bl) with a exact in FP32
__device__ __forceinline__ void df_mac1(dfl& acc, float a, float bh, float bl) {
    const float p = a * bh;
    float e = fmaf(a, bh, -p);
    e = fmaf(a, bl, e);
    float s, t;
    two_sum(acc.h, p, s, t);
    acc.h = s;
    acc.l += t + e;
}

// (ah + al) * (bh + bl), normalised
__device__ __forceinline__ dfl df_mul(float ah, float al, float bh, float bl) {
    const float p = ah * bh;
    float e = fmaf(ah, bh, -p);
    e = fmaf(ah, bl, e);
    e = fmaf(al, bh, e);
    dfl r;
    quick_two_sum(p, e, r.h, r.l);
    return r;
}

// Two FP32 operations per instruction (packed pairs, sm_100 and later), each
// rounded as the single one is.  They run at the same rate per lane, so they
// save issue slots, not pipe cycles.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(reinterpret_cast<unsigned long long&>(d))
        : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)),
          "l"(reinterpret_cast<const unsigned long long&>(c)));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long&>(d))
        : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long&>(d))
        : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
    return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

// two double-floats
struct dfl2 {
    float2 h, l;
};

// df_mac1 on both halves, the same operations in the same order: acc += a (bh +
// bl), nbh = -bh (the product enters as its negative, which the sums subtract)
__device__ __forceinline__ void df_mac1_2(dfl2& acc, float2 a, float2 bh, float2 nbh, float2 bl) {
    const float2 np = mul2(a, nbh);
    float2 e = fma2(a, bh, np);
    e = fma2(a, bl, e);
    const float2 s = sub2(acc.h, np);
    const float2 bb = sub2(s, acc.h);
    const float2 t = sub2(sub2(acc.h, sub2(s, bb)), add2(np, bb));
    acc.h = s;
    acc.l = add2(acc.l, add2(t, e));
}

// df_mac on both halves: acc += (ah + al) (bh + bl)
__device__ __forceinline__ void df_mac_2(dfl2& acc, float2 ah, float2 al, float2 bh, float2 nbh, float2 bl) {
    const float2 np = mul2(ah, nbh);
    float2 e = fma2(ah, bh, np);
    e = fma2(ah, bl, e);
    e = fma2(al, bh, e);
    const float2 s = sub2(acc.h, np);
    const float2 bb = sub2(s, acc.h);
    const float2 t = sub2(sub2(acc.h, sub2(s, bb)), add2(np, bb));
    acc.h = s;
    acc.l = add2(acc.l, add2(t, e));
}

// df_mul on both halves
__device__ __forceinline__ dfl2 df_mul_2(float2 ah, float2 al, float2 bh, float2 bl) {
    const float2 p = mul2(ah, bh);
    float2 e = fma2(ah, bh, make_float2(-p.x, -p.y));
    e = fma2(ah, bl, e);
    e = fma2(al, bh, e);
    dfl2 r;
    r.h = add2(p, e);
    r.l = sub2(e, sub2(r.h, p));
    return r;
}

__device__ __forceinline__ dfl2 df_norm_2(dfl2 a) {
    dfl2 r;
    r.h = add2(a.h, a.l);
    r.l = sub2(a.l, sub2(r.h, a.h));
    return r;
}

// nearest double-float of an FP64 value (FP64 units: use outside hot loops)
__device__ __forceinline__ float2 df_split(double x) {
    const float h = __double2float_rn(x);
    const float l = __double2float_rn(x - (double)h);
    return make_float2(h, l);
}

__device__ __forceinline__ double df_join(float h, float l) { return (double)h + (double)l; }

}  // namespace mwi
