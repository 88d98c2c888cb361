// Double-float arithmetic: a value is the unevaluated sum hi + lo of two FP32 numbers (|lo| <= ulp(hi)/2),
// about 48 significant bits.  Sums use the error-free two-sum transformation (Knuth), products the
// FMA-based two-product (p = a*b, e = fma(a, b, -p) exactly), followed by renormalisation
// (Dekker's fast two-sum).  Everything runs on the FP32 units, which on this GPU have 64 times the
// FP64 throughput; the J/K kernels use it for the quartets that need FP64-class accuracy.
//
// Within an expression sums and products stay unnormalised (df32u): the low part may exceed half an ulp of
// the high one, which costs the next sum nothing, and the three instructions of Dekker's sum are spent once,
// when the value is stored or multiplied.  a b + c d takes 19 instructions instead of 25, a Boys term 12
// instead of 15, a b + c d + e (f - g h) 46 instead of 61.  (H2O)_32 / 6-31G*, launches one at a time: (pp|pp)
// 382 -> 295 us, (pp|ps) 480 -> 376, (dp|ds) 564 -> 457, (ps|ss) 714 -> 661.
#pragma once
#include <cuda_runtime.h>

struct df32u;
struct df32 {
    float hi, lo;
    __device__ __forceinline__ df32() {}
    __device__ __forceinline__ constexpr df32(float h, float l) : hi(h), lo(l) {}
    __device__ __forceinline__ explicit df32(int v) : hi((float)v), lo(0.f) {}
    __device__ __forceinline__ explicit df32(float v) : hi(v), lo(0.f) {}
    __device__ __forceinline__ explicit df32(double v);   // after d2f_alu / f2d_alu
};

__device__ __forceinline__ df32 df_fast_two_sum(float a, float b)
{
    const float s = a + b;
    return df32(s, b - (s - a));
}

__device__ __forceinline__ df32 df_two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    return df32(s, (a - (s - bb)) + (b - bb));
}

// hi + lo before normalisation
struct df32u {
    float hi, lo;
    __device__ __forceinline__ constexpr df32u(float h, float l) : hi(h), lo(l) {}
    __device__ __forceinline__ constexpr df32u(df32 v) : hi(v.hi), lo(v.lo) {}
    __device__ __forceinline__ operator df32() const { return df_fast_two_sum(hi, lo); }
};

__device__ __forceinline__ df32u operator+(df32u a, df32u b)
{
    const df32 s = df_two_sum(a.hi, b.hi);
    return df32u(s.hi, s.lo + (a.lo + b.lo));
}

__device__ __forceinline__ df32 operator-(df32 a) { return df32(-a.hi, -a.lo); }
__device__ __forceinline__ df32u operator-(df32u a) { return df32u(-a.hi, -a.lo); }
__device__ __forceinline__ df32u operator-(df32u a, df32u b) { return a + (-b); }

__device__ __forceinline__ df32u operator*(df32 a, df32 b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df32u(p, e);
}

__device__ __forceinline__ df32& operator+=(df32& a, df32u b) { a = a + b; return a; }
__device__ __forceinline__ df32& operator-=(df32& a, df32u b) { a = a - b; return a; }
__device__ __forceinline__ df32& operator*=(df32& a, df32 b) { a = a * b; return a; }
__device__ __forceinline__ bool operator!=(df32 a, df32 b) { return a.hi != b.hi || a.lo != b.lo; }
__device__ __forceinline__ bool operator<(df32 a, double b) { return a.hi < (float)b; }

// a + b for |a| >= |b| (8 instructions instead of 11)
__device__ __forceinline__ df32 df_add_smaller(df32 a, df32u b)
{
    const float s = a.hi + b.hi;
    const float e = b.hi - (s - a.hi);
    return df_fast_two_sum(s, e + (a.lo + b.lo));
}

// reciprocal root without the scaling of subnormal arguments (three instructions less; a subnormal gives infinity)
__device__ __forceinline__ float rsqrt_ftz(float a)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return y;
}

// a^(-1/2): FP32 reciprocal root, one FP32 Newton step, then y (1 + r/2 + 3/8 r^2) with r = 1 - a y^2
// (|r| < 2e-7) formed to double-float accuracy.  a > 0 (and no subnormal).
__device__ __forceinline__ df32 df_rsqrt(df32 a)
{
    float y = rsqrt_ftz(a.hi);
    y = fmaf(0.5f * y, fmaf(-a.hi * y, y, 1.0f), y);
    const float ph = y * y, pl = fmaf(y, y, -ph);
    const float mh = a.hi * ph;
    float ml = fmaf(a.hi, ph, -mh);
    ml = fmaf(a.hi, pl, ml);
    ml = fmaf(a.lo, ph, ml);
    const float r = (1.0f - mh) - ml;
    return df_fast_two_sum(y, y * (r * fmaf(0.375f, r, 0.5f)));
}

__device__ __forceinline__ df32 df_shfl_xor(df32 v, int o)
{
    return df32(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}

// element type of the density copy a J/K kernel of arithmetic type R reads (D itself for FP64,
// FP32-rounded for FP32, hi / lo pairs for double-float)
template <typename R> struct DElem { typedef double T; };
template <> struct DElem<float> { typedef float T; };
template <> struct DElem<df32> { typedef float2 T; };
