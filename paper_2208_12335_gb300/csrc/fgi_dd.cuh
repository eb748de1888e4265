// Double-float arithmetic: a value is the unevaluated sum hi + lo of two
// FP32 numbers (about 48 significant bits).  Built from the error-free
// transformations of Dekker (1971) and Knuth (TAOCP vol. 2): the exact
// rounding error of a sum from six additions, of a product from one FMA.
// Used where FP32 rounding would be systematic across many grid points
// (the radial spline and its normalisation), at a fraction of the cost of
// GB300's FP64 pipe.  Relies on IEEE FP32 without reassociation (nvcc's
// default; explicit fmaf where an FMA is meant).
#pragma once
#include <cuda_runtime.h>

namespace fgi {

struct df {
    float hi, lo;
};

__device__ __forceinline__ df df_two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}

__device__ __forceinline__ df df_fast_two_sum(float a, float b)   // |a| >= |b|
{
    const float s = a + b;
    return {s, b - (s - a)};
}

__device__ __forceinline__ df df_two_prod(float a, float b)
{
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}

// Sum with one error-free transformation (the high parts) and a rounded sum
// of the low parts: error within about 2^-48 (|a| + |b|) instead of
// 2^-48 |a + b|.  Exact enough for sums of one sign, and for differences of
// grid coordinates, whose rounding differs from point to point.
__device__ __forceinline__ df df_add_sloppy(df a, df b)
{
    const df s = df_two_sum(a.hi, b.hi);
    return df_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}

__device__ __forceinline__ df df_sub_sloppy(df a, df b) { return df_add_sloppy(a, df{-b.hi, -b.lo}); }

__device__ __forceinline__ df df_mul(df a, df b)
{
    df p = df_two_prod(a.hi, b.hi);
    p.lo = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, p.lo));
    return df_fast_two_sum(p.hi, p.lo);
}

__device__ __forceinline__ df df_mul_f(df a, float b)
{
    df p = df_two_prod(a.hi, b);
    p.lo = fmaf(a.lo, b, p.lo);
    return df_fast_two_sum(p.hi, p.lo);
}

// The same product without the final renormalisation: hi = fl(a.hi b) and
// lo the rest, |lo| up to about two ulps of hi.  For consumers that use the
// pair only as the sum hi + lo (the split into BF16 terms).
__device__ __forceinline__ df df_mul_f_raw(df a, float b)
{
    const float p = a.hi * b;
    return {p, fmaf(a.lo, b, fmaf(a.hi, b, -p))};
}

// sqrt by one Newton correction of the FP32 root (IEEE sqrtf)
__device__ __forceinline__ df df_sqrt(df a)
{
    if (a.hi <= 0.f) return {0.f, 0.f};
    const float r = sqrtf(a.hi);
    const float e = fmaf(-r, r, a.hi) + a.lo;
    return df_fast_two_sum(r, e * (0.5f / r));
}

// 1/a by one Newton correction of the FP32 reciprocal
__device__ __forceinline__ df df_rcp(df a)
{
    const float r = 1.0f / a.hi;
    float e = fmaf(-a.hi, r, 1.0f);
    e = fmaf(-a.lo, r, e);
    return df_fast_two_sum(r, e * r);
}

// 1/sqrt(a) from an approximation y (relative error up to ~2^-20): with
// rho = 1 - a y^2 (from exact products, to about 2^-46 absolute),
// 1/sqrt(a) = y (1 - rho)^(-1/2) = y (1 + rho/2 + 3 rho^2/8 + O(rho^3)).
// Host-callable so that tests can check it against FP64 with a perturbed y.
__host__ __device__ __forceinline__ df df_rsqrt_refine(df a, float y)
{
    const float y2h = y * y;
    const float y2l = fmaf(y, y, -y2h);
    const float ph = a.hi * y2h;
    const float pl = fmaf(a.hi, y2h, -ph);
    // 1 - ph is exact (ph is within a factor two of 1)
    const float rho = ((1.f - ph) - pl) - fmaf(a.hi, y2l, a.lo * y2h);
    const float c = y * (rho * fmaf(0.375f, rho, 0.5f));
    const float s = y + c;
    return {s, c - (s - y)};
}

#if defined(__CUDACC__)
// 1/sqrt(a) for a > 0 (a.hi a normal FP32 number): the FP32 approximation
// rsqrtf refined once
__device__ __forceinline__ df df_rsqrt(df a) { return df_rsqrt_refine(a, rsqrtf(a.hi)); }
#endif

__host__ __device__ __forceinline__ df df_from_double(double x)
{
    const float hi = (float)x;
    return {hi, (float)(x - (double)hi)};
}

#if defined(__CUDACC__)
// ---- pairs of FP32 numbers, one instruction for both: the FMA pipe takes two
// cycles for it, the issue slots are halved.  Each half is rounded as the
// scalar operation would be.
struct pk {
    unsigned long long v;
};
__device__ __forceinline__ pk pk_make(float a, float b)
{
    pk r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ pk pk_dup(float a) { return pk_make(a, a); }
__device__ __forceinline__ float2 pk_get(pk a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ pk operator+(pk a, pk b)
{
    pk r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ pk operator*(pk a, pk b)
{
    pk r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ pk fma2(pk a, pk b, pk c)
{
    pk r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ pk operator-(pk a) { return pk{a.v ^ 0x8000000080000000ull}; }
__device__ __forceinline__ pk operator-(pk a, pk b) { return fma2(b, pk_dup(-1.f), a); }   // one rounding, as a - b

// two double-floats, and the operations above on them, step by step
struct df2 {
    pk hi, lo;
};
__device__ __forceinline__ df2 df2_two_sum(pk a, pk b)
{
    const pk s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ df2 df2_fast_two_sum(pk a, pk b)
{
    const pk s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ df2 df2_add_sloppy(df2 a, df2 b)
{
    const df2 s = df2_two_sum(a.hi, b.hi);
    return df2_fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__device__ __forceinline__ df2 df2_mul(df2 a, df2 b)
{
    const pk p = a.hi * b.hi;
    return df2_fast_two_sum(p, fma2(a.hi, b.lo, fma2(a.lo, b.hi, fma2(a.hi, b.hi, -p))));
}
__device__ __forceinline__ df2 df2_rsqrt(df2 a)                   // df_rsqrt_refine
{
    const float2 ah = pk_get(a.hi);
    const pk y = pk_make(rsqrtf(ah.x), rsqrtf(ah.y)), y2h = y * y, y2l = fma2(y, y, -y2h);
    const pk ph = a.hi * y2h, pl = fma2(a.hi, y2h, -ph);
    const pk rho = ((pk_dup(1.f) - ph) - pl) - fma2(a.hi, y2l, a.lo * y2h);
    const pk c = y * (rho * fma2(pk_dup(0.375f), rho, pk_dup(0.5f)));
    const pk s = y + c;
    return {s, c - (s - y)};
}
#endif

}  // namespace fgi
