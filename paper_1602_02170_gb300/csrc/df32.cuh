// Double-float arithmetic: a value is the unevaluated sum hi + lo of two
// FP32 numbers with |lo| <= ulp(hi)/2, giving about 46 significant bits on
// the FP32 pipes.  Built from the classic error-free transformations:
// Knuth's two-sum (the exact rounding error of a + b), the fast two-sum of
// Dekker for |a| >= |b|, and the exact product error of a * b obtained with a
// fused multiply-add.
//
// GB300 runs FP64 at a small fraction of its FP32 rate; the pair kernel in
// double-float reaches FP64-class accuracy for the refinement residuals of
// the mixed-precision solver at a fraction of the FP64 kernel's time.
#pragma once

#include <cuda_runtime.h>

namespace mb {

// 1/sqrt(x) in FP32 for normal x: the hardware estimate without the scaling
// of denormal arguments that rsqrtf() adds.
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct dfl {
    float hi, lo;

    __host__ __device__ constexpr dfl() : hi(0.f), lo(0.f) {}
    __host__ __device__ constexpr dfl(float h, float l) : hi(h), lo(l) {}
    // exact split of a double into hi + lo (constant-folded for literals)
    __host__ __device__ constexpr dfl(double d)
        : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ constexpr dfl(int i) : dfl((double)i) {}
};

__device__ __forceinline__ dfl two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return dfl(s, e);
}

__device__ __forceinline__ dfl fast_two_sum(float a, float b)
{
    const float s = a + b;
    return dfl(s, b - (s - a));
}

// Addition in the "sloppy" form of Bailey's QD library (an exact two-sum of
// the high parts, the low parts added in FP32), here without the closing
// renormalisation: 8 FP32 operations instead of 20 for the form that also
// two-sums the low parts and renormalises twice.  The result hi + lo is not
// normalised (lo may exceed half an ulp of hi); every operation here accepts
// such operands, and subtraction, accumulation (+=) and the reciprocal square
// root renormalise.  The absolute error is within a few 2^-48 (|a| + |b|), so
// relative accuracy is lost only where a and b nearly cancel, and then only
// relative to the operands, which is what the pair sums need (about 1e-13 of
// each term).
__device__ __forceinline__ dfl operator+(dfl a, dfl b)
{
    const dfl s = two_sum(a.hi, b.hi);
    return dfl(s.hi, s.lo + (a.lo + b.lo));
}

__device__ __forceinline__ dfl operator-(dfl a) { return dfl(-a.hi, -a.lo); }
// Subtraction renormalises: it forms the separations of nearby positions,
// where hi nearly cancels and the unnormalised lo would be large relative to
// the difference.
__device__ __forceinline__ dfl operator-(dfl a, dfl b)
{
    const dfl s = two_sum(a.hi, -b.hi);
    return fast_two_sum(s.hi, s.lo + (a.lo - b.lo));
}

// Product without the final renormalisation: lo may reach a few ulp of hi
// instead of half an ulp.  Every consumer (addition, product, conversion to
// double) takes such operands without loss beyond ~2^-46 relative.
__device__ __forceinline__ dfl operator*(dfl a, dfl b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return dfl(p, e);
}

// Accumulation renormalises (fast two-sum after the sloppy addition): a
// running sum over thousands of terms would otherwise let lo grow and lose
// bits in its FP32 additions.
__device__ __forceinline__ dfl &operator+=(dfl &a, dfl b)
{
    const dfl s = two_sum(a.hi, b.hi);
    a = fast_two_sum(s.hi, s.lo + (a.lo + b.lo));
    return a;
}

__device__ __forceinline__ double to_double(dfl a) { return (double)a.hi + (double)a.lo; }

// ---------------------------------------------------------------------------
// Two double-float values in the halves of float2s.  One paired instruction
// does the work of two, so the FMA pipe and not the issue of instructions
// bounds code written with these (negated operands cost nothing).
__device__ __forceinline__ float2 splat2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

struct dfl2 {
    float2 hi, lo;

    __host__ __device__ dfl2() : hi{0.f, 0.f}, lo{0.f, 0.f} {}
    __host__ __device__ dfl2(float2 h, float2 l) : hi(h), lo(l) {}
    // the same value in both halves
    __host__ __device__ dfl2(dfl a) : hi{a.hi, a.hi}, lo{a.lo, a.lo} {}
};

__device__ __forceinline__ dfl2 two_sum(float2 a, float2 b)
{
    const float2 s = add2(a, b), bb = sub2(s, a);
    return dfl2(s, add2(sub2(a, sub2(s, bb)), sub2(b, bb)));
}

__device__ __forceinline__ dfl2 fast_two_sum(float2 a, float2 b)
{
    const float2 s = add2(a, b);
    return dfl2(s, sub2(b, sub2(s, a)));
}

// Sums and products as for dfl: unnormalised (8 and 4 instructions);
// subtraction renormalises (11).
__device__ __forceinline__ dfl2 operator+(dfl2 a, dfl2 b)
{
    const dfl2 s = two_sum(a.hi, b.hi);
    return dfl2(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ dfl2 operator-(dfl2 a) { return dfl2(neg2(a.hi), neg2(a.lo)); }
__device__ __forceinline__ dfl2 operator-(dfl2 a, dfl2 b)
{
    const dfl2 s = two_sum(a.hi, neg2(b.hi));
    return fast_two_sum(s.hi, add2(s.lo, sub2(a.lo, b.lo)));
}
__device__ __forceinline__ dfl2 operator*(dfl2 a, dfl2 b)
{
    const float2 p = mul2(a.hi, b.hi);
    return dfl2(p, fma2(a.lo, b.hi, fma2(a.hi, b.lo, fma2(a.hi, b.hi, neg2(p)))));
}
// accumulation renormalises, as for dfl (11)
__device__ __forceinline__ dfl2 &operator+=(dfl2 &a, dfl2 b)
{
    const dfl2 s = two_sum(a.hi, b.hi);
    a = fast_two_sum(s.hi, add2(s.lo, add2(a.lo, b.lo)));
    return a;
}
// a + b for |a| >= |b| (5), a c for c exact in FP32 (3), a c for c a power of
// two (2), a + c (7)
__device__ __forceinline__ dfl2 add_ordered(dfl2 a, dfl2 b)
{
    const dfl2 s = fast_two_sum(a.hi, b.hi);
    return dfl2(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ dfl2 mulf(dfl2 a, float c)
{
    const float2 c2 = splat2(c), p = mul2(a.hi, c2);
    return dfl2(p, fma2(a.lo, c2, fma2(a.hi, c2, neg2(p))));
}
__device__ __forceinline__ dfl2 mul_pow2(dfl2 a, float c)
{
    return dfl2(mul2(a.hi, splat2(c)), mul2(a.lo, splat2(c)));
}
__device__ __forceinline__ dfl2 addf(dfl2 a, float c)
{
    const dfl2 s = two_sum(a.hi, splat2(c));
    return dfl2(s.hi, add2(s.lo, a.lo));
}
// a + c for c below an ulp or so of what a is added to next: into lo (1)
__device__ __forceinline__ dfl2 add_lo(dfl2 a, float2 c) { return dfl2(a.hi, add2(a.lo, c)); }
__device__ __forceinline__ void renorm(dfl2 &a) { a = fast_two_sum(a.hi, a.lo); }

// x^-1/2: the FP32 estimate y0 of x.hi and one step of Householder's cubic
// iteration y0 + y0 r (1/2 + 3/8 r), r = 1 - x y0^2 formed as an FP32 number
// from exact products (y0^2 = s + t, x_hi s = p + e; 1 - p is exact, p being
// within 2^-20 of 1).  x may be unnormalised: its lo part enters r, and what
// it adds to r (a few 2^-24) leaves a truncation error far below 2^-48.
__device__ __forceinline__ dfl2 rsqrt_df(dfl2 x)
{
    const float2 y0 = make_float2(rsqrt_ftz(x.hi.x), rsqrt_ftz(x.hi.y));
    const float2 s = mul2(y0, y0), t = fma2(y0, y0, neg2(s));
    const float2 p = mul2(x.hi, s), e = fma2(x.hi, s, neg2(p));
    const float2 q = fma2(x.hi, t, mul2(x.lo, s));
    const float2 r = sub2(sub2(sub2(splat2(1.f), p), e), q);
    return fast_two_sum(y0, mul2(y0, mul2(r, fma2(r, splat2(0.375f), splat2(0.5f)))));
}

// Sum of both halves in FP64.
__device__ __forceinline__ double sum_halves(dfl2 a)
{
    return ((double)a.hi.x + (double)a.hi.y) + ((double)a.lo.x + (double)a.lo.y);
}

}  // namespace mb
