// df64.cuh -- double-float arithmetic on the float32 pipe, for the
// float64-class form of the predictor (WT_FP64_DF).
//
// A value is carried as h + l with |l| <= ulp(h)/2: 48 significant bits,
// float64 accuracy to within a factor of 32, at float32 rates (the GB300's
// float64 pipe runs at a small fraction of its float32 rate). The building
// blocks are the two error-free transforms: Knuth's two-sum (a + b = s + e
// exactly) and the FMA product error (a b = p + e exactly, e = fma(a, b, -p)).
// Sums and products are renormalised with Dekker's fast two-sum; the sum
// drops the rounding error of the low parts' addition (absolute error below
// 2^-47 of the operands), the product drops l_a l_b (below 2^-48 of it).
#pragma once

#include "wt_internal.cuh"

namespace wt {

struct DF {
    float h, l;
};

__device__ __forceinline__ DF df_renorm(float s, float e)
{
    const float h = __fadd_rn(s, e);
    return DF{h, __fsub_rn(e, __fsub_rn(h, s))};
}

__device__ __forceinline__ DF df_add(DF a, DF b)
{
    float s, e;
    two_sum(a.h, b.h, s, e);
    return df_renorm(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}

__device__ __forceinline__ DF df_add_f(DF a, float b)
{
    float s, e;
    two_sum(a.h, b, s, e);
    return df_renorm(s, __fadd_rn(e, a.l));
}

__device__ __forceinline__ DF df_neg(DF a) { return DF{-a.h, -a.l}; }

__device__ __forceinline__ DF df_mul(DF a, DF b)
{
    const float p = __fmul_rn(a.h, b.h);
    const float e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)));
    return df_renorm(p, e);
}

// times a power of two: exact
__device__ __forceinline__ DF df_scale(DF a, float pow2) { return DF{__fmul_rn(a.h, pow2), __fmul_rn(a.l, pow2)}; }

__device__ __forceinline__ double df_to_double(DF a) { return static_cast<double>(a.h) + static_cast<double>(a.l); }

__device__ __forceinline__ DF df_from_double(double x)
{
    const float h = __double2float_rn(x);
    return DF{h, __double2float_rn(x - static_cast<double>(h))};
}

// Sum of many double-floats: sum + x with the head's rounding error and the
// low parts gathered in the low part, not renormalised. The head's sum is
// error-free; the low part holds rounding errors and low parts only, so its
// own rounding stays 2^-24 below theirs. Eight operations against df_add's 11.
__device__ __forceinline__ void df_accumulate(DF& sum, float xh, float xl)
{
    float s, e;
    two_sum(sum.h, xh, s, e);
    sum.h = s;
    sum.l = __fadd_rn(sum.l, __fadd_rn(e, xl));
}

// a b as an unevaluated p + e (df_mul without the renormalisation).
__device__ __forceinline__ void df_product_raw(DF a, DF b, float& p, float& e)
{
    p = __fmul_rn(a.h, b.h);
    e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)));
}

__device__ __forceinline__ void df_accumulate_product(DF& sum, DF a, DF b)
{
    float p, e;
    df_product_raw(a, b, p, e);
    df_accumulate(sum, p, e);
}

// 2 pi as a double-float (the float32 rounding and its remainder)
constexpr float kTwoPiH = 6.2831854820251465f, kTwoPiL = -1.7484555314695172e-07f;

// exp(i 2 pi t) as double-floats (unevaluated sums, the low part within a few
// ulp of the head) for t = th + tl turns, |th| <= 1/2 and tl small (the phase
// of phase_turns_df). The table method of the float64 form (P. T. P. Tang, ACM
// TOMS 15(2), 1989) carried out in double-float: k = rint(1024 t), f = (th -
// k/1024) + tl (the difference exact, the sum error-free), x = 2 pi f, |x| <=
// 0.0031,
//   sin x = x - x^3/6 + x^5/120,  cos x - 1 = -x^2/2 + x^4/24
// (truncated below 6e-22 and 2e-18), x and x^2 in double-float and the rest,
// below 5e-9 and 4e-12, in float32 (rounded below 3e-16); then the rotation of
// the table entry C + i S, tab[k mod 1024] = (C h, C l, S h, S l), by the small
// angle, C + (C (cos x - 1) - S sin x) and S + (S (cos x - 1) + C sin x), whose
// two products are added to the entry's head error-free one after the other.
// 74 operations of the float32 pipe; with 256 entries, where x^3 and the
// cosine itself need double-floats renormalised at every step, 135. With the
// sums left unnormalised (df_accumulate) the medium regrouped sum went from
// 9.4 to 6.7 ms at the same error (2e-12).
__device__ __forceinline__ void sincos_turns_df(float th, float tl, const float4* __restrict__ tab, DF& s, DF& c)
{
    const float k = rintf(__fmul_rn(__fadd_rn(th, tl), 1024.0f));
    float fh, fl;
    two_sum(__fmaf_rn(k, -0.0009765625f, th), tl, fh, fl);
    const float4 e = tab[static_cast<int>(k) & 1023];
    const float xh = __fmul_rn(fh, kTwoPiH);
    const float xe = __fmaf_rn(fh, kTwoPiL, __fmaf_rn(fl, kTwoPiH, __fmaf_rn(fh, kTwoPiH, -xh)));
    const float q = __fmul_rn(xh, xh);
    const float qe = __fmaf_rn(__fadd_rn(xh, xh), xe, __fmaf_rn(xh, xh, -q));
    const DF sx{xh, __fmaf_rn(__fmul_rn(xh, q), __fmaf_rn(q, 8.3333333333333333e-3f, -1.6666666666666667e-1f), xe)};
    const DF cm{__fmul_rn(-0.5f, q), __fmaf_rn(__fmul_rn(q, q), 4.1666666666666667e-2f, __fmul_rn(-0.5f, qe))};
    const DF C{e.x, e.y}, S{e.z, e.w};
    float p, pe;
    c = C;
    df_product_raw(S, sx, p, pe);
    df_accumulate(c, -p, -pe);
    df_product_raw(C, cm, p, pe);
    df_accumulate(c, p, pe);
    s = S;
    df_product_raw(C, sx, p, pe);
    df_accumulate(s, p, pe);
    df_product_raw(S, cm, p, pe);
    df_accumulate(s, p, pe);
}

constexpr int kDfTableEntries = 1024;

static __device__ const float4 kSinCosDF[kDfTableEntries] =
#include "sincos_table_df.inc"
    ;

// The table of exp(i 2 pi k/1024), k = 0 .. 1023, as double-floats, copied by
// the CTA's threads into shared memory.
__device__ __forceinline__ void load_sincos_table_df(float4* tab)
{
#pragma unroll 4
    for (int i = threadIdx.x; i < kDfTableEntries; i += blockDim.x) tab[i] = __ldg(&kSinCosDF[i]);
}

}  // namespace wt
