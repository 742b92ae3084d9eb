// df64.cuh -- double-float arithmetic on the float32 pipe, for the
// float64-class form of the predictor (WT_FP64_DF).
//
// A value is carried as h + l with |l| <= ulp(h)/2: 48 significant bits,
// float64 accuracy to within a factor of 32, at float32 rates (the GB300's
// float64 pipe runs at a small fraction of its float32 rate). The building
// blocks are the two error-free transforms: Knuth's two-sum (a + b = s + e
// exactly) and the FMA product error (a b = p + e exactly, e = fma(a, b, -p)).
// Sums gather the heads' rounding errors and the low parts in the low part and
// are renormalised (Dekker's fast two-sum) after a few terms; a product drops
// l_a l_b (below 2^-48 of it).
#pragma once

#include "wt_internal.cuh"

namespace wt {

struct DF {
    float h, l;
};

// times a power of two: exact
__device__ __forceinline__ DF df_scale(DF a, float pow2) { return DF{__fmul_rn(a.h, pow2), __fmul_rn(a.l, pow2)}; }

__device__ __forceinline__ double df_to_double(DF a) { return static_cast<double>(a.h) + static_cast<double>(a.l); }

// Sum of many double-floats: sum + x with the head's rounding error and the
// low parts gathered in the low part, not renormalised. The head's sum is
// error-free; the low part holds rounding errors and low parts only, so its
// own rounding stays 2^-24 below theirs as long as few terms gather there. A
// long sum is taken in blocks of a few terms (df_product of the first,
// df_accumulate_product of the others), each then added to the whole, which is
// renormalised: a block's head is small, and so are its roundings. The error of
// sums of 20, 200, 2 000 terms of random flux, RMS, in 1e-15 of the fluxes' sum:
// renormalised at every term (11 operations, not eight) 1.22, 1.07, 0.97;
// one sum renormalised every eight terms 1.77, 1.57, 1.55; blocks of four,
// renormalised too, 1.20, 0.64, 0.52; two such side by side, added to each other
// and then to the whole, 1.21, 0.54, 0.41.
__device__ __forceinline__ void df_accumulate(DF& sum, float xh, float xl)
{
    float s, e;
    two_sum(sum.h, xh, s, e);
    sum.h = s;
    sum.l = __fadd_rn(sum.l, __fadd_rn(e, xl));
}

__device__ __forceinline__ void df_renorm(DF& x)
{
    const float h = __fadd_rn(x.h, x.l);
    x.l = __fsub_rn(x.l, __fsub_rn(h, x.h));
    x.h = h;
}

// a b as an unevaluated p + e.
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

__device__ __forceinline__ DF df_product(DF a, DF b)
{
    DF r;
    df_product_raw(a, b, r.h, r.l);
    return r;
}

// sum + a block's sum, renormalised.
__device__ __forceinline__ void df_add_block(DF& sum, DF block)
{
    df_accumulate(sum, block.h, block.l);
    df_renorm(sum);
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
// cosine itself need double-floats renormalised at every step, 135. Emulated over
// 4e6 phases the error is 1.08e-15 RMS, 9.3e-15 at most (256 entries: 1.16e-15,
// 9.1e-15).
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

// ---- two visibilities at once -------------------------------------------------
// The same operations on packed pairs, element 0 one visibility and element 1
// another: the float32 pipe takes a pair every two cycles in one issue slot, so
// half of them are left for the records, the table and the sweep. A pair cannot be negated for free, so products are formed with their
// heads negated (from a factor that is kept negated) and subtracted.
struct DFP {
    float2 h, l;
};

__device__ __forceinline__ DFP dfp_zero() { return DFP{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

// sum + (-nh + l), as df_accumulate.
__device__ __forceinline__ void dfp_accumulate_neg(DFP& sum, float2 nh, float2 l)
{
    const float2 s = sub2(sum.h, nh);
    const float2 bp = sub2(s, sum.h);                         // what of -nh arrived
    const float2 e = sub2(sub2(sum.h, sub2(s, bp)), add2(nh, bp));
    sum.h = s;
    sum.l = add2(sum.l, add2(e, l));
}

// sum + x.
__device__ __forceinline__ void dfp_accumulate(DFP& sum, const DFP& x)
{
    float2 s, e;
    two_sum2(sum.h, x.h, s, e);
    sum.h = s;
    sum.l = add2(sum.l, add2(e, x.l));
}

// a b = -np + e, na = -a.h.
__device__ __forceinline__ void dfp_product(const DFP& a, float2 na, const DFP& b, float2& np, float2& e)
{
    np = mul2(na, b.h);
    e = fma2(a.h, b.l, fma2(a.l, b.h, fma2(a.h, b.h, np)));
}

__device__ __forceinline__ void dfp_renorm(DFP& x)
{
    const float2 h = add2(x.h, x.l);
    x.l = sub2(x.l, sub2(h, x.h));
    x.h = h;
}

// A factor common to both elements, with its negated head.
struct DFS {
    DFP v;
    float2 nh;
};
__device__ __forceinline__ DFS dfs(float h, float l) { return DFS{DFP{bcast2(h), bcast2(l)}, bcast2(-h)}; }

__device__ __forceinline__ void dfp_accumulate_product(DFP& sum, const DFS& a, const DFP& b)
{
    float2 np, e;
    dfp_product(a.v, a.nh, b, np, e);
    dfp_accumulate_neg(sum, np, e);
}

// a b, to be the first of a block.
__device__ __forceinline__ DFP dfp_product(const DFS& a, const DFP& b)
{
    float2 np, e;
    dfp_product(a.v, a.nh, b, np, e);
    return DFP{sub2(make_float2(0.f, 0.f), np), e};
}

__device__ __forceinline__ void dfp_add_block(DFP& sum, const DFP& block)
{
    dfp_accumulate(sum, block);
    dfp_renorm(sum);
}

// phase_turns_df2 with the phase as th + tl.
__device__ __forceinline__ void phase_turns_dfp(const DF2& u, const DF2& v, const DF2& w, F2 su, F2 sv, F2 sw1,
                                                float2& th, float2& tl)
{
    float2 q1, t1, q2, t2, q3, t3, a, ea, b, eb;
    df_product2n(u, su, q1, t1);
    df_product2n(v, sv, q2, t2);
    df_product2n(w, sw1, q3, t3);
    two_sum2(q1, q2, a, ea);
    two_sum2(a, q3, b, eb);
    th = sub2(make_float2(rintf(b.x), rintf(b.y)), b);
    tl = sub2(add2(add2(t1, t2), sub2(t3, ea)), eb);
}

// sincos_turns_df of two phases.
__device__ __forceinline__ void sincos_turns_dfp(float2 th, float2 tl, const float4* __restrict__ tab, DFP& s, DFP& c)
{
    const float2 t = mul2(add2(th, tl), bcast2(1024.0f));
    const float2 k = make_float2(rintf(t.x), rintf(t.y));
    float2 fh, fl;
    two_sum2(fma2(k, bcast2(-0.0009765625f), th), tl, fh, fl);
    const float4 e0 = tab[static_cast<int>(k.x) & 1023], e1 = tab[static_cast<int>(k.y) & 1023];
    const float2 xh = mul2(fh, bcast2(kTwoPiH)), nx = mul2(fh, bcast2(-kTwoPiH));
    const float2 xe = fma2(fh, bcast2(kTwoPiL), fma2(fl, bcast2(kTwoPiH), fma2(fh, bcast2(kTwoPiH), nx)));
    const float2 nq = mul2(nx, xh);                            // -x^2
    const float2 qe = fma2(add2(xh, xh), xe, fma2(xh, xh, nq));
    // sin x = x - x^3/6 + x^5/120, cos x - 1 = -x^2/2 + x^4/24
    const DFP sx{xh, fma2(mul2(xh, nq), fma2(nq, bcast2(8.3333333333333333e-3f), bcast2(1.6666666666666667e-1f)), xe)};
    const DFP cm{mul2(nq, bcast2(0.5f)),
                 fma2(mul2(nq, nq), bcast2(4.1666666666666667e-2f), mul2(qe, bcast2(-0.5f)))};
    const float2 ncm = mul2(nq, bcast2(-0.5f));
    const DFP C{make_float2(e0.x, e1.x), make_float2(e0.y, e1.y)}, S{make_float2(e0.z, e1.z), make_float2(e0.w, e1.w)};
    float2 np, e;
    c = C;
    dfp_product(sx, nx, S, np, e);                             // -S sin x: head np, low -e
    {
        float2 sum, err;
        two_sum2(c.h, np, sum, err);
        c.h = sum;
        c.l = add2(c.l, sub2(err, e));
    }
    dfp_product(cm, ncm, C, np, e);
    dfp_accumulate_neg(c, np, e);
    s = S;
    dfp_product(sx, nx, C, np, e);
    dfp_accumulate_neg(s, np, e);
    dfp_product(cm, ncm, S, np, e);
    dfp_accumulate_neg(s, np, e);
}

__device__ __forceinline__ double2 dfp_vis(const DFP& re, const DFP& im, int k)
{
    return k == 0 ? make_double2(static_cast<double>(re.h.x) + static_cast<double>(re.l.x),
                                 static_cast<double>(im.h.x) + static_cast<double>(im.l.x))
                  : make_double2(static_cast<double>(re.h.y) + static_cast<double>(re.l.y),
                                 static_cast<double>(im.h.y) + static_cast<double>(im.l.y));
}

constexpr int kDfTableEntries = 1024;

static __device__ const float4 kSinCosDF[kDfTableEntries] =
#include "sincos_table_df.inc"
    ;

// The table of exp(i 2 pi k/1024), k = 0 .. 1023, as double-floats, copied by
// the CTA's threads into shared memory.
__device__ __forceinline__ void load_sincos_table_df(float4* tab)
{
#pragma unroll 16
    for (int i = threadIdx.x; i < kDfTableEntries; i += blockDim.x) tab[i] = __ldg(&kSinCosDF[i]);
}

}  // namespace wt
