// Refined-FP32 determinant step (GBS_FP32_REFINED).
//
// Below the FP64 pivots of U the elimination runs on unevaluated pairs of FP32
// numbers (about 48 significant bits): a product of two pairs is split by FMAs, and
// "entry minus products" is summed with two-sums into a leading part and a
// gathered remainder (Acc), normalised only where it becomes a factor.
//
// The leaf. With X the (c2, j) block of the Schur complement after eliminating the
// prefix and c3, and the c2 pivot factored as Pi2 = [[1, 0], [l, 1]]
// diag(1/i0^2, 1/i1^2) [[1, l], [0, 1]], the rows a = i0 X_0, b = i1 (X_1 - l X_0)
// give the leaf's block Sch_j = D - a a^T - b b^T, and
//   P0(S) / P0(S') = det(Sch_j)^{-1/2} = r0 (1 + eta),
// r0 the FP32 reciprocal square root and eta its residual's correction (eta also
// carries the low part of the determinant: one step of refinement to FP64
// accuracy). Bound by FP32 issue, about 240 instructions a leaf. The block's three
// sums are normalised before the determinant (9 of them; M = 144, kmax = 5: 10.56 ->
// 10.72 ms the call): without that, P0 of two-mode squeezed pairs was off by 1.0e-10
// at r = 3, with it by 1.6e-12 (M = 8 to 66, relative, largest).
#pragma once
#include <cuda_runtime.h>

namespace gbs {

// FP32 value as FP64, assembled from its bits on the integer pipe (GB300 runs
// FP32<->FP64 conversions on its narrow FP64 pipe). Zero and subnormal inputs
// give a signed zero; inputs here are finite.
__device__ __forceinline__ double f2d_bits(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xffu;
    const unsigned long long sign = (unsigned long long)(b & 0x80000000u) << 32;
    const unsigned long long r =
        sign | ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)(b & 0x7fffffu) << 29);
    return __longlong_as_double((long long)(e == 0u ? sign : r));
}

// FP64 value truncated to FP32 (toward zero: relative error below 2^-23),
// assembled from its bits on the integer pipe. Finite inputs in FP32's normal
// range only; any other input (zero, below 2^-126, at or above 2^128, inf, NaN)
// gives 0.
__device__ __forceinline__ float d2f_bits(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu) - 896;
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned r = (hi & 0x80000000u) | ((unsigned)e << 23) | m;
    return (e > 0 && e < 255) ? __uint_as_float(r) : 0.f;
}

// Double-float (unevaluated FP32 pair) value h + l.
struct DF {
    float h, l;
};
__device__ __forceinline__ DF df_norm(float s, float t) {  // fast two-sum, |s| >= |t|
    const float r = __fadd_rn(s, t);
    return DF{r, __fsub_rn(t, __fsub_rn(r, s))};
}
// a * b, not normalised (the low part holds the product's rounding error and the
// cross terms)
__device__ __forceinline__ DF df_mulu(DF a, DF b) {
    const float p = a.h * b.h;
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e));
    return DF{p, e};
}
__device__ __forceinline__ DF df_mul(DF a, DF b) {
    const DF p = df_mulu(a, b);
    return df_norm(p.h, p.l);
}

__device__ __forceinline__ void split_df(double x, float &h, float &l) {
    h = __double2float_rn(x);
    l = __double2float_rn(x - (double)h);
}

// x truncated to FP32 and the rest (below FP32's normal range: the rounded value alone).
__device__ __forceinline__ float2 pair_of_double(double x) {
    const float h = d2f_bits(x);
    return make_float2(h, __double2float_rn(x - f2d_bits(h)));
}

// Running sum s + t, not normalised.
struct Acc {
    float s, t;
};
__device__ __forceinline__ DF acc_norm(Acc a) { return df_norm(a.s, a.t); }
// acc -= a * b (two-product by FMA, two-sum; a.l b.l dropped, below 2^-48 of it)
__device__ __forceinline__ void acc_sub(Acc &c, DF a, DF b) {
    const DF p = df_mulu(a, b);
    const float s = __fadd_rn(c.s, -p.h);
    const float bb = __fsub_rn(s, c.s);
    const float err = __fadd_rn(__fsub_rn(c.s, __fsub_rn(s, bb)), __fsub_rn(-p.h, bb));
    c.s = s;
    c.t = __fadd_rn(c.t, __fsub_rn(err, p.l));
}
// acc -= a^2 where acc stays positive, a diagonal element (so |acc| >= a^2 and the
// fast two-sum is exact)
__device__ __forceinline__ void acc_sub_sq(Acc &c, DF a) {
    const float p = a.h * a.h;
    const float q = __fmaf_rn(a.h, a.l + a.l, __fmaf_rn(a.h, a.h, -p));
    const float s = __fsub_rn(c.s, p);
    const float err = __fsub_rn(__fsub_rn(c.s, s), p);
    c.s = s;
    c.t = __fadd_rn(c.t, __fsub_rn(err, q));
}

// 1 / sqrt(x) = y (1 + eta), x = h + l > 0 normal: the hardware's approximation
// and its residual, eta exact to about 2^-46.
__device__ __forceinline__ void df_rsqrt(DF x, float &y, float &eta) {
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x.h));
    const float q = y * y;
    const float ql = __fmaf_rn(y, y, -q);
    const float rho = __fmaf_rn(-x.l, q, __fmaf_rn(-x.h, ql, __fmaf_rn(-x.h, q, 1.f)));
    eta = rho * __fmaf_rn(0.375f, rho, 0.5f);
}
__device__ __forceinline__ DF df_rsqrt(DF x) {
    float y, eta;
    df_rsqrt(x, y, eta);
    return df_norm(y, y * eta);
}

// 2x2 pivot [[d00, d01], [d01, d11]] as [[1, 0], [l, 1]] diag(1/i0^2, 1/i1^2) [[1, l], [0, 1]].
struct Piv {
    DF i0, l, i1;
};
// 2x2 blocks of pairs, and of running sums.
struct DFBlk {
    DF a00, a01, a10, a11;
};
struct ABlk {
    Acc a00, a01, a10, a11;
};
struct ASym {
    Acc s00, s01, s11;
};
__device__ __forceinline__ Piv pivot_of(const ASym &d, bool &ok) {
    const DF a = acc_norm(d.s00), b = acc_norm(d.s01);
    Piv p;
    p.i0 = df_rsqrt(a);
    p.l = df_mul(df_mul(b, p.i0), p.i0);
    Acc c = d.s11;
    acc_sub(c, p.l, b);
    const DF q = acc_norm(c);
    p.i1 = df_rsqrt(q);
    ok = a.h > 0.f && q.h > 0.f;
    return p;
}

// c -= x^T y for one pivot row's elements (x0, x1), (y0, y1).
__device__ __forceinline__ void acc_sub_row(ABlk &c, DF x0, DF x1, DF y0, DF y1) {
    acc_sub(c.a00, x0, y0);
    acc_sub(c.a01, x0, y1);
    acc_sub(c.a10, x1, y0);
    acc_sub(c.a11, x1, y1);
}

// The pivot rows of a block X below a factored pivot: i0 X_0 and i1 (X_1 - l X_0).
__device__ __forceinline__ DFBlk pivot_rows(ABlk x, const Piv &p) {
    const DF x0 = acc_norm(x.a00), x1 = acc_norm(x.a01);
    acc_sub(x.a10, p.l, x0);
    acc_sub(x.a11, p.l, x1);
    return DFBlk{df_mulu(p.i0, x0), df_mulu(p.i0, x1), df_mulu(p.i1, acc_norm(x.a10)), df_mulu(p.i1, acc_norm(x.a11))};
}

// d - w^T w for a symmetric block d and the two pivot rows w.
__device__ __forceinline__ ASym acc_sub_gram(ASym d, const DFBlk &w) {
    acc_sub_sq(d.s00, w.a00);
    acc_sub(d.s01, w.a00, w.a01);
    acc_sub_sq(d.s11, w.a01);
    acc_sub_sq(d.s00, w.a10);
    acc_sub(d.s01, w.a10, w.a11);
    acc_sub_sq(d.s11, w.a11);
    return d;
}

// det(Sch_j)^{-1/2} = r0 (1 + eta) of one leaf, S the (c2, j) block of the Schur
// complement after eliminating U, z2 and zj the pivot rows of c3 at c2 and j, d =
// the j block after c3 and pv the c2 pivot after c3; ok = false if the leaf's
// block is not positive definite.
__device__ __forceinline__ void refined_leaf_factor(ABlk S, const DFBlk &z2, const DFBlk &zj, const ASym &d,
                                                    const Piv &pv, float &r0, float &eta, bool &ok) {
    acc_sub_row(S, z2.a00, z2.a01, zj.a00, zj.a01);
    acc_sub_row(S, z2.a10, z2.a11, zj.a10, zj.a11);
    const ASym sch = acc_sub_gram(d, pivot_rows(S, pv));
    // normalised first: where the elimination cancels (j's two-mode squeezed partner in
    // the prefix) the remainders are not small beside the leading parts, and the
    // products below drop what is of second order in them
    const DF a = acc_norm(sch.s00), b = acc_norm(sch.s01), c = acc_norm(sch.s11);
    // det = a c - b^2 (a c >= b^2: the fast two-sum is exact)
    const DF p = df_mulu(a, c);
    const float q = b.h * b.h;
    const float ql = __fmaf_rn(b.h, b.l + b.l, __fmaf_rn(b.h, b.h, -q));
    const float s = __fsub_rn(p.h, q);
    const float err = __fsub_rn(__fsub_rn(p.h, s), q);
    ok = a.h > 0.f && s > 0.f;
    df_rsqrt(DF{s, __fadd_rn(err, __fsub_rn(p.l, ql))}, r0, eta);
}

// P0(S) = P0(S') r0 (1 + eta): two FP64 operations.
__device__ __forceinline__ double refined_leaf_p0(double P0Sp, float r0, float eta) {
    const double u = P0Sp * f2d_bits(r0);
    return fma(u, f2d_bits(eta), u);
}

}  // namespace gbs
