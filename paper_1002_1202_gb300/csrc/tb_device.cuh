// Device functions shared by the kernels of tb_kernels.cu (grid-wide panels)
// and tb_slice.cu (column slices): complex and double-float arithmetic and
// the scalars of the recurrences.
#pragma once

#include "tb_internal.h"

namespace tb {
namespace {

__device__ __forceinline__ double2 cmk(double r, double i) { return make_double2(r, i); }
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return cmk(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return cmk(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return cmk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// complex division by Smith's method (no intermediate overflow of |b|^2)
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    if (fabs(b.x) >= fabs(b.y)) {
        double r = b.y / b.x, den = b.x + b.y * r;
        return cmk((a.x + a.y * r) / den, (a.y - a.x * r) / den);
    }
    double r = b.x / b.y, den = b.y + b.x * r;
    return cmk((a.x * r + a.y) / den, (a.y * r - a.x) / den);
}

// Double-float products for FP64-accurate SpMVs on FP32 units (mixed path).
// A value is carried as hi + lo (two FP32 numbers, |lo| <= ulp(hi)/2).
// acc += s * x: the rounded product p = sh*xh and its exact error
// fma(sh, xh, -p) (Dekker / Ogita-Rump-Oishi error-free transformations),
// the cross terms sh*xl + sl*xh (sl*xl is below the working accuracy), and a
// two-sum of hi + p whose error goes to lo.  The _rn intrinsics keep the
// compiler from contracting these steps into FMAs, which would break the
// error terms.  Relative accuracy of a sum of n products ~ n * 2^-46.
// df_mac2 does this for a (re, im) pair that shares s, in packed FP32
// instructions (two lanes each, round-to-nearest per lane: each lane
// computes exactly the scalar sequence); a - b is a + (-b), which is exact.
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ void df_mac2(float2& hi, float2& lo, float sh, float sl, float2 xh, float2 xl) {
    const float2 s2h = make_float2(sh, sh), s2l = make_float2(sl, sl);
    const float2 pr = __fmul2_rn(s2h, xh);
    float2 e = __ffma2_rn(s2h, xh, neg2(pr));
    e = __ffma2_rn(s2h, xl, e);
    e = __ffma2_rn(s2l, xh, e);
    const float2 t = __fadd2_rn(hi, pr);
    const float2 bp = __fadd2_rn(t, neg2(hi));
    const float2 err = __fadd2_rn(__fadd2_rn(hi, neg2(__fadd2_rn(t, neg2(bp)))), __fadd2_rn(pr, neg2(bp)));
    hi = t;
    lo = __fadd2_rn(lo, __fadd2_rn(err, e));
}

// complex double -> (re_hi, im_hi, re_lo, im_lo): the hi and lo pairs are
// the two float2 operands of df_mac2
__device__ __forceinline__ float4 df_split(double2 v) {
    const float rh = (float)v.x, ih = (float)v.y;
    return make_float4(rh, ih, (float)(v.x - (double)rh), (float)(v.y - (double)ih));
}

// Scalars of outer step n of one column from m = u'_n^T W (one thread):
// asig = m / t_n, and the factors of the update
//     u_{n+1} = g (W - asig u_n) - f u_{n-1},  g = 1 / (nu_n s), f = B_n / (nu_{n-1} s),
// scaled by s = B_n (1 at the first step), so that nu_{n+1} = B_{n+1} / s stays
// near one however the residuals shrink.  False (and the column is
// deactivated) when t_n is not positive and finite, or when the seed shift
// z_s makes the pivot of its own recurrence vanish (a real shift on a level):
// D_n = z_s - a_n - B_n^2 / D_{n-1}.
__device__ __forceinline__ bool lanczos_step_scalars(ColState& cs, double m, double2 zs) {
    const double asig = m / cs.t;
    double2 D = make_double2((zs.x - cs.sigma) - asig, zs.y);
    if (cs.iters > 0) {
        D.x -= cs.B * cs.B * cs.sinv.x;
        D.y -= cs.B * cs.B * cs.sinv.y;
    }
    if (!(cs.t > 0.0) || !isfinite(m) || !isfinite(cs.t) || (D.x == 0.0 && D.y == 0.0)) {
        cs.active = 0;
        return false;
    }
    const double s = cs.iters > 0 ? cs.B : 1.0;
    cs.asig = asig;
    cs.s = s;
    cs.g = 1.0 / (cs.nu * s);
    cs.f = cs.iters > 0 ? cs.B / (cs.nu_prev * s) : 0.0;
    return true;
}

// Shift k of a column at outer step n: the pivot of the tridiagonal z_k - T,
//     D_n = z_k - a_n - B_n^2 / D_{n-1},
// the step's coefficients alpha = zeta_n / D_n and l = B_{n+1} / D_n, and
// zeta_{n+1} = l zeta_n, |zeta_{n+1}| ||u^_{n+1}|| being the residual of
// shift k (the collinear residual of Eq. collinear): the COCG iterates of
// shift k for whatever seed, with one complex division per shift and step.
// Im D_n has the sign of Im z_k and at least its size, so no pivot vanishes
// off the real axis.
struct ShiftCoef {
    double2 inv, al, l, zeta;
};
__device__ __forceinline__ ShiftCoef shift_coef(double2 z, double sigma, double asig, double B, double Bn,
                                                double2 pinv, double2 zeta) {
    const double B2 = B * B;
    const double2 D = cmk((z.x - sigma) - asig - B2 * pinv.x, z.y - B2 * pinv.y);
    ShiftCoef c;
    const double den = D.x * D.x + D.y * D.y;
    const double id = 1.0 / den;
    c.inv = cmk(D.x * id, -D.y * id);
    c.al = cmul(zeta, c.inv);
    c.l = cmk(Bn * c.inv.x, Bn * c.inv.y);
    c.zeta = cmk(Bn * c.al.x, Bn * c.al.y);
    return c;
}

}  // namespace
}  // namespace tb
