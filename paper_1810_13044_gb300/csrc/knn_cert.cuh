// The rounding bounds that decide which columns of a distance tile a row must
// keep, shared by the tensor-core sweep and its rerank.
//
// For a row p and a column q, D = ||xt_p - xt_q|| of the rounded operands, dt
// the tile's value for D^2 and d = ||x_p - x_q||:
//   |dt - D^2| <= coef (|xt_p| + |xt_q|)^2   (tile arithmetic, norms)
//   |D - d|    <= rho_p + rho_q              (operand rounding)
//   rho_q <= min(rmax, kap |xt_q|)           (largest rho, largest rho / |v|)
//
// Reach.  If k columns q' != p have dt <= dk, each has
//   D <= sqrt(dk) + sc (2 |xt_p| + D), sc = sqrt(coef), as |xt_q'| <= |xt_p| + D,
// which bounds |xt_q'|, with it D <= D1, and d <= s1 = D1 + rho_p + rho_q'.
// The k nearest by the float32 distances (each off by at most err_exact) then
// all have d <= sk = s1 (1 + 2.02 err_exact).
//
// Certificate.  Let every column a row did not list have D^2 >= T (or dt >= T)
// and K be the k-th exact distance of the listed ones, inflated by its
// rounding.  A column with |y_q| >= |y_p| + sqrt(K) (y = x - mu) is farther; any
// other has |xt_q| <= (|xt_p| + rho_p + sqrt(K)) / (1 - kap), which bounds its
// rho and the error delta of its dt, so the row is complete if
//   sqrt(T - delta) - rho_p - rho_q > sqrt(K).
//
// Threshold.  cert_thr(dk) is the T for which that holds if sqrt(K) turns out
// at most sqrt(dk) + eta times the rounding bounds, eta = 4 / sqrt(D) (at most
// 1): rho bounds the length of a rounding error, whose component along x_p -
// x_q, which moves D, is about 1 / sqrt(D) of that.  With the full bound (eta =
// 1) a row of the 1e6 x 128 manifolds keeps twice the columns; with eta = 0.2
// 1172 of 19870 rows of 9 features fail the certificate.  It grows with dk, so a row
// may drop columns at or above cert_thr of any earlier, larger dk.
// All steps are float32 with relative slack 1e-5 over their few roundings,
// and 1e-30 absolute for squares that underflow.
#pragma once

#include <math.h>

#include "slk_internal.cuh"

namespace {

struct CertConsts {
    float coef, sc, inv_sc, rmax, kap, inv_kap, snmax, ex, sn_infl, eta;
};

// gam: error of a tile's dot product relative to |xt_p| |xt_q|; maxima as
// float bits (norm^2, rho, rho / |v|).
__device__ __forceinline__ CertConsts cert_make(double gam, int Dp, int D, unsigned nmax_bits,
                                                unsigned rmax_bits, unsigned kappa_bits) {
    const double u = 5.9604644775390625e-08;
    CertConsts c;
    c.coef = (float)((gam + (double)(Dp / 32 + 5) * u) * (1.0 + 1e-6));
    c.sc = sqrtf(c.coef) * 1.000001f;
    c.inv_sc = c.sc < 0.5f ? 1.00001f / (1.f - c.sc) : __int_as_float(0x7f800000);
    c.rmax = __uint_as_float(rmax_bits) * 1.000001f;
    const float kappa = __uint_as_float(kappa_bits);
    c.kap = kappa < 0.25f ? kappa / (1.f - kappa) * 1.00001f : __int_as_float(0x7f800000);
    c.inv_kap = kappa < 0.25f ? 1.00001f / (1.f - c.kap) : __int_as_float(0x7f800000);
    c.sn_infl = (float)(1.0 + (double)(Dp / 32 + 8) * u + 1e-6);
    c.snmax = sqrtf(__uint_as_float(nmax_bits)) * c.sn_infl;
    c.ex = (float)(1.0 + 2.02 * 1.01 * (double)(D + 8) * u + 1e-6);
    c.eta = fminf(1.f, 4.f * rsqrtf((float)D));
    return c;
}

// sk of the derivation above: no q of the k nearest is farther than this.
__device__ __forceinline__ float cert_reach(const CertConsts& c, float sp, float rp, float dk) {
    const float d = fmaxf(dk, 0.f);
    const float b0 = (sqrtf(d) + 2.f * c.sc * sp) * c.inv_sc;
    const float q1 = fminf(sp + b0, c.snmax);
    const float t1 = sp + q1;
    const float s1 = sqrtf(d + c.coef * t1 * t1) + rp + fminf(c.rmax, c.kap * q1);
    return s1 * c.ex * 1.00001f;
}

// sqrt(T) that certifies a row whose k-th exact distance is at most sk, less
// the error of dt: sk + rho_p + rho_q and delta.
__device__ __forceinline__ void cert_need(const CertConsts& c, float sp, float rp, float sk, float& root,
                                          float& delta) {
    const float q2 = fminf((sp + rp + sk) * c.inv_kap, c.snmax);
    const float t2 = sp + q2;
    root = (sk + rp + fminf(c.rmax, c.kap * q2)) * 1.00001f;
    delta = c.coef * t2 * t2 * 1.00001f;
}

// The row's threshold (above; sp >= |xt_p|, rp >= rho_p).
__device__ __forceinline__ float cert_thr(const CertConsts& c, float sp, float rp, float dk) {
    if (!(dk < __int_as_float(0x7f800000))) return __int_as_float(0x7f800000);
    const float d = sqrtf(fmaxf(dk, 0.f));
    const float rq = fminf(c.rmax, c.kap * (sp + d));
    const float t1 = 2.f * sp + d;
    float root, delta;
    cert_need(c, sp, rp, sqrtf(fmaxf(dk, 0.f) + c.eta * c.coef * t1 * t1) * c.ex + c.eta * (rp + rq), root, delta);
    return (root * root + delta) * 1.00001f + 1e-30f;
}

// Whether a row is complete: dk the k-th exact distance, T as above.
__device__ __forceinline__ bool cert_ok(const CertConsts& c, float sp, float rp, float dk, float T) {
    float root, delta;
    cert_need(c, sp, rp, sqrtf(dk) * c.ex * 1.00001f, root, delta);
    return T > (root * root + delta) * 1.00001f;
}

}  // namespace
