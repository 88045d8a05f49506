// Local-density exchange-correlation per point: Slater exchange and the
// Perdew-Zunger 1981 fit (PRB 23, 5048), unpolarised.
#pragma once

namespace jdft {

// Conversions of normal numbers in FP32's range by integer instructions (the
// conversion instructions take a slot of the FP64 pipe each): truncated to 24 bits,
// and exact.
__device__ __forceinline__ float short_of(double x) {
    const int hi = __double2hiint(x);
    return __int_as_float((int)(((uint32_t)(hi - (896 << 20)) << 3) | ((uint32_t)__double2loint(x) >> 29)));
}
__device__ __forceinline__ double long_of(float x) {
    const int b = __float_as_int(x);
    return __hiloint2double((b >> 3) + (896 << 20), b << 29);
}

// Energy per electron e and potential v at density n (both zero for n <= 0).  A call,
// not inlined: the epilogues evaluate a dozen points per lane and few need it.
static __device__ __noinline__ void lda_pz_plain(double n, double& e, double& v) {
    if (!(n > 0.0)) { e = 0.0; v = 0.0; return; }
    const double cx = -0.73855876638202240588423003065;   // -(3/4)(3/pi)^{1/3}
    const double kr = 0.62035049089940001666800681204778;  // (3/(4 pi))^{1/3}
    const double third = 1.0 / 3.0;
    const double c = cbrt(n);
    const double ex = cx * c;
    const double rs = kr / c;
    double ec, vc;
    if (rs >= 1.0) {
        const double g = -0.1423, b1 = 1.0529, b2 = 0.3334;
        const double sq = sqrt(rs);
        const double iden = 1.0 / (1.0 + b1 * sq + b2 * rs);
        ec = g * iden;
        // r_s de_c/dr_s = -g (b1 sqrt(r_s) / 2 + b2 r_s) / den^2
        const double rdec = -g * (0.5 * b1 * sq + b2 * rs) * iden * iden;
        vc = ec - third * rdec;
    } else {
        const double A = 0.0311, B = -0.048, C = 0.0020, D = -0.0116;
        const double lr = log(rs);
        ec = A * lr + B + C * rs * lr + D * rs;
        // r_s de_c/dr_s = A + r_s (C (ln r_s + 1) + D)
        const double rdec = A + rs * (C * (lr + 1.0) + D);
        vc = ec - third * rdec;
    }
    e = ex + ec;
    v = (4.0 * third) * ex + vc;
}

// The same with the FP64 pipe's work cut to about 25 instructions where r_s >= 1
// (n <= 0.2387, nearly every point of a cell): t = n^(-1/6) from an FP32 estimate
// with one step of Householder's method (d = 1 - n t^6 is below 2^-16, the terms
// kept reach d^3), from which n^(1/3) and the fit in t (sqrt(r_s) and r_s are
// multiples of t and t^2) are products, and the reciprocal of the fit's denominator
// from an FP32 one with two terms of the geometric series.  What bounds the epilogue
// is still the FP64 pipe: 25 instructions for each of two million points are 90 us of
// a 128^3 box.  Emulated against 80 bits, e and v are off by 0.7 to 0.9 units of 2^-53
// (root mean square), as the plain form is with a correctly rounded cube root.
__device__ __forceinline__ void lda_pz(double n, double& e, double& v) {
    if (!(n > 1e-30 && n < 0.23)) { lda_pz_plain(n, e, v); return; }
    const double cx = -0.73855876638202240588423003065;
    const double g = -0.1423;
    const double p1 = 0.82928859141663966846;  // b1 sqrt(kr) and b2 kr of the plain form
    const double p2 = 0.20682485366585996556;
    const double t0 = long_of(exp2f(__log2f(short_of(n)) * (-1.0f / 6.0f)));
    const double t3 = (t0 * t0) * t0;  // the square is exact: t0 has 24 bits
    const double w = n * t3;
    const double d = fma(-w, t3, 1.0);
    // t = t0 (1 - d)^(-1/6) and n^(1/3) = n t0^4 (1 - d)^(-2/3), each by its own series: the
    // fourth power of t would multiply its rounding by four.  n t0^4 is formed from d's own
    // n t0^3, whose roundings d takes out again but for a third.
    const double t = fma(t0, d * fma(d, fma(d, 91.0 / 1296.0, 7.0 / 72.0), 1.0 / 6.0), t0);
    const double c0 = w * t0;
    const double c = fma(c0, d * fma(d, fma(d, 40.0 / 81.0, 5.0 / 9.0), 2.0 / 3.0), c0);
    const double den = fma(fma(t, p2, p1), t, 1.0);
    double r = long_of(__fdividef(1.0f, short_of(den)));
    const double f = fma(-den, r, 1.0);
    r = fma(r, fma(f, f, f), r);
    const double ec = g * r;
    // v_c = e_c - (r_s/3) de_c/dr_s = e_c (1 + (b1 sqrt(r_s)/2 + b2 r_s) / (3 den))
    const double vc = fma(ec * (t * r), fma(t, p2 / 3.0, p1 / 6.0), ec);
    e = fma(cx, c, ec);
    v = fma((4.0 / 3.0) * cx, c, vc);
}

}  // namespace jdft
