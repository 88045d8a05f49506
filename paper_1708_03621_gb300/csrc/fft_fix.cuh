// Line FFTs of FP64 data in 64-bit fixed point.
//
// What bounds an FP64 transform here is the FP64 pipe: 2 instructions per clock
// and SM (a probe of independent chains measured DFMA and DADD at 2.0, 64-bit
// integer additions at 65, 32 x 32 + 64 multiply-adds at 29 per clock and SM).
// A transform is mostly additions, so a line is converted once to 64-bit
// integers with a common power-of-two scale, transformed with integer
// additions and wide multiply-adds, and converted back.  Conversions are
// integer bit work too: the conversion instructions run at the FP64 rate.
//
// Scale: with L1 = sum over the line of |Re| + |Im|, every intermediate value
// of the transform is a sum of inputs times numbers of modulus at most 1, so
// its components stay below sqrt(2) L1.  The scale puts L1 just below 2^60:
// nothing can overflow.  Values are cut toward zero at a unit: a line of normal random
// values keeps 3.8, 2.0, 1.0 and 0.0 bits more than FP64's 53 below its largest component
// at 12, 48, 128 and 256 values, one with most of its values small more.  Roundings
// are half to one unit of 2^-60 L1 each, where FP64 rounds every operation to
// 2^-53 of its result: against the line's norm the transform's error is no larger than
// the FP64 one's (tests/test_gpu_fixfft.py).
//
// Measured (H C, FP64 blocks): 64 bands on a 128^3 box 39.45 -> 28.06 ms, 16 bands
// on 48^3 486 -> 432 us, the projector products included; error against 64-bit
// references unchanged (1.5e-16 and 1.4e-16 of the result's norm).
//
// Values: an infinity or NaN in a line makes the whole line's output NaN (the
// FP64 transform spreads it over the line too).  Lines below 2^-959 are scaled
// up first, results outside the normal range scaled back by an FP64 multiply.
#pragma once

#include "fft.cuh"

namespace jdft {

using i64 = long long;

// The "scalar type" of the fixed-point transforms: complex values are
// longlong2, twiddles int4 {Re hi, Re lo, Im hi, Im lo} with
// w = hi 2^-30 + lo 2^-62, lo in (-2^31, 2^31).
struct fix64 {};
template <> struct cplx<fix64> { using type = longlong2; };
template <typename T> struct twiddle { using type = c_t<T>; };
template <> struct twiddle<fix64> { using type = int4; };
template <typename T> using tw_t = typename twiddle<T>::type;

// Split of an integer multiple of 2^-62 into the two words.
struct FixW {
    int h, l;
};
__host__ __device__ constexpr FixW fix_split(i64 q) {
    return FixW{(int)((q + (i64(1) << 31)) >> 32),
                (int)(q - ((q + (i64(1) << 31)) >> 32) * (i64(1) << 32))};
}
// cos and sin values of the butterflies in units of 2^-62 (rounded to nearest)
constexpr i64 kFixC8 = 4260642322793532497ll;    // cos(pi/8)
constexpr i64 kFixS8 = 1764815834521887442ll;    // sin(pi/8)
constexpr i64 kFixH = 3260954456333195553ll;     // cos(pi/4)
constexpr i64 kFixS3 = 3993837246235628775ll;    // sqrt(3)/2
constexpr i64 kFixC51 = 1425089352415399811ll;   // cos(2 pi/5)
constexpr i64 kFixC52 = -3730932361629093763ll;  // cos(4 pi/5)
constexpr i64 kFixS51 = 4385974038932618941ll;   // sin(2 pi/5)
constexpr i64 kFixS52 = 2710681029835013083ll;   // sin(4 pi/5)
// cos and sin of 2 pi k/9, k = 1, 2, 4
constexpr i64 kFixC91 = 3532756447825785444ll, kFixS91 = 2964334632409774423ll;
constexpr i64 kFixC92 = 800810873071977681ll, kFixS92 = 4541624145405292212ll;
constexpr i64 kFixC94 = -4333567320897763126ll, kFixS94 = 1577289512995517789ll;

// x = h 2^32 + l with both words signed.
__device__ __forceinline__ void fix_words(i64 x, int& h, int& l) {
    l = (int)x;
    h = (int)(x >> 32) - (l >> 31);
}
// Product sums: hi collects word products h h (weight 2^2 after the scaling by
// 2^-62), mid the cross products (weight 2^-30, started at half a unit); the
// products of low words (below one unit) are dropped.
constexpr i64 kFixHalf = i64(1) << 29;
__device__ __forceinline__ i64 fix_sum(i64 hi, i64 mid) { return (hi << 2) + (mid >> 30); }

// a real constant times a value (|x| < 2^61)
__device__ __forceinline__ i64 fix_mul(i64 x, FixW w) {
    int h, l;
    fix_words(x, h, l);
    return fix_sum((i64)h * w.h, (i64)h * w.l + ((i64)l * w.h + kFixHalf));
}
__device__ __forceinline__ longlong2 cscale(longlong2 a, FixW w) {
    return make_longlong2(fix_mul(a.x, w), fix_mul(a.y, w));
}
// a w and a conj(w) (components below 2^61: the four cross products of a
// component stay below 2^63)
__device__ __forceinline__ longlong2 cmul(longlong2 a, int4 w) {
    int xh, xl, yh, yl;
    fix_words(a.x, xh, xl);
    fix_words(a.y, yh, yl);
    const int nh = -w.z, nl = -w.w;
    const i64 rh = (i64)xh * w.x + (i64)yh * nh;
    const i64 rm = (i64)xh * w.y + ((i64)xl * w.x + ((i64)yh * nl + ((i64)yl * nh + kFixHalf)));
    const i64 ih = (i64)xh * w.z + (i64)yh * w.x;
    const i64 im = (i64)xh * w.w + ((i64)xl * w.z + ((i64)yh * w.y + ((i64)yl * w.x + kFixHalf)));
    return make_longlong2(fix_sum(rh, rm), fix_sum(ih, im));
}
__device__ __forceinline__ longlong2 cmulc(longlong2 a, int4 w) {
    return cmul(a, make_int4(w.x, w.y, -w.z, -w.w));
}

template <int SIGN>
__device__ __forceinline__ void dft3_fix(longlong2* v) {
    constexpr FixW h = fix_split(kFixS3);
    const longlong2 t1 = cadd(v[1], v[2]);
    const longlong2 t2 = cscale(cmul_i<SIGN>(csub(v[1], v[2])), h);
    const longlong2 m = make_longlong2(v[0].x - ((t1.x + 1) >> 1), v[0].y - ((t1.y + 1) >> 1));
    v[0] = cadd(v[0], t1);
    v[1] = cadd(m, t2);
    v[2] = csub(m, t2);
}

template <int SIGN>
__device__ __forceinline__ void dft5_fix(longlong2* v) {
    constexpr FixW c1 = fix_split(kFixC51), c2 = fix_split(kFixC52), s1 = fix_split(kFixS51), s2 = fix_split(kFixS52);
    const longlong2 a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
    const longlong2 a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
    const longlong2 x0 = v[0];
    const longlong2 p1 = cadd(x0, cadd(cscale(a1, c1), cscale(a2, c2)));
    const longlong2 p2 = cadd(x0, cadd(cscale(a1, c2), cscale(a2, c1)));
    const longlong2 q1 = cmul_i<SIGN>(cadd(cscale(b1, s1), cscale(b2, s2)));
    const longlong2 q2 = cmul_i<SIGN>(csub(cscale(b1, s2), cscale(b2, s1)));
    v[0] = cadd(x0, cadd(a1, a2));
    v[1] = cadd(p1, q1);
    v[4] = csub(p1, q1);
    v[2] = cadd(p2, q2);
    v[3] = csub(p2, q2);
}

// (1 + SIGN i) a / sqrt 2 and (-1 + SIGN i) a / sqrt 2
template <int SIGN>
__device__ __forceinline__ longlong2 rot45_fix(longlong2 a) {
    constexpr FixW h = fix_split(kFixH);
    return make_longlong2(fix_mul(a.x - SIGN * a.y, h), fix_mul(a.y + SIGN * a.x, h));
}
template <int SIGN>
__device__ __forceinline__ longlong2 rot135_fix(longlong2 a) {
    constexpr FixW h = fix_split(kFixH);
    return make_longlong2(fix_mul(-a.x - SIGN * a.y, h), fix_mul(SIGN * a.x - a.y, h));
}

// W9^k, k = 1, 2, 4
template <int SIGN>
__device__ __forceinline__ longlong2 rot9_fix(longlong2 a, int k) {
    constexpr FixW c1 = fix_split(kFixC91), s1 = fix_split(SIGN * kFixS91), c2 = fix_split(kFixC92),
                   s2 = fix_split(SIGN * kFixS92), c4 = fix_split(kFixC94), s4 = fix_split(SIGN * kFixS94);
    if (k == 0) return a;
    if (k == 1) return cmul(a, make_int4(c1.h, c1.l, s1.h, s1.l));
    if (k == 2) return cmul(a, make_int4(c2.h, c2.l, s2.h, s2.l));
    return cmul(a, make_int4(c4.h, c4.l, s4.h, s4.l));
}

template <int SIGN>
__device__ __forceinline__ void dft8_fix(longlong2* v) {
    longlong2 e[4] = {v[0], v[2], v[4], v[6]};
    longlong2 o[4] = {v[1], v[3], v[5], v[7]};
    dft4<fix64, SIGN>(e);
    dft4<fix64, SIGN>(o);
    const longlong2 w1 = rot45_fix<SIGN>(o[1]), w2 = cmul_i<SIGN>(o[2]), w3 = rot135_fix<SIGN>(o[3]);
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cadd(e[1], w1);
    v[5] = csub(e[1], w1);
    v[2] = cadd(e[2], w2);
    v[6] = csub(e[2], w2);
    v[3] = cadd(e[3], w3);
    v[7] = csub(e[3], w3);
}

// a exp(SIGN i pi e / 8), e = n1 k1 in 0 .. 9
template <int SIGN>
__device__ __forceinline__ longlong2 rot16_fix(longlong2 a, int e) {
    constexpr FixW c = fix_split(kFixC8), s = fix_split(SIGN > 0 ? kFixS8 : -kFixS8);
    constexpr FixW nc = fix_split(-kFixC8), ns = fix_split(SIGN > 0 ? -kFixS8 : kFixS8);
    constexpr FixW ss = fix_split(kFixS8), cc = fix_split(SIGN > 0 ? kFixC8 : -kFixC8);
    switch (e) {
        case 0: return a;
        case 1: return cmul(a, make_int4(c.h, c.l, s.h, s.l));
        case 2: return rot45_fix<SIGN>(a);
        case 3: return cmul(a, make_int4(ss.h, ss.l, cc.h, cc.l));
        case 4: return cmul_i<SIGN>(a);
        case 6: return rot135_fix<SIGN>(a);
        default: return cmul(a, make_int4(nc.h, nc.l, ns.h, ns.l));  // e = 9
    }
}

template <int SIGN>
__device__ __forceinline__ void dft16_fix(longlong2* v) {
    longlong2 a[4][4];
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) {
        longlong2 w[4] = {v[n1], v[n1 + 4], v[n1 + 8], v[n1 + 12]};
        dft4<fix64, SIGN>(w);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) a[n1][k1] = rot16_fix<SIGN>(w[k1], n1 * k1);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        longlong2 w[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
        dft4<fix64, SIGN>(w);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = w[k2];
    }
}

template <int SIGN, int R>
__device__ __forceinline__ void dft_fix(longlong2* v) {
    if constexpr (R == 2) dft2<fix64, SIGN>(v);
    else if constexpr (R == 3) dft3_fix<SIGN>(v);
    else if constexpr (R == 4) dft4<fix64, SIGN>(v);
    else if constexpr (R == 5) dft5_fix<SIGN>(v);
    else if constexpr (R == 8) dft8_fix<SIGN>(v);
    else if constexpr (R == 16) dft16_fix<SIGN>(v);
}

// ---------------------------------------------------------------------------
// Conversions.  A line's integers stand for x 2^q.
// ---------------------------------------------------------------------------
struct FixScale {
    int q;     // binary weight of a unit
    bool bad;  // the line holds an infinity or NaN
};

__device__ __forceinline__ int fix_abs_hi(double x) { return __double2hiint(x) & 0x7fffffff; }

// |x| relative to 2^(emax - 1023), truncated to 21 significant bits (0 below 2^-126 of it)
__device__ __forceinline__ float fix_relative(double x, int bias) {
    return __int_as_float(max(fix_abs_hi(x) - bias, 0) << 3);
}

// x's significand shifted to the line's unit (see fix_line_in), truncated toward zero
__device__ __forceinline__ i64 fix_encode(double x, int nbase) {
    const int hi = __double2hiint(x);
    const int n = min(nbase - ((hi >> 20) & 0x7ff), 63);
    const uint64_t m = (((uint64_t)(uint32_t)((hi & 0xfffff) | 0x100000)) << 32) | (uint32_t)__double2loint(x);
    const i64 u = (i64)((m << 7) >> n);
    const i64 s = (i64)(hi >> 31);
    return (u ^ s) - s;
}

// x 2^q as a double, rounded to nearest (q in the range where the result is normal)
__device__ __forceinline__ double fix_decode(i64 x, int q) {
    const int s = (int)(x >> 63);
    const i64 sm = (i64)s;
    const uint64_t a = (uint64_t)((x ^ sm) - sm);
    const int lz = __clzll((i64)a);
    const uint64_t r = ((a << ((lz - 1) & 63)) + 0x200) >> 10;
    const int field = 1085 + q - lz;  // exponent field less one: r carries the implicit bit
    int hi = (int)(r >> 32) + (field << 20);
    hi = a == 0 ? 0 : hi;
    return __hiloint2double(hi | (s & 0x80000000), (int)r);
}

// Maximum and sum over the TL lanes of a line (lane l belongs to line l mod LPW,
// LPW = 32 / TL; lanes past TL LPW belong to none).
template <int TL>
__device__ __forceinline__ int line_max(int x) {
    constexpr int LPW = 32 / TL;
    if constexpr ((TL & (TL - 1)) == 0) {
#pragma unroll
        for (int m = LPW; m < 32; m <<= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, m));
        return x;
    } else {
        const int lane = threadIdx.x & 31;
        int r = x;
#pragma unroll
        for (int i = 1; i < TL; ++i) {
            const int s = lane + i * LPW;
            r = max(r, __shfl_sync(0xffffffffu, x, s < TL * LPW ? s : s - TL * LPW));
        }
        return r;
    }
}
template <int TL>
__device__ __forceinline__ float line_sum(float x) {
    constexpr int LPW = 32 / TL;
    if constexpr ((TL & (TL - 1)) == 0) {
#pragma unroll
        for (int m = LPW; m < 32; m <<= 1) x += __shfl_xor_sync(0xffffffffu, x, m);
        return x;
    } else {
        // every lane adds in the same order (from the line's first lane), so all lanes get the same scale
        const int line = (threadIdx.x & 31) % LPW;
        float r = 0.f;
#pragma unroll
        for (int i = 0; i < TL; ++i) r += __shfl_sync(0xffffffffu, x, line + i * LPW);
        return r;
    }
}

// E values per lane of lines of TL lanes: v becomes integers.
template <int E, int TL>
__device__ __forceinline__ FixScale fix_line_in(const double2* v, longlong2* x) {
    int amax = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) amax = max(amax, max(fix_abs_hi(v[e].x), fix_abs_hi(v[e].y)));
    amax = line_max<TL>(amax);
    int emax = amax >> 20;
    const bool bad = emax == 0x7ff;
    int up = 0;
    double2 w[E];
#pragma unroll
    for (int e = 0; e < E; ++e) w[e] = v[e];
    if (__any_sync(0xffffffffu, amax > 0 && emax < 64)) {
        // tiny lines: scaled up exactly by 2^512
        up = (amax > 0 && emax < 64) ? 512 : 0;
        const double f = __hiloint2double((1023 + up) << 20, 0);
        amax = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            w[e].x *= f;
            w[e].y *= f;
            amax = max(amax, max(fix_abs_hi(w[e].x), fix_abs_hi(w[e].y)));
        }
        amax = line_max<TL>(amax);
        emax = amax >> 20;
    }
    emax = max(emax, 64);  // all-zero lines
    const int bias = (emax - 127) * (1 << 20);
    float s = 1e-30f;
#pragma unroll
    for (int e = 0; e < E; ++e) s += fix_relative(w[e].x, bias) + fix_relative(w[e].y, bias);
    s = line_sum<TL>(s);
    // L1 < 2^(es + 1) 2^(emax - 1023), with a margin for the truncated terms and the float sum
    const int es = max((__float_as_int(s * 1.0001f) >> 23) - 127, 0);
    // x = 1.f 2^(ex - 1023) becomes 1.f 2^(59 - es - (emax - ex)): L1 < 2^60 units
    const int nbase = es + emax;
#pragma unroll
    for (int e = 0; e < E; ++e) x[e] = make_longlong2(fix_encode(w[e].x, nbase), fix_encode(w[e].y, nbase));
    return FixScale{es + emax - 1082 - up, bad};
}

template <int E>
__device__ __forceinline__ void fix_line_out(const longlong2* x, double2* v, FixScale sc) {
    // results are normal for q in [-1018, 960]; outside, convert at a nearer q and scale
    const int q = min(max(sc.q, -1018), 960);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = make_double2(fix_decode(x[e].x, q), fix_decode(x[e].y, q));
    if (__any_sync(0xffffffffu, sc.bad || q != sc.q)) {
        double f = __hiloint2double((1023 + sc.q - q) << 20, 0);
        if (sc.bad) f = __hiloint2double(0x7ff80000, 0);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e].x *= f;
            v[e].y *= f;
        }
    }
}

}  // namespace jdft
