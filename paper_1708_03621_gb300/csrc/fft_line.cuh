// Register line FFTs of any compiled length: the transforms of fft_reg.cuh without
// its requirement that the lanes of a line divide the warp and share the
// butterflies evenly, so that lengths with factors 3 and 5 are served too.
//
// A line of N values has TL lanes (any number up to 32; a warp serves LPW =
// 32 / TL lines, lane l being position l / LPW of line l mod LPW, the lanes past
// TL LPW idle).  A stage of radix R has N / R butterflies, which the lanes take in
// turns; a lane without one skips the arithmetic, and its values are invalid
// (in_valid, out_valid).  The stages are those of the Stockham transform in
// fft_reg.cuh, with radices 6, 9 and 10 as well (fewer stages: each costs an
// exchange through shared memory).  FP64 lines run in fixed point (fft_fix.cuh).
#pragma once

#include "fft_reg.cuh"

namespace jdft {

// 6 = 3 x 2 and 10 = 5 x 2 by the prime-factor map: with n = 3 a + 2 b mod 6 and
// k = 3 a' + 4 b' mod 6 (10: n = 5 a + 2 b, k = 5 a' + 6 b'), W6^(n k) = W2^(a a') W3^(b b').
template <typename T, int SIGN>
__device__ __forceinline__ void dft6_any(c_t<T>* v);
template <typename T, int SIGN>
__device__ __forceinline__ void dft9_any(c_t<T>* v);
template <typename T, int SIGN>
__device__ __forceinline__ void dft10_any(c_t<T>* v);

template <typename T, int SIGN, int R>
__device__ __forceinline__ void dft_any(c_t<T>* v) {
    if constexpr (R == 6) dft6_any<T, SIGN>(v);
    else if constexpr (R == 9) dft9_any<T, SIGN>(v);
    else if constexpr (R == 10) dft10_any<T, SIGN>(v);
    else dft_r<T, SIGN, R>(v);
}

template <typename T, int SIGN>
__device__ __forceinline__ void dft6_any(c_t<T>* v) {
    c_t<T> a[3] = {v[0], v[2], v[4]}, b[3] = {v[3], v[5], v[1]};
    dft_r<T, SIGN, 3>(a);
    dft_r<T, SIGN, 3>(b);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[(4 * k) % 6] = cadd(a[k], b[k]);
        v[(3 + 4 * k) % 6] = csub(a[k], b[k]);
    }
}

template <typename T, int SIGN>
__device__ __forceinline__ void dft10_any(c_t<T>* v) {
    c_t<T> a[5] = {v[0], v[2], v[4], v[6], v[8]}, b[5] = {v[5], v[7], v[9], v[1], v[3]};
    dft_r<T, SIGN, 5>(a);
    dft_r<T, SIGN, 5>(b);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        v[(6 * k) % 10] = cadd(a[k], b[k]);
        v[(5 + 6 * k) % 10] = csub(a[k], b[k]);
    }
}

// a exp(SIGN 2 pi i k / 9), k = 0, 1, 2, 4
template <typename T, int SIGN>
__device__ __forceinline__ c_t<T> rot9(c_t<T> a, int k) {
    if constexpr (std::is_same<T, fix64>::value) {
        return rot9_fix<SIGN>(a, k);
    } else {
        if (k == 0) return a;
        const T c = k == 1 ? T(0.76604444311897803520) : k == 2 ? T(0.17364817766693034885) : T(-0.93969262078590838405);
        const T s = (k == 1 ? T(0.64278760968653932632) : k == 2 ? T(0.98480775301220805937) : T(0.34202014332566873304)) *
                    T(SIGN);
        return mk<T>(a.x * c - a.y * s, a.x * s + a.y * c);
    }
}

template <typename T, int SIGN>
__device__ __forceinline__ void dft9_any(c_t<T>* v) {
    c_t<T> a[3][3];
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) {
        c_t<T> w[3] = {v[n1], v[n1 + 3], v[n1 + 6]};
        dft_r<T, SIGN, 3>(w);
#pragma unroll
        for (int k1 = 0; k1 < 3; ++k1) a[n1][k1] = rot9<T, SIGN>(w[k1], n1 * k1);
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
        c_t<T> w[3] = {a[0][k1], a[1][k1], a[2][k1]};
        dft_r<T, SIGN, 3>(w);
#pragma unroll
        for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = w[k2];
    }
}

constexpr int per_lane(int N, int TL, int R) { return (N / R + TL - 1) / TL; }
// Whether every lane of the warp has a butterfly in every turn of a radix-R stage;
// otherwise each turn checks its index (lanes past TL LPW have t past N).
constexpr bool all_busy(int N, int TL, int R) { return 32 % TL == 0 && (N / R) % TL == 0; }

// One stage (NS, R): inputs and outputs v[u R + r] of butterfly j = t + TL u.
// ADJ: the adjoint stage (the DFT, then the twiddles), of sign SIGN.
template <typename T, int N, int TL, int SIGN, int NS, int R, bool ADJ>
__device__ __forceinline__ void any_stage(c_t<T>* v, int t, const tw_t<T>* __restrict__ W) {
    constexpr int B = N / R, U = per_lane(N, TL, R);
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int j = t + TL * u;
        if (!all_busy(N, TL, R) && j >= B) continue;
        if constexpr (ADJ) dft_any<T, SIGN, R>(v + u * R);
        const int k = j % NS;
        if (NS > 1 && k != 0) {
            tw_t<T> w[R];
            stage_twiddles<T, R>(w, k * (N / (NS * R)), W);
#pragma unroll
            for (int r = 1; r < R; ++r) v[u * R + r] = SIGN > 0 ? cmul(v[u * R + r], w[r]) : cmulc(v[u * R + r], w[r]);
        }
        if constexpr (!ADJ) dft_any<T, SIGN, R>(v + u * R);
    }
}

// Moves values between the output places of stage (NS, R) and the input places of
// the next stage, radix R2; TO: from the former to the latter, else back.
template <typename T, int N, int TL, int NS, int R, int R2, bool TO>
__device__ __forceinline__ void any_exchange(c_t<T>* v, int t, c_t<T>* scr) {
    auto outputs = [&](auto&& f) {
#pragma unroll
        for (int u = 0; u < per_lane(N, TL, R); ++u) {
            const int j = t + TL * u, k = j % NS;
            if (!all_busy(N, TL, R) && j >= N / R) continue;
#pragma unroll
            for (int r = 0; r < R; ++r) f(v[u * R + r], scr[padx((j - k) * R + k + r * NS)]);
        }
    };
    auto inputs = [&](auto&& f) {
#pragma unroll
        for (int u = 0; u < per_lane(N, TL, R2); ++u) {
            const int j = t + TL * u;
            if (!all_busy(N, TL, R2) && j >= N / R2) continue;
#pragma unroll
            for (int r = 0; r < R2; ++r) f(v[u * R2 + r], scr[padx(j + r * (N / R2))]);
        }
    };
    auto store = [](c_t<T>& a, c_t<T>& s) { s = a; };
    auto load = [](c_t<T>& a, c_t<T>& s) { a = s; };
    __syncwarp();
    if constexpr (TO) outputs(store);
    else inputs(store);
    __syncwarp();
    if constexpr (TO) inputs(load);
    else outputs(load);
}

template <typename T, int N, int TL, int SIGN, int NS, int R, int... Rest>
struct AnyRunner {
    static __device__ __forceinline__ void run(c_t<T>* v, int t, c_t<T>* scr, const tw_t<T>* __restrict__ W) {
        any_stage<T, N, TL, SIGN, NS, R, false>(v, t, W);
        if constexpr (sizeof...(Rest) > 0) {
            any_exchange<T, N, TL, NS, R, FirstRadix<Rest...>::value, true>(v, t, scr);
            AnyRunner<T, N, TL, SIGN, NS * R, Rest...>::run(v, t, scr, W);
        }
    }
    // the adjoint flow graph, of sign SIGN
    static __device__ __forceinline__ void adjoint(c_t<T>* v, int t, c_t<T>* scr, const tw_t<T>* __restrict__ W) {
        if constexpr (sizeof...(Rest) > 0) {
            AnyRunner<T, N, TL, SIGN, NS * R, Rest...>::adjoint(v, t, scr, W);
            any_exchange<T, N, TL, NS, R, FirstRadix<Rest...>::value, false>(v, t, scr);
        }
        any_stage<T, N, TL, SIGN, NS, R, true>(v, t, W);
    }
};

template <int NS, int R, int... Rest>
struct LastStage {
    static constexpr int ns = LastStage<NS * R, Rest...>::ns, radix = LastStage<NS * R, Rest...>::radix;
};
template <int NS, int R>
struct LastStage<NS, R> {
    static constexpr int ns = NS, radix = R;
};
template <int N, int TL, int... R>
constexpr int any_values() {
    int e = 0;
    ((e = per_lane(N, TL, R) * R > e ? per_lane(N, TL, R) * R : e), ...);
    return e;
}

// run: from the input layout to the output layout, sign +1 or -1; adjoint: sign
// SIGN from the output layout back to the input layout.  Invalid values must be
// zero on entry of an FP64 transform (they take part in the line's scale).
template <typename T, int N, int TL_, int SP, class RadList>
struct AnyLine;
template <typename T, int N, int TL_, int SP, int R0, int... R>
struct AnyLine<T, N, TL_, SP, Rad<R0, R...>> {
    static constexpr int TL = TL_, LPW = 32 / TL, E = any_values<N, TL, R0, R...>(), SPACING = SP;
    static_assert(RadInfo<R0, R...>::prod == N, "radices must multiply to N");
    static constexpr int kRL = LastStage<1, R0, R...>::radix, kNSL = LastStage<1, R0, R...>::ns;
    static __device__ __forceinline__ bool in_valid(int t, int e) {
        return e / R0 < per_lane(N, TL, R0) && t + TL * (e / R0) < N / R0;
    }
    static __device__ __forceinline__ int in_index(int t, int e) { return t + TL * (e / R0) + (e % R0) * (N / R0); }
    static __device__ __forceinline__ bool out_valid(int t, int e) {
        return e / kRL < per_lane(N, TL, kRL) && t + TL * (e / kRL) < N / kRL;
    }
    static __device__ __forceinline__ int out_index(int t, int e) {
        const int j = t + TL * (e / kRL), k = j % kNSL;
        return (j - k) * kRL + k + (e % kRL) * kNSL;
    }
    template <int SIGN>
    static __device__ __forceinline__ void run(c_t<T>* v, int t, c_t<T>* scr, const c_t<T>* __restrict__ W) {
        if constexpr (std::is_same<T, double>::value) {
            longlong2 x[E];
            const FixScale sc = fix_line_in<E, TL>(v, x);
            AnyRunner<fix64, N, TL, SIGN, 1, R0, R...>::run(x, t, reinterpret_cast<longlong2*>(scr),
                                                            reinterpret_cast<const int4*>(W));
            fix_line_out<E>(x, v, sc);
        } else {
            AnyRunner<T, N, TL, SIGN, 1, R0, R...>::run(v, t, scr, W);
        }
    }
    template <int SIGN>
    static __device__ __forceinline__ void adjoint(c_t<T>* v, int t, c_t<T>* scr, const c_t<T>* __restrict__ W) {
        if constexpr (std::is_same<T, double>::value) {
            longlong2 x[E];
            const FixScale sc = fix_line_in<E, TL>(v, x);
            AnyRunner<fix64, N, TL, SIGN, 1, R0, R...>::adjoint(x, t, reinterpret_cast<longlong2*>(scr),
                                                                reinterpret_cast<const int4*>(W));
            fix_line_out<E>(x, v, sc);
        } else {
            AnyRunner<T, N, TL, SIGN, 1, R0, R...>::adjoint(v, t, scr, W);
        }
    }
};

// Per length: lanes, elements between the scratch lines of a warp (8-byte and
// 16-byte values) and radices.  Two stages where the factors allow, up to 16 values a
// lane (FP64: 64 registers of them), and as few idle lanes as that leaves; the
// spacings are those with the fewest shared-memory wavefronts over a transform's
// exchanges, counted access by access (128 values: half those of an odd spacing).
template <typename T, int N> struct AnyCfg;
#define JDFT_ANY(N_, TL_, SP8, SP16, ...)                                           \
    template <typename T>                                                           \
    struct AnyCfg<T, N_> {                                                          \
        static constexpr int TL = TL_;                                              \
        static constexpr int SPACING = std::is_same<T, double>::value ? SP16 : SP8; \
        using R = Rad<__VA_ARGS__>;                                                 \
        static_assert(SPACING >= padded_line(N_), "scratch lines must not overlap"); \
    };
JDFT_ANY(12, 4, 14, 13, 4, 3)
JDFT_ANY(16, 4, 18, 17, 4, 4)
JDFT_ANY(24, 6, 29, 29, 4, 6)
JDFT_ANY(25, 5, 39, 29, 5, 5)
JDFT_ANY(27, 3, 33, 29, 9, 3)
JDFT_ANY(30, 6, 45, 37, 5, 6)
JDFT_ANY(32, 4, 34, 35, 8, 4)
JDFT_ANY(36, 6, 41, 45, 6, 6)
JDFT_ANY(40, 5, 55, 43, 8, 5)
JDFT_ANY(45, 5, 55, 47, 9, 5)
JDFT_ANY(48, 8, 54, 54, 8, 6)
JDFT_ANY(50, 5, 55, 55, 10, 5)
JDFT_ANY(54, 6, 71, 61, 9, 6)
JDFT_ANY(60, 6, 77, 69, 10, 6)
JDFT_ANY(64, 8, 68, 70, 8, 8)
JDFT_ANY(72, 9, 76, 83, 9, 8)
JDFT_ANY(75, 5, 87, 81, 5, 5, 3)
JDFT_ANY(80, 10, 87, 86, 10, 8)
JDFT_ANY(81, 9, 91, 91, 9, 9)
JDFT_ANY(90, 10, 100, 99, 10, 9)
JDFT_ANY(96, 8, 103, 102, 4, 4, 6)
JDFT_ANY(100, 10, 108, 110, 10, 10)
JDFT_ANY(108, 9, 123, 115, 6, 6, 3)
JDFT_ANY(120, 8, 132, 130, 8, 5, 3)
JDFT_ANY(125, 9, 132, 139, 5, 5, 5)
JDFT_ANY(128, 8, 140, 140, 16, 8)
JDFT_ANY(256, 16, 280, 276, 16, 16)
#undef JDFT_ANY
// FP64: 16 lanes of 8 values in three stages, which leaves more warps an SM (see RegCfg)
template <>
struct AnyCfg<double, 128> {
    static constexpr int TL = 16, SPACING = 140;
    using R = Rad<8, 4, 4>;
};

template <typename T, int N>
using LineOf = AnyLine<T, N, AnyCfg<T, N>::TL, AnyCfg<T, N>::SPACING, typename AnyCfg<T, N>::R>;

}  // namespace jdft
