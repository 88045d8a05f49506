// Lane and shared-memory layout of the register line FFTs (fft_reg.cuh) per
// compiled length, shared by the plane and z passes and the field transforms.
#pragma once

#include <type_traits>

#include "fft_reg.cuh"

namespace jdft {

// i mod N in [0, N) for either sign of i: one bit mask when N is a power of
// two (two's complement), else a remainder and a correction.
template <int N>
__device__ __forceinline__ int wrapn(int i) {
    if constexpr ((N & (N - 1)) == 0) {
        return i & (N - 1);
    } else {
        const int r = i % N;
        return r < 0 ? r + N : r;
    }
}

// Shared-memory layout of the register-FFT kernels.  A warp's 8-byte shared
// access is served in two halves of 16 lanes and a 16-byte access in four
// quarters of 8 lanes; lanes of one group that hit different addresses in the
// same bank slot (16 eight-byte or 8 sixteen-byte slots per 128 bytes) cost
// one wavefront each.  The constants below are the ones with the fewest such
// conflicts over every shared access of these kernels, counted access by
// access (plane_layout.py beside this package prints them); the 128^3 FP32
// plane pass has none.
//
// Lanes: a line of N values is split over TL = N / E lanes and a warp serves
// LPW = 32 / TL lines; lane l takes position l / LPW of line l % LPW, so a
// half-warp covers several lines at once and several consecutive rows or
// columns of the plane array.
template <int N, int E>
struct Lanes {
    static constexpr int TL = N / E, LPW = 32 / TL;
    static __device__ __forceinline__ int line(int lane) { return lane % LPW; }
    static __device__ __forceinline__ int pos(int lane) { return lane / LPW; }
};

// Elements between the LPW scratch lines of one warp (each line needs
// padded_line(N)).
template <typename T, int N>
struct ScratchSpacing;
#define JDFT_SPACING_OF(T, N, SP)                                                           \
    template <>                                                                             \
    struct ScratchSpacing<T, N> {                                                           \
        static constexpr int value = SP;                                                    \
        static_assert(SP >= padded_line(N), "scratch lines of one warp must not overlap"); \
    };
JDFT_SPACING_OF(float, 12, 13)
JDFT_SPACING_OF(float, 16, 17)
JDFT_SPACING_OF(float, 40, 43)
JDFT_SPACING_OF(float, 48, 54)
JDFT_SPACING_OF(float, 64, 68)
JDFT_SPACING_OF(float, 80, 86)
JDFT_SPACING_OF(float, 128, 140)
JDFT_SPACING_OF(float, 256, 280)
JDFT_SPACING_OF(double, 12, 13)
JDFT_SPACING_OF(double, 16, 17)
JDFT_SPACING_OF(double, 40, 43)
JDFT_SPACING_OF(double, 48, 51)
JDFT_SPACING_OF(double, 64, 70)
JDFT_SPACING_OF(double, 80, 85)
JDFT_SPACING_OF(double, 128, 138)
JDFT_SPACING_OF(double, 256, 276)
#undef JDFT_SPACING_OF

// Line shapes per compiled length: E values per lane and the radix list.
template <int N> struct FastCfg;
template <> struct FastCfg<12> { static constexpr int E = 12; using R = Rad<4, 3>; };
template <> struct FastCfg<16> { static constexpr int E = 16; using R = Rad<16>; };
template <> struct FastCfg<40> { static constexpr int E = 20; using R = Rad<2, 4, 5>; };
template <> struct FastCfg<48> { static constexpr int E = 12; using R = Rad<4, 4, 3>; };
template <> struct FastCfg<64> { static constexpr int E = 8; using R = Rad<8, 8>; };
template <> struct FastCfg<80> { static constexpr int E = 20; using R = Rad<4, 4, 5>; };
template <> struct FastCfg<128> { static constexpr int E = 16; using R = Rad<16, 8>; };
template <> struct FastCfg<256> { static constexpr int E = 16; using R = Rad<16, 16>; };


// The shape a length's transform of type T uses.  FP64 lines of 128 values take 16
// lanes of 8 values in three stages: a lane's integers then fit 128 registers, so a
// plane block of 16 warps does (8 warps of 16-value lanes kept 1.5 instructions a
// clock in flight).
template <typename T, int N> struct RegCfg : FastCfg<N> {};
template <> struct RegCfg<double, 128> { static constexpr int E = 8; using R = Rad<8, 4, 4>; };

#define JDFT_FAST_LENGTHS(X) X(12) X(16) X(40) X(48) X(64) X(80) X(128) X(256)

// The table the register line FFTs of type T read: the fixed-point one for FP64.
template <typename T>
const c_t<T>* reg_table(const c_t<T>* tw_base, const FftPlan& p) {
    return tw_base + (std::is_same<T, double>::value ? p.fx_offset : p.tw_offset);
}

}  // namespace jdft
