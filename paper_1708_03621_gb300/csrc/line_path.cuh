// The chain of the Hamiltonian one line transform per launch, for boxes that no
// fused plane kernel is compiled for.
//
// What bounded the generic plane kernels on such boxes: FP64 ones the FP64 pipe,
// all of them the runtime index arithmetic, the shared-memory round trip of every
// radix pass and the block barriers between passes, with one block to a plane.  Here
// each axis is one launch of register line FFTs of compiled length (fft_line.cuh),
// every warp on its own lines: sphere columns along z, the sphere's rows along axis
// 1, columns along axis 0 with the potential between the inverse and forward
// transforms, and back.  The two intermediates keep z fastest,
//     col[b][c][j2]  (sphere columns),  row[b][r][j1][j2]  (sphere rows x axis 1),
// so that the lines of a warp are neighbours along z and every access of the axis-1
// and axis-0 passes covers whole sectors; so do the real-space boxes of I and J.
#pragma once

#include "chain.cuh"

namespace jdft {

// Geometry of a band chunk; tables as in ChainGeom.
struct LineArgs {
    int S0, S1, S2, ncols, nrows, i0min, i1min, nb;
    const int *col_start, *row_col_start, *row_i1lo, *pw_z;
};

template <typename T, int N>
struct LinePath {
    // C (sphere) -> col: axis 2, N = S2
    static jdft_status zinv(const LineArgs& g, const c_t<T>* C, int ldc, c_t<T>* col, const c_t<T>* tw, const FftPlan& p,
                            cudaStream_t st);
    // col -> out: forward along axis 2; kin != nullptr: out = omega (kin C + scale y), else out = scale y
    static jdft_status zfwd(const LineArgs& g, const c_t<T>* col, const c_t<T>* C, int ldc, c_t<T>* out, int ldo,
                            const T* kin, T omega, T scale, const c_t<T>* tw, const FftPlan& p, cudaStream_t st);
    // col -> row (sign +1) and row -> col (sign -1) along axis 1, N = S1
    static jdft_status rows(const LineArgs& g, int sign, c_t<T>* col, c_t<T>* row, const c_t<T>* tw, const FftPlan& p,
                            cudaStream_t st);
    // row -> row along axis 0, N = S0: inverse, times V (natural order), forward
    static jdft_status apply(const LineArgs& g, c_t<T>* row, const T* V, const c_t<T>* tw, const FftPlan& p,
                             cudaStream_t st);
    // row -> psi = scale * inverse, and psi -> row, along axis 0
    static jdft_status full(const LineArgs& g, int sign, c_t<T>* row, c_t<T>* psi, T scale, const c_t<T>* tw,
                            const FftPlan& p, cudaStream_t st);
    // n_r += w sum_b f_b |inverse along axis 0|^2
    static jdft_status density(const LineArgs& g, const c_t<T>* row, const double* f, double w, double* n_r,
                               const c_t<T>* tw, const FftPlan& p, cudaStream_t st);
};

#define JDFT_LINE_LENGTHS(X)                                                                                          \
    X(12) X(16) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64) X(72) X(75) X(80) X(81) \
        X(90) X(96) X(100) X(108) X(120) X(125) X(128) X(256)

inline bool line_length(int n) {
#define JDFT_CASE(N) \
    if (n == N) return true;
    JDFT_LINE_LENGTHS(JDFT_CASE)
#undef JDFT_CASE
    return false;
}

// Evaluates an expression in the constant N for the compiled length n
// (JDFT_ERR_UNSUPPORTED where there is none).
#define JDFT_LINE_CASE_(N_, ...)   \
    case N_: {                     \
        constexpr int N = N_;      \
        return __VA_ARGS__;        \
    }
#define JDFT_LINE_DISPATCH(n, ...)                                                                                   \
    [&]() -> jdft_status {                                                                                           \
        switch (n) {                                                                                                 \
            JDFT_LINE_CASE_(12, __VA_ARGS__) JDFT_LINE_CASE_(16, __VA_ARGS__) JDFT_LINE_CASE_(24, __VA_ARGS__)       \
            JDFT_LINE_CASE_(25, __VA_ARGS__) JDFT_LINE_CASE_(27, __VA_ARGS__) JDFT_LINE_CASE_(30, __VA_ARGS__)       \
            JDFT_LINE_CASE_(32, __VA_ARGS__) JDFT_LINE_CASE_(36, __VA_ARGS__) JDFT_LINE_CASE_(40, __VA_ARGS__)       \
            JDFT_LINE_CASE_(45, __VA_ARGS__) JDFT_LINE_CASE_(48, __VA_ARGS__) JDFT_LINE_CASE_(50, __VA_ARGS__)       \
            JDFT_LINE_CASE_(54, __VA_ARGS__) JDFT_LINE_CASE_(60, __VA_ARGS__) JDFT_LINE_CASE_(64, __VA_ARGS__)       \
            JDFT_LINE_CASE_(72, __VA_ARGS__) JDFT_LINE_CASE_(75, __VA_ARGS__) JDFT_LINE_CASE_(80, __VA_ARGS__)       \
            JDFT_LINE_CASE_(81, __VA_ARGS__) JDFT_LINE_CASE_(90, __VA_ARGS__) JDFT_LINE_CASE_(96, __VA_ARGS__)       \
            JDFT_LINE_CASE_(100, __VA_ARGS__) JDFT_LINE_CASE_(108, __VA_ARGS__) JDFT_LINE_CASE_(120, __VA_ARGS__)    \
            JDFT_LINE_CASE_(125, __VA_ARGS__) JDFT_LINE_CASE_(128, __VA_ARGS__) JDFT_LINE_CASE_(256, __VA_ARGS__)    \
        }                                                                                                            \
        return JDFT_ERR_UNSUPPORTED;                                                                                 \
    }()

}  // namespace jdft
