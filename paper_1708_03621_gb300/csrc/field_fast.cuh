// Full-box field transforms with register line FFTs (fft_line.cuh), for the
// axis lengths those are compiled for.
//
// What bounded the shared-memory Stockham passes: FP64 ones the FP64 pipe, FP32
// ones the issue of their index arithmetic, shared-memory round trips and block
// barriers (two to three passes a line, each read and written through shared
// memory with runtime divisions).  Here a warp takes 32 / TL lines, loads them
// straight into registers (a lane's values N / E lines' width apart: every
// 32-byte sector is used whole), transforms them with one or two exchanges
// through its own scratch and stores them; there is no block barrier.  FP64
// lines run in fixed point (fft_fix.cuh).
//
// The density and the potentials of the Hartree chain are real, so the chain
// keeps the half box m2 = 0 .. S2 / 2: a warp's line slots each take two real lines
// a, b along axis 2 as a + i b, and the halves' spectra come apart by symmetry
// (A_k = (Z_k + conj Z_-k) / 2, B_k = (Z_k - conj Z_-k) / 2i).  Every pass of the
// chain moves and transforms half of what the complex box takes.
//
// Measured on a 128^3 box: Kohn-Sham potential 898 -> 320 us (half of it the LDA
// epilogue: FP64 arithmetic per point, see field_lda.cuh); an FP32 conjugate-gradient
// iteration of the dielectric solve, its direction formed in the gradient pass and
// its sums finished by each launch's last block, 424 -> 193 us (two axis-1 passes 59
// -> 24 each, gradient and direction 91 -> 43, eps 86 -> 29, divergence 94 -> 44, update
// 44 -> 31), the solve 50 -> 23.6 ms.
#pragma once

#include "common.cuh"

namespace jdft {

// Lines of one axis: line l = o * inner + i starts at o * ostride + i * istride,
// its elements es apart.
struct LineGeom {
    int nlines, inner;
    int64_t ostride, istride, es;
};

// Cell data of the kernels that form G: columns b_d of B (row-major), box edges.
struct FieldCell {
    double B[9];
    int S[3];
};

// A conjugate-gradient direction formed on the way into the gradient pass:
// d <- K r + (*rz_new / *rz_old) d, K the Coulomb kernel.
template <typename T>
struct DirectionArgs {
    const c_t<T>* r;  // null: d as it is
    const double *rz_new, *rz_old;
};

// A sum over the blocks of a launch: each block's partial sum, the last block to
// finish adding them in block order into *out (deterministic) and resetting *count.
struct BlockSum {
    double* partial;
    unsigned* count;  // zero before the launch
    double* out;
};

// T = double or float, N = the transformed axis's length; `tw` is the basis's
// twiddle array of type T (all lengths), p the axis's plan.  Defined in
// field_fast_impl.cuh and instantiated per type and length in field_fast_*.cu.
template <typename T, int N>
struct FieldFast {
    // out = scale * transform of sign `sign` of in, `batch` boxes bstride apart
    static jdft_status axis(const char* name, int sign, const c_t<T>* in, c_t<T>* out, const LineGeom& g, T scale,
                            int batch, int64_t bstride, const c_t<T>* tw, const FftPlan& p, cudaStream_t st);
    // axis 0: Y_c = I_0 (i G_c X), c = 0, 1, 2, with X updated first if dir says so
    static jdft_status grad(c_t<T>* X, const DirectionArgs<T>& dir, c_t<T>* Y, const FieldCell& q, int64_t bstride, const c_t<T>* tw,
                            const FftPlan& p, cudaStream_t st);
    // axis 2 of three boxes: inverse, times eps, forward, in place
    static jdft_status eps(c_t<T>* Y, const T* eps, int nlines, int64_t bstride, const c_t<T>* tw, const FftPlan& p,
                           cudaStream_t st);
    // axis 0: out = scale sum_c i G_c F_0(Y_c); with din, sum = sum of Re conj(din) out
    static jdft_status div(const c_t<T>* Y, const c_t<T>* din, c_t<T>* out, const FieldCell& q, int64_t bstride,
                           double scale, const BlockSum& sum, const c_t<T>* tw, const FftPlan& p, cudaStream_t st);
};

// The Hartree chain's end passes (FP64, N = S2 or S0), on the half box of
// S0 x S1 x (S2 / 2 + 1) values.
template <int N>
struct HartreeFast {
    // axis 2: real box -> half box
    static jdft_status forward2(const double* n, double2* half, int nlines, const double2* tw, const FftPlan& p,
                                cudaStream_t st);
    // axis 0: forward, times the Coulomb kernel / N, inverse, in place; sum (unless its out is null) of
    // sum_scale K |n~|^2
    static jdft_status kernel0(double2* half, const FieldCell& q, const BlockSum& sum, double sum_scale,
                               const double2* tw, const FftPlan& p, cudaStream_t st);
    // axis 2: half box -> V (vion == nullptr), or vion + V + v_xc(n) with sum (unless its out is null) of
    // sum_scale n e_xc(n)
    static jdft_status inverse2(const double2* half, double* V, const double* n, const double* vion,
                                const BlockSum& sum, double sum_scale, int nlines, const double2* tw, const FftPlan& p,
                                cudaStream_t st);
};

}  // namespace jdft
