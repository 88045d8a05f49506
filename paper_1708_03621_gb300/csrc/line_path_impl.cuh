// Kernels and launchers of line_path.cuh, instantiated per length in line_path_*.cu.
#pragma once

#include <algorithm>

#include "fft_lanes.cuh"
#include "fft_line.cuh"
#include "line_path.cuh"
#include "profile.cuh"

namespace jdft {
namespace lp {

constexpr int kWarps = 4, kThreads = 32 * kWarps;

template <typename T, int N>
struct Ctx {
    using F = LineOf<T, N>;
    static constexpr int LPB = kWarps * F::LPW;  // lines per block
    static constexpr size_t SMEM = (N + (size_t)LPB * F::SPACING) * sizeof(c_t<T>);
    // position in the line (past N for idle lanes, whose values are all invalid), line of the block
    int t, line;
    c_t<T>*W, *scr;
    __device__ __forceinline__ Ctx(unsigned char* smem, const c_t<T>* __restrict__ tw) {
        W = reinterpret_cast<c_t<T>*>(smem);
        for (int i = threadIdx.x; i < N; i += kThreads) W[i] = tw[i];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        t = lane < F::TL * F::LPW ? lane / F::LPW : 2 * N;
        line = warp * F::LPW + lane % F::LPW;
        scr = W + N + line * F::SPACING;
        __syncthreads();
    }
};

template <typename T, int N>
__global__ void __launch_bounds__(kThreads)
    zinv_kernel(LineArgs g, const c_t<T>* __restrict__ C, int ldc, c_t<T>* __restrict__ col,
                const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using K = Ctx<T, N>;
    using F = typename K::F;
    K k(smem, tw);
    const int c = blockIdx.x * K::LPB + k.line, b = blockIdx.y;
    const bool act = c < g.ncols;
    int q0 = 0, cnt = 0, z0 = 0;
    if (act) {
        q0 = g.col_start[c];
        cnt = g.col_start[c + 1] - q0;
        z0 = g.pw_z[q0];
    }
    const c_t<T>* Cb = C + (size_t)b * ldc + q0;
    c_t<T> v[F::E];
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        const int off = wrapn<N>(F::in_index(k.t, e) - z0);
        v[e] = F::in_valid(k.t, e) && off < cnt ? Cb[off] : mk<T>(T(0), T(0));
    }
    F::template run<+1>(v, k.t, k.scr, k.W);
    if (act) {
        c_t<T>* o = col + ((size_t)b * g.ncols + c) * N;
#pragma unroll
        for (int e = 0; e < F::E; ++e)
            if (F::out_valid(k.t, e)) o[F::out_index(k.t, e)] = v[e];
    }
}

template <typename T, int N>
__global__ void __launch_bounds__(kThreads)
    zfwd_kernel(LineArgs g, const c_t<T>* __restrict__ col, const c_t<T>* __restrict__ C, int ldc,
                c_t<T>* __restrict__ out, int ldo, const T* __restrict__ kin, T omega, T scale,
                const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using K = Ctx<T, N>;
    using F = typename K::F;
    K k(smem, tw);
    const int c = blockIdx.x * K::LPB + k.line, b = blockIdx.y;
    const bool act = c < g.ncols;
    const c_t<T>* in = col + ((size_t)b * g.ncols + (act ? c : 0)) * N;
    c_t<T> v[F::E];
#pragma unroll
    for (int e = 0; e < F::E; ++e)
        v[e] = act && F::in_valid(k.t, e) ? in[F::in_index(k.t, e)] : mk<T>(T(0), T(0));
    F::template run<-1>(v, k.t, k.scr, k.W);
    if (!act) return;
    const int q0 = g.col_start[c], cnt = g.col_start[c + 1] - q0, z0 = g.pw_z[q0];
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        const int off = wrapn<N>(F::out_index(k.t, e) - z0);
        if (!F::out_valid(k.t, e) || off >= cnt) continue;
        const int q = q0 + off;
        c_t<T> r;
        if (kin) {
            const c_t<T> cq = C[(size_t)b * ldc + q];
            const T kq = kin[q];
            r = mk<T>(omega * (kq * cq.x + scale * v[e].x), omega * (kq * cq.y + scale * v[e].y));
        } else {
            r = mk<T>(scale * v[e].x, scale * v[e].y);
        }
        out[(size_t)b * ldo + q] = r;
    }
}

// Lines (r, j2), j2 fastest, blockIdx.y = band.
template <typename T, int N, int SIGN>
__global__ void __launch_bounds__(kThreads)
    rows_kernel(LineArgs g, c_t<T>* __restrict__ col, c_t<T>* __restrict__ row, const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using K = Ctx<T, N>;
    using F = typename K::F;
    K k(smem, tw);
    const int l = blockIdx.x * K::LPB + k.line, b = blockIdx.y;
    const bool act = l < g.nrows * g.S2;
    const int r = act ? l / g.S2 : 0, j2 = act ? l - r * g.S2 : 0;
    const int cs = g.row_col_start[r], cnt = g.row_col_start[r + 1] - cs, lo = g.row_i1lo[r];
    c_t<T>* cp = col + ((size_t)b * g.ncols + cs) * g.S2 + j2;
    c_t<T>* rp = row + (((size_t)b * g.nrows + r) * N) * g.S2 + j2;
    c_t<T> v[F::E];
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        const int i = F::in_index(k.t, e);
        v[e] = mk<T>(T(0), T(0));
        if (act && F::in_valid(k.t, e)) {
            if constexpr (SIGN > 0) {
                const int off = wrapn<N>(i - lo);
                if (off < cnt) v[e] = cp[(size_t)off * g.S2];
            } else {
                v[e] = rp[(size_t)i * g.S2];
            }
        }
    }
    F::template run<SIGN>(v, k.t, k.scr, k.W);
    if (!act) return;
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        if (!F::out_valid(k.t, e)) continue;
        const int i = F::out_index(k.t, e);
        if constexpr (SIGN > 0) {
            rp[(size_t)i * g.S2] = v[e];
        } else {
            const int off = wrapn<N>(i - lo);
            if (off < cnt) cp[(size_t)off * g.S2] = v[e];
        }
    }
}

// Lines (j1, j2), j2 fastest: element r of a line at row[(b nrows + r) S1 S2 + l].
template <typename T, int N, class F>
__device__ __forceinline__ void load_rows(const LineArgs& g, const c_t<T>* rp, int ps, bool act, int t, c_t<T>* v) {
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        const int r = wrapn<N>(F::in_index(t, e) - g.i0min);
        v[e] = act && F::in_valid(t, e) && r < g.nrows ? rp[(size_t)r * ps] : mk<T>(T(0), T(0));
    }
}

template <typename T, int N>
__global__ void __launch_bounds__(kThreads, 3)
    apply_kernel(LineArgs g, c_t<T>* __restrict__ row, const T* __restrict__ V, const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using K = Ctx<T, N>;
    using F = typename K::F;
    K k(smem, tw);
    const int ps = g.S1 * g.S2, l = blockIdx.x * K::LPB + k.line, b = blockIdx.y;
    const bool act = l < ps;
    c_t<T>* rp = row + (size_t)b * g.nrows * ps + l;
    c_t<T> v[F::E];
    load_rows<T, N, F>(g, rp, ps, act, k.t, v);
    F::template run<+1>(v, k.t, k.scr, k.W);
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        if (act && F::out_valid(k.t, e)) {
            const T s = V[(size_t)F::out_index(k.t, e) * ps + l];
            v[e].x *= s;
            v[e].y *= s;
        } else {
            v[e] = mk<T>(T(0), T(0));
        }
    }
    F::template adjoint<-1>(v, k.t, k.scr, k.W);
    if (!act) return;
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        const int r = wrapn<N>(F::in_index(k.t, e) - g.i0min);
        if (F::in_valid(k.t, e) && r < g.nrows) rp[(size_t)r * ps] = v[e];
    }
}

template <typename T, int N, int SIGN>
__global__ void __launch_bounds__(kThreads)
    full_kernel(LineArgs g, c_t<T>* __restrict__ row, c_t<T>* __restrict__ psi, T scale,
                const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using K = Ctx<T, N>;
    using F = typename K::F;
    K k(smem, tw);
    const int ps = g.S1 * g.S2, l = blockIdx.x * K::LPB + k.line, b = blockIdx.y;
    const bool act = l < ps;
    c_t<T>* rp = row + (size_t)b * g.nrows * ps + l;
    c_t<T>* pp = psi + (size_t)b * N * ps + l;
    c_t<T> v[F::E];
    if constexpr (SIGN > 0) {
        load_rows<T, N, F>(g, rp, ps, act, k.t, v);
    } else {
#pragma unroll
        for (int e = 0; e < F::E; ++e)
            v[e] = act && F::in_valid(k.t, e) ? pp[(size_t)F::in_index(k.t, e) * ps] : mk<T>(T(0), T(0));
    }
    F::template run<SIGN>(v, k.t, k.scr, k.W);
    if (!act) return;
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        if (!F::out_valid(k.t, e)) continue;
        const int j = F::out_index(k.t, e);
        if constexpr (SIGN > 0) {
            pp[(size_t)j * ps] = mk<T>(scale * v[e].x, scale * v[e].y);
        } else {
            const int r = wrapn<N>(j - g.i0min);
            if (r < g.nrows) rp[(size_t)r * ps] = v[e];
        }
    }
}

template <typename T, int N>
__global__ void __launch_bounds__(kThreads, 3)
    density_kernel(LineArgs g, const c_t<T>* __restrict__ row, int per, const double* __restrict__ f, double w,
                   double* __restrict__ n_r, const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using K = Ctx<T, N>;
    using F = typename K::F;
    K k(smem, tw);
    const int ps = g.S1 * g.S2, l = blockIdx.x * K::LPB + k.line;
    const bool act = l < ps;
    double acc[F::E];
#pragma unroll
    for (int e = 0; e < F::E; ++e) acc[e] = 0.0;
    const int bA = blockIdx.y * per, bB = min(g.nb, bA + per);
#pragma unroll 1
    for (int b = bA; b < bB; ++b) {
        const double fb = f[b];
        c_t<T> v[F::E];
        load_rows<T, N, F>(g, row + (size_t)b * g.nrows * ps + l, ps, act, k.t, v);
        F::template run<+1>(v, k.t, k.scr, k.W);
#pragma unroll
        for (int e = 0; e < F::E; ++e)
            acc[e] += fb * ((double)v[e].x * (double)v[e].x + (double)v[e].y * (double)v[e].y);
        __syncwarp();
    }
    if (!act) return;
    const bool atomic = gridDim.y > 1;
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        if (!F::out_valid(k.t, e)) continue;
        double* d = n_r + (size_t)F::out_index(k.t, e) * ps + l;
        if (atomic) atomicAdd(d, w * acc[e]);
        else *d += w * acc[e];
    }
}

template <typename T, int N, typename Kern, typename... A>
static jdft_status launch(const char* name, Kern kern, int lines, int batch, cudaStream_t st, A... args) {
    using K = Ctx<T, N>;
    cudaError_t e = set_smem_attr((const void*)kern, K::SMEM);
    if (e != cudaSuccess) return set_error(JDFT_ERR_CUDA, std::string(name) + ": " + cudaGetErrorString(e));
    {
        Trace tr_(name, st);
        kern<<<dim3((lines + K::LPB - 1) / K::LPB, batch), kThreads, K::SMEM, st>>>(args...);
    }
    return check_launch(name);
}

}  // namespace lp

template <typename T, int N>
jdft_status LinePath<T, N>::zinv(const LineArgs& g, const c_t<T>* C, int ldc, c_t<T>* col, const c_t<T>* tw,
                                 const FftPlan& p, cudaStream_t st) {
    return lp::launch<T, N>("line_z_inverse", lp::zinv_kernel<T, N>, g.ncols, g.nb, st, g, C, ldc, col,
                            reg_table<T>(tw, p));
}
template <typename T, int N>
jdft_status LinePath<T, N>::zfwd(const LineArgs& g, const c_t<T>* col, const c_t<T>* C, int ldc, c_t<T>* out, int ldo,
                                 const T* kin, T omega, T scale, const c_t<T>* tw, const FftPlan& p, cudaStream_t st) {
    return lp::launch<T, N>("line_z_forward", lp::zfwd_kernel<T, N>, g.ncols, g.nb, st, g, col, C, ldc, out, ldo, kin,
                            omega, scale, reg_table<T>(tw, p));
}
template <typename T, int N>
jdft_status LinePath<T, N>::rows(const LineArgs& g, int sign, c_t<T>* col, c_t<T>* row, const c_t<T>* tw,
                                 const FftPlan& p, cudaStream_t st) {
    const c_t<T>* t = reg_table<T>(tw, p);
    return sign > 0 ? lp::launch<T, N>("line_rows_inverse", lp::rows_kernel<T, N, +1>, g.nrows * g.S2, g.nb, st, g, col,
                                       row, t)
                    : lp::launch<T, N>("line_rows_forward", lp::rows_kernel<T, N, -1>, g.nrows * g.S2, g.nb, st, g, col,
                                       row, t);
}
template <typename T, int N>
jdft_status LinePath<T, N>::apply(const LineArgs& g, c_t<T>* row, const T* V, const c_t<T>* tw, const FftPlan& p,
                                  cudaStream_t st) {
    return lp::launch<T, N>("line_columns", lp::apply_kernel<T, N>, g.S1 * g.S2, g.nb, st, g, row, V,
                            reg_table<T>(tw, p));
}
template <typename T, int N>
jdft_status LinePath<T, N>::full(const LineArgs& g, int sign, c_t<T>* row, c_t<T>* psi, T scale, const c_t<T>* tw,
                                 const FftPlan& p, cudaStream_t st) {
    const c_t<T>* t = reg_table<T>(tw, p);
    return sign > 0 ? lp::launch<T, N>("line_box_inverse", lp::full_kernel<T, N, +1>, g.S1 * g.S2, g.nb, st, g, row,
                                       psi, scale, t)
                    : lp::launch<T, N>("line_box_forward", lp::full_kernel<T, N, -1>, g.S1 * g.S2, g.nb, st, g, row,
                                       psi, scale, t);
}
template <typename T, int N>
jdft_status LinePath<T, N>::density(const LineArgs& g, const c_t<T>* row, const double* f, double w, double* n_r,
                                    const c_t<T>* tw, const FftPlan& p, cudaStream_t st) {
    // band groups so that the grid covers the GPU a few times
    const int blocks = (g.S1 * g.S2 + lp::Ctx<T, N>::LPB - 1) / lp::Ctx<T, N>::LPB;
    int groups = std::max(1, std::min(g.nb, (152 * 8 + blocks - 1) / blocks));
    const int per = (g.nb + groups - 1) / groups;
    groups = (g.nb + per - 1) / per;
    return lp::launch<T, N>("line_density", lp::density_kernel<T, N>, g.S1 * g.S2, groups, st, g, row, per, f, w, n_r,
                            reg_table<T>(tw, p));
}

}  // namespace jdft
