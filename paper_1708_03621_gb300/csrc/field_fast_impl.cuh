// Kernels and launchers of field_fast.cuh; included by the field_fast_*.cu
// translation units, which instantiate them per type and length.
#pragma once

#include "block_sum.cuh"
#include "fft_lanes.cuh"
#include "fft_line.cuh"
#include "field_fast.cuh"
#include "field_lda.cuh"
#include "profile.cuh"

namespace jdft {
namespace ff {

// Warps per block: the transforms need no block barrier, so small blocks, as
// many per SM as registers and scratch allow, leave the shortest last wave.
template <typename T>
constexpr int kWarps = std::is_same<T, double>::value ? 4 : 8;
constexpr double kFourPi = 12.566370614359172953850573533118;  // and what it is short of 4 pi
constexpr double kFourPiLo = 4.8985871965894128e-16;

__device__ __forceinline__ int fold(int m, int S) { return m < (S + 1) / 2 ? m : m - S; }

template <typename T, int N>
struct Line {
    using F = LineOf<T, N>;
    static constexpr int E = F::E, TL = F::TL;
    static constexpr int THREADS = 32 * kWarps<T>;
    static constexpr int LPB = kWarps<T> * F::LPW;  // lines per block
    static constexpr size_t SMEM = (N + (size_t)LPB * F::SPACING) * sizeof(c_t<T>);
    // this thread's position in its line (past N for idle lanes, whose values are all invalid), its line
    // within the block, the table and the line's scratch
    int t, line;
    const c_t<T>* W;
    c_t<T>* scr;
    __device__ __forceinline__ Line(unsigned char* smem, const c_t<T>* __restrict__ tw) {
        c_t<T>* w = reinterpret_cast<c_t<T>*>(smem);
        for (int i = threadIdx.x; i < N; i += THREADS) w[i] = tw[i];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        t = lane < TL * F::LPW ? lane / F::LPW : 2 * N;
        line = warp * F::LPW + lane % F::LPW;
        scr = w + N + line * F::SPACING;
        W = w;
        __syncthreads();
    }
};

// The forward transform is the inverse one with real and imaginary parts swapped on
// both sides: one compiled transform serves both signs.
template <typename T, int N>
__global__ void __launch_bounds__(Line<T, N>::THREADS)
    axis_kernel(const c_t<T>* in, c_t<T>* out, LineGeom g, int forward, T scale, int64_t bstride,
                const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using L = Line<T, N>;
    using F = typename L::F;
    L ln(smem, tw);
    const int l = blockIdx.x * L::LPB + ln.line;
    const bool act = l < g.nlines;
    const int o = l / g.inner, i = l - o * g.inner;
    const int64_t base = blockIdx.y * bstride + o * g.ostride + i * g.istride;
    c_t<T> v[L::E];
#pragma unroll
    for (int e = 0; e < L::E; ++e) {
        v[e] = mk<T>(T(0), T(0));
        if (act && F::in_valid(ln.t, e)) {
            const c_t<T> x = in[base + F::in_index(ln.t, e) * g.es];
            v[e] = forward ? mk<T>(x.y, x.x) : x;
        }
    }
    F::template run<+1>(v, ln.t, ln.scr, ln.W);
    if (!act) return;
#pragma unroll
    for (int e = 0; e < L::E; ++e) {
        if (!F::out_valid(ln.t, e)) continue;
        const c_t<T> y = forward ? mk<T>(v[e].y, v[e].x) : v[e];
        out[base + F::out_index(ln.t, e) * g.es] = mk<T>(scale * y.x, scale * y.y);
    }
}

// G of a line of axis 0 (its parts from axes 1 and 2).
template <typename T>
__device__ __forceinline__ void line_G(const FieldCell& q, int l, int S2, T* G) {
    const int m1 = l / S2, m2 = l - m1 * S2;
    const double f1 = fold(m1, q.S[1]), f2 = fold(m2, q.S[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) G[c] = (T)(f1 * q.B[3 * c + 1] + f2 * q.B[3 * c + 2]);
}

template <typename T, int N>
__global__ void __launch_bounds__(Line<T, N>::THREADS)
    grad_kernel(c_t<T>* X, DirectionArgs<T> dir, c_t<T>* __restrict__ Y, FieldCell q, int64_t bstride,
                const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using L = Line<T, N>;
    using F = typename L::F;
    L ln(smem, tw);
    const int es = q.S[1] * q.S[2];
    const int l = blockIdx.x * L::LPB + ln.line;
    const bool act = l < es;
    T G[3];
    line_G<T>(q, act ? l : 0, q.S[2], G);
    // The direction (saves a launch and a pass over d): each lane updates the values it reads below, in
    // groups whose loads are all in flight before the first store.
    if (dir.r && act) {
        const T beta = (T)(*dir.rz_new / *dir.rz_old);
        constexpr int GR = L::E % 8 == 0 ? 8 : L::E % 6 == 0 ? 6 : L::E % 5 == 0 ? 5 : L::E % 3 == 0 ? 3 : 1;
#pragma unroll
        for (int e0 = 0; e0 < L::E; e0 += GR) {
            c_t<T> r[GR], d[GR];
#pragma unroll
            for (int i = 0; i < GR; ++i) {
                r[i] = d[i] = mk<T>(T(0), T(0));
                if (F::in_valid(ln.t, e0 + i)) {
                    const int64_t a = l + (int64_t)F::in_index(ln.t, e0 + i) * es;
                    r[i] = dir.r[a];
                    d[i] = X[a];
                }
            }
#pragma unroll
            for (int i = 0; i < GR; ++i) {
                if (!F::in_valid(ln.t, e0 + i)) continue;
                const int j = F::in_index(ln.t, e0 + i);
                const T f0 = (T)fold(j, N);
                const T gx = f0 * (T)q.B[0] + G[0], gy = f0 * (T)q.B[3] + G[1], gz = f0 * (T)q.B[6] + G[2];
                const T g2 = gx * gx + gy * gy + gz * gz;
                const T K = g2 > (T)0 ? (T)kFourPi / g2 : (T)0;
                X[l + (int64_t)j * es] = mk<T>(K * r[i].x + beta * d[i].x, K * r[i].y + beta * d[i].y);
            }
        }
    }
    // X is read again for each component: it stays in L1, and the registers go to the transform
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
        const T b0 = (T)q.B[3 * c], g0 = c == 0 ? G[0] : c == 1 ? G[1] : G[2];
        c_t<T> v[L::E];
#pragma unroll
        for (int e = 0; e < L::E; ++e) {
            const int j = F::in_index(ln.t, e);
            const c_t<T> x = act && F::in_valid(ln.t, e) ? X[l + (int64_t)j * es] : mk<T>(T(0), T(0));
            const T Gc = (T)fold(j, N) * b0 + g0;
            v[e] = mk<T>(-Gc * x.y, Gc * x.x);
        }
        F::template run<+1>(v, ln.t, ln.scr, ln.W);
        if (act) {
            c_t<T>* Yc = Y + c * bstride + l;
#pragma unroll
            for (int e = 0; e < L::E; ++e)
                if (F::out_valid(ln.t, e)) Yc[(int64_t)F::out_index(ln.t, e) * es] = v[e];
        }
        __syncwarp();
    }
}

template <typename T, int N>
__global__ void __launch_bounds__(Line<T, N>::THREADS)
    eps_kernel(c_t<T>* __restrict__ Y, const T* __restrict__ eps, int nlines, int64_t bstride,
               const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using L = Line<T, N>;
    using F = typename L::F;
    L ln(smem, tw);
    const int l = blockIdx.x * L::LPB + ln.line;
    const bool act = l < nlines;
    c_t<T>* y = Y + blockIdx.y * bstride + (int64_t)l * N;
    c_t<T> v[L::E];
#pragma unroll
    for (int e = 0; e < L::E; ++e)
        v[e] = act && F::in_valid(ln.t, e) ? y[F::in_index(ln.t, e)] : mk<T>(T(0), T(0));
    F::template run<+1>(v, ln.t, ln.scr, ln.W);
    const T* el = eps + (int64_t)(act ? l : 0) * N;
#pragma unroll
    for (int e = 0; e < L::E; ++e) {
        const T s = F::out_valid(ln.t, e) ? el[F::out_index(ln.t, e)] : T(0);
        // invalid slots hold leftovers of the earlier stages: zero, not a product, since they may not be finite
        v[e] = F::out_valid(ln.t, e) ? mk<T>(s * v[e].x, s * v[e].y) : mk<T>(T(0), T(0));
    }
    // the forward transform as the inverse's adjoint: from the layout the inverse left to the one it read
    F::template adjoint<-1>(v, ln.t, ln.scr, ln.W);
    if (act) {
#pragma unroll
        for (int e = 0; e < L::E; ++e)
            if (F::in_valid(ln.t, e)) y[F::in_index(ln.t, e)] = v[e];
    }
}

template <typename T, int N>
__global__ void __launch_bounds__(Line<T, N>::THREADS)
    div_kernel(const c_t<T>* __restrict__ Y, const c_t<T>* __restrict__ din, c_t<T>* __restrict__ out, FieldCell q,
               int64_t bstride, double scale, BlockSum sum, const c_t<T>* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using L = Line<T, N>;
    using F = typename L::F;
    L ln(smem, tw);
    const int es = q.S[1] * q.S[2];
    const int l = blockIdx.x * L::LPB + ln.line;
    const bool act = l < es;
    T G[3];
    line_G<T>(q, act ? l : 0, q.S[2], G);
    c_t<T> acc[L::E];
#pragma unroll
    for (int e = 0; e < L::E; ++e) acc[e] = mk<T>(T(0), T(0));
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
        const T b0 = (T)q.B[3 * c], g0 = c == 0 ? G[0] : c == 1 ? G[1] : G[2];
        const c_t<T>* Yc = Y + c * bstride + l;
        c_t<T> v[L::E];
#pragma unroll
        for (int e = 0; e < L::E; ++e)
            v[e] = act && F::in_valid(ln.t, e) ? Yc[(int64_t)F::in_index(ln.t, e) * es] : mk<T>(T(0), T(0));
        F::template run<-1>(v, ln.t, ln.scr, ln.W);
#pragma unroll
        for (int e = 0; e < L::E; ++e) {
            const T Gc = (T)fold(F::out_index(ln.t, e), N) * b0 + g0;
            acc[e].x -= Gc * v[e].y;
            acc[e].y += Gc * v[e].x;
        }
        __syncwarp();
    }
    RunningSum<T> part;
    const T sc = (T)scale;
    if (act) {
#pragma unroll
        for (int e = 0; e < L::E; ++e) {
            if (!F::out_valid(ln.t, e)) continue;
            const int64_t a = l + (int64_t)F::out_index(ln.t, e) * es;
            const c_t<T> r = mk<T>(sc * acc[e].x, sc * acc[e].y);
            out[a] = r;
            if (din) {
                const c_t<T> d = din[a];
                part.add(d.x * r.x + d.y * r.y);
            }
        }
    }
    const double total = part.total();
    if (din) finish_sum<1, L::THREADS>(&total, sum, 1.0);
}

// ---- the Hartree chain on the half box -----------------------------------------
// Line slot p holds the real lines a = 2 p and b = 2 p + 1 as a + i b.
template <int N>
__global__ void __launch_bounds__(Line<double, N>::THREADS)
    hartree_forward2_kernel(const double* __restrict__ n, double2* __restrict__ half, int nlines,
                            const double2* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using L = Line<double, N>;
    using F = typename L::F;
    constexpr int H = N / 2 + 1;
    L ln(smem, tw);
    const int a = 2 * (blockIdx.x * L::LPB + ln.line);
    const bool actA = a < nlines, actB = a + 1 < nlines;
    const double* na = n + (int64_t)a * N;
    double2 v[L::E];
#pragma unroll
    for (int e = 0; e < L::E; ++e) {
        const int j = F::in_index(ln.t, e);
        const bool ok = F::in_valid(ln.t, e);
        v[e] = make_double2(actA && ok ? na[j] : 0.0, actB && ok ? na[N + j] : 0.0);
    }
    F::template run<-1>(v, ln.t, ln.scr, ln.W);
    __syncwarp();
#pragma unroll
    for (int e = 0; e < L::E; ++e)
        if (F::out_valid(ln.t, e)) ln.scr[padx(F::out_index(ln.t, e))] = v[e];
    __syncwarp();
    double2* ha = half + (int64_t)a * H;
    for (int k = ln.t; k < H; k += L::TL) {
        const double2 z = ln.scr[padx(k)], w = ln.scr[padx(k == 0 ? 0 : N - k)];
        if (actA) ha[k] = make_double2(0.5 * (z.x + w.x), 0.5 * (z.y - w.y));
        if (actB) ha[H + k] = make_double2(0.5 * (z.y + w.y), 0.5 * (w.x - z.x));
    }
}

// c / |G|^2 (0 at G = 0): the FP32 reciprocal, one Newton step, the product with c and
// that product's own residual, so that the result is rounded once (a factor rounded
// twice, or c's own rounding, biases every coefficient of a shell alike); half the
// FP64 instructions of a division where it is in range.  Against long double the
// Kohn-Sham potential of a 128^3 box is off by 1.4e-16 of its norm (2.6e-16 with a
// division and FP64 transforms).
struct Coulomb {
    double hi, lo;  // c
};
static __device__ __noinline__ double coulomb_plain(double c, double g2) { return g2 > 0.0 ? c / g2 : 0.0; }
__device__ __forceinline__ double coulomb_of(Coulomb c, double g2) {
    if (!(g2 > 1e-30 && g2 < 1e30)) return coulomb_plain(c.hi, g2);
    double r = long_of(__fdividef(1.0f, short_of(g2)));
    r = fma(fma(-g2, r, 1.0), r, r);
    const double k = c.hi * r;
    return fma(fma(-g2, k, c.hi) + c.lo, r, k);
}
__device__ __forceinline__ double norm2(const FieldCell& q, double f0, double lx, double ly, double lz) {
    const double x = fma(f0, q.B[0], lx), y = fma(f0, q.B[3], ly), z = fma(f0, q.B[6], lz);
    return fma(x, x, fma(y, y, z * z));
}

// c = 4 pi / N of the box's N points.
template <int N>
__global__ void __launch_bounds__(Line<double, N>::THREADS)
    hartree_kernel0_kernel(double2* __restrict__ half, FieldCell q, Coulomb c, BlockSum sum, double sum_scale,
                           const double2* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using L = Line<double, N>;
    using F = typename L::F;
    L ln(smem, tw);
    const int H = q.S[2] / 2 + 1, es = q.S[1] * H;
    const int l = blockIdx.x * L::LPB + ln.line;
    const bool act = l < es;
    const int m1 = act ? l / H : 0, m2 = act ? l - m1 * H : 0;
    double2 v[L::E];
#pragma unroll
    for (int e = 0; e < L::E; ++e)
        v[e] = act && F::in_valid(ln.t, e) ? half[l + (int64_t)F::in_index(ln.t, e) * es] : make_double2(0.0, 0.0);
    F::template run<-1>(v, ln.t, ln.scr, ln.W);
    double G[3], Gm[3];
    line_G<double>(q, m1 * q.S[2] + m2, q.S[2], G);
    // the mirror slot -m of the full box: a Nyquist index folds to -S/2 on both sides, so on
    // those slots the mirror's |G|^2 differs in skewed cells; the real potential sees the mean
    const bool ny1 = 2 * m1 == q.S[1], ny2 = 2 * m2 == q.S[2];
    line_G<double>(q, (ny1 ? m1 : m1 == 0 ? 0 : q.S[1] - m1) * q.S[2] + (ny2 ? m2 : m2 == 0 ? 0 : q.S[2] - m2), q.S[2],
                   Gm);
    double part = 0.0;
#pragma unroll
    for (int e = 0; e < L::E; ++e) {
        if (!F::out_valid(ln.t, e)) {
            v[e] = make_double2(0.0, 0.0);
            continue;
        }
        const int t = F::out_index(ln.t, e);
        double K = coulomb_of(c, norm2(q, (double)fold(t, N), G[0], G[1], G[2]));
        if (ny1 || ny2 || 2 * t == N) {
            const int tm = 2 * t == N || t == 0 ? t : N - t;
            K = 0.5 * (K + coulomb_of(c, norm2(q, (double)fold(tm, N), Gm[0], Gm[1], Gm[2])));
        }
        part = fma(K, fma(v[e].x, v[e].x, v[e].y * v[e].y), part);
        v[e].x *= K;
        v[e].y *= K;
    }
    // slots with 0 < m2 < S2/2 stand for their mirrors too
    part *= m2 == 0 || ny2 ? 1.0 : 2.0;
    F::template adjoint<+1>(v, ln.t, ln.scr, ln.W);
    if (act) {
#pragma unroll
        for (int e = 0; e < L::E; ++e)
            if (F::in_valid(ln.t, e)) half[l + (int64_t)F::in_index(ln.t, e) * es] = v[e];
    }
    if (!act) part = 0.0;
    if (sum.out) finish_sum<1, L::THREADS>(&part, sum, sum_scale);
}

template <int N, bool KS>
__global__ void __launch_bounds__(Line<double, N>::THREADS)
    hartree_inverse2_kernel(const double2* __restrict__ half, double* __restrict__ V, const double* __restrict__ n,
                            const double* __restrict__ vion, BlockSum sum, double sum_scale, int nlines,
                            const double2* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem[];
    using L = Line<double, N>;
    using F = typename L::F;
    constexpr int H = N / 2 + 1;
    L ln(smem, tw);
    const int a = 2 * (blockIdx.x * L::LPB + ln.line);
    const bool actA = a < nlines, actB = a + 1 < nlines;
    const double2* ha = half + (int64_t)a * H;
    double2 v[L::E];
#pragma unroll
    for (int e = 0; e < L::E; ++e) {
        const int j = F::in_index(ln.t, e), k = 2 * j <= N ? j : N - j;
        const bool ok = F::in_valid(ln.t, e);
        double2 A = actA && ok ? ha[k] : make_double2(0.0, 0.0), B = actB && ok ? ha[H + k] : make_double2(0.0, 0.0);
        if (k == 0 || 2 * k == N) A.y = B.y = 0.0;  // real for real lines
        v[e] = 2 * j <= N ? make_double2(A.x - B.y, A.y + B.x) : make_double2(A.x + B.y, B.x - A.y);
    }
    F::template run<+1>(v, ln.t, ln.scr, ln.W);
    double part = 0.0;
#pragma unroll
    for (int e = 0; e < L::E; ++e) {
        if (!F::out_valid(ln.t, e)) continue;
        const int64_t j = (int64_t)a * N + F::out_index(ln.t, e);
        if constexpr (KS) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 0 ? actA : actB) {
                    const int64_t i = j + h * N;
                    const double nj = n[i];
                    double ee, vx;
                    lda_pz(nj, ee, vx);
                    V[i] = vion[i] + (h ? v[e].y : v[e].x) + vx;
                    part = fma(nj, ee, part);
                }
            }
        } else {
            if (actA) V[j] = v[e].x;
            if (actB) V[j + N] = v[e].y;
        }
    }
    if constexpr (KS) {
        if (sum.out) finish_sum<1, L::THREADS>(&part, sum, sum_scale);
    }
}

template <typename T, int N, typename K, typename... A>
static jdft_status launch(const char* name, K kern, int lines, int batch, cudaStream_t st, A... args) {
    using L = Line<T, N>;
    cudaError_t e = set_smem_attr((const void*)kern, L::SMEM);
    if (e != cudaSuccess) return set_error(JDFT_ERR_CUDA, std::string(name) + ": " + cudaGetErrorString(e));
    {
        Trace tr_(name, st);
        kern<<<dim3((lines + L::LPB - 1) / L::LPB, batch), L::THREADS, L::SMEM, st>>>(args...);
    }
    return check_launch(name);
}

}  // namespace ff

template <typename T, int N>
jdft_status FieldFast<T, N>::axis(const char* name, int sign, const c_t<T>* in, c_t<T>* out, const LineGeom& g, T scale,
                                  int batch, int64_t bstride, const c_t<T>* tw, const FftPlan& p, cudaStream_t st) {
    const c_t<T>* t = reg_table<T>(tw, p);
    return ff::launch<T, N>(name, ff::axis_kernel<T, N>, g.nlines, batch, st, in, out, g, sign < 0 ? 1 : 0, scale,
                            bstride, t);
}
template <typename T, int N>
jdft_status FieldFast<T, N>::grad(c_t<T>* X, const DirectionArgs<T>& dir, c_t<T>* Y, const FieldCell& q,
                                  int64_t bstride, const c_t<T>* tw, const FftPlan& p, cudaStream_t st) {
    return ff::launch<T, N>("pcm_grad_axis0", ff::grad_kernel<T, N>, q.S[1] * q.S[2], 1, st, X, dir, Y, q, bstride,
                            reg_table<T>(tw, p));
}
template <typename T, int N>
jdft_status FieldFast<T, N>::eps(c_t<T>* Y, const T* eps, int nlines, int64_t bstride, const c_t<T>* tw,
                                 const FftPlan& p, cudaStream_t st) {
    return ff::launch<T, N>("pcm_eps_axis2", ff::eps_kernel<T, N>, nlines, 3, st, Y, eps, nlines, bstride,
                            reg_table<T>(tw, p));
}
template <typename T, int N>
jdft_status FieldFast<T, N>::div(const c_t<T>* Y, const c_t<T>* din, c_t<T>* out, const FieldCell& q, int64_t bstride,
                                 double scale, const BlockSum& sum, const c_t<T>* tw, const FftPlan& p,
                                 cudaStream_t st) {
    return ff::launch<T, N>("pcm_div_axis0", ff::div_kernel<T, N>, q.S[1] * q.S[2], 1, st, Y, din, out, q, bstride,
                            scale, sum, reg_table<T>(tw, p));
}

template <int N>
jdft_status HartreeFast<N>::forward2(const double* n, double2* half, int nlines, const double2* tw, const FftPlan& p,
                                     cudaStream_t st) {
    return ff::launch<double, N>("field_fft_axis2", ff::hartree_forward2_kernel<N>, (nlines + 1) / 2, 1, st, n, half,
                                 nlines, reg_table<double>(tw, p));
}
template <int N>
jdft_status HartreeFast<N>::kernel0(double2* half, const FieldCell& q, const BlockSum& sum, double sum_scale,
                                    const double2* tw, const FftPlan& p, cudaStream_t st) {
    const double box = (double)N * q.S[1] * q.S[2];
    ff::Coulomb c{ff::kFourPi / box, 0.0};
    c.lo = (fma(-c.hi, box, ff::kFourPi) + ff::kFourPiLo) / box;
    return ff::launch<double, N>("hartree_kernel_axis0", ff::hartree_kernel0_kernel<N>, q.S[1] * (q.S[2] / 2 + 1), 1, st,
                                 half, q, c, sum, sum_scale / box, reg_table<double>(tw, p));
}
template <int N>
jdft_status HartreeFast<N>::inverse2(const double2* half, double* V, const double* n, const double* vion,
                                     const BlockSum& sum, double sum_scale, int nlines, const double2* tw,
                                     const FftPlan& p, cudaStream_t st) {
    const int slots = (nlines + 1) / 2;
    if (vion)
        return ff::launch<double, N>("ks_potential_axis2", ff::hartree_inverse2_kernel<N, true>, slots, 1, st, half, V,
                                     n, vion, sum, sum_scale, nlines, reg_table<double>(tw, p));
    return ff::launch<double, N>("field_fft_axis2", ff::hartree_inverse2_kernel<N, false>, slots, 1, st, half, V, n,
                                 vion, sum, sum_scale, nlines, reg_table<double>(tw, p));
}

}  // namespace jdft
