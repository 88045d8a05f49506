// Complex GEMMs on the CUDA cores (FP64 and FP32): the projector products
// P^dag C and P (D B) of the nonlocal pseudopotential term (JDFTx paper,
// Sec. 2.2, pseudopotentials), and the subspace matrices C^dag H C and
// C^dag O C of the band minimiser (Sec. 2.1, Minimize; O diagonal in the
// plane-wave basis).
#include <algorithm>

#include <type_traits>

#include "gemm.cuh"
#include "profile.cuh"

namespace jdft {

// ---------------------------------------------------------------------------
// C^dag-style product with split K, for the shapes whose FP64 products are too
// small for the sliced ones.  FP64: bound by the FP64 pipe (2
// multiply-adds per clock and SM), so what counts is that every SM has work and
// no lane multiplies padding.  A block of four warps holds a TM x TN tile (16 or
// 32 each way, whichever pads less) and a range of K in chunks of 32; each warp
// takes a quarter of a chunk's K with the whole tile in its registers (lanes
// 8 x 4, TM/8 x TN/4 outputs each), so one shared-memory read feeds 5 to 11
// multiply-adds.  The warps' sums meet in shared memory, the blocks' in FP64 atomics.
// Against a 32 x 32 tile of 256 threads with 2 x 2 outputs each and at least 64
// K to a block, 16 x 16 over 4 259 plane waves took 142 us and takes 22 (event times),
// 27 before a complex multiply-add was written as four fused instructions (mad).
// ---------------------------------------------------------------------------
constexpr int CN_BK = 32, CN_WARPS = 4;

__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }

template <typename T, int TM, int TN>
__global__ void __launch_bounds__(32 * CN_WARPS)
    zgemm_cn_kernel(int M, int N, int K, int kchunk, const c_t<T>* __restrict__ A, int lda,
                    const c_t<T>* __restrict__ B, int ldb, double2* __restrict__ out, int ldo, double scale) {
    constexpr int PM = TM / 8, PN = TN / 4, THREADS = 32 * CN_WARPS;
    constexpr int STAGE = CN_BK * (TM + 1 + TN + 1);
    constexpr int ELEMS = STAGE > CN_WARPS * TM * TN ? STAGE : CN_WARPS * TM * TN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    c_t<T>* As = reinterpret_cast<c_t<T>*>(smem_raw);  // [CN_BK][TM + 1]
    c_t<T>* Bs = As + CN_BK * (TM + 1);                // [CN_BK][TN + 1]
    static_assert(ELEMS * sizeof(c_t<T>) <= 64 * 1024, "shared memory of a block");
    const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
    const int kA = blockIdx.z * kchunk, kB = min(K, kA + kchunk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lm = lane >> 2, ln = lane & 3;
    c_t<T> acc[PM][PN];
#pragma unroll
    for (int i = 0; i < PM; ++i)
#pragma unroll
        for (int j = 0; j < PN; ++j) acc[i][j] = mk<T>(T(0), T(0));
    for (int k0 = kA; k0 < kB; k0 += CN_BK) {
        // a warp reads 32 consecutive K values of one row
        for (int e = threadIdx.x; e < (TM + TN) * CN_BK; e += THREADS) {
            const int r = e / CN_BK, kk = e % CN_BK, k = k0 + kk;
            c_t<T> v = mk<T>(T(0), T(0));
            if (r < TM) {
                if (m0 + r < M && k < kB) v = A[(size_t)(m0 + r) * lda + k];
                As[kk * (TM + 1) + r] = v;
            } else {
                if (n0 + r - TM < N && k < kB) v = B[(size_t)(n0 + r - TM) * ldb + k];
                Bs[kk * (TN + 1) + r - TM] = v;
            }
        }
        __syncthreads();
        const int kn = min(CN_BK, kB - k0);
#pragma unroll 2
        for (int kk = warp; kk < kn; kk += CN_WARPS) {
            c_t<T> a[PM], b[PN];
#pragma unroll
            for (int i = 0; i < PM; ++i) a[i] = As[kk * (TM + 1) + lm + 8 * i];
#pragma unroll
            for (int j = 0; j < PN; ++j) b[j] = Bs[kk * (TN + 1) + ln + 4 * j];
#pragma unroll
            for (int i = 0; i < PM; ++i)
#pragma unroll
                for (int j = 0; j < PN; ++j) {
                    // conj(a) * b, as four multiply-adds (summing the two products first would make six)
                    acc[i][j].x = mad(a[i].y, b[j].y, mad(a[i].x, b[j].x, acc[i][j].x));
                    acc[i][j].y = mad(-a[i].y, b[j].x, mad(a[i].x, b[j].y, acc[i][j].y));
                }
        }
        __syncthreads();
    }
    c_t<T>* red = As;  // [warp][m][n]
#pragma unroll
    for (int i = 0; i < PM; ++i)
#pragma unroll
        for (int j = 0; j < PN; ++j) red[(warp * TM + lm + 8 * i) * TN + ln + 4 * j] = acc[i][j];
    __syncthreads();
    for (int e = threadIdx.x; e < TM * TN; e += THREADS) {
        const int m = m0 + e / TN, n = n0 + e % TN;
        if (m >= M || n >= N) continue;
        double x = 0.0, y = 0.0;
#pragma unroll
        for (int w = 0; w < CN_WARPS; ++w) {
            const c_t<T> v = red[w * TM * TN + e];
            x += (double)v.x;
            y += (double)v.y;
        }
        atomicAdd(&out[(size_t)m * ldo + n].x, scale * x);
        atomicAdd(&out[(size_t)m * ldo + n].y, scale * y);
    }
}

template <typename T, int TM, int TN>
static jdft_status launch_zgemm_cn(int M, int N, int K, const c_t<T>* A, int lda, const c_t<T>* B, int ldb,
                                   double2* out, int ldo, double scale, cudaStream_t st) {
    const int tiles = ((M + TM - 1) / TM) * ((N + TN - 1) / TN);
    // enough K splits for two blocks per SM (one for a single tile: fewer atomics), each at least 16 deep
    int splits = tiles == 1 ? 152 : (304 + tiles - 1) / tiles;
    splits = std::min(splits, std::max(1, K / 16));
    int kchunk = (K + splits - 1) / splits;
    kchunk = (kchunk + CN_WARPS - 1) / CN_WARPS * CN_WARPS;
    splits = (K + kchunk - 1) / kchunk;
    dim3 grid((M + TM - 1) / TM, (N + TN - 1) / TN, splits);
    const size_t smem = std::max<size_t>(CN_BK * (TM + 1 + TN + 1), CN_WARPS * TM * TN) * sizeof(c_t<T>);
    cudaError_t e = set_smem_attr((const void*)zgemm_cn_kernel<T, TM, TN>, smem);
    if (e != cudaSuccess) return set_error(JDFT_ERR_CUDA, std::string("zgemm_cn: ") + cudaGetErrorString(e));
    {
        Trace tr_("zgemm_cn", st);
        zgemm_cn_kernel<T, TM, TN><<<grid, 32 * CN_WARPS, smem, st>>>(M, N, K, kchunk, A, lda, B, ldb, out, ldo, scale);
    }
    return check_launch("zgemm_cn");
}

// FP32 blocks: the multiply-adds are cheap and latency counts, so a block of eight
// warps shares its staged K (16 deep), each thread with P x P outputs of a 16 P square
// tile, four blocks to an SM.  The tiles above, with four warps a block and two blocks
// an SM, tie with P = 2 at 44 x 13 over 6 600 plane waves (18.6 us) and lose on large
// blocks (spinor H C of 64 bands on 128^3 with 256 projectors 3.29 ms; with P = 4 here
// and cgemm_nn_kernel below 2.08 ms).
constexpr int CNF_BK = 16;

template <int P>
__global__ void __launch_bounds__(256)
    cgemm_cn_kernel(int M, int N, int K, int kchunk, const float2* __restrict__ A, int lda, const float2* __restrict__ B,
                    int ldb, double2* __restrict__ out, int ldo, double scale) {
    constexpr int TILE = 16 * P;
    __shared__ float2 As[CNF_BK][TILE + 1];
    __shared__ float2 Bs[CNF_BK][TILE + 1];
    const int m0 = blockIdx.x * TILE, n0 = blockIdx.y * TILE;
    const int kA = blockIdx.z * kchunk, kB = min(K, kA + kchunk);
    const int tm = threadIdx.x / 16, tn = threadIdx.x % 16;
    float2 acc[P][P];
#pragma unroll
    for (int i = 0; i < P; ++i)
#pragma unroll
        for (int j = 0; j < P; ++j) acc[i][j] = make_float2(0.f, 0.f);
    for (int k0 = kA; k0 < kB; k0 += CNF_BK) {
#pragma unroll
        for (int e = threadIdx.x; e < TILE * CNF_BK; e += 256) {
            const int r = e / CNF_BK, kk = e % CNF_BK;
            const int m = m0 + r, n = n0 + r, k = k0 + kk;
            As[kk][r] = (m < M && k < kB) ? A[(size_t)m * lda + k] : make_float2(0.f, 0.f);
            Bs[kk][r] = (n < N && k < kB) ? B[(size_t)n * ldb + k] : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < CNF_BK; ++kk) {
            float2 a[P], b[P];
#pragma unroll
            for (int i = 0; i < P; ++i) a[i] = As[kk][tm + 16 * i];
#pragma unroll
            for (int j = 0; j < P; ++j) b[j] = Bs[kk][tn + 16 * j];
#pragma unroll
            for (int i = 0; i < P; ++i)
#pragma unroll
                for (int j = 0; j < P; ++j) {
                    if constexpr (P == 2) {
                        // the shorter chain: four outputs a thread hardly hide two additions in a row (two
                        // products of 32 x 32 over 19 808: 41.5 us, 47.9 with the form below; H C of 4 bands
                        // with 256 projectors on 62 759 the other way, 308 and 280)
                        acc[i][j].x += a[i].x * b[j].x + a[i].y * b[j].y;
                        acc[i][j].y += a[i].x * b[j].y - a[i].y * b[j].x;
                    } else {
                        acc[i][j].x = mad(a[i].y, b[j].y, mad(a[i].x, b[j].x, acc[i][j].x));
                        acc[i][j].y = mad(-a[i].y, b[j].x, mad(a[i].x, b[j].y, acc[i][j].y));
                    }
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < P; ++i)
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const int m = m0 + tm + 16 * i, n = n0 + tn + 16 * j;
            if (m < M && n < N) {
                atomicAdd(&out[(size_t)m * ldo + n].x, scale * (double)acc[i][j].x);
                atomicAdd(&out[(size_t)m * ldo + n].y, scale * (double)acc[i][j].y);
            }
        }
}

template <int P>
static jdft_status launch_cgemm_cn(int M, int N, int K, const float2* A, int lda, const float2* B, int ldb, double2* out,
                                   int ldo, double scale, cudaStream_t st) {
    constexpr int TILE = 16 * P;
    const int mt = (M + TILE - 1) / TILE, nt = (N + TILE - 1) / TILE;
    // enough K splits for about 4 blocks per SM, each at least 64 deep
    int splits = std::max(1, (152 * 4 + mt * nt - 1) / (mt * nt));
    splits = std::min(splits, std::max(1, K / 64));
    int kchunk = (K + splits - 1) / splits;
    kchunk = (kchunk + CNF_BK - 1) / CNF_BK * CNF_BK;
    splits = (K + kchunk - 1) / kchunk;
    {
        Trace tr_("zgemm_cn", st);
        cgemm_cn_kernel<P><<<dim3(mt, nt, splits), 256, 0, st>>>(M, N, K, kchunk, A, lda, B, ldb, out, ldo, scale);
    }
    return check_launch("zgemm_cn");
}

template <>
jdft_status zgemm_cn<float>(int M, int N, int K, const float2* A, int lda, const float2* B, int ldb, double2* out,
                            int ldo, double scale, cudaStream_t st) {
    if (M == 0 || N == 0 || K == 0) return JDFT_OK;
    // 64-wide tiles where they are more than half full both ways and the product is long enough for
    // their larger blocks (two products, P = 2 / 4: 64 x 64 over 4 259 34 / 49 us, over 19 808 67 / 74,
    // over 62 759 156 / 154; 128 x 128 over 19 808 190 / 155, over 62 759 604 / 436)
    if (M > 32 && N > 32 && (double)M * N * K > 1e8) return launch_cgemm_cn<4>(M, N, K, A, lda, B, ldb, out, ldo, scale, st);
    return launch_cgemm_cn<2>(M, N, K, A, lda, B, ldb, out, ldo, scale, st);
}

template <>
jdft_status zgemm_cn<double>(int M, int N, int K, const double2* A, int lda, const double2* B, int ldb, double2* out,
                             int ldo, double scale, cudaStream_t st) {
    using T = double;
    if (M == 0 || N == 0 || K == 0) return JDFT_OK;
    // 16-wide tiles where a 32-wide one would be at most half full at the edge
    const bool m16 = (M - 1) % 32 < 16, n16 = (N - 1) % 32 < 16;
    if (m16 && n16) return launch_zgemm_cn<T, 16, 16>(M, N, K, A, lda, B, ldb, out, ldo, scale, st);
    if (m16) return launch_zgemm_cn<T, 16, 32>(M, N, K, A, lda, B, ldb, out, ldo, scale, st);
    if (n16) return launch_zgemm_cn<T, 32, 16>(M, N, K, A, lda, B, ldb, out, ldo, scale, st);
    return launch_zgemm_cn<T, 32, 32>(M, N, K, A, lda, B, ldb, out, ldo, scale, st);
}

// ---------------------------------------------------------------------------
// out[n][m] += sum_i A[i][m] Bm[i][n].  A block holds 32 m x 16 n, warp w the
// columns 4 w .. 4 w + 3: a lane owns one m, reads A straight from global memory
// (32 consecutive values a warp, sixteen rows in flight) and Bm, staged 64 rows deep, by broadcast.
// Small blocks, because N is small where this kernel is used and M/32 of them
// just fill the SMs: 16 x 16 over 4 259 rows 40 -> 23 us in FP64 against 64 m to a
// block, which used 67 SMs, and 18 with four fused instructions a multiply-add.
// ---------------------------------------------------------------------------
constexpr int NN_BM = 32, NN_PN = 4, NN_WARPS = 4, NN_BN = NN_PN * NN_WARPS, NN_BK = 64;

template <typename T>
__global__ void __launch_bounds__(32 * NN_WARPS)
    zgemm_nn_kernel(int M, int N, int K, const c_t<T>* __restrict__ A, int lda, const c_t<T>* __restrict__ Bm, int ldb,
                    c_t<T>* __restrict__ out, int ldo, bool accumulate) {
    __shared__ __align__(16) c_t<T> Bs[NN_BK][NN_BN];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m = blockIdx.x * NN_BM + lane, n0 = blockIdx.y * NN_BN;
    c_t<T> acc[NN_PN];
#pragma unroll
    for (int j = 0; j < NN_PN; ++j) acc[j] = mk<T>(T(0), T(0));
    for (int k0 = 0; k0 < K; k0 += NN_BK) {
        for (int e = threadIdx.x; e < NN_BK * NN_BN; e += 32 * NN_WARPS) {
            const int kk = e / NN_BN, c = e % NN_BN;
            Bs[kk][c] = (n0 + c < N && k0 + kk < K) ? Bm[(size_t)(k0 + kk) * ldb + n0 + c] : mk<T>(T(0), T(0));
        }
        __syncthreads();
        const int kn = min(NN_BK, K - k0);
        if (m < M) {
            const c_t<T>* Ak = A + (size_t)k0 * lda + m;
#pragma unroll 16
            for (int kk = 0; kk < kn; ++kk) {
                const c_t<T> a = Ak[(size_t)kk * lda];
#pragma unroll
                for (int j = 0; j < NN_PN; ++j) {
                    const c_t<T> b = Bs[kk][warp * NN_PN + j];
                    acc[j].x = mad(-a.y, b.y, mad(a.x, b.x, acc[j].x));
                    acc[j].y = mad(a.y, b.x, mad(a.x, b.y, acc[j].y));
                }
            }
        }
        __syncthreads();
    }
    if (m < M) {
#pragma unroll
        for (int j = 0; j < NN_PN; ++j) {
            const int n = n0 + warp * NN_PN + j;
            if (n < N) out[(size_t)n * ldo + m] = accumulate ? cadd(out[(size_t)n * ldo + m], acc[j]) : acc[j];
        }
    }
}

// FP32 blocks on many plane waves: A's tile staged as well, 256 threads of 2 m x 8 n
// each (128 x 32 outputs a block), so that A is read once per 32 columns instead of
// once per 16 and a shared-memory read feeds 6 multiply-adds (FP32 H C of 64 bands with
// 256 projectors on 62 759 plane waves, both products: 1 179 -> 993 us against 64 m x
// 16 n a block).
constexpr int NNF_BM = 128, NNF_BN = 32, NNF_BK = 16;

__global__ void __launch_bounds__(256)
    cgemm_nn_kernel(int M, int N, int K, const float2* __restrict__ A, int lda, const float2* __restrict__ Bm, int ldb,
                    float2* __restrict__ out, int ldo, bool accumulate) {
    __shared__ float2 As[NNF_BK][NNF_BM];
    __shared__ float2 Bs[NNF_BK][NNF_BN];
    const int m0 = blockIdx.x * NNF_BM, n0 = blockIdx.y * NNF_BN;
    const int tm = threadIdx.x % 64, tq = threadIdx.x / 64;  // rows tm and tm + 64, columns 8 tq .. 8 tq + 7
    float2 acc[2][8];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = make_float2(0.f, 0.f);
    for (int k0 = 0; k0 < K; k0 += NNF_BK) {
#pragma unroll
        for (int e = threadIdx.x; e < NNF_BK * NNF_BM; e += 256) {
            const int kk = e / NNF_BM, r = e % NNF_BM;
            const int m = m0 + r, k = k0 + kk;
            As[kk][r] = (m < M && k < K) ? A[(size_t)k * lda + m] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int e = threadIdx.x; e < NNF_BK * NNF_BN; e += 256) {
            const int kk = e / NNF_BN, c = e % NNF_BN;
            const int n = n0 + c, k = k0 + kk;
            Bs[kk][c] = (n < N && k < K) ? Bm[(size_t)k * ldb + n] : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < NNF_BK; ++kk) {
            const float2 a0 = As[kk][tm], a1 = As[kk][tm + 64];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float2 b = Bs[kk][tq * 8 + j];
                acc[0][j].x = mad(-a0.y, b.y, mad(a0.x, b.x, acc[0][j].x));
                acc[0][j].y = mad(a0.y, b.x, mad(a0.x, b.y, acc[0][j].y));
                acc[1][j].x = mad(-a1.y, b.y, mad(a1.x, b.x, acc[1][j].x));
                acc[1][j].y = mad(a1.y, b.x, mad(a1.x, b.y, acc[1][j].y));
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int m = m0 + tm + 64 * i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int n = n0 + tq * 8 + j;
            if (n < N) out[(size_t)n * ldo + m] = accumulate ? cadd(out[(size_t)n * ldo + m], acc[i][j]) : acc[i][j];
        }
    }
}

template <typename T>
jdft_status zgemm_nn_acc(int M, int N, int K, const c_t<T>* A, int lda, const c_t<T>* Bm, int ldb, c_t<T>* out,
                         int ldo, cudaStream_t st, bool accumulate) {
    if (M == 0 || N == 0) return JDFT_OK;
    if (K == 0) {
        if (!accumulate)
            for (int n = 0; n < N; ++n)
                JDFT_CUDA_TRY(cudaMemsetAsync(out + (size_t)n * ldo, 0, (size_t)M * sizeof(c_t<T>), st));
        return JDFT_OK;
    }
    if constexpr (std::is_same<T, float>::value) {
        // two blocks for every SM, and more than half of the 32 columns
        const int mt = (M + NNF_BM - 1) / NNF_BM, nt = (N + NNF_BN - 1) / NNF_BN;
        if (N > 16 && (int64_t)mt * nt >= 304) {
            {
                Trace tr_("zgemm_nn", st);
                cgemm_nn_kernel<<<dim3(mt, nt), 256, 0, st>>>(M, N, K, A, lda, Bm, ldb, out, ldo, accumulate);
            }
            return check_launch("zgemm_nn");
        }
    }
    dim3 grid((M + NN_BM - 1) / NN_BM, (N + NN_BN - 1) / NN_BN);
    {
        Trace tr_("zgemm_nn", st);
        zgemm_nn_kernel<T><<<grid, 32 * NN_WARPS, 0, st>>>(M, N, K, A, lda, Bm, ldb, out, ldo, accumulate);
    }
    return check_launch("zgemm_nn");
}

// Bd[i][b] = sum_j D[i][j] Bc[j][b], rounded to the product type; D as ELL
// rows (w entries of column index and value per row).
template <typename T>
__global__ void dmul_kernel(int nproj, int nb, int w, const int* __restrict__ Dcol, const double* __restrict__ Dval,
                            const double2* __restrict__ Bc, c_t<T>* __restrict__ Bd) {
    const int total = nproj * nb;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int i = e / nb, b = e % nb;
        double re = 0.0, im = 0.0;
        for (int q = 0; q < w; ++q) {
            const double d = Dval[(size_t)i * w + q];
            const double2 x = Bc[(size_t)Dcol[(size_t)i * w + q] * nb + b];
            re += d * x.x;
            im += d * x.y;
        }
        Bd[e] = mk<T>((T)re, (T)im);
    }
}

bool gemm_nn_inplace_ok(jdft_prec prec, int N) {
    if (prec == JDFT_BF16X3) return N <= 256;
    if (prec == JDFT_TF32X3) return N <= 128;
    return false;  // the CUDA-core products tile N in 16-column blocks
}

size_t nonlocal_workspace_bytes(int nproj, int nb, size_t elem, int npw, jdft_prec prec, bool split_c,
                                bool partials) {
    if (nproj == 0) return 0;
    const size_t a = ((size_t)nproj * nb * sizeof(double2) + 255) / 256 * 256;
    const size_t b = ((size_t)nproj * nb * elem + 255) / 256 * 256;
    const size_t c = split_c && tcx_eligible(prec, nproj, nb) ? (tcx_split_bytes(nb, npw) + 255) / 256 * 256 : 0;
    // the split of (D P^dag C)'s transpose for P (D P^dag C) on split operands
    const size_t d = tcx_eligible(prec, nproj, nb) ? (tcx_split_bytes(nb, nproj) + 255) / 256 * 256 : 0;
    const size_t e = partials && tcx_eligible(prec, nproj, nb) ? tcx_cn_partial_bytes(nproj, nb, npw) : 0;
    return a + b + c + d + e;
}

template <typename T>
static const c_t<T>* proj_ptr(const KSphere& sp);
template <> const double2* proj_ptr<double>(const KSphere& sp) { return (const double2*)sp.P; }
template <> const float2* proj_ptr<float>(const KSphere& sp) { return (const float2*)sp.P32; }

bool nonlocal_small(const KSphere& sp, int nb, jdft_prec prec) {
    if (prec == JDFT_FP64) return !sl_eligible(sp.nproj, nb, sp.npw);
    return !tcx_eligible(prec, sp.nproj, nb) && (size_t)sp.nproj * nb * sp.npw < (size_t)64 << 20;
}

template <typename T>
jdft_status nonlocal_accumulate(const KSphere& sp, const void* C, int ldc, void* HC, int ldhc, int nb,
                                jdft_prec prec, void* work, cudaStream_t st, bool split_c, const void* Csplit,
                                bool partials, ProductScratch* scratch, int phases) {
    if (sp.nproj == 0 || nb == 0) return JDFT_OK;
    double2* Bc = (double2*)work;
    const size_t abytes = ((size_t)sp.nproj * nb * sizeof(double2) + 255) / 256 * 256;
    const size_t bbytes = ((size_t)sp.nproj * nb * sizeof(c_t<T>) + 255) / 256 * 256;
    c_t<T>* Bd = (c_t<T>*)((char*)work + abytes);
    jdft_status s;
    const bool split_ops = std::is_same<T, float>::value && (split_c || Csplit) && sp.Psplit &&
                           tcx_eligible(prec, sp.nproj, nb);
    const size_t cbytes = split_c && tcx_eligible(prec, sp.nproj, nb)
                              ? (tcx_split_bytes(nb, sp.npw) + 255) / 256 * 256 : 0;
    if (phases & kNonlocalProject) {
        JDFT_CUDA_TRY(cudaMemsetAsync(Bc, 0, (size_t)sp.nproj * nb * sizeof(double2), st));
        if (split_ops) {
            const void* Cs = Csplit;
            if (!Cs) {
                void* own = (char*)work + abytes + bbytes;
                if ((s = tcx_split((const float2*)C, ldc, nb, sp.npw, own, st))) return s;
                Cs = own;
            }
            const size_t dbytes = (tcx_split_bytes(nb, sp.nproj) + 255) / 256 * 256;
            void* part = partials ? (char*)work + abytes + bbytes + cbytes + dbytes : nullptr;
            s = tcx_cn(sp.nproj, nb, sp.npw, sp.Psplit, Cs, Bc, nb, 1.0, st, part,
                       partials ? tcx_cn_partial_bytes(sp.nproj, nb, sp.npw) : 0);
        } else {
            s = gemm_cn<T>(prec, sp.nproj, nb, sp.npw, proj_ptr<T>(sp), sp.npw, (const c_t<T>*)C, ldc, Bc, nb, 1.0, st,
                           scratch);
        }
        if (s != JDFT_OK) return s;
        {
            Trace tr_("dmul", st);
            dmul_kernel<T><<<std::min(152 * 8, (sp.nproj * nb + 255) / 256), 256, 0, st>>>(sp.nproj, nb, sp.Dw, sp.Dcol,
                                                                                            sp.Dval, Bc, Bd);
        }
        if ((s = check_launch("dmul"))) return s;
    }
    if (!(phases & kNonlocalAdd)) return JDFT_OK;
    if (split_ops && sp.Psplit_t) {
        // HC += P (D P^dag C): P's transposed split (made with the projectors) and that of D P^dag C
        void* Bt = (char*)work + abytes + bbytes + cbytes;
        if ((s = tcx_split_t((const float2*)Bd, nb, nb, sp.nproj, Bt, st))) return s;
        return tcx_nn(sp.npw, nb, sp.nproj, sp.Psplit_t, Bt, (float2*)HC, ldhc, true, st);
    }
    return gemm_nn_acc<T>(prec, sp.npw, nb, sp.nproj, proj_ptr<T>(sp), sp.npw, Bd, nb, (c_t<T>*)HC, ldhc, st, true, scratch);
}

template <>
jdft_status gemm_cn<double>(jdft_prec, int M, int N, int K, const double2* A, int lda, const double2* B, int ldb,
                            double2* out, int ldo, double alpha, cudaStream_t st, ProductScratch* scratch) {
    if (scratch && sl_eligible(M, N, K)) {
        const jdft_status s = sl_zgemm_cn(M, N, K, A, lda, B, ldb, out, ldo, alpha, *scratch, st);
        if (s != JDFT_ERR_UNSUPPORTED) return s;
    }
    return zgemm_cn<double>(M, N, K, A, lda, B, ldb, out, ldo, alpha, st);
}
template <>
jdft_status gemm_cn<float>(jdft_prec prec, int M, int N, int K, const float2* A, int lda, const float2* B, int ldb,
                           double2* out, int ldo, double alpha, cudaStream_t st, ProductScratch*) {
    if (prec == JDFT_TF32X3 || prec == JDFT_BF16X3)
        return tc_zgemm_cn(M, N, K, A, lda, B, ldb, out, ldo, alpha, prec == JDFT_BF16X3, st);
    return zgemm_cn<float>(M, N, K, A, lda, B, ldb, out, ldo, alpha, st);
}
template <>
jdft_status gemm_nn_acc<double>(jdft_prec, int M, int N, int K, const double2* A, int lda, const double2* Bm, int ldb,
                                double2* out, int ldo, cudaStream_t st, bool accumulate, ProductScratch* scratch) {
    if (scratch && sl_eligible(M, N, K)) {
        const jdft_status s = sl_zgemm_nn(M, N, K, A, lda, Bm, ldb, out, ldo, accumulate, *scratch, st);
        if (s != JDFT_ERR_UNSUPPORTED) return s;
    }
    return zgemm_nn_acc<double>(M, N, K, A, lda, Bm, ldb, out, ldo, st, accumulate);
}
template <>
jdft_status gemm_nn_acc<float>(jdft_prec prec, int M, int N, int K, const float2* A, int lda, const float2* Bm, int ldb,
                               float2* out, int ldo, cudaStream_t st, bool accumulate, ProductScratch*) {
    if (prec == JDFT_TF32X3 || prec == JDFT_BF16X3)
        return tc_zgemm_nn_acc(M, N, K, A, lda, Bm, ldb, out, ldo, prec == JDFT_BF16X3, st, accumulate);
    return zgemm_nn_acc<float>(M, N, K, A, lda, Bm, ldb, out, ldo, st, accumulate);
}

template jdft_status zgemm_nn_acc<double>(int, int, int, const double2*, int, const double2*, int, double2*, int,
                                          cudaStream_t, bool);
template jdft_status zgemm_nn_acc<float>(int, int, int, const float2*, int, const float2*, int, float2*, int,
                                         cudaStream_t, bool);
template jdft_status nonlocal_accumulate<double>(const KSphere&, const void*, int, void*, int, int, jdft_prec, void*,
                                                 cudaStream_t, bool, const void*, bool, ProductScratch*, int);
template jdft_status nonlocal_accumulate<float>(const KSphere&, const void*, int, void*, int, int, jdft_prec, void*,
                                                cudaStream_t, bool, const void*, bool, ProductScratch*, int);

}  // namespace jdft

using namespace jdft;

extern "C" jdft_status jdft_subspace(jdft_basis_t b, int ik, const void* C, int ldc, const void* HC, int ldhc, int nb,
                                     void* CHC, void* COC, jdft_prec prec, void* stream) {
    clear_error();
    JDFT_CHECK_ARG(b, "null basis");
    JDFT_CHECK_ARG(ik >= 0 && ik < b->nk, "k-point index out of range");
    JDFT_CHECK_ARG(nb >= 0, "nb must be >= 0");
    JDFT_CHECK_ARG(prec >= JDFT_FP64 && prec <= JDFT_BF16X3, "unknown precision");
    if (nb == 0) return JDFT_OK;
    const int npw = b->ks[ik].npw;
    JDFT_CHECK_ARG(C && ldc >= npw, "bad C block");
    JDFT_CHECK_ARG(!CHC || (HC && ldhc >= npw), "bad HC block");
    JDFT_CHECK_ARG(((uintptr_t)CHC % 16) == 0 && ((uintptr_t)COC % 16) == 0, "outputs must be 16-byte aligned");
    cudaStream_t st = (cudaStream_t)stream;
    jdft_status s = JDFT_OK;
    if (prec == JDFT_BF16X3 && tcx_eligible(prec, nb, nb)) {
        // split C (and HC) once into BF16 planes in the basis workspace; both
        // products read the split C
        // (and room for the products' split-K partial tiles after them)
        const size_t cb = (tcx_split_bytes(nb, npw) + 255) / 256 * 256;
        const size_t pb = tcx_cn_partial_bytes(nb, nb, npw);
        const size_t sb = CHC ? 2 * cb : cb;
        if ((s = ensure_workspace(b, sb + pb))) return s;
        char* ws = (char*)b->work.ptr;
        if ((s = tcx_split((const float2*)C, ldc, nb, npw, ws, st))) return s;
        if (CHC) {
            if ((s = tcx_split((const float2*)HC, ldhc, nb, npw, ws + cb, st))) return s;
            JDFT_CUDA_TRY(cudaMemsetAsync(CHC, 0, (size_t)nb * nb * sizeof(double2), st));
            if ((s = tcx_cn(nb, nb, npw, ws, ws + cb, (double2*)CHC, nb, 1.0, st, ws + sb, pb))) return s;
        }
        if (COC) {
            JDFT_CUDA_TRY(cudaMemsetAsync(COC, 0, (size_t)nb * nb * sizeof(double2), st));
            if ((s = tcx_cn(nb, nb, npw, ws, ws, (double2*)COC, nb, b->omega, st, ws + sb, pb, true)))
                return s;
        }
        return JDFT_OK;
    }
    if (CHC) {
        JDFT_CUDA_TRY(cudaMemsetAsync(CHC, 0, (size_t)nb * nb * sizeof(double2), st));
        s = (prec == JDFT_FP64)
                ? gemm_cn<double>(prec, nb, nb, npw, (const double2*)C, ldc, (const double2*)HC, ldhc, (double2*)CHC,
                                  nb, 1.0, st, &b->subwork)
                : gemm_cn<float>(prec, nb, nb, npw, (const float2*)C, ldc, (const float2*)HC, ldhc, (double2*)CHC, nb, 1.0,
                                  st);
        if (s != JDFT_OK) return s;
    }
    if (COC) {
        JDFT_CUDA_TRY(cudaMemsetAsync(COC, 0, (size_t)nb * nb * sizeof(double2), st));
        s = (prec == JDFT_FP64)
                ? gemm_cn<double>(prec, nb, nb, npw, (const double2*)C, ldc, (const double2*)C, ldc, (double2*)COC, nb,
                                  b->omega, st, &b->subwork)
                : gemm_cn<float>(prec, nb, nb, npw, (const float2*)C, ldc, (const float2*)C, ldc, (double2*)COC, nb,
                                  b->omega, st);
    }
    return s;
}
