// FP64 complex products on the tensor cores, from operands cut into exact
// 7-bit slices (included by tc_gemm.cu, whose barriers and wait limits it uses).
//
// What bounds an FP64 product on the CUDA cores is the FP64 pipe: 2 multiply-adds
// per clock and SM, 1.26 TFLOP/s over the chip.  BF16 tensor products run three
// orders of magnitude faster, and are exact on small integers: so each row of an
// operand is scaled by a power of two to 62-bit integers, written in nine signed
// base-128 digits
//     x = 2^(e - 61) sum_{i = 1..9} d_i 2^(7 (9 - i)),   -64 <= d_i <= 64,
// (BF16 holds the digits exactly), and the product is the sum over digit pairs
// with i + j <= 10 (45 pairs, each four real products): error-free products of
// slices as in Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 95 (2012), and
// Mukunoki et al., ISC 2020 (with FP16 tensor cores).  A product of digits is at
// most 2^12 and FP32 sums of integers are exact up to 2^24, so a block sums
// 2 (D - 1) K <= 4096 products (D = i + j) in tensor memory before the sum is
// taken out as an integer.  What is dropped (digits below 2^-62 of a row's
// largest value, pairs beyond 10) is below 2^-62 of the rows' largest products: over
// the block shapes here the results are nearer to extended precision than the
// FP64 sums they replace.
//
// Launches: row maxima, slices (36 bytes a complex value) of both operands, the
// products, and the sum of the blocks' integers (128 bits) into the FP64 output.
// A unit of work (block) is a 128 x NT output tile, a pair of digit sums (D, D - 1)
// and a range of K: at step j it adds A_j B_(D-j) to the first and
// A_(j-1) B_(D-j) to the second accumulator, so each slice is staged once for
// two products; three steps share a stage, copied by one bulk copy per operand.
// Tensor memory holds 2 x 2 x NT columns.
//
// Measured (event times, against the CUDA-core products): overlap, subspace matrix
// and rotation of 120 bands of 27 000 plane waves 19.86 -> 1.32 ms, error against
// 64-bit references 6.7e-16 -> 5.9e-16 (the Cholesky factorisation between them
// takes 0.35 ms); H C of 64 bands on a 128^3 box with 256 projectors 28.06 -> 7.64 ms
// when they came in, their two launches of products 0.65 ms each then and 0.58 now.
#pragma once

namespace jdft {

constexpr int SL_N = 9;                 // slices of an operand
constexpr int SL_BITS = 7;
constexpr int SL_GROUPS = 5;            // digit sums (10, 9), (8, 7), (6, 5), (4, 3), (2)
constexpr int SL_PLANES = 2 * SL_N;     // Re and Im of each slice
constexpr int SL_STAGES = 4;
constexpr int SL_RUN = 3;               // slices per stage and operand, one copy each
constexpr int SL_THREADS = 128;
constexpr int SL_BIAS = 1 << 13;        // of stored exponents (0: none)
constexpr int SL_BAD = 1 << 20;         // exponent of a row with an infinity or NaN
__host__ __device__ constexpr int sl_top(int g) { return 10 - 2 * g; }              // larger digit sum of group g
__host__ __device__ constexpr int sl_limit(int g) { return 2048 / (sl_top(g) - 1) / TCX_KC; }  // K chunks per unit

// How the K range is cut per group: per[g] chunks to a unit, first[g] the
// group's first unit (first[SL_GROUPS]: units in all).
struct SlPlan {
    int per[SL_GROUPS];
    int first[SL_GROUPS + 1];
};

// ---- row maxima -------------------------------------------------------------
// Exponents are exponent fields (1 for zeros and denormals, whose significands have no
// implicit bit) plus SL_BIAS, so that 0 means none.  `shift` scales the summed index: value
// k counts as 2^(sign (shift[k] - SL_BIAS)) times itself, with sign -1 for one operand and
// +1 for the other (see sl_zgemm_nn).
__device__ __forceinline__ int sl_field(int hi) { return max((hi >> 20) & 0x7ff, 1); }
__device__ __forceinline__ int sl_shift(const int* __restrict__ shift, int sign, int k) {
    return shift ? sign * (shift[k] - SL_BIAS) : 0;
}
// The exponent that a row of largest component v has at least: SL_BAD for an infinity or NaN.
__device__ __forceinline__ int sl_exponent(double2 v, int shift) {
    const int x = __double2hiint(v.x) & 0x7fffffff, y = __double2hiint(v.y) & 0x7fffffff, hi = max(x, y);
    if ((hi >> 20) == 0x7ff) return SL_BAD;
    return (hi | __double2loint(v.x) | __double2loint(v.y)) == 0 ? 0 : sl_field(hi) + shift + SL_BIAS;
}

// ex[r] = largest exponent over the row's K values (FINITE: of those without an infinity or NaN).
template <bool FINITE>
__global__ void __launch_bounds__(256) sl_rowmax_kernel(const double2* __restrict__ X, size_t ld, int K,
                                                        const int* __restrict__ shift, int sign,
                                                        int* __restrict__ ex) {
    const double2* x = X + (size_t)blockIdx.x * ld;
    int m = 0;
    for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < K; k += gridDim.y * blockDim.x) {
        const int e = sl_exponent(x[k], sl_shift(shift, sign, k));
        if (!FINITE || e != SL_BAD) m = max(m, e);
    }
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&ex[blockIdx.x], m);
}
// The same of the transpose: row r, value k at X[k * ld + r]; blockIdx.y strides over k.
__global__ void __launch_bounds__(256) sl_rowmax_t_kernel(const double2* __restrict__ X, size_t ld, int rows, int K,
                                                          const int* __restrict__ shift, int sign,
                                                          int* __restrict__ ex) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    int m = 0;
    for (int k = blockIdx.y; k < K; k += gridDim.y)
        m = max(m, sl_exponent(X[(size_t)k * ld + r], sl_shift(shift, sign, k)));
    atomicMax(&ex[r], m);
}

// ---- slices -------------------------------------------------------------------
// Layout: [chunk of 16 K][block of RB rows][plane][RB x 16 values], the rows of a
// plane as core matrices (as in the split blocks above).  The planes of consecutive
// slices of a row block are one contiguous run, so a stage of three steps takes one
// bulk copy per operand and one barrier, in place of four copies and a barrier a step
// (products of 120 x 120 over 27 000: 162 -> 147 us a launch; of 256 x 64 over a 128^3
// box's plane waves: 651 -> 582 us).
// One thread per row and 8 consecutive K values: a 16-byte core-matrix row of
// each of the 18 planes.
template <bool TRANS>
__global__ void __launch_bounds__(256) sl_slice_kernel(const double2* __restrict__ X, size_t ld, int rows, int K,
                                                       int rows_pad, int RB, int nkc, const int* __restrict__ ex,
                                                       const int* __restrict__ shift, int sign,
                                                       __nv_bfloat16* __restrict__ out) {
    const int per_chunk = rows_pad * 2;
    const int64_t total = (int64_t)per_chunk * nkc;
    const size_t P = (size_t)RB * TCX_KC;  // elements between planes
    const int nrb = rows_pad / RB;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int kc = (int)(i / per_chunk), u = (int)(i - (int64_t)kc * per_chunk);
        const int r8 = u & 7, h = (u >> 3) & 1, g = u >> 4;
        const int r = g * 8 + r8, k0 = kc * TCX_KC + h * 8;
        uint64_t d[2][8];
        // the digits' offsets: 64 in each place makes them non-negative
        constexpr uint64_t kOffset = 64ull * ((1ull << 0) + (1ull << 7) + (1ull << 14) + (1ull << 21) + (1ull << 28) +
                                              (1ull << 35) + (1ull << 42) + (1ull << 49) + (1ull << 56));
        const int emax = r < rows ? ex[r] - SL_BIAS : 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            double2 v = make_double2(0.0, 0.0);
            int sh = 0;
            if (r < rows && k0 + j < K) {
                v = TRANS ? X[(size_t)(k0 + j) * ld + r] : X[(size_t)r * ld + k0 + j];
                sh = sl_shift(shift, sign, k0 + j);
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const double x = c ? v.y : v.x;
                const int hi = __double2hiint(x);
                // (a zero may lie above its row's exponent: as unsigned, the shift is then 63 too)
                const int n = (int)min((uint32_t)(emax - sl_field(hi) - sh), 63u);
                const uint64_t m = ((uint64_t)(uint32_t)((hi & 0xfffff) | ((hi & 0x7ff00000) ? 0x100000 : 0)) << 32) |
                                   (uint32_t)__double2loint(x);
                const int64_t t = (int64_t)((m << 8) >> n), s = (int64_t)(hi >> 31);
                d[c][j] = (uint64_t)((t ^ s) - s) + kOffset;
            }
        }
        const int rb = r / RB;
        __nv_bfloat16* o = out + ((size_t)kc * nrb + rb) * SL_PLANES * P + (size_t)((r - rb * RB) & ~7) * TCX_KC + h * 64 +
                           r8 * 8;
        const __nv_bfloat162 off = __floats2bfloat162_rn(192.f, 192.f);
#pragma unroll
        for (int s = 0; s < SL_N; ++s) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t w[4];
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    // bits of the BF16 numbers 128 + digit + 64, less 192
                    const uint32_t a = (uint32_t)(d[c][j] >> (7 * (SL_N - 1 - s))) & 127u;
                    const uint32_t b = (uint32_t)(d[c][j + 1] >> (7 * (SL_N - 1 - s))) & 127u;
                    const uint32_t bits = 0x43004300u | a | (b << 16);
                    const __nv_bfloat162 z = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&bits), off);
                    w[j / 2] = *reinterpret_cast<const uint32_t*>(&z);
                }
                *reinterpret_cast<uint4*>(o + (size_t)(2 * s + c) * P) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
}

// ---- products -------------------------------------------------------------------
template <int NT>
struct SlLayout {
    static constexpr int A_PL = TCX_PLANE;
    static constexpr int B_PL = NT * TCX_KC * 2;
    static constexpr int A_SL = 2 * A_PL, B_SL = 2 * B_PL;  // one slice: Re and Im
    static constexpr int B_OFF = SL_RUN * A_SL;
    static constexpr int STAGE = SL_RUN * (A_SL + B_SL);
    static constexpr int BAR_OFF = SL_STAGES * STAGE;
    static constexpr int SMEM = BAR_OFF + 512 + 1024;
    static constexpr uint32_t NCOLS = 4 * NT;
    static_assert(NCOLS <= 512 && SMEM <= 227 * 1024, "one block per SM");
};

// The pieces of the issuing thread's loop, on shared-memory addresses and descriptor words.
__device__ __forceinline__ bool sl_wait(uint32_t bar, uint32_t parity, uint64_t* generic, uint64_t wait_ns) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok && wait_ns) return true;
    return tc::mbar_wait_ns(generic, parity, wait_ns);
}
__device__ __forceinline__ void sl_mma(uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t hi, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(alo), "r"(blo), "r"(hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void sl_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// CONJ: Re = Ar.Br + Ai.Bi, Im = Ar.Bi - Ai.Br (conj(A) B); else Re = Ar.Br - Ai.Bi, Im = Ar.Bi + Ai.Br.
// part: [tile][unit][column][row] of (Re, Im) integers, S_D + 2^7 S_(D-1).
template <int NT, bool CONJ>
__global__ void __launch_bounds__(SL_THREADS, 1)
    sl_mma_kernel(const char* __restrict__ As, const char* __restrict__ Bs, int nrbA, int nrbB, int nkc, int mtiles,
                  SlPlan plan, int2* __restrict__ part) {
    using L = SlLayout<NT>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
    uint64_t* empty = full + SL_STAGES;
    uint64_t* accbar = empty + SL_STAGES;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(accbar + 1);
    volatile int* flags = reinterpret_cast<volatile int*>(tslot + 1);  // 0: failed, 1: stages loaded, 2: steps issued
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int unit = blockIdx.x, tile = blockIdx.y;
    int g = 0;
    while (g + 1 < SL_GROUPS && unit >= plan.first[g + 1]) ++g;
    const int D = sl_top(g), steps = D - 1;
    const int c0 = (unit - plan.first[g]) * plan.per[g], c1 = min(nkc, c0 + plan.per[g]);
    const int mt = tile % mtiles, nt = tile / mtiles;
    const int runs = (steps + SL_RUN - 1) / SL_RUN;  // stages per chunk
    const int total = (c1 - c0) * runs;              // at least one: the plan has no empty units
    if (tid == 0) {
        for (int s = 0; s < SL_STAGES; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(accbar, 1);
        flags[0] = 0;
        flags[1] = 0;
        flags[2] = 0;
        tc::mbar_fence_init();
    }
    if (warp == 2) tc::tmem_alloc(tslot, L::NCOLS);
    tc::tc_fence_before_sync();
    __syncthreads();
    tc::tc_fence_after_sync();
    const uint32_t tmem = *tslot;
    const unsigned long long wait_ns = g_tc_wait_ns;
    if (tid == 0) {
        // steps j = j0 .. j0 + n - 1 of a chunk to a stage: slices j of A (ascending) and D - j of B
        // (1-based; copied ascending, so step i of the stage finds its slice of B at place n - 1 - i)
        int it = 0, s = 0;
        uint32_t par = 1;
        for (int kc = c0; kc < c1 && !flags[0]; ++kc) {
            const char* pa = As + ((size_t)kc * nrbA + mt) * SL_N * L::A_SL;
            const char* pb = Bs + ((size_t)kc * nrbB + nt) * SL_N * L::B_SL;
            for (int j0 = 1; j0 <= steps; j0 += SL_RUN, ++it) {
                const int n = min(SL_RUN, steps - j0 + 1);
                if (!tc::mbar_wait_ns(&empty[s], par, wait_ns)) {
                    flags[0] = 1;
                    break;
                }
                unsigned char* st = smem + s * L::STAGE;
                tc::mbar_arrive_expect_tx(&full[s], (uint32_t)(n * (L::A_SL + L::B_SL)));
                bulk_load(st, pa + (size_t)(j0 - 1) * L::A_SL, n * L::A_SL, &full[s]);
                bulk_load(st + L::B_OFF, pb + (size_t)(D - j0 - n) * L::B_SL, n * L::B_SL, &full[s]);
                if (++s == SL_STAGES) {
                    s = 0;
                    par ^= 1u;
                }
            }
        }
        flags[1] = it;
    } else if (tid == 32) {
        // One thread issues every product: its loop works on descriptor words, of which only the low one
        // differs from slice to slice (descriptors built anew for each product: 120 x 120 over 27 000 took
        // 203 us a launch, with these words 162).
        constexpr uint32_t idesc = tc::instr_desc(1u, TCX_M, NT);
        constexpr uint32_t idesc_neg = idesc | (1u << 13);  // negate A
        const uint64_t d0 = tc::smem_desc(tc::smem_addr(smem), 128, 256);
        const uint32_t dhi = (uint32_t)(d0 >> 32);
        constexpr uint32_t AI = L::A_PL >> 4, BI = L::B_PL >> 4, AS = L::A_SL >> 4, BS = L::B_SL >> 4, ST = L::STAGE >> 4;
        const uint32_t fullbar = tc::smem_addr(full), emptybar = tc::smem_addr(empty);
        const uint32_t re = tmem, im = tmem + NT, re1 = tmem + 2 * NT, im1 = tmem + 3 * NT;
        uint32_t stage = (uint32_t)d0, prev = 0, s = 0, sp = 0, par = 0, acc = 0, acc1 = 0;
        int it = 0;
        for (int kc = c0; kc < c1 && !flags[0]; ++kc) {
            for (int j0 = 1; j0 <= steps; j0 += SL_RUN, ++it) {
                const int n = min(SL_RUN, steps - j0 + 1);
                if (!sl_wait(fullbar + 8 * s, par, &full[s], wait_ns)) {
                    flags[0] = 1;
                    break;
                }
                tc::tc_fence_after_sync();
                uint32_t a = stage, b = stage + (L::B_OFF >> 4) + (n - 1) * BS;
                for (int i = 0; i < n; ++i, a += AS, b -= BS) {
                    // this step's slice of A into the sum D, the previous one's into D - 1
                    sl_mma(re, a, b, dhi, idesc, acc);
                    sl_mma(im, a, b + BI, dhi, idesc, acc);
                    sl_mma(re, a + AI, b + BI, dhi, CONJ ? idesc : idesc_neg, 1u);
                    sl_mma(im, a + AI, b, dhi, CONJ ? idesc_neg : idesc, 1u);
                    acc = 1u;
                    if (j0 + i > 1) {
                        sl_mma(re1, prev, b, dhi, idesc, acc1);
                        sl_mma(im1, prev, b + BI, dhi, idesc, acc1);
                        sl_mma(re1, prev + AI, b + BI, dhi, CONJ ? idesc : idesc_neg, 1u);
                        sl_mma(im1, prev + AI, b, dhi, CONJ ? idesc_neg : idesc, 1u);
                        acc1 = 1u;
                        // the previous stage's last slice of A has been used twice now
                        if (i == 0) sl_commit(emptybar + 8 * sp);
                    }
                    prev = a;
                }
                if (j0 + SL_RUN > steps) sl_commit(emptybar + 8 * s);  // the chunk's last stage is not needed again
                sp = s;
                if (++s == SL_STAGES) {
                    s = 0;
                    par ^= 1u;
                    stage = (uint32_t)d0;
                } else {
                    stage += ST;
                }
            }
        }
        flags[2] = it;
        if (it == total) tc::mma_commit(accbar);
    }
    __syncthreads();
    const int loaded = flags[1], issued = flags[2];
    int ok = flags[0] == 0 && issued == total;
    if (ok) ok = __syncthreads_and(tc::mbar_wait_ns(accbar, 0u, wait_ns) ? 1 : 0);
    if (!ok) {
        // drain: copies issued but never consumed, and every product issued
        if (tid == 0) {
            for (int it = issued; it < loaded; ++it)
                tc::mbar_wait_ns(&full[it % SL_STAGES], (uint32_t)((it / SL_STAGES) & 1), TC_DRAIN_NS);
        }
        if (tid == 32) {
            if (issued < total) tc::mma_commit(accbar);
            tc::mbar_wait_ns(accbar, 0u, TC_DRAIN_NS);
        }
        __syncthreads();
    }
    tc::tc_fence_after_sync();
    if (ok) {
        int2* P = part + ((size_t)tile * plan.first[SL_GROUPS] + unit) * (size_t)(NT * TCX_M) + warp * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int col = 0; col < NT; col += 16) {
            float a[16], b[16];
            int re[16], im[16];
            tc::tmem_ld16(lane_base + col, a);
            tc::tmem_ld16(lane_base + NT + col, b);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                re[i] = __float2int_rn(a[i]);
                im[i] = __float2int_rn(b[i]);
            }
            if (steps > 1) {
                tc::tmem_ld16(lane_base + 2 * NT + col, a);
                tc::tmem_ld16(lane_base + 3 * NT + col, b);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    // |S_D| <= 2^24 and |S_(D-1)| <= 2^24 (D - 2) / (D - 1): the sum fits 32 bits
                    re[i] += __float2int_rn(a[i]) * (1 << SL_BITS);
                    im[i] += __float2int_rn(b[i]) * (1 << SL_BITS);
                }
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) P[(size_t)(col + i) * TCX_M] = make_int2(re[i], im[i]);
        }
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    if (warp == 2) tc::tmem_dealloc(tmem, L::NCOLS);
    if (!ok && tid == 0) atomicExch(&g_tc_status, (int)JDFT_ERR_TIMEOUT);
}

// ---- sums -------------------------------------------------------------------------
// t 2^q rounded to a double
__device__ __forceinline__ double sl_to_double(__int128 t, int q) {
    const bool neg = t < 0;
    unsigned __int128 a = neg ? (unsigned __int128)(-t) : (unsigned __int128)t;
    const uint64_t h = (uint64_t)(a >> 64);
    const uint64_t l = (uint64_t)a;
    const int drop = h ? 64 - __clzll((long long)h) + 2 : (l >> 62) ? 2 : 0;  // to at most 62 bits
    uint64_t m = (uint64_t)(a >> drop);
    if (a != ((unsigned __int128)m << drop)) m |= 1;          // sticky: the rounding below sees what was dropped
    const int qq = q + drop, qc = min(max(qq, -1018), 960);
    double x = fix_decode(neg ? -(i64)m : (i64)m, qc);
    if (qc != qq) x *= __hiloint2double((1023 + min(max(qq - qc, -1022), 1023)) << 20, 0);
    return x;
}

// Block (columns j .. of a tile): thread (row r, q) sums units q, q + RZ, ... of
// its output with 64-bit integers per group, the RZ sums meet in 128 bits.
// out[m * sm + n * sn] (+)= scale * sum.
template <int RZ>
__global__ void __launch_bounds__(TCX_M* RZ)
    sl_reduce_kernel(const int2* __restrict__ part, SlPlan plan, int NT, int mtiles, int M, int N,
                     const int* __restrict__ exA, const int* __restrict__ exB, double2* __restrict__ out, size_t sm,
                     size_t sn, double scale, int accumulate) {
    __shared__ longlong2 sum[RZ > 1 ? RZ : 1][2][RZ > 1 ? TCX_M : 1];
    const int r = threadIdx.x, q = threadIdx.y;
    const int col = blockIdx.x, tile = blockIdx.y;
    const int m = (tile % mtiles) * TCX_M + r, n = (tile / mtiles) * NT + col;
    if (n >= N) return;  // the whole block
    const int units = plan.first[SL_GROUPS];
    const size_t ustride = (size_t)NT * TCX_M;
    const int2* p = part + (size_t)tile * units * ustride + (size_t)col * TCX_M + r;
    __int128 re = 0, im = 0;
#pragma unroll
    for (int g = 0; g < SL_GROUPS; ++g) {
        i64 x = 0, y = 0;
        for (int u = plan.first[g] + q; u < plan.first[g + 1]; u += RZ) {
            const int2 v = p[(size_t)u * ustride];
            x += v.x;
            y += v.y;
        }
        re += (__int128)x << (2 * SL_BITS * g);
        im += (__int128)y << (2 * SL_BITS * g);
    }
    if constexpr (RZ > 1) {
        sum[q][0][r] = make_longlong2((i64)(uint64_t)re, (i64)(re >> 64));
        sum[q][1][r] = make_longlong2((i64)(uint64_t)im, (i64)(im >> 64));
        __syncthreads();
        if (q > 0) return;
        re = 0;
        im = 0;
#pragma unroll
        for (int i = 0; i < RZ; ++i) {
            const longlong2 a = sum[i][0][r], b = sum[i][1][r];
            re += ((__int128)a.y << 64) | (unsigned __int128)(uint64_t)a.x;
            im += ((__int128)b.y << 64) | (unsigned __int128)(uint64_t)b.x;
        }
    }
    if (m >= M) return;
    // a slice's last digit is worth 2^(exponent - 1083) of its row, the sums are in units of 2^56 of their product
    const int eA = exA[m], eB = exB[n];
    const int w = (eA - SL_BIAS - 1083) + (eB - SL_BIAS - 1083) + 56;
    double2 v = make_double2(scale * sl_to_double(re, w), scale * sl_to_double(im, w));
    if (eA == SL_BAD || eB == SL_BAD) v.x = v.y = __hiloint2double(0x7ff80000, 0);
    double2* o = out + (size_t)m * sm + (size_t)n * sn;
    if (accumulate) {
        const double2 old = *o;
        v.x += old.x;
        v.y += old.y;
    }
    *o = v;
}

// ---- host ---------------------------------------------------------------------------
// Units of the largest size the sums allow, or up to four times smaller: the
// choice whose waves of blocks, each as long as its largest unit, end first.
static SlPlan sl_plan(int nkc, int tiles) {
    constexpr int kOverhead = 180;  // of a unit, in products: barriers, tensor memory, the integers out
    SlPlan best{};
    int64_t best_cost = -1;
    for (int f = 16; f >= 4; --f) {
        SlPlan p;
        p.first[0] = 0;
        int64_t longest = 0;
        for (int g = 0; g < SL_GROUPS; ++g) {
            const int top = std::max(1, std::min(sl_limit(g), nkc) * f / 16);
            const int n = (nkc + top - 1) / top;
            p.per[g] = (nkc + n - 1) / n;
            p.first[g + 1] = p.first[g] + (nkc + p.per[g] - 1) / p.per[g];
            longest = std::max<int64_t>(longest, (int64_t)p.per[g] * 4 * (2 * sl_top(g) - 3));
        }
        const int64_t waves = ((int64_t)p.first[SL_GROUPS] * tiles + 151) / 152;
        const int64_t cost = waves * (longest + kOverhead);
        if (best_cost < 0 || cost < best_cost) {
            best = p;
            best_cost = cost;
        }
    }
    return best;
}
static int sl_units_max(int nkc, int tiles) { return sl_plan(nkc, tiles).first[SL_GROUPS]; }
static int sl_nt(int N) { return N <= 32 ? 32 : N <= 64 ? 64 : 128; }
static size_t sl_align(size_t b) { return (b + 255) / 256 * 256; }
static size_t sl_block_bytes(int rows_pad, int K) {
    return sl_align((size_t)rows_pad * tcx_chunks(K) * TCX_KC * SL_PLANES * 2);
}

// Scratch budget of a product: larger ones run in panels (of K for conj(A) B, of
// output rows for A B).
constexpr size_t SL_BUDGET = size_t(1) << 30;

// Whether the slices are the faster way: estimated times of both (microseconds).
// Slices: 54 for the launches, reading both operands twice and writing their padded
// slices at 3.5 TB/s, and per tile of 128 rows 3.6 ns a K and, for five blocks' start
// and end, 4 us on each of 152 SMs.  CUDA cores: 10 for the launch and 8 flops a padded
// output and K at 1 TFLOP/s.  Measured (conj(A) B of 4 259 plane waves, CUDA cores /
// slices): 32 x 32 50 / 67, 40 x 40 108 / 67; of 19 778: 16 x 16 53 / 154, 32 x 32
// 165 / 160; H C with 128 projectors on 4 259: 16 bands 193 / 225, 32 bands 364 / 274.
bool sl_eligible(int M, int N, int K) {
    const int NT = sl_nt(N), ntiles = (N + NT - 1) / NT;
    const double m = tcx_rows_pad(M), n = (double)ntiles * NT, k = K, tiles = m / TCX_M * ntiles;
    const double slices = 54.0 + (36.0 * (m + n) + 32.0 * ((double)M + N)) * k / 3.5e6 +
                          tiles * (3.6e-3 * k + 5 * 4.0 / 152);
    const double M16 = (M + 15) / 16 * 16, N16 = (N + 15) / 16 * 16;
    return slices < 10.0 + 8.0 * M16 * N16 * k / 1.0e6;
}

template <int NT, bool CONJ>
static jdft_status sl_launch_nt(const void* As, const void* Bs, int nrbA, int nrbB, int nkc, int mtiles, int tiles,
                                const SlPlan& plan, int2* part, cudaStream_t st) {
    auto kern = sl_mma_kernel<NT, CONJ>;
    cudaError_t e = set_smem_attr((const void*)kern, SlLayout<NT>::SMEM);
    if (e != cudaSuccess) return set_error(JDFT_ERR_CUDA, std::string("sl_mma: ") + cudaGetErrorString(e));
    {
        Trace tr_("sl_mma", st);
        kern<<<dim3(plan.first[SL_GROUPS], tiles), SL_THREADS, SlLayout<NT>::SMEM, st>>>(
            (const char*)As, (const char*)Bs, nrbA, nrbB, nkc, mtiles, plan, part);
    }
    return check_launch("sl_mma");
}

template <bool CONJ>
static jdft_status sl_product(const void* As, const void* Bs, int M, int N, int NT, int nkc, const int* exA,
                              const int* exB, void* partial, double2* out, size_t sm, size_t sn, double scale,
                              bool accumulate, cudaStream_t st) {
    const int mtiles = tcx_rows_pad(M) / TCX_M, ntiles = (N + NT - 1) / NT, tiles = mtiles * ntiles;
    const SlPlan plan = sl_plan(nkc, tiles);
    int2* part = (int2*)partial;
    jdft_status s;
    if (NT == 32) s = sl_launch_nt<32, CONJ>(As, Bs, mtiles, ntiles, nkc, mtiles, tiles, plan, part, st);
    else if (NT == 64) s = sl_launch_nt<64, CONJ>(As, Bs, mtiles, ntiles, nkc, mtiles, tiles, plan, part, st);
    else s = sl_launch_nt<128, CONJ>(As, Bs, mtiles, ntiles, nkc, mtiles, tiles, plan, part, st);
    if (s != JDFT_OK) return s;
    {
        Trace tr_("sl_reduce", st);
        const dim3 grid(std::min(NT, N), tiles);
        if (plan.first[SL_GROUPS] > 24)
            sl_reduce_kernel<8><<<grid, dim3(TCX_M, 8), 0, st>>>(part, plan, NT, mtiles, M, N, exA, exB, out, sm, sn,
                                                                 scale, accumulate);
        else
            sl_reduce_kernel<1><<<grid, dim3(TCX_M, 1), 0, st>>>(part, plan, NT, mtiles, M, N, exA, exB, out, sm, sn,
                                                                 scale, accumulate);
    }
    return check_launch("sl_reduce");
}

// Exponents of an operand's rows (K values a row; trans: X[k * ld + r]).
static jdft_status sl_exponents(const double2* X, size_t ld, int rows, int K, bool trans, const int* shift, int sign,
                                int* ex, cudaStream_t st, bool finite = false) {
    JDFT_CUDA_TRY(cudaMemsetAsync(ex, 0, (size_t)rows * sizeof(int), st));
    Trace tr_("sl_rowmax", st);
    if (trans) {
        const int bx = (rows + 255) / 256;
        sl_rowmax_t_kernel<<<dim3(bx, std::max(1, std::min(K, 152 * 8 / bx))), 256, 0, st>>>(X, ld, rows, K, shift,
                                                                                            sign, ex);
    } else {
        const dim3 grid(rows, std::max(1, std::min((K + 1023) / 1024, 152 * 8 / rows)));
        if (finite) sl_rowmax_kernel<true><<<grid, 256, 0, st>>>(X, ld, K, shift, sign, ex);
        else sl_rowmax_kernel<false><<<grid, 256, 0, st>>>(X, ld, K, shift, sign, ex);
    }
    return check_launch("sl_rowmax");
}

// Slices of an operand from its rows' exponents, its rows padded to blocks of RB.
static jdft_status sl_slice(const double2* X, size_t ld, int rows, int RB, int K, bool trans, const int* shift,
                            int sign, const int* ex, void* slices, cudaStream_t st) {
    const int nkc = tcx_chunks(K), rows_pad = (rows + RB - 1) / RB * RB;
    const int64_t total = (int64_t)rows_pad * 2 * nkc;
    const int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
    Trace tr_("sl_slice", st);
    if (trans)
        sl_slice_kernel<true><<<grid, 256, 0, st>>>(X, ld, rows, K, rows_pad, RB, nkc, ex, shift, sign,
                                                    (__nv_bfloat16*)slices);
    else
        sl_slice_kernel<false><<<grid, 256, 0, st>>>(X, ld, rows, K, rows_pad, RB, nkc, ex, shift, sign,
                                                     (__nv_bfloat16*)slices);
    return check_launch("sl_slice");
}

jdft_status sl_zgemm_cn(int M, int N, int K, const double2* A, int lda, const double2* B, int ldb, double2* out,
                        int ldo, double scale, ProductScratch& scratch, cudaStream_t st) {
    const int NT = sl_nt(N);
    const bool same = A == B && lda == ldb && M == N && NT == TCX_M;  // one set of slices
    const int rpA = tcx_rows_pad(M), rpB = (N + NT - 1) / NT * NT;
    const int tiles = rpA / TCX_M * ((N + NT - 1) / NT);
    const size_t mx = sl_align((size_t)(M + N) * sizeof(int));
    auto bytes = [&](int k) {
        return mx + sl_block_bytes(rpA, k) + (same ? 0 : sl_block_bytes(rpB, k)) +
               sl_align((size_t)tiles * sl_units_max(tcx_chunks(k), tiles) * NT * TCX_M * sizeof(int2));
    };
    int kp = K;
    while (kp > 2048 && bytes(kp) > SL_BUDGET) kp = (kp / 2 + TCX_KC - 1) / TCX_KC * TCX_KC;
    void* ws = scratch.get(std::max(bytes(kp), K % kp ? bytes(K % kp) : 0));
    if (!ws) return JDFT_ERR_UNSUPPORTED;
    jdft_status s;
    int* exA = (int*)ws;
    int* exB = same ? exA : exA + M;
    for (int k0 = 0; k0 < K; k0 += kp) {
        const int k = std::min(kp, K - k0);
        char* As = (char*)ws + mx;
        char* Bs = same ? As : As + sl_block_bytes(rpA, k);
        char* part = Bs + sl_block_bytes(rpB, k);
        if ((s = sl_exponents(A + k0, lda, M, k, false, nullptr, 0, exA, st))) return s;
        if ((s = sl_slice(A + k0, lda, M, TCX_M, k, false, nullptr, 0, exA, As, st))) return s;
        if (!same) {
            if ((s = sl_exponents(B + k0, ldb, N, k, false, nullptr, 0, exB, st))) return s;
            if ((s = sl_slice(B + k0, ldb, N, NT, k, false, nullptr, 0, exB, Bs, st))) return s;
        }
        if ((s = sl_product<true>(As, Bs, M, N, NT, tcx_chunks(k), exA, exB, part, out, ldo, 1, scale, true, st)))
            return s;
    }
    return JDFT_OK;
}

// The summed index is scaled first: column k of A by 2^-s_k and row k of B by 2^s_k, s_k the
// exponent of the column's largest value (exponents only, so exact).  A row of A is one plane
// wave over all bands or projectors, and their norms may be anything: cut against the largest
// of them, a small band's coefficients would lose the bits that its large entries of B bring
// back (bands with norms spread over 1e12, rotated by L^-dag, came out orthonormal to 7e-7).
// Scaled, the columns of A are alike, and each column of the output is off by 2^-60 of its own
// largest contributions, whatever the scales.  It costs one more reading of A.
jdft_status sl_zgemm_nn(int M, int N, int K, const double2* A, int lda, const double2* Bm, int ldb, double2* out,
                        int ldo, bool accumulate, ProductScratch& scratch, cudaStream_t st) {
    const int NT = sl_nt(N);
    const int rpB = (N + NT - 1) / NT * NT;
    const int nkc = tcx_chunks(K);
    const size_t head = sl_align((size_t)(M + N + K) * sizeof(int));  // exponents
    auto bytes = [&](int m) {
        const int rpA = tcx_rows_pad(m), tiles = rpA / TCX_M * (rpB / NT);
        return head + sl_block_bytes(rpA, K) + sl_block_bytes(rpB, K) +
               sl_align((size_t)tiles * sl_units_max(nkc, tiles) * NT * TCX_M * sizeof(int2));
    };
    int mp = M;
    while (mp > 4096 && bytes(mp) > SL_BUDGET) mp = (mp / 2 + TCX_M - 1) / TCX_M * TCX_M;
    // smaller panels cut K finer: the last panel may need as much as a full one
    const int last = M % mp;
    void* ws = scratch.get(std::max(bytes(mp), last ? bytes(last) : 0));
    if (!ws) return JDFT_ERR_UNSUPPORTED;
    jdft_status s;
    int* shift = (int*)ws;
    int* exB = shift + K;
    int* exA = exB + N;
    char* Bs = (char*)ws + head;
    char* As = Bs + sl_block_bytes(rpB, K);
    if ((s = sl_exponents(A, lda, K, M, false, nullptr, 0, shift, st, true))) return s;
    if ((s = sl_exponents(Bm, ldb, N, K, true, shift, +1, exB, st))) return s;
    if ((s = sl_slice(Bm, ldb, N, NT, K, true, shift, +1, exB, Bs, st))) return s;
    for (int m0 = 0; m0 < M; m0 += mp) {
        const int m = std::min(mp, M - m0);
        char* part = As + sl_block_bytes(tcx_rows_pad(m), K);
        if ((s = sl_exponents(A + m0, lda, m, K, true, shift, -1, exA, st))) return s;
        if ((s = sl_slice(A + m0, lda, m, TCX_M, K, true, shift, -1, exA, As, st))) return s;
        if ((s = sl_product<false>(As, Bs, m, N, NT, nkc, exA, exB, part, out + m0, 1, ldo, 1.0, accumulate, st)))
            return s;
    }
    return JDFT_OK;
}

}  // namespace jdft
