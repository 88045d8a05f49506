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
// taken out as an integer.
//
// What is dropped: a row's largest component becomes an integer of 2^60 to 2^61 and all of
// them are cut toward zero to integers, 2^-58 of the product of the two rows' largest at
// worst for each real product; the digit pairs beyond 10 are up to 8 2^12 2^49 = 2^64 of
// its 2^120 or more, 2^-56.  Both have either sign, and over the block shapes here the
// results are nearer to extended precision than the FP64 sums they replace.  But the bound
// is relative to the rows' maxima, not to the sum of the terms' absolute values as in FP64:
// sl_zgemm_cn and sl_zgemm_nn scale the summed index where that would show.
//
// Launches: row exponents, slices (36 bytes a complex value) of both operands, the
// products, and the sum of the blocks' integers (128 bits) into the FP64 output; for A B
// the exponents of A's columns first, for conj(A) B of two operands a look at the columns
// of the largest values (and a reading of both operands and two more launches, which return
// at once in ordinary products).
// A unit of work (block) is a 128 x NT output tile, a pair of digit sums (D, D - 1)
// and a range of K: at step j it adds A_j B_(D-j) to the first and
// A_(j-1) B_(D-j) to the second accumulator, so each slice is staged once for
// two products; three steps share a stage, copied by one bulk copy per operand.
// Tensor memory holds 2 x 2 x NT columns.
//
// Measured (event times, against the CUDA-core products): overlap, subspace matrix
// and rotation of 120 bands of 27 000 plane waves 19.86 -> 1.33 ms, error against
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
// Cut against the rows as they are, an entry is off by about 2^-61 |a| |b| of its rows' norms, FP64 sums by 2^-53
// of their terms: equal where the terms are 2^-8 of the product of the rows' maxima.  Scaled from 2^-4 down.
constexpr int SL_NEAR = 2 * SL_BIAS - 4;
__host__ __device__ constexpr int sl_top(int g) { return 10 - 2 * g; }              // larger digit sum of group g
__host__ __device__ constexpr int sl_limit(int g) { return 2048 / (sl_top(g) - 1) / TCX_KC; }  // K chunks per unit

// How the K range is cut per group: per[g] chunks to a unit, first[g] the
// group's first unit (first[SL_GROUPS]: units in all).
struct SlPlan {
    int per[SL_GROUPS];
    int first[SL_GROUPS + 1];
};

// ---- exponents of the rows ------------------------------------------------------
// Exponents are exponent fields (1 for zeros and denormals, whose significands have no
// implicit bit) plus SL_BIAS, so that 0 means none.  The summed index may be scaled first:
// value k of one operand counts as 2^-s_k and of the other as 2^s_k times itself, with
// shift[k] = s_k + SL_BIAS.
struct SlScale {
    const int* shift;  // null: no scaling
    const int* near;   // null: scale; else only where the word is below SL_NEAR (see sl_balance_kernel)
    __device__ __forceinline__ bool on() const { return shift && (!near || *near < SL_NEAR); }
};
// An operand's rows: exponents, and where the index is scaled those of the scaled rows.
struct SlRows {
    const int *ex, *scaled;  // scaled null: ex are the scaled rows' already
    SlScale scale;
    int sign;  // of s_k
    __device__ __forceinline__ const int* pick(bool on) const { return on && scaled ? scaled : ex; }
};
__device__ __forceinline__ int sl_field(int hi) { return max((hi >> 20) & 0x7ff, 1); }
// The exponent that a row holding v has at least: SL_BAD for an infinity or NaN.
__device__ __forceinline__ int sl_exponent(double2 v, int shift) {
    const int x = __double2hiint(v.x) & 0x7fffffff, y = __double2hiint(v.y) & 0x7fffffff, hi = max(x, y);
    if ((hi >> 20) == 0x7ff) return SL_BAD;
    return (hi | __double2loint(v.x) | __double2loint(v.y)) == 0 ? 0 : sl_field(hi) + shift + SL_BIAS;
}

// ex[r] = largest exponent over the K values of row r: first A's rows, then B's (signs -1
// and +1 of the shift).  FINITE: of the values without an infinity or NaN.  at (or null):
// the exponent and the place of such a value, as one word.
template <bool FINITE>
__global__ void __launch_bounds__(256) sl_rowmax_kernel(const double2* __restrict__ A, size_t lda, int rowsA,
                                                        const double2* __restrict__ B, size_t ldb, int K, SlScale sc,
                                                        int* __restrict__ ex, unsigned long long* __restrict__ at) {
    const bool on = sc.on();
    if (sc.shift && !on) return;
    const int r = blockIdx.x;
    const double2* x = r < rowsA ? A + (size_t)r * lda : B + (size_t)(r - rowsA) * ldb;
    const int sign = r < rowsA ? -1 : 1;
    int m = 0, place = 0;
    for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < K; k += gridDim.y * blockDim.x) {
        const int e = sl_exponent(x[k], on ? sign * (sc.shift[k] - SL_BIAS) : 0);
        if (e > m && (!FINITE || e != SL_BAD)) {
            m = e;
            place = k;
        }
    }
    const int top = __reduce_max_sync(0xffffffffu, m);
    const unsigned who = __ballot_sync(0xffffffffu, m == top);
    if ((threadIdx.x & 31) == __ffs(who) - 1) {
        atomicMax(&ex[r], top);
        if (at) atomicMax(&at[r], (unsigned long long)top << 32 | (unsigned)place);
    }
}
// The same of a transpose: row r, value k at X[k * ld + r]; blockIdx.y strides over k.
__global__ void __launch_bounds__(256) sl_rowmax_t_kernel(const double2* __restrict__ X, size_t ld, int rows, int K,
                                                          const int* __restrict__ shift, int sign,
                                                          int* __restrict__ ex) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    int m = 0;
    for (int k = blockIdx.y; k < K; k += gridDim.y)
        m = max(m, sl_exponent(X[(size_t)k * ld + r], sign * (shift[k] - SL_BIAS)));
    atomicMax(&ex[r], m);
}

// The scaling of the summed index of conj(A) B: s_k half the difference of the columns'
// largest exponents a_k and b_k, each value's taken relative to its row's.  Scaled, value k
// of a row is at most 2^((a_k + b_k) / 2) of the row's largest, so max (a_k + b_k), kept
// in *near (plus 2 SL_BIAS), is what the scaling gains over cutting the rows as they are.
// sl_near_kernel looks at the columns of the rows' largest values first: in an ordinary
// product one of them holds a large value of the other operand too, and nothing else is
// read (H C of 64 bands with 256 projectors on 62 759 plane waves: 6 237 us with both operands
// read a second time, 6 190 so).  One warp a row.
__global__ void __launch_bounds__(256) sl_near_kernel(const double2* __restrict__ A, size_t lda, int rowsA,
                                                      const double2* __restrict__ B, size_t ldb, int rowsB,
                                                      const int* __restrict__ ex,
                                                      const unsigned long long* __restrict__ at,
                                                      int* __restrict__ near) {
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= rowsA + rowsB || ex[r] == 0 || ex[r] == SL_BAD) return;
    const bool ofA = r < rowsA;
    const double2* x = (ofA ? B : A) + (unsigned)at[r];
    const size_t ld = ofA ? ldb : lda;
    const int* e = ex + (ofA ? rowsA : 0);
    int g = 0;
    for (int n = lane; n < (ofA ? rowsB : rowsA); n += 32) {
        const int v = sl_exponent(x[n * ld], 0);
        if (v != 0 && e[n] != SL_BAD) g = max(g, v - e[n] + 2 * SL_BIAS);
    }
    g = __reduce_max_sync(0xffffffffu, g);
    if (lane == 0) atomicMax(near, g);
}
// 32 columns a block, its warps sharing the rows.
__global__ void __launch_bounds__(256) sl_balance_kernel(const double2* __restrict__ A, size_t lda, int rowsA,
                                                         const double2* __restrict__ B, size_t ldb, int rowsB, int K,
                                                         const int* __restrict__ ex, int* __restrict__ shift,
                                                         int* __restrict__ near) {
    __shared__ int top[2][8][32];
    constexpr int kNone = -(1 << 24);
    // the word rises while blocks run: the block decides as one
    if (__syncthreads_or(*(volatile const int*)near >= SL_NEAR)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = blockIdx.x * 32 + lane;
    int m[2] = {kNone, kNone};
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        const double2* x = (o ? B : A) + k;
        const size_t ld = o ? ldb : lda;
        const int rows = k < K ? (o ? rowsB : rowsA) : 0;
        const int* e = ex + (o ? rowsA : 0);
#pragma unroll 4
        for (int r = warp; r < rows; r += 8) {
            const int v = sl_exponent(x[r * ld], 0), row = e[r];
            if (v != 0 && row != SL_BAD) m[o] = max(m[o], v - row);
        }
        top[o][warp][lane] = m[o];
    }
    __syncthreads();
    if (warp) return;
#pragma unroll
    for (int w = 1; w < 8; ++w) {
        m[0] = max(m[0], top[0][w][lane]);
        m[1] = max(m[1], top[1][w][lane]);
    }
    const bool both = m[0] > kNone && m[1] > kNone;
    if (k < K) shift[k] = (both ? (m[0] - m[1]) >> 1 : 0) + SL_BIAS;
    int g = both ? m[0] + m[1] + 2 * SL_BIAS : 0;
    for (int o = 16; o > 0; o >>= 1) g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
    if (lane == 0) atomicMax(near, g);
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
                                                       int rows_pad, int RB, int nkc, SlRows sr,
                                                       __nv_bfloat16* __restrict__ out) {
    const bool on = sr.scale.on();
    const int* __restrict__ ex = sr.pick(on);
    const int* __restrict__ shift = sr.scale.shift;
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
                if (on) sh = sr.sign * (shift[k0 + j] - SL_BIAS);
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
// part: [tile - tile0][unit][column][row] of (Re, Im) integers, S_D + 2^7 S_(D-1).
template <int NT, bool CONJ>
__global__ void __launch_bounds__(SL_THREADS, 1)
    sl_mma_kernel(const char* __restrict__ As, const char* __restrict__ Bs, int nrbA, int nrbB, int nkc, int mtiles,
                  int tile0, SlPlan plan, int2* __restrict__ part, int* __restrict__ gave_up) {
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
    const int mt = (tile0 + tile) % mtiles, nt = (tile0 + tile) / mtiles;
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
    if (!ok && tid == 0) {
        // the block's part holds whatever was there before: the sums below must not use it
        atomicExch(gave_up, 1);
        atomicExch(&g_tc_status, (int)JDFT_ERR_TIMEOUT);
    }
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
// out[m * sm + n * sn] (+)= scale * sum, NaN where a block of the product gave up, which
// *failed (or null) then says as well.
template <int RZ>
__global__ void __launch_bounds__(TCX_M* RZ)
    sl_reduce_kernel(const int2* __restrict__ part, SlPlan plan, int NT, int mtiles, int tile0, int M, int N,
                     SlRows ra, SlRows rb, double2* __restrict__ out, size_t sm,
                     size_t sn, double scale, int accumulate, const int* __restrict__ gave_up,
                     int* __restrict__ failed) {
    __shared__ longlong2 sum[RZ > 1 ? RZ : 1][2][RZ > 1 ? TCX_M : 1];
    const int r = threadIdx.x, q = threadIdx.y;
    const int col = blockIdx.x, tile = blockIdx.y;
    const int m = ((tile0 + tile) % mtiles) * TCX_M + r, n = ((tile0 + tile) / mtiles) * NT + col;
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
    const bool on = ra.scale.on();
    const int eA = ra.pick(on)[m], eB = rb.pick(on)[n];
    const int w = (eA - SL_BIAS - 1083) + (eB - SL_BIAS - 1083) + 56;
    double2 v = make_double2(scale * sl_to_double(re, w), scale * sl_to_double(im, w));
    const bool incomplete = *gave_up != 0;
    if (eA == SL_BAD || eB == SL_BAD || incomplete) v.x = v.y = __hiloint2double(0x7ff80000, 0);
    if (incomplete && failed && m + n == 0) *failed = (int)JDFT_ERR_TIMEOUT;
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

// Scratch of a product is at most SL_BUDGET (the largest that ProductScratch grows to of
// itself): larger ones run in panels, of K for conj(A) B and of output rows and columns for
// A B, and in groups of output tiles.
constexpr size_t SL_BUDGET = ProductScratch::kMost;
// Partial sums of `group` tiles.
static size_t sl_partial_bytes(int nkc, int group, int NT) {
    return sl_align((size_t)group * sl_units_max(nkc, group) * NT * TCX_M * sizeof(int2));
}
// The largest group of `tiles` whose partial sums fit, by halving (0: none).
static int sl_group(int nkc, int tiles, int NT, size_t room) {
    int g = tiles;
    while (g > 1 && sl_partial_bytes(nkc, g, NT) > room) g = (g + 1) / 2;
    return sl_partial_bytes(nkc, g, NT) <= room ? g : 0;
}

// Whether the slices are the faster way: estimated times of both (microseconds).
// Slices: 54 for the launches, reading both operands twice (three times for A of A B) and
// writing their padded slices at 3.5 TB/s, and per tile of 128 rows 3.6 ns a K and, for five blocks' start
// and end, 4 us on each of 152 SMs.  CUDA cores: 10 for the launch and 8 flops a padded
// output and K at 1 TFLOP/s.  Measured (conj(A) B of 4 259 plane waves, CUDA cores /
// slices, the mean of one and of two operands): 32 x 32 51 / 69, 40 x 40 109 / 69; of
// 19 778: 16 x 16 52 / 152, 32 x 32 166 / 161; H C with 128 projectors on 4 259: 16 bands
// 193 / 240, 32 bands 364 / 288.
bool sl_eligible(int M, int N, int K) {
    const int NT = sl_nt(N), ntiles = (N + NT - 1) / NT;
    const double m = tcx_rows_pad(M), n = (double)ntiles * NT, k = K, tiles = m / TCX_M * ntiles;
    const double slices = 54.0 + (36.0 * (m + n) + 32.0 * ((double)M + N)) * k / 3.5e6 +
                          tiles * (3.6e-3 * k + 5 * 4.0 / 152);
    const double M16 = (M + 15) / 16 * 16, N16 = (N + 15) / 16 * 16;
    return slices < 10.0 + 8.0 * M16 * N16 * k / 1.0e6;
}

template <int NT, bool CONJ>
static jdft_status sl_launch_nt(const void* As, const void* Bs, int nrbA, int nrbB, int nkc, int mtiles, int tile0,
                                int tiles, const SlPlan& plan, int2* part, int* gave_up, cudaStream_t st) {
    auto kern = sl_mma_kernel<NT, CONJ>;
    cudaError_t e = set_smem_attr((const void*)kern, SlLayout<NT>::SMEM);
    if (e != cudaSuccess) return set_error(JDFT_ERR_CUDA, std::string("sl_mma: ") + cudaGetErrorString(e));
    {
        Trace tr_("sl_mma", st);
        kern<<<dim3(plan.first[SL_GROUPS], tiles), SL_THREADS, SlLayout<NT>::SMEM, st>>>(
            (const char*)As, (const char*)Bs, nrbA, nrbB, nkc, mtiles, tile0, plan, part, gave_up);
    }
    return check_launch("sl_mma");
}

// `group` output tiles at a time, as many as the partial sums have room for.
template <bool CONJ>
static jdft_status sl_product(const void* As, const void* Bs, int M, int N, int NT, int nkc, int group, const SlRows& ra,
                              const SlRows& rb, void* partial, double2* out, size_t sm, size_t sn, double scale,
                              bool accumulate, int* gave_up, int* failed, cudaStream_t st) {
    const int mtiles = tcx_rows_pad(M) / TCX_M, ntiles = (N + NT - 1) / NT, all = mtiles * ntiles;
    int2* part = (int2*)partial;
    for (int t0 = 0; t0 < all; t0 += group) {
        const int tiles = std::min(group, all - t0);
        const SlPlan plan = sl_plan(nkc, group);
        jdft_status s;
        if (NT == 32)
            s = sl_launch_nt<32, CONJ>(As, Bs, mtiles, ntiles, nkc, mtiles, t0, tiles, plan, part, gave_up, st);
        else if (NT == 64)
            s = sl_launch_nt<64, CONJ>(As, Bs, mtiles, ntiles, nkc, mtiles, t0, tiles, plan, part, gave_up, st);
        else
            s = sl_launch_nt<128, CONJ>(As, Bs, mtiles, ntiles, nkc, mtiles, t0, tiles, plan, part, gave_up, st);
        if (s != JDFT_OK) return s;
        {
            Trace tr_("sl_reduce", st);
            const dim3 grid(std::min(NT, N), tiles);
            if (plan.first[SL_GROUPS] > 24)
                sl_reduce_kernel<8><<<grid, dim3(TCX_M, 8), 0, st>>>(part, plan, NT, mtiles, t0, M, N, ra, rb, out, sm,
                                                                     sn, scale, accumulate, gave_up, failed);
            else
                sl_reduce_kernel<1><<<grid, dim3(TCX_M, 1), 0, st>>>(part, plan, NT, mtiles, t0, M, N, ra, rb, out, sm,
                                                                     sn, scale, accumulate, gave_up, failed);
        }
        if ((s = check_launch("sl_reduce"))) return s;
    }
    return JDFT_OK;
}

// Exponents of an operand's rows (K values a row) into ex, zeroed before; `finite` and sc as in the kernel.
static jdft_status sl_exponents(const double2* A, size_t lda, int rowsA, const double2* B, size_t ldb, int rowsB, int K,
                                SlScale sc, int* ex, cudaStream_t st, bool finite = false,
                                unsigned long long* at = nullptr) {
    const int rows = rowsA + rowsB;
    const dim3 grid(rows, std::max(1, std::min((K + 1023) / 1024, 152 * 8 / rows)));
    Trace tr_("sl_rowmax", st);
    if (finite) sl_rowmax_kernel<true><<<grid, 256, 0, st>>>(A, lda, rowsA, B, ldb, K, sc, ex, at);
    else sl_rowmax_kernel<false><<<grid, 256, 0, st>>>(A, lda, rowsA, B, ldb, K, sc, ex, at);
    return check_launch("sl_rowmax");
}
static jdft_status sl_exponents_t(const double2* X, size_t ld, int rows, int K, const int* shift, int sign, int* ex,
                                  cudaStream_t st) {
    const int bx = (rows + 255) / 256;
    Trace tr_("sl_rowmax", st);
    sl_rowmax_t_kernel<<<dim3(bx, std::max(1, std::min(K, 152 * 8 / bx))), 256, 0, st>>>(X, ld, rows, K, shift, sign,
                                                                                        ex);
    return check_launch("sl_rowmax");
}

// Slices of an operand (trans: X[k * ld + r]) from its rows' exponents, its rows padded to blocks of RB.
static jdft_status sl_slice(const double2* X, size_t ld, int rows, int RB, int K, bool trans, const SlRows& sr,
                            void* slices, cudaStream_t st) {
    const int nkc = tcx_chunks(K), rows_pad = (rows + RB - 1) / RB * RB;
    const int64_t total = (int64_t)rows_pad * 2 * nkc;
    const int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
    Trace tr_("sl_slice", st);
    if (trans)
        sl_slice_kernel<true><<<grid, 256, 0, st>>>(X, ld, rows, K, rows_pad, RB, nkc, sr, (__nv_bfloat16*)slices);
    else
        sl_slice_kernel<false><<<grid, 256, 0, st>>>(X, ld, rows, K, rows_pad, RB, nkc, sr, (__nv_bfloat16*)slices);
    return check_launch("sl_slice");
}

// Rows are cut against their own largest value, so the error of an entry is relative to the
// product of the two rows' norms, as that of FP64 sums is where the rows' large values meet.
// Where they do not (C falling and H C rising over the plane waves: the products of the
// terms are far below the product of the rows' maxima), the summed index is scaled first
// (sl_balance_kernel).  One product C^dag C needs none: its operands are alike.
jdft_status sl_zgemm_cn(int M, int N, int K, const double2* A, int lda, const double2* B, int ldb, double2* out,
                        int ldo, double scale, ProductScratch& scratch, cudaStream_t st) {
    const int NT = sl_nt(N);
    const bool twin = A == B && lda == ldb && M == N;
    const bool same = twin && NT == TCX_M;  // one set of slices
    const int rpA = tcx_rows_pad(M), rpB = (N + NT - 1) / NT * NT;
    const int tiles = rpA / TCX_M * ((N + NT - 1) / NT);
    // places of the rows' largest values, exponents of the rows, of the scaled rows, whether a block gave up, the
    // gain, the shifts
    const int rows = M + N, words = 2 * rows + (twin ? 0 : 2 * rows + 1) + 1;
    const size_t head = sl_align(((size_t)words + (twin ? 0 : K)) * sizeof(int));
    auto slices = [&](int k) { return head + sl_block_bytes(rpA, k) + (same ? 0 : sl_block_bytes(rpB, k)); };
    // K panels of which the slices take at most three quarters of the budget, tiles for the rest
    int kp = K, group = 0;
    for (;; kp = (kp / 2 + TCX_KC - 1) / TCX_KC * TCX_KC) {
        const size_t b = slices(kp);
        group = b < SL_BUDGET ? sl_group(tcx_chunks(kp), tiles, NT, SL_BUDGET - b) : 0;
        if (group == tiles || (group && b <= SL_BUDGET / 4 * 3) || kp <= 256) break;
    }
    // (a last panel of fewer chunks may cut them finer)
    auto bytes = [&](int k) { return k ? slices(k) + sl_partial_bytes(tcx_chunks(k), group, NT) : 0; };
    while (group > 1 && bytes(K % kp) > SL_BUDGET) group = (group + 1) / 2;
    void* ws = group ? scratch.get(std::max(bytes(kp), bytes(K % kp)), st) : nullptr;
    if (!ws) return JDFT_ERR_UNSUPPORTED;
    const ScratchUse use{scratch, st};
    jdft_status s;
    unsigned long long* at = twin ? nullptr : (unsigned long long*)ws;
    int* ex = (int*)ws + (twin ? 0 : 2 * rows);
    int *scaled = ex + rows, *gave_up = scaled + rows, *near = gave_up + 1, *shift = near + 1;
    const SlScale none{nullptr, nullptr}, sc = twin ? none : SlScale{shift, near};
    const SlRows ra{ex, twin ? nullptr : scaled, sc, -1};
    const SlRows rb = twin ? ra : SlRows{ex + M, scaled + M, sc, +1};
    for (int k0 = 0; k0 < K; k0 += kp) {
        const int k = std::min(kp, K - k0);
        char* As = (char*)ws + head;
        char* Bs = same ? As : As + sl_block_bytes(rpA, k);
        char* part = Bs + sl_block_bytes(rpB, k);
        JDFT_CUDA_TRY(cudaMemsetAsync(ws, 0, words * sizeof(int), st));
        if ((s = sl_exponents(A + k0, lda, M, B + k0, ldb, twin ? 0 : N, k, none, ex, st, false, at))) return s;
        if (!twin) {
            {
                Trace tr_("sl_balance", st);
                sl_near_kernel<<<(rows + 7) / 8, 256, 0, st>>>(A + k0, lda, M, B + k0, ldb, N, ex, at, near);
                sl_balance_kernel<<<(k + 31) / 32, 256, 0, st>>>(A + k0, lda, M, B + k0, ldb, N, k, ex, shift, near);
            }
            if ((s = check_launch("sl_balance"))) return s;
            if ((s = sl_exponents(A + k0, lda, M, B + k0, ldb, N, k, sc, scaled, st))) return s;
        }
        if ((s = sl_slice(A + k0, lda, M, TCX_M, k, false, ra, As, st))) return s;
        if (!same && (s = sl_slice(B + k0, ldb, N, NT, k, false, rb, Bs, st))) return s;
        if ((s = sl_product<true>(As, Bs, M, N, NT, tcx_chunks(k), group, ra, rb, part, out, ldo, 1, scale, true,
                                   gave_up, scratch.failed, st)))
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
    const int nkc = tcx_chunks(K);
    const size_t head = sl_align((size_t)(M + N + K + 1) * sizeof(int));  // exponents, and whether a block gave up
    auto slices = [&](int m, int n) {
        return head + sl_block_bytes(tcx_rows_pad(m), K) + sl_block_bytes((n + NT - 1) / NT * NT, K);
    };
    auto tiles_of = [&](int m, int n) { return tcx_rows_pad(m) / TCX_M * ((n + NT - 1) / NT); };
    // panels of rows (and, where one row block beside B's slices is too much, of columns) of which the slices take
    // at most three quarters of the budget, tiles for the rest
    int mp = M, np = N, group = 0;
    for (;;) {
        const size_t b = slices(mp, np);
        const int tiles = tiles_of(mp, np);
        group = b < SL_BUDGET ? sl_group(nkc, tiles, NT, SL_BUDGET - b) : 0;
        if (group == tiles || (group && b <= SL_BUDGET / 4 * 3)) break;
        if (mp > 4096 || (mp > TCX_M && np <= NT)) mp = (mp / 2 + TCX_M - 1) / TCX_M * TCX_M;
        else if (np > NT) np = (np / 2 + NT - 1) / NT * NT;
        else break;
    }
    if (!group) return JDFT_ERR_UNSUPPORTED;
    // (a smaller last panel has no more tiles, and its partial sums are laid out by the same plan)
    void* ws = scratch.get(slices(mp, np) + sl_partial_bytes(nkc, group, NT), st);
    if (!ws) return JDFT_ERR_UNSUPPORTED;
    const ScratchUse use{scratch, st};
    jdft_status s;
    int* gave_up = (int*)ws;
    int* shift = gave_up + 1;
    int* exB = shift + K;
    int* exA = exB + N;
    char* As = (char*)ws + head;
    char* Bs = As + sl_block_bytes(tcx_rows_pad(mp), K);
    char* part = Bs + sl_block_bytes((np + NT - 1) / NT * NT, K);
    JDFT_CUDA_TRY(cudaMemsetAsync(ws, 0, head, st));
    const SlScale none{nullptr, nullptr}, sc{shift, nullptr};
    if ((s = sl_exponents(A, lda, K, nullptr, 0, 0, M, none, shift, st, true))) return s;
    if ((s = sl_exponents_t(Bm, ldb, N, K, shift, +1, exB, st))) return s;
    if ((s = sl_exponents_t(A, lda, M, K, shift, -1, exA, st))) return s;
    for (int n0 = 0; n0 < N; n0 += np) {
        const int n = std::min(np, N - n0);
        const SlRows rb{exB + n0, nullptr, sc, +1};
        if ((s = sl_slice(Bm + n0, ldb, n, NT, K, true, rb, Bs, st))) return s;
        for (int m0 = 0; m0 < M; m0 += mp) {
            const int m = std::min(mp, M - m0);
            const SlRows ra{exA + m0, nullptr, sc, -1};
            if ((mp < M || n0 == 0) && (s = sl_slice(A + m0, lda, m, TCX_M, K, true, ra, As, st))) return s;
            if ((s = sl_product<false>(As, Bs, m, n, NT, nkc, group, ra, rb, part, out + (size_t)n0 * ldo + m0, 1, ldo,
                                       1.0, accumulate, gave_up, scratch.failed, st)))
                return s;
        }
    }
    return JDFT_OK;
}

}  // namespace jdft
