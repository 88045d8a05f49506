// One thread's running sum of T values, no less accurate however many there are: FP32
// sums carry their rounding errors in a second word (Knuth's two-sum), FP64 ones are
// plain.  FP32 additions beside loads from memory cost nothing there, conversions to FP64
// (two a value, at the rate of its multiply-adds) would.
#pragma once

#ifdef __CUDACC__
#define JDFT_HD __host__ __device__ __forceinline__
#else
#define JDFT_HD inline
#endif

namespace jdft {

template <typename T>
struct RunningSum {
    T s = 0;
    JDFT_HD void add(T a) { s += a; }
    JDFT_HD double total() const { return s; }
};

template <>
struct RunningSum<float> {
    float s = 0.f, c = 0.f;
    // an addition of its own: a product in `a` must not be contracted into it
    static JDFT_HD float sum(float a, float b) {
#ifdef __CUDA_ARCH__
        return __fadd_rn(a, b);
#else
        return a + b;
#endif
    }
    JDFT_HD void add(float a) {
        const float t = sum(s, a), z = sum(t, -s);
        c = sum(c, sum(sum(s, -sum(t, -z)), sum(a, -z)));
        s = t;
    }
    JDFT_HD double total() const { return (double)s + (double)c; }
};

}  // namespace jdft
