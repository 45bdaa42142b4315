// pk_sums.h -- sums of FP32 numbers held as unevaluated sums of FP32 numbers
// (pk_lognormal.cu).  Not installed.
#pragma once

#include <math.h>

namespace pk {

// One rounding each, never contracted (host: compile with -ffp-contract=off).
#ifdef __CUDA_ARCH__
#define PK_FADD(a, b) __fadd_rn(a, b)
#define PK_FMUL(a, b) __fmul_rn(a, b)
#else
#define PK_FADD(a, b) ((a) + (b))
#define PK_FMUL(a, b) ((a) * (b))
#endif

// a + b = s + e exactly (Knuth's two-sum).
__host__ __device__ __forceinline__ float two_sum(float a, float b, float *e) {
    const float s = PK_FADD(a, b), bb = PK_FADD(s, -a);
    *e = PK_FADD(PK_FADD(a, -PK_FADD(s, -bb)), PK_FADD(b, -bb));
    return s;
}

// Sum of squares in three parts (some 72 bits): the square and every addition split
// exactly but for the last part's.  Largest errors of fifty sums of 430 and of 8192
// squares (a draw of 512^3 cells takes 215 a thread, of 2048^3 14000): 0 and 9e-17; in
// two parts 3e-13 and 5e-12, in FP64 0 (the squares there had 46 bits) and 9e-14.  Two
// cells per instruction (packed FP32) took longer.
struct SquareSum {
    float h = 0.0f, m = 0.0f, l = 0.0f;
    __host__ __device__ __forceinline__ void add(float x) {
        const float p = PK_FMUL(x, x), pe = fmaf(x, x, -p);
        float e, e2;
        h = two_sum(h, p, &e);
        m = two_sum(m, e, &e);
        m = two_sum(m, pe, &e2);
        l = PK_FADD(l, PK_FADD(e, e2));
    }
    __host__ __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
};

}  // namespace pk
