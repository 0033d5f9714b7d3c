// Arithmetic shared by the data-parallel FMM kernels.
#pragma once
#include <cuda_runtime.h>

#include "fmm_internal.h"

namespace gtap {
namespace fmm {
namespace {   // internal linkage: every translation unit gets its own copy

template <class R> struct Ops;
template <> struct Ops<double> {
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double rsq(double a) { return rsqrt(a); }
    static __device__ __forceinline__ double coef(const TermEntry& t) { return t.coef64; }
};
template <> struct Ops<float> {
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float rsq(float a) { return rsqrtf(a); }
    static __device__ __forceinline__ float coef(const TermEntry& t) { return t.coef32; }
};

// Compensated accumulator (Kahan) for float; plain sum for double.
template <class R> struct Acc {
    R s = 0, c = 0;
    __device__ __forceinline__ void add(R v) {
        if constexpr (sizeof(R) == 4) {
            const R y = Ops<R>::sub(v, c);
            const R t = Ops<R>::add(s, y);
            c = Ops<R>::sub(Ops<R>::sub(t, s), y);
            s = t;
        } else {
            s += v;
        }
    }
};

// Coefficients are ordered by order |n|, then by y + z, then by z.
__host__ __device__ constexpr int cidx(int a, int b, int c) {
    return (a + b + c) * (a + b + c + 1) * (a + b + c + 2) / 6 + (b + c) * (b + c + 1) / 2 + c;
}

}  // namespace
}  // namespace fmm
}  // namespace gtap
