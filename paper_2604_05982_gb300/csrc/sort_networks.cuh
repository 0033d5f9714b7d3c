// Register sorting networks shared by the thread-mode and block-mode sorts.
// Every index is a constant after unrolling, so the arrays stay in registers.
#pragma once
#include <cstdint>

namespace gtap {

// Bitonic sort of ITEMS keys (a power of two), ascending.
template <int ITEMS>
__device__ __forceinline__ void sort_registers(uint32_t (&x)[ITEMS]) {
#pragma unroll
    for (int k = 2; k <= ITEMS; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int l = i ^ j;
                if (l > i) {
                    const bool up = (i & k) == 0;
                    const uint32_t lo = min(x[i], x[l]), hi = max(x[i], x[l]);
                    x[i] = up ? lo : hi;
                    x[l] = up ? hi : lo;
                }
            }
        }
    }
}

// The N smallest of two ascending sequences a and b, ascending, into a.  The
// element-wise minimum of a and reversed b holds exactly the N smallest of the
// 2N keys and is bitonic (Batcher's bitonic merge, first half-cleaner); the
// remaining half-cleaners sort it.  Only key values are produced, so which of
// two equal keys is taken does not matter.
template <int N>
__device__ __forceinline__ void lowest_of_two_sorted(uint32_t (&a)[N], const uint32_t (&b)[N]) {
#pragma unroll
    for (int k = 0; k < N; ++k) a[k] = min(a[k], b[N - 1 - k]);
#pragma unroll
    for (int j = N / 2; j > 0; j >>= 1) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            if ((k & j) == 0) {
                const uint32_t x = a[k], y = a[k + j];
                a[k] = min(x, y);
                a[k + j] = max(x, y);
            }
        }
    }
}

}  // namespace gtap
