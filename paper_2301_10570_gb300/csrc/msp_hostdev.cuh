// msp_hostdev.cuh -- arithmetic that host and kernels share, or that the tests run
// on the host: plain C++ without CUDA headers.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define MSP_HD __host__ __device__ __forceinline__
#else
#define MSP_HD inline
#endif

namespace msp {

// whether the bytes [a, a + na) and [b, b + nb) meet
inline bool meets(const void* a, int64_t na, const void* b, int64_t nb) {
    const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
    return pa < pb + (uintptr_t)nb && pb < pa + (uintptr_t)na;
}

// What a traversal tile counts (children, split, near-field and far pairs) as
// the W words of its look-back, which adds them modulo 2^62.  The pairs of a
// depth lie in the pair table (at most 2^31 - 1), so two of their counts share a
// word; a depth's children may be 64 times as many and have a word of their own:
// their number has to be exact beyond the table too, or the depths that do not
// fit would not be seen.  W = 2 where no pair can be far, else 3.
template <int W>
MSP_HD void trav_pack(const int (&tot)[4], long long (&w)[W]) {
    w[0] = tot[0];
    w[1] = (long long)tot[1] << 31 | tot[2];
    if (W > 2) w[W - 1] = tot[3];
}

template <int W>
MSP_HD void trav_unpack(const long long (&w)[W], long long (&ex)[4]) {
    ex[0] = w[0];
    ex[1] = w[1] >> 31;
    ex[2] = w[1] & ((1ll << 31) - 1);
    ex[3] = W > 2 ? w[W - 1] : 0;
}

// The sum of N compensated totals get(0 .. N-1).  Up to four are added in order
// (three roundings); more with their rounding errors collected (Knuth's exact
// sum of two), so that the sum stays within a rounding or two of the exact one:
// added in order, 16 warps' totals put u of networks of 21,000 neurons 1.59e-7 off
// (relative, over all neurons) where four warps' had been 1.50e-7; this is 1.48e-7.
template <int N, class Get>
MSP_HD float sum_totals(Get get) {
    float s = get(0), lost = 0.f;
    for (int k = 1; k < N; ++k) {
        const float v = get(k), t = s + v;
        if (N > 4) {
            const float b = t - s;
            lost += (s - (t - b)) + (v - b);
        }
        s = t;
    }
    return N > 4 ? s + lost : s;
}

}  // namespace msp
