// Which taps of an interpolation window lie on the spectrum (k5_refine.cu).  No CUDA needed: the bounds
// are checked on the host too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define FDAS_HD __host__ __device__ __forceinline__
#else
#define FDAS_HD inline
#endif

namespace fdas {

struct TapRange {
    int lo, hi;      // tap offsets lo .. hi; none when lo > hi
};

// The offsets j in [-m/2, m - m/2) with 0 <= k0 + j < nb.  Anchors reach +-2^52 (a point is accepted up to
// |r| = 4.5e15), so the bounds meet in 64 bits; when any offset is left, both lie inside the window.
FDAS_HD TapRange taps_on_spectrum(int64_t k0, int m, int64_t nb) {
    const int half = m / 2;
    const int64_t lo = k0 < half ? -k0 : -(int64_t)half;
    const int64_t hi = nb - 1 - k0 < m - half - 1 ? nb - 1 - k0 : (int64_t)(m - half - 1);
    if (lo > hi) return {0, -1};
    return {(int)lo, (int)hi};
}

// The part of `on`, folded (j -> -j) when neg, that lies in jl .. jh.
FDAS_HD TapRange taps_between(TapRange on, bool neg, int jl, int jh) {
    if (on.lo > on.hi) return {0, -1};
    const int lo = neg ? -on.hi : on.lo, hi = neg ? -on.lo : on.hi;
    return {jl > lo ? jl : lo, jh < hi ? jh : hi};
}

}  // namespace fdas
