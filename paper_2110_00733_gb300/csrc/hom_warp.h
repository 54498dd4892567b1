// hom_warp.h -- which lanes a butterfly sum over part of a warp takes from.
// Plain C++, so that the rule can be run on the host.
#pragma once

#ifdef __CUDACC__
#define HOM_HD __host__ __device__
#else
#define HOM_HD
#endif

namespace hom {

// lanes of warp `warp` that a block of `threads` threads launched
HOM_HD constexpr int warp_lanes(int threads, int warp) {
    const int left = threads - 32 * warp;
    return left >= 32 ? 32 : (left > 0 ? left : 0);
}

// Whether `lane` adds the value of lane ^ off in the step `off` (16, 8, .. 1) of a
// butterfly sum over the first n lanes of a warp.  A lane beyond n was never
// launched, and what a shuffle from it returns is undefined.  Lane 0 ends with the
// sum of all n: a lane o < off takes o + off where that exists, and where it does
// not, neither does any lane that one stands for.
HOM_HD constexpr bool sum_takes(int lane, int off, int n) { return (lane ^ off) < n; }

}  // namespace hom
