// wo_feat.cuh - the points of a half-spectrum plane as the estimator's
// features walk them (host and device: the offsets are tested on the host).
#pragma once
#include <limits.h>

namespace wo {

// Point p = y Xh + x of a plane's rows 0 .. Y/2, as offsets in the plane: the
// point itself and its row's mirror image, the point at Y - y (-1: none, the
// rows 0 and Y/2).
template <class I>
struct FeatPoint {
  I at, mirror;
};

template <class I>
__host__ __device__ inline FeatPoint<I> feat_point(I p, int Y, int Xh, int* y, int* x) {
  *y = (int)(p / Xh);
  *x = (int)(p - (I)*y * Xh);
  return {p, (*y > 0 && *y < Y - *y) ? (I)(Y - *y) * Xh + *x : (I)-1};
}

// Planes of more points than an int counts (a step of the walk, 128 points,
// may pass the last one) take 64-bit offsets; the others 32-bit ones, which
// take half the shared memory and integer instructions.
__host__ __device__ inline bool feat_wide(int Y, int Xh) { return (long long)Y * Xh > INT_MAX - 128; }

}  // namespace wo
