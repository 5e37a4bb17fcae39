// Arithmetic of the learned partitioner's kernels (tests/reciprocal_check.cu).
#pragma once

namespace vx {

// 1 / d for 1 <= d <= 6e34: CUDA's fast division and one step of Householder's
// third-order iteration for the reciprocal, r (1 + e + e^2) with e = 1 - d r.
// From the fast division's two units in the last place the step leaves an error of
// 2^-45 before the last rounding, so all but about one result in a million are the
// correctly rounded ones, and those are off by one unit.  (__frcp_rn looks for
// special cases, which keeps the 32 reciprocals of a lane from overlapping: 300
// training steps take 2.01 ms with it, 1.70 with this, 1.64 with the fast
// division alone.)
__device__ __forceinline__ float reciprocal(float d) {
  const float r = __fdividef(1.f, d), e = fmaf(-d, r, 1.f);
  return fmaf(r, fmaf(e, e, e), r);
}

}  // namespace vx
