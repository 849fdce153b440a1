// Index arithmetic shared by the device code.
#pragma once

namespace ttns {

// n / d for 0 <= n < 2^24 through a float reciprocal, corrected to the exact quotient
// (the float estimate is within 2 of it); 64-bit integer division is emulated and slow.
__device__ __forceinline__ int fdivu(int n, int d, float inv) {
  int q = __float2int_rz((float)n * inv);
  int r = n - q * d;
  if (r < 0) { --q; r += d; }
  if (r < 0) { --q; r += d; }
  if (r >= d) { ++q; r -= d; }
  if (r >= d) { ++q; }
  return q;
}

}  // namespace ttns
