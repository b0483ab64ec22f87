// Warp sums of several values at once.
#pragma once

namespace tlr {

// Sums of P (a power of two, at most 32) values over the warp by halving exchanges, in a fixed order:
// afterwards lane l holds the sum of value l / (32 / P).  About one addition per value for P = 32, where
// P butterflies take five (an FP64 addition occupies the warp's FP64 pipe for 64 clocks).
template <int P>
__device__ __forceinline__ double warp_sums(double (&v)[P], int lane) {
  int o = 16;
#pragma unroll
  for (int n = P; n > 1; n /= 2, o /= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const double keep = up ? v[i + n / 2] : v[i], send = up ? v[i] : v[i + n / 2];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (int q = 16 / P; q; q /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], q);
  return v[0];
}

}  // namespace tlr
