// Positions of the sample rows of a set (plain C++, also compiled by the host tests).
#pragma once

#ifdef __CUDACC__
#define CA_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define CA_HOST_DEVICE inline
#endif

namespace ca {

// floor(j s / D) for j < D, D a power of two: j (s / D) + floor(j (s mod D) / D), whose products stay below 2^31 for
// every s (j s itself leaves 32 bits from 33.8 million rows at D = 128).
template <int D>
CA_HOST_DEVICE int sample_position(int j, int s) {
  static_assert(D > 0 && (D & (D - 1)) == 0, "a power of two");
  const unsigned uj = (unsigned)j, us = (unsigned)s;
  return (int)(uj * (us / D) + uj * (us % D) / D);
}

}  // namespace ca
