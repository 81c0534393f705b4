// The arithmetic of the index sums, apart from the kernel so that it can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define RESTKV_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define RESTKV_HOST_DEVICE inline
#endif

namespace restkv {

// Adds to `sum` those of the indices i .. i + 3 whose key (x, y, z, w) lies above `limit`, in 32 bits as far as they go (a 64-bit
// sum for every key took twice the instructions): four indices at a time below 2^30, which kShort promises, otherwise two.  (Two at a
// time for all rows: adaptive window, 20011 rows 115.1 -> 115.4 us.)
template <bool kShort>
RESTKV_HOST_DEVICE void add_indices_above(unsigned long long& sum, unsigned int i, unsigned int x, unsigned int y, unsigned int z,
                                          unsigned int w, unsigned int limit) {
  unsigned int part = 0u;
  if (x > limit) part += i;
  if (y > limit) part += i + 1u;
  if (!kShort) {
    sum += part;
    part = 0u;
  }
  if (z > limit) part += i + 2u;
  if (w > limit) part += i + 3u;
  sum += part;
}

}  // namespace restkv
