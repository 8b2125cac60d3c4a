// fw_rows.h -- stepping through the entries of a CSR row (device code; plain
// C++ on the host).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define FW_ROWS_INLINE __device__ __forceinline__
#else
#define FW_ROWS_INLINE inline
#endif

namespace fw {

// Calls f(i) for the entries i = s + t, s + t + step, ... of the row of d
// entries that begins at s.  A graph holds up to 2^31 - 1 entries, so an int32
// index one step past a row's end may not exist: the place in the row is
// counted instead, in 32 unsigned bits (d + step < 2^32).
template <class F>
FW_ROWS_INLINE void for_entries(int32_t s, int32_t d, int32_t t, int32_t step, F f) {
  for (uint32_t k = (uint32_t)t; k < (uint32_t)d; k += (uint32_t)step) f((int32_t)((uint32_t)s + k));
}

}  // namespace fw
