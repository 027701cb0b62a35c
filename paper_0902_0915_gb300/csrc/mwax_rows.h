// Aligned 16-byte units of a sample buffer that may end inside one (shared by
// the row copy's kernel and its host test).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MWAX_HD __host__ __device__ __forceinline__
#else
#define MWAX_HD inline
#endif

namespace mwax {

struct Unit16 {
  uint32_t w[4];
};

// The bytes of the unit at p (16-byte aligned) that lie before `end`, zeros after
// them; nothing from `end` on is read.  load.unit(p) reads 16 bytes, load.byte(p) one.
// WHOLE: the unit lies before `end`, the caller says.
template <bool WHOLE, class Load>
MWAX_HD Unit16 unit_before(const uint8_t *p, const uint8_t *end, const Load &load) {
  if (WHOLE || end - p >= 16) return load.unit(p);
  Unit16 u = {{0, 0, 0, 0}};
  for (int w = 0; w < 4; ++w)
    for (int k = 0; k < 4; ++k)
      if (p + 4 * w + k < end) u.w[w] |= (uint32_t)load.byte(p + 4 * w + k) << (8 * k);
  return u;
}

// The two aligned units that hold the n (1 .. 16) bytes at `at`; the second is
// only read where they reach it.  WHOLE: at least 15 bytes follow them before `end`.
// Returns how far into the first unit they start.
template <bool WHOLE, class Load>
MWAX_HD int units_of(const uint8_t *at, int n, const uint8_t *end, const Load &load, Unit16 &a, Unit16 &b) {
  const int s = (int)(reinterpret_cast<uintptr_t>(at) & 15);
  a = unit_before<WHOLE>(at - s, end, load);
  b = Unit16{{0, 0, 0, 0}};
  if (s + n > 16) b = unit_before<WHOLE>(at - s + 16, end, load);
  return s;
}

}  // namespace mwax
