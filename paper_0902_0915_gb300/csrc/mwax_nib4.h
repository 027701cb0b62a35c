// mwax_nib4.h -- 4-bit samples to E4M3 operand codes (device code, shared by
// the unpack kernel and the correlate kernel's fused pair mode).
#pragma once

#include <stdint.h>

namespace mwax {

// Value of one unit of an operand code: E4M3 codes 0x00 .. 0x0F are the
// subnormals and the first binade, i x 2^-9 for code i, and bit 7 is the sign.
// So the code of the integer n x 2^-9, |n| <= 15, is sign and magnitude as they
// are: no float arithmetic makes it.  Products are exact multiples of 2^-18,
// and so are the FP32 sums as long as they stay below 2^24 units.
constexpr float kNib4Units = 262144.f;  // 2^18: accumulator value -> integer

// Four samples (nibbles, two's complement, low = re, high = im) -> the four re
// and the four im codes.  With s = 0xFF in the bytes of negative values, the
// magnitude is (n ^ s) + 1 in four bits and the sign bit 0x80: (n ^ s) & 0x0F
// plus s & 0x81 (no carry leaves a byte).  10 instructions, three of them on the
// FMA pipe, against 17 for biased halves converted to E4M3 by the hardware.
__device__ __forceinline__ uint32_t byte_signs(uint32_t x) {  // bit 7 of each byte replicated
  uint32_t s;
  asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(s) : "r"(x));
  return s;
}
__device__ __forceinline__ uint32_t nib4_re(uint32_t w) {
  const uint32_t s = byte_signs(w << 4);
  return ((w ^ s) & 0x0F0F0F0Fu) + (s & 0x81818181u);
}
__device__ __forceinline__ uint32_t nib4_im(uint32_t w) {
  const uint32_t s = byte_signs(w);
  return (((w >> 4) ^ s) & 0x0F0F0F0Fu) + (s & 0x81818181u);
}

}  // namespace mwax
