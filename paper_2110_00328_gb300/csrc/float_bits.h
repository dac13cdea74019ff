// float_bits.h -- conversions between float and double on their bits, without the
// conversion instructions, which are ones of the 1/64-rate FP64 pipe.
#pragma once

#ifdef __CUDACC__
#define MG_HD __host__ __device__ __forceinline__
#else
#define MG_HD inline
#endif

namespace mg {

// The float nearest a double of high word hi and low word lo (ties to even), for doubles
// that round to a normal float and for zeros; *ok = false for the others.
MG_HD unsigned d2f_nearest_bits(unsigned hi, unsigned lo, bool* ok) {
  const unsigned a = hi & 0x7fffffffu;
  // exponent and leading 23 bits of the fraction, rebiased; the 29 bits below decide
  const unsigned m = ((a << 3) | (lo >> 29)) - (896u << 23);
  const unsigned r = m + (((lo & 0x1fffffffu) + 0x0fffffffu + (m & 1u)) >> 29);
  const bool zero = (a | lo) == 0;
  *ok = zero || (a >= (897u << 20) && a < (1151u << 20) && r < 0x7f800000u);
  return (zero ? 0u : r) | (hi & 0x80000000u);
}

}  // namespace mg
