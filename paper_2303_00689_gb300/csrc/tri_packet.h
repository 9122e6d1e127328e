// The tagged double of the FP64 tridiagonalisation's packets: 64 bits that hold a double and one
// bit that says which column it is of.  A double uses all 64 bits, but only half of its
// exponents occur: with bit 62 (the exponent's highest) free for the tag,
//  * 2^-766 <= |x| < 2^257 is stored with its exponent moved down by 256: all of its bits.
//    (Sums over a row of products of the Fock matrix's elements: those of 10^38 eV and, since the
//    square of a reflector's row underflows below 10^-154, couplings of less than 10^-77 eV are
//    outside.)
//  * every other value (zero, infinities and NaN among them) as the upper 52 of its 63 bits below
//    the sign, under an exponent field of zero: 41 bits of the significand.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define KX_PACKET_FN __host__ __device__ __forceinline__
#else
#define KX_PACKET_FN inline
#endif

namespace kx {

constexpr uint64_t kPacketTag = 1ull << 62;

KX_PACKET_FN uint64_t packet_encode(uint64_t b, uint64_t tag) {
  const uint64_t sign = b & (1ull << 63), mag = b ^ sign;
  const unsigned ex = (unsigned)(mag >> 52);
  const uint64_t body = (ex - 257u < 1023u) ? mag - (256ull << 52) : mag >> 11;
  return sign | body | tag;
}
KX_PACKET_FN uint64_t packet_decode(uint64_t x) {
  const uint64_t sign = x & (1ull << 63), body = x & (kPacketTag - 1);
  return sign | ((body >> 52) ? body + (256ull << 52) : body << 11);
}

}  // namespace kx
