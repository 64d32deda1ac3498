// Correctly rounded FP64 products by integer operations (internal).
//
// An FP64 instruction of a warp holds its quarter of the SM for 64 clocks; the integer units take
// 64 lanes a clock beside it.  A product of two normal numbers is one 64 x 64 -> 128 bit
// multiplication, a normalising shift and a rounding of its upper half to 53 bits with everything
// below as the sticky bit -- the bits of the IEEE product -- in about 30 integer instructions, the
// time of one FP64 instruction on the other pipe.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define SAAMG_HD __host__ __device__ __forceinline__
#else
#define SAAMG_HD inline
#endif

namespace saamg {

// A non-negative number sig / 2^63 * 2^e: sig has its top bit set and its low 11 bits clear (53
// significant bits), or is 0.
struct Unpacked {
  uint64_t sig;
  int e;
};

SAAMG_HD uint64_t mul_hi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

SAAMG_HD int clz64(uint64_t a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// The nearest 53-bit integer to sig / 2^11 (sticky: the number is a little above sig), ties to even
SAAMG_HD uint64_t round53(uint64_t sig, bool sticky) {
  const uint64_t h = (sig >> 1) | (sig & 1u) | (sticky ? 1u : 0u);  // room for the carry
  return (h + 0x1ffu + ((h >> 10) & 1u)) >> 10;
}

// f / 2^64 (at most 53 significant bits)
SAAMG_HD Unpacked unpack_fraction(uint64_t f) {
  Unpacked u;
  const int lz = clz64(f);
  u.sig = f ? f << lz : 0u;
  u.e = -1 - lz;
  return u;
}

// 1 - f / 2^64, rounded
SAAMG_HD Unpacked unpack_complement(uint64_t f) {
  Unpacked u;
  const uint64_t g = 0u - f;  // 2^64 - f, and 0 for f = 0
  const int lz = clz64(g);
  const uint64_t r = g ? round53(g << lz, false) : 0u;
  const bool carry = (r >> 53) != 0;  // rounded up to a power of two
  u.sig = g && !carry ? r << 11 : 0x8000000000000000ull;
  u.e = g ? -1 - lz + (carry ? 1 : 0) : 0;
  return u;
}

// The product's significand rounded to 53 bits in [2^52, 2^53] and its exponent
SAAMG_HD uint64_t mul53(uint64_t a, uint64_t b, int& e) {
  uint64_t hi = mul_hi64(a, b), lo = a * b;
  if (hi >> 63) {
    e += 1;
  } else {
    hi = (hi << 1) | (lo >> 63);
    lo <<= 1;
  }
  return round53(hi, lo != 0u);
}

SAAMG_HD Unpacked mul_unpacked(Unpacked a, Unpacked b) {
  Unpacked u;
  u.e = a.e + b.e;
  const uint64_t r = mul53(a.sig, b.sig, u.e);
  const bool carry = (r >> 53) != 0;
  u.sig = carry ? 0x8000000000000000ull : r << 11;
  u.e += carry ? 1 : 0;
  if (a.sig == 0u || b.sig == 0u) u.sig = 0u;
  return u;
}

// The bits of the double u is (normal range)
SAAMG_HD uint64_t pack_bits(Unpacked u) {
  return u.sig ? ((uint64_t)(u.e + 1022) << 52) + (u.sig >> 11) : 0u;
}

// The bits of RN(w v) for the double with bits v; ok is false where the operands are not both
// normal or the product leaves the normal range (the caller multiplies then); a product by a zero v
// is +0
SAAMG_HD uint64_t mul_bits(Unpacked w, uint64_t v, bool& ok) {
  const int ev = (int)((v >> 52) & 0x7ffu);
  const uint64_t m = v & 0xfffffffffffffull;
  int e = ev + w.e;  // exponent field of the product, less the carry of mul53
  const bool zero = ev == 0 && m == 0u;
  ok = zero || (ev != 0 && ev != 0x7ff && w.sig != 0u && e >= 1 && e <= 2045);
  const uint64_t r = mul53(w.sig, (m | 0x10000000000000ull) << 11, e);
  const uint64_t p = ((uint64_t)(e - 1) << 52) + r;  // r's top bit adds one to the field
  return zero ? 0u : p | (v & 0x8000000000000000ull);
}

}  // namespace saamg
