// GF(2^64) = GR(2, 64): an element is one word, bit c = coefficient of x^c, modulus
// f = x^64 + x^4 + x^3 + x + 1.
#pragma once
#include "common.cuh"

namespace mpc3 {

// 32 x 32 -> 64-bit carry-less product from integer multiplies on bits spaced 4 apart (the
// "multiplication with holes" of T. Pornin's constant-time GHASH): with x_k = x & (0x11111111 << k),
// the integer product x_i y_j has partial-product bits only in the columns p = i + j (mod 4),
// at most 8 in a column, so each column count fits in the 4 bits p .. p + 3 and bit p is its
// parity.  The XOR of the four products with i + j = k (mod 4), kept at those columns, gives the
// carry-less product's bits there.
__host__ __device__ __forceinline__ u64 clmul32(unsigned x, unsigned y) {
  const unsigned m = 0x11111111u;
  const unsigned x0 = x & m, x1 = x & (m << 1), x2 = x & (m << 2), x3 = x & (m << 3);
  const unsigned y0 = y & m, y1 = y & (m << 1), y2 = y & (m << 2), y3 = y & (m << 3);
  auto mw = [](unsigned a, unsigned b) { return (u64)a * (u64)b; };
  const u64 z0 = mw(x0, y0) ^ mw(x1, y3) ^ mw(x2, y2) ^ mw(x3, y1);
  const u64 z1 = mw(x0, y1) ^ mw(x1, y0) ^ mw(x2, y3) ^ mw(x3, y2);
  const u64 z2 = mw(x0, y2) ^ mw(x1, y1) ^ mw(x2, y0) ^ mw(x3, y3);
  const u64 z3 = mw(x0, y3) ^ mw(x1, y2) ^ mw(x2, y1) ^ mw(x3, y0);
  const u64 M = 0x1111111111111111ull;
  return (z0 & M) | (z1 & (M << 1)) | (z2 & (M << 2)) | (z3 & (M << 3));
}

// a b in GF(2^64) = GF(2)[x] / (x^64 + x^4 + x^3 + x + 1): the 128-bit carry-less product by one
// Karatsuba step over 32-bit halves, then the reduction
__host__ __device__ __forceinline__ u64 gf_mul(u64 a, u64 b) {
  const unsigned a0 = (unsigned)a, a1 = (unsigned)(a >> 32);
  const unsigned b0 = (unsigned)b, b1 = (unsigned)(b >> 32);
  const u64 l = clmul32(a0, b0), h = clmul32(a1, b1);
  const u64 mid = clmul32(a0 ^ a1, b0 ^ b1) ^ l ^ h;
  u64 lo = l ^ (mid << 32);
  const u64 hi = h ^ (mid >> 32);
  // x^64 = x^4 + x^3 + x + 1: fold hi twice (the second fold has at most 4 bits)
  const u64 h2 = (hi >> 60) ^ (hi >> 61) ^ (hi >> 63);
  lo ^= hi ^ (hi << 1) ^ (hi << 3) ^ (hi << 4);
  lo ^= h2 ^ (h2 << 1) ^ (h2 << 3) ^ (h2 << 4);
  return lo;
}

__host__ __device__ inline u64 gf_pow(u64 a, unsigned long long e) {
  u64 r = 1;
  while (e) {
    if (e & 1) r = gf_mul(r, a);
    a = gf_mul(a, a);
    e >>= 1;
  }
  return r;
}

__host__ __device__ __forceinline__ u64 gf_inv(u64 a) { return gf_pow(a, ~0ull - 1ull); }   // a^(2^64 - 2)

// a x in GF(2^64): a shift, and x^4 + x^3 + x + 1 for the x^64 that it carries out
__host__ __device__ __forceinline__ u64 gf_mulx(u64 a) {
  return (a << 1) ^ ((0ull - (a >> 63)) & 0x1Bull);
}

}  // namespace mpc3
