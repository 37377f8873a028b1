// Block-cooperative products in GR(2^64, 64) by 64 P threads, for the single-element steps of the
// verification (challenges, claims, weights), which are chains of dependent products: their time
// is the latency of one product, so a product is spread over P threads per coefficient.
#pragma once
#include "common.cuh"

namespace mpc3 {

// What coefficient c of the reduction subtracts from lo[c], from the coefficients hi (64 ..).
__device__ __forceinline__ u64 gr_carry_at(const u64* hi, int c) {
  u64 v = 0;
  if (c < 63) v += hi[c];
  if (c >= 1) v += hi[c - 1];
  if (c >= 3) v += hi[c - 3];
  if (c >= 4) v += hi[c - 4];
  if (c < 7) {   // H2 = (h_60 + h_61, h_61 + h_62, h_62), at the shifts 0, 1, 3, 4 of g
    const u64 h0 = hi[60], h1 = hi[61], h2 = hi[62];
    if ((0x1B >> c) & 1) v -= h0 + h1;
    if ((0x36 >> c) & 1) v -= h1 + h2;
    if ((0x6C >> c) & 1) v -= h2;
  }
  return v;
}

// Coefficient c of the reduction mod f of a 127-coefficient product (lo: coefficients 0..63, hi:
// 64..126, hi[63] ignored): lo - H g + g H2 with x^64 = -g = -(x^4 + x^3 + x + 1), H2 the three
// coefficients that H g carries past 63.
__device__ __forceinline__ u64 gr_reduce_at(const u64* lo, const u64* hi, int c) {
  return lo[c] - gr_carry_at(hi, c);
}

// lo += product terms of coefficient t, hi += those of coefficient 64 + t, over the factors
// a_i, i0 <= i < i0 + N.  The terms with i <= t belong to lo: one running sum, its value after
// i = t kept, so that the additions stay inside the multiply-adds.
template <int N>
__device__ __forceinline__ void gr_mac_part(const u64* a, const u64* b, int t, int i0, u64& lo,
                                            u64& hi) {
  u64 s = 0, l = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const int i = i0 + k;
    s += a[i] * b[(t - i) & 63];
    if (i == t) l = s;
  }
  if (t >= i0 + N) l = s;
  lo += l;
  hi += s - l;
}

// The sum of the P parts' (lo, hi) and its reduction: every thread of the block calls it (sub =
// the thread's index in its group of 64 P, scr = the group's 128 P words); returns coefficient
// sub of the result to the threads sub < 64.  A thread whose group has no product passes zeros.
template <int P>
__device__ __forceinline__ u64 gr_finish(u64 lo, u64 hi, u64* scr, int sub) {
  const int t = sub & 63, part = sub >> 6;
  scr[part * 128 + t] = lo;
  scr[part * 128 + 64 + t] = hi;
  __syncthreads();
  if (P > 1) {
    if (sub < 128) {
      u64 v = scr[sub];
#pragma unroll
      for (int p = 1; p < P; ++p) v += scr[p * 128 + sub];
      scr[sub] = v;
    }
    __syncthreads();
  }
  const u64 r = sub < 64 ? gr_reduce_at(scr, scr + 64, sub) : 0ull;
  __syncthreads();
  return r;
}

// a * b by a group of 64 P threads; all threads of the block call it (a, b in shared memory).
template <int P>
__device__ __forceinline__ u64 gr_mul_par(const u64* a, const u64* b, u64* scr, int sub) {
  u64 lo = 0, hi = 0;
  gr_mac_part<64 / P>(a, b, sub & 63, (sub >> 6) * (64 / P), lo, hi);
  return gr_finish<P>(lo, hi, scr, sub);
}

// The terms of coefficients 2 l and 2 l + 1 (lo) and of 64 + 2 l, 65 + 2 l (hi) over the factors a_i,
// i0 <= i < i0 + N (both even): a warp, lane l, takes all coefficients.  a, b 16-byte aligned: with
// two coefficients a lane a pair of b serves four multiply-adds, half the shared-memory reads of
// gr_mac_part, which bound blocks of many products.
struct Gr2 {
  u64 lo[2] = {0, 0}, hi[2] = {0, 0};
  __device__ __forceinline__ void sub(const Gr2& o) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      lo[q] -= o.lo[q];
      hi[q] -= o.hi[q];
    }
  }
};
template <int N>
__device__ __forceinline__ void gr_mac2(const u64* a, const u64* b, int l, int i0, Gr2& g) {
  u64 s0 = 0, s1 = 0, l0 = 0, l1 = 0;
  ulonglong2 p = *reinterpret_cast<const ulonglong2*>(b + ((2 * l - i0) & 63));
#pragma unroll
  for (int k = 0; k < N; k += 2) {
    const int i = i0 + k;
    const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(a + i);
    const ulonglong2 n = *reinterpret_cast<const ulonglong2*>(b + ((2 * l - i - 2) & 63));
    s0 += f.x * p.x;   // b_(2l - i)
    s1 += f.x * p.y;   // b_(2l + 1 - i)
    if (i == 2 * l) l0 = s0;
    s0 += f.y * n.y;   // b_(2l - i - 1)
    s1 += f.y * p.x;   // b_(2l - i)
    if (i == 2 * l) l1 = s1;
    p = n;
  }
  if (2 * l >= i0 + N) {
    l0 = s0;
    l1 = s1;
  }
  g.lo[0] += l0;
  g.lo[1] += l1;
  g.hi[0] += s0 - l0;
  g.hi[1] += s1 - l1;
}

// Coefficient t of x v and of x^2 v (x^64 = -(x^4 + x^3 + x + 1)).
__device__ __forceinline__ u64 gr_x_at(const u64* v, int t) {
  u64 r = t > 0 ? v[t - 1] : 0ull;
  if (t == 0 || t == 1 || t == 3 || t == 4) r -= v[63];
  return r;
}
__device__ __forceinline__ u64 gr_x2_at(const u64* v, int t) {
  u64 r = t > 1 ? v[t - 2] : 0ull;
  if (t == 0 || t == 1 || t == 3 || t == 4) r -= v[62];
  if (t == 1 || t == 2 || t == 4 || t == 5) r -= v[63];
  return r;
}

// Entry (i, t) of the multiplication matrix of a: coefficient t of a x^i, 0 <= i < 64.
__device__ __forceinline__ u64 gr_mulmat_at(const u64* a, int i, int t) {
  // a x^i = sum_m a_m x^(m + i); coefficient 64 + m of the unreduced product is a_(64 + m - i)
  // for m < i, else 0
  auto h = [&](int m) -> u64 { return (m >= 0 && m < i) ? a[64 + m - i] : 0ull; };
  auto hg = [&](int s) -> u64 { return h(s) + h(s - 1) + h(s - 3) + h(s - 4); };
  u64 v = (t >= i ? a[t - i] : 0ull) - hg(t);
  if (t < 7) {
    const u64 h0 = hg(64), h1 = hg(65), h2 = hg(66);
    auto q = [&](int m) -> u64 { return m == 0 ? h0 : m == 1 ? h1 : m == 2 ? h2 : 0ull; };
    v += q(t) + q(t - 1) + q(t - 3) + q(t - 4);
  }
  return v;
}

}  // namespace mpc3
