// Compare-select of the non-linear layers (Sec. 4.3): everything between its two openings in one
// launch per stage.  edaBits -> Delta = d - r opened -> MSB carry circuit -> e opened -> B2A and the
// selection.
//
// All of it is elementwise in the element (or in the word of 64 elements) and bound by latency at
// the sizes of a request, by memory and the streams at a layer's.  As one kernel per protocol step
// with a copy per message, it was about 120 launches and copies a stage, and 160 more that gathered
// the triples for the verification; here the kernels write the triples where the verification reads
// them, and the sharings that only feed the next step (the arithmetic sharings of public-seed bits,
// r' = b1 + b2 - 2 b1 b2, <r>) stay in registers.
//
// Layouts: Boolean sharings are bit-sliced (64 elements per word, planes of W = np / 64 words);
// edaBit bit i of element e is bit i np + e of its planes, word (i np + e) / 64.  Component order
// P0.[r]_1, P0.[r]_2, P1.m, P1.[r]_1, P2.m, P2.[r]_2.
#include "kernels.h"

namespace mpc3 {

namespace {

constexpr int TPB = 256;

// One Pi_Mult (Fig. MultP): x y for one element, from the streams' words; g2x, p1x, p2x corrupt the
// messages P0 -> P2, P1 -> P2, P2 -> P1 (0: intact).
__device__ __forceinline__ void mult1(const u64 (&x)[6], const u64 (&y)[6], u64 r1, u64 r2, u64 g1,
                                      u64 g2x, u64 p1x, u64 p2x, u64 (&z)[6]) {
  const u64 g2 = ((x[0] + x[1]) * (y[0] + y[1]) + r1 + r2 - g1) ^ g2x;   // as P2 receives it
  const u64 p1 = g1 - x[2] * y[3] - y[2] * x[3];
  const u64 p2 = x[4] * y[4] - x[4] * y[5] - y[4] * x[5] + g2;
  z[0] = z[3] = r1;
  z[1] = z[5] = r2;
  z[2] = p1 + (p2 ^ p2x);
  z[4] = p2 + (p1 ^ p1x);
}

__device__ __forceinline__ u64 bit_of(const u64* w, long long i) {
  return (w[i >> 6] >> (i & 63)) & 1ull;
}

// The public-seed bits: blockIdx.y = 0..2 the edaBits' planes (np words), 3..5 the daBits' (W words).
__global__ void __launch_bounds__(TPB) k_cs_bits(const CompareSelect a) {
  grid_dep();
  const int q = blockIdx.y % 3, da = blockIdx.y / 3;
  const long long n = da ? a.np / 64 : a.np;
  u64* out = da ? a.da[q] : a.eda[q];
  const Key& key = q == 0 ? a.k01 : q == 1 ? a.k02 : a.k12;
  const u32 tag = make_tag(da ? P_DABIT : P_EDABIT, q == 0 ? C_R1 : q == 1 ? C_R2 : C_M12);
  const long long stride = (long long)gridDim.x * TPB;
  for (long long b = blockIdx.x * (long long)TPB + threadIdx.x; b * 8 < n; b += stride) {
    u64 w[8];
    prf_block8(key, tag, a.obj, (u64)b, w);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (b * 8 + j < n) out[b * 8 + j] = w[j];
  }
}

// The edaBit bit products b1 b2 of all 64 np bits, eight consecutive ones a thread.
__global__ void __launch_bounds__(TPB) k_cs_products(const CompareSelect a) {
  grid_dep();
  const long long N = 64 * a.np, nb = N / 8;
  for (long long b = blockIdx.x * (long long)TPB + threadIdx.x; b < nb; b += (long long)gridDim.x * TPB) {
    u64 r1[8], r2[8], g1[8];
    prf_block8(a.k01, make_tag(P_EDA_MULT, C_R1), a.obj, (u64)b, r1);
    prf_block8(a.k02, make_tag(P_EDA_MULT, C_R2), a.obj, (u64)b, r2);
    prf_block8(a.k01, make_tag(P_EDA_MULT, C_G1), a.obj, (u64)b, g1);
    const long long j0 = b * 8;
    const unsigned b1 = (unsigned)(a.eda[0][j0 >> 6] >> (j0 & 63));
    const unsigned b2 = (unsigned)(a.eda[1][j0 >> 6] >> (j0 & 63));
    u64 z[6][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const u64 n1 = 0ull - ((b1 >> j) & 1u), n2 = 0ull - ((b2 >> j) & 1u);   // [r] = -bit, m = 0
      const u64 x[6] = {n1, 0, 0, n1, 0, 0}, y[6] = {0, n2, 0, 0, 0, n2};
      u64 w[6];
      mult1(x, y, r1[j], r2[j], g1[j], j0 + j == a.fault[0].idx ? a.fault[0].mask : 0ull,
            j0 + j == a.fault[1].idx ? a.fault[1].mask : 0ull,
            j0 + j == a.fault[2].idx ? a.fault[2].mask : 0ull, w);
#pragma unroll
      for (int c = 0; c < 6; ++c) z[c][j] = w[c];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
      for (int j = 0; j < 8; j += 2)
        *reinterpret_cast<ulonglong2*>(a.eprod + c * N + j0 + j) = make_ulonglong2(z[c][j], z[c][j + 1]);
  }
}

// r' = b1 + b2 - 2 b1 b2 of edaBit product j, component c (n1, n2: minus the bits)
__device__ __forceinline__ u64 rprime(int c, u64 n1, u64 n2, u64 z) {
  const u64 lin = (c == 0 || c == 3) ? n1 : (c == 1 || c == 5) ? n2 : 0ull;
  return lin - 2ull * z;
}

// z = sum_i m_i 2^(i+1) r'_i (Pi_Inner: <m_i> has no mask), r = sum_i 2^i (m_i + r'_i) - z, and
// Delta's sharing d - r with d = a - b (stored: the selection's first operand).  A block takes 32
// elements, eight threads an element for eight bits each; its threads 0..95 draw the streams.
__global__ void __launch_bounds__(TPB) k_cs_inner(const CompareSelect a) {
  grid_dep();
  __shared__ u64 red[8][8][33], str[3][32];
  const long long np = a.np, N = 64 * np, e0 = (long long)blockIdx.x * 32;
  const int l = threadIdx.x & 31, g = threadIdx.x >> 5;
  const long long e = e0 + l;
  u64 s1 = 0, s2 = 0, acc[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = g * 8 + k;
    const long long j = (long long)i * np + e;
    const u64 n1 = 0ull - bit_of(a.eda[0], j), n2 = 0ull - bit_of(a.eda[1], j), m = bit_of(a.eda[2], j);
    u64 rp[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      rp[c] = rprime(c, n1, n2, a.eprod[c * N + j]);
      acc[c] += (rp[c] + ((c == 2 || c == 4) ? m : 0ull)) << i;
    }
    // P1: -(m_x [r_y]_1 + m_y [r_x]_1), [r_x]_1 = 0;  P2: m_x m_y - m_x [r_y]_2 - m_y [r_x]_2
    if (i < 63) {
      s1 -= m * (rp[3] << (i + 1));
      s2 += m * (rp[4] << (i + 1)) - m * (rp[5] << (i + 1));
    }
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) red[g][c][l] = acc[c];
  red[g][6][l] = s1;
  red[g][7][l] = s2;
  if (g < 3)
    str[g][l] = prf_word(g == 1 ? a.k02 : a.k01,
                         make_tag(P_EDA_INNER, g == 0 ? C_R1 : g == 1 ? C_R2 : C_G1), a.obj, (u64)e);
  __syncthreads();
  if (g < 6) {   // component g of element e
    const int c = g;
    const u64 r1 = str[0][l], r2 = str[1][l], g1 = str[2][l];
    u64 v = 0, z;
#pragma unroll
    for (int q = 0; q < 8; ++q) v += red[q][c][l];
    if (c == 2 || c == 4) {
      u64 p1 = g1, p2 = r1 + r2 - g1;   // Gamma = [r_z]_1 + [r_z]_2: <m_i> has no mask
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        p1 += red[q][6][l];
        p2 += red[q][7][l];
      }
      z = p1 + p2;
    } else {
      z = (c == 0 || c == 3) ? r1 : r2;
    }
    const u64 av = a.a.p && e < a.a.valid ? a.a.p[c * a.a.stride + e] : 0ull;
    const u64 bv = a.b.p && e < a.b.valid ? a.b.p[c * a.b.stride + e] : 0ull;
    a.ez[c * np + e] = z;
    a.mx[2][c * a.nm + e] = av - bv;
    a.dd[c * np + e] = av - bv - (v - z);
  }
}

// The daBits: t = b1 b2, r' = b1 + b2 - 2 t, u = r' b3, r = r' + b3 - 2 u, and the first two triples.
__global__ void __launch_bounds__(TPB) k_cs_dabits(const CompareSelect a) {
  grid_dep();
  const long long np = a.np, nm = a.nm, stride = (long long)gridDim.x * TPB;
  for (long long b = blockIdx.x * (long long)TPB + threadIdx.x; b * 8 < np; b += stride) {
    const long long e0 = b * 8;
    const unsigned b1 = (unsigned)(a.da[0][e0 >> 6] >> (e0 & 63));
    const unsigned b2 = (unsigned)(a.da[1][e0 >> 6] >> (e0 & 63));
    const unsigned b3 = (unsigned)(a.da[2][e0 >> 6] >> (e0 & 63));
    u64 r1[8], r2[8], g1[8], t[6][8];
    prf_block8(a.k01, make_tag(P_DA_MULT1, C_R1), a.obj, (u64)b, r1);
    prf_block8(a.k02, make_tag(P_DA_MULT1, C_R2), a.obj, (u64)b, r2);
    prf_block8(a.k01, make_tag(P_DA_MULT1, C_G1), a.obj, (u64)b, g1);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const u64 n1 = 0ull - ((b1 >> j) & 1u), n2 = 0ull - ((b2 >> j) & 1u);
      const u64 x[6] = {n1, 0, 0, n1, 0, 0}, y[6] = {0, n2, 0, 0, 0, n2};
      u64 z[6];
      mult1(x, y, r1[j], r2[j], g1[j], 0, 0, 0, z);
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        a.mx[0][c * nm + e0 + j] = x[c];
        a.my[0][c * nm + e0 + j] = y[c];
        a.mz[0][c * nm + e0 + j] = z[c];
        t[c][j] = rprime(c, n1, n2, z[c]);
      }
    }
    prf_block8(a.k01, make_tag(P_DA_MULT2, C_R1), a.obj, (u64)b, r1);
    prf_block8(a.k02, make_tag(P_DA_MULT2, C_R2), a.obj, (u64)b, r2);
    prf_block8(a.k01, make_tag(P_DA_MULT2, C_G1), a.obj, (u64)b, g1);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const u64 m = (b3 >> j) & 1u;
      const u64 x[6] = {t[0][j], t[1][j], t[2][j], t[3][j], t[4][j], t[5][j]}, y[6] = {0, 0, m, 0, m, 0};
      u64 z[6];
      mult1(x, y, r1[j], r2[j], g1[j], 0, 0, 0, z);
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        a.mx[1][c * nm + e0 + j] = x[c];
        a.my[1][c * nm + e0 + j] = y[c];
        a.mz[1][c * nm + e0 + j] = z[c];
        a.rad[c * np + e0 + j] = x[c] + y[c] - 2ull * z[c];
      }
    }
  }
}

// MSB of d = Delta + r by a carry tree over the bit planes, and e = [d >= 0] XOR (daBit r).  The
// words w are independent: a block takes four of them (32-byte runs of the triples), thread (plane,
// word).  Leaves: G_i = r_i AND Delta_i, P_i = r_i XOR Delta_i for i < 63, leaf 63 = (0, 1).  Level l
// joins neighbours: X = [P_hi ; P_hi], Y = [G_lo ; P_lo] over 2 C planes (C at the root), Z = X AND Y
// (Fig. MultP over Z_2), G' = G_hi XOR Z, P' = Z of the second half.
__global__ void __launch_bounds__(TPB) k_cs_msb(const CompareSelect a) {
  grid_dep();
  __shared__ u64 G[6][64][4], P[6][64][4];
  const long long W = a.np / 64;
  const int wl = threadIdx.x & 3, p = threadIdx.x >> 2;
  const long long w = (long long)blockIdx.x * 4 + wl;
  const bool in = w < W;
  const u64 b1 = in ? a.eda[0][p * W + w] : 0ull, b2 = in ? a.eda[1][p * W + w] : 0ull;
  const u64 bm = in ? a.eda[2][p * W + w] : 0ull, d = in ? a.dpl[p * W + w] : 0ull;
  const u64 rb[6] = {b1, b2, bm, b1, bm, b2};
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const bool m = c == 2 || c == 4;
    G[c][p][wl] = p < 63 ? rb[c] & d : 0ull;
    P[c][p][wl] = p < 63 ? (m ? rb[c] ^ d : rb[c]) : (m ? ~0ull : 0ull);
  }
  long long off = a.and_off;
#pragma unroll 1
  for (int l = 1; l <= 6; ++l) {
    const int C = 32 >> (l - 1), planes = l == 6 ? C : 2 * C;
    const bool on = p < planes;
    u64 z[6] = {0, 0, 0, 0, 0, 0}, gh[6];
    __syncthreads();
    if (on) {
      const int k = p < C ? p : p - C;
      u64 x[6], y[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        x[c] = P[c][2 * k + 1][wl];
        y[c] = p < C ? G[c][2 * k][wl] : P[c][2 * k][wl];
        gh[c] = G[c][2 * k + 1][wl];
      }
      const u64 i = (u64)p * W + w, obj = a.obj + (u64)l;
      const u64 r1 = prf_word(a.k01, make_tag(P_AND, C_R1), obj, i);
      const u64 r2 = prf_word(a.k02, make_tag(P_AND, C_R2), obj, i);
      const u64 g1 = prf_word(a.k01, make_tag(P_AND, C_G1), obj, i);
      // P0 -> P2: [Gamma]_2; the first level's is the AND messages' fault site
      const u64 g2 = ((x[0] ^ x[1]) & (y[0] ^ y[1])) ^ r1 ^ r2 ^ g1 ^
                     (l == 1 && (long long)i == a.fault[3].idx ? a.fault[3].mask : 0ull);
      const u64 p1 = (x[2] & y[3]) ^ (y[2] & x[3]) ^ g1;
      const u64 p2 = (x[4] & y[4]) ^ (x[4] & y[5]) ^ (y[4] & x[5]) ^ g2;
      z[0] = z[3] = r1;
      z[1] = z[5] = r2;
      z[2] = z[4] = p1 ^ p2;
      if (in) {
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          const long long o = c * a.and_words + off + (long long)i;
          a.ax[o] = x[c];
          a.ay[o] = y[c];
          a.az[o] = z[c];
        }
      }
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        if (p < C) G[c][p][wl] = gh[c] ^ z[c];
        else P[c][p - C][wl] = z[c];
      }
    }
    off += (long long)planes * W;
  }
  __syncthreads();
  if (p == 63 && in) {   // msb = r_63 XOR Delta_63 XOR carry; [d >= 0] = NOT msb
    const u64 q1 = a.da[0][w], q2 = a.da[1][w], qm = a.da[2][w];
    const u64 q[6] = {q1, q2, qm, q1, qm, q2};
#pragma unroll
    for (int c = 0; c < 6; ++c)
      a.e[c * W + w] = rb[c] ^ G[c][0][wl] ^ q[c] ^ ((c == 2 || c == 4) ? ~d : 0ull);
  }
}

// B2A of e (opened: dbits) and the selection out = b + d [a >= b], with the third triple.
__global__ void __launch_bounds__(TPB) k_cs_select(const CompareSelect a) {
  grid_dep();
  const long long np = a.np, nm = a.nm, stride = (long long)gridDim.x * TPB;
  for (long long b = blockIdx.x * (long long)TPB + threadIdx.x; b * 8 < np; b += stride) {
    const long long e0 = b * 8;
    const unsigned bits = (unsigned)(a.dbits[e0 >> 6] >> (e0 & 63));
    u64 r1[8], r2[8], g1[8];
    prf_block8(a.k01, make_tag(P_NL_MULT, C_R1), a.obj, (u64)b, r1);
    prf_block8(a.k02, make_tag(P_NL_MULT, C_R2), a.obj, (u64)b, r2);
    prf_block8(a.k01, make_tag(P_NL_MULT, C_G1), a.obj, (u64)b, g1);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const long long e = e0 + j;
      const bool bit = (bits >> j) & 1u;
      u64 x[6], y[6], z[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const u64 r = a.rad[c * np + e];
        x[c] = a.mx[2][c * nm + e];
        y[c] = bit ? ((c == 2 || c == 4) ? 1ull : 0ull) - r : r;
      }
      mult1(x, y, r1[j], r2[j], g1[j], 0, 0, 0, z);
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        a.my[2][c * nm + e] = y[c];
        a.mz[2][c * nm + e] = z[c];
        if (e < a.out_n)
          a.out[c * a.out_ld + e] = z[c] + (a.b.p && e < a.b.valid ? a.b.p[c * a.b.stride + e] : 0ull);
      }
    }
  }
}

inline unsigned grid_for(long long threads) {
  long long g = (threads + TPB - 1) / TPB;
  return (unsigned)(g < 1 ? 1 : g > 152 * 32 ? 152 * 32 : g);
}

}  // namespace

void launch_cs_open_delta(cudaStream_t st, const CompareSelect& a) {
  launch_dep(k_cs_bits, dim3(grid_for((a.np + 7) / 8), 6), TPB, 0, st, a);
  launch_dep(k_cs_products, grid_for(8 * a.np), TPB, 0, st, a);
  launch_dep(k_cs_inner, (unsigned)(a.np / 32), TPB, 0, st, a);
}

void launch_cs_open_bit(cudaStream_t st, const CompareSelect& a) {
  launch_dep(k_cs_dabits, grid_for(a.np / 8), TPB, 0, st, a);
  launch_dep(k_cs_msb, (unsigned)((a.np / 64 + 3) / 4), TPB, 0, st, a);
}

void launch_cs_select(cudaStream_t st, const CompareSelect& a) {
  launch_dep(k_cs_select, grid_for(a.np / 8), TPB, 0, st, a);
}

}  // namespace mpc3
