// Pi_MultVerify (Fig. PPEV) over GF(2^64) of the AND gates of a non-linear layer.
//
// The batch has D = 64 nw gates: x_i = r^i X_i, y_i = Y_i, z = sum r^i Z_i, with X, Y, Z shared bits
// (bit i % 64 of word i / 64).  Like the batches over GR(2^64, 64) (gr_block.cu) its first three
// rounds need no field vectors: with blocks of eight gates, i = 8 b + j, R_b = r^(8b) and the bits
//   w^0 = (X0 ^ X1)_j (Y0 ^ Y1)_j',  w^1 = X2_j Y3_j' ^ X3_j Y2_j',
//   w^2 = X4_j (Y4 ^ Y5)_j' ^ X5_j Y4_j'      (the parties' cross terms; index = share component)
// every party sum of the rounds 1..3 is a sum of V_j W_j' S^p_{j,j'}, S^p_{j,j'} = sum_b R_b w^p, and
// the vectors after them are x_b = R_b (sum_j X_{b,j} V_j) and y_b = sum_j Y_{b,j} W_j: one look-up
// in 256 subset sums each, and one product for x.  Per gate that is 24 masked XORs and 6/8 products
// where materialising and folding took about 40 products (a product is 48 integer multiply-adds).
// 8.2 M gates: 0.7 ms, against 3.9 ms.
//
// Every launch ends with the step that needs its sums (h(0), h(x), the opened zeta, the next claim)
// in whichever block finishes last, so a round is one launch that folds by the round before's zeta
// and sums; the last rounds (up to GF_TAIL elements), Pi_InnerVerify and the hash comparisons of
// every Pi_Rec are one block's work.  As separate launches a round was about 14 of them: a batch of
// 16000 gates took 0.75 ms, now 0.12 ms.
#include "gf.cuh"
#include "kernels.h"

namespace mpc3 {

namespace {

constexpr int GF_TAIL = 500;          // elements that enter the last block's rounds (12 x 4000 bytes)
constexpr u64 GF_X = 2ull;

struct Coef {
  u64 ixx1;   // 1 / (x (x + 1))
};

// Words of GfWork::st, per round k >= 1 at 9 k: the streams H0 (r1, r2, g1), H2 (r1, r2, g1) and
// zeta (r1, r2, m); round 0: r (r1, r2, m), Delta (r1, r2, g1), alpha (r1, r2, m).
__device__ __forceinline__ u64 round_stream(const GfVerify& a, int k, int q) {
  const u32 purpose = k == 0 ? (q < 3 ? P_VER_R : q < 6 ? P_VER_DELTA : P_VER_ALPHA)
                             : (q < 3 ? P_VER_H0 : q < 6 ? P_VER_H2 : P_VER_ZETA);
  const bool m12 = q % 3 == 2 && (k == 0 ? (q < 3 || q >= 6) : q >= 6);   // third word: m or [Gamma]_1
  const u32 comp = q % 3 == 0 ? C_R1 : q % 3 == 1 ? C_R2 : m12 ? C_M12 : C_G1;
  return prf_word(q % 3 == 1 ? a.k02 : m12 ? a.k12 : a.k01, make_tag(purpose, comp),
                  a.obj + (u64)k, 0);
}

// The end of round k on the threads c < 6 of a warp: s = the party sums at 0 (3) and at x (3).  h(0)
// and h(x) as secure inner products (P0 sends Gamma - [Gamma]_1; [m]_1, [m]_2 exchanged), zeta
// opened, the next claim.  L0 + L1 + L2 = 1 at the points 0, 1, x, so z' = h(0) + L1 z + L2 (h(x) +
// h(0)) with L2 = (zeta^2 + zeta) / (x (x + 1)), L1 = (zeta^2 + x zeta) / (1 + x) = x L2 + zeta.
__device__ __forceinline__ void gf_tail(const GfVerify& a, int k, const u64* s, const u64* st, u64* z,
                                        u64* zeta_out, const Coef cf, int c) {
  const u64 zeta = st[8] ^ st[6] ^ st[7] ^ (k == a.xrec ? a.xmask : 0ull);   // P1's opening
  u64 h[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const u64 r1 = st[3 * q], r2 = st[3 * q + 1], g1 = st[3 * q + 2];
    const u64 m1 = s[3 * q + 1] ^ g1;                            // P1
    const u64 m2 = s[3 * q + 2] ^ (s[3 * q] ^ r1 ^ r2 ^ g1);     // P2, with [Gamma]_2
    h[q] = (c == 0 || c == 3) ? r1 : (c == 1 || c == 5) ? r2 : m1 ^ m2;
  }
  const u64 l2 = gf_mul(gf_mul(zeta, zeta) ^ zeta, cf.ixx1);
  const u64 l1 = gf_mulx(l2) ^ zeta;
  z[c] = h[0] ^ gf_mul(l1, z[c]) ^ gf_mul(l2, h[1] ^ h[0]);
  if (c == 0) *zeta_out = zeta;
  if (a.trace) {
    u64* t = a.trace + (long long)(k - 1) * a.trace_ld;
    if (c == 0) t[0] = zeta;
    t[1 + c] = h[0];
    t[7 + c] = h[1];
  }
}

// XOR of v over the block's warps: thread 0 of each warp adds it to *out (shared or global).
__device__ __forceinline__ void warp_xor_to(u64 v, u64* out) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v ^= __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v)
    atomicXor(reinterpret_cast<unsigned long long*>(out), (unsigned long long)v);
}

// true in every thread of the block that finishes last (its earlier atomics and writes, and all
// other blocks', are visible to it)
__device__ bool last_block(unsigned* count) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(count, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// The party sums of one pair (u0, u1), (v0, v1) of elements (6 components): at 0 the even elements,
// at x f(x) = f(0) + x (f(0) + f(1)).
__device__ __forceinline__ void pair_sums(const u64 (&x0)[6], const u64 (&x1)[6],
                                          const u64 (&y0)[6], const u64 (&y1)[6], u64 (&s)[6]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    u64 u[6], v[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      u[c] = q ? x0[c] ^ gf_mulx(x0[c] ^ x1[c]) : x0[c];
      v[c] = q ? y0[c] ^ gf_mulx(y0[c] ^ y1[c]) : y0[c];
    }
    s[3 * q] ^= gf_mul(u[0] ^ u[1], v[0] ^ v[1]);
    s[3 * q + 1] ^= gf_mul(u[2], v[3]) ^ gf_mul(v[2], u[3]);
    s[3 * q + 2] ^= gf_mul(u[4], v[4] ^ v[5]) ^ gf_mul(v[4], u[5]);
  }
}

// r and its powers R_b = r^(8 b), b < nb (8 a thread, from the squares); block 0 also draws every
// stream word of the rounds.
__global__ void __launch_bounds__(256) k_gf_setup(const GfVerify a, long long nb) {
  grid_dep();
  __shared__ u64 sq[40], st[3];
  const int tid = threadIdx.x;
  if (tid < 3) st[tid] = round_stream(a, 0, tid);
  __syncthreads();
  if (tid == 0) {
    u64 r = st[2] ^ st[0] ^ st[1] ^ (a.xrec == 0 ? a.xmask : 0ull);
    if (blockIdx.x == 0) a.w->r = r;
    r = gf_mul(r, r);
    r = gf_mul(r, r);
    for (int k = 0; k < 40 && (k == 0 || (nb >> k) > 0); ++k) {
      r = gf_mul(r, r);
      sq[k] = r;                     // r^(8 2^k)
    }
  }
  if (blockIdx.x == 0)
    for (int i = tid; i < 9 * (a.R + 1); i += 256) a.st[i] = round_stream(a, i / 9, i % 9);
  __syncthreads();
  const long long b0 = ((long long)blockIdx.x * 256 + tid) * 8;
  if (b0 >= nb) return;
  u64 p = 1;
  for (int k = 3; (b0 >> k) > 0; ++k)
    if ((b0 >> k) & 1) p = gf_mul(p, sq[k]);
#pragma unroll 1
  for (int j = 0; j < 8 && b0 + j < nb; ++j) {
    a.pw[b0 + j] = p;
    p = gf_mul(p, sq[0]);
  }
}

// S^p_{j,j'} (192 sums) and the claim's sum_b R_b Z_{c,b,j} (48), then rounds 1..3 in the last block.
// A block takes contiguous words, 16 at a time through shared memory; thread t keeps sum t: its eight
// bits of a word are one AND/XOR of the shifted words, each of them masks one R_b.  Bound by the
// masked XORs (about 6 instructions for each).
__global__ void __launch_bounds__(256) k_gf_sums(const GfVerify a, const Coef cf) {
  grid_dep();
  constexpr int NB = 16;
  __shared__ u64 raw[18][NB], pw[NB * 8];
  const int tid = threadIdx.x, p = tid >> 6, j = (tid >> 3) & 7, k = tid & 7;
  const long long nw = a.nw;
  const long long w0 = nw * blockIdx.x / gridDim.x, w1 = nw * (blockIdx.x + 1) / gridDim.x;
  u64 acc = 0;
  for (long long w = w0; w < w1; w += NB) {
    const int cnt = (int)(w1 - w < NB ? w1 - w : NB);
    __syncthreads();
    for (int i = tid; i < 18 * NB; i += 256) {
      const int c = i / NB, e = i % NB;
      const u64* src = c < 6 ? a.X : c < 12 ? a.Y : a.Z;
      raw[c][e] = e < cnt ? src[(c % 6) * nw + w + e] : 0ull;
    }
    for (int i = tid; i < NB * 8; i += 256) pw[i] = i < cnt * 8 ? a.pw[w * 8 + i] : 0ull;
    __syncthreads();
    for (int e = 0; e < cnt; ++e) {
      u64 v = 0;
      if (p == 0) v = ((raw[0][e] ^ raw[1][e]) >> j) & ((raw[6][e] ^ raw[7][e]) >> k);
      else if (p == 1) v = ((raw[2][e] >> j) & (raw[9][e] >> k)) ^ ((raw[3][e] >> j) & (raw[8][e] >> k));
      else if (p == 2) v = ((raw[4][e] >> j) & ((raw[10][e] ^ raw[11][e]) >> k)) ^
                           ((raw[5][e] >> j) & (raw[10][e] >> k));
      else if (tid < 240) v = raw[12 + (tid - 192) / 8][e] >> k;
#pragma unroll
      for (int q = 0; q < 8; ++q) acc ^= pw[e * 8 + q] & (0ull - ((v >> (8 * q)) & 1ull));
    }
  }
  if (tid < 240) atomicXor(reinterpret_cast<unsigned long long*>(a.w->S + tid), (unsigned long long)acc);
  if (!last_block(&a.w->count[0])) return;
  // ---- rounds 1 .. 3 ----
  __shared__ u64 V[8], W[8], s9[9], z[6], s6[6], zeta, T[8];
  const u64 S = tid < 240 ? __ldcg(a.w->S + tid) : 0ull;
  if (tid == 0) {
    const u64 r = a.w->r;
    u64 t = 1;
    for (int q = 0; q < 8; ++q) {
      T[q] = t;
      t = gf_mul(t, r);
    }
  }
  __syncthreads();
  if (tid < 8) {
    V[tid] = T[tid];
    W[tid] = 1;
  }
  if (tid >= 192) {   // the claim: eight lanes a component
    u64 v = tid < 240 ? gf_mul(T[k], S) : 0ull;
#pragma unroll
    for (int o = 4; o; o >>= 1) v ^= __shfl_xor_sync(0xffffffffu, v, o);
    if (tid < 240 && k == 0) z[(tid - 192) >> 3] = v;
  }
  for (int rd = 1; rd <= 3; ++rd) {
    if (tid < 9) s9[tid] = 0;
    __syncthreads();
    if (p < 3) {   // a warp has one p
      const u64 v = (j >> rd) == (k >> rd) ? gf_mul(gf_mul(V[j], W[k]), S) : 0ull;
      const int cls = ((j >> (rd - 1)) & 1) + ((k >> (rd - 1)) & 1);
#pragma unroll
      for (int q = 0; q < 3; ++q) warp_xor_to(cls == q ? v : 0ull, s9 + q * 3 + p);   // even, cross, odd
    }
    __syncthreads();
    if (tid < 3) {   // at x: (1 + x)^2 even + (1 + x) x cross + x^2 odd
      const u64 e = s9[tid], c = s9[3 + tid], o = s9[6 + tid];
      s6[tid] = e;
      s6[3 + tid] = e ^ gf_mulx(c) ^ gf_mulx(gf_mulx(e ^ c ^ o));
    }
    __syncthreads();
    if (tid < 6) gf_tail(a, rd, s6, a.st + 9 * rd, z, &zeta, cf, tid);
    __syncthreads();
    if (tid < 16) {
      u64* X = tid < 8 ? V : W;
      X[tid & 7] = gf_mul(X[tid & 7], zeta ^ (((tid >> (rd - 1)) & 1) ? 0ull : 1ull));
    }
    __syncthreads();
  }
  if (tid < 8) {
    a.w->V[tid] = V[tid];
    a.w->W[tid] = W[tid];
  }
  if (tid < 6) a.w->z[tid] = z[tid];
}

// The vectors after three rounds (element b = 8 w + q from byte q of word w) and round 4.
__global__ void __launch_bounds__(256) k_gf_vectors(const GfVerify a, const Coef cf, u64* x, u64* y) {
  grid_dep();
  __shared__ u64 tv[256], tw[256], V[8], W[8];
  const int tid = threadIdx.x;
  if (tid < 8) {
    V[tid] = a.w->V[tid];
    W[tid] = a.w->W[tid];
  }
  __syncthreads();
  u64 v = 0, w = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    v ^= V[q] & (0ull - ((tid >> q) & 1ull));
    w ^= W[q] & (0ull - ((tid >> q) & 1ull));
  }
  tv[tid] = v;
  tw[tid] = w;
  __syncthreads();
  const long long nb = 8 * a.nw;
  u64 s[6] = {0, 0, 0, 0, 0, 0};
  for (long long i = blockIdx.x * 256ll + tid; i < nb / 2; i += gridDim.x * 256ll) {
    const long long wd = i >> 2;
    const int sh = (int)(i & 3) * 16;
    const u64 R0 = a.pw[2 * i], R1 = a.pw[2 * i + 1];
    u64 x0[6], x1[6], y0[6], y1[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const unsigned bx = (unsigned)(a.X[c * a.nw + wd] >> sh), by = (unsigned)(a.Y[c * a.nw + wd] >> sh);
      x0[c] = gf_mul(R0, tv[bx & 255]);
      x1[c] = gf_mul(R1, tv[(bx >> 8) & 255]);
      y0[c] = tw[by & 255];
      y1[c] = tw[(by >> 8) & 255];
      *reinterpret_cast<ulonglong2*>(x + c * nb + 2 * i) = make_ulonglong2(x0[c], x1[c]);
      *reinterpret_cast<ulonglong2*>(y + c * nb + 2 * i) = make_ulonglong2(y0[c], y1[c]);
    }
    pair_sums(x0, x1, y0, y1, s);
  }
  u64* S = a.w->sums + 6 * 4;
#pragma unroll
  for (int q = 0; q < 6; ++q) warp_xor_to(s[q], S + q);
  if (!last_block(&a.w->count[4])) return;
  __shared__ u64 s6[6];
  if (tid < 6) s6[tid] = __ldcg(S + tid);
  __syncthreads();
  if (tid < 6) gf_tail(a, 4, s6, a.st + 9 * 4, a.w->z, &a.w->zeta, cf, tid);
}

// Folds D elements (stride ld) by the last zeta into (D + 1) / 2 (stride ldo), a_2i + zeta (a_2i +
// a_2i+1), and takes round k's sums of them.  A thread makes two folded elements: 24 products for
// the folds and 16 for the sums.
__global__ void __launch_bounds__(128)
k_gf_round(const GfVerify a, const Coef cf, int k, long long D, const u64* x,
           const u64* y, long long ld, u64* __restrict__ xo, u64* __restrict__ yo,
           long long ldo) {
  grid_dep();
  const long long Dh = (D + 1) / 2, np = (Dh + 1) / 2;
  const u64 zeta = a.w->zeta;
  u64 s[6] = {0, 0, 0, 0, 0, 0};
  for (long long i = blockIdx.x * 128ll + threadIdx.x; i < np; i += gridDim.x * 128ll) {
    u64 f[2][2][6];
#pragma unroll
    for (int side = 0; side < 2; ++side)
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const u64* in = (side ? y : x) + c * ld;
        u64* out = (side ? yo : xo) + c * ldo;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const long long e = 4 * i + 2 * h;
          const u64 u = e < D ? in[e] : 0ull, v = e + 1 < D ? in[e + 1] : 0ull;
          const u64 w = u ^ gf_mul(zeta, u ^ v);
          f[side][h][c] = w;
          if (2 * i + h < Dh) out[2 * i + h] = w;
        }
      }
    pair_sums(f[0][0], f[0][1], f[1][0], f[1][1], s);
  }
  u64* S = a.w->sums + 6 * k;
#pragma unroll
  for (int q = 0; q < 6; ++q) warp_xor_to(s[q], S + q);
  if (!last_block(&a.w->count[k])) return;
  __shared__ u64 s6[6];
  if (threadIdx.x < 6) s6[threadIdx.x] = __ldcg(S + threadIdx.x);
  __syncthreads();
  if (threadIdx.x < 6) gf_tail(a, k, s6, a.st + 9 * k, a.w->z, &a.w->zeta, cf, threadIdx.x);
}

// H of one word (Pi_Rec of a field element)
__device__ void sha256_word(u64 w, u32 h[8]) {
  u32 blk[16];
  sha256_init(h);
  blk[0] = bswap32((u32)w);
  blk[1] = bswap32((u32)(w >> 32));
  blk[2] = 0x80000000u;
#pragma unroll
  for (int q = 3; q < 15; ++q) blk[q] = 0;
  blk[15] = 64u;
  sha256_compress(h, blk);
}

// From round k's opened zeta and its D elements: the rounds k + 1 .. R, Pi_InnerVerify (Fig. DPV) and
// the hash comparisons, by one block.  A fold is one product a thread and component, the sums one
// product a thread.
__global__ void __launch_bounds__(512)
k_gf_last(const GfVerify a, const Coef cf, int k, long long D0, const u64* x, const u64* y,
          long long ld) {
  grid_dep();
  __shared__ u64 buf[12][GF_TAIL];
  __shared__ u64 s6[6], z[6], zeta, sd[3], dl;
  __shared__ u32 bad;
  const int tid = threadIdx.x;
  int D = (int)((D0 + 1) / 2);
  if (tid < 6) z[tid] = a.w->z[tid];
  if (tid == 0) {
    zeta = a.w->zeta;
    bad = 0;
  }
  __syncthreads();
  for (int i = tid; i < 12 * D; i += 512) {
    const int c = i / D, e = i % D;
    const u64* in = (c < 6 ? x + c * ld : y + (c - 6) * ld);
    const u64 u = in[2 * e], v = 2 * e + 1 < D0 ? in[2 * e + 1] : 0ull;
    buf[c][e] = u ^ gf_mul(zeta, u ^ v);
  }
  __syncthreads();
  for (++k; k <= a.R; ++k) {
    const int Dh = (D + 1) / 2;
    if (tid < 6) s6[tid] = 0;
    __syncthreads();
    // ten products a pair: five at 0, five at x, 32 pairs a warp
    for (int w = tid >> 5; w < 10 * ((Dh + 31) / 32); w += 16) {
      const int t = w % 10, e = (w / 10) * 32 + (tid & 31), q = t >= 5, m = t % 5;
      u64 r = 0;
      if (e < Dh) {
        auto at = [&](int c) -> u64 {
          const u64 u = buf[c][2 * e];
          return q ? u ^ gf_mulx(u ^ (2 * e + 1 < D ? buf[c][2 * e + 1] : 0ull)) : u;
        };
        const u64 u = m == 0 ? at(0) ^ at(1) : m == 1 ? at(2) : m == 2 ? at(3) : m == 3 ? at(4) : at(5);
        const u64 v = m == 0 ? at(6) ^ at(7) : m == 1 ? at(9) : m == 2 ? at(8) : m == 3 ? at(10) ^ at(11)
                                                                                       : at(10);
        r = gf_mul(u, v);
      }
      warp_xor_to(r, s6 + 3 * q + (m == 0 ? 0 : m < 3 ? 1 : 2));
    }
    __syncthreads();
    if (tid < 6) gf_tail(a, k, s6, a.st + 9 * k, z, &zeta, cf, tid);
    __syncthreads();
    u64 f[6];   // 12 Dh <= 6 GF_TAIL < 6 * 512
#pragma unroll
    for (int n = 0; n < 6; ++n) {
      const int i = tid + 512 * n, c = i / Dh, e = i % Dh;
      f[n] = 0;
      if (c < 12) {
        const u64 u = buf[c][2 * e], v = 2 * e + 1 < D ? buf[c][2 * e + 1] : 0ull;
        f[n] = u ^ gf_mul(zeta, u ^ v);
      }
    }
    __syncthreads();
#pragma unroll
    for (int n = 0; n < 6; ++n) {
      const int i = tid + 512 * n, c = i / Dh, e = i % Dh;
      if (c < 12) buf[c][e] = f[n];
    }
    D = Dh;
    __syncthreads();
  }
  // ---- Pi_InnerVerify: x' = x alpha, Delta = sum x'_i y_i + alpha z opened ----
  if (tid < 3) sd[tid] = 0;
  __syncthreads();
  const u64 a1 = a.st[6], a2 = a.st[7], am = a.st[8];   // alpha: [r]_1, [r]_2, m
  for (int i0 = 0; i0 <= D; i0 += 512) {
    const int i = i0 + tid;
    u64 u0 = 0, u1 = 0, u2 = 0, u3 = 0, u4 = 0, u5 = 0;
    if (i < D) {
      const u64 r1 = prf_word(a.k01, make_tag(P_VER_XA, C_R1), a.obj, (u64)i);
      const u64 r2 = prf_word(a.k02, make_tag(P_VER_XA, C_R2), a.obj, (u64)i);
      const u64 g1 = prf_word(a.k01, make_tag(P_VER_XA, C_G1), a.obj, (u64)i);
      const u64 g2 = gf_mul(buf[0][i] ^ buf[1][i], a1 ^ a2) ^ r1 ^ r2 ^ g1;               // P0 -> P2
      const u64 m1 = gf_mul(buf[2][i], a1) ^ gf_mul(am, buf[3][i]) ^ g1;                  // P1
      const u64 m2 = gf_mul(buf[4][i], am ^ a2) ^ gf_mul(am, buf[5][i]) ^ g2;             // P2
      u0 = u3 = r1;
      u1 = u5 = r2;
      u2 = u4 = m1 ^ m2;
    } else if (i == D) {
      u0 = u3 = a1;
      u1 = u5 = a2;
      u2 = u4 = am;
    }
    auto v = [&](int c) -> u64 { return i < D ? buf[6 + c][i] : z[c]; };   // u = 0 past D
    const u64 t0 = gf_mul(u0 ^ u1, v(0) ^ v(1));
    const u64 t1 = gf_mul(u2, v(3)) ^ gf_mul(v(2), u3);
    const u64 t2 = gf_mul(u4, v(4) ^ v(5)) ^ gf_mul(v(4), u5);
    warp_xor_to(t0, sd);
    warp_xor_to(t1, sd + 1);
    warp_xor_to(t2, sd + 2);
  }
  __syncthreads();
  const u64 d1 = a.st[3], d2 = a.st[4], dg = a.st[5];
  if (tid == 0) {
    const u64 m1 = sd[1] ^ dg, m2 = sd[2] ^ (sd[0] ^ d1 ^ d2 ^ dg);
    dl = m1 ^ m2;                        // m of Delta
    const u64 delta = dl ^ d1 ^ d2 ^ (a.xrec == a.R + 1 ? a.xmask : 0ull);   // P1's opening
    if (a.trace) a.trace[(long long)a.R * a.trace_ld] = delta;
    if (delta) atomicOr(a.status, a.flag_verify);
  }
  __syncthreads();
  // The hashes of every Pi_Rec (r, the zetas, Delta): of message h thread 2 h hashes what its hasher
  // holds, thread 2 h + 1 what the receiver got, which is the same word unless a fault corrupts it
  // ([r]_2 at P1).
  for (int i0 = 0; i0 < 6 * (a.R + 2); i0 += 512) {
    const int i = i0 + tid, rec = i / 6, msg = (i % 6) >> 1;
    u64 w = 0;
    if (rec <= a.R) w = a.st[rec == 0 ? msg : 9 * rec + 6 + msg];
    else if (rec == a.R + 1) w = msg == 0 ? d1 : msg == 1 ? d2 : dl;
    if (rec == a.xrec && msg == 1 && (i & 1)) w ^= a.xmask;
    u32 h[8];
    sha256_word(w, h);
    bool diff = false;
#pragma unroll
    for (int q = 0; q < 8; ++q) diff |= __shfl_xor_sync(0xffffffffu, h[q], 1) != h[q];
    if (diff) bad = 1;
  }
  __syncthreads();
  if (tid == 0 && bad) atomicOr(a.status, a.flag_abort);
}

}  // namespace

void launch_gf_verify(cudaStream_t st, const GfVerify& a) {
  static const Coef cf = [] {
    return Coef{gf_inv(gf_mul(GF_X, GF_X ^ 1ull))};
  }();
  const long long nb = 8 * a.nw;
  cudaMemsetAsync(a.w, 0, sizeof(GfWork), st);
  launch_dep(k_gf_setup, (unsigned)((nb + 2047) / 2048), 256, 0, st, a, nb);
  long long g = (a.nw + 15) / 16;
  launch_dep(k_gf_sums, (unsigned)(g < 608 ? g : 608), 256, 0, st, a, cf);
  g = (nb / 2 + 255) / 256;
  u64 *x = a.x[0], *y = a.y[0], *xo = a.x[1], *yo = a.y[1];
  launch_dep(k_gf_vectors, (unsigned)(g < 1216 ? g : 1216), 256, 0, st, a, cf, x, y);
  long long D = nb, ld = nb;
  int k = 4;
  for (; (D + 1) / 2 > GF_TAIL; ++k) {
    const long long Dh = (D + 1) / 2, ldo = Dh;
    g = ((Dh + 1) / 2 + 127) / 128;
    launch_dep(k_gf_round, (unsigned)(g < 2432 ? g : 2432), 128, 0, st, a, cf, k + 1, D, x, y, ld, xo,
               yo, ldo);
    u64* t = x; x = xo; xo = t;
    t = y; y = yo; yo = t;
    D = Dh;
    ld = ldo;
  }
  launch_dep(k_gf_last, 1, 512, 0, st, a, cf, k, D, x, y, ld);
}

}  // namespace mpc3
