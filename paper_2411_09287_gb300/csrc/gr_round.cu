// The single-element steps of the batched verification over GR(2^64, 64), one launch per protocol
// round: everything of a Pi_Reduce round between its party sums and its folds (k_round_tail), the
// revealed challenges, the opened Delta, and the hashes of their Pi_Rec calls.
//
// These steps are chains of products of single GR elements: they move a few KB and are bound by
// latency alone.  As separate launches (reduction of the Gram blocks, quadratic combination, two
// inner-product finishes, the random sharing, Pi_Rec with its SHA-256, Lagrange weights, the next
// claim, the fold matrix, three trace copies) a round took about 95 us of kernel time, 20 us of it
// SHA-256 on one thread per digest.  Fused, with the products by the interpolation points x and
// 1 - x as shifts, the Lagrange weights from one square and one product, and the hash comparisons
// of all of a batch's Pi_Rec calls in one launch at its end, a round's tail is one launch.
#include "gr_mul.cuh"
#include "kernels.h"

namespace mpc3 {

namespace {

// The 64 words (8 ChaCha20 blocks) of a stream into w; threads lane = 0..7 each write 8 words.
__device__ __forceinline__ void stream64(const Key& k, u32 tag, u64 obj, int lane, u64* w) {
  u64 o[8];
  prf_block8(k, tag, obj, (u64)lane, o);
#pragma unroll
  for (int j = 0; j < 8; ++j) w[lane * 8 + j] = o[j];
}

// The messages of Pi_Rec of a shared element with streams (r1, r2, m), for the batch's hash
// comparison: rows of 64 words: the three values as their senders hold them ([r]_1, [r]_2, m at
// P0, P0, P1), as their hashers hold them ([r]_1 at P1, [r]_2 at P2, m at P2), and [r]_2 as it
// arrived at P1.
constexpr int REC_ROWS = 7;

// One Pi_Reduce round after its party sums (Fig. Reduce): h(0) and h(p2) by secure GR inner
// products, zeta' drawn and opened, the next claim z' = L0 h(0) + L1 (z - h(0)) + L2 h(p2), the
// fold element f and its multiplication matrix.  Block c < 6 computes component c of h(0), h(p2)
// and z'; block 6 the matrix, the Pi_Rec messages and the next round's cleared sums and zero rows; in a
// round over a matrix S (nvw > 0) the blocks from 7 on take the weights V_j, W_j, two each: times 1 - f
// or f by bit vwbit of j.  Every block derives zeta' from its streams, so that no block waits for another.
//
// L0 + L1 + L2 = 1 in both readings of the third point, hence z' = h(0) + L1 (z - 2 h(0)) +
// L2 (h(p2) - h(0)), with (points 0, 1, x) L2 = (z^2 - z) / (x (x - 1)), L1 = z - (z^2 - z) / x -
// L2, z = zeta'; (points 0, 1, 2) L2 = 2 z^2 - z, L1 = 4 z - 4 z^2, zeta = 2 zeta'.
//
// Everything that the keys alone decide (the streams, zeta', the Lagrange weights: a ChaCha20 block
// and two dependent products, half of the kernel's latency) comes before grid_dep, while the
// predecessor still runs; no memory that a kernel of the chain writes is touched there.
__global__ void __launch_bounds__(512) k_round_tail(const RoundTail a) {
  __shared__ u64 st[9][64];       // streams: H0 (r1, r2, g1), H2 (r1, r2, g1), zeta (r1, r2, m)
  __shared__ u64 zt[64], sq[64], L1[64], L2[64], inv[64], va[64], vb[64];
  __shared__ u64 S[9][64];        // reduced party sums: ee (3 parties), cross, oo
  __shared__ u64 scr[2][4 * 128];
  const int tid = threadIdx.x, blk = blockIdx.x;
  const int t = tid & 63, sub = tid & 255, grp = tid >> 8;
  if (tid < 72 && (blk < 7 || tid >= 48)) {
    const int s = tid >> 3, q = s % 3, g = s / 3;
    const u32 purpose = g == 0 ? P_VER_H0 : g == 1 ? P_VER_H2 : P_VER_ZETA;
    const Key& key = q == 0 ? a.k01 : q == 1 ? a.k02 : (g == 2 ? a.k12 : a.k01);
    const u32 comp = q == 0 ? C_R1 : q == 1 ? C_R2 : (g == 2 ? C_M12 : C_G1);
    stream64(key, make_tag(purpose, comp), a.obj, tid & 7, st[s]);
  } else if (tid >= 128 && tid < 192) {
    inv[t] = a.inv[t];   // a constant of the context
  }
  __syncthreads();
  if (tid < 64) {   // P1's opening: m - [r]_1 - [r]_2 as received
    const u64 r2 = st[7][t] ^ (t == a.fault.idx ? a.fault.mask : 0ull);
    zt[t] = st[8][t] - st[6][t] - r2;
  }
  __syncthreads();
  if (blk < 6) {
    // z^2 (the second group idles), then L2
    u64 r = gr_mul_par<4>(zt, zt, scr[grp], sub);
    if (tid < 64) sq[t] = a.mode == 1 ? r : r - zt[t];   // z^2, or z^2 - z
    __syncthreads();
    if (a.mode == 1) {
      if (tid < 64) {
        L2[t] = 2 * sq[t] - zt[t];
        L1[t] = 4 * zt[t] - 4 * sq[t];
      }
    } else {
      r = gr_mul_par<4>(inv, sq, scr[grp], sub);
      if (tid < 64) {
        // (z^2 - z) / x: the coefficients move down one, the constant term times
        // x^-1 = -(x^63 + x^3 + x^2 + 1)
        u64 u = t < 63 ? sq[t + 1] : 0ull;
        if (t == 0 || t == 2 || t == 3 || t == 63) u -= sq[0];
        L2[t] = r;
        L1[t] = zt[t] - u - r;
      }
    }
  }
  grid_dep();
  if (blk == 6) {
    __shared__ u64 fe[64];
    if (tid < 64) {
      const u64 f = a.mode == 1 ? 2 * zt[t] : zt[t];
      fe[t] = f;
      a.coef[t] = f;
      a.coef[384 + t] = (t == 0 ? 1ull : 0ull) - f;
      a.zp[t] = zt[t];
      if (a.trace) a.trace[t] = zt[t];
    } else if (tid < 128) {
      u64* l = a.rec;
      l[t] = st[6][t];             // [r]_1 sent by P0
      l[64 + t] = st[7][t];        // [r]_2 sent by P0
      l[128 + t] = st[8][t];       // m sent by P1
      l[192 + t] = st[6][t];       // [r]_1 held by P1
      l[256 + t] = st[7][t];       // [r]_2 held by P2
      l[320 + t] = st[8][t];       // m held by P2
      l[384 + t] = st[7][t] ^ (t == a.fault.idx ? a.fault.mask : 0ull);   // [r]_2 received by P1
    }
    __syncthreads();
    for (int i = tid; i < 4096; i += 512) a.MM[i] = gr_mulmat_at(fe, i >> 6, i & 63);
    for (long long i = tid; i < a.nzero; i += 512) a.zero[i] = 0ull;
    for (int i = tid; i < 12 * 64; i += 512)
      if (a.pad[i >> 6]) a.pad[i >> 6][i & 63] = 0ull;
    return;
  }
  if (blk > 6) {
    __shared__ u64 w[2][64], e[2][64];
    const int i = 2 * (blk - 7) + grp, j = i < a.nvw ? i : i - a.nvw;
    u64* X = (i < a.nvw ? a.V : a.W) + j * 64;
    if (sub < 64) {
      const u64 f = a.mode == 1 ? 2 * zt[t] : zt[t];
      w[grp][t] = ((j >> a.vwbit) & 1) ? f : (t == 0 ? 1ull : 0ull) - f;
      e[grp][t] = X[t];
    }
    __syncthreads();
    const u64 v = gr_mul_par<4>(w[grp], e[grp], scr[grp], sub);
    if (sub < 64) X[t] = v;
    return;
  }
  const bool msg = blk == 2 || blk == 4;   // the components m, which take the party sums
  if (msg) {
    for (int i = tid; i < 9 * 64; i += 512) {
      const int q = i >> 6, c = i & 63;
      const u64* s0 = a.sums + (q < 6 ? q : q + 3) * a.ld;   // ee, S01, oo
      u64 v = a.ld == 128 ? gr_reduce_at(s0, s0 + 64, c) : s0[c];
      if (q >= 3 && q < 6) {   // cross: S01 + S10
        const u64* s1 = a.sums + (q + 3) * a.ld;
        v += a.ld == 128 ? gr_reduce_at(s1, s1 + 64, c) : s1[c];
      }
      S[q][c] = v;
    }
  }
  __syncthreads();
  u64 r;
  u64 h0 = 0, z = 0;
  if (tid < 64) {
    u64 h2;
    if (msg) {
      // P0: Gamma = S0 + r1 + r2, sends Gamma - g1 to P2; P1: S1 + g1; P2: S2 + (received)
      u64 q[3], e[3];
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const u64 *s00 = S[p], *sx = S[3 + p], *s11 = S[6 + p];
        e[p] = s00[t];
        if (a.mode == 1) {   // p2 = 2: (1 - p2)^2 = 1, (1 - p2) p2 = -2, p2^2 = 4
          q[p] = s00[t] - 2 * sx[t] + 4 * s11[t];
        } else {             // p2 = x: S00 + x (Sx - 2 S00) + x^2 (S00 - Sx + S11)
          q[p] = s00[t] + gr_x_at(sx, t) - 2 * gr_x_at(s00, t) + gr_x2_at(s00, t) -
                 gr_x2_at(sx, t) + gr_x2_at(s11, t);
        }
      }
      const u64 g20 = e[0] + st[0][t] + st[1][t] - st[2][t];
      h0 = (e[1] + st[2][t]) + (e[2] + g20);
      const u64 g22 = q[0] + st[3][t] + st[4][t] - st[5][t];
      h2 = (q[1] + st[5][t]) + (q[2] + g22);
    } else {
      const int s = (blk == 0 || blk == 3) ? 0 : 1;   // [r]_1 or [r]_2
      h0 = st[s][t];
      h2 = st[3 + s][t];
    }
    z = a.z[blk * 64 + t];
    va[t] = z - 2 * h0;
    vb[t] = h2 - h0;
    if (a.trace) {
      a.trace[64 + blk * 64 + t] = h0;
      a.trace[448 + blk * 64 + t] = h2;
    }
  }
  __syncthreads();
  r = gr_mul_par<4>(grp ? L2 : L1, grp ? vb : va, scr[grp], sub);
  if (grp == 1 && sub < 64) sq[t] = r;
  __syncthreads();
  if (tid < 64) a.zo[blk * 64 + t] = h0 + r + sq[t];
}

// <v> random GR element (streams of `purpose`), opened with Pi_Rec; its messages go to rec.
__global__ void __launch_bounds__(64)
k_reveal(Key k01, Key k02, Key k12, u32 purpose, u64 obj, const MsgFault fault, u64* __restrict__ out,
         u64* __restrict__ rec) {
  __shared__ u64 st[3][64];
  const int t = threadIdx.x;
  if (t < 24) {
    const int s = t >> 3;
    stream64(s == 0 ? k01 : s == 1 ? k02 : k12,
             make_tag(purpose, s == 0 ? C_R1 : s == 1 ? C_R2 : C_M12), obj, t & 7, st[s]);
  }
  __syncthreads();
  grid_dep();   // the streams come from the keys alone
  const u64 r1 = st[0][t], r2 = st[1][t], m = st[2][t];
  const u64 r2in = r2 ^ (t == fault.idx ? fault.mask : 0ull);
  rec[t] = r1;
  rec[64 + t] = r2;
  rec[128 + t] = m;
  rec[192 + t] = r1;
  rec[256 + t] = r2;
  rec[320 + t] = m;
  rec[384 + t] = r2in;
  out[t] = m - r1 - r2in;
}

// The vectors' part of a Pi_Reduce round on a short claim, in one launch: the fold by the last round's
// f (fold set: a_2e + f (a_2e+1 - a_2e), D elements into ceil(D / 2)), and this round's party sums over
// the pairs of what it leaves (sums not null): blocks S00, S11 and the cross sum S01 + S10 as (e + o)(e'
// + o') - S00 - S11, 127 unreduced coefficients each.  A block takes one pair: its 24 products one a
// warp, then an eighth of each of the fifteen products of the sums a warp.  Bound by latency; on
// the tensor cores, whose tiles want 128 rows and whose kernels first split their operands, the two
// Gram launches and the fold of such a round took 36 us at 512 elements, this 16 us, 13 without the fold
// (20 and 15 us with a coefficient a thread and a load an operand and multiply-add).
__global__ void __launch_bounds__(256) k_small_round(const SmallRound a) {
  grid_dep();
  __shared__ __align__(16) u64 f[64], v[2][12][64], d[8][64], red[9][128];
  const int tid = threadIdx.x, t = tid & 63, g = tid >> 6, wp = tid >> 5, l = tid & 31;
  const long long pair = blockIdx.x;
  if (a.fold) {
    if (tid < 64) f[t] = a.f[t];
    __syncthreads();
    for (int i = wp; i < 24; i += 8) {   // (element, component): three of each warp
      const int e = i / 12, c = i % 12;
      const u64* src = a.in[c];
      const long long s0 = 2 * (2 * pair + e);
      ulonglong2 base = make_ulonglong2(0, 0), r = base;
      if (src && s0 < a.D) {   // uniform over the warp
        base = reinterpret_cast<const ulonglong2*>(src + s0 * 64)[l];
        if (s0 + 1 < a.D) r = reinterpret_cast<const ulonglong2*>(src + (s0 + 1) * 64)[l];
        *reinterpret_cast<ulonglong2*>(&d[wp][2 * l]) = make_ulonglong2(r.x - base.x, r.y - base.y);
        __syncwarp();
        Gr2 m;
        gr_mac2<64>(f, d[wp], l, 0, m);
        __syncwarp();
        u64* scr = d[wp];   // coefficients 64 .. 126
        scr[2 * l] = m.hi[0];
        scr[2 * l + 1] = m.hi[1];
        __syncwarp();
        r.x = base.x + m.lo[0] - gr_carry_at(scr, 2 * l);
        r.y = base.y + m.lo[1] - gr_carry_at(scr, 2 * l + 1);
        __syncwarp();
        reinterpret_cast<ulonglong2*>(a.out[c] + (2 * pair + e) * 64)[l] = r;
      }
      *reinterpret_cast<ulonglong2*>(&v[e][c][2 * l]) = r;
    }
  } else {
    for (int i = g; i < 24; i += 4) {
      const int e = i / 12, c = i % 12;
      const long long s0 = 2 * pair + e;
      v[e][c][t] = a.in[c] && s0 < a.D ? a.in[c][s0 * 64 + t] : 0ull;
    }
  }
  __syncthreads();
  if (!a.sums) return;
  // the parties' factors: P0 r_u, r_v; P2 m_v - [r_v]_2 (in places that are not needed any more)
  if (tid < 128) {
    const int e = tid >> 6;
    v[e][0][t] += v[e][1][t];
    v[e][6][t] += v[e][7][t];
    v[e][1][t] = v[e][10][t] - v[e][11][t];
  }
  __syncthreads();
  // sums over even, odd and even + odd elements; pairs of components (u, v) of x at c, of y at 6 + c;
  // warp wp takes the factors 8 wp .. 8 wp + 7 of every product
  Gr2 m[9];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (k == 2) {
      __syncthreads();
      for (int i = g; i < 12; i += 4) v[0][i][t] += v[1][i][t];
      __syncthreads();
    }
    u64(*w)[64] = v[k == 1 ? 1 : 0];
    Gr2 n;
    if ((a.in[0] || a.in[1]) && (a.in[6] || a.in[7])) gr_mac2<8>(w[0], w[6], l, wp * 8, m[3 * k]);
    if (a.in[2] && a.in[9]) gr_mac2<8>(w[2], w[9], l, wp * 8, n);
    if (a.in[8] && a.in[3]) gr_mac2<8>(w[8], w[3], l, wp * 8, n);
    m[3 * k + 1].sub(n);
    n = Gr2();
    if (a.in[4] && (a.in[10] || a.in[11])) gr_mac2<8>(w[4], w[1], l, wp * 8, m[3 * k + 2]);
    if (a.in[10] && a.in[5]) gr_mac2<8>(w[10], w[5], l, wp * 8, n);
    m[3 * k + 2].sub(n);
  }
  for (int p = 0; p < 8; ++p) {
    if (wp == p) {
#pragma unroll
      for (int q = 0; q < 9; ++q) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          red[q][2 * l + h] = m[q].lo[h] + (p ? red[q][2 * l + h] : 0ull);
          red[q][64 + 2 * l + h] = m[q].hi[h] + (p ? red[q][64 + 2 * l + h] : 0ull);
        }
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < 9 * 128; i += 256) {
    const int q = i >> 7, c = i & 127, k = q / 3, p = q % 3;
    u64 s = red[q][c];
    if (k == 2) s -= red[p][c] + red[3 + p][c];
    // S00 at 0, the cross sum at 3, S11 at 9 (blocks of 128 words)
    const int blk = (k == 0 ? 0 : k == 1 ? 9 : 3) + p;
    if (s)
      atomicAdd(reinterpret_cast<unsigned long long*>(a.sums + blk * 128 + c), (unsigned long long)s);
  }
}

// The end of Pi_InnerVerify in the block that finishes last: the inner product from the sums in acc, Delta
// opened, the status.  Every thread of the block calls it; st is 3 x 64 words of shared memory.
__device__ void inner_verify_open(const InnerVerify& a, u64 (*st)[64]) {
  __shared__ int last;
  const int tid = threadIdx.x, t = tid & 63;
  __threadfence();
  __syncthreads();
  if (tid == 0)
    last = atomicAdd(reinterpret_cast<unsigned long long*>(a.acc + 192), 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid < 24) {
    const int q = tid >> 3;
    stream64(q == 1 ? a.k02 : a.k01, make_tag(P_VER_DELTA, q == 0 ? C_R1 : q == 1 ? C_R2 : C_G1),
             a.obj, tid & 7, st[q]);
  }
  __syncthreads();
  if (tid >= 64) return;
  const u64 r1 = st[0][t], r2 = st[1][t], g1 = st[2][t];
  const u64 g2 = __ldcg(a.acc + t) + r1 + r2 - g1;                          // P0 -> P2
  const u64 m = (__ldcg(a.acc + 64 + t) + g1) + (__ldcg(a.acc + 128 + t) + g2);   // P1 <-> P2
  const u64 r2in = r2 ^ (t == a.fault.idx ? a.fault.mask : 0ull);
  a.rec[t] = r1;
  a.rec[64 + t] = r2;
  a.rec[128 + t] = m;
  a.rec[192 + t] = r1;
  a.rec[256 + t] = r2;
  a.rec[320 + t] = m;
  a.rec[384 + t] = r2in;
  const u64 d = m - r1 - r2in;
  if (a.trace) a.trace[t] = d;
  if (d != 0ull) atomicOr(a.status, a.flag);
}

// Pi_InnerVerify (Fig. DPV) on a claim of D elements, in one launch.  Row i < D: x'_i = alpha x_i
// (alpha random, shared, never opened) by Pi_Mult over GR, whose messages are Gamma_i - [Gamma_i]_1
// (P0 -> P2) and the two halves of m (P1 <-> P2); row D: alpha against -z.  Every block takes some
// rows and adds their party sums of sum_i x'_i y_i - alpha z,
//   S0 = sum r_u r_v, S1 = -sum (m_u [r_v]_1 + m_v [r_u]_1), S2 = sum m_u (m_v - [r_v]_2) - m_v [r_u]_2,
// to acc; the last one finishes the inner product, opens Delta (messages to rec) and sets `flag` in
// *status unless it is zero.  A row is ten GR products: the five of x'_i are added before they are
// reduced, so it is two dependent products and one ChaCha20 block of latency, about 8 us with the
// opening.  As separate launches (streams, multiplication matrices, three small GEMMs, messages,
// copies of x' and y, Gram sums, reductions: 40 launches) it took 150-200 us a batch.
__global__ void __launch_bounds__(256) k_inner_verify(const InnerVerify a) {
  __shared__ u64 al[6][64];           // r1, r2, m of alpha; r_a, m - r2
  __shared__ u64 u[6][64], v[6][64], st[3][64], scr[4 * 128];
  const int tid = threadIdx.x, t = tid & 63, i0 = (tid >> 6) * 16;
  if (tid < 24) {
    const int q = tid >> 3;
    stream64(q == 0 ? a.k01 : q == 1 ? a.k02 : a.k12,
             make_tag(P_VER_ALPHA, q == 0 ? C_R1 : q == 1 ? C_R2 : C_M12), a.obj, tid & 7, al[q]);
  }
  __syncthreads();
  if (tid < 64) {
    al[3][t] = al[0][t] + al[1][t];
    al[4][t] = al[2][t] - al[1][t];
  }
  grid_dep();   // alpha comes from the keys alone
  u64 lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  for (long long i = blockIdx.x; i <= a.D; i += gridDim.x) {
    __syncthreads();
    for (int e = tid; e < 6 * 64; e += 256) {
      const int c = e >> 6, w = e & 63;
      if (i < a.D) {
        u[c][w] = a.x[c] ? a.x[c][i * 64 + w] : 0ull;
        v[c][w] = a.y[c] ? a.y[c][i * 64 + w] : 0ull;
      } else {
        u[c][w] = al[c == 0 || c == 3 ? 0 : c == 1 || c == 5 ? 1 : 2][w];
        v[c][w] = 0ull - a.z[e];
      }
    }
    if (i < a.D) {   // u = x_i becomes x'_i; uniform over the block
      if (tid >= 232) {   // masks and [Gamma]_1, words 64 i .. 64 i + 63 of their streams
        const int q = (tid - 232) >> 3, l = tid & 7;
        u64 o[8];
        prf_block8(q == 1 ? a.k02 : a.k01, make_tag(P_VER_XA, q == 0 ? C_R1 : q == 1 ? C_R2 : C_G1),
                   a.obj, (u64)i * 8 + l, o);
#pragma unroll
        for (int w = 0; w < 8; ++w) st[q][l * 8 + w] = o[w];
      }
      __syncthreads();
      if (tid < 64) u[0][t] += u[1][t];   // r_x = [r]_1 + [r]_2 at P0
      __syncthreads();
      u64 gl = 0, gh = 0, nl = 0, nh = 0;
      gr_mac_part<16>(u[0], al[3], t, i0, gl, gh);   // P0: r_x r_a
      gr_mac_part<16>(u[4], al[4], t, i0, gl, gh);   // P2: m_x (m_a - [r_a]_2)
      gr_mac_part<16>(u[2], al[0], t, i0, nl, nh);   // P1: -(m_x [r_a]_1 + m_a [r_x]_1)
      gr_mac_part<16>(u[3], al[2], t, i0, nl, nh);
      gr_mac_part<16>(u[5], al[2], t, i0, nl, nh);   // P2: -[r_x]_2 m_a
      const u64 r = gr_finish<4>(gl - nl, gh - nh, scr, tid);
      if (tid < 64) {
        // Gamma = r_x r_a + r1 + r2; [m]_1 + [m]_2 takes [Gamma]_1 + (Gamma - [Gamma]_1)
        const u64 r1 = st[0][t], r2 = st[1][t], g1 = st[2][t], g2 = r1 + r2 - g1;
        const u64 m = r + g1 + g2;
        u[0][t] = r1; u[1][t] = r2; u[2][t] = m;
        u[3][t] = r1; u[4][t] = m; u[5][t] = r2;
      }
    }
    __syncthreads();
    if (tid < 64) {
      u[0][t] += u[1][t];
      v[0][t] += v[1][t];
      v[1][t] = v[4][t] - v[5][t];
    }
    __syncthreads();
    u64 nl = 0, nh = 0;
    gr_mac_part<16>(u[0], v[0], t, i0, lo[0], hi[0]);
    gr_mac_part<16>(u[2], v[3], t, i0, nl, nh);
    gr_mac_part<16>(v[2], u[3], t, i0, nl, nh);
    lo[1] -= nl; hi[1] -= nh;
    nl = nh = 0;
    gr_mac_part<16>(u[4], v[1], t, i0, lo[2], hi[2]);
    gr_mac_part<16>(v[4], u[5], t, i0, nl, nh);
    lo[2] -= nl; hi[2] -= nh;
  }
  __syncthreads();
  for (int q = 0; q < 3; ++q) {
    const u64 r = gr_finish<4>(lo[q], hi[q], scr, tid);
    if (tid < 64)
      atomicAdd(reinterpret_cast<unsigned long long*>(a.acc + q * 64 + t), (unsigned long long)r);
  }
  inner_verify_open(a, st);
}

// g += a b over the 64 factors (a, b in shared memory, 16-byte aligned), 16 at a time.
__device__ __forceinline__ void gr_mac_row(const u64* a, const u64* b, int l, Gr2& g) {
#pragma unroll 1
  for (int i0 = 0; i0 < 64; i0 += 16) gr_mac2<16>(a, b, l, i0, g);
}

// The same on long claims (few rounds asked for): a warp takes a row, two coefficients a lane.  Bound by
// the multiply-adds, where the form above, a row a block, is bound by its barriers and by two
// shared-memory reads for each multiply-add.  Products with an absent (zero) component are left out, as
// in the Gram sums.
constexpr int IVL_WARPS = 4;
__global__ void __launch_bounds__(IVL_WARPS * 32, 5) k_inner_verify_long(const InnerVerify a) {
  __shared__ __align__(16) u64 al[5][64];               // r1, r2, m of alpha; r_a, m - r2
  __shared__ __align__(16) u64 U[IVL_WARPS][5][64];     // r_x, m_x (P1), [r]_1, m_x (P2), [r]_2; then x'
  __shared__ __align__(16) u64 V[IVL_WARPS][5][64];     // r_y, m_y (P1), [r]_1, m_y (P2), m_y - [r]_2
  __shared__ __align__(16) u64 ST[IVL_WARPS][3][64];
  const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
  if (tid < 24) {
    const int q = tid >> 3;
    stream64(q == 0 ? a.k01 : q == 1 ? a.k02 : a.k12,
             make_tag(P_VER_ALPHA, q == 0 ? C_R1 : q == 1 ? C_R2 : C_M12), a.obj, tid & 7, al[q]);
  }
  __syncthreads();
  if (tid < 64) {
    al[3][tid] = al[0][tid] + al[1][tid];
    al[4][tid] = al[2][tid] - al[1][tid];
  }
  __syncthreads();
  grid_dep();   // alpha comes from the keys alone
  u64(*u)[64] = U[w], (*v)[64] = V[w], (*st)[64] = ST[w];
  auto get = [&](const u64* src, long long i) {
    return src ? reinterpret_cast<const ulonglong2*>(src + i * 64)[l] : make_ulonglong2(0, 0);
  };
  auto put = [&](u64* dst, u64 x, u64 y) {
    *reinterpret_cast<ulonglong2*>(dst + 2 * l) = make_ulonglong2(x, y);
  };
  Gr2 acc[3];
  const long long stride = (long long)gridDim.x * IVL_WARPS;
  for (long long i = blockIdx.x * (long long)IVL_WARPS + w; i <= a.D; i += stride) {
    const bool row = i < a.D;   // uniform over the warp; the last one is alpha against -z
    __syncwarp();
    ulonglong2 y[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      y[c] = row ? get(a.y[c], i) : get(a.z + c * 64, 0);
      if (!row) y[c] = make_ulonglong2(0ull - y[c].x, 0ull - y[c].y);
    }
    put(v[0], y[0].x + y[1].x, y[0].y + y[1].y);
    put(v[1], y[2].x, y[2].y);
    put(v[2], y[3].x, y[3].y);
    put(v[3], y[4].x, y[4].y);
    put(v[4], y[4].x - y[5].x, y[4].y - y[5].y);
    if (row) {
      const ulonglong2 x0 = get(a.x[0], i), x1 = get(a.x[1], i), x2 = get(a.x[2], i), x3 = get(a.x[3], i),
                       x4 = get(a.x[4], i), x5 = get(a.x[5], i);
      put(u[0], x0.x + x1.x, x0.y + x1.y);
      put(u[1], x2.x, x2.y);
      put(u[2], x3.x, x3.y);
      put(u[3], x4.x, x4.y);
      put(u[4], x5.x, x5.y);
      if (l < 24) {   // masks and [Gamma]_1, words 64 i .. 64 i + 63 of their streams
        const int q = l >> 3;
        u64 o[8];
        prf_block8(q == 1 ? a.k02 : a.k01, make_tag(P_VER_XA, q == 0 ? C_R1 : q == 1 ? C_R2 : C_G1),
                   a.obj, (u64)i * 8 + (l & 7), o);
#pragma unroll
        for (int k = 0; k < 8; ++k) st[q][(l & 7) * 8 + k] = o[k];
      }
      __syncwarp();
      Gr2 g, n;
      if (a.x[0] || a.x[1]) gr_mac_row(u[0], al[3], l, g);   // P0: r_x r_a
      if (a.x[4]) gr_mac_row(u[3], al[4], l, g);             // P2: m_x (m_a - [r_a]_2)
      if (a.x[2]) gr_mac_row(u[1], al[0], l, n);             // P1: -(m_x [r_a]_1 + m_a [r_x]_1)
      if (a.x[3]) gr_mac_row(u[2], al[2], l, n);
      if (a.x[5]) gr_mac_row(u[4], al[2], l, n);             // P2: -[r_x]_2 m_a
      g.sub(n);
      __syncwarp();
      put(u[0], g.hi[0], g.hi[1]);
      __syncwarp();
      u64 m[2], r1[2], r2[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        // Gamma = r_x r_a + r1 + r2; [m]_1 + [m]_2 takes [Gamma]_1 + (Gamma - [Gamma]_1)
        r1[h] = st[0][2 * l + h];
        r2[h] = st[1][2 * l + h];
        const u64 g1 = st[2][2 * l + h], g2 = r1[h] + r2[h] - g1;
        m[h] = g.lo[h] - gr_carry_at(u[0], 2 * l + h) + g1 + g2;
      }
      __syncwarp();
      put(u[0], r1[0] + r2[0], r1[1] + r2[1]);
      put(u[1], m[0], m[1]);
      put(u[2], r1[0], r1[1]);
      put(u[3], m[0], m[1]);
      put(u[4], r2[0], r2[1]);
    } else {
      put(u[0], al[3][2 * l], al[3][2 * l + 1]);
      put(u[1], al[2][2 * l], al[2][2 * l + 1]);
      put(u[2], al[0][2 * l], al[0][2 * l + 1]);
      put(u[3], al[2][2 * l], al[2][2 * l + 1]);
      put(u[4], al[1][2 * l], al[1][2 * l + 1]);
    }
    __syncwarp();
    auto has = [&](int c) { return !row || a.y[c]; };
    Gr2 n1, n2;
    if (has(0) || has(1)) gr_mac_row(u[0], v[0], l, acc[0]);
    if (has(3)) gr_mac_row(u[1], v[2], l, n1);
    if (has(2)) gr_mac_row(v[1], u[2], l, n1);
    if (has(4) || has(5)) gr_mac_row(u[3], v[4], l, acc[2]);
    if (has(4)) gr_mac_row(v[3], u[4], l, n2);
    acc[1].sub(n1);
    acc[2].sub(n2);
  }
  // the warps' sums: lo in the rows 0 .. 2 of u, hi in those of v
  __syncwarp();
  for (int q = 0; q < 3; ++q) {
    put(u[q], acc[q].lo[0], acc[q].lo[1]);
    put(v[q], acc[q].hi[0], acc[q].hi[1]);
  }
  __syncthreads();
  for (int e = tid; e < 2 * 192; e += IVL_WARPS * 32) {
    u64(*X)[5][64] = e < 192 ? U : V;
    const int q = (e % 192) >> 6, c = e & 63;
    u64 r = X[0][q][c];
    for (int k = 1; k < IVL_WARPS; ++k) r += X[k][q][c];
    X[0][q][c] = r;
  }
  __syncthreads();
  for (int e = tid; e < 192; e += IVL_WARPS * 32)
    atomicAdd(reinterpret_cast<unsigned long long*>(a.acc + e),
              (unsigned long long)gr_reduce_at(U[0][e >> 6], V[0][e >> 6], e & 63));
  inner_verify_open(a, ST[0]);
}


// The hash comparisons of n Pi_Rec calls of single GR elements (one block each): P1 sends H([r]_1)
// to P2, P2 sends H(m) to P0 and H([r]_2) to P1, and every receiver hashes what it received; a
// mismatch sets `flag` in *status.  Six digests of 512 bytes: the message schedules (plus round
// constants) of all 6 x 9 blocks first, by one thread each, then six threads run the rounds, whose
// dependent chain is what the launch takes.
__global__ void __launch_bounds__(64)
k_rec_hash(const u64* log, u32* status, u32 flag) {
  grid_dep();
  constexpr int LD = 55;             // words of one schedule step, 54 used
  __shared__ u32 wk[64 * LD];
  __shared__ u32 dig[6][8];
  const u64* rec = log + (long long)blockIdx.x * (REC_ROWS * 64);
  const int tid = threadIdx.x;
  if (tid < 54) {
    const int hsh = tid / 9, b = tid % 9;
    // P1's [r]_1, P2's m, P2's [r]_2; received: [r]_1 at P2, m at P0, [r]_2 at P1
    const int row = hsh == 0 ? 3 : hsh == 1 ? 5 : hsh == 2 ? 4 : hsh == 3 ? 0 : hsh == 4 ? 2 : 6;
    u32 w[16];
    if (b < 8) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const u64 v = rec[row * 64 + b * 8 + q];
        w[2 * q] = bswap32((u32)v);
        w[2 * q + 1] = bswap32((u32)(v >> 32));
      }
    } else {   // padding of a 512-byte message
#pragma unroll
      for (int q = 0; q < 16; ++q) w[q] = 0;
      w[0] = 0x80000000u;
      w[15] = 4096u;
    }
#pragma unroll
    for (int i = 0; i < 64; ++i) {
      u32 v = w[i & 15];
      if (i >= 16) {
        const u32 w15 = w[(i - 15) & 15], w2 = w[(i - 2) & 15];
        v += (rotr32(w15, 7) ^ rotr32(w15, 18) ^ (w15 >> 3)) + w[(i - 7) & 15] +
             (rotr32(w2, 17) ^ rotr32(w2, 19) ^ (w2 >> 10));
        w[i & 15] = v;
      }
      wk[i * LD + tid] = v + SHA_K[i];
    }
  }
  __syncthreads();
  if (tid < 6) {
    u32 h[8];
    sha256_init(h);
#pragma unroll 1
    for (int b = 0; b < 9; ++b) {
      const u32* W = wk + tid * 9 + b;
      u32 s[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) s[q] = h[q];
#pragma unroll 16
      for (int i = 0; i < 64; ++i) {
        const u32 S1 = rotr32(s[4], 6) ^ rotr32(s[4], 11) ^ rotr32(s[4], 25);
        const u32 ch = (s[4] & s[5]) ^ (~s[4] & s[6]);
        const u32 t1 = (s[7] + W[i * LD]) + S1 + ch;
        const u32 S0 = rotr32(s[0], 2) ^ rotr32(s[0], 13) ^ rotr32(s[0], 22);
        const u32 mj = (s[0] & s[1]) ^ (s[0] & s[2]) ^ (s[1] & s[2]);
        s[7] = s[6]; s[6] = s[5]; s[5] = s[4]; s[4] = s[3] + t1;
        s[3] = s[2]; s[2] = s[1]; s[1] = s[0]; s[0] = t1 + S0 + mj;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) h[q] += s[q];
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) dig[tid][q] = h[q];
  }
  __syncthreads();
  if (tid < 8 && (dig[0][tid] != dig[3][tid] || dig[1][tid] != dig[4][tid] ||
                  dig[2][tid] != dig[5][tid]))
    atomicOr(status, flag);
}

// One of the first rounds of a batch evaluated from a matrix S_{j,j'}, j, j' < n (the truncation
// batch's and the edaBits' bit pairs, n = 64: S_{j,j'} = sum_e R_e b1_{e,j} b2_{e,j'}; blocks of
// ring words, n <= 16, one matrix per party): with V_j, W_j the accumulated weights of the x and y
// side, the sums over the pairs (j, j') of one 2^k-block
//   out[2 a + b] += sum_{bit k-1 of j = a, of j' = b} V_j W_j' S_{j,j'},  192 words apart, party p
// at 64 p (the round's S00, S01, S10, S11; out must be zero on entry).  Block (j, c, p) takes the
// c-th eight j' of j's 2^k-block: the eight products share one reduction, so a block runs three
// dependent products' latency.  One thread group per j ran 2^k + 5 products one after another:
// 201 us for k = 6, 461 us for the six rounds of a bit batch.
__global__ void __launch_bounds__(256)
k_weighted_sums(const u64* V, const u64* W, const u64* S,
                int n, int k, u64* __restrict__ out) {
  grid_dep();
  __shared__ u64 w[8][64], s[8][64], T[2][64], v[64], scr[4 * 128];
  const int tid = threadIdx.x, t = tid & 63, part = tid >> 6;
  const int j = blockIdx.x, sh = k - 1, bs = 1 << k;
  const int m = bs < 8 ? bs : 8;
  const int j0 = (j & ~(bs - 1)) + blockIdx.y * 8;
  S += (long long)blockIdx.z * n * n * 64;
  for (int i = tid; i < m * 64; i += 256) {
    w[i >> 6][i & 63] = W[(j0 + (i >> 6)) * 64 + (i & 63)];
    s[i >> 6][i & 63] = S[((long long)j * n + j0 + (i >> 6)) * 64 + (i & 63)];
  }
  if (tid < 64) v[t] = V[j * 64 + t];
  __syncthreads();
  // halves of the block: with eight j' of a larger block they all lie in one half
  u64 lo[2] = {0, 0}, hi[2] = {0, 0};
  for (int q = 0; q < m; ++q) {
    u64 l = 0, h = 0;
    gr_mac_part<16>(w[q], s[q], t, part * 16, l, h);
    if (((j0 + q) >> sh) & 1) { lo[1] += l; hi[1] += h; }
    else { lo[0] += l; hi[0] += h; }
  }
  const int aj = (j >> sh) & 1;
  for (int b = 0; b < 2; ++b) {
    if (m == 8 && bs > 8 && (((j0 >> sh) & 1) != b)) continue;   // uniform over the block
    const u64 r = gr_finish<4>(lo[b], hi[b], scr, tid);
    if (tid < 64) T[b][t] = r;
    __syncthreads();
    const u64 y = gr_mul_par<4>(v, T[b], scr, tid);
    if (tid < 64)
      atomicAdd(reinterpret_cast<unsigned long long*>(out + 192 * (2 * aj + b) + 64 * blockIdx.z + t),
                (unsigned long long)y);
  }
}

// 64 words of zeros at each of the 12 rows (null: none)
__global__ void __launch_bounds__(768) k_zero_rows(const ZeroRows r) {
  grid_dep();
  u64* p = r.p[threadIdx.x >> 6];
  if (p) p[threadIdx.x & 63] = 0ull;
}

}  // namespace

void launch_zero_rows(cudaStream_t st, const ZeroRows& r) { launch_dep(k_zero_rows, 1, 768, 0, st, r); }

void launch_round_tail(cudaStream_t st, const RoundTail& a) {
  launch_dep(k_round_tail, 7 + a.nvw, 512, 0, st, a);
}

void launch_reveal(cudaStream_t st, Key k01, Key k02, Key k12, u32 purpose, u64 obj,
                   const MsgFault& fault, u64* out, u64* rec) {
  launch_dep(k_reveal, 1, 64, 0, st, k01, k02, k12, purpose, obj, fault, out, rec);
}

void launch_small_round(cudaStream_t st, const SmallRound& a) {
  const long long n = a.fold ? (a.D + 1) / 2 : a.D;
  launch_dep(k_small_round, (unsigned)((n + 1) / 2), 256, 0, st, a);
}

// Elements from which a claim takes a warp a row.  A verification of 2^16 products, by the elements that
// are left for this step: 1024: 444 us with a block a row, 465 with a warp; 2048: 422, 420; 4096: 412,
// 388; of 2^18 products with all of them left 7.50 ms, 6.35; of 2^19 truncations with 2^22 left (two
// components a side) 122 ms, 57.
constexpr long long IV_LONG = 2048;

void launch_inner_verify(cudaStream_t st, const InnerVerify& a) {
  if (a.D >= IV_LONG) {   // up to five blocks an SM
    const long long g = (a.D + IVL_WARPS) / IVL_WARPS;
    launch_dep(k_inner_verify_long, (unsigned)(g < 152 * 5 ? g : 152 * 5), IVL_WARPS * 32, 0, st, a);
    return;
  }
  const long long n = a.D + 1;   // four blocks an SM at most: rows beyond that are looped over
  launch_dep(k_inner_verify, (unsigned)(n < 608 ? n : 608), 256, 0, st, a);
}

void launch_rec_hash(cudaStream_t st, const u64* log, int n, u32* status, u32 flag) {
  if (n <= 0) return;
  static_assert(REC_ROWS * 64 == REC_WORDS, "record size");
  launch_dep(k_rec_hash, n, 64, 0, st, log, status, flag);
}

void launch_weighted_sums(cudaStream_t st, const u64* V, const u64* W, const u64* S, int n, int k,
                          int np, u64* out) {
  const int bs = 1 << k;
  launch_dep(k_weighted_sums, dim3(n, bs < 8 ? 1 : bs / 8, np), 256, 0, st, V, W, S, n, k, out);
}

}  // namespace mpc3
