// The first rounds of a verification batch whose vectors are ring words times known weights.
//
// After Pi_Tran (Fig. MTP) a batch has x_i = w_i X_i and y_i = lift(Y_i), with X_i, Y_i shares in
// Z_2^64 and w_i a public GR element (r^i, or r^(i / 64) for the edaBit inner products).  The first
// K rounds of Pi_Reduce (at most 3, or 4 for long batches) fold blocks of B = 2^K elements with public
// weights, so they need no GR vector at all: with w_i = R_b T_j (i = B b + j) and
//   S^p_{j,j'} = sum_b R_b word^p_{b,j,j'},
//   word^0 = (X0 + X1)_j (Y0 + Y1)_j',  word^1 = -(X2_j Y3_j' + X3_j Y2_j'),
//   word^2 = X4_j (Y4 - Y5)_j' - X5_j Y4_j'   (the parties' cross terms; index = share component)
// every party sum of round k is sum V_j W_j' S^p_{j,j'} over the pairs (j, j') of one 2^k-block,
// V_j starting as T_j and W_j as 1, each multiplied by 1 - f or f after a round.  The vectors after
// K rounds are x_b = sum_j X_{b,j} (R_b V_j) and y_b = sum_j Y_{b,j} W_j.
//
// Per element this costs 3 B + 6 scalar-times-element sums for the S and the claim, one GR product
// (R_b V_j) and 12 scalar-times-element sums for the vectors, and 512 (1 + 12 / B) bytes of vectors,
// where materialising and folding takes 9 GR products, 10 Gram terms and 12 x 512 bytes of vectors
// several times over.  The sums grow with B, what the dense rounds still do shrinks with it: B = 8 on
// the CUDA cores (this file), B = 16 for long batches, whose sums run on the tensor cores (blk_sums_tc:
// a product of the blocks' words and R); a batch of 2^20 triples: 4.06 ms with B = 8 on the tensor
// cores, 3.38 ms with 16.
#include "gr_mul.cuh"
#include "kernels.h"

namespace mpc3 {

namespace {

// S and (CLAIM) the sums Z_{c,j} = sum_b R_b Z_c[B b + j] of the claim.  Rows of 64 words: party,
// j, j' (parties 1 and 2 only without MASK: x has no masks, X0 = X1 = X3 = X5 = 0), then c, j.
// Blocks take contiguous ranges of b, NB at a time: the words of the NB blocks in shared memory
// (from the staged shares), then thread t of the eight 64-thread groups adds coefficient t of the
// group's rows.  Bound by the multiply-adds (3 IMADs each).
template <int B, bool FULL>
struct BlkRows {
  static constexpr int NP = FULL ? 3 : 2;
  static constexpr int S = NP * B * B;
  static constexpr int N = S + (FULL ? 6 * B : 0);
  static constexpr int PER = (N + 7) / 8;      // rows of a group
  static constexpr int PAD = 8 * ((PER + 1) / 2 * 2);
};

template <int B, bool FULL>
__global__ void __launch_bounds__(512)
k_blk_sums(const BlkIn in, long long nb, int sh, const u64* R, u64* __restrict__ out) {
  grid_dep();
  using Rows = BlkRows<B, FULL>;
  constexpr int NB = 8;
  constexpr int G = Rows::PAD / 8;             // rows of a group, even
  constexpr int NC = FULL ? 18 : 8;            // staged share components
  __shared__ __align__(16) u64 wd[NB][Rows::PAD];
  __shared__ u64 raw[NC][NB * B];
  const int tid = threadIdx.x, t = tid & 63, g = tid >> 6;
  const long long b0 = nb * blockIdx.x / gridDim.x, b1 = nb * (blockIdx.x + 1) / gridDim.x;
  u64 acc[G];
#pragma unroll
  for (int q = 0; q < G; ++q) acc[q] = 0;
  for (long long b = b0; b < b1; b += NB) {
    const int cnt = (int)(b1 - b < NB ? b1 - b : NB);
    __syncthreads();
    for (int i = tid; i < NC * NB * B; i += 512) {
      const int c = i / (NB * B), e = i % (NB * B);
      const long long idx = b * B + e;
      const u64* src;
      if (FULL) src = c < 6 ? in.x[c] : c < 12 ? in.y[c - 6] : in.z + (c - 12) * in.ldz;
      else src = c == 0 ? in.x[2] : c == 1 ? in.x[4] : in.y[c - 2];
      raw[c][e] = (e < cnt * B && idx < in.D) ? src[idx] : 0ull;
    }
    __syncthreads();
    for (int i = tid; i < NB * Rows::PAD; i += 512) {
      const int bb = i / Rows::PAD, slot = i % Rows::PAD;
      const int row = (slot / G) * Rows::PER + slot % G;   // group's rows are contiguous
      u64 w = 0;
      if (slot % G < Rows::PER && row < Rows::N) {
        if (row < Rows::S) {
          const int p = row / (B * B) + (FULL ? 0 : 1);
          const int j = bb * B + (row / B) % B, k = bb * B + row % B;
          if (FULL) {
            if (p == 0) w = (raw[0][j] + raw[1][j]) * (raw[6][k] + raw[7][k]);
            else if (p == 1) w = 0ull - (raw[2][j] * raw[9][k] + raw[3][j] * raw[8][k]);
            else w = raw[4][j] * (raw[10][k] - raw[11][k]) - raw[5][j] * raw[10][k];
          } else {
            if (p == 1) w = 0ull - raw[0][j] * raw[5][k];
            else w = raw[1][j] * (raw[6][k] - raw[7][k]);
          }
        } else if (FULL) {
          const int q = row - Rows::S;
          w = raw[12 + q / B][bb * B + q % B];
        }
      }
      wd[bb][slot] = w;
    }
    __syncthreads();
    for (int bb = 0; bb < cnt; ++bb) {
      const u64 r = R[((b + bb) >> sh) * 64 + t];
#pragma unroll
      for (int q = 0; q < G; q += 2) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&wd[bb][g * G + q]);
        acc[q] += w.x * r;
        acc[q + 1] += w.y * r;
      }
    }
  }
  if (b0 < b1) {
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const int row = g * Rows::PER + q;
      if (q < Rows::PER && row < Rows::N)
        atomicAdd(reinterpret_cast<unsigned long long*>(out + row * 64 + t),
                  (unsigned long long)acc[q]);
    }
  }
}

// out[c][j] += sum_w R[w] Z_c[64 w + j] for the 6 components (the claim of a bit batch): 384 rows,
// 48 a group, as above.
__global__ void __launch_bounds__(512)
k_words_sums(const u64* z, long long ldz, long long nw, const u64* R,
             u64* __restrict__ out) {
  grid_dep();
  constexpr int NB = 8, G = 48;
  __shared__ __align__(16) u64 wd[NB][384];
  const int tid = threadIdx.x, t = tid & 63, g = tid >> 6;
  const long long b0 = nw * blockIdx.x / gridDim.x, b1 = nw * (blockIdx.x + 1) / gridDim.x;
  u64 acc[G];
#pragma unroll
  for (int q = 0; q < G; ++q) acc[q] = 0;
  for (long long b = b0; b < b1; b += NB) {
    const int cnt = (int)(b1 - b < NB ? b1 - b : NB);
    __syncthreads();
    for (int i = tid; i < NB * 384; i += 512) {
      const int c = i / (NB * 64), e = i % (NB * 64);
      wd[e >> 6][c * 64 + (e & 63)] = e < cnt * 64 ? z[c * ldz + b * 64 + e] : 0ull;
    }
    __syncthreads();
    for (int bb = 0; bb < cnt; ++bb) {
      const u64 r = R[(b + bb) * 64 + t];
#pragma unroll
      for (int q = 0; q < G; q += 2) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&wd[bb][g * G + q]);
        acc[q] += w.x * r;
        acc[q + 1] += w.y * r;
      }
    }
  }
  if (b0 < b1) {
#pragma unroll
    for (int q = 0; q < G; ++q)
      atomicAdd(reinterpret_cast<unsigned long long*>(out + (g * G + q) * 64 + t),
                (unsigned long long)acc[q]);
  }
}

// z_c += sum_j T_j Zr[c n + j] over the eight j of block (c, y): the claim from its row sums.
__global__ void __launch_bounds__(256)
k_blk_claim(const u64* T, const u64* Zr, int n, u64* __restrict__ z) {
  grid_dep();
  __shared__ u64 a[8][64], b[8][64], scr[4 * 128];
  const int tid = threadIdx.x, c = blockIdx.x, j0 = blockIdx.y * 8;
  const int cnt = n - j0 < 8 ? n - j0 : 8;
  for (int i = tid; i < cnt * 64; i += 256) {
    a[i >> 6][i & 63] = T[j0 * 64 + i];
    b[i >> 6][i & 63] = Zr[((long long)c * n + j0) * 64 + i];
  }
  __syncthreads();
  u64 lo = 0, hi = 0;
  for (int j = 0; j < cnt; ++j) gr_mac_part<16>(a[j], b[j], tid & 63, (tid >> 6) * 16, lo, hi);
  const u64 r = gr_finish<4>(lo, hi, scr, tid);
  if (tid < 64)
    atomicAdd(reinterpret_cast<unsigned long long*>(z + c * 64 + tid), (unsigned long long)r);
}

// out_c[b] = sum_{j < B} in_c[B b + j] G_j, G_j row (b >> sh) B + j of Gt (ROWS) or row j for every
// b, for the present components (words at or past D read as 0).  A warp takes an element, two
// coefficients a lane; VEC: 16-byte loads of the words (16-byte aligned components, B even).  Bound by
// the rows written; with 64 threads an element and a load a word it was bound by those loads (a load
// for each multiply-add): 264 us for 131072 edaBit blocks, now 182 us.
template <int B, bool ROWS, bool VEC>
__global__ void __launch_bounds__(256)
k_blk_combine(const BlkVec in, const BlkOut out, long long D, long long nb, int sh,
              const u64* Gt) {
  grid_dep();
  const int t = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * 8;
  u64 G[B][2];
  auto load_g = [&](const u64* g) {
#pragma unroll
    for (int j = 0; j < B; ++j) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(g + j * 64 + 2 * t);
      G[j][0] = v.x;
      G[j][1] = v.y;
    }
  };
  if (!ROWS) load_g(Gt);
  for (long long b = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); b < nb; b += stride) {
    if (ROWS) load_g(Gt + (b >> sh) * B * 64);
    const bool whole = (b + 1) * B <= D;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const u64* w = in.c[c];
      if (!w) continue;
      w += b * B;
      u64 s[B];
      if (VEC && whole) {
#pragma unroll
        for (int j = 0; j < B; j += 2) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(w + j);
          s[j] = v.x;
          s[j + 1 < B ? j + 1 : j] = v.y;
        }
      } else {
#pragma unroll
        for (int j = 0; j < B; ++j) s[j] = (whole || b * B + j < D) ? w[j] : 0ull;
      }
      u64 v0 = 0, v1 = 0;
#pragma unroll
      for (int j = 0; j < B; ++j) {
        v0 += s[j] * G[j][0];
        v1 += s[j] * G[j][1];
      }
      *reinterpret_cast<ulonglong2*>(out.c[c] + b * 64 + 2 * t) = make_ulonglong2(v0, v1);
    }
  }
}

// rows i < n of 64 words: the element 1
__global__ void k_ones(int n, u64* __restrict__ out) {
  grid_dep();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i < n * 64) out[i] = (i & 63) == 0 ? 1ull : 0ull;
}

inline unsigned blk_grid(long long nb) {
  long long g = (nb + 7) / 8;
  return (unsigned)(g > 152 ? 152 : g);
}

}  // namespace

int blk_rows(int B, bool full) { return (full ? 3 : 2) * B * B + (full ? 6 * B : 0); }

void launch_blk_sums(cudaStream_t st, const BlkIn& in, int B, bool full, long long nb, int sh,
                     const u64* R, u64* out) {
  const unsigned g = blk_grid(nb);
  auto go = [&](auto kern) { launch_dep(kern, g, 512, 0, st, in, nb, sh, R, out); };
  if (full) {
    if (B == 1) go(k_blk_sums<1, true>);
    else if (B == 2) go(k_blk_sums<2, true>);
    else if (B == 4) go(k_blk_sums<4, true>);
    else go(k_blk_sums<8, true>);
  } else {
    if (B == 1) go(k_blk_sums<1, false>);
    else if (B == 2) go(k_blk_sums<2, false>);
    else if (B == 4) go(k_blk_sums<4, false>);
    else go(k_blk_sums<8, false>);
  }
}

void launch_words_sums(cudaStream_t st, const u64* z, long long ldz, long long nw, const u64* R,
                       u64* out) {
  launch_dep(k_words_sums, blk_grid(nw), 512, 0, st, z, ldz, nw, R, out);
}

void launch_blk_claim(cudaStream_t st, const u64* T, const u64* Zr, int n, u64* z) {
  launch_dep(k_blk_claim, dim3(6, (unsigned)((n + 7) / 8)), 256, 0, st, T, Zr, n, z);
}

void launch_blk_combine(cudaStream_t st, const BlkVec& in, const BlkOut& out, int B, bool rows,
                        long long D, long long nb, int sh, const u64* G) {
  long long g = (nb + 7) / 8;
  if (g > 152 * 8) g = 152 * 8;
  bool vec = B >= 8;   // 16-byte loads of all components, or of none
  for (int c = 0; c < 6; ++c) vec = vec && (reinterpret_cast<uintptr_t>(in.c[c]) & 15) == 0;
  auto go = [&](auto kern) { launch_dep(kern, (unsigned)g, 256, 0, st, in, out, D, nb, sh, G); };
  if (rows) {
    if (B == 1) go(k_blk_combine<1, true, false>);
    else if (B == 2) go(k_blk_combine<2, true, false>);
    else if (B == 4) go(k_blk_combine<4, true, false>);
    else if (B == 16) go(vec ? k_blk_combine<16, true, true> : k_blk_combine<16, true, false>);
    else go(vec ? k_blk_combine<8, true, true> : k_blk_combine<8, true, false>);
  } else {
    if (B == 1) go(k_blk_combine<1, false, false>);
    else if (B == 2) go(k_blk_combine<2, false, false>);
    else if (B == 4) go(k_blk_combine<4, false, false>);
    else if (B == 16) go(vec ? k_blk_combine<16, false, true> : k_blk_combine<16, false, false>);
    else go(vec ? k_blk_combine<8, false, true> : k_blk_combine<8, false, false>);
  }
}

void launch_ones(cudaStream_t st, int n, u64* out) {
  launch_dep(k_ones, (n * 64 + 255) / 256, 256, 0, st, n, out);
}

}  // namespace mpc3
