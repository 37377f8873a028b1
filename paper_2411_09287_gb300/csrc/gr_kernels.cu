// Kernels on GR(2^64, 64) elements for the batched verification (Sec. 3):
//   random <.>^{l[x]} sharings (Pi_<.>^{l[x]}), powers r^i (Fig. MTP), reduction of Gram sums,
//   row scalings and sums, and the helpers of the truncation-pair batch (weights u_j and the
//   materialisation of the folded vectors).  The steps on single elements are in gr_round.cu.
// A GR element is 64 consecutive u64 coefficients.  A <.>^{l[x]}-shared vector of D elements uses
// the 6-component layout with component c at [c*D*64, (c+1)*D*64).
#include "gr_mul.cuh"
#include "kernels.h"

namespace mpc3 {

namespace {

constexpr int TPB = 256;

inline unsigned grid_for(long long n) {
  long long g = (n + TPB - 1) / TPB;
  if (g > (1ll << 20)) g = 1ll << 20;
  if (g < 1) g = 1;
  return (unsigned)g;
}

// ---- powers ---------------------------------------------------------------------------------
// Block b writes table[16 b .. 16 b + 15]: the squares a^(2^k) by one half of the block while the
// other multiplies the ones of 16 b's bits into a^(16 b), then four doublings of the row count
// (row 2^k + i = row i a^(2^k)), the block's threads spread over the products of each.  A block is a
// chain of about log2(n) + 4 products, so its time is their latency: 13.7 us for 1024
// rows (16.3 with 256 threads).
constexpr int POW_ROWS = 16, POW_LG = 4;
__global__ void __launch_bounds__(512)
k_gr_powers(const u64* a, long long n, u64* __restrict__ table) {
  grid_dep();
  __shared__ u64 rows[POW_ROWS][64], P[64], Pk[POW_LG][64], scr[8 * 128];
  const int tid = threadIdx.x, t = tid & 63;
  const long long start = (long long)blockIdx.x * POW_ROWS;
  if (tid < 64) {
    P[t] = a[t];
    rows[0][t] = t == 0 ? 1ull : 0ull;
  }
  __syncthreads();
  const int half = tid >> 8, quarter = tid >> 7, g = tid >> 6;
  for (int k = 0; k < POW_LG || (start >> k); ++k) {   // P = a^(2^k)
    const bool bit = (start >> k) & 1;
    if (k < POW_LG && tid < 64) Pk[k][t] = P[t];
    const u64 r = gr_mul_par<4>(half ? rows[0] : P, P, scr + half * 512, tid & 255);
    if ((tid & 255) < 64) {
      if (!half) P[t] = r;
      else if (bit) rows[0][t] = r;
    }
    __syncthreads();
  }
  u64 r = gr_mul_par<8>(rows[0], Pk[0], scr, tid);
  if (tid < 64) rows[1][t] = r;
  __syncthreads();
  r = gr_mul_par<4>(rows[half], Pk[1], scr + half * 512, tid & 255);
  if ((tid & 255) < 64) rows[2 + half][t] = r;
  __syncthreads();
  r = gr_mul_par<2>(rows[quarter], Pk[2], scr + quarter * 256, tid & 127);
  if ((tid & 127) < 64) rows[4 + quarter][t] = r;
  __syncthreads();
  r = gr_mul_par<1>(rows[g], Pk[3], scr + g * 128, t);
  rows[8 + g][t] = r;
  __syncthreads();
  for (int i = g; i < POW_ROWS && start + i < n; i += 8) table[(start + i) * 64 + t] = rows[i][t];
}

__global__ void __launch_bounds__(256) k_gr_mul1(const u64* a, const u64* b, u64* out) {
  grid_dep();
  __shared__ u64 sa[64], sb[64], scr[4 * 128];
  const int t = threadIdx.x;
  if (t < 64) sa[t] = a[t];
  else if (t < 128) sb[t - 64] = b[t - 64];
  __syncthreads();
  const u64 r = gr_mul_par<4>(sa, sb, scr, t);
  if (t < 64) out[t] = r;
}

// out_c = a_c + r b_c, one block per c
__global__ void __launch_bounds__(256)
k_gr_axpy(const u64* r, const u64* a, const u64* b,
          u64* __restrict__ out) {
  grid_dep();
  __shared__ u64 x[64], y[64], scr[4 * 128];
  const int t = threadIdx.x, c = blockIdx.x;
  if (t < 64) x[t] = r[t];
  else if (t < 128) y[t - 64] = b[c * 64 + t - 64];
  __syncthreads();
  const u64 p = gr_mul_par<4>(x, y, scr, t);
  if (t < 64) out[c * 64 + t] = a[c * 64 + t] + p;
}

// M[i] = multiplication matrix of the GR element src + i * stride, for i < n (one block each).
__global__ void __launch_bounds__(256)
k_gr_mulmat_batch(const u64* src, long long stride, u64* M) {
  grid_dep();
  __shared__ u64 e[64];
  if (threadIdx.x < 64) e[threadIdx.x] = src[blockIdx.x * stride + threadIdx.x];
  __syncthreads();
  u64* dst = M + (long long)blockIdx.x * 4096;
  for (int i = threadIdx.x; i < 64 * 64; i += blockDim.x) dst[i] = gr_mulmat_at(e, i >> 6, i & 63);
}

// out[c * rows + r] = in[r * cols + c] for r < rows, c < cols; entries with r * cols + c >= n
// read as 0 (32 x 32 tiles through shared memory).
__global__ void k_word_transpose(long long rows, long long cols, long long n, const u64* in,
                                 u64* out) {
  grid_dep();
  __shared__ u64 tile[32][33];
  const long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 256 threads: 8 rows per pass
  for (int k = ty; k < 32; k += 8) {
    const long long r = r0 + k, c = c0 + tx;
    const long long i = r * cols + c;
    tile[k][tx] = (r < rows && c < cols && i < n) ? in[i] : 0ull;
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    const long long c = c0 + k, r = r0 + tx;
    if (c < cols && r < rows) out[c * rows + r] = tile[tx][k];
  }
}

// out[i] = src[idx(i)] for rows of 64 words, idx(i) = ((i mul) / div) mod m (m = 0: no mod).
__global__ void k_gather_rows_affine(long long n, const u64* src, long long mul,
                                     long long div, long long m, u64* __restrict__ out) {
  grid_dep();
  for (long long i = blockIdx.x; i < n; i += gridDim.x) {
    long long idx = (i * mul) / div;
    if (m) idx %= m;
    out[i * 64 + threadIdx.x] = src[idx * 64 + threadIdx.x];
  }
}

// out[i] = sum_{h < n} in[h ld + i] for i < m words.
__global__ void __launch_bounds__(256)
k_sum_blocks(long long m, long long n, long long ld, const u64* in,
             u64* __restrict__ out) {
  grid_dep();
  const long long i = blockIdx.x * 256ll + threadIdx.x;
  if (i >= m) return;
  u64 v = 0;
#pragma unroll 8
  for (long long h = 0; h < n; ++h) v += in[h * ld + i];
  out[i] = v;
}

// out[c] = sum_{h < nper} in[c nper + h] for c < ncomp (rows of 64 words).
__global__ void k_block_rowsum(long long nper, const u64* in, u64* __restrict__ out) {
  grid_dep();
  const long long c = blockIdx.x;
  u64 v = 0;
#pragma unroll 8
  for (long long h = 0; h < nper; ++h) v += in[(c * nper + h) * 64 + threadIdx.x];
  out[c * 64 + threadIdx.x] = v;
}

// ---- inverse of the interpolation constant (Pi_Reduce with points 0, 1, x) --------------------
__device__ u64 gf2_64_mul(u64 a, u64 b) {   // GF(2)[x]/(x^64 + x^4 + x^3 + x + 1)
  u64 r = 0;
  for (int i = 63; i >= 0; --i) {
    const u64 top = r >> 63;
    r = (r << 1) ^ (top ? 0x1Bull : 0ull);
    if ((b >> i) & 1) r ^= a;
  }
  return r;
}

// out = (x (x - 1))^-1: the GF(2^64) inverse a^(2^64 - 2) of the residue, then Newton steps
// y <- y (2 - a y).
__global__ void k_gr_inverse(u64* out) {
  grid_dep();
  __shared__ u64 a[64], y[64], t1[64], scr[128];
  __shared__ u64 ybits;
  const int t = threadIdx.x;
  a[t] = t == 2 ? 1ull : t == 1 ? ~0ull : 0ull;   // x^2 - x
  __syncthreads();
  if (t == 0) {
    u64 bits = 0;
    for (int c = 0; c < 64; ++c) bits |= (a[c] & 1ull) << c;
    u64 acc = 1, p = bits;
    for (int k = 1; k < 64; ++k) {
      p = gf2_64_mul(p, p);
      acc = gf2_64_mul(acc, p);
    }
    ybits = acc;
  }
  __syncthreads();
  y[t] = (ybits >> t) & 1ull;
  __syncthreads();
  for (int it = 0; it < 7; ++it) {
    gr_mul_block(a, y, t1, scr);            // t1 = a y
    t1[t] = ((t == 0) ? 2ull : 0ull) - t1[t];
    __syncthreads();
    gr_mul_block(y, t1, y, scr);            // y = y (2 - a y)
  }
  out[t] = y[t];
}

// ---- fold of Gram sums ------------------------------------------------------------------------
// P: n matrices of 64x64 (P[a][b] = sum u_a v_b); out: n reduced GR elements.
__global__ void k_gr_fold_reduce(const u64* P, u64* __restrict__ out) {
  grid_dep();
  __shared__ u64 prod[128];
  const u64* M = P + (long long)blockIdx.x * 4096;
  const int s = threadIdx.x;   // 128 threads
  u64 v = 0;
  if (s < 127) {
    const int a0 = (s < 64) ? 0 : s - 63;
    const int a1 = (s < 64) ? s : 63;
    for (int a = a0; a <= a1; ++a) v += M[a * 64 + (s - a)];
  }
  prod[s] = (s < 127) ? v : 0ull;
  __syncthreads();
  if (s < 64) {
    const u64* h = prod + 64;
    u64 r = prod[s] - gr_hg(h, s);
    if (s < 7) {
      u64 h2[3];
      for (int m = 0; m < 3; ++m) h2[m] = gr_hg(h, 64 + m);
      u64 g = 0;
      if (s < 3) g += h2[s];
      if (s - 1 >= 0 && s - 1 < 3) g += h2[s - 1];
      if (s - 3 >= 0 && s - 3 < 3) g += h2[s - 3];
      if (s - 4 >= 0 && s - 4 < 3) g += h2[s - 4];
      r += g;
    }
    out[(long long)blockIdx.x * 64 + s] = r;
  }
}

__global__ void k_neg_copy(const u64* a, long long n, u64* __restrict__ out) {
  grid_dep();
  for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < n;
       w += (long long)gridDim.x * blockDim.x)
    out[w] = 0ull - a[w];
}

// ---- truncation-pair batch --------------------------------------------------------------------
// u_j = c_j + r c'_j with c_j = -2^(j+1), c'_j = -2 w_j (w_j the weight of bit j in >>_arith t).
__global__ void k_trunc_u(const u64* r, int t, u64* __restrict__ u) {
  grid_dep();
  const int j = blockIdx.x;
  const int c = threadIdx.x;
  u64 cj = 0ull - (2ull << j);                         // -2^(j+1) mod 2^64 (0 for j = 63)
  if (j == 63) cj = 0;
  u64 wj = 0;
  if (j >= t && j < 63) wj = 1ull << (j - t);
  if (j == 63) {
    wj = (1ull << (63 - t));
    for (int i = 64 - t; i < 64; ++i) wj += 1ull << i;
  }
  const u64 cpj = 0ull - 2 * wj;
  u[j * 64 + c] = r[c] * cpj + ((c == 0) ? cj : 0ull);
}

// Materialise a folded truncation-batch vector after kd rounds:
// out[e * (64 >> kd) + jp] = [R_e *] sum_{j >> kd == jp} VW_j * (-bit_j(words[e])).
// 256 threads = 4 groups of 64; group g handles every 4th output, thread t of a group computes
// coefficient t.  The product R_e * X uses one uniform 64-step loop per thread: step i adds
// R_i X_{(t-i) mod 64} to the low coefficient t (i <= t) or to the high coefficient 64 + t
// (i > t), followed by the reduction mod f.  VW in shared memory; R (optional) holds r^(2e).
__global__ void __launch_bounds__(256)
k_trunc_materialize(long long E, const u64* words, const u64* VW,
                    const u64* R, int kd, u64* __restrict__ out) {
  grid_dep();
  __shared__ u64 vw[64 * 64];
  __shared__ u64 xs[4][64], rr[4][64], hp[4][64];
  const int tid = threadIdx.x;
  const int g = tid >> 6, t = tid & 63;
  for (int i = tid; i < 4096; i += blockDim.x) vw[i] = VW[i];
  __syncthreads();
  const int per = 64 >> kd;
  const int bs = 1 << kd;
  const long long nout = E * per;
  for (long long ob = (long long)blockIdx.x * 4; ob < nout; ob += (long long)gridDim.x * 4) {
    const long long o = ob + g;
    const bool live = o < nout;
    u64 s = 0;
    long long e = 0;
    if (live) {
      e = o / per;
      const int jp = (int)(o % per);
      const u64 w = words[e] >> (jp * bs);
      for (int q = 0; q < bs; ++q)
        if ((w >> q) & 1ull) s -= vw[(jp * bs + q) * 64 + t];
    }
    if (R) {
      xs[g][t] = s;
      rr[g][t] = live ? R[e * 64 + t] : 0ull;
      __syncthreads();
      u64 lo = 0, hi = 0;
#pragma unroll 8
      for (int i = 0; i < 64; ++i) {
        const u64 pr = rr[g][i] * xs[g][(t - i) & 63];
        if (i <= t) lo += pr; else hi += pr;
      }
      hp[g][t] = (t < 63) ? hi : 0ull;   // coefficient 64 + t of the product (t = 63: none)
      __syncthreads();
      const u64* h = hp[g];
      s = lo - gr_hg(h, t);
      if (t < 7) {
        u64 h2[3];
        for (int m = 0; m < 3; ++m) h2[m] = gr_hg(h, 64 + m);
        u64 gg = 0;
        if (t < 3) gg += h2[t];
        if (t - 1 >= 0 && t - 1 < 3) gg += h2[t - 1];
        if (t - 3 >= 0 && t - 3 < 3) gg += h2[t - 3];
        if (t - 4 >= 0 && t - 4 < 3) gg += h2[t - 4];
        s += gg;
      }
    }
    if (live) out[o * 64 + t] = s;
    if (R) __syncthreads();   // xs/rr/hp are rewritten by the next iteration
  }
}


// out[e] = a[e] * b[e] in GR(2^64, 64) for e < n (rows of 64 words; out may alias a or b).
// One warp per element: lane l forms the product coefficients 4l .. 4l + 3 with a sliding window
// over b (zero-padded in shared memory, so no bounds tests), then the warp reduces mod f.  Word j
// of the padded b sits at j + j / 8, which makes the lanes' window loads (4 words apart)
// conflict-free.
__device__ __forceinline__ int padj(int j) { return j + (j >> 3); }

__global__ void __launch_bounds__(256)
k_gr_mul_rows(long long n, const u64* a, const u64* b, u64* out) {
  grid_dep();
  __shared__ u64 sa[8][64], sbp[8][216], sc[8][128];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  for (int i = l; i < 216; i += 32) sbp[w][i] = 0;
  __syncwarp();
  const long long stride = (long long)gridDim.x * 8;
  for (long long e = (long long)blockIdx.x * 8 + w; e < n; e += stride) {
    sa[w][l] = a[e * 64 + l];
    sa[w][l + 32] = a[e * 64 + l + 32];
    sbp[w][padj(64 + l)] = b[e * 64 + l];
    sbp[w][padj(96 + l)] = b[e * 64 + l + 32];
    __syncwarp();
    const int k0 = 4 * l;
    // window w_m = b[k0 + m - i] = padded word 64 + k0 + m - i
    u64 w0 = sbp[w][padj(64 + k0)], w1 = sbp[w][padj(65 + k0)], w2 = sbp[w][padj(66 + k0)],
        w3 = sbp[w][padj(67 + k0)];
    u64 c0 = 0, c1 = 0, c2 = 0, c3 = 0;
#pragma unroll
    for (int i = 0; i < 64; ++i) {
      const u64 ai = sa[w][i];
      c0 += ai * w0;
      c1 += ai * w1;
      c2 += ai * w2;
      c3 += ai * w3;
      w3 = w2;
      w2 = w1;
      w1 = w0;
      w0 = sbp[w][padj(63 + k0 - i)];
    }
    sc[w][k0] = c0;
    sc[w][k0 + 1] = c1;
    sc[w][k0 + 2] = c2;
    sc[w][k0 + 3] = c3;
    __syncwarp();
    const u64* h = sc[w] + 64;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int t = l + 32 * half;
      u64 v = sc[w][t] - gr_hg(h, t);
      if (t < 7) {
        u64 h2[3];
        for (int m = 0; m < 3; ++m) h2[m] = gr_hg(h, 64 + m);
        u64 g = 0;
        if (t < 3) g += h2[t];
        if (t - 1 >= 0 && t - 1 < 3) g += h2[t - 1];
        if (t - 3 >= 0 && t - 3 < 3) g += h2[t - 3];
        if (t - 4 >= 0 && t - 4 < 3) g += h2[t - 4];
        v += g;
      }
      out[e * 64 + t] = v;
    }
    __syncwarp();
  }
}

// out[c] += sum_{e < n} A[c][e] * R[e] for c < nrows <= NR: GR elements R[e] (rows of 64 words)
// scaled by ring scalars and summed (e.g. sum_e r^(2e) p_c[e] for the truncation batch).  Each
// block takes a contiguous slice of e, 256 e at a time: the slice of A is staged in shared memory
// as [e][c] (a broadcast read per e), and the four 64-thread groups take every fourth e, thread t
// coefficient t of every row c; the groups' sums are added in shared memory, then atomically.
// Bound by the rows of R (512 bytes an e) once the grid fills the GPU; 4096 e a block left one
// block for the smallest batches and 256 for 2^20 (361 and 413 us).
template <int NR>
__global__ void __launch_bounds__(256)
k_scalar_gr_sum(long long n, const u64* A, long long lda, int nrows,
                const u64* R, u64* __restrict__ out) {
  grid_dep();
  __shared__ __align__(16) u64 as[256][NR];
  const int t = threadIdx.x & 63, grp = threadIdx.x >> 6;
  const long long per = (n + gridDim.x - 1) / gridDim.x;
  const long long e0 = per * blockIdx.x;
  const long long e1 = (e0 + per < n) ? e0 + per : n;
  u64 acc[NR];
#pragma unroll
  for (int c = 0; c < NR; ++c) acc[c] = 0;
  for (long long eb = e0; eb < e1; eb += 256) {
    const int cnt = (int)(e1 - eb < 256 ? e1 - eb : 256);
    __syncthreads();
    for (int i = threadIdx.x; i < NR * 256; i += 256) {
      const int c = i >> 8, k = i & 255;
      as[k][c] = (c < nrows && k < cnt) ? A[c * lda + eb + k] : 0ull;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = grp; k < cnt; k += 4) {
      const u64 r = R[(eb + k) * 64 + t];
#pragma unroll
      for (int c = 0; c < NR; c += 2) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&as[k][c]);
        acc[c] += w.x * r;
        acc[c + 1] += w.y * r;
      }
    }
  }
  __syncthreads();
  u64* red = &as[0][0];   // [grp][c][t]: 4 x NR x 64 of the 256 x NR words
#pragma unroll
  for (int c = 0; c < NR; ++c) red[(grp * NR + c) * 64 + t] = acc[c];
  __syncthreads();
  for (int i = threadIdx.x; i < nrows * 64; i += 256) {
    const u64 v = red[i] + red[NR * 64 + i] + red[2 * NR * 64 + i] + red[3 * NR * 64 + i];
    atomicAdd(reinterpret_cast<unsigned long long*>(out + i), (unsigned long long)v);
  }
}

}  // namespace

// ---- launchers --------------------------------------------------------------------------------
void launch_gr_powers(cudaStream_t st, const u64* a, long long n, u64* table) {
  if (n <= 0) return;
  launch_dep(k_gr_powers, (unsigned)((n + POW_ROWS - 1) / POW_ROWS), 512, 0, st, a, n, table);
}

void launch_gr_mul1(cudaStream_t st, const u64* a, const u64* b, u64* out) {
  launch_dep(k_gr_mul1, 1, 256, 0, st, a, b, out);
}

void launch_gr_axpy(cudaStream_t st, int n, const u64* r, const u64* a, const u64* b, u64* out) {
  if (n > 0) launch_dep(k_gr_axpy, n, 256, 0, st, r, a, b, out);
}

void launch_gr_mulmat_batch(cudaStream_t st, long long n, const u64* src, long long stride,
                            u64* M) {
  if (n <= 0) return;
  launch_dep(k_gr_mulmat_batch, (unsigned)n, 256, 0, st, src, stride, M);
}

void launch_word_transpose(cudaStream_t st, long long rows, long long cols, long long n,
                           const u64* in, u64* out) {
  if (rows <= 0 || cols <= 0) return;
  dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((rows + 31) / 32));
  launch_dep(k_word_transpose, grid, 256, 0, st, rows, cols, n, in, out);
}

void launch_gather_rows_affine(cudaStream_t st, long long n, const u64* src, long long mul,
                               long long div, long long m, u64* out) {
  if (n <= 0) return;
  launch_dep(k_gather_rows_affine, (unsigned)(n < 65536 ? n : 65536), 64, 0, st, n, src, mul, div, m, out);
}

void launch_block_rowsum(cudaStream_t st, int ncomp, long long nper, const u64* in, u64* out) {
  if (ncomp <= 0) return;
  launch_dep(k_block_rowsum, (unsigned)ncomp, 64, 0, st, nper, in, out);
}

void launch_sum_blocks(cudaStream_t st, long long m, long long n, long long ld, const u64* in,
                       u64* out) {
  if (m <= 0) return;
  launch_dep(k_sum_blocks, (unsigned)((m + 255) / 256), 256, 0, st, m, n, ld, in, out);
}

void launch_gr_inverse(cudaStream_t st, u64* out) { launch_dep(k_gr_inverse, 1, 64, 0, st, out); }

void launch_gr_fold_reduce(cudaStream_t st, const u64* P, int n, u64* out) {
  if (n <= 0) return;
  launch_dep(k_gr_fold_reduce, n, 128, 0, st, P, out);
}

void launch_neg_copy(cudaStream_t st, const u64* a, long long n, u64* out) {
  if (n <= 0) return;
  launch_dep(k_neg_copy, grid_for(n), TPB, 0, st, a, n, out);
}

void launch_trunc_u(cudaStream_t st, const u64* r, int t, u64* u) {
  launch_dep(k_trunc_u, 64, 64, 0, st, r, t, u);
}

void launch_trunc_materialize(cudaStream_t st, long long E, const u64* words, const u64* VW,
                              const u64* R, int kd, u64* out) {
  if (E <= 0) return;
  long long nout = E * (64 >> kd);
  long long g = (nout + 3) / 4;
  if (g > 152 * 16) g = 152 * 16;
  launch_dep(k_trunc_materialize, (unsigned)g, 256, 0, st, E, words, VW, R, kd, out);
}

void launch_gr_mul_rows(cudaStream_t st, long long n, const u64* a, const u64* b, u64* out) {
  if (n <= 0) return;
  long long g = (n + 7) / 8;
  if (g > 152 * 8) g = 152 * 8;
  launch_dep(k_gr_mul_rows, (unsigned)g, 256, 0, st, n, a, b, out);
}

void launch_scalar_gr_sum(cudaStream_t st, long long n, const u64* A, long long lda, int nrows,
                          const u64* R, u64* out) {
  if (n <= 0 || nrows <= 0) return;
  // 64 e a block while the batch is small, then eight blocks an SM
  long long g = (n + 63) / 64;
  if (g > 152 * 8) g = 152 * 8;
  auto go = [&](auto kern) { launch_dep(kern, (unsigned)g, 256, 0, st, n, A, lda, nrows, R, out); };
  if (nrows <= 2) go(k_scalar_gr_sum<2>);
  else if (nrows <= 6) go(k_scalar_gr_sum<6>);
  else if (nrows <= 12) go(k_scalar_gr_sum<12>);
  else go(k_scalar_gr_sum<16>);
}

}  // namespace mpc3
