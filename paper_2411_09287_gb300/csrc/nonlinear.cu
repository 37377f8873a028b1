// Elementwise kernels of the non-linear layers (Sec. 4.3) and of the layer-level calls.
#include "kernels.h"

namespace mpc3 {

namespace {

constexpr int TPB = 256;
inline unsigned grid_for(long long n) {
  long long g = (n + TPB - 1) / TPB;
  if (g < 1) g = 1;
  if (g > 152 * 32) g = 152 * 32;
  return (unsigned)g;
}
#define GRID_STRIDE(i, n) \
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (n); i += (long long)gridDim.x * blockDim.x)

// out = a - b (sub = 1) or a + b (sub = 0) over n words
__global__ void k_addsub(long long n, const u64* a, const u64* b, int sub,
                         u64* __restrict__ out) {
  grid_dep();
  GRID_STRIDE(i, n) { out[i] = sub ? a[i] - b[i] : a[i] + b[i]; }
}

// Pi_Tran of the edaBit inner products (rows e of dimension 64, weight r^(e0 + e) on row e) as ring
// words: entry (e0 + e) 64 + i of xm is the bit m_i of element e (components 2 and 4 of <m_i>, which
// has no mask), of component c of y 2^(i+1) <r'_i> with r' = b1 + b2 - 2 b1 b2 from the bits and the
// shared products.  The sources are plane-major: a 64 x 32 tile goes through shared memory, so that
// reads run along e and writes along i.
__global__ void __launch_bounds__(TPB)
k_eda_words(const u64* b1, const u64* b2, const u64* mbits,
            const u64* eprod, long long np, long long e0, long long ldy,
            u64* __restrict__ xm, u64* __restrict__ y) {
  grid_dep();
  __shared__ u64 tile[64][33];
  const long long N = 64 * np, eb = (long long)blockIdx.x * 32;
  const int q = blockIdx.y, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const u64* bits = q == 6 ? mbits : (q == 0 || q == 3) ? b1 : (q == 1 || q == 5) ? b2 : nullptr;
  for (int i = ty; i < 64; i += TPB / 32) {
    const long long j = (long long)i * np + eb + tx;   // np is a multiple of 64
    const u64 bit = bits ? (bits[j >> 6] >> (j & 63)) & 1ull : 0ull;
    u64 v = bit;
    if (q < 6) v = i < 63 ? (0ull - bit - 2ull * eprod[q * N + j]) << (i + 1) : 0ull;
    tile[i][tx] = v;
  }
  __syncthreads();
  u64* dst = (q < 6 ? y + q * ldy : xm) + (e0 + eb) * 64;
  for (int k = threadIdx.x; k < 64 * 32; k += TPB) dst[k] = tile[k & 63][k >> 6];
}

// 2x2 max-pool operands: for every window w = (b, ch, i, j) of a (B C, H, W) tensor (one
// component of n = B C H W words), left = [a ; c], right = [b ; d] with a = [2i][2j],
// b = [2i][2j+1], c = [2i+1][2j], d = [2i+1][2j+1]; nw windows, stage width np.
__global__ void k_window_gather(const u64* x, long long BC, long long H, long long W,
                                long long np, u64* __restrict__ left, u64* __restrict__ right) {
  grid_dep();
  const long long H2 = H / 2, W2 = W / 2, nw = BC * H2 * W2, n = BC * H * W;
  GRID_STRIDE(t, 6 * nw) {
    const int c = (int)(t / nw);
    const long long w = t % nw;
    const long long bc = w / (H2 * W2), ij = w % (H2 * W2), i = ij / W2, j = ij % W2;
    const u64* src = x + c * n + (bc * H + 2 * i) * W + 2 * j;
    left[c * np + w] = src[0];
    right[c * np + w] = src[1];
    left[c * np + nw + w] = src[W];
    right[c * np + nw + w] = src[W + 1];
  }
}

// out[c][k] = idx[k] >= 0 ? xs[c][idx[k]] : 0 for the six components (a local linear map)
__global__ void k_gather(const u64* xs, long long n_in, const long long* idx,
                         long long n_out, u64* __restrict__ out) {
  grid_dep();
  GRID_STRIDE(t, 6 * n_out) {
    const int c = (int)(t / n_out);
    const long long k = t % n_out;
    const long long j = idx[k];
    out[t] = (j >= 0 && j < n_in) ? xs[c * n_in + j] : 0ull;
  }
}

}  // namespace

// ---- launchers ------------------------------------------------------------------------------
void launch_addsub(cudaStream_t st, long long n, const u64* a, const u64* b, int sub, u64* out) {
  if (n <= 0) return;
  launch_dep(k_addsub, grid_for(n), TPB, 0, st, n, a, b, sub, out);
}
void launch_eda_words(cudaStream_t st, const u64* const bits[3], const u64* eprod, long long np,
                      long long e0, long long ldy, u64* xm, u64* y) {
  launch_dep(k_eda_words, dim3((unsigned)(np / 32), 7), TPB, 0, st, bits[0], bits[1], bits[2], eprod, np,
             e0, ldy, xm, y);
}

void launch_window_gather(cudaStream_t st, const u64* x, long long BC, long long H, long long W,
                          long long np, u64* left, u64* right) {
  launch_dep(k_window_gather, grid_for(6 * BC * (H / 2) * (W / 2)), TPB, 0, st, x, BC, H, W, np, left,
             right);
}

void launch_gather(cudaStream_t st, const u64* xs, long long n_in, const long long* idx,
                   long long n_out, u64* out) {
  if (n_out <= 0) return;
  launch_dep(k_gather, grid_for(6 * n_out), TPB, 0, st, xs, n_in, idx, n_out, out);
}

}  // namespace mpc3
