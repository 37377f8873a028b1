// Kernels of the non-linear layers (Sec. 4.3): Boolean <.>^1 sharings over Z_2 stored bit-sliced
// (64 elements per u64 word, planes of n_pad / 64 words), AND gates (Pi_Mult over Z_2), the pieces
// of daBits / edaBits / the MSB carry circuit / B2A.
//
// Layouts.  A Boolean sharing of nw words is 6 nw words, component c at [c nw, (c+1) nw) in the
// order P0.[r]_1, P0.[r]_2, P1.m, P1.[r]_1, P2.m, P2.[r]_2 (as for arithmetic sharings).  A
// Boolean stream's bit i is bit i % 64 of ChaCha20 word i / 64, so word w of a bit-sliced
// operand is stream word w.
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

// ---- AND gates (Fig. MultP over Z_2: + and - are XOR, products are AND) ------------------------
__global__ void k_and_offline(const u64* __restrict__ xs, const u64* __restrict__ ys, long long nw,
                              Key k01, Key k02, u32 tr1, u32 tr2, u32 tg1, u64 obj,
                              u64* __restrict__ zs, u64* __restrict__ g2_out) {
  GRID_STRIDE(i, nw) {
    const u64 r1 = prf_word(k01, tr1, obj, (u64)i);
    const u64 r2 = prf_word(k02, tr2, obj, (u64)i);
    const u64 g1 = prf_word(k01, tg1, obj, (u64)i);
    const u64 rx = xs[i] ^ xs[nw + i];
    const u64 ry = ys[i] ^ ys[nw + i];
    g2_out[i] = (rx & ry) ^ r1 ^ r2 ^ g1;   // [Gamma]_2 = Gamma - [Gamma]_1, P0 -> P2
    zs[i] = r1;
    zs[nw + i] = r2;
    zs[3 * nw + i] = r1;
    zs[5 * nw + i] = r2;
  }
}

__global__ void k_and_online(const u64* __restrict__ xs, const u64* __restrict__ ys, long long nw,
                             Key k01, u32 tg1, u64 obj, const u64* __restrict__ g2_in,
                             u64* __restrict__ p1_out, u64* __restrict__ p2_out) {
  GRID_STRIDE(i, nw) {
    const u64 g1 = prf_word(k01, tg1, obj, (u64)i);
    p1_out[i] = (xs[2 * nw + i] & ys[3 * nw + i]) ^ (ys[2 * nw + i] & xs[3 * nw + i]) ^ g1;
    const u64 mx = xs[4 * nw + i], my = ys[4 * nw + i];
    p2_out[i] = (mx & my) ^ (mx & ys[5 * nw + i]) ^ (my & xs[5 * nw + i]) ^ g2_in[i];
  }
}

__global__ void k_xor_finish(long long nw, const u64* __restrict__ p1_own, const u64* __restrict__ p1_in,
                             const u64* __restrict__ p2_own, const u64* __restrict__ p2_in,
                             u64* __restrict__ zs) {
  GRID_STRIDE(i, nw) {
    zs[2 * nw + i] = p1_own[i] ^ p1_in[i];
    zs[4 * nw + i] = p2_own[i] ^ p2_in[i];
  }
}

// ---- bits <-> arithmetic sharings ---------------------------------------------------------------
// out (6 n arithmetic words) = the sharing of the n bits: kind 0 (eta01 bits): [r]_1 = -b;
// kind 1 (eta02 bits): [r]_2 = -b; kind 2 (eta12 bits): m = b (reading A1).
__global__ void k_bits_to_arith(const u64* __restrict__ bits, long long n, int kind, u64* __restrict__ out) {
  GRID_STRIDE(i, n) {
    const u64 b = (bits[i >> 6] >> (i & 63)) & 1ull;
    const u64 nb = 0ull - b;
    out[i] = kind == 0 ? nb : 0ull;
    out[n + i] = kind == 1 ? nb : 0ull;
    out[2 * n + i] = kind == 2 ? b : 0ull;
    out[3 * n + i] = kind == 0 ? nb : 0ull;
    out[4 * n + i] = kind == 2 ? b : 0ull;
    out[5 * n + i] = kind == 1 ? nb : 0ull;
  }
}

// out = a + b - 2 c over all words (linear combination of sharings)
__global__ void k_lin_apb_m2c(long long n, const u64* __restrict__ a, const u64* __restrict__ b,
                              const u64* __restrict__ c, u64* __restrict__ out) {
  GRID_STRIDE(i, n) { out[i] = a[i] + b[i] - 2ull * c[i]; }
}

// ---- edaBit inner products: z_e = sum_i m_{i,e} (2^(i+1) r'_{i,e}), plane-major inputs ---------
// X = <m_i> (only m components non-zero), Y = r' (all components); Pi_Inner (Fig. DPP) per e.
// P0's part: Gamma_e = sum_i r_{x,i} r_{y,i} + [r_z]_1 + [r_z]_2 with r_x = [r]_1 + [r]_2 = 0 for
// every <m_i> (an eta12 bit has no mask), so Gamma_e is the output mask itself.
__global__ void k_eda_inner_offline(long long np, Key k01, Key k02, u32 tr1, u32 tr2, u32 tg1,
                                    u64 obj, u64* __restrict__ zs, u64* __restrict__ g2_out) {
  GRID_STRIDE(e, np) {
    const u64 r1 = prf_word(k01, tr1, obj, (u64)e);
    const u64 r2 = prf_word(k02, tr2, obj, (u64)e);
    const u64 g1 = prf_word(k01, tg1, obj, (u64)e);
    g2_out[e] = r1 + r2 - g1;
    zs[e] = r1;
    zs[np + e] = r2;
    zs[3 * np + e] = r1;
    zs[5 * np + e] = r2;
  }
}

__device__ __forceinline__ u64 shl_mod(u64 v, int s) { return s < 64 ? v << s : 0ull; }

__global__ void k_eda_inner_online(const u64* __restrict__ mbits, const u64* __restrict__ rp,
                                   long long np, Key k01, u32 tg1, u64 obj,
                                   const u64* __restrict__ g2_in, u64* __restrict__ p1_out,
                                   u64* __restrict__ p2_out) {
  const long long N = 64 * np;
  GRID_STRIDE(e, np) {
    u64 s1 = 0, s2 = 0;
    for (int i = 0; i < 64; ++i) {
      const long long j = (long long)i * np + e;
      const u64 m = (mbits[j >> 6] >> (j & 63)) & 1ull;   // m_x of <m_i> (P1 and P2 copies)
      const int sh = i + 1;
      const u64 ry1 = shl_mod(rp[3 * N + j], sh);
      const u64 my2 = shl_mod(rp[4 * N + j], sh), ry2 = shl_mod(rp[5 * N + j], sh);
      // P1: -(m_x [r_y]_1 + m_y [r_x]_1), [r_x]_1 = 0;  P2: m_x m_y - m_x [r_y]_2 - m_y [r_x]_2
      s1 -= m * ry1;
      s2 += m * my2 - m * ry2;
    }
    p1_out[e] = s1 + prf_word(k01, tg1, obj, (u64)e);
    p2_out[e] = s2 + g2_in[e];
  }
}

// ra = sum_i 2^i (<m_i> + <r'_i>) - <z>   (all six components)
__global__ void k_eda_compose(const u64* __restrict__ mbits, const u64* __restrict__ rp,
                              const u64* __restrict__ z, long long np, u64* __restrict__ ra) {
  const long long N = 64 * np;
  GRID_STRIDE(t, 6 * np) {
    const int c = (int)(t / np);
    const long long e = t % np;
    u64 acc = 0;
    for (int i = 0; i < 64; ++i) {
      const long long j = (long long)i * np + e;
      const u64 m = (c == 2 || c == 4) ? (mbits[j >> 6] >> (j & 63)) & 1ull : 0ull;
      acc += (m + rp[c * N + j]) << i;
    }
    ra[c * np + e] = acc - z[c * np + e];
  }
}

// ---- MSB carry circuit ------------------------------------------------------------------------
// Leaves: G_i = r[i] AND Delta_i (all components), P_i = r[i] XOR Delta_i (m components), i < 63;
// leaf 63 = (0, 1).  rbits, G, P: Boolean sharings of 64 planes of W words; dplanes: 64 x W.
__global__ void k_msb_leaves(const u64* __restrict__ rbits, const u64* __restrict__ dplanes, long long W,
                             u64* __restrict__ G, u64* __restrict__ P) {
  const long long NW = 64 * W;
  GRID_STRIDE(t, NW) {
    const int i = (int)(t / W);
    const u64 d = dplanes[t];
    for (int c = 0; c < 6; ++c) {
      const u64 r = rbits[c * NW + t];
      const bool m = (c == 2 || c == 4);
      if (i < 63) {
        G[c * NW + t] = r & d;
        P[c * NW + t] = m ? (r ^ d) : r;
      } else {
        G[c * NW + t] = 0;
        P[c * NW + t] = m ? ~0ull : 0ull;
      }
    }
  }
}

// Level inputs: X = [P_hi(k), k < C ; P_hi(k), k < C (not at the root)],
//               Y = [G_lo(k) ; P_lo(k)], hi = 2k + 1, lo = 2k.  G, P have 2C planes.
__global__ void k_msb_gather(const u64* __restrict__ G, const u64* __restrict__ P, int C, int root,
                             long long W, u64* __restrict__ X, u64* __restrict__ Y) {
  const int planes = root ? C : 2 * C;
  const long long nin = 2ll * C * W, nout = (long long)planes * W;
  GRID_STRIDE(t, nout) {
    const int p = (int)(t / W);
    const long long w = t % W;
    const int k = p < C ? p : p - C;
    for (int c = 0; c < 6; ++c) {
      X[c * nout + t] = P[c * nin + (long long)(2 * k + 1) * W + w];
      Y[c * nout + t] = p < C ? G[c * nin + (long long)(2 * k) * W + w]
                              : P[c * nin + (long long)(2 * k) * W + w];
    }
  }
}

// G'(k) = G_hi(k) XOR Z(k), P'(k) = Z(C + k)
__global__ void k_msb_combine(const u64* __restrict__ G, const u64* __restrict__ Z, int C, int root,
                              long long W, u64* __restrict__ Gout, u64* __restrict__ Pout) {
  const long long nin = 2ll * C * W, nz = (long long)(root ? C : 2 * C) * W, nout = (long long)C * W;
  GRID_STRIDE(t, nout) {
    const int k = (int)(t / W);
    const long long w = t % W;
    for (int c = 0; c < 6; ++c) {
      Gout[c * nout + t] = G[c * nin + (long long)(2 * k + 1) * W + w] ^ Z[c * nz + t];
      if (!root) Pout[c * nout + t] = Z[c * nz + (long long)(C + k) * W + w];
    }
  }
}

// msb = r[63] XOR G_root XOR Delta_63 (public, m components); ge = NOT msb when `negate`.
__global__ void k_msb_out(const u64* __restrict__ rbits, const u64* __restrict__ Groot,
                          const u64* __restrict__ d63, long long W, int negate, u64* __restrict__ out) {
  const long long NW = 64 * W;
  GRID_STRIDE(w, W) {
    for (int c = 0; c < 6; ++c) {
      u64 v = rbits[c * NW + 63 * W + w] ^ Groot[c * W + w];
      if (c == 2 || c == 4) v ^= d63[w] ^ (negate ? ~0ull : 0ull);
      out[c * W + w] = v;
    }
  }
}

// Boolean XOR of two sharings of nw words (6 nw words each)
__global__ void k_bxor(long long n6, const u64* __restrict__ a, const u64* __restrict__ b, u64* __restrict__ out) {
  GRID_STRIDE(i, n6) { out[i] = a[i] ^ b[i]; }
}

// B2A: out = Delta + (1 - 2 Delta) ra for public bits Delta (n elements, packed)
__global__ void k_b2a_apply(const u64* __restrict__ dbits, const u64* __restrict__ ra, long long n,
                            u64* __restrict__ out) {
  GRID_STRIDE(t, 6 * n) {
    const int c = (int)(t / n);
    const long long e = t % n;
    const u64 d = (dbits[e >> 6] >> (e & 63)) & 1ull;
    u64 v = d ? 0ull - ra[t] : ra[t];
    if (d && (c == 2 || c == 4)) v += 1ull;
    out[t] = v;
  }
}

// out = a - b (sub = 1) or a + b (sub = 0) over n words
__global__ void k_addsub(long long n, const u64* __restrict__ a, const u64* __restrict__ b, int sub,
                         u64* __restrict__ out) {
  GRID_STRIDE(i, n) { out[i] = sub ? a[i] - b[i] : a[i] + b[i]; }
}

// Pi_Tran of the edaBit inner products (rows e of dimension 64, weight r^(e0 + e) on row e) as ring
// words: entry (e0 + e) 64 + i of xm is the bit m_i of element e (components 2 and 4 of <m_i>,
// which has no mask), of component c of y 2^(i+1) <r'_i>.  The sources are plane-major: a 64 x 32
// tile goes through shared memory, so that reads run along e and writes along i.
__global__ void __launch_bounds__(TPB)
k_eda_words(const u64* __restrict__ mbits, const u64* __restrict__ rp, long long np, long long e0,
            long long ldy, u64* __restrict__ xm, u64* __restrict__ y) {
  __shared__ u64 tile[64][33];
  const long long N = 64 * np, eb = (long long)blockIdx.x * 32;
  const int q = blockIdx.y, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int i = ty; i < 64; i += TPB / 32) {
    const long long j = (long long)i * np + eb + tx;   // np is a multiple of 64
    tile[i][tx] = q < 6 ? shl_mod(rp[q * N + j], i + 1) : (mbits[j >> 6] >> (j & 63)) & 1ull;
  }
  __syncthreads();
  u64* dst = (q < 6 ? y + q * ldy : xm) + (e0 + eb) * 64;
  for (int k = threadIdx.x; k < 64 * 32; k += TPB) dst[k] = tile[k & 63][k >> 6];
}

// 2x2 max-pool operands: for every window w = (b, ch, i, j) of a (B C, H, W) tensor (one
// component of n = B C H W words), left = [a ; c], right = [b ; d] with a = [2i][2j],
// b = [2i][2j+1], c = [2i+1][2j], d = [2i+1][2j+1]; nw windows, stage width np.
__global__ void k_window_gather(const u64* __restrict__ x, long long BC, long long H, long long W,
                                long long np, u64* __restrict__ left, u64* __restrict__ right) {
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
__global__ void k_gather(const u64* __restrict__ xs, long long n_in, const long long* __restrict__ idx,
                         long long n_out, u64* __restrict__ out) {
  GRID_STRIDE(t, 6 * n_out) {
    const int c = (int)(t / n_out);
    const long long k = t % n_out;
    const long long j = idx[k];
    out[t] = (j >= 0 && j < n_in) ? xs[c * n_in + j] : 0ull;
  }
}

}  // namespace

// ---- launchers ------------------------------------------------------------------------------
void launch_and_offline(cudaStream_t st, const u64* xs, const u64* ys, long long nw, Key k01, Key k02,
                        u32 purpose, u64 obj, u64* zs, u64* g2_out) {
  if (nw <= 0) return;
  k_and_offline<<<grid_for(nw), TPB, 0, st>>>(xs, ys, nw, k01, k02, make_tag(purpose, C_R1),
                                              make_tag(purpose, C_R2), make_tag(purpose, C_G1), obj,
                                              zs, g2_out);
}
void launch_and_online(cudaStream_t st, const u64* xs, const u64* ys, long long nw, Key k01,
                       u32 purpose, u64 obj, const u64* g2_in, u64* p1_out, u64* p2_out) {
  if (nw <= 0) return;
  k_and_online<<<grid_for(nw), TPB, 0, st>>>(xs, ys, nw, k01, make_tag(purpose, C_G1), obj, g2_in,
                                             p1_out, p2_out);
}
void launch_xor_finish(cudaStream_t st, long long nw, const u64* p1_own, const u64* p1_in,
                       const u64* p2_own, const u64* p2_in, u64* zs) {
  if (nw <= 0) return;
  k_xor_finish<<<grid_for(nw), TPB, 0, st>>>(nw, p1_own, p1_in, p2_own, p2_in, zs);
}
void launch_bits_to_arith(cudaStream_t st, const u64* bits, long long n, int kind, u64* out) {
  if (n <= 0) return;
  k_bits_to_arith<<<grid_for(n), TPB, 0, st>>>(bits, n, kind, out);
}
void launch_lin_apb_m2c(cudaStream_t st, long long n, const u64* a, const u64* b, const u64* c, u64* out) {
  if (n <= 0) return;
  k_lin_apb_m2c<<<grid_for(n), TPB, 0, st>>>(n, a, b, c, out);
}
void launch_eda_inner_offline(cudaStream_t st, long long np, Key k01, Key k02, u64 obj, u64* zs,
                              u64* g2_out) {
  k_eda_inner_offline<<<grid_for(np), TPB, 0, st>>>(np, k01, k02, make_tag(P_EDA_INNER, C_R1),
                                                    make_tag(P_EDA_INNER, C_R2),
                                                    make_tag(P_EDA_INNER, C_G1), obj, zs, g2_out);
}
void launch_eda_inner_online(cudaStream_t st, const u64* mbits, const u64* rp, long long np, Key k01,
                             u64 obj, const u64* g2_in, u64* p1_out, u64* p2_out) {
  k_eda_inner_online<<<grid_for(np), TPB, 0, st>>>(mbits, rp, np, k01, make_tag(P_EDA_INNER, C_G1),
                                                   obj, g2_in, p1_out, p2_out);
}
void launch_eda_compose(cudaStream_t st, const u64* mbits, const u64* rp, const u64* z, long long np,
                        u64* ra) {
  k_eda_compose<<<grid_for(6 * np), TPB, 0, st>>>(mbits, rp, z, np, ra);
}
void launch_msb_leaves(cudaStream_t st, const u64* rbits, const u64* dplanes, long long W, u64* G,
                       u64* P) {
  k_msb_leaves<<<grid_for(64 * W), TPB, 0, st>>>(rbits, dplanes, W, G, P);
}
void launch_msb_gather(cudaStream_t st, const u64* G, const u64* P, int C, int root, long long W,
                       u64* X, u64* Y) {
  k_msb_gather<<<grid_for((long long)(root ? C : 2 * C) * W), TPB, 0, st>>>(G, P, C, root, W, X, Y);
}
void launch_msb_combine(cudaStream_t st, const u64* G, const u64* Z, int C, int root, long long W,
                        u64* Gout, u64* Pout) {
  k_msb_combine<<<grid_for((long long)C * W), TPB, 0, st>>>(G, Z, C, root, W, Gout, Pout);
}
void launch_msb_out(cudaStream_t st, const u64* rbits, const u64* Groot, const u64* d63, long long W,
                    int negate, u64* out) {
  k_msb_out<<<grid_for(W), TPB, 0, st>>>(rbits, Groot, d63, W, negate, out);
}
void launch_bxor(cudaStream_t st, long long n6, const u64* a, const u64* b, u64* out) {
  if (n6 <= 0) return;
  k_bxor<<<grid_for(n6), TPB, 0, st>>>(n6, a, b, out);
}
void launch_b2a_apply(cudaStream_t st, const u64* dbits, const u64* ra, long long n, u64* out) {
  k_b2a_apply<<<grid_for(6 * n), TPB, 0, st>>>(dbits, ra, n, out);
}
void launch_addsub(cudaStream_t st, long long n, const u64* a, const u64* b, int sub, u64* out) {
  if (n <= 0) return;
  k_addsub<<<grid_for(n), TPB, 0, st>>>(n, a, b, sub, out);
}
void launch_eda_words(cudaStream_t st, const u64* mbits, const u64* rp, long long np, long long e0,
                      long long ldy, u64* xm, u64* y) {
  k_eda_words<<<dim3((unsigned)(np / 32), 7), TPB, 0, st>>>(mbits, rp, np, e0, ldy, xm, y);
}

void launch_window_gather(cudaStream_t st, const u64* x, long long BC, long long H, long long W,
                          long long np, u64* left, u64* right) {
  k_window_gather<<<grid_for(6 * BC * (H / 2) * (W / 2)), TPB, 0, st>>>(x, BC, H, W, np, left, right);
}

void launch_gather(cudaStream_t st, const u64* xs, long long n_in, const long long* idx,
                   long long n_out, u64* out) {
  if (n_out <= 0) return;
  k_gather<<<grid_for(6 * n_out), TPB, 0, st>>>(xs, n_in, idx, n_out, out);
}

}  // namespace mpc3
