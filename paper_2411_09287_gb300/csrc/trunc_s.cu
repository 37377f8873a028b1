// The matrix S_{j,j'} = sum_e r^(2e) b1_{e,j} b2_{e,j'} of the truncation-pair batch on the
// 5th-generation tensor cores (tcgen05.mma kind::f8f6f4, e4m3 operands, f32 accumulators in
// tensor memory), exactly.
//
// Why: in the consolidated trunc-pair claim (index i = 64 e + j), P0's cross-term sums of the first
// six Pi_Reduce rounds (Fig. Reduce) are all linear combinations of S with public GR weights, so
// S is computed once per layer.  Writing r^(2e) = T_hi[e_hi] T_lo[e_lo] with e = e_hi L + e_lo:
//   S_hi[e_hi][(j,j')] = sum_{e_lo} T_lo[e_lo] b1_{e,j} b2_{e,j'}     (this file, tensor cores)
//   S[(j,j')]          = sum_{e_hi} T_hi[e_hi] S_hi[e_hi][(j,j')]
// The second sum is a GR-matrix product of the blocks in place and a sum over them, or, on the CUDA
// cores, one u64 GEMM over the blocks and the reduction of its products (k_fold_reduce_strided).
// Exactness: each u64 coefficient v of T_lo is written as v = sum_l d_l 32^l mod 2^64 with 13 limbs,
// -16 <= d_l <= 15 (d_12 the top four bits); e4m3 has four significant bits, so every integer from
// -16 to 16 is exact in it, as are the bits, and an accumulator sums at most L <= 2^16 terms, so
// every f32 partial sum is an exact integer of at most 2^20; the limbs are recombined mod 2^64 when
// the e_lo loop ends.  13 limbs take 39.4 ms for 2^24 outputs, 16
// unsigned ones of 4 bits (N = 256) 41.2; 12 (radix 43) need divisions that cost small batches 60 us.
// What bounds it is the pair bits' way through shared memory beside the MMAs' reads: without the stores
// of A it took 16% less.
//
// Operands, both K-major (K = e):
//   A (M = 128 pairs per accumulator): byte (p, e) = e4m3(b1_{e,j} AND b2_{e,j'}), generated in
//     shared memory by four warps from bit-transposed words BT[j][e / 64] (bit e % 64);
//   B (N = 208 limb columns): TL8[c][e_lo] = e4m3(limb c % 13 of coefficient c / 13 of T_lo[e_lo]),
//     loaded by TMA (128-byte swizzle).
// CTA = 256 pairs (j = 4 blockIdx.x .. +3, all j') x 208 limb columns (16 coefficients) x one e_hi
// block; two accumulators (pairs 0..127 and 128..255 of the tile) take 208 of 256 TMEM columns each.
// Warps 0-3 generate A and drain TMEM at the end, warp 4 issues the TMA loads, warp 5 the MMAs;
// a 3-stage ring of 58 KB (two A tiles + one B tile per stage) keeps the three roles apart.
// Every mbarrier wait is bounded; a failure sets err_flag in *err and the CTA lets its copies and
// MMAs finish (bounded), frees its tensor memory and returns without writing.
#include <cstring>

#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "gr_mul.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace mpc3 {

namespace {

using namespace tc;

constexpr int S_LIMBS = TRUNC_LIMBS;
constexpr int S_KC = 128;                  // e per chunk (one 128-byte swizzled row)
constexpr int S_TPAIRS = 256;              // pairs per CTA (two accumulators of 128)
constexpr int S_TCOLS = 16 * S_LIMBS;      // limb columns per CTA (16 coefficients)
constexpr int S_ATILE = 128 * S_KC;        // 16 KB
constexpr int S_BTILE = S_TCOLS * S_KC;    // 26 KB
static_assert(S_BTILE % 1024 == 0 && S_TCOLS % 16 == 0 && S_TCOLS <= 256, "swizzle atoms, MMA N");
constexpr int S_STAGE = 2 * S_ATILE + S_BTILE;
constexpr int S_NST = 3;
constexpr int S_THREADS = 6 * 32;
constexpr size_t S_SMEM = (size_t)S_NST * S_STAGE + 1024;

// kind::f8f6f4: f32 accumulator, e4m3 A and B (format 0), both K-major, M = 128, N = 208
constexpr unsigned S_IDESC = (1u << 4) | ((unsigned)(S_TCOLS >> 3) << 17) | ((unsigned)(128 >> 4) << 24);

template <int ACC>
__device__ __forceinline__ void mma_f8(unsigned d_tmem, u64 adesc, u64 bdesc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(S_IDESC), "n"(ACC));
}

// 4 bits -> 4 bytes of e4m3 1.0 (0x38) or 0: the multiply spreads bit b to byte b (no carries)
__device__ __forceinline__ unsigned nibble_bytes(unsigned nib) {
  return ((nib * 0x00204081u) & 0x01010101u) * 0x38u;
}

// TL8[c * L + e] = e4m3(limb c % 13 of coefficient c / 13 of T_lo[e]), e < L.  A block takes 64 e:
// their words go through shared memory, thread (coefficient, 16 e) then writes 16 bytes of each of
// its coefficient's 13 rows.  Adding sum_{l < 12} 16 * 32^l makes the limbs plain 5-bit fields less
// 16; a field n becomes the f16 1024 + n by its bits, and two of them an e4m3 pair by one conversion.
// Bound by the writes.  (Each thread gathering its 16 words with a stride of 512 bytes and a table in
// constant memory, indexed per thread: 231 us for L = 2^16, now 33-43 us.)
__global__ void __launch_bounds__(256)
k_limb_table(const u64* Tlo, long long L, unsigned char* __restrict__ TL8) {
  grid_dep();
  __shared__ u64 tile[64][65];
  const long long e0 = (long long)blockIdx.x * 64;   // L is a multiple of 64
  for (int i = threadIdx.x; i < 4096; i += 256) tile[i >> 6][i & 63] = Tlo[e0 * 64 + i];
  __syncthreads();
  const int coeff = threadIdx.x & 63, eq = (threadIdx.x >> 6) * 16;
  u64 bias = 0;
#pragma unroll
  for (int l = 0; l < S_LIMBS - 1; ++l) bias += 16ull << (5 * l);
  u64 v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = tile[eq + i][coeff] + bias;
  unsigned char* out = TL8 + (long long)coeff * S_LIMBS * L + e0 + eq;
#pragma unroll
  for (int l = 0; l < S_LIMBS; ++l) {
    const __half2 off = __float2half2_rn(l < S_LIMBS - 1 ? 1040.0f : 1024.0f);
    unsigned o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const unsigned n = ((unsigned)(v[2 * i] >> (5 * l)) & 31u) |
                         (((unsigned)(v[2 * i + 1] >> (5 * l)) & 31u) << 16) | 0x64006400u;
      __half2 h;
      memcpy(&h, &n, 4);
      h = __hsub2(h, off);
      o[i] = __nv_cvt_halfraw2_to_fp8x2(h, __NV_SATFINITE, __NV_E4M3);
    }
    uint4 q;
    q.x = o[0] | (o[1] << 16); q.y = o[2] | (o[3] << 16);
    q.z = o[4] | (o[5] << 16); q.w = o[6] | (o[7] << 16);
    *reinterpret_cast<uint4*>(out + l * L) = q;
  }
}

// BT[j * nw + w] = bits j of words[64 w .. 64 w + 63] (bit i = word 64 w + i).  A warp transposes
// the 64 x 64 bits of one w by exchanging halves (lane t holds words t and t + 32: one exchange in
// the thread, five with lanes t ^ 16 .. t ^ 1); a block's 16 w leave through shared memory, so that
// the rows are written 128 bytes at a time.  (64 threads gathering 64 bits each and writing 8 bytes
// a row: 318 us for 2^24 words, now 84 us.)
constexpr int BT_W = 16;
__global__ void __launch_bounds__(32 * BT_W)
k_bit_transpose(const u64* words, long long nw, u64* __restrict__ BT) {
  grid_dep();
  __shared__ u64 rows[64][BT_W + 1];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const long long w0 = (long long)blockIdx.x * BT_W;
  u64 a = 0, b = 0;
  if (w0 + wl < nw) {
    a = words[(w0 + wl) * 64 + lane];
    b = words[(w0 + wl) * 64 + 32 + lane];
  }
  // words t and t + 32: the off-diagonal 32-bit halves change places
  const u64 t0 = (a & 0xFFFFFFFFull) | (b << 32);
  b = (a >> 32) | (b & 0xFFFFFFFF00000000ull);
  a = t0;
  auto step = [&](int s, u64 m) {   // m: the low s bits of every 2 s
    const bool up = lane & s;
    const u64 ax = __shfl_xor_sync(0xffffffffu, a, s), bx = __shfl_xor_sync(0xffffffffu, b, s);
    a = up ? ((a & ~m) | ((ax >> s) & m)) : ((a & m) | ((ax & m) << s));
    b = up ? ((b & ~m) | ((bx >> s) & m)) : ((b & m) | ((bx & m) << s));
  };
  step(16, 0x0000FFFF0000FFFFull);
  step(8, 0x00FF00FF00FF00FFull);
  step(4, 0x0F0F0F0F0F0F0F0Full);
  step(2, 0x3333333333333333ull);
  step(1, 0x5555555555555555ull);
  rows[lane][wl] = a;
  rows[lane + 32][wl] = b;
  __syncthreads();
  for (int i = threadIdx.x; i < 64 * BT_W; i += 32 * BT_W) {
    const int j = i / BT_W, w = i % BT_W;
    if (w0 + w < nw) BT[(long long)j * nw + w0 + w] = rows[j][w];
  }
}

__global__ void __launch_bounds__(S_THREADS, 1)
k_trunc_s_tc(const __grid_constant__ CUtensorMap tmB, const u64* B1T,
             const u64* B2T, long long nw, long long L, u64* __restrict__ S_hi,
             unsigned* __restrict__ err, unsigned err_flag) {
  grid_dep();
  extern __shared__ unsigned char dsm[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(dsm) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) u64 fullb[S_NST], fulla[S_NST], empty[S_NST], done_bar;
  __shared__ unsigned tmem_slot;
  __shared__ int abort_flag;
  volatile int* abort = &abort_flag;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int pt = blockIdx.x, ct = blockIdx.y;
  const long long ehi = blockIdx.z;
  const int nchunks = (int)(L / S_KC);

  if (tid == 0) {
    for (int i = 0; i < S_NST; ++i) {
      mbar_init(&fullb[i], 1);
      mbar_init(&fulla[i], 4);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&done_bar, 1);
    abort_flag = 0;
    mbar_init_fence();
  }
  if (warp == 0) tmem_alloc(&tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = tmem_slot;

  auto fail = [&]() {
    *abort = 1;
    atomicOr(err, err_flag);
  };

  if (warp == 4) {
    // ---- TMA producer: limb-table tile (208 columns x 128 e) per chunk ----
    if (lane == 0) {
      int last = -1;
      for (int c = 0; c < nchunks; ++c) {
        const int st = c % S_NST;
        if (c >= S_NST && !mbar_wait(&empty[st], (unsigned)(((c / S_NST) + 1) & 1), abort)) {
          fail();
          break;
        }
        mbar_expect_tx(&fullb[st], (unsigned)S_BTILE);
        tma_load_2d(base + st * S_STAGE + 2 * S_ATILE, &tmB, &fullb[st], c * S_KC, ct * S_TCOLS);
        last = c;
      }
      for (int c = last; c >= 0 && c > last - S_NST; --c)
        mbar_wait_plain(&fullb[c % S_NST], (unsigned)((c / S_NST) & 1));
    }
  } else if (warp == 5) {
    // ---- MMA issuer ----
    if (lane == 0) {
      const u64 d0 = smem_desc(base, 128);
      for (int c = 0; c < nchunks; ++c) {
        const int st = c % S_NST;
        const unsigned par = (unsigned)((c / S_NST) & 1);
        if (!mbar_wait(&fullb[st], par, abort) || !mbar_wait(&fulla[st], par, abort)) {
          fail();
          break;
        }
        tc_fence_after();
        const u64 ds = d0 + (u64)((st * S_STAGE) >> 4);
        const u64 db = ds + (u64)((2 * S_ATILE) >> 4);
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          const u64 da = ds + (u64)((a * S_ATILE) >> 4);
#pragma unroll
          for (int k = 0; k < S_KC / 32; ++k) {
            if (c == 0 && k == 0) mma_f8<0>(tmem + (unsigned)(a * 256), da + 2 * k, db + 2 * k);
            else mma_f8<1>(tmem + (unsigned)(a * 256), da + 2 * k, db + 2 * k);
          }
        }
        mma_commit(&empty[st]);
      }
      mma_commit(&done_bar);
      mbar_wait_plain(&done_bar, 0u);
    }
  } else {
    // ---- A generators (warps 0-3), then the drain ----
    const int jp = tid & 63, jj = tid >> 6;          // row tid of both tiles: j' and j offset
    const u64* b2row = B2T + (long long)jp * nw;
    const u64* b1row0 = B1T + (long long)(4 * pt + jj) * nw;
    const u64* b1row1 = B1T + (long long)(4 * pt + 2 + jj) * nw;
    const int r7 = tid & 7;
    const int roff = (tid >> 3) * 1024 + r7 * 128;
    const long long w0 = ehi * (L / 64);
    // A chunk's words (two of each row, 16-byte aligned: nw and L / 64 are even) are loaded while the
    // chunk before is written: loaded after the wait for a free stage, they put a load's latency into
    // every chunk (4096^2 outputs: 44.3 ms, 39.4 with them ahead).
    ulonglong2 nb2 = make_ulonglong2(0, 0), nb10 = nb2, nb11 = nb2;
    auto load_words = [&](int c) {
      const long long w = w0 + 2 * c;
      nb2 = *reinterpret_cast<const ulonglong2*>(b2row + w);
      nb10 = *reinterpret_cast<const ulonglong2*>(b1row0 + w);
      nb11 = *reinterpret_cast<const ulonglong2*>(b1row1 + w);
    };
    if (nchunks > 0) load_words(0);
    bool ok = true;
    for (int c = 0; c < nchunks && ok; ++c) {
      const int st = c % S_NST;
      const u64 m[2][2] = {{nb10.x & nb2.x, nb10.y & nb2.y}, {nb11.x & nb2.x, nb11.y & nb2.y}};
      if (c + 1 < nchunks) load_words(c + 1);
      if (c >= S_NST) {
        ok = __all_sync(0xffffffffu, mbar_wait(&empty[st], (unsigned)(((c / S_NST) + 1) & 1), abort));
        if (!ok) break;
      }
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        unsigned char* row = base + st * S_STAGE + a * S_ATILE + roff;
#pragma unroll
        for (int q = 0; q < 8; ++q) {             // 16 e per 16-byte chunk, swizzled position
          const unsigned bits = (unsigned)(m[a][q >> 2] >> (16 * (q & 3))) & 0xFFFFu;
          uint4 v;
          v.x = nibble_bytes(bits & 15u);
          v.y = nibble_bytes((bits >> 4) & 15u);
          v.z = nibble_bytes((bits >> 8) & 15u);
          v.w = nibble_bytes(bits >> 12);
          *reinterpret_cast<uint4*>(row + ((q ^ r7) << 4)) = v;
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&fulla[st]);
    }
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&done_bar, 0u, abort));
    if (ok && !*abort) {
      tc_fence_after();
      const unsigned tl = tmem + ((unsigned)(warp * 32) << 16);
#pragma unroll 1
      for (int a = 0; a < 2; ++a) {
        const long long pair = (long long)pt * S_TPAIRS + a * 128 + warp * 32 + lane;
        u64* out = S_hi + (ehi * 4096 + pair) * 64 + ct * 16;
#pragma unroll 1
        for (int cc = 0; cc < 16; ++cc) {
          unsigned v[16];
          tmem_ld16(tl + (unsigned)(a * 256 + cc * S_LIMBS), v);   // 13 of 16 columns
          tmem_ld_wait();
          u64 sum = 0;
#pragma unroll
          for (int l = 0; l < S_LIMBS; ++l)   // exact: |limb sum| <= 2^20, + 1.5 2^23 keeps it integral
            sum += (u64)(long long)(int)(__float_as_uint(__uint_as_float(v[l]) + 12582912.0f) -
                                         0x4B400000u) << (5 * l);
          out[cc] = sum;
        }
      }
    } else if (!ok && lane == 0) {
      fail();
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// out[p][c] = reduce(sum_{a+b=s} P[a*ld + p*64 + b]), one pair p a block.
__global__ void __launch_bounds__(128) k_fold_reduce_strided(const u64* P, long long ld, u64* out) {
  grid_dep();
  __shared__ u64 prod[128];
  const long long p = blockIdx.x;
  const int s = threadIdx.x;
  u64 v = 0;
  if (s < 127) {
    const int a0 = (s < 64) ? 0 : s - 63;
    const int a1 = (s < 64) ? s : 63;
    for (int a = a0; a <= a1; ++a) v += P[a * ld + p * 64 + (s - a)];
  }
  prod[s] = v;
  __syncthreads();
  if (s < 64) out[p * 64 + s] = gr_reduce_at(prod, prod + 64, s);
}

}  // namespace

void launch_trunc_limb_table(cudaStream_t st, const u64* Tlo, long long L, unsigned char* TL8) {
  launch_dep(k_limb_table, (unsigned)(L / 64), 256, 0, st, Tlo, L, TL8);
}

void launch_trunc_bit_transpose(cudaStream_t st, const u64* words, long long Epad, u64* BT) {
  const long long nw = Epad / 64;
  launch_dep(k_bit_transpose, (unsigned)((nw + BT_W - 1) / BT_W), 32 * BT_W, 0, st, words, nw, BT);
}

int launch_trunc_s_tc(cudaStream_t st, const u64* B1T, const u64* B2T, long long Epad,
                      const unsigned char* TL8, long long L, long long nhi, u64* S_hi,
                      unsigned* err, unsigned err_flag) {
  auto enc = encode_fn();
  if (!enc || L % S_KC != 0) return -2;
  CUtensorMap mb;
  cuuint64_t dims[2] = {(cuuint64_t)L, 64 * S_LIMBS};
  cuuint64_t strides[1] = {(cuuint64_t)L};
  cuuint32_t box[2] = {(cuuint32_t)S_KC, (cuuint32_t)S_TCOLS};
  cuuint32_t es[2] = {1, 1};
  if (enc(&mb, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<unsigned char*>(TL8), dims, strides,
          box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return -2;
  set_max_dynamic_smem(reinterpret_cast<const void*>(k_trunc_s_tc), (int)S_SMEM);
  dim3 grid(4096 / S_TPAIRS, 64 * S_LIMBS / S_TCOLS, (unsigned)nhi);
  launch_dep(k_trunc_s_tc, grid, S_THREADS, S_SMEM, st, mb, B1T, B2T, Epad / 64, L, S_hi, err, err_flag);
  return 0;
}

void launch_fold_reduce_strided(cudaStream_t st, const u64* P, long long ld, int npairs, u64* out) {
  launch_dep(k_fold_reduce_strided, npairs, 128, 0, st, P, ld, out);
}

}  // namespace mpc3
