// Host-side launchers of libmpc3's kernels (internal interface between the protocol code in
// api.cu and the kernels).  Every launcher enqueues on `st` and returns nothing; launch errors
// are collected by the protocol code with cudaGetLastError().
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace mpc3 {

// ---- u64 GEMM on CUDA cores ----------------------------------------------------------------
// An operand is value(r, c) = scale * (p0[r, c] + s1 * p1[r, c]) with element (r, c) stored at
// p[r*ld + c] (trans = 0) or p[c*ld + r] (trans = 1); p1 may be null.
struct Opnd {
  const u64* p0;
  const u64* p1;
  long long ld;
  u64 s1;
  u64 scale;
  int trans;
};
struct GemmTerm {
  Opnd A;   // M x K
  Opnd B;   // K x N
};
// out[i] = acc_sign*acc + add0[i] + add1[i] + prf_sign*PRF(key, tag, obj, i), i = r*ldc + c,
// or, with atomic = 1, out[r*ldc + c] += acc_sign*acc (split-K accumulation).
struct Epi {
  int atomic;
  u64 acc_sign;
  const u64* add0;
  long long ld_add0;   // row stride of add0 (0: same index as out)
  const u64* add1;
  u64 prf_sign;
  Key key;
  u32 tag;
  u64 obj;
  u64* out;
  long long ldc;
};
// Up to GRAM_BATCH_MAX independent 64 x 64 Gram sums out_i += sign_i sum_k A_i[:, k] B_i[k, :]
// (each a one-term product, K deep, with an atomic epilogue) in one launch.
constexpr int GRAM_BATCH_MAX = 8;
void gemm_u64_gram_batch(cudaStream_t st, long long K, int n, const GemmTerm* terms,
                         const Epi* epis, int nsplit);
// C(M x N) = sum over terms of A_t (M x K) * B_t (K x N), then the epilogue.  nsplit > 1 splits
// K across grid.z and requires epi.atomic = 1.
void gemm_u64(cudaStream_t st, long long M, long long N, long long K, int nterms,
              const GemmTerm* terms, const Epi& epi, int nsplit);

// ---- exact u64 GEMM on the tcgen05 tensor cores (limb_gemm_tc.cu) ---------------------------
// Same contract as gemm_u64 without split-K (epi.atomic must be 0) and with an epilogue on whole rows
// only (ldc = N; add0 at out's index); returns -1 otherwise and for terms of different layouts, -2 if
// the tensor maps cannot be encoded.  scratch: limb_tc_scratch_bytes(M, N, K, nterms) bytes,
// 256-byte aligned (the bf16 digit planes of both operands).  A bounded wait that expires
// sets err_flag in *err and leaves the output undefined.
size_t limb_tc_scratch_bytes(long long M, long long N, long long K, int nterms);
// ev0 / ev1 (may be null) are recorded on st around the tensor-core kernel alone.
// Groups of A's rows: row r is row r % rows of group r / rows, the groups `stride` words apart and the
// rows from `valid` on zeros (rows = 0: no groups).
struct GemmGroups {
  long long rows = 0, valid = 0, stride = 0;
};
int limb_gemm_tc(cudaStream_t st, long long M, long long N, long long K, int nterms,
                 const GemmTerm* terms, const Epi& epi, void* scratch, unsigned* err,
                 unsigned err_flag, cudaEvent_t ev0, cudaEvent_t ev1, int split_min = 0,
                 const GemmGroups& groups = GemmGroups{});

// Row map of a GR matrix product: logical row rho sits at word offset (rho % q) s1 + (rho / q) s2
// (q = 0: rho s1).  q must be a multiple of 128.
struct GrRowMap {
  long long q, s1, s2;
};
// GR-matrix product on the tensor cores, exact: out[rho][c] = add0[rho][c] +
// sum_k A[rho][k] M[k][c] (k, c < 64, M row-major 64 x 64) for rows rho < R.  A row rho at
// p0 + in(rho) (minus p1 + in(rho): s1 must be -1 when p1 is given; returns -1 otherwise), or
// with a_bits the bits of the word p0[in(rho)]; matrix rho / mrows at Mmat + 4096 (rho / mrows)
// (mrows = 0: one matrix, else a multiple of 128); out row rho at out + om(rho), written only
// when om(rho) < out_lim (0: no limit); add0 (may be null) row rho at add0 + rho ld_add0
// (0: 64).  Needs 16-byte aligned bases and even row strides (returns -1 otherwise).
struct GrMMArgs {
  long long R;
  const u64* p0;
  const u64* p1;
  u64 s1;
  GrRowMap in;
  int a_bits;
  const u64* Mmat;
  long long mrows;
  const u64* add0;
  long long ld_add0;
  u64* out;
  GrRowMap om;
  long long out_lim;
  long long qvalid;   // > 0: only rows with rho % in.q < qvalid exist (padded segments)
  int add0_in;        // add0 row rho at add0 + in(rho) (the input map) instead of rho ld_add0
  int tma;            // 1: the A rows of the plain and fold modes are loaded by TMA; 2: and the
                      // A operand sits in tensor memory
  int drain_warps;    // 8 (default) or 16 drain warps
  int out_tma;        // set by the launcher: bit-operand tiles leave by TMA stores (tensor map of
                      // out and om in place of p1's)
};
int gr_matmul_tc_ex(cudaStream_t st, const GrMMArgs& a, unsigned* err, unsigned err_flag);

// One job of a batched tensor-core Gram launch.  u = a0 + sa1 a1 and v = b0 + sb1 b1 (a1, b1 may
// be null; every pointer 16-byte aligned) are vectors of GR elements (rows of 64 words,
// contiguous); over their Dh element pairs (2i, 2i + 1) the job adds, mod 2^64,
//   P[0] += sign C(u_e, v_e),  P[off_oo] += sign C(u_o, v_o),  P[off_x] += sign (C(u_e, v_o) + C(u_o, v_e))
// with C(u, v) = sum_i u_i v_i as its 127 unreduced product coefficients (a block of 128 words).
struct GramJob {
  const u64* a0;
  const u64* a1;
  u64 sa1;
  const u64* b0;
  const u64* b1;
  u64 sb1;
  u64* P;
  u64 sign;
};
constexpr int GRAM_JOBS_MAX = 8;
struct GramJobs {
  GramJob j[GRAM_JOBS_MAX];
  int n;
  long long off_oo, off_x;   // word offsets of the odd-odd and cross blocks from a job's P
};
// Every job of `jobs`: one launch for the single-source jobs and one for those with a second
// source (nsplit: CTAs per parity shared by a launch's jobs, 0 = half the SMs).  Returns -1 for a
// bad job (null or misaligned pointers), 0 otherwise.
int gram_jobs_tc(cudaStream_t st, long long Dh, const GramJobs& jobs, unsigned* err,
                 unsigned err_flag, int nsplit = 0);
// The single-source job of x and y with P = party 0's blocks of a round's sums (S00 at 0, the
// cross sum at 3 * 128, S11 at 9 * 128).  Returns -1 for misaligned inputs.
int gram3_tc(cudaStream_t st, long long Dh, const u64* x, const u64* y, u64* P, unsigned* err,
             unsigned err_flag, int nsplit = 0);

// A fault of one message: word idx XORed with mask where it arrives (idx < 0: none).
struct MsgFault {
  long long idx = -1;
  u64 mask = 0;
};

// ---- single-element steps of the verification (gr_round.cu) ---------------------------------
// Words of one opened element's record: the copies that Pi_Rec's hashes compare.
constexpr int REC_WORDS = 7 * 64;
struct RoundTail {
  const u64* sums;      // 12 blocks of party sums (S00, S01, S10, S11; three parties each)
  int ld;               // words per block: 64 (reduced) or 128 (unreduced coefficients)
  int mode;             // MPC_REDUCE_POINT_X or MPC_REDUCE_POINT_2
  Key k01, k02, k12;
  u64 obj;              // the round's stream object
  const u64* inv;       // (x (x - 1))^-1
  const u64* z;         // the claim entering the round, 6 x 64
  u64* zo;              // the next claim (not z)
  u64* coef;            // the fold element f at 0, 1 - f at 384
  u64* MM;              // the multiplication matrix of f
  u64* zp;              // the opened zeta'
  u64* rec;             // this Pi_Rec's record (REC_WORDS)
  MsgFault fault;       // of the opening's P0 -> P1 message
  u64* zero;            // nzero words cleared for the next round
  long long nzero;
  u64* trace;           // zeta' | h(0) | h(p2) of the round, or null
  u64 *V, *W;           // nvw elements each (nvw = 0: none), times f or 1 - f by bit vwbit of j
  int nvw, vwbit;
  u64* pad[12];         // rows of 64 words to clear (null: none): past the folded vectors' odd ends
};
struct ZeroRows {
  u64* p[12];
};
void launch_zero_rows(cudaStream_t st, const ZeroRows& r);
void launch_round_tail(cudaStream_t st, const RoundTail& a);
// A random GR element of the streams of (purpose, obj), opened into out; record in rec.
void launch_reveal(cudaStream_t st, Key k01, Key k02, Key k12, u32 purpose, u64 obj,
                   const MsgFault& fault, u64* out, u64* rec);
// A round's fold and party sums on a claim of D elements, for short claims.
struct SmallRound {
  const u64* in[12];    // x's components, then y's (null = zero)
  u64* out[12];         // folded (fold set)
  const u64* f;
  long long D;
  bool fold;
  u64* sums;            // 12 blocks of 128 words, added into (S01 + S10 in S01's place), or null
};
void launch_small_round(cudaStream_t st, const SmallRound& a);
// Pi_InnerVerify of a claim of D elements: x, y component pointers (null = zero), z the claim (6 x
// 64), acc 193 words that are zero on entry (party sums and a count of finished blocks).  Delta is
// opened into trace (when not null); `flag` in *status unless it is zero.
struct InnerVerify {
  const u64 *x[6], *y[6];
  const u64* z;
  long long D;
  Key k01, k02, k12;
  u64 obj;
  u64* acc;
  u64* rec;             // this Pi_Rec's record (REC_WORDS)
  MsgFault fault;       // of the opening's P0 -> P1 message
  u64* trace;
  u32* status;
  u32 flag;
};
constexpr int IV_ACC_WORDS = 193;
void launch_inner_verify(cudaStream_t st, const InnerVerify& a);
// The hash comparisons of n records: `flag` in *status on a mismatch.
void launch_rec_hash(cudaStream_t st, const u64* log, int n, u32* status, u32 flag);
// Round k's sums S00, S01, S10, S11 of np parties (party p at 64 p, the four 192 words apart; added
// into out) of rounds over a matrix S[p][j][j'] of n x n GR elements with weights V_j, W_j.
void launch_weighted_sums(cudaStream_t st, const u64* V, const u64* W, const u64* S, int n, int k,
                          int np, u64* out);

// ---- elementwise protocol kernels (prf_kernels.cu) ------------------------------------------
void launch_share_input(cudaStream_t st, const u64* x, long long n, Key k01, Key k02, u64 obj,
                        u64* s6, u64* p0_out_m);
void launch_fill_masks(cudaStream_t st, long long n, Key k01, Key k02, u32 purpose, u64 obj,
                       u64* s6);
void launch_mult_offline(cudaStream_t st, const u64* xs, const u64* ys, long long n, Key k01,
                         Key k02, u64 obj, u64* zs, u64* p0_out_g2);
void launch_mult_online(cudaStream_t st, const u64* xs, const u64* ys, long long n, Key k01,
                        u64 obj, const u64* p2_in_g2, u64* p1_out, u64* p2_out);
// m = own + received for P1 and P2; with t >= 0 also writes the truncated m (>>_arith t) into
// out_s6 (P1.m, P2.m components) when out_s6 != null.
void launch_exchange_finish(cudaStream_t st, long long n, const u64* p1_own, const u64* p1_in,
                            const u64* p2_own, const u64* p2_in, u64* zs, int t, u64* outs);
// row_keys (device, one object id per output row of N outputs, or null): the truncation bits of
// output e come from the streams of object row_keys[e / N] at word e mod N
void launch_trunc_p0(cudaStream_t st, long long E, Key k01, Key k02, u64 obj, int t, u64* zpre,
                     u64* zout, u64* pq, u64* p0_out_gp2, u64* p0_out_gq2, u64* p1_out_mp,
                     u64* p1_out_mq, const u64* row_keys, long long N);
void launch_trunc_finish(cudaStream_t st, long long E, Key k01, Key k02, u64 obj, int t,
                         const u64* p1_in_mp, const u64* p1_in_mq, const u64* p2_in_mp,
                         const u64* p2_in_mq, const u64* p2_gp2, const u64* p2_gq2,
                         const u64* p1_mp1, const u64* p1_mq1, u64* zpre, u64* zout, u64* pq,
                         const u64* row_keys, long long N);
void launch_xor_one(cudaStream_t st, u64* p, u64 mask);
// The messages of Pi_Rec of a sharing xs and (out not null) P1's opening: in_p2_r1 = P0.[r]_1, in_p1_r2
// = P0.[r]_2 (with the fault), in_p0_m = P1.m, out = P1.m - P1.[r]_1 - in_p1_r2 (XOR for a Boolean
// sharing).
void launch_rec_messages(cudaStream_t st, const u64* xs, long long n, const MsgFault& fault, bool boolean,
                         u64* in_p2_r1, u64* in_p1_r2, u64* in_p0_m, u64* out);
// The opening alone, from the received in_p1_r2.
void launch_rec_open(cudaStream_t st, const u64* xs, const u64* in_p1_r2, long long n, bool boolean,
                     u64* out);

// ---- SHA-256 Merkle hash (sha_kernels.cu) ---------------------------------------------------
// Merkle hash of Pi_Rec: 1024-byte leaves, subtree roots of 64 aligned leaves per CTA.
constexpr long long HASH_LEAF_BYTES = 1024;
constexpr long long HASH_CTA_LEAVES = 64;
constexpr long long hash_scratch_words_for(long long n) {
  return 16 * (((8 * n + HASH_LEAF_BYTES - 1) / HASH_LEAF_BYTES > 1
                    ? (8 * n + HASH_LEAF_BYTES - 1) / HASH_LEAF_BYTES
                    : 1) +
               HASH_CTA_LEAVES - 1) /
         HASH_CTA_LEAVES;
}
// The digests of njobs arrays of n words each: one launch over all leaves, one for the trees (a
// Pi_Rec hashes six arrays, which as launches of their own ran one after another).
struct HashJobs {
  const u64* data[6];
  u32* scratch[6];   // hash_scratch_words(n) 32-bit words each
  u32* digest[6];    // 8 words each
};
void launch_hash_jobs(cudaStream_t st, const HashJobs& jobs, int njobs, long long n);
// digest (8 words) of the n-word array; scratch needs hash_scratch_words(n) 32-bit words.
void launch_hash_u64(cudaStream_t st, const u64* data, long long n, u32* scratch, u32* digest);
void launch_digest_check(cudaStream_t st, const u32* a0, const u32* b0, const u32* a1,
                         const u32* b1, const u32* a2, const u32* b2, u32* status, u32 flag);
size_t hash_scratch_words(long long n);
// Pi_Rec of the sharing xs of n words (arguments as launch_rec_messages): the messages, the opening and
// the six hashes, of what P1, P2, P2 hold ([r]_1, m, [r]_2) and of what P2, P0, P1 received; a mismatch
// sets `flag` in *status.  out may lie in xs.
struct RecBufs {
  u64 *in_p2_r1, *in_p1_r2, *in_p0_m;   // n words each
  u32* hs[6];                           // hash_scratch_words(n) 32-bit words each
  u32* dg;                              // 6 x 8
};
void launch_rec(cudaStream_t st, const u64* xs, long long n, const MsgFault& fault, bool boolean,
                const RecBufs& b, u64* out, u32* status, u32 flag);

// ---- GR(2^64, 64) kernels (gr_kernels.cu) ---------------------------------------------------
void launch_gr_powers(cudaStream_t st, const u64* a, long long n, u64* table);
void launch_gr_mul1(cudaStream_t st, const u64* a, const u64* b, u64* out);
// out_c = a_c + r b_c for n GR elements (rows of 64 words)
void launch_gr_axpy(cudaStream_t st, int n, const u64* r, const u64* a, const u64* b, u64* out);
// out = (x (x - 1))^-1, the constant of the Lagrange weights at the points 0, 1, x
void launch_gr_inverse(cudaStream_t st, u64* out);
void launch_gr_fold_reduce(cudaStream_t st, const u64* P, int n, u64* out);
void launch_neg_copy(cudaStream_t st, const u64* a, long long n, u64* out);
void launch_trunc_u(cudaStream_t st, const u64* r, int t, u64* u);
// out[c] += sum_{e < n} A[c * lda + e] * R[e] (R: n GR elements), c < nrows <= 16, atomically
void launch_scalar_gr_sum(cudaStream_t st, long long n, const u64* A, long long lda, int nrows,
                          const u64* R, u64* out);
// out[e] = a[e] * b[e] (GR products of n row pairs; out may alias a or b)
void launch_gr_mul_rows(cudaStream_t st, long long n, const u64* a, const u64* b, u64* out);
// out[i] = src[idx(i)] (rows of 64 words), idx(i) = ((i mul) / div) mod m (m = 0: no mod).
void launch_gather_rows_affine(cudaStream_t st, long long n, const u64* src, long long mul,
                               long long div, long long m, u64* out);
// out[c] = sum over h < nper of in[c nper + h] (rows of 64 words), c < ncomp.
void launch_block_rowsum(cudaStream_t st, int ncomp, long long nper, const u64* in, u64* out);
// out[i] = sum over h < n of in[h ld + i], i < m words.
void launch_sum_blocks(cudaStream_t st, long long m, long long n, long long ld, const u64* in,
                       u64* out);
// M + 4096 i = multiplication matrix (M[b][c] = coefficient c of g x^b) of g = src + i stride,
// i < n.
void launch_gr_mulmat_batch(cudaStream_t st, long long n, const u64* src, long long stride,
                            u64* M);
// out (cols x rows) = transpose of in viewed as rows x cols; source indices >= n read as 0.
void launch_word_transpose(cudaStream_t st, long long rows, long long cols, long long n,
                           const u64* in, u64* out);
void launch_trunc_materialize(cudaStream_t st, long long E, const u64* words, const u64* VW,
                              const u64* R, int kd, u64* out);
// PRF words off .. off + n - 1 of one stream into out[0 .. n) (e.g. the truncation bits b1, b2
// of the outputs of one verification chunk)
void launch_prf_words(cudaStream_t st, long long n, Key key, u32 tag, u64 obj, u64* out,
                      long long off = 0);
// the same for a row-keyed truncation-bit stream: word e = word e mod N of object row_keys[e / N]
void launch_prf_words_keyed(cudaStream_t st, long long n, Key key, u32 tag, const u64* row_keys,
                            long long N, u64* out, long long off);

// ---- first rounds of a batch of weighted ring words (gr_block.cu) ----------------------------
struct BlkIn {            // share components of x, y (words) and of the claim z (ldz words apart)
  const u64* x[6];
  const u64* y[6];
  const u64* z;
  long long ldz;
  long long D;            // words of a component; words past D read as 0
};
struct BlkVec {
  const u64* c[6];
};
struct BlkOut {
  u64* c[6];
};
// Rows of launch_blk_sums: the parties' B x B sums, then (full) the claim's 6 x B.
int blk_rows(int B, bool full);
// out (blk_rows x 64 words, accumulated): S^p_{j,j'} and Z_{c,j} over the blocks b < nb of B words,
// weight R[b >> sh].  full: every component and the claim; else x has components 2 and 4 only and
// the rows are those of parties 1 and 2.
void launch_blk_sums(cudaStream_t st, const BlkIn& in, int B, bool full, long long nb, int sh,
                     const u64* R, u64* out);
// The same sums for full batches (sh = 0) and the edaBits' (sh = 2) with B = 16, on the tensor cores:
// a product of the blocks' words (nw columns, those of a weight added) and R.  scratch:
// blk_sums_tc_bytes(full, nw), 256-byte aligned; 0, or not 0 when the tensor maps cannot be encoded.
size_t blk_sums_tc_bytes(bool full, long long nw);
int blk_sums_tc(cudaStream_t st, const BlkIn& in, bool full, long long nw, const u64* R, u64* out,
                void* scratch, unsigned* err, unsigned err_flag, int split_min);
// out[c][j] (6 x 64 elements, accumulated) = sum over w < nw of R[w] z[c ldz + 64 w + j].
void launch_words_sums(cudaStream_t st, const u64* z, long long ldz, long long nw, const u64* R,
                       u64* out);
// z_c += sum over j < n of T_j Zr[c n + j] (6 components).
void launch_blk_claim(cudaStream_t st, const u64* T, const u64* Zr, int n, u64* z);
// out_c[b] = sum over j < B of in_c[B b + j] G[row], row = (b >> sh) B + j (rows) or j, b < nb.
void launch_blk_combine(cudaStream_t st, const BlkVec& in, const BlkOut& out, int B, bool rows,
                        long long D, long long nb, int sh, const u64* G);
// n rows holding the element 1
void launch_ones(cudaStream_t st, int n, u64* out);

// ---- trunc-batch S matrix on the tensor cores (trunc_s.cu) ----------------------------------
constexpr int TRUNC_LIMBS = 13;   // e4m3 limbs of a u64
void launch_trunc_limb_table(cudaStream_t st, const u64* Tlo, long long L, unsigned char* TL8);
// BT[j][w] = bit j of words[64 w + i] at bit i, for w < Epad / 64
void launch_trunc_bit_transpose(cudaStream_t st, const u64* words, long long Epad, u64* BT);
// S_hi[e_hi][64 j + j'][coeff] for e_hi < nhi; returns -2 if the tensor map cannot be encoded.
// A bounded wait that expires sets err_flag in *err (the output is then undefined).
int launch_trunc_s_tc(cudaStream_t st, const u64* B1T, const u64* B2T, long long Epad,
                      const unsigned char* TL8, long long L, long long nhi, u64* S_hi,
                      unsigned* err, unsigned err_flag);

// out[p] = the reduced product whose terms are P[a ld + 64 p + b] (a, b < 64), for npairs p.
void launch_fold_reduce_strided(cudaStream_t st, const u64* P, long long ld, int npairs, u64* out);

// ---- compare-select of the non-linear layers (compare.cu) --------------------------------------
struct CsView {          // component c of element e at p[c stride + e], 0 for e >= valid or p = null
  const u64* p;
  long long stride, valid;
};
// One stage of np elements (a multiple of 64): out = max(a, b).
struct CompareSelect {
  CsView a, b;
  u64* out;              // component c of element e < out_n at c out_ld + e
  long long out_ld, out_n;
  long long np;
  Key k01, k02, k12;
  u64 obj;               // the stage's stream object (AND level l: + l)
  MsgFault fault[4];     // edaBit products' GAMMA2, MZ1, MZ2; the first AND level's [Gamma]_2
  u64 *eda[3], *da[3];   // bit planes of the public-seed bits: np words each, np / 64 words each
  u64 *eprod, *ez;       // edaBit products (6 x 64 np) and inner products (6 np)
  u64* dd;               // 6 np: Delta's sharing to open
  u64 *mx[3], *my[3], *mz[3];   // the daBit products' and the selection's triples, components nm apart
  long long nm;
  u64* rad;              // 6 np: the daBits' arithmetic sharing
  const u64* dpl;        // the opened Delta's bit planes
  u64 *ax, *ay, *az;     // AND triples, components and_words apart, this stage's from and_off
  long long and_off, and_words;
  u64* e;                // 6 np / 64: Boolean sharing to open
  const u64* dbits;      // e opened
};
// The three parts around the openings of dd and e.
void launch_cs_open_delta(cudaStream_t st, const CompareSelect& a);
void launch_cs_open_bit(cudaStream_t st, const CompareSelect& a);
void launch_cs_select(cudaStream_t st, const CompareSelect& a);

// ---- non-linear layers (nonlinear.cu) -----------------------------------------------------------
void launch_addsub(cudaStream_t st, long long n, const u64* a, const u64* b, int sub, u64* out);
// The edaBit inner-product batch's ring words (see nonlinear.cu): bits m into xm, 2^(i+1) r' into y
// (component c at c ldy), entry (e0 + e) 64 + i.
void launch_eda_words(cudaStream_t st, const u64* const bits[3], const u64* eprod, long long np,
                      long long e0, long long ldy, u64* xm, u64* y);
void launch_gather(cudaStream_t st, const u64* xs, long long n_in, const long long* idx,
                   long long n_out, u64* out);
void launch_window_gather(cudaStream_t st, const u64* x, long long BC, long long H, long long W,
                          long long np, u64* left, u64* right);
// ---- Pi_MultVerify of AND gates over GF(2^64) (gf_verify.cu) ----------------------------------
constexpr int GF_MAX_ROUNDS = 60;
struct GfWork {          // cleared by launch_gf_verify
  u64 S[240], V[8], W[8], z[6], zeta, r;
  u64 sums[6 * (GF_MAX_ROUNDS + 1)];
  u32 count[GF_MAX_ROUNDS + 1];
};
struct GfVerify {
  const u64 *X, *Y, *Z;  // the triples: 6 x nw words each, bit i of the 64 nw gates = bit i % 64
  long long nw;          // at least 125
  int R;                 // rounds, at least 4, to at most 64 elements
  Key k01, k02, k12;
  u64 obj;               // the batch's stream object (round k: + k)
  u64* pw;               // 8 nw words
  u64* st;               // 9 (R + 1) words
  GfWork* w;
  u64 *x[2], *y[2];      // 48 nw and 24 nw words each
  u64* trace;            // zeta | h(0) | h(x) of round k at (k - 1) trace_ld, Delta at R trace_ld; or null
  long long trace_ld;
  u32* status;
  u32 flag_verify, flag_abort;   // Delta != 0; a hash mismatch
  int xrec;              // fault: the P0 -> P1 message of opening xrec (0: r, k: zeta of round k, R + 1:
  u64 xmask;             // Delta; -1: none) is XORed with xmask
};
void launch_gf_verify(cudaStream_t st, const GfVerify& a);
// ---- layer-level calls (layer_kernels.cu) ----------------------------------------------------
// Geometry of a convolution: NCHW input (B, C, H, W), kh x kw kernel, stride, zero padding; the
// output is Ho x Wo per image.
struct ConvGeom {
  long long B, C, H, W, kh, kw, stride, pad, Ho, Wo;
};
// out[i] = floor(x[i] 2^k) (saturating, NaN -> 0) / out[i] = (signed) v[i] / 2^k
void launch_encode_fixed(cudaStream_t st, const double* x, long long n, int k, u64* out);
void launch_decode_fixed(cudaStream_t st, const u64* v, long long n, int k, double* out);
// the im2col rows of all six components of x: cols holds 6 (B Ho Wo) (C kh kw) words
void launch_im2col(cudaStream_t st, const u64* x, const ConvGeom& g, u64* cols);
// the mask-switch differences of a standalone truncation and its online shift
void launch_trunc_remask(cudaStream_t st, const u64* xs, const u64* rx, long long n, u64* d1_p1,
                         u64* d2_p2, u64* d1_p0, u64* d2_p0);
void launch_trunc_online(cudaStream_t st, const u64* xs, long long n, const u64* d1,
                         const u64* d2_at_p1, const u64* d1_at_p2, const u64* d2, int t,
                         u64* out);

// test hook: one thread's bounded wait (limit `cycles`) on an mbarrier nothing arrives at
void launch_wait_expires(cudaStream_t st, long long cycles, unsigned* err, unsigned err_flag);

}  // namespace mpc3
