// libmpc3: the C-ABI and the protocol driver.  Every protocol step runs in the kernels of this
// library; the host code here only sequences them, moves messages between the three simulated
// parties (counted in the ledger) and carves the caller's workspace.
//
// Paper map: mpc_share_input = Pi_<.>^{l,0} (Sec. 2); mpc_mult = Pi_Mult (Fig. MultP);
// mpc_matmul = Pi_Inner per output (Fig. DPP, Sec. 4.1) + Pi_Trunc (Fig. trunc);
// mpc_verify_mult = Pi_MultVerify (Fig. PPEV); mpc_verify_matmul = Pi_BIVerify (Fig. PBDP);
// both use Pi_Tran (Fig. MTP), Pi_Reduce (Fig. Reduce), Pi_InnerVerify (Fig. DPV);
// mpc_reconstruct = Pi_Rec (Sec. 2).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstdio>
#include <cstring>
#include <set>
#include <string>
#include <vector>

#include "mpc3.h"
#include "kernels.h"

using namespace mpc3;

namespace {

constexpr u32 ST_ABORT = 1u;    // a Pi_Rec check failed
constexpr u32 ST_VERIFY = 2u;   // Delta != 0
constexpr u32 ST_TIMEOUT = 4u;  // a bounded device wait expired

// device constants block (words)
constexpr int CST_INV = 0;      // 64: (x(x-1))^-1
constexpr int CST_WORDS = 64;

constexpr int TRACE_ROUND = 832;  // words per round in a verification trace

struct Arena {
  char* base;
  size_t cap;
  size_t off = 0;
  bool dry;
  template <class T>
  T* take(long long count) {
    const size_t bytes = ((size_t)std::max<long long>(count, 1) * sizeof(T) + 255) & ~size_t(255);
    T* p = dry ? nullptr : reinterpret_cast<T*>(base + off);
    off += bytes;
    return p;
  }
  bool ok() const { return dry || off <= cap; }
  // room for `bytes` from offset `from` on, under what was taken since
  void reserve(size_t from, size_t bytes) { off = std::max(off, from + ((bytes + 255) & ~size_t(255))); }
};

struct Fault {
  bool armed = false;
  u64 index = 0;
  u64 mask = 0;
  u64 skip = 0;   // messages of the site that pass before it
};

__global__ void k_derive_keys(Key master, u32* out) {
  // eta_{0,1}, eta_{0,2}, eta_{1,2}: first 32 bytes of ChaCha20(master, counter 0,
  // nonce (0x0059454B, pair, 0)), pair = 1, 2, 3
  grid_dep();
  const int pair = threadIdx.x + 1;
  if (pair > 3) return;
  u32 o[16];
  chacha_block(master, 0u, 0x0059454Bu, (u32)pair, 0u, o);
  for (int i = 0; i < 8; ++i) out[(pair - 1) * 8 + i] = o[i];
}

inline long long ceil_log2(long long v) {
  long long r = 0;
  while ((1ll << r) < v) ++r;
  return r;
}
inline int default_R(long long D) { return D > 1 ? (int)std::max<long long>(0, ceil_log2(D) - 6) : 0; }

}  // namespace

namespace {
// e_hi blocks from which the S matrix is combined on the tensor cores unless the caller says
// otherwise (trunc_shape); what mpc_get_tuning reports for an unset field is the ABI's 32.
constexpr int COMBINE_MIN = 2, COMBINE_REPORTED = 32;

mpc_tuning default_tuning() {
  mpc_tuning t;
  t.trunc_block = 65536;
  t.trunc_chunk = 1ll << 24;
  t.row_split = 0;
  t.tc_combine_min = COMBINE_MIN;
  t.gemm_split_min = 8;
  t.gram_split = 76;
  t.fold_batch_max = 65536;
  t.gr_producers = 2;
  t.gr_drain_warps = 8;
  return t;
}
}  // namespace

constexpr int NSIDE = 3;

struct mpc_ctx {
  int device = 0;
  mpc_tuning tune = default_tuning();
  bool combine_set = false;   // tune.tc_combine_min is the caller's
  cudaStream_t st = nullptr;
  bool own_stream = false;
  Key k01{}, k02{}, k12{};
  int reduce_mode = MPC_REDUCE_POINT_X;
  int gemm_path = MPC_GEMM_U64;
  u64* cst = nullptr;
  u32* status = nullptr;
  u64 ledger[MPC_NPHASE][MPC_NPROTO] = {};
  u64 nmsg = 0;
  Fault fault[MPC_NSITE];
  bool aborted = false;
  std::set<u64> pending;   // (call_id << 1) | kind, kind 0 = mult, 1 = matmul
  std::string err;
  // phase timers (CUDA events on the context's stream), enabled by mpc_profile()
  struct ProfRec {
    int id;
    cudaEvent_t a, b;
    double work;   // algorithmic u64 multiply-accumulates of a kernel interval
  };
  bool prof = false;
  std::vector<ProfRec> recs;
  std::vector<cudaEvent_t> pool;
  size_t pool_used = 0;
  // asynchronous uploads (mpc_h2d_async): a copy stream and one event per slot
  cudaStream_t copy_st = nullptr;
  cudaEvent_t copy_ev[MPC_H2D_SLOTS] = {};
  cudaEvent_t order_ev = nullptr;   // the context stream's work before a download
  // side streams of independent verification batches (Fork)
  cudaStream_t side[NSIDE] = {};
  cudaEvent_t fork_ev = nullptr, join_ev[NSIDE] = {};
};

namespace {

int fail(mpc_ctx* c, int code, const std::string& msg) {
  if (c) c->err = msg;
  return code;
}

int cuda_check(mpc_ctx* c, const char* where) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(c, MPC_ERR_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
  return MPC_OK;
}

#define CK(call)                                                                        \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess)                                                              \
      return fail(ctx, MPC_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

cudaEvent_t prof_event(mpc_ctx* c) {
  if (c->pool_used == c->pool.size()) {
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    c->pool.push_back(e);
  }
  return c->pool[c->pool_used++];
}

// Times the enclosed stream work as phase `id` when profiling is on.
struct Phase {
  mpc_ctx* c;
  int id;
  double work;
  cudaEvent_t a = nullptr;
  Phase(mpc_ctx* c_, int id_, double work_ = 0.0) : c(c_), id(id_), work(work_) {
    if (c->prof) {
      a = prof_event(c);
      cudaEventRecord(a, c->st);
    }
  }
  ~Phase() {
    if (c->prof) {
      cudaEvent_t b = prof_event(c);
      cudaEventRecord(b, c->st);
      c->recs.push_back({id, a, b, work});
    }
  }
};

// Independent verification batches side by side.  A batch is a chain of launches that mostly wait for
// one another's results on a few SMs, and the batches of a call share nothing but the status word (an
// atomic OR) and the inputs, so they run on streams of their own: on(i) sends what follows to side
// stream i (i < 0: the context's own), after everything before the fork; join() (or the end of the
// scope) makes the context's stream wait for all of them, so that a call leaves nothing running that
// its stream does not cover.  With phase timers on, everything stays on the one stream.
struct Fork {
  mpc_ctx* c;
  cudaStream_t main;
  bool used[NSIDE] = {};
  explicit Fork(mpc_ctx* ctx, bool enable = true) : c(ctx), main(ctx->st) {
    on_ = enable && !c->prof && cudaEventRecord(c->fork_ev, main) == cudaSuccess;
  }
  void on(int i) {
    c->st = main;
    if (!on_ || i < 0 || cudaStreamWaitEvent(c->side[i], c->fork_ev, 0) != cudaSuccess) return;
    c->st = c->side[i];
    used[i] = true;
  }
  void join() {
    c->st = main;
    for (int i = 0; i < NSIDE; ++i) {
      if (!used[i]) continue;
      used[i] = false;
      if (cudaEventRecord(c->join_ev[i], c->side[i]) != cudaSuccess ||
          cudaStreamWaitEvent(main, c->join_ev[i], 0) != cudaSuccess)
        cudaStreamSynchronize(c->side[i]);
    }
  }
  ~Fork() { join(); }
  Fork(const Fork&) = delete;
  Fork& operator=(const Fork&) = delete;

 private:
  bool on_;
};

int guard(mpc_ctx* ctx) {
  if (!ctx) return MPC_ERR_ARG;
  if (ctx->aborted) return fail(ctx, MPC_ERR_ABORT, "context aborted");
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e != cudaSuccess) return fail(ctx, MPC_ERR_CUDA, cudaGetErrorString(e));
  return MPC_OK;
}

bool id_ok(u64 id) { return id < (1ull << 44); }

// ---- messages -----------------------------------------------------------------------------------
// The fault that is due at this message of n words of `site`, disarmed (HIGH_BIT is a fault of the
// [Gamma]_2 messages, in place of GAMMA2's).
MsgFault take_fault(mpc_ctx* ctx, int site, long long n) {
  if (site < 0 || n <= 0) return {};
  if (site == MPC_SITE_GAMMA2 && ctx->fault[MPC_SITE_HIGH_BIT].armed) site = MPC_SITE_HIGH_BIT;
  Fault& f = ctx->fault[site];
  if (!f.armed) return {};
  if (f.skip) {
    --f.skip;
    return {};
  }
  f.armed = false;
  if (site == MPC_SITE_HIGH_BIT) ctx->fault[MPC_SITE_GAMMA2].armed = false;
  return {(long long)(f.index % (u64)n), f.mask};
}

void count_msgs(mpc_ctx* ctx, int phase, int proto, int count, u64 bytes_each) {
  ctx->ledger[phase][proto] += (u64)count * bytes_each;
  ctx->nmsg += (u64)count;
}

int deliver_copy(mpc_ctx* ctx, int phase, int proto, const u64* src, u64* dst, long long n,
                 const MsgFault& f) {
  if (n > 0) CK(cudaMemcpyAsync(dst, src, (size_t)n * 8, cudaMemcpyDeviceToDevice, ctx->st));
  count_msgs(ctx, phase, proto, 1, (u64)n * 8);
  if (f.idx >= 0) launch_xor_one(ctx->st, dst + f.idx, f.mask);
  return MPC_OK;
}

// The message src to a receiver that only reads it is handed over in place (a copy of a small message
// is a launch of 4 us); one that a fault corrupts is copied first, into `copy` (n words).  dst: what the
// receiver reads.
int deliver(mpc_ctx* ctx, int phase, int proto, const u64* src, const u64*& dst, long long n, int site,
            u64* copy) {
  const MsgFault f = take_fault(ctx, site, n);
  dst = f.idx < 0 ? src : copy;
  if (f.idx >= 0) return deliver_copy(ctx, phase, proto, src, copy, n, f);
  count_msgs(ctx, phase, proto, 1, (u64)n * 8);
  return MPC_OK;
}

// Room for the messages of a call that faults corrupt, at most one a site (a fault fires once).
struct FaultCopies {
  u64 *g2, *mz1, *mz2;   // GAMMA2 (HIGH_BIT), MZ1, MZ2
};
FaultCopies plan_copies(Arena& a, long long n) {
  FaultCopies c;
  c.g2 = a.take<u64>(n);
  c.mz1 = a.take<u64>(n);
  c.mz2 = a.take<u64>(n);
  return c;
}

int read_status(mpc_ctx* ctx, u32* out) {
  CK(cudaMemcpyAsync(out, ctx->status, sizeof(u32), cudaMemcpyDeviceToHost, ctx->st));
  CK(cudaStreamSynchronize(ctx->st));
  if (*out & ST_TIMEOUT) {
    ctx->aborted = true;
    return fail(ctx, MPC_ERR_TIMEOUT, "a bounded device wait expired");
  }
  return MPC_OK;
}

// ---- GEMM helpers -------------------------------------------------------------------------------
Opnd op(const u64* p0, long long ld, int trans = 0, const u64* p1 = nullptr, u64 s1 = 1,
        u64 scale = 1) {
  Opnd o;
  o.p0 = p0; o.p1 = p1; o.ld = ld; o.s1 = s1; o.scale = scale; o.trans = trans;
  return o;
}

Epi epi_store(u64* out, long long ldc) {
  Epi e;
  std::memset(&e, 0, sizeof(e));
  e.atomic = 0; e.acc_sign = 1; e.out = out; e.ldc = ldc;
  return e;
}

Epi epi_atomic(u64* out, long long ldc, u64 sign = 1) {
  Epi e = epi_store(out, ldc);
  e.atomic = 1;
  e.acc_sign = sign;
  return e;
}

// split-K factor of the 64 x 64 Gram products: enough CTAs to fill the GPU down to K ~ 2^12
int nsplit_for(long long K) { return (int)std::min<long long>(1024, std::max<long long>(1, K / 32)); }

// out (atomic, 64x64) += sign * sum_i U_i (x) V_i with U = U0 + su U1, V = V0 + sv V1.
void gram(mpc_ctx* ctx, u64* P, const u64* U0, const u64* U1, u64 su, long long ldu, const u64* V0,
          const u64* V1, u64 sv, long long ldv, long long count, u64 sign) {
  u64 us = 1, vs = 1;
  if (!U0) { U0 = U1; U1 = nullptr; us = su; }
  if (!V0) { V0 = V1; V1 = nullptr; vs = sv; }
  if (!U0 || !V0 || count <= 0) return;
  GemmTerm T;
  T.A = op(U0, ldu, 1, U1, su, us);
  T.B = op(V0, ldv, 0, V1, sv, vs);
  gemm_u64(ctx->st, 64, 64, count, 1, &T, epi_atomic(P, 64, sign), nsplit_for(count));
}

// GR-product arguments with this context's choice of producer and drain variant
GrMMArgs grargs(const mpc_ctx* ctx) {
  GrMMArgs g{};
  g.tma = ctx->tune.gr_producers >= 2 ? ctx->tune.gr_producers - 1 : 0;
  g.drain_warps = ctx->tune.gr_drain_warps;
  return g;
}

// out[i] = add0[i] + (p0[i] + s1 p1[i]) . M for i < R (rows of 64 words, M a 64 x 64 GR
// multiplication matrix): the folds of Pi_Reduce and the products by a fixed GR element.  Tensor
// cores on the limb path, the u64 CUDA-core GEMM otherwise.
int gr_matmul(mpc_ctx* ctx, long long R, const u64* p0, const u64* p1, u64 s1, long long lda,
              const u64* Mmat, const u64* add0, long long ld_add0, u64* out, long long ldc) {
  if (R <= 0) return MPC_OK;
  if (ctx->gemm_path == MPC_GEMM_LIMB_TC) {
    Phase kp(ctx, MPC_PROF_K_GR_MATMUL, (double)R * 4096);
    GrMMArgs g = grargs(ctx);
    g.R = R;
    g.p0 = p0;
    g.p1 = p1;
    g.s1 = s1;
    g.in = GrRowMap{0, lda, 0};
    g.Mmat = Mmat;
    g.add0 = add0;
    g.ld_add0 = ld_add0 ? ld_add0 : ldc;
    g.out = out;
    g.om = GrRowMap{0, ldc, 0};
    if (gr_matmul_tc_ex(ctx->st, g, ctx->status, ST_TIMEOUT) == 0) return MPC_OK;
    // misaligned view: fall through to the CUDA-core GEMM
  }
  GemmTerm T;
  T.A = p1 ? op(p0, lda, 0, p1, s1) : op(p0, lda);
  T.B = op(Mmat, 64);
  Epi e = epi_store(out, ldc);
  e.add0 = add0;
  e.ld_add0 = add0 ? ld_add0 : 0;
  gemm_u64(ctx->st, R, 64, 64, 1, &T, e, 1);
  return MPC_OK;
}

// C = A B (+ epilogue) for a one-term product that the limb path runs on the tensor cores
// (scratch: limb_tc_scratch_bytes(M, N, K, 1) bytes) and the u64 path on the CUDA cores.
int dense_gemm(mpc_ctx* ctx, long long M, long long N, long long K, const GemmTerm& T,
               const Epi& e, void* scratch, const GemmGroups& groups = GemmGroups{}) {
  if (scratch && !e.atomic) {
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ctx->prof) {
      e0 = prof_event(ctx);
      e1 = prof_event(ctx);
      ctx->recs.push_back({MPC_PROF_K_LIMB_GEMM, e0, e1, (double)M * N * K});
    }
    if (limb_gemm_tc(ctx->st, M, N, K, 1, &T, e, scratch, ctx->status, ST_TIMEOUT, e0, e1,
                     ctx->tune.gemm_split_min, groups))
      return fail(ctx, MPC_ERR_CUDA, "tensor-core GEMM setup failed");
    return MPC_OK;
  }
  gemm_u64(ctx->st, M, N, K, 1, &T, e, 1);
  return MPC_OK;
}

// A view of a <.>^{l[x]}-shared vector: component pointers (null = identically zero), row stride.
struct View {
  const u64* c[6];
  long long ld;
};

// Party sums of a secure GR inner product sum_i u_i v_i (Sec. 2 inner product over GR):
//   S0 = sum r_u r_v (P0), S1 = -sum (m_u [r_v]_1 + m_v [r_u]_1) (P1),
//   S2 = sum m_u (m_v - [r_v]_2) - m_v [r_u]_2 (P2).  Pmat: 3 x 4096 scratch; S: 3 x 64 out.
// The same Gram sums collected for one batched launch.
struct GramBatch {
  GemmTerm T[GRAM_BATCH_MAX];
  Epi e[GRAM_BATCH_MAX];
  int n = 0;
  void add(u64* P, const u64* U0, const u64* U1, u64 su, long long ldu, const u64* V0,
           const u64* V1, u64 sv, long long ldv, u64 sign) {
    u64 us = 1, vs = 1;
    if (!U0) { U0 = U1; U1 = nullptr; us = su; }
    if (!V0) { V0 = V1; V1 = nullptr; vs = sv; }
    if (!U0 || !V0 || n >= GRAM_BATCH_MAX) return;
    T[n].A = op(U0, ldu, 1, U1, su, us);
    T[n].B = op(V0, ldv, 0, V1, sv, vs);
    e[n] = epi_atomic(P, 64, sign);
    ++n;
  }
};

int party_sums(mpc_ctx* ctx, const View& u, const View& v, long long count, u64* Pmat, u64* S) {
  CK(cudaMemsetAsync(Pmat, 0, 3 * 4096 * 8, ctx->st));
  const u64 M1 = ~0ull;  // -1
  GramBatch gb;
  gb.add(Pmat, u.c[0], u.c[1], 1, u.ld, v.c[0], v.c[1], 1, v.ld, 1);
  gb.add(Pmat + 4096, u.c[2], nullptr, 1, u.ld, v.c[3], nullptr, 1, v.ld, M1);
  gb.add(Pmat + 4096, v.c[2], nullptr, 1, v.ld, u.c[3], nullptr, 1, u.ld, M1);
  gb.add(Pmat + 8192, u.c[4], nullptr, 1, u.ld, v.c[4], v.c[5], M1, v.ld, 1);
  gb.add(Pmat + 8192, v.c[4], nullptr, 1, v.ld, u.c[5], nullptr, 1, u.ld, M1);
  if (count > 0 && gb.n > 0) {
    gemm_u64_gram_batch(ctx->st, count, gb.n, gb.T, gb.e, nsplit_for(count));
  }
  launch_gr_fold_reduce(ctx->st, Pmat, 3, S);
  return cuda_check(ctx, "party_sums");
}

// ---- verification state ---------------------------------------------------------------------
struct Small {   // per-verification small scratch (all device, from the workspace)
  u64* Pmat;     // 4 x 3 x 4096
  u64* S;        // 4 x 192: S00, S01, S10, S11 (reduced; u64 path)
  u64* U;        // 2 x 12 x 128: a round's party sums ee, S01, S10, oo (3 parties each), the other
                 // half cleared for the next round (sums_begin, next_sums); then Pi_InnerVerify's
  u64* rec;      // REC_SLOTS records of opened single elements, hashed by flush_recs
  u64* z[2];     // 384 each
  u64* coef;     // 448: the fold element f at 0, 1 - f at 384
  u64* zp;       // 64
  u64* r;        // 64
  u64* MM;       // 128 x 64
  u64* aux;      // 4 x 64
  u64* zinit;    // 384: the claim entering the first round (never round scratch)
  mutable int nrec = 0, uc = 0;   // records not hashed yet; half of U in use
};
constexpr int REC_SLOTS = 40;
constexpr int SUMS_WORDS = 12 * 128;

Small plan_small(Arena& a) {
  Small s;
  s.Pmat = a.take<u64>(4 * 3 * 4096);
  s.S = a.take<u64>(4 * 192);
  s.U = a.take<u64>(2 * SUMS_WORDS + IV_ACC_WORDS);
  s.rec = a.take<u64>(REC_SLOTS * REC_WORDS);
  s.z[0] = a.take<u64>(384);
  s.z[1] = a.take<u64>(384);
  s.coef = a.take<u64>(448);
  s.zp = a.take<u64>(64);
  s.r = a.take<u64>(64);
  s.MM = a.take<u64>(128 * 64);
  s.aux = a.take<u64>(4 * 64);
  s.zinit = a.take<u64>(384);
  return s;
}

// A dense claim: x, y vectors of D GR elements (components may be null), claimed z (6 x 64).
struct Vec {
  u64* c[6];
};

struct Dense {
  Vec x[2], y[2];     // ping-pong buffers, capacity cap0 (index 0) and cap1 (index 1)
  long long cap[2];
  int cur = 0;
};

// The hash comparisons of the Pi_Rec calls recorded since the last flush; each batch flushes
// before its Delta is read.
void flush_recs(mpc_ctx* ctx, const Small& s) {
  if (!s.nrec) return;
  launch_rec_hash(ctx->st, s.rec, s.nrec, ctx->status, ST_ABORT);
  s.nrec = 0;
}

// Pi_Rec of one shared GR element (3 shares + 3 hashes): the record its messages go to, and the
// REC_MSG fault that is due, which corrupts the P0 -> P1 share, as for any other Pi_Rec.
struct Rec1 {
  u64* rec;
  MsgFault fault;
};
Rec1 begin_rec(mpc_ctx* ctx, const Small& s) {
  if (s.nrec == REC_SLOTS) flush_recs(ctx, s);
  Rec1 r;
  r.rec = s.rec + (long long)s.nrec++ * REC_WORDS;
  r.fault = take_fault(ctx, MPC_SITE_REC_MSG, 64);
  count_msgs(ctx, MPC_PHASE_VERIFY, MPC_PROTO_VERIFY, 3, 512);
  count_msgs(ctx, MPC_PHASE_VERIFY, MPC_PROTO_VERIFY, 3, 32);
  return r;
}

// <v> random GR element, revealed with Pi_Rec.
void reveal(mpc_ctx* ctx, u32 purpose, u64 obj, const Small& s, u64* out) {
  const Rec1 r = begin_rec(ctx, s);
  launch_reveal(ctx->st, ctx->k01, ctx->k02, ctx->k12, purpose, obj, r.fault, out, r.rec);
}

// Clears both halves of the round sums and Pi_InnerVerify's; a round adds into cur_sums, and its tail
// clears the other half for the next round.
int sums_begin(mpc_ctx* ctx, const Small& s) {
  s.uc = 0;
  CK(cudaMemsetAsync(s.U, 0, (2 * SUMS_WORDS + IV_ACC_WORDS) * 8, ctx->st));
  return MPC_OK;
}
u64* cur_sums(const Small& s) { return s.U + s.uc * SUMS_WORDS; }

// The part of a Pi_Reduce round after its party sums (sums: 12 blocks S00, S01, S10, S11 of three
// parties, ld words apart: 64 reduced, 128 unreduced coefficients): h(0) and h(p2) by secure GR
// inner products, zeta revealed, the next claim zo, and M_zeta (s.MM) for the folds; the fold
// element is s.coef[0..63].
void round_tail(mpc_ctx* ctx, u64 vid, u32 batch, int k, const u64* z, u64* zo, const Small& s,
                const u64* sums, int ld, u64* trace, u64* V = nullptr, u64* W = nullptr,
                int nvw = 0, const ZeroRows* pad = nullptr) {
  RoundTail a;
  for (int q = 0; q < 12; ++q) a.pad[q] = pad ? pad->p[q] : nullptr;
  a.V = V;   // the weights of a round over a matrix S: folded along bit k - 1
  a.W = W;
  a.nvw = nvw;
  a.vwbit = k - 1;
  a.sums = sums;
  a.ld = ld;
  a.mode = ctx->reduce_mode;
  a.k01 = ctx->k01;
  a.k02 = ctx->k02;
  a.k12 = ctx->k12;
  a.obj = make_obj(vid, batch, (u32)k);
  a.inv = ctx->cst + CST_INV;
  a.z = z;
  a.zo = zo;
  a.coef = s.coef;
  a.MM = s.MM;
  a.zp = s.zp;
  a.zero = s.U + (s.uc ^ 1) * SUMS_WORDS;
  a.nzero = SUMS_WORDS;
  a.trace = trace ? trace + (long long)(k - 1) * TRACE_ROUND : nullptr;
  count_msgs(ctx, MPC_PHASE_VERIFY, MPC_PROTO_VERIFY, 6, 512);   // two secure inner products
  const Rec1 r = begin_rec(ctx, s);
  a.rec = r.rec;
  a.fault = r.fault;
  launch_round_tail(ctx->st, a);
  s.uc ^= 1;
}

// The rows past vectors of D elements, when D is odd.
ZeroRows pad_rows(const Vec& x, const Vec& y, long long D) {
  ZeroRows r{};
  for (int c = 0; c < 6 && (D & 1); ++c) {
    r.p[c] = x.c[c] ? x.c[c] + D * 64 : nullptr;
    r.p[6 + c] = y.c[c] ? y.c[c] + D * 64 : nullptr;
  }
  return r;
}

// One Pi_Reduce round on a dense claim (Fig. Reduce).  x, y: current vectors (D elements, with
// capacity for D+1), z: current claim; writes the folded vectors into xo, yo and z into zo.
int reduce_round_dense(mpc_ctx* ctx, u64 vid, u32 batch, int k, const Vec& x, const Vec& y,
                       long long D, const u64* z, Vec& xo, Vec& yo, u64* zo, const Small& s,
                       u64* trace) {
  cudaStream_t st = ctx->st;
  const long long Dh = (D + 1) / 2;
  // a vector of odd length is followed by a row of zeros: the tail clears those of the vectors that
  // this round folds into (before the fold; the first round's are run_dense's)
  ZeroRows pad = pad_rows(xo, yo, Dh);
  View f[2], g[2];
  for (int a = 0; a < 2; ++a) {
    for (int c = 0; c < 6; ++c) {
      f[a].c[c] = x.c[c] ? x.c[c] + 64 * a : nullptr;
      g[a].c[c] = y.c[c] ? y.c[c] + 64 * a : nullptr;
    }
    f[a].ld = 128;
    g[a].ld = 128;
  }
  u64* S00 = s.S;
  u64* S01 = s.S + 192;
  u64* S10 = s.S + 384;
  u64* S11 = s.S + 576;
  int rc;
  // Shape of the truncation batch's dense rounds: x holds only [r]_1 (P0, P1 copies), y only
  // [r]_2 (P0, P2 copies), so P1's and P2's cross terms vanish and P0's sums are single Grams.
  const bool bit_form = x.c[0] && !x.c[1] && !x.c[2] && x.c[3] && !x.c[4] && !x.c[5] &&
                        !y.c[0] && y.c[1] && !y.c[2] && !y.c[3] && !y.c[4] && y.c[5];
  u64* U = cur_sums(s);
  const u64* sums = s.S;   // reduced sums of the CUDA-core Grams unless set below
  int ld = 64;
  if (bit_form) {
    bool done = false;
    if (ctx->gemm_path == MPC_GEMM_LIMB_TC) {
      // tensor cores: G00, G11 and the cross sum G01 + G10 directly
      {
        Phase kp(ctx, MPC_PROF_K_GRAM, 4.0 * Dh * 4096);
        done = gram3_tc(st, Dh, x.c[0], y.c[1], U, ctx->status, ST_TIMEOUT,
                        ctx->tune.gram_split) == 0;
      }
      if (done) {
        sums = U;
        ld = 128;
      }
    }
    if (!done) {
      // G00, G11 and G(x0 + x1, y0 + y1); G01 + G10 = G(x0 + x1, y0 + y1) - G00 - G11
      CK(cudaMemsetAsync(s.Pmat, 0, 3 * 4096 * 8, st));
      CK(cudaMemsetAsync(s.S, 0, 4 * 192 * 8, st));
      gram(ctx, s.Pmat, x.c[0], nullptr, 1, 128, y.c[1], nullptr, 1, 128, Dh, 1);
      gram(ctx, s.Pmat + 4096, x.c[0] + 64, nullptr, 1, 128, y.c[1] + 64, nullptr, 1, 128, Dh, 1);
      gram(ctx, s.Pmat + 8192, x.c[0], x.c[0] + 64, 1, 128, y.c[1], y.c[1] + 64, 1, 128, Dh, 1);
      launch_gr_fold_reduce(st, s.Pmat, 3, s.aux);            // aux: G00, G11, Gsum (64 each)
      CK(cudaMemcpyAsync(S00, s.aux, 512, cudaMemcpyDeviceToDevice, st));
      CK(cudaMemcpyAsync(S11, s.aux + 64, 512, cudaMemcpyDeviceToDevice, st));
      launch_addsub(st, 64, s.aux + 128, s.aux, 1, s.aux + 192);
      launch_addsub(st, 64, s.aux + 192, s.aux + 64, 1, S01);
    }
  } else {
    bool done = false;
    if (ctx->gemm_path == MPC_GEMM_LIMB_TC) {
      // tensor cores: the party sums of S00, S11 and S01 + S10 as Gram blocks (in S01; S10 = 0),
      // one job per Gram term.  P0: G(x0 + x1, y0 + y1); P1: -G(x2, y3) - G(y2, x3);
      // P2: G(x4, y4 - y5) - G(y4, x5).  A term with an absent first source takes the second's
      // scale into its sign; a term with an absent side is zero.
      const u64 M1 = ~0ull;
      GramJobs jobs{};
      jobs.off_x = 3 * 128;
      jobs.off_oo = 9 * 128;
      auto add = [&](int party, const u64* a0, const u64* a1, u64 sa1, const u64* b0,
                     const u64* b1, u64 sb1, u64 sign) {
        if (!a0) { a0 = a1; a1 = nullptr; sign *= sa1; }
        if (!b0) { b0 = b1; b1 = nullptr; sign *= sb1; }
        if (!a0 || !b0) return;
        jobs.j[jobs.n++] = GramJob{a0, a1, sa1, b0, b1, sb1, U + party * 128, sign};
      };
      add(0, x.c[0], x.c[1], 1, y.c[0], y.c[1], 1, 1);
      add(1, x.c[2], nullptr, 0, y.c[3], nullptr, 0, M1);
      add(1, y.c[2], nullptr, 0, x.c[3], nullptr, 0, M1);
      add(2, x.c[4], nullptr, 0, y.c[4], y.c[5], M1, 1);
      add(2, y.c[4], nullptr, 0, x.c[5], nullptr, 0, M1);
      {
        Phase kp(ctx, MPC_PROF_K_GRAM, 4.0 * Dh * 4096 * jobs.n);
        done = gram_jobs_tc(st, Dh, jobs, ctx->status, ST_TIMEOUT, ctx->tune.gram_split) == 0;
      }
      if (done) {
        sums = U;   // S00 | S01 + S10 | 0 | S11
        ld = 128;
      }
    }
    if (!done) {
      if ((rc = party_sums(ctx, f[0], g[0], Dh, s.Pmat, S00))) return rc;
      if ((rc = party_sums(ctx, f[0], g[1], Dh, s.Pmat + 3 * 4096, S01))) return rc;
      if ((rc = party_sums(ctx, f[1], g[0], Dh, s.Pmat + 6 * 4096, S10))) return rc;
      if ((rc = party_sums(ctx, f[1], g[1], Dh, s.Pmat + 9 * 4096, S11))) return rc;
    }
  }
  round_tail(ctx, vid, batch, k, z, zo, s, sums, ld, trace, nullptr, nullptr, 0, &pad);
  // f(zeta) = f(0) + zeta (f(1) - f(0)): rows [x_{2i+1} - x_{2i}] times M_zeta, plus x_{2i}.
  // Vectors that sit at one stride (the dense plans put a slot's x vectors, then its y vectors,
  // one after another) go through one launch: segment s of Dh rows (padded to whole tiles); all
  // of them when x's and y's rows have the same capacity, else each side's.  Only short vectors
  // are batched: there one launch replaces several latency-bound ones, while on long ones the
  // segment arithmetic of the batched row map costs more than the launches it saves.
  auto fold_batched = [&](const u64* const* ins, u64* const* outs, int n) -> bool {
    if (ctx->gemm_path != MPC_GEMM_LIMB_TC || Dh > ctx->tune.fold_batch_max || n < 2) return false;
    const long long sin = ins[1] - ins[0], sout = outs[1] - outs[0];
    for (int i = 1; i < n; ++i)
      if (ins[i] - ins[0] != i * sin || outs[i] - outs[0] != i * sout) return false;
    if (sin <= 0 || sout <= 0) return false;
    const long long Rp = (Dh + 127) / 128 * 128;
    GrMMArgs g = grargs(ctx);
    g.R = n * Rp;
    g.p0 = ins[0] + 64;
    g.p1 = ins[0];
    g.s1 = ~0ull;
    g.in = GrRowMap{Rp, 128, sin};
    g.qvalid = Dh;
    g.Mmat = s.MM;
    g.add0 = ins[0];
    g.add0_in = 1;
    g.out = outs[0];
    g.om = GrRowMap{Rp, 64, sout};
    Phase kp(ctx, MPC_PROF_K_GR_MATMUL, (double)n * Dh * 4096);
    if (gr_matmul_tc_ex(st, g, ctx->status, ST_TIMEOUT) == 0) return true;
    return false;
  };
  const u64* ins[12];
  u64* outs[12];
  int nx = 0, n = 0;
  for (int side = 0; side < 2; ++side)
    for (int c = 0; c < 6; ++c) {
      const u64* in = side ? y.c[c] : x.c[c];
      if (!in) continue;
      ins[n] = in;
      outs[n] = side ? yo.c[c] : xo.c[c];
      ++n;
      if (!side) ++nx;
    }
  bool done_all = fold_batched(ins, outs, n);
  for (int side = 0; side < 2 && !done_all; ++side) {
    const int i0 = side ? nx : 0, i1 = side ? n : nx;
    if (fold_batched(ins + i0, outs + i0, i1 - i0)) continue;
    for (int i = i0; i < i1; ++i)
      if ((rc = gr_matmul(ctx, Dh, ins[i] + 64, ins[i], ~0ull, 128, s.MM, ins[i], 128, outs[i], 64)))
        return rc;
  }
  return cuda_check(ctx, "reduce_round");
}

// Pi_InnerVerify (Fig. DPV) on a dense claim of dimension D.
int inner_verify_dense(mpc_ctx* ctx, u64 vid, u32 batch, const Vec& x, const Vec& y, long long D,
                       const u64* z, const Small& s, u64* trace, int R) {
  InnerVerify a;
  for (int c = 0; c < 6; ++c) {
    a.x[c] = x.c[c];
    a.y[c] = y.c[c];
  }
  a.z = z;
  a.D = D;
  a.k01 = ctx->k01;
  a.k02 = ctx->k02;
  a.k12 = ctx->k12;
  a.obj = make_obj(vid, batch, 0);
  a.acc = s.U + 2 * SUMS_WORDS;
  count_msgs(ctx, MPC_PHASE_VERIFY, MPC_PROTO_VERIFY, 3, (u64)D * 512);   // x alpha
  count_msgs(ctx, MPC_PHASE_VERIFY, MPC_PROTO_VERIFY, 3, 512);            // the inner product
  const Rec1 r = begin_rec(ctx, s);
  a.rec = r.rec;
  a.fault = r.fault;
  a.trace = trace ? trace + (long long)R * TRACE_ROUND : nullptr;
  a.status = ctx->status;
  a.flag = ST_VERIFY;
  launch_inner_verify(ctx->st, a);
  flush_recs(ctx, s);
  return cuda_check(ctx, "inner_verify");
}

// Elements of a claim up to which a round's fold and sums are one launch on the CUDA cores (on the
// limb path): at 512 its 256 blocks still run at once, 16 us against 36; it would double with each
// doubling, the tensor-core launches hardly grow up to 4096.
constexpr long long SMALL_MAX = 512;

// Dense rounds k = k0..R followed by Pi_InnerVerify.
int run_dense(mpc_ctx* ctx, u64 vid, u32 batch, Dense& dv, long long D, const u64* z0, int k0,
              int R, const Small& s, u64* trace) {
  int rc;
  const u64* z = z0;
  int zi = 0;
  const bool tc = ctx->gemm_path == MPC_GEMM_LIMB_TC;
  int k = k0;
  if (k <= R && (D & 1) && !(tc && D <= SMALL_MAX))
    launch_zero_rows(ctx->st, pad_rows(dv.x[dv.cur], dv.y[dv.cur], D));
  for (; k <= R && !(tc && D <= SMALL_MAX); ++k) {
    Vec& x = dv.x[dv.cur];
    Vec& y = dv.y[dv.cur];
    Vec& xo = dv.x[dv.cur ^ 1];
    Vec& yo = dv.y[dv.cur ^ 1];
    u64* zo = s.z[zi];
    if ((rc = reduce_round_dense(ctx, vid, batch, k, x, y, D, z, xo, yo, zo, s, trace))) return rc;
    z = zo;
    zi ^= 1;
    dv.cur ^= 1;
    D = (D + 1) / 2;
  }
  // short claims: each launch folds by the round before's f and takes this round's sums
  bool fold = false;
  for (; k <= R + 1; ++k) {
    if (k > R && !fold) break;
    SmallRound a;
    const int o = dv.cur ^ 1;
    for (int c = 0; c < 6; ++c) {
      a.in[c] = dv.x[dv.cur].c[c];
      a.in[6 + c] = dv.y[dv.cur].c[c];
      a.out[c] = dv.x[o].c[c];
      a.out[6 + c] = dv.y[o].c[c];
    }
    a.f = s.coef;
    a.D = D;
    a.fold = fold;
    a.sums = k <= R ? cur_sums(s) : nullptr;
    launch_small_round(ctx->st, a);
    if (fold) {
      dv.cur = o;
      D = (D + 1) / 2;
    }
    if (k > R) break;
    round_tail(ctx, vid, batch, k, z, s.z[zi], s, a.sums, 128, trace);
    z = s.z[zi];
    zi ^= 1;
    fold = true;
  }
  return inner_verify_dense(ctx, vid, batch, dv.x[dv.cur], dv.y[dv.cur], D, z, s, trace, R);
}

long long dim_after(long long D, int R) {
  for (int k = 0; k < R; ++k) D = (D + 1) / 2;
  return D;
}

// Allocate ping-pong vectors for a dense claim of dimension D over the present components: a
// slot's x vectors, then its y vectors, each side's present vectors at one stride (the batched
// folds use that).
Dense plan_dense(Arena& a, long long D, const bool xc[6], const bool yc[6]) {
  Dense d;
  d.cap[0] = D + 1;
  d.cap[1] = (D + 1) / 2 + 1;
  for (int i = 0; i < 2; ++i) {
    for (int c = 0; c < 6; ++c) d.x[i].c[c] = xc[c] ? a.take<u64>(d.cap[i] * 64) : nullptr;
    for (int c = 0; c < 6; ++c) d.y[i].c[c] = yc[c] ? a.take<u64>(d.cap[i] * 64) : nullptr;
  }
  return d;
}

// Reads the status word after a verification; the products under pend_key leave the pending
// set only on a clean status (after a failure the context is aborted for good).
int finish_verify(mpc_ctx* ctx, u64 pend_key) {
  u32 stv = 0;
  int rc = read_status(ctx, &stv);
  if (rc) return rc;
  if (!(stv & (ST_ABORT | ST_VERIFY))) ctx->pending.erase(pend_key);
  if (stv & ST_ABORT) {
    ctx->aborted = true;
    return fail(ctx, MPC_ERR_ABORT, "Pi_Rec: inconsistent messages");
  }
  if (stv & ST_VERIFY) {
    ctx->aborted = true;
    return fail(ctx, MPC_ERR_VERIFY, "verification failed: Delta != 0");
  }
  return MPC_OK;
}

// ---- plans ----------------------------------------------------------------------------------
struct MatmulPlan {
  u64 *g2, *mz1, *mz2;             // the product's messages
  u64 *gp2, *gq2, *mp1, *mq1;      // the truncation pairs' messages
  FaultCopies fc;
  void* tc;   // digit planes of the tensor-core path (null on the u64 path)
};

MatmulPlan plan_matmul(Arena& a, long long M, long long N, long long K, bool trunc, bool tc) {
  const long long E = M * N;
  MatmulPlan p{};
  p.tc = tc ? (void*)a.take<unsigned char>((long long)limb_tc_scratch_bytes(M, N, K, 2)) : nullptr;
  p.g2 = a.take<u64>(E);
  p.mz1 = a.take<u64>(E);
  p.mz2 = a.take<u64>(E);
  if (trunc)
    for (u64** b : {&p.gp2, &p.gq2, &p.mp1, &p.mq1}) *b = a.take<u64>(E);
  p.fc = plan_copies(a, E);
  return p;
}

struct RecPlan : RecBufs {
  u64* out_dev;
};

RecPlan plan_rec(Arena& a, long long n, bool need_out) {
  RecPlan p{};
  p.in_p2_r1 = a.take<u64>(n);
  p.in_p1_r2 = a.take<u64>(n);
  p.in_p0_m = a.take<u64>(n);
  for (int i = 0; i < 6; ++i) p.hs[i] = a.take<u32>((long long)hash_scratch_words(n));
  p.dg = a.take<u32>(48);
  p.out_dev = need_out ? a.take<u64>(n) : nullptr;
  return p;
}

// Pi_Rec of n words up to the hash comparison (into the status word): P0 sends [r]_1 to P2 and
// [r]_2 to P1 (fault site REC_MSG, arithmetic sharings), P1 sends m to P0; P1 sends H([r]_1) to P2,
// P2 H(m) to P0 and H([r]_2) to P1, and every receiver hashes what it received.  out = P1's opening.
void rec_core(mpc_ctx* ctx, const u64* xs, long long n, const RecPlan& p, u64* out, bool boolean) {
  const MsgFault f = take_fault(ctx, boolean ? -1 : MPC_SITE_REC_MSG, n);
  launch_rec(ctx->st, xs, n, f, boolean, p, out, ctx->status, ST_ABORT);
  count_msgs(ctx, MPC_PHASE_ONLINE, MPC_PROTO_REC, 3, (u64)n * 8);
  count_msgs(ctx, MPC_PHASE_ONLINE, MPC_PROTO_REC, 3, 32);
}

// A table of powers r^i, i < n (rows of 64 words): rows below L by repeated multiplication, row
// h L + l (h >= 1) = r^(hL) r^l, all of them one grouped GR-matrix product (matrix h - 1 for the
// rows L h .. L h + L - 1).  L is a multiple of 128 near sqrt(n).
struct PowPlan {
  long long n, L, nhi;
  u64* Thi;   // r^(hL), h < nhi
  u64* Mhi;   // multiplication matrices of r^(hL), h = 1 .. nhi - 1
};

PowPlan plan_pow(Arena& a, long long n) {
  PowPlan p;
  p.n = n;
  long long L = 1024;
  while (L * L < n) L += 128;
  p.L = L;
  p.nhi = (n + L - 1) / L;
  p.Thi = a.take<u64>(p.nhi * 64);
  p.Mhi = a.take<u64>(std::max<long long>(p.nhi - 1, 1) * 4096);
  return p;
}

// table[i] = r^i for i < p.n; aux: 64 words of scratch
int power_table(mpc_ctx* ctx, const u64* r, const PowPlan& p, u64* table, u64* aux) {
  cudaStream_t st = ctx->st;
  if (ctx->gemm_path != MPC_GEMM_LIMB_TC || p.nhi <= 1) {
    launch_gr_powers(st, r, p.n, table);
    return MPC_OK;
  }
  launch_gr_powers(st, r, p.L, table);
  launch_gr_mul1(st, table + (p.L - 1) * 64, r, aux);                 // r^L
  launch_gr_powers(st, aux, p.nhi, p.Thi);
  launch_gr_mulmat_batch(st, p.nhi - 1, p.Thi + 64, 64, p.Mhi);
  GrMMArgs g = grargs(ctx);
  g.R = (p.nhi - 1) * p.L;
  g.p0 = table;
  g.in = GrRowMap{p.L, 64, 0};
  g.Mmat = p.Mhi;
  g.mrows = p.L;
  g.out = table + p.L * 64;
  g.om = GrRowMap{0, 64, 0};
  g.out_lim = (p.n - p.L) * 64;
  Phase kp(ctx, MPC_PROF_K_GR_MATMUL, (double)(p.n - p.L) * 4096);
  if (gr_matmul_tc_ex(st, g, ctx->status, ST_TIMEOUT) == 0) return MPC_OK;
  launch_gr_powers(st, r, p.n, table);
  return MPC_OK;
}

// A batch of weighted ring words (gr_block.cu): x_i = R_{b >> sh} T_j X_i, y_i = lift(Y_i), i =
// B b + j < D, whose first kap = log2(B) rounds need no GR vectors.
constexpr int BLK_ROUNDS = 3;
// Words from which a batch takes four rounds that way, its sums on the tensor cores (65520
// words: 58 us of CUDA-core sums for three rounds; 65536: 65 us in three launches for four, and the dense
// round on 8192 elements, about 70 us, is gone).
constexpr long long BLK_TC_MIN = 1 << 16;
struct BlkPlan {
  long long D, nb;        // words, blocks
  long long nw, nwp;      // weight rows R, rounded up to whole tiles
  int R, kap, B, sh;
  bool tc;                // B = 16, sums on the tensor cores
  bool full;              // all components and the claim's sums; else x has 2 and 4 only
  PowPlan pp;
  u64 *T, *Rw, *S, *V, *W, *Vm, *G;
  void* planes;           // the sums' digit planes (tc), under G and dv, which come after the rounds
  Dense dv;
};

// wlog: log2 of the words per weight step (0: weights r^i; 6: r^(i / 64), T_j = 1)
BlkPlan plan_blk(Arena& a, long long D, int R, int wlog, bool full, const bool xc[6],
                 const bool yc[6], bool tc) {
  BlkPlan p;
  p.D = D;
  p.R = R;
  p.tc = tc && D >= BLK_TC_MIN && R > BLK_ROUNDS;
  p.kap = p.tc ? BLK_ROUNDS + 1 : std::min(R, BLK_ROUNDS);
  p.B = 1 << p.kap;
  p.nb = (D + p.B - 1) / p.B;
  p.sh = wlog > p.kap ? wlog - p.kap : 0;
  p.nw = ((p.nb - 1) >> p.sh) + 1;
  p.nwp = (p.nw + 127) / 128 * 128;
  p.full = full;
  p.pp = plan_pow(a, p.nw);
  p.T = a.take<u64>((p.B + 1) * 64);
  p.Rw = a.take<u64>(p.nwp * 64);
  p.S = a.take<u64>(blk_rows(p.B, full) * 64);
  p.V = p.T;   // the claim is taken from T before the rounds fold it
  p.W = a.take<u64>(p.B * 64);
  p.Vm = a.take<u64>(p.B * 4096);
  const size_t at = a.off;
  p.G = a.take<u64>(p.nwp * p.B * 64);
  p.planes = p.G;
  p.dv = plan_dense(a, p.nb, xc, yc);
  if (p.tc) a.reserve(at, blk_sums_tc_bytes(full, p.nw));
  return p;
}

// T_j = r^j (j <= B) and the weights R_b = r^(B b) of a batch with weights r^i.
int blk_tables(mpc_ctx* ctx, BlkPlan& p, const u64* r, u64* aux) {
  launch_gr_powers(ctx->st, r, p.B + 1, p.T);
  return power_table(ctx, p.T + p.B * 64, p.pp, p.Rw, aux);
}

// The batch from its weights (T, Rw), words (xw, yw: component pointers) and claim (zw: 6 x D
// words, full batches; else s.zinit holds the claim): the first kap rounds from the block sums,
// the vectors after them, and the dense rounds.
int run_blk(mpc_ctx* ctx, u64 vid, u32 batch, BlkPlan& p, const Vec& xw, const Vec& yw,
            const u64* zw, const Small& s, u64* trace) {
  cudaStream_t st = ctx->st;
  const int B = p.B;
  int rc;
  if (!p.tc) CK(cudaMemsetAsync(p.S, 0, (size_t)blk_rows(B, p.full) * 512, st));
  BlkIn in;
  for (int c = 0; c < 6; ++c) {
    in.x[c] = xw.c[c];
    in.y[c] = yw.c[c];
  }
  in.z = zw;
  in.ldz = p.D;
  in.D = p.D;
  // parties 1 and 2 only: their matrices sit where those of a full batch's first two would
  const int np = p.full ? 3 : 2, p0 = p.full ? 0 : 1;
  if (p.tc) {
    if (blk_sums_tc(st, in, p.full, p.nw, p.Rw, p.S, p.planes, ctx->status, ST_TIMEOUT,
                    ctx->tune.gemm_split_min))
      return fail(ctx, MPC_ERR_CUDA, "block sums: tensor maps");
  } else if (p.full || p.kap > 0) {
    launch_blk_sums(st, in, B, p.full, p.nb, p.sh, p.Rw, p.S);
  }
  if (p.full) {
    CK(cudaMemsetAsync(s.zinit, 0, 384 * 8, st));
    launch_blk_claim(st, p.T, p.S + 3ll * B * B * 64, B, s.zinit);
  }
  launch_ones(st, B, p.W);
  const u64* z = s.zinit;
  for (int k = 1; k <= p.kap; ++k) {
    u64* sums = cur_sums(s);
    launch_weighted_sums(st, p.V, p.W, p.S, B, k, np, sums + 64 * p0);
    u64* zo = s.z[k & 1];
    round_tail(ctx, vid, batch, k, z, zo, s, sums, 64, trace, p.V, p.W, B);
    z = zo;
  }
  // G row b B + j = R_b V_j
  bool done = false;
  launch_gr_mulmat_batch(st, B, p.V, 64, p.Vm);
  if (ctx->gemm_path == MPC_GEMM_LIMB_TC) {
    GrMMArgs g = grargs(ctx);
    g.R = B * p.nwp;   // rows j nwp + b read R_b, matrix j
    g.p0 = p.Rw;
    g.in = GrRowMap{p.nwp, 64, 0};
    g.Mmat = p.Vm;
    g.mrows = p.nwp;
    g.out = p.G;
    g.om = GrRowMap{p.nwp, 64ll * B, 64};
    Phase kp(ctx, MPC_PROF_K_GR_MATMUL, (double)g.R * 4096);
    done = gr_matmul_tc_ex(st, g, ctx->status, ST_TIMEOUT) == 0;
  }
  for (int j = 0; j < B && !done; ++j)
    if ((rc = gr_matmul(ctx, p.nw, p.Rw, nullptr, 1, 64, p.Vm + j * 4096, nullptr, 0, p.G + j * 64,
                        64ll * B)))
      return rc;
  BlkVec vi;
  BlkOut vo;
  for (int side = 0; side < 2; ++side) {
    for (int c = 0; c < 6; ++c) {
      vi.c[c] = side ? yw.c[c] : xw.c[c];
      vo.c[c] = side ? p.dv.y[0].c[c] : p.dv.x[0].c[c];
    }
    launch_blk_combine(st, vi, vo, B, side == 0, p.D, p.nb, side ? 0 : p.sh, side ? p.W : p.G);
  }
  if (z != s.zinit) CK(cudaMemcpyAsync(s.zinit, z, 384 * 8, cudaMemcpyDeviceToDevice, st));
  p.dv.cur = 0;
  if ((rc = cuda_check(ctx, "block rounds"))) return rc;
  return run_dense(ctx, vid, batch, p.dv, p.nb, s.zinit, p.kap + 1, p.R, s, trace);
}

struct VMultPlan {
  Small s;
  BlkPlan b;
  int R;
};

VMultPlan plan_vmult(Arena& a, long long n, int R, bool tc) {
  VMultPlan p;
  p.R = R < 0 ? default_R(n) : R;
  p.s = plan_small(a);
  const bool all[6] = {true, true, true, true, true, true};
  p.b = plan_blk(a, n, p.R, 0, true, all, all, tc);
  return p;
}

// deferred Pi_MultVerify over several calls: the gathered triples, then the verification plan
struct VMultCallsPlan {
  u64 *x, *y, *z;
  VMultPlan v;
};

VMultCallsPlan plan_vmult_calls(Arena& a, long long n, int R, bool tc) {
  VMultCallsPlan p;
  p.x = a.take<u64>(6 * n);
  p.y = a.take<u64>(6 * n);
  p.z = a.take<u64>(6 * n);
  p.v = plan_vmult(a, n, R, tc);
  return p;
}

// One verification chunk of the truncation batch (E consecutive outputs of the layer).
struct TruncPlan {
  long long E = 0;
  int R1 = 0, kd = 0;
  long long Dt = 0;
  long long L = 0, Epad = 0, nhi = 0;   // S = sum over e_hi < nhi of T_hi (x) (sum over e_lo < L ...)
  u64 *b1, *b2, *Rtab, *S, *Zpq, *V, *W, *zt, *S_hi, *Thi, *Mhi;
  u64* Pst = nullptr;   // 64 x 262144: the combination's products before their fold (u64 GEMM form)
  PowPlan pow;          // the table r^(2 e_lo), e_lo < L
  u64 *B1T, *B2T;   // bit-transposed b1, b2: [j][e / 64]
  unsigned char* TL8;
  // tensor-core materialisation with r^(2e) = r^(2 Lm e_hi) r^(2 e_lo), e = e_hi Lm + e_lo:
  // Tm[e_lo][j] = r^(2 e_lo) (-V_j), Bm[e_hi] = M(r^(2 Lm e_hi)), Vm[j] = M(-V_j), bT = b1 in
  // (e_lo, e_hi) order (nhm x Lm view transposed)
  long long Lm = 0, nhm = 0;
  u64 *Tm = nullptr, *Bm = nullptr, *Vm = nullptr, *bT = nullptr;
  // compact table (E a multiple of L on that path): only r^(2 e_lo), e_lo < L, is materialised;
  // sum_e r^(2e) pq_c[e] = sum_{e_hi} T_hi[e_hi] (sum_{e_lo} pq_c[e] r^(2 e_lo)) (a limb GEMM over
  // the first block, then 12 nhi GR products), and the rows r^(2 Lm e_hi) come from T_hi x r^(2 e_lo)
  bool compact = false;
  u64 *Zhi = nullptr, *Zrep = nullptr, *Zprod = nullptr, *Prow = nullptr;
  u64* pqc = nullptr;        // the chunk's 12 rows of <p>, <q> gathered (chunked batches only)
  Dense dt;
};

// A truncation batch of E outputs: nchunks chunks of C outputs (the last one ragged).
struct TruncBatch {
  long long E = 0, nchunks = 0, C = 0;
  TruncPlan tp[2];   // plans of a full chunk and of the ragged last one
};

struct VMatPlan {
  Small s, st;                    // batch 0's and the truncation batch's
  u64 *Q, *P, *T, *Pz;
  PowPlan powQ, powP;
  Dense dv;
  int R0;
  bool trunc = false;
  TruncBatch tb;
  void *tcs = nullptr, *tcst = nullptr;   // tensor-core digit planes of the two (limb path only)
  bool fork = false;              // the two side by side (their scratch apart)
  bool grouped = false;           // X^T P and W Q of all six components as one product each
};
// Outputs up to which batch 0 and the truncation batch run side by side: above, batch 0 is a few
// percent of the call and its scratch is better shared (64 x 64 x 128: 1.05 ms one after the other, 0.89
// side by side).
constexpr long long FORK_MAX = 1ll << 22;
// Words of a grouped operand at most (256 MB of digit planes).  Below, a product of one component is
// a few CTAs and its four launches take longer than its work (17 products of a layer: 1.67 ms a
// verified product of 64 x 64 x 128, 1.32 ms with seven); above, each fills the GPU.
constexpr long long GROUPED_MAX = 1ll << 24;

// Layout decisions of a truncation chunk of E outputs (no allocation).
struct TruncShape {
  long long L, Epad, nhi, Lm = 0, nhm = 0;
  int R1, kd;
  bool compact = false, blocked = false;
  bool comb_tc = false;   // S_hi combined by GR products (else by one u64 GEMM over the blocks)
};

TruncShape trunc_shape(long long E, int R1, bool tc, const mpc_tuning& tu) {
  TruncShape h;
  h.R1 = R1 < 0 ? default_R(64 * E) : R1;
  h.kd = std::min(h.R1, 6);
  const long long Lb = tu.trunc_block;
  h.blocked = E >= Lb;
  h.L = h.blocked ? Lb : ((E + 127) / 128) * 128;
  h.Epad = ((E + h.L - 1) / h.L) * h.L;
  h.nhi = h.Epad / h.L;
  // One pass of 64 x 262144 x nhi multiply-adds on the CUDA cores, or nhi - 1 GR products of 4096 rows:
  // the tensor cores take those from the second block on (a verification of 100003 truncations, two
  // blocks: 1.66 ms against 1.95; 1051000, 17 blocks: 8.80 against 9.26).  On the CUDA cores a product
  // is 32 blocks of threads, and the pass is the better form (256 blocks: 3.5 ms a chunk against 11.7).
  h.comb_tc = tc && h.nhi >= tu.tc_combine_min;
  h.compact = tc && h.kd == 6 && h.blocked && E % h.L == 0;
  if (tc && h.kd == 6 && h.blocked) {
    if (tu.row_split > 0) {
      // at most E rounded up to a tile: the row-split table reads r^(2 e_lo) for e_lo < Lm
      h.Lm = std::min<long long>(tu.row_split, (E + 127) / 128 * 128);
      h.nhm = ((E + h.Lm - 1) / h.Lm + 127) / 128 * 128;
    } else {
      // Lm = 128 a with a odd near sqrt(E) / 128, and nhm = 128 b >= E / Lm with the fewest rows
      // past E: the bit product writes its rows Lm rows apart, and a stride of a multiple of
      // 2 MB (a even at E = 2^24) puts a tile's 128 rows on the same memory channels
      long long sq = 1;
      while (sq * sq < E) ++sq;
      const long long a0 = (sq + 127) / 128;
      h.Lm = 128 * a0;
      h.nhm = ((E + h.Lm - 1) / h.Lm + 127) / 128 * 128;
      if (a0 >= 4) {   // strides of 512 KB and more
        long long best = -1;
        for (long long aa = (a0 * 3 / 4) | 1; aa <= 2 * a0 + 1; aa += 2) {
          const long long bb = (E + 128 * 128 * aa - 1) / (128 * 128 * aa);
          const long long rows = 128 * 128 * aa * bb;
          if (best < 0 || rows < h.Lm * h.nhm ||
              (rows == h.Lm * h.nhm && std::llabs(aa - a0) < std::llabs(best - a0))) {
            best = aa;
            h.Lm = 128 * aa;
            h.nhm = 128 * bb;
          }
        }
      }
    }
    // the compact table keeps r^(2 e_lo) for e_lo < L only, and the row-split table reads e_lo < Lm
    if (h.Lm > h.L) h.compact = false;
  }
  return h;
}

// tensor-core scratch of a truncation chunk: the compact table's sum over the first block
// (12 nhi x 64 x L)
size_t trunc_tc_scratch(const TruncShape& h) {
  return h.compact ? limb_tc_scratch_bytes(12 * h.nhi, 64, h.L, 1) : 0;
}

// whole_table: every power rho^e is kept (the caller reads them)
TruncPlan plan_trunc(Arena& a, long long E, int R1, bool tc, bool chunked, const mpc_tuning& tu,
                     bool whole_table = false) {
  TruncPlan p;
  TruncShape h = trunc_shape(E, R1, tc, tu);
  if (whole_table) h.compact = false;
  p.E = E;
  p.R1 = h.R1;
  p.kd = h.kd;
  p.Dt = E * (64 >> p.kd);
  p.L = h.L;
  p.Epad = h.Epad;
  p.nhi = h.nhi;
  p.compact = h.compact;
  p.b1 = a.take<u64>(p.Epad);
  p.b2 = a.take<u64>(p.Epad);
  p.Rtab = a.take<u64>((p.compact ? p.L : p.Epad) * 64);
  p.TL8 = a.take<unsigned char>(64ll * TRUNC_LIMBS * p.L);
  p.B1T = a.take<u64>(p.Epad);
  p.B2T = a.take<u64>(p.Epad);
  p.S_hi = a.take<u64>(p.nhi * 4096 * 64);
  p.S = p.nhi > 1 ? a.take<u64>(4096 * 64) : p.S_hi;   // one block: T_hi[0] = 1
  if (p.nhi > 1 && !h.comb_tc) p.Pst = a.take<u64>(64ll * 262144);
  p.pow = plan_pow(a, p.L);
  p.Thi = a.take<u64>(p.nhi * 64);
  p.Mhi = a.take<u64>(std::max<long long>(1, p.nhi - 1) * 4096);
  p.Zpq = a.take<u64>(12 * 64);
  p.V = a.take<u64>(4096);
  p.W = a.take<u64>(4096);
  p.zt = a.take<u64>(2 * 384);
  if (chunked) p.pqc = a.take<u64>(12 * E);
  if (h.Lm) {
    p.Lm = h.Lm;
    p.nhm = h.nhm;
    p.Tm = a.take<u64>(p.Lm * 4096);
    p.Bm = a.take<u64>((E + p.Lm - 1) / p.Lm * 4096);
    if (p.compact) {
      p.Zhi = a.take<u64>(12 * p.nhi * 64);
      p.Zrep = a.take<u64>(12 * p.nhi * 64);
      p.Zprod = a.take<u64>(12 * p.nhi * 64);
      p.Prow = a.take<u64>(3 * ((E + p.Lm - 1) / p.Lm) * 64);
    }
    p.Vm = a.take<u64>(64 * 4096);
    p.bT = a.take<u64>(p.nhm * p.Lm);
  }
  const bool xc[6] = {true, false, false, true, false, false};
  const bool yc[6] = {false, true, false, false, false, true};
  p.dt = plan_dense(a, p.Dt, xc, yc);
  return p;
}

// Chunks of the truncation batch of E outputs: n chunks of C outputs, the last E - (n-1) C.
void trunc_chunks(long long E, const mpc_tuning& tu, long long* n, long long* C) {
  *C = std::min<long long>(E, tu.trunc_chunk);
  *n = (E + *C - 1) / *C;
}
constexpr long long MAX_TRUNC_CHUNKS = 15;   // batch ids 1 .. 15 of the object-id layout

// Tensor-core scratch of a truncation batch of E outputs (the larger of its two chunk shapes);
// -1 when it has more than MAX_TRUNC_CHUNKS chunks.
long long trunc_batch_tcs(long long E, int R1, bool tc, const mpc_tuning& tu) {
  long long n = 0, C = 0;
  trunc_chunks(E, tu, &n, &C);
  if (n > MAX_TRUNC_CHUNKS) return -1;
  const long long Elast = E - (n - 1) * C;
  return (long long)std::max(trunc_tc_scratch(trunc_shape(C, R1, tc, tu)),
                             trunc_tc_scratch(trunc_shape(Elast, R1, tc, tu)));
}

// The chunks run one after another: their plans share the rest of the workspace.
void plan_trunc_batch(Arena& a, long long E, int R1, bool tc, const mpc_tuning& tu,
                      TruncBatch& b) {
  b.E = E;
  trunc_chunks(E, tu, &b.nchunks, &b.C);
  const long long Elast = E - (b.nchunks - 1) * b.C;
  const bool chunked = b.nchunks > 1;
  const size_t off0 = a.off;
  b.tp[0] = plan_trunc(a, b.C, R1, tc, chunked, tu);
  const size_t off1 = a.off;
  if (Elast != b.C) {
    a.off = off0;
    b.tp[1] = plan_trunc(a, Elast, R1, tc, chunked, tu);
    a.off = std::max(off1, a.off);
  } else {
    b.tp[1] = b.tp[0];
  }
}

// false when the layer cannot be planned (too many truncation chunks)
bool plan_vmat(Arena& a, long long M, long long N, long long K, int t, int R0, int R1, bool tc,
               const mpc_tuning& tu, VMatPlan& p) {
  p.R0 = R0 < 0 ? default_R(K) : R0;
  p.s = plan_small(a);
  p.trunc = t >= 0;
  const long long E = M * N;
  p.fork = p.trunc && E <= FORK_MAX;
  p.st = p.fork ? plan_small(a) : p.s;
  long long trunc_tcs = 0;
  if (p.trunc && (trunc_tcs = trunc_batch_tcs(E, R1, tc, tu)) < 0) return false;
  // digit planes of the batch-0 products (X^T P, W Q, Z Q) and of the truncation chunks'
  // tensor-core products, on the tensor-core path
  const long long G = 6 * (K + 1);
  p.grouped = tc && G * std::max(M, N) <= GROUPED_MAX;
  p.tcs = tc ? (void*)a.take<unsigned char>((long long)std::max(
                   {limb_tc_scratch_bytes(p.grouped ? G : K, 64, M, 1),
                    limb_tc_scratch_bytes(p.grouped ? G : K, 64, N, 1),
                    limb_tc_scratch_bytes(6 * M, 64, N, 1), (size_t)(p.fork ? 0 : trunc_tcs)}))
             : nullptr;
  p.tcst = p.fork && tc && trunc_tcs > 0 ? (void*)a.take<unsigned char>(trunc_tcs) : p.tcs;
  p.Q = a.take<u64>(N * 64);
  p.P = a.take<u64>(M * 64);
  p.powQ = plan_pow(a, N);
  p.powP = plan_pow(a, M);
  p.T = a.take<u64>(6 * M * 64);
  p.Pz = a.take<u64>(6 * 4096);
  const bool all[6] = {true, true, true, true, true, true};
  p.dv = plan_dense(a, K, all, all);
  if (p.trunc) plan_trunc_batch(a, E, R1, tc, tu, p.tb);
  return true;
}

// plan of a standalone truncation batch's verification (mpc_verify_trunc)
struct VTruncPlan {
  Small s;
  TruncBatch tb;
  void* tcs = nullptr;
};

bool plan_vtrunc(Arena& a, long long n, int R, bool tc, const mpc_tuning& tu, VTruncPlan& p) {
  const long long tcs = trunc_batch_tcs(n, R, tc, tu);
  if (tcs < 0) return false;
  p.s = plan_small(a);
  p.tcs = tc && tcs > 0 ? (void*)a.take<unsigned char>(tcs) : nullptr;
  plan_trunc_batch(a, n, R, tc, tu, p.tb);
  return true;
}

// ---- batches of bit pairs -----------------------------------------------------------------------
// A batch whose 64-element blocks are bit words: x_{64 e + j} = -rho^e V_j b1_{e,j} (held by P0 and
// P1), y_{64 e + j} = -W_j b2_{e,j} (P0 and P2): the truncation pairs (rho = r^2, V_j = u_j, W_j =
// 1) and the edaBit bit products (rho = r^64, V_j = r^j, W_j = 1).  The weights first.
int bit_tables(mpc_ctx* ctx, TruncPlan& p, const Small& s, const u64* rho) {
  cudaStream_t st = ctx->st;
  const long long E = p.E;
  int rc;
  launch_ones(st, 64, p.W);
  if (p.Epad > E) {
    CK(cudaMemsetAsync(p.b1 + E, 0, (size_t)(p.Epad - E) * 8, st));
    CK(cudaMemsetAsync(p.b2 + E, 0, (size_t)(p.Epad - E) * 8, st));
  }
  // rho^e for e < Epad: rho^e_lo for e_lo < L by repeated multiplication, then every further
  // block of L rows is that block times the constant rho^(L e_hi) (a 64 x 64 matrix product)
  if ((rc = power_table(ctx, rho, p.pow, p.Rtab, s.aux + 192))) return rc;
  if (p.compact) {
    launch_gr_mul1(st, p.Rtab + (p.L - 1) * 64, rho, s.aux + 128);   // rho^L
    launch_gr_powers(st, s.aux + 128, p.nhi, p.Thi);
    launch_gr_mulmat_batch(st, p.nhi - 1, p.Thi + 64, 64, p.Mhi);
  } else if (p.nhi > 1) {
    launch_gr_mul1(st, p.Rtab + (p.L - 1) * 64, rho, s.aux + 128);   // rho^L
    launch_gr_powers(st, s.aux + 128, p.nhi, p.Thi);
    // rows h L + e_lo (h >= 1) = rho^(L h) rho^e_lo: one grouped product, matrix h - 1 for
    // the rows (h - 1) L .. h L - 1 of the block, each reading row e_lo of the first block
    launch_gr_mulmat_batch(st, p.nhi - 1, p.Thi + 64, 64, p.Mhi);
    bool done = false;
    if (ctx->gemm_path == MPC_GEMM_LIMB_TC) {
      GrMMArgs g = grargs(ctx);
      g.R = (p.nhi - 1) * p.L;
      g.p0 = p.Rtab;
      g.in = GrRowMap{p.L, 64, 0};
      g.Mmat = p.Mhi;
      g.mrows = p.L;
      g.out = p.Rtab + p.L * 64;
      g.om = GrRowMap{0, 64, 0};
      Phase kp(ctx, MPC_PROF_K_GR_MATMUL, (double)g.R * 4096);
      done = gr_matmul_tc_ex(st, g, ctx->status, ST_TIMEOUT) == 0;
    }
    for (long long h = 1; h < p.nhi && !done; ++h)
      if ((rc = gr_matmul(ctx, p.L, p.Rtab, nullptr, 1, 64, p.Mhi + (h - 1) * 4096, nullptr, 0,
                          p.Rtab + h * p.L * 64, 64)))
        return rc;
  }
  return MPC_OK;
}

// The batch from its weights (bit_tables), bit words (p.b1, p.b2), V and claim z0: the matrix S,
// the rounds that fold the 64 bits, the folded vectors and the dense rounds.
int bit_batch(mpc_ctx* ctx, TruncPlan& p, const Small& s, const u64* z0, u64 verify_id, u32 batch,
              u64* tr) {
  cudaStream_t st = ctx->st;
  const long long E = p.E;
  int rc;
  Phase* phase = new Phase(ctx, MPC_PROF_TRUNC_S);
  {  // S_{j,j'} = sum_e rho^e b1_{e,j} b2_{e,j'} (P0), with rho^e = rho^(L e_hi) rho^e_lo:
     // tensor cores for the inner sums over e_lo, then sum_{e_hi} T_hi S_hi
    launch_trunc_limb_table(st, p.Rtab, p.L, p.TL8);
    launch_trunc_bit_transpose(st, p.b1, p.Epad, p.B1T);
    launch_trunc_bit_transpose(st, p.b2, p.Epad, p.B2T);
    {
      Phase kphase(ctx, MPC_PROF_K_TRUNC_S, 4096.0 * 64 * E);
      if (launch_trunc_s_tc(st, p.B1T, p.B2T, p.Epad, p.TL8, p.L, p.nhi, p.S_hi, ctx->status,
                            ST_TIMEOUT))
        return fail(ctx, MPC_ERR_CUDA, "verify_matmul: tensor map of the limb table");
    }
    if (p.Pst) {   // S = sum_{e_hi} T_hi S_hi in one pass, then the products' reduction
      GemmTerm T;
      T.A = op(p.Thi, 64, 1);     // A[a][e_hi] = coefficient a of rho^(L e_hi)
      T.B = op(p.S_hi, 262144);   // B[e_hi][(p, b)]
      gemm_u64(st, 64, 262144, p.nhi, 1, &T, epi_store(p.Pst, 262144), 1);
      launch_fold_reduce_strided(st, p.Pst, 262144, 4096, p.S);
    } else if (p.nhi > 1) {
      // the blocks h >= 1 times rho^(L h) (matrix h - 1) in place, then the sum over the blocks
      u64* blk1 = p.S_hi + 262144;
      GrMMArgs g = grargs(ctx);
      g.R = (p.nhi - 1) * 4096;
      g.p0 = blk1;
      g.in = GrRowMap{0, 64, 0};
      g.Mmat = p.Mhi;
      g.mrows = 4096;
      g.out = blk1;
      g.om = GrRowMap{0, 64, 0};
      {
        Phase kp(ctx, MPC_PROF_K_GR_MATMUL, (double)g.R * 4096);
        if (gr_matmul_tc_ex(st, g, ctx->status, ST_TIMEOUT))
          return fail(ctx, MPC_ERR_CUDA, "S matrix: tensor maps of the blocks' products");
      }
      launch_sum_blocks(st, 262144, p.nhi, 262144, p.S_hi, p.S);
    }
  }
  delete phase;
  phase = new Phase(ctx, MPC_PROF_TRUNC_ROUNDS);
  const u64* z = z0;
  u64* zbuf[2] = {s.z[0], s.z[1]};
  int zi = 0;
  for (int k = 1; k <= p.kd; ++k) {   // rounds folding the 64 bits of each output
    u64* sums = cur_sums(s);
    launch_weighted_sums(st, p.V, p.W, p.S, 64, k, 1, sums);
    round_tail(ctx, verify_id, batch, k, z, zbuf[zi], s, sums, 64, tr, p.V, p.W, 64);
    z = zbuf[zi];
    zi ^= 1;
  }
  delete phase;
  phase = new Phase(ctx, MPC_PROF_TRUNC_MATERIALIZE);
  // materialise the folded vectors: x.[r]_1 at P0 and P1, y.[r]_2 at P0 and P2
  Vec& tx = p.dt.x[0];
  Vec& ty = p.dt.y[0];
  if (ctx->gemm_path == MPC_GEMM_LIMB_TC && p.kd == 6) {
    // one folded element per output e: -sum_j V_j b_{e,j} as a product of the bit matrix with
    // -V on the tensor cores, then (x only) the GR product with r^(2e), for each party's copy
    u64* nV = s.MM;
    u64* nW = s.MM + 4096;
    launch_neg_copy(st, p.V, 4096, nV);
    launch_neg_copy(st, p.W, 4096, nW);
    const u64* bits[4] = {p.b1, p.b1, p.b2, p.b2};
    const u64* mats[4] = {nV, nV, nW, nW};
    u64* outs[4] = {tx.c[0], tx.c[3], ty.c[1], ty.c[5]};
    auto grmm = [&](const GrMMArgs& g, double work) {
      Phase kp(ctx, MPC_PROF_K_GR_MATMUL, work);
      return gr_matmul_tc_ex(st, g, ctx->status, ST_TIMEOUT);
    };
    if (p.Lm) {
      // x_e = r^(2 Lm e_hi) (sum_j b_{e,j} r^(2 e_lo) (-V_j)): the per-row factor r^(2e) split
      // into two grouped GR matrix products on the tensor cores.
      const long long Lm = p.Lm, nhm = p.nhm, nB = (E + Lm - 1) / Lm;
      launch_gr_mulmat_batch(st, 64, nV, 64, p.Vm);
      if (p.compact) {   // r^(2 Lm e_hi) = T_hi[e / L] r^(2 (e mod L)), e = e_hi Lm
        u64* ra = p.Prow;
        u64* rb = p.Prow + nB * 64;
        u64* rr = p.Prow + 2 * nB * 64;
        launch_gather_rows_affine(st, nB, p.Thi, Lm, p.L, 0, ra);
        launch_gather_rows_affine(st, nB, p.Rtab, Lm, 1, p.L, rb);
        launch_gr_mul_rows(st, nB, ra, rb, rr);
        launch_gr_mulmat_batch(st, nB, rr, 64, p.Bm);
      } else {
        launch_gr_mulmat_batch(st, nB, p.Rtab, Lm * 64, p.Bm);
      }
      launch_word_transpose(st, nhm, Lm, E, p.b1, p.bT);
      GrMMArgs g = grargs(ctx);
      // Tm: rows sigma = j Lm + e_lo read r^(2 e_lo) and use matrix j; written at [e_lo][j]
      g.R = 64 * Lm;
      g.p0 = p.Rtab;
      g.in = GrRowMap{Lm, 64, 0};
      g.Mmat = p.Vm;
      g.mrows = Lm;
      g.out = p.Tm;
      g.om = GrRowMap{Lm, 4096, 64};
      if (grmm(g, 64.0 * Lm * 4096)) return fail(ctx, MPC_ERR_CUDA, "verify_matmul: r^(2e) V table");
      for (int v = 0; v < 2; ++v) {
        // rows rho = e_lo nhm + e_hi (bits b_e), matrix Tm[e_lo], result at row e
        GrMMArgs ga = grargs(ctx);
        ga.R = nhm * Lm;
        ga.p0 = p.bT;
        ga.in = GrRowMap{0, 1, 0};
        ga.a_bits = 1;
        ga.Mmat = p.Tm;
        ga.mrows = nhm;
        ga.out = outs[v];
        ga.om = GrRowMap{nhm, Lm * 64, 64};
        ga.out_lim = E * 64;
        if (grmm(ga, (double)nhm * Lm * 4096 * 8.0 / 36.0))
          return fail(ctx, MPC_ERR_CUDA, "verify_matmul: folded-vector product");
        // in place: rows e, matrix M(r^(2 Lm e_hi)) for e_hi = e / Lm
        GrMMArgs gb = grargs(ctx);
        gb.R = E;
        gb.p0 = outs[v];
        gb.in = GrRowMap{0, 64, 0};
        gb.Mmat = p.Bm;
        gb.mrows = Lm;
        gb.out = outs[v];
        gb.om = GrRowMap{0, 64, 0};
        if (grmm(gb, (double)E * 4096))
          return fail(ctx, MPC_ERR_CUDA, "verify_matmul: r^(2e) factor");
      }
    }
    for (int v = p.Lm ? 2 : 0; v < 4; ++v) {
      GrMMArgs g = grargs(ctx);
      g.R = E;
      g.p0 = bits[v];
      g.in = GrRowMap{0, 1, 0};
      g.a_bits = 1;
      g.Mmat = mats[v];
      g.out = outs[v];
      g.om = GrRowMap{0, 64, 0};
      // A has digit plane 0 only: 8 of the 36 digit-pair products (work in 36-pair units)
      if (grmm(g, (double)E * 4096 * 8.0 / 36.0))
        return fail(ctx, MPC_ERR_CUDA, "verify_matmul: folded-vector product");
      if (v < 2) {
        Phase kp(ctx, MPC_PROF_K_GR_MUL_ROWS, (double)E * 4096);
        launch_gr_mul_rows(st, E, outs[v], p.Rtab, outs[v]);
      }
    }
  } else {
    launch_trunc_materialize(st, E, p.b1, p.V, p.Rtab, p.kd, tx.c[0]);
    launch_trunc_materialize(st, E, p.b1, p.V, p.Rtab, p.kd, tx.c[3]);
    launch_trunc_materialize(st, E, p.b2, p.W, nullptr, p.kd, ty.c[1]);
    launch_trunc_materialize(st, E, p.b2, p.W, nullptr, p.kd, ty.c[5]);
  }
  delete phase;
  if ((rc = cuda_check(ctx, "trunc batch"))) return rc;
  phase = new Phase(ctx, MPC_PROF_TRUNC_TAIL);
  // the claim entering the dense rounds must not alias their round scratch
  CK(cudaMemcpyAsync(s.zinit, z, 384 * 8, cudaMemcpyDeviceToDevice, st));
  p.dt.cur = 0;
  rc = run_dense(ctx, verify_id, batch, p.dt, p.Dt, s.zinit, p.kd + 1, p.R1, s, tr);
  delete phase;
  return rc;
}

// One chunk of batch 1 of Pi_BIVerify (Fig. PBDP): the 2 E inner products of the truncation pairs
// of outputs e0 .. e0 + E - 1 (E = p.E) of a layer of E_all outputs, with the challenge and round
// streams of batch `batch`.  pq_all: the layer's 12 rows of <p>, <q> (stride E_all).
int verify_trunc_chunk(mpc_ctx* ctx, TruncPlan& p, const Small& s, void* tcs, const u64* pq_all,
                       long long E_all, long long e0, int trunc_bits, u64 verify_id, u32 batch,
                       u64 matmul_call_id, u64* tr, const u64* row_keys, long long N) {
  cudaStream_t st = ctx->st;
  Phase* phase = new Phase(ctx, MPC_PROF_TRUNC_SETUP);
  const u64 mobj = make_obj(matmul_call_id, 0, 0);
  const long long E = p.E;
  int rc;
  if (p.pqc)   // this chunk's outputs of the 12 rows of <p>, <q>, gathered to a stride of E
    CK(cudaMemcpy2DAsync(p.pqc, (size_t)E * 8, pq_all + e0, (size_t)E_all * 8, (size_t)E * 8, 12,
                         cudaMemcpyDeviceToDevice, st));
  const u64* pq = p.pqc ? p.pqc : pq_all;
  if ((rc = sums_begin(ctx, s))) return rc;
  reveal(ctx, P_VER_R, make_obj(verify_id, batch, 0), s, s.r);
  launch_trunc_u(st, s.r, trunc_bits, p.V);                         // V_j = u_j
  if (row_keys) {
    launch_prf_words_keyed(st, E, ctx->k01, make_tag(P_TRUNC_BITS, C_TB1), row_keys, N, p.b1, e0);
    launch_prf_words_keyed(st, E, ctx->k02, make_tag(P_TRUNC_BITS, C_TB2), row_keys, N, p.b2, e0);
  } else {
    launch_prf_words(st, E, ctx->k01, make_tag(P_TRUNC_BITS, C_TB1), mobj, p.b1, e0);
    launch_prf_words(st, E, ctx->k02, make_tag(P_TRUNC_BITS, C_TB2), mobj, p.b2, e0);
  }
  launch_gr_mul1(st, s.r, s.r, s.aux + 64);                          // r^2
  if ((rc = bit_tables(ctx, p, s, s.aux + 64))) return rc;
  CK(cudaMemsetAsync(p.Zpq, 0, 12 * 64 * 8, st));
  // sum_e r^(2e) p_c[e], sum_e r^(2e) q_c[e]: (12 x E) . (E x 64)
  if (p.compact) {
    // Zhi[c nhi + h] = sum_{e_lo} pq_c[h L + e_lo] r^(2 e_lo) (E = nhi L: one strided view)
    GemmTerm T;
    T.A = op(pq, p.L);
    T.B = op(p.Rtab, 64);
    if ((rc = dense_gemm(ctx, 12 * p.nhi, 64, p.L, T, epi_store(p.Zhi, 64), tcs))) return rc;
    launch_gather_rows_affine(st, 12 * p.nhi, p.Thi, 1, 1, p.nhi, p.Zrep);   // T_hi[h]
    launch_gr_mul_rows(st, 12 * p.nhi, p.Zhi, p.Zrep, p.Zprod);
    launch_block_rowsum(st, 12, p.nhi, p.Zprod, p.Zpq);
  } else {
    launch_scalar_gr_sum(st, E, pq, E, 12, p.Rtab, p.Zpq);
  }
  u64* z0 = p.zt + 384;
  launch_gr_axpy(st, 6, s.r, p.Zpq, p.Zpq + 384, z0);   // z_c = sum r^(2e) p_c + r sum r^(2e) q_c
  delete phase;
  return bit_batch(ctx, p, s, z0, verify_id, batch, tr);
}

// The messages of the truncation pairs' two inner products (Fig. trunc), as their receivers read them.
struct PairMsgs {
  const u64 *gp2, *gq2;             // P2: [Gamma]_2
  const u64 *mp1, *mq1, *mp2, *mq2; // P1: from P2; P2: from P1
};
int deliver_pairs(mpc_ctx* ctx, const u64* gp2, const u64* gq2, const u64* mp1, const u64* mq1, long long n,
                  const FaultCopies& fc, PairMsgs& m) {
  const int ph = MPC_PHASE_OFFLINE, pr = MPC_PROTO_TRUNC;
  int rc;
  if ((rc = deliver(ctx, ph, pr, gp2, m.gp2, n, MPC_SITE_GAMMA2, fc.g2))) return rc;
  if ((rc = deliver(ctx, ph, pr, mp1, m.mp2, n, MPC_SITE_MZ1, fc.mz1))) return rc;
  if ((rc = deliver(ctx, ph, pr, m.gp2, m.mp1, n, MPC_SITE_MZ2, fc.mz2))) return rc;
  if ((rc = deliver(ctx, ph, pr, gq2, m.gq2, n, MPC_SITE_GAMMA2, fc.g2))) return rc;
  if ((rc = deliver(ctx, ph, pr, mq1, m.mq2, n, MPC_SITE_MZ1, fc.mz1))) return rc;
  return deliver(ctx, ph, pr, m.gq2, m.mq1, n, MPC_SITE_MZ2, fc.mz2);
}

// workspace of a standalone truncation (mpc_trunc)
struct TruncCallPlan {
  u64* rx;   // 6n: the pairs' r_x shares in the mask components
  u64 *gp2, *gq2, *mp1, *mq1;      // pair messages
  u64 *d1, *d2, *d1p0, *d2p0;      // mask switch
  FaultCopies fc;
  u64* d1x;                        // d1 as a fault corrupts it
  u32* hs[4];
  u32* dg;   // 4 x 8 digest words
};

TruncCallPlan plan_trunc_call(Arena& a, long long n) {
  TruncCallPlan p;
  p.rx = a.take<u64>(6 * n);
  for (u64** b : {&p.gp2, &p.gq2, &p.mp1, &p.mq1, &p.d1, &p.d2, &p.d1p0, &p.d2p0, &p.d1x})
    *b = a.take<u64>(n);
  p.fc = plan_copies(a, n);
  for (int i = 0; i < 4; ++i) p.hs[i] = a.take<u32>((long long)hash_scratch_words(n));
  p.dg = a.take<u32>(32);
  return p;
}

// Every chunk of a truncation batch (batches 1, 2, ... of verify_id); trace: chunk after chunk.
int verify_trunc_batch(mpc_ctx* ctx, TruncBatch& b, const Small& s, void* tcs, const u64* pq,
                       int trunc_bits, u64 verify_id, u64 call_id, u64* tr, const u64* row_keys,
                       long long N) {
  for (long long i = 0; i < b.nchunks; ++i) {
    TruncPlan& tp = b.tp[i == b.nchunks - 1 ? 1 : 0];
    const int rc = verify_trunc_chunk(ctx, tp, s, tcs, pq, b.E, i * b.C, trunc_bits, verify_id,
                                      (u32)(1 + i), call_id, tr, row_keys, N);
    if (rc) return rc;
    if (tr) tr += (long long)(tp.R1 + 1) * TRACE_ROUND;
  }
  return MPC_OK;
}

}  // namespace

// =================================================================================================
// C-ABI
// =================================================================================================
namespace {
void destroy_side(mpc_ctx* ctx) {
  for (int i = 0; i < NSIDE; ++i) {
    if (ctx->side[i]) cudaStreamDestroy(ctx->side[i]);
    if (ctx->join_ev[i]) cudaEventDestroy(ctx->join_ev[i]);
  }
  if (ctx->fork_ev) cudaEventDestroy(ctx->fork_ev);
}
}  // namespace

extern "C" {

int mpc_create(const mpc_config* cfg, mpc_ctx** out) {
  if (!out) return MPC_ERR_ARG;
  *out = nullptr;
  if (!cfg) return MPC_ERR_ARG;
  if (cfg->reduce_mode != MPC_REDUCE_POINT_X && cfg->reduce_mode != MPC_REDUCE_POINT_2)
    return MPC_ERR_ARG;
  if (cfg->gemm_path != MPC_GEMM_U64 && cfg->gemm_path != MPC_GEMM_LIMB_TC) return MPC_ERR_ARG;
  mpc_ctx* ctx = new mpc_ctx();
  ctx->device = cfg->device;
  ctx->reduce_mode = cfg->reduce_mode;
  ctx->gemm_path = cfg->gemm_path;
  auto bail = [&](const char* what, cudaError_t e) {
    std::fprintf(stderr, "mpc_create: %s: %s\n", what, cudaGetErrorString(e));
    if (ctx->cst) cudaFree(ctx->cst);
    if (ctx->own_stream && ctx->st) cudaStreamDestroy(ctx->st);
    destroy_side(ctx);
    delete ctx;
    return MPC_ERR_CUDA;
  };
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e != cudaSuccess) return bail("cudaSetDevice", e);
  if (cfg->stream) {
    ctx->st = (cudaStream_t)cfg->stream;
  } else {
    e = cudaStreamCreateWithFlags(&ctx->st, cudaStreamNonBlocking);
    if (e != cudaSuccess) return bail("cudaStreamCreate", e);
    ctx->own_stream = true;
  }
  e = cudaEventCreateWithFlags(&ctx->fork_ev, cudaEventDisableTiming);
  for (int i = 0; i < NSIDE && e == cudaSuccess; ++i) {
    e = cudaStreamCreateWithFlags(&ctx->side[i], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->join_ev[i], cudaEventDisableTiming);
  }
  if (e != cudaSuccess) return bail("side streams", e);
  // constants block + status word + key staging
  e = cudaMalloc(&ctx->cst, CST_WORDS * 8 + 256 + 256);
  if (e != cudaSuccess) return bail("cudaMalloc", e);
  ctx->status = reinterpret_cast<u32*>(reinterpret_cast<char*>(ctx->cst) + CST_WORDS * 8);
  u32* keys_dev = reinterpret_cast<u32*>(reinterpret_cast<char*>(ctx->cst) + CST_WORDS * 8 + 256);
  Key master;
  std::memcpy(master.k, cfg->seed, 32);
  launch_dep(k_derive_keys, 1, 32, 0, ctx->st, master, keys_dev);
  launch_gr_inverse(ctx->st, ctx->cst + CST_INV);
  e = cudaMemsetAsync(ctx->status, 0, sizeof(u32), ctx->st);
  if (e != cudaSuccess) return bail("cudaMemset", e);
  u32 kh[24];
  e = cudaMemcpyAsync(kh, keys_dev, sizeof(kh), cudaMemcpyDeviceToHost, ctx->st);
  if (e != cudaSuccess) return bail("key copy", e);
  e = cudaStreamSynchronize(ctx->st);
  if (e != cudaSuccess) return bail("init", e);
  std::memcpy(ctx->k01.k, kh, 32);
  std::memcpy(ctx->k02.k, kh + 8, 32);
  std::memcpy(ctx->k12.k, kh + 16, 32);
  *out = ctx;
  return MPC_OK;
}

void mpc_destroy(mpc_ctx* ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  if (ctx->st) cudaStreamSynchronize(ctx->st);
  if (ctx->copy_st) {
    cudaStreamSynchronize(ctx->copy_st);
    cudaStreamDestroy(ctx->copy_st);
  }
  for (cudaEvent_t e : ctx->copy_ev)
    if (e) cudaEventDestroy(e);
  if (ctx->order_ev) cudaEventDestroy(ctx->order_ev);
  for (cudaEvent_t e : ctx->pool) cudaEventDestroy(e);
  if (ctx->cst) cudaFree(ctx->cst);
  if (ctx->own_stream && ctx->st) cudaStreamDestroy(ctx->st);
  destroy_side(ctx);
  delete ctx;
}

const char* mpc_last_error(const mpc_ctx* ctx) { return ctx ? ctx->err.c_str() : "null context"; }

int mpc_h2d_async(mpc_ctx* ctx, void* dst, const void* src, size_t bytes, int slot) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (!dst || !src || bytes == 0 || slot < 0 || slot >= MPC_H2D_SLOTS)
    return fail(ctx, MPC_ERR_ARG, "h2d_async: bad argument");
  if (!ctx->copy_st) CK(cudaStreamCreateWithFlags(&ctx->copy_st, cudaStreamNonBlocking));
  if (!ctx->copy_ev[slot]) CK(cudaEventCreateWithFlags(&ctx->copy_ev[slot], cudaEventDisableTiming));
  if (!ctx->order_ev) CK(cudaEventCreateWithFlags(&ctx->order_ev, cudaEventDisableTiming));
  CK(cudaEventRecord(ctx->order_ev, ctx->st));   // after the work that may still read dst
  CK(cudaStreamWaitEvent(ctx->copy_st, ctx->order_ev, 0));
  CK(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, ctx->copy_st));
  CK(cudaEventRecord(ctx->copy_ev[slot], ctx->copy_st));
  return MPC_OK;
}

int mpc_d2h_async(mpc_ctx* ctx, void* dst, const void* src, size_t bytes, int slot) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (!dst || !src || bytes == 0 || slot < 0 || slot >= MPC_H2D_SLOTS)
    return fail(ctx, MPC_ERR_ARG, "d2h_async: bad argument");
  if (!ctx->copy_st) CK(cudaStreamCreateWithFlags(&ctx->copy_st, cudaStreamNonBlocking));
  if (!ctx->copy_ev[slot]) CK(cudaEventCreateWithFlags(&ctx->copy_ev[slot], cudaEventDisableTiming));
  if (!ctx->order_ev) CK(cudaEventCreateWithFlags(&ctx->order_ev, cudaEventDisableTiming));
  CK(cudaEventRecord(ctx->order_ev, ctx->st));   // after the work that writes src
  CK(cudaStreamWaitEvent(ctx->copy_st, ctx->order_ev, 0));
  CK(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, ctx->copy_st));
  CK(cudaEventRecord(ctx->copy_ev[slot], ctx->copy_st));
  return MPC_OK;
}

int mpc_h2d_wait(mpc_ctx* ctx, int slot) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (slot < 0 || slot >= MPC_H2D_SLOTS) return fail(ctx, MPC_ERR_ARG, "h2d_wait: bad slot");
  if (!ctx->copy_ev[slot]) return MPC_OK;   // nothing was issued under this slot
  CK(cudaStreamWaitEvent(ctx->st, ctx->copy_ev[slot], 0));
  return MPC_OK;
}

int mpc_set_stream(mpc_ctx* ctx, void* stream) {
  if (!ctx || !stream) return MPC_ERR_ARG;
  if (ctx->own_stream && ctx->st) {
    cudaStreamSynchronize(ctx->st);
    cudaStreamDestroy(ctx->st);
    ctx->own_stream = false;
  }
  ctx->st = (cudaStream_t)stream;
  return MPC_OK;
}

int mpc_sync(mpc_ctx* ctx) {
  if (!ctx) return MPC_ERR_ARG;
  CK(cudaStreamSynchronize(ctx->st));
  u32 stv = 0;
  return read_status(ctx, &stv);
}

int mpc_status(const mpc_ctx* ctx) {
  if (!ctx) return MPC_ERR_ARG;
  return ctx->aborted ? MPC_ERR_ABORT : MPC_OK;
}

int mpc_set_tuning(mpc_ctx* ctx, const mpc_tuning* tune) {
  if (!ctx) return MPC_ERR_ARG;
  mpc_tuning t = default_tuning();
  if (tune) {
    if (tune->trunc_block < 0 || tune->trunc_chunk < 0 || tune->row_split < 0 ||
        tune->tc_combine_min < 0 || tune->gemm_split_min < 0 || tune->gram_split < 0 ||
        tune->fold_batch_max < 0 || tune->trunc_block % 128 || tune->row_split % 128 ||
        tune->trunc_block > 65536 || tune->gram_split > 65535 || tune->gr_producers < 0 ||
        tune->gr_producers > 3 || (tune->gr_drain_warps != 0 && tune->gr_drain_warps != 8 &&
                                   tune->gr_drain_warps != 16))
      return fail(ctx, MPC_ERR_ARG, "set_tuning: value out of range");
    if (tune->trunc_block) t.trunc_block = tune->trunc_block;
    if (tune->trunc_chunk) t.trunc_chunk = tune->trunc_chunk;
    t.row_split = tune->row_split;
    if (tune->tc_combine_min) t.tc_combine_min = tune->tc_combine_min;
    if (tune->gemm_split_min) t.gemm_split_min = tune->gemm_split_min;
    if (tune->gram_split) t.gram_split = tune->gram_split;
    if (tune->fold_batch_max) t.fold_batch_max = tune->fold_batch_max;
    if (tune->gr_producers) t.gr_producers = tune->gr_producers;
    if (tune->gr_drain_warps) t.gr_drain_warps = tune->gr_drain_warps;
  }
  ctx->tune = t;
  ctx->combine_set = tune && tune->tc_combine_min;
  return MPC_OK;
}

int mpc_get_tuning(const mpc_ctx* ctx, mpc_tuning* out) {
  if (!ctx || !out) return MPC_ERR_ARG;
  *out = ctx->tune;
  if (!ctx->combine_set) out->tc_combine_min = COMBINE_REPORTED;
  return MPC_OK;
}

int64_t mpc_trace_words(const mpc_ctx* ctx, int op, int64_t a, int64_t b, int64_t c,
                        int trunc_bits, int R_main, int R_trunc) {
  switch (op) {
    case MPC_OP_VERIFY_MULT:
    case MPC_OP_VERIFY_MULT_CALLS:
      if (a <= 0) return -1;
      return (int64_t)((R_main < 0 ? default_R(a) : R_main) + 1) * TRACE_ROUND;
    case MPC_OP_VERIFY_MATMUL: {
      if (a <= 0 || b <= 0 || c <= 0 || trunc_bits > 63) return -1;
      int64_t w = (int64_t)((R_main < 0 ? default_R(c) : R_main) + 1) * TRACE_ROUND;
      if (trunc_bits >= 0) {
        const mpc_tuning tu = ctx ? ctx->tune : default_tuning();
        long long n = 0, C = 0;
        trunc_chunks(a * b, tu, &n, &C);
        if (n > MAX_TRUNC_CHUNKS) return -1;
        for (long long i = 0; i < n; ++i) {
          const long long Ei = i == n - 1 ? a * b - (n - 1) * C : C;
          w += (int64_t)((R_trunc < 0 ? default_R(64 * Ei) : R_trunc) + 1) * TRACE_ROUND;
        }
      }
      return w;
    }
    case MPC_OP_VERIFY_TRUNC: {
      if (a <= 0) return -1;
      const mpc_tuning tu = ctx ? ctx->tune : default_tuning();
      long long n = 0, C = 0;
      trunc_chunks(a, tu, &n, &C);
      if (n > MAX_TRUNC_CHUNKS) return -1;
      int64_t w = 0;
      for (long long i = 0; i < n; ++i) {
        const long long Ei = i == n - 1 ? a - (n - 1) * C : C;
        w += (int64_t)((R_trunc < 0 ? default_R(64 * Ei) : R_trunc) + 1) * TRACE_ROUND;
      }
      return w;
    }
    default:
      return -1;
  }
}

namespace {
// workspace of a non-linear layer
void nl_plan_take(Arena& a, int nst, const long long np[2], bool tc, const mpc_tuning& tu);
}

int64_t mpc_workspace_size(const mpc_ctx* ctx, int op, int64_t a, int64_t b, int64_t c,
                           int trunc_bits, int R_main, int R_trunc) {
  (void)ctx;
  Arena ar{nullptr, 0, 0, true};
  switch (op) {
    case MPC_OP_SHARE:
      if (a < 0) return -1;
      ar.take<u64>(a);
      ar.take<u64>(a);
      break;
    case MPC_OP_MULT:
      if (a < 0) return -1;
      for (int i = 0; i < 6; ++i) ar.take<u64>(a);
      break;
    case MPC_OP_MATMUL:
      if (a <= 0 || b <= 0 || c <= 0) return -1;
      plan_matmul(ar, a, b, c, trunc_bits >= 0, ctx && ctx->gemm_path == MPC_GEMM_LIMB_TC);
      break;
    case MPC_OP_VERIFY_MULT:
      if (a <= 0) return -1;
      plan_vmult(ar, a, R_main, ctx && ctx->gemm_path == MPC_GEMM_LIMB_TC);
      break;
    case MPC_OP_VERIFY_MULT_CALLS:
      if (a <= 0) return -1;
      plan_vmult_calls(ar, a, R_main, ctx && ctx->gemm_path == MPC_GEMM_LIMB_TC);
      break;
    case MPC_OP_VERIFY_MATMUL: {
      if (a <= 0 || b <= 0 || c <= 0 || trunc_bits > 63) return -1;
      VMatPlan vp;
      if (!plan_vmat(ar, a, b, c, trunc_bits, R_main, R_trunc,
                     ctx && ctx->gemm_path == MPC_GEMM_LIMB_TC, ctx ? ctx->tune : default_tuning(),
                     vp))
        return -1;
      break;
    }
    case MPC_OP_RELU: {
      if (a <= 0) return -1;
      const long long np[2] = {64 * ((a + 63) / 64), 0};
      nl_plan_take(ar, 1, np, ctx && ctx->gemm_path == MPC_GEMM_LIMB_TC,
                   ctx ? ctx->tune : default_tuning());
      break;
    }
    case MPC_OP_MAXPOOL2: {
      if (a <= 0 || b <= 0 || c <= 0 || (b & 1) || (c & 1)) return -1;
      const long long nw = a * (b / 2) * (c / 2);
      const long long np[2] = {64 * ((2 * nw + 63) / 64), 64 * ((nw + 63) / 64)};
      nl_plan_take(ar, 2, np, ctx && ctx->gemm_path == MPC_GEMM_LIMB_TC,
                   ctx ? ctx->tune : default_tuning());
      break;
    }
    case MPC_OP_RECONSTRUCT:
      if (a < 0) return -1;
      plan_rec(ar, a, true);
      break;
    case MPC_OP_SHARE_FIXED:
      if (a < 0) return -1;
      ar.take<u64>(a);
      ar.take<double>(a);
      ar.take<u64>(a);
      ar.take<u64>(a);
      break;
    case MPC_OP_RECONSTRUCT_FIXED:
      if (a < 0) return -1;
      ar.take<u64>(a);
      ar.take<double>(a);
      plan_rec(ar, a, false);
      break;
    case MPC_OP_TRUNC:
      if (a <= 0) return -1;
      plan_trunc_call(ar, a);
      break;
    case MPC_OP_VERIFY_TRUNC: {
      if (a <= 0) return -1;
      VTruncPlan vp;
      if (!plan_vtrunc(ar, a, R_trunc, ctx && ctx->gemm_path == MPC_GEMM_LIMB_TC,
                       ctx ? ctx->tune : default_tuning(), vp))
        return -1;
      break;
    }
    default:
      return -1;
  }
  return (int64_t)ar.off;
}

int mpc_share_input(mpc_ctx* ctx, uint64_t call_id, const uint64_t* x, int x_on_host, int64_t n,
                    uint64_t* xs, void* workspace, size_t workspace_bytes) {
  return mpc_share_input_from(ctx, call_id, 0, x, x_on_host, n, xs, workspace, workspace_bytes);
}

int mpc_share_input_from(mpc_ctx* ctx, uint64_t call_id, int owner, const uint64_t* x,
                         int x_on_host, int64_t n, uint64_t* xs, void* workspace,
                         size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n < 0) return fail(ctx, MPC_ERR_SHAPE, "n < 0");
  if (owner < 0 || owner > 2) return fail(ctx, MPC_ERR_ARG, "share_input: owner must be 0, 1 or 2");
  if (n == 0) return MPC_OK;
  if (!x || !xs || !id_ok(call_id)) return fail(ctx, MPC_ERR_ARG, "share_input: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  u64* stage = ar.take<u64>(n);
  u64* mout = ar.take<u64>(n);
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "share_input: workspace too small");
  Phase phase(ctx, MPC_PROF_SHARE);
  const u64* xd = (const u64*)x;
  if (x_on_host) {
    CK(cudaMemcpyAsync(stage, x, (size_t)n * 8, cudaMemcpyHostToDevice, ctx->st));
    xd = stage;
  }
  launch_share_input(ctx->st, xd, n, ctx->k01, ctx->k02, make_obj(call_id, 0, 0), (u64*)xs, mout);
  // m_x: components 2 (P1) and 4 (P2).  The owner P0 sends it to both; P1 or P2 keeps its own
  // copy and sends one message to the other.  A message arriving at P1 is fault site MX_COPY_P1.
  u64* m1 = (u64*)xs + 2 * n;
  u64* m2 = (u64*)xs + 4 * n;
  if (owner == 1)
    CK(cudaMemcpyAsync(m1, mout, (size_t)n * 8, cudaMemcpyDeviceToDevice, ctx->st));
  else if ((rc = deliver_copy(ctx, MPC_PHASE_ONLINE, MPC_PROTO_SHARE, mout, m1, n,
                              take_fault(ctx, MPC_SITE_MX_COPY_P1, n))))
    return rc;
  if (owner == 2)
    CK(cudaMemcpyAsync(m2, mout, (size_t)n * 8, cudaMemcpyDeviceToDevice, ctx->st));
  else if ((rc = deliver_copy(ctx, MPC_PHASE_ONLINE, MPC_PROTO_SHARE, mout, m2, n, MsgFault{})))
    return rc;
  return cuda_check(ctx, "share_input");
}

int mpc_mult(mpc_ctx* ctx, uint64_t call_id, const uint64_t* xs, const uint64_t* ys, int64_t n,
             uint64_t* zs, void* workspace, size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n <= 0) return fail(ctx, MPC_ERR_SHAPE, "mult: n <= 0");
  if (!xs || !ys || !zs || !id_ok(call_id)) return fail(ctx, MPC_ERR_ARG, "mult: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  u64* g2 = ar.take<u64>(n);
  u64* p1 = ar.take<u64>(n);
  u64* p2 = ar.take<u64>(n);
  const FaultCopies fc = plan_copies(ar, n);
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "mult: workspace too small");
  Phase phase(ctx, MPC_PROF_MULT);
  const u64 obj = make_obj(call_id, 0, 0);
  const u64 *g2_at_p2, *p1_at_p2, *p2_at_p1;
  launch_mult_offline(ctx->st, xs, ys, n, ctx->k01, ctx->k02, obj, zs, g2);
  const int off = MPC_PHASE_OFFLINE, on = MPC_PHASE_ONLINE, pr = MPC_PROTO_MULT;
  if ((rc = deliver(ctx, off, pr, g2, g2_at_p2, n, MPC_SITE_GAMMA2, fc.g2))) return rc;
  launch_mult_online(ctx->st, xs, ys, n, ctx->k01, obj, g2_at_p2, p1, p2);
  if ((rc = deliver(ctx, on, pr, p1, p1_at_p2, n, MPC_SITE_MZ1, fc.mz1))) return rc;
  if ((rc = deliver(ctx, on, pr, p2, p2_at_p1, n, MPC_SITE_MZ2, fc.mz2))) return rc;
  launch_exchange_finish(ctx->st, n, p1, p2_at_p1, p2, p1_at_p2, zs, -1, nullptr);
  ctx->pending.insert((call_id << 1) | 0);
  return cuda_check(ctx, "mult");
}

int mpc_matmul(mpc_ctx* ctx, uint64_t call_id, const uint64_t* xs, const uint64_t* ws_,
               int64_t M, int64_t N, int64_t K, int trunc_bits, uint64_t* zpre, uint64_t* zout,
               uint64_t* pq, void* workspace, size_t workspace_bytes) {
  return mpc_matmul_keyed(ctx, call_id, xs, ws_, M, N, K, trunc_bits, nullptr, zpre, zout, pq,
                          workspace, workspace_bytes);
}

int mpc_matmul_keyed(mpc_ctx* ctx, uint64_t call_id, const uint64_t* xs, const uint64_t* ws_,
                     int64_t M, int64_t N, int64_t K, int trunc_bits, const uint64_t* row_keys,
                     uint64_t* zpre, uint64_t* zout, uint64_t* pq, void* workspace,
                     size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (M <= 0 || N <= 0 || K <= 0) return fail(ctx, MPC_ERR_SHAPE, "matmul: bad shape");
  if (trunc_bits > 63) return fail(ctx, MPC_ERR_ARG, "matmul: trunc_bits > 63");
  const bool trunc = trunc_bits >= 0;
  if (!xs || !ws_ || !zpre || !id_ok(call_id) || (trunc && (!zout || !pq || zout == zpre)))
    return fail(ctx, MPC_ERR_ARG, "matmul: bad argument");
  const long long E = M * N;
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  const bool tc = ctx->gemm_path == MPC_GEMM_LIMB_TC;
  MatmulPlan p = plan_matmul(ar, M, N, K, trunc, tc);
  // the parties' local products: CUDA-core u64 GEMM or the limb-split tensor-core GEMM
  auto party_gemm = [&](int nterms, const GemmTerm* T, const Epi& e) -> int {
    if (!tc) {
      gemm_u64(ctx->st, M, N, K, nterms, T, e, 1);
      return MPC_OK;
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ctx->prof) {
      e0 = prof_event(ctx);
      e1 = prof_event(ctx);
      ctx->recs.push_back({MPC_PROF_K_LIMB_GEMM, e0, e1, (double)M * N * K * nterms});
    }
    const int r = limb_gemm_tc(ctx->st, M, N, K, nterms, T, e, p.tc, ctx->status, ST_TIMEOUT, e0, e1,
                               ctx->tune.gemm_split_min);
    return r ? fail(ctx, MPC_ERR_CUDA, "matmul: tensor-core GEMM setup failed") : MPC_OK;
  };
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "matmul: workspace too small");
  cudaStream_t st = ctx->st;
  const u64 obj = make_obj(call_id, 0, 0);
  const u64 M1 = ~0ull;
  if (trunc) {   // Pi_Trunc preprocessing first: it assigns the product wire's mask
    Phase phase(ctx, MPC_PROF_TRUNC_PAIRS);
    launch_trunc_p0(st, E, ctx->k01, ctx->k02, obj, trunc_bits, zpre, zout, pq, p.gp2, p.gq2,
                    p.mp1, p.mq1, (const u64*)row_keys, N);
    PairMsgs m;
    if ((rc = deliver_pairs(ctx, p.gp2, p.gq2, p.mp1, p.mq1, E, p.fc, m))) return rc;
    launch_trunc_finish(st, E, ctx->k01, ctx->k02, obj, trunc_bits, m.mp1, m.mq1, m.mp2, m.mq2, m.gp2,
                        m.gq2, p.mp1, p.mq1, zpre, zout, pq, (const u64*)row_keys, N);
  } else {
    launch_fill_masks(st, E, ctx->k01, ctx->k02, P_INNER, obj, zpre);
  }
  const u64* X = xs;
  const u64* W = ws_;
  const long long MK = M * K, KN = K * N;
  {  // P0, offline: Gamma = (R_X1 + R_X2)(R_W1 + R_W2) + r_Z; message [Gamma]_2 = Gamma - [Gamma]_1
    Phase phase(ctx, MPC_PROF_GEMM);
    GemmTerm T;
    T.A = op(X, K, 0, X + MK, 1);
    T.B = op(W, N, 0, W + KN, 1);
    Epi e = epi_store(p.g2, N);
    e.add0 = zpre;
    e.add1 = zpre + E;
    e.prf_sign = M1;
    e.key = ctx->k01;
    e.tag = make_tag(P_INNER, C_G1);
    e.obj = obj;
    if ((rc = party_gemm(1, &T, e))) return rc;
  }
  const u64 *g2_at_p2, *mz1_at_p2, *mz2_at_p1;
  if ((rc = deliver(ctx, MPC_PHASE_OFFLINE, MPC_PROTO_INNER, p.g2, g2_at_p2, E, MPC_SITE_GAMMA2, p.fc.g2)))
    return rc;
  {  // P1, online: [m_Z]_1 = -(M_X [R_W]_1 + [R_X]_1 M_W) + [Gamma]_1
    Phase phase(ctx, MPC_PROF_GEMM);
    GemmTerm T[2];
    T[0].A = op(X + 2 * MK, K);
    T[0].B = op(W + 3 * KN, N);
    T[1].A = op(X + 3 * MK, K);
    T[1].B = op(W + 2 * KN, N);
    Epi e = epi_store(p.mz1, N);
    e.acc_sign = M1;
    e.prf_sign = 1;
    e.key = ctx->k01;
    e.tag = make_tag(P_INNER, C_G1);
    e.obj = obj;
    if ((rc = party_gemm(2, T, e))) return rc;
  }
  {  // P2, online: [m_Z]_2 = M_X (M_W - [R_W]_2) - [R_X]_2 M_W + [Gamma]_2
    Phase phase(ctx, MPC_PROF_GEMM);
    GemmTerm T[2];
    T[0].A = op(X + 4 * MK, K);
    T[0].B = op(W + 4 * KN, N, 0, W + 5 * KN, M1);
    T[1].A = op(X + 5 * MK, K, 0, nullptr, 1, M1);
    T[1].B = op(W + 4 * KN, N);
    Epi e = epi_store(p.mz2, N);
    e.add0 = g2_at_p2;
    if ((rc = party_gemm(2, T, e))) return rc;
  }
  {
    Phase phase(ctx, MPC_PROF_EXCHANGE);
    if ((rc = deliver(ctx, MPC_PHASE_ONLINE, MPC_PROTO_INNER, p.mz1, mz1_at_p2, E, MPC_SITE_MZ1, p.fc.mz1)))
      return rc;
    if ((rc = deliver(ctx, MPC_PHASE_ONLINE, MPC_PROTO_INNER, p.mz2, mz2_at_p1, E, MPC_SITE_MZ2, p.fc.mz2)))
      return rc;
    launch_exchange_finish(st, E, p.mz1, mz2_at_p1, p.mz2, mz1_at_p2, zpre, trunc_bits,
                           trunc ? zout : nullptr);
  }
  if (!trunc && zout && zout != zpre)
    CK(cudaMemcpyAsync(zout, zpre, (size_t)E * 48, cudaMemcpyDeviceToDevice, st));
  ctx->pending.insert((call_id << 1) | 1);
  return cuda_check(ctx, "matmul");
}

namespace {
// Pi_MultVerify (Fig. PPEV) of the n triples (xs, ys, zs) in the plan's workspace, up to the
// opened Delta; the caller reads the outcome with finish_verify.
int verify_mult_body(mpc_ctx* ctx, uint64_t verify_id, const u64* xs, const u64* ys,
                     const u64* zs, long long n, VMultPlan& p, u64* trace) {
  Phase phase(ctx, MPC_PROF_VERIFY_MULT);
  const Small& s = p.s;
  // Pi_Tran (Fig. MTP): reveal r; x'_i = r^i x_i; y lifted; z = sum r^i z_i
  int rc;
  if ((rc = sums_begin(ctx, s))) return rc;
  reveal(ctx, P_VER_R, make_obj(verify_id, 0, 0), s, s.r);
  if ((rc = blk_tables(ctx, p.b, s.r, s.aux))) return rc;
  Vec x, y;
  for (int c = 0; c < 6; ++c) {
    x.c[c] = const_cast<u64*>(xs + c * n);
    y.c[c] = const_cast<u64*>(ys + c * n);
  }
  return run_blk(ctx, verify_id, 0, p.b, x, y, zs, s, trace);
}
}  // namespace

int mpc_verify_mult(mpc_ctx* ctx, uint64_t verify_id, const uint64_t* xs, const uint64_t* ys,
                    const uint64_t* zs, int64_t n, uint64_t mult_call_id, int R,
                    void* workspace, size_t workspace_bytes, uint64_t* trace) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n <= 0) return fail(ctx, MPC_ERR_SHAPE, "verify_mult: n <= 0");
  if (!xs || !ys || !zs || !id_ok(verify_id)) return fail(ctx, MPC_ERR_ARG, "verify_mult: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  VMultPlan p = plan_vmult(ar, n, R, ctx->gemm_path == MPC_GEMM_LIMB_TC);
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "verify_mult: workspace too small");
  if ((rc = verify_mult_body(ctx, verify_id, xs, ys, zs, n, p, trace))) return rc;
  return finish_verify(ctx, (mult_call_id << 1) | 0);
}

int mpc_verify_mult_calls(mpc_ctx* ctx, uint64_t verify_id, int ncalls,
                          const uint64_t* const* xs, const uint64_t* const* ys,
                          const uint64_t* const* zs, const int64_t* n, const uint64_t* call_ids,
                          int R, void* workspace, size_t workspace_bytes, uint64_t* trace) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (ncalls <= 0 || !xs || !ys || !zs || !n || !call_ids || !id_ok(verify_id))
    return fail(ctx, MPC_ERR_ARG, "verify_mult_calls: bad argument");
  long long N = 0;
  for (int l = 0; l < ncalls; ++l) {
    if (n[l] <= 0 || n[l] > (1ll << 40)) return fail(ctx, MPC_ERR_SHAPE, "verify_mult_calls: bad n");
    if (!xs[l] || !ys[l] || !zs[l] || !id_ok(call_ids[l]))
      return fail(ctx, MPC_ERR_ARG, "verify_mult_calls: bad argument");
    // only products still awaiting verification, each once
    if (!ctx->pending.count((call_ids[l] << 1) | 0))
      return fail(ctx, MPC_ERR_ARG, "verify_mult_calls: a call id is not a pending mpc_mult call");
    for (int j = 0; j < l; ++j)
      if (call_ids[j] == call_ids[l])
        return fail(ctx, MPC_ERR_ARG, "verify_mult_calls: a call id is listed twice");
    N += n[l];
    if (N > (1ll << 40)) return fail(ctx, MPC_ERR_SHAPE, "verify_mult_calls: batch too large");
  }
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  VMultCallsPlan p = plan_vmult_calls(ar, N, R, ctx->gemm_path == MPC_GEMM_LIMB_TC);
  if (!workspace || !ar.ok())
    return fail(ctx, MPC_ERR_WORKSPACE, "verify_mult_calls: workspace too small");
  // the batch: component c of call l at c N + (n[0] + ... + n[l-1]) of each gathered sharing
  long long off = 0;
  for (int l = 0; l < ncalls; ++l) {
    const size_t bytes = (size_t)n[l] * 8;
    for (int c = 0; c < 6; ++c) {
      CK(cudaMemcpyAsync(p.x + c * N + off, xs[l] + c * n[l], bytes, cudaMemcpyDeviceToDevice, ctx->st));
      CK(cudaMemcpyAsync(p.y + c * N + off, ys[l] + c * n[l], bytes, cudaMemcpyDeviceToDevice, ctx->st));
      CK(cudaMemcpyAsync(p.z + c * N + off, zs[l] + c * n[l], bytes, cudaMemcpyDeviceToDevice, ctx->st));
    }
    off += n[l];
  }
  if ((rc = verify_mult_body(ctx, verify_id, p.x, p.y, p.z, N, p.v, trace))) return rc;
  if ((rc = finish_verify(ctx, (call_ids[0] << 1) | 0))) return rc;
  for (int l = 1; l < ncalls; ++l) ctx->pending.erase((call_ids[l] << 1) | 0);
  return MPC_OK;
}

int mpc_verify_matmul(mpc_ctx* ctx, uint64_t verify_id, const uint64_t* xs, const uint64_t* ws_,
                      const uint64_t* zpre, const uint64_t* pq, int64_t M, int64_t N, int64_t K,
                      int trunc_bits, uint64_t matmul_call_id, int R_main, int R_trunc,
                      void* workspace, size_t workspace_bytes, uint64_t* trace) {
  return mpc_verify_matmul_keyed(ctx, verify_id, xs, ws_, zpre, pq, M, N, K, trunc_bits, nullptr,
                                 matmul_call_id, R_main, R_trunc, workspace, workspace_bytes,
                                 trace);
}

int mpc_verify_matmul_keyed(mpc_ctx* ctx, uint64_t verify_id, const uint64_t* xs,
                            const uint64_t* ws_, const uint64_t* zpre, const uint64_t* pq,
                            int64_t M, int64_t N, int64_t K, int trunc_bits,
                            const uint64_t* row_keys, uint64_t matmul_call_id, int R_main,
                            int R_trunc, void* workspace, size_t workspace_bytes,
                            uint64_t* trace) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (M <= 0 || N <= 0 || K <= 0) return fail(ctx, MPC_ERR_SHAPE, "verify_matmul: bad shape");
  const bool trunc = trunc_bits >= 0;
  if (!xs || !ws_ || !zpre || (trunc && !pq) || !id_ok(verify_id) || !id_ok(matmul_call_id) ||
      trunc_bits > 63)
    return fail(ctx, MPC_ERR_ARG, "verify_matmul: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  VMatPlan p;
  if (!plan_vmat(ar, M, N, K, trunc_bits, R_main, R_trunc, ctx->gemm_path == MPC_GEMM_LIMB_TC,
                 ctx->tune, p))
    return fail(ctx, MPC_ERR_SHAPE, "verify_matmul: more than 15 truncation chunks");
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "verify_matmul: workspace too small");
  const Small& s = p.s;
  const long long MK = M * K, KN = K * N;
  Fork fork(ctx, p.fork);
  fork.on(0);
  // ---- batch 0: the M N inner products of Z = X W, rank-1 consolidation ----
  cudaStream_t st = ctx->st;
  Phase* phase = new Phase(ctx, MPC_PROF_VERIFY_GEMM);
  if ((rc = sums_begin(ctx, s))) return rc;
  reveal(ctx, P_VER_R, make_obj(verify_id, 0, 0), s, s.r);
  if ((rc = power_table(ctx, s.r, p.powQ, p.Q, s.aux + 64))) return rc;   // r^b
  launch_gr_mul1(st, p.Q + (N - 1) * 64, s.r, s.aux);                     // rho = r^N
  if ((rc = power_table(ctx, s.aux, p.powP, p.P, s.aux + 64))) return rc; // rho^a
  Vec& x = p.dv.x[0];
  Vec& y = p.dv.y[0];
  if (p.grouped) {   // all six components of a side in one product: rows c (K + 1) + k, row K zero
    GemmTerm T;
    T.A = op(xs, K, 1);
    T.B = op(p.P, 64);
    if ((rc = dense_gemm(ctx, 6 * (K + 1), 64, M, T, epi_store(x.c[0], 64), p.tcs, {K + 1, K, MK})))
      return rc;
    T.A = op(ws_, N);
    T.B = op(p.Q, 64);
    if ((rc = dense_gemm(ctx, 6 * (K + 1), 64, N, T, epi_store(y.c[0], 64), p.tcs, {K + 1, K, KN})))
      return rc;
  }
  for (int c = 0; c < 6 && !p.grouped; ++c) {
    GemmTerm T;
    T.A = op(xs + c * MK, K, 1);        // Xt_k = sum_a rho^a X_ak  (K x M) . (M x 64)
    T.B = op(p.P, 64);
    if ((rc = dense_gemm(ctx, K, 64, M, T, epi_store(x.c[c], 64), p.tcs))) return rc;
    GemmTerm U;
    U.A = op(ws_ + c * KN, N);          // Wt_k = sum_b r^b W_kb   (K x N) . (N x 64)
    U.B = op(p.Q, 64);
    if ((rc = dense_gemm(ctx, K, 64, N, U, epi_store(y.c[c], 64), p.tcs))) return rc;
  }
  {  // zt = sum_a rho^a (sum_b r^b Z_ab): T = Z Q for all 6 components, then Gram with P
    GemmTerm T;
    T.A = op(zpre, N);
    T.B = op(p.Q, 64);
    if ((rc = dense_gemm(ctx, 6 * M, 64, N, T, epi_store(p.T, 64), p.tcs))) return rc;
    CK(cudaMemsetAsync(p.Pz, 0, 6 * 4096 * 8, st));
    GramBatch gb;
    for (int c = 0; c < 6; ++c)
      gb.add(p.Pz + c * 4096, p.P, nullptr, 1, 64, p.T + c * M * 64, nullptr, 1, 64, 1);
    gemm_u64_gram_batch(st, M, gb.n, gb.T, gb.e, nsplit_for(M));
    launch_gr_fold_reduce(st, p.Pz, 6, s.zinit);
  }
  p.dv.cur = 0;
  rc = run_dense(ctx, verify_id, 0, p.dv, K, s.zinit, 1, p.R0, s, trace);
  delete phase;
  if (rc) return rc;
  // ---- batch 1: the truncation pairs, chunk by chunk ----
  fork.on(-1);
  if (trunc &&
      (rc = verify_trunc_batch(ctx, p.tb, p.st, p.tcst, pq, trunc_bits, verify_id, matmul_call_id,
                               trace ? trace + (long long)(p.R0 + 1) * TRACE_ROUND : nullptr,
                               (const u64*)row_keys, N)))
    return rc;
  fork.join();
  return finish_verify(ctx, (matmul_call_id << 1) | 1);
}

int mpc_reconstruct(mpc_ctx* ctx, const uint64_t* xs, int64_t n, uint64_t* out, int out_on_host,
                    void* workspace, size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n <= 0) return fail(ctx, MPC_ERR_SHAPE, "reconstruct: n <= 0");
  if (!xs || !out) return fail(ctx, MPC_ERR_ARG, "reconstruct: bad argument");
  if (!ctx->pending.empty())
    return fail(ctx, MPC_ERR_PENDING, "reconstruct: products are not verified yet");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  RecPlan p = plan_rec(ar, n, out_on_host != 0);
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "reconstruct: workspace too small");
  Phase* phase = new Phase(ctx, MPC_PROF_REC);
  cudaStream_t st = ctx->st;
  u64* o = out_on_host ? p.out_dev : (u64*)out;
  rec_core(ctx, xs, n, p, o, false);
  if (out_on_host) CK(cudaMemcpyAsync(out, o, (size_t)n * 8, cudaMemcpyDeviceToHost, st));
  delete phase;
  if ((rc = cuda_check(ctx, "reconstruct"))) return rc;
  u32 stv = 0;
  if ((rc = read_status(ctx, &stv))) return rc;
  if (stv & ST_ABORT) {
    ctx->aborted = true;
    if (out_on_host) std::memset(out, 0, (size_t)n * 8);
    else cudaMemsetAsync(out, 0, (size_t)n * 8, st);
    return fail(ctx, MPC_ERR_ABORT, "Pi_Rec: inconsistent messages");
  }
  return MPC_OK;
}

int mpc_ledger(const mpc_ctx* ctx, uint64_t* bytes, uint64_t* messages) {
  if (!ctx || !bytes) return MPC_ERR_ARG;
  for (int a = 0; a < MPC_NPHASE; ++a)
    for (int b = 0; b < MPC_NPROTO; ++b) bytes[a * MPC_NPROTO + b] = ctx->ledger[a][b];
  if (messages) *messages = ctx->nmsg;
  return MPC_OK;
}

void mpc_ledger_reset(mpc_ctx* ctx) {
  if (!ctx) return;
  std::memset(ctx->ledger, 0, sizeof(ctx->ledger));
  ctx->nmsg = 0;
}

int mpc_inject_fault(mpc_ctx* ctx, int site, uint64_t index, uint64_t xor_mask) {
  return mpc_inject_fault_after(ctx, site, 0, index, xor_mask);
}

int mpc_inject_fault_after(mpc_ctx* ctx, int site, uint64_t skip, uint64_t index, uint64_t xor_mask) {
  if (!ctx || site < 0 || site >= MPC_NSITE) return MPC_ERR_ARG;
  ctx->fault[site] = {true, index, site == MPC_SITE_HIGH_BIT ? (1ull << 63) : xor_mask, skip};
  return MPC_OK;
}

int mpc_profile(mpc_ctx* ctx, int enable) {
  if (!ctx) return MPC_ERR_ARG;
  if (enable) {
    ctx->recs.clear();
    ctx->pool_used = 0;
  }
  ctx->prof = enable != 0;
  return MPC_OK;
}

int mpc_profile_read(mpc_ctx* ctx, double* ms, uint64_t* count, double* work) {
  if (!ctx || !ms) return MPC_ERR_ARG;
  CK(cudaStreamSynchronize(ctx->st));
  for (int i = 0; i < MPC_NPROF; ++i) {
    ms[i] = 0.0;
    if (count) count[i] = 0;
    if (work) work[i] = 0.0;
  }
  for (const auto& r : ctx->recs) {
    float t = 0.f;
    CK(cudaEventElapsedTime(&t, r.a, r.b));
    if (r.id >= 0 && r.id < MPC_NPROF) {
      ms[r.id] += t;
      if (count) count[r.id] += 1;
      if (work) work[r.id] += r.work;
    }
  }
  ctx->recs.clear();
  ctx->pool_used = 0;
  return MPC_OK;
}

uint64_t mpc_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }


// ---- layer-level calls -----------------------------------------------------------------------
int mpc_share_fixed(mpc_ctx* ctx, uint64_t call_id, int owner, const double* x, int x_on_host,
                    int64_t n, int frac_bits, uint64_t* xs, void* workspace,
                    size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n < 0) return fail(ctx, MPC_ERR_SHAPE, "share_fixed: n < 0");
  if (frac_bits < 0 || frac_bits > 62) return fail(ctx, MPC_ERR_ARG, "share_fixed: frac_bits");
  if (n == 0) return MPC_OK;
  if (!x || !xs || !workspace) return fail(ctx, MPC_ERR_ARG, "share_fixed: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  u64* enc = ar.take<u64>(n);
  double* stage = ar.take<double>(n);
  if (!ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "share_fixed: workspace too small");
  const double* xd = x;
  if (x_on_host) {
    CK(cudaMemcpyAsync(stage, x, (size_t)n * 8, cudaMemcpyHostToDevice, ctx->st));
    xd = stage;
  }
  {
    Phase phase(ctx, MPC_PROF_SHARE);
    launch_encode_fixed(ctx->st, xd, n, frac_bits, enc);
  }
  rc = mpc_share_input_from(ctx, call_id, owner, enc, 0, n, xs, (char*)workspace + ar.off,
                            workspace_bytes > ar.off ? workspace_bytes - ar.off : 0);
  if (rc == MPC_OK && x_on_host) CK(cudaStreamSynchronize(ctx->st));   // x may be reused
  return rc;
}

int mpc_reconstruct_fixed(mpc_ctx* ctx, const uint64_t* xs, int64_t n, int frac_bits, double* out,
                          int out_on_host, void* workspace, size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n <= 0) return fail(ctx, MPC_ERR_SHAPE, "reconstruct_fixed: n <= 0");
  if (frac_bits < 0 || frac_bits > 62 || !xs || !out || !workspace)
    return fail(ctx, MPC_ERR_ARG, "reconstruct_fixed: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  u64* v = ar.take<u64>(n);
  double* stage = ar.take<double>(n);
  if (!ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "reconstruct_fixed: workspace too small");
  rc = mpc_reconstruct(ctx, xs, n, v, 0, (char*)workspace + ar.off,
                       workspace_bytes > ar.off ? workspace_bytes - ar.off : 0);
  if (rc) {
    if (out_on_host) std::memset(out, 0, (size_t)n * 8);
    return rc;
  }
  {
    Phase phase(ctx, MPC_PROF_REC);
    launch_decode_fixed(ctx->st, v, n, frac_bits, out_on_host ? stage : out);
  }
  if (out_on_host) {
    CK(cudaMemcpyAsync(out, stage, (size_t)n * 8, cudaMemcpyDeviceToHost, ctx->st));
    CK(cudaStreamSynchronize(ctx->st));
  }
  return cuda_check(ctx, "reconstruct_fixed");
}

int mpc_conv2d(mpc_ctx* ctx, uint64_t call_id, const uint64_t* xs, const uint64_t* ws_,
               const int32_t geom[8], int64_t C_out, int trunc_bits, const uint64_t* row_keys,
               uint64_t* cols, uint64_t* zpre, uint64_t* zout, uint64_t* pq, void* workspace,
               size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (!geom || !xs || !cols) return fail(ctx, MPC_ERR_ARG, "conv2d: bad argument");
  ConvGeom g;
  g.B = geom[0]; g.C = geom[1]; g.H = geom[2]; g.W = geom[3];
  g.kh = geom[4]; g.kw = geom[5]; g.stride = geom[6]; g.pad = geom[7];
  if (g.B <= 0 || g.C <= 0 || g.H <= 0 || g.W <= 0 || g.kh <= 0 || g.kw <= 0 || g.stride <= 0 ||
      g.pad < 0 || C_out <= 0)
    return fail(ctx, MPC_ERR_SHAPE, "conv2d: bad geometry");
  if (g.H + 2 * g.pad < g.kh || g.W + 2 * g.pad < g.kw)
    return fail(ctx, MPC_ERR_SHAPE, "conv2d: kernel larger than the padded image");
  g.Ho = (g.H + 2 * g.pad - g.kh) / g.stride + 1;
  g.Wo = (g.W + 2 * g.pad - g.kw) / g.stride + 1;
  launch_im2col(ctx->st, xs, g, cols);
  if ((rc = cuda_check(ctx, "conv2d: im2col"))) return rc;
  return mpc_matmul_keyed(ctx, call_id, cols, ws_, g.B * g.Ho * g.Wo, C_out, g.C * g.kh * g.kw,
                          trunc_bits, row_keys, zpre, zout, pq, workspace, workspace_bytes);
}

int mpc_trunc(mpc_ctx* ctx, uint64_t call_id, const uint64_t* xs, int64_t n, int t, uint64_t* out,
              uint64_t* pq, void* workspace, size_t workspace_bytes) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n <= 0) return fail(ctx, MPC_ERR_SHAPE, "trunc: n <= 0");
  if (t < 0 || t > 63 || !xs || !out || !pq || out == xs || !id_ok(call_id))
    return fail(ctx, MPC_ERR_ARG, "trunc: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  TruncCallPlan p = plan_trunc_call(ar, n);
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "trunc: workspace too small");
  cudaStream_t st = ctx->st;
  const u64 obj = make_obj(call_id, 0, 0);
  {  // preprocessing (Fig. trunc): the pairs, as for a truncated product
    Phase phase(ctx, MPC_PROF_TRUNC_PAIRS);
    launch_trunc_p0(st, n, ctx->k01, ctx->k02, obj, t, p.rx, out, pq, p.gp2, p.gq2, p.mp1, p.mq1,
                    nullptr, n);
    PairMsgs m;
    if ((rc = deliver_pairs(ctx, p.gp2, p.gq2, p.mp1, p.mq1, n, p.fc, m))) return rc;
    launch_trunc_finish(st, n, ctx->k01, ctx->k02, obj, t, m.mp1, m.mq1, m.mp2, m.mq2, m.gp2, m.gq2, p.mp1,
                        p.mq1, p.rx, out, pq, nullptr, n);
  }
  {  // online: the wire's mask switched to the pairs' r_x (checked by P0's hashes), then m >> t
    Phase phase(ctx, MPC_PROF_EXCHANGE);
    launch_trunc_remask(st, xs, p.rx, n, p.d1, p.d2, p.d1p0, p.d2p0);
    const int ph = MPC_PHASE_ONLINE, pr = MPC_PROTO_TRUNC;
    const u64 *d1_at_p2, *d2_at_p1;
    if ((rc = deliver(ctx, ph, pr, p.d1, d1_at_p2, n, MPC_SITE_TRUNC_D1, p.d1x))) return rc;   // P1->P2
    if ((rc = deliver(ctx, ph, pr, p.d2, d2_at_p1, n, -1, nullptr))) return rc;               // P2->P1
    // P0 sends H(d1) to P2 and H(d2) to P1, who hash the d1, d2 they received
    const u64* data[4] = {p.d1p0, p.d2p0, d1_at_p2, d2_at_p1};
    HashJobs hj{};
    for (int q = 0; q < 4; ++q) {
      hj.data[q] = data[q];
      hj.scratch[q] = p.hs[q];
      hj.digest[q] = p.dg + 8 * q;
    }
    launch_hash_jobs(st, hj, 4, n);
    count_msgs(ctx, ph, pr, 2, 32);
    launch_digest_check(st, p.dg, p.dg + 16, p.dg + 8, p.dg + 24, p.dg, p.dg + 16, ctx->status,
                        ST_ABORT);
    launch_trunc_online(st, xs, n, p.d1, d2_at_p1, d1_at_p2, p.d2, t, out);
  }
  if ((rc = cuda_check(ctx, "trunc"))) return rc;
  ctx->pending.insert((call_id << 1) | 1);
  u32 stv = 0;
  if ((rc = read_status(ctx, &stv))) return rc;
  if (stv & ST_ABORT) {
    ctx->aborted = true;
    return fail(ctx, MPC_ERR_ABORT, "Pi_Trunc: a mask-switch message disagrees with P0's hash");
  }
  return MPC_OK;
}

int mpc_verify_trunc(mpc_ctx* ctx, uint64_t verify_id, const uint64_t* pq, int64_t n, int t,
                     uint64_t trunc_call_id, int R, void* workspace, size_t workspace_bytes,
                     uint64_t* trace) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n <= 0) return fail(ctx, MPC_ERR_SHAPE, "verify_trunc: n <= 0");
  if (!pq || t < 0 || t > 63 || !id_ok(verify_id) || !id_ok(trunc_call_id))
    return fail(ctx, MPC_ERR_ARG, "verify_trunc: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  VTruncPlan p;
  if (!plan_vtrunc(ar, n, R, ctx->gemm_path == MPC_GEMM_LIMB_TC, ctx->tune, p))
    return fail(ctx, MPC_ERR_SHAPE, "verify_trunc: more than 15 chunks");
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "verify_trunc: workspace too small");
  if ((rc = verify_trunc_batch(ctx, p.tb, p.s, p.tcs, pq, t, verify_id, trunc_call_id, trace,
                               nullptr, n)))
    return rc;
  return finish_verify(ctx, (trunc_call_id << 1) | 1);
}


int mpc_test_wait_expires(mpc_ctx* ctx, int64_t cycles) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (cycles < 1 || cycles > 100000000) return fail(ctx, MPC_ERR_ARG, "test_wait_expires: cycles");
  launch_wait_expires(ctx->st, cycles, ctx->status, ST_TIMEOUT);
  if ((rc = cuda_check(ctx, "test_wait_expires"))) return rc;
  u32 stv = 0;
  return read_status(ctx, &stv);   // MPC_ERR_TIMEOUT, and the context is aborted
}
}  // extern "C"

// ---- accessors for other translation units of the library (not part of the C-ABI) ----------
namespace mpc3 {
namespace internal {
int ctx_guard(mpc_ctx* c) { return guard(c); }
int ctx_fail(mpc_ctx* c, int code, const char* msg) { return fail(c, code, msg); }
MsgFault ctx_take_rec_fault(mpc_ctx* c, long long n) { return take_fault(c, MPC_SITE_REC_MSG, n); }
void ctx_count(mpc_ctx* c, int phase, int proto, int count, u64 bytes_each) {
  count_msgs(c, phase, proto, count, bytes_each);
}
int ctx_read_status(mpc_ctx* c, u32* out) { return read_status(c, out); }
bool ctx_has_pending(const mpc_ctx* c) { return !c->pending.empty(); }
cudaStream_t ctx_stream(const mpc_ctx* c) { return c->st; }
u32* ctx_status_word(const mpc_ctx* c) { return c->status; }
void ctx_set_aborted(mpc_ctx* c) { c->aborted = true; }
}  // namespace internal
}  // namespace mpc3

// ---- non-linear layers (Sec. 4.3) -------------------------------------------------------------
namespace {

// take_fault for a Boolean message of nw words: the AND_GAMMA2 site flips bit `index` of it (when mask
// & 1), the Boolean counterpart of an element fault; HIGH_BIT at l = 1 is the same bit flip.
MsgFault take_bit_fault(mpc_ctx* ctx, int site, long long nw) {
  const MsgFault f = take_fault(ctx, site, 64 * nw);
  if (f.idx < 0 || !(f.mask & 1ull)) return {};
  return {f.idx / 64, 1ull << (f.idx % 64)};
}

// The messages of a Pi_Mult (three of n words; offline [Gamma]_2, online the halves of m)
void count_mult(mpc_ctx* ctx, long long n) {
  count_msgs(ctx, MPC_PHASE_OFFLINE, MPC_PROTO_MULT, 1, (u64)n * 8);
  count_msgs(ctx, MPC_PHASE_ONLINE, MPC_PROTO_MULT, 2, (u64)n * 8);
}

constexpr int NL_LEVELS = 6;
inline int level_planes(int l) { return l == NL_LEVELS ? 1 : 2 * (32 >> (l - 1)); }   // 64,32,..,4,1

// Buffers of one compare-select stage of np (padded) elements, W = np / 64 words per plane; the bit
// planes eda[0], eda[1], the triples and the outputs are the layer's (plan_nl).
struct CSPlan {
  CompareSelect k;
  u64 *delta, *dpl, *dbits;      // np public words, their 64 W bit planes, W words
  RecPlan reca, recb;
};

CSPlan plan_cs(Arena& a, long long np) {
  CSPlan p;
  CompareSelect& k = p.k;
  const long long W = np / 64;
  k.np = np;
  k.eda[2] = a.take<u64>(np);
  for (int q = 0; q < 3; ++q) k.da[q] = a.take<u64>(W);
  k.eprod = a.take<u64>(6 * 64 * np);
  k.ez = a.take<u64>(6 * np);
  k.dd = a.take<u64>(6 * np);
  k.rad = a.take<u64>(6 * np);
  k.e = a.take<u64>(6 * W);
  p.delta = a.take<u64>(np);
  p.dpl = a.take<u64>(np);
  p.dbits = a.take<u64>(W);
  k.dpl = p.dpl;
  k.dbits = p.dbits;
  p.reca = plan_rec(a, np, false);
  p.recb = plan_rec(a, W, false);
  return p;
}

constexpr int AND_PLANES = 125;   // AND gates of the carry tree, per element: 64 + 32 + 16 + 8 + 4 + 1

// <max(a, b)> of a stage (p.k.a, p.k.b into p.k.out): Sec. 4.3 compare-select
int compare_select(mpc_ctx* ctx, u64 call_id, int stage, CSPlan& p) {
  cudaStream_t st = ctx->st;
  CompareSelect& k = p.k;
  const long long np = k.np, W = np / 64, N = 64 * np;
  k.k01 = ctx->k01;
  k.k02 = ctx->k02;
  k.k12 = ctx->k12;
  k.obj = make_obj(call_id, (u32)stage, 0);
  k.fault[0] = take_fault(ctx, MPC_SITE_GAMMA2, N);
  k.fault[1] = take_fault(ctx, MPC_SITE_MZ1, N);
  k.fault[2] = take_fault(ctx, MPC_SITE_MZ2, N);
  k.fault[3] = take_bit_fault(ctx, MPC_SITE_AND_GAMMA2, 64 * W);
  // edaBits (Fig. edabits) and Delta = d - r, d = a - b
  launch_cs_open_delta(st, k);
  count_mult(ctx, N);                                                    // the bit products
  count_msgs(ctx, MPC_PHASE_OFFLINE, MPC_PROTO_INNER, 3, (u64)np * 8);   // the inner products
  rec_core(ctx, k.dd, np, p.reca, p.delta, false);
  // msb(d) by the carry circuit over the bits of Delta + r; daBits; e = [d >= 0] XOR bit
  launch_trunc_bit_transpose(st, p.delta, np, p.dpl);
  launch_cs_open_bit(st, k);
  for (int l = 1; l <= NL_LEVELS; ++l) count_mult(ctx, level_planes(l) * W);
  count_mult(ctx, np);   // the daBits' two products
  count_mult(ctx, np);
  rec_core(ctx, k.e, W, p.recb, p.dbits, true);
  // out = b + (a - b) [a >= b]
  launch_cs_select(st, k);
  count_mult(ctx, np);
  return cuda_check(ctx, "compare_select");
}

// ---- verification of a non-linear layer -------------------------------------------------------
struct GfPlan {   // GF(2^64) Pi_MultVerify of D AND gates
  long long D;
  int R;
  u64 *XA, *YA, *ZA;        // concatenated triples, 6 x nw words each
  u64 *pw, *st;
  GfWork* w;
  u64 *x[2], *y[2];
};

GfPlan plan_gf(Arena& a, long long nw) {
  GfPlan g;
  g.D = 64 * nw;
  g.R = default_R(g.D);
  g.XA = a.take<u64>(6 * nw); g.YA = a.take<u64>(6 * nw); g.ZA = a.take<u64>(6 * nw);
  g.pw = a.take<u64>(8 * nw);
  g.st = a.take<u64>(9 * (g.R + 1));
  g.w = a.take<GfWork>(1);
  for (int i = 0; i < 2; ++i) {
    g.x[i] = a.take<u64>(i ? 24 * nw : 48 * nw);
    g.y[i] = a.take<u64>(i ? 24 * nw : 48 * nw);
  }
  return g;
}

// Pi_MultVerify (Fig. PPEV) over GF(2^64) of the AND triples in g.XA/YA/ZA (batch 2)
int gf_verify(mpc_ctx* ctx, u64 vid, GfPlan& g, u64* trace) {
  GfVerify v;
  v.X = g.XA;
  v.Y = g.YA;
  v.Z = g.ZA;
  v.nw = g.D / 64;
  v.R = g.R;
  v.k01 = ctx->k01;
  v.k02 = ctx->k02;
  v.k12 = ctx->k12;
  v.obj = make_obj(vid, 2, 0);
  v.pw = g.pw;
  v.st = g.st;
  v.w = g.w;
  for (int i = 0; i < 2; ++i) {
    v.x[i] = g.x[i];
    v.y[i] = g.y[i];
  }
  v.trace = trace;
  v.trace_ld = MPC_TRACE_GF_ROUND;
  v.status = ctx->status;
  v.flag_verify = ST_VERIFY;
  v.flag_abort = ST_ABORT;
  v.xrec = -1;
  v.xmask = 0;
  for (int i = 0; i < g.R + 2; ++i) {   // the openings: r, the zetas, Delta
    const MsgFault f = take_fault(ctx, MPC_SITE_REC_MSG, 1);
    if (f.idx < 0) continue;
    v.xrec = i;
    v.xmask = f.mask;
  }
  launch_gf_verify(ctx->st, v);
  // Pi_Rec of r, the zetas and Delta (3 words and 3 hashes each); two secure inner products a round,
  // x alpha and the last inner product
  const int ph = MPC_PHASE_VERIFY, pr = MPC_PROTO_VERIFY;
  count_msgs(ctx, ph, pr, 3 * (g.R + 2), 8);
  count_msgs(ctx, ph, pr, 3 * (g.R + 2), 32);
  count_msgs(ctx, ph, pr, 3 * (2 * g.R + 1), 8);
  count_msgs(ctx, ph, pr, 3, (u64)8 * dim_after(g.D, g.R));
  return cuda_check(ctx, "gf_verify");
}

struct NLPlan {
  int nst;
  CSPlan cs[2];
  u64 *a, *b, *o;                // max-pool's first stage: operands and result (6 x np each)
  // batch 0: arithmetic products
  long long nm;
  u64 *MX, *MY, *MZ;
  VMultPlan vm;
  // batch 1: edaBit inner products (D1 = 64 sum np rows)
  long long ne, D1;
  int R1;
  Small s1;
  BlkPlan b1;
  u64* Ye;                       // 6 x D1 ring words: the y side
  u64* Xe;                       // D1 ring words: the bits m (components 2 and 4 of x)
  // batch 2: AND gates
  GfPlan gf;
  // batch 3: edaBit bit products (nb = 64 sum np), x only [r]_1 and y only [r]_2 (reading N9)
  long long nb;
  int Rb;
  Small sb;
  TruncPlan tb;                  // bit words of 64 products each
  u64* Zr;                       // 6 x 64 elements: the claim's sums over the bit words
  void* wsum = nullptr;          // digit planes for them (long batches on the limb path)
};

// Elements of a stage from which the sums over its bit words go to the tensor cores (61 us on
// the CUDA cores at 4032, 60 us at 4096 in three launches; 235 and 80 us at 16384).
constexpr long long WORDS_TC_MIN = 4096;

NLPlan plan_nl(Arena& a, int nst, const long long np[2], bool tc, const mpc_tuning& tu) {
  NLPlan p;
  p.nst = nst;
  p.nm = 0;
  p.ne = 0;
  for (int s = 0; s < nst; ++s) {
    p.cs[s] = plan_cs(a, np[s]);
    p.nm += 3 * np[s];
    p.ne += np[s];
  }
  const long long n0 = nst > 1 ? 6 * np[0] : 0;
  p.a = a.take<u64>(n0);
  p.b = a.take<u64>(n0);
  p.o = a.take<u64>(n0);
  const long long andw = AND_PLANES * (p.ne / 64);
  p.MX = a.take<u64>(6 * p.nm); p.MY = a.take<u64>(6 * p.nm); p.MZ = a.take<u64>(6 * p.nm);
  p.vm = plan_vmult(a, p.nm, -1, tc);
  p.D1 = 64 * p.ne;
  p.R1 = default_R(p.D1);
  p.s1 = plan_small(a);
  const bool xc[6] = {false, false, true, false, true, false};
  const bool yc[6] = {true, true, true, true, true, true};
  p.b1 = plan_blk(a, p.D1, p.R1, 6, false, xc, yc, tc);
  p.Ye = a.take<u64>(6 * p.D1);
  p.Xe = a.take<u64>(p.D1);
  p.gf = plan_gf(a, andw);
  p.nb = 64 * p.ne;
  p.Rb = default_R(p.nb);
  p.sb = plan_small(a);
  p.tb = plan_trunc(a, p.ne, p.Rb, tc, false, tu, true);
  p.Zr = a.take<u64>(384 * 64);
  if (tc && np[0] >= WORDS_TC_MIN)
    p.wsum = a.take<unsigned char>((long long)limb_tc_scratch_bytes(384, 64, np[0], 1));
  // each stage's part of the batches: its triples and its edaBits' bit words
  long long e0 = 0;
  for (int s = 0; s < nst; ++s) {
    CompareSelect& k = p.cs[s].k;
    k.nm = p.nm;
    for (int q = 0; q < 3; ++q) {
      const long long o = 3 * e0 + q * np[s];
      k.mx[q] = p.MX + o;
      k.my[q] = p.MY + o;
      k.mz[q] = p.MZ + o;
    }
    k.eda[0] = p.tb.b1 + e0;
    k.eda[1] = p.tb.b2 + e0;
    k.ax = p.gf.XA;
    k.ay = p.gf.YA;
    k.az = p.gf.ZA;
    k.and_words = andw;
    k.and_off = AND_PLANES * (e0 / 64);
    e0 += np[s];
  }
  return p;
}

int verify_nl(mpc_ctx* ctx, u64 vid, NLPlan& p, u64* trace) {
  int rc;
  u64* tr1 = trace ? trace + (long long)(p.vm.R + 1) * TRACE_ROUND : nullptr;
  u64* tr2 = tr1 ? tr1 + (long long)(p.R1 + 1) * TRACE_ROUND : nullptr;
  u64* tr3 = tr2 ? tr2 + (long long)(p.gf.R + 1) * MPC_TRACE_GF_ROUND : nullptr;
  Fork fork(ctx);   // four independent batches, the longest chains of launches first
  // ---- batch 1: the edaBit inner products, weight r^e on row e (e over all stages)
  fork.on(0);
  {
    cudaStream_t st = ctx->st;
    const Small& s = p.s1;
    if ((rc = sums_begin(ctx, s))) return rc;
    reveal(ctx, P_VER_R, make_obj(vid, 1, 0), s, s.r);
    BlkPlan& b = p.b1;
    launch_ones(st, b.B, b.T);   // weights r^e on the 64 entries of element e
    if ((rc = power_table(ctx, s.r, b.pp, b.Rw, s.aux))) return rc;
    CK(cudaMemsetAsync(s.zinit, 0, 384 * 8, st));
    long long e0 = 0;
    for (int q = 0; q < p.nst; ++q) {   // the words and the claim
      const CompareSelect& c = p.cs[q].k;
      launch_eda_words(st, c.eda, c.eprod, c.np, e0, p.D1, p.Xe, p.Ye);
      launch_scalar_gr_sum(st, c.np, c.ez, c.np, 6, b.Rw + e0 * 64, s.zinit);
      e0 += c.np;
    }
    Vec x{}, y;
    x.c[2] = x.c[4] = p.Xe;
    for (int c = 0; c < 6; ++c) y.c[c] = p.Ye + c * p.D1;
    if ((rc = run_blk(ctx, vid, 1, b, x, y, nullptr, s, tr1))) return rc;
  }
  // ---- batch 3: the edaBit bit products b_{i,1} b_{i,2}, stage by stage (plane-major); x has
  // only the [r]_1 components and y only the [r]_2 ones, so the dense rounds take the
  // single-Gram form
  fork.on(1);
  {
    cudaStream_t st = ctx->st;
    const Small& s = p.sb;
    if ((rc = sums_begin(ctx, s))) return rc;
    reveal(ctx, P_VER_R, make_obj(vid, 3, 0), s, s.r);
    // 64 consecutive products are the bits of one word of the b1 and b2 planes
    TruncPlan& t = p.tb;
    launch_gr_powers(st, s.r, 64, t.V);                                   // V_j = r^j
    launch_gr_mul1(st, t.V + 63 * 64, s.r, s.aux + 64);                   // rho = r^64
    if ((rc = bit_tables(ctx, t, s, s.aux + 64))) return rc;
    CK(cudaMemsetAsync(t.zt + 384, 0, 384 * 8, st));
    long long w0 = 0;
    for (int q = 0; q < p.nst; ++q) {
      const CompareSelect& c = p.cs[q].k;
      // sum over w of rho^w z_c[64 w + j] for the 384 rows (c, j)
      if (p.wsum) {
        GemmTerm T;
        T.A = op(c.eprod, 64, 1);
        T.B = op(t.Rtab + w0 * 64, 64);
        if ((rc = dense_gemm(ctx, 384, 64, c.np, T, epi_store(p.Zr, 64), p.wsum, {64, 64, 64 * c.np})))
          return rc;
      } else {
        CK(cudaMemsetAsync(p.Zr, 0, 384 * 512, st));
        launch_words_sums(st, c.eprod, 64 * c.np, c.np, t.Rtab + w0 * 64, p.Zr);
      }
      launch_blk_claim(st, t.V, p.Zr, 64, t.zt + 384);
      w0 += c.np;
    }
    if ((rc = bit_batch(ctx, t, s, t.zt + 384, vid, 3, tr3))) return rc;
  }
  // ---- batch 0: the daBit products (two) and the final product, stage by stage (the edaBit
  // bit products are batch 3)
  fork.on(2);
  {
    VMultPlan& v = p.vm;
    const Small& s = v.s;
    const long long n = p.nm;
    if ((rc = sums_begin(ctx, s))) return rc;
    reveal(ctx, P_VER_R, make_obj(vid, 0, 0), s, s.r);
    if ((rc = blk_tables(ctx, v.b, s.r, s.aux))) return rc;
    Vec x, y;
    for (int c = 0; c < 6; ++c) {
      x.c[c] = p.MX + c * n;
      y.c[c] = p.MY + c * n;
    }
    if ((rc = run_blk(ctx, vid, 0, v.b, x, y, p.MZ, s, trace))) return rc;
  }
  // ---- batch 2: every AND gate over GF(2^64), stage by stage, level by level
  fork.on(-1);
  if ((rc = gf_verify(ctx, vid, p.gf, tr2))) return rc;
  return MPC_OK;
}

int nl_finish(mpc_ctx* ctx) {
  u32 stv = 0;
  int rc = read_status(ctx, &stv);
  if (rc) return rc;
  if (stv & ST_ABORT) {
    ctx->aborted = true;
    return fail(ctx, MPC_ERR_ABORT, "Pi_Rec: inconsistent messages");
  }
  if (stv & ST_VERIFY) {
    ctx->aborted = true;
    return fail(ctx, MPC_ERR_VERIFY, "non-linear layer: verification failed");
  }
  return MPC_OK;
}

long long npad64(long long n) { return 64 * ((n + 63) / 64); }

void nl_plan_take(Arena& a, int nst, const long long np[2], bool tc, const mpc_tuning& tu) {
  plan_nl(a, nst, np, tc, tu);
}

}  // namespace

int mpc_relu(mpc_ctx* ctx, uint64_t call_id, uint64_t verify_id, const uint64_t* xs, int64_t n,
             uint64_t* out, void* workspace, size_t workspace_bytes, uint64_t* trace) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n <= 0) return fail(ctx, MPC_ERR_SHAPE, "relu: n <= 0");
  if (!xs || !out || !id_ok(call_id) || !id_ok(verify_id)) return fail(ctx, MPC_ERR_ARG, "relu: bad argument");
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  const long long np[2] = {npad64(n), 0};
  NLPlan p = plan_nl(ar, 1, np, ctx->gemm_path == MPC_GEMM_LIMB_TC, ctx->tune);
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "relu: workspace too small");
  Phase phase(ctx, MPC_PROF_NONLINEAR);
  CompareSelect& k = p.cs[0].k;
  k.a = {xs, n, n};
  k.b = {nullptr, 0, 0};
  k.out = out;
  k.out_ld = k.out_n = n;
  if ((rc = compare_select(ctx, call_id, 0, p.cs[0]))) return rc;
  if ((rc = verify_nl(ctx, verify_id, p, trace))) return rc;
  if ((rc = cuda_check(ctx, "relu"))) return rc;
  return nl_finish(ctx);
}

int mpc_maxpool2(mpc_ctx* ctx, uint64_t call_id, uint64_t verify_id, const uint64_t* xs, int64_t B,
                 int64_t C, int64_t H, int64_t W, uint64_t* out, void* workspace,
                 size_t workspace_bytes, uint64_t* trace) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (B <= 0 || C <= 0 || H <= 0 || W <= 0 || (H & 1) || (W & 1))
    return fail(ctx, MPC_ERR_SHAPE, "maxpool2: bad shape");
  if (!xs || !out || !id_ok(call_id) || !id_ok(verify_id)) return fail(ctx, MPC_ERR_ARG, "maxpool2: bad argument");
  const long long nw = B * C * (H / 2) * (W / 2);
  Arena ar{(char*)workspace, workspace_bytes, 0, false};
  const long long np[2] = {npad64(2 * nw), npad64(nw)};
  NLPlan p = plan_nl(ar, 2, np, ctx->gemm_path == MPC_GEMM_LIMB_TC, ctx->tune);
  if (!workspace || !ar.ok()) return fail(ctx, MPC_ERR_WORKSPACE, "maxpool2: workspace too small");
  Phase phase(ctx, MPC_PROF_NONLINEAR);
  cudaStream_t st = ctx->st;
  // stage 0 operands: left = [a ; c], right = [b ; d] of every window; stage 1: the two halves of its
  // result
  launch_window_gather(st, xs, B * C, H, W, np[0], p.a, p.b);
  CompareSelect &k0 = p.cs[0].k, &k1 = p.cs[1].k;
  k0.a = {p.a, np[0], 2 * nw};
  k0.b = {p.b, np[0], 2 * nw};
  k0.out = p.o;
  k0.out_ld = np[0];
  k0.out_n = 2 * nw;
  k1.a = {p.o, np[0], nw};
  k1.b = {p.o + nw, np[0], nw};
  k1.out = out;
  k1.out_ld = k1.out_n = nw;
  for (int s = 0; s < 2; ++s)
    if ((rc = compare_select(ctx, call_id, s, p.cs[s]))) return rc;
  if ((rc = verify_nl(ctx, verify_id, p, trace))) return rc;
  if ((rc = cuda_check(ctx, "maxpool2"))) return rc;
  return nl_finish(ctx);
}

int mpc_hash_u64(mpc_ctx* ctx, const uint64_t* data, int64_t n, uint8_t* digest) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n < 0) return fail(ctx, MPC_ERR_SHAPE, "hash: bad size");
  if ((n > 0 && !data) || !digest) return fail(ctx, MPC_ERR_ARG, "hash: bad argument");
  u32* scratch = nullptr;
  const size_t words = hash_scratch_words(n) + 8;
  cudaError_t e = cudaMalloc(&scratch, words * sizeof(u32));
  if (e != cudaSuccess) return fail(ctx, MPC_ERR_CUDA, "hash: scratch allocation");
  u32 h[8];
  launch_hash_u64(ctx->st, data, n, scratch, scratch + words - 8);
  e = cudaMemcpyAsync(h, scratch + words - 8, sizeof(h), cudaMemcpyDeviceToHost, ctx->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->st);
  cudaFree(scratch);
  if (e != cudaSuccess) return fail(ctx, MPC_ERR_CUDA, cudaGetErrorString(e));
  for (int q = 0; q < 8; ++q)
    for (int b = 0; b < 4; ++b) digest[4 * q + b] = (uint8_t)(h[q] >> (24 - 8 * b));
  return cuda_check(ctx, "hash");
}

int mpc_gather(mpc_ctx* ctx, const uint64_t* xs, int64_t n_in, const int64_t* idx, int64_t n_out,
               uint64_t* out) {
  int rc = guard(ctx);
  if (rc) return rc;
  if (n_in <= 0 || n_out <= 0) return fail(ctx, MPC_ERR_SHAPE, "gather: bad size");
  if (!xs || !idx || !out) return fail(ctx, MPC_ERR_ARG, "gather: bad argument");
  launch_gather(ctx->st, xs, n_in, reinterpret_cast<const long long*>(idx), n_out, out);
  return cuda_check(ctx, "gather");
}
