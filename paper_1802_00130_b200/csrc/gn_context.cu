// Host side of the C ABI (include/gn.h): context, workspaces, and the launch sequences for the
// stored forward pass, f / gradient over row batches, the full and block-diagonal Gauss-Newton
// products, and conjugate gradient.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/gn.h"
#include "gn_kernels.h"

// Named ranges around the phases of the path (stored forward pass, f / gradient, products, CG solve) for timeline
// tools; compiled in only with -DGN_NVTX (paper_1802_00130_b200/build.py: GN_NVTX=1 in the environment).
#ifdef GN_NVTX
#include <nvtx3/nvToolsExt.h>
namespace {
struct PhaseRange {
  explicit PhaseRange(const char* name) { nvtxRangePushA(name); }
  ~PhaseRange() { nvtxRangePop(); }
};
}  // namespace
#define GN_PHASE(name) PhaseRange gn_phase_range_(name)
#else
#define GN_PHASE(name) do { } while (0)
#endif

using namespace gn;

struct gn_ctx {
  int L = 0;
  std::vector<int> w;               // n_0..n_L
  double C = 1.0;
  int64_t l = 0;
  const float* dX = nullptr;
  const float* dY = nullptr;
  gn_precision prec = GN_FP32_ACCURATE;
  cudaStream_t st = nullptr;
  // side stream: the bias column sums and the n_L-row weight block of a layer are independent of the layer's large
  // contractions and small enough to run beside them; they are forked off after the layer's delta is ready and
  // joined before the product (or row batch) ends
  cudaStream_t st2 = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  bool side_enabled = true, side_open = false, side_region = false;
  int64_t n = 0;
  std::vector<int64_t> w_off, b_off;  // [m], m = 1..L (entry 0 unused)
  int64_t batch_rows = 32768;
  bool have_theta = false, have_sub = false;

  float* theta = nullptr;
  // subsample
  int64_t nS = 0, capS = 0;
  int32_t* idx = nullptr;
  std::vector<float*> Z;    // Z[0] = X_S, Z[m] = [nS][n_m]
  // RZ[m], DS[m]: forward directional derivatives and backward quantities d(.)/d s^m, [|S|][n_m]; once the
  // propagate form of the block-diagonal product has been asked for they are m |S| rows deep (its L streams
  // stacked along rows), see ensure_stacked
  std::vector<float*> RZ;
  std::vector<float*> DS;
  bool stacked = false;     // RZ / DS hold m * capS rows (else capS rows)
  // stored Jacobian factors d z^L / d s^m on the subsample (block-diagonal product, Section 3.3.1)
  std::vector<float*> DF;   // DF[m] = [nS * n_L][n_m], m = 1..L-1
  int64_t capF = 0;         // rows of S the factor buffers hold
  bool factors_valid = false;
  int bd_method = 0;        // 0 choose, 1 propagate L stacked streams, 2 stored factors
  int bd_expect = 0;        // products the running solver may still ask for (0 outside a solver)
  int bd_count = 0;         // propagate-form products since the factors were last invalidated
  // variable partition (Section 3.1): split[m] contiguous neuron groups in layer m; all ones = one block per layer
  std::vector<int> split;
  bool has_split = false;
  int P = 0;                // number of partitions = sum_m split[m-1] split[m]
  float* SU = nullptr; float* SQ = nullptr; int64_t capSplit = 0;   // per-group right-hand sides and results
  int cg_min = 0;           // termination rule of Section 4.4 for block-diagonal solves
  double cg_share = 1.0;
  // row-batch workspace of f / grad
  int64_t capB = 0;
  std::vector<float*> Zb, Db;
  // reductions
  float* colsum_scratch = nullptr; int64_t colsum_cap = 0;
  float* thin_scratch = nullptr; int64_t thin_cap = 0;
  float* sk_ws = nullptr; int* sk_flags = nullptr;   // stream-K workspace of the tensor-core kernel
  bool sk_enabled = true;
  bool group_enabled = true;   // independent contractions of a layer as one launch (TF32 mode)
  // consecutive layers of a pass as one launch with tile-level dependencies (TF32 mode): 0 never, 1 the stored forward
  // pass (where it measured 8 % faster), 2 also the forward R pass of a product (where cutting left-over tiles along K,
  // which a chained launch does not do, measured as fast or faster)
  int chain_level = 1;
  bool split_k_enabled = true; // weight blocks of the stored-factor product as two chained parts of the rows
  int64_t cut_for_nS = -1, cut_rows = 0;   // rows of the first part, chosen once per subsample size
  bool cut_for_half = false;                 // ... and kind of operands
  bool fly_enabled = true;                 // last hidden layer's factor formed on the fly in the stored-factor product
  int back_chain = 2;                      // hidden layers of a backward pass as one chained launch: 0 never, 1 always, 2 where it pays
  int* chain_ctr = nullptr; int64_t chain_ctr_cap = 0;   // finished-tile counters of such a launch
  // FP32-accurate contractions on the tensor cores (gemm_f16x3.cu): two FP16 parts of every operand
  int acc_method = 0;        // 0 choose (tensor cores where they are faster), 1 FP32 FMA only, 2 as 0
  bool x3_usable = true;     // cleared if the tensor-core kernel could not be launched
  uint64_t theta_epoch = 1, sub_epoch = 1;   // bumped whenever theta / the stored activations are rewritten
  // [hi part: cap elements][lo part: cap elements][exponents of the cells, in whole 16 bytes]
  struct SplitBuf {
    uint16_t* p = nullptr; int64_t cap = 0;
    int8_t* cells() const { return reinterpret_cast<int8_t*>(p + 2 * cap); }
    static int64_t elements(int64_t cap) { return 2 * cap + (split_cell_bytes(cap) + 15) / 16 * 8; }
  };
  // Parts kept until the matrix changes: of matrices inside theta (kind 1) and the stored Z_m (kind 2), and, for the
  // length of one launch sequence, inside the product's v (kind 3) and the row batch's X and Z_m (kind 4).  The key is
  // the matrix's place in those, never an address of the caller's.  Whole layers' matrices have their place in one
  // allocation per kind (arena), anything else (a sub-block of a split structure) a buffer of its own.
  struct SplitEntry { int kind; int64_t key; int64_t rows; int cols; int64_t ld; uint64_t epoch; SplitBuf buf; bool in_arena; };
  std::vector<SplitEntry> split_cache;
  uint16_t* arena[5] = {nullptr, nullptr, nullptr, nullptr, nullptr}; int64_t arena_rows[5] = {0, 0, 0, 0, 0};
  const float* cur_v = nullptr;                            // the vector of the product in progress
  const float* cur_x = nullptr;                            // the rows of X of the batch in progress
  struct SplitSlot {         // parts of any other operand: one slot per operand role, overwritten by the next use
    const float* src = nullptr; int64_t rows = 0; int cols = 0; int64_t ld = 0; SplitBuf buf;
    uint64_t seq = 0;        // contraction (gemm_seq) that wrote these parts
  };
  SplitSlot split_slot[4];
  SplitOperand h_ops[4];                                   // of the contraction being launched
  uint64_t parts_epoch = 1;
  bool split_together = true;                              // a contraction's operands in one splitting launch (else one each)
  bool own_capture = false, foreign_capture = false;       // the solver's step / the caller is capturing the stream
  uint64_t gemm_seq = 0;     // counts contractions (run_gemm calls)
  // FP16 copies of the matrices that TF32 contractions of a large pass read (HalfInfo in gn_kernels.h): of the stored activations
  // and theta's weights until these change, of everything else for the length of a pass.  One entry per FP32 matrix it stands for.
  struct HalfBuf {
    uint16_t* p = nullptr; int64_t cap = 0;                  // (cap: elements of an allocation of its own, 0: borrowed memory)
    const float* base = nullptr; int64_t rows = 0; int cols = 0;   // the matrix the copy is of
    int info = 0;                                            // index into half_info
    bool valid = false, info_valid = false;                  // the copy, and its info, belong to what the matrix now holds
  };
  enum HalfSet { kHZ, kHV, kHRZ, kHDS, kHZb, kHDb, kHW, kHF, kHalfSets };   // (kHV[0]: all of a vector, its scale; kHZb[0]: the rows of X of a batch; kHF: factors)
  std::vector<HalfBuf> half_buf[kHalfSets];
  HalfInfo* half_info = nullptr; unsigned* half_acc = nullptr; unsigned long long* half_sums = nullptr;
  uint16_t* half_weights = nullptr; std::vector<int64_t> half_at;   // the copies of theta's weights, then of a vector's; where layer m's starts
  struct HalfSums { int64_t v_rows, rows, cols; };
  std::vector<HalfSums> half_sums_at; int64_t half_sums_v = 0, half_sums_n = 0;   // where a layer's sums are in half_sums: a vector's (the first half_sums_v), theta's
  int half_mode = 1;         // 0 never, 1 where a pass is large enough, 2 wherever it can be done
  bool half_usable = true;   // cleared if a copy's memory could not be had
  bool half_now = false;     // the pass in progress works with copies
  uint64_t half_theta_epoch = 0;
  float* small_scratch = nullptr; int64_t small_cap = 0;     // blocks' sums of a small network's pass
  bool small_enabled = true;
  int small_tf32 = -1;         // a TF32 context's passes are all small ones (-1: not looked at yet)
  double* partial = nullptr; int64_t partial_cap = 0;
  // What the host reads at a synchronisation, in one device block with one pinned mirror, so that sync() brings all of
  // it in one copy: scalars ([0] loss, [1] theta^T theta, [4..8] Newton's products), the solver's state, and the error
  // words ([0] gather index error, [1] tensor-core pipeline timeout code).
  struct Status { double scal[16]; CgControl ctl; int err[2]; };
  Status* status = nullptr; Status* h_status = nullptr;
  double* dscal = nullptr; double* hscal = nullptr;      // (into status and h_status, as the pointers below)
  int* err_flag = nullptr; int* h_err = nullptr;
  gn_status sticky = GN_OK;  // a launch-time failure that must surface at the next check
  // CG
  float* cg_r = nullptr; float* cg_p = nullptr; float* cg_q = nullptr;
  CgControl* cg_ctl = nullptr; CgControl* h_ctl = nullptr;   // device-resident solver state and its mirror
  double* cg_hist = nullptr; int cg_hist_cap = 0;            // squared residual norms, one per step
  // One CG step (product + the three vector kernels) as a CUDA graph, for problems small enough that issuing the
  // step's ~20 launches from the host takes as long as running them: captured from the second step of a
  // fixed-length solve and replayed for the rest; kept across solves while nothing it has baked in changes.
  struct CgGraph {
    cudaGraphExec_t exec = nullptr;
    uint64_t alloc_gen = 0, dispatch_gen = 0; int64_t nS = 0; float coef = 0.f; const float* d = nullptr; int stored = 0, method = 0, n_seg = 0;
    int64_t launches = 0;
  };
  CgGraph cg_graph[2];
  bool graph_enabled = true, graph_ok = true;
  int64_t graph_replays = 0;
  bool own_stream = false;     // no stream was given: the context made one (stream capture cannot use the legacy default stream)
  uint64_t alloc_gen = 1;      // bumped by every device allocation and release of the context
  // bumped by whatever sends contractions another way.  A captured step relies on the directly run first step of its
  // solve for what that step leaves behind (split parts of theta and of the activations): it may only be replayed after a
  // first step that went the same way
  uint64_t dispatch_gen = 1;
  float* tmp_a = nullptr; float* tmp_b = nullptr;  // staging for *_host calls
  float* nt[4] = {nullptr, nullptr, nullptr, nullptr};  // Newton iteration: g, d, G d / G dbar, trial theta
  CgChunk* chunks[2] = {nullptr, nullptr}; int n_chunks[2] = {0, 0};
  CgSeg* segs[2] = {nullptr, nullptr}; int64_t segs_cap[2] = {0, 0};   // per-segment scalars: full system, block systems

  // optional per-GEMM timing
  struct EvPair { cudaEvent_t a, b; double flop; int kind; };
  std::vector<EvPair> ev;
  size_t ev_used = 0;
  bool profiling = false;

  int64_t bytes = 0;
  int64_t launches = 0;
  std::string err;
  struct Owned { void* p; int64_t bytes; };
  std::vector<Owned> owned;     // every device allocation of the context with its accounted size
  int fail_alloc_in = 0;        // test hook: the fail_alloc_in-th device allocation from now is refused (0 = off)
};

namespace {

gn_status fail(gn_ctx* c, gn_status s, const std::string& msg) {
  if (c) c->err = msg;
  return s;
}

gn_status cuda_fail(gn_ctx* c, cudaError_t e, const char* where) {
  return fail(c, e == cudaErrorMemoryAllocation ? GN_ENOMEM : GN_ECUDA,
              std::string(where) + ": " + cudaGetErrorString(e));
}

#define GN_CUDA(c, call)                                          \
  do {                                                            \
    cudaError_t e__ = (call);                                     \
    if (e__ != cudaSuccess) return cuda_fail((c), e__, #call);    \
  } while (0)

#define GN_TRY(expr)                      \
  do {                                    \
    gn_status s__ = (expr);               \
    if (s__ != GN_OK) return s__;         \
  } while (0)

constexpr int kCanaryByte = 0xA5;
bool half_release(gn_ctx* c);

template <class T>
gn_status dev_alloc(gn_ctx* c, T** p, int64_t count) {
  *p = nullptr;
  if (count <= 0) count = 1;
  void* q = nullptr;
  for (;;) {
    std::string why;
    if (c->fail_alloc_in > 0 && --c->fail_alloc_in == 0) {
      why = "device allocation of " + std::to_string(count * (int64_t)sizeof(T)) + " bytes refused (injected)";
    } else {
      // 256 bytes of slack: the tensor-core kernel's 3-D TMA boxes may read up to 124 bytes past the last
      // row of an MN-major operand
      const cudaError_t e = cudaMalloc(&q, (size_t)count * sizeof(T) + 256);
      if (e == cudaSuccess) break;
      cudaGetLastError();
      why = "cudaMalloc of " + std::to_string(count * (int64_t)sizeof(T)) + " bytes: " + cudaGetErrorString(e);
    }
    if (!half_release(c)) return fail(c, GN_ENOMEM, why);      // (FP16 copies make room for what is needed)
  }
  // the last 128 bytes of the slack are a canary: nothing of the library may write there (gn_debug_check_canaries)
  if (cudaMemset(static_cast<char*>(q) + (size_t)count * sizeof(T) + 128, kCanaryByte, 128) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(q);
    return fail(c, GN_ECUDA, "cudaMemset of a fresh allocation failed");
  }
  c->bytes += count * (int64_t)sizeof(T);
  ++c->alloc_gen;
  c->owned.push_back({q, count * (int64_t)sizeof(T)});
  *p = static_cast<T*>(q);
  return GN_OK;
}

// Frees a context allocation (null is fine); the accounted size is the one recorded when it was made.
template <class T>
void dev_free(gn_ctx* c, T*& p, int64_t = 0) {
  if (!p) return;
  for (auto& o : c->owned)
    if (o.p == (void*)p) { c->bytes -= o.bytes; o.p = nullptr; o.bytes = 0; break; }
  cudaFree(p);
  p = nullptr;
  ++c->alloc_gen;
  // keep the registry from growing without bound across many regrowths
  if (c->owned.size() > 4096) {
    size_t k = 0;
    for (size_t i = 0; i < c->owned.size(); ++i) if (c->owned[i].p) c->owned[k++] = c->owned[i];
    c->owned.resize(k);
  }
}

gn_status check_launch(gn_ctx* c, const char* where) {
  if (c->sticky != GN_OK) { gn_status s = c->sticky; c->sticky = GN_OK; return s; }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, where);
  return GN_OK;
}

// Side stream: everything enqueued on the main stream so far happens before what follows on the side stream.
cudaStream_t side_fork(gn_ctx* c) {
  if (!c->side_enabled || !c->st2) return c->st;
  cudaEventRecord(c->ev_fork, c->st);
  cudaStreamWaitEvent(c->st2, c->ev_fork, 0);
  c->side_open = true;
  return c->st2;
}
// ... and everything on the side stream so far happens before what follows on the main stream.
void side_join(gn_ctx* c) {
  if (!c->side_open) return;
  cudaEventRecord(c->ev_join, c->st2);
  cudaStreamWaitEvent(c->st, c->ev_join, 0);
  c->side_open = false;
}
// A launch sequence that uses the side stream: inside it, every kernel that works in the side stream's scratch
// buffers (column sums, the n_L-row weight block) goes to the side stream, so those buffers have one user at a
// time; the join happens on every way out.
struct SideJoin {
  gn_ctx* c;
  explicit SideJoin(gn_ctx* ctx) : c(ctx) { c->side_region = true; }
  ~SideJoin() { side_join(c); c->side_region = false; }
};

// The vector of a product in progress (its layers' parts are kept for the length of the product).
struct CurrentVector {
  gn_ctx* c;
  CurrentVector(gn_ctx* ctx, const float* v) : c(ctx) { c->cur_v = v; }
  ~CurrentVector() { c->cur_v = nullptr; }
};

// Before a workspace that side-stream kernels may still read is released.
void quiesce(gn_ctx* c) {
  cudaStreamSynchronize(c->st);
  if (c->st2) cudaStreamSynchronize(c->st2);
}

// Synchronise the stream; also fetch the status block and look at the tensor-core pipeline's timeout word.
gn_status sync(gn_ctx* c, const char* where) {
  cudaError_t e = cudaMemcpyAsync(c->h_status, c->status, sizeof(gn_ctx::Status), cudaMemcpyDeviceToHost, c->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->st);
  if (e != cudaSuccess) return cuda_fail(c, e, where);
  if (c->h_err[1] != 0) {
    const int code = c->h_err[1];
    cudaMemsetAsync(c->err_flag + 1, 0, sizeof(int), c->st);
    // a launch that gave up may have left arrival counts of its K-sliced tiles behind
    if (c->sk_flags) cudaMemsetAsync(c->sk_flags, 0, sizeof(int) * gemm_tf32_workspace_flags(), c->st);
    return fail(c, GN_ETIMEOUT, std::string(where) + ": a bounded wait in the tensor-core pipeline ran out (role " +
                                    std::to_string(code) + "); results are invalid");
  }
  return GN_OK;
}

gn_status ensure_sk_workspace(gn_ctx* c);

void run_gemm_kind(gn_ctx* c, const GemmArgs& g, int kind, cudaStream_t st = nullptr) {
  if (!st) st = c->st;
  gn_ctx::EvPair* e = nullptr;
  if (c->profiling) {
    if (c->ev_used == c->ev.size()) {
      gn_ctx::EvPair p{};
      if (cudaEventCreate(&p.a) == cudaSuccess && cudaEventCreate(&p.b) == cudaSuccess) c->ev.push_back(p);
    }
    if (c->ev_used < c->ev.size()) {
      e = &c->ev[c->ev_used++];
      e->flop = 2.0 * g.M * (double)g.N * ((double)g.K1 + (g.A2 ? (double)g.K2 : 0.0));
      // the one-CTA tensor-core kernel (n_L-wide and small-M shapes, bound by memory) is counted apart from the
      // CTA-pair kernel that carries the large contractions
      e->kind = (kind == 0 && !(g.two_cta >= 0 ? g.two_cta != 0 : (g.M > 128 && g.N >= 128))) ? 4 : kind;
      cudaEventRecord(e->a, st);
    }
  }
  if (kind == 0) {
    ensure_sk_workspace(c);   // first tensor-core launch of this context: stream-K workspace
    const bool sk = c->sk_enabled && g.two_cta != 2;
    GemmArgs g2 = g;
    if (g2.two_cta == 2) g2.two_cta = 1;
    const int r = launch_gemm_tf32(g2, c->err_flag + 1, sk ? c->sk_ws : nullptr, sk ? c->sk_flags : nullptr, st);
    if (r < 0) { c->sticky = GN_ECUDA; c->err = "cuTensorMapEncodeTiled failed"; }
    else c->launches += r;
  } else if (kind == 3) {
    const int r = launch_gemm_f16x3(g, c->h_ops, c->sk_ws, c->err_flag + 1, st);
    if (r < 0) { c->sticky = GN_ECUDA; c->err = "the FP32-accurate tensor-core kernel could not be launched"; c->x3_usable = false; ++c->dispatch_gen; }
    else c->launches += r;
  } else if (kind == 2) {
    c->launches += launch_gemm_thin(g, c->thin_scratch, st);
  } else {
    c->launches += launch_gemm_ffma(g, st);
  }
  if (e) cudaEventRecord(e->b, st);
}

gn_status ensure_sk_workspace(gn_ctx* c) {
  if (!c->sk_ws && c->sk_enabled) {
    if (dev_alloc(c, &c->sk_ws, gemm_tf32_workspace_floats()) != GN_OK ||
        dev_alloc(c, &c->sk_flags, (int64_t)gemm_tf32_workspace_flags()) != GN_OK ||
        cudaMemsetAsync(c->sk_flags, 0, sizeof(int) * gemm_tf32_workspace_flags(), c->st) != cudaSuccess) {
      c->sk_ws = nullptr; c->sk_flags = nullptr; c->sk_enabled = false; ++c->dispatch_gen;
    }
  }
  return c->sk_ws ? GN_OK : GN_ENOMEM;
}

inline int64_t round8(int64_t x) { return (x + 7) & ~(int64_t)7; }

bool split_buf_reserve(gn_ctx* c, gn_ctx::SplitBuf& b, int64_t need) {
  if (need <= b.cap) return true;
  cudaStreamSynchronize(c->st);   // an earlier contraction may still be reading the old buffer
  dev_free(c, b.p);
  b.cap = 0;
  if (dev_alloc(c, &b.p, gn_ctx::SplitBuf::elements(need)) != GN_OK) return false;
  b.cap = need;
  return true;
}

// The parts of kind `kind` (0: of every kind) that have a buffer of their own go, and, with `all`, the whole kind's.
void drop_kept_parts(gn_ctx* c, int kind, bool all) {
  for (size_t i = 0; i < c->split_cache.size();) {
    const gn_ctx::SplitEntry& e = c->split_cache[i];
    if ((kind == 0 || e.kind == kind) && (all || !e.in_arena)) {
      if (!e.in_arena) dev_free(c, c->split_cache[i].buf.p);
      c->split_cache.erase(c->split_cache.begin() + (long)i);
    } else {
      ++i;
    }
  }
  if (!all) return;
  dev_free(c, c->arena[kind]);
  c->arena_rows[kind] = 0;
}

// Buffer of the kept parts of a whole layer's matrix inside the kind's arena: kinds 1 and 3 hold every W^m-shaped
// matrix, kinds 2 and 4 the operands z^0 .. z^{L-1} of the subsample and of the row batch at their workspaces' capacity - on a
// TF32 context only those that TMA cannot address in one of their contractions (the layer's two widths, and where its weights
// start), since nothing else is split there.  False if the matrix has no place there.
bool arena_buffer(gn_ctx* c, int kind, int64_t key, int64_t rows, int cols, int64_t ld, gn_ctx::SplitBuf* out) {
  const bool vec = kind == 1 || kind == 3;
  const int64_t cap_rows = kind == 2 ? c->capS : kind == 4 ? c->capB : 0;
  int64_t total = 0, at = -1, size = 0;
  for (int m = 0; m < c->L; ++m) {
    const int64_t n = vec ? (int64_t)c->w[m + 1] * round8(c->w[m]) : cap_rows * round8(c->w[m]);
    const int64_t k = vec ? c->w_off[m + 1] : (int64_t)m << 48;
    if (c->prec == GN_TF32 && c->w[m] % 4 == 0 && c->w[m + 1] % 4 == 0 && (!vec || c->w_off[m + 1] % 4 == 0)) continue;
    if (key == k && cols == c->w[m] && ld == c->w[m] && rows <= (vec ? c->w[m + 1] : cap_rows)) { at = total; size = n; }
    total += gn_ctx::SplitBuf::elements(n);
  }
  if (at < 0) return false;
  if (!c->arena[kind]) {
    if (dev_alloc(c, &c->arena[kind], total) != GN_OK) return false;
    c->arena_rows[kind] = cap_rows;
  } else if (c->arena_rows[kind] != cap_rows) {
    return false;
  }
  out->p = c->arena[kind] + at; out->cap = size;
  return true;
}

// Place of `src` in a matrix set whose parts are kept (SplitEntry::kind), or 0.  Of the activations only what starts in the
// first row has one: a place per row offset would be one per subsample size.
int split_kind(const gn_ctx* c, const float* src, int64_t* key, uint64_t* epoch) {
  if (src >= c->theta && src < c->theta + c->n) { *key = src - c->theta; *epoch = c->theta_epoch; return 1; }
  for (int m = 0; m <= c->L; ++m)
    if (c->Z[m] && src >= c->Z[m] && src < c->Z[m] + c->w[m]) {
      *key = ((int64_t)m << 48) + (src - c->Z[m]); *epoch = c->sub_epoch;
      return 2;
    }
  *epoch = c->parts_epoch;
  if (c->cur_v && src >= c->cur_v && src < c->cur_v + c->n) { *key = src - c->cur_v; return 3; }
  if (c->cur_x && src >= c->cur_x && src < c->cur_x + c->w[0]) { *key = src - c->cur_x; return 4; }
  for (int m = 1; m <= c->L; ++m)
    if (c->Zb[m] && src >= c->Zb[m] && src < c->Zb[m] + c->w[m]) { *key = ((int64_t)m << 48) + (src - c->Zb[m]); return 4; }
  return 0;
}

// The two FP16 parts of the stored matrix [rows][cols] (leading dimension ld) that serves as an operand: in `out`, with
// the splitting job they still need, if any, appended to `jobs`.  Matrices of the kept kinds are split once per epoch;
// anything else goes through the slot of its operand role (0 = A1, 1 = B1, 2 = A2, 3 = B2) and is split again on every
// use unless the caller vouches (reuse) that the contraction just before this one read this very operand,
// unchanged.  The caller's word is checked: the parts are taken over only if that previous contraction is
// the one that wrote the slot (it may have gone to another kernel and left the slot alone).
constexpr int64_t kMaxTransientSplitFloats = 1500LL * 1000 * 1000;   // 6 GB for both parts

bool split_operand(gn_ctx* c, const float* src, int64_t rows, int cols, int64_t ld, int role, bool reuse,
                   SplitOperand* out, std::vector<SplitJob>& jobs) {
  const int64_t ldo = round8(cols);
  int64_t key = 0;
  uint64_t epoch = 0;
  const int kind = split_kind(c, src, &key, &epoch);
  // (theta and the stored activations are split whatever their size: their parts serve many contractions)
  if (kind != 1 && kind != 2 && rows * ldo > kMaxTransientSplitFloats) return false;
  gn_ctx::SplitBuf* buf = nullptr;
  bool fresh = false;
  if (kind != 0) {
    // one entry per place: a matrix that comes back with another shape (a subsample of another size in the same
    // buffers) replaces the old parts instead of adding to them
    gn_ctx::SplitEntry* e = nullptr;
    for (auto& x : c->split_cache)
      if (x.kind == kind && x.key == key) { e = &x; break; }
    if (!e) {
      if (c->split_cache.size() >= 4096) return false;
      gn_ctx::SplitEntry x{};
      x.kind = kind; x.key = key;
      x.in_arena = arena_buffer(c, kind, key, rows, cols, ld, &x.buf);
      c->split_cache.push_back(x);
      e = &c->split_cache.back();
    }
    // (a caller that captures its calls replays them after theta or the subsample have changed: a graph of the caller's
    // splits everything it reads, and records nothing as split that has not run)
    fresh = !c->foreign_capture && e->epoch == epoch && e->rows == rows && e->cols == cols && e->ld == ld;
    if (!fresh) {
      e->epoch = 0;
      if (rows * ldo > e->buf.cap) {
        if (e->in_arena) { e->buf = gn_ctx::SplitBuf{}; e->in_arena = false; }
        if (!split_buf_reserve(c, e->buf, rows * ldo)) return false;
      }
      e->rows = rows; e->cols = cols; e->ld = ld; e->epoch = c->foreign_capture ? 0 : epoch;
    }
    buf = &e->buf;
  } else {
    gn_ctx::SplitSlot& sl = c->split_slot[role];
    fresh = reuse && sl.seq != 0 && sl.seq + 1 == c->gemm_seq && sl.src == src && sl.rows == rows && sl.cols == cols &&
            sl.ld == ld && sl.buf.p;
    if (!fresh) {
      sl.src = nullptr; sl.seq = 0;
      int64_t want = rows * ldo;
      if (want > sl.buf.cap) {       // (grow at once to what this role will meet in the current workspaces)
        int64_t widest = 0;
        for (int m = 1; m < c->L; ++m) widest = std::max<int64_t>(widest, round8(c->w[m]));
        if (role == 0) want = std::max(want, std::max(c->nS, c->capB) * widest);
        if (!split_buf_reserve(c, sl.buf, want)) return false;
      }
      sl.src = src; sl.rows = rows; sl.cols = cols; sl.ld = ld;
    }
    sl.seq = c->gemm_seq;
    buf = &sl.buf;
  }
  out->hi = buf->p; out->lo = buf->p + buf->cap; out->ld = ldo; out->cells = buf->cells(); out->cells_ld = (cols + 127) / 128;
  if (!fresh) {
    SplitJob j{};
    j.src = src; j.rows = rows; j.cols = cols; j.ld = ld;
    j.hi = buf->p; j.lo = buf->p + buf->cap; j.ld_out = ldo; j.cells = buf->cells();
    jobs.push_back(j);
  }
  return true;
}

void run_splits(gn_ctx* c, const std::vector<SplitJob>& jobs) {
  const size_t together = c->split_together ? kSplitSegs : 1;
  for (size_t i = 0; i < jobs.size(); i += together) {
    const int r = launch_split_f16(jobs.data() + i, (int)std::min<size_t>(together, jobs.size() - i), c->st);
    if (r < 0) { c->sticky = GN_ECUDA; c->err = "an operand could not be split"; return; }
    c->launches += r;
  }
}

// Stored matrices: A is [M][K] (K-major) or [K][M]; B is [N][K] (K-major) or [K][N].
struct OperandView { const float* p; int64_t rows; int cols; int64_t ld; };
OperandView operand_view(const GemmArgs& g, int role) {
  const int K = role < 2 ? g.K1 : g.K2;
  if (role % 2 == 0) {
    const float* p = role == 0 ? g.A1 : g.A2;
    const int64_t ld = role == 0 ? g.lda1 : g.lda2;
    return g.a_kmajor ? OperandView{p, g.M, K, ld} : OperandView{p, K, g.M, ld};
  }
  const float* p = role == 1 ? g.B1 : g.B2;
  const int64_t ld = role == 1 ? g.ldb1 : g.ldb2;
  return g.b_kmajor ? OperandView{p, g.N, K, ld} : OperandView{p, K, g.N, ld};
}

// FP32-accurate contraction on the FP16 tensor cores.  False if it has to go to the FP32 FMA GEMM.  Chunks of 128
// terms (about 4e-7 of the result) on FP32-accurate contexts at the shapes of whole CTA-pair tiles, of 64 terms
// (about 2e-7, below what a chain of K FP32 additions leaves) where the alternative is the FMA GEMM.
bool run_gemm_f16x3(gn_ctx* c, const GemmArgs& args) {
  GemmArgs g = args;
  g.chunk_kb = c->prec == GN_FP32_ACCURATE && g.M > 128 && g.N >= 128 ? 2 : 1;
  if (!c->x3_usable || !gemm_f16x3_usable() || g.K1 < 1 || (g.A2 && g.K2 < 1)) return false;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  c->foreign_capture = !c->own_capture && cudaStreamIsCapturing(c->st, &cap) == cudaSuccess && cap != cudaStreamCaptureStatusNone;
  if (!c->sk_enabled || (gemm_f16x3_workspace_floats(g) > 0 && ensure_sk_workspace(c) != GN_OK)) g.whole_tiles = true;
  std::vector<SplitJob> jobs;
  SplitOperand ops[4];
  for (int role = 0; role < (g.A2 ? 4 : 2); ++role) {
    const OperandView v = operand_view(g, role);
    if (!split_operand(c, v.p, v.rows, v.cols, v.ld, role, role == 0 && g.a1_split_fresh, &ops[role], jobs)) {
      run_splits(c, jobs);                       // (what has been recorded as split must be)
      return false;
    }
  }
  run_splits(c, jobs);
  for (int k = 0; k < 4; ++k) c->h_ops[k] = ops[k];
  run_gemm_kind(c, g, 3);
  return true;
}

// Whether the tensor-core form is the faster way to FP32 accuracy.  The FP32 FMA GEMM walks K alone in 128 x 128
// tiles: about 10 us plus 0.12 us per unit of K and round of tiles (17 us at K = 37, 53 at 333).  The tensor-core form
// pays for splitting its operands before it starts (a launch, 4 to 6 us, and its bytes) and about 6 us of ramp; the 14 us
// charged here date from when a split took two launches, so the line lies a little on the FMA GEMM's side.
bool wants_f16x3(const gn_ctx* c, const GemmArgs& g) {
  if (!c->x3_usable || !gemm_f16x3_usable()) return false;
  if (c->prec == GN_FP32_ACCURATE && c->acc_method == 1) return false;
  const double K = (double)g.K1 + (g.A2 ? g.K2 : 0);
  const double blocks = ((g.M + 127) / 128) * (double)((g.N + 127) / 128);
  const double rounds = blocks <= 148.0 ? 1.0 : blocks / 148.0;
  const double fma_us = 10.0 + rounds * K * 0.12;
  return gemm_f16x3_estimate_us(g) + 14.0 + (g.M + (double)g.N) * K * 8.0 / 4.0e6 * 0.5 < fma_us;
}

// Whether a contraction goes to the TF32 kernels: on a TF32 context every one whose operands TMA can address, whatever its
// sizes.  The gradient (K or M up to a row batch) and the products (|S|) of one solve have to round the same operator (see
// small_pass); with the weight blocks of narrow layers in FP32 accuracy from some K on, as an earlier rule had it, they did not
// (300-120-80-40: the 80 x 120 block above about 1150 rows).
bool on_tf32(const gn_ctx* c, const GemmArgs& g) { return c->prec == GN_TF32 && gemm_tf32_eligible(g); }

// Whether run_gemm will send a contraction to that form.
bool goes_f16x3(const gn_ctx* c, const GemmArgs& g) {
  return gemm_thin_kind(g) == THIN_NONE && !on_tf32(c, g) && wants_f16x3(c, g);
}

// Kernel choice: streaming kernels for the n_L-wide shapes (both precisions: they are exact FP32), the TF32
// tensor-core kernel in TF32 mode when TMA can address the operands; everything else is computed to FP32 accuracy, by
// the FP16 tensor-core kernel or the FP32 FMA GEMM, whichever is the faster at that size.
void run_gemm(gn_ctx* c, const GemmArgs& g, cudaStream_t st = nullptr) {
  ++c->gemm_seq;
  const ThinKind thin = gemm_thin_kind(g);
  // In TF32 mode the n_L-wide forward products go to the tensor-core kernel as one 32- or 64-column
  // tile: TMA streams A about 2.5x faster than the SIMT streaming kernel does (measured) - once there are enough
  // 128-row tiles to occupy the SMs; below 48 tiles (a CTA walks its whole K range alone, 53 us at K = 4000 whatever
  // the row count) the streaming kernel, one warp per four rows, is the faster one (3000 rows: 3-4 % of a product).
  const bool thin_n_on_tensor = thin == THIN_N && c->prec == GN_TF32 && gemm_tf32_eligible(g) && g.M >= 48 * 128;
  if (thin != THIN_NONE && !thin_n_on_tensor) {
    const int64_t need = gemm_thin_scratch_floats(g);
    if (need > c->thin_cap) {
      quiesce(c);
      dev_free(c, c->thin_scratch, c->thin_cap);
      c->thin_cap = 0;
      if (dev_alloc(c, &c->thin_scratch, need) != GN_OK) { c->sticky = GN_ENOMEM; return; }
      c->thin_cap = need;
    }
    // the n_L-row weight block streams its operands once and shares nothing with the layer's other contraction
    if (thin == THIN_M && c->side_region && !st) st = side_fork(c);
    run_gemm_kind(c, g, 2, st);
    return;
  }
  if (on_tf32(c, g)) { run_gemm_kind(c, g, 0, st); return; }
  if (!st && wants_f16x3(c, g) && run_gemm_f16x3(c, g)) return;
  run_gemm_kind(c, g, 1, st);
}

// The parts of the operands in `roles` (bit per role) of several contractions that will go to the FP32-accurate
// tensor-core kernel, in one splitting launch instead of one per contraction.  Kept kinds only.
void presplit(gn_ctx* c, const GemmArgs* gs, int n, unsigned roles) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (!c->own_capture && cudaStreamIsCapturing(c->st, &cap) == cudaSuccess && cap != cudaStreamCaptureStatusNone) return;
  c->foreign_capture = false;
  std::vector<SplitJob> jobs;
  for (int i = 0; i < n; ++i) {
    const GemmArgs& g = gs[i];
    if (!goes_f16x3(c, g)) continue;
    for (int role = 0; role < (g.A2 ? 4 : 2); ++role) {
      const OperandView v = operand_view(g, role);
      int64_t key = 0;
      uint64_t epoch = 0;
      SplitOperand op;
      if ((roles >> role & 1) && split_kind(c, v.p, &key, &epoch) != 0) split_operand(c, v.p, v.rows, v.cols, v.ld, role, false, &op, jobs);
    }
  }
  run_splits(c, jobs);
}

// ---- FP16 copies ---------------------------------------------------------------------------------
using HalfBuf = gn_ctx::HalfBuf;

int half_info_index(const gn_ctx* c, int set, int m) { return set * (c->L + 1) + m; }

bool half_setup(gn_ctx* c) {
  if (c->half_info) return true;
  const int64_t n = (int64_t)gn_ctx::kHalfSets * (c->L + 1);
  if (dev_alloc(c, &c->half_info, n) != GN_OK) return false;
  c->half_at.assign((size_t)c->L + 2, 0);
  for (int m = 1; m <= c->L; ++m) c->half_at[(size_t)m + 1] = c->half_at[(size_t)m] + c->w[m] * round8(c->w[m - 1]);
  c->half_sums_at.assign((size_t)c->L + 1, {});
  c->half_sums_n = 0;
  for (int m = 1; m <= c->L; ++m) { c->half_sums_at[(size_t)m].v_rows = c->half_sums_n; c->half_sums_n += c->w[m]; }
  c->half_sums_v = c->half_sums_n;
  for (int m = 1; m <= c->L; ++m) {
    c->half_sums_at[(size_t)m].rows = c->half_sums_n;
    c->half_sums_at[(size_t)m].cols = c->half_sums_n + c->w[m];
    c->half_sums_n += c->w[m] + c->w[m - 1];
  }
  if (dev_alloc(c, &c->half_acc, (int64_t)kHalfSegs + 1) != GN_OK || dev_alloc(c, &c->half_weights, 2 * c->half_at.back()) != GN_OK ||
      dev_alloc(c, &c->half_sums, c->half_sums_n) != GN_OK) {
    dev_free(c, c->half_weights); dev_free(c, c->half_acc); dev_free(c, c->half_info);
    return false;
  }
  cudaMemsetAsync(c->half_info, 0, sizeof(HalfInfo) * (size_t)n, c->st);
  cudaMemsetAsync(c->half_acc, 0, sizeof(unsigned) * (kHalfSegs + 1), c->st);
  return true;
}

// Where the copy of entry m of a set has its place in memory that is there anyway: weights and vectors in theirs, and in FP32
// memory of the context that holds nothing meanwhile, with as many rows and columns: a copy of R z^m is read before delta s^m is
// written, and one of delta s^m is written when R z^m has been read for the last time.
uint16_t* half_lender(const gn_ctx* c, int set, int m) {
  if (set == gn_ctx::kHW) return c->half_weights + c->half_at[(size_t)m];
  if (set == gn_ctx::kHV) return c->half_weights + c->half_at.back() + c->half_at[(size_t)m];
  if (m < 1 || m >= c->L) return nullptr;
  return reinterpret_cast<uint16_t*>(set == gn_ctx::kHRZ ? c->DS[(size_t)m] : set == gn_ctx::kHDS ? c->RZ[(size_t)m] : nullptr);
}

// Room for a copy of a rows x cols matrix at `base` (copy: it will have one, and not an info alone).
bool half_reserve(gn_ctx* c, HalfBuf& b, int set, int m, const float* base, int64_t rows, int cols, int64_t cap_rows, bool copy = true) {
  if (!half_setup(c)) return false;
  const int64_t need = copy ? std::max(rows, cap_rows) * round8(cols) : 0;
  if (uint16_t* lent = half_lender(c, set, m)) {
    b.p = lent;
  } else if (need > b.cap) {
    if (b.cap > 0) { quiesce(c); dev_free(c, b.p); }
    b.p = nullptr; b.cap = 0; b.valid = false;
    if (dev_alloc(c, &b.p, need) != GN_OK) return false;
    b.cap = need;
  }
  b.base = base; b.rows = rows; b.cols = cols; b.info = half_info_index(c, set, m);
  b.valid = b.info_valid = false;
  return true;
}

void half_invalidate(gn_ctx* c, int set) {
  for (auto& b : c->half_buf[set]) { b.base = nullptr; b.valid = b.info_valid = false; }
}
void half_drop(gn_ctx* c, int set) {
  for (auto& b : c->half_buf[set]) {
    if (b.cap > 0) dev_free(c, b.p);
    b.p = nullptr; b.cap = 0; b.base = nullptr; b.valid = b.info_valid = false;
  }
}
// No room: the passes go on without copies until the next subsample, whose memory may be another.
void half_give_up(gn_ctx* c) {
  quiesce(c);
  for (int set = 0; set < gn_ctx::kHalfSets; ++set) half_drop(c, set);
  dev_free(c, c->half_weights); dev_free(c, c->half_sums); dev_free(c, c->half_acc); dev_free(c, c->half_info);
  c->half_usable = false; c->half_now = false; c->half_theta_epoch = 0; ++c->dispatch_gen;
}
// Something that a call cannot do without has found no room: whether copies could be let go for it.  (Not inside a pass with
// copies, whose operands point to them: or_without_copies is for that.)
bool half_release(gn_ctx* c) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (!c->half_info || c->half_now) return false;
  if (cudaStreamIsCapturing(c->st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return false;
  half_give_up(c);
  return true;
}
// A pass, and once more without copies if it has run out of memory with them.
template <class Pass>
gn_status or_without_copies(gn_ctx* c, Pass pass) {
  const gn_status s = pass();
  return s == GN_ENOMEM && half_release(c) ? pass() : s;
}

HalfMat half_mat(const gn_ctx* c, const HalfBuf& b) {
  HalfMat h;
  h.p = b.p; h.ld = round8(b.cols); h.info = c->half_info + b.info;
  return h;
}
// The copy of the matrix at `src` with leading dimension ld, possibly a part of a larger one that starts on a copy's 16 bytes.
bool half_find(const gn_ctx* c, const float* src, int64_t ld, HalfMat* out, bool info_only) {
  for (int set = 0; set < gn_ctx::kHalfSets; ++set)
    for (const HalfBuf& b : c->half_buf[set]) {
      if (!(info_only ? b.info_valid : b.valid) || b.cols != ld || src < b.base || src >= b.base + b.rows * b.cols) continue;
      const int64_t off = src - b.base, r = off / ld, col = off - r * ld;
      if (!info_only && col % 8 != 0) return false;
      *out = half_mat(c, b);
      out->p = info_only ? nullptr : b.p + r * out->ld + col;
      return true;
    }
  return false;
}

bool suits_half(const GemmArgs& g) {
  return gemm_thin_kind(g) == THIN_NONE && g.M > 128 && g.N >= 128 && g.two_cta != 0 && gemm_tf32_eligible(g);
}
// The streaming kernel of a short K reads FP32 and can write its result's copy.
bool thin_with_copy(const GemmArgs& g) { return gemm_thin_kind(g) == THIN_K && !g.bias && !g.cin && !g.sigmoid; }
// The copies of a contraction's operands, if it can be computed from them and all are there.
void attach_half(const gn_ctx* c, GemmArgs& g) {
  if (!c->half_now) return;
  if (thin_with_copy(g)) {                  // (what bounds its result)
    if (!half_find(c, g.A1, g.lda1, &g.h[0], true) || !half_find(c, g.B1, g.ldb1, &g.h[1], true)) g.h[0] = g.h[1] = HalfMat{};
    return;
  }
  if (!suits_half(g)) return;
  bool all = true;
  for (int role = 0; role < (g.A2 ? 4 : 2); ++role) {
    const float* p = role == 0 ? g.A1 : role == 1 ? g.B1 : role == 2 ? g.A2 : g.B2;
    const int64_t ld = role == 0 ? g.lda1 : role == 1 ? g.ldb1 : role == 2 ? g.lda2 : g.ldb2;
    if (!half_find(c, p, ld, &g.h[role], false)) {
      all = false;
      if (!half_find(c, p, ld, &g.h[role], true)) g.h[role] = HalfMat{};
    }
  }
  g.half = all;
}
// ... and the copy of its result, which it writes (attach_half comes first).  The result is the matrix of `b`.
void attach_half_out(const gn_ctx* c, GemmArgs& g, HalfBuf& b) {
  b.valid = b.info_valid = false;
  if (!c->half_now || !(suits_half(g) || thin_with_copy(g)) || !b.p || b.base != g.D || b.cols != g.ldd) return;
  for (int role = 0; role < (g.A2 ? 4 : 2); ++role)
    if (!g.h[role].info) return;
  g.hout = half_mat(c, b);
  b.valid = b.info_valid = true;
}

// Copies by passes of their own.  infos: one largest-magnitude job per scale; every matrix of `bufs` is then copied.  The infos
// from `reset` on are cleared on the way.
// (With no such job the infos hold what the matrices' writers have reported.)
// set: kHW or kHV, whose copies' rows (and, of theta, columns) are summed as well: they bound what is computed from them.
bool half_convert(gn_ctx* c, const std::vector<HalfAmaxJob>& amax, const std::vector<HalfBuf*>& bufs, int reset = 0, int n_reset = 0,
                  int set = gn_ctx::kHalfSets) {
  const bool theta = set == gn_ctx::kHW, vec = set == gn_ctx::kHV;
  unsigned long long* const sums = c->half_sums + (theta ? c->half_sums_v : 0);
  const int64_t n_sums = theta ? c->half_sums_n - c->half_sums_v : vec ? c->half_sums_v : 0;
  for (size_t i = 0; i < amax.size(); i += kHalfSegs) {
    const int r = launch_half_amax(amax.data() + i, (int)std::min<size_t>(kHalfSegs, amax.size() - i), c->half_acc, c->half_info + reset, i == 0 ? n_reset : 0, sums, i == 0 ? n_sums : 0, c->st);
    if (r < 0) { c->sticky = GN_ECUDA; c->err = "FP16 copies could not be made"; return false; }
    c->launches += r;
  }
  std::vector<HalfCopyJob> jobs;
  for (HalfBuf* b : bufs) {
    HalfCopyJob j{b->base, b->rows, b->cols, (int64_t)b->cols, half_mat(c, *b), amax.empty()};
    if (theta || vec) {
      const gn_ctx::HalfSums& at = c->half_sums_at[(size_t)(b->info - half_info_index(c, set, 0))];
      j.row_sums = c->half_sums + (theta ? at.rows : at.v_rows);
      if (theta) j.col_sums = c->half_sums + at.cols;
      if (vec) j.from = c->half_info + half_info_index(c, set, 0);
    }
    jobs.push_back(j);
  }
  for (size_t i = 0; i < jobs.size(); i += kHalfSegs) {
    const int r = launch_half_copy(jobs.data() + i, (int)std::min<size_t>(kHalfSegs, jobs.size() - i), c->st);
    if (r < 0) { c->sticky = GN_ECUDA; c->err = "FP16 copies could not be made"; return false; }
    c->launches += r;
  }
  for (HalfBuf* b : bufs) b->valid = b->info_valid = true;
  return true;
}

// Layers whose weights are an operand of a contraction that suits_half.
bool half_layer(const gn_ctx* c, int m) { return c->w[m] >= 128 && c->w[m] % 4 == 0 && c->w[m - 1] % 4 == 0 && c->w_off[m] % 4 == 0; }
// Whether a pass over `rows` rows is to work with copies.  They cost launches of their own (v, X, the output layer's delta), bytes
// that grow with the weights, and the chained form of the pass; what they save grows with the rows times the weights.  Times with
// copies over times without, network (weights), at 2000 / 4000 / 8000 / 16000 rows; theta new in every pass for f and the gradient:
//                               full product           stored-factor product  gradient               f
//   784-500-500-10 (0.65e6)     .97 1.12 1.05 .82      1.05 .94 .88 .83       1.03 1.14 1.05 .87     1.27 1.22 1.11 1.22
//   784-800-800-10 (1.3e6)      .93 1.08  .97 .81      1.08 .97 .93 .90        .99 1.09 1.01 .86     1.12 1.12 1.14 1.13
//   784-1000x3-10 (2.8e6)       .93 1.09  .85 .79      1.09 1.07 .99 .92      1.00 1.09  .84 .77     1.08 1.13 1.09 1.01
//   3072-1000-1000-10 (4.1e6)   .99 1.08  .86 .81      1.02 .96 .87 .90        .97 1.01  .94 .89     1.13 1.10 1.13 1.11
//   784-2000x3-10 (9.6e6)      1.02  .85  .87 .78      1.00 .95 .92 .89       1.07  .86  .80 .78     1.13  .99  .89  .83
//   1024-4096x4-100 (55e6)      .85  .76               -                       .86  .75              1.00  .86
// (at 1000 and 500 rows of the last: 0.94 and 1.12 for the product, 1.19 and 1.20 for f.)  But for block products, where all layers have
// as many contractions (784-1000-16 at 12000 rows: 0.84), the first layer counts half: it has half of the others', and a copy of X to pay
// for (288-2200-59 at 26013 rows: 1.04).
enum HalfKind { kHalfStored, kHalfProduct, kHalfGrad, kHalfFun };   // block products through stored factors; full product, factors; ...
bool half_pays(HalfKind kind, double rows, double weights) {
  if (weights < (kind == kHalfStored ? 5e5 : 4e5)) return false;
  if (kind == kHalfFun) return rows * weights >= 6.5e10;
  return rows >= (kind == kHalfStored ? 3000.0 : 12000.0) || (rows >= 1000.0 && rows * weights >= 1.8e10);
}
bool half_wanted(gn_ctx* c, int64_t rows, HalfKind kind) {
  if (c->prec != GN_TF32 || c->half_mode == 0 || !c->half_usable || rows <= 128 || c->L < 2) return false;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  // (what a caller captures is replayed after theta has changed: such a graph reads the FP32 matrices)
  if (!c->own_capture && cudaStreamIsCapturing(c->st, &cap) == cudaSuccess && cap != cudaStreamCaptureStatusNone) return false;
  double weights = 0.0;
  for (int m = 1; m <= c->L; ++m)
    if (half_layer(c, m)) weights += (m == 1 && kind != kHalfStored ? 0.5 : 1.0) * c->w[m - 1] * c->w[m];
  return weights > 0.0 && (c->half_mode == 2 || half_pays(kind, (double)rows, weights));
}
// A pass that works with copies, or not.  What is known at its end beyond theta and the stored activations is forgotten: a copy is
// found by the address of its matrix, and the next pass may meet another matrix there (of the caller, or in memory that the
// context has let go and got again).
struct HalfPass {
  gn_ctx* c;
  HalfPass(gn_ctx* ctx, bool on) : c(ctx) { c->half_now = on; }
  ~HalfPass() {
    c->half_now = false;
    for (int set = 0; set < gn_ctx::kHalfSets; ++set)
      if (set != gn_ctx::kHZ && set != gn_ctx::kHW) half_invalidate(c, set);
  }
};

// theta's weights, once per theta.
void half_theta(gn_ctx* c) {
  if (!c->half_now || c->half_theta_epoch == c->theta_epoch) return;
  std::vector<HalfAmaxJob> amax;
  std::vector<HalfBuf*> bufs;
  half_invalidate(c, gn_ctx::kHW);
  for (int m = 1; m <= c->L; ++m) {
    HalfBuf& b = c->half_buf[gn_ctx::kHW][(size_t)m];
    const bool copy = half_layer(c, m) || (c->w[m - 1] >= 128 && c->w[m] > 16 && c->w[m] % 4 == 0 && c->w[m - 1] % 4 == 0 && c->w_off[m] % 4 == 0);
    // (of the output layer's weights at least the largest magnitude, which bounds the last hidden layer's delta)
    if (!copy && m < c->L) continue;
    if (!half_reserve(c, b, gn_ctx::kHW, m, c->theta + c->w_off[m], c->w[m], c->w[m - 1], 0)) { half_give_up(c); return; }
    amax.push_back(HalfAmaxJob{b.base, b.rows * b.cols, c->half_info + b.info});
    if (copy) bufs.push_back(&b);
  }
  if (!half_convert(c, amax, bufs, 0, 0, gn_ctx::kHW)) return;
  c->half_buf[gn_ctx::kHW][(size_t)c->L].info_valid = true;
  c->half_theta_epoch = c->theta_epoch;
}

// The vector of a product; the infos of what the product computes start afresh.
void half_vector(gn_ctx* c, const float* v) {
  if (!c->half_now) return;
  std::vector<HalfBuf*> bufs;
  for (int m = 1; m <= c->L; ++m) {
    if (!half_layer(c, m)) continue;
    HalfBuf& b = c->half_buf[gn_ctx::kHV][(size_t)m];
    if (!half_reserve(c, b, gn_ctx::kHV, m, v + c->w_off[m], c->w[m], c->w[m - 1], 0)) { half_give_up(c); return; }
    bufs.push_back(&b);
  }
  const std::vector<HalfAmaxJob> amax{HalfAmaxJob{v, c->n, c->half_info + half_info_index(c, gn_ctx::kHV, 0)}};
  // (one scale for all of v: that of entry 0, which the layers' infos take over)
  half_convert(c, amax, bufs, half_info_index(c, gn_ctx::kHV, 1), 3 * (c->L + 1) - 1, gn_ctx::kHV);
}

// A copy of one matrix that something else than a contraction with a copy of its own has written.
void half_matrix(gn_ctx* c, int set, int m, const float* base, int64_t rows, int cols, int64_t cap_rows, bool copy, int reset = 0, int n_reset = 0) {
  if (!c->half_now) return;
  HalfBuf& b = c->half_buf[set][(size_t)m];
  if (!half_reserve(c, b, set, m, base, rows, cols, cap_rows, copy)) { half_give_up(c); return; }
  std::vector<HalfBuf*> bufs;
  if (copy) bufs.push_back(&b);
  if (half_convert(c, {HalfAmaxJob{base, rows * cols, c->half_info + b.info}}, bufs, reset, n_reset)) b.info_valid = true;
}

// Room for the copies of the layers' matrices `mats` (1 .. top) that a pass over `rows` rows writes.
bool half_room(gn_ctx* c, int set, const std::vector<float*>& mats, int top, int64_t rows, int64_t cap_rows) {
  if (!c->half_now) return false;
  for (int m = 1; m <= top; ++m)
    if (c->w[m] >= 128 && c->w[m] % 4 == 0 &&
        !half_reserve(c, c->half_buf[set][(size_t)m], set, m, mats[(size_t)m], rows, c->w[m], cap_rows)) { half_give_up(c); return false; }
  return true;
}

// Independent contractions issued together (any order is allowed).  In TF32 mode those that suit the CTA-pair
// kernel go out in launches of up to three problems with a common work list (the tiles of one fill the partial
// last wave of another); everything else runs one after the other, in the order given.
void run_gemm_group(gn_ctx* c, const GemmArgs* gs, int n) {
  constexpr int kMax = 3;      // (more than three independent problems per launch gained nothing measurable)
  bool taken[16] = {false};
  if (n >= 2 && n <= 16 && c->prec == GN_TF32 && c->group_enabled) {
    GemmArgs pick[kMax];
    int idx[kMax], np = 0;
    auto flush = [&]() {
      if (np >= 2 && gemm_tf32_group_eligible(pick, np)) {
        c->gemm_seq += (uint64_t)np;
        gn_ctx::EvPair* e = nullptr;
        if (c->profiling) {
          if (c->ev_used == c->ev.size()) {
            gn_ctx::EvPair p{};
            if (cudaEventCreate(&p.a) == cudaSuccess && cudaEventCreate(&p.b) == cudaSuccess) c->ev.push_back(p);
          }
          if (c->ev_used < c->ev.size()) {
            e = &c->ev[c->ev_used++];
            e->flop = 0.0;
            for (int i = 0; i < np; ++i)
              e->flop += 2.0 * pick[i].M * (double)pick[i].N * ((double)pick[i].K1 + (pick[i].A2 ? (double)pick[i].K2 : 0.0));
            e->kind = 0;
            cudaEventRecord(e->a, c->st);
          }
        }
        const int r = launch_gemm_tf32_group(pick, np, nullptr, nullptr, nullptr, 0, c->err_flag + 1, c->st);
        if (r < 0) { c->sticky = GN_ECUDA; c->err = "cuTensorMapEncodeTiled failed"; }
        else c->launches += r;
        if (e) cudaEventRecord(e->b, c->st);
        for (int i = 0; i < np; ++i) taken[idx[i]] = true;
      }
      np = 0;
    };
    for (int i = 0; i < n; ++i) {
      if (gemm_thin_kind(gs[i]) != THIN_NONE || !gemm_tf32_group_eligible(&gs[i], 1)) continue;
      pick[np] = gs[i]; idx[np] = i; ++np;
      if (np == kMax) flush();
    }
    flush();
  }
  presplit(c, gs, n, 0xf);
  for (int i = 0; i < n; ++i)
    if (i >= 16 || !taken[i]) run_gemm(c, gs[i]);
}

// (the new buffer is obtained before the old one is let go: the solver and the dot products use c->partial
// without asking for it again, so a refused allocation must leave the old buffer in place)
// The layers of a pass, each reading what the one before it writes (dep[i] = index of that earlier problem, -1 for
// none; dep_all[i]: it reads all of that output, not just the rows of its own tile).  In TF32 mode a run of
// consecutive problems that suit the CTA-pair kernel goes out as ONE launch in which a tile starts as soon as the
// tiles it reads are stored, so a layer's first tiles run beside the previous layer's last ones; everything else
// runs one after the other, in the order given (which is a valid order by construction).
void run_gemm_chain(gn_ctx* c, const GemmArgs* gs, const int* dep, const int* dep_all, int n, int level = 1) {
  int i = 0;
  while (i < n) {
    int j = i;
    if (c->prec == GN_TF32 && c->chain_level >= level) {
      while (j < n && j - i < kGemmGroupMax && gemm_thin_kind(gs[j]) == THIN_NONE && gemm_tf32_group_eligible(&gs[j], 1)) ++j;
    }
    if (j - i >= 2) {
      const int cnt = j - i;
      int64_t panels = 0;
      for (int k = i; k < j; ++k) panels = std::max<int64_t>(panels, (gs[k].M + 255) / 256);
      const int stride = (int)panels + 1;
      if (!c->chain_ctr || (int64_t)kGemmGroupMax * stride > c->chain_ctr_cap) {
        quiesce(c);
        dev_free(c, c->chain_ctr);
        c->chain_ctr_cap = 0;
        if (dev_alloc(c, &c->chain_ctr, (int64_t)kGemmGroupMax * stride) == GN_OK) c->chain_ctr_cap = (int64_t)kGemmGroupMax * stride;
      }
      int ldep[kGemmGroupMax], lall[kGemmGroupMax];
      // (what an earlier launch wrote is complete by stream order: no dependency inside this launch)
      for (int k = 0; k < cnt; ++k) { ldep[k] = dep[i + k] < i ? -1 : dep[i + k] - i; lall[k] = dep_all[i + k]; }
      if (c->chain_ctr) {
        gn_ctx::EvPair* e = nullptr;
        if (c->profiling) {
          if (c->ev_used == c->ev.size()) {
            gn_ctx::EvPair pnew{};
            if (cudaEventCreate(&pnew.a) == cudaSuccess && cudaEventCreate(&pnew.b) == cudaSuccess) c->ev.push_back(pnew);
          }
          if (c->ev_used < c->ev.size()) {
            e = &c->ev[c->ev_used++];
            e->flop = 0.0;
            for (int k = i; k < j; ++k)
              e->flop += 2.0 * gs[k].M * (double)gs[k].N * ((double)gs[k].K1 + (gs[k].A2 ? (double)gs[k].K2 : 0.0));
            e->kind = 0;
            cudaEventRecord(e->a, c->st);
          }
        }
        const int r = launch_gemm_tf32_group(gs + i, cnt, ldep, lall, c->chain_ctr, stride, c->err_flag + 1, c->st);
        if (e) cudaEventRecord(e->b, c->st);
        if (r >= 0) {
          c->launches += r + 1;             // (the clearing of the counters counts as a launch)
          c->gemm_seq += (uint64_t)cnt;
          i = j;
          continue;
        }
        if (e) --c->ev_used;                // nothing was launched: drop the event pair
      }
    }
    run_gemm(c, gs[i]);
    ++i;
  }
}

gn_status ensure_partials(gn_ctx* c, int64_t count) {
  if (count <= c->partial_cap) return GN_OK;
  double* fresh = nullptr;
  GN_TRY(dev_alloc(c, &fresh, count));
  cudaStreamSynchronize(c->st);
  dev_free(c, c->partial);
  c->partial = fresh;
  c->partial_cap = count;
  return GN_OK;
}

// Scratch of the column sums: two slots of equal size (slot 1 starts at colsum_cap / 2), so that the sums of two
// layers can run at the same time on two streams.
gn_status ensure_colsum(gn_ctx* c, int64_t rows, int cols) {
  const int64_t need = 2 * ((colsum_scratch_floats(rows, cols) + 3) / 4 * 4);
  if (need <= c->colsum_cap) return GN_OK;
  quiesce(c);
  dev_free(c, c->colsum_scratch, c->colsum_cap);
  c->colsum_cap = 0;
  GN_TRY(dev_alloc(c, &c->colsum_scratch, need));
  c->colsum_cap = need;
  return GN_OK;
}

// Whole passes of a small network in one launch (small_net.cu): the description for `rows` rows, and whether the pass
// is to go that way.
enum SmallKind { kSmallGv = 0, kSmallBlock = 1, kSmallGrad = 2, kSmallFun = 3, kSmallForward = 4 };
bool small_pass(gn_ctx* c, SmallKind kind, int64_t rows, SmallNet* a) {
  if (!c->small_enabled || c->L > kSmallLayers || c->n > 60000) return false;
  *a = SmallNet{};
  a->L = c->L; a->n = (int)c->n; a->rows = rows;
  for (int m = 0; m <= c->L; ++m) a->w[m] = c->w[m];
  for (int m = 1; m <= c->L; ++m) { a->w_off[m] = (int)c->w_off[m]; a->b_off[m] = (int)c->b_off[m]; }
  a->theta = c->theta;
  if (c->prec != GN_TF32) return small_net_fits(*a, kind);
  // On a TF32 context all passes go this way or none: the gradient and the products of one solve have to round the
  // same operator.  An exact gradient beside TF32 products (or the other way round) leaves an error in the first residual
  // that is not along the gradient, and conjugate gradient amplifies it (96-100-50-200-1: iterates off by 1.4e-3 instead
  // of 1e-4 although every single result was the more accurate one).
  if (c->has_split || c->bd_method == 2) return false;
  if (c->small_tf32 < 0) {
    SmallNet all = *a;
    all.rows = c->l;
    c->small_tf32 = 1;
    for (int k = kSmallGv; k <= kSmallForward; ++k)
      if (!small_net_fits(all, k)) c->small_tf32 = 0;
  }
  return c->small_tf32 && (rows <= c->l || small_net_fits(*a, kind));
}

gn_status run_small_pass(gn_ctx* c, SmallKind kind, SmallNet& a, float alpha, const float* cin, float beta, float* out, double* loss_out) {
  if (kind != kSmallForward) {
    const int64_t blocks = small_net_blocks(a.rows);
    const int64_t need = (blocks * 2 + 3) / 4 * 4 + blocks * a.n;            // the losses (doubles), then the sums
    if (need > c->small_cap) {
      quiesce(c);
      dev_free(c, c->small_scratch);
      c->small_cap = 0;
      GN_TRY(dev_alloc(c, &c->small_scratch, need));
      c->small_cap = need;
    }
    a.loss = reinterpret_cast<double*>(c->small_scratch);
    a.scratch = c->small_scratch + (blocks * 2 + 3) / 4 * 4;
  }
  const int r = launch_small_net(a, kind, alpha, cin, beta, out, loss_out, c->st);
  if (r < 0) return fail(c, GN_ECUDA, "the small network's pass could not be launched");
  c->launches += r;
  return GN_OK;
}

// First neuron of group g when a layer of n neurons is cut into `groups` contiguous groups.
int group_lo(int n, int groups, int g) { return (int)(((long long)g * n) / groups); }

const float* Wm(const gn_ctx* c, const float* vec, int m) { return vec + c->w_off[m]; }
const float* bm(const gn_ctx* c, const float* vec, int m) { return vec + c->b_off[m]; }

// Eq. (xtoz): Zout[m] = sigma(Zout[m-1] W^m + 1 b^mT), m = 1..L, over `rows` rows; Zout[0] = Z0.
// With copies (half_now): of Z0 as `set`'s entry 0, of the Z_m, all written here; cap_rows as of the buffers Zout.
void forward_pass(gn_ctx* c, const float* Z0, int64_t rows, std::vector<float*>& Zout, int set, int64_t cap_rows) {
  half_theta(c);
  half_invalidate(c, set);
  if (c->half_now) {
    // infos of what is about to be written, to be cleared: of Z_1 .. Z_L, and of a batch's deltas, which follow
    const int reset = half_info_index(c, set, 1), n_reset = set == gn_ctx::kHZb ? 2 * c->L + 1 : c->L;
    if (half_layer(c, 1)) half_matrix(c, set, 0, Z0, rows, c->w[0], cap_rows, true, reset, n_reset);
    else cudaMemsetAsync(c->half_info + reset, 0, sizeof(HalfInfo) * (size_t)n_reset, c->st);
    // (z^{L-1} is an operand of the output layer's contractions alone)
    half_room(c, set, Zout, half_layer(c, c->L) ? c->L - 1 : c->L - 2, rows, cap_rows);
  }
  std::vector<GemmArgs> gs((size_t)c->L);
  std::vector<int> dep((size_t)c->L), dep_all((size_t)c->L, 0);
  for (int m = 1; m <= c->L; ++m) {
    GemmArgs& g = gs[(size_t)m - 1];
    g.M = (int)rows; g.N = c->w[m];
    g.A1 = m == 1 ? Z0 : Zout[m - 1]; g.lda1 = c->w[m - 1];
    g.B1 = Wm(c, c->theta, m); g.ldb1 = c->w[m - 1]; g.K1 = c->w[m - 1];
    g.a_kmajor = true; g.b_kmajor = true;
    g.D = Zout[m]; g.ldd = c->w[m];
    g.bias = bm(c, c->theta, m);
    g.sigmoid = m < c->L;
    attach_half(c, g);
    if (m < c->L) attach_half_out(c, g, c->half_buf[set][(size_t)m]);
    dep[(size_t)m - 1] = m - 2;          // layer m reads the rows layer m - 1 writes
  }
  presplit(c, gs.data(), c->L, 0x2);       // theta's weights
  run_gemm_chain(c, gs.data(), dep.data(), dep_all.data(), c->L);
}

// Parameter-space half of the backward pass for one layer (Eqs. xtow-g, xtow-g-bias, and their
// Jacobian twins of Section 4.2): out_W = alpha ds^T Zprev + beta cin_W, out_b = alpha 1^T ds + beta cin_b.
GemmArgs weight_block_args(const gn_ctx* c, int m, const float* ds, const float* Zprev, int64_t rows, float alpha,
                           const float* cin, float beta, float* out, bool padded = true) {
  GemmArgs g;
  g.mn_padded = padded;   // ds and Zprev are context-owned (padded) unless the caller says otherwise
  g.M = c->w[m]; g.N = c->w[m - 1];
  g.A1 = ds; g.lda1 = c->w[m]; g.a_kmajor = false;
  g.B1 = Zprev; g.ldb1 = c->w[m - 1]; g.b_kmajor = false;
  g.K1 = (int)rows;
  g.alpha = alpha;
  g.cin = cin + c->w_off[m]; g.ld_cin = c->w[m - 1]; g.beta = beta;
  g.D = out + c->w_off[m]; g.ldd = c->w[m - 1];
  attach_half(c, g);
  return g;
}

// on_main: on the context's stream, in the second scratch slot, instead of the side stream and the first.
gn_status bias_block(gn_ctx* c, int m, const float* ds, int64_t rows, float alpha, const float* cin, float beta,
                     float* out, bool on_main = false) {
  GN_TRY(ensure_colsum(c, rows, c->w[m]));
  c->launches += launch_colsum(ds, rows, c->w[m], c->w[m], alpha, cin + c->b_off[m], beta, out + c->b_off[m],
                               c->colsum_scratch + (on_main ? c->colsum_cap / 2 : 0), on_main ? c->st : side_fork(c));
  return GN_OK;
}

gn_status weight_block(gn_ctx* c, int m, const float* ds, const float* Zprev, int64_t rows, float alpha,
                       const float* cin, float beta, float* out, bool padded = true) {
  // (the bias sums first: forked to the side stream before the contraction is enqueued, they run beside it)
  GN_TRY(bias_block(c, m, ds, rows, alpha, cin, beta, out));
  run_gemm(c, weight_block_args(c, m, ds, Zprev, rows, alpha, cin, beta, out, padded));
  return GN_OK;
}

// Activation-space half (Eq. communi-g / communi-jaco followed by Eq. ztox-g):
// dst = (ds W^mT) * sigma'(z^{m-1}), rows stacked modulo z_rows.
GemmArgs backward_data_args(gn_ctx* c, int m, const float* ds, int64_t rows, const float* Zprev, int64_t z_rows,
                            float* dst, bool ds_just_used = false) {
  GemmArgs g;
  g.a1_split_fresh = ds_just_used;   // the weight block of the same layer has just read these very rows of ds
  g.M = (int)rows; g.N = c->w[m - 1];
  g.A1 = ds; g.lda1 = c->w[m]; g.a_kmajor = true;
  g.B1 = Wm(c, c->theta, m); g.ldb1 = c->w[m - 1]; g.b_kmajor = false;
  g.K1 = c->w[m];
  g.dsig = Zprev; g.ld_dsig = c->w[m - 1]; g.dsig_rows = (int)z_rows;
  g.D = dst; g.ldd = c->w[m - 1];
  g.mn_padded = true;     // B is the context's own (padded) copy of theta
  attach_half(c, g);
  for (int set : {(int)gn_ctx::kHDS, (int)gn_ctx::kHDb}) {
    HalfBuf& b = c->half_buf[set][(size_t)m - 1];
    if (b.p && b.base == dst) attach_half_out(c, g, b);
  }
  return g;
}

// Both halves for layer m from the same ds: the weight block over `w_rows` rows starting at ds_w, and (above the
// first layer) the activation gradient over `d_rows` rows starting at ds_d.  The two contractions are independent.
gn_status layer_backward(gn_ctx* c, int m, const float* ds_w, int64_t w_rows, const float* ds_d, int64_t d_rows,
                         const float* Zprev, int64_t z_rows, float alpha, const float* cin, float beta, float* out,
                         float* dst, bool w_padded = true) {
  GemmArgs gs[2];
  int n = 0;
  gs[n++] = weight_block_args(c, m, ds_w, Zprev, w_rows, alpha, cin, beta, out, w_padded);
  if (m > 1) gs[n++] = backward_data_args(c, m, ds_d, d_rows, Zprev, z_rows, dst, ds_w == ds_d && w_rows == d_rows);
  GN_TRY(bias_block(c, m, ds_w, w_rows, alpha, cin, beta, out));
  run_gemm_group(c, gs, n);
  return GN_OK;
}

// Layers m_top .. 1 of a backward pass over `rows` rows, delta s^{m_top} = ds_top being complete: every layer's
// activation gradient (Eqs. communi-g, ztox-g) into DSbuf[m - 1] and its weight and bias blocks (Eqs. xtow-g,
// xtow-g-bias) into `out`.  In TF32 mode the contractions go out as ONE chain, [activation gradient, weight block] per
// layer: an activation-gradient tile waits for the tiles of its row panel one layer up, a weight block for all of
// them, and the pairs' loads are levelled over the whole pass instead of per layer (one ramp, one exposed
// epilogue and one ragged last round instead of one per layer).  The bias sums of the layers below m_top can
// then only start when the chain has ended.  zprev[m - 1] = z^{m-1}; layer 1 takes w1_rows rows (the caller adds
// the rest) of an operand that is padded or not (w1_padded).
gn_status backward_hidden_layers(gn_ctx* c, int m_top, const float* ds_top, const std::vector<const float*>& zprev,
                                 std::vector<float*>& DSbuf, int64_t rows, float alpha, const float* cin, float beta,
                                 float* out, int64_t w1_rows, bool w1_padded) {
  if (m_top < 1) return GN_OK;
  // One launch instead of one per layer saves the ramp, the exposed last epilogue and the ragged last round of
  // every layer, but it has to end with layer 1's weight block, whose tiles are as long as the pass has rows, and
  // the lower layers' bias sums wait for all of it: measured at 784-2000-2000-2000-10, it wins below about 4000
  // rows (full product 0.40 -> 0.37 ms at 1500 rows, 0.56 -> 0.52 at 3000; 784-300-300-10 0.161 -> 0.143) and loses
  // above (0.94 -> 1.00 at 6000, 1.13 -> 1.30 at 8000).
  int widest = 0;
  for (int m = 1; m <= m_top; ++m) widest = std::max(widest, c->w[m]);
  const bool chain = c->back_chain == 1 || (c->back_chain == 2 && (double)rows * widest <= 7.0e6);
  // (with copies never as a chain: a copy's scale comes from the largest delta of the layer above, known when that is complete)
  if (!(c->prec == GN_TF32 && chain && m_top >= 2) || c->half_now) {
    const float* ds = ds_top;
    for (int m = m_top; m >= 1; --m) {
      const int64_t wr = m == 1 ? w1_rows : rows;
      if (m == 1) GN_TRY(weight_block(c, 1, ds, zprev[0], wr, alpha, cin, beta, out, w1_padded));
      else GN_TRY(layer_backward(c, m, ds, wr, ds, rows, zprev[(size_t)m - 1], rows, alpha, cin, beta, out, DSbuf[(size_t)m - 1]));
      if (m > 1) ds = DSbuf[(size_t)m - 1];
    }
    return GN_OK;
  }
  std::vector<GemmArgs> gs;
  std::vector<int> dep, dep_all;
  GN_TRY(bias_block(c, m_top, ds_top, m_top == 1 ? w1_rows : rows, alpha, cin, beta, out));   // (its operand is ready now)
  int producer = -1;                        // index of the problem that writes delta s^m
  const float* ds = ds_top;
  for (int m = m_top; m >= 1; --m) {
    int next_producer = -1;
    if (m > 1) {
      gs.push_back(backward_data_args(c, m, ds, rows, zprev[(size_t)m - 1], rows, DSbuf[(size_t)m - 1], true));
      dep.push_back(producer); dep_all.push_back(0);
      next_producer = (int)gs.size() - 1;
    }
    gs.push_back(weight_block_args(c, m, ds, zprev[(size_t)m - 1], m == 1 ? w1_rows : rows, alpha, cin, beta, out,
                                   m == 1 ? w1_padded : true));
    dep.push_back(producer); dep_all.push_back(1);
    producer = next_producer;
    if (m > 1) ds = DSbuf[(size_t)m - 1];
  }
  run_gemm_chain(c, gs.data(), dep.data(), dep_all.data(), (int)gs.size());
  // (nothing is left to hide these sums behind: they alternate between the side stream and this one, each with its
  // own scratch, so that two of them run at a time)
  for (int m = m_top - 1; m >= 1; --m)
    GN_TRY(bias_block(c, m, DSbuf[(size_t)m], m == 1 ? w1_rows : rows, alpha, cin, beta, out, ((m_top - 1 - m) & 1) != 0));
  return GN_OK;
}

// Copies of a backward pass (`deltas` as of set kHDS or kHDb): room for those that contractions write, with the largest
// magnitude of the output layer's delta where the first of them has to bound its result from it ...
void half_deltas(gn_ctx* c, int set, const float* top, const std::vector<float*>& deltas, int64_t rows, int64_t cap_rows) {
  if (!c->half_now || !half_room(c, set, deltas, c->L - 1, rows, cap_rows)) return;
  half_matrix(c, set, c->L, top, rows, c->w[c->L], cap_rows, false);
}
// ... and of the last hidden layer's delta, if it was written by something that wrote no copy.
void half_top_delta(gn_ctx* c, int set, const std::vector<float*>& deltas, int64_t rows, int64_t cap_rows) {
  const int m = c->L - 1;
  if (!c->half_now || c->half_buf[set][(size_t)m].valid || c->w[m] < 128 || c->w[m] % 4 != 0) return;
  half_matrix(c, set, m, deltas[(size_t)m], rows, c->w[m], cap_rows, true);
}

// out = coef v + (1/|S|) J^T (2 J v) over the stored subsample (Eq. sampled-Gauss).
gn_status product_full_pass(gn_ctx* c, const float* v, float* out, float coef) {
  GN_PHASE("G v");
  SmallNet small;
  if (small_pass(c, kSmallGv, c->nS, &small)) {
    small.v = v;
    for (int m = 0; m < c->L; ++m) small.z[m] = c->Z[m];
    GN_TRY(run_small_pass(c, kSmallGv, small, (float)(1.0 / (double)c->nS), v, coef, out, nullptr));
    return check_launch(c, "G v");
  }
  SideJoin side_guard(c);
  CurrentVector current(c, v);
  ++c->parts_epoch;
  const int L = c->L;
  const int64_t nS = c->nS;
  HalfPass half_guard(c, half_wanted(c, nS, kHalfProduct));
  half_theta(c);
  half_vector(c, v);
  half_room(c, gn_ctx::kHRZ, c->RZ, L - 1, nS, c->capS);
  {
    std::vector<GemmArgs> gs((size_t)L);
    std::vector<int> dep((size_t)L), dep_all((size_t)L, 0);
    for (int m = 1; m <= L; ++m) {
      GemmArgs& g = gs[(size_t)m - 1];
      g.M = (int)nS; g.N = c->w[m];
      if (m == 1) {
        g.A1 = c->Z[0]; g.lda1 = c->w[0]; g.B1 = Wm(c, v, 1); g.ldb1 = c->w[0]; g.K1 = c->w[0];
      } else {
        g.A1 = c->RZ[m - 1]; g.lda1 = c->w[m - 1]; g.B1 = Wm(c, c->theta, m); g.ldb1 = c->w[m - 1]; g.K1 = c->w[m - 1];
        g.A2 = c->Z[m - 1];  g.lda2 = c->w[m - 1]; g.B2 = Wm(c, v, m);        g.ldb2 = c->w[m - 1]; g.K2 = c->w[m - 1];
      }
      g.bias = bm(c, v, m);
      if (m < L) { g.dsig = c->Z[m]; g.ld_dsig = c->w[m]; g.dsig_rows = (int)nS; }
      else g.alpha = 2.f;                                   // B = 2I
      g.D = c->RZ[m]; g.ldd = c->w[m];
      attach_half(c, g);
      if (m < L && half_layer(c, m + 1)) {
        g.h_next[0] = c->half_info + half_info_index(c, gn_ctx::kHZ, m);
        g.h_next[1] = c->half_info + half_info_index(c, gn_ctx::kHV, m + 1);
        g.h_next[2] = c->half_info + half_info_index(c, gn_ctx::kHW, m + 1);
        attach_half_out(c, g, c->half_buf[gn_ctx::kHRZ][(size_t)m]);
      }
      dep[(size_t)m - 1] = m - 2;        // R z^{m-1} of the layer below
    }
    presplit(c, gs.data(), L, 0xf);
    // (with copies never as a chain, see backward_hidden_layers)
    run_gemm_chain(c, gs.data(), dep.data(), dep_all.data(), L, c->half_now ? 3 : 2);
  }
  const float inv = (float)(1.0 / (double)nS);
  std::vector<const float*> zprev((size_t)L);
  for (int m = 1; m <= L; ++m) zprev[(size_t)m - 1] = c->Z[m - 1];
  // the output layer (streaming kernels at n_L <= 16) on its own, the hidden layers as one pass
  half_deltas(c, gn_ctx::kHDS, c->RZ[L], c->DS, nS, c->capS);
  GN_TRY(layer_backward(c, L, c->RZ[L], nS, c->RZ[L], nS, c->Z[L - 1], nS, inv, v, coef, out, L > 1 ? c->DS[L - 1] : nullptr));
  if (L > 1) {
    half_top_delta(c, gn_ctx::kHDS, c->DS, nS, c->capS);
    GN_TRY(backward_hidden_layers(c, L - 1, c->DS[L - 1], zprev, c->DS, nS, inv, v, coef, out, nS, true));
  }
  return check_launch(c, "G v");
}
gn_status product_full(gn_ctx* c, const float* v, float* out, float coef) {
  return or_without_copies(c, [&] { return product_full_pass(c, v, out, coef); });
}

// Eq. (approx-jaco), one block per layer.  The perturbation of layer k is pushed to the output and
// pulled back to layer k only; the L streams are stacked along rows, stream j occupying rows
// [(j-1)|S|, j|S|) of every buffer at or above layer j, so each layer runs one stacked GEMM.
// The propagate form stacks its L streams along rows: the first time it is asked for, RZ_m and DS_m are regrown
// to m |S| rows (contexts that only ever use the full product and the stored factors never pay for that).
gn_status ensure_stacked(gn_ctx* c) {
  if (c->stacked) return GN_OK;
  quiesce(c);
  for (int m = 1; m <= c->L; ++m) { dev_free(c, c->RZ[m]); dev_free(c, c->DS[m]); }
  c->stacked = true;
  for (int m = 1; m <= c->L; ++m) {
    gn_status st = dev_alloc(c, &c->RZ[m], (int64_t)m * c->capS * c->w[m]);
    if (st == GN_OK && m < c->L) st = dev_alloc(c, &c->DS[m], (int64_t)m * c->capS * c->w[m]);
    if (st != GN_OK) {
      // leave a consistent, empty state: the next set_subsample allocates afresh
      for (int k = 1; k <= c->L; ++k) { dev_free(c, c->RZ[k]); dev_free(c, c->DS[k]); }
      drop_kept_parts(c, 2, true);
      half_invalidate(c, gn_ctx::kHZ);
      for (int k = 0; k <= c->L; ++k) dev_free(c, c->Z[k]);
      dev_free(c, c->idx);
      c->capS = 0; c->have_sub = false; c->factors_valid = false;
      return st;
    }
  }
  return GN_OK;
}

gn_status product_blockdiag(gn_ctx* c, const float* v, float* out, float coef) {
  GN_TRY(ensure_stacked(c));
  SideJoin side_guard(c);
  CurrentVector current(c, v);
  ++c->parts_epoch;
  const int L = c->L;
  const int64_t nS = c->nS;
  for (int k = 1; k <= L; ++k) {
    // the streams that entered below layer k move up one layer; stream k enters (disjoint rows of R z^k: independent)
    GemmArgs gs[2];
    int n = 0;
    if (k > 1) {
      GemmArgs& g = gs[n++];
      g.M = (int)((k - 1) * nS); g.N = c->w[k];
      g.A1 = c->RZ[k - 1]; g.lda1 = c->w[k - 1]; g.B1 = Wm(c, c->theta, k); g.ldb1 = c->w[k - 1]; g.K1 = c->w[k - 1];
      if (k < L) { g.dsig = c->Z[k]; g.ld_dsig = c->w[k]; g.dsig_rows = (int)nS; }
      else g.alpha = 2.f;
      g.D = c->RZ[k]; g.ldd = c->w[k];
    }
    GemmArgs& g = gs[n++];
    g.M = (int)nS; g.N = c->w[k];
    g.A1 = c->Z[k - 1]; g.lda1 = c->w[k - 1]; g.B1 = Wm(c, v, k); g.ldb1 = c->w[k - 1]; g.K1 = c->w[k - 1];
    g.bias = bm(c, v, k);
    if (k < L) { g.dsig = c->Z[k]; g.ld_dsig = c->w[k]; g.dsig_rows = (int)nS; }
    else g.alpha = 2.f;
    g.D = c->RZ[k] + (k - 1) * nS * c->w[k]; g.ldd = c->w[k];
    run_gemm_group(c, gs, n);
  }
  const float* cur = c->RZ[L];
  const float inv = (float)(1.0 / (double)nS);
  for (int k = L; k >= 1; --k) {
    const float* dsk = cur + (k - 1) * nS * c->w[k];
    GN_TRY(layer_backward(c, k, dsk, nS, cur, (k - 1) * nS, c->Z[k - 1], nS, inv, v, coef, out,
                          k > 1 ? c->DS[k - 1] : nullptr));
    if (k > 1) cur = c->DS[k - 1];
  }
  return check_launch(c, "block-diagonal G v");
}

// ---- block-diagonal product through stored factors (the paper's own mechanism, Sections 3.3.1 and 4.2)
bool stored_factors_applicable(const gn_ctx* c) {
  if (c->L < 2 || c->w[c->L] > 16) return false;
  if ((int64_t)c->w[c->L] * c->nS > 65535LL * 128) return false;
  int64_t bytes = 0;
  for (int m = 1; m < c->L; ++m) bytes += (int64_t)c->nS * c->w[c->L] * c->w[m] * 4;
  return bytes <= 32LL * 1000 * 1000 * 1000;
}

// D^{L-1} from the linear output layer, then D^{m-1} = (D^m W^{mT}) * sigma'(z^{m-1}) on |S| n_L rows
// (Eqs. communi-jaco, ztox-jaco, Jelement-store).  Done once per (theta, S).
gn_status ensure_factors(gn_ctx* c) {
  if (c->factors_valid) return GN_OK;
  GN_PHASE("Jacobian factors");
  ++c->parts_epoch;
  const int L = c->L, nL = c->w[L];
  const int64_t nS = c->nS;
  if (nS > c->capF) {
    GN_TRY(sync(c, "factors"));
    for (int m = 1; m < L; ++m) dev_free(c, c->DF[m], c->capF * nL * c->w[m]);
    c->capF = 0;
    for (int m = 1; m < L; ++m) GN_TRY(dev_alloc(c, &c->DF[m], nS * nL * c->w[m]));
    c->capF = nS;
  }
  c->launches += launch_factor_last(Wm(c, c->theta, L), c->Z[L - 1], nS, nL, c->w[L - 1], c->DF[L - 1], c->st);
  HalfPass half_guard(c, L >= 3 && half_wanted(c, nS * nL, kHalfProduct));
  half_theta(c);
  // (the factors' copies are the largest: where they find no room the recurrence goes on without, and the other copies stay)
  const auto room = [&](int m) {
    if (half_reserve(c, c->half_buf[gn_ctx::kHF][(size_t)m], gn_ctx::kHF, m, c->DF[m], nS * nL, c->w[m], 0)) return true;
    quiesce(c);
    half_drop(c, gn_ctx::kHF);
    c->half_now = false;
    return false;
  };
  if (L >= 3 && c->w[L - 1] >= 128 && c->half_now && room(L - 1))
    half_matrix(c, gn_ctx::kHF, L - 1, c->DF[L - 1], nS * nL, c->w[L - 1], 0, true, half_info_index(c, gn_ctx::kHF, 0), L - 1);
  for (int m = L - 1; m >= 2; --m) {
    GemmArgs g;
    g.M = (int)(nS * nL); g.N = c->w[m - 1];
    g.A1 = c->DF[m]; g.lda1 = c->w[m]; g.a_kmajor = true;
    g.B1 = Wm(c, c->theta, m); g.ldb1 = c->w[m - 1]; g.b_kmajor = false;
    g.K1 = c->w[m];
    g.dsig = c->Z[m - 1]; g.ld_dsig = c->w[m - 1]; g.dsig_rows = (int)nS; g.dsig_div = nL;
    g.D = c->DF[m - 1]; g.ldd = c->w[m - 1];
    g.mn_padded = true;
    attach_half(c, g);
    if (m - 1 >= 2 && c->half_now && c->w[m - 1] >= 128 && c->w[m - 1] % 4 == 0) {
      if (room(m - 1)) attach_half_out(c, g, c->half_buf[gn_ctx::kHF][(size_t)m - 1]);
      else g.half = false;
    }
    run_gemm(c, g);
  }
  c->factors_valid = true;
  return check_launch(c, "Jacobian factors");
}

gn_status product_blockdiag_stored(gn_ctx* c, const float* v, float* out, float coef) {
  SideJoin side_guard(c);
  CurrentVector current(c, v);
  ++c->parts_epoch;
  GN_TRY(ensure_factors(c));
  const int L = c->L, nL = c->w[L];
  const int64_t nS = c->nS;
  const float inv = (float)(1.0 / (double)nS);
  HalfPass half_guard(c, half_wanted(c, nS, kHalfStored));
  half_vector(c, v);
  constexpr int kGroup = 3;
  // The layers' chains are independent of one another, so each stage is issued for all layers together.
  // 1. u_i = V^{mT} z^{m-1,i} + c^m for every row (the inner sum of Eq. direct-JV-cost); at m = L, D = I and B = 2I
  for (int m0 = 1; m0 <= L; m0 += kGroup) {
    GemmArgs gs[kGroup];
    int n = 0;
    for (int m = m0; m <= L && m < m0 + kGroup; ++m) {
      GemmArgs& g = gs[n++];
      g.M = (int)nS; g.N = c->w[m];
      g.A1 = c->Z[m - 1]; g.lda1 = c->w[m - 1]; g.B1 = Wm(c, v, m); g.ldb1 = c->w[m - 1]; g.K1 = c->w[m - 1];
      g.bias = bm(c, v, m);
      if (m == L) g.alpha = 2.f;
      g.D = c->RZ[m]; g.ldd = c->w[m];
      attach_half(c, g);
    }
    run_gemm_group(c, gs, n);
  }
  // 2. q_i = D_i^T 2 D_i u_i per sample (Eqs. direct-JV-cost, JTv)
  // (the factor of the last hidden layer is W^L * sigma'(z^{L-1}): formed on the fly where the kernel allows it,
  // the stored copy being needed only as the operand of the recurrence that builds the factors below it)
  for (int m = 1; m < L; ++m) {
    int done = 0;
    HalfInfo* const info = c->half_now && factor_apply_reports(nL, c->w[m]) ? c->half_info + half_info_index(c, gn_ctx::kHDS, m) : nullptr;
    if (m == L - 1 && c->fly_enabled)
      done = launch_factor_apply_last(Wm(c, c->theta, L), c->Z[L - 1], c->RZ[m], nS, nL, c->w[m], c->DS[m], info, c->st);
    if (!done) done = launch_factor_apply(c->DF[m], c->RZ[m], nS, nL, c->w[m], 1, 1, 0, c->DS[m], info, c->st);
    c->launches += done;
  }
  if (c->half_now) {
    std::vector<HalfBuf*> bufs;
    for (int m = 1; m < L && c->half_now; ++m) {
      if (c->w[m] <= 128 || c->w[m] % 4 != 0 || c->w[m - 1] < 128 || c->w[m - 1] % 4 != 0 || !factor_apply_reports(nL, c->w[m])) continue;
      HalfBuf& b = c->half_buf[gn_ctx::kHDS][(size_t)m];
      if (!half_reserve(c, b, gn_ctx::kHDS, m, c->DS[m], nS, c->w[m], c->capS)) { half_give_up(c); break; }
      bufs.push_back(&b);
    }
    if (c->half_now && !bufs.empty()) half_convert(c, {}, bufs);
  }
  // 3. the weight and bias blocks.  The bias sums and the n_L-row weight block go first: they run on the side
  // stream beside the large weight blocks, which is only possible if they are forked before those are enqueued.
  for (int m = 1; m <= L; ++m)
    GN_TRY(bias_block(c, m, m < L ? c->DS[m] : c->RZ[m], nS, inv, v, coef, out));
  // The weight blocks are few long tiles (64 of 375 k-blocks per 2000 x 2000 layer at
  // |S| = 12000: 160 tiles on 74 pairs for three layers leave a third of the last round idle), so with a long enough
  // K each block is cut into two parts of the rows: the first writes alpha Z^T Q + beta v, the second adds
  // its alpha Z^T Q to that (a chained launch: a second-part tile waits for the first-part tiles of its row panel).
  // More and shorter tiles fill the rounds better, and a short second part fills them best (the long tiles go
  // first, the short ones level the loads): the cut is the one of 1/2, 5/8, 3/4 of the rows for which the host's
  // work list comes out shortest.  The order of the two partial sums is fixed.
  bool tf32_operands = true;                                  // (the FP32-accurate kernel cuts K by itself)
  for (int m = 0; m < L; ++m) tf32_operands = tf32_operands && c->w[m] % 4 == 0;
  const bool halves = c->prec == GN_TF32 && c->chain_level >= 1 && c->split_k_enabled && nS >= 4096 && L - 1 >= 1 && L - 1 <= kGroup && tf32_operands;
  if (halves) {
    GemmArgs gs[2 * kGroup];
    int dep[2 * kGroup], dep_all[2 * kGroup];
    int n = 0;
    const int nl = L - 1;                                     // the hidden layers' blocks (the n_L-row block is a streaming kernel)
    if (c->cut_for_nS != nS || c->cut_for_half != c->half_now) {
      double best = -1.0;
      for (int eighths = 4; eighths <= 6; ++eighths) {
        const int64_t r = (nS * eighths / 8 + 63) / 64 * 64;  // first part: a whole number of k-blocks
        int Ms[2 * kGroup], Ns[2 * kGroup], Ks[2 * kGroup];
        for (int part = 0; part < 2; ++part)
          for (int m = 1; m <= nl; ++m) {
            const int k = part * nl + m - 1;
            Ms[k] = c->w[m]; Ns[k] = c->w[m - 1]; Ks[k] = (int)(part == 0 ? r : nS - r);
            if (c->half_now) Ks[k] = (Ks[k] + 1) / 2;         // (k-blocks of twice the terms)
          }
        const double t = gemm_tf32_group_makespan(2 * nl, Ms, Ns, Ks, 1);
        if (t >= 0.0 && (best < 0.0 || t < best)) { best = t; c->cut_rows = r; }
      }
      if (best < 0.0) c->cut_rows = (nS / 2 + 63) / 64 * 64;
      c->cut_for_nS = nS; c->cut_for_half = c->half_now;
    }
    const int64_t h0 = c->cut_rows;
    for (int part = 0; part < 2; ++part)
      for (int m = 1; m <= nl; ++m) {
        const int64_t r0 = part == 0 ? 0 : h0, rows = part == 0 ? h0 : nS - h0;
        GemmArgs g = weight_block_args(c, m, c->DS[m] + r0 * c->w[m], c->Z[m - 1] + r0 * c->w[m - 1], rows, inv,
                                       part == 0 ? v : out, part == 0 ? coef : 1.f, out);
        dep[n] = part == 0 ? -1 : m - 1;                      // the first-half problem of the same layer
        dep_all[n] = 0;
        gs[n++] = g;
      }
    run_gemm(c, weight_block_args(c, L, c->RZ[L], c->Z[L - 1], nS, inv, v, coef, out));
    run_gemm_chain(c, gs, dep, dep_all, n);
  } else {
    for (int m0 = 1; m0 <= L; m0 += kGroup) {
      GemmArgs gs[kGroup];
      int n = 0;
      for (int m = m0; m <= L && m < m0 + kGroup; ++m)
        gs[n++] = weight_block_args(c, m, m < L ? c->DS[m] : c->RZ[m], c->Z[m - 1], nS, inv, v, coef, out);
      run_gemm_group(c, gs, n);
    }
  }
  return check_launch(c, "block-diagonal G v (stored factors)");
}

// Eq. (approx-jaco) for a split structure, in the order of Section 4.2.  Layer m with s_a groups below and s_b
// groups at it: stream a holds U_a = Z_{m-1}[:, T_a] V^m[T_a, :] (+ c^m for the first group, which owns the
// biases); one pass over the stored factors turns every (stream a, group b) slice into
// Q_a[:, T_b] = D[:, :, T_b]^T 2 D[:, :, T_b] U_a[:, T_b]; then out_W[T_a, :] = Z_{m-1}[:, T_a]^T Q_a / |S|.
// At the output layer D = I, so Q_a = 2 U_a.
gn_status product_split(gn_ctx* c, const float* v, float* out, float coef) {
  SideJoin side_guard(c);
  CurrentVector current(c, v);
  ++c->parts_epoch;
  const int L = c->L, nL = c->w[L];
  const int64_t nS = c->nS;
  if (L >= 2) {
    if (nL > 32) return fail(c, GN_EINVAL, "a split structure needs n_L <= 32 (stored Jacobian factors)");
    if ((int64_t)nL * nS > 65535LL * 128) return fail(c, GN_EINVAL, "n_L * |S| exceeds 8 388 480 rows");
    GN_TRY(ensure_factors(c));
  }
  int64_t need = 0;
  for (int m = 1; m <= L; ++m) {
    const int64_t f = (int64_t)c->split[m - 1] * nS * c->w[m];
    if (f > need) need = f;
  }
  if (need > c->capSplit) {
    GN_TRY(sync(c, "split workspace"));
    dev_free(c, c->SU, c->capSplit); dev_free(c, c->SQ, c->capSplit);
    c->capSplit = 0;
    GN_TRY(dev_alloc(c, &c->SU, need));
    GN_TRY(dev_alloc(c, &c->SQ, need));
    c->capSplit = need;
  }
  const float inv = (float)(1.0 / (double)nS);
  HalfPass half_guard(c, half_wanted(c, nS, kHalfStored));
  half_vector(c, v);
  std::vector<GemmArgs> batch;
  for (int m = 1; m <= L; ++m) {
    const int sa = c->split[m - 1], sb = c->split[m], np = c->w[m - 1], nm = c->w[m];
    const int64_t stride = nS * nm;
    // (the copy of the layer's results lies in R z^m's memory, which has room for two streams' in FP16)
    const bool copy = c->half_now && m < L && sa <= 2 && nm > 128 && nm % 8 == 0 && factor_apply_reports(nL, (nm + sb - 1) / sb);
    for (int a = 0; a < sa; ++a) {
      const int t0 = group_lo(np, sa, a), t1 = group_lo(np, sa, a + 1);
      GemmArgs g;
      g.M = (int)nS; g.N = nm;
      g.A1 = c->Z[m - 1] + t0; g.lda1 = np; g.B1 = Wm(c, v, m) + t0; g.ldb1 = np; g.K1 = t1 - t0;
      if (a == 0) g.bias = bm(c, v, m);
      if (m == L) g.alpha = 2.f;                          // B = 2I
      g.D = c->SU + a * stride; g.ldd = nm;
      attach_half(c, g);
      batch.push_back(g);
    }
    // the groups' contractions are independent of one another: up to sixteen at a time to the group launcher
    for (size_t b0 = 0; b0 < batch.size(); b0 += 16) run_gemm_group(c, batch.data() + b0, (int)std::min<size_t>(16, batch.size() - b0));
    batch.clear();
    const float* Q = c->SU;
    if (m < L) {
      side_join(c);                                         // (the layer below's bias sums read what this overwrites)
      c->launches += launch_factor_apply(c->DF[m], c->SU, nS, nL, nm, sb, sa, stride, c->SQ,
                                         copy ? c->half_info + half_info_index(c, gn_ctx::kHDS, m) : nullptr, c->st);
      Q = c->SQ;
    }
    if (copy) {
      HalfBuf& b = c->half_buf[gn_ctx::kHDS][(size_t)m];
      if (half_reserve(c, b, gn_ctx::kHDS, m, Q, sa * nS, nm, 0)) half_convert(c, {}, {&b});
      else half_give_up(c);
    }
    // the bias sums on the side stream, beside this layer's weight blocks and the next layer's first contractions
    GN_TRY(ensure_colsum(c, nS, nm));
    c->launches += launch_colsum(Q, nS, nm, nm, inv, v + c->b_off[m], coef, out + c->b_off[m], c->colsum_scratch, side_fork(c));
    for (int a = 0; a < sa; ++a) {
      const int t0 = group_lo(np, sa, a), t1 = group_lo(np, sa, a + 1);
      GemmArgs g;
      g.mn_padded = true;                                   // both operands are context-owned
      g.M = nm; g.N = t1 - t0;
      g.A1 = Q + a * stride; g.lda1 = nm; g.a_kmajor = false;
      g.B1 = c->Z[m - 1] + t0; g.ldb1 = np; g.b_kmajor = false;
      g.K1 = (int)nS;
      g.alpha = inv;
      g.cin = v + c->w_off[m] + t0; g.ld_cin = np; g.beta = coef;
      g.D = out + c->w_off[m] + t0; g.ldd = np;
      attach_half(c, g);
      batch.push_back(g);
    }
    for (size_t b0 = 0; b0 < batch.size(); b0 += 16) run_gemm_group(c, batch.data() + b0, (int)std::min<size_t>(16, batch.size() - b0));
    batch.clear();
    half_invalidate(c, gn_ctx::kHDS);                       // (the next layer's results take the same place)
  }
  return check_launch(c, "partition-wise G v");
}

// Choosing between the two forms when the caller has not: building the factors costs about as much as
// five to six propagate-form products and saves about a third of each later one, so they are built when
// a solver announces at least kFactorBreakEven products, or once that many single products have been
// asked for on the same (theta, S), counting the one at hand; after that every product uses them.
constexpr int kFactorBreakEven = 8;

gn_status product_blockdiag_pass(gn_ctx* c, const float* v, float* out, float coef) {
  GN_PHASE("block-diagonal G v");
  if (c->has_split) return product_split(c, v, out, coef);
  SmallNet small;
  if (c->bd_method != 2 && small_pass(c, kSmallBlock, c->nS, &small)) {
    small.v = v;
    for (int m = 0; m < c->L; ++m) small.z[m] = c->Z[m];
    GN_TRY(run_small_pass(c, kSmallBlock, small, (float)(1.0 / (double)c->nS), v, coef, out, nullptr));
    return check_launch(c, "block-diagonal G v");
  }
  bool stored = c->bd_method == 2;
  if (c->bd_method == 0 && stored_factors_applicable(c))
    stored = c->factors_valid || c->bd_expect >= kFactorBreakEven || c->bd_count + 1 >= kFactorBreakEven;
  if (stored && c->L >= 2 && c->w[c->L] <= 16) return product_blockdiag_stored(c, v, out, coef);
  ++c->bd_count;
  return product_blockdiag(c, v, out, coef);
}
gn_status product_blockdiag_any(gn_ctx* c, const float* v, float* out, float coef) {
  return or_without_copies(c, [&] { return product_blockdiag_pass(c, v, out, coef); });
}

gn_status ensure_batch(gn_ctx* c) {
  const int64_t rows = c->batch_rows < c->l ? c->batch_rows : c->l;
  if (rows <= c->capB) return GN_OK;
  quiesce(c);
  drop_kept_parts(c, 4, true);
  for (int m = 1; m <= c->L; ++m) { dev_free(c, c->Zb[m], c->capB * c->w[m]); dev_free(c, c->Db[m], c->capB * c->w[m]); }
  c->capB = 0;
  for (int m = 1; m <= c->L; ++m) {
    GN_TRY(dev_alloc(c, &c->Zb[m], rows * c->w[m]));
    GN_TRY(dev_alloc(c, &c->Db[m], rows * c->w[m]));
  }
  c->capB = rows;
  return GN_OK;
}

// f from the summed loss and theta^T theta on the device.
gn_status read_loss(gn_ctx* c, double* f_host) {
  GN_TRY(check_launch(c, "f / grad"));
  GN_TRY(sync(c, "f / grad"));
  *f_host = c->hscal[1] / (2.0 * c->C) + c->hscal[0] / (double)c->l;
  return GN_OK;
}

// f and (optionally) the gradient over all rows in row batches (Section 6.1 in its one-GPU form).
gn_status fun_grad_pass(gn_ctx* c, float* d_grad, double* f_host) {
  GN_PHASE("f / gradient");
  SmallNet small;
  if (small_pass(c, d_grad ? kSmallGrad : kSmallFun, c->l, &small)) {
    small.z[0] = c->dX; small.Y = c->dY; small.theta_sq = c->dscal + 1;
    GN_TRY(run_small_pass(c, d_grad ? kSmallGrad : kSmallFun, small, (float)(1.0 / (double)c->l), c->theta, (float)(1.0 / c->C), d_grad, c->dscal));
    return f_host ? read_loss(c, f_host) : check_launch(c, "grad");
  }
  GN_TRY(ensure_batch(c));
  const int L = c->L;
  const int64_t Rb = c->capB;
  const int64_t nb = (c->l + Rb - 1) / Rb;
  const int64_t per_batch = loss_num_partials(Rb * c->w[L]);
  GN_TRY(ensure_partials(c, per_batch * nb + (c->n + kCgChunk - 1) / kCgChunk + 16));
  const float inv_l = (float)(1.0 / (double)c->l);
  const float inv_C = (float)(1.0 / c->C);
  struct CurrentBatch { gn_ctx* c; ~CurrentBatch() { c->cur_x = nullptr; } } current{c};
  for (int64_t b = 0; b < nb; ++b) {
    const int64_t r0 = b * Rb;
    const int64_t rows = (c->l - r0 < Rb) ? c->l - r0 : Rb;
    const float* X0 = c->dX + r0 * c->w[0];
    c->cur_x = X0;
    ++c->parts_epoch;           // the batch buffers are rewritten
    HalfPass half_guard(c, half_wanted(c, rows, d_grad ? kHalfGrad : kHalfFun));
    forward_pass(c, X0, rows, c->Zb, gn_ctx::kHZb, c->capB);
    c->launches += launch_loss_delta(c->Zb[L], c->dY + r0 * c->w[L], rows * c->w[L], d_grad ? c->Db[L] : nullptr,
                                     c->partial + b * per_batch, c->st);
    {
      // only the last batch can be shorter than Rb: zero the partial slots it does not write
      const int used = loss_num_partials(rows * c->w[L]);
      if (used < per_batch)
        GN_CUDA(c, cudaMemsetAsync(c->partial + b * per_batch + used, 0, (per_batch - used) * sizeof(double), c->st));
    }
    if (d_grad) {
      SideJoin side_guard(c);     // the next batch overwrites what the side stream reads
      const float* cin0 = b == 0 ? c->theta : d_grad;
      const float beta0 = b == 0 ? inv_C : 1.f;
      std::vector<const float*> zprev((size_t)L);
      for (int m = 1; m <= L; ++m) zprev[(size_t)m - 1] = m == 1 ? X0 : c->Zb[m - 1];
      // layer 1 reads the caller's X, which has no slack after its last row: in the last batch all but the final
      // 32 rows use the TF32 kernel's padded fast path, the rest is added by a second, unpadded contraction
      const bool last = r0 + rows == c->l;
      // (a copy of X has the slack)
      const bool tail = last && rows > 64 && c->prec == GN_TF32 && c->w[0] % 4 == 0 && c->w[1] % 4 == 0 &&
                        !(c->half_now && c->half_buf[gn_ctx::kHZb][0].valid && c->w[1] > 128 && c->w[0] >= 128);
      const int64_t head = tail ? rows - 32 : rows;
      if (L > 1) {
        half_deltas(c, gn_ctx::kHDb, c->Db[L], c->Db, rows, c->capB);
        GN_TRY(layer_backward(c, L, c->Db[L], rows, c->Db[L], rows, c->Zb[L - 1], rows, inv_l, cin0, beta0, d_grad, c->Db[L - 1]));
        half_top_delta(c, gn_ctx::kHDb, c->Db, rows, c->capB);
        GN_TRY(backward_hidden_layers(c, L - 1, c->Db[L - 1], zprev, c->Db, rows, inv_l, cin0, beta0, d_grad, head, tail || !last));
      } else {
        GN_TRY(weight_block(c, 1, c->Db[1], X0, head, inv_l, cin0, beta0, d_grad, tail || !last));
      }
      if (tail)
        GN_TRY(weight_block(c, 1, c->Db[1] + head * c->w[1], X0 + head * c->w[0], 32, inv_l, d_grad, 1.f, d_grad, false));
    }
  }
  if (f_host) {
    c->launches += launch_sum_partials(c->partial, (int)(per_batch * nb), c->dscal + 0, false, c->st);
    // theta^T theta with the CG dot kernel over the single-segment chunk table
    double* tp = c->partial + per_batch * nb;
    c->launches += launch_cg_dot(c->theta, c->theta, c->chunks[0], c->n_chunks[0], tp, nullptr, 0, nullptr, c->st);
    c->launches += launch_sum_partials(tp, c->n_chunks[0], c->dscal + 1, false, c->st);
    return read_loss(c, f_host);
  }
  return check_launch(c, "grad");
}
gn_status fun_grad(gn_ctx* c, float* d_grad, double* f_host) {
  return or_without_copies(c, [&] { return fun_grad_pass(c, d_grad, f_host); });
}

gn_status ensure_tmp(gn_ctx* c) {
  if (!c->tmp_a) GN_TRY(dev_alloc(c, &c->tmp_a, c->n));
  if (!c->tmp_b) GN_TRY(dev_alloc(c, &c->tmp_b, c->n));
  return GN_OK;
}

gn_status need_product_state(gn_ctx* c) {
  if (!c->have_theta) return fail(c, GN_ESTATE, "theta has not been set");
  if (!c->have_sub) return fail(c, GN_ESTATE, "no current subsample (set it after theta)");
  return GN_OK;
}

void push_range(std::vector<CgChunk>& h, int64_t a, int64_t b, int seg) {
  for (int64_t k = a; k < b; k += kCgChunk) {
    CgChunk ch;
    ch.start = k; ch.len = (int32_t)((b - k < kCgChunk) ? b - k : kCgChunk); ch.seg = seg;
    h.push_back(ch);
  }
}

// Chunk table of the block systems.  One block per layer: the layer's run of theta.  With a split structure:
// partition (group a of layer m-1, group b of layer m) owns, in every row j of group b of the stored
// [n_m][n_{m-1}] matrix, the columns of group a; b^m_j goes with the first group of layer m-1.
// Partitions are numbered layer by layer, inside a layer by a * split[m] + b.
void block_chunks(const gn_ctx* c, std::vector<CgChunk>& h) {
  if (!c->has_split) {
    for (int s = 0; s < c->L; ++s) push_range(h, c->w_off[s + 1], s + 1 < c->L ? c->w_off[s + 2] : c->n, s);
    return;
  }
  int base = 0;
  for (int m = 1; m <= c->L; ++m) {
    const int sa = c->split[m - 1], sb = c->split[m], np = c->w[m - 1], nm = c->w[m];
    for (int b = 0; b < sb; ++b) {
      const int j0 = group_lo(nm, sb, b), j1 = group_lo(nm, sb, b + 1);
      if (sa == 1) {
        push_range(h, c->w_off[m] + (int64_t)j0 * np, c->w_off[m] + (int64_t)j1 * np, base + b);
      } else {
        for (int a = 0; a < sa; ++a) {
          const int t0 = group_lo(np, sa, a), t1 = group_lo(np, sa, a + 1);
          for (int j = j0; j < j1; ++j) push_range(h, c->w_off[m] + (int64_t)j * np + t0, c->w_off[m] + (int64_t)j * np + t1, base + a * sb + b);
        }
      }
      push_range(h, c->b_off[m] + j0, c->b_off[m] + j1, base + b);
    }
    base += sa * sb;
  }
}

// Chunk tables are kept sorted by segment, and every segment records where its chunks start, so that the
// per-segment reductions touch only their own partial sums.
gn_status build_chunks(gn_ctx* c, bool block_only) {
  for (int mode = block_only ? 1 : 0; mode < 2; ++mode) {
    std::vector<CgChunk> h;
    if (mode == 0) push_range(h, 0, c->n, 0);
    else block_chunks(c, h);
    std::stable_sort(h.begin(), h.end(), [](const CgChunk& a, const CgChunk& b) { return a.seg < b.seg; });
    const int n_seg = mode == 0 ? 1 : c->P;
    std::vector<CgSeg> segs((size_t)n_seg);
    for (auto& sg : segs) { std::memset(&sg, 0, sizeof(CgSeg)); }
    for (size_t i = 0; i < h.size(); ++i) {
      CgSeg& sg = segs[(size_t)h[i].seg];
      if (sg.count == 0) sg.first = (int)i;
      ++sg.count;
    }
    // room for the partial sums of the new table, then the new tables, then the swap: a refused allocation
    // leaves the old tables (and the structure they belong to) in use
    GN_TRY(ensure_partials(c, 2 * (int64_t)h.size() + 64));
    CgChunk* d_chunks = nullptr;
    CgSeg* d_segs = nullptr;
    gn_status st = dev_alloc(c, &d_chunks, (int64_t)h.size());
    if (st == GN_OK) st = dev_alloc(c, &d_segs, (int64_t)n_seg);
    if (st == GN_OK && (cudaMemcpy(d_chunks, h.data(), h.size() * sizeof(CgChunk), cudaMemcpyHostToDevice) != cudaSuccess ||
                        cudaMemcpy(d_segs, segs.data(), segs.size() * sizeof(CgSeg), cudaMemcpyHostToDevice) != cudaSuccess)) {
      cudaGetLastError();
      st = fail(c, GN_ECUDA, "copy of the chunk tables failed");
    }
    if (st != GN_OK) { dev_free(c, d_chunks); dev_free(c, d_segs); return st; }
    dev_free(c, c->chunks[mode]);
    dev_free(c, c->segs[mode]);
    c->chunks[mode] = d_chunks; c->n_chunks[mode] = (int)h.size();
    c->segs[mode] = d_segs; c->segs_cap[mode] = n_seg;
  }
  return GN_OK;
}

}  // namespace

extern "C" {

gn_status gn_create(gn_ctx** out, int L, const int32_t* widths, double C, int64_t l, const float* dX,
                    const float* dY, gn_precision prec, void* cuda_stream) {
  if (!out) return GN_EINVAL;
  *out = nullptr;
  if (L < 1 || L > 64 || !widths || !(C > 0.0) || l < 1 || !dX || !dY) return GN_EINVAL;
  if (prec != GN_TF32 && prec != GN_FP32_ACCURATE) return GN_EINVAL;
  for (int m = 0; m <= L; ++m)
    if (widths[m] < 1) return GN_EINVAL;
  if (l > 0x7fffffffLL) return GN_EINVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return GN_ECUDA; }
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) { cudaGetLastError(); return GN_ECUDA; }
  if (prop.major != 10) return GN_ECUDA;  // kernels are built for sm_100a only
  gn_ctx* c = new (std::nothrow) gn_ctx();
  if (!c) return GN_ENOMEM;
  c->L = L;
  c->w.assign(widths, widths + L + 1);
  c->C = C; c->l = l; c->dX = dX; c->dY = dY; c->prec = prec;
  c->st = static_cast<cudaStream_t>(cuda_stream);
  if (!c->st) {
    // a blocking stream of the context's own: it orders itself with work on the legacy default stream the way
    // CUDA's blocking streams do, so a caller that works on that stream sees no difference
    if (cudaStreamCreate(&c->st) != cudaSuccess) { cudaGetLastError(); delete c; return GN_ECUDA; }
    c->own_stream = true;
  }
  c->w_off.assign(L + 2, 0); c->b_off.assign(L + 2, 0);
  int64_t off = 0;
  for (int m = 1; m <= L; ++m) {
    c->w_off[m] = off; off += (int64_t)c->w[m - 1] * c->w[m];
    c->b_off[m] = off; off += c->w[m];
  }
  c->n = off;
  c->Z.assign(L + 1, nullptr); c->RZ.assign(L + 1, nullptr); c->DS.assign(L + 1, nullptr);
  c->DF.assign(L + 1, nullptr);
  c->Zb.assign(L + 1, nullptr); c->Db.assign(L + 1, nullptr);
  for (auto& set : c->half_buf) set.resize((size_t)L + 1);
  c->split.assign(L + 1, 1); c->has_split = false; c->P = L;
  gn_status s = GN_OK;
  do {
    if ((s = dev_alloc(c, &c->theta, c->n)) != GN_OK) break;
    if ((s = dev_alloc(c, &c->cg_r, c->n)) != GN_OK) break;
    if ((s = dev_alloc(c, &c->cg_p, c->n)) != GN_OK) break;
    if ((s = dev_alloc(c, &c->cg_q, c->n)) != GN_OK) break;
    if ((s = dev_alloc(c, &c->status, 1)) != GN_OK) break;
    if (cudaMemset(c->status, 0, sizeof(gn_ctx::Status)) != cudaSuccess) { s = GN_ECUDA; break; }
    if (cudaMallocHost(&c->h_status, sizeof(gn_ctx::Status)) != cudaSuccess) { s = GN_ENOMEM; break; }
    std::memset(c->h_status, 0, sizeof(gn_ctx::Status));
    c->dscal = c->status->scal; c->hscal = c->h_status->scal;
    c->cg_ctl = &c->status->ctl; c->h_ctl = &c->h_status->ctl;
    c->err_flag = c->status->err; c->h_err = c->h_status->err;
    if (cudaStreamCreateWithFlags(&c->st2, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming) != cudaSuccess) { s = GN_ECUDA; break; }
    if ((s = build_chunks(c, false)) != GN_OK) break;
  } while (0);
  if (s != GN_OK) { gn_destroy(c); return s; }
  *out = c;
  return GN_OK;
}

gn_status gn_destroy(gn_ctx* c) {
  if (!c) return GN_OK;
  quiesce(c);
  for (auto& g : c->cg_graph) if (g.exec) cudaGraphExecDestroy(g.exec);
  if (c->own_stream) cudaStreamDestroy(c->st);
  if (c->st2) cudaStreamDestroy(c->st2);
  if (c->ev_fork) cudaEventDestroy(c->ev_fork);
  if (c->ev_join) cudaEventDestroy(c->ev_join);
  for (auto& o : c->owned)
    if (o.p) cudaFree(o.p);
  for (auto& p : c->ev) { cudaEventDestroy(p.a); cudaEventDestroy(p.b); }
  if (c->h_status) cudaFreeHost(c->h_status);
  cudaGetLastError();
  delete c;
  return GN_OK;
}

int64_t gn_num_params(const gn_ctx* c) { return c ? c->n : -1; }
const char* gn_last_error(const gn_ctx* c) { return c ? c->err.c_str() : "null context"; }
int64_t gn_workspace_bytes(const gn_ctx* c) { return c ? c->bytes : -1; }
int64_t gn_kernel_launches(const gn_ctx* c) { return c ? c->launches : -1; }
int64_t gn_graph_replays(const gn_ctx* c) { return c ? c->graph_replays : -1; }

gn_status gn_set_batch_rows(gn_ctx* c, int64_t rows) {
  if (!c) return GN_EINVAL;
  if (rows < 1) return fail(c, GN_EINVAL, "batch rows must be >= 1");
  c->batch_rows = rows;
  if ((rows < c->l ? rows : c->l) != c->capB && c->capB > 0) {
    // shrink or grow on next use: drop the old workspace now so memory stays bounded
    quiesce(c);
      drop_kept_parts(c, 4, true);
    for (int m = 1; m <= c->L; ++m) { dev_free(c, c->Zb[m], c->capB * c->w[m]); dev_free(c, c->Db[m], c->capB * c->w[m]); }
    c->capB = 0;
  }
  return GN_OK;
}

gn_status gn_set_blockdiag_method(gn_ctx* c, int method) {
  if (!c) return GN_EINVAL;
  if (method < 0 || method > 2) return fail(c, GN_EINVAL, "method must be 0 (choose), 1 (propagate) or 2 (stored factors)");
  if (method == 2 && (c->L < 2 || c->w[c->L] > 16))
    return fail(c, GN_EINVAL, "stored factors need at least two layers and n_L <= 16");
  c->bd_method = method;
  return GN_OK;
}

gn_status gn_set_accurate_method(gn_ctx* c, int method) {
  if (!c) return GN_EINVAL;
  if (method < 0 || method > 2) return fail(c, GN_EINVAL, "method must be 0 (choose), 1 (FP32 FMA) or 2 (as 0)");
  if (c->acc_method != method) ++c->dispatch_gen;
  c->acc_method = method;
  return GN_OK;
}

gn_status gn_set_split(gn_ctx* c, const int32_t* split) {
  if (!c) return GN_EINVAL;
  if (!split) return fail(c, GN_EINVAL, "split is NULL");
  int64_t P = 0;
  bool any = false;
  for (int m = 0; m <= c->L; ++m) {
    if (split[m] < 1 || split[m] > c->w[m]) return fail(c, GN_EINVAL, "split[m] must lie in [1, n_m]");
    if (split[m] > 1) any = true;
    if (m >= 1) P += (int64_t)split[m - 1] * split[m];
  }
  if (P > 1024) return fail(c, GN_EINVAL, "more than 1024 partitions");
  if (any && c->L >= 2 && c->w[c->L] > 32) return fail(c, GN_EINVAL, "a split structure needs n_L <= 32 (stored Jacobian factors)");
  GN_TRY(sync(c, "set_split"));
  const std::vector<int> old_split = c->split;
  const bool old_has = c->has_split;
  const int old_P = c->P;
  c->split.assign(split, split + c->L + 1);
  c->has_split = any;
  c->P = (int)P;
  const gn_status st = build_chunks(c, true);
  if (st == GN_OK) drop_kept_parts(c, 0, false);     // (of the sub-blocks of the structure that has gone)
  if (st != GN_OK) { c->split = old_split; c->has_split = old_has; c->P = old_P; }   // the old tables are still in place
  return st;
}

int32_t gn_num_partitions(const gn_ctx* c) { return c ? c->P : -1; }

gn_status gn_set_cg_termination(gn_ctx* c, int32_t cg_min, double finished_share) {
  if (!c) return GN_EINVAL;
  if (cg_min < 0) return fail(c, GN_EINVAL, "cg_min must be >= 0");
  if (!(finished_share > 0.0 && finished_share <= 1.0)) return fail(c, GN_EINVAL, "finished_share must lie in (0, 1]");
  c->cg_min = cg_min; c->cg_share = finished_share;
  return GN_OK;
}

gn_status gn_set_theta(gn_ctx* c, const float* d_theta) {
  if (!c) return GN_EINVAL;
  if (!d_theta) return fail(c, GN_EINVAL, "theta is NULL");
  GN_CUDA(c, cudaMemcpyAsync(c->theta, d_theta, c->n * sizeof(float), cudaMemcpyDeviceToDevice, c->st));
  ++c->theta_epoch;
  c->have_theta = true;
  c->have_sub = false;
  return GN_OK;
}

gn_status gn_set_theta_host(gn_ctx* c, const float* h_theta) {
  if (!c) return GN_EINVAL;
  if (!h_theta) return fail(c, GN_EINVAL, "theta is NULL");
  GN_CUDA(c, cudaMemcpyAsync(c->theta, h_theta, c->n * sizeof(float), cudaMemcpyHostToDevice, c->st));
  ++c->theta_epoch;
  GN_TRY(sync(c, "set_theta_host"));
  c->have_theta = true;
  c->have_sub = false;
  return GN_OK;
}

static gn_status set_subsample_pass(gn_ctx* c, const int32_t* idx, int64_t nS, cudaMemcpyKind kind) {
  GN_PHASE("set_subsample");
  if (!idx) return fail(c, GN_EINVAL, "idx is NULL");
  if (nS < 1) return fail(c, GN_EINVAL, "the subsample must have at least one row");
  if (!c->have_theta) return fail(c, GN_ESTATE, "theta has not been set");
  if ((int64_t)c->L * nS > 65535LL * 128) return fail(c, GN_EINVAL, "L * |S| exceeds 8 388 480 rows");
  c->have_sub = false;
  c->factors_valid = false;
  c->bd_count = 0;
  ++c->sub_epoch;             // the stored activations are about to be rewritten
  half_invalidate(c, gn_ctx::kHZ);
  ++c->parts_epoch;
  if (nS > c->capS) {
    GN_TRY(sync(c, "set_subsample"));
    drop_kept_parts(c, 2, true);      // the stored activations move: their parts are made anew
    half_drop(c, gn_ctx::kHZ);
      dev_free(c, c->idx, c->capS);
    for (int m = 0; m <= c->L; ++m) dev_free(c, c->Z[m], c->capS * c->w[m]);
    for (int m = 1; m <= c->L; ++m) { dev_free(c, c->RZ[m], m * c->capS * c->w[m]); dev_free(c, c->DS[m], m * c->capS * c->w[m]); }
    c->capS = 0;
    GN_TRY(dev_alloc(c, &c->idx, nS));
    for (int m = 0; m <= c->L; ++m) GN_TRY(dev_alloc(c, &c->Z[m], nS * c->w[m]));
    for (int m = 1; m <= c->L; ++m) {
      const int64_t depth = c->stacked ? m : 1;
      GN_TRY(dev_alloc(c, &c->RZ[m], depth * nS * c->w[m]));
      if (m < c->L) GN_TRY(dev_alloc(c, &c->DS[m], depth * nS * c->w[m]));
    }
    c->capS = nS;
  }
  c->nS = nS;
  GN_CUDA(c, cudaMemcpyAsync(c->idx, idx, nS * sizeof(int32_t), kind, c->st));
  GN_CUDA(c, cudaMemsetAsync(c->err_flag, 0, sizeof(int), c->st));
  SmallNet small;
  if (small_pass(c, kSmallForward, nS, &small)) {
    small.z[0] = c->dX; small.idx = c->idx; small.x_rows = c->l; small.err_flag = c->err_flag;
    for (int m = 0; m <= c->L; ++m) small.z_out[m] = c->Z[m];
    GN_TRY(run_small_pass(c, kSmallForward, small, 0.f, nullptr, 0.f, nullptr, nullptr));
  } else {
    c->launches += launch_gather_rows(c->dX, c->l, c->w[0], c->idx, nS, c->Z[0], c->err_flag, c->st);
    // (copies of the stored activations are there for the products)
    const bool blocks = c->w[c->L] <= 16 || c->has_split;
    HalfPass half_guard(c, half_wanted(c, nS, kHalfProduct) || (blocks && half_wanted(c, nS, kHalfStored)));
    forward_pass(c, c->Z[0], nS, c->Z, gn_ctx::kHZ, c->capS);
  }
  GN_TRY(check_launch(c, "set_subsample"));
  GN_TRY(sync(c, "set_subsample"));
  if (*c->h_err) return fail(c, GN_EINVAL, "a subsample index lies outside [0, l)");
  c->have_sub = true;
  return GN_OK;
}

static gn_status set_subsample_impl(gn_ctx* c, const int32_t* idx, int64_t nS, cudaMemcpyKind kind) {
  if (!c) return GN_EINVAL;
  if (!c->half_usable) { c->half_usable = true; ++c->dispatch_gen; }
  return or_without_copies(c, [&] { return set_subsample_pass(c, idx, nS, kind); });
}

gn_status gn_set_subsample(gn_ctx* c, const int32_t* d_idx, int64_t nS) {
  return set_subsample_impl(c, d_idx, nS, cudaMemcpyDeviceToDevice);
}
gn_status gn_set_subsample_host(gn_ctx* c, const int32_t* h_idx, int64_t nS) {
  return set_subsample_impl(c, h_idx, nS, cudaMemcpyHostToDevice);
}

gn_status gn_fun(gn_ctx* c, double* f_host) {
  if (!c) return GN_EINVAL;
  if (!f_host) return fail(c, GN_EINVAL, "f_host is NULL");
  if (!c->have_theta) return fail(c, GN_ESTATE, "theta has not been set");
  return fun_grad(c, nullptr, f_host);
}

gn_status gn_grad(gn_ctx* c, float* d_grad, double* f_host) {
  if (!c) return GN_EINVAL;
  if (!d_grad) return fail(c, GN_EINVAL, "grad is NULL");
  if (!c->have_theta) return fail(c, GN_ESTATE, "theta has not been set");
  return fun_grad(c, d_grad, f_host);
}

gn_status gn_grad_host(gn_ctx* c, float* h_grad, double* f_host) {
  if (!c) return GN_EINVAL;
  if (!h_grad) return fail(c, GN_EINVAL, "grad is NULL");
  if (!c->have_theta) return fail(c, GN_ESTATE, "theta has not been set");
  GN_TRY(ensure_tmp(c));
  GN_TRY(fun_grad(c, c->tmp_b, f_host));
  GN_CUDA(c, cudaMemcpyAsync(h_grad, c->tmp_b, c->n * sizeof(float), cudaMemcpyDeviceToHost, c->st));
  return sync(c, "grad_host");
}

gn_status gn_Gv(gn_ctx* c, const float* d_v, float* d_out) {
  if (!c) return GN_EINVAL;
  if (!d_v || !d_out) return fail(c, GN_EINVAL, "v / out is NULL");
  if (d_v == d_out) return fail(c, GN_EINVAL, "v and out must not overlap");
  GN_TRY(need_product_state(c));
  return product_full(c, d_v, d_out, (float)(1.0 / c->C));
}

gn_status gn_Gv_blockdiag(gn_ctx* c, const float* d_v, float* d_out) {
  if (!c) return GN_EINVAL;
  if (!d_v || !d_out) return fail(c, GN_EINVAL, "v / out is NULL");
  if (d_v == d_out) return fail(c, GN_EINVAL, "v and out must not overlap");
  GN_TRY(need_product_state(c));
  return product_blockdiag_any(c, d_v, d_out, (float)(1.0 / c->C));
}

static gn_status product_host(gn_ctx* c, const float* h_v, float* h_out, bool blockdiag) {
  if (!c) return GN_EINVAL;
  if (!h_v || !h_out) return fail(c, GN_EINVAL, "v / out is NULL");
  GN_TRY(need_product_state(c));
  GN_TRY(ensure_tmp(c));
  GN_CUDA(c, cudaMemcpyAsync(c->tmp_a, h_v, c->n * sizeof(float), cudaMemcpyHostToDevice, c->st));
  const float coef = (float)(1.0 / c->C);
  GN_TRY(blockdiag ? product_blockdiag_any(c, c->tmp_a, c->tmp_b, coef) : product_full(c, c->tmp_a, c->tmp_b, coef));
  GN_CUDA(c, cudaMemcpyAsync(h_out, c->tmp_b, c->n * sizeof(float), cudaMemcpyDeviceToHost, c->st));
  return sync(c, "product_host");
}

gn_status gn_Gv_host(gn_ctx* c, const float* h_v, float* h_out) { return product_host(c, h_v, h_out, false); }
gn_status gn_Gv_blockdiag_host(gn_ctx* c, const float* h_v, float* h_out) { return product_host(c, h_v, h_out, true); }

gn_status gn_cg_solve(gn_ctx* c, const float* d_g, double lambda, int blockdiag, int max_iter, double tol,
                      float* d_d, int* iters_host, float* d_iterates, double* resnorm_host) {
  GN_PHASE("CG solve");
  if (!c) return GN_EINVAL;
  if (!d_g || !d_d) return fail(c, GN_EINVAL, "g / d is NULL");
  if (max_iter < 1) return fail(c, GN_EINVAL, "max_iter must be >= 1");
  if (!(lambda >= 0.0)) return fail(c, GN_EINVAL, "lambda must be >= 0");
  GN_TRY(need_product_state(c));
  const int mode = blockdiag ? 1 : 0;
  const int n_seg = blockdiag ? c->P : 1;
  const CgChunk* ch = c->chunks[mode];
  const int nc = c->n_chunks[mode];
  const float coef = (float)(1.0 / c->C + lambda);
  CgSeg* seg = c->segs[mode];
  // device-resident solver state: ticket, step count, residual history
  if (max_iter + 1 > c->cg_hist_cap) {
    GN_TRY(sync(c, "cg history"));
    dev_free(c, c->cg_hist, c->cg_hist_cap);
    c->cg_hist_cap = 0;
    GN_TRY(dev_alloc(c, &c->cg_hist, (int64_t)max_iter + 1));
    c->cg_hist_cap = max_iter + 1;
  }
  CgControl h0{};
  h0.hist = c->cg_hist; h0.hist_cap = max_iter + 1;
  *c->h_ctl = h0;
  GN_CUDA(c, cudaMemcpyAsync(c->cg_ctl, c->h_ctl, sizeof(CgControl), cudaMemcpyHostToDevice, c->st));
  // The host has to look at the scalars after every step only if something may end the solve early: a stop
  // tolerance, or the termination rule of Section 4.4.  Otherwise all max_iter steps are enqueued without waiting
  // (a system that converges exactly freezes, and the steps after that change nothing).
  const bool rule44 = blockdiag && (c->cg_min > 0 || c->cg_share < 1.0);
  const bool watch = tol > 0.0 || rule44;

  c->launches += launch_cg_init(d_g, d_d, c->cg_r, c->cg_p, ch, nc, c->partial, seg, n_seg, tol, c->cg_ctl, c->st);
  GN_TRY(check_launch(c, "cg init"));
  double active = 1.0;
  if (watch) {
    GN_TRY(sync(c, "cg init"));
    active = c->h_ctl->out[1];
  }
  int it = 0;
  c->bd_expect = blockdiag ? max_iter : 0;
  struct Reset { int* p; ~Reset() { *p = 0; } } reset_expect{&c->bd_expect};
  auto one_step = [&]() -> gn_status {
    GN_TRY(blockdiag ? product_blockdiag_any(c, c->cg_p, c->cg_q, coef) : product_full(c, c->cg_p, c->cg_q, coef));
    c->launches += launch_cg_dot(c->cg_p, c->cg_q, ch, nc, c->partial, seg, n_seg, c->cg_ctl, c->st);
    c->launches += launch_cg_update(c->cg_p, c->cg_q, d_d, c->cg_r, ch, nc, seg, n_seg, tol, c->partial, c->cg_ctl, c->st);
    c->launches += launch_cg_direction(c->cg_r, c->cg_p, ch, nc, seg, c->st);
    return check_launch(c, "cg step");
  };
  // Fixed-length solve of a small problem: the step's launches are issued once, into a graph, and replayed.
  double step_flop = 0.0;
  for (int m = 1; m <= c->L; ++m) step_flop += (m == 1 ? 4.0 : 8.0) * (double)c->w[m - 1] * c->w[m] * (double)c->nS;
  const bool use_graph = !watch && !d_iterates && !c->profiling && c->graph_enabled && c->graph_ok && max_iter >= 4 &&
                         step_flop < 120e9;
  gn_ctx::CgGraph& cgg = c->cg_graph[mode];
  while (it < max_iter && active > 0.5) {
    // Section 4.4: all partitions stop once cg_min steps are done and the stated share of them have finished
    if (rule44 && it >= c->cg_min && (double)n_seg - active >= c->cg_share * (double)n_seg) break;
    if (use_graph && it >= 1) {
      // (the first step ran as plain launches: every workspace it needs exists and the stored factors are built)
      const bool fits = cgg.exec && cgg.alloc_gen == c->alloc_gen && cgg.dispatch_gen == c->dispatch_gen && cgg.nS == c->nS && cgg.coef == coef && cgg.d == d_d &&
                        cgg.stored == (c->factors_valid ? 1 : 0) && cgg.method == c->bd_method && cgg.n_seg == n_seg;
      if (!fits) {
        if (cgg.exec) { cudaGraphExecDestroy(cgg.exec); cgg.exec = nullptr; }
        const int64_t before = c->launches;
        const uint64_t gen = c->alloc_gen;
        cudaGraph_t graph = nullptr;
        gn_status st = GN_OK;
        if (cudaStreamBeginCapture(c->st, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
          c->own_capture = true;
          st = one_step();
          c->own_capture = false;
          const cudaError_t e = cudaStreamEndCapture(c->st, &graph);
          if (st == GN_OK && e == cudaSuccess && graph && gen == c->alloc_gen &&
              cudaGraphInstantiate(&cgg.exec, graph, 0) == cudaSuccess) {
            cgg.alloc_gen = gen; cgg.dispatch_gen = c->dispatch_gen; cgg.nS = c->nS; cgg.coef = coef; cgg.d = d_d; cgg.stored = c->factors_valid ? 1 : 0;
            cgg.method = c->bd_method; cgg.n_seg = n_seg; cgg.launches = c->launches - before;
          } else {
            cgg.exec = nullptr;
          }
          if (graph) cudaGraphDestroy(graph);
          c->launches = before;              // nothing has run yet: the captured step runs when the graph is launched
        }
        cudaGetLastError();
        if (!cgg.exec) {                     // capture is not available here: plain launches from now on
          c->graph_ok = false;
          c->sticky = GN_OK;
          GN_TRY(one_step());
          ++it;
          continue;
        }
      }
      if (c->graph_ok && cgg.exec) {
        GN_CUDA(c, cudaGraphLaunch(cgg.exec, c->st));
        c->launches += cgg.launches;
        ++c->graph_replays;
        ++it;
        continue;
      }
    }
    GN_TRY(one_step());
    if (d_iterates)
      GN_CUDA(c, cudaMemcpyAsync(d_iterates + (int64_t)it * c->n, d_d, c->n * sizeof(float), cudaMemcpyDeviceToDevice, c->st));
    if (watch) {
      GN_TRY(sync(c, "cg step"));
      active = c->h_ctl->out[1];
    }
    ++it;
  }
  // the state at the end: steps in which a segment was still active, and the residual history
  if (!watch) GN_TRY(sync(c, "cg solve"));     // (a watched solve has just read it)
  const int steps = watch ? it : c->h_ctl->steps;
  if (iters_host) *iters_host = steps;
  if (resnorm_host) {
    const int len = c->h_ctl->hist_len < steps + 1 ? c->h_ctl->hist_len : steps + 1;
    GN_CUDA(c, cudaMemcpy(resnorm_host, c->cg_hist, (size_t)len * sizeof(double), cudaMemcpyDeviceToHost));
    for (int k = 0; k < len; ++k) resnorm_host[k] = sqrt(resnorm_host[k]);
  }
  return GN_OK;
}

gn_status gn_cg_solve_host(gn_ctx* c, const float* h_g, double lambda, int blockdiag, int max_iter, double tol,
                           float* h_d, int* iters_host, double* resnorm_host) {
  if (!c) return GN_EINVAL;
  if (!h_g || !h_d) return fail(c, GN_EINVAL, "g / d is NULL");
  GN_TRY(need_product_state(c));
  GN_TRY(ensure_tmp(c));
  GN_CUDA(c, cudaMemcpyAsync(c->tmp_a, h_g, c->n * sizeof(float), cudaMemcpyHostToDevice, c->st));
  GN_TRY(gn_cg_solve(c, c->tmp_a, lambda, blockdiag, max_iter, tol, c->tmp_b, iters_host, nullptr, resnorm_host));
  GN_CUDA(c, cudaMemcpyAsync(h_d, c->tmp_b, c->n * sizeof(float), cudaMemcpyDeviceToHost, c->st));
  return sync(c, "cg_solve_host");
}

gn_status gn_profile(gn_ctx* c, int enable) {
  if (!c) return GN_EINVAL;
  c->profiling = enable != 0;
  return GN_OK;
}

gn_status gn_profile_read(gn_ctx* c, double* gemm_ms, double* gemm_flop, int64_t* gemm_launches) {
  if (!c) return GN_EINVAL;
  GN_TRY(sync(c, "profile_read"));
  double ms[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, flop[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  int64_t cnt[5] = {0, 0, 0, 0, 0};
  for (size_t i = 0; i < c->ev_used; ++i) {
    float t = 0.f;
    const int k = c->ev[i].kind < 0 || c->ev[i].kind > 4 ? 1 : c->ev[i].kind;
    if (cudaEventElapsedTime(&t, c->ev[i].a, c->ev[i].b) == cudaSuccess) ms[k] += t;
    flop[k] += c->ev[i].flop;
    cnt[k] += 1;
  }
  for (int k = 0; k < 5; ++k) {
    if (gemm_ms) gemm_ms[k] = ms[k];
    if (gemm_flop) gemm_flop[k] = flop[k];
    if (gemm_launches) gemm_launches[k] = cnt[k];
  }
  c->ev_used = 0;
  cudaGetLastError();
  return GN_OK;
}

static gn_status debug_gemm_impl(gn_ctx* c, int kind, GemmArgs g);

gn_status gn_debug_gemm(gn_ctx* c, int kind, int M, int N, int K, const float* dA, int64_t lda, int a_kmajor,
                        const float* dB, int64_t ldb, int b_kmajor, float* dD, int64_t ldd) {
  return gn_debug_gemm_epilogue(c, kind, M, N, K, dA, lda, a_kmajor, dB, ldb, b_kmajor, dD, ldd, nullptr, 0, nullptr, 0,
                                1.f, nullptr, 0, 0.f);
}

gn_status gn_debug_gemm_epilogue(gn_ctx* c, int kind, int M, int N, int K, const float* dA, int64_t lda, int a_kmajor,
                                 const float* dB, int64_t ldb, int b_kmajor, float* dD, int64_t ldd, const float* d_bias,
                                 int sigmoid, const float* d_dsig, int64_t ld_dsig, float alpha, const float* d_cin,
                                 int64_t ld_cin, float beta) {
  if (!c) return GN_EINVAL;
  if (!dA || !dB || !dD || M < 1 || N < 1 || K < 1 || kind < 0 || kind > 9) return fail(c, GN_EINVAL, "bad GEMM arguments");
  if ((d_dsig && ld_dsig < N) || (d_cin && ld_cin < N)) return fail(c, GN_EINVAL, "leading dimension of an epilogue operand below N");
  GemmArgs g;
  g.M = M; g.N = N; g.K1 = K;
  g.A1 = dA; g.lda1 = lda; g.a_kmajor = a_kmajor != 0;
  g.B1 = dB; g.ldb1 = ldb; g.b_kmajor = b_kmajor != 0;
  g.D = dD; g.ldd = ldd;
  g.bias = d_bias; g.sigmoid = sigmoid != 0;
  if (d_dsig) { g.dsig = d_dsig; g.ld_dsig = ld_dsig; g.dsig_rows = M; }
  g.alpha = alpha;
  if (d_cin) { g.cin = d_cin; g.ld_cin = ld_cin; g.beta = beta; }
  return debug_gemm_impl(c, kind, g);
}

static gn_status debug_gemm_impl(gn_ctx* c, int kind, GemmArgs g) {
  // kinds 3..6 are the tensor-core kernel with options: 3 = MN-major operands declared padded,
  // 4 = one CTA per tile forced, 5 = CTA pair per tile forced, 6 = as 5 without splitting tiles
  // between pairs (all with padded operands)
  ++c->parts_epoch;
  if (kind == 7 || kind == 8) {   // FP32-accurate tensor-core form: 7 = shapes that fill a CTA-pair tile only, 8 = any
    ++c->gemm_seq;
    if ((kind == 7 && (g.M <= 128 || g.N < 128)) || !run_gemm_f16x3(c, g)) return fail(c, GN_EINVAL, "the FP32-accurate tensor-core form does not take this problem");
    GN_TRY(check_launch(c, "debug_gemm"));
    return sync(c, "debug_gemm");
  }
  if (kind == 9) {                // CTA pair per tile, FP16 copies of the operands
    HalfPass half_guard(c, true);
    if (!suits_half(g)) return fail(c, GN_EINVAL, "operands do not qualify for FP16 copies");
    for (int role = 0; role < 2; ++role) {
      const OperandView v = operand_view(g, role);
      if (v.ld != v.cols) return fail(c, GN_EINVAL, "FP16 copies are of whole matrices");
      half_matrix(c, gn_ctx::kHF, role, v.p, v.rows, v.cols, 0, true);
    }
    if (!c->half_now) return fail(c, GN_ENOMEM, "no room for FP16 copies");
    attach_half(c, g);
    c->factors_valid = false;
    if (!g.half) return fail(c, GN_EINVAL, "operands do not qualify for FP16 copies");
    kind = 5;
  }
  g.mn_padded = (kind >= 3);
  if (kind == 4) g.two_cta = 0;
  if (kind == 5) g.two_cta = 1;
  if (kind == 6) g.two_cta = 2;   // CTA pair per tile, whole tiles only (no stream-K split)
  if (kind >= 3) kind = 0;
  if (kind == 0 && !gemm_tf32_eligible(g)) return fail(c, GN_EINVAL, "operands do not qualify for the tensor-core kernel");
  if (kind == 2) {
    if (gemm_thin_kind(g) == THIN_NONE) return fail(c, GN_EINVAL, "operands do not qualify for a streaming kernel");
    run_gemm(c, g);
  } else {
    run_gemm_kind(c, g, kind);
  }
  GN_TRY(check_launch(c, "debug_gemm"));
  return sync(c, "debug_gemm");
}

// x^T y into device scalar slot (fixed-order double-precision sum of per-chunk partials)
static void dot_to_slot(gn_ctx* c, const float* x, const float* y, int slot) {
  c->launches += launch_cg_dot(x, y, c->chunks[0], c->n_chunks[0], c->partial, nullptr, 0, nullptr, c->st);
  c->launches += launch_sum_partials(c->partial, c->n_chunks[0], c->dscal + slot, false, c->st);
}

gn_status gn_newton_iter(gn_ctx* c, float* d_theta, const int32_t* d_idx, int64_t nS, float* d_dir,
                         const gn_newton_params* prm, gn_newton_report* rep) {
  if (!c) return GN_EINVAL;
  if (!d_theta || !d_idx || !d_dir || !prm || !rep) return fail(c, GN_EINVAL, "NULL argument");
  if (!(prm->lambda >= 0.0) || prm->cg_max < 1 || !(prm->eta > 0.0 && prm->eta < 1.0) || prm->max_backtrack < 0 ||
      !(prm->drop > 0.0) || !(prm->boost > 0.0))
    return fail(c, GN_EINVAL, "bad Newton parameters");
  for (int i = 0; i < 4; ++i)
    if (!c->nt[i]) GN_TRY(dev_alloc(c, &c->nt[i], c->n));
  float* g = c->nt[0]; float* d = c->nt[1]; float* Gx = c->nt[2]; float* trial = c->nt[3];
  const float inv_C = (float)(1.0 / c->C);
  std::memset(rep, 0, sizeof(*rep));

  GN_TRY(gn_set_theta(c, d_theta));
  GN_TRY(gn_set_subsample(c, d_idx, nS));
  double f0 = 0.0;
  GN_TRY(fun_grad(c, g, &f0));
  int its = 0;
  GN_TRY(gn_cg_solve(c, g, prm->lambda, prm->blockdiag, prm->cg_max, prm->sigma, d, &its, nullptr, nullptr));
  // entries of the two-variable system on the full G^S (Eq. sol-comp)
  GN_TRY(product_full(c, d, Gx, inv_C));
  dot_to_slot(c, d, Gx, 4);          // a  = d^T G d
  dot_to_slot(c, d_dir, Gx, 5);      // b  = dbar^T G d
  GN_TRY(product_full(c, d_dir, Gx, inv_C));
  dot_to_slot(c, d_dir, Gx, 6);      // c  = dbar^T G dbar
  dot_to_slot(c, g, d, 7);           // g^T d
  dot_to_slot(c, g, d_dir, 8);       // g^T dbar
  GN_TRY(check_launch(c, "newton: direction combination"));
  GN_TRY(sync(c, "newton: direction combination"));
  const double a = c->hscal[4], b = c->hscal[5], cc = c->hscal[6], gd = c->hscal[7], gdb = c->hscal[8];
  double beta1 = 1.0, beta2 = 0.0;
  const double det = a * cc - b * b;
  if (det > prm->eps) { beta1 = (-gd * cc + b * gdb) / det; beta2 = (-a * gdb + b * gd) / det; }
  // d <- beta1 d + beta2 dbar, kept in d_dir (it is the next iteration's dbar)
  c->launches += launch_axpby(c->n, (float)beta1, d, (float)beta2, d_dir, d_dir, c->st);
  const double gTd = beta1 * gd + beta2 * gdb;
  const double dGd = beta1 * beta1 * a + 2.0 * beta1 * beta2 * b + beta2 * beta2 * cc;
  // back-tracking line search (Eq. linesearch-condition)
  double alpha = 1.0, f1 = 0.0;
  int backtracks = 0;
  for (;;) {
    c->launches += launch_axpby(c->n, 1.f, d_theta, (float)alpha, d_dir, trial, c->st);
    GN_TRY(gn_set_theta(c, trial));
    GN_TRY(fun_grad(c, nullptr, &f1));
    if (f1 <= f0 + prm->eta * alpha * gTd || backtracks >= prm->max_backtrack) break;
    alpha *= 0.5;
    ++backtracks;
  }
  GN_CUDA(c, cudaMemcpyAsync(d_theta, trial, c->n * sizeof(float), cudaMemcpyDeviceToDevice, c->st));
  GN_TRY(sync(c, "newton: update"));
  const double rho = (f1 - f0) / (alpha * gTd + 0.5 * alpha * alpha * dGd);
  double lam = prm->lambda;
  if (rho > 0.75) lam *= prm->drop;
  else if (!(rho >= 0.25)) lam *= prm->boost;
  rep->f_before = f0; rep->f_after = f1; rep->alpha = alpha; rep->beta1 = beta1; rep->beta2 = beta2;
  rep->rho = rho; rep->gTd = gTd; rep->dGd = dGd; rep->lambda_next = lam;
  rep->cg_iters = its; rep->backtracks = backtracks;
  return GN_OK;
}

gn_status gn_debug_option(gn_ctx* c, int option, int value) {
  if (!c) return GN_EINVAL;
  if (option == 2) { if (value < 0) return fail(c, GN_EINVAL, "count must be >= 0"); c->fail_alloc_in = value; return GN_OK; }
  if (option >= 0 && option <= 11) ++c->dispatch_gen;
  if (option == 11) { c->half_mode = value < 0 ? 0 : (value > 2 ? 2 : value); return GN_OK; }
  if (option == 3) { quiesce(c); c->side_enabled = value != 0; return GN_OK; }
  if (option == 7) { c->split_k_enabled = value != 0; return GN_OK; }
  if (option == 8) { c->back_chain = value < 0 ? 0 : (value > 2 ? 2 : value); return GN_OK; }
  if (option == 10) { c->small_enabled = value != 0; return GN_OK; }
  if (option == 9) { c->fly_enabled = value != 0; return GN_OK; }
  if (option == 6) { c->graph_enabled = value != 0; return GN_OK; }
  if (option == 5) { c->split_together = value != 0; return GN_OK; }
  if (option == 4) { c->chain_level = value < 0 ? 0 : (value > 2 ? 2 : value); return GN_OK; }
  if (option == 0) c->group_enabled = value != 0;
  else if (option == 1) c->sk_enabled = value != 0 && c->sk_enabled;
  else return fail(c, GN_EINVAL, "unknown option");
  return GN_OK;
}

int32_t gn_debug_plan_group(int32_t n, const int32_t* M, const int32_t* N, const int32_t* K, int32_t pairs, int32_t keep_order,
                            int32_t* counts, int32_t* waves, int32_t* order, int32_t* tiles) {
  if (!M || !N || !K || !counts || !waves || !order || !tiles) return -1;
  return gemm_tf32_plan_group(n, M, N, K, pairs, keep_order, counts, waves, order, tiles);
}

gn_status gn_debug_copies(gn_ctx* c, int64_t* known, int64_t* refused) {
  if (!c || !known || !refused) return GN_EINVAL;
  *known = *refused = 0;
  GN_TRY(sync(c, "copies"));
  if (!c->half_info) return GN_OK;
  std::vector<HalfInfo> host((size_t)gn_ctx::kHalfSets * (c->L + 1));
  GN_CUDA(c, cudaMemcpy(host.data(), c->half_info, sizeof(HalfInfo) * host.size(), cudaMemcpyDeviceToHost));
  for (const HalfInfo& i : host) { *known += i.amax != 0u; *refused += i.bad != 0u; }
  return GN_OK;
}

gn_status gn_debug_check_canaries(gn_ctx* c, int64_t* n_checked) {
  if (!c) return GN_EINVAL;
  GN_TRY(sync(c, "canary check"));
  if (c->st2) cudaStreamSynchronize(c->st2);
  unsigned char host[128];
  int64_t checked = 0;
  for (const auto& o : c->owned) {
    if (!o.p) continue;
    GN_CUDA(c, cudaMemcpy(host, static_cast<const char*>(o.p) + o.bytes + 128, 128, cudaMemcpyDeviceToHost));
    for (int i = 0; i < 128; ++i)
      if (host[i] != kCanaryByte)
        return fail(c, GN_ECUDA, "the guard bytes after a workspace of " + std::to_string(o.bytes) + " bytes were overwritten (offset " +
                                     std::to_string(i) + " past its slack)");
    ++checked;
  }
  if (n_checked) *n_checked = checked;
  return GN_OK;
}

gn_status gn_debug_timeout_probe(gn_ctx* c, double limit_ms) {
  if (!c) return GN_EINVAL;
  if (!(limit_ms > 0.0) || limit_ms > 1000.0) return fail(c, GN_EINVAL, "limit must be in (0, 1000] ms");
  c->launches += launch_timeout_probe(c->err_flag + 1, (unsigned long long)(limit_ms * 1e6), c->st);
  GN_TRY(check_launch(c, "timeout probe"));
  return sync(c, "timeout probe");
}

gn_status gn_debug_activations(gn_ctx* c, int m, float* d_out) {
  if (!c) return GN_EINVAL;
  if (!d_out || m < 1 || m > c->L) return fail(c, GN_EINVAL, "bad layer / NULL output");
  GN_TRY(need_product_state(c));
  GN_CUDA(c, cudaMemcpyAsync(d_out, c->Z[m], c->nS * c->w[m] * sizeof(float), cudaMemcpyDeviceToDevice, c->st));
  return GN_OK;
}

}  // extern "C"
