// Internal launch interface between the host logic (gn_context.cu) and the kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace gn {

// One dense contraction with a fused epilogue:
//
//   acc[m][n] = sum_k A1(m,k) B1(k,n)  (+ sum_k A2(m,k) B2(k,n) when A2 != nullptr)
//   t = acc + bias[n]                   (bias != nullptr)
//   t = 1 / (1 + exp(-t))               (sigmoid)
//   t = t * zc (1 - zc)                 (dsig != nullptr; zc = dsig[((m / dsig_div) % dsig_rows) * ld_dsig + n])
//   t = alpha * t
//   t = t + beta * cin[m * ld_cin + n]  (cin != nullptr)
//   D[m * ldd + n] = t
//
// A operands: a_kmajor -> A(m,k) = A[m * lda + k], else A(m,k) = A[k * lda + m].
// B operands: b_kmajor -> B(k,n) = B[n * ldb + k], else B(k,n) = B[k * ldb + n].
// Both pairs share layouts but have their own K and leading dimensions.
//
// FP16 copies.  The tensor core reads a TF32 operand as its 11 leading significant bits.  FP16 has as many, so a copy
// X 2^e in FP16, rounded to nearest as TMA rounds on its way to TF32, holds the same operand (up to the power of two) wherever
// X 2^e is a normal FP16 number, takes half the bytes and is multiplied at twice the rate.  HalfInfo, in device memory, says
// which power of two, how large the matrix's largest magnitude is, and whether the copy may be used: `bad` is set by whoever
// writes it when an element overflows, is infinite or NaN, or when a whole run of a row or of a column lies so low that FP16's
// denormals would cost it precision (kHalfLeast).  The contraction kernels look at it and read the FP32 matrix instead.
// row1, col1: largest sum of the magnitudes of a row and of a column, in units of 2^(-e - 4) (0: not known).
struct alignas(16) HalfInfo { int e; unsigned amax; unsigned bad; unsigned pad; unsigned long long row1, col1; };
// Copy of a matrix, stored with leading dimension ld (a multiple of 8, 16-byte aligned, followed by >= 128 readable bytes).
struct HalfMat { void* p = nullptr; int64_t ld = 0; HalfInfo* info = nullptr; };
// A run of elements of a row (32 or 128) or column (16, or more) whose largest scaled magnitude is below this (and not zero) makes
// a copy bad: above it the rounding of a denormal, at most 2^-25, stays below the 2^-12 by which rounding to 11 bits changes the
// run's largest element.  (Runs of 2 and 8 elements were too short: a few saturated neurons have them, and one run decides over a
// whole matrix.  For the same reason what a contraction leaves over at the end of a row or column, shorter than a run, is not judged
// by itself: the row's or column's runs are.)
constexpr float kHalfLeast = 1.220703125e-4f;   // 2^-13

struct GemmArgs {
  int M = 0, N = 0;
  const float* A1 = nullptr; const float* B1 = nullptr; int K1 = 0; int64_t lda1 = 0, ldb1 = 0;
  const float* A2 = nullptr; const float* B2 = nullptr; int K2 = 0; int64_t lda2 = 0, ldb2 = 0;
  bool a1_split_fresh = false;   // caller's word that A1 is, unchanged, the A1 of the previous contraction
  int chunk_kb = 1;              // FP32-accurate tensor-core form: 64-term k-blocks per accumulation in tensor memory
  bool whole_tiles = false;      // ... without K slices (no workspace)
  bool a_kmajor = true, b_kmajor = true;
  bool mn_padded = false;  // every MN-major operand is followed by >= 128 readable bytes
  int two_cta = -1;        // tensor-core kernel: -1 choose, 0 one CTA per tile, 1 CTA pair per 256-row tile
  float* D = nullptr; int64_t ldd = 0;
  const float* bias = nullptr;
  bool sigmoid = false;
  const float* dsig = nullptr; int64_t ld_dsig = 0; int dsig_rows = 1; int dsig_div = 1;
  float alpha = 1.f;
  const float* cin = nullptr; int64_t ld_cin = 0; float beta = 0.f;
  // CTA-pair kernel, and for hout the streaming kernel of a short K as well (no bias, no cin).  half: every operand has a copy in h (A1, B1, A2, B2).  hout: a copy of D is written as well, scaled
  // by a bound on D from the operands' infos (all in h, with or without copies; the second pair's matrices, or the only pair's,
  // bound the bias too); h_next: infos of what the next contraction adds to hout's product (see out_exponent).
  bool half = false;
  HalfMat h[4];
  HalfMat hout;
  const HalfInfo* h_next[3] = {nullptr, nullptr, nullptr};
};

// FP32 fused-multiply-add GEMM (any shape, any alignment).  Returns launches made.
int launch_gemm_ffma(const GemmArgs& g, cudaStream_t st);

// TF32 tensor-core GEMM (tcgen05 + TMA).  Operands must be 16-byte aligned with leading dimensions
// that are multiples of 4 floats (TMA strides); gemm_tf32_eligible says whether a problem qualifies.
// *err_flag receives a non-zero code if a bounded device-side wait ran out.  Returns launches made,
// or -1 if a tensor map could not be encoded.
// sk_ws / sk_flags: optional workspace of gemm_tf32_workspace_floats() floats and
// gemm_tf32_workspace_flags() ints that lets the two-CTA kernel cut the tiles left over after its whole
// waves along K over the CTA pairs; pass nullptr to keep whole tiles.  The flags must be zero before the
// first launch; every launch that completes leaves them zero again (after a launch that gave up on a
// bounded wait they must be cleared by the caller).
bool gemm_tf32_eligible(const GemmArgs& g);
int64_t gemm_tf32_workspace_floats();
int gemm_tf32_workspace_flags();
int launch_gemm_tf32(const GemmArgs& g, int* err_flag, float* sk_ws, int* sk_flags, cudaStream_t st);
// Up to six problems, each suited to the CTA-pair kernel (M > 128, N >= 128), as ONE launch whose pairs walk a
// common, host-balanced work list.  Whole tiles only.
//   dep_prob == nullptr: independent problems, longest tiles first; the tiles of one fill the partial last wave
//   of another.
//   dep_prob != nullptr: a chain in the given order; problem i reads, as its FIRST A operand (row panels) or, with
//   dep_all[i] != 0, as an operand whose K runs over the producer's rows, the output of problem dep_prob[i] < i
//   (-1: none).  The consumer's tiles wait (bounded) for the producer's, so the layers of a pass overlap instead
//   of each draining the GPU.  `done`: device scratch of n * done_stride ints (done_stride > M / 256 + 1),
//   cleared by the call.
// Returns launches made, or -1 if the group cannot run this way (run the problems one by one, in order).
constexpr int kGemmGroupMax = 6;
bool gemm_tf32_group_eligible(const GemmArgs* gs, int n);
int launch_gemm_tf32_group(const GemmArgs* gs, int n, const int* dep_prob, const int* dep_all, int* done,
                           int done_stride, int* err_flag, cudaStream_t st);

// The work list of such a launch, computed without a device (see gemm_tf32.cu); for tests of the host logic.
int gemm_tf32_plan_group(int n, const int* M, const int* N, const int* K, int pairs, int keep_order, int* counts,
                         int* waves, int* order_out, int* tiles_out);
double gemm_tf32_group_makespan(int n, const int* M, const int* N, const int* K, int keep_order);

// FP16 copies by passes of their own (half_copy.cu), at most kHalfSegs matrices a launch.  launch_half_amax starts an info
// afresh from the largest magnitude of `count` consecutive floats and clears the n_reset infos from `reset` on; acc:
// kHalfSegs + 1 words, zero before the first launch and after every one; the n_sums words from `sums` on are cleared as well.
// launch_half_copy writes the copies and marks the bad ones.  Both return launches made, or -1.
constexpr int kHalfSegs = 8;
struct HalfAmaxJob { const float* src; int64_t count; HalfInfo* info; };
// fresh: the info holds the largest magnitude alone (whoever wrote the matrix has reported it): the scale is said here.
// from: the info that has the scale, if it is not the copy's own (which is told scale and largest magnitude then).  row_sums,
// col_sums: `rows` and `cols` words, zero: the sums of magnitudes are formed there, the largest goes into the info.
struct HalfCopyJob {
  const float* src; int64_t rows; int cols; int64_t ld; HalfMat out; bool fresh = false;
  const HalfInfo* from = nullptr; unsigned long long* row_sums = nullptr; unsigned long long* col_sums = nullptr;
};
int launch_half_amax(const HalfAmaxJob* jobs, int n, unsigned* acc, HalfInfo* reset, int n_reset, unsigned long long* sums, int64_t n_sums, cudaStream_t st);
int launch_half_copy(const HalfCopyJob* jobs, int n, cudaStream_t st);

// FP32-accurate contraction on the FP16 tensor cores (gemm_f16x3.cu): any shape and alignment, because it reads
// split copies of its operands.
//   SplitOperand  the two FP16 parts of a stored matrix X (leading dimension a multiple of 8, 16-byte aligned) and one
//                 byte per 128 x 128 cell of it, cells_ld of them per 128 rows: the exponent e of X 2^e = hi + lo, or the mark
//                 that the parts do not hold the cell and the contraction is to read X itself, which GemmArgs points to.
//   SplitJob      one matrix to be split.
// ops: A1, B1, A2, B2.  ws: gemm_f16x3_workspace_floats(g) floats (K slices; never more than
// gemm_tf32_workspace_floats()).  Both return launches made, or -1 if the launch failed.
struct SplitOperand { const void* hi = nullptr; const void* lo = nullptr; int64_t ld = 0; const int8_t* cells = nullptr; int cells_ld = 0; };
struct SplitJob {
  const float* src; int64_t rows; int cols; int64_t ld;
  void* hi; void* lo; int64_t ld_out; int8_t* cells;
};
// Bytes that hold the cells of any matrix of at most `cap` elements with its rows rounded up to 8: cap / 4096 where it has a
// cell's rows and columns or more, else one per 128 rows (of 8 elements at least) or columns.
inline int64_t split_cell_bytes(int64_t cap) { return cap / 128 + 16; }
constexpr int kSplitSegs = 8;
bool gemm_f16x3_usable();
double gemm_f16x3_estimate_us(const GemmArgs& g);
int64_t gemm_f16x3_workspace_floats(const GemmArgs& g);
int launch_gemm_f16x3(const GemmArgs& g, const SplitOperand* ops, float* ws, int* err_flag, cudaStream_t st);
int launch_split_f16(const SplitJob* jobs, int n, cudaStream_t st);

// Whole passes of a small network (small_net.cu).  kind 0: G^S v, 1: block-diagonal G^S v, 2: loss and gradient, 3: loss,
// 4: row gather and stored forward pass.  The blocks' sums go to scratch (small_net_blocks(rows) * n floats) and their losses to
// loss (one double per block); launch_small_net then writes out = alpha * sum + beta * cin and *loss_out.  theta_sq (kinds 2, 3)
// receives theta^T theta.  Returns launches made, or -1 if a launch failed.
constexpr int kSmallLayers = 8;
constexpr double kSmallUs = 42.0;       // estimated time up to which a pass goes this way (see small_net_fits) ...
constexpr double kSmallUsPerElement = 20e-6;   // ... and what is added to it per row and neuron
struct SmallNet {
  int L, n;
  int w[kSmallLayers + 1], w_off[kSmallLayers + 1], b_off[kSmallLayers + 1];
  int64_t rows;
  const float* theta; const float* v;
  const float* z[kSmallLayers];         // z^0 .. z^{L-1} of the subsample (kinds 0, 1), or z[0] = X (2, 3, 4)
  float* z_out[kSmallLayers + 1];       // kind 4: where the gathered rows and z^1 .. z^L go
  const int32_t* idx; int64_t x_rows; int* err_flag;   // kind 4
  const float* Y;
  float* scratch; double* loss; double* theta_sq;
};
int64_t small_net_blocks(int64_t rows);
bool small_net_fits(const SmallNet& a, int kind);
int launch_small_net(const SmallNet& a, int kind, float alpha, const float* cin, float beta, float* out, double* loss_out, cudaStream_t st);

// Streaming FP32 kernels for contractions with one dimension <= 16 (the n_L-wide output layer).
// gemm_thin_kind says which of them (if any) takes a problem; THIN_M needs a scratch buffer of
// gemm_thin_scratch_floats(g) floats.  launch_gemm_thin returns the launches made (0 = not taken).
enum ThinKind { THIN_NONE = 0, THIN_N = 1, THIN_M = 2, THIN_K = 3 };
ThinKind gemm_thin_kind(const GemmArgs& g);
int64_t gemm_thin_scratch_floats(const GemmArgs& g);
int launch_gemm_thin(const GemmArgs& g, float* scratch, cudaStream_t st);

// A one-CTA kernel whose bounded wait (limit_ns) can never be satisfied: writes code 9 to *err_flag.
int launch_timeout_probe(int* err_flag, unsigned long long limit_ns, cudaStream_t st);

// ---- vector / memory-bound kernels -------------------------------------------------------------
// Row gather dst[r][:] = src[idx[r]][:]; rows with idx outside [0, src_rows) are zero-filled and
// *err_flag is set to 1.
int launch_gather_rows(const float* src, int64_t src_rows, int cols, const int32_t* idx, int64_t n_idx,
                       float* dst, int* err_flag, cudaStream_t st);

// out[j] = alpha * sum_r A[r * lda + j] + beta * cin[j]  (cin may be nullptr), j < cols.
// scratch: at least colsum_scratch_floats(rows, cols) floats.
int64_t colsum_scratch_floats(int64_t rows, int cols);
int launch_colsum(const float* A, int64_t rows, int cols, int64_t lda, float alpha, const float* cin,
                  float beta, float* out, float* scratch, cudaStream_t st);

// Squared loss and its derivative for a row batch: delta = 2 (Z - Y) (delta may be nullptr),
// partial[b] = sum over the block's elements of (Z - Y)^2 in double.  Returns blocks via *n_partials.
int loss_num_partials(int64_t count);
int launch_loss_delta(const float* Z, const float* Y, int64_t count, float* delta, double* partial,
                      cudaStream_t st);

// Fixed-order double-precision sum of `count` partials: *out (+)= sum.
int launch_sum_partials(const double* partial, int count, double* out, bool accumulate, cudaStream_t st);

// out[i] = a x[i] + b y[i]; out may be x or y.
int launch_axpby(int64_t n, float a, const float* x, float b, const float* y, float* out, cudaStream_t st);

// Stored Jacobian factors (d z^L / d s^m per sample, Section 3.3.1).  D is [rows * nL][n] with row i * nL + u.
// factor_last: D[(i, u)][t] = WL[u * n + t] * z (1 - z), z = Zprev[i * n + t]   (layer L-1 from the linear output layer)
int launch_factor_last(const float* WL, const float* Zprev, int64_t rows, int nL, int n, float* D, cudaStream_t st);
// factor_apply, for every neuron group T_b of the layer (groups contiguous, boundaries floor(b n / groups)) and
// every stream a (U and Q hold `streams` matrices [rows][n], stream_stride floats apart):
//   p_u = sum_{j in T_b} D[(i,u)][j] U_a[i][j];  Q_a[i][j] = 2 sum_u D[(i,u)][j] p_u for j in T_b
// (Eqs. direct-JV-cost, JTv; B = 2I).  n_L <= 32.  info (may be null): its amax is raised to Q's largest magnitude.
// factor_apply_reports: whether asking for it costs less than the copies save (columns of the widest group).  Not where the general form
// has n_L above 10: fewer registers, more samples in flight, D out of L2 (512-3000-3000-16 at 4000 rows, a product with copies
// and without: 1156 and 1106 us, 1395 and 1188 split in two; with n_L = 10 700 and 727).
inline bool factor_apply_reports(int nL, int widest) { return nL <= 10 || widest <= 1024; }
int launch_factor_apply(const float* D, const float* U, int64_t rows, int nL, int n, int groups, int streams,
                        int64_t stream_stride, float* Q, HalfInfo* info, cudaStream_t st);
int launch_factor_apply_last(const float* WL, const float* Zprev, const float* U, int64_t rows, int nL, int n, float* Q,
                             HalfInfo* info, cudaStream_t st);

// ---- conjugate gradient ------------------------------------------------------------------------
// The n coordinates are cut into chunks, each inside one segment (one segment for the full system,
// one per layer for the block-diagonal systems).  Partial sums are per chunk, combined per segment
// in a fixed order in double precision.
struct CgChunk { int64_t start; int32_t len; int32_t seg; };
constexpr int kCgChunk = 4096;

struct CgSeg {           // per-segment scalars, device resident
  double rho;            // r^T r
  double pq;             // p^T q
  double gnorm2;         // ||g||^2
  float alpha, beta;
  int active;
  int first, count;      // this segment's chunks are entries [first, first + count) of the (segment-sorted) chunk table
  int pad;
};

// Device-resident state of one solve: where the kernels that end in a dot product take their tickets, what the
// last scalar update left for the host (sum of rho over segments, number of active segments), the number of steps
// in which some segment was still active, and the history of squared residual norms.
struct CgControl {
  unsigned int ticket;   // zero between launches
  int steps;
  int hist_len, hist_cap;
  double* hist;
  double out[2];
};

// r = -g, p = r, d = 0, partial[c] = sum r^2; then rho = gnorm2 = sum, active = rho > 0 && (tol <= 0 || tol < 1) per segment
int launch_cg_init(const float* g, float* d, float* r, float* p, const CgChunk* chunks, int n_chunks,
                   double* partial, CgSeg* seg, int n_seg, double tol, CgControl* ctl, cudaStream_t st);
// partial[c] = sum p q; with seg != nullptr also pq = sum, alpha = active ? rho / pq : 0 per segment
// (seg == nullptr: partials only, ctl unused)
int launch_cg_dot(const float* p, const float* q, const CgChunk* chunks, int n_chunks, double* partial,
                  CgSeg* seg, int n_seg, CgControl* ctl, cudaStream_t st);
// d += alpha p, r -= alpha q, partial[c] = sum r^2 (alpha per segment); then rho_new = sum, beta = rho_new / rho,
// rho = rho_new, active &= !(sqrt(rho) <= tol ||g||) per segment
int launch_cg_update(const float* p, const float* q, float* d, float* r, const CgChunk* chunks,
                     int n_chunks, CgSeg* seg, int n_seg, double tol, double* partial, CgControl* ctl, cudaStream_t st);
// p = r + beta p   (beta per segment)
int launch_cg_direction(const float* r, float* p, const CgChunk* chunks, int n_chunks, const CgSeg* seg,
                        cudaStream_t st);

}  // namespace gn
