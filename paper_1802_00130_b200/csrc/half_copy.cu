// FP16 copies of matrices (see HalfInfo in gn_kernels.h), by passes of their own: the largest magnitude, then the copy.  Copies
// of what a contraction computes are written by its epilogue instead (gemm_tf32.cu).
//
// Both are bound by HBM: 4 bytes read per element, then 4 read (from L2 where the matrix fits) and 2 written.
#include <cuda_fp16.h>

#include "gn_kernels.h"
#include "half_common.cuh"
#include "tc_common.cuh"

namespace gn {
namespace {

struct AmaxSeg { const float* src; long long count; HalfInfo* info; int vec; };
struct AmaxList { int n; AmaxSeg s[kHalfSegs]; HalfInfo* reset; int n_reset; unsigned long long* sums; long long n_sums; unsigned* acc; };

// Every block looks at its share of every matrix; the last block to finish writes the infos (acc[k]: largest magnitude of matrix
// k so far, acc[kHalfSegs]: blocks finished).
__global__ void __launch_bounds__(512) half_amax_kernel(const __grid_constant__ AmaxList list) {
  __shared__ unsigned warp_max[16];
  __shared__ int last;
  grid_dep_wait();
  grid_dep_launch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long stride = (long long)gridDim.x * 512;
  for (long long i = (long long)blockIdx.x * 512 + tid; i < list.n_sums; i += stride) list.sums[i] = 0ull;
  for (int k = 0; k < list.n; ++k) {
    const float* const src = dep(list.s[k].src);
    const long long n = list.s[k].count;
    unsigned m = 0u;
    long long i = (long long)blockIdx.x * 512 + tid;
    if (list.s[k].vec) {
      const float4* const q = reinterpret_cast<const float4*>(src);
      const long long n4 = n >> 2;
      for (; i + 3 * stride < n4; i += 4 * stride) {
        float4 x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = __ldg(q + i + j * stride);
#pragma unroll
        for (int j = 0; j < 4; ++j) m = max(m, max(max(magnitude(x[j].x), magnitude(x[j].y)), max(magnitude(x[j].z), magnitude(x[j].w))));
      }
      for (; i < n4; i += stride) {
        const float4 x = __ldg(q + i);
        m = max(m, max(max(magnitude(x.x), magnitude(x.y)), max(magnitude(x.z), magnitude(x.w))));
      }
      i = n4 * 4 + (long long)blockIdx.x * 512 + tid;
    }
    for (; i < n; i += stride) m = max(m, magnitude(__ldg(src + i)));
    m = __reduce_max_sync(0xffffffffu, m);
    __syncthreads();
    if (lane == 0) warp_max[warp] = m;
    __syncthreads();
    if (warp == 0) {
      m = __reduce_max_sync(0xffffffffu, warp_max[lane & 15]);
      if (lane == 0) atomicMax(list.acc + k, m);
    }
  }
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(list.acc + kHalfSegs, 1u) == gridDim.x - 1 ? 1 : 0;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  for (int k = tid; k < list.n_reset; k += 512) list.reset[k] = HalfInfo{0, 0u, 0u, 0u, 0ull, 0ull};
  if (tid < list.n) {
    const unsigned m = __ldcg(list.acc + tid);
    *list.s[tid].info = HalfInfo{half_exponent(m), m, m >= 0x7f800000u ? 1u : 0u, 0u, 0ull, 0ull};
    list.acc[tid] = 0u;
  }
  if (tid == 0) list.acc[kHalfSegs] = 0u;
}

// A block copies 128 rows x 128 columns, a warp 16 of the rows, a thread 4 of the columns (all requested before the first is
// used).  The runs looked at for kHalfLeast are a row's 128 and a column's 16 elements; the last of a row or column starts as far
// back as it needs to be whole (what it has in common with the one before is written twice, the same).
//
// Sums of magnitudes, where they are asked for, are formed as whole numbers (a thread's part rounded up), so that the order in which
// the blocks add theirs does not matter; whoever adds takes the sum so far to the maximum, and the last to add has the whole
// one.  A vector of 9.6e6 elements takes 19 us, 12 without them.
constexpr int COPY_CELL = 128, COPY_ROWS = 16;
struct CopySeg { const float* src; long long rows; int cols; long long ld; __half* out; long long ld_out; HalfInfo* info; int cells_ld, cell0, vec, fresh; const HalfInfo* from; unsigned long long* row_sums; unsigned long long* col_sums; };
struct CopyList { int n; CopySeg s[kHalfSegs]; };

// The largest of a warp's sums to the maximum at `to`.
__device__ __forceinline__ void report_sum(unsigned long long* to, unsigned long long sum, int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum = max(sum, __shfl_xor_sync(0xffffffffu, sum, o));
  if (lane == 0 && sum > __ldcg(to)) atomicMax(to, sum);
}

__global__ void __launch_bounds__(256) half_copy_kernel(const __grid_constant__ CopyList list) {
  grid_dep_wait();
  grid_dep_launch();
  int k = 0;
  while (k + 1 < list.n && (int)blockIdx.x >= list.s[k + 1].cell0) ++k;
  const CopySeg& s = list.s[k];
  const float* const src = dep(s.src);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cell = (int)blockIdx.x - s.cell0, rc = cell / s.cells_ld;
  const int c_own = (cell - rc * s.cells_ld) * COPY_CELL;
  const int c0 = s.cols >= COPY_CELL && s.cols % 4 == 0 ? min(c_own, s.cols - COPY_CELL) : c_own;
  const long long r_own = (long long)rc * COPY_CELL + warp * COPY_ROWS;
  const long long r0 = s.rows >= COPY_ROWS && r_own < s.rows ? min(r_own, s.rows - COPY_ROWS) : r_own;
  const int skip_c = c_own - c0, skip_r = (int)(r_own - r0);      // columns and rows that are others' as well
  const int c = c0 + 4 * lane, left = s.cols - c;
  const int n_rows = (int)max(0ll, min((long long)COPY_ROWS, s.rows - r0));
  float4 x[COPY_ROWS];
  const float* q = src + r0 * s.ld + c;
#pragma unroll
  for (int i = 0; i < COPY_ROWS; ++i, q += s.ld) {
    x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < n_rows && left > 0) {
      if (s.vec) {
        x[i] = __ldg(reinterpret_cast<const float4*>(q));
      } else {
        x[i].x = __ldg(q);
        if (left > 1) x[i].y = __ldg(q + 1);
        if (left > 2) x[i].z = __ldg(q + 2);
        if (left > 3) x[i].w = __ldg(q + 3);
      }
    }
  }
  int e = 0;
  if (s.fresh) {
    const unsigned m = __ldcg(&s.info->amax);
    e = half_exponent(m);
    if (cell == 0 && threadIdx.x == 0) {
      __stcg(&s.info->e, e);
      if (m >= 0x7f800000u) atomicOr(&s.info->bad, 1u);
    }
  } else if (s.from) {
    const int4 f = __ldcg(reinterpret_cast<const int4*>(s.from));
    e = f.x;
    if (cell == 0 && threadIdx.x == 0) {
      __stcg(&s.info->e, e);
      __stcg(&s.info->amax, (unsigned)f.y);
      if (f.z) atomicOr(&s.info->bad, 1u);
    }
  } else {
    e = __ldcg(&s.info->e);
  }
  const float sc = half_scale(e);
  float col[4] = {0.f, 0.f, 0.f, 0.f}, col_sum[4] = {0.f, 0.f, 0.f, 0.f};
  unsigned row_sum = 0u;                          // of this warp's row number `lane`
  HalfCheck check;
  __half* o = s.out + r0 * s.ld_out + c;
#pragma unroll
  for (int i = 0; i < COPY_ROWS; ++i, o += s.ld_out) {
    const float y[4] = {x[i].x * sc, x[i].y * sc, x[i].z * sc, x[i].w * sc};
    float row = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) { col[j] = fmaxf(col[j], fabsf(y[j])); row = fmaxf(row, fabsf(y[j])); }
    if (s.row_sums) {
      const float mine = 4 * lane < skip_c ? 0.f : fabsf(y[0]) + fabsf(y[1]) + fabsf(y[2]) + fabsf(y[3]);
      const unsigned part = __reduce_add_sync(0xffffffffu, __float2uint_ru(mine * (float)(1 << kHalfNormExp)));
      if (lane == i) row_sum = part;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) col_sum[j] += i < skip_r ? 0.f : fabsf(y[j]);
    check.run(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(row))));
    if (i < n_rows && left > 0) {                 // (ld_out is a multiple of 8: a whole group always fits)
      const __half2 a = __floats2half2_rn(y[0], y[1]), b = __floats2half2_rn(y[2], y[3]);
      *reinterpret_cast<uint2*>(o) = make_uint2(*reinterpret_cast<const unsigned*>(&a), *reinterpret_cast<const unsigned*>(&b));
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) check.run(col[j]);
  if (__any_sync(0xffffffffu, check.bad()) && lane == 0) atomicOr(&s.info->bad, 1u);
  if (s.row_sums) {
    unsigned long long sum = lane >= skip_r && lane < n_rows ? atomicAdd(s.row_sums + r0 + lane, (unsigned long long)row_sum) + row_sum : 0ull;
    report_sum(&s.info->row1, sum, lane);
  }
  if (s.col_sums) {
    __shared__ unsigned part[COPY_CELL];
    if (threadIdx.x < COPY_CELL) part[threadIdx.x] = 0u;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) atomicAdd(part + 4 * lane + j, __float2uint_ru(col_sum[j] * (float)(1 << kHalfNormExp)));
    __syncthreads();
    if (threadIdx.x < COPY_CELL) {
      const int cc = c0 + (int)threadIdx.x;
      unsigned long long sum = cc >= c_own && cc < s.cols ? atomicAdd(s.col_sums + cc, (unsigned long long)part[threadIdx.x]) + part[threadIdx.x] : 0ull;
      report_sum(&s.info->col1, sum, lane);
    }
  }
}

}  // namespace

int launch_half_amax(const HalfAmaxJob* jobs, int n, unsigned* acc, HalfInfo* reset, int n_reset, unsigned long long* sums, int64_t n_sums, cudaStream_t st) {
  if (n < 1 || n > kHalfSegs) return -1;
  AmaxList list{};
  list.n = n; list.reset = reset; list.n_reset = n_reset; list.sums = sums; list.n_sums = n_sums; list.acc = acc;
  long long total = 0;
  for (int i = 0; i < n; ++i) {
    list.s[i] = AmaxSeg{jobs[i].src, (long long)jobs[i].count, jobs[i].info, aligned16(jobs[i].src) ? 1 : 0};
    total += jobs[i].count;
  }
  long long blocks = (total + 4095) / 4096;        // (two groups of 4 per thread at least: a small matrix is a chain of round trips)
  if (blocks > 2LL * num_sms()) blocks = 2LL * num_sms();
  return launch_pdl(half_amax_kernel, (int)blocks, 512, 0, st, list) == cudaSuccess ? 1 : -1;
}

int launch_half_copy(const HalfCopyJob* jobs, int n, cudaStream_t st) {
  if (n < 1 || n > kHalfSegs) return -1;
  CopyList list{};
  long long cells = 0;
  for (int i = 0; i < n; ++i) {
    const HalfCopyJob& j = jobs[i];
    CopySeg& s = list.s[list.n++];
    s.src = j.src; s.rows = j.rows; s.cols = j.cols; s.ld = j.ld;
    s.out = static_cast<__half*>(j.out.p); s.ld_out = j.out.ld; s.info = j.out.info;
    s.cells_ld = (j.cols + COPY_CELL - 1) / COPY_CELL;
    s.cell0 = (int)cells; s.fresh = j.fresh ? 1 : 0; s.from = j.from; s.row_sums = j.row_sums; s.col_sums = j.col_sums;
    s.vec = j.cols % 4 == 0 && j.ld % 4 == 0 && aligned16(j.src);
    cells += (j.rows + COPY_CELL - 1) / COPY_CELL * s.cells_ld;
    if (cells > 0x7fffffff) return -1;
  }
  return launch_pdl(half_copy_kernel, (int)cells, 256, 0, st, list) == cudaSuccess ? 1 : -1;
}

}  // namespace gn
