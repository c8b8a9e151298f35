// FP32-accurate contractions on the FP16 tensor cores (sm_100a).
//
// Every operand X arrives as two FP16 matrices, cut into cells of 128 x 128 elements with an exponent e each:
// X 2^e = hi + lo, hi = rn16(X 2^e), lo = rn16(X 2^e - hi), where 2^e takes the largest element of the cell to [2^14, 2^15).
// hi and lo carry 11 significant bits each, so |X - (hi + lo) 2^-e| <= 2^-23 |x| for elements down to 2^-16 of the cell's
// largest, and <= 2^-39 of that below.  A logical product A B is Alo Bhi + Ahi Blo + Ahi Bhi (the dropped Alo Blo is below
// 2^-22 |a b|).
//
// A cell is as long as a chunk of K (below) at most and as wide as a CTA's rows, so the exponents cost the main loop nothing:
// what a chunk adds to the running sums is multiplied by a power of two anyway, which now belongs to the chunk's cells.
// A cell with a row or a column that lies wholly below 2^-20 of its largest element, or with an infinity or NaN, is marked by
// the splitting pass instead, and the epilogue warps compute the chunks that meet it as FP32 FMAs from the operands
// themselves (fma_chunk): the range of a matrix costs time, not precision.  Why 2^-20: at that limit the elements of the row
// or column are off by 5e-7 of its largest (root mean square), which is what an FP32 sum of some thousand terms leaves; and
// the deltas of a scalar output, an outer product, have a row below 2^-18 in one of seventy products over 2000 rows.
//
// Why FP16 and not TF32 parts: the two formats have the same 11-bit significand, but kind::f16 runs at twice the rate
// of kind::tf32 and its parts are half the bytes, so the three products cost 1.5 TF32 products instead of 3 and the
// parts together are no larger than the FP32 operand.  What TF32 parts have and FP16 parts lack is exponent range;
// the exponent per cell puts the range where the cell is.
//
// The tensor core adds into its FP32 accumulator with truncation, a bias that grows with the number of additions, so
// the K range is cut into chunks of 64 or 128 terms; each chunk is accumulated in tensor memory on its own (two
// 256-column accumulators alternate) and the epilogue warps add the chunks into running sums held in registers, in
// FP32 with round-to-nearest.  Inside a k-block the small products go first, so only a third of the additions
// meet a full-size accumulator.  Measured against float64 on N(0, 1) operands: 1.5e-7 to 2.8e-7 for K = 64 to 32768 with
// chunks of 64 terms (the FP32 FMA GEMM: 1.4e-7 to 3.2e-6), 3.8e-7 to 4.2e-7 with 128, which is 5 to 10 % faster.
//
//   warps 0..3   (56 registers)   0 = TMA producer, 1 = MMA issuer, 2 = tensor-memory allocation, 3 idle
//   warps 4..11  (224 registers)  epilogue, two warps per 32-lane quadrant of tensor memory
//
// A CTA pair computes a 256 x bn tile (tcgen05.mma.cta_group::2), CTA r staging its 128 rows of A and half of the B
// tile; the pair protocol is that of gemm_tf32.cu.  Tiles left over after the whole rounds of the pairs are cut along K
// into slices whose partial sums go to a workspace and are added, in slice order, by a second kernel that also runs
// the epilogue options (no CTA waits for another one's slice).
#include <cuda_fp16.h>

#include "gn_kernels.h"
#include "tc_common.cuh"

namespace gn {
namespace {

constexpr int H_BM = 128, H_BK = 64, H_BN_MAX = 256;
constexpr int H_THREADS = 384, H_STAGES = 3;
constexpr int H_PART_BYTES = H_BM * H_BK * 2;             // 16 KB: 128 rows x 64 FP16
constexpr int H_STAGE_BYTES = 4 * H_PART_BYTES;           // A hi, A lo, B-half hi, B-half lo
constexpr int H_REGS_LOW = 56, H_REGS_HIGH = 224;         // 128 * 56 + 256 * 224 = 384 * 168
constexpr int H_STG_BYTES = 8 * 32 * 32 * 4;              // one 32 x 32 staging tile per epilogue warp
constexpr int H_SMEM_BYTES = H_STAGES * H_STAGE_BYTES + H_STG_BYTES + 1024 + 256;
static_assert(H_SMEM_BYTES <= 232448, "more shared memory than a block can have");

struct HEpilogue {
  int M, N;
  float* D; long long ldd;
  const float* bias; int sigmoid;
  const float* dsig; long long ld_dsig; int dsig_rows, dsig_div, dsig_direct;
  float alpha;
  const float* cin; long long ld_cin; float beta;
  int vec;                                   // N % 4 == 0; D, bias, dsig, cin 16-byte aligned, leading dimensions % 4 == 0
};

struct HParams {
  HEpilogue e;
  int n_pairs;                               // logical operand pairs accumulated into one tile (1 or 2)
  int kblocks[2];
  int a_mn, b_mn;
  // of A1, B1, A2, B2: the cells' exponents (kMarked: see the top), row by row of the stored matrix, and the matrix itself
  const int8_t* cells[4]; int cells_ld[4];
  const float* src[4]; long long ld_src[4];
  int K[2];
  int chunk_log;                             // log2 of the k-blocks per accumulation in tensor memory (0 or 1)
  int chunks0;                               // chunks of the first operand pair
  // work list: items 0 .. whole - 1 are whole tiles, then slice sl of left-over tile j (tile whole + j) is item
  // whole + sl * rem + j; pair q takes items q, q + P, ...
  int bn, tiles_n, whole, rem, slices, items, P;
  float* ws;                                 // partial sums of the left-over tiles: [slices][rem][256][bn]
  int* err;
};

struct HMaps { CUtensorMap m[8]; };          // per pair: A hi, A lo, B hi, B lo

constexpr int CELL = 128;                    // = H_BM = the longest chunk of K
constexpr int kMarked = 127;
constexpr unsigned FAR_LOG = 20;             // see the top
// Exponent e of the scale 2^e for a cell whose largest magnitude has this bit pattern: -113 .. 126, 0 for a cell of zeros.
__device__ __forceinline__ int scale_exponent(unsigned amax_bits) {
  const int p = (int)(amax_bits >> 23) - 127;             // (denormals: -127)
  return amax_bits ? min(14 - p, 126) : 0;
}
__device__ __forceinline__ float exp2_int(int e) {        // 2^e, -149 <= e <= 127
  return __uint_as_float(e < -126 ? 1u << (e + 149) : (unsigned)(e + 127) << 23);
}

__device__ __forceinline__ void mma2_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}

// The epilogue as it is after grid_dep_wait (see dep()).
__device__ __forceinline__ HEpilogue after_wait(const HEpilogue& in) {
  HEpilogue e = in;
  e.bias = dep(e.bias); e.dsig = dep(e.dsig); e.cin = dep(e.cin);
  return e;
}

__device__ __forceinline__ long long dsig_row(const HEpilogue& e, int m) {
  return e.dsig_direct ? m : (m / e.dsig_div) % e.dsig_rows;
}

__device__ __forceinline__ float finish(const HEpilogue& e, float x, float bz, float z, float c) {
  x += bz;
  if (e.sigmoid) x = sigmoid_from(expf(-x));
  if (e.dsig) x *= z * (1.f - z);
  x *= e.alpha;
  if (e.cin) x = fmaf(e.beta, c, x);
  return x;
}

// Place of columns 4 q .. 4 q + 3 of row r in a staging tile: the 16-byte groups of a row are permuted by the row's low
// bits, so that a column of groups, a row of groups and a row of single elements are all free of bank conflicts.
__device__ __forceinline__ uint32_t stg_at(uint32_t stg, int r, int q) { return stg + (uint32_t)(r * 128 + ((q ^ (r & 7)) << 4)); }
// (through shared-space addresses: behind a generic pointer the compiler must keep every read of the tile behind the
// global store before it, one latency per row)
__device__ __forceinline__ void stg_put(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
template <int W>
__device__ __forceinline__ void stg_get(uint32_t a, float* v) {
  if (W == 4)
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[W > 1 ? 1 : 0]), "=f"(v[W > 2 ? 2 : 0]), "=f"(v[W > 3 ? 3 : 0]) : "r"(a));
  else
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[0]) : "r"(a));
}

// W floats, read where the call stands.
template <int W>
__device__ __forceinline__ void load_now(const float* p, float* v) {
  if (W == 4)
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[W > 1 ? 1 : 0]), "=f"(v[W > 2 ? 2 : 0]), "=f"(v[W > 3 ? 3 : 0]) : "l"(p));
  else
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v[0]) : "l"(p));
}

// A warp's share of a finished tile through the epilogue options and out: `n_mine` chunks of 32 rows x 32 columns, 64
// columns apart from column nb0 on, read back from tensor memory at `ta` (lane = row) and turned through the warp's
// staging tile so that accesses to global memory are whole rows of 128 bytes whatever the alignment of the matrices.
// VEC (16-byte aligned rows, N a multiple of 4): lane l takes columns 4 (l % 8) .. + 3 of rows l / 8, l / 8 + 4, ...;
// otherwise lane = column, one row per access.  MODE fixes the options at compile time: 0 = alpha * x (+ bias), 1 =
// sigmoid, 2 = times the sigmoid derivative of dsig, 3 = plus beta * cin, 4 = any combination.  Eight warps with
// nothing to hide latency behind: what bounds this is the operand's round trips, so the operand of modes 2 and 3 is
// requested for a whole chunk before the first use.  That takes registers the 128 running sums would not leave, hence
// their detour through the tensor memory they came from, and the kernel is compiled per form so that no form's
// registers are another's spills.  (Requested 2 to 4 rows at a time beside the sums, all forms in one kernel: 12000 x
// 2000 x 2000 with dsig 319 us, now 236; 4001 x 1201 x 617 with unaligned rows 83, now 58.)
template <int MODE, bool VEC>
__device__ __forceinline__ void store_tile(const HEpilogue& e, uint32_t stg, uint32_t ta, int n_mine, int m0, int rows, int nb0, int lane) {
  constexpr int W = VEC ? 4 : 1, STEP = VEC ? 4 : 1, IT = 32 / STEP;
  constexpr bool ONE_OP = MODE == 2 || MODE == 3;
  const int col = VEC ? (lane & 7) * 4 : lane, r_first = VEC ? lane >> 3 : 0;
  const bool use_sigm = MODE == 4 ? e.sigmoid != 0 : MODE == 1;
  const bool use_dsig = MODE == 4 ? e.dsig != nullptr : MODE == 2;
  const bool use_cin = MODE == 4 ? e.cin != nullptr : MODE == 3;
  float op[ONE_OP ? IT : 1][W];
#pragma unroll 1
  for (int j = 0; j < n_mine; ++j) {
    const int n = nb0 + 64 * j + col;
    if (ONE_OP) {
      // rows and columns past the end read the last ones: with a condition around it the compiler moves each load down
      // to its use, one round trip per row
      const int nc = min(n, e.N - W);
      const float* const src = MODE == 2 ? e.dsig + nc : e.cin + nc;
      const long long ld = MODE == 2 ? e.ld_dsig : e.ld_cin;
#pragma unroll
      for (int i = 0; i < IT; ++i) {
        const int m = m0 + min(r_first + i * STEP, rows - 1);
        load_now<W>(src + (MODE == 2 ? dsig_row(e, m) : (long long)m) * ld, op[ONE_OP ? i : 0]);
      }
    }
    {
      float v[32];
      tmem_ld32(ta + (uint32_t)(64 * j), v);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        stg_put(stg_at(stg, lane, i >> 2), v[i], v[i + 1], v[i + 2], v[i + 3]);
      __syncwarp();
    }
    float xs[IT][W];                           // the whole chunk out of the staging tile before the first store
#pragma unroll
    for (int i = 0; i < IT; ++i) stg_get<W>(stg_at(stg, r_first + i * STEP, VEC ? lane & 7 : lane >> 2) + (VEC ? 0u : (lane & 3) * 4u), xs[i]);
    if (n < e.N) {
      float bz[W];
#pragma unroll
      for (int q = 0; q < W; ++q) bz[q] = 0.f;
      if (e.bias) {
        if (VEC) *reinterpret_cast<float4*>(bz) = __ldg(reinterpret_cast<const float4*>(e.bias + n));
        else bz[0] = __ldg(e.bias + n);
      }
#pragma unroll
      for (int i = 0; i < IT; ++i) {
        float z[W], c[W];
        if (MODE == 4) {                       // (rows past the end read the last one)
          const int m = m0 + min(r_first + i * STEP, rows - 1);
          if (use_dsig) load_now<W>(e.dsig + dsig_row(e, m) * e.ld_dsig + n, z);
          if (use_cin) load_now<W>(e.cin + (long long)m * e.ld_cin + n, c);
        }
#pragma unroll
        for (int q = 0; q < W; ++q) {
          float t = xs[i][q] + bz[q];
          if (use_sigm) t = sigmoid_from(expf(-t));
          if (use_dsig) { const float zz = MODE == 4 ? z[q] : op[ONE_OP ? i : 0][q]; t *= zz * (1.f - zz); }
          t *= e.alpha;
          if (use_cin) t = fmaf(e.beta, MODE == 4 ? c[q] : op[ONE_OP ? i : 0][q], t);
          xs[i][q] = t;
        }
      }
      // (the stores in a loop of their own, whole chunks without a test per row: with rows that are no multiple of four
      // floats every element is a store of its own, and what surrounds it counts)
      float* d = e.D + (long long)(m0 + r_first) * e.ldd + n;
      const long long step = STEP * e.ldd;
      if (rows == 32) {
#pragma unroll
        for (int i = 0; i < IT; ++i, d += step) {
          if (VEC) *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(xs[i]);
          else d[0] = xs[i][0];
        }
      } else {
#pragma unroll
        for (int i = 0; i < IT; ++i, d += step)
          if (r_first + i * STEP < rows) {
            if (VEC) *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(xs[i]);
            else d[0] = xs[i][0];
          }
      }
    }
  }
}

// Piece `i` of the chunk list of a K range: chunks of 1 or 2 k-blocks that never straddle the two operand pairs.
struct ChunkPos { int pair, kb0, kb1; };
__device__ __forceinline__ ChunkPos chunk_at(const HParams& p, int i) {
  ChunkPos c;
  c.pair = i >= p.chunks0 ? 1 : 0;
  c.kb0 = (i - (c.pair ? p.chunks0 : 0)) << p.chunk_log;
  c.kb1 = min(p.kblocks[c.pair], c.kb0 + (1 << p.chunk_log));
  return c;
}
__device__ __forceinline__ int chunk_count(const HParams& p) {
  return p.chunks0 + (p.n_pairs > 1 ? (p.kblocks[1] + p.chunk_log) >> p.chunk_log : 0);
}

// Item of the work list: its tile, its chunks c0 .. c1 - 1, and, for a K slice, where its partial sums go (else -1).
struct Item { int tile, c0, c1, slot; };
__device__ __forceinline__ Item item_at(const HParams& p, int i, int n_chunks) {
  if (i < p.whole) return Item{i, 0, n_chunks, -1};
  const int k = i - p.whole, sl = k / p.rem;
  return Item{p.whole + k - sl * p.rem, (int)((long long)n_chunks * sl / p.slices), (int)((long long)n_chunks * (sl + 1) / p.slices), k};
}

// Where a lane finds the exponents of the chunks it looks up for its warp in this tile: lanes 0..3 of the cells of B under the
// warp's four 32-column groups, lane 4 of A's cell of the CTA's rows (lanes without a cell repeat a neighbour's).
struct CellWalk { const int8_t* at[2]; int step[2]; };
__device__ __forceinline__ CellWalk cell_walk(const HParams& p, int m_cta, int n_warp, int n_cc_mine, int lane) {
  const bool is_a = lane >= 4;
  const int c = (is_a ? min(m_cta, p.e.M - 1) : min(n_warp + 64 * min(lane, max(n_cc_mine, 1) - 1), p.e.N - 1)) / CELL;
  CellWalk w;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int op = 2 * s + (is_a ? 0 : 1), ld = p.cells_ld[op];
    const bool k_rows = is_a ? p.a_mn : p.b_mn;            // K runs over the rows of the stored matrix
    w.step[s] = k_rows ? ld : 1;
    w.at[s] = p.cells[op] + (k_rows ? (long long)c : (long long)c * ld);
  }
  return w;
}
__device__ __forceinline__ int cell_exponent(const HParams& p, const CellWalk& w, int ch) {
  const int s = ch >= p.chunks0 ? 1 : 0, k = ((ch - (s ? p.chunks0 : 0)) << p.chunk_log) >> 1;      // (two k-blocks per cell)
  return __ldcg((s ? w.at[1] : w.at[0]) + (long long)k * (s ? w.step[1] : w.step[0]));
}

__device__ __forceinline__ void stg_put1(uint32_t a, float x) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory"); }

// A chunk of K as FP32 FMAs: sum_k A(m, k) B(k, n) for the warp's 32 rows from m_warp on and its groups of 32 columns, 64 apart
// from n_warp on, added to the running sums at `sums` in tensor memory (lane = row).  16 terms at a time go through the warp's
// staging tile, A's and B's 16 x 32 each; a thread takes 4 rows x 8 columns, three 16-byte reads for 32 FMAs.  Not meant
// to be fast: 12000 x 2000 x 2000 takes 0.21 ms with no cell marked, 0.71 ms with one column of A far below the others and
// 7.5 ms with every cell marked (the FMA GEMM: 2.3 ms).
__device__ __forceinline__ void fma_chunk(const HParams& p, const ChunkPos cp, uint32_t stg, int m_warp, int n_warp, int n_groups, int lane, uint32_t sums) {
  const float* const A = dep(p.src[2 * cp.pair]);
  const float* const B = dep(p.src[2 * cp.pair + 1]);
  const long long lda = p.ld_src[2 * cp.pair], ldb = p.ld_src[2 * cp.pair + 1];
  const int k_end = min(p.K[cp.pair], cp.kb1 * H_BK), M = p.e.M, N = p.e.N;
  const int k_of = lane & 15, mn_of = lane >> 4;           // K-major operands: 16 terms of two rows per access
#pragma unroll 1
  for (int j = 0; j < n_groups; ++j) {
    const int n0 = n_warp + 64 * j;
    float acc[4][8];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
    float a[16], b[16];
    const auto fetch = [&](int k0) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int ka = p.a_mn ? k0 + i : k0 + k_of, m = m_warp + (p.a_mn ? lane : 2 * i + mn_of);
        a[i] = ka < k_end && m < M ? __ldg(A + (p.a_mn ? ka * lda + m : m * lda + ka)) : 0.f;
        const int kb = p.b_mn ? k0 + i : k0 + k_of, n = n0 + (p.b_mn ? lane : 2 * i + mn_of);
        b[i] = kb < k_end && n < N ? __ldg(B + (p.b_mn ? kb * ldb + n : n * ldb + kb)) : 0.f;
      }
    };
    fetch(cp.kb0 * H_BK);
#pragma unroll 1
    for (int k0 = cp.kb0 * H_BK; k0 < k_end; k0 += 16) {
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int ra = p.a_mn ? i : k_of, m = p.a_mn ? lane : 2 * i + mn_of;
        stg_put1(stg_at(stg, ra, m >> 2) + (m & 3) * 4u, a[i]);
        const int rb = p.b_mn ? i : k_of, n = p.b_mn ? lane : 2 * i + mn_of;
        stg_put1(stg_at(stg, 16 + rb, n >> 2) + (n & 3) * 4u, b[i]);
      }
      __syncwarp();
      if (k0 + 16 < k_end) fetch(k0 + 16);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        float x[4], y[8];
        stg_get<4>(stg_at(stg, k, lane >> 2), x);
        stg_get<4>(stg_at(stg, 16 + k, 2 * (lane & 3)), y);
        stg_get<4>(stg_at(stg, 16 + k, 2 * (lane & 3) + 1), y + 4);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(x[u], y[v], acc[u][v]);
      }
    }
    __syncwarp();                                          // the block's sums, turned to lane = row
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        stg_put(stg_at(stg, (lane >> 2) * 4 + u, 2 * (lane & 3) + h), acc[u][4 * h], acc[u][4 * h + 1], acc[u][4 * h + 2], acc[u][4 * h + 3]);
    __syncwarp();
    float run[32];
    tmem_ld32(sums + (uint32_t)(64 * j), run);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float x[4];
      stg_get<4>(stg_at(stg, lane, q), x);
#pragma unroll
      for (int u = 0; u < 4; ++u) run[4 * q + u] += x[u];
    }
    tmem_st32(sums + (uint32_t)(64 * j), run);
    tmem_st_wait();
    __syncwarp();
  }
}

template <int MODE, bool VEC>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(H_THREADS, 1)
gemm_f16x3_kernel(const __grid_constant__ HMaps maps, const __grid_constant__ HParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + H_STAGES * H_STAGE_BYTES + H_STG_BYTES);
  uint64_t* empty = full + H_STAGES;
  uint64_t* acc_full = empty + H_STAGES;   // [2]
  uint64_t* acc_empty = acc_full + 2;      // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1;
  const int bn = p.bn, hb = p.bn >> 1;                     // hb: columns of B staged by each CTA
  const int n_chunks = chunk_count(p);

  if (threadIdx.x == 0) {
    for (int s = 0; s < H_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 16); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();
  grid_dep_launch();

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(H_REGS_LOW));
    if (warp == 0) {
      // ---------------------------------------------------------------- producer (both CTAs)
      const int b_chunks = p.b_mn ? (hb + 63) / 64 : 0;    // MN-major B: 64-column boxes
      const uint32_t b_bytes = p.b_mn ? (uint32_t)b_chunks * 8192u : (uint32_t)hb * 128u;
      const uint32_t pair_tx = 4u * (H_PART_BYTES + b_bytes);            // two CTAs x (hi + lo) x (A + B half)
      int it = 0;
      bool ok = true;
      for (int item = pair; item < p.items && ok; item += p.P) {
        const Item w = item_at(p, item, n_chunks);
        const int m0 = (w.tile / p.tiles_n) * (2 * H_BM) + (int)rank * H_BM;
        const int n0 = (w.tile % p.tiles_n) * bn + (int)rank * hb;
        for (int ch = w.c0; ch < w.c1 && ok; ++ch) {
          const ChunkPos cp = chunk_at(p, ch);
          const CUtensorMap* mp = &maps.m[4 * cp.pair];
          for (int kb = cp.kb0; kb < cp.kb1; ++kb, ++it) {
            const int s = it % H_STAGES;
            const uint32_t ph = (it / H_STAGES) & 1;
            int good = 1;
            if (lane == 0) good = wait_or_abort(&empty[s], ph ^ 1, abort_flag, p.err, 1) ? 1 : 0;
            good = __shfl_sync(0xffffffffu, good, 0);
            if (!good) { ok = false; break; }
            if (rank == 0 && lane == 0) mbar_expect_tx(&full[s], pair_tx);
            __syncwarp();
            const uint32_t full_leader = map_to_cta(smem_u32(&full[s]), 0);
            const int k0 = kb * H_BK;
            uint8_t* sa = smem + s * H_STAGE_BYTES;        // A hi | A lo | B hi | B lo
            uint8_t* sb = sa + 2 * H_PART_BYTES;
            if (!p.a_mn) {
              if (lane < 2) tma2_load_2d(sa + lane * H_PART_BYTES, &mp[lane], k0, m0, full_leader);
            } else if (lane < 4) {                         // lane = 2 * part + 64-row box
              tma2_load_2d(sa + (lane >> 1) * H_PART_BYTES + (lane & 1) * 8192, &mp[lane >> 1], m0 + 64 * (lane & 1), k0, full_leader);
            }
            if (!p.b_mn) {
              if (lane >= 8 && lane < 10) tma2_load_2d(sb + (lane - 8) * H_PART_BYTES, &mp[2 + lane - 8], k0, n0, full_leader);
            } else if (lane >= 8 && lane < 12 && (lane & 1) < b_chunks) {
              const int q = lane - 8;
              tma2_load_2d(sb + (q >> 1) * H_PART_BYTES + (q & 1) * 8192, &mp[2 + (q >> 1)], n0 + 64 * (q & 1), k0, full_leader);
            }
          }
        }
      }
    } else if (warp == 1 && rank == 0 && lane == 0) {
      // ---------------------------------------------------------------- MMA issuer (leader CTA only)
      // instruction descriptor: D = F32, A = B = F16, majors, N >> 3, M >> 4
      const uint32_t idesc = (1u << 4) | ((uint32_t)(p.a_mn ? 1 : 0) << 15) | ((uint32_t)(p.b_mn ? 1 : 0) << 16) |
                             ((uint32_t)(bn >> 3) << 17) | ((uint32_t)((2 * H_BM) >> 4) << 24);
      // K-major: 64 K elements per 128-byte row, one MMA (K = 16) advances 32 B; MN-major: 64-column chunks of 64 rows of
      // 128 B (8 KB), one MMA advances 16 rows.  8-row groups are 1024 B apart in both.
      const uint32_t a_lbo = p.a_mn ? 8192 : 16, b_lbo = p.b_mn ? 8192 : 16;
      const uint32_t a_step = p.a_mn ? 2048 : 32, b_step = p.b_mn ? 2048 : 32;
      int it = 0, ci = 0;                          // ring position, running chunk count (accumulator phase)
      bool ok = true;
      for (int item = pair; item < p.items && ok; item += p.P) {
        const Item w = item_at(p, item, n_chunks);
        for (int ch = w.c0; ch < w.c1 && ok; ++ch, ++ci) {
          const ChunkPos cp = chunk_at(p, ch);
          const int buf = ci & 1;
          const uint32_t aph = (ci >> 1) & 1;
          ok = wait_or_abort(&acc_empty[buf], aph ^ 1, abort_flag, p.err, 4);
          if (!ok) break;
          tc_fence_after();
          const uint32_t tmem_d = tmem_base + (uint32_t)(buf * H_BN_MAX);
          for (int kb = cp.kb0; kb < cp.kb1; ++kb, ++it) {
            const int s = it % H_STAGES;
            const uint32_t ph = (it / H_STAGES) & 1;
            ok = wait_or_abort(&full[s], ph, abort_flag, p.err, 2);
            if (!ok) break;
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + s * H_STAGE_BYTES);
            const uint32_t sb = sa + 2 * H_PART_BYTES;
            uint32_t acc = kb > cp.kb0 ? 1u : 0u;
#pragma unroll
            for (int k = 0; k < H_BK / 16; ++k) {          // small terms first
              const uint64_t ah = make_desc(sa + k * a_step, a_lbo, 1024, 2);
              const uint64_t al = make_desc(sa + H_PART_BYTES + k * a_step, a_lbo, 1024, 2);
              const uint64_t bh = make_desc(sb + k * b_step, b_lbo, 1024, 2);
              const uint64_t bl = make_desc(sb + H_PART_BYTES + k * b_step, b_lbo, 1024, 2);
              mma2_f16(tmem_d, al, bh, idesc, acc);
              mma2_f16(tmem_d, ah, bl, idesc, 1u);
              acc = 1u;
            }
#pragma unroll
            for (int k = 0; k < H_BK / 16; ++k) {
              const uint64_t ah = make_desc(sa + k * a_step, a_lbo, 1024, 2);
              const uint64_t bh = make_desc(sb + k * b_step, b_lbo, 1024, 2);
              mma2_f16(tmem_d, ah, bh, idesc, 1u);
            }
            mma2_commit_both(&empty[s]);
          }
          if (ok) mma2_commit_both(&acc_full[buf]);
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(H_REGS_HIGH));
    // ------------------------------------------------------------------ epilogue (warps 4..11, both CTAs)
    const int quad = warp & 3;
    const int half = (warp - 4) >> 2;
    const uint32_t stg = smem_u32(smem + H_STAGES * H_STAGE_BYTES) + (uint32_t)(warp - 4) * 4096u;
    int ci = 0;
    bool alive = true;
    for (int item = pair; item < p.items && alive; item += p.P) {
      const Item w = item_at(p, item, n_chunks);
      const int m0 = (w.tile / p.tiles_n) * (2 * H_BM) + (int)rank * H_BM + quad * 32, n0 = (w.tile % p.tiles_n) * bn;
      const int n_cc = min(bn / 32, (p.e.N - n0 + 31) / 32);     // column chunks of this tile that exist
      float run[4][32];                                          // this warp's chunks: half, half + 2, half + 4, half + 6
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 32; ++i) run[j][i] = 0.f;
      const CellWalk walk = cell_walk(p, m0 - quad * 32, n0 + half * 32, (n_cc - half + 1) / 2, lane);
      int exps = cell_exponent(p, walk, w.c0);                   // exponents of the cells of the chunk to come
      for (int ch = w.c0; ch < w.c1; ++ch, ++ci) {
        const int buf = ci & 1;
        const uint32_t aph = (ci >> 1) & 1;
        const bool by_fma = __any_sync(0xffffffffu, exps == kMarked);
        // what undoes the scales of this chunk's cells, per 32-column group: 2^-shift
        int shift[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) shift[j] = __shfl_sync(0xffffffffu, exps, 4) + __shfl_sync(0xffffffffu, exps, j);
        if (ch + 1 < w.c1) exps = cell_exponent(p, walk, ch + 1);       // (on its way while this chunk is waited for)
        int good = 1;
        if (lane == 0) good = wait_or_abort(&acc_full[buf], aph, abort_flag, p.err, 3) ? 1 : 0;
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) { alive = false; break; }
        tc_fence_after();
        // two 32-column reads in flight at a time (a read of columns past the tile is harmless: it is never stored)
        const uint32_t ta = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * H_BN_MAX + half * 32);
        if (by_fma) {                                            // (the sums wait in tensor memory: the buffer is free)
#pragma unroll
          for (int j = 0; j < 4; ++j) tmem_st32(ta + (uint32_t)(j * 64), run[j]);
          tmem_st_wait();
          fma_chunk(p, chunk_at(p, ch), stg, m0, n0 + half * 32, (n_cc - half + 1) / 2, lane, ta);
#pragma unroll
          for (int j = 0; j < 4; ++j) tmem_ld_32x32b_x32(ta + (uint32_t)(j * 64), run[j]);
          tmem_ld_wait();
        } else {
#pragma unroll
          for (int j = 0; j < 4; j += 2) {
            if (half + 2 * j < n_cc) {                           // warp-uniform
              float v[64];
              tmem_ld_32x32b_x32(ta + (uint32_t)(j * 64), v);
              tmem_ld_32x32b_x32(ta + (uint32_t)(j * 64 + 64), v + 32);
              tmem_ld_wait();
              if (abs(shift[j]) > 126 || abs(shift[j + 1]) > 126) {      // (out of a factor's range: in two steps)
                const float g0 = exp2_int(-shift[j] / 2), g1 = exp2_int(-shift[j + 1] / 2);
#pragma unroll
                for (int i = 0; i < 32; ++i) { v[i] *= g0; v[32 + i] *= g1; }
                shift[j] += -shift[j] / 2; shift[j + 1] += -shift[j + 1] / 2;
              }
              const float f0 = exp2_int(-shift[j]), f1 = exp2_int(-shift[j + 1]);
#pragma unroll
              for (int i = 0; i < 32; ++i) {
                run[j][i] = fmaf(v[i], f0, run[j][i]);
                run[j + 1][i] = fmaf(v[32 + i], f1, run[j + 1][i]);
              }
            }
          }
        }
        if (ch + 1 == w.c1) break;                               // (the last buffer takes the finished sums first)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(smem_u32(&acc_empty[buf]), 0));
      }
      if (!alive) break;
      const int buf = ci & 1;
      ++ci;
      const uint32_t ta = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * H_BN_MAX + half * 32);
      const int n_mine = (n_cc - half + 1) / 2;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < n_mine) tmem_st32(ta + (uint32_t)(j * 64), run[j]);
      tmem_st_wait();
      if (m0 < p.e.M) {                                          // warp-uniform
        const int rows = min(32, p.e.M - m0), nb0 = n0 + half * 32;
        if (w.slot >= 0) {                                       // (the workspace holds whole tiles)
          float* o = p.ws + ((long long)w.slot * (2 * H_BM) + (int)rank * H_BM + quad * 32 + (lane >> 3)) * bn + half * 32 + (lane & 7) * 4;
#pragma unroll 1
          for (int j = 0; j < n_mine; ++j) {
            float v[32];
            tmem_ld32(ta + (uint32_t)(64 * j), v);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 32; i += 4)
              stg_put(stg_at(stg, lane, i >> 2), v[i], v[i + 1], v[i + 2], v[i + 3]);
            __syncwarp();
            float x[8][4];
#pragma unroll
            for (int r = 0; r < 8; ++r) stg_get<4>(stg_at(stg, 4 * r + (lane >> 3), lane & 7), x[r]);
#pragma unroll
            for (int r = 0; r < 8; ++r)
              __stcg(reinterpret_cast<float4*>(o + 4 * r * bn + 64 * j), make_float4(x[r][0], x[r][1], x[r][2], x[r][3]));
          }
        } else {
          store_tile<MODE, VEC>(after_wait(p.e), stg, ta, n_mine, m0, rows, nb0, lane);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(smem_u32(&acc_empty[buf]), 0));
    }
  }
  tc_fence_before();
  cluster_sync_all();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

// Sum of the K slices of the left-over tiles, slice 0 first, and the epilogue.  blockIdx.x = 32-column chunk of a left-over
// tile, warp = row, lane = column; bound by the reads of the workspace, which the kernel before it has left in L2.
__global__ void __launch_bounds__(256) slice_sum_kernel(const HEpilogue epi, const float* __restrict__ ws, int whole, int rem, int slices,
                                                        int tiles_n, int bn) {
  grid_dep_wait();
  grid_dep_launch();
  const HEpilogue e = after_wait(epi);
  ws = dep(ws);
  const int lane = threadIdx.x & 31;
  const int per_tile = bn / 32;
  const int j = blockIdx.x / per_tile, c = (blockIdx.x - j * per_tile) * 32 + lane;
  const int t = whole + j;
  const int m0 = (t / tiles_n) * (2 * H_BM), n = (t % tiles_n) * bn + c;
  if (n < e.N) {
    const float bz = e.bias ? __ldg(e.bias + n) : 0.f;
    const long long step = (long long)rem * (2 * H_BM) * bn;
    const int rows = min(2 * H_BM, e.M - m0);
    for (int r = blockIdx.y * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.y * 8) {
      const int m = m0 + r;
      const float* w = ws + ((long long)j * (2 * H_BM) + r) * bn + c;
      const float z = e.dsig ? __ldg(e.dsig + dsig_row(e, m) * e.ld_dsig + n) : 0.f;
      const float cv = e.cin ? __ldg(e.cin + (long long)m * e.ld_cin + n) : 0.f;
      float s = 0.f;
#pragma unroll 8
      for (int k = 0; k < slices; ++k) s += __ldcg(w + k * step);
      e.D[(long long)m * e.ldd + n] = finish(e, s, bz, z, cv);
    }
  }
}

// ---- splitting -----------------------------------------------------------------------------------
// Up to kSplitSegs matrices per launch, a cluster of four blocks per cell: a block holds 32 rows of it in registers (4 groups of
// 4 columns per thread, all requested before the first is used), the cluster finds its largest element, and every block writes
// its parts, so a matrix is read once.  (A last column of cells of at most 32 columns has a block per cell, four to a cluster.)  Bound by its memory traffic where there is some and by the chain of load, exchange
// and store where there is not.  12000 x 2000:
// 43 us (192 MB; a pass for one maximum of the whole matrix and one for the parts took 22 + 45), 2500 x 1000: 6.2 us (3.9 +
// 5.3), 300 x 300: 3.5 us (2.3 + 2.8).  A block of 512 threads per cell: 36, 8.4 and 4.9 us.
constexpr int SPLIT_THREADS = 256, SPLIT_BLOCKS = 4, SPLIT_ROWS = CELL / SPLIT_BLOCKS / (SPLIT_THREADS / 32);   // rows of a warp
struct SplitSeg {
  const float* src; long long rows; int cols; long long ld;
  __half* hi; __half* lo; long long ld_out;
  int8_t* cells; int cells_ld;
  int rows_ld;                               // 128-row panels
  int wide, wide_ld;                         // clusters with a cell each, of them per panel; then clusters of four narrow cells
  int cluster0, vec;
};
struct SplitList { int n; SplitSeg s[kSplitSegs]; };

// columns c .. c + 3 of a row of which `left` are there
__device__ __forceinline__ float4 load_group(const float* q, int left, int vec) {
  if (vec) return __ldg(reinterpret_cast<const float4*>(q));
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
  x.x = __ldg(q);
  if (left > 1) x.y = __ldg(q + 1);
  if (left > 2) x.z = __ldg(q + 2);
  if (left > 3) x.w = __ldg(q + 3);
  return x;
}

__device__ __forceinline__ void split4(float4 x, float sc, uint2& h, uint2& l) {
  const float2 a = make_float2(x.x * sc, x.y * sc), b = make_float2(x.z * sc, x.w * sc);
  const __half2 ha = __float22half2_rn(a), hb = __float22half2_rn(b);
  const float2 fa = __half22float2(ha), fb = __half22float2(hb);
  const __half2 la = __float22half2_rn(make_float2(a.x - fa.x, a.y - fa.y)), lb = __float22half2_rn(make_float2(b.x - fb.x, b.y - fb.y));
  h.x = *reinterpret_cast<const unsigned*>(&ha); h.y = *reinterpret_cast<const unsigned*>(&hb);
  l.x = *reinterpret_cast<const unsigned*>(&la); l.y = *reinterpret_cast<const unsigned*>(&lb);
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void put_remote(const void* at, uint32_t rank, unsigned x) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_to_cta(smem_u32(at), rank)), "r"(x) : "memory");
}

__device__ __forceinline__ unsigned magnitude(float x) { return __float_as_uint(x) & 0x7fffffffu; }

__global__ void __cluster_dims__(SPLIT_BLOCKS, 1, 1) __launch_bounds__(SPLIT_THREADS) split_f16_kernel(const __grid_constant__ SplitList list) {
  constexpr int WARPS = SPLIT_THREADS / 32;
  __shared__ unsigned col_max[CELL];                       // of this block's rows: largest magnitude per column,
  __shared__ unsigned warp_max[WARPS], warp_row[WARPS];    // largest, and smallest of the rows' largest (less one, so that a row of zeros is the largest)
  __shared__ unsigned all_max[SPLIT_BLOCKS];               // what the blocks tell every block, and block 0
  __shared__ unsigned all_row[SPLIT_BLOCKS], all_col[SPLIT_BLOCKS][CELL];
  cluster_arrive();                                        // (no block writes to another before that one runs)
  grid_dep_wait();
  grid_dep_launch();
  const int cluster = blockIdx.x / SPLIT_BLOCKS;
  const int rank = (int)cluster_ctarank();
  int k = 0;
  while (k + 1 < list.n && cluster >= list.s[k + 1].cluster0) ++k;
  const SplitSeg& s = list.s[k];
  const float* const src = dep(s.src);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the cluster's cell, or (narrow, at most 32 columns: a block holds all of one) this block's
  const int at_seg = cluster - s.cluster0;
  const bool solo = at_seg >= s.wide;
  const int panel = solo ? (at_seg - s.wide) * SPLIT_BLOCKS + rank : at_seg / s.wide_ld, ct = solo ? s.cells_ld - 1 : at_seg - panel * s.wide_ld;
  // lanes that share a row (8, 16 or 32 groups of 4 columns, as the cell has columns), rows of an access
  const int width = s.cols - ct * CELL, lanes_log = solo ? 3 : width <= 64 ? 4 : 5, lanes = 1 << lanes_log, rpi = 32 >> lanes_log;
  const int g = lane & (lanes - 1), c = ct * CELL + 4 * g, left = s.cols - c;
  const int warp_rows = solo ? 4 * SPLIT_ROWS : SPLIT_ROWS;
  const long long r0 = (long long)panel * CELL + (solo ? warp : rank * WARPS + warp) * warp_rows + (lane >> lanes_log);
  const int n_mine = left > 0 ? (int)min((s.rows - r0 + rpi - 1) >> (5 - lanes_log), (long long)(warp_rows >> (5 - lanes_log))) : 0;   // this thread's groups
  float4 x[SPLIT_ROWS];
  {
    const float* q = src + r0 * s.ld + c;
    const long long step = rpi * s.ld;
    const int vec = s.vec;
#pragma unroll
    for (int i = 0; i < SPLIT_ROWS; ++i, q += step)
      x[i] = i < n_mine ? load_group(q, left, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (tid < CELL) col_max[tid] = 0u;
  __syncthreads();
  unsigned largest = 0u, row_min = 0xffffffffu, col[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < SPLIT_ROWS; ++i) {
    const unsigned m[4] = {magnitude(x[i].x), magnitude(x[i].y), magnitude(x[i].z), magnitude(x[i].w)};
#pragma unroll
    for (int q = 0; q < 4; ++q) col[q] = max(col[q], m[q]);
    unsigned row = max(max(m[0], m[1]), max(m[2], m[3]));
    if (lanes == 32) {
      row = __reduce_max_sync(0xffffffffu, row);
    } else {
      for (int o = lanes >> 1; o > 0; o >>= 1) row = max(row, __shfl_xor_sync(0xffffffffu, row, o));
    }
    largest = max(largest, row);
    row_min = min(row_min, row - 1u);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (col[q]) atomicMax(&col_max[4 * g + q], col[q]);
  if (lanes < 32) {
    largest = __reduce_max_sync(0xffffffffu, largest);
    row_min = __reduce_min_sync(0xffffffffu, row_min);
  }
  if (lane == 0) { warp_max[warp] = largest; warp_row[warp] = row_min; }
  cluster_wait();
  __syncthreads();
  if (warp == 0) {
    largest = __reduce_max_sync(0xffffffffu, warp_max[lane & (WARPS - 1)]);
    row_min = __reduce_min_sync(0xffffffffu, warp_row[lane & (WARPS - 1)]);
    // (a block that has a cell to itself fills all places, its own)
    if (lane < SPLIT_BLOCKS) put_remote(&all_max[solo ? lane : rank], solo ? rank : lane, largest);
    else if (lane < 2 * SPLIT_BLOCKS && (solo || lane == SPLIT_BLOCKS)) put_remote(&all_row[solo ? lane - SPLIT_BLOCKS : rank], solo ? rank : 0, row_min);
  } else if (tid >= SPLIT_THREADS - CELL) {
    const int t = tid & (CELL - 1);
    if (!solo) put_remote(&all_col[rank][t], 0, col_max[t]);
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  largest = max(max(all_max[0], all_max[1]), max(all_max[2], all_max[3]));
  const int e = scale_exponent(largest);
  if (largest < 0x7f800000u) {                             // (infinities, NaN: nobody reads the parts)
    const float sc = exp2_int(e);
    long long at = r0 * s.ld_out + c;
    const long long step = rpi * s.ld_out;
    __half* const hi = s.hi;
    __half* const lo = s.lo;
#pragma unroll
    for (int i = 0; i < SPLIT_ROWS; ++i, at += step)
      if (i < n_mine) {
        uint2 h, l;
        split4(x[i], sc, h, l);                            // (ld_out is a multiple of 8: a whole group always fits)
        *reinterpret_cast<uint2*>(hi + at) = h;
        *reinterpret_cast<uint2*>(lo + at) = l;
      }
  }
  if (solo ? panel >= s.rows_ld : rank != 0) return;
  // Marked: a row or a column whose largest element is not zero but below 2^-20 of the cell's, or anything infinite or NaN.
  const unsigned least = largest > (FAR_LOG << 23) ? largest - (FAR_LOG << 23) : 1u;
  bool far = largest >= 0x7f800000u;
  if (tid < CELL) {
    const unsigned m = solo ? col_max[tid] : max(max(all_col[0][tid], all_col[1][tid]), max(all_col[2][tid], all_col[3][tid]));
    far = far || (m != 0u && m < least);
  }
  if (tid < SPLIT_BLOCKS) far = far || all_row[tid] < least - 1u;                 // (0xffffffff: only zeros)
  far = __syncthreads_or(far) != 0;
  if (tid == 0) s.cells[(long long)panel * s.cells_ld + ct] = (int8_t)(far ? kMarked : e);
}

// 2-D map over a row-major [rows][cols] FP16 matrix with leading dimension ld; box = 64 columns x box_r rows.
bool make_half_map(CUtensorMap* m, const void* base, long long rows, long long cols, long long ld, int box_r) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_r};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct HPlan { int bn, whole, rem, slices; double us; };

int chunks_of(const GemmArgs& g, int chunk_kb) {
  const int kc = chunk_kb * H_BK;                          // (1 or 2 k-blocks)
  return (g.K1 + kc - 1) / kc + (g.A2 ? (g.K2 + kc - 1) / kc : 0);
}

// Tile width, and the K slices of the tiles left over after the whole rounds of the CTA pairs, with the shortest
// estimated time: a k-block takes time proportional to 96 + bn columns (0.9 us at 256, bound by its MMAs and the
// shared-memory feed), an item a ramp and its epilogue, and slices a second kernel that reads the partial sums back.
// (12000 x 2000 x 2000, 376 tiles on 74 pairs: 245 us in six rounds, 218 us with the last six tiles cut in twelve.)
HPlan plan_f16x3(const GemmArgs& g) {
  const int pairs = num_sms() / 2;
  const long long tiles_m = (g.M + 2 * H_BM - 1) / (2 * H_BM);
  const int kb = chunks_of(g, 1);
  const int nc = chunks_of(g, g.chunk_kb);
  HPlan best{256, 0, 0, 1, -1.0};
  const int widths[] = {256, 192, 128, 64, 32};
  for (int bn : widths) {
    if (bn > 32 && bn / 2 >= g.N) continue;                // a narrower tile covers N
    const long long tiles = tiles_m * ((g.N + bn - 1) / bn);
    const double t_kb = 0.9 * (96 + bn) / 352.0, t_item = 3.0 + 5.0 * bn / 256.0;
    const long long rounds = tiles / pairs, rem = tiles - rounds * pairs;
    const double t_whole = rounds * (kb * t_kb + t_item);
    const double t = t_whole + (rem ? kb * t_kb + t_item : 0.0);
    if (best.us < 0.0 || t < 0.98 * best.us) best = HPlan{bn, (int)tiles, 0, 1, t};
    if (rem == 0 || g.whole_tiles) continue;
    for (int s = 2; s <= nc && s <= 64 && rem * s <= pairs; ++s) {
      const double per_slice = (kb + s - 1) / s + (g.chunk_kb - 1);
      const double sliced = t_whole + per_slice * t_kb + t_item + 3.0 + (s + 2.0) * rem * bn * 1024.0 / 3.0e6;
      if (sliced < 0.98 * best.us) best = HPlan{bn, (int)(rounds * pairs), (int)rem, s, sliced};
    }
  }
  return best;
}

HEpilogue make_epilogue(const GemmArgs& g) {
  HEpilogue e{};
  e.M = g.M; e.N = g.N; e.D = g.D; e.ldd = g.ldd; e.bias = g.bias; e.sigmoid = g.sigmoid ? 1 : 0;
  e.dsig = g.dsig; e.ld_dsig = g.ld_dsig; e.dsig_rows = g.dsig_rows > 0 ? g.dsig_rows : 1; e.dsig_div = g.dsig_div > 0 ? g.dsig_div : 1;
  e.dsig_direct = e.dsig_div == 1 && e.dsig_rows >= g.M;
  e.alpha = g.alpha; e.cin = g.cin; e.ld_cin = g.ld_cin; e.beta = g.beta;
  e.vec = g.N % 4 == 0 && aligned16(g.D) && g.ldd % 4 == 0 && (!g.bias || aligned16(g.bias)) && (!g.dsig || (aligned16(g.dsig) && g.ld_dsig % 4 == 0)) &&
          (!g.cin || (aligned16(g.cin) && g.ld_cin % 4 == 0));
  return e;
}

}  // namespace

namespace {
typedef void (*HKernel)(const HMaps, const HParams);
// [2 * mode + vec], see store_tile
HKernel const kKernels[10] = {
    gemm_f16x3_kernel<0, false>, gemm_f16x3_kernel<0, true>, gemm_f16x3_kernel<1, false>, gemm_f16x3_kernel<1, true>,
    gemm_f16x3_kernel<2, false>, gemm_f16x3_kernel<2, true>, gemm_f16x3_kernel<3, false>, gemm_f16x3_kernel<3, true>,
    gemm_f16x3_kernel<4, false>, gemm_f16x3_kernel<4, true>};
}  // namespace

// The register split of the kernel (128 x 56 + 256 x 224) must not exceed what the block is launched with, and the
// kernel needs its dynamic shared memory granted: checked once per device.
bool gemm_f16x3_usable() {
  static std::atomic<signed char> state[64];
  return once_per_device(state, [] {
    bool ok = encode_fn() != nullptr;
    for (HKernel k : kKernels) {
      cudaFuncAttributes fa;
      ok = ok && cudaFuncGetAttributes(&fa, k) == cudaSuccess && fa.numRegs * H_THREADS >= 128 * H_REGS_LOW + 256 * H_REGS_HIGH &&
           cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, H_SMEM_BYTES) == cudaSuccess;
    }
    return ok;
  });
}

double gemm_f16x3_estimate_us(const GemmArgs& g) { return plan_f16x3(g).us; }

int64_t gemm_f16x3_workspace_floats(const GemmArgs& g) {
  const HPlan pl = plan_f16x3(g);
  return (int64_t)(pl.slices > 1 ? pl.slices : 0) * pl.rem * (2 * H_BM) * pl.bn;
}

int launch_gemm_f16x3(const GemmArgs& g, const SplitOperand* ops, float* ws, int* err_flag, cudaStream_t st) {
  if (!gemm_f16x3_usable()) return -1;
  const HPlan pl = plan_f16x3(g);
  if (pl.slices > 1 && !ws) return -1;
  const int n_pairs = g.A2 ? 2 : 1;
  const int Ks[2] = {g.K1, g.A2 ? g.K2 : 0};
  HMaps maps;
  HParams p{};
  for (int s = 0; s < 2; ++s) {
    const int src = s < n_pairs ? s : 0;                   // unused second pair: repeat the first (never read)
    const SplitOperand& a = ops[2 * src];
    const SplitOperand& b = ops[2 * src + 1];
    for (int h = 0; h < 2; ++h) {
      const void* ap = h ? a.lo : a.hi;
      const void* bp = h ? b.lo : b.hi;
      bool ok = g.a_kmajor ? make_half_map(&maps.m[4 * s + h], ap, g.M, Ks[src], a.ld, H_BM)
                           : make_half_map(&maps.m[4 * s + h], ap, Ks[src], g.M, a.ld, H_BK);
      ok = ok && (g.b_kmajor ? make_half_map(&maps.m[4 * s + 2 + h], bp, g.N, Ks[src], b.ld, pl.bn / 2)
                             : make_half_map(&maps.m[4 * s + 2 + h], bp, Ks[src], g.N, b.ld, H_BK));
      if (!ok) return -1;
    }
    p.kblocks[s] = s < n_pairs ? (Ks[s] + H_BK - 1) / H_BK : 0;
    for (int q = 0; q < 2; ++q) {
      p.cells[2 * s + q] = ops[2 * src + q].cells;
      p.cells_ld[2 * s + q] = ops[2 * src + q].cells_ld;
    }
    p.src[2 * s] = src ? g.A2 : g.A1; p.ld_src[2 * s] = src ? g.lda2 : g.lda1;
    p.src[2 * s + 1] = src ? g.B2 : g.B1; p.ld_src[2 * s + 1] = src ? g.ldb2 : g.ldb1;
    p.K[s] = Ks[src];
  }
  p.e = make_epilogue(g);
  p.n_pairs = n_pairs;
  p.a_mn = g.a_kmajor ? 0 : 1; p.b_mn = g.b_kmajor ? 0 : 1;
  p.bn = pl.bn;
  p.tiles_n = (g.N + pl.bn - 1) / pl.bn;
  p.chunk_log = g.chunk_kb - 1;
  p.chunks0 = (p.kblocks[0] + p.chunk_log) >> p.chunk_log;
  p.whole = pl.whole; p.rem = pl.rem; p.slices = pl.slices;
  p.items = p.whole + p.rem * p.slices;
  const int pairs = num_sms() / 2;
  p.P = p.items < pairs ? p.items : pairs;
  p.ws = ws;
  p.err = err_flag;
  // (left-over tiles' slices store raw sums: with no whole tile in the list every form of the kernel is the same)
  const int n_opt = (p.e.sigmoid ? 1 : 0) + (p.e.dsig ? 1 : 0) + (p.e.cin ? 1 : 0);
  const int mode = p.whole == 0 || n_opt == 0 ? 0 : n_opt > 1 ? 4 : p.e.sigmoid ? 1 : p.e.dsig ? 2 : 3;
  if (launch_pdl(kKernels[2 * mode + (p.e.vec ? 1 : 0)], 2 * p.P, H_THREADS, H_SMEM_BYTES, st, maps, p) != cudaSuccess) return -1;
  if (p.rem == 0) return 1;
  const int gx = p.rem * (p.bn / 32);
  int gy = (148 * 8 + gx - 1) / gx;
  if (gy > 32) gy = 32;
  if (launch_pdl_grid(slice_sum_kernel, dim3((unsigned)gx, (unsigned)gy), 256, 0, st, p.e, (const float*)ws, p.whole, p.rem, p.slices, p.tiles_n, p.bn) != cudaSuccess)
    return -1;
  return 2;
}

int launch_split_f16(const SplitJob* jobs, int n, cudaStream_t st) {
  if (n < 1 || n > kSplitSegs) return -1;
  SplitList list{};
  long long clusters = 0;
  for (int i = 0; i < n; ++i) {
    const SplitJob& j = jobs[i];
    SplitSeg& s = list.s[list.n++];
    s.src = j.src; s.rows = j.rows; s.cols = j.cols; s.ld = j.ld;
    s.hi = static_cast<__half*>(j.hi); s.lo = static_cast<__half*>(j.lo); s.ld_out = j.ld_out;
    s.cells = j.cells; s.cells_ld = (j.cols + CELL - 1) / CELL;
    s.vec = j.cols % 4 == 0 && j.ld % 4 == 0 && aligned16(j.src);
    const bool narrow = j.cols - (s.cells_ld - 1) * CELL <= 32;
    const long long panels = (j.rows + CELL - 1) / CELL;
    if (panels * s.cells_ld > 0x7fffffff / SPLIT_BLOCKS) return -1;
    s.rows_ld = (int)panels;
    s.wide_ld = s.cells_ld - (narrow ? 1 : 0);
    s.wide = (int)panels * s.wide_ld;
    s.cluster0 = (int)clusters;
    clusters += s.wide + (narrow ? (panels + SPLIT_BLOCKS - 1) / SPLIT_BLOCKS : 0);
    if (clusters > 0x7fffffff / SPLIT_BLOCKS) return -1;
  }
  return launch_pdl(split_f16_kernel, (int)clusters * SPLIT_BLOCKS, SPLIT_THREADS, 0, st, list) == cudaSuccess ? 1 : -1;
}

}  // namespace gn
