// FP32-accurate contractions on the FP16 tensor cores (sm_100a).
//
// Every operand X arrives as two FP16 matrices, X 2^e = hi + lo with hi = rn16(X 2^e), lo = rn16(X 2^e - hi), where the
// power of two 2^e takes the largest element of X to [2^14, 2^15).  hi and lo carry 11 significant bits each, so
// |X - (hi + lo) 2^-e| <= 2^-23 |x| for elements down to 2^-18 of the largest one and <= 2^-40 max|X| below that.  A
// logical product A B is Alo Bhi + Ahi Blo + Ahi Bhi (the dropped Alo Blo is below 2^-22 |a b|).
//
// Why FP16 and not TF32 parts: the two formats have the same 11-bit significand, but kind::f16 runs at twice the rate
// of kind::tf32 and its parts are half the bytes, so the three products cost 1.5 TF32 products instead of 3 and the
// parts together are no larger than the FP32 operand.  What TF32 parts have and FP16 parts lack is exponent range;
// the scale per operand puts the range where the operand is.
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
  unsigned* amax_out;                        // |D| maximum (bit pattern) is accumulated here when set
};

struct HParams {
  HEpilogue e;
  int n_pairs;                               // logical operand pairs accumulated into one tile (1 or 2)
  int kblocks[2];
  int a_mn, b_mn;
  const unsigned* amax[4];                   // bit pattern of max|X| of A1, B1, A2, B2
  unsigned* reset[4];                        // accumulators of fused maxima to be cleared for their next use
  int chunk_kb;                              // k-blocks per accumulation in tensor memory
  // work list: items 0 .. whole - 1 are whole tiles, then slice sl of left-over tile j (tile whole + j) is item
  // whole + sl * rem + j; pair q takes items q, q + P, ...
  int bn, tiles_n, whole, rem, slices, items, P;
  float* ws;                                 // partial sums of the left-over tiles: [slices][rem][256][bn]
  int* err;
};

struct HMaps { CUtensorMap m[8]; };          // per pair: A hi, A lo, B hi, B lo

// Exponent e of the scale 2^e for an operand whose largest magnitude has this bit pattern.
__device__ __forceinline__ int scale_exponent(unsigned amax_bits) {
  const int p = (int)(amax_bits >> 23) - 127;             // (zero and denormals: -127)
  return min(14 - p, 126);
}
__device__ __forceinline__ float exp2_int(int e) {        // 2^e, 0 below the normal range
  return e < -126 ? 0.f : __uint_as_float((unsigned)(min(e, 127) + 127) << 23);
}
__device__ __forceinline__ unsigned finite_magnitude(float x) {
  const unsigned b = __float_as_uint(x) & 0x7fffffffu;
  return b < 0x7f800000u ? b : 0u;                        // infinities and NaN do not set the scale
}

__device__ __forceinline__ void mma2_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
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
__device__ __forceinline__ void store_tile(const HEpilogue& e, uint32_t stg, uint32_t ta, int n_mine, int m0, int rows, int nb0, int lane, unsigned& mag) {
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
      // (the record and the stores in loops of their own, whole chunks without a test per row: with rows that are no
      // multiple of four floats every element is a store of its own, and what surrounds it counts)
      if (e.amax_out) {
#pragma unroll
        for (int i = 0; i < IT; ++i)
#pragma unroll
          for (int q = 0; q < W; ++q)
            if (r_first + i * STEP < rows) mag = max(mag, finite_magnitude(xs[i][q]));
      }
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

// Piece `i` of the chunk list of a K range: chunks of chunk_kb k-blocks that never straddle the two operand pairs.
struct ChunkPos { int pair, kb0, kb1; };
__device__ __forceinline__ ChunkPos chunk_at(const HParams& p, int i) {
  const int n0 = (p.kblocks[0] + p.chunk_kb - 1) / p.chunk_kb;
  ChunkPos c;
  c.pair = i >= n0 ? 1 : 0;
  c.kb0 = (i - (c.pair ? n0 : 0)) * p.chunk_kb;
  c.kb1 = min(p.kblocks[c.pair], c.kb0 + p.chunk_kb);
  return c;
}
__device__ __forceinline__ int chunk_count(const HParams& p) {
  int n = (p.kblocks[0] + p.chunk_kb - 1) / p.chunk_kb;
  if (p.n_pairs > 1) n += (p.kblocks[1] + p.chunk_kb - 1) / p.chunk_kb;
  return n;
}

// Item of the work list: its tile, its chunks c0 .. c1 - 1, and, for a K slice, where its partial sums go (else -1).
struct Item { int tile, c0, c1, slot; };
__device__ __forceinline__ Item item_at(const HParams& p, int i, int n_chunks) {
  if (i < p.whole) return Item{i, 0, n_chunks, -1};
  const int k = i - p.whole, sl = k / p.rem;
  return Item{p.whole + k - sl * p.rem, (int)((long long)n_chunks * sl / p.slices), (int)((long long)n_chunks * (sl + 1) / p.slices), k};
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
      if (blockIdx.x == 0 && lane < 4 && p.reset[lane]) *p.reset[lane] = 0u;
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
    // what undoes the operands' scales: pair i's products are true values times 2^-E_i; sums are kept relative to
    // the largest E (the other pair's factor is a power of two below one), which is undone once per tile
    const int E0 = -(scale_exponent(__ldcg(p.amax[0])) + scale_exponent(__ldcg(p.amax[1])));
    const int E1 = p.n_pairs > 1 ? -(scale_exponent(__ldcg(p.amax[2])) + scale_exponent(__ldcg(p.amax[3]))) : E0;
    const int E = max(E0, E1);
    const float f0 = exp2_int(E0 - E), f1 = exp2_int(E1 - E);
    const float u0 = exp2_int(E / 2), u1 = exp2_int(E - E / 2);
    const HEpilogue& e = p.e;
    unsigned mag = 0u;
    int ci = 0;
    bool alive = true;
    for (int item = pair; item < p.items && alive; item += p.P) {
      const Item w = item_at(p, item, n_chunks);
      const int m0 = (w.tile / p.tiles_n) * (2 * H_BM) + (int)rank * H_BM + quad * 32, n0 = (w.tile % p.tiles_n) * bn;
      const int n_cc = min(bn / 32, (e.N - n0 + 31) / 32);       // column chunks of this tile that exist
      float run[4][32];                                          // this warp's chunks: half, half + 2, half + 4, half + 6
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 32; ++i) run[j][i] = 0.f;
      for (int ch = w.c0; ch < w.c1; ++ch, ++ci) {
        const int buf = ci & 1;
        const uint32_t aph = (ci >> 1) & 1;
        const float f = chunk_at(p, ch).pair ? f1 : f0;
        int good = 1;
        if (lane == 0) good = wait_or_abort(&acc_full[buf], aph, abort_flag, p.err, 3) ? 1 : 0;
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) { alive = false; break; }
        tc_fence_after();
        // two 32-column reads in flight at a time (a read of columns past the tile is harmless: it is never stored)
        const uint32_t ta = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * H_BN_MAX + half * 32);
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
          if (half + 2 * j < n_cc) {                             // warp-uniform
            float v[64];
            tmem_ld_32x32b_x32(ta + (uint32_t)(j * 64), v);
            tmem_ld_32x32b_x32(ta + (uint32_t)(j * 64 + 64), v + 32);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              run[j][i] = fmaf(v[i], f, run[j][i]);
              run[j + 1][i] = fmaf(v[32 + i], f, run[j + 1][i]);
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
        if (j < n_mine) {
#pragma unroll
          for (int i = 0; i < 32; ++i) run[j][i] = run[j][i] * u0 * u1;
          tmem_st32(ta + (uint32_t)(j * 64), run[j]);
        }
      tmem_st_wait();
      if (m0 < e.M) {                                            // warp-uniform
        const int rows = min(32, e.M - m0), nb0 = n0 + half * 32;
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
          store_tile<MODE, VEC>(e, stg, ta, n_mine, m0, rows, nb0, lane, mag);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(smem_u32(&acc_empty[buf]), 0));
    }
    if (e.amax_out) {
      mag = __reduce_max_sync(0xffffffffu, mag);
      if (lane == 0 && mag) atomicMax(e.amax_out, mag);
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
__global__ void __launch_bounds__(256) slice_sum_kernel(const HEpilogue e, const float* __restrict__ ws, int whole, int rem, int slices,
                                                        int tiles_n, int bn) {
  grid_dep_wait();
  grid_dep_launch();
  const int lane = threadIdx.x & 31;
  const int per_tile = bn / 32;
  const int j = blockIdx.x / per_tile, c = (blockIdx.x - j * per_tile) * 32 + lane;
  const int t = whole + j;
  const int m0 = (t / tiles_n) * (2 * H_BM), n = (t % tiles_n) * bn + c;
  unsigned mag = 0u;
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
      const float x = finish(e, s, bz, z, cv);
      e.D[(long long)m * e.ldd + n] = x;
      mag = max(mag, finite_magnitude(x));
    }
  }
  if (e.amax_out) {
    mag = __reduce_max_sync(0xffffffffu, mag);
    if (lane == 0 && mag) atomicMax(e.amax_out, mag);
  }
}

// ---- splitting -----------------------------------------------------------------------------------
// Up to kSplitSegs matrices per launch.  A thread takes 4 consecutive columns; a block of 256 threads covers 256 / per_row
// rows at a time (or one row in several steps), with the thread's place in that pattern fixed so that the loop
// has no division.  Four rows are requested before the first is used.
struct SplitSeg {
  const float* src; long long rows; int cols; long long ld;
  __half* hi; __half* lo; long long ld_out;
  unsigned* part; int n_part;                // maxima of the blocks of the first pass (or the producer's one maximum)
  unsigned* bits;                            // the operand's maximum, for the contraction
  int block0, blocks, vec;
};
struct SplitList { int n; SplitSeg s[kSplitSegs]; };

__device__ __forceinline__ float4 load_group(const SplitSeg& s, long long r, int c) {
  const float* q = s.src + r * s.ld + c;
  if (s.vec) return __ldg(reinterpret_cast<const float4*>(q));
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
  x.x = __ldg(q);
  if (c + 1 < s.cols) x.y = __ldg(q + 1);
  if (c + 2 < s.cols) x.z = __ldg(q + 2);
  if (c + 3 < s.cols) x.w = __ldg(q + 3);
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

template <bool SPLIT>
__global__ void __launch_bounds__(256) split_f16_kernel(const __grid_constant__ SplitList list) {
  __shared__ unsigned sh[8];
  grid_dep_wait();
  grid_dep_launch();
  int k = 0;
  while (k + 1 < list.n && (int)blockIdx.x >= list.s[k + 1].block0) ++k;
  const SplitSeg& s = list.s[k];
  const int blk = blockIdx.x - s.block0;
  const int tid = threadIdx.x;
  float sc = 1.f;
  if (SPLIT) {
    unsigned m = 0u;
    for (int i = tid; i < s.n_part; i += 256) m = max(m, __ldcg(s.part + i));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((tid & 31) == 0) sh[tid >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) m = max(m, sh[i]);
    if (blk == 0 && tid == 0) *s.bits = m;
    sc = exp2_int(scale_exponent(m));
  }
  const int per_row = (s.cols + 3) >> 2;
  const int rpb = per_row < 256 ? 256 / per_row : 1;       // rows a block covers at a time
  const int r_off = per_row < 256 ? tid / per_row : 0;
  const int g0 = per_row < 256 ? tid - r_off * per_row : tid;
  unsigned mag = 0u;
  if (r_off < rpb) {
    const long long step = (long long)s.blocks * rpb;
    for (long long r0 = (long long)blk * rpb + r_off; r0 < s.rows; r0 += 4 * step) {
      for (int g = g0; g < per_row; g += 256) {
        float4 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          x[i] = r0 + i * step < s.rows ? load_group(s, r0 + i * step, 4 * g) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (!SPLIT) {
            mag = max(mag, max(max(finite_magnitude(x[i].x), finite_magnitude(x[i].y)),
                               max(finite_magnitude(x[i].z), finite_magnitude(x[i].w))));
          } else if (r0 + i * step < s.rows) {
            uint2 h, l;
            split4(x[i], sc, h, l);                        // (ld_out is a multiple of 8: a whole group always fits)
            *reinterpret_cast<uint2*>(s.hi + (r0 + i * step) * s.ld_out + 4 * g) = h;
            *reinterpret_cast<uint2*>(s.lo + (r0 + i * step) * s.ld_out + 4 * g) = l;
          }
        }
      }
    }
  }
  if (!SPLIT) {
    mag = __reduce_max_sync(0xffffffffu, mag);
    if ((tid & 31) == 0) sh[tid >> 5] = mag;
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int i = 1; i < 8; ++i) mag = max(mag, sh[i]);
      s.part[blk] = mag;
    }
  }
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
  const int kc = chunk_kb * H_BK;
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

HEpilogue make_epilogue(const GemmArgs& g, unsigned* amax_out) {
  HEpilogue e{};
  e.M = g.M; e.N = g.N; e.D = g.D; e.ldd = g.ldd; e.bias = g.bias; e.sigmoid = g.sigmoid ? 1 : 0;
  e.dsig = g.dsig; e.ld_dsig = g.ld_dsig; e.dsig_rows = g.dsig_rows > 0 ? g.dsig_rows : 1; e.dsig_div = g.dsig_div > 0 ? g.dsig_div : 1;
  e.dsig_direct = e.dsig_div == 1 && e.dsig_rows >= g.M;
  e.alpha = g.alpha; e.cin = g.cin; e.ld_cin = g.ld_cin; e.beta = g.beta;
  e.vec = g.N % 4 == 0 && aligned16(g.D) && g.ldd % 4 == 0 && (!g.bias || aligned16(g.bias)) && (!g.dsig || (aligned16(g.dsig) && g.ld_dsig % 4 == 0)) &&
          (!g.cin || (aligned16(g.cin) && g.ld_cin % 4 == 0));
  e.amax_out = amax_out;
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

int launch_gemm_f16x3(const GemmArgs& g, const SplitOperand* ops, float* ws, unsigned* amax_out, int* err_flag, cudaStream_t st) {
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
      p.amax[2 * s + q] = ops[2 * src + q].amax;
      p.reset[2 * s + q] = s < n_pairs ? ops[2 * s + q].reset : nullptr;
    }
  }
  p.e = make_epilogue(g, amax_out);
  p.n_pairs = n_pairs;
  p.a_mn = g.a_kmajor ? 0 : 1; p.b_mn = g.b_kmajor ? 0 : 1;
  p.bn = pl.bn;
  p.tiles_n = (g.N + pl.bn - 1) / pl.bn;
  p.chunk_kb = g.chunk_kb;
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

int launch_split_f16(const SplitJob* jobs, int n, unsigned* part, cudaStream_t st) {
  if (n < 1 || n > kSplitSegs) return -1;
  SplitList all{}, need{};
  int blocks_all = 0, blocks_need = 0;
  for (int i = 0; i < n; ++i) {
    const SplitJob& j = jobs[i];
    SplitSeg s{};
    s.src = j.src; s.rows = j.rows; s.cols = j.cols; s.ld = j.ld;
    s.hi = static_cast<__half*>(j.hi); s.lo = static_cast<__half*>(j.lo); s.ld_out = j.ld_out;
    s.bits = j.bits;
    s.vec = j.cols % 4 == 0 && j.ld % 4 == 0 && aligned16(j.src);
    const int per_row = (j.cols + 3) / 4;
    const int rpb = per_row < 256 ? 256 / per_row : 1;
    long long b = (j.rows + rpb - 1) / rpb;
    b = (b + 3) / 4;                                       // (four rows in flight per thread)
    if (b < 1) b = 1;
    if (b > kSplitBlocks / n) b = kSplitBlocks / n;
    s.blocks = (int)b;
    s.block0 = blocks_all;
    blocks_all += s.blocks;
    if (j.acc) {                                           // the producer's epilogue has left the maximum
      s.part = j.acc; s.n_part = 1;
    } else {
      s.part = part + s.block0; s.n_part = s.blocks;
      SplitSeg q = s;
      q.block0 = blocks_need;
      blocks_need += q.blocks;
      need.s[need.n++] = q;
    }
    all.s[all.n++] = s;
  }
  int launches = 0;
  if (need.n) {
    if (launch_pdl(split_f16_kernel<false>, blocks_need, 256, 0, st, need) != cudaSuccess) return -1;
    ++launches;
  }
  if (launch_pdl(split_f16_kernel<true>, blocks_all, 256, 0, st, all) != cudaSuccess) return -1;
  return launches + 1;
}

}  // namespace gn
