// TF32 tensor-core GEMM for sm_100a: tcgen05.mma with the accumulator in tensor memory, operands
// staged in shared memory by TMA (128-byte swizzle), fused epilogue read back with tcgen05.ld.
//
// Operands of the CTA-pair kernel may also be FP16 copies (see HalfInfo in gn_kernels.h): the same numbers up to a power of two, in
// half the bytes and at twice the rate.  18944 x 2048 x 2048: 241 us with TF32 operands, 141 us with copies; 16384 x
// 4096 x 4096: 801 and 433 us, 1270 TFLOP/s.
//
// Persistent kernels.  One CTA per SM, each walking 128 x bn output tiles (the CTA-pair kernel further down).  Warp roles:
//   warp 0      TMA producer: fills a ring of STAGES operand buffers (issue spread over lanes)
//   warp 1      MMA issuer   (one elected lane): 4 x (128 x bn x 8) tcgen05.mma per ring slot
//   warps 2..9  epilogue: two warps per 32-lane quadrant of tensor memory, alternating over the
//               tile's 32-column chunks; registers only (shared-memory bandwidth belongs to the
//               MMA and TMA), all of a chunk's global reads issued before the accumulator is read
// Two accumulators alternate in tensor memory, so a tile's epilogue overlaps the next tile's MMAs.
// Up to two (A, B) operand pairs are accumulated into the same tile (the forward directional
// derivative needs R z^{m-1} W^m + z^{m-1} V^m in one accumulator).
//
// Operand layouts in shared memory (32-bit elements, rows of 128 B):
//   K-major  : rows = M (or N) index, 32 consecutive K elements per row; plain 128-byte swizzle
//              (16-byte units permuted over 8 rows).  Descriptor: stride between 8-row groups
//              1024 B; one MMA (K = 8) advances 32 B inside the row.
//   MN-major : the global operand is [K][MN] with MN contiguous; it is staged as chunks of 32 MN
//              elements, each chunk = BK rows (K index) of 128 B.  32-bit MN-major operands must
//              use the 128-byte swizzle with 32-byte atoms (32-byte units permuted over 4 rows), in
//              the tensor map and in the descriptor alike.  Descriptor: leading-dimension offset =
//              chunk size (BK * 128 B), stride between 4-row groups 512 B; one MMA (K = 8)
//              advances 1024 B.
// Every wait on an mbarrier is bounded: after about two seconds the waiting role records an error
// code in global memory and the CTA drains and exits (tensor memory is always released).
#include <cuda_fp16.h>

#include "gn_kernels.h"
#include "half_common.cuh"
#include "tc_common.cuh"

namespace gn {
namespace {

constexpr int BM = 128, BK = 32, BN_MAX = 256;
constexpr int A_STAGE_BYTES = BM * BK * 4;  // 16 KB

struct Tf32Params {
  // (what the producer and the MMA issuer look at before their first instruction stands together: parameters are read through
  // the constant cache, and every line of it that is new to an SM costs some hundred cycles)
  int M, N;
  int kblocks[2];
  int a_mn, b_mn;
  int a_3d, b_3d;       // MN-major operand fetched with one 3-D box per stage (needs a padded operand)
  int bn;               // tile width: multiple of 32, 32 <= bn <= 256
  int tiles_n, tiles;
  // work list of the two-CTA kernel: pair q runs tiles q, q + P, ... for `waves` full waves of P tiles;
  // the `rem` tiles left over are each cut along K into `slices` parts, one per pair, done before the
  // pair's whole tiles (slices == 1: whole tiles, done last)
  int P, waves, rem, slices;
  // FP16 copies (CTA-pair kernel): half = every operand has one, k-blocks of 64 terms, K; further down the infos of A1, B1, A2, B2,
  // where the copy of D goes (copy_out), its info, and the infos of GemmArgs::h_next
  int half, copy_out;
  int khalf[2];
  int K[2];
  float alpha;
  int sigmoid;
  int vec_epi;          // D, bias, dsig, cin all 16-byte aligned with leading dimensions % 4 == 0, N % 4 == 0
  float* D; long long ldd;
  const float* bias;
  const float* dsig; long long ld_dsig; int dsig_rows, dsig_div;
  const float* cin; long long ld_cin; float beta;
  const HalfInfo* hin[4];
  __half* Dh; long long ldh; HalfInfo* hout;
  const HalfInfo* hnext[3];
  int* err;
  float* sk_ws;          // [P][2][128][256] raw partial accumulators of the sliced tiles, slot = pair
  int* sk_flags;         // [P] arrival counters, one per sliced tile; zero between launches (the kernel resets them)
};

// Up to MAX_GROUP independent problems in one launch of the two-CTA kernel.  Pair q runs, problem after problem,
// its tiles of the problem's whole waves (q, q + P, ...) and then tiles rstart[g][q] .. rstart[g][q + 1] - 1 of the
// tiles left over after those waves; the host deals the left-over tiles so that the pairs' total loads come out even
// (longest tiles first), which lets the short tiles of one problem fill the partial last wave of another.
constexpr int MAX_GROUP = 6;
constexpr int MAX_PAIRS_LAUNCH = 80;        // >= SMs / 2
//
// A launch with one problem may cut left-over tiles along K, one with several may chain them, and neither has the code of the other;
// one without FP16 copies (HALF false) has nothing of theirs, neither maps nor code.  Parameters are copied at every launch: with 9 KB
// of them in all launches (six problems and the maps of their copies; one problem without copies takes 1 KB) a full CG step
// of 54-40-2540-14 with 883 rows took 163 us instead of 155, a 700 x 50 product 4 us more.
template <int NP>
struct GroupParams {
  int n_prob;
  Tf32Params pr[NP];
  unsigned short rstart[NP][MAX_PAIRS_LAUNCH + 1];
  // Dependent problems in one launch (a chain of layers): problem g may read, as an operand, what problem
  // dep_prob[g] (earlier in the list) writes.  dep_all[g] == 0: a tile of g needs the producer's tiles of the
  // same 256-row panel (its A rows are the producer's output rows); dep_all[g] == 1: it needs all of them (its
  // K runs over the producer's rows).  The epilogue warps of a producer count finished tiles per panel
  // (signal bit 0) and in total (bit 1) in `done`; the TMA warps of a consumer wait, bounded, for the count.
  // Every pair works through the problems in list order and all pairs are resident, so a wait is always for
  // work that is running or about to run on another pair.
  int dep_prob[NP];
  int dep_all[NP];
  int signal[NP];
  // (bit 30 of a counter: a copy written by these tiles may not be used)
  int* done;                 // [n_prob][done_stride]: entry i < done_stride - 1 counts panel i, the last entry all tiles
  int done_stride;
};
template <int NP, bool HALF>
struct GroupMaps { CUtensorMap m[NP][HALF ? 8 : 4]; };   // per problem: A0, B0, A1, B1, then the same of their FP16 copies

__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
// Persistent kernel: CTA b works on tiles b, b + gridDim.x, ...  Tile = 128 rows x p.bn columns
// (p.bn a multiple of 32, at most 256).  Two accumulators of 256 tensor-memory columns alternate so
// that the epilogue of one tile overlaps the MMAs of the next.
template <int STAGES>
__global__ void __launch_bounds__(320, 1)
gemm_tf32_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmB0,
                 const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                 const Tf32Params p) {
  constexpr int B_STAGE_MAX = BN_MAX * BK * 4;
  constexpr int STAGE_BYTES = A_STAGE_BYTES + B_STAGE_MAX;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;   // [2]
  uint64_t* acc_empty = acc_full + 2;    // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total_kb = p.kblocks[0] + p.kblocks[1];
  const int bn = p.bn;
  const uint32_t stage_tx = A_STAGE_BYTES + (uint32_t)bn * BK * 4;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 8); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {  // all 512 tensor-memory columns: two 128 x 256 FP32 accumulators
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();
  grid_dep_launch();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (TMA issue spread over lanes)
    int it = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x) {
      const int m0 = (t / p.tiles_n) * BM, n0 = (t % p.tiles_n) * bn;
      for (int kb = 0; kb < total_kb; ++kb, ++it) {
        const int s = it % STAGES;
        const uint32_t ph = (it / STAGES) & 1;
        int good = 1;
        if (lane == 0) good = wait_or_abort(&empty[s], ph ^ 1, abort_flag, p.err, 1) ? 1 : 0;
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) { ok = false; break; }
        if (lane == 0) mbar_expect_tx(&full[s], stage_tx);
        __syncwarp();
        const int pair = kb < p.kblocks[0] ? 0 : 1;
        const int k0 = (pair == 0 ? kb : kb - p.kblocks[0]) * BK;
        const CUtensorMap* ma = pair == 0 ? &tmA0 : &tmA1;
        const CUtensorMap* mb = pair == 0 ? &tmB0 : &tmB1;
        uint8_t* sa = smem + s * STAGE_BYTES;
        uint8_t* sb = sa + A_STAGE_BYTES;
        if (!p.a_mn) {
          if (lane == 0) tma_load_2d(sa, ma, k0, m0, &full[s]);
        } else if (p.a_3d) {
          if (lane == 0) tma_load_3d(sa, ma, 0, k0, m0 / 32, &full[s]);
        } else if (lane < BM / 32) {
          tma_load_2d(sa + lane * (BK * 128), ma, m0 + 32 * lane, k0, &full[s]);
        }
        if (!p.b_mn) {
          if (lane == 8) tma_load_2d(sb, mb, k0, n0, &full[s]);
        } else if (p.b_3d) {
          if (lane == 8) tma_load_3d(sb, mb, 0, k0, n0 / 32, &full[s]);
        } else if (lane >= 8 && lane < 8 + bn / 32) {
          const int c = lane - 8;
          tma_load_2d(sb + c * (BK * 128), mb, n0 + 32 * c, k0, &full[s]);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------------------------------------------------------- MMA issuer
      // instruction descriptor: D = F32, A = B = TF32, majors, N >> 3, M >> 4
      const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(p.a_mn ? 1 : 0) << 15) |
                             ((uint32_t)(p.b_mn ? 1 : 0) << 16) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      const uint32_t a_lbo = p.a_mn ? BK * 128 : 16, b_lbo = p.b_mn ? BK * 128 : 16;
      const uint32_t a_step = p.a_mn ? 1024 : 32, b_step = p.b_mn ? 1024 : 32;
      const uint32_t a_sbo = p.a_mn ? 512 : 1024, b_sbo = p.b_mn ? 512 : 1024;
      const uint32_t a_lay = p.a_mn ? 1 : 2, b_lay = p.b_mn ? 1 : 2;
      int it = 0, ti = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x, ++ti) {
        const int buf = ti & 1;
        const uint32_t aph = (ti >> 1) & 1;
        ok = wait_or_abort(&acc_empty[buf], aph ^ 1, abort_flag, p.err, 4);   // epilogue has drained this accumulator
        if (!ok) break;
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(buf * BN_MAX);
        for (int kb = 0; kb < total_kb; ++kb, ++it) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1;
          ok = wait_or_abort(&full[s], ph, abort_flag, p.err, 2);
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + s * STAGE_BYTES);
          const uint32_t sb = sa + A_STAGE_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 8; ++k) {
            const uint64_t ad = make_desc(sa + k * a_step, a_lbo, a_sbo, a_lay);
            const uint64_t bd = make_desc(sb + k * b_step, b_lbo, b_sbo, b_lay);
            mma_tf32(tmem_d, ad, bd, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          mma_commit(&empty[s]);  // frees the slot once these MMAs have read it
        }
        if (ok) mma_commit(&acc_full[buf]);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9)
    // Two warps per tensor-memory quadrant; the pair alternates over the tile's 32-column chunks.
    const int quad = warp & 3;            // tensor-memory lanes 32*quad .. 32*quad+31 are this warp's
    const int half = (warp - 2) >> 2;     // 0 or 1: which chunks of the tile this warp takes
    const float* const bias = dep(p.bias);
    const float* const dsig = dep(p.dsig);
    const float* const cin = dep(p.cin);
    int ti = 0;
    for (int t = blockIdx.x; t < p.tiles; t += gridDim.x, ++ti) {
      const int m0 = (t / p.tiles_n) * BM, n0 = (t % p.tiles_n) * bn;
      const int buf = ti & 1;
      const uint32_t aph = (ti >> 1) & 1;
      int good = 1;
      if (lane == 0) good = wait_or_abort(&acc_full[buf], aph, abort_flag, p.err, 3) ? 1 : 0;
      good = __shfl_sync(0xffffffffu, good, 0);
      if (!good) break;
      tc_fence_after();
      // Registers only: the MMA's operand reads and the TMA writes already use all of the shared-memory
      // bandwidth, so staging the tile through shared memory would starve.  Lane = row; every lane
      // moves 16 bytes per access and a row's 128 bytes are completed by consecutive accesses.
      const int m = m0 + quad * 32 + lane;
      const bool m_ok = m < p.M;
      const float* zrow = dsig ? dsig + (long long)((m / p.dsig_div) % p.dsig_rows) * p.ld_dsig : nullptr;
      const float* crow = cin ? cin + (long long)m * p.ld_cin : nullptr;
      float* drow = p.D + (long long)m * p.ldd;
      for (int c = half; c < bn / 32; c += 2) {
        const int nb = n0 + c * 32;
        if (nb >= p.N) break;               // warp-uniform
        const bool full = p.vec_epi && nb + 32 <= p.N;   // warp-uniform: whole chunk in range and 16-byte aligned
        float4 zc[8], ci[8];
        if (full && m_ok) {                 // all global reads of the chunk in flight before anything waits
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            zc[q] = zrow ? __ldg(reinterpret_cast<const float4*>(zrow + nb) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
            ci[q] = crow ? __ldg(reinterpret_cast<const float4*>(crow + nb) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
        float v[32];
        tmem_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * BN_MAX + c * 32), v);
        if (!m_ok) continue;
        if (full) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            float4 bz = make_float4(0.f, 0.f, 0.f, 0.f);
            if (bias) bz = __ldg(reinterpret_cast<const float4*>(bias + nb) + q);
            float x[4] = {v[4 * q] + bz.x, v[4 * q + 1] + bz.y, v[4 * q + 2] + bz.z, v[4 * q + 3] + bz.w};
            const float z[4] = {zc[q].x, zc[q].y, zc[q].z, zc[q].w};
            const float cc[4] = {ci[q].x, ci[q].y, ci[q].z, ci[q].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (p.sigmoid) x[j] = 1.f / (1.f + __expf(-x[j]));
              if (zrow) x[j] *= z[j] * (1.f - z[j]);
              x[j] *= p.alpha;
              if (crow) x[j] = fmaf(p.beta, cc[j], x[j]);
            }
            reinterpret_cast<float4*>(drow + nb)[q] = make_float4(x[0], x[1], x[2], x[3]);
          }
        } else {                             // ragged or unaligned chunk: element by element
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const int n = nb + j;
            if (n < p.N) {
              float x = v[j] + (bias ? __ldg(bias + n) : 0.f);
              if (p.sigmoid) x = 1.f / (1.f + __expf(-x));
              if (zrow) { const float z = __ldg(zrow + n); x *= z * (1.f - z); }
              x *= p.alpha;
              if (crow) x = fmaf(p.beta, __ldg(crow + n), x);
              drow[n] = x;
            }
          }
        }
      }
      // this warp has read its quadrant of the accumulator: let the MMA issuer reuse it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

// ------------------------------------------------------------------------------------------------
// Two-CTA variant: a cluster of two CTAs (two SMs) computes one 256 x bn tile with
// tcgen05.mma.cta_group::2.  CTA r of the pair owns rows [128 r, 128 r + 128) of the tile (its A block
// and its accumulator) and stages half of the B tile (bn/2 rows); the tensor cores of both SMs read
// both halves.  Per k-block each SM therefore moves 16 KB + 16 KB instead of 16 KB + 32 KB through
// shared memory, which is what limits the one-CTA kernel.
// Protocol: both producers wait on their own empty[s] (released in both CTAs by a multicast commit),
// only the leader (rank 0) arms full[s] with the bytes of both CTAs, and both CTAs' TMA loads complete
// on the leader's full[s].  MMAs are issued by the leader only.  acc_full[b] is multicast to both
// CTAs; all 32 epilogue warps of the pair arrive on the leader's acc_empty[b].  Sixteen epilogue warps per CTA, four per scheduler,
// because their time is latency (12000 x 2000 x 784 on copies with the sigmoid: 105 us with eight, 63 us with sixteen), at 96 registers,
// which leaves room on the SM for a block of the column-sum kernel that runs beside this one (576 x 96 + 256 x 40 = 65536).
//
// Work list: with T tiles on P pairs, pair q runs tiles q, q + P, ... for the floor(T / P) full waves, so
// that all pairs move through neighbouring tiles together (tiles of one A panel are read at the same
// time and hit in L2).  The T mod P tiles left over are each cut along K into up to 16 slices, one per
// pair, and a pair does its slice before its whole tiles.  The pairs of a sliced tile store their raw
// accumulators in a workspace, count themselves in on the tile's flag, wait (bounded) until all slices
// have arrived, and then each sums one share of the tile's column chunks over all slices, in slice
// order, and runs the epilogue on it - all of this on the epilogue warps while the MMA issuer is already
// working on the pair's first whole tile in the other accumulator.  The order of every sum is fixed, so
// results are deterministic.
__device__ __forceinline__ void mma2_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
// The same with FP16 operands (K = 16 per instruction: as many bytes of operands and as long, twice the terms).
__device__ __forceinline__ void mma2_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
// ... adding to the accumulator times 2^-S
template <int S>
__device__ __forceinline__ void mma2_f16_scaled(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.eq.b32 p, 0, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p, %4;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "n"(S) : "memory");
}
__device__ __forceinline__ void mma2_f16_shift(int s, uint32_t d, uint64_t a, uint64_t b, uint32_t i) {
  switch (s) {
    case 1: mma2_f16_scaled<1>(d, a, b, i); break;
    case 2: mma2_f16_scaled<2>(d, a, b, i); break;
    case 3: mma2_f16_scaled<3>(d, a, b, i); break;
    case 4: mma2_f16_scaled<4>(d, a, b, i); break;
    case 5: mma2_f16_scaled<5>(d, a, b, i); break;
    case 6: mma2_f16_scaled<6>(d, a, b, i); break;
    case 7: mma2_f16_scaled<7>(d, a, b, i); break;
    case 8: mma2_f16_scaled<8>(d, a, b, i); break;
    case 9: mma2_f16_scaled<9>(d, a, b, i); break;
    case 10: mma2_f16_scaled<10>(d, a, b, i); break;
    case 11: mma2_f16_scaled<11>(d, a, b, i); break;
    case 12: mma2_f16_scaled<12>(d, a, b, i); break;
    case 13: mma2_f16_scaled<13>(d, a, b, i); break;
    case 14: mma2_f16_scaled<14>(d, a, b, i); break;
    default: mma2_f16_scaled<15>(d, a, b, i); break;
  }
}

constexpr int BK_HALF = 64;                    // K elements of a 128-byte row of FP16
constexpr unsigned kBadPanel = 1u << 30;       // in a counter of finished tiles: their rows of the copy may not be used

// What the producer finds out about a problem from the copies' infos (all of them in a few lines of L2, which thousands of
// warps must not read per tile).  use: its tiles are computed from the copies; 2^sum0, 2^sum1: scale of A1 B1 and of A2 B2.  With
// two operand pairs the second goes first, and the first instruction of the first brings the sums to its scale (scale-input-d: exact,
// but downwards only, and by at most 2^-15: a second scaled instruction would scale the first one's own products as well).  A
// pair of pairs further apart is computed from the FP32 matrices.  out: exponent of the scale of D's copy.
constexpr int kMaxScaleStep = 15;
struct HalfUse { int use, sum0, sum1, out; };

// Exponent of the scale of D's copy: |D| is bounded by A's largest magnitude times the largest sum of magnitudes that an output
// column of B has (K times B's largest magnitude where that is not known), and 2^e takes the bound below 2^15.  On 784-2000-2000-2000-10
// with 3000 rows the largest elements then lie at 2^9 to 2^11, with dense and with sparse weights (K times the largest magnitude left them at
// 2^6 to 2^8 and 2^2 to 2^5: runs below kHalfLeast in five of nine copies of a sparse network).  Sigmoids need no
// bound.  Where the next contraction adds A2 B2 to the product of this copy with W (hnext: infos of A2, B2, W), its scale must not
// be above theirs.
constexpr int kSigmoidExp = 15;
__device__ __forceinline__ int out_exponent(const Tf32Params& p, const int (&e)[4], const unsigned (&m)[4]) {
  if (p.sigmoid) return kSigmoidExp;
  float bound = 0.f;
#pragma unroll
  for (int s = 0; s < 2; ++s)
    if (p.K[s] > 0) {
      const HalfInfo* const b = p.hin[2 * s + 1];
      const unsigned long long sum = __ldcg(p.b_mn ? &b->col1 : &b->row1);
      bound += __uint_as_float(m[2 * s]) * (sum ? half_norm(sum, e[2 * s + 1]) : (float)p.K[s] * __uint_as_float(m[2 * s + 1]));
    }
  if (p.bias) bound += __uint_as_float(p.K[1] > 0 ? m[3] : m[1]);
  bound *= fabsf(p.alpha) * (p.dsig ? 0.25f : 1.f);
  const int out = half_exponent(__float_as_uint(bound) & 0x7fffffffu);
  return p.hnext[0] ? min(out, max(-kHalfMaxExp, __ldcg(&p.hnext[0]->e) + __ldcg(&p.hnext[1]->e) - __ldcg(&p.hnext[2]->e))) : out;
}
// a1_here: A1's copy is written by this very launch (a sigmoid's; the tiles say with the counter whether it may be used).
__device__ __forceinline__ HalfUse half_use(const Tf32Params& p, bool a1_here) {
  HalfUse u{0, 0, 0, 0};
  if (!p.half && !p.copy_out) return u;
  const int n = p.K[1] > 0 ? 4 : 2;
  int e[4] = {0, 0, 0, 0};
  unsigned amax[4] = {0u, 0u, 0u, 0u}, bad = 0u;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (k < n) {
      const int4 i = __ldcg(reinterpret_cast<const int4*>(p.hin[k]));
      const bool here = k == 0 && a1_here;
      e[k] = here ? kSigmoidExp : i.x;
      amax[k] = here ? __float_as_uint(1.f) : (unsigned)i.y;
      if (!here) bad |= (unsigned)i.z;
    }
  if (p.half) {
    u.sum0 = e[0] + e[1]; u.sum1 = n == 4 ? e[2] + e[3] : u.sum0;
    u.use = bad == 0u && abs(u.sum0) <= kHalfMaxExp && abs(u.sum1) <= kHalfMaxExp && u.sum1 >= u.sum0 && u.sum1 - u.sum0 <= kMaxScaleStep;
  }
  if (p.copy_out) u.out = out_exponent(p, e, amax);
  return u;
}

// Word from the producer to its CTA's epilogue warps, one per tile, tagged with the tile's place in the pair's work list: form of
// the operands, exponent that undoes the scale of the sums, exponent of the scale of D's copy.  The ring of words is longer
// than the producer can be ahead: two tiles in tensor memory, the operand slots, the tile it is at.
constexpr int TILE_WORDS = 16;
__device__ __forceinline__ int tile_word(int wi, int use, int un, int out) { return use | (un + 128) << 1 | (out + 128) << 9 | ((wi + 1) & 0x3fff) << 17; }

struct Work { int prob, tile, sl, sliced; };

// Its k-blocks: all, or slice sl of them.
__device__ __forceinline__ void k_range(const Tf32Params& p, const Work& w, bool half, int& kb0, int& kb1) {
  const int total = half ? p.khalf[0] + p.khalf[1] : p.kblocks[0] + p.kblocks[1];
  kb0 = w.sliced ? (int)((long long)total * w.sl / p.slices) : 0;
  kb1 = w.sliced ? (int)((long long)total * (w.sl + 1) / p.slices) : total;
}
// Counter of finished tiles that a tile's first A operand (its row panel) or K operand (all) waits for.
template <int NP>
__device__ __forceinline__ const int* dep_counter(const GroupParams<NP>& gp, const Work& w) {
  const int d = gp.dep_prob[w.prob];
  return gp.done + (long long)d * gp.done_stride + (gp.dep_all[w.prob] ? gp.done_stride - 1 : w.tile / gp.pr[w.prob].tiles_n);
}

// idx-th piece of work of CTA pair `pair` (see Tf32Params and GroupParams); false when the pair has no more.
// A single problem whose left-over tiles are cut along K: the pair does its slice FIRST; the store of the partial
// accumulator, the wait for the other slices and the fix-up epilogue then run on the epilogue warps underneath the
// MMAs of the pair's first whole tile instead of being exposed at the end of the kernel.
template <int NP>
__device__ __forceinline__ bool next_work(const GroupParams<NP>& gp, int pair, int idx, Work& w) {
  if (NP == 1 && gp.pr[0].slices >= 2) {
    const Tf32Params& p = gp.pr[0];
    w.prob = 0;
    if (pair < p.rem * p.slices) {
      if (idx == 0) {
        const int j = pair / p.slices;
        w.tile = p.waves * p.P + j;
        w.sl = pair - j * p.slices;
        w.sliced = 1;
        return true;
      }
      --idx;
    }
    if (idx >= p.waves) return false;
    w.tile = idx * p.P + pair; w.sl = 0; w.sliced = 0;
    return true;
  }
  for (int g = 0; g < (NP == 1 ? 1 : gp.n_prob); ++g) {
    const Tf32Params& p = gp.pr[g];
    const int r0 = gp.rstart[g][pair], n_rem = gp.rstart[g][pair + 1] - r0;
    if (idx < p.waves + n_rem) {
      w.prob = g; w.sl = 0; w.sliced = 0;
      w.tile = idx < p.waves ? idx * p.P + pair : p.waves * p.P + r0 + (idx - p.waves);
      return true;
    }
    idx -= p.waves + n_rem;
  }
  return false;
}

// Epilogue of a warp's 16 x 32 pieces of a tile, on 16-byte aligned rows, in the fragment layout of tmem_ld_16x256b_x4: value
// v[4j + 2e + i] is element (row 8e + lane / 4, column 8j + 2 (lane % 4) + i).  Sixteen warps run this beside the main loop, four per
// scheduler; each waits for its operands most of the time, so the warps' number and the loads they keep in flight are
// what counts (a piece's operands are requested before the piece before it is computed), and after that the instruction stream.
// MODE fixes the options at compile time: 0 = alpha * acc (+ bias), 1 = sigmoid, 2 = times the sigmoid derivative of `dsig`,
// 3 = plus beta * cin.  (Combinations, none of them on the path, go element by element: epilogue_ragged.)
struct EpiArgs {
  float un;                  // what undoes the scale of the sums (1 for TF32 operands)
  float hsc;                 // scale of D's copy
};

// Row of dsig that belongs to row m (m itself without a division where it can be).
__device__ __forceinline__ long long dsig_row(const Tf32Params& p, int m) {
  return p.dsig_div == 1 && p.dsig_rows >= p.M ? m : (m / p.dsig_div) % p.dsig_rows;
}

// This warp's pieces of a tile: column chunks first, first + step, ... below end of the 16 rows whose element 0 this thread holds in
// row m (and m + 8); column nb0 + 32 c of this thread in chunk c.  slices > 0: a tile cut along K, its partial sums at ws.
struct PieceRun { uint32_t taddr; int m, nb0, first, step, end; const float* ws; int slices; };

// The sums of a piece: from tensor memory, or of the slices' partials, slice 0 first.
__device__ __forceinline__ void piece_sums(const PieceRun& r, int c, float (&v)[16]) {
  if (r.slices == 0) {
    tmem_ld_16x256b_x4(r.taddr + (uint32_t)(c * 32), v);
    tmem_ld_wait();
    return;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = 0.f;
  for (int s2 = 0; s2 < r.slices; ++s2) {
    const float* wsr = r.ws + c * 32 + (long long)s2 * (2 * BM * BN_MAX);
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 x = __ldcg(reinterpret_cast<const float2*>(wsr + (8 * e) * BN_MAX + 8 * j));
        v[4 * j + 2 * e] += x.x; v[4 * j + 2 * e + 1] += x.y;
      }
  }
}

// The runs of a copy that are looked at are a piece's 32 elements of a row and 16 of a column.  A thread has 8 and 2 of them; only if
// these lie low (`check` says so, for some thread of the warp) is the piece looked at as a whole: read back from D, which the
// same threads have just written, so that the common case pays for a vote and holds nothing more in registers.
__device__ __noinline__ bool low_piece(const float* drow, long long ldd, int rows, int n, int N, float hsc) {
  const int lane = threadIdx.x & 31;
  const bool whole_col = rows + lane / 4 >= 16, whole_row = n - 2 * (lane & 3) + 32 <= N;
  float y[2][8];
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int j = 0; j < 8; ++j)
      y[e][j] = 8 * e < rows && n + 8 * (j / 2) + j % 2 < N ? fabsf(drow[8 * e * ldd + 8 * (j / 2) + j % 2] * hsc) : 0.f;
  HalfCheck check;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) m = fmaxf(m, y[e][j]);
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    if (whole_row) check.run(m);
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    float m = fmaxf(y[0][j], y[1][j]);
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 4));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    if (whole_col) check.run(m);
  }
  return __any_sync(0xffffffffu, check.low_run());
}
// A piece is done: its low runs, if it has any, belong to longer ones that are not low, or make the copy bad.
__device__ __forceinline__ void end_piece(const Tf32Params& p, const PieceRun& r, int c, float hsc, HalfCheck& check) {
  if (!__any_sync(0xffffffffu, check.low_run())) return;
  check.low = low_piece(p.D + (long long)r.m * p.ldd + r.nb0 + c * 32, p.ldd, p.M - r.m, r.nb0 + c * 32, p.N, hsc) ? 0u : 0xffffffffu;
}

// HALF: D's FP16 copy is written too.  Two threads swap halves of what they hold so that a store covers whole 32-byte sectors.
template <int MODE, bool HALF>
__device__ __forceinline__ void epilogue_pieces(const Tf32Params& p, const EpiArgs& a, const PieceRun& r, int lane, HalfCheck& check) {
  constexpr bool ONE_OP = MODE == 2 || MODE == 3;
  const int N = p.N;
  const bool ok[2] = {r.m < p.M, r.m + 8 < p.M};
  const float* orow[2] = {nullptr, nullptr};   // this thread's rows of dsig (mode 2) or of cin (mode 3)
  if (ONE_OP) {
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (ok[e]) orow[e] = (MODE == 3 ? dep(p.cin) + (long long)(r.m + 8 * e) * p.ld_cin : dep(p.dsig) + dsig_row(p, r.m + 8 * e) * p.ld_dsig) + r.nb0;
  }
  const float* const bias = dep(p.bias);
  float* const drow = p.D + (long long)r.m * p.ldd + r.nb0;
#pragma unroll 1
  for (int c = r.first; c < r.end; c += r.step) {
    bool in[4];                                // (N is a multiple of four: a thread's pair, and what it stores of a copy, is in or out)
#pragma unroll
    for (int j = 0; j < 4; ++j) in[j] = r.nb0 + c * 32 + 8 * j < N;
    float2 op[ONE_OP ? 8 : 1];                 // [4e + j], requested before anything is waited for
    if (ONE_OP) {
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float2 x = make_float2(0.f, 0.f);
          // (cin: L2-coherent read, in a chained launch it may have been written by another pair of this very launch)
          if (ok[e] && in[j]) x = MODE == 3 ? __ldcg(reinterpret_cast<const float2*>(orow[e] + c * 32 + 8 * j)) : __ldg(reinterpret_cast<const float2*>(orow[e] + c * 32 + 8 * j));
          op[ONE_OP ? 4 * e + j : 0] = x;
        }
    }
    float2 bz[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) bz[j] = bias && in[j] ? __ldg(reinterpret_cast<const float2*>(bias + r.nb0 + c * 32 + 8 * j)) : make_float2(0.f, 0.f);
    float v[16];
    piece_sums(r, c, v);
    unsigned hv[2][HALF ? 4 : 1];
    float row[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float c0 = 0.f, c1 = 0.f;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float x0 = fmaf(v[4 * j + 2 * e], a.un, bz[j].x), x1 = fmaf(v[4 * j + 2 * e + 1], a.un, bz[j].y);
        if (MODE == 1) { x0 = sigmoid_from(__expf(-x0)); x1 = sigmoid_from(__expf(-x1)); }
        if (MODE == 2) {
          const float2 z = op[ONE_OP ? 4 * e + j : 0];
          x0 *= z.x * (1.f - z.x); x1 *= z.y * (1.f - z.y);
        }
        x0 *= p.alpha; x1 *= p.alpha;
        if (MODE == 3) {
          const float2 cc = op[ONE_OP ? 4 * e + j : 0];
          x0 = fmaf(p.beta, cc.x, x0); x1 = fmaf(p.beta, cc.y, x1);
        }
        if (ok[e] && in[j]) *reinterpret_cast<float2*>(drow + 8 * e * p.ldd + c * 32 + 8 * j) = make_float2(x0, x1);
        if (HALF) {
          const float y0 = ok[e] && in[j] ? x0 * a.hsc : 0.f, y1 = ok[e] && in[j] ? x1 * a.hsc : 0.f;
          row[e] = max3_abs(row[e], y0, y1);
          if (e == 0) { c0 = y0; c1 = y1; } else { check.run(max3_abs(c0, y0, y0)); check.run(max3_abs(c1, y1, y1)); }
          const __half2 y = __floats2half2_rn(y0, y1);
          hv[e][HALF ? j : 0] = *reinterpret_cast<const unsigned*>(&y);
        }
      }
    }
    if (HALF) {
      const bool odd = lane & 1;
      __half* const hrow = p.Dh + (long long)r.m * p.ldh + r.nb0 + c * 32 + (odd ? 6 : 0);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        check.run(row[e]);
#pragma unroll
        for (int j = 0; j < 4; j += 2) {       // even lanes: columns 8 j + 0..3 or 4..7, odd lanes the same of 8 (j + 1)
          const unsigned mine = odd ? hv[e][HALF ? j + 1 : 0] : hv[e][HALF ? j : 0];
          const unsigned other = __shfl_xor_sync(0xffffffffu, odd ? hv[e][HALF ? j : 0] : hv[e][HALF ? j + 1 : 0], 1);
          if (ok[e] && (odd ? in[j + 1] : in[j])) *reinterpret_cast<uint2*>(hrow + 8 * e * p.ldh + 8 * j) = odd ? make_uint2(other, mine) : make_uint2(mine, other);
        }
      }
      end_piece(p, r, c, a.hsc, check);
    }
  }
}

// The same of pieces that are ragged or unaligned, or that combine options, element by element.
template <bool HALF>
__device__ __forceinline__ HalfCheck epilogue_ragged(const Tf32Params& p, const EpiArgs& a, const PieceRun& r) {
  HalfCheck check;
  const int N = p.N;
  const float* const bias = p.bias ? dep(p.bias) + r.nb0 : nullptr;
  const float* const dsig = dep(p.dsig);
  const float* const cin = dep(p.cin);
  const float* zrow[2] = {nullptr, nullptr};   // this thread's rows of dsig and cin
  const float* crow[2] = {nullptr, nullptr};
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (r.m + 8 * e < p.M) {
      if (dsig) zrow[e] = dsig + dsig_row(p, r.m + 8 * e) * p.ld_dsig + r.nb0;
      if (cin) crow[e] = cin + (long long)(r.m + 8 * e) * p.ld_cin + r.nb0;
    }
  float* const drow = p.D + (long long)r.m * p.ldd + r.nb0;
#pragma unroll 1
  for (int c = r.first; c < r.end; c += r.step) {
    float v[16];
    piece_sums(r, c, v);
    float row[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int n = c * 32 + 8 * j + i;
        float col = 0.f;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (r.nb0 + n < N && r.m + 8 * e < p.M) {
            float x = fmaf(v[4 * j + 2 * e + i], a.un, bias ? __ldg(bias + n) : 0.f);
            if (p.sigmoid) x = sigmoid_from(__expf(-x));
            if (dsig) { const float z = __ldg(zrow[e] + n); x *= z * (1.f - z); }
            x *= p.alpha;
            if (cin) x = fmaf(p.beta, __ldcg(crow[e] + n), x);
            drow[8 * e * p.ldd + n] = x;
            if (HALF && p.copy_out) {
              const float y = x * a.hsc;
              row[e] = max3_abs(row[e], y, y);
              col = max3_abs(col, y, y);
              p.Dh[(long long)(r.m + 8 * e) * p.ldh + r.nb0 + n] = __float2half_rn(y);
            }
          }
        }
        if (HALF && p.copy_out) check.run(col);
      }
    if (HALF && p.copy_out) { check.run(row[0]); check.run(row[1]); end_piece(p, r, c, a.hsc, check); }
  }
  return check;
}

constexpr int PAIR_EPI_WARPS = 16, PAIR_THREADS = 64 + 32 * PAIR_EPI_WARPS;
constexpr int B2_STAGE_MAX = (BN_MAX / 2) * BK * 4;          // 16 KB: this CTA's half of the B tile
constexpr int STAGE2_BYTES = A_STAGE_BYTES + B2_STAGE_MAX;   // 32 KB

template <int STAGES, int NP, bool HALF>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PAIR_THREADS, 1)
gemm_tf32_2cta_kernel(const __grid_constant__ GroupMaps<NP, HALF> gm, const __grid_constant__ GroupParams<NP> gp) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE2_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;   // [2]
  uint64_t* acc_empty = acc_full + 2;    // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* tile_words = reinterpret_cast<volatile int*>(tmem_slot + 2);  // [TILE_WORDS]
  volatile int* tile_form = tile_words + TILE_WORDS;   // [STAGES], from the producer to the MMA issuer with a
                                                                              // tile's first slot: 1 = FP16 copies, + 2 x scale step
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1;
  int* const err = gp.pr[0].err;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * PAIR_EPI_WARPS); }
    *abort_flag = 0;
    if (HALF)
      for (int i = 0; i < TILE_WORDS; ++i) tile_words[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {  // both CTAs of the pair allocate all 512 columns, same warp, same destination offset
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_sync_all();      // barriers of both CTAs are initialised before anyone signals across the pair
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();
  grid_dep_launch();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (both CTAs)
    int s = 0;                                 // ring slot and its phase
    uint32_t ph = 0;
    bool ok = true;
    Work w;
    HalfUse hu{0, 0, 0, 0};
    int hu_prob = -1;
    for (int wi = 0; ok && next_work(gp, pair, wi, w); ++wi) {
      const Tf32Params& p = gp.pr[w.prob];
      const int bn = p.bn, hb = p.bn >> 1;                     // hb: B rows staged by each CTA
      const int t = w.tile;
      const int m0 = (t / p.tiles_n) * (2 * BM) + (int)rank * BM;
      const int n0 = (t % p.tiles_n) * bn + (int)rank * hb;
      const int dp = NP > 1 ? gp.dep_prob[w.prob] : -1;
      const bool a1_here = HALF && dp >= 0 && p.half && gp.pr[dp].hout == p.hin[0];
      int bad_panel = 0;
      if (dp >= 0) {
        // an operand of this tile is written by an earlier problem of this launch: wait until its tiles are stored
        const int* const ctr = dep_counter(gp, w);
        const int want = 2 * PAIR_EPI_WARPS * (gp.dep_all[w.prob] ? gp.pr[dp].tiles : gp.pr[dp].tiles_n);
        int good = 1;
        if (lane == 0) {
          const unsigned long long t0 = globaltimer();
          int seen;
          while (((seen = ld_acquire_gpu(ctr)) & (int)(kBadPanel - 1u)) < want) {
            if (*abort_flag || globaltimer() - t0 > WAIT_LIMIT_NS) { atomicCAS(err, 0, 6); *abort_flag = 1; good = 0; break; }
            __nanosleep(100);
          }
          if (seen & (int)kBadPanel) good |= 2;
        }
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!(good & 1)) { ok = false; break; }
        bad_panel = good >> 1;
        asm volatile("fence.proxy.async.global;" ::: "memory");   // the stores were generic, the loads below are TMA's
        __syncwarp();
      }
      if (HALF && w.prob != hu_prob) { hu = half_use(p, a1_here); hu_prob = w.prob; }
      const bool half = HALF && hu.use != 0 && !(a1_here && bad_panel);
      int kb0, kb1;
      k_range(p, w, half, kb0, kb1);
      if (HALF && lane == 0)     // (a slice may end before the first operand pair)
        tile_words[wi % TILE_WORDS] = tile_word(wi, half ? 1 : 0, half ? -(p.khalf[1] > 0 && kb1 <= p.khalf[1] ? hu.sum1 : hu.sum0) : 0, hu.out);
      const int first = half && p.khalf[1] > 0 ? 1 : 0;        // operand pair that goes first
      const int n_first = half ? p.khalf[first] : p.kblocks[0];
      // (an FP16 box covers 128 bytes of a row too: a slot holds 64 terms instead of 32.  MN-major copies are staged in chunks of 64
      // columns: a half tile of 96 takes two, each with a box of its own because it does not start on a multiple of 64)
      const int b_boxes = half && p.b_mn ? (hb + 63) / 64 : 0;
      const uint32_t pair_tx = 2u * (A_STAGE_BYTES + (b_boxes ? (uint32_t)b_boxes * 8192u : (uint32_t)hb * BK * 4));
      const int a_boxes = half || !p.a_mn || p.a_3d ? 1 : BM / 32;
      const bool one_box = a_boxes == 1 && (half ? b_boxes < 2 || hb % 64 == 0 : !p.b_mn || p.b_3d);
      if (one_box) {
        // one thread, and nothing in the loop that need not be there (as for the MMA issuer)
        int good = 1;
        if (lane == 0) {
          const CUtensorMap* const maps = gm.m[w.prob] + (half ? 4 : 0);
          const int bk = half ? BK_HALF : BK, am = m0 / (half ? 64 : 32), bm = n0 / (half ? 64 : 32);
          const bool a3 = p.a_mn != 0, b3 = p.b_mn != 0;
          for (int kb = kb0; kb < kb1; ++kb) {
            if (!wait_or_abort(&empty[s], ph ^ 1, abort_flag, err, 1)) { good = 0; break; }
            if (rank == 0) {
              if (HALF && kb == kb0) tile_form[s] = half ? 1 | (hu.sum1 - hu.sum0) << 1 : 0;
              mbar_expect_tx(&full[s], pair_tx);
            }
            const uint32_t full_leader = map_to_cta(smem_u32(&full[s]), 0);
            const int pr = kb < n_first ? first : first ^ 1;
            const int k0 = (kb < n_first ? kb : kb - n_first) * bk;
            uint8_t* sa = smem + s * STAGE2_BYTES;
            if (a3) tma2_load_3d(sa, maps + 2 * pr, 0, k0, am, full_leader);
            else tma2_load_2d(sa, maps + 2 * pr, k0, m0, full_leader);
            if (b3) tma2_load_3d(sa + A_STAGE_BYTES, maps + 2 * pr + 1, 0, k0, bm, full_leader);
            else tma2_load_2d(sa + A_STAGE_BYTES, maps + 2 * pr + 1, k0, n0, full_leader);
            if (++s == STAGES) { s = 0; ph ^= 1u; }
          }
        }
        good = __shfl_sync(0xffffffffu, good, 0);
        s = __shfl_sync(0xffffffffu, s, 0);
        ph = __shfl_sync(0xffffffffu, ph, 0);
        if (!good) { ok = false; break; }
        continue;
      }
      for (int kb = kb0; kb < kb1; ++kb) {
        int good = 1;
        if (lane == 0) good = wait_or_abort(&empty[s], ph ^ 1, abort_flag, err, 1) ? 1 : 0;
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) { ok = false; break; }
        if (rank == 0 && lane == 0) {
          if (HALF && kb == kb0) tile_form[s] = half ? 1 | (hu.sum1 - hu.sum0) << 1 : 0;
          mbar_expect_tx(&full[s], pair_tx);
        }
        __syncwarp();
        const uint32_t full_leader = map_to_cta(smem_u32(&full[s]), 0);
        const int pr = kb < n_first ? first : first ^ 1;
        const int kk = kb < n_first ? kb : kb - n_first;
        uint8_t* sa = smem + s * STAGE2_BYTES;
        uint8_t* sb = sa + A_STAGE_BYTES;
        if (++s == STAGES) { s = 0; ph ^= 1u; }
        if (half) {
          const CUtensorMap* ma = &gm.m[w.prob][HALF ? 4 + 2 * pr : 0];
          const CUtensorMap* mb = ma + 1;
          const int k0 = kk * BK_HALF;
          if (lane == 0) {
            if (!p.a_mn) tma2_load_2d(sa, ma, k0, m0, full_leader);
            else tma2_load_3d(sa, ma, 0, k0, m0 / 64, full_leader);
          } else if (lane == 8) {
            if (!p.b_mn) tma2_load_2d(sb, mb, k0, n0, full_leader);
            else if (hb % 64 == 0) tma2_load_3d(sb, mb, 0, k0, n0 / 64, full_leader);
            else tma2_load_2d(sb, mb, n0, k0, full_leader);
          } else if (lane == 9 && p.b_mn && hb % 64 != 0) {
            tma2_load_2d(sb + 8192, mb, n0 + 64, k0, full_leader);
          }
          continue;
        }
        const int k0 = kk * BK;
        const CUtensorMap* ma = &gm.m[w.prob][2 * pr];
        const CUtensorMap* mb = &gm.m[w.prob][2 * pr + 1];
        if (!p.a_mn) {
          if (lane == 0) tma2_load_2d(sa, ma, k0, m0, full_leader);
        } else if (p.a_3d) {
          if (lane == 0) tma2_load_3d(sa, ma, 0, k0, m0 / 32, full_leader);
        } else if (lane < BM / 32) {
          tma2_load_2d(sa + lane * (BK * 128), ma, m0 + 32 * lane, k0, full_leader);
        }
        if (!p.b_mn) {
          if (lane == 8) tma2_load_2d(sb, mb, k0, n0, full_leader);
        } else if (p.b_3d) {
          if (lane == 8) tma2_load_3d(sb, mb, 0, k0, n0 / 32, full_leader);
        } else if (lane >= 8 && lane < 8 + hb / 32) {
          const int c = lane - 8;
          tma2_load_2d(sb + c * (BK * 128), mb, n0 + 32 * c, k0, full_leader);
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && lane == 0) {
      // ---------------------------------------------------------------- MMA issuer (leader CTA only)
      int s = 0, ti = 0;                       // ring slot and its phase, tiles done
      uint32_t ph = 0;
      bool ok = true;
      Work w;
      for (int wi = 0; ok && next_work(gp, pair, wi, w); ++wi, ++ti) {
        const Tf32Params& p = gp.pr[w.prob];
        const uint32_t shape = (1u << 4) | ((uint32_t)(p.a_mn ? 1 : 0) << 15) | ((uint32_t)(p.b_mn ? 1 : 0) << 16) |
                               ((uint32_t)(p.bn >> 3) << 17) | ((uint32_t)((2 * BM) >> 4) << 24);
        const int buf = ti & 1;
        const uint32_t aph = (ti >> 1) & 1;
        ok = wait_or_abort(&acc_empty[buf], aph ^ 1, abort_flag, err, 4);
        if (!ok) break;
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)(buf * BN_MAX);
        int form = 0;
        if (HALF && p.half) {                  // (comes with the tile's first operands)
          ok = wait_or_abort(&full[s], ph, abort_flag, err, 2);
          if (!ok) break;
          form = tile_form[s];
        }
        const bool half = HALF && form != 0;
        int kb0, kb1;
        k_range(p, w, half, kb0, kb1);
        // scale step: before the first k-block of the first operand pair, where one of the second went before it
        const int step_at = (form >> 1) > 0 && p.khalf[1] > kb0 && p.khalf[1] < kb1 ? p.khalf[1] : -1;
        const uint32_t idesc = shape | (half ? 0u : (2u << 7) | (2u << 10));       // operands: FP16 or TF32
        // MN-major: chunks of 64 (32) columns, BK_HALF (BK) rows of 128 bytes each
        const uint32_t chunk = half ? BK_HALF * 128 : BK * 128, mn_sbo = half ? 1024 : 512, mn_lay = half ? 2 : 1;
        const uint64_t mn_step = (half ? 2048 : 1024) >> 4;
        const uint64_t a_step = p.a_mn ? mn_step : 32 >> 4, b_step = p.b_mn ? mn_step : 32 >> 4;       // (descriptors count in 16 bytes)
        const uint32_t base = smem_u32(smem);
        const uint64_t a0 = make_desc(base, p.a_mn ? chunk : 16, p.a_mn ? mn_sbo : 1024, p.a_mn ? mn_lay : 2);
        const uint64_t b0 = make_desc(base + A_STAGE_BYTES, p.b_mn ? chunk : 16, p.b_mn ? mn_sbo : 1024, p.b_mn ? mn_lay : 2);
        uint32_t acc = 0u;
        // One thread issues everything, and what it takes per k-block (descriptors made anew, ring arithmetic, all forms of the
        // scale step in the loop: 680 cycles with TF32 operands, 900 with FP16) was what bounded the main loop, where the
        // instructions themselves need 512: so nothing is in the loop that need not be there.
        for (int kb = kb0; ok && kb < kb1;) {
          const int end = kb < step_at ? step_at : kb1;
          if (half) {
            if (kb == step_at) {
              if (!wait_or_abort(&full[s], ph, abort_flag, err, 2)) { ok = false; break; }
              tc_fence_after();
              const uint64_t ad = a0 + (uint64_t)(s * (STAGE2_BYTES >> 4)), bd = b0 + (uint64_t)(s * (STAGE2_BYTES >> 4));
              mma2_f16_shift(form >> 1, tmem_d, ad, bd, idesc);
              for (int k = 1; k < 4; ++k) mma2_f16(tmem_d, ad + k * a_step, bd + k * b_step, idesc, 1u);
              mma2_commit_both(&empty[s]);
              if (++s == STAGES) { s = 0; ph ^= 1u; }
              ++kb;
            }
#pragma unroll 1
            for (; kb < end; ++kb) {
              if (!wait_or_abort(&full[s], ph, abort_flag, err, 2)) { ok = false; break; }
              tc_fence_after();
              const uint64_t ad = a0 + (uint64_t)(s * (STAGE2_BYTES >> 4)), bd = b0 + (uint64_t)(s * (STAGE2_BYTES >> 4));
              mma2_f16(tmem_d, ad, bd, idesc, acc);
              acc = 1u;
              mma2_f16(tmem_d, ad + a_step, bd + b_step, idesc, 1u);
              mma2_f16(tmem_d, ad + 2 * a_step, bd + 2 * b_step, idesc, 1u);
              mma2_f16(tmem_d, ad + 3 * a_step, bd + 3 * b_step, idesc, 1u);
              mma2_commit_both(&empty[s]);
              if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
          } else {
#pragma unroll 1
            for (; kb < end; ++kb) {
              if (!wait_or_abort(&full[s], ph, abort_flag, err, 2)) { ok = false; break; }
              tc_fence_after();
              const uint64_t ad = a0 + (uint64_t)(s * (STAGE2_BYTES >> 4)), bd = b0 + (uint64_t)(s * (STAGE2_BYTES >> 4));
              mma2_tf32(tmem_d, ad, bd, idesc, acc);
              acc = 1u;
              mma2_tf32(tmem_d, ad + a_step, bd + b_step, idesc, 1u);
              mma2_tf32(tmem_d, ad + 2 * a_step, bd + 2 * b_step, idesc, 1u);
              mma2_tf32(tmem_d, ad + 3 * a_step, bd + 3 * b_step, idesc, 1u);
              mma2_commit_both(&empty[s]);
              if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
          }
        }
        if (ok) mma2_commit_both(&acc_full[buf]);
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..17, both CTAs)
    // Fragment layout: see epilogue_pieces.
    const int quad = warp & 3;
    const int sub = (warp - 2) >> 2;             // of the quadrant's four warps: rows 16 (sub % 2) .., every other column chunk
    const int hh = sub & 1, half = sub >> 1;
    const int rsub = 16 * hh + (lane >> 2), csub = (lane & 3) * 2;
    int ti = 0;
    Work w;
    int amax_prob = -1;
    unsigned amax_seen = 0u;                     // largest magnitude this warp has reported of that problem's copy
    for (int wi = 0; next_work(gp, pair, wi, w); ++wi, ++ti) {
      const Tf32Params& p = gp.pr[w.prob];
      const int bn = p.bn;
      const int t = w.tile;
      const int m0 = (t / p.tiles_n) * (2 * BM) + (int)rank * BM, n0 = (t % p.tiles_n) * bn;
      const int buf = ti & 1;
      const uint32_t aph = (ti >> 1) & 1;
      int good = 1;
      if (lane == 0) good = wait_or_abort(&acc_full[buf], aph, abort_flag, err, 3) ? 1 : 0;
      good = __shfl_sync(0xffffffffu, good, 0);
      if (!good) break;
      tc_fence_after();
      // (the producer has left the tile's word before it asked for the first operands: this loop ends at once)
      int word = 0;
      if (HALF) {
        if (lane == 0) {
          const unsigned long long t0 = globaltimer();
          while (((word = tile_words[wi % TILE_WORDS]) >> 17) != ((wi + 1) & 0x3fff)) {
            if (*abort_flag || globaltimer() - t0 > WAIT_LIMIT_NS) { atomicCAS(err, 0, 7); *abort_flag = 1; word = 0; break; }
          }
        }
        word = __shfl_sync(0xffffffffu, word, 0);
        if (word == 0) break;
      }
      const float un = HALF && word & 1 ? half_scale((word >> 1 & 0xff) - 128) : 1.f;
      const int out_e = (word >> 9 & 0xff) - 128;
      const int n_chunks = min(bn / 32, (p.N - n0 + 31) / 32);   // column chunks of this tile that exist
      const uint32_t tq = tmem_base + ((uint32_t)(quad * 32 + 16 * hh) << 16) + (uint32_t)(buf * BN_MAX);
      int sl = 0, grp = 0;                                       // slice index and first pair of the tile's group
      const bool sliced = NP == 1 && w.sliced;
      if (sliced) {
        grp = (pair / p.slices) * p.slices;
        sl = pair - grp;
        // (a tile of few rows or columns is few warps' work, and the others take no part in the count)
        if (m0 + quad * 32 + 16 * hh >= p.M || half >= n_chunks) {
          if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(smem_u32(&acc_empty[buf]), 0));
          continue;
        }
        // 1. raw accumulator of this slice to the workspace slot of this pair
        float* wsw = p.sk_ws + (((long long)pair * 2 + rank) * BM + quad * 32 + rsub) * BN_MAX + csub;
        for (int c = half; c < n_chunks; c += 2) {
          float v[16];
          tmem_ld_16x256b_x4(tq + (uint32_t)(c * 32), v);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              __stcg(reinterpret_cast<float2*>(wsw + (long long)(8 * e) * BN_MAX + c * 32 + 8 * j),
                     make_float2(v[4 * j + 2 * e] * un, v[4 * j + 2 * e + 1] * un));
        }
        // the accumulator is free again; the tensor pipe has no further use for it in this pair
        tc_fence_before();
        __threadfence();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_cluster_relaxed(map_to_cta(smem_u32(&acc_empty[buf]), 0));
          int* flag_w = p.sk_flags + pair / p.slices;
          atomicAdd(flag_w, 1);
          // 2. wait until the warps of both CTAs of every slice of this tile have stored theirs (16 rows, every other chunk each)
          const volatile int* flag = flag_w;
          const int want = (min(2 * BM, p.M - (t / p.tiles_n) * (2 * BM)) + 15) / 16 * min(2, n_chunks) * p.slices;
          const unsigned long long t0 = globaltimer();
          while (*flag < want) {
            if (*abort_flag || globaltimer() - t0 > WAIT_LIMIT_NS) { atomicCAS(err, 0, 5); *abort_flag = 1; good = 0; break; }
            __nanosleep(200);   // up to thirty-two warps per pair poll the same word: keep them off the L2 while the pair's MMAs run
          }
          __threadfence();
          // 3. count out again: the last of the tile's warps to have seen the full count puts the flag back to
          // zero for the next launch (no memset between launches; the count only grows until then, so nobody
          // still waiting can miss it)
          if (good && atomicAdd(flag_w, 1) == 2 * want - 1) *reinterpret_cast<volatile int*>(flag_w) = 0;
        }
        good = __shfl_sync(0xffffffffu, good, 0);
        if (!good) break;
      }
      bool bad_out = false;
      {
        const int mq = m0 + quad * 32 + rsub;                    // this thread's rows are mq and mq + 8
        EpiArgs ea;
        const bool copy_out = HALF && p.copy_out;
        ea.un = sliced ? 1.f : un; ea.hsc = half_scale(out_e);
        HalfCheck check;
        const int n_opt = (p.sigmoid ? 1 : 0) + (p.dsig ? 1 : 0) + (p.cin ? 1 : 0);
        const int mode = n_opt == 0 ? 0 : n_opt > 1 ? 4 : p.sigmoid ? 1 : p.dsig ? 2 : 3;
        // whole tile: this warp's chunks are half, half + 2, ...; sliced tile: the pair's share of the
        // chunks is sl, sl + slices, ..., dealt alternately to the two warps of these rows
        const int c_first = sliced ? sl + half * p.slices : half;
        const int c_step = sliced ? 2 * p.slices : 2;
        const int n_slices = sliced ? p.slices : 0;
        const float* const ws0 = sliced ? p.sk_ws + (((long long)grp * 2 + rank) * BM + quad * 32 + rsub) * BN_MAX + csub : nullptr;
        // (options of one kind on 16-byte aligned rows; anything else element by element)
        const PieceRun run{tq, mq, n0 + csub, c_first, c_step, n_chunks, ws0, n_slices};
        if (!p.vec_epi || mode == 4) {
          check = epilogue_ragged<HALF>(p, ea, run);
        } else if (copy_out) {                                            // (only ever set with mode 1 or 2)
          if (mode == 1) epilogue_pieces<1, true>(p, ea, run, lane, check);
          else epilogue_pieces<2, true>(p, ea, run, lane, check);
        } else {
          switch (mode) {
            case 0: epilogue_pieces<0, false>(p, ea, run, lane, check); break;
            case 1: epilogue_pieces<1, false>(p, ea, run, lane, check); break;
            case 2: epilogue_pieces<2, false>(p, ea, run, lane, check); break;
            case 3: epilogue_pieces<3, false>(p, ea, run, lane, check); break;
            default: break;
          }
        }
        if (copy_out) {
          // this warp's word on the copy: the largest magnitude, and whether it may be used (the scale is said once)
          const unsigned high = __reduce_max_sync(0xffffffffu, check.high);
          bad_out = __any_sync(0xffffffffu, check.bad());
          if (w.prob != amax_prob) { amax_prob = w.prob; amax_seen = 0u; }
          if (lane == 0) {
            if (t == 0 && warp == 2 && rank == 0) {
              __stcg(&p.hout->e, out_e);
              if (p.sigmoid) __stcg(&p.hout->amax, __float_as_uint(1.f));
            }
            if (!p.sigmoid && high > amax_seen) atomicMax(&p.hout->amax, __float_as_uint(__uint_as_float(high) * half_scale(-out_e)));
            if (bad_out) atomicOr(&p.hout->bad, 1u);
          }
          amax_seen = max(amax_seen, high);
        }
      }
      if (!sliced) {       // (a sliced tile released its accumulator right after storing it)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(smem_u32(&acc_empty[buf]), 0));
      }
      if (NP > 1 && gp.signal[w.prob]) {
        // a later problem of this launch reads this tile: publish this warp's stores, then count the warp in
        __threadfence();
        asm volatile("fence.proxy.async.global;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          int* base = gp.done + (long long)w.prob * gp.done_stride;
          if (gp.signal[w.prob] & 1) { if (bad_out) atomicOr(base + t / p.tiles_n, (int)kBadPanel); atomicAdd(base + t / p.tiles_n, 1); }
          if (gp.signal[w.prob] & 2) { if (bad_out) atomicOr(base + gp.done_stride - 1, (int)kBadPanel); atomicAdd(base + gp.done_stride - 1, 1); }
        }
      }
    }
  }
  tc_fence_before();
  cluster_sync_all();      // neither CTA leaves (or frees tensor memory) while the other may still use it
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

// One CTA waits on an mbarrier that nothing ever arrives on, with the same bounded-wait code the GEMM
// roles use but a caller-chosen limit; it must record its code and return.  Exercises the path from a
// timed-out device wait to GN_ETIMEOUT on the host without hanging anything.
__global__ void timeout_probe_kernel(int* err, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const unsigned long long t0 = globaltimer();
    while (!mbar_test_wait(&bar, 0)) {
      if (globaltimer() - t0 > limit_ns) { atomicCAS(err, 0, 9); break; }
    }
  }
}

// ---- host side ---------------------------------------------------------------------------------
// 2-D map over a row-major [rows][cols] float matrix with leading dimension ld; box = (box_c, box_r).
bool make_map(CUtensorMap* m, const float* base, long long rows, long long cols, long long ld, int box_c, int box_r,
              CUtensorMapSwizzle swz) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
  cuuint32_t box[2] = {(cuuint32_t)box_c, (cuuint32_t)box_r};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_TFLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// The maps of FP16 copies: 2-D as above, box = 64 columns x box_r rows, and 3-D as below, chunks of 64 columns, BK_HALF rows.
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
bool make_half_map_mn3d(CUtensorMap* m, const void* base, long long K, long long MN, long long ld, int chunks) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {64, (cuuint64_t)K, (cuuint64_t)((MN + 63) / 64)};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, 128};
  cuuint32_t box[3] = {64, (cuuint32_t)BK_HALF, (cuuint32_t)chunks};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3-D view of a row-major [K][MN] matrix (MN contiguous): (32 inner columns, K rows, MN/32 column chunks).
// One box (32, BK, chunks) lands in shared memory as `chunks` consecutive [BK][32] blocks.  The last
// chunk of a row may extend past MN (into the next row, or up to 124 bytes past the last row), so the
// operand must be followed by that much readable memory.
bool make_map_mn3d(CUtensorMap* m, const float* base, long long K, long long MN, long long ld, int chunks) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {32, (cuuint64_t)K, (cuuint64_t)((MN + 31) / 32)};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 4, 128};
  cuuint32_t box[3] = {32, (cuuint32_t)BK, (cuuint32_t)chunks};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_TFLOAT32, 3, const_cast<float*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

constexpr int kStages = 4;
constexpr int kSmemBytes = kStages * (A_STAGE_BYTES + BN_MAX * BK * 4) + 1024 + 256;

// Tile width against wave quantisation: every CTA runs ceil(tiles / SMs) tiles.  Measured tile times
// on B200 fit (320 + bn) units: the operand pipeline is latency-bound, so a narrower tile is only
// slightly cheaper and the width that minimises the number of waves usually wins.
int choose_bn(int M, int N) {
  const long long tiles_m = (M + BM - 1) / BM;
  const int sms = num_sms();
  int best = 256;
  long long best_cost = -1;
  for (int bn = 256; bn >= 128; bn -= 32) {
    const long long tiles = tiles_m * ((N + bn - 1) / bn);
    const long long cost = ((tiles + sms - 1) / sms) * (320 + bn);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = bn; }
  }
  if (N <= 64) best = 64;
  if (N <= 32) best = 32;
  return best;
}

}  // namespace

int launch_timeout_probe(int* err_flag, unsigned long long limit_ns, cudaStream_t st) {
  timeout_probe_kernel<<<1, 32, 0, st>>>(err_flag, limit_ns);
  return 1;
}

bool gemm_tf32_eligible(const GemmArgs& g) {
  if (g.M < 1 || g.N < 1) return false;
  if (!aligned16(g.A1) || !aligned16(g.B1) || g.lda1 % 4 || g.ldb1 % 4) return false;
  if (g.A2 && (!aligned16(g.A2) || !aligned16(g.B2) || g.lda2 % 4 || g.ldb2 % 4)) return false;
  if (!encode_fn()) return false;
  return true;
}

constexpr int kStages2 = 6;
constexpr int kMaxSlices = 16;   // K slices per left-over tile
constexpr int kSmemBytes2 = kStages2 * STAGE2_BYTES + 1024 + 512;

// Two-CTA tile width (a multiple of 64 so that each CTA's half is whole 32-column chunks).  With the
// work split evenly over the pairs (stream-K) only the padding of N to whole tiles costs anything;
// without it the number of waves decides as well.
int choose_bn2(int M, int N, bool stream_k, int fixed_cost = 320) {
  const long long tiles_m = (M + 2 * BM - 1) / (2 * BM);
  const int pairs = num_sms() / 2;
  int best = 256;
  long long best_cost = -1;
  for (int bn = 256; bn >= 128; bn -= 64) {
    const long long tiles_n = (N + bn - 1) / bn;
    const long long tiles = tiles_m * tiles_n;
    const long long cost = (stream_k ? tiles_n : (tiles + pairs - 1) / pairs) * (fixed_cost + bn);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = bn; }
  }
  return best;
}

int64_t gemm_tf32_workspace_floats() { return (int64_t)(num_sms() / 2) * 2 * BM * BN_MAX; }
int gemm_tf32_workspace_flags() { return num_sms() / 2; }

namespace {

// Tensor maps and kernel parameters of one problem for a given tile width (two_cta: 256 x bn tiles of a CTA pair).
// maps: four, and four more of the copies if there are any.
bool setup_problem(const GemmArgs& g, bool two_cta, int bn, int* err_flag, CUtensorMap* maps, Tf32Params& p) {
  CUtensorMap* const half_maps = maps + 4;
  const int b_rows = two_cta ? bn / 2 : bn;      // B rows staged per CTA
  const float* As[2] = {g.A1, g.A2};
  const float* Bs[2] = {g.B1, g.B2};
  const int Ks[2] = {g.K1, g.A2 ? g.K2 : 0};
  const long long lda[2] = {g.lda1, g.lda2}, ldb[2] = {g.ldb1, g.ldb2};
  for (int s = 0; s < 2; ++s) {
    const int src = As[s] ? s : 0;  // unused second pair: repeat the first (never dereferenced)
    bool ok;
    const CUtensorMapSwizzle kmaj = CU_TENSOR_MAP_SWIZZLE_128B, mnmaj = CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B;
    if (g.a_kmajor)      ok = make_map(&maps[2 * s], As[src], g.M, Ks[src], lda[src], BK, BM, kmaj);
    else if (g.mn_padded) ok = make_map_mn3d(&maps[2 * s], As[src], Ks[src], g.M, lda[src], BM / 32);
    else                 ok = make_map(&maps[2 * s], As[src], Ks[src], g.M, lda[src], 32, BK, mnmaj);
    if (g.b_kmajor)      ok = ok && make_map(&maps[2 * s + 1], Bs[src], g.N, Ks[src], ldb[src], BK, b_rows, kmaj);
    else if (g.mn_padded) ok = ok && make_map_mn3d(&maps[2 * s + 1], Bs[src], Ks[src], g.N, ldb[src], b_rows / 32);
    else                 ok = ok && make_map(&maps[2 * s + 1], Bs[src], Ks[src], g.N, ldb[src], 32, BK, mnmaj);
    if (!ok) return false;
  }
  p = Tf32Params{};
  p.M = g.M; p.N = g.N;
  p.kblocks[0] = (Ks[0] + BK - 1) / BK;
  p.kblocks[1] = (Ks[1] + BK - 1) / BK;
  p.a_mn = g.a_kmajor ? 0 : 1; p.b_mn = g.b_kmajor ? 0 : 1;
  p.a_3d = (p.a_mn && g.mn_padded) ? 1 : 0; p.b_3d = (p.b_mn && g.mn_padded) ? 1 : 0;
  p.D = g.D; p.ldd = g.ldd;
  p.bias = g.bias; p.sigmoid = g.sigmoid;
  p.dsig = g.dsig; p.ld_dsig = g.ld_dsig; p.dsig_rows = g.dsig_rows > 0 ? g.dsig_rows : 1; p.dsig_div = g.dsig_div > 0 ? g.dsig_div : 1;
  p.alpha = g.alpha;
  p.cin = g.cin; p.ld_cin = g.ld_cin; p.beta = g.beta;
  p.vec_epi = g.N % 4 == 0 && aligned16(g.D) && (g.ldd % 4 == 0) && (!g.bias || aligned16(g.bias)) &&
              (!g.dsig || (aligned16(g.dsig) && g.ld_dsig % 4 == 0)) &&
              (!g.cin || (aligned16(g.cin) && g.ld_cin % 4 == 0));
  for (int s = 0; s < 2; ++s) p.K[s] = Ks[s];
  if (two_cta && (g.half || g.hout.p)) {
    for (int k = 0; k < (g.A2 ? 4 : 2); ++k) p.hin[k] = g.h[k].info;
    if (g.half) {
      for (int s = 0; s < (g.A2 ? 2 : 1); ++s) {
        const HalfMat& a = g.h[2 * s];
        const HalfMat& b = g.h[2 * s + 1];
        bool ok = g.a_kmajor ? make_half_map(&half_maps[2 * s], a.p, g.M, Ks[s], a.ld, BM)
                             : make_half_map_mn3d(&half_maps[2 * s], a.p, Ks[s], g.M, a.ld, BM / 64);
        if (g.b_kmajor) ok = ok && make_half_map(&half_maps[2 * s + 1], b.p, g.N, Ks[s], b.ld, b_rows);
        else if (b_rows % 64 == 0) ok = ok && make_half_map_mn3d(&half_maps[2 * s + 1], b.p, Ks[s], g.N, b.ld, b_rows / 64);
        else ok = ok && make_half_map(&half_maps[2 * s + 1], b.p, Ks[s], g.N, b.ld, BK_HALF);
        if (!ok) return false;
        p.khalf[s] = (Ks[s] + BK_HALF - 1) / BK_HALF;
      }
      p.half = 1;
    }
    if (g.hout.p) {
      p.Dh = static_cast<__half*>(g.hout.p); p.ldh = g.hout.ld; p.hout = g.hout.info; p.copy_out = 1;
      for (int k = 0; k < 3; ++k) p.hnext[k] = g.h_next[k];
    }
  }
  p.bn = bn;
  p.tiles_n = (g.N + bn - 1) / bn;
  p.tiles = ((g.M + (two_cta ? 2 : 1) * BM - 1) / ((two_cta ? 2 : 1) * BM)) * p.tiles_n;
  p.err = err_flag;
  p.slices = 1;
  return true;
}

void set_kernel_attributes() {
  static std::atomic<signed char> state[64];
  once_per_device(state, [] {
    return cudaFuncSetAttribute(gemm_tf32_kernel<kStages>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) == cudaSuccess &&
           cudaFuncSetAttribute(gemm_tf32_2cta_kernel<kStages2, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes2) == cudaSuccess &&
           cudaFuncSetAttribute(gemm_tf32_2cta_kernel<kStages2, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes2) == cudaSuccess &&
           cudaFuncSetAttribute(gemm_tf32_2cta_kernel<kStages2, MAX_GROUP, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes2) == cudaSuccess &&
           cudaFuncSetAttribute(gemm_tf32_2cta_kernel<kStages2, MAX_GROUP, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes2) == cudaSuccess;
  });
}

// One launch of the CTA-pair kernel; maps: eight per problem, the last four unused without copies.
template <int NP, bool HALF>
void launch_pair(const GroupParams<NP>& gp, const CUtensorMap (*maps)[8], int ctas, cudaStream_t st) {
  GroupMaps<NP, HALF> gm;
  for (int k = 0; k < gp.n_prob; ++k)
    for (int j = 0; j < (HALF ? 8 : 4); ++j) gm.m[k][j] = maps[k][j];
  launch_pdl(gemm_tf32_2cta_kernel<kStages2, NP, HALF>, ctas, PAIR_THREADS, kSmemBytes2, st, gm, gp);
}

inline bool suits_pair_kernel(const GemmArgs& g) { return g.M > BM && g.N >= 128; }

}  // namespace

namespace {
// k-blocks of a tile: 128 bytes of a row each, whatever the operands' type, and as long to multiply
int kblocks_of(const GemmArgs& g) {
  const int bk = g.half ? BK_HALF : BK;
  return (g.K1 + bk - 1) / bk + (g.A2 ? (g.K2 + bk - 1) / bk : 0);
}
// K slices for the tiles left over after the whole waves of a problem with `tiles` tiles of `total_kb` k-blocks on
// `pairs` CTA pairs (1 = whole tiles).  A sliced tile pays for a store and a re-read of its partial accumulators
// and for the wait between them, about as much as 25 to 30 k-blocks of main loop (measured: a 25-k-block tile is
// faster whole even when its wave is nearly empty, a 63-k-block tile gains from 2 slices on), so a tile is cut only
// if that saves more than this.
int choose_slices(int tiles, int total_kb, int pairs) {
  int rem = tiles % pairs;
  if (tiles < pairs) rem = tiles;
  if (rem == 0) return 1;
  int sl = pairs / rem;
  if (sl > kMaxSlices) sl = kMaxSlices;
  if (sl > total_kb) sl = total_kb;
  while (sl >= 2 && total_kb / sl < 4) --sl;
  if (sl < 2) return 1;
  return (double)total_kb * (1.0 - 1.0 / sl) >= 30.0 ? sl : 1;
}
}  // namespace

int launch_gemm_tf32(const GemmArgs& g, int* err_flag, float* sk_ws, int* sk_flags, cudaStream_t st) {
  set_kernel_attributes();
  const int pairs = num_sms() / 2;
  const int total_kb_all = kblocks_of(g);
  bool two_cta = g.two_cta >= 0 ? g.two_cta != 0 : suits_pair_kernel(g);
  if (!two_cta && g.two_cta < 0 && sk_ws && sk_flags) {
    // A result of at most 128 rows or fewer than 128 columns leaves part of a pair's tile empty, but the pair kernel can
    // cut a long K (the weight block of a narrow layer, or of an output layer wider than the streaming kernels take) where
    // the one-CTA kernel walks it alone on a few SMs, at about 0.5 us per k-block: 100 x 4096 x 32768 took 566 us there,
    // 64 x 64 x 60000 about 900.  A slice costs 0.45 us per k-block and 16 us on top.
    const int bn2 = choose_bn2(g.M, g.N, true);
    const int tiles = ((g.M + 2 * BM - 1) / (2 * BM)) * ((g.N + bn2 - 1) / bn2);
    const int sl = choose_slices(tiles, total_kb_all, pairs);
    two_cta = sl >= 2 && tiles <= pairs && 0.45 * total_kb_all / sl + 16.0 < 0.5 * total_kb_all;
  }
  bool stream_k = two_cta && sk_ws && sk_flags;
  int bn = two_cta ? choose_bn2(g.M, g.N, stream_k) : choose_bn(g.M, g.N);
  if (stream_k) {
    // the width chosen for an even split of the work only stands if the left-over tiles will in fact be cut
    const int tiles = ((g.M + 2 * BM - 1) / (2 * BM)) * ((g.N + bn - 1) / bn);
    if (choose_slices(tiles, total_kb_all, pairs) < 2) { stream_k = false; bn = choose_bn2(g.M, g.N, false); }
  }
  if (two_cta) {
    CUtensorMap maps[1][8];
    GroupParams<1> gp = {};                    // (no dependencies, no signals)
    gp.n_prob = 1;
    Tf32Params& p = gp.pr[0];
    if (!setup_problem(g, true, bn, err_flag, maps[0], p)) return -1;
    const int total_kb = total_kb_all;
    p.sk_ws = sk_ws; p.sk_flags = sk_flags;
    p.P = p.tiles < pairs ? p.tiles : pairs;
    p.waves = p.tiles / p.P;
    p.rem = p.tiles - p.waves * p.P;
    int launch_pairs = p.P;
    if (stream_k) {
      const int sl = choose_slices(p.tiles, total_kb, pairs);
      if (sl >= 2) {
        if (p.tiles < pairs) { p.P = pairs; p.waves = 0; p.rem = p.tiles; }   // no full wave: every tile is cut
        p.slices = sl;
        if (p.waves == 0) launch_pairs = p.rem * p.slices;
      }
    }
    for (int q = 0; q <= MAX_PAIRS_LAUNCH; ++q) gp.rstart[0][q] = (unsigned short)(q < p.rem ? q : p.rem);
    if (p.half || p.copy_out) launch_pair<1, true>(gp, maps, 2 * launch_pairs, st);
    else launch_pair<1, false>(gp, maps, 2 * launch_pairs, st);
  } else {
    CUtensorMap maps[4];
    Tf32Params p;
    if (!setup_problem(g, false, bn, err_flag, maps, p)) return -1;
    const int grid = p.tiles < num_sms() ? p.tiles : num_sms();
    launch_pdl(gemm_tf32_kernel<kStages>, grid, 320, kSmemBytes, st, maps[0], maps[1], maps[2], maps[3], p);
  }
  return 1;
}

bool gemm_tf32_group_eligible(const GemmArgs* gs, int n) {
  if (n < 1 || n > MAX_GROUP || num_sms() / 2 > MAX_PAIRS_LAUNCH) return false;
  for (int i = 0; i < n; ++i)
    if (!gemm_tf32_eligible(gs[i]) || !suits_pair_kernel(gs[i]) || gs[i].two_cta == 0) return false;
  return true;
}

namespace {

// Tiles of problem slot k of a group (cost `cost` each) dealt to the P pairs on top of the loads they carry
// already: as many whole waves (tiles q, q + P, ... for every pair q) as every pair takes anyway, the rest as
// contiguous runs of the left-over tiles, so that the loads come out as even as whole tiles allow.
void deal_tiles(GroupParams<MAX_GROUP>& gp, int k, double cost, int P, double* load) {
  Tf32Params& p = gp.pr[k];
  p.P = P;
  int cnt[MAX_PAIRS_LAUNCH];
  // lowest level L with sum_q floor((L - load_q) / cost) >= tiles, by bisection on L
  double lo = 0.0, hi = 0.0;
  for (int q = 0; q < P; ++q) if (load[q] > hi) hi = load[q];
  hi += cost * (p.tiles / P + 2);
  for (int iter = 0; iter < 60; ++iter) {
    const double mid = 0.5 * (lo + hi);
    long long have = 0;
    for (int q = 0; q < P; ++q) if (mid > load[q]) have += (long long)((mid - load[q]) / cost);
    if (have >= p.tiles) hi = mid; else lo = mid;
  }
  long long have = 0;
  for (int q = 0; q < P; ++q) { cnt[q] = hi > load[q] ? (int)((hi - load[q]) / cost) : 0; have += cnt[q]; }
  // more than needed (several pairs cross a multiple of `cost` at the same level): take back from the fullest
  while (have > p.tiles) {
    int worst = -1;
    for (int q = 0; q < P; ++q)
      if (cnt[q] > 0 && (worst < 0 || load[q] + cnt[q] * cost > load[worst] + cnt[worst] * cost)) worst = q;
    --cnt[worst]; --have;
  }
  while (have < p.tiles) {                    // (rounding in the bisection)
    int best = 0;
    for (int q = 1; q < P; ++q)
      if (load[q] + cnt[q] * cost < load[best] + cnt[best] * cost) best = q;
    ++cnt[best]; ++have;
  }
  int waves = cnt[0];
  for (int q = 1; q < P; ++q) if (cnt[q] < waves) waves = cnt[q];
  p.waves = waves;
  p.rem = p.tiles - waves * P;
  int run = 0;
  for (int q = 0; q < P; ++q) { gp.rstart[k][q] = (unsigned short)run; run += cnt[q] - waves; load[q] += cnt[q] * cost; }
  for (int q = P; q <= MAX_PAIRS_LAUNCH; ++q) gp.rstart[k][q] = (unsigned short)run;
}

// time of one tile in k-blocks of a 256-wide tile: operand bytes per k-block (the feed bounds the main loop) plus a fixed part
double tile_cost(const Tf32Params& p) {
  return (p.half ? p.khalf[0] + p.khalf[1] : p.kblocks[0] + p.kblocks[1]) * (256.0 + p.bn) / 512.0 + 8.0;
}

}  // namespace

// Several problems in one launch of the CTA-pair kernel.
//   Independent problems (dep_prob == nullptr): taken longest tile first, the pairs' loads evened out on the host,
//   so the short tiles of one problem fill the partial last wave of another.
//   A chain (dep_prob[i] = index of the earlier problem whose output problem i reads, or -1; dep_all[i] != 0 if it
//   needs all of that output rather than the 256-row panel of its own tile): kept in the given order, every pair
//   works through the problems one after the other, and the head of a problem overlaps the tail of the one before.
//   `done` is a zeroed-by-this-call array of n * done_stride ints, done_stride > the number of 256-row panels.
int launch_gemm_tf32_group(const GemmArgs* gs, int n, const int* dep_prob, const int* dep_all, int* done,
                           int done_stride, int* err_flag, cudaStream_t st) {
  if (!gemm_tf32_group_eligible(gs, n)) return -1;
  set_kernel_attributes();
  CUtensorMap maps[MAX_GROUP][8];
  GroupParams<MAX_GROUP> gp = {};
  const int pairs = num_sms() / 2;
  struct Item { int src; double cost; };
  Item order[MAX_GROUP];
  Tf32Params tmp[MAX_GROUP];
  CUtensorMap tmaps[MAX_GROUP][8];
  long long total_tiles = 0;
  bool half = false;
  for (int i = 0; i < n; ++i) {
    const int bn = choose_bn2(gs[i].M, gs[i].N, true);
    if (!setup_problem(gs[i], true, bn, err_flag, tmaps[i], tmp[i])) return -1;
    half = half || tmp[i].half || tmp[i].copy_out;
    if (tmp[i].tiles > 60000) return -1;       // (left-over tile indices are 16-bit)
    order[i].src = i;
    order[i].cost = tile_cost(tmp[i]);
    total_tiles += tmp[i].tiles;
  }
  const bool chain = dep_prob != nullptr;
  if (chain) {
    if (!done) return -1;
    for (int i = 0; i < n; ++i) {
      if (dep_prob[i] >= i) return -1;
      if (dep_prob[i] >= 0 && !dep_all[i] && gs[dep_prob[i]].M != gs[i].M) return -1;   // panels must coincide
      if ((gs[i].M + 2 * BM - 1) / (2 * BM) + 1 > done_stride) return -1;
    }
  } else {
    for (int i = 1; i < n; ++i)                 // insertion sort, longest tile first (stable)
      for (int j = i; j > 0 && order[j].cost > order[j - 1].cost; --j) { Item t = order[j]; order[j] = order[j - 1]; order[j - 1] = t; }
  }
  const int P = total_tiles < pairs ? (int)total_tiles : pairs;
  double load[MAX_PAIRS_LAUNCH];
  for (int q = 0; q < P; ++q) load[q] = 0.0;
  gp.n_prob = n;
  gp.done = done; gp.done_stride = done_stride;
  for (int k = 0; k < MAX_GROUP; ++k) { gp.dep_prob[k] = -1; gp.dep_all[k] = 0; gp.signal[k] = 0; }
  for (int k = 0; k < n; ++k) {
    const int i = order[k].src;
    gp.pr[k] = tmp[i];
    for (int j = 0; j < (half ? 8 : 4); ++j) maps[k][j] = tmaps[i][j];
    deal_tiles(gp, k, order[k].cost, P, load);
    if (chain && dep_prob[i] >= 0) {            // (a chain keeps its order: slot == index)
      gp.dep_prob[k] = dep_prob[i];
      gp.dep_all[k] = dep_all[i] ? 1 : 0;
      gp.signal[dep_prob[i]] |= dep_all[i] ? 2 : 1;
    }
  }
  if (chain && cudaMemsetAsync(done, 0, sizeof(int) * (size_t)n * done_stride, st) != cudaSuccess) return -1;
  if (half) launch_pair<MAX_GROUP, true>(gp, maps, 2 * P, st);
  else launch_pair<MAX_GROUP, false>(gp, maps, 2 * P, st);
  return 1;
}

// Host-only view of the work list a grouped launch would use (no device needed): for problems of the given shapes
// on `pairs` CTA pairs, counts[k * pairs + q] = tiles of the k-th problem IN LAUNCH ORDER that pair q runs,
// waves[k] = how many of them are whole waves (tiles q, q + pairs, ...), order[k] = index of that problem in the
// caller's list, tiles[k] = its tile count.  keep_order != 0 keeps the caller's order (a chain).  Returns the number
// of pairs the launch would use, or -1 for bad arguments.
namespace {
int plan_group_impl(int n, const int* M, const int* N, const int* K, int pairs, int keep_order, int* counts,
                    int* waves, int* order_out, int* tiles_out, double* makespan) {
  if (n < 1 || n > MAX_GROUP || pairs < 1 || pairs > MAX_PAIRS_LAUNCH) return -1;
  GroupParams<MAX_GROUP> gp = {};
  struct Item { int src; double cost; };
  Item order[MAX_GROUP];
  Tf32Params tmp[MAX_GROUP];
  long long total_tiles = 0;
  for (int i = 0; i < n; ++i) {
    if (M[i] < 1 || N[i] < 1 || K[i] < 1) return -1;
    const int bn = choose_bn2(M[i], N[i], true);
    tmp[i] = Tf32Params{};
    tmp[i].bn = bn;
    tmp[i].kblocks[0] = (K[i] + BK - 1) / BK;
    tmp[i].tiles_n = (N[i] + bn - 1) / bn;
    tmp[i].tiles = ((M[i] + 2 * BM - 1) / (2 * BM)) * tmp[i].tiles_n;
    order[i].src = i;
    order[i].cost = tile_cost(tmp[i]);
    total_tiles += tmp[i].tiles;
  }
  if (!keep_order)
    for (int i = 1; i < n; ++i)
      for (int j = i; j > 0 && order[j].cost > order[j - 1].cost; --j) { Item t = order[j]; order[j] = order[j - 1]; order[j - 1] = t; }
  const int P = total_tiles < pairs ? (int)total_tiles : pairs;
  double load[MAX_PAIRS_LAUNCH];
  for (int q = 0; q < P; ++q) load[q] = 0.0;
  for (int k = 0; k < n; ++k) {
    gp.pr[k] = tmp[order[k].src];
    deal_tiles(gp, k, order[k].cost, P, load);
    if (waves) waves[k] = gp.pr[k].waves;
    if (order_out) order_out[k] = order[k].src;
    if (tiles_out) tiles_out[k] = gp.pr[k].tiles;
    if (counts)
      for (int q = 0; q < pairs; ++q)
        counts[k * pairs + q] = q < P ? gp.pr[k].waves + (gp.rstart[k][q + 1] - gp.rstart[k][q]) : 0;
  }
  if (makespan) {
    *makespan = 0.0;
    for (int q = 0; q < P; ++q) if (load[q] > *makespan) *makespan = load[q];
  }
  return P;
}
}  // namespace

int gemm_tf32_plan_group(int n, const int* M, const int* N, const int* K, int pairs, int keep_order, int* counts,
                         int* waves, int* order_out, int* tiles_out) {
  return plan_group_impl(n, M, N, K, pairs, keep_order, counts, waves, order_out, tiles_out, nullptr);
}

// Load of the fullest CTA pair, in k-blocks of a 256-wide tile, if the problems went out as one grouped
// (keep_order == 0) or chained launch on this device; negative for bad arguments.  Host arithmetic only.
double gemm_tf32_group_makespan(int n, const int* M, const int* N, const int* K, int keep_order) {
  double ms = 0.0;
  if (plan_group_impl(n, M, N, K, num_sms() / 2, keep_order, nullptr, nullptr, nullptr, nullptr, &ms) < 0) return -1.0;
  return ms;
}

}  // namespace gn
