// Whole passes of small networks in one launch: a block takes 32 rows through all layers with the weights in shared
// memory, so a product or a gradient is two launches (pass, sum over the blocks) instead of fifteen to thirty.
//
// Such networks are bound by launches and latency: at 20-16-16-4 with 64 rows the chain of contraction, column-sum and
// streaming kernels takes 52 us for 0.5 MFLOP, nearly all of it launch overhead, and the 128 x 128 tiles of the FMA GEMM
// are mostly padding.  Used where theta (and v) and the rows' activations fit into one block's shared memory and the
// arithmetic is small enough not to need the tensor cores (small_net_fits).  FP32 arithmetic throughout; the blocks'
// weight and bias sums are added in block order, in double.
//
// Activations are kept transposed, [neuron][row] with 36 floats per neuron: a thread owns one neuron and four rows, reads
// the rows as one 16-byte access and the weight as a broadcast (forward, backward), and the sums over rows read 16
// bytes of both operands (36 = 4 mod 32 keeps eight neighbouring neurons on different banks).
#include "gn_kernels.h"
#include "tc_common.cuh"

namespace gn {
namespace {

constexpr int SN_ROWS = 32, SN_LD = 36, SN_THREADS = 256;
constexpr size_t SN_SMEM_MAX = 232448 - 1024;    // (the reductions' static arrays come on top)

enum { SN_GV = 0, SN_BLOCK = 1, SN_GRAD = 2, SN_FUN = 3, SN_FORWARD = 4 };

__host__ __device__ constexpr bool sn_has_v(int kind) { return kind == SN_GV || kind == SN_BLOCK; }

// Shared-memory floats: W of every layer (rows padded to an odd length) and b, the same of v, z^0 .. z^{L-1}, two buffers
// of the widest layer.
size_t sn_smem_floats(const SmallNet& a, int kind) {
  size_t wts = 0, z = 0, widest = 0;
  for (int m = 1; m <= a.L; ++m) {
    wts += (size_t)a.w[m] * (a.w[m - 1] | 1) + a.w[m];
    if ((size_t)a.w[m] > widest) widest = a.w[m];
  }
  wts = (wts + 3) / 4 * 4;
  for (int m = 0; m < a.L; ++m) z += a.w[m];
  return wts * (sn_has_v(kind) ? 2 : 1) + (z + 2 * widest) * SN_LD;
}

__device__ __forceinline__ float4 fma4(float a, float4 x, float4 c) {
  return make_float4(fmaf(a, x.x, c.x), fmaf(a, x.y, c.y), fmaf(a, x.z, c.z), fmaf(a, x.w, c.w));
}
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ float dsig(float z) { return z * (1.f - z); }
__device__ __forceinline__ float4 mul_dsig(float4 x, float4 z) {
  return make_float4(x.x * dsig(z.x), x.y * dsig(z.y), x.z * dsig(z.z), x.w * dsig(z.w));
}

// sum_k x[k][rows] W[j][k] for neuron j and four rows
__device__ __forceinline__ float4 dot_rows(const float* W, const float* xt, int n_in, int g, float4 acc) {
#pragma unroll 4
  for (int k = 0; k < n_in; ++k) acc = fma4(W[k], ld4(xt + k * SN_LD + 4 * g), acc);
  return acc;
}

// delta^{m-1} = (delta^m W^{mT}) * sigma'(z^{m-1}) (Eqs. communi-g, ztox-g)
__device__ __forceinline__ void back_layer(const float* W, int ldw, int n_m, int n_prev, const float* dt, const float* zt, float* out) {
  for (int i = threadIdx.x; i < n_prev * 8; i += SN_THREADS) {
    const int k = i >> 3, g = i & 7;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int j = 0; j < n_m; ++j) acc = fma4(W[j * ldw + k], ld4(dt + j * SN_LD + 4 * g), acc);
    st4(out + k * SN_LD + 4 * g, mul_dsig(acc, ld4(zt + k * SN_LD + 4 * g)));
  }
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float c) { return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, c)))); }

// This block's rows' share of delta^T z (two neurons of each side per thread) and 1^T delta (Eqs. xtow-g, xtow-g-bias)
__device__ __forceinline__ void weight_sums(const float* dt, const float* zt, int n_m, int n_prev, float* pw, float* pb) {
  const int hk = (n_prev + 1) / 2, hj = (n_m + 1) / 2;
  for (int i = threadIdx.x; i < hj * hk; i += SN_THREADS) {
    const int j0 = i / hk, k0 = i - j0 * hk, j1 = j0 + hj < n_m ? j0 + hj : j0, k1 = k0 + hk < n_prev ? k0 + hk : k0;
    float s00 = 0.f, s01 = 0.f, s10 = 0.f, s11 = 0.f;
#pragma unroll
    for (int r = 0; r < SN_ROWS; r += 4) {
      const float4 d0 = ld4(dt + j0 * SN_LD + r), d1 = ld4(dt + j1 * SN_LD + r), z0 = ld4(zt + k0 * SN_LD + r), z1 = ld4(zt + k1 * SN_LD + r);
      s00 = dot4(d0, z0, s00); s01 = dot4(d0, z1, s01); s10 = dot4(d1, z0, s10); s11 = dot4(d1, z1, s11);
    }
    pw[(long long)j0 * n_prev + k0] = s00;
    if (k1 != k0) pw[(long long)j0 * n_prev + k1] = s01;
    if (j1 != j0) pw[(long long)j1 * n_prev + k0] = s10;
    if (j1 != j0 && k1 != k0) pw[(long long)j1 * n_prev + k1] = s11;
  }
  for (int j = threadIdx.x; j < n_m; j += SN_THREADS) {
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < SN_ROWS; r += 4) { const float4 d = ld4(dt + j * SN_LD + r); s += (d.x + d.y) + (d.z + d.w); }
    pb[j] = s;
  }
}

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[SN_THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int i = 0; i < SN_THREADS / 32; ++i) t += sh[i];
  return t;
}

template <int KIND>
__global__ void __launch_bounds__(SN_THREADS) small_net_kernel(const __grid_constant__ SmallNet a) {
  extern __shared__ __align__(16) float sm[];
  grid_dep_wait();
  grid_dep_launch();
  const float* const theta = dep(a.theta);
  const float* const v = dep(a.v);
  const float* const Y = dep(a.Y);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int L = a.L;
  const long long row0 = (long long)blockIdx.x * SN_ROWS;
  const int cnt = (int)min((long long)SN_ROWS, a.rows - row0);
  // ---- layout: W and b of theta, of v, z^0 .. z^{L-1}, two buffers
  int wo[kSmallLayers + 1], zo[kSmallLayers + 1], wts = 0, zt_total = 0, widest = 0;
#pragma unroll
  for (int m = 1; m <= kSmallLayers; ++m)
    if (m <= L) { wo[m] = wts; wts += a.w[m] * (a.w[m - 1] | 1) + a.w[m]; widest = max(widest, a.w[m]); }
  wts = (wts + 3) / 4 * 4;
#pragma unroll
  for (int m = 0; m < kSmallLayers; ++m)
    if (m < L) { zo[m] = zt_total; zt_total += a.w[m] * SN_LD; }
  float* const ws = sm;
  float* const vs = sm + wts;
  float* const zs = sm + wts * (sn_has_v(KIND) ? 2 : 1);
  float* cur = zs + zt_total;
  float* nxt = cur + widest * SN_LD;
  // ---- weights in, rows in
  double tt = 0.0;
#pragma unroll
  for (int m = 1; m <= kSmallLayers; ++m)
    if (m <= L) {
      const int np = a.w[m - 1], ldw = np | 1;
      for (int j = warp; j < a.w[m]; j += SN_THREADS / 32)
        for (int k = lane; k < np; k += 32) {
          const float t = __ldg(theta + a.w_off[m] + j * np + k);
          ws[wo[m] + j * ldw + k] = t;
          if (KIND == SN_GRAD || KIND == SN_FUN) tt += (double)t * t;
          if (sn_has_v(KIND)) vs[wo[m] + j * ldw + k] = __ldg(v + a.w_off[m] + j * np + k);
        }
      for (int j = tid; j < a.w[m]; j += SN_THREADS) {
        const float t = __ldg(theta + a.b_off[m] + j);
        ws[wo[m] + a.w[m] * ldw + j] = t;
        if (KIND == SN_GRAD || KIND == SN_FUN) tt += (double)t * t;
        if (sn_has_v(KIND)) vs[wo[m] + a.w[m] * ldw + j] = __ldg(v + a.b_off[m] + j);
      }
    }
  if ((KIND == SN_GRAD || KIND == SN_FUN) && blockIdx.x == 0) {
    tt = block_sum(tt);
    if (tid == 0) *a.theta_sq = tt;
  }
#pragma unroll
  for (int m = 0; m < (sn_has_v(KIND) ? kSmallLayers : 1); ++m)
    if (m < L) {
      const float* const zm = dep(a.z[m]);
      for (int r = warp; r < SN_ROWS; r += SN_THREADS / 32) {
        const float* src = zm;
        bool ok = r < cnt;
        if (KIND == SN_FORWARD && ok) {
          const long long s = a.idx[row0 + r];
          ok = s >= 0 && s < a.x_rows;
          if (!ok && lane == 0) atomicExch(a.err_flag, 1);
          src += (ok ? s : 0) * a.w[0];
        } else {
          src += (row0 + (ok ? r : 0)) * a.w[m];
        }
        for (int k = lane; k < a.w[m]; k += 32) {
          const float x = ok ? __ldg(src + k) : 0.f;
          zs[zo[m] + k * SN_LD + r] = x;
          if (KIND == SN_FORWARD && r < cnt) a.z_out[0][(row0 + r) * a.w[0] + k] = x;
        }
      }
    }
  __syncthreads();

  if (KIND == SN_GRAD || KIND == SN_FUN || KIND == SN_FORWARD) {
    // ---- forward pass (Eq. xtoz)
#pragma unroll
    for (int m = 1; m <= kSmallLayers; ++m)
      if (m <= L) {
        const int np = a.w[m - 1], ldw = np | 1, n = a.w[m];
        float* const out = m < L ? zs + zo[m < kSmallLayers ? m : 0] : cur;
        for (int i = tid; i < n * 8; i += SN_THREADS) {
          const int j = i >> 3, g = i & 7;
          const float b = ws[wo[m] + n * ldw + j];
          float4 s = dot_rows(ws + wo[m] + j * ldw, zs + zo[m - 1], np, g, make_float4(b, b, b, b));
          if (m < L) s = make_float4(sigmoid_from(expf(-s.x)), sigmoid_from(expf(-s.y)), sigmoid_from(expf(-s.z)), sigmoid_from(expf(-s.w)));
          st4(out + j * SN_LD + 4 * g, s);
        }
        __syncthreads();
        if (KIND == SN_FORWARD)
          for (int r = warp; r < cnt; r += SN_THREADS / 32)
            for (int j = lane; j < n; j += 32) a.z_out[m][(row0 + r) * n + j] = out[j * SN_LD + r];
      }
    if (KIND == SN_FORWARD) return;
    // ---- squared loss and its derivative
    double loss = 0.0;
    for (int r = warp; r < SN_ROWS; r += SN_THREADS / 32)
      for (int j = lane; j < a.w[L]; j += 32) {
        float d = 0.f;
        if (r < cnt) {
          d = cur[j * SN_LD + r] - __ldg(Y + (row0 + r) * a.w[L] + j);
          loss += (double)d * d;
        }
        cur[j * SN_LD + r] = 2.f * d;
      }
    loss = block_sum(loss);            // (ends with every thread past its part of `cur`)
    if (tid == 0) a.loss[blockIdx.x] = loss;
    if (KIND == SN_FUN) return;
    __syncthreads();
  }
  float* const part = a.scratch + (long long)blockIdx.x * a.n;

  if (KIND == SN_GV) {
    // ---- forward directional derivative, both operand pairs of a layer in one sum
#pragma unroll
    for (int m = 1; m <= kSmallLayers; ++m)
      if (m <= L) {
        const int np = a.w[m - 1], ldw = np | 1, n = a.w[m];
        for (int i = tid; i < n * 8; i += SN_THREADS) {
          const int j = i >> 3, g = i & 7;
          const float c = vs[wo[m] + n * ldw + j];
          float4 s = dot_rows(vs + wo[m] + j * ldw, zs + zo[m - 1], np, g, make_float4(c, c, c, c));
          if (m > 1) s = dot_rows(ws + wo[m] + j * ldw, cur, np, g, s);
          if (m < L) {
            s = mul_dsig(s, ld4(zs + zo[m < kSmallLayers ? m : 0] + j * SN_LD + 4 * g));
          } else {                     // B = 2I; rows past the end count for nothing
            s.x = 4 * g + 0 < cnt ? 2.f * s.x : 0.f; s.y = 4 * g + 1 < cnt ? 2.f * s.y : 0.f;
            s.z = 4 * g + 2 < cnt ? 2.f * s.z : 0.f; s.w = 4 * g + 3 < cnt ? 2.f * s.w : 0.f;
          }
          st4(nxt + j * SN_LD + 4 * g, s);
        }
        __syncthreads();
        float* const t = cur; cur = nxt; nxt = t;
      }
  }
  if (KIND == SN_GV || KIND == SN_GRAD) {
    // ---- backward pass
#pragma unroll
    for (int m = kSmallLayers; m >= 1; --m)
      if (m <= L) {
        const int np = a.w[m - 1], ldw = np | 1, n = a.w[m];
        weight_sums(cur, zs + zo[m - 1], n, np, part + a.w_off[m], part + a.b_off[m]);
        if (m > 1) back_layer(ws + wo[m], ldw, n, np, cur, zs + zo[m - 1], nxt);
        __syncthreads();
        float* const t = cur; cur = nxt; nxt = t;
      }
  }
  if (KIND == SN_BLOCK) {
    // ---- one stream per layer: the layer's own perturbation to the output and back to that layer (Eq. approx-jaco)
    for (int s = 1; s <= L; ++s) {
#pragma unroll
      for (int m = 1; m <= kSmallLayers; ++m)
        if (m >= s && m <= L) {
          const int np = a.w[m - 1], ldw = np | 1, n = a.w[m];
          for (int i = tid; i < n * 8; i += SN_THREADS) {
            const int j = i >> 3, g = i & 7;
            float4 x;
            if (m == s) {
              const float c = vs[wo[m] + n * ldw + j];
              x = dot_rows(vs + wo[m] + j * ldw, zs + zo[m - 1], np, g, make_float4(c, c, c, c));
            } else {
              x = dot_rows(ws + wo[m] + j * ldw, cur, np, g, make_float4(0.f, 0.f, 0.f, 0.f));
            }
            if (m < L) {
              x = mul_dsig(x, ld4(zs + zo[m < kSmallLayers ? m : 0] + j * SN_LD + 4 * g));
            } else {
              x.x = 4 * g + 0 < cnt ? 2.f * x.x : 0.f; x.y = 4 * g + 1 < cnt ? 2.f * x.y : 0.f;
              x.z = 4 * g + 2 < cnt ? 2.f * x.z : 0.f; x.w = 4 * g + 3 < cnt ? 2.f * x.w : 0.f;
            }
            st4(nxt + j * SN_LD + 4 * g, x);
          }
          __syncthreads();
          float* const t = cur; cur = nxt; nxt = t;
        }
#pragma unroll
      for (int m = kSmallLayers; m >= 1; --m)
        if (m >= s && m <= L) {
          const int np = a.w[m - 1], ldw = np | 1, n = a.w[m];
          if (m == s) {
            weight_sums(cur, zs + zo[m - 1], n, np, part + a.w_off[m], part + a.b_off[m]);
          } else {
            back_layer(ws + wo[m], ldw, n, np, cur, zs + zo[m - 1], nxt);
            __syncthreads();
            float* const t = cur; cur = nxt; nxt = t;
          }
        }
      __syncthreads();
    }
  }
}

// out = alpha * (sum of the blocks' sums, in block order) + beta * cin, and the loss.  A block takes 32 coordinates (lane);
// warp w adds blocks w, w + 8, ... and the eight sums are added in warp order, all in double.
__global__ void __launch_bounds__(256) small_sum_kernel(const float* __restrict__ part, int blocks, int n, float alpha, const float* cin,
                                                        float beta, float* out, const double* __restrict__ loss, double* loss_out) {
  __shared__ double sh[8][33];
  grid_dep_wait();
  grid_dep_launch();
  part = dep(part); loss = dep(loss);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (out) {
    const int i = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (i < n) {
#pragma unroll 4
      for (int b = w; b < blocks; b += 8) s += (double)__ldg(part + (long long)b * n + i);
    }
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0 && i < n) {
      double t = sh[0][lane];
#pragma unroll
      for (int k = 1; k < 8; ++k) t += sh[k][lane];
      out[i] = fmaf(beta, cin[i], alpha * (float)t);
    }
  }
  if (loss_out && blockIdx.x == 0) {
    __syncthreads();
    double s = 0.0;
    for (int b = threadIdx.x; b < blocks; b += 256) s += loss[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sh[0][w] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int k = 0; k < 8; ++k) t += sh[0][k];
      *loss_out = t;
    }
  }
}

typedef void (*SmallKernel)(const SmallNet);
SmallKernel const kSmall[5] = {small_net_kernel<0>, small_net_kernel<1>, small_net_kernel<2>, small_net_kernel<3>, small_net_kernel<4>};

bool small_usable() {
  static std::atomic<signed char> state[64];
  return once_per_device(state, [] {
    bool ok = true;
    for (SmallKernel k : kSmall) ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SN_SMEM_MAX) == cudaSuccess;
    return ok;
  });
}

}  // namespace

int64_t small_net_blocks(int64_t rows) { return (rows + SN_ROWS - 1) / SN_ROWS; }

// The pass fits if its weights and 32 rows of activations do (227 KB), the blocks' sums take at most 32 MB, and the
// estimated time stays below what the chain of kernels needs to be launched and to move the rows' activations.  Measured
// (product, this way / the chain): 37-53-19-7 with 5000 rows 32 / 135 us, 60000 rows 159 / 318; 64-64-64-10 with 5000 rows
// 69 / 101, 20000 rows 170 / 159; 100-100-10 with 1000 rows 41 / 52, 5000 rows 80 / 60; 784-16-10 with 1000 rows 38 / 59, 5000
// rows 74 / 72.
bool small_net_fits(const SmallNet& a, int kind) {
  if (a.L < 1 || a.L > kSmallLayers || !small_usable()) return false;
  const size_t smem = sn_smem_floats(a, kind) * sizeof(float);
  if (smem > SN_SMEM_MAX) return false;
  const int64_t blocks = small_net_blocks(a.rows);
  if (blocks * a.n > 8 * 1000 * 1000) return false;
  double macs = 0.0, own = 0.0;
  for (int m = 1; m <= a.L; ++m) { own = (double)a.w[m - 1] * a.w[m]; macs += own; }
  macs *= kind == SN_GV ? 4.0 : kind == SN_BLOCK ? 1.0 + a.L : kind == SN_GRAD ? 3.0 : 1.0;
  int per_sm = (int)(SN_SMEM_MAX / (smem + 1024));
  if (per_sm > 4) per_sm = 4;
  if (per_sm > (blocks + 147) / 148) per_sm = (int)((blocks + 147) / 148);
  if (per_sm < 1) per_sm = 1;
  const double rounds = (double)((blocks + 148 * per_sm - 1) / (148 * per_sm));
  const double block_us = 3.0 + smem / 1.0e5 + 32.0 * macs * per_sm / 60.0e3;
  double width = 0.0;
  for (int m = 1; m <= a.L; ++m) width += a.w[m];
  return rounds * block_us <= kSmallUs + kSmallUsPerElement * width * (double)a.rows;
}

int launch_small_net(const SmallNet& a, int kind, float alpha, const float* cin, float beta, float* out, double* loss_out, cudaStream_t st) {
  const int blocks = (int)small_net_blocks(a.rows);
  if (launch_pdl(kSmall[kind], blocks, SN_THREADS, (int)(sn_smem_floats(a, kind) * sizeof(float)), st, a) != cudaSuccess) return -1;
  if (kind == SN_FORWARD) return 1;
  const int grid = out ? (a.n + 31) / 32 : 1;
  if (launch_pdl(small_sum_kernel, grid, 256, 0, st, (const float*)a.scratch, blocks, a.n, alpha, cin, beta, out, (const double*)a.loss, loss_out) != cudaSuccess)
    return -1;
  return 2;
}

}  // namespace gn
