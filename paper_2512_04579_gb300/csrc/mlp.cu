// mlp.cu -- the learned warm start: a small MLP that maps an initial state to
// a nominal control sequence mu (U_0 of Algorithm 1) and one log sampling
// scale per control step (Sigma_0), trained on solutions of plain GN-MPPI with
// a Gaussian negative log-likelihood.  Training and inference run in these
// kernels.  Every product -- forward, input gradient, weight gradient -- is a
// tcgen05 GEMM on the sm_103a tensor cores: its operands are stored as a BF16
// head plane and a BF16 remainder plane (K-major rows, loaded by TMA), each
// product is formed from three BF16 passes (head x head + head x remainder +
// remainder x head, FP32 accumulation in TMEM, FP32-level accuracy), and the
// epilogue fuses the bias, GELU (keeping the pre-activation) or the GELU'
// factor of the layer below and writes the next products' operand planes.  Weights optionally rounded to BF16 (their
// remainder plane is then zero) for the forward and input-gradient products.
// Then the loss and its output gradient, column sums for the bias gradients,
// and Adam with bias correction.  Parameter layout per layer: W [d_out][d_in]
// row-major, then b [d_out].
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/gnmppi.h"
#include "common.cuh"
#include "tc_ptx.cuh"

namespace gnm {
namespace {

constexpr int kMaxLayers = 8;

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_df(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// One product x[i][j] = sum_k A[i][k] B[j][k] (i < M, j < N, k < K) with the
// epilogue `mode`: 0 x += bias[j]; 1 z = x + bias[j], x = GELU(z); 2 x *=
// GELU'(zprev); 3 none; and with x stored where the pointers are not NULL:
//   C   [M][ldc] FP32; P (head, remainder) [M][ldp] BF16: the next product's operand;
//   PT  [N][ldt] the planes' transposes (the weight gradients' operands);
//   XT  [N][ldt] FP32 transposed (the bias gradients' sums); ZT [N][ldt] z transposed.
struct MlpTc {
  int M, N, K, mode;
  const float* bias;
  float* C;
  int64_t ldc;
  __nv_bfloat16 *Ph, *Pl;
  int64_t ldp;
  __nv_bfloat16 *PTh, *PTl;
  float *XT, *ZT;
  const float* ZTprev;
  int64_t ldt;
};
// The products of one launch: operand maps (A head, A remainder, B head, B
// remainder) and the first tile of each; tile t of product g covers rows 128
// (t / tn) and columns cols (t % tn).
template <int NB>
struct MlpBatch {
  CUtensorMap map[NB][4];
  MlpTc g[NB];
  int tile0[NB + 1];
  int count, cols, stages;  // output columns per tile (32, 64 or 128), ring depth
};

constexpr int kTcBox = 128 * 128;  // one 128-row x 64-value BF16 box (128-byte rows), 16 KB
constexpr int kTcRing = 160 * 1024;
constexpr int kTcMaxStages = 4;
constexpr int kTcSmem = kTcRing + 1024 + 256 + 4 * 32 * 33 * 4;  // ring, barriers, GELU' inputs

// One 128 x cols output tile per CTA.  Warp 0 lane 0 issues the TMA loads of
// the four operand boxes of a 64-value k-block into a ring, warp 1 lane 0 the
// three BF16 passes (M = 128, N = cols, K = 16 per MMA) into one TMEM
// accumulator; warps 0-3 read it back, one TMEM lane per output row, apply the
// epilogue and store the transposed outputs (32 consecutive rows per warp
// store) from registers and the row-major ones through a padded shared-memory
// transpose.  The network's products are small (a batch of 1024: 2 x 1024 x 256
// x 256 flops at most), so a launch is latency: starting up, one or two
// microseconds of load latency, the epilogue.  Hence narrow tiles (cols = 32
// spreads 1024 x 256 outputs over 64 SMs), the operand planes written by the
// epilogue that has the values in registers instead of by a pass of their own,
// the operand maps encoded with the handle, start-up beside the previous
// kernel's tail, and the weight gradients of all layers in one launch: a
// training step at batch 1024 takes 174 us in 13 launches, 550 in 31 before; one
// inference 49 us in 6, 77 in 10 (batch 4096: 95, 123).  Every wait is bounded; a wait that runs out sets
// *err and the CTA winds down.
template <int NB>
__global__ void __launch_bounds__(128, 1) k_mlp_tc(const __grid_constant__ MlpBatch<NB> p, int* __restrict__ err) {
  int gi = 0;
  while (gi + 1 < p.count && (int)blockIdx.x >= p.tile0[gi + 1]) ++gi;
  const MlpTc& g = p.g[gi];
  const int tn = (g.N + p.cols - 1) / p.cols, tile = blockIdx.x - p.tile0[gi];
  const int i0 = tile / tn * 128, j0 = tile % tn * p.cols;
  const int nkb = (g.K + 63) / 64, stages = p.stages;
  const int bbox = p.cols * 128, stage_bytes = 2 * (kTcBox + bbox);
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + kTcRing);
  // bars[0..4): full, [4..8): empty, [8]: done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kTcMaxStages + 1);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2 * kTcMaxStages + 1; ++s) mbar_init(su32(bars + s), 1);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                 "r"(128)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t done = su32(bars + 2 * kTcMaxStages);
  // the next product may start up now; the previous kernel's results are complete past the wait
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer
    int issued = 0;
    for (int kb = 0; kb < nkb; ++kb) {
      const int s = kb % stages, round = kb / stages;
      if (kb >= stages && !mbar_wait(su32(bars + kTcMaxStages + s), (round - 1) & 1, abort, true)) {
        *abort = 1;
        atomicExch(err, 1);
        break;
      }
      const uint32_t full = su32(bars + s);
      mbar_expect_tx(full, (uint32_t)stage_bytes);
      const uint32_t d = su32(base + s * stage_bytes);
      tma_load(d, &p.map[gi][0], full, kb * 64, i0);
      tma_load(d + kTcBox, &p.map[gi][1], full, kb * 64, i0);
      tma_load(d + 2 * kTcBox, &p.map[gi][2], full, kb * 64, j0);
      tma_load(d + 2 * kTcBox + bbox, &p.map[gi][3], full, kb * 64, j0);
      ++issued;
    }
    for (int kb = (issued > stages ? issued - stages : 0); kb < issued; ++kb)
      mbar_wait(su32(bars + kb % stages), (kb / stages) & 1, abort, false);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    const uint32_t id = idesc<true>(min(p.cols, (g.N - j0 + 15) / 16 * 16));
    for (int kb = 0; kb < nkb; ++kb) {
      const int s = kb % stages, round = kb / stages;
      if (!mbar_wait(su32(bars + s), round & 1, abort, true)) {
        *abort = 1;
        atomicExch(err, 1);
        break;
      }
      tc_fence_after();
      const uint32_t a0 = su32(base + s * stage_bytes);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t xa = a0 + k * 32, xb = a0 + 2 * kTcBox + k * 32;
        mma<true>(tmem, sdesc(xa), sdesc(xb), id, (kb > 0 || k > 0) ? 1u : 0u);
        mma<true>(tmem, sdesc(xa), sdesc(xb + bbox), id, 1u);
        mma<true>(tmem, sdesc(xa + kTcBox), sdesc(xb), id, 1u);
      }
      mma_commit(su32(bars + kTcMaxStages + s));
    }
    mma_commit(done);
  }
  __syncwarp();

  // what the epilogue reads is fetched a chunk ahead, the first while the MMAs run
  const int row0 = i0 + warp * 32, i = row0 + lane;
  const bool in = i < g.M;
  float bj = 0.f;
  float* zp = reinterpret_cast<float*>(base + kTcRing + 256) + (warp * 32 + lane) * 33;
  auto fetch = [&](int jc) {
    if (g.mode <= 1) bj = jc + lane < g.N ? g.bias[jc + lane] : 0.f;
    if (g.mode == 2) {
#pragma unroll 16
      for (int q = 0; q < 32; ++q) zp[q] = (in && jc + q < g.N) ? g.ZTprev[(int64_t)(jc + q) * g.ldt + i] : 0.f;
    }
  };
  fetch(j0);
  const bool ok = mbar_wait(done, 0, abort, false);
  tc_fence_after();
  if (__all_sync(0xffffffffu, ok && !*abort)) {
    float* stg = reinterpret_cast<float*>(base) + warp * 32 * 33;
    float* own = stg + lane * 33;
#pragma unroll 1
    for (int c = 0; c * 32 < p.cols && j0 + c * 32 < g.N; ++c) {  // uniform over the warp
      const int jc = j0 + c * 32;
      {
        uint32_t v[32];
        tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c * 32), v);
#pragma unroll
        for (int q = 0; q < 32; ++q) own[q] = __uint_as_float(v[q]);
      }
      if (c > 0) fetch(jc);
      // eight columns at a time, the arithmetic without branches so that their
      // chains overlap (a branch per entry cost 400 cycles each)
#pragma unroll 1
      for (int q0 = 0; q0 < 32; q0 += 8) {
        float x[8], z[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          x[e] = own[q0 + e];
          const float b = __shfl_sync(0xffffffffu, bj, q0 + e);
          if (g.mode <= 1) x[e] += b;
          z[e] = x[e];
        }
        if (g.mode == 1) {
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] = gelu_f(z[e]);
        } else if (g.mode == 2) {
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] *= gelu_df(zp[q0 + e]);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int j = jc + q0 + e;
          own[q0 + e] = x[e];
          const int64_t t = (int64_t)j * g.ldt + i;
          if (!in || j >= g.N || !GNM_IN(t, (int64_t)g.N * g.ldt + (g.ldt ? 0 : g.M))) continue;
          if (g.ZT) g.ZT[t] = z[e];
          if (g.XT) g.XT[t] = x[e];
          if (g.PTh) {
            const __nv_bfloat16 h = __float2bfloat16_rn(x[e]);
            g.PTh[t] = h;
            g.PTl[t] = __float2bfloat16_rn(x[e] - __bfloat162float(h));
          }
        }
      }
      __syncwarp();
      const int j = jc + lane;
      if (j < g.N) {
#pragma unroll 4
        for (int rr = 0; rr < 32; ++rr) {
          const int r = row0 + rr;
          if (r >= g.M) break;
          const float x = stg[rr * 33 + lane];
          if (g.C && GNM_IN((int64_t)r * g.ldc + j, (int64_t)g.M * g.ldc)) g.C[(int64_t)r * g.ldc + j] = x;
          if (g.Ph && GNM_IN((int64_t)r * g.ldp + j, (int64_t)g.M * g.ldp)) {
            const __nv_bfloat16 h = __float2bfloat16_rn(x);
            g.Ph[(int64_t)r * g.ldp + j] = h;
            g.Pl[(int64_t)r * g.ldp + j] = __float2bfloat16_rn(x - __bfloat162float(h));
          }
        }
      }
      __syncwarp();
    }
  } else if (threadIdx.x == 0) {
    atomicExch(err, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128) : "memory");
  }
}

// Stores of one 32 x 32 tile of an FP32 array: BF16 head / remainder planes
// hi[r ld + c] = bf16(x), lo[r ld + c] = bf16(x - hi) (0 when zero_lo, for
// BF16-exact weights), and, when hiT is not NULL, those of the transpose,
// hiT[c ldt + r].  Blocks of (32, 8) threads: thread (x, y) holds rows y, y + 8,
// ... of column x in v[].
struct PlaneOut {
  __nv_bfloat16 *hi, *lo;
  int64_t ld;
  __nv_bfloat16 *hiT, *loT;
  int64_t ldt;
};
__device__ __forceinline__ void store_planes(const PlaneOut& o, const float* v, int r0, int c0, int rows, int cols,
                                             int zero_lo) {
  __shared__ __nv_bfloat16 sh[32][33], sl[32][33];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int rr = threadIdx.y + 8 * q, r = r0 + rr, c = c0 + threadIdx.x;
    const float x = (r < rows && c < cols) ? v[q] : 0.f;
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    const __nv_bfloat16 l = zero_lo ? __float2bfloat16_rn(0.f) : __float2bfloat16_rn(x - __bfloat162float(h));
    if (r < rows && c < cols) {
      o.hi[(int64_t)r * o.ld + c] = h;
      o.lo[(int64_t)r * o.ld + c] = l;
    }
    sh[rr][threadIdx.x] = h;
    sl[rr][threadIdx.x] = l;
  }
  if (!o.hiT) return;  // uniform
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int cc = threadIdx.y + 8 * q, c = c0 + cc, r = r0 + threadIdx.x;
    if (c < cols && r < rows) {
      o.hiT[(int64_t)c * o.ldt + r] = sh[threadIdx.x][cc];
      o.loT[(int64_t)c * o.ldt + r] = sl[threadIdx.x][cc];
    }
  }
}

// Planes of h0 = (x - mean) / std in FP32, x given in FP64.
__global__ void __launch_bounds__(256) k_mlp_input(const double* __restrict__ X, int B, int d0,
                                                   const float* __restrict__ mean, const float* __restrict__ stdv,
                                                   PlaneOut o) {
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, c = c0 + threadIdx.x;
  float v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = r0 + threadIdx.y + 8 * q;
    v[q] = (r < B && c < d0) ? ((float)X[(int64_t)r * d0 + c] - mean[c]) / stdv[c] : 0.f;
  }
  store_planes(o, v, r0, c0, B, d0, 0);
}

// Gaussian NLL and dL/dy of one 32-sample x 32-output tile: thread (x, y) takes
// output column c0 + x of samples y, y + 8, ...  Columns below nmu are dL/dmu;
// column nmu + k is dL/ds_k, the sum over its step's nu components in order, and
// also forms the step's loss.  Per tile with scale columns and sample the loss
// terms go to part[tile][b].  dL/dy leaves as planes, as transposed planes and as FP32
// transposed XT [dL][ldt].  (One thread per sample and 200 dependent FP64 sums
// took a quarter of a training step.)
__global__ void __launch_bounds__(256) k_mlp_nll(const float* __restrict__ Y, int B, int dL, int nmu, int nu,
                                                 const double* __restrict__ T, PlaneOut o, float* __restrict__ XT,
                                                 double* __restrict__ part) {
  __shared__ float sx[32][33];
  const int b0 = blockIdx.y * 32, c0 = blockIdx.x * 32, col = c0 + threadIdx.x;
  const float invB = 1.0f / (float)B;
  float v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int b = b0 + threadIdx.y + 8 * q;
    double loss = 0.0;
    float d = 0.f;
    if (b < B && col < dL) {
      const float* y = Y + (int64_t)b * dL;
      const double* t = T + (int64_t)b * nmu;
      const int k = col < nmu ? col / nu : col - nmu;
      const float s = y[nmu + k];
      const float w = expf(-2.0f * s);
      if (col < nmu) {
        const float e = (float)t[col] - y[col];
        d = -e * w * invB;
      } else {
        for (int j = k * nu; j < (k + 1) * nu; ++j) {
          const float e = (float)t[j] - y[j];
          loss += 0.5 * (double)e * (double)e * (double)w + (double)s;
          d += (1.0f - e * e * w) * invB;
        }
      }
    }
    for (int o2 = 16; o2 > 0; o2 >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o2);
    const int pt = (int)blockIdx.x - nmu / 32;
    if (threadIdx.x == 0 && pt >= 0 && b < B) part[(int64_t)pt * B + b] = loss;
    v[q] = d;
    sx[threadIdx.y + 8 * q][threadIdx.x] = d;
  }
  __syncthreads();
  for (int q = 0; q < 4; ++q) {
    const int c = c0 + threadIdx.y + 8 * q, b = b0 + threadIdx.x;
    if (c < dL && b < B) XT[(int64_t)c * o.ldt + b] = sx[threadIdx.x][threadIdx.y + 8 * q];
  }
  store_planes(o, v, b0, c0, B, dL, 0);
}

// Deterministic sum of n doubles into out[0] (one block).
__global__ void k_sum(const double* x, int64_t n, double scale, double* out) {
  __shared__ double red[1024];
  double s = 0.0;
#pragma unroll 4
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0] * scale;
}

// Per-layer arrays of the kernels that run over all layers at once.
struct MlpLayers {
  int L;
  int dout[kMaxLayers], din[kMaxLayers];
  int64_t off[kMaxLayers];         // parameter offset of the layer
  const float* XT[kMaxLayers];     // output gradient, transposed [dout][ldt]
  PlaneOut W[kMaxLayers];          // weight planes and their transposes
  int tile0[kMaxLayers + 1];       // 32 x 32 weight tiles before the layer
  int col0[kMaxLayers + 1];        // output columns before the layer
};

// Bias gradients of all layers: gb[j] = sum_b dZ[b][j], b in order; a warp per
// column, each lane holding 32 rows in turn (one thread per column walked the
// batch's rows one load at a time).
__global__ void __launch_bounds__(128) k_colsum(MlpLayers m, int B, int64_t ldt, float* __restrict__ g) {
  const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (w >= m.col0[m.L]) return;
  int l = 0;
  while (w >= m.col0[l + 1]) ++l;
  const int j = w - m.col0[l];
  const float* x = m.XT[l] + (int64_t)j * ldt;
  float s = 0.f;
  for (int b0 = 0; b0 < B; b0 += 256) {
    float v[8];  // 256 rows' loads in flight at once
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = b0 + 32 * k + lane < B ? x[b0 + 32 * k + lane] : 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int nb = min(32, B - b0 - 32 * k);
      if (nb == 32) {
#pragma unroll
        for (int q = 0; q < 32; ++q) s += __shfl_sync(0xffffffffu, v[k], q);
      } else {
        for (int q = 0; q < nb; ++q) s += __shfl_sync(0xffffffffu, v[k], q);
      }
    }
  }
  if (lane == 0) g[m.off[l] + (int64_t)m.dout[l] * m.din[l] + j] = s;
}

struct AdamArgs {
  float *p, *m, *v;
  const float* g;
  float lr, b1, b2, eps, c1, c2;
  int update, zero_lo;  // update 0: only the planes, from the parameters as they are
};
__device__ __forceinline__ float adam(const AdamArgs& a, int64_t i) {
  if (!a.update) return a.p[i];
  const float gi = a.g[i];
  const float mi = a.b1 * a.m[i] + (1.f - a.b1) * gi;
  const float vi = a.b2 * a.v[i] + (1.f - a.b2) * gi * gi;
  a.m[i] = mi;
  a.v[i] = vi;
  const float pi = a.p[i] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
  a.p[i] = pi;
  return pi;
}
// Adam over all parameters and the refreshed weight planes in the same pass:
// blocks below tile0[L] take a 32 x 32 weight tile, the others biases.
__global__ void __launch_bounds__(256) k_adam(MlpLayers m, AdamArgs a) {
  const int nt = m.tile0[m.L];
  if ((int)blockIdx.x >= nt) {
    const int w = (blockIdx.x - nt) * 256 + threadIdx.y * 32 + threadIdx.x;
    if (w >= m.col0[m.L]) return;
    int l = 0;
    while (w >= m.col0[l + 1]) ++l;
    adam(a, m.off[l] + (int64_t)m.dout[l] * m.din[l] + (w - m.col0[l]));
    return;
  }
  int l = 0;
  while ((int)blockIdx.x >= m.tile0[l + 1]) ++l;
  const int t = blockIdx.x - m.tile0[l], tc = (m.din[l] + 31) / 32;
  const int r0 = t / tc * 32, c0 = t % tc * 32, c = c0 + threadIdx.x;
  float v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = r0 + threadIdx.y + 8 * q;
    v[q] = (r < m.dout[l] && c < m.din[l]) ? adam(a, m.off[l] + (int64_t)r * m.din[l] + c) : 0.f;
  }
  store_planes(m.W[l], v, r0, c0, m.dout[l], m.din[l], a.zero_lo);
}

__global__ void k_d2f(const double* x, int64_t n, float* y) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (float)x[i];
}
__global__ void k_f2d(const float* x, int64_t n, double* y, double scale) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (double)x[i] * scale;
}

// U0 = y_scale * mu, sigma_j = clamp(y_scale * exp(s_{j / nu}), lo, hi)
__global__ void k_warm(const float* Y, int B, int dL, int nmu, int nu, float yscale, double lo, double hi, double* U0,
                       double* sig) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)B * nmu) return;
  const int b = (int)(t / nmu), j = (int)(t % nmu);
  const float* y = Y + (int64_t)b * dL;
  U0[t] = (double)(yscale * y[j]);
  sig[t] = fmin(hi, fmax(lo, (double)(yscale * expf(y[nmu + j / nu]))));
}

}  // namespace
GNM_CHECK_ACCESSOR(check_count_mlp)
}  // namespace gnm

using namespace gnm;

struct gnmppi_mlp_s {
  int L = 0;
  int dims[kMaxLayers + 1] = {0};
  int nu = 1, nmu = 0, bf16 = 0, max_batch = 0;
  int64_t np = 0;
  int64_t off[kMaxLayers + 1] = {0};  // parameter offset of layer l (1-based)
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  float *xmean = nullptr, *xstd = nullptr;
  float yscale = 1.f;
  float* Y = nullptr;                    // network outputs [B][d_L]
  float* ZT[kMaxLayers + 1] = {nullptr};  // hidden pre-activations, transposed [d_l][ldb]
  float* XT[kMaxLayers + 1] = {nullptr};  // output gradients, transposed [d_l][ldb]
  // BF16 head / remainder planes of the tensor-core operands: activations
  // H_l [B][ldh l] and their transposes [d_l][ldb] (l < L), weights W_l
  // [d_l][ldh l-1] and their transposes [d_{l-1}][ldh l], output gradients
  // dZ_l [B][ldh l] and their transposes [d_l][ldb]
  __nv_bfloat16 *Hh[kMaxLayers + 1] = {nullptr}, *Hl[kMaxLayers + 1] = {nullptr};
  __nv_bfloat16 *HTh[kMaxLayers + 1] = {nullptr}, *HTl[kMaxLayers + 1] = {nullptr};
  __nv_bfloat16 *Wh[kMaxLayers + 1] = {nullptr}, *Wl[kMaxLayers + 1] = {nullptr};
  __nv_bfloat16 *WTh[kMaxLayers + 1] = {nullptr}, *WTl[kMaxLayers + 1] = {nullptr};
  __nv_bfloat16 *Dh[kMaxLayers + 1] = {nullptr}, *Dl[kMaxLayers + 1] = {nullptr};
  __nv_bfloat16 *DTh[kMaxLayers + 1] = {nullptr}, *DTl[kMaxLayers + 1] = {nullptr};
  int64_t ldh[kMaxLayers + 1] = {0};
  int64_t ldb = 0;
  int nsm = 1;
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  // pinned host memory the kernels write: set when a bounded wait of the
  // tensor-core GEMM ran out; the minibatch loss
  int* h_err = nullptr;
  double* h_loss = nullptr;
  // operand maps, by tile width 32 << c: [l][0]: layer l's forward product,
  // [l][1]: its input gradient (their row extents are max_batch: rows past the
  // batch only reach output rows that are not stored); and the weight
  // gradients', whose depth is the batch, for the last batch size
  CUtensorMap maps[3][kMaxLayers + 1][2][4];
  CUtensorMap gw_maps[3][kMaxLayers][4];
  int gw_B = 0;
  double* loss_b = nullptr;  // per 32-output tile and sample
  int t = 0;
  std::vector<void*> allocs;
  std::string err;
};

static thread_local char g_mlp_err[512];

static gnmppi_status mfail(gnmppi_mlp_t h, gnmppi_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  if (h) h->err = buf;
  else snprintf(g_mlp_err, sizeof(g_mlp_err), "%s", buf);
  return st;
}

#define MCK(call)                                                                                             \
  do {                                                                                                        \
    cudaError_t e_ = (call);                                                                                  \
    if (e_ != cudaSuccess) return mfail(h, GNMPPI_E_CUDA, "%s: %s", #call, cudaGetErrorString(e_));            \
  } while (0)
#define MCKL() MCK(cudaGetLastError())

template <typename P>
static gnmppi_status malloc_(gnmppi_mlp_t h, P** ptr, size_t bytes) {
  if (cudaMalloc((void**)ptr, bytes < 16 ? 16 : bytes) != cudaSuccess) {
    cudaGetLastError();
    return mfail(h, GNMPPI_E_NOMEM, "cudaMalloc(%zu) failed", bytes);
  }
  h->allocs.push_back((void*)*ptr);
  MCK(cudaMemsetAsync(*ptr, 0, bytes < 16 ? 16 : bytes, h->stream));
  return GNMPPI_OK;
}

static gnmppi_status refresh_weights(gnmppi_mlp_t h);
static bool encode_maps(gnmppi_mlp_t h);

extern "C" const char* gnmppi_mlp_last_error(gnmppi_mlp_t h) { return h ? h->err.c_str() : g_mlp_err; }

extern "C" void gnmppi_mlp_destroy(gnmppi_mlp_t h) {
  if (!h) return;
  if (h->stream) cudaStreamSynchronize(h->stream);
  for (void* q : h->allocs) cudaFree(q);
  if (h->h_err) cudaFreeHost(h->h_err);
  if (h->h_loss) cudaFreeHost(h->h_loss);
  if (h->own_stream) cudaStreamDestroy(h->stream);
  delete h;
}

extern "C" gnmppi_status gnmppi_mlp_create(int32_t nlayers, const int32_t* dims, int32_t nu, int32_t weights_bf16,
                                           int32_t max_batch, void* cuda_stream, gnmppi_mlp_t* out) {
  if (!out || !dims) return mfail(nullptr, GNMPPI_E_ARG, "dims and out must not be NULL");
  *out = nullptr;
  if (nlayers < 1 || nlayers > kMaxLayers) return mfail(nullptr, GNMPPI_E_ARG, "nlayers must be in 1..%d", kMaxLayers);
  for (int l = 0; l <= nlayers; ++l)
    if (dims[l] < 1 || dims[l] > 65536) return mfail(nullptr, GNMPPI_E_ARG, "layer widths must be in 1..65536");
  if (nu < 1 || dims[nlayers] % (nu + 1) != 0)
    return mfail(nullptr, GNMPPI_E_ARG, "output width must be n_mu + n_mu/nu (a multiple of nu + 1)");
  if (max_batch < 1) return mfail(nullptr, GNMPPI_E_ARG, "max_batch must be >= 1");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
    cudaGetLastError();
    return mfail(nullptr, GNMPPI_E_CUDA, "no CUDA device available");
  }
  gnmppi_mlp_t h = new gnmppi_mlp_s();
  h->L = nlayers;
  for (int l = 0; l <= nlayers; ++l) h->dims[l] = dims[l];
  h->nu = nu;
  h->nmu = dims[nlayers] / (nu + 1) * nu;
  h->bf16 = weights_bf16 ? 1 : 0;
  h->max_batch = max_batch;
  int64_t np = 0;
  for (int l = 1; l <= nlayers; ++l) {
    h->off[l] = np;
    np += (int64_t)dims[l] * dims[l - 1] + dims[l];
  }
  h->np = np;
  if (cuda_stream) {
    h->stream = (cudaStream_t)cuda_stream;
  } else {
    if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete h;
      return mfail(nullptr, GNMPPI_E_CUDA, "cudaStreamCreate failed");
    }
    h->own_stream = true;
  }
  gnmppi_status st;
#define MA(ptr, bytes)                                          \
  if ((st = malloc_(h, &(ptr), (bytes))) != GNMPPI_OK) {        \
    snprintf(g_mlp_err, sizeof(g_mlp_err), "%s", h->err.c_str()); \
    gnmppi_mlp_destroy(h);                                      \
    return st;                                                  \
  }
  MA(h->p, 4 * np);
  MA(h->g, 4 * np);
  MA(h->m, 4 * np);
  MA(h->v, 4 * np);
  MA(h->xmean, 4 * (size_t)dims[0]);
  MA(h->xstd, 4 * (size_t)dims[0]);
  // BF16 operand planes; row strides rounded up to 8 values (16 bytes, the TMA stride rule)
  auto r8 = [](int64_t x) { return (x + 7) / 8 * 8; };
  h->ldb = r8(max_batch);
  for (int l = 0; l <= nlayers; ++l) h->ldh[l] = r8(dims[l]);
  MA(h->Y, 4 * (size_t)max_batch * dims[nlayers]);
  for (int l = 0; l < nlayers; ++l) {
    MA(h->Hh[l], 2 * (size_t)max_batch * h->ldh[l]);
    MA(h->Hl[l], 2 * (size_t)max_batch * h->ldh[l]);
    MA(h->HTh[l], 2 * (size_t)dims[l] * h->ldb);
    MA(h->HTl[l], 2 * (size_t)dims[l] * h->ldb);
  }
  for (int l = 1; l <= nlayers; ++l) {
    MA(h->Wh[l], 2 * (size_t)dims[l] * h->ldh[l - 1]);
    MA(h->Wl[l], 2 * (size_t)dims[l] * h->ldh[l - 1]);
    MA(h->WTh[l], 2 * (size_t)dims[l - 1] * h->ldh[l]);
    MA(h->WTl[l], 2 * (size_t)dims[l - 1] * h->ldh[l]);
    MA(h->Dh[l], 2 * (size_t)max_batch * h->ldh[l]);
    MA(h->Dl[l], 2 * (size_t)max_batch * h->ldh[l]);
    MA(h->DTh[l], 2 * (size_t)dims[l] * h->ldb);
    MA(h->DTl[l], 2 * (size_t)dims[l] * h->ldb);
    MA(h->XT[l], 4 * (size_t)dims[l] * h->ldb);
    if (l < nlayers) MA(h->ZT[l], 4 * (size_t)dims[l] * h->ldb);
  }
  MA(h->loss_b, 8 * (size_t)max_batch * ((dims[nlayers] + 31) / 32));
#undef MA
  {
    void* fn = nullptr;
    int dev = 0;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn ||
        cudaFuncSetAttribute(k_mlp_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem) != cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_tc<kMaxLayers>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem) !=
            cudaSuccess ||
        cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaMallocHost((void**)&h->h_err, sizeof(int)) != cudaSuccess ||
        cudaMallocHost((void**)&h->h_loss, sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      gnmppi_mlp_destroy(h);
      return mfail(nullptr, GNMPPI_E_CUDA, "tensor-core GEMM set-up failed (cuTensorMapEncodeTiled, shared memory)");
    }
    h->encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    *h->h_err = 0;
  }
  if (!encode_maps(h)) {
    gnmppi_mlp_destroy(h);
    return mfail(nullptr, GNMPPI_E_CUDA, "cuTensorMapEncodeTiled failed (MLP operand)");
  }
  std::vector<float> one(dims[0], 1.f);
  if (cudaMemcpyAsync(h->xstd, one.data(), 4 * one.size(), cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
      cudaStreamSynchronize(h->stream) != cudaSuccess) {
    gnmppi_mlp_destroy(h);
    return mfail(nullptr, GNMPPI_E_CUDA, "initialising the MLP failed");
  }
  *out = h;
  return GNMPPI_OK;
}

extern "C" int64_t gnmppi_mlp_num_params(gnmppi_mlp_t h) { return h ? h->np : 0; }


static gnmppi_status to_device_f(gnmppi_mlp_t h, int32_t mem, const double* src, int64_t n, float* dst) {
  const double* dsrc = src;
  double* tmp = nullptr;
  if (mem == GNMPPI_MEM_HOST) {
    MCK(cudaMallocAsync((void**)&tmp, 8 * (size_t)n, h->stream));
    MCK(cudaMemcpyAsync(tmp, src, 8 * (size_t)n, cudaMemcpyHostToDevice, h->stream));
    dsrc = tmp;
  }
  k_d2f<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>(dsrc, n, dst);
  MCKL();
  if (tmp) MCK(cudaFreeAsync(tmp, h->stream));
  MCK(cudaStreamSynchronize(h->stream));
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_set_params(gnmppi_mlp_t h, int32_t mem, const double* params, int64_t count) {
  if (!h || !params) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (count != h->np) return mfail(h, GNMPPI_E_ARG, "expected %lld parameters", (long long)h->np);
  gnmppi_status st = to_device_f(h, mem, params, count, h->p);
  if (st != GNMPPI_OK) return st;
  if ((st = refresh_weights(h)) != GNMPPI_OK) return st;
  MCK(cudaMemsetAsync(h->m, 0, 4 * (size_t)h->np, h->stream));
  MCK(cudaMemsetAsync(h->v, 0, 4 * (size_t)h->np, h->stream));
  h->t = 0;
  MCK(cudaStreamSynchronize(h->stream));
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_get_params(gnmppi_mlp_t h, int32_t mem, double* params, int64_t count) {
  if (!h || !params) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (count != h->np) return mfail(h, GNMPPI_E_ARG, "expected %lld parameters", (long long)h->np);
  double* dst = params;
  if (mem == GNMPPI_MEM_HOST) MCK(cudaMallocAsync((void**)&dst, 8 * (size_t)count, h->stream));
  k_f2d<<<(unsigned)((count + 255) / 256), 256, 0, h->stream>>>(h->p, count, dst, 1.0);
  MCKL();
  if (mem == GNMPPI_MEM_HOST) {
    MCK(cudaMemcpyAsync(params, dst, 8 * (size_t)count, cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaFreeAsync(dst, h->stream));
  }
  MCK(cudaStreamSynchronize(h->stream));
  return GNMPPI_OK;
}

// Copy an FP32 device array out as doubles into `mem` memory.
static gnmppi_status out_f(gnmppi_mlp_t h, int32_t mem, const float* src, int64_t n, double* dst_user) {
  double* dst = dst_user;
  if (mem == GNMPPI_MEM_HOST) MCK(cudaMallocAsync((void**)&dst, 8 * (size_t)n, h->stream));
  k_f2d<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>(src, n, dst, 1.0);
  MCKL();
  if (mem == GNMPPI_MEM_HOST) {
    MCK(cudaMemcpyAsync(dst_user, dst, 8 * (size_t)n, cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaFreeAsync(dst, h->stream));
  }
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_get_state(gnmppi_mlp_t h, int32_t mem, double* params, double* m1, double* m2,
                                              int64_t count, int32_t* step) {
  if (!h || !params || !m1 || !m2 || !step) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (count != h->np) return mfail(h, GNMPPI_E_ARG, "expected %lld parameters", (long long)h->np);
  gnmppi_status st;
  if ((st = out_f(h, mem, h->p, count, params)) != GNMPPI_OK) return st;
  if ((st = out_f(h, mem, h->m, count, m1)) != GNMPPI_OK) return st;
  if ((st = out_f(h, mem, h->v, count, m2)) != GNMPPI_OK) return st;
  MCK(cudaStreamSynchronize(h->stream));
  *step = h->t;
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_set_state(gnmppi_mlp_t h, int32_t mem, const double* params, const double* m1,
                                              const double* m2, int64_t count, int32_t step) {
  if (!h || !params || !m1 || !m2) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (count != h->np) return mfail(h, GNMPPI_E_ARG, "expected %lld parameters", (long long)h->np);
  if (step < 0) return mfail(h, GNMPPI_E_ARG, "step must be >= 0");
  gnmppi_status st;
  if ((st = to_device_f(h, mem, params, count, h->p)) != GNMPPI_OK) return st;
  if ((st = to_device_f(h, mem, m1, count, h->m)) != GNMPPI_OK) return st;
  if ((st = to_device_f(h, mem, m2, count, h->v)) != GNMPPI_OK) return st;
  if ((st = refresh_weights(h)) != GNMPPI_OK) return st;
  MCK(cudaStreamSynchronize(h->stream));
  h->t = step;
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_set_normalization(gnmppi_mlp_t h, const double* x_mean, const double* x_std,
                                                      double y_scale) {
  if (!h || !x_mean || !x_std) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (!(y_scale > 0.0)) return mfail(h, GNMPPI_E_ARG, "y_scale must be > 0");
  std::vector<float> m(h->dims[0]), s(h->dims[0]);
  for (int i = 0; i < h->dims[0]; ++i) {
    if (!(x_std[i] > 0.0)) return mfail(h, GNMPPI_E_ARG, "x_std must be > 0");
    m[i] = (float)x_mean[i];
    s[i] = (float)x_std[i];
  }
  MCK(cudaMemcpyAsync(h->xmean, m.data(), 4 * m.size(), cudaMemcpyHostToDevice, h->stream));
  MCK(cudaMemcpyAsync(h->xstd, s.data(), 4 * s.size(), cudaMemcpyHostToDevice, h->stream));
  MCK(cudaStreamSynchronize(h->stream));
  h->yscale = (float)y_scale;
  return GNMPPI_OK;
}

// K-major BF16 plane [rows][ld] as a TMA operand: boxes of 64 values x `box`
// rows, 128-byte swizzle, zero fill outside the `cols` x `rows` extent.
static bool encode_plane(gnmppi_mlp_t h, CUtensorMap* m, const __nv_bfloat16* p, int64_t cols, int64_t rows,
                         int64_t ld, int box) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t boxd[2] = {64, (cuuint32_t)box};
  cuuint32_t estr[2] = {1, 1};
  return h->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(p), dims, strides, boxd, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Maps of C = A B^T: A [M][K] (planes Ah, Al, row stride lda), B [N][K] (planes
// Bh, Bl, row stride ldb), for output tiles of `cols` columns.
static bool encode_product(gnmppi_mlp_t h, CUtensorMap* m, const __nv_bfloat16* Ah, const __nv_bfloat16* Al, int64_t lda,
                           int64_t M, const __nv_bfloat16* Bh, const __nv_bfloat16* Bl, int64_t ldb, int64_t N,
                           int64_t K, int cols) {
  return encode_plane(h, m, Ah, K, M, lda, 128) && encode_plane(h, m + 1, Al, K, M, lda, 128) &&
         encode_plane(h, m + 2, Bh, K, N, ldb, cols) && encode_plane(h, m + 3, Bl, K, N, ldb, cols);
}
static bool encode_maps(gnmppi_mlp_t h) {
  for (int c = 0; c < 3; ++c)
    for (int l = 1; l <= h->L; ++l) {
      const int64_t din = h->dims[l - 1], dout = h->dims[l], B = h->max_batch;
      if (!encode_product(h, h->maps[c][l][0], h->Hh[l - 1], h->Hl[l - 1], h->ldh[l - 1], B, h->Wh[l], h->Wl[l],
                          h->ldh[l - 1], dout, din, 32 << c) ||
          !encode_product(h, h->maps[c][l][1], h->Dh[l], h->Dl[l], h->ldh[l], B, h->WTh[l], h->WTl[l], h->ldh[l], din,
                          dout, 32 << c))
        return false;
    }
  return true;
}

// Launch the products g[0..count) (outputs, epilogue and M, N, K); maps(c, k):
// the operand maps of product k for tiles of 32 << c columns.  Tiles of 32
// columns while they leave no SM a second one, else wider: a CTA spends as long
// starting up as multiplying.
template <int NB, class Maps>
static gnmppi_status tc_gemm(gnmppi_mlp_t h, const MlpTc* g, int count, const Maps& maps) {
  MlpBatch<NB> p;
  p.count = count;
  int c = 0;
  for (;; ++c) {
    p.cols = 32 << c;
    p.tile0[0] = 0;
    for (int k = 0; k < count; ++k)
      p.tile0[k + 1] = p.tile0[k] + (g[k].M + 127) / 128 * ((g[k].N + p.cols - 1) / p.cols);
    if (c == 2 || p.tile0[count] <= h->nsm) break;
  }
  const int stage = 2 * (kTcBox + p.cols * 128);
  p.stages = kTcRing / stage < kTcMaxStages ? kTcRing / stage : kTcMaxStages;
  for (int k = 0; k < count; ++k) {
    p.g[k] = g[k];
    memcpy(p.map[k], maps(c, k), sizeof(p.map[k]));
  }
  // starts up beside the previous kernel's tail (it waits for that kernel before reading its results)
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)p.tile0[count]);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = kTcSmem;
  cfg.stream = h->stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  MCK(cudaLaunchKernelEx(&cfg, k_mlp_tc<NB>, p, h->h_err));
  return GNMPPI_OK;
}

static MlpLayers layers(gnmppi_mlp_t h) {
  MlpLayers m{};
  m.L = h->L;
  for (int l = 1; l <= h->L; ++l) {
    const int k = l - 1, din = h->dims[k], dout = h->dims[l];
    m.dout[k] = dout;
    m.din[k] = din;
    m.off[k] = h->off[l];
    m.XT[k] = h->XT[l];
    m.W[k] = PlaneOut{h->Wh[l], h->Wl[l], h->ldh[k], h->WTh[l], h->WTl[l], h->ldh[l]};
    m.tile0[l] = m.tile0[k] + (din + 31) / 32 * ((dout + 31) / 32);
    m.col0[l] = m.col0[k] + dout;
  }
  return m;
}

// One Adam step (update) and the weight planes W_l and W_l^T from the FP32
// master parameters (the remainder plane is zero when the products use
// BF16-rounded weights).
static gnmppi_status adam_planes(gnmppi_mlp_t h, AdamArgs a) {
  const MlpLayers m = layers(h);
  a.p = h->p;
  a.m = h->m;
  a.v = h->v;
  a.g = h->g;
  a.zero_lo = h->bf16;
  const int bias_blocks = a.update ? (m.col0[m.L] + 255) / 256 : 0;
  k_adam<<<(unsigned)(m.tile0[m.L] + bias_blocks), dim3(32, 8), 0, h->stream>>>(m, a);
  MCKL();
  return GNMPPI_OK;
}
static gnmppi_status refresh_weights(gnmppi_mlp_t h) { return adam_planes(h, AdamArgs{}); }

// End of a call: wait for it and check the tensor-core error word.
static gnmppi_status finish(gnmppi_mlp_t h) {
  MCK(cudaStreamSynchronize(h->stream));
  if (*h->h_err) {
    *h->h_err = 0;
    return mfail(h, GNMPPI_E_TIMEOUT, "a bounded wait in the MLP's tensor-core GEMM ran out");
  }
  return GNMPPI_OK;
}

// Forward pass of B samples already in device memory (FP64), outputs in Y;
// `train` also writes what the gradients use: the transposed activation planes
// and the hidden pre-activations.
static gnmppi_status forward(gnmppi_mlp_t h, const double* dX, int B, bool train) {
  const int d0 = h->dims[0];
  const PlaneOut in{h->Hh[0], h->Hl[0], h->ldh[0], train ? h->HTh[0] : nullptr, h->HTl[0], h->ldb};
  k_mlp_input<<<dim3((unsigned)((d0 + 31) / 32), (unsigned)((B + 31) / 32)), dim3(32, 8), 0, h->stream>>>(
      dX, B, d0, h->xmean, h->xstd, in);
  MCKL();
  for (int l = 1; l <= h->L; ++l) {
    const int din = h->dims[l - 1], dout = h->dims[l];
    const bool hidden = l < h->L;
    MlpTc q{};
    q.M = B;
    q.N = dout;
    q.K = din;
    q.bias = h->p + h->off[l] + (int64_t)dout * din;
    q.mode = hidden ? 1 : 0;
    if (hidden) {
      q.Ph = h->Hh[l];
      q.Pl = h->Hl[l];
      q.ldp = h->ldh[l];
      if (train) {
        q.PTh = h->HTh[l];
        q.PTl = h->HTl[l];
        q.ZT = h->ZT[l];
        q.ldt = h->ldb;
      }
    } else {
      q.C = h->Y;
      q.ldc = dout;
    }
    gnmppi_status st = tc_gemm<1>(h, &q, 1, [&](int c, int) { return h->maps[c][l][0]; });
    if (st != GNMPPI_OK) return st;
  }
  return GNMPPI_OK;
}

// Loss and gradient of B samples (device FP64 inputs) into h->g and h->h_loss.
static gnmppi_status loss_grad(gnmppi_mlp_t h, const double* dX, const double* dT, int B) {
  gnmppi_status st = forward(h, dX, B, true);
  if (st != GNMPPI_OK) return st;
  const int L = h->L, dL = h->dims[L];
  const int ct = (dL + 31) / 32;
  const PlaneOut out{h->Dh[L], h->Dl[L], h->ldh[L], h->DTh[L], h->DTl[L], h->ldb};
  k_mlp_nll<<<dim3((unsigned)ct, (unsigned)((B + 31) / 32)), dim3(32, 8), 0, h->stream>>>(h->Y, B, dL, h->nmu, h->nu,
                                                                                         dT, out, h->XT[L], h->loss_b);
  MCKL();
  k_sum<<<1, 1024, 0, h->stream>>>(h->loss_b, (int64_t)(ct - h->nmu / 32) * B, 1.0 / B, h->h_loss);
  MCKL();
  for (int l = L; l > 1; --l) {
    // dz_{l-1}[b][i] = (sum_o dz_l[b][o] W_l[o][i]) * GELU'(z_{l-1}[b][i])
    MlpTc q{};
    q.M = B;
    q.N = h->dims[l - 1];
    q.K = h->dims[l];
    q.mode = 2;
    q.ZTprev = h->ZT[l - 1];
    q.ldt = h->ldb;
    q.XT = h->XT[l - 1];
    q.PTh = h->DTh[l - 1];
    q.PTl = h->DTl[l - 1];
    if (l > 2) {  // the next product down reads the row-major planes
      q.Ph = h->Dh[l - 1];
      q.Pl = h->Dl[l - 1];
      q.ldp = h->ldh[l - 1];
    }
    if ((st = tc_gemm<1>(h, &q, 1, [&](int c, int) { return h->maps[c][l][1]; })) != GNMPPI_OK) return st;
  }
  // gW_l[o][i] = sum_b dz_l[b][o] h_{l-1}[b][i]: the transposed planes, K = B
  if (h->gw_B != B) {
    h->gw_B = 0;
    for (int c = 0; c < 3; ++c)
      for (int l = 1; l <= L; ++l)
        if (!encode_product(h, h->gw_maps[c][l - 1], h->DTh[l], h->DTl[l], h->ldb, h->dims[l], h->HTh[l - 1],
                            h->HTl[l - 1], h->ldb, h->dims[l - 1], B, 32 << c))
          return mfail(h, GNMPPI_E_CUDA, "cuTensorMapEncodeTiled failed (MLP operand)");
    h->gw_B = B;
  }
  MlpTc q[kMaxLayers] = {};
  for (int l = 1; l <= L; ++l) {
    MlpTc& x = q[l - 1];
    x.M = h->dims[l];
    x.N = h->dims[l - 1];
    x.K = B;
    x.mode = 3;
    x.C = h->g + h->off[l];
    x.ldc = h->dims[l - 1];
  }
  if ((st = tc_gemm<kMaxLayers>(h, q, L, [&](int c, int k) { return h->gw_maps[c][k]; })) != GNMPPI_OK) return st;
  const MlpLayers m = layers(h);
  k_colsum<<<(unsigned)((m.col0[L] + 3) / 4), 128, 0, h->stream>>>(m, B, h->ldb, h->g);
  MCKL();
  return GNMPPI_OK;
}

static gnmppi_status stage_in(gnmppi_mlp_t h, int32_t mem, const double* src, int64_t n, const double** dptr,
                              double** tmp) {
  *tmp = nullptr;
  *dptr = src;
  if (mem == GNMPPI_MEM_HOST) {
    MCK(cudaMallocAsync((void**)tmp, 8 * (size_t)(n > 0 ? n : 1), h->stream));
    MCK(cudaMemcpyAsync(*tmp, src, 8 * (size_t)n, cudaMemcpyHostToDevice, h->stream));
    *dptr = *tmp;
  }
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_forward(gnmppi_mlp_t h, int32_t mem, const double* X, int32_t B, double* Y) {
  if (!h || !X || !Y) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (B < 1 || B > h->max_batch) return mfail(h, GNMPPI_E_ARG, "B must be in 1..%d", h->max_batch);
  const double* dX;
  double* tx;
  gnmppi_status st = stage_in(h, mem, X, (int64_t)B * h->dims[0], &dX, &tx);
  if (st != GNMPPI_OK) return st;
  if ((st = forward(h, dX, B, false)) != GNMPPI_OK) return st;
  const int64_t n = (int64_t)B * h->dims[h->L];
  double* dY = Y;
  if (mem == GNMPPI_MEM_HOST) MCK(cudaMallocAsync((void**)&dY, 8 * (size_t)n, h->stream));
  k_f2d<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>(h->Y, n, dY, 1.0);
  MCKL();
  if (mem == GNMPPI_MEM_HOST) {
    MCK(cudaMemcpyAsync(Y, dY, 8 * (size_t)n, cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaFreeAsync(dY, h->stream));
  }
  if (tx) MCK(cudaFreeAsync(tx, h->stream));
  return finish(h);
}

extern "C" gnmppi_status gnmppi_mlp_loss_grad(gnmppi_mlp_t h, int32_t mem, const double* X, const double* T,
                                              int32_t B, double* loss, double* grad) {
  if (!h || !X || !T) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (B < 1 || B > h->max_batch) return mfail(h, GNMPPI_E_ARG, "B must be in 1..%d", h->max_batch);
  const double *dX, *dT;
  double *tx, *tt;
  gnmppi_status st = stage_in(h, mem, X, (int64_t)B * h->dims[0], &dX, &tx);
  if (st == GNMPPI_OK) st = stage_in(h, mem, T, (int64_t)B * h->nmu, &dT, &tt);
  if (st != GNMPPI_OK) return st;
  if ((st = loss_grad(h, dX, dT, B)) != GNMPPI_OK) return st;
  if (grad) {
    double* dg = grad;
    if (mem == GNMPPI_MEM_HOST) MCK(cudaMallocAsync((void**)&dg, 8 * (size_t)h->np, h->stream));
    k_f2d<<<(unsigned)((h->np + 255) / 256), 256, 0, h->stream>>>(h->g, h->np, dg, 1.0);
    MCKL();
    if (mem == GNMPPI_MEM_HOST) {
      MCK(cudaMemcpyAsync(grad, dg, 8 * (size_t)h->np, cudaMemcpyDeviceToHost, h->stream));
      MCK(cudaFreeAsync(dg, h->stream));
    }
  }
  if (tx) MCK(cudaFreeAsync(tx, h->stream));
  if (tt) MCK(cudaFreeAsync(tt, h->stream));
  if ((st = finish(h)) != GNMPPI_OK) return st;
  if (loss) *loss = *h->h_loss;
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_train_step(gnmppi_mlp_t h, int32_t mem, const double* X, const double* T,
                                               int32_t B, double lr, double* loss) {
  if (!h || !X || !T) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (B < 1 || B > h->max_batch) return mfail(h, GNMPPI_E_ARG, "B must be in 1..%d", h->max_batch);
  if (!(lr > 0.0)) return mfail(h, GNMPPI_E_ARG, "lr must be > 0");
  const double *dX, *dT;
  double *tx, *tt;
  gnmppi_status st = stage_in(h, mem, X, (int64_t)B * h->dims[0], &dX, &tx);
  if (st == GNMPPI_OK) st = stage_in(h, mem, T, (int64_t)B * h->nmu, &dT, &tt);
  if (st != GNMPPI_OK) return st;
  if ((st = loss_grad(h, dX, dT, B)) != GNMPPI_OK) return st;
  h->t += 1;
  const double b1 = 0.9, b2 = 0.999;
  AdamArgs a{};
  a.lr = (float)lr;
  a.b1 = (float)b1;
  a.b2 = (float)b2;
  a.eps = 1e-8f;
  a.c1 = (float)(1.0 - std::pow(b1, h->t));
  a.c2 = (float)(1.0 - std::pow(b2, h->t));
  a.update = 1;
  if ((st = adam_planes(h, a)) != GNMPPI_OK) return st;
  if (tx) MCK(cudaFreeAsync(tx, h->stream));
  if (tt) MCK(cudaFreeAsync(tt, h->stream));
  if ((st = finish(h)) != GNMPPI_OK) return st;
  if (loss) *loss = *h->h_loss;
  return GNMPPI_OK;
}

extern "C" gnmppi_status gnmppi_mlp_warm_start(gnmppi_mlp_t h, int32_t mem, const double* X, int32_t B,
                                               double sigma_min, double sigma_max, double* U0, double* sigma) {
  if (!h || !X || !U0 || !sigma) return mfail(h, GNMPPI_E_ARG, "NULL argument");
  if (!(sigma_min > 0.0) || !(sigma_max >= sigma_min)) return mfail(h, GNMPPI_E_ARG, "need 0 < sigma_min <= sigma_max");
  if (B < 1 || B > h->max_batch) return mfail(h, GNMPPI_E_ARG, "B must be in 1..%d", h->max_batch);
  const double* dX;
  double* tx;
  gnmppi_status st = stage_in(h, mem, X, (int64_t)B * h->dims[0], &dX, &tx);
  if (st != GNMPPI_OK) return st;
  if ((st = forward(h, dX, B, false)) != GNMPPI_OK) return st;
  const int64_t n = (int64_t)B * h->nmu;
  double *dU = U0, *dS = sigma;
  if (mem == GNMPPI_MEM_HOST) {
    MCK(cudaMallocAsync((void**)&dU, 8 * (size_t)n, h->stream));
    MCK(cudaMallocAsync((void**)&dS, 8 * (size_t)n, h->stream));
  }
  k_warm<<<(unsigned)((n + 255) / 256), 256, 0, h->stream>>>(h->Y, B, h->dims[h->L], h->nmu, h->nu, h->yscale,
                                                             sigma_min, sigma_max, dU, dS);
  MCKL();
  if (mem == GNMPPI_MEM_HOST) {
    MCK(cudaMemcpyAsync(U0, dU, 8 * (size_t)n, cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaMemcpyAsync(sigma, dS, 8 * (size_t)n, cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaFreeAsync(dU, h->stream));
    MCK(cudaFreeAsync(dS, h->stream));
  }
  if (tx) MCK(cudaFreeAsync(tx, h->stream));
  return finish(h);
}
