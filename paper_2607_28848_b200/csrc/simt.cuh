// Plain CUDA-core kernels of the multi-LoRA layer, templated on the storage type.  They are the
// product path for fp32 layers (small layers; every product in fp32 FMA) and, for bf16 layers,
// a slow cross-check of the tensor-core kernels that shares none of their index arithmetic.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dropout.cuh"
#include "ptx.cuh"

namespace mlora {
namespace simt {

// The kernels here wait for the launch in front as the first thing they do, and let the next one start its own launch at once:
// between short kernels that is where the time goes (launch to launch 4.7 us without it).
__device__ __forceinline__ void wait_then_trigger() {
  ptx::grid_dependency_wait();
  ptx::grid_launch_dependents();
}

__device__ __forceinline__ float ld(const float* p) { return *p; }
__device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void st(float* p, float v) { *p = v; }
__device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// Out[t, q] = (scale?) * sum_k In[t, k] P_a(t)[q, k]; one warp per (row, q); rows without an
// adapter get zeros, and so do rows whose id lies outside [-1, n_adapters) (the planned path has
// validated its ids on the host; a caller-supplied device table has not been looked at by anyone).  Fine-tuning rows (row_save >= 0) also write u_save (unscaled) and x_save;
// with dropout on, their products skip the dropped columns and count 1 / (1 - p).
template <typename T>
__global__ void shrink_kernel(const T* In, int64_t ld_in, int D, int R, const T* P_all, const float* scale,
                              const int32_t* row_adapter, const int32_t* row_save, float* Out,
                              T* x_save, float* u_save, int64_t save_base, int n_rows, int n_adapters,
                              const DropArgs drop) {
  wait_then_trigger();
  const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= n_rows * R) return;
  const int t = wid / R, q = wid % R;
  int a = row_adapter[t];
  if (a >= n_adapters) a = -1;
  const int sv = row_save ? row_save[t] : -1;
  float acc = 0.f;
  if (a >= 0) {
    const T* x = In + (size_t)t * ld_in;
    const T* p = P_all + ((size_t)a * R + q) * D;
    if (drop.thr != 0 && sv >= 0) {
      for (int k = lane; k < D; k += 32)
        if (drop_keep(drop, (uint32_t)sv, (uint32_t)k)) acc = fmaf(ld(x + k), ld(p + k), acc);
    } else {
      for (int k = lane; k < D; k += 32) acc = fmaf(ld(x + k), ld(p + k), acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (drop.thr != 0 && sv >= 0) acc *= drop.keep_scale;
  }
  if (lane == 0) {
    Out[(size_t)t * R + q] = (a >= 0 && scale) ? acc * scale[a] : acc;
    if (sv >= 0 && u_save) u_save[(size_t)(save_base + sv) * R + q] = acc;
  }
  if (sv >= 0 && x_save && q == 0) {
    const T* x = In + (size_t)t * ld_in;
    T* d = x_save + (size_t)(save_base + sv) * D;
    for (int k = lane; k < D; k += 32) d[k] = x[k];
  }
}

// Out[m, n] = sum_k In[m, k] Wop(k, n) + sum_q P[m, q] sc L_a(m)[q, n], one thread per element, tiles of 8 rows x 32 columns.
// W_KMAJOR: Wop(k, n) = W[n * ldw + k]; else Wop(k, n) = W[k * ldw + n].
// With `drop` on (input gradient only) the low-rank term of element (m, n) is kept or dropped
// as the branch input (m, n) was in the forward.
// Bound by shared-memory reads: both operands lie with k innermost, so four steps of k take two 16-byte reads (a pitch of 36
// floats spreads the columns over the banks), and 8-row tiles spread a small layer over 64 SMs instead of 16 (64 x 256 x 256:
// 13.2 us with 32-row tiles before, 5.0 now).  A weight element comes from the L2 four times as often per row as with 32-row
// tiles, which costs less than the reads saved at every size measured: fp32 forward + backward of 16 to 4096 rows, 256 to 4096
// wide, 1.03 to 2.4 times as fast (4096 rows 4096 -> 4096 34.7 -> 31.3 ms), the allocation-free bf16 forward of 1 to 512 rows
// 1.03 to 3.7 times (512 rows 4096 -> 4096 2.54 -> 2.19 ms).  The sums run over k in the same order as before.
constexpr int GEMM_ROWS = 8;
struct GemmTile {
  __align__(16) float in[2][GEMM_ROWS][32];
  __align__(16) float w[2][32][36];                    // [n local][k local]
};
// Base product of element (m0 + threadIdx.y, n0 + threadIdx.x); the whole block calls it.
template <typename T, bool W_KMAJOR>
__device__ __forceinline__ float tile_product(GemmTile& s, const T* In, int64_t ld_in, const T* W, int64_t ldw, int m0, int n0, int M,
                                              int N, int K) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int m = m0 + ty, n = n0 + tx;
  float next_in, next_w[32 / GEMM_ROWS];
  auto load = [&](int k0) {
    next_in = (m < M && k0 + tx < K) ? ld(In + (size_t)m * ld_in + k0 + tx) : 0.f;
#pragma unroll
    for (int i = 0; i < 32 / GEMM_ROWS; ++i) {
      const int r = ty + GEMM_ROWS * i;                          // W_KMAJOR: local column, k = tx; else local k, column = tx
      if (W_KMAJOR) next_w[i] = (n0 + r < N && k0 + tx < K) ? ld(W + (size_t)(n0 + r) * ldw + k0 + tx) : 0.f;
      else          next_w[i] = (k0 + r < K && n < N) ? ld(W + (size_t)(k0 + r) * ldw + n) : 0.f;
    }
  };
  float acc = 0.f;
  load(0);
  for (int k0 = 0, buf = 0; k0 < K; k0 += 32, buf ^= 1) {        // two buffers: one barrier per 32 steps of k
    s.in[buf][ty][tx] = next_in;
#pragma unroll
    for (int i = 0; i < 32 / GEMM_ROWS; ++i) {
      const int r = ty + GEMM_ROWS * i;
      if (W_KMAJOR) s.w[buf][r][tx] = next_w[i];
      else          s.w[buf][tx][r] = next_w[i];
    }
    __syncthreads();
    if (k0 + 32 < K) load(k0 + 32);
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(&s.in[buf][ty][k]), w = *reinterpret_cast<const float4*>(&s.w[buf][tx][k]);
      acc = fmaf(x.x, w.x, acc); acc = fmaf(x.y, w.y, acc); acc = fmaf(x.z, w.z, acc); acc = fmaf(x.w, w.w, acc);
    }
  }
  return acc;
}
// The base product plus the low-rank term of element (m, n): P = the row's rank-R values, a = its adapter.
template <typename T>
__device__ __forceinline__ float add_low_rank(float acc, const float* P, int a, const float* scale, const T* L_all, int m, int n, int N,
                                              int R, const DropArgs& drop) {
  const float sc = scale ? scale[a] : 1.0f;
  float lo = 0.f;
#pragma unroll 8
  for (int q = 0; q < R; ++q) lo = fmaf(P[q], ld(L_all + ((size_t)a * R + q) * N + n), lo);
  if (drop.thr != 0) lo = drop_keep(drop, (uint32_t)m, (uint32_t)n) ? lo * drop.keep_scale : 0.f;
  return fmaf(sc, lo, acc);
}
template <typename T, bool W_KMAJOR>
__global__ void __launch_bounds__(32 * GEMM_ROWS)
gemm_lora_kernel(const T* In, int64_t ld_in, const T* W, int64_t ldw, const T* L_all,
                                 const float* P, const float* scale, const int32_t* row_adapter,
                                 T* Out, int64_t ld_out, int M, int N, int K, int R, int n_adapters,
                                 const DropArgs drop) {
  wait_then_trigger();
  __shared__ GemmTile s;
  const int n0 = blockIdx.x * 32, n = n0 + threadIdx.x;
  for (int m0 = (int)blockIdx.y * GEMM_ROWS; m0 < M; m0 += (int)gridDim.y * GEMM_ROWS) {
    const int m = m0 + threadIdx.y;
    const int a = (row_adapter && m < M) ? row_adapter[m] : -1;
    float acc = tile_product<T, W_KMAJOR>(s, In, ld_in, W, ldw, m0, n0, M, N, K);
    if (m < M && n < N) {
      if (a >= 0 && a < n_adapters)          // an id outside the adapter tables counts as no adapter
        acc = add_low_rank(acc, P + (size_t)m * R, a, scale, L_all, m, n, N, R, drop);
      st(Out + (size_t)m * ld_out + n, acc);
    }
    __syncthreads();                          // the buffers are the next rows' now
  }
}
inline dim3 gemm_grid(int M, int N) {
  const int y = (M + GEMM_ROWS - 1) / GEMM_ROWS;
  return dim3((N + 31) / 32, y < 65535 ? y : 65535);
}

// G[slot, q, j] (+)= sum over the slot's rows of sc P[t, q] Q[t, j]; one thread per (q, j).
// With `drop` on (dA only: Q = the saved branch input) element (t, j) of Q is kept or dropped.
template <typename T>
struct GradTask {
  const float* P;
  const float* scale;
  const T* Q;
  int64_t ldq;
  float* G;
  int32_t R, D, n_slots, accumulate;
  const int32_t *slot_chunk_off, *chunk_row0, *chunk_nrows, *slot_adapter;
  DropArgs drop;
};
template <typename T>
__device__ __forceinline__ void grad_element(const GradTask<T>& g, int slot, int q, int j) {
  if (j >= g.D) return;
  const float sc = (g.scale ? g.scale[g.slot_adapter[slot]] : 1.0f) * (g.drop.thr != 0 ? g.drop.keep_scale : 1.0f);
  float acc = 0.f;
  for (int ch = g.slot_chunk_off[slot]; ch < g.slot_chunk_off[slot + 1]; ++ch) {
    const int r0 = g.chunk_row0[ch], nr = g.chunk_nrows[ch];
    const float* P = g.P + (size_t)r0 * g.R + q;
    const T* Q = g.Q + (size_t)r0 * g.ldq + j;
    if (g.drop.thr == 0) {
      int t = 0;
      for (; t + 16 <= nr; t += 16) {          // sixteen rows in flight
        float p[16], x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) { p[i] = P[(size_t)(t + i) * g.R]; x[i] = ld(Q + (size_t)(t + i) * g.ldq); }
#pragma unroll
        for (int i = 0; i < 16; ++i) acc = fmaf(p[i] * sc, x[i], acc);
      }
      for (; t < nr; ++t) acc = fmaf(P[(size_t)t * g.R] * sc, ld(Q + (size_t)t * g.ldq), acc);
    } else {
      for (int t = 0; t < nr; ++t)
        if (drop_keep(g.drop, (uint32_t)(r0 + t), (uint32_t)j)) acc = fmaf(P[(size_t)t * g.R] * sc, ld(Q + (size_t)t * g.ldq), acc);
    }
  }
  float* dst = g.G + ((size_t)slot * g.R + q) * g.D + j;
  *dst = g.accumulate ? *dst + acc : acc;
}
template <typename T>
__global__ void grad_kernel(const GradTask<T> g) {
  wait_then_trigger();
  grad_element(g, (int)blockIdx.z, (int)blockIdx.y, (int)(blockIdx.x * blockDim.x + threadIdx.x));
}

// ---- small fp32 layers: the same arithmetic in fewer launches ------------------------------------
// A pass over a layer of a few hundred columns takes less time than launching its kernels, so the rank-R products move into the
// kernels that use them: the forward is one launch, the backward two (64 rows 256 -> 256, rank 8, forward + backward: 28.7 us
// with six launches, 21.5 with their set-up overlapped, 19.0 here).  Every sum has the terms and the order of the kernels above.

// sum_k x[k] p[k] as shrink_kernel adds it (over a warp), for NQ rows of p at a time; with dropout the dropped columns are skipped.
template <int NQ, typename T>
__device__ __forceinline__ void row_dots(const T* x, const T* p, int D, int lane, const DropArgs& drop, int sv, float (&acc)[NQ]) {
#pragma unroll
  for (int i = 0; i < NQ; ++i) acc[i] = 0.f;
  const bool dropping = drop.thr != 0 && sv >= 0;
#pragma unroll 4
  for (int k = lane; k < D; k += 32) {
    const float xv = ld(x + k);
    const bool keep = !dropping || drop_keep(drop, (uint32_t)sv, (uint32_t)k);
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const float pv = ld(p + (size_t)i * D + k);
      if (keep) acc[i] = fmaf(xv, pv, acc[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
    if (dropping) acc[i] *= drop.keep_scale;
  }
}

// Forward: every block of 8 rows x 32 columns computes its rows' rank-R values itself, one warp per row; the blocks of the first
// columns save them and the rows.  R is at most 128.
template <typename T>
__global__ void __launch_bounds__(32 * GEMM_ROWS)
small_forward_kernel(const T* In, int64_t ld_in, const T* W, int64_t ldw, const T* A_all, const T* B_all, const float* scale,
                     const int32_t* row_adapter, const int32_t* row_save, T* Out, int64_t ld_out, T* x_save, float* u_save,
                     int64_t save_base, int M, int N, int K, int R, const DropArgs drop) {
  wait_then_trigger();
  __shared__ GemmTile s;
  __shared__ float U[GEMM_ROWS][128];
  const int lane = threadIdx.x, ty = threadIdx.y;
  const int m0 = (int)blockIdx.y * GEMM_ROWS, m = m0 + ty, n0 = blockIdx.x * 32, n = n0 + lane;
  const int a = m < M ? row_adapter[m] : -1;
  const int sv = m < M && row_save ? row_save[m] : -1;
  const T* x = In + (size_t)m * ld_in;
  if (a >= 0) {
    const T* p = A_all + (size_t)a * R * K;
    int q = 0;
    for (; q + 8 <= R; q += 8) {
      float u[8];
      row_dots<8>(x, p + (size_t)q * K, K, lane, drop, sv, u);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (lane == i) U[ty][q + i] = u[i];
    }
    if (q + 4 <= R) {
      float u[4];
      row_dots<4>(x, p + (size_t)q * K, K, lane, drop, sv, u);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (lane == i) U[ty][q + i] = u[i];
      q += 4;
    }
    for (; q < R; ++q) {
      float u[1];
      row_dots<1>(x, p + (size_t)q * K, K, lane, drop, sv, u);
      if (lane == 0) U[ty][q] = u[0];
    }
    __syncwarp();
  }
  if (sv >= 0 && blockIdx.x == 0) {
    if (u_save)
      for (int q = lane; q < R; q += 32) u_save[(size_t)(save_base + sv) * R + q] = a >= 0 ? U[ty][q] : 0.f;
    if (x_save)
      for (int k = lane; k < K; k += 32) x_save[(size_t)(save_base + sv) * K + k] = x[k];
  }
  float acc = tile_product<T, false>(s, In, ld_in, W, ldw, m0, n0, M, N, K);
  if (m < M && n < N) {
    if (a >= 0) acc = add_low_rank(acc, U[ty], a, scale, B_all, m, n, N, R, DropArgs{0, 0, 1.0f});
    st(Out + (size_t)m * ld_out + n, acc);
  }
}

// Backward, first launch: the blocks [0, grad_blocks) compute dB - first, since each walks the slot's rows one after the other -
// and the ones behind them V = s dY B^T (a warp per value, as shrink_kernel), which dB does not need.
template <typename T>
__device__ __noinline__ void grad_block(const GradTask<T>& g, int block) {
  const int strips = (g.D + 255) / 256, strip = block % strips, rest = block / strips;
  grad_element(g, rest / g.R, rest % g.R, strip * 256 + (int)(threadIdx.y * 32 + threadIdx.x));
}
template <typename T>
__global__ void __launch_bounds__(32 * GEMM_ROWS)
small_backward_v_kernel(const T* dY, int64_t lddy, int D, const T* B_all, const float* scale, const int32_t* row_adapter, float* V,
                        int n_rows, int grad_blocks, const GradTask<T> dB) {
  wait_then_trigger();
  if ((int)blockIdx.x < grad_blocks) { grad_block(dB, (int)blockIdx.x); return; }
  const int R = dB.R, w = ((int)blockIdx.x - grad_blocks) * GEMM_ROWS + threadIdx.y, lane = threadIdx.x;
  if (w >= n_rows * R) return;
  const int t = w / R, q = w % R, a = row_adapter[t];
  float v[1] = {0.f};
  if (a >= 0) row_dots<1>(dY + (size_t)t * lddy, B_all + ((size_t)a * R + q) * D, D, lane, DropArgs{0, 0, 1.0f}, -1, v);
  if (lane == 0) V[(size_t)t * R + q] = a >= 0 ? v[0] * scale[a] : 0.f;
}
// Second launch: the blocks [0, grad_blocks) compute dA, the ones behind them dX.
template <typename T>
__global__ void __launch_bounds__(32 * GEMM_ROWS)
small_backward_x_kernel(const T* dY, int64_t lddy, const T* W, int64_t ldw, const T* A_all, const float* V, const int32_t* row_adapter,
                        T* dX, int64_t lddx, int M, int N, int K, int grad_blocks, const GradTask<T> dA) {
  wait_then_trigger();
  __shared__ GemmTile s;
  if ((int)blockIdx.x < grad_blocks) { grad_block(dA, (int)blockIdx.x); return; }
  const int tile = (int)blockIdx.x - grad_blocks;
  const int col_tiles = (N + 31) / 32;
  const int m0 = tile / col_tiles * GEMM_ROWS, n0 = tile % col_tiles * 32;
  const int m = m0 + threadIdx.y, n = n0 + threadIdx.x;
  const int a = m < M ? row_adapter[m] : -1;
  float acc = tile_product<T, true>(s, dY, lddy, W, ldw, m0, n0, M, N, K);
  if (m < M && n < N) {
    if (a >= 0) acc = add_low_rank<T>(acc, V + (size_t)m * dA.R, a, nullptr, A_all, m, n, N, dA.R, dA.drop);
    st(dX + (size_t)m * lddx + n, acc);
  }
}

// One AdamW update of the adapters of the fine-tuning slots; element i of slot g, rank row q,
// column j.  `which` = blockIdx.y: 0 -> the A matrices (width d_in), 1 -> the B matrices (d_out).
struct AdamwSide {
  const float* grad;   // [n_slots, R, D]
  float* master;       // [n_slots, R, D]
  float* m;
  float* v;
  void* weights;       // [n_adapters, R, D] in the layer's storage type
  int32_t D;
};
struct AdamwArgs {
  AdamwSide side[2];
  const int32_t* slot_adapter;
  int32_t n_slots, R;
  float lr, beta1, beta2, eps, wd, inv_bc1, inv_bc2;   // inv_bc = 1 / (1 - beta^t)
};

template <typename T>
__global__ void adamw_kernel(const AdamwArgs a) {
  wait_then_trigger();
  const AdamwSide& s = a.side[blockIdx.y];
  const int64_t per_slot = (int64_t)a.R * s.D;
  const int64_t total4 = (int64_t)a.n_slots * per_slot / 4;           // D is a multiple of 4
  for (int64_t i4 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i4 < total4; i4 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = i4 * 4;
    const int slot = (int)(i / per_slot);
    const int64_t off = i - (int64_t)slot * per_slot;
    const float4 g = *reinterpret_cast<const float4*>(s.grad + i);
    float4 w = *reinterpret_cast<const float4*>(s.master + i);
    float4 m = *reinterpret_cast<const float4*>(s.m + i);
    float4 v = *reinterpret_cast<const float4*>(s.v + i);
    float* gw = reinterpret_cast<float*>(const_cast<float4*>(&g));
    float *pw = reinterpret_cast<float*>(&w), *pm = reinterpret_cast<float*>(&m), *pv = reinterpret_cast<float*>(&v);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float wk = pw[k] - a.lr * a.wd * pw[k];
      const float mk = a.beta1 * pm[k] + (1.0f - a.beta1) * gw[k];
      const float vk = a.beta2 * pv[k] + (1.0f - a.beta2) * gw[k] * gw[k];
      wk -= a.lr * (mk * a.inv_bc1) / (sqrtf(vk * a.inv_bc2) + a.eps);
      pw[k] = wk; pm[k] = mk; pv[k] = vk;
    }
    *reinterpret_cast<float4*>(s.master + i) = w;
    *reinterpret_cast<float4*>(s.m + i) = m;
    *reinterpret_cast<float4*>(s.v + i) = v;
    T* dst = reinterpret_cast<T*>(s.weights) + (int64_t)a.slot_adapter[slot] * per_slot + off;
#pragma unroll
    for (int k = 0; k < 4; ++k) st(dst + k, pw[k]);
  }
}

}  // namespace simt
}  // namespace mlora
