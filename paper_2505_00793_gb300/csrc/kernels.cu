// Elementwise, row and update kernels of the mixed-mode sweep (HBM-bound work).
//
//  * per-example loss seeds with the tangent per-example loss (the mixed term of Eq. 7 for
//    per-example weights) and d eta_{t,b} = sigmoid'(eta_{t,b}) * l'_b / B;
//  * the fused per-layer update kernel: the inner-step update of Eq. 2 (rollout, SGD,
//    heavy ball or Adam) or the adjoint update of the reverse sweep (Eq. 5 with the Hessian
//    product supplied by the forward-over-reverse pass, and the elementwise reverse of the
//    optimiser step), each fused with the cast of the next step's parameters / tangent into
//    the bf16 GEMM operand copies;
//  * the chain loss of the motivating example, in both HVP modes;
//  * the reverse-over-reverse element kernels, column fills and a deterministic sum.
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include "device_math.cuh"
#include "internal.h"
#include "launch.cuh"

namespace mf {

int g_pdl = 1;
namespace {

constexpr int TILE = 32, TROWS = 8;

template <typename T>
__global__ void fill_cols_kernel(const ColFill f, int rows) {
  pdl_entry();
  const int n = blockIdx.y;
  T* dst = static_cast<T*>(f.dst[n]);
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x)
    dst[static_cast<int64_t>(r) * f.ld[n] + f.col[n]] = to_t<T>(f.value[n]);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// One warp per example row.  Squared loss l = 1/2 mean_o (f - y)^2; softmax CE
// l = logsumexp(f) - f_y.  Seeds scaled by w_b / B.
template <typename T>
__device__ __forceinline__ void loss_seed_row(const LossArgs& a, int row, int lane) {
  const int C = a.cols;
  const float* f = a.F + static_cast<int64_t>(row) * C;
  const float* fd = a.Fd ? a.Fd + static_cast<int64_t>(row) * C : nullptr;
  float w = 1.f, sg = 0.f;
  if (a.ex_w) w = a.ex_w[row];
  else if (a.eta_w) { sg = 1.f / (1.f + expf(-a.eta_w[row])); w = sg; }
  const float scale = w * a.inv_norm;
  T* dF = static_cast<T*>(a.dF);
  T* dFd = static_cast<T*>(a.dFd);
  const int64_t orow = static_cast<int64_t>(row) * a.ldo;
  float l = 0.f, ld = 0.f;
  if (a.loss == 0) {
    const float* y = a.Yf + static_cast<int64_t>(row) * C;
    const float invC = 1.f / static_cast<float>(C);
    float s2 = 0.f, s1 = 0.f;
    for (int c = lane; c < C; c += 32) {
      const float r = f[c] - y[c];
      s2 += r * r;
      if (fd) s1 += r * fd[c];
      if (dF) dF[orow + c] = to_t<T>(scale * r * invC);
      if (fd && dFd) dFd[orow + c] = to_t<T>(scale * fd[c] * invC);
    }
    l = 0.5f * warp_sum(s2) * invC;
    ld = warp_sum(s1) * invC;
  } else {
    const int y = a.Yi[row];
    if (y < 0 || y >= C) {
      if (lane == 0 && a.status) atomicMax(a.status, 1);
      return;
    }
    float mx = -INFINITY;
    for (int c = lane; c < C; c += 32) mx = fmaxf(mx, f[c]);
    mx = warp_max(mx);
    float se = 0.f;
    for (int c = lane; c < C; c += 32) se += expf(f[c] - mx);
    se = warp_sum(se);
    const float lse = mx + logf(se);
    float pf = 0.f;
    if (fd) {
      for (int c = lane; c < C; c += 32) pf += expf(f[c] - lse) * fd[c];
      pf = warp_sum(pf);
    }
    for (int c = lane; c < C; c += 32) {
      const float pc = expf(f[c] - lse);
      if (dF) dF[orow + c] = to_t<T>(scale * (pc - (c == y ? 1.f : 0.f)));
      if (fd && dFd) dFd[orow + c] = to_t<T>(scale * pc * (fd[c] - pf));
    }
    l = lse - f[y];
    if (fd) ld = pf - fd[y];
  }
  if (lane == 0) {
    if (a.l) a.l[row] = l;
    if (a.ld) a.ld[row] = ld;
    if (a.d_eta && a.eta_w) a.d_eta[row] = sg * (1.f - sg) * ld * a.inv_norm;
  }
}

template <typename T>
__global__ void loss_seed_kernel(const LossArgs a) {
  pdl_entry();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row < a.rows) loss_seed_row<T>(a, row, threadIdx.x & 31);
}

// The same for wide rows, one block per row: a warp crossed a wide row in strided passes one
// load at a time (512 rows x 4096, squared error: 75 us; one block per row with sixteen-byte
// loads in flight: 7 us).  From 129 columns on, where both take the same time at few rows;
// a 1000-way cross-entropy at 1000 rows takes its call from 56 to 30 us.
constexpr int LB_THREADS = 256, kBlockLossCols = 128;

// Sum (or maximum) over the block, in every thread.
template <bool MAX>
__device__ __forceinline__ float block_reduce(float v, float* red) {
  v = MAX ? warp_max(v) : warp_sum(v);
  __syncthreads();   // red may still be read
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = red[0];
#pragma unroll
  for (int i = 1; i < LB_THREADS / 32; ++i) r = MAX ? fmaxf(r, red[i]) : r + red[i];
  return r;
}

// n (1 or 4) consecutive floats of p at c
template <int N>
__device__ __forceinline__ void ldn(float (&x)[N], const float* p, int c) {
  if constexpr (N == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p + c);
    x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
  } else {
    x[0] = p[c];
  }
}
template <typename T, int N>
__device__ __forceinline__ void stn(T* p, int64_t c, const float (&x)[N]) {
  if constexpr (N == 1) {
    p[c] = to_t<T>(x[0]);
  } else if constexpr (sizeof(T) == 2) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(x[0], x[1]), hi = __floats2bfloat162_rn(x[2], x[3]);
    uint2 v;
    v.x = *reinterpret_cast<uint32_t*>(&lo);
    v.y = *reinterpret_cast<uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(p + c) = v;
  } else {
    *reinterpret_cast<float4*>(p + c) = make_float4(x[0], x[1], x[2], x[3]);
  }
}

template <typename T, int N>
__global__ void __launch_bounds__(LB_THREADS) loss_seed_block_kernel(const LossArgs a) {
  pdl_entry();
  __shared__ float red[LB_THREADS / 32];
  const int row = blockIdx.x, C = a.cols;
  const float* f = a.F + static_cast<int64_t>(row) * C;
  const float* fd = a.Fd ? a.Fd + static_cast<int64_t>(row) * C : nullptr;
  float w = 1.f, sg = 0.f;
  if (a.ex_w) w = a.ex_w[row];
  else if (a.eta_w) { sg = 1.f / (1.f + expf(-a.eta_w[row])); w = sg; }
  const float scale = w * a.inv_norm;
  T* dF = a.dF ? static_cast<T*>(a.dF) + static_cast<int64_t>(row) * a.ldo : nullptr;
  T* dFd = fd && a.dFd ? static_cast<T*>(a.dFd) + static_cast<int64_t>(row) * a.ldo : nullptr;
  const int c0 = threadIdx.x * N;
  constexpr int STEP = LB_THREADS * N;
  float l = 0.f, ld = 0.f;
  if (a.loss == 0) {
    const float* y = a.Yf + static_cast<int64_t>(row) * C;
    const float invC = 1.f / static_cast<float>(C);
    float s2 = 0.f, s1 = 0.f;
#pragma unroll 4
    for (int c = c0; c < C; c += STEP) {
      float fv[N], yv[N], dv[N] = {}, o[N];
      ldn(fv, f, c);
      ldn(yv, y, c);
      if (fd) ldn(dv, fd, c);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const float r = fv[j] - yv[j];
        s2 += r * r;
        s1 += r * dv[j];
        o[j] = scale * r * invC;
        dv[j] = scale * dv[j] * invC;
      }
      if (dF) stn<T, N>(dF, c, o);
      if (dFd) stn<T, N>(dFd, c, dv);
    }
    l = 0.5f * block_reduce<false>(s2, red) * invC;
    ld = block_reduce<false>(s1, red) * invC;
  } else {
    const int y = a.Yi[row];
    if (y < 0 || y >= C) {
      if (threadIdx.x == 0 && a.status) atomicMax(a.status, 1);
      return;
    }
    float mx = -INFINITY, se = 0.f, pf = 0.f;
#pragma unroll 4
    for (int c = c0; c < C; c += STEP) {
      float fv[N];
      ldn(fv, f, c);
#pragma unroll
      for (int j = 0; j < N; ++j) mx = fmaxf(mx, fv[j]);
    }
    mx = block_reduce<true>(mx, red);
#pragma unroll 4
    for (int c = c0; c < C; c += STEP) {
      float fv[N];
      ldn(fv, f, c);
#pragma unroll
      for (int j = 0; j < N; ++j) se += expf(fv[j] - mx);
    }
    const float lse = mx + logf(block_reduce<false>(se, red));
    if (fd) {
#pragma unroll 4
      for (int c = c0; c < C; c += STEP) {
        float fv[N], dv[N];
        ldn(fv, f, c);
        ldn(dv, fd, c);
#pragma unroll
        for (int j = 0; j < N; ++j) pf += expf(fv[j] - lse) * dv[j];
      }
      pf = block_reduce<false>(pf, red);
    }
#pragma unroll 4
    for (int c = c0; c < C; c += STEP) {
      float fv[N], dv[N] = {}, o[N];
      ldn(fv, f, c);
      if (fd) ldn(dv, fd, c);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const float pc = expf(fv[j] - lse);
        o[j] = scale * (pc - (c + j == y ? 1.f : 0.f));
        dv[j] = scale * pc * (dv[j] - pf);
      }
      if (dF) stn<T, N>(dF, c, o);
      if (dFd) stn<T, N>(dFd, c, dv);
    }
    l = lse - f[y];
    if (fd) ld = pf - fd[y];
  }
  if (threadIdx.x == 0) {
    if (a.l) a.l[row] = l;
    if (a.ld) a.ld[row] = ld;
    if (a.d_eta && a.eta_w) a.d_eta[row] = sg * (1.f - sg) * ld * a.inv_norm;
  }
}

// Motivating example of Section 3 (Eq. 8): the model output is f = x theta followed by the
// elementwise recursion y_0 = f, y_i = i (2 + sin y_{i-1})^cos y_{i-1}, i = 1..M, and
// l_b = mean_o (y_M - t)^2.  Per element the recursion is carried with its first and second
// derivatives in f (y', y''), so the loss seed 2/C r y' and its tangent 2/C (y'^2 + r y'') f'
// come out of one pass; nothing of the recursion is stored.  One block per example.
template <bool SECOND>
__device__ __forceinline__ void chain_eval(float f, int M, float& y, float& d1, float& d2) {
  y = f; d1 = 1.f; d2 = 0.f;
  for (int i = 1; i <= M; ++i) {
    float sn, cs;
    sincosf(y, &sn, &cs);
    const float b = 2.f + sn;                 // >= 1
    const float lb = logf(b);
    const float g1 = -sn * lb + cs * cs / b;  // d/dy [cos y log(2 + sin y)]
    const float yi = static_cast<float>(i) * expf(cs * lb);
    const float f1 = yi * g1;
    if constexpr (SECOND) {
      const float g2 = -cs * lb - 3.f * sn * cs / b - cs * cs * cs / (b * b);
      d2 = yi * (g1 * g1 + g2) * d1 * d1 + f1 * d2;
    }
    d1 = f1 * d1;
    y = yi;
  }
}

// Bound by the instructions of sincosf, logf, expf and the divisions of each step.  Without a
// tangent the second derivatives are not formed: 1024 x 4096 at M = 3, primal 65 -> 39 us, dual
// 53 us.
template <typename T, bool DUAL, int N>
__global__ void __launch_bounds__(LB_THREADS) chain_loss_kernel(const LossArgs a) {
  pdl_entry();
  __shared__ float red[LB_THREADS / 32];
  const int row = blockIdx.x;
  const int C = a.cols;
  const float* f = a.F + static_cast<int64_t>(row) * C;
  const float* fd = DUAL ? a.Fd + static_cast<int64_t>(row) * C : nullptr;
  const float* t = a.Yf + static_cast<int64_t>(row) * C;
  float w = 1.f, sg = 0.f;
  if (a.ex_w) w = a.ex_w[row];
  else if (a.eta_w) { sg = 1.f / (1.f + expf(-a.eta_w[row])); w = sg; }
  const float invC = 1.f / static_cast<float>(C);
  const float scale = w * a.inv_norm;
  T* dF = a.dF ? static_cast<T*>(a.dF) + static_cast<int64_t>(row) * a.ldo : nullptr;
  T* dFd = DUAL && a.dFd ? static_cast<T*>(a.dFd) + static_cast<int64_t>(row) * a.ldo : nullptr;
  float s2 = 0.f, s1 = 0.f;
  bool bad = false;
  for (int c = threadIdx.x * N; c < C; c += LB_THREADS * N) {
    float fv[N], tv[N], dv[N] = {}, o[N], od[N];
    ldn(fv, f, c);
    ldn(tv, t, c);
    if constexpr (DUAL) ldn(dv, fd, c);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      float y, d1, d2;
      chain_eval<DUAL>(fv[j], a.chain, y, d1, d2);
      const float r = y - tv[j];
      bad |= !isfinite(y) || !isfinite(d1);
      s2 += r * r;
      o[j] = scale * 2.f * invC * r * d1;
      if constexpr (DUAL) {
        const float ad = d1 * dv[j];
        s1 += r * ad;
        od[j] = scale * 2.f * invC * (d1 * ad + r * d2 * dv[j]);
      }
    }
    if (dF) stn<T, N>(dF, c, o);
    if constexpr (DUAL) {
      if (dFd) stn<T, N>(dFd, c, od);
    }
  }
  if (bad && a.status) atomicMax(a.status, DEV_NONFINITE);
  const float l = block_reduce<false>(s2, red) * invC;
  const float ld = DUAL ? block_reduce<false>(s1, red) * 2.f * invC : 0.f;
  if (threadIdx.x == 0) {
    if (a.l) a.l[row] = l;
    if (a.ld) a.ld[row] = ld;
    if (a.d_eta && a.eta_w) a.d_eta[row] = sg * (1.f - sg) * ld * a.inv_norm;
  }
}

// The same loss by reverse-over-reverse (Algorithm 1's schedule applied inside the chain).
// ror = 1, primal: forward y_i = phi_i(y_{i-1}) recording y_0..y_{M-1}, then the backward
// ybar_M = c r, ybar_{i-1} = ybar_i phi_i'(y_{i-1}) recording ybar_1..ybar_M, with
// c = 2 w / (B C) and phi_i' = y_i (d/dy)[cos y log(2 + sin y)]; dF = ybar_0.
// ror = 2, adjoint of that backward along a_0 = Fd (the incoming adjoint of ybar_0): forward
// a_i = a_{i-1} phi_i'(y_{i-1}) leaving yhat_{i-1} = a_{i-1} ybar_i phi_i''(y_{i-1}) in
// ybar_i's slot, then yhat_M = c a_M and back yhat_{i-1} += yhat_i phi_i'(y_{i-1});
// dFd = yhat_0, and ld = 2/C sum r a_M.  Both phases read the tape back instead of carrying
// derivatives, so the tape (2 M floats per element) is what this mode holds beyond the
// mixed mode.  Tape slot k of element e = row * C + c is at tape[k * rows * C + e].
__device__ __forceinline__ float chain_step(int i, float y, float& g1, float& g2) {
  float sn, cs;
  sincosf(y, &sn, &cs);
  const float b = 2.f + sn;
  const float lb = logf(b);
  g1 = -sn * lb + cs * cs / b;
  g2 = -cs * lb - 3.f * sn * cs / b - cs * cs * cs / (b * b);
  return static_cast<float>(i) * expf(cs * lb);
}

template <typename T>
__global__ void chain_ror_kernel(const LossArgs a) {
  pdl_entry();
  __shared__ float red[2][8];
  const int row = blockIdx.x;
  const int C = a.cols, M = a.chain;
  const int64_t E = static_cast<int64_t>(a.rows) * C;
  const float* f = a.F + static_cast<int64_t>(row) * C;
  const float* t = a.Yf + static_cast<int64_t>(row) * C;
  float w = 1.f, sg = 0.f;
  if (a.ex_w) w = a.ex_w[row];
  else if (a.eta_w) { sg = 1.f / (1.f + expf(-a.eta_w[row])); w = sg; }
  const float invC = 1.f / static_cast<float>(C);
  const float cw = w * a.inv_norm * 2.f * invC;
  const int64_t orow = static_cast<int64_t>(row) * a.ldo;
  float s2 = 0.f, s1 = 0.f;
  bool bad = false;
  float g1, g2;
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float* tp = a.tape + static_cast<int64_t>(row) * C + c;   // slot k at tp[k * E]
    if (a.ror == 1) {
      float y = f[c];
      for (int i = 1; i <= M; ++i) {
        tp[(i - 1) * E] = y;
        y = chain_step(i, y, g1, g2);
      }
      const float yM = y;
      const float r = yM - t[c];
      s2 += r * r;
      float yb = cw * r;
      for (int i = M; i >= 1; --i) {
        tp[(M + i - 1) * E] = yb;
        const float yi = i == M ? yM : tp[i * E];
        chain_step(i, tp[(i - 1) * E], g1, g2);
        yb *= yi * g1;
      }
      bad |= !isfinite(yM) || !isfinite(yb);
      if (a.dF) static_cast<T*>(a.dF)[orow + c] = to_t<T>(yb);
    } else {
      float ad = a.Fd[static_cast<int64_t>(row) * C + c];
      const float yM = chain_step(M, tp[(M - 1) * E], g1, g2);
      for (int i = 1; i <= M; ++i) {
        const float yi = i == M ? yM : tp[i * E];
        chain_step(i, tp[(i - 1) * E], g1, g2);
        float* slot = tp + (M + i - 1) * E;
        *slot = ad * *slot * yi * (g1 * g1 + g2);
        ad *= yi * g1;
      }
      const float r = yM - t[c];
      s1 += r * ad;
      float yh = cw * ad;
      for (int i = M; i >= 1; --i) {
        const float yi = i == M ? yM : tp[i * E];
        chain_step(i, tp[(i - 1) * E], g1, g2);
        yh = tp[(M + i - 1) * E] + yh * yi * g1;
      }
      bad |= !isfinite(yh);
      if (a.dFd) static_cast<T*>(a.dFd)[orow + c] = to_t<T>(yh);
    }
  }
  if (bad && a.status) atomicMax(a.status, DEV_NONFINITE);
  s2 = warp_sum(s2);
  s1 = warp_sum(s1);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { red[0][wid] = s2; red[1][wid] = s1; }
  __syncthreads();
  if (threadIdx.x == 0) {
    float l = 0.f, ld = 0.f;
    for (int k = 0; k < static_cast<int>(blockDim.x >> 5); ++k) { l += red[0][k]; ld += red[1][k]; }
    if (a.ror == 1) {
      if (a.l) a.l[row] = l * invC;
    } else {
      ld *= 2.f * invC;
      if (a.ld) a.ld[row] = ld;
      if (a.d_eta && a.eta_w) a.d_eta[row] = sg * (1.f - sg) * ld * a.inv_norm;
    }
  }
}

__global__ void sum_scaled_kernel(const float* __restrict__ x, int n, float scale,
                                  float* __restrict__ out) {
  pdl_entry();
  __shared__ float red[32];
  float s = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    v = warp_sum(v);
    if (threadIdx.x == 0) out[0] = v * scale;
  }
}

// Four consecutive parameters per thread, UPD_ELEMS per block, blocks assigned to layers by
// tab.tile0.  A layer whose offset and width are multiples of 4 moves them as float4 (and
// its operand copies as four-element stores in one row); others go element by element.
__device__ __forceinline__ void ld4(float (&x)[4], const float* p, int64_t k, bool vec, int cnt) {
  if (vec) {
    const float4 t = *reinterpret_cast<const float4*>(p + k);
    x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = j < cnt ? p[k + j] : 0.f;
  }
}

__device__ __forceinline__ void st4(float* p, int64_t k, const float (&x)[4], bool vec, int cnt) {
  if (vec) {
    *reinterpret_cast<float4*>(p + k) = make_float4(x[0], x[1], x[2], x[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < cnt) p[k + j] = x[j];
  }
}

template <typename T>
__device__ __forceinline__ void st_copy(T* W, int64_t e0, int r0, int dout, int din, int ldw,
                                        const float (&x)[4], bool vec, int cnt) {
  if (vec) {   // four elements of row r0
    if (r0 >= din) return;
    T* q = W + static_cast<int64_t>(r0) * ldw + (e0 - static_cast<int64_t>(r0) * dout);
    if constexpr (sizeof(T) == 2) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(x[0], x[1]);
      __nv_bfloat162 hi = __floats2bfloat162_rn(x[2], x[3]);
      uint2 v;
      v.x = *reinterpret_cast<uint32_t*>(&lo);
      v.y = *reinterpret_cast<uint32_t*>(&hi);
      *reinterpret_cast<uint2*>(q) = v;
    } else {
      *reinterpret_cast<float4*>(q) = make_float4(x[0], x[1], x[2], x[3]);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j >= cnt) break;
      const int64_t e = e0 + j;
      const int r = static_cast<int>(e / dout), c = static_cast<int>(e % dout);
      if (r < din) W[static_cast<int64_t>(r) * ldw + c] = to_t<T>(x[j]);
    }
  }
}

// f(mode, adam) of an update as types.
#pragma nv_exec_check_disable
template <class F>
__host__ __device__ __forceinline__ void with_update_mode(const LayerUpdArgs& a, F&& f) {
  using R = std::integral_constant<int, LU_ROLLOUT>;
  using A = std::integral_constant<int, LU_ADJOINT>;
  if (a.mode == LU_ROLLOUT && a.adam) f(R{}, std::true_type{});
  else if (a.mode == LU_ROLLOUT) f(R{}, std::false_type{});
  else if (a.mode == LU_ADJOINT && a.adam) f(A{}, std::true_type{});
  else if (a.mode == LU_ADJOINT) f(A{}, std::false_type{});
  else f(std::integral_constant<int, LU_CAST>{}, std::false_type{});
}

// Tiles blk .. blk + NQ - 1 of the update over the whole vector, by UPD_THREADS threads tid
// (red: one float a warp; sync: their barrier), whose loads are all issued before the first
// result is needed.  Memory traffic bounds it (about 85% of the copy bandwidth on vectors of
// 537 MB), so a vector that no later operation reads is not written and one that would be zeros
// is not read: u' where its operand copy serves the products, and the sum of the first
// learning-rate gradients.  One kernel per mode, so that each has the registers of its own
// vectors only, and its layer table read from constant memory (a per-thread copy of it in local
// memory cost more than the search for the layer): against one kernel for all modes, a call of
// 2 steps on eight 4096-wide layers with momentum and per-parameter rates 7.33 -> 6.80 ms.
template <typename T, int MODE, bool ADAM, int NQ, class Sync>
__device__ __forceinline__ void layer_update_block(const LayerTable& tab, const LayerUpdArgs& a,
                                                   int blk, int tid, float* red, Sync sync) {
  // the layer of the first tile: the last l with tile0[l] <= blk (binary search)
  int l = 0;
  {
    int hi = tab.n - 1;
    while (l < hi) {
      const int mid = (l + hi + 1) >> 1;
      if (blk >= tab.tile0[mid]) l = mid;
      else hi = mid - 1;
    }
  }
  struct Pos { int l, dout, cnt; bool vec; int64_t n, e0, k; };
  auto place = [&](int lay, int q) {
    Pos z;
    z.l = lay;
    z.dout = tab.dout[lay];
    z.n = static_cast<int64_t>(tab.rows[lay]) * z.dout;
    z.e0 = (static_cast<int64_t>(blk + q - tab.tile0[lay]) * UPD_THREADS + tid) * 4;
    z.cnt = static_cast<int>(z.n - z.e0 < 4 ? z.n - z.e0 : 4);
    z.vec = a.vec_ok && z.cnt == 4 && (tab.off[lay] & 3) == 0 && (z.dout & 3) == 0;
    z.k = tab.off[lay] + z.e0;
    return z;
  };
  const bool cast_w = (MODE == LU_ROLLOUT) || (MODE == LU_CAST && !a.cast_src_to_u) ||
                      (MODE == LU_ADJOINT && a.cast_src);
  const bool cast_u = (MODE == LU_CAST && a.cast_src_to_u) || (MODE == LU_ADJOINT && a.u_out);
  const bool need_lr = MODE == LU_ROLLOUT ||
                       (MODE == LU_ADJOINT && ((ADAM && a.adam_pre) || a.m_adj || a.u_out));
  constexpr bool plain = !ADAM;
  // Inputs of one tile: the rollout's theta, g, m, v; the adjoint's theta_bar, Hu and (plain)
  // m_adj, u_in, d_plr, cast_src; the cast's source.  The pointers may alias in place, so
  // every one of them is read before the tile's first store.
  struct In { float lr[4], x0[4], x1[4], x2[4], x3[4], x4[4], x5[4]; } in[NQ];
  int lay[NQ];
  bool on[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    if (q > 0)
      while (l + 1 < tab.n && blk + q >= tab.tile0[l + 1]) ++l;
    lay[q] = l;
    const Pos z = place(l, q);
    on[q] = z.e0 < z.n;
    In& i = in[q];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      i.lr[j] = i.x0[j] = i.x1[j] = i.x2[j] = i.x3[j] = i.x4[j] = i.x5[j] = 0.f;
    if (!on[q]) continue;
    if (a.lr.plr && need_lr) ld4(i.lr, a.lr.plr, z.k, z.vec, z.cnt);
    if (MODE == LU_ROLLOUT) {
      ld4(i.x0, a.theta, z.k, z.vec, z.cnt);
      ld4(i.x1, a.g, z.k, z.vec, z.cnt);
      if (a.m) ld4(i.x2, a.m, z.k, z.vec, z.cnt);
      if (ADAM && a.v) ld4(i.x3, a.v, z.k, z.vec, z.cnt);
    } else if (MODE == LU_ADJOINT) {
      ld4(i.x0, a.theta_bar, z.k, z.vec, z.cnt);
      if (a.Hu) ld4(i.x1, a.Hu, z.k, z.vec, z.cnt);
      if (plain && a.m_adj) ld4(i.x2, a.m_adj, z.k, z.vec, z.cnt);
      if (plain && a.u_out && a.u_in) ld4(i.x3, a.u_in, z.k, z.vec, z.cnt);
      if (plain && a.m_adj && a.d_plr && !a.plr_first) ld4(i.x4, a.d_plr, z.k, z.vec, z.cnt);
      if (plain && a.cast_src) ld4(i.x5, a.cast_src, z.k, z.vec, z.cnt);
    } else {
      ld4(i.x0, a.cast_src, z.k, z.vec, z.cnt);
    }
  }
  bool bad = false;
  float acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    acc[q] = 0.f;
    if (!on[q]) continue;
    const Pos z = place(lay[q], q);
    const int l = z.l, dout = z.dout, cnt = z.cnt, din = tab.din[l];
    const bool vec = z.vec;
    const int64_t n = z.n, e0 = z.e0, k = z.k;
    In& i = in[q];
    // the float32 tangent of an element that its operand copy serves (the quads of a vector
    // access lie in one row)
    const int r0 = n <= 0xffffffffLL
                       ? static_cast<int>(static_cast<uint32_t>(e0) / static_cast<uint32_t>(dout))
                       : static_cast<int>(e0 / dout);
    const bool u_kept = !(a.u_copy && vec && tab.U[l] && r0 < din);
    float vw[4] = {0.f, 0.f, 0.f, 0.f}, vu[4] = {0.f, 0.f, 0.f, 0.f};
    float lr[4];
    if (a.lr.plr && need_lr) {
#pragma unroll
      for (int j = 0; j < 4; ++j) lr[j] = expf(i.lr[j]);
    } else {
      const float l0 = a.lr.slr ? expf(a.lr.slr[0]) : a.lr.alpha;
#pragma unroll
      for (int j = 0; j < 4; ++j) lr[j] = l0;
    }
    if (MODE == LU_ROLLOUT) {
      const float(&th)[4] = i.x0, (&g)[4] = i.x1, (&m)[4] = i.x2, (&v)[4] = i.x3;
      float mn[4], vn[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (ADAM) {
          mn[j] = a.b1 * m[j] + (1.f - a.b1) * g[j];
          vn[j] = a.b2 * v[j] + (1.f - a.b2) * g[j] * g[j];
          vw[j] = th[j] - lr[j] * (mn[j] / a.c1) / (sqrtf(vn[j] / a.c2) + a.eps);
        } else {
          mn[j] = a.mu * m[j] + g[j];
          vn[j] = 0.f;
          vw[j] = th[j] - lr[j] * mn[j];
        }
        bad |= j < cnt && !isfinite(vw[j]);
      }
      st4(a.theta_out, k, vw, vec, cnt);
      if (a.m_out) st4(a.m_out, k, mn, vec, cnt);
      if (ADAM && a.v_out) st4(a.v_out, k, vn, vec, cnt);
    } else if (MODE == LU_ADJOINT) {
      float(&tb)[4] = i.x0, (&dp)[4] = i.x4;
      const float(&hu)[4] = i.x1, (&ma)[4] = i.x2, (&ui)[4] = i.x3;
      if (plain && a.cast_src) {
#pragma unroll
        for (int j = 0; j < 4; ++j) vw[j] = i.x5[j];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        tb[j] += hu[j];
        bad |= j < cnt && !isfinite(tb[j]);
      }
      st4(a.theta_bar_out ? a.theta_bar_out : a.theta_bar, k, tb, vec, cnt);
      float contrib[4] = {0.f, 0.f, 0.f, 0.f};
      bool have_contrib = false;
      if (ADAM && a.adam_pre) {
        // reverse of Adam step j from its outputs m1 = m_{j+1}, v1 = v_{j+1} (see LayerUpdArgs)
        float m1[4], v1[4], mp[4] = {0.f, 0.f, 0.f, 0.f};
        float mb[4] = {0.f, 0.f, 0.f, 0.f}, vb[4] = {0.f, 0.f, 0.f, 0.f};
        ld4(m1, a.m_adj, k, vec, cnt);
        ld4(v1, a.v_adj, k, vec, cnt);
        if (a.m_prev) ld4(mp, a.m_prev, k, vec, cnt);
        if (a.bar_in) {
          ld4(mb, a.mbar, k, vec, cnt);
          ld4(vb, a.vbar, k, vec, cnt);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float sq = sqrtf(v1[j] / a.c2);
          const float den = sq + a.eps;
          const float s = -lr[j] * tb[j];
          // at v = 0 (where m = g = 0) the sqrt term is 0
          const float Mb = mb[j] + s / (a.c1 * den);
          const float Vb = vb[j] - (sq > 0.f ? s * m1[j] / (a.c1 * den * den * 2.f * sq * a.c2) : 0.f);
          const float g = (m1[j] - a.b1 * mp[j]) / (1.f - a.b1);
          vu[j] = (1.f - a.b1) * Mb + 2.f * (1.f - a.b2) * g * Vb;
          mb[j] = a.b1 * Mb;
          vb[j] = a.b2 * Vb;
          contrib[j] = -lr[j] * (m1[j] / a.c1) / den * tb[j];
          bad |= j < cnt && !isfinite(vu[j]);
        }
        if (u_kept) st4(a.u_out, k, vu, vec, cnt);
        st4(a.mbar, k, mb, vec, cnt);
        st4(a.vbar, k, vb, vec, cnt);
        have_contrib = true;
      } else if (plain) {
        if (a.m_adj) {
#pragma unroll
          for (int j = 0; j < 4; ++j) contrib[j] = -lr[j] * ma[j] * tb[j];
          have_contrib = true;
        }
        if (a.u_out) {
#pragma unroll
          for (int j = 0; j < 4; ++j) vu[j] = a.mu * ui[j] - lr[j] * tb[j];
          if (u_kept) st4(a.u_out, k, vu, vec, cnt);
        }
      }
      if (have_contrib) {
        if (a.d_plr) {
          if (!plain && !a.plr_first) ld4(dp, a.d_plr, k, vec, cnt);
#pragma unroll
          for (int j = 0; j < 4; ++j) dp[j] += contrib[j];
          st4(a.d_plr, k, dp, vec, cnt);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[q] += j < cnt ? contrib[j] : 0.f;
        }
      }
      if (!plain && a.cast_src) ld4(vw, a.cast_src, k, vec, cnt);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) vu[j] = vw[j] = i.x0[j];
    }
    if (cast_w && tab.W[l]) st_copy<T>(static_cast<T*>(tab.W[l]), e0, r0, dout, din, tab.ldw[l], vw, vec, cnt);
    if (cast_u && tab.U[l]) st_copy<T>(static_cast<T*>(tab.U[l]), e0, r0, dout, din, tab.ldw[l], vu, vec, cnt);
  }
  if (bad && a.status) atomicMax(a.status, DEV_NONFINITE);
  if (a.partials) {   // one deterministic partial sum per tile (scalar log-lr)
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      if (blk + q >= tab.tile0[tab.n]) break;
      const float w = warp_sum(acc[q]);
      if ((tid & 31) == 0) red[tid >> 5] = w;
      sync();
      if (tid < 32) {
        float v = tid < UPD_THREADS / 32 ? red[tid] : 0.f;
        v = warp_sum(v);
        if (tid == 0) a.partials[blk + q] = v;
      }
      sync();   // red may be used again
    }
  }
}

// The table and the arguments stay in constant memory: indexed by a run-time layer, a by-value
// copy of them went to each thread's local memory.
template <typename T, int MODE, bool ADAM, int NQ>
__global__ void __launch_bounds__(UPD_THREADS) layer_update_kernel(
    const __grid_constant__ LayerTable tab, const __grid_constant__ LayerUpdArgs a) {
  pdl_entry();
  __shared__ float red[UPD_THREADS / 32];
  layer_update_block<T, MODE, ADAM, NQ>(tab, a, static_cast<int>(blockIdx.x) * NQ,
                                  static_cast<int>(threadIdx.x), red, [] { __syncthreads(); });
}

// Reverse-over-reverse, forward layer order: from dzbar (the adjoint of the backward's dz)
// and the stored derivatives D1 = phi'(z), D2 = phi''(z):
//   dabar = dzbar D1  (T, row-major [rows][ld]),  zpart = dzbar D2 da.
template <typename T>
__global__ void ror_fwd_elem_kernel(const float* __restrict__ dzbar, const float* __restrict__ D1,
                                    const float* __restrict__ D2, const float* __restrict__ dA,
                                    int rows, int cols, T* __restrict__ dab, int ld,
                                    float* __restrict__ zpart) {
  pdl_entry();
  const int c = blockIdx.x * TILE + threadIdx.x;
  for (int i = threadIdx.y; i < TILE; i += TROWS) {
    const int r = blockIdx.y * TILE + i;
    if (r < rows && c < cols) {
      const int64_t o = static_cast<int64_t>(r) * cols + c;
      zpart[o] = dzbar[o] * D2[o] * dA[o];
      dab[static_cast<int64_t>(r) * ld + c] = to_t<T>(dzbar[o] * D1[o]);
    }
  }
}

// Reverse-over-reverse, reverse layer order:  zbar = zpart + abar D1  (T, [rows][ld]).
template <typename T>
__global__ void ror_bwd_elem_kernel(const float* __restrict__ zpart,
                                    const float* __restrict__ abar, const float* __restrict__ D1,
                                    int rows, int cols, T* __restrict__ zb, int ld) {
  pdl_entry();
  const int c = blockIdx.x * TILE + threadIdx.x;
  for (int i = threadIdx.y; i < TILE; i += TROWS) {
    const int r = blockIdx.y * TILE + i;
    if (r < rows && c < cols) {
      const int64_t o = static_cast<int64_t>(r) * cols + c;
      zb[static_cast<int64_t>(r) * ld + c] = to_t<T>(zpart[o] + abar[o] * D1[o]);
    }
  }
}

__global__ void fill_kernel(float* p, int64_t n, float v) {
  pdl_entry();
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    p[i] = v;
}

// ---- small float32 models: a whole call as one block's program ---------------------------
// Every operation of a small MLP's call takes one block a fraction of a microsecond, and a
// launch of its own three: the launches, not the work, are what such a call costs.  The block
// walks the recorded operations in order with a barrier between them.  The call's workspace
// lives in the block's shared memory (pointers into the workspace are moved there when the
// program is read): from global memory, whose lines a store drops from L1, each operation
// waited two round trips to L2.  Each is the operation of the kernel it stands for: the loss
// and update share their device code, a GEMM is one output per thread with its products added
// in K order.  What is left is the instructions of one block: splitting K over lanes or more
// threads per block issued more of them and ran slower.
// 16-32-1 at B = 8, T = 4 (70 operations): meta-gradient 185 us as launches, 108 us with the
// workspace in global memory, 85 us; its Hessian-vector product 27 -> 17 us.
constexpr int SP_THREADS = 512, SP_GROUPS = SP_THREADS / UPD_THREADS;
static_assert(SP_THREADS >= kSmallOps && SP_THREADS >= kMaxLayers, "a thread per operation");

__device__ __forceinline__ void small_gemm(const GemmArgs& g) {
  const bool dual = (g.terms & (T_C1_A1B0 | T_C1_A0B1)) != 0;
  const int K = g.K, N = g.N, total = g.M * N;
  const int da = g.a_mn ? g.lda0 : 1, db = g.b_mn ? g.ldb0 : 1;   // the pairs share a stride
  const int ra = g.a_mn ? 1 : g.lda0, rb = g.b_mn ? 1 : g.ldb0;
  for (int o = threadIdx.x; o < total; o += SP_THREADS) {
    const int m = o / N, n = o - m * N;
    auto dot = [&](const void* A, const void* B, float acc) {
      const float* a = static_cast<const float*>(A) + m * ra;
      const float* b = static_cast<const float*>(B) + n * rb;
#pragma unroll 8
      for (int k = 0; k < K; ++k, a += da, b += db) acc = fmaf(*a, *b, acc);
      return acc;
    };
    float acc0 = 0.f, acc1 = 0.f;
    if (g.terms & T_C0_A0B0) acc0 = dot(g.A0, g.B0, acc0);
    if (g.terms & T_C0_A1B0) acc0 = dot(g.A1, g.B0, acc0);
    if (g.terms & T_C0_A0B1) acc0 = dot(g.A0, g.B1, acc0);
    if (g.terms & T_C0_A1B1) acc0 = dot(g.A1, g.B1, acc0);
    if (g.terms & T_C1_A1B0) acc1 = dot(g.A1, g.B0, acc1);
    if (g.terms & T_C1_A0B1) acc1 = dot(g.A0, g.B1, acc1);
    const EpiOut r = epi_eval(g.epi, m, n, acc0, acc1, g.bias0, g.bias1, dual);
    if (g.C0) g.C0[m * g.ldc0 + n] = r.c0;
    if (g.C1) g.C1[m * g.ldc1 + n] = r.c1;
    if (g.epi.mode != EPI_STORE) {
      if (g.epi.A) static_cast<float*>(g.epi.A)[m * g.epi.lda + n] = r.o0;
      if (dual && g.epi.Ad) static_cast<float*>(g.epi.Ad)[m * g.epi.lda + n] = r.o1;
    }
  }
}

// Copy n bytes (a multiple of 16) of the kernel parameters or of global memory to or from
// shared memory, 16 bytes per thread.  Through generic addresses: as indexed constant loads
// the parameters would come one word at a time.
__device__ __forceinline__ void copy16(void* dst, const void* src, int n) {
  for (int o = threadIdx.x * 16; o < n; o += SP_THREADS * 16) {
    uint4 v;
    asm volatile("ld.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(static_cast<const char*>(src) + o));
    *reinterpret_cast<uint4*>(static_cast<char*>(dst) + o) = v;
  }
}

struct MovePtr {   // a pointer into the workspace -> the same place in its shared-memory image
  char* base; char* image; int64_t bytes;
  template <typename P>
  __device__ __forceinline__ void operator()(P*& p) const {
    char* q = reinterpret_cast<char*>(const_cast<void*>(static_cast<const void*>(p)));
    if (q >= base && q < base + bytes) p = reinterpret_cast<P*>(image + (q - base));
  }
};

__device__ __forceinline__ void move_op(SmallOp& op, const MovePtr& mv) {
  switch (op.kind) {
    case SMALL_GEMM: {
      GemmArgs& g = *reinterpret_cast<GemmArgs*>(op.data);
      mv(g.A0); mv(g.A1); mv(g.B0); mv(g.B1); mv(g.C0); mv(g.C1); mv(g.bias0); mv(g.bias1);
      mv(g.epi.A); mv(g.epi.Ad); mv(g.epi.Z); mv(g.epi.Zd);
      break;
    }
    case SMALL_LOSS: {
      LossArgs& a = *reinterpret_cast<LossArgs*>(op.data);
      mv(a.F); mv(a.Fd); mv(a.Yf); mv(a.Yi); mv(a.eta_w); mv(a.ex_w); mv(a.l); mv(a.ld);
      mv(a.d_eta); mv(a.dF); mv(a.dFd);
      break;
    }
    case SMALL_UPDATE: {
      LayerUpdArgs& a = *reinterpret_cast<LayerUpdArgs*>(op.data);
      mv(a.cast_src); mv(a.theta); mv(a.m); mv(a.g); mv(a.theta_out); mv(a.m_out); mv(a.theta_bar);
      mv(a.Hu); mv(a.m_adj); mv(a.u_in); mv(a.u_out); mv(a.d_plr); mv(a.partials); mv(a.lr.plr);
      mv(a.lr.slr); mv(a.v); mv(a.v_out); mv(a.v_adj); mv(a.m_prev); mv(a.mbar); mv(a.vbar);
      break;
    }
    case SMALL_COPY: {
      SmallCopy& c = *reinterpret_cast<SmallCopy*>(op.data);
      mv(c.dst); mv(c.src);
      break;
    }
    case SMALL_SUM: {
      SmallSum& a = *reinterpret_cast<SmallSum*>(op.data);
      mv(a.x); mv(a.out);
      break;
    }
    default: {
      SmallRor& a = *reinterpret_cast<SmallRor*>(op.data);
      mv(a.x); mv(a.D1); mv(a.D2); mv(a.dA); mv(a.zpart); mv(a.out);
    }
  }
}

__global__ void __launch_bounds__(SP_THREADS, 1) small_program_kernel(
    const __grid_constant__ SmallProgram prog) {
  __shared__ float red[SP_THREADS / 32];
  extern __shared__ __align__(256) char image[];   // the workspace, then the program
  SmallProgram& sp = *reinterpret_cast<SmallProgram*>(image + prog.ws_bytes);
  LayerTable& tab = sp.tab;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, grp = tid / UPD_THREADS;
  const int n = prog.n;
  copy16(&sp, &prog, static_cast<int>(offsetof(SmallProgram, op)) + n * static_cast<int>(sizeof(SmallOp)));
  __syncthreads();
  const MovePtr mv{static_cast<char*>(prog.ws), image, prog.ws_bytes};
  if (tid < n) move_op(sp.op[tid], mv);
  if (tid < tab.n) { mv(tab.W[tid]); mv(tab.U[tid]); }
  pdl_entry();
  if (prog.load) copy16(image, prog.ws, prog.ws_bytes);   // left there by the call's last program
  __syncthreads();
  for (int i = 0; i < n; ++i) {
    const SmallOp& op = sp.op[i];
    switch (op.kind) {
      case SMALL_GEMM: small_gemm(*reinterpret_cast<const GemmArgs*>(op.data)); break;
      case SMALL_LOSS: {
        const LossArgs& a = *reinterpret_cast<const LossArgs*>(op.data);
        for (int row = warp; row < a.rows; row += SP_THREADS / 32) loss_seed_row<float>(a, row, lane);
        break;
      }
      case SMALL_UPDATE: {   // a group of UPD_THREADS threads per block of the update
        const LayerUpdArgs& a = *reinterpret_cast<const LayerUpdArgs*>(op.data);
        auto tiles = [&](auto mode, auto adam) __attribute__((always_inline)) {
          for (int b = grp; b < tab.tile0[tab.n]; b += SP_GROUPS)
            layer_update_block<float, decltype(mode)::value, decltype(adam)::value, 1>(
                tab, a, b, tid % UPD_THREADS, red + grp * (UPD_THREADS / 32),
                [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(UPD_THREADS) : "memory"); });
        };
        with_update_mode(a, tiles);
        break;
      }
      case SMALL_COPY: {   // rows x cols floats; a null source writes value
        const SmallCopy& c = *reinterpret_cast<const SmallCopy*>(op.data);
        for (int e = tid; e < c.rows * c.cols; e += SP_THREADS) {
          const int r = e / c.cols, x = e % c.cols;
          c.dst[r * c.ldd + x] = c.src ? c.src[r * c.lds + x] : c.value;
        }
        break;
      }
      case SMALL_SUM: {
        const SmallSum& a = *reinterpret_cast<const SmallSum*>(op.data);
        float v = 0.f;
        for (int e = tid; e < a.n; e += SP_THREADS) v += a.x[e];
        v = warp_sum(v);
        if (lane == 0) red[warp] = v;
        __syncthreads();
        if (warp == 0) {
          v = warp_sum(lane < SP_THREADS / 32 ? red[lane] : 0.f);
          if (lane == 0) a.out[0] = v * a.scale;
        }
        break;
      }
      case SMALL_ROR_FWD: {
        const SmallRor& a = *reinterpret_cast<const SmallRor*>(op.data);
        for (int e = tid; e < a.rows * a.cols; e += SP_THREADS) {
          const int at = e / a.cols * a.ld + e % a.cols;
          a.zpart[e] = a.x[e] * a.D2[e] * a.dA[e];
          a.out[at] = a.x[e] * a.D1[e];
        }
        break;
      }
      case SMALL_ROR_BWD: {
        const SmallRor& a = *reinterpret_cast<const SmallRor*>(op.data);
        for (int e = tid; e < a.rows * a.cols; e += SP_THREADS) {
          const int at = e / a.cols * a.ld + e % a.cols;
          a.out[at] = a.zpart[e] + a.x[e] * a.D1[e];
        }
        break;
      }
    }
    __syncthreads();
  }
  if (prog.save) copy16(prog.ws, image, prog.ws_bytes);
}

}  // namespace

cudaError_t small_program(const SmallProgram& prog, cudaStream_t s) {
  if (prog.n == 0) return cudaSuccess;
  static PerDeviceOnce attr_once;
  const cudaError_t e = attr_once.run([](int&) {
    return cudaFuncSetAttribute(small_program_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kSmallImage + static_cast<int>(sizeof(SmallProgram)));
  });
  if (e != cudaSuccess) return e;
  return launch_k(small_program_kernel, dim3(1), dim3(SP_THREADS),
                  prog.ws_bytes + sizeof(SmallProgram), s, prog);
}

template <typename T>
void fill_cols(const ColFill& f, int rows, cudaStream_t s) {
  if (f.n == 0 || rows <= 0) return;
  launch_k(fill_cols_kernel<T>, dim3((rows + 255) / 256, f.n), dim3(256), 0, s, f, rows);
}

template <typename T>
void loss_seed(const LossArgs& a, cudaStream_t s) {
  if (!loss_ready(a)) return;
  // sixteen-byte access where every row is a multiple of it
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const bool vec = !(a.cols & 3) && !(a.ldo & 3) && al(a.F) && al(a.Fd) && al(a.Yf) && al(a.dF) && al(a.dFd);
  const dim3 rows(a.rows), block(LB_THREADS);
  if (a.loss == 2) {
    if (a.ror && a.tape && a.chain > 0 && (a.ror == 1 || a.Fd)) {
      launch_k(chain_ror_kernel<T>, rows, dim3(256), 0, s, a);
    } else if (a.Fd) {
      if (vec) launch_k(chain_loss_kernel<T, true, 4>, rows, block, 0, s, a);
      else launch_k(chain_loss_kernel<T, true, 1>, rows, block, 0, s, a);
    } else {
      if (vec) launch_k(chain_loss_kernel<T, false, 4>, rows, block, 0, s, a);
      else launch_k(chain_loss_kernel<T, false, 1>, rows, block, 0, s, a);
    }
    return;
  }
  if (a.cols > kBlockLossCols) {
    if (vec) launch_k(loss_seed_block_kernel<T, 4>, rows, block, 0, s, a);
    else launch_k(loss_seed_block_kernel<T, 1>, rows, block, 0, s, a);
    return;
  }
  const int warps = 8;
  launch_k(loss_seed_kernel<T>, dim3((a.rows + warps - 1) / warps), dim3(warps * 32), 0, s, a);
}

void sum_scaled(const float* x, int n, float scale, float* out, cudaStream_t s) {
  launch_k(sum_scaled_kernel, dim3(1), dim3(1024), 0, s, x, n, scale, out);
}

// float4 access only when every vector the call touches is 16-byte aligned (caller pointers
// such as theta or eta + offset need not be)
bool update_vec_ok(const LayerUpdArgs& a) {
  uintptr_t any = 0;
  for (const void* p : {static_cast<const void*>(a.cast_src), static_cast<const void*>(a.theta),
                        static_cast<const void*>(a.m), static_cast<const void*>(a.g),
                        static_cast<const void*>(a.theta_out), static_cast<const void*>(a.m_out),
                        static_cast<const void*>(a.theta_bar), static_cast<const void*>(a.theta_bar_out),
                        static_cast<const void*>(a.Hu),
                        static_cast<const void*>(a.m_adj), static_cast<const void*>(a.u_in),
                        static_cast<const void*>(a.u_out), static_cast<const void*>(a.d_plr),
                        static_cast<const void*>(a.lr.plr), static_cast<const void*>(a.v),
                        static_cast<const void*>(a.v_out), static_cast<const void*>(a.v_adj),
                        static_cast<const void*>(a.m_prev), static_cast<const void*>(a.mbar),
                        static_cast<const void*>(a.vbar)})
    any |= reinterpret_cast<uintptr_t>(p);
  return (any & 15) == 0;
}

template <typename T>
void layer_update(const LayerTable& tab, const LayerUpdArgs& args, cudaStream_t s) {
  const int blocks = tab.tile0[tab.n];
  if (blocks <= 0) return;
  LayerUpdArgs a = args;
  a.vec_ok = update_vec_ok(a);
  // A cast has one load a tile, so a block takes four tiles (a Hessian-vector product with 92
  // million parameters: 2407 us with one, 2365 with four); the other modes have up to
  // six and lose more to the registers of a second tile (8 x 4096 layers: rollout 6.83 -> 6.98
  // ms a call with two, adjoint -> 7.28).
  with_update_mode(a, [&](auto mode, auto adam) {
    constexpr int MODE = decltype(mode)::value, NQ = MODE == LU_CAST ? 4 : 1;
    launch_k(layer_update_kernel<T, MODE, decltype(adam)::value, NQ>,
             dim3((blocks + NQ - 1) / NQ), dim3(UPD_THREADS), 0, s, tab, a);
  });
}

template <typename T>
void ror_fwd_elem(const float* dzbar, const float* D1, const float* D2, const float* dA, int rows,
                  int cols, T* dab, int ld, float* zpart, cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return;
  dim3 grid((cols + TILE - 1) / TILE, (rows + TILE - 1) / TILE);
  launch_k(ror_fwd_elem_kernel<T>, dim3(grid), dim3(TILE, TROWS), 0, s, dzbar, D1, D2, dA, rows,
           cols, dab, ld, zpart);
}

template <typename T>
void ror_bwd_elem(const float* zpart, const float* abar, const float* D1, int rows, int cols,
                  T* zb, int ld, cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return;
  dim3 grid((cols + TILE - 1) / TILE, (rows + TILE - 1) / TILE);
  launch_k(ror_bwd_elem_kernel<T>, dim3(grid), dim3(TILE, TROWS), 0, s, zpart, abar, D1, rows,
           cols, zb, ld);
}

void fill(float* p, int64_t n, float v, cudaStream_t s) {
  if (n <= 0) return;
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  launch_k(fill_kernel, dim3(static_cast<int>(b)), dim3(256), 0, s, p, n, v);
}

#define MF_INST(T)                                                                 \
  template void fill_cols<T>(const ColFill&, int, cudaStream_t);                  \
  template void loss_seed<T>(const LossArgs&, cudaStream_t);                      \
  template void layer_update<T>(const LayerTable&, const LayerUpdArgs&, cudaStream_t);        \
  template void ror_fwd_elem<T>(const float*, const float*, const float*, const float*, int, int, \
                                T*, int, float*, cudaStream_t);                                  \
  template void ror_bwd_elem<T>(const float*, const float*, const float*, int, int, T*, int,     \
                                cudaStream_t);
MF_INST(float)
MF_INST(__nv_bfloat16)
#undef MF_INST

}  // namespace mf
