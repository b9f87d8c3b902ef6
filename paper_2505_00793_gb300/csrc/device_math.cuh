// Device helpers shared by the GEMM epilogues and the elementwise kernels.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include "internal.h"

namespace mf {

template <typename T> __device__ __forceinline__ T to_t(float x);
template <> __device__ __forceinline__ float to_t<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 to_t<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

// phi, phi', phi'' of the hidden activations.
//   tanh:  phi' = 1 - t^2,                     phi'' = -2 t (1 - t^2)
//   GELU:  phi = x Phi(x), phi' = Phi + x pdf,  phi'' = pdf (2 - x^2)
//   SiLU:  phi = x s(x),  phi' = s (1 + x (1 - s)),  phi'' = s (1 - s) (2 + x (1 - 2 s))
__device__ __forceinline__ void act_eval(int act, float z, float& f, float& d1, float& d2) {
  switch (act) {
    case ACT_TANH: {
      const float t = tanhf(z);
      f = t; d1 = 1.f - t * t; d2 = -2.f * t * d1;
      break;
    }
    case ACT_GELU: {
      const float cdf = 0.5f * (1.f + erff(z * 0.70710678118654752f));
      const float pdf = 0.39894228040143268f * expf(-0.5f * z * z);
      f = z * cdf; d1 = cdf + z * pdf; d2 = pdf * (2.f - z * z);
      break;
    }
    case ACT_SILU: {
      const float sg = 1.f / (1.f + expf(-z));
      f = z * sg; d1 = sg * (1.f + z * (1.f - sg));
      d2 = sg * (1.f - sg) * (2.f + z * (1.f - 2.f * sg));
      break;
    }
    default:
      f = z; d1 = 1.f; d2 = 0.f;
  }
}

// Per-element epilogue of a dual GEMM (shared by the tensor-core and SIMT kernels).
//  EPI_STORE:   C0 = acc0 + bias0, C1 = acc1 + bias1.
//  EPI_ACT_FWD: z = acc0 + bias0, z' = acc1 + bias1 ->
//               a = phi(z), a' = phi'(z) z'  -> A, Ad (row-major), and what the backward pass
//               needs of z, in place of z itself: phi'(z) -> C0 and, where C1 is given,
//               phi''(z) z' (dual) or phi''(z) (primal, GemmArgs::keep_d2) -> C1, float32.  The
//               activation is evaluated once per element and pass instead of again in the
//               backward.
//  EPI_ACT_BWD: da = acc0, da' = acc1, the stored derivatives read from Z, Zd ->
//               dz = Z da, dz' = Zd da + Z da'  -> A, Ad.
struct EpiOut {
  float c0, c1;     // float32 outputs for C0 / C1
  float o0, o1;     // values for A / Ad
};

__device__ __forceinline__ EpiOut epi_bwd(float acc0, float acc1, float d1, float e, bool dual) {
  EpiOut r;
  r.c0 = acc0; r.c1 = acc1;
  r.o0 = d1 * acc0;
  r.o1 = dual ? e * acc0 + d1 * acc1 : 0.f;
  return r;
}

// f, d1, d2 = phi, phi', phi'' at z
__device__ __forceinline__ EpiOut epi_fwd(float f, float d1, float d2, float zd, bool dual) {
  EpiOut r;
  r.c0 = d1;
  r.c1 = dual ? d2 * zd : d2;
  r.o0 = f;
  r.o1 = dual ? d1 * zd : 0.f;
  return r;
}

__device__ __forceinline__ EpiOut epi_eval(const EpiParams& e, int m, int n, float acc0,
                                           float acc1, const float* bias0, const float* bias1,
                                           bool dual) {
  if (e.mode == EPI_ACT_BWD) {
    const int64_t at = static_cast<int64_t>(m) * e.ldz + n;
    return epi_bwd(acc0, acc1, e.Z[at], dual ? e.Zd[at] : 0.f, dual);
  }
  const float z = acc0 + (bias0 ? bias0[n] : 0.f);
  const float zd = acc1 + (bias1 ? bias1[n] : 0.f);
  if (e.mode == EPI_ACT_FWD) {
    float f, d1, d2;
    act_eval(e.act, z, f, d1, d2);
    return epi_fwd(f, d1, d2, zd, dual);
  }
  EpiOut r;
  r.c0 = z; r.c1 = zd;
  r.o0 = r.o1 = 0.f;
  return r;
}

// Compile-time specialisations of act_eval / epi_eval (one activation, one epilogue mode per
// kernel instance: the per-element code stays small).
template <int ACT>
__device__ __forceinline__ void act_eval_t(float z, float& f, float& d1, float& d2) {
  if constexpr (ACT == ACT_TANH) {
    const float t = tanhf(z);
    f = t; d1 = 1.f - t * t; d2 = -2.f * t * d1;
  } else if constexpr (ACT == ACT_GELU) {
    const float cdf = 0.5f * (1.f + erff(z * 0.70710678118654752f));
    const float pdf = 0.39894228040143268f * expf(-0.5f * z * z);
    f = z * cdf; d1 = cdf + z * pdf; d2 = pdf * (2.f - z * z);
  } else if constexpr (ACT == ACT_SILU) {
    const float sg = 1.f / (1.f + expf(-z));
    f = z * sg; d1 = sg * (1.f + z * (1.f - sg));
    d2 = sg * (1.f - sg) * (2.f + z * (1.f - 2.f * sg));
  } else {
    f = z; d1 = 1.f; d2 = 0.f;
  }
}

// The per-element arithmetic of epi_eval_t on values already loaded: x0, x1 the stored
// derivatives (EPI_ACT_BWD); b0, b1 the biases (0 when absent).
template <int MODE, int ACT>
__device__ __forceinline__ EpiOut epi_core_t(float acc0, float acc1, float x0, float x1,
                                             float b0, float b1, bool dual) {
  if constexpr (MODE == EPI_ACT_BWD) return epi_bwd(acc0, acc1, x0, x1, dual);
  const float z = acc0 + b0;
  const float zd = acc1 + b1;
  if constexpr (MODE == EPI_ACT_FWD) {
    float f, d1, d2;
    act_eval_t<ACT>(z, f, d1, d2);
    return epi_fwd(f, d1, d2, zd, dual);
  }
  EpiOut r;
  r.c0 = z; r.c1 = zd;
  r.o0 = r.o1 = 0.f;
  return r;
}

template <int MODE, int ACT>
__device__ __forceinline__ EpiOut epi_eval_t(const EpiParams& e, int m, int n, float acc0,
                                             float acc1, const float* bias0,
                                             const float* bias1, bool dual) {
  if constexpr (MODE == EPI_ACT_BWD) {
    const float z = e.Z[static_cast<int64_t>(m) * e.ldz + n];
    const float zd = dual ? e.Zd[static_cast<int64_t>(m) * e.ldz + n] : 0.f;
    return epi_core_t<MODE, ACT>(acc0, acc1, z, zd, 0.f, 0.f, dual);
  } else {
    return epi_core_t<MODE, ACT>(acc0, acc1, 0.f, 0.f, bias0 ? bias0[n] : 0.f,
                                 bias1 ? bias1[n] : 0.f, dual);
  }
}

}  // namespace mf
