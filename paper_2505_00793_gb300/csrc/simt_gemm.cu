// Float32 dual GEMM on the CUDA cores, for the float32-precision path (results checked at
// 1e-4 relative error, below what bf16 or tf32 operands allow).  Same term semantics and
// fused epilogues as the tensor-core kernel: C_j = sum of selected X Y^T products, then the
// per-element epilogue of device_math.cuh.
//
// What bounds it: the FMA pipes (128 per clock and SM) for large products, the latency of a
// short chain of loads for the small ones that fill a meta-gradient of a small model.
//  * Every operand a product mask uses is staged once per K block and all its terms run from
//    that stage, so a dual product reads four tiles for three products.
//  * Tiles come through cp.async in a four-stage ring, four-byte copies that transpose a
//    K-major operand on the way and sixteen-byte ones for an MN-major operand, both
//    coalesced; shared memory holds every operand as [k][row].
//  * A lane owns 8 x TN outputs per accumulator; products are packed two rows at a time
//    (fma.rn.f32x2), each lane of the pair rounding like fmaf.
//  * Three tiles: 128 x 128 (8 warps), 64 x 64 (two groups of 4 warps that split each K
//    block) and 32 x 32 (8 warps that split each K block), and a split of K over a cluster
//    of up to 8 CTAs whose partial tiles meet in distributed shared memory; the sums run in
//    a fixed order, so results are deterministic.
// Measured against one 64 x 64 tile per block that ran a mask's terms one after the other
// from single-buffered tiles: the layers of a 784-1023-1023-500-10 Hessian-vector
// product at 500 rows 8.31 -> 0.59 ms, four training steps of a 4 x 256 transformer
// (1024 tokens) 65.8 -> 4.8 ms; large products run at 38-52 TFLOP/s (4096x4096x1024: the
// FMA pipes active 71% of the time) where they ran at 2.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "device_math.cuh"
#include "internal.h"
#include "launch.cuh"

namespace mf {
namespace {

constexpr int PAD = 4;       // floats after each k row of a staged tile
constexpr int STAGES = 4;

struct SimtParams {
  int M, N, K, tiles_n, split;
  unsigned terms;
  const float* A[2]; int lda[2];
  const float* B[2]; int ldb[2];
  int a_mn, b_mn;                  // MN-major operands: X[row][k] at k * ld + row
  int a_vec, b_vec;                // MN-major rows may be copied 16 bytes at a time
  float* C[2]; int ldc[2]; const float* bias[2];
  int c_vec, e_vec;                // C0/C1 and A/Ad rows may be stored as float4
  EpiParams epi;
  int64_t bsA[2], bsB[2], bsC[2];  // batch strides (blockIdx.z / split = batch index)
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp4(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(dst)), "l"(src),
               "r"(ok ? 4 : 0));
}
__device__ __forceinline__ void cp16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
               "r"(bytes));
}
__device__ __forceinline__ uint64_t dup2(float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(b));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t& c, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ float4 ld_remote4(uint32_t addr, uint32_t rank) {
  uint32_t ra;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(ra)
               : "memory");
  return v;
}

// Rows [r0, r0 + R) x K block [k0, k0 + BK) of one operand into S[k][R + PAD], zero outside
// the operand (rows at or past `rows`, k at or past `K`).
template <int R, int BK, int THREADS>
__device__ __forceinline__ void stage_tile(float* S, const float* X, int ld, bool mn, bool vec,
                                           int r0, int rows, int k0, int K) {
  constexpr int LDS = R + PAD;
  if (!mn) {
#pragma unroll
    for (int i = threadIdx.x; i < R * BK; i += THREADS) {
      const int k = i % BK, r = i / BK;
      const bool ok = r0 + r < rows && k0 + k < K;
      cp4(S + k * LDS + r, ok ? X + static_cast<int64_t>(r0 + r) * ld + k0 + k : X, ok);
    }
  } else if (vec) {
#pragma unroll
    for (int i = threadIdx.x; i < R / 4 * BK; i += THREADS) {
      const int r = i % (R / 4) * 4, k = i / (R / 4);
      const int left = rows - r0 - r;
      const bool ok = left > 0 && k0 + k < K;
      cp16(S + k * LDS + r, ok ? X + static_cast<int64_t>(k0 + k) * ld + r0 + r : X,
           !ok ? 0 : left >= 4 ? 16 : left * 4);
    }
  } else {
#pragma unroll
    for (int i = threadIdx.x; i < R * BK; i += THREADS) {
      const int r = i % R, k = i / R;
      const bool ok = r0 + r < rows && k0 + k < K;
      cp4(S + k * LDS + r, ok ? X + static_cast<int64_t>(k0 + k) * ld + r0 + r : X, ok);
    }
  }
}

// WM x WN warps of 32 x (8 TN) outputs each, KS such groups that split every K block of BK.
// TERMS: the product mask (T_ALL: taken from p.terms at run time).
template <int WM, int WN, int TN, int KS, int BK, unsigned TERMS>
struct Cfg {
  static constexpr int BM = 32 * WM, BN = 8 * TN * WN, THREADS = 32 * WM * WN * KS;
  static constexpr int NACC = (TERMS & (T_C1_A1B0 | T_C1_A0B1)) ? 2 : 1;
  static constexpr bool A0 = TERMS & (T_C0_A0B0 | T_C0_A0B1 | T_C1_A0B1);
  static constexpr bool A1 = TERMS & (T_C0_A1B0 | T_C1_A1B0 | T_C0_A1B1);
  static constexpr bool B0 = TERMS & (T_C0_A0B0 | T_C0_A1B0 | T_C1_A1B0);
  static constexpr bool B1 = TERMS & (T_C0_A0B1 | T_C1_A0B1 | T_C0_A1B1);
  static constexpr int TA = BK * (BM + PAD), TB = BK * (BN + PAD);   // floats per staged tile
  static constexpr int OA1 = A0 ? TA : 0, OB0 = OA1 + (A1 ? TA : 0), OB1 = OB0 + (B0 ? TB : 0);
  static constexpr int STAGE = OB1 + (B1 ? TB : 0);
  static constexpr int LDT = BN + PAD;                               // partial tile rows
  static constexpr int TILE = NACC * BM * LDT;
  static constexpr int SMEM = (STAGES * STAGE > KS * TILE ? STAGES * STAGE : KS * TILE) * 4;
};

template <int WM, int WN, int TN, int KS, int BK, unsigned TERMS>
__global__ void __launch_bounds__(32 * WM * WN * KS)
    simt_dual_gemm_kernel(const __grid_constant__ SimtParams p) {
  using C = Cfg<WM, WN, TN, KS, BK, TERMS>;
  constexpr int BM = C::BM, BN = C::BN, THREADS = C::THREADS, NACC = C::NACC;
  extern __shared__ __align__(16) float sm[];
  const unsigned terms = TERMS == T_ALL ? p.terms : TERMS;
  const int S = p.split, rank = S > 1 ? static_cast<int>(cta_rank()) : 0;
  const int64_t bz = blockIdx.z / S;
  const int m0 = static_cast<int>(blockIdx.x) / p.tiles_n * BM;
  const int n0 = static_cast<int>(blockIdx.x) % p.tiles_n * BN;
  const float* A0 = p.A[0] + bz * p.bsA[0];
  const float* A1 = p.A[1] + bz * p.bsA[1];
  const float* B0 = p.B[0] + bz * p.bsB[0];
  const float* B1 = p.B[1] + bz * p.bsB[1];
  const bool useA0 = C::A0 && (TERMS != T_ALL || (terms & (T_C0_A0B0 | T_C0_A0B1 | T_C1_A0B1)));
  const bool useA1 = C::A1 && (TERMS != T_ALL || (terms & (T_C0_A1B0 | T_C1_A1B0 | T_C0_A1B1)));
  const bool useB0 = C::B0 && (TERMS != T_ALL || (terms & (T_C0_A0B0 | T_C0_A1B0 | T_C1_A1B0)));
  const bool useB1 = C::B1 && (TERMS != T_ALL || (terms & (T_C0_A0B1 | T_C1_A0B1 | T_C0_A1B1)));
  const int nkb = (p.K + BK - 1) / BK;
  const int kb0 = static_cast<int>(static_cast<int64_t>(nkb) * rank / S);
  const int kb1 = static_cast<int>(static_cast<int64_t>(nkb) * (rank + 1) / S);

  auto load = [&](int kb) {
    if (kb < kb1) {
      float* st = sm + (kb - kb0) % STAGES * C::STAGE;
      const int k0 = kb * BK;
      if (useA0) stage_tile<BM, BK, THREADS>(st, A0, p.lda[0], p.a_mn, p.a_vec, m0, p.M, k0, p.K);
      if (useA1) stage_tile<BM, BK, THREADS>(st + C::OA1, A1, p.lda[1], p.a_mn, p.a_vec, m0, p.M, k0, p.K);
      if (useB0) stage_tile<BN, BK, THREADS>(st + C::OB0, B0, p.ldb[0], p.b_mn, p.b_vec, n0, p.N, k0, p.K);
      if (useB1) stage_tile<BN, BK, THREADS>(st + C::OB1, B1, p.ldb[1], p.b_mn, p.b_vec, n0, p.N, k0, p.K);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // lane -> rows lr*4 + {0..3, 16..19} of the warp's 32, columns lc*4 + {0..3} (and + 32)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slice = warp / (WM * WN), wm = warp % (WM * WN) / WN, wn = warp % WN;
  const int lr = lane >> 3, lc = lane & 7;
  const int ra = wm * 32 + lr * 4, cb = wn * 8 * TN + lc * 4;
  uint64_t acc[NACC][4][TN] = {};

  pdl_entry();
#pragma unroll
  for (int i = 0; i < STAGES - 1; ++i) load(kb0 + i);
  for (int kb = kb0; kb < kb1; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();
    load(kb + STAGES - 1);   // into the stage every thread finished reading before the barrier
    const float* st = sm + (kb - kb0) % STAGES * C::STAGE;
#pragma unroll
    for (int q = 0; q < BK / KS; ++q) {
      const int kk = slice * (BK / KS) + q;
      uint64_t a0[4], a1[4];
      float b0[TN], b1[TN];
      auto lda = [&](uint64_t (&a)[4], int off) {
        const float* s = st + off + kk * (BM + PAD) + ra;
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(s);
        const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(s + 16);
        a[0] = x.x; a[1] = x.y; a[2] = y.x; a[3] = y.y;
      };
      auto ldb = [&](float (&b)[TN], int off) {
        const float* s = st + off + kk * (BN + PAD) + cb;
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
          const float4 v = *reinterpret_cast<const float4*>(s + j * 8);
          b[j] = v.x; b[j + 1] = v.y; b[j + 2] = v.z; b[j + 3] = v.w;
        }
      };
      auto mul = [&](int j, const uint64_t (&a)[4], const float (&b)[TN]) {
#pragma unroll
        for (int n = 0; n < TN; ++n) {
          const uint64_t bb = dup2(b[n]);
#pragma unroll
          for (int i = 0; i < 4; ++i) fma2(acc[j][i][n], a[i], bb);
        }
      };
      if (useA0) lda(a0, 0);
      if (useA1) lda(a1, C::OA1);
      if (useB0) ldb(b0, C::OB0);
      if (useB1) ldb(b1, C::OB1);
      if ((TERMS & T_C0_A0B0) && (terms & T_C0_A0B0)) mul(0, a0, b0);
      if ((TERMS & T_C0_A1B0) && (terms & T_C0_A1B0)) mul(0, a1, b0);
      if ((TERMS & T_C0_A0B1) && (terms & T_C0_A0B1)) mul(0, a0, b1);
      if ((TERMS & T_C0_A1B1) && (terms & T_C0_A1B1)) mul(0, a1, b1);
      if ((TERMS & T_C1_A1B0) && (terms & T_C1_A1B0)) mul(NACC - 1, a1, b0);
      if ((TERMS & T_C1_A0B1) && (terms & T_C1_A0B1)) mul(NACC - 1, a0, b1);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();   // the stages are free: partial tiles [slice][acc][BM][BN + PAD]

  float* part = sm + slice * C::TILE;
#pragma unroll
  for (int j = 0; j < NACC; ++j)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float* row = part + (j * BM + ra + (i < 4 ? i : i + 12)) * C::LDT + cb;
#pragma unroll
      for (int n = 0; n < TN; n += 4) {
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint64_t w = acc[j][i >> 1][n + k];
          v[k] = __uint_as_float(static_cast<uint32_t>(i & 1 ? w >> 32 : w));
        }
        *reinterpret_cast<float4*>(row + n * 8) = make_float4(v[0], v[1], v[2], v[3]);
      }
    }
  __syncthreads();

  // sum the slices (and, over the cluster, the ranks) in order, then the epilogue
  constexpr int GROUPS = BM * BN / 4;
  auto local4 = [&](int j, int r, int c) {
    float4 s = *reinterpret_cast<const float4*>(sm + (j * BM + r) * C::LDT + c);
#pragma unroll
    for (int k = 1; k < KS; ++k) {
      const float4 t = *reinterpret_cast<const float4*>(sm + k * C::TILE + (j * BM + r) * C::LDT + c);
      s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
    }
    return s;
  };
  if (S > 1) {
    if (KS > 1) {
      for (int g = threadIdx.x; g < NACC * GROUPS; g += THREADS) {
        const int j = g / GROUPS, r = g % GROUPS / (BN / 4), c = g % (BN / 4) * 4;
        *reinterpret_cast<float4*>(sm + (j * BM + r) * C::LDT + c) = local4(j, r, c);
      }
    }
    cluster_sync();
  }
  const bool dual = (terms & (T_C1_A1B0 | T_C1_A0B1)) != 0;
  const EpiParams& e = p.epi;
  float* EA = static_cast<float*>(e.A);
  float* EAd = static_cast<float*>(e.Ad);
  const int share = GROUPS / S;
  for (int g = rank * share + threadIdx.x; g < (rank + 1) * share; g += THREADS) {
    const int r = g / (BN / 4), c = g % (BN / 4) * 4;
    const int gm = m0 + r, gn = n0 + c;
    if (gm >= p.M || gn >= p.N) continue;
    float x[2][4] = {};
#pragma unroll
    for (int j = 0; j < NACC; ++j) {
      float4 s;
      if (S == 1) {
        s = local4(j, r, c);
      } else {
        const uint32_t at = smem_addr(sm + (j * BM + r) * C::LDT + c);
        s = ld_remote4(at, 0);
        for (int k = 1; k < S; ++k) {
          const float4 t = ld_remote4(at, k);
          s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
        }
      }
      x[j][0] = s.x; x[j][1] = s.y; x[j][2] = s.z; x[j][3] = s.w;
    }
    const int cnt = p.N - gn < 4 ? p.N - gn : 4;
    float c0[4] = {}, c1[4] = {}, o0[4] = {}, o1[4] = {};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k >= cnt) break;
      const EpiOut o = epi_eval(e, gm, gn + k, x[0][k], x[1][k], p.bias[0], p.bias[1], dual);
      c0[k] = o.c0; c1[k] = o.c1; o0[k] = o.o0; o1[k] = o.o1;
    }
    auto put = [&](float* q, int64_t at, const float (&v)[4], bool vec) {
      if (vec && cnt == 4) {
        *reinterpret_cast<float4*>(q + at) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < cnt) q[at + k] = v[k];
      }
    };
    if (p.C[0]) put(p.C[0] + bz * p.bsC[0], static_cast<int64_t>(gm) * p.ldc[0] + gn, c0, p.c_vec);
    if (p.C[1]) put(p.C[1] + bz * p.bsC[1], static_cast<int64_t>(gm) * p.ldc[1] + gn, c1, p.c_vec);
    if (e.mode != EPI_STORE) {
      if (EA) put(EA, static_cast<int64_t>(gm) * e.lda + gn, o0, p.e_vec);
      if (dual && EAd) put(EAd, static_cast<int64_t>(gm) * e.lda + gn, o1, p.e_vec);
    }
  }
  if (S > 1) cluster_sync();   // no CTA's partial tile goes away while another reads it
}

template <int WM, int WN, int TN, int KS, int BK, unsigned TERMS>
cudaError_t launch_cfg(const SimtParams& p, int batch, cudaStream_t s) {
  using C = Cfg<WM, WN, TN, KS, BK, TERMS>;
  auto* kernel = simt_dual_gemm_kernel<WM, WN, TN, KS, BK, TERMS>;
  static PerDeviceOnce attr_once;
  cudaError_t e = attr_once.run([&](int&) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  });
  if (e != cudaSuccess) return e;
  SimtParams q = p;
  q.tiles_n = (p.N + C::BN - 1) / C::BN;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(q.tiles_n * ((p.M + C::BM - 1) / C::BM), 1, batch * p.split);
  cfg.blockDim = dim3(C::THREADS);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = g_pdl ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = p.split;
  cfg.attrs = attr;
  cfg.numAttrs = p.split > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, q);
}

enum Tile { T128 = 0, T64 = 1, T32 = 2 };

template <unsigned TERMS>
cudaError_t launch_tile(const SimtParams& p, int tile, int batch, cudaStream_t s) {
  if (tile == T128) return launch_cfg<4, 2, 8, 1, 8, TERMS>(p, batch, s);
  if (tile == T64) return launch_cfg<2, 2, 4, 2, 16, TERMS>(p, batch, s);
  return launch_cfg<1, 1, 4, 8, 32, TERMS>(p, batch, s);
}

}  // namespace

cudaError_t simt_gemm(const GemmArgs& a, cudaStream_t s) {
  if (a.M <= 0 || a.N <= 0) return cudaSuccess;
  if (a.batch > 1 && a.epi.mode != EPI_STORE) return cudaErrorInvalidValue;
  SimtParams p;
  memset(&p, 0, sizeof(p));
  p.M = a.M; p.N = a.N; p.K = a.K; p.terms = a.terms & T_ALL;
  p.A[0] = static_cast<const float*>(a.A0); p.lda[0] = a.lda0;
  p.A[1] = static_cast<const float*>(a.A1); p.lda[1] = a.lda1;
  p.B[0] = static_cast<const float*>(a.B0); p.ldb[0] = a.ldb0;
  p.B[1] = static_cast<const float*>(a.B1); p.ldb[1] = a.ldb1;
  p.C[0] = a.C0; p.ldc[0] = a.ldc0; p.bias[0] = a.bias0;
  p.C[1] = writes_c1(a) ? a.C1 : nullptr; p.ldc[1] = a.ldc1; p.bias[1] = a.bias1;
  p.epi = a.epi;
  p.a_mn = a.a_mn ? 1 : 0;
  p.b_mn = a.b_mn ? 1 : 0;
  p.bsA[0] = a.bsA0; p.bsA[1] = a.bsA1; p.bsB[0] = a.bsB0; p.bsB[1] = a.bsB1;
  p.bsC[0] = a.bsC0; p.bsC[1] = a.bsC1;
  const int batch = a.batch < 1 ? 1 : a.batch;
  // sixteen-byte access only where every address is a multiple of it
  auto ok16 = [&](const void* x, int ld, int64_t bs) {
    return !x || (!(reinterpret_cast<uintptr_t>(x) & 15) && !(ld & 3) && (batch == 1 || !(bs & 3)));
  };
  p.a_vec = ok16(a.A0, a.lda0, a.bsA0) && ok16(a.A1, a.lda1, a.bsA1);
  p.b_vec = ok16(a.B0, a.ldb0, a.bsB0) && ok16(a.B1, a.ldb1, a.bsB1);
  p.c_vec = ok16(a.C0, a.ldc0, a.bsC0) && ok16(a.C1, a.ldc1, a.bsC1);
  p.e_vec = ok16(a.epi.A, a.epi.lda, 0) && ok16(a.epi.Ad, a.epi.lda, 0);

  // Tile and K split by a cost in clocks, fitted to one GB300 (1.93 GHz): the clocks a CTA
  // takes per k and product term when it has its SM to itself (latency of the staged loads
  // and barriers) and when the SM is full of such CTAs (the FMA pipes), the epilogue's clocks
  // per output, and the fixed cost of a launch and of a cluster exchange.  Within 12% of the
  // best of all tiles and splits on 20 shapes from 8x32x16 to 4096x4096x1024 (times in us,
  // 128 / 64 / 32 tile at its best split): 256x1024x1024 32 / 20 / 23, 1024x256x256 14 / 9 / 9,
  // dual 500x10x500 26 / 12 / 9, dual 500x1023x1023 84 / 91 / 114, batched 32 x 128x64x128
  // 10 / 7 / 6, tangent 4096x4096x1024 1329 / 1446 / 1919.
  const int edge[3] = {128, 64, 32};
  const double alone[3] = {210.0, 75.0, 21.0}, full[3] = {185.0, 52.0, 20.0};
  const double exchange[4] = {0.0, 3500.0, 5500.0, 9000.0};
  const int nacc = p.terms & (T_C1_A1B0 | T_C1_A0B1) ? 2 : 1;
  double best = 0.0;
  int tile = T64;
  p.split = 1;
  for (int t = 0; t < 3; ++t) {
    const int64_t tiles = static_cast<int64_t>((a.M + edge[t] - 1) / edge[t]) *
                          ((a.N + edge[t] - 1) / edge[t]) * batch;
    for (int j = 0; j < (t == T128 ? 3 : 4); ++j) {
      const int S = 1 << j;
      if (S > 1 && (tiles * S > 304 || a.K < 32 * S)) break;
      const double n = static_cast<double>((tiles * S + 151) / 152);   // on the busiest SM
      const double k = static_cast<double>((a.K + S - 1) / S) * term_count(a.terms);
      const double cost = exchange[j] + k * std::max(alone[t], n * full[t]) +
                          0.4 * n * nacc * edge[t] * edge[t];
      if (best == 0.0 || cost < best) { best = cost; tile = t; p.split = S; }
    }
  }
  cudaError_t e;
  switch (p.terms) {
    case T_C0_A0B0: e = launch_tile<T_C0_A0B0>(p, tile, batch, s); break;
    case T_C0_A0B1: e = launch_tile<T_C0_A0B1>(p, tile, batch, s); break;
    case T_C0_A1B0 | T_C0_A0B1: e = launch_tile<T_C0_A1B0 | T_C0_A0B1>(p, tile, batch, s); break;
    case T_C0_A0B0 | T_C0_A1B1: e = launch_tile<T_C0_A0B0 | T_C0_A1B1>(p, tile, batch, s); break;
    case T_C0_A0B0 | T_C1_A0B1: e = launch_tile<T_C0_A0B0 | T_C1_A0B1>(p, tile, batch, s); break;
    case T_C0_A0B0 | T_C1_A1B0 | T_C1_A0B1:
      e = launch_tile<T_C0_A0B0 | T_C1_A1B0 | T_C1_A0B1>(p, tile, batch, s);
      break;
    default: e = launch_tile<T_ALL>(p, tile, batch, s); break;
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace mf
