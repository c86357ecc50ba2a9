// SIMT kernels of the FP64 and FP32 paths: register-blocked batched GEMM
// for the mu-mode products (Sec. 2, Eq. 5), the stage-1 right-hand side
// W = sum_mu U x_mu A_mu + G(U, V) (Eq. 6, Eq. 11) and the stage-2 reaction
// difference D = G(U2, V2) - G(U, V) (Eq. 11).
#include <cuda_runtime.h>
#include <stdint.h>

#include <math.h>

#include <algorithm>

#include "adr_internal.h"
#include "pointwise.cuh"

namespace adr {

// Programmatic dependent launch: a kernel of a step waits for its predecessors
// before it touches memory, and lets the next one be scheduled when only its
// own last stores are left.  Not before: the next kernel's blocks would then be
// placed while this one's hold most SMs, several to each that is free (FP64
// 64^2, 128 blocks a launch, us a step: trigger at the start 28.5, before the
// epilogue 17.4, before the last stores 15.3, after them 15.8; no programmatic
// launches 30).  Shared memory padded so that a block has its SM to itself does
// it too (16.3), but keeps the launches of other streams off the SMs (eight
// 64^2 solves on eight streams 64.7; 37.7 without the padding).
__device__ __forceinline__ void simt_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void simt_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
static cudaError_t simt_launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                               Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

template <typename T>
__global__ void __launch_bounds__(128) rhs_kernel(PointwiseArgsT<T> a, const T* __restrict__ u,
                                                  const T* __restrict__ v, T* __restrict__ wu,
                                                  T* __restrict__ wv) {
  simt_wait();
  const int i1 = blockIdx.x * blockDim.x + threadIdx.x;
  if (i1 >= (int)a.n[0]) return;
  const int i2 = blockIdx.y, i3 = blockIdx.z;
  const int64_t idx = ((int64_t)i3 * a.n[1] + i2) * a.n[0] + i1;
  T x, y;
  rhs_point<T>(a, u, v, idx, i1, i2, i3, x, y);
  wu[idx] = x;
  wv[idx] = y;
  simt_trigger();
}

template <typename T>
__global__ void __launch_bounds__(256) rdiff_kernel(PointwiseArgsT<T> a, const T* __restrict__ u,
                                                    const T* __restrict__ v,
                                                    const T* __restrict__ u2,
                                                    const T* __restrict__ v2, T* __restrict__ du,
                                                    T* __restrict__ dv) {
  simt_wait();
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < a.N;
       idx += (int64_t)gridDim.x * blockDim.x) {
    react_diff<T>(a.rx, u[idx], v[idx], u2[idx], v2[idx], du[idx], dv[idx]);
  }
  simt_trigger();
}

// Lawson2b (Eq. 7) pointwise stages: x = u + scale G^u(u, v) (both
// components), and u += scale G^u(u2, v2).
template <typename T>
__global__ void __launch_bounds__(256) lawson_pre_kernel(PointwiseArgsT<T> a, const T* __restrict__ u,
                                                         const T* __restrict__ v, T scale,
                                                         T* __restrict__ xu, T* __restrict__ xv) {
  simt_wait();
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < a.N;
       idx += (int64_t)gridDim.x * blockDim.x) {
    T gu, gv;
    const T uu = u[idx], vv = v[idx];
    react<T>(a.rx, uu, vv, gu, gv);
    xu[idx] = uu + scale * gu;
    xv[idx] = vv + scale * gv;
  }
  simt_trigger();
}

template <typename T>
__global__ void __launch_bounds__(256) lawson_post_kernel(PointwiseArgsT<T> a,
                                                          const T* __restrict__ u2,
                                                          const T* __restrict__ v2, T scale,
                                                          T* __restrict__ u, T* __restrict__ v) {
  simt_wait();
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < a.N;
       idx += (int64_t)gridDim.x * blockDim.x) {
    T gu, gv;
    react<T>(a.rx, u2[idx], v2[idx], gu, gv);
    u[idx] += scale * gu;
    v[idx] += scale * gv;
  }
  simt_trigger();
}

// Threads of a flat block: 64 in FP64, so that a grid of a few thousand points
// covers all SMs (two FP64 operations a clock each).
template <typename T>
constexpr int kFlatThreads = sizeof(T) == 8 ? 64 : 256;
template <typename T>
static dim3 pointwise_grid(int64_t N) {
  const int64_t b = (N + kFlatThreads<T> - 1) / kFlatThreads<T>;
  const int64_t cap = 152 * 16 * (256 / kFlatThreads<T>);
  return dim3((unsigned)(b < cap ? (b < 1 ? 1 : b) : cap));
}

template <typename T>
cudaError_t launch_rhs(const PointwiseArgsT<T>& a, const T* u, const T* v, T* wu, T* wv,
                       cudaStream_t s) {
  dim3 grid((unsigned)((a.n[0] + 127) / 128), (unsigned)a.n[1], (unsigned)(a.d == 3 ? a.n[2] : 1));
  return simt_launch(rhs_kernel<T>, grid, dim3(128), 0, s, a, u, v, wu, wv);
}

template <typename T>
cudaError_t launch_rdiff(const PointwiseArgsT<T>& a, const T* u, const T* v, const T* u2, const T* v2,
                         T* du, T* dv, cudaStream_t s) {
  return simt_launch(rdiff_kernel<T>, pointwise_grid<T>(a.N), dim3(kFlatThreads<T>), 0, s, a, u, v, u2, v2, du, dv);
}

template <typename T>
cudaError_t launch_lawson_pre(const PointwiseArgsT<T>& a, const T* u, const T* v, T scale, T* xu,
                              T* xv, cudaStream_t s) {
  return simt_launch(lawson_pre_kernel<T>, pointwise_grid<T>(a.N), dim3(kFlatThreads<T>), 0, s, a, u, v, scale, xu, xv);
}

template <typename T>
cudaError_t launch_lawson_post(const PointwiseArgsT<T>& a, const T* u2, const T* v2, T scale, T* u,
                               T* v, cudaStream_t s) {
  return simt_launch(lawson_post_kernel<T>, pointwise_grid<T>(a.N), dim3(kFlatThreads<T>), 0, s, a, u2, v2, scale, u, v);
}

template cudaError_t launch_lawson_pre<float>(const PointwiseArgsT<float>&, const float*,
                                              const float*, float, float*, float*, cudaStream_t);
template cudaError_t launch_lawson_pre<double>(const PointwiseArgsT<double>&, const double*,
                                               const double*, double, double*, double*,
                                               cudaStream_t);
template cudaError_t launch_lawson_post<float>(const PointwiseArgsT<float>&, const float*,
                                               const float*, float, float*, float*, cudaStream_t);
template cudaError_t launch_lawson_post<double>(const PointwiseArgsT<double>&, const double*,
                                                const double*, double, double*, double*,
                                                cudaStream_t);
template cudaError_t launch_rhs<float>(const PointwiseArgsT<float>&, const float*, const float*, float*,
                                       float*, cudaStream_t);
template cudaError_t launch_rhs<double>(const PointwiseArgsT<double>&, const double*, const double*,
                                        double*, double*, cudaStream_t);
template cudaError_t launch_rdiff<float>(const PointwiseArgsT<float>&, const float*, const float*,
                                         const float*, const float*, float*, float*,
                                         cudaStream_t);
template cudaError_t launch_rdiff<double>(const PointwiseArgsT<double>&, const double*, const double*,
                                          const double*, const double*, double*, double*,
                                          cudaStream_t);

// ---------------------------------------------------------------- GEMM
// One CTA computes a BM x BN tile of C, a thread a TM x TN block of it.  A and
// B panels of KC values of K go through ST shared-memory stages by cp.async,
// ST - 1 of them requested ahead: the products of the small plans (K of a few
// dozen to a few hundred) are one or two stages long, so a launch pays one
// memory round trip instead of one per 8 values of K.  Every output is one
// chain of FMAs over k = 0, 1, ..., K - 1, whatever the tile (KS such chains
// where the tile's K is split).
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// bytes <= B are copied, the rest of the B bytes zero-filled
template <int B>
__device__ __forceinline__ void cp_async(void* dst, const void* src, int bytes) {
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(bytes)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_addr(dst)), "l"(src), "n"(B),
                 "r"(bytes)
                 : "memory");
}
// rows x cols values of a row-major matrix (leading dimension ld) from src
// into dst (row pitch PITCH), rows and columns beyond nr, nc as zeros
template <typename T, int ROWS, int COLS, int PITCH, int THREADS, bool VEC>
__device__ __forceinline__ void load_panel(T* dst, const T* src, int64_t ld, int nr, int nc) {
  constexpr int V = VEC ? 16 / (int)sizeof(T) : 1, CV = COLS / V;
#pragma unroll
  for (int i0 = 0; i0 < ROWS * CV; i0 += THREADS) {
    const int i = i0 + threadIdx.x;
    if (ROWS * CV % THREADS != 0 && i >= ROWS * CV) break;
    const int r = i / CV, c = i % CV * V;
    const int n = r < nr ? min(V, max(0, nc - c)) : 0;
    cp_async<V * (int)sizeof(T)>(dst + r * PITCH + c, n > 0 ? src + r * ld + c : src, n * (int)sizeof(T));
  }
}

// KS: groups of threads that share the tile's K (each takes every KS-th run
// of V values of a stage); their sums are added in order at the end.
template <typename T, int BM_, int BN_, int TM_, int TN_, int KC_, int ST_, int KS_ = 1>
struct GemmCfg {
  static constexpr int BM = BM_, BN = BN_, TM = TM_, TN = TN_, KC = KC_, ST = ST_, KS = KS_;
  static constexpr int V = 16 / (int)sizeof(T);            // values per 16 bytes
  static constexpr int GROUP = (BM / TM) * (BN / TN);      // threads of one group
  static constexpr int THREADS = GROUP * KS;
  static constexpr int PA = KC + V, PB = BN + V;           // row pitches
  static constexpr int STAGE = BM * PA + KC * PB;          // values
  static constexpr int SMEM = ST * STAGE * (int)sizeof(T);
};

template <typename T, typename C>
__global__ void __launch_bounds__(C::THREADS) gemm_kernel(const __grid_constant__ GemmArgs g) {
  constexpr int BM = C::BM, BN = C::BN, TM = C::TM, TN = C::TN, KC = C::KC, ST = C::ST, V = C::V;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  simt_wait();
  const int z = blockIdx.z;
  const int comp = z / g.batch;
  const int p = z - comp * g.batch;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const T* __restrict__ A = (const T*)g.A[comp] + (int64_t)p * g.a_bs + (int64_t)m0 * g.lda;
  const T* __restrict__ B = (const T*)g.B[comp] + (int64_t)p * g.b_bs + n0;
  // 16-byte copies where every row of the operand starts on 16 bytes
  const bool va = (((uintptr_t)A | (uintptr_t)(g.lda * (int64_t)sizeof(T))) & 15) == 0;
  const bool vb = (((uintptr_t)B | (uintptr_t)(g.ldb * (int64_t)sizeof(T))) & 15) == 0;
  const int nk = (g.K + KC - 1) / KC;
  auto load = [&](int kt) {
    if (kt < nk) {
      T* st = sm + kt % ST * C::STAGE;
      const int k0 = kt * KC;
      if (va)
        load_panel<T, BM, KC, C::PA, C::THREADS, true>(st, A + k0, g.lda, g.M - m0, g.K - k0);
      else
        load_panel<T, BM, KC, C::PA, C::THREADS, false>(st, A + k0, g.lda, g.M - m0, g.K - k0);
      T* sb = st + BM * C::PA;
      if (vb)
        load_panel<T, KC, BN, C::PB, C::THREADS, true>(sb, B + (int64_t)k0 * g.ldb, g.ldb, g.K - k0, g.N - n0);
      else
        load_panel<T, KC, BN, C::PB, C::THREADS, false>(sb, B + (int64_t)k0 * g.ldb, g.ldb, g.K - k0, g.N - n0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int kg = threadIdx.x / C::GROUP, gt = threadIdx.x % C::GROUP;
  const int tx = gt % (BN / TN), ty = gt / (BN / TN);
  // a thread's columns: groups of min(TN, 4) neighbours spread over the tile;
  // its rows: BM / TM apart
  constexpr int G = TN < 4 ? TN : 4;
  auto col = [&](int j) { return (j / G) * (BN / (TN / G)) + tx * G + j % G; };
  auto row = [&](int i) { return i * (BM / TM) + ty; };
  T acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = (T)0;
#pragma unroll
  for (int s = 0; s < ST - 1; ++s) load(s);
  for (int kt = 0; kt < nk; ++kt) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();  // stage kt landed; stage kt - 1 is read by nobody any more
    load(kt + ST - 1);
    const T* as = sm + kt % ST * C::STAGE;
    const T* bs = as + BM * C::PA;
    const int kend = min(KC, g.K - kt * KC);
#pragma unroll 2
    for (int k = kg * V; k < kend; k += C::KS * V) {
      T a[TM][V], b[V][TN];
#pragma unroll
      for (int i = 0; i < TM; ++i)
        *reinterpret_cast<float4*>(&a[i][0]) = *reinterpret_cast<const float4*>(as + row(i) * C::PA + k);
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int j = 0; j < TN; j += G) {
          const T* src = bs + (k + q) * C::PB + col(j);
          if constexpr (G * sizeof(T) == 16)
            *reinterpret_cast<float4*>(&b[q][j]) = *reinterpret_cast<const float4*>(src);
          else
#pragma unroll
            for (int e = 0; e < G; ++e) b[q][j + e] = src[e];
        }
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i][q], b[q][j], acc[i][j]);
    }
  }
  if constexpr (C::KS > 1) {
    static_assert(TM == 1 && TN == 1, "split contractions: one output a thread");
    __syncthreads();
    sm[threadIdx.x] = acc[0][0];
    __syncthreads();
    if (kg != 0) return;
#pragma unroll
    for (int q = 1; q < C::KS; ++q) acc[0][0] += sm[q * C::GROUP + gt];
  }
  // out = alpha acc + beta base + beta2 base2
  T* __restrict__ Co = (T*)g.C[comp] + (int64_t)p * g.c_bs;
  const T* base = g.base[comp] ? (const T*)g.base[comp] + (int64_t)p * g.c_bs : nullptr;
  const T* base2 = g.base2[comp] ? (const T*)g.base2[comp] + (int64_t)p * g.c_bs : nullptr;
  const T alpha = (T)g.alpha, beta = (T)g.beta, beta2 = (T)g.beta2;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int r = m0 + row(i);
    if (r >= g.M) continue;
    T extra[TN];  // the row's base values before any store (C may be the base)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = n0 + col(j);
      const int64_t o = (int64_t)r * g.ldc + c;
      T x = (T)0;
      if (c < g.N) {
        if (base) x += beta * base[o];
        if (base2) x += beta2 * base2[o];
      }
      extra[j] = x;
    }
    if (i == TM - 1) simt_trigger();
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = n0 + col(j);
      if (c < g.N) Co[(int64_t)r * g.ldc + c] = alpha * acc[i][j] + extra[j];
    }
  }
}

template <typename T, typename C>
static cudaError_t run_gemm(const GemmArgs& g, cudaStream_t s) {
  const dim3 grid((g.N + C::BN - 1) / C::BN, (g.M + C::BM - 1) / C::BM, g.batch * g.ncomp);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
  if constexpr (C::SMEM > 48 * 1024) {  // an attribute of the kernel on the current device
    const cudaError_t e =
        cudaFuncSetAttribute(gemm_kernel<T, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
  }
  return simt_launch(gemm_kernel<T, C>, grid, dim3(C::THREADS), C::SMEM, s, g);
}

// FP64: an SM retires two FMAs a clock (a warp's takes one of its four units
// 64 clocks), so what counts is that the tiles divide evenly over the SMs and
// that every unit has a warp: 8 x 8 tiles, K split two ways; four ways where
// an SM has one tile at most.  us a step, ETD2RKds, 64 x 64 tiles with an 8 x 8
// kernel for small plans (before) / K in two / in four:
//   32^2 33.8 / 15.6 / 15.2   64^2 44.0 / 19.0 / 17.8   128^2 74.7 / 47.9 / 49.4
//   256^2 276 / 252 / 251     512^2 1821 / 1781 / 1795  1024^2 16567 / 13920 / 13986
//   32^3 60.5 / 46.0 / 51.2   64^3 415 / 403 / 414      160^3 17024 / 13469 / 13677
// (16 x 16 tiles: 48.8, 280, 1835, 13917; 45.3, 403, 13330.)  What is left
// above the FMA time (256^2: 232 us) is the pointwise kernels and launches.
// (Measured with an earlier trigger; with the present one, above, 32^2 12.8,
// 64^2 15.3, 128^2 45.3.)
template <>
cudaError_t launch_gemm_simt<double>(const GemmArgs& g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  using S8 = GemmCfg<double, 8, 8, 1, 1, 64, 3, 2>;
  using S8x4 = GemmCfg<double, 8, 8, 1, 1, 64, 3, 4>;
  using S64 = GemmCfg<double, 64, 64, 4, 4, 16, 3>;
  const int64_t rows = (g.M + 7) / 8;
  if (rows > 65535) return run_gemm<double, S64>(g, s);  // a launch's limit
  if (rows * ((g.N + 7) / 8) * g.batch * g.ncomp <= 152) return run_gemm<double, S8x4>(g, s);
  return run_gemm<double, S8>(g, s);
}

// FP32: larger blocks per thread reuse more of each shared-memory load, but
// leave SMs idle sooner.  Clocks of a launch on tiles of configuration C: with
// w tiles on the fullest SM, `rate` FMAs a clock at w >> h, less where few
// warps hide each other's latency.
template <typename C>
static double gemm_clocks(const GemmArgs& g, double rate, double h) {
  const double tiles = (double)((g.N + C::BN - 1) / C::BN) * ((g.M + C::BM - 1) / C::BM) * g.batch * g.ncomp;
  return (ceil(tiles / 152.0) + h) * C::BM * C::BN * g.K / rate;
}

// Rates and h from us a step, 128 x 128 tiles (before) / 32 x 32 / 64 x 32 /
// 64 x 64 / 128 x 128:
//   128^2 42.0 / 20.7 / 27.6 / 34.8 / 90.5    384^2 231 / 57.6 / 55.7 / 75.5 / 213
//   512^2 361 / 131 / 109 / 97.2 / 275        1024^2 716 / 814 / 569 / 551 / 527
//   1500^2 2203 / 2527 / 1542 / 1571 / 1365   64^3 107 / 54.4 / 47.1 / 42.9 / 79.6
//   96^3 191 / 159 / 128 / 134 / 139          160^3 1271 / 916 / 664 / 685 / 916
// Where an SM has one 8 x 8 tile at most, those, K split four ways as in FP64:
// such launches are one chain of latencies.  us a step, first kernel of this
// path / the rule above / 8 x 8:
//   3^3 12.0 / 14.7 / 12.1    9^3 16.0 / 17.8 / 14.6    3^2 10.2 / 11.4 / 10.1
//   32^2 13.1 / 12.0 / 10.2   64^2 17.9 / 14.2 / 10.8   300 x 8 38.0 / 21.3 / 13.7
//   16^3 21.3 / 15.7 / 14.4
template <>
cudaError_t launch_gemm_simt<float>(const GemmArgs& g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  using S8x4 = GemmCfg<float, 8, 8, 1, 1, 64, 3, 4>;
  using S32 = GemmCfg<float, 32, 32, 2, 2, 64, 3>;
  using S64n = GemmCfg<float, 64, 32, 4, 4, 32, 3>;
  using S64 = GemmCfg<float, 64, 64, 4, 4, 32, 3>;
  using S128 = GemmCfg<float, 128, 128, 8, 8, 16, 3>;
  if ((int64_t)((g.M + 7) / 8) * ((g.N + 7) / 8) * g.batch * g.ncomp <= 152) return run_gemm<float, S8x4>(g, s);
  const double c[4] = {gemm_clocks<S32>(g, 40.0, 0.5), gemm_clocks<S64n>(g, 62.0, 0.65),
                       gemm_clocks<S64>(g, 72.0, 0.4), gemm_clocks<S128>(g, 82.0, 0.1)};
  int best = 3;
  for (int i = 2; i >= 0; --i) {
    const int64_t bm = i == 0 ? 32 : 64;
    if (c[i] < c[best] && (g.M + bm - 1) / bm <= 65535) best = i;
  }
  switch (best) {
    case 0: return run_gemm<float, S32>(g, s);
    case 1: return run_gemm<float, S64n>(g, s);
    case 2: return run_gemm<float, S64>(g, s);
    default: return run_gemm<float, S128>(g, s);
  }
}

}  // namespace adr
