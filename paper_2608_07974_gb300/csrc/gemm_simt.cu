// CUDA-core GEMM with fp32 accumulation: the fp32 path (the tiny fp32 workload needs fp32
// accuracy, which rules out TF32 tensor cores) and the reference the tensor-core GEMM is tested
// against. Row-major operands; the three modes of ops.h. fp32 operands with 16-byte aligned rows run the
// pipelined kernel of the second half; every other case (bf16 shapes outside the tensor-core rules, odd
// strides) the plain one.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "ops.h"

namespace zl {

namespace {
constexpr int BM = 64, BN = 64, BK = 16;

template <typename T, int MODE>
__device__ __forceinline__ float ldA(const T* A, int M, int K, int m, int k) {
  if (m >= M || k >= K) return 0.f;
  return MODE == 2 ? to_f(A[(size_t)k * M + m]) : to_f(A[(size_t)m * K + k]);
}
template <typename T, int MODE>
__device__ __forceinline__ float ldB(const T* B, int N, int K, int k, int n) {
  if (n >= N || k >= K) return 0.f;
  return MODE == 0 ? to_f(B[(size_t)n * K + k]) : to_f(B[(size_t)k * N + n]);
}

template <typename T, typename TC, int MODE>
__global__ void __launch_bounds__(256) gemm_simt_k(int M, int N, int K, const T* __restrict__ A,
                                                   const T* __restrict__ B, TC* C,
                                                   const float* __restrict__ bias, const TC* R, float alpha,
                                                   int rmode) {
  __shared__ float As[BK][BM + 4];
  __shared__ float Bs[BK][BN + 4];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int bm = blockIdx.y * BM, bn = blockIdx.x * BN;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int e = tid + 256 * r;
      if (MODE == 2) { const int k = e / BM, m = e % BM; As[k][m] = ldA<T, MODE>(A, M, K, bm + m, k0 + k); }
      else { const int m = e / BK, k = e % BK; As[k][m] = ldA<T, MODE>(A, M, K, bm + m, k0 + k); }
      if (MODE == 0) { const int n = e / BK, k = e % BK; Bs[k][n] = ldB<T, MODE>(B, N, K, k0 + k, bn + n); }
      else { const int k = e / BN, n = e % BN; Bs[k][n] = ldB<T, MODE>(B, N, K, k0 + k, bn + n); }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = As[k][ty + 16 * i]; b[i] = Bs[k][tx + 16 * i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = bm + ty + 16 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = bn + tx + 16 * j;
      if (n >= N) continue;
      const size_t o = (size_t)m * N + n;
      float v = alpha * acc[i][j];
      if (MODE == 2) {
        reinterpret_cast<float*>(C)[o] += v;
      } else {
        if (bias) v += bias[n];
        if (R) v = rmode ? v * gelu_tanh_grad(to_f(R[o]), std::is_same<TC, bf16>::value) : v + to_f(R[o]);
        C[o] = from_f<TC>(v);
      }
    }
  }
}

template <typename T>
void gemm_simt_t(int mode, int M, int N, int K, const void* A, const void* B, void* C, const float* bias,
                 const void* R, cudaStream_t s, float alpha, int rmode) {
  dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM), block(256);
  if (mode == 0)
    gemm_simt_k<T, T, 0><<<grid, block, 0, s>>>(M, N, K, (const T*)A, (const T*)B, (T*)C, bias, (const T*)R, alpha,
                                                 rmode);
  else if (mode == 1)
    gemm_simt_k<T, T, 1><<<grid, block, 0, s>>>(M, N, K, (const T*)A, (const T*)B, (T*)C, bias, (const T*)R,
                                                 alpha, rmode);
  else
    gemm_simt_k<T, float, 2><<<grid, block, 0, s>>>(M, N, K, (const T*)A, (const T*)B, (float*)C, nullptr, nullptr,
                                                    alpha, 0);
}
}  // namespace

namespace {
// ------------------------------------------------------------------------------------------------
// fp32, 16-byte aligned rows. A CTA of 256 threads computes a BT x BT tile, 4 x 4 per thread; with BT = 32
// four groups of 64 threads share the tile, each taking a quarter of every k block, and a cluster of up to
// four CTAs along z shares the tile's K range; the partial sums meet in a fixed order (groups through
// shared memory, CTAs through distributed shared memory). Operands come in three cp.async stages in the
// layout they have in memory: rows of k (padded by 4) where k is contiguous, rows of m or n where it is not,
// so nothing is transposed.
// What bounds it at the sizes it is for (256 tokens, widths 128-688) is latency: the plain kernel waited for the
// loads of one 16-deep k block before the next, about 28 us a product; the 32-wide tiles and the K split give
// such products enough CTAs (256 x 128: 32 tiles, up to 128 CTAs). The tiny fp32 step (4 layers, d 128, 4 x 64
// tokens, K = 2) with this, the fused update and the attention kernels in tiles: 1.37 -> 0.49 ms.
// ------------------------------------------------------------------------------------------------
constexpr int FST = 3;   // stages

template <int BT>
struct FCfg {
  static constexpr int KG = BT == 32 ? 4 : 1;          // k groups
  static constexpr int FK = BT == 32 ? 64 : 32;        // k block
  static constexpr int LDK = FK + 4, LDM = BT + 4;     // row pitches (floats): k contiguous; m / n contiguous
  static constexpr int OPND = BT * LDK > FK * LDM ? BT * LDK : FK * LDM;
  static constexpr int SMEM = FST * 2 * OPND * 4;
  static_assert(SMEM >= KG * BT * BT * 4, "the partial tiles reuse the stages");
};

__device__ __forceinline__ void cp16(float* dst, const float* src, bool ok) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// One operand's block: rows r0 .. of `rows` (m or n), k from k0 below k1. KC: k is contiguous (row pitch `ld`
// = K), else m / n is (ld = rows). Out-of-range pieces become zeros (their source stays the array's start).
template <int BT, bool KC>
__device__ __forceinline__ void f32_stage(float* dst, const float* src, int ld, int rows, int r0, int k0, int k1) {
  using C_ = FCfg<BT>;
  constexpr int PER = KC ? C_::FK / 4 : BT / 4;                 // 16-byte pieces per stored row
  constexpr int N = (KC ? BT : C_::FK) * PER;
  for (int e = threadIdx.x; e < N; e += 256) {
    const int a = e / PER, b = (e % PER) * 4;
    const int r = r0 + (KC ? a : b), k = k0 + (KC ? b : a);
    const bool ok = r < rows && k < k1;
    const size_t o = KC ? (size_t)r * ld + k : (size_t)k * ld + r;
    cp16(dst + a * (KC ? C_::LDK : C_::LDM) + b, src + (ok ? o : 0), ok);
  }
}

struct F32Epi {
  const float* bias;
  const float* R;
  float alpha;
  int rmode;
  GemmUpdate u;   // UPD: the AdamW step of the tensor (theta = C) instead of the accumulation
};

// KC operands end at a multiple of 4 (K % 4 == 0) and so do m / n contiguous ones, so no 16-byte piece
// straddles an end. kps: the K range of one CTA of the cluster (a multiple of 4).
template <int MODE, int BT, bool UPD>
__global__ void __launch_bounds__(256) gemm_f32_k(int M, int N, int K, const float* __restrict__ A,
                                                  const float* __restrict__ B, float* C, int kps, const F32Epi ep) {
  using C_ = FCfg<BT>;
  constexpr bool AKC = MODE != 2, BKC = MODE == 0;
  constexpr int KG = C_::KG, FK = C_::FK, TT = BT / 4;   // TT x TT threads per group
  extern __shared__ __align__(16) float sm[];
  pdl_wait();
  pdl_trigger();
  const int g = threadIdx.x / (TT * TT), t = threadIdx.x % (TT * TT), tx = t % TT, ty = t / TT;
  const int bm = blockIdx.y * BT, bn = blockIdx.x * BT;
  const int kb = blockIdx.z * kps, ke = min(K, kb + kps);
  const int nk = ke > kb ? (ke - kb + FK - 1) / FK : 0;
  auto stage = [&](int i) {
    if (i < nk) {
      float* a = sm + (i % FST) * 2 * C_::OPND;
      f32_stage<BT, AKC>(a, A, AKC ? K : M, M, bm, kb + i * FK, ke);
      f32_stage<BT, BKC>(a + C_::OPND, B, BKC ? K : N, N, bn, kb + i * FK, ke);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[4][4] = {};
  stage(0);
  stage(1);
  for (int i = 0; i < nk; ++i) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();   // block i has landed; every thread is done with the buffer that block i + 2 takes
    stage(i + 2);
    const float* as = sm + (i % FST) * 2 * C_::OPND;
    const float* bs = as + C_::OPND;
#pragma unroll 4
    for (int k = g * (FK / KG); k < (g + 1) * (FK / KG); k += 4) {
      // thread rows: 4 ty + r of an m-contiguous operand, ty + TT r of a k-contiguous one (no bank conflicts)
      float4 a[4], b[4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
        a[r] = *reinterpret_cast<const float4*>(AKC ? as + (ty + TT * r) * C_::LDK + k : as + (k + r) * C_::LDM + 4 * ty);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        b[r] = *reinterpret_cast<const float4*>(BKC ? bs + (tx + TT * r) * C_::LDK + k : bs + (k + r) * C_::LDM + 4 * tx);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float av[4], bv[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          av[r] = AKC ? (&a[r].x)[q] : (&a[q].x)[r];
          bv[r] = BKC ? (&b[r].x)[q] : (&b[q].x)[r];
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(av[r], bv[c], acc[r][c]);
      }
    }
  }
  // the groups' partial tiles, then (cluster) the CTAs', summed in order by the threads of each output
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      sm[g * BT * BT + (AKC ? ty + TT * r : 4 * ty + r) * BT + (BKC ? tx + TT * c : 4 * tx + c)] = acc[r][c];
  __syncthreads();
  const unsigned nz = gridDim.z, rank = blockIdx.z;
  if (KG > 1) {
    for (int e = threadIdx.x; e < BT * BT; e += 256) {
      float v = sm[e];
#pragma unroll
      for (int q = 1; q < KG; ++q) v += sm[q * BT * BT + e];
      sm[e] = v;
    }
    __syncthreads();
  }
  if (nz > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  AdamHP hpv;
  if (UPD) hpv = adam_hp(ep.u.hp, ep.u.b1, ep.u.b2, ep.u.eps, ep.u.wd);
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);
  for (int e = (int)rank * 256 + threadIdx.x; e < BT * BT; e += (int)nz * 256) {   // each CTA its share
    const int m = bm + e / BT, n = bn + e % BT;
    float v = 0.f;
    if (nz > 1) {
      for (unsigned q = 0; q < nz; ++q) {
        uint32_t ra;
        float x;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(sbase + 4u * (uint32_t)e), "r"(q));
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(ra) : "memory");
        v += x;
      }
    } else {
      v = sm[e];
    }
    if (m >= M || n >= N) continue;
    const size_t o = (size_t)m * N + n;
    v *= ep.alpha;
    if (UPD) {
      const size_t so = ep.u.blk ? blk_index((size_t)m, (size_t)n, (size_t)N) : o;
      float th = ep.u.theta[so], mm = ep.u.m[so], vv = ep.u.v[so];
      adamw_elem(th, mm, vv, __fmul_rn(v, ep.u.gscale), hpv);
      ep.u.theta[so] = th;
      ep.u.m[so] = mm;
      ep.u.v[so] = vv;
    } else if (MODE == 2) {
      C[o] += v;
    } else {
      if (ep.bias) v += ep.bias[n];
      if (ep.R) v = ep.rmode ? v * gelu_tanh_grad(ep.R[o], false) : v + ep.R[o];
      C[o] = v;
    }
  }
  // no CTA leaves while another still reads its shared memory
  if (nz > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int MODE, int BT, bool UPD>
bool launch_f32(int M, int N, int K, const float* A, const float* B, float* C, const F32Epi& ep, int ks, cudaStream_t s) {
  using C_ = FCfg<BT>;
  auto kern = gemm_f32_k<MODE, BT, UPD>;
  static const bool attr =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM) == cudaSuccess;
  if (!attr) {
    cudaGetLastError();
    return false;
  }
  const int kps = ((K + ks - 1) / ks + 3) / 4 * 4;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((N + BT - 1) / BT), (unsigned)((M + BT - 1) / BT), (unsigned)ks);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = C_::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 1;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = (unsigned)ks;
  cfg.attrs = at;
  cfg.numAttrs = ks > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, M, N, K, A, B, C, kps, ep) == cudaSuccess;
}

// 64-wide tiles where they fill the SMs twice over (each thread then works on one tile alone); else 32-wide ones
// with K shared by 2 or 4 CTAs while that keeps every CTA a k block of 64 and the CTAs within one wave.
template <int MODE, bool UPD>
bool run_f32(int M, int N, int K, const float* A, const float* B, float* C, const F32Epi& ep, cudaStream_t s) {
  auto al16 = [](const void* p) { return ((uintptr_t)p & 15u) == 0; };
  const bool rows_ok = MODE == 0 ? K % 4 == 0 : MODE == 1 ? K % 4 == 0 && N % 4 == 0 : M % 4 == 0 && N % 4 == 0;
  if (!rows_ok || !al16(A) || !al16(B) || M < 1 || N < 1 || K < 1 || (M + 31) / 32 > 65535) return false;
  const long t64 = (long)((M + 63) / 64) * ((N + 63) / 64), t32 = (long)((M + 31) / 32) * ((N + 31) / 32);
  const long sms = sm_count();
  if (t64 >= 2 * sms) return launch_f32<MODE, 64, UPD>(M, N, K, A, B, C, ep, 1, s);
  int ks = 1;
  while (ks < 4 && t32 * ks * 2 <= 2 * sms && K / (ks * 2) >= 64) ks *= 2;
  return launch_f32<MODE, 32, UPD>(M, N, K, A, B, C, ep, ks, s);
}
}  // namespace

bool gemm_f32_update(int M, int N, int K, const void* A, const void* B, const GemmUpdate& u, cudaStream_t s) {
  if (u.g || u.comp) return false;
  if (!run_f32<2, true>(M, N, K, (const float*)A, (const float*)B, u.theta, F32Epi{nullptr, nullptr, 1.f, 0, u}, s))
    return false;
  note_launch(1);
  return true;
}

void gemm_simt(int dt, int mode, int M, int N, int K, const void* A, const void* B, void* C, const float* bias,
               const void* R, cudaStream_t s, float alpha, int rmode) {
  note_launch(1);
  if (M <= 0 || N <= 0) return;
  if (dt == F32) {
    const F32Epi ep{bias, (const float*)R, alpha, rmode, GemmUpdate{}};
    const float *a = (const float*)A, *b = (const float*)B;
    if (mode == 0 ? run_f32<0, false>(M, N, K, a, b, (float*)C, ep, s)
                  : mode == 1 ? run_f32<1, false>(M, N, K, a, b, (float*)C, ep, s)
                              : run_f32<2, false>(M, N, K, a, b, (float*)C, ep, s))
      return;
    gemm_simt_t<float>(mode, M, N, K, A, B, C, bias, R, s, alpha, rmode);
  } else {
    gemm_simt_t<bf16>(mode, M, N, K, A, B, C, bias, R, s, alpha, rmode);
  }
}

}  // namespace zl

namespace zl {
// GEMM dispatch: the tensor-core kernel where it applies, else the CUDA-core kernel.
void gemm(int dt, int mode, int M, int N, int K, const void* A, const void* B, void* C, const float* bias,
          const void* R, cudaStream_t s, unsigned* err, cudaMemPool_t pool, float alpha, int rmode) {
  if (dt == BF16 && gemm_tc(mode, M, N, K, A, B, C, bias, R, err, s, pool, alpha, rmode)) return;
  gemm_simt(dt, mode, M, N, K, A, B, C, bias, R, s, alpha, rmode);
}
}  // namespace zl
