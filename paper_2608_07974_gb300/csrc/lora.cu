// The skinny products of LoRA at rank 16 (bf16): 16 output columns or rows, so the time is the reading of the wide
// operand once. Both kernels stream it through a ring of cp.async stages and multiply with m16n8k16 (the tensor cores
// are nearly idle: 16 of a tcgen05 tile's 64 to 256 columns would be used).
#include <algorithm>

#include "common.cuh"
#include "ops.h"

namespace zl {

namespace {
constexpr int RW = 8;    // warps per CTA
constexpr int RST = 4;   // stages

__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4t(uint32_t* r, const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
// 16 bytes to shared memory; !ok: zeros (the source is not read).
__device__ __forceinline__ void cp16(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ------------------------------------------------------------------------------------------------
// U [N, 16] = scale * X [N, K] W [16, K]^T. A CTA forms 16 MT rows. A stage is 256 k's of its rows and of W; warp w
// takes k's 32 w .. 32 w + 31 of every stage and the warps' partial sums are added in order at the end. The order of k
// inside 32 does not matter as long as both operands agree on it, so every lane reads 16 contiguous bytes (eight k's,
// the four k pairs of two m16n8k16 steps) straight into its fragments: rows g and g + 8 of X, rows g and g + 8 of W.
// Bound by HBM (2 N K bytes): 4096 tokens, K = 2048 / 5632 / 11264 6.2 / 12.4 / 22.5 us (launch included; 4.1 TB/s at
// the last). Loads straight into fragments, a batch of four per warp at a time and W read by every 16 rows, waited
// for each batch in full: 9.4 / 25 / 45 us.
// ------------------------------------------------------------------------------------------------
constexpr int kDownK = 256, kDownPitch = kDownK * 2 + 64;   // bytes per row: two rows' 64-byte pieces span the banks

template <int MT>
struct DownCfg {
  static constexpr int ROWS = 16 * MT + 16, STAGE = ROWS * kDownPitch, SMEM = RST * STAGE;
  static_assert(SMEM >= MT * RW * 16 * 17 * 4, "the partial sums reuse the stages");
};

template <int MT>
__global__ void __launch_bounds__(32 * RW) rank16_k(const bf16* __restrict__ X, const bf16* __restrict__ W,
                                                    bf16* __restrict__ U, int N, int K, float scale) {
  using C_ = DownCfg<MT>;
  extern __shared__ __align__(16) uint8_t sm[];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int r0 = blockIdx.x * 16 * MT, nst = (K + kDownK - 1) / kDownK;
  auto stage = [&](int i) {   // a warp copies a row's 512 bytes at once
    if (i < nst) {
      uint8_t* d = sm + (i % RST) * C_::STAGE + lane * 16;
      const int k = i * kDownK + lane * 8;
      const bool ok = k < K;   // K % 8 == 0: a piece's eight k's are all inside or all outside
#pragma unroll
      for (int j = 0; j < C_::ROWS / RW; ++j) {
        const int r = warp + RW * j;   // rows past N are not stored
        const bf16* src = r < 16 * MT ? X + (size_t)min(r0 + r, N - 1) * K : W + (size_t)(r - 16 * MT) * K;
        cp16(d + r * kDownPitch, src + (ok ? k : 0), ok);
      }
    }
    cp_commit();
  };
  float acc[MT][2][4] = {};
#pragma unroll
  for (int i = 0; i < RST - 1; ++i) stage(i);
  for (int i = 0; i < nst; ++i) {
    cp_wait<RST - 2>();
    __syncthreads();   // stage i has landed; every warp is done with the one that stage i + RST - 1 takes
    stage(i + RST - 1);
    const uint8_t* s = sm + (i % RST) * C_::STAGE + warp * 64 + t * 16;
    const uint4 p = *reinterpret_cast<const uint4*>(s + (16 * MT + g) * kDownPitch);
    const uint4 q = *reinterpret_cast<const uint4*>(s + (16 * MT + g + 8) * kDownPitch);
#pragma unroll
    for (int m = 0; m < MT; ++m) {
      const uint4 a = *reinterpret_cast<const uint4*>(s + (16 * m + g) * kDownPitch);
      const uint4 b = *reinterpret_cast<const uint4*>(s + (16 * m + g + 8) * kDownPitch);
      const uint32_t f0[4] = {a.x, b.x, a.y, b.y}, f1[4] = {a.z, b.z, a.w, b.w};
      mma16816(acc[m][0], f0, p.x, p.y);
      mma16816(acc[m][1], f0, q.x, q.y);
      mma16816(acc[m][0], f1, p.z, p.w);
      mma16816(acc[m][1], f1, q.z, q.w);
    }
  }
  cp_wait<0>();
  __syncthreads();
  float(*part)[RW][16][17] = reinterpret_cast<float(*)[RW][16][17]>(sm);
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      part[m][warp][g + 8 * (e >> 1)][2 * t + (e & 1)] = acc[m][0][e];
      part[m][warp][g + 8 * (e >> 1)][8 + 2 * t + (e & 1)] = acc[m][1][e];
    }
  __syncthreads();
  const int r = threadIdx.x >> 4, n = threadIdx.x & 15;
#pragma unroll
  for (int m = 0; m < MT; ++m) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < RW; ++w) v += part[m][w][r][n];
    const int row = r0 + 16 * m + r;
    if (row < N) U[(size_t)row * 16 + n] = __float2bfloat16_rn(v * scale);
  }
}

// ------------------------------------------------------------------------------------------------
// G [16, C] += U [N, 16]^T Y [N, C], fp32. A CTA takes 64 columns; a cluster of up to eight along y shares the
// tokens, so that narrow matrices fill the SMs. A stage is 128 tokens (16 per warp); ldmatrix transposes both operands.
// The warps' partial sums are added in order through shared memory, then the cluster's in order through distributed
// shared memory, onto G: no partials in HBM and no second launch. Bound by HBM (2 N C bytes) when wide, by the latency
// of its start and its sums when narrow: 4096 tokens, C = 2048 / 5632 / 11264 8.9 / 19.1 / 28.2 us; the tensor-core
// GEMM on mostly padding tiles, its partials and their reduction 12.6 / 20.0 / 23.3 us plus the workspace's
// allocation (the whole 1.1B LoRA step of 4096 tokens is 1% slower with the GEMM for the widths of 5632 and 11264). 128-column
// tiles, one CTA per SM: 10.7 / 17.9 / 27.0 us.
// ------------------------------------------------------------------------------------------------
constexpr int kGradC = 64, kGradT = 16 * RW;   // columns; tokens per stage, 16 a warp
constexpr int kGradE = 16 * kGradC / (32 * RW);   // outputs per thread when one CTA forms them all
constexpr int kGradPitch = kGradC * 2 + 16, kGradUPitch = 48;   // bytes per token: eight rows of 16 bytes span the banks
constexpr int kGradStage = kGradT * (kGradPitch + kGradUPitch), kGradSmem = RST * kGradStage;
static_assert(kGradSmem >= RW * 16 * kGradC * 4, "the partial sums reuse the stages");

__global__ void __launch_bounds__(32 * RW) rank16_grad_k(const bf16* __restrict__ U, const bf16* __restrict__ Y,
                                                         float* __restrict__ G, int N, int C, int tokens) {
  extern __shared__ __align__(16) uint8_t sm[];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = blockIdx.x * kGradC, n0 = blockIdx.y * tokens, n1 = min(N, n0 + tokens);
  const int nst = n1 > n0 ? (n1 - n0 + kGradT - 1) / kGradT : 0;
  auto stage = [&](int i) {
    if (i < nst) {
      uint8_t* d = sm + (i % RST) * kGradStage;
      const int nb = n0 + i * kGradT;
#pragma unroll
      for (int j = 0; j < kGradT * (kGradC / 8) / (32 * RW); ++j) {   // Y: eight 16-byte pieces a token
        const int e = threadIdx.x + 32 * RW * j, r = e / (kGradC / 8), c = e % (kGradC / 8) * 8;
        const bool ok = nb + r < n1 && c0 + c < C;
        cp16(d + r * kGradPitch + c * 2, Y + (ok ? (size_t)(nb + r) * C + c0 + c : 0), ok);
      }
      const int r = threadIdx.x >> 1, c = (threadIdx.x & 1) * 8;   // U: two
      const bool ok = nb + r < n1;
      cp16(d + kGradT * kGradPitch + r * kGradUPitch + c * 2, U + (ok ? (size_t)(nb + r) * 16 + c : 0), ok);
    }
    cp_commit();
  };
  static_assert(kGradT * 2 == 32 * RW, "one piece of U per thread");
  float acc[8][4] = {};
#pragma unroll
  for (int i = 0; i < RST - 1; ++i) stage(i);
  // the CTA's share of the outputs, up to four a thread: G is read ahead of the sums
  const int nz = (int)gridDim.y, share = 16 * kGradC / nz, e0 = (int)blockIdx.y * share + (int)threadIdx.x;
  float old[kGradE];
  auto out = [&](int u, float** o) {   // whether output u of this thread exists, and where
    const int e = e0 + 32 * RW * u, c = c0 + e % kGradC;
    *o = G + (size_t)(e / kGradC) * C + c;
    return (int)threadIdx.x + 32 * RW * u < share && c < C;
  };
#pragma unroll
  for (int u = 0; u < kGradE; ++u) {
    float* o;
    old[u] = out(u, &o) ? *o : 0.f;
  }
  // lane l addresses row l % 8 of 8 x 8 block l / 8: tokens first for Y (blocks 0, 1), ranks first for U
  const int blk = lane >> 3, br = lane & 7;
  const int yo = (16 * warp + (blk & 1) * 8 + br) * kGradPitch + (blk >> 1) * 16;
  const int uo = kGradT * kGradPitch + (16 * warp + (blk >> 1) * 8 + br) * kGradUPitch + (blk & 1) * 16;
  for (int i = 0; i < nst; ++i) {
    cp_wait<RST - 2>();
    __syncthreads();
    stage(i + RST - 1);
    const uint8_t* s = sm + (i % RST) * kGradStage;
    uint32_t a[4];
    ldsm4t(a, s + uo);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t b[4];
      ldsm4t(b, s + yo + j * 32);
      mma16816(acc[2 * j], a, b[0], b[1]);
      mma16816(acc[2 * j + 1], a, b[2], b[3]);
    }
  }
  cp_wait<0>();
  __syncthreads();
  float* part = reinterpret_cast<float*>(sm);   // [warp][16][kGradC]
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      *reinterpret_cast<float2*>(part + (warp * 16 + g + 8 * h) * kGradC + 8 * j + 2 * t) =
          make_float2(acc[j][2 * h], acc[j][2 * h + 1]);
  __syncthreads();
  for (int e = threadIdx.x; e < 16 * kGradC; e += 32 * RW) {
    float v = part[e];
#pragma unroll
    for (int w = 1; w < RW; ++w) v += part[w * 16 * kGradC + e];
    part[e] = v;
  }
  if (nz > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  else __syncthreads();
#pragma unroll
  for (int u = 0; u < kGradE; ++u) {
    float* o;
    if (!out(u, &o)) continue;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(part) + 4u * (uint32_t)(e0 + 32 * RW * u);
    float x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      x[q] = 0.f;
      if (q < nz) {
        uint32_t ra;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(base), "r"(q));
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x[q]) : "r"(ra) : "memory");
      }
    }
    float v = x[0];
#pragma unroll
    for (int q = 1; q < 8; ++q) v += x[q];
    *o = old[u] + v;
  }
  // no CTA leaves while another still reads its shared memory
  if (nz > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

bool al16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

template <int MT>
bool launch_down(const bf16* X, const bf16* W, bf16* U, int N, int K, float scale, cudaStream_t s) {
  using C_ = DownCfg<MT>;
  static const bool attr =
      cudaFuncSetAttribute(rank16_k<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM) == cudaSuccess;
  if (!attr) {
    cudaGetLastError();
    return false;
  }
  note_launch(1);
  return launch_pdl(rank16_k<MT>, (N + 16 * MT - 1) / (16 * MT), 32 * RW, C_::SMEM, s, X, W, U, N, K, scale) == cudaSuccess;
}
}  // namespace

// 32 rows a CTA (W is read half as often) unless CTAs of 16 fit the SMs one each: there W comes from L2 beside an X
// that no other CTA of the SM waits for.
bool rank16_down(const void* X, const void* W, void* U, int N, int K, float scale, cudaStream_t s) {
  if (N < 1 || K < 8 || K % 8 != 0 || !al16(X) || !al16(W)) return false;
  const bf16 *x = (const bf16*)X, *w = (const bf16*)W;
  return (N + 15) / 16 <= sm_count() ? launch_down<1>(x, w, (bf16*)U, N, K, scale, s)
                                     : launch_down<2>(x, w, (bf16*)U, N, K, scale, s);
}

bool rank16_grad(const void* U, const void* Y, float* G, int N, int C, cudaStream_t s) {
  if (N < 1 || C < 8 || C % 8 != 0 || !al16(U) || !al16(Y)) return false;
  static const bool attr =
      cudaFuncSetAttribute(rank16_grad_k, cudaFuncAttributeMaxDynamicSharedMemorySize, kGradSmem) == cudaSuccess;
  if (!attr) {
    cudaGetLastError();
    return false;
  }
  // tokens shared by up to eight CTAs while all CTAs are resident at once (two per SM) and each has a full stage
  const int tiles = (C + kGradC - 1) / kGradC;
  int nz = 1;
  while (nz < 8 && tiles * nz * 2 <= 2 * sm_count() && N / (nz * 2) >= kGradT) nz *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tiles, (unsigned)nz);
  cfg.blockDim = dim3(32 * RW);
  cfg.dynamicSmemBytes = kGradSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 1;
  at[1].val.clusterDim.y = (unsigned)nz;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = nz > 1 ? 2 : 1;
  note_launch(1);
  return cudaLaunchKernelEx(&cfg, rank16_grad_k, (const bf16*)U, (const bf16*)Y, G, N, C, (N + nz - 1) / nz) == cudaSuccess;
}

}  // namespace zl
