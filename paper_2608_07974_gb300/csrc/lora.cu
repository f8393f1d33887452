// The skinny product of LoRA: 16 output columns, so the time is the reading of X once.
#include <algorithm>

#include "common.cuh"
#include "ops.h"

namespace zl {

namespace {
constexpr int RW = 8;   // warps per CTA, sharing the K range of 16 rows

__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A CTA forms 16 rows of U. Its warps take 32-deep chunks of K in turn (chunk c: warp c % 8, so neighbouring warps
// read neighbouring 64-byte pieces of a row) and add their partial sums in order at the end. The order of k inside
// a chunk does not matter as long as both operands agree on it, so every lane loads 16 contiguous bytes (eight k's,
// the four k pairs of two m16n8k16 steps) straight into its fragments: rows g and g + 8 of X, rows g and g + 8 of W.
// Bound by HBM (2 N K bytes); the tensor-core GEMM it replaces here ran one 128 x 64 tile column with most of
// its B tile padding, and a split-K reduction after it.
__global__ void __launch_bounds__(32 * RW) rank16_k(const bf16* __restrict__ X, const bf16* __restrict__ W,
                                                    bf16* __restrict__ U, int N, int K, float scale) {
  __shared__ float part[RW][16][17];
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int r0 = blockIdx.x * 16;
  const bf16* xa = X + (size_t)min(r0 + g, N - 1) * K + 8 * t;       // (rows past N are not stored)
  const bf16* xb = X + (size_t)min(r0 + g + 8, N - 1) * K + 8 * t;
  const bf16* wa = W + (size_t)g * K + 8 * t;
  const bf16* wb = W + (size_t)(g + 8) * K + 8 * t;
  const uint4 z = make_uint4(0, 0, 0, 0);
  float d0[4] = {}, d1[4] = {};
  constexpr int UN = 4;   // chunks in flight per warp
  for (int c = warp * 32; c < K; c += 32 * RW * UN) {
    uint4 a[UN], b[UN], p[UN], q[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const int k = c + u * 32 * RW;
      const bool ok = k + 8 * t < K;   // K % 8 == 0: a lane's eight k's are all inside or all outside
      a[u] = ok ? __ldg(reinterpret_cast<const uint4*>(xa + k)) : z;
      b[u] = ok ? __ldg(reinterpret_cast<const uint4*>(xb + k)) : z;
      p[u] = ok ? __ldg(reinterpret_cast<const uint4*>(wa + k)) : z;
      q[u] = ok ? __ldg(reinterpret_cast<const uint4*>(wb + k)) : z;
    }
#pragma unroll
    for (int u = 0; u < UN; ++u) {
      const uint32_t f0[4] = {a[u].x, b[u].x, a[u].y, b[u].y}, f1[4] = {a[u].z, b[u].z, a[u].w, b[u].w};
      mma16816(d0, f0, p[u].x, p[u].y);
      mma16816(d1, f0, q[u].x, q[u].y);
      mma16816(d0, f1, p[u].z, p[u].w);
      mma16816(d1, f1, q[u].z, q[u].w);
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    part[warp][g + 8 * (e >> 1)][2 * t + (e & 1)] = d0[e];
    part[warp][g + 8 * (e >> 1)][8 + 2 * t + (e & 1)] = d1[e];
  }
  __syncthreads();
  const int r = threadIdx.x >> 4, n = threadIdx.x & 15;
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < RW; ++w) s += part[w][r][n];
  if (r0 + r < N) U[(size_t)(r0 + r) * 16 + n] = __float2bfloat16_rn(s * scale);
}
}  // namespace

void launch_rank16(const void* X, const void* W, void* U, int N, int K, float scale, cudaStream_t s) {
  note_launch(1);
  launch_pdl(rank16_k, (N + 15) / 16, 32 * RW, 0, s, (const bf16*)X, (const bf16*)W, (bf16*)U, N, K, scale);
}

}  // namespace zl
