// Causal attention on the 5th-generation tensor cores (sm_103a), head dims 64 and 128: a one-pass forward
// with lazy rescaling and a two-kernel backward (dQ; dK and dV).
//
// A tile is 128 rows of one (batch, head), one CTA per tile, the longest tiles first. TMA brings a tile's
// fixed operands once and streams the 128-row blocks of the other side (128-byte swizzle; a 3-D tensor map
// over [batch, token, feature] reads rows past the sequence end as zeros); one elected lane of the MMA warp
// issues tcgen05.mma with fp32 accumulators in TMEM; the elementwise warps own TMEM lane quadrants (one row
// per thread). What the elementwise warps hand back to the tensor cores (P, dS) goes into TMEM as the A
// operand, over the scores that it was made from, so it never passes through shared memory. The products
// are issued in the order in which they depend on each other's TMEM columns, and the tensor pipe runs them
// in that order. Every mbarrier wait is bounded (about 2 s); on expiry the kernel raises ZL_DEVERR_TIMEOUT
// and unwinds.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "ops.h"
#include "tcgen05.cuh"

namespace zl {
namespace tg {
using namespace tc;

constexpr int QB = 128;     // rows of a tile and of a streamed block
constexpr float kL2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Bounded wait of a producer that unwinds: lets a copy it issued land before the CTA exits.
__device__ __forceinline__ void drain1(uint64_t* bar, int parity) {
  if (parity < 0) return;
  const unsigned long long t0 = gtimer();
  while (!mbar_test(bar, (uint32_t)parity) && gtimer() - t0 < 100000000ull) {
  }
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(dst)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

// Warp 1 after the final __syncthreads: waits (bounded) for the last MMAs, frees the TMEM.
__device__ __forceinline__ void tmem_release(uint64_t* fin, uint32_t tmem, uint32_t cols) {
  if ((threadIdx.x & 31) == 0) drain1(fin, 0);
  __syncwarp();
  fence_after();
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

// 128 rows x HD columns of one head from `m` into a tile of HD / 64 blocks of [128 rows][64 columns].
template <int HD>
__device__ __forceinline__ void load_tile(uint8_t* dst, const CUtensorMap* m, uint64_t* bar, int col, int row, int b) {
#pragma unroll
  for (int c = 0; c < HD / 64; ++c) tma3d(dst + c * 16384, m, bar, col + 64 * c, row, b);
}

// D[128 x 128] = A[128 x HD] B[128 x HD]^T, both K-major tiles of load_tile.
template <int HD>
__device__ __forceinline__ void mma_nt(uint32_t d, uint32_t a, uint32_t b) {
  constexpr uint32_t id = idesc_f16(128, 128, false, false);
#pragma unroll
  for (int ks = 0; ks < HD / 16; ++ks) {
    const uint32_t o = (ks / 4) * 16384 + (ks % 4) * 32;
    mma_bf16(d, sdesc(a + o, 16, 1024), sdesc(b + o, 16, 1024), id, ks > 0 ? 1u : 0u);
  }
}

// D[128 x HD] (+)= A[128 x 128] B[128 x HD]: A in TMEM, each group of CW score columns holding its bf16
// pairs in the group's first CW / 2 columns; B a tile of load_tile read MN-major (16-row steps 2 KB apart).
template <int HD, int CW>
__device__ __forceinline__ void mma_ta(uint32_t d, uint32_t a, uint32_t b, bool acc) {
  constexpr uint32_t id = idesc_f16(128, HD, false, true);
#pragma unroll
  for (int ks = 0; ks < 8; ++ks)
    mma_bf16_ta(d, a + (ks * 16 / CW) * CW + (ks * 16 % CW) / 2, sdesc(b + ks * 2048, 16384, 1024), id,
                (acc || ks > 0) ? 1u : 0u);
}

// This warp's 32 rows x HD fp32 columns at TMEM address `t` (this lane's row), times `f`, as bf16 through the
// staging area `st` (HD / 64 boxes of 32 rows x 128 bytes, 128-byte swizzle) to rows row0 .. of `m`; box c0
// .. c1 - 1 only. Rows past the sequence end are clipped by the map (a box with none inside is skipped).
__device__ __forceinline__ void store_rows(uint32_t t, float f, uint8_t* st, const CUtensorMap* m, int col, int row0,
                                           int b, int S, int c0, int c1, int lane) {
  for (int c = c0; c < c1; ++c) {
    uint8_t* box = st + c * 4096;
    uint32_t u[64];
    tmem_ld64u(t + (uint32_t)(64 * c), u);
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      uint32_t w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        w[e] = pack2(__uint_as_float(u[8 * p + 2 * e]) * f, __uint_as_float(u[8 * p + 2 * e + 1]) * f);
      *reinterpret_cast<uint4*>(box + lane * 128 + ((p ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    fence_async_smem();
    __syncwarp();
    if (lane == 0 && row0 < S) tma_store3d(m, box, col + 64 * c, row0, b);
  }
  if (lane == 0) {   // the staging area outlives the copies' reads of it; the writes land by the kernel's end
    bulk_commit();
    bulk_wait_read0();
  }
}

// ==============================================================================================
// Forward, one pass with lazy rescaling. Per 128-key block j: S = Q K_j^T (TMEM), the softmax warps (half
// a query row per thread, the two halves' maxima exchanged through shared memory) turn S into P =
// 2^(s - m) in place, O += P V_j. The running maximum m moves only
// when the block maximum exceeds it by more than 8 (log2 units): P then stays at most 256 (exact in fp32
// sums, the usual bf16 rounding), and O and the row sum l are rescaled (in TMEM / registers) only on such
// a move. At the end O / l is the softmax-weighted sum and m + log2 l the row's log-sum-exp.
//
// One block's chain S -> softmax -> P V is serial (S, P and O share 256 TMEM columns), and two CTAs per SM
// (256 columns and at most 113 KB of shared memory each) fill each other's gaps: while one is in its
// softmax, the other's products run. What bounds it: the softmax phase (about 1,450 cycles a block with its
// hand-offs, of which 512 are the exponentials) against 1,024 cycles of products at head dim 128. Measured
// against one persistent CTA per SM with P in shared memory: B 2, S 1024, 32 heads of 128 36.8 -> 22.7 us
// (755 TFLOP/s); B 1, S 4096 1,250 TFLOP/s; B 4, S 2048, 32 / 4 heads of 64 103 us (665 TFLOP/s). Four
// softmax warps with whole rows (no exchange) measured 1-3% slower.
// ==============================================================================================
template <int HD>
struct FCfg {
  static constexpr int T = 128 * HD * 2;                // one tile
  static constexpr int NST = HD == 64 ? 2 : 1;          // K and V buffers
  static constexpr int XBYTES = (2 * 2 * 128 + 2 * 128) * 4;   // maxima [2 buffers][2 halves][rows], sums [2][rows]
  static constexpr int SMEM = T + NST * 2 * T + XBYTES + 256 + 1024;
  static constexpr int NSW = 8;                         // softmax warps: two per lane quadrant, 64 keys each
  static constexpr int NTHR = 64 + 32 * NSW;            // TMA warp, MMA warp, softmax warps
  static constexpr uint32_t OCOL = 128, COLS = 256;
  static_assert(SMEM + 1024 <= 233472 / 2, "two CTAs per SM");
  static_assert(OCOL + HD <= COLS, "TMEM columns");
};

template <int HD>
__global__ void __launch_bounds__(FCfg<HD>::NTHR, 2)
    attn_fwd_k(const __grid_constant__ CUtensorMap tqkv, const __grid_constant__ CUtensorMap tout,
               float* __restrict__ lse, int S, int H, int Hkv, float scale, unsigned* err) {
  using C_ = FCfg<HD>;
  constexpr int NST = C_::NST;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sq = smem;                       // Q, at the end the staging of the output
  uint8_t* sk = sq + C_::T;                 // [NST] K
  uint8_t* sv = sk + NST * C_::T;           // [NST] V
  float* xmax = (float*)(sv + NST * C_::T);   // [2][2][128]
  float* xsum = xmax + 512;                   // [2][128]
  uint64_t* kfull = (uint64_t*)(xsum + 256);
  uint64_t* kempty = kfull + NST;
  uint64_t* vfull = kempty + NST;
  uint64_t* vempty = vfull + NST;
  uint64_t* qfull = vempty + NST;
  uint64_t* sfull = qfull + 1;
  uint64_t* pfull = sfull + 1;
  uint64_t* ofull = pfull + 1;
  uint64_t* fin = ofull + 1;
  uint32_t* tbase = (uint32_t*)(fin + 1);
  volatile int* abort_flag = (volatile int*)(tbase + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.x, b = blockIdx.y, qb = gridDim.z - 1 - blockIdx.z;   // longest first
  const int kvh = h / (H / Hkv), q0 = qb * QB, nkb = qb + 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&kfull[s], 1);
      mbar_init(&kempty[s], 1);
      mbar_init(&vfull[s], 1);
      mbar_init(&vempty[s], 1);
    }
    mbar_init(qfull, 1);
    mbar_init(sfull, 1);
    mbar_init(pfull, C_::NSW);
    mbar_init(ofull, 1);
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(tbase, C_::COLS);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tbase;
  pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    // ---------------- TMA producer (whole warp, one elected lane issues) ----------------
    const int xk = (H + kvh) * HD, xv = (H + Hkv + kvh) * HD;
    const bool leader = elect_one();
    if (leader) {
      mbar_expect_tx(qfull, C_::T);
      load_tile<HD>(sq, &tqkv, qfull, h * HD, q0, b);
    }
    bool ok = true;
    int kp[NST], vp[NST];   // parity of the last fill of each buffer, -1 if none
#pragma unroll
    for (int s = 0; s < NST; ++s) kp[s] = vp[s] = -1;
    for (int j = 0; ok && j < nkb; ++j) {
      const int st = j % NST;
      const uint32_t ph = (uint32_t)(j / NST) & 1u;
      if (!uwait(&kempty[st], ph ^ 1u, abort_flag, err)) { ok = false; break; }
      kp[st] = (int)ph;
      if (leader) {
        mbar_expect_tx(&kfull[st], C_::T);
        load_tile<HD>(sk + st * C_::T, &tqkv, &kfull[st], xk, j * QB, b);
      }
      __syncwarp();
      if (!uwait(&vempty[st], ph ^ 1u, abort_flag, err)) { ok = false; break; }
      vp[st] = (int)ph;
      if (leader) {
        mbar_expect_tx(&vfull[st], C_::T);
        load_tile<HD>(sv + st * C_::T, &tqkv, &vfull[st], xv, j * QB, b);
      }
      __syncwarp();
    }
    if (!ok && lane == 0) {   // unwinding: let the copies in flight land before the CTA exits
#pragma unroll
      for (int s = 0; s < NST; ++s) {
        drain1(&kfull[s], kp[s]);
        drain1(&vfull[s], vp[s]);
      }
      drain1(qfull, 0);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (whole warp, one elected lane issues and commits) ----------------
    const uint32_t q_addr = su32(sq), k_addr = su32(sk), v_addr = su32(sv);
    const bool leader = elect_one();
    bool ok = uwait(qfull, 0, abort_flag, err);
    for (int j = 0; ok && j < nkb; ++j) {
      const int st = j % NST;
      const uint32_t ph = (uint32_t)(j / NST) & 1u;
      if (!uwait(&kfull[st], ph, abort_flag, err)) { ok = false; break; }
      fence_after();
      if (leader) {   // over P of block j - 1, which its P V product (issued before) reads first
        mma_nt<HD>(tmem, q_addr, k_addr + st * C_::T);
        mma_commit(sfull);
        mma_commit(&kempty[st]);
      }
      __syncwarp();
      if (!uwait(&vfull[st], ph, abort_flag, err) || !uwait(pfull, (uint32_t)j & 1u, abort_flag, err)) {
        ok = false;
        break;
      }
      fence_after();
      if (leader) {
        mma_ta<HD, 32>(tmem + C_::OCOL, tmem, v_addr + st * C_::T, j > 0);
        mma_commit(&vempty[st]);
        if (j == nkb - 1) mma_commit(ofull);
      }
      __syncwarp();
    }
    if (leader) mma_commit(fin);   // every MMA of the leader completes before TMEM is released
    __syncwarp();
  } else {
    // ---------------- softmax and output: warps 2..9, half a query row per thread ----------------
    const int quad = warp & 3, half = (warp - 2) >> 2;    // TMEM lane quadrant; key half of every block
    const int r = quad * 32 + lane, q = q0 + r;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t ts = trow + (uint32_t)(64 * half);
    const float sl2 = scale * kL2e;
    const uint64_t SL2 = f2(sl2, sl2);
    // After a failed wait the loop only runs on over whatever TMEM holds (both warps of a quadrant pass every
    // named barrier); nothing is stored.
    bool ok = true;
    float m = -INFINITY;                                  // running maximum (log2 units)
    uint64_t la = f2(0.f, 0.f), lb = la;                  // this half's row sum, in four parts
    for (int j = 0; j < nkb; ++j) {
      if (ok && !uwait(sfull, (uint32_t)j & 1u, abort_flag, err)) ok = false;
      uint32_t v[64];
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      fence_after();
      tmem_ld64u(ts, v);
      if (j == nkb - 1) {   // the diagonal block: keys after the query (and past the end) are masked
        const int kmax = min(q, S - 1) - j * QB - 64 * half;
#pragma unroll
        for (int e = 0; e < 64; ++e)
          if (e > kmax) v[e] = 0xff800000u;
      }
#pragma unroll
      for (int e = 0; e < 64; e += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) mx[u] = fmaxf(mx[u], __uint_as_float(v[e + u]));
      }
      const float mh = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sl2;
      // the partner half's maximum (double-buffered by block parity; one barrier per block)
      float* xm = xmax + (j & 1) * 256;
      xm[half * 128 + r] = mh;
      asm volatile("bar.sync %0, 64;" ::"r"(1 + quad) : "memory");
      const float mnew = fmaxf(m, fmaxf(mh, xm[(1 - half) * 128 + r]));
      const bool move = mnew > m + 8.f;   // also true on the first block (m = -inf)
      // the previous P V product completed before this S, which was issued after it
      if (j > 0 && __any_sync(0xffffffffu, move)) {   // rescale this half of the O row (warp-wide TMEM access)
        const float a = move ? ex2(m - mnew) : 1.f;
        la = mul2(la, f2(a, a));
        lb = mul2(lb, f2(a, a));
#pragma unroll 1
        for (int c = half * (HD / 2); c < (half + 1) * (HD / 2); c += 32) {
          float o[32];
          tmem_ld32(trow + C_::OCOL + (uint32_t)c, o);
#pragma unroll
          for (int e = 0; e < 32; ++e) o[e] *= a;
          tmem_st32(trow + C_::OCOL + (uint32_t)c, o);
        }
      }
      if (move) m = mnew;
      const uint64_t NM = f2(-m, -m);
#pragma unroll
      for (int c = 0; c < 64; c += 32) {   // P of 32 keys into the first 16 of their 32 columns
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          const float2 x = uf2(fma2(f2(__uint_as_float(v[c + e]), __uint_as_float(v[c + e + 1])), SL2, NM));
          const float2 y = uf2(fma2(f2(__uint_as_float(v[c + e + 2]), __uint_as_float(v[c + e + 3])), SL2, NM));
          const float p0 = ex2(x.x), p1 = ex2(x.y), p2 = ex2(y.x), p3 = ex2(y.y);   // masked scores are -inf: 0
          la = add2(la, f2(p0, p1));
          lb = add2(lb, f2(p2, p3));
          pk[e / 2] = pack2(p0, p1);
          pk[e / 2 + 1] = pack2(p2, p3);
        }
        tmem_st16u(ts + (uint32_t)c, pk);
      }
      tmem_st_wait();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(pfull);
    }
    // output: both halves use the same m; O / (l_0 + l_1), log-sum-exp m + log2(l_0 + l_1)
    const float2 ls = uf2(add2(la, lb));
    xsum[half * 128 + r] = ls.x + ls.y;
    asm volatile("bar.sync %0, 64;" ::"r"(1 + quad) : "memory");
    const float lt = xsum[r] + xsum[128 + r];
    const float inv = lt > 0.f ? 1.f / lt : 0.f;
    if (ok && uwait(ofull, 0, abort_flag, err)) {
      fence_after();
      // one 64-column box per warp (head dim 64: the first warp of a quadrant has the only one)
      if (half < HD / 64)
        store_rows(trow + C_::OCOL, inv, sq + quad * (HD / 64) * 4096, &tout, h * HD, q0 + quad * 32, b, S, half,
                   half + 1, lane);
      if (q < S && half == 0) lse[((size_t)b * H + h) * S + q] = (lt > 0.f ? m + log2f(lt) : INFINITY) * kLn2;
    }
  }

  fence_before();
  __syncthreads();
  if (warp == 1) tmem_release(fin, tmem, C_::COLS);
}

// ==============================================================================================
// Backward: two kernels, each a fixed-order sum per output row (no atomics), 128-row blocks.
//   dQ kernel: one CTA per 128 queries; per key block j: S = Q K_j^T, dP = dO V_j^T,
//              dS = P * (dP - D), dQ += dS K_j; also writes D = rowsum(dO * O).
//   dK/dV kernel: one CTA per 128 keys of one KV head (and a share of its query heads); per query block i:
//              S^T = K Q_i^T, dP^T = V dO_i^T, dV += P^T dO_i, dK += dS^T Q_i.
// Sixteen elementwise warps, four per TMEM lane quadrant, 32 score columns each. P and dS go back into TMEM as
// bf16, over the scores they come from (each warp over its own columns), as the A operands of the
// accumulating products: nothing but the TMA tiles is in shared memory. The elementwise warps alternate
// between the P and the dS phase of a block, and the products of the other operand run under each phase.
// What bounds it: the P phase (about 1,100-1,400 cycles a block: TMEM reads, 512 cycles of exponentials, the
// conversion and the TMEM writes), the hand-offs (about 280 cycles from the last warp's arrival to the next
// product, 400-550 from the last product to the warps) and, at short sequences, each tile's first loads and
// its output. Measured against P and dS in shared memory (64-row blocks at head dim 128), both kernels
// together: B 2, S 1024, 32 heads of 128 127 -> 86 us; B 8, S 512, 12 heads of 64 46 -> 34.6 us; B 4, S 2048,
// 32 / 4 heads of 64 540 -> 300 us. Eight elementwise warps with 64 columns each measured 10-15% slower.
// ==============================================================================================
constexpr int NEW = 16;
constexpr int NTHR_B = 64 + 32 * NEW;

template <int HD>
struct BCfg {
  static constexpr int T = 128 * HD * 2;
  // dQ kernel: K_j is held until its dQ product, V_j only until its dP product
  static constexpr int NK = HD == 64 ? 4 : 3, NV = HD == 64 ? 4 : 2;
  static constexpr int SMEM_DQ = (2 + NK + NV) * T + 128 * 4 + 256 + 1024;   // Q, dO | K | V | D | barriers | align
  // dK/dV kernel: stages of (Q_i, dO_i) with their statistics (-lse2, D), and score buffers
  static constexpr int NST = HD == 64 ? 4 : 2, NSB = HD == 64 ? 2 : 1;
  static constexpr int SMEM_DKV = (2 + NST * 2) * T + NST * 2 * 128 * 4 + 256 + 1024;
  static_assert(SMEM_DQ <= 232448 && SMEM_DKV <= 232448, "shared memory per CTA");
  static_assert((NSB + 1) * 128 + 2 * HD <= 512, "TMEM columns");
};

// dQ (and D) kernel. TMEM: S 0-127, dP two buffers 128-383, dQ 384 .. 384 + HD.
template <int HD>
__global__ void __launch_bounds__(NTHR_B, 1)
    attn_bwd_dq_k(const __grid_constant__ CUtensorMap tqkv, const __grid_constant__ CUtensorMap tdo,
                  const __grid_constant__ CUtensorMap tdq, const bf16* __restrict__ outp,
                  const bf16* __restrict__ dout, const float* __restrict__ lse, float* __restrict__ Dv, int S, int H,
                  int Hkv, float scale, unsigned* err) {
  using C_ = BCfg<HD>;
  constexpr int NK = C_::NK, NV = C_::NV;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sq = smem;                             // Q, at the end the staging of dQ
  uint8_t* sdo = sq + C_::T;
  uint8_t* sk = sdo + C_::T;                      // [NK] K
  uint8_t* sv = sk + NK * C_::T;                  // [NV] V
  float* sD = (float*)(sv + NV * C_::T);          // [128] D
  uint64_t* kfull = (uint64_t*)(sD + 128);
  uint64_t* kempty = kfull + NK;
  uint64_t* vfull = kempty + NK;
  uint64_t* vempty = vfull + NV;
  uint64_t* qfull = vempty + NV;
  uint64_t* sfull = qfull + 1;
  uint64_t* sread = sfull + 1;                    // the elementwise warps have S in registers
  uint64_t* dpfull = sread + 1;                   // [2]
  uint64_t* dsfull = dpfull + 2;                  // [2] (the warps may be a block ahead of the MMA warp's wait)
  uint64_t* ofull = dsfull + 2;
  uint64_t* fin = ofull + 1;
  uint32_t* tbase = (uint32_t*)(fin + 1);
  volatile int* abort_flag = (volatile int*)(tbase + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.x, b = blockIdx.y, qb = gridDim.z - 1 - blockIdx.z;   // longest first
  const int kvh = h / (H / Hkv), q0 = qb * QB, nkb = qb + 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NK; ++s) { mbar_init(&kfull[s], 1); mbar_init(&kempty[s], 1); }
    for (int s = 0; s < NV; ++s) { mbar_init(&vfull[s], 1); mbar_init(&vempty[s], 1); }
    mbar_init(qfull, 1);
    mbar_init(sfull, 1);
    mbar_init(sread, NEW);
    mbar_init(&dpfull[0], 1);
    mbar_init(&dpfull[1], 1);
    mbar_init(&dsfull[0], NEW);
    mbar_init(&dsfull[1], NEW);
    mbar_init(ofull, 1);
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(tbase, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tbase;
  constexpr uint32_t DP = 128, DQ = 384;
  pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    const int xk = (H + kvh) * HD, xv = (H + Hkv + kvh) * HD;
    const bool leader = elect_one();
    if (leader) {
      mbar_expect_tx(qfull, 2 * C_::T);
      load_tile<HD>(sq, &tqkv, qfull, h * HD, q0, b);
      load_tile<HD>(sdo, &tdo, qfull, h * HD, q0, b);
    }
    bool ok = true;
    int kp[NK], vp[NV];   // parity of the last fill of each buffer, -1 if none
#pragma unroll
    for (int s = 0; s < NK; ++s) kp[s] = -1;
#pragma unroll
    for (int s = 0; s < NV; ++s) vp[s] = -1;
    for (int j = 0; j < nkb; ++j) {
      const int ks = j % NK, vs = j % NV;
      const uint32_t kph = (uint32_t)(j / NK) & 1u, vph = (uint32_t)(j / NV) & 1u;
      if (!uwait(&kempty[ks], kph ^ 1u, abort_flag, err)) { ok = false; break; }
      kp[ks] = (int)kph;
      if (leader) {
        mbar_expect_tx(&kfull[ks], C_::T);
        load_tile<HD>(sk + ks * C_::T, &tqkv, &kfull[ks], xk, j * QB, b);
      }
      __syncwarp();
      if (!uwait(&vempty[vs], vph ^ 1u, abort_flag, err)) { ok = false; break; }
      vp[vs] = (int)vph;
      if (leader) {
        mbar_expect_tx(&vfull[vs], C_::T);
        load_tile<HD>(sv + vs * C_::T, &tqkv, &vfull[vs], xv, j * QB, b);
      }
      __syncwarp();
    }
    if (!ok && lane == 0) {   // unwinding: let the copies in flight land before the CTA exits
#pragma unroll
      for (int s = 0; s < NK; ++s) drain1(&kfull[s], kp[s]);
#pragma unroll
      for (int s = 0; s < NV; ++s) drain1(&vfull[s], vp[s]);
      drain1(qfull, 0);
    }
  } else if (warp == 1) {
    // S_{j+1} and dP_{j+1} are issued as soon as S_j has been read into registers, ahead of dQ += dS_j K_j, so
    // they run under the dS phase of block j. dP_{j+1} overwrites dS_{j-1}, whose product was issued before.
    const uint32_t q_addr = su32(sq), do_addr = su32(sdo), k_addr = su32(sk), v_addr = su32(sv);
    const bool leader = elect_one();   // issues every product and every commit that tracks them
    bool ok = uwait(qfull, 0, abort_flag, err);
    auto scores = [&](int j) -> bool {   // S_j, then dP_j
      const int ks = j % NK, vs = j % NV;
      if (!uwait(&kfull[ks], (uint32_t)(j / NK) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD>(tmem, q_addr, k_addr + ks * C_::T);
        mma_commit(sfull);
      }
      __syncwarp();
      if (!uwait(&vfull[vs], (uint32_t)(j / NV) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD>(tmem + DP + 128 * (j & 1), do_addr, v_addr + vs * C_::T);
        mma_commit(&dpfull[j & 1]);
        mma_commit(&vempty[vs]);
      }
      __syncwarp();
      return true;
    };
    ok = ok && scores(0);
    for (int j = 0; ok && j < nkb; ++j) {
      if (j + 1 < nkb && (!uwait(sread, (uint32_t)j & 1u, abort_flag, err) || !scores(j + 1))) { ok = false; break; }
      if (!uwait(&dsfull[j & 1], (uint32_t)(j >> 1) & 1u, abort_flag, err)) { ok = false; break; }
      fence_after();
      if (leader) {
        const int ks = j % NK;
        mma_ta<HD, 32>(tmem + DQ, tmem + DP + 128 * (j & 1), k_addr + ks * C_::T, j > 0);
        mma_commit(&kempty[ks]);
      }
      __syncwarp();
    }
    if (leader) {
      if (ok) mma_commit(ofull);
      mma_commit(fin);
    }
    __syncwarp();
  } else {
    const int quad = warp & 3, qq = (warp - 2) >> 2;   // TMEM lane quadrant, 32-column quarter
    const int r = quad * 32 + lane;
    const int q = q0 + r;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(32 * qq);
    const size_t si = ((size_t)b * H + h) * S + min(q, S - 1);
    const float nlse2 = q < S ? -lse[si] * kL2e : -INFINITY;
    {   // D = rowsum(dO * O), eight rows per warp: LR lanes per row, 16 bytes of O and dO each
      constexpr int LR = HD / 8, RPL = 32 / LR;
      const int w = warp - 2, sub = lane / LR;
      uint4 o4[8 / RPL], g4[8 / RPL];
#pragma unroll
      for (int u = 0; u < 8 / RPL; ++u) {
        const int row = min(q0 + 8 * w + u * RPL + sub, S - 1);
        const size_t o = ((size_t)b * S + row) * ((size_t)H * HD) + (size_t)h * HD + (lane % LR) * 8;
        o4[u] = *reinterpret_cast<const uint4*>(outp + o);
        g4[u] = *reinterpret_cast<const uint4*>(dout + o);
      }
#pragma unroll
      for (int u = 0; u < 8 / RPL; ++u) {
        const uint32_t ow[4] = {o4[u].x, o4[u].y, o4[u].z, o4[u].w}, gw[4] = {g4[u].x, g4[u].y, g4[u].z, g4[u].w};
        uint64_t acc = f2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc = fma2(bf2_to_f2(ow[e]), bf2_to_f2(gw[e]), acc);
        const float2 a2 = uf2(acc);
        float a = a2.x + a2.y;
#pragma unroll
        for (int x = LR / 2; x > 0; x >>= 1) a += __shfl_xor_sync(0xffffffffu, a, x);
        const int lr = 8 * w + u * RPL + sub;
        if (lane % LR == 0) {
          sD[lr] = a;
          if (q0 + lr < S) Dv[((size_t)b * H + h) * S + q0 + lr] = a;
        }
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * NEW) : "memory");
    const float Dq = sD[r];
    const uint64_t SL2 = f2(scale * kL2e, scale * kL2e), NL = f2(nlse2, nlse2), DD = f2(Dq, Dq);
    bool ok = true;
    for (int j = 0; j < nkb; ++j) {
      if (!uwait(sfull, (uint32_t)j & 1u, abort_flag, err)) { ok = false; break; }
      fence_after();
      uint32_t p[32];   // S, then P (fp32 bits)
      tmem_ld32u(trow, p);
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sread);
      if (j == nkb - 1) {   // the diagonal block: keys after the query are masked
        const int kmax = r - 32 * qq;
#pragma unroll
        for (int e = 0; e < 32; ++e)
          if (e > kmax) p[e] = 0xff800000u;
      }
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        const float2 x = uf2(fma2(f2(__uint_as_float(p[e]), __uint_as_float(p[e + 1])), SL2, NL));
        p[e] = __float_as_uint(ex2(x.x));
        p[e + 1] = __float_as_uint(ex2(x.y));
      }
      if (!uwait(&dpfull[j & 1], (uint32_t)(j >> 1) & 1u, abort_flag, err)) { ok = false; break; }
      fence_after();
      const uint32_t tdp = trow + DP + 128u * (uint32_t)(j & 1);
      uint32_t dp[32], pk[16];
      tmem_ld32u(tdp, dp);
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        const float2 ds = uf2(mul2(f2(__uint_as_float(p[e]), __uint_as_float(p[e + 1])),
                                   sub2(f2(__uint_as_float(dp[e]), __uint_as_float(dp[e + 1])), DD)));
        pk[e / 2] = pack2(ds.x, ds.y);
      }
      tmem_st16u(tdp, pk);
      tmem_st_wait();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&dsfull[j & 1]);
    }
    if (ok && uwait(ofull, 0, abort_flag, err)) {
      fence_after();
      // one 64-column box for each of the quadrant's first HD / 64 warps
      if (qq < HD / 64)
        store_rows(tmem + ((uint32_t)(quad * 32) << 16) + DQ, scale, sq + quad * (HD / 64) * 4096, &tdq, h * HD,
                   q0 + quad * 32, b, S, qq, qq + 1, lane);
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) tmem_release(fin, tmem, 512);
}

// dK / dV kernel. One CTA per 128 keys of one KV head and `hpc` of its query heads (blockIdx.x = kvh *
// (group / hpc) + share): with hpc == group bf16 straight into dqkv, else fp32 partials part[2][shares of all
// KV heads][B * S][HD] (dK unscaled), summed per group afterwards. TMEM: NSB buffers of
// S^T / P^T, then dP^T / dS^T, dV, dK.
template <int HD>
__global__ void __launch_bounds__(NTHR_B, 1)
    attn_bwd_dkv_k(const __grid_constant__ CUtensorMap tqkv, const __grid_constant__ CUtensorMap tdo,
                   const __grid_constant__ CUtensorMap tdkv, const float* __restrict__ lse,
                   const float* __restrict__ Dv, int S, int H, int Hkv, int hpc, float scale, float* __restrict__ part,
                   unsigned* err) {
  using C_ = BCfg<HD>;
  constexpr int NST = C_::NST, NSB = C_::NSB;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sk = smem;                             // K and V, at the end the staging of dK and dV
  uint8_t* sv = sk + C_::T;
  uint8_t* sst = sv + C_::T;                      // stage s: Q_i at s * 2 T, dO_i after it
  float* stats = (float*)(sst + NST * 2 * C_::T); // stage s: -lse2[128], D[128]
  uint64_t* full = (uint64_t*)(stats + NST * 2 * 128);
  uint64_t* empty = full + NST;
  uint64_t* kvfull = empty + NST;
  uint64_t* sfull = kvfull + 1;                   // [NSB]
  uint64_t* pfull = sfull + NSB;                  // [NSB] (with two, a block ahead of the MMA warp's wait)
  uint64_t* dpfull = pfull + NSB;
  uint64_t* dsfull = dpfull + 1;
  uint64_t* ofull = dsfull + 1;
  uint64_t* fin = ofull + 1;
  uint32_t* tbase = (uint32_t*)(fin + 1);
  volatile int* abort_flag = (volatile int*)(tbase + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.y, kb = blockIdx.z;   // key block 0 (the longest) first
  const int shares = H / Hkv / hpc, kvh = blockIdx.x / shares;
  const int h0 = kvh * (H / Hkv) + (blockIdx.x % shares) * hpc;   // first query head
  const int k0 = kb * QB;
  const int per_head = (S + QB - 1) / QB - kb;     // query blocks kb .. : the causal ones
  const int nit = hpc * per_head;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) { mbar_init(&full[s], 2); mbar_init(&empty[s], 1); }
    mbar_init(kvfull, 1);
    for (int s = 0; s < NSB; ++s) mbar_init(&sfull[s], 1);
    for (int s = 0; s < NSB; ++s) mbar_init(&pfull[s], NEW);
    mbar_init(dpfull, 1);
    mbar_init(dsfull, NEW);
    mbar_init(ofull, 1);
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(tbase, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tbase;
  constexpr uint32_t DP = NSB * 128, DVC = DP + 128, DKC = DVC + HD;
  pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    // one elected lane: TMA of K, V once and of (Q_i, dO_i) per block; every lane: four of the block's
    // -lse2 and D, loaded one block ahead
    const bool leader = elect_one();
    if (leader) {
      mbar_expect_tx(kvfull, 2 * C_::T);
      load_tile<HD>(sk, &tqkv, kvfull, (H + kvh) * HD, k0, b);
      load_tile<HD>(sv, &tqkv, kvfull, (H + Hkv + kvh) * HD, k0, b);
    }
    int issued[NST];
#pragma unroll
    for (int s = 0; s < NST; ++s) issued[s] = -1;
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    float nl[4], dd[4];
    auto fetch = [&](int it) {
      const size_t row = ((size_t)b * H + h0 + it / per_head) * S;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int qq = (kb + it % per_head) * QB + lane * 4 + u;
        nl[u] = qq < S ? -lse[row + qq] * kL2e : -INFINITY;
        dd[u] = qq < S ? Dv[row + qq] : 0.f;
      }
    };
    fetch(0);
    for (int it = 0; it < nit; ++it) {
      const int h = h0 + it / per_head, qi0 = (kb + it % per_head) * QB;
      if (!uwait(&empty[stage], phase ^ 1u, abort_flag, err)) { ok = false; break; }
      issued[stage] = (int)phase;
      if (leader) {
        mbar_expect_tx(&full[stage], 2 * C_::T);
        uint8_t* st = sst + stage * 2 * C_::T;
        load_tile<HD>(st, &tqkv, &full[stage], h * HD, qi0, b);
        load_tile<HD>(st + C_::T, &tdo, &full[stage], h * HD, qi0, b);
      }
      float* sl = stats + stage * 256;
      *reinterpret_cast<float4*>(sl + lane * 4) = make_float4(nl[0], nl[1], nl[2], nl[3]);
      *reinterpret_cast<float4*>(sl + 128 + lane * 4) = make_float4(dd[0], dd[1], dd[2], dd[3]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[stage]);
      if (it + 1 < nit) fetch(it + 1);
      if (++stage == NST) { stage = 0; phase ^= 1u; }
    }
    if (!ok && lane == 0) {
#pragma unroll
      for (int s = 0; s < NST; ++s) drain1(&full[s], issued[s]);
      drain1(kvfull, 0);
    }
  } else if (warp == 1) {
    // Order per block: dV += P_i dO_i, S_{i + NSB} over P_i, dK += dS_i Q_i, dP_{i+1} over dS_i. With two score
    // buffers S is always ready before its P phase begins; with one (head dim 128, where the accumulators
    // take half of TMEM) the dV product and S_{i+1} run under the dS phase.
    const uint32_t k_addr = su32(sk), v_addr = su32(sv), st_addr = su32(sst);
    const bool leader = elect_one();   // issues every product and every commit that tracks them
    bool ok = uwait(kvfull, 0, abort_flag, err);
    auto scores = [&](int it) -> bool {   // S^T_it into its buffer
      const int st = it % NST, sb = it % NSB;
      if (!uwait(&full[st], (uint32_t)(it / NST) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD>(tmem + 128 * sb, k_addr, st_addr + st * 2 * C_::T);
        mma_commit(&sfull[sb]);
      }
      __syncwarp();
      return true;
    };
    auto dprobs = [&](int it) {   // dP^T_it (its stage has been waited for)
      if (leader) {
        mma_nt<HD>(tmem + DP, v_addr, st_addr + (it % NST) * 2 * C_::T + C_::T);
        mma_commit(dpfull);
      }
      __syncwarp();
    };
    ok = ok && scores(0);
    if (ok) dprobs(0);
    if (ok && NSB == 2 && nit > 1) ok = scores(1);
    for (int it = 0; ok && it < nit; ++it) {
      const int st = it % NST, sb = it % NSB;
      const uint32_t qa = st_addr + st * 2 * C_::T;
      if (!uwait(&pfull[sb], (uint32_t)(it / NSB) & 1u, abort_flag, err)) { ok = false; break; }
      fence_after();
      if (leader) mma_ta<HD, 32>(tmem + DVC, tmem + 128 * sb, qa + C_::T, it > 0);
      __syncwarp();
      if (it + NSB < nit && !scores(it + NSB)) { ok = false; break; }
      if (!uwait(dsfull, (uint32_t)it & 1u, abort_flag, err)) { ok = false; break; }
      fence_after();
      if (leader) {
        mma_ta<HD, 32>(tmem + DKC, tmem + DP, qa, it > 0);
        mma_commit(&empty[st]);
      }
      __syncwarp();
      if (it + 1 < nit) dprobs(it + 1);
    }
    if (leader) {
      if (ok) mma_commit(ofull);
      mma_commit(fin);
    }
    __syncwarp();
  } else {
    const int quad = warp & 3, qq = (warp - 2) >> 2;     // TMEM lane quadrant, 32-column quarter
    const int r = quad * 32 + lane;                       // key row = TMEM lane
    const int key = k0 + r;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(32 * qq);
    const uint64_t SL2 = f2(scale * kL2e, scale * kL2e);
    // Only the causal mask is applied: queries >= S have -lse2 = -inf (P = 0) and D = 0, and rows of
    // keys >= S are never stored.
    bool ok = true;
    for (int it = 0; it < nit; ++it) {
      const int stage = it % NST, sb = it % NSB;
      if (!uwait(&sfull[sb], (uint32_t)(it / NSB) & 1u, abort_flag, err)) { ok = false; break; }
      fence_after();
      // this stage's statistics: its full phase has completed (the S product waited on it); the wait orders
      // the producer's stores before these loads
      if (!uwait(&full[stage], (uint32_t)(it / NST) & 1u, abort_flag, err)) { ok = false; break; }
      const float4* sl4 = reinterpret_cast<const float4*>(stats + stage * 256 + 32 * qq);
      const float4* sd4 = sl4 + 32;
      uint32_t p[32], pk[16];   // S, then P (fp32 bits)
      tmem_ld32u(trow + 128u * (uint32_t)sb, p);
      if (it % per_head == 0) {   // the diagonal block: queries before the key are masked
        const int qlo = r - 32 * qq;
#pragma unroll
        for (int e = 0; e < 32; ++e)
          if (e < qlo) p[e] = 0xff800000u;
      }
#pragma unroll
      for (int e = 0; e < 32; e += 4) {
        const float4 l = sl4[e / 4];
        const float2 xa = uf2(fma2(f2(__uint_as_float(p[e]), __uint_as_float(p[e + 1])), SL2, f2(l.x, l.y)));
        const float2 xb = uf2(fma2(f2(__uint_as_float(p[e + 2]), __uint_as_float(p[e + 3])), SL2, f2(l.z, l.w)));
        const float p0 = ex2(xa.x), p1 = ex2(xa.y), p2 = ex2(xb.x), p3 = ex2(xb.y);
        p[e] = __float_as_uint(p0);
        p[e + 1] = __float_as_uint(p1);
        p[e + 2] = __float_as_uint(p2);
        p[e + 3] = __float_as_uint(p3);
        pk[e / 2] = pack2(p0, p1);
        pk[e / 2 + 1] = pack2(p2, p3);
      }
      tmem_st16u(trow + 128u * (uint32_t)sb, pk);
      tmem_st_wait();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&pfull[sb]);
      if (!uwait(dpfull, (uint32_t)it & 1u, abort_flag, err)) { ok = false; break; }
      fence_after();
      uint32_t dp[32];
      tmem_ld32u(trow + DP, dp);
#pragma unroll
      for (int e = 0; e < 32; e += 4) {
        const float4 d = sd4[e / 4];
        const float2 da = uf2(mul2(f2(__uint_as_float(p[e]), __uint_as_float(p[e + 1])),
                                   sub2(f2(__uint_as_float(dp[e]), __uint_as_float(dp[e + 1])), f2(d.x, d.y))));
        const float2 db = uf2(mul2(f2(__uint_as_float(p[e + 2]), __uint_as_float(p[e + 3])),
                                   sub2(f2(__uint_as_float(dp[e + 2]), __uint_as_float(dp[e + 3])), f2(d.z, d.w))));
        pk[e / 2] = pack2(da.x, da.y);
        pk[e / 2 + 1] = pack2(db.x, db.y);
      }
      tmem_st16u(trow + DP, pk);
      tmem_st_wait();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(dsfull);
    }
    if (ok && uwait(ofull, 0, abort_flag, err)) {
      fence_after();
      const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
      const int which = qq >> 1;   // 0 dK, 1 dV; two warps of the quadrant each
      const uint32_t tc = tl + (which ? DVC : DKC);
      if (part) {   // half of the columns per warp
        const size_t NS = (size_t)gridDim.y * S;
        float* pr = part + ((which ? (size_t)gridDim.x * NS : 0) + (size_t)blockIdx.x * NS + (size_t)b * S +
                            min(key, S - 1)) * HD;
        for (int c = (qq & 1) * (HD / 2); c < ((qq & 1) + 1) * (HD / 2); c += 32) {
          uint32_t u[32];
          tmem_ld32u(tc + (uint32_t)c, u);
          if (key < S) {
#pragma unroll
            for (int e = 0; e < 32; e += 4)
              *reinterpret_cast<uint4*>(pr + c + e) = make_uint4(u[e], u[e + 1], u[e + 2], u[e + 3]);
          }
        }
      } else if ((qq & 1) < HD / 64) {   // one 64-column box per warp
        const int x = (which ? H + Hkv + kvh : H + kvh) * HD;
        store_rows(tc, which ? 1.f : scale, (which ? sv : sk) + quad * (HD / 64) * 4096, &tdkv, x, k0 + quad * 32, b, S,
                   qq & 1, (qq & 1) + 1, lane);
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) tmem_release(fin, tmem, 512);
}

PFN_cuTensorMapEncodeTiled_v12000 g_enc = nullptr;
int g_nsm = 0;

bool enc_init() {
  static int avail = -1;
  if (avail >= 0) return avail == 1;
  avail = 0;
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  cudaDeviceGetAttribute(&g_nsm, cudaDevAttrMultiProcessorCount, dev);
  if (major != 10 || minor != 3 || g_nsm < 1) return false;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qr;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qr) != cudaSuccess ||
      qr != cudaDriverEntryPointSuccess || !fn)
    return false;
  g_enc = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  avail = 1;
  return true;
}

// 3-D map over qkv viewed as [B][S][W] bf16 (W = (H + 2 Hkv) hd), box [1][rows][64], 128-byte swizzle.
bool qkv_map(CUtensorMap* m, const void* qkv, int B, int S, int W, int rows) {
  cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)S, (cuuint64_t)B};
  cuuint64_t strides[2] = {(cuuint64_t)W * 2, (cuuint64_t)S * W * 2};
  cuuint32_t box[3] = {64u, (cuuint32_t)rows, 1u};
  cuuint32_t es[3] = {1, 1, 1};
  return g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(qkv), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Query heads per CTA of the dK / dV kernel, a divisor of the group: a KV head's whole group in one CTA needs
// no partials (fp32, 2 B S hd per query head, written and read back), but its longest tile (every query block
// of every head) must not outlast the others: at most 0.6 of an SM's mean share of the blocks.
int dkv_heads_per_cta(int B, int Hkv, int group, int nqb) {
  const double mean = 0.5 * B * Hkv * (double)group * nqb * (nqb + 1) / g_nsm;   // blocks per SM
  for (int hpc = group; hpc > 1; --hpc)
    if (group % hpc == 0 && (double)hpc * nqb <= 0.6 * mean) return hpc;
  return 1;
}

template <int HD>
bool bwd_launch(const void* qkv, const void* out, const void* dout, const float* lse, float* D, void* dqkv, int B,
                int S, int H, int Hkv, cudaStream_t s, cudaMemPool_t pool, unsigned* err, float scale) {
  using C_ = BCfg<HD>;
  static bool attr = false;
  auto kq = attn_bwd_dq_k<HD>;
  auto kkv = attn_bwd_dkv_k<HD>;
  if (!attr) {
    if (cudaFuncSetAttribute(kq, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM_DQ) != cudaSuccess ||
        cudaFuncSetAttribute(kkv, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM_DKV) != cudaSuccess)
      return false;
    attr = true;
  }
  const int W = (H + 2 * Hkv) * HD, Wo = H * HD;
  CUtensorMap mq, mdo, mst;   // loads of 128-row boxes; stores of 32-row boxes
  if (!qkv_map(&mq, qkv, B, S, W, 128) || !qkv_map(&mdo, dout, B, S, Wo, 128) || !qkv_map(&mst, dqkv, B, S, W, 32))
    return false;
  const int nqb = (S + QB - 1) / QB, group = H / Hkv;
  const int hpc = dkv_heads_per_cta(B, Hkv, group, nqb), shares = group / hpc;
  float* part = nullptr;
  if (shares > 1) {   // a KV head's query heads over several CTAs, then a fixed-order reduction
    const size_t bytes = 2ull * Hkv * shares * B * S * HD * sizeof(float);
    cudaError_t e = pool ? cudaMallocFromPoolAsync((void**)&part, bytes, pool, s) : cudaMallocAsync((void**)&part, bytes, s);
    if (e != cudaSuccess) { cudaGetLastError(); return false; }
  }
  cudaError_t e = launch_pdl(kq, dim3(H, B, nqb), NTHR_B, C_::SMEM_DQ, s, mq, mdo, mst, (const bf16*)out, (const bf16*)dout,
                             lse, D, S, H, Hkv, scale, err);
  if (e == cudaSuccess)
    e = launch_pdl(kkv, dim3(Hkv * shares, B, nqb), NTHR_B, C_::SMEM_DKV, s, mq, mdo, mst, (const float*)lse,
                   (const float*)D, S, H, Hkv, hpc, scale, part, err);
  if (part) {
    if (e == cudaSuccess) launch_reduce_dkv(part, dqkv, B * S, H, Hkv, shares, HD, scale, s);
    cudaFreeAsync(part, s);
  }
  return e == cudaSuccess;
}

template <int HD>
bool fwd_launch(const void* qkv, void* out, float* lse, int B, int S, int H, int Hkv, cudaStream_t s, unsigned* err,
                float scale) {
  using C_ = FCfg<HD>;
  static bool attr = false;
  auto kern = attn_fwd_k<HD>;
  if (!attr) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM) != cudaSuccess) return false;
    attr = true;
  }
  CUtensorMap mq, mo;
  if (!qkv_map(&mq, qkv, B, S, (H + 2 * Hkv) * HD, 128) || !qkv_map(&mo, out, B, S, H * HD, 32)) return false;
  return launch_pdl(kern, dim3(H, B, (S + QB - 1) / QB), C_::NTHR, C_::SMEM, s, mq, mo, lse, S, H, Hkv, scale, err) ==
         cudaSuccess;
}

}  // namespace tg

// Returns false when the shape is outside this kernel (head dim 64 or 128, alignment, no sm_103a); the
// caller uses the mma.sync kernel then. scale: the softmax scale (1 / sqrt of the true head dim when the
// heads are zero-padded up to hd).
bool attn_fwd_tcgen05(const void* qkv, void* out, float* lse, int B, int S, int H, int Hkv, int hd, cudaStream_t s,
                      unsigned* err, float scale) {
  if (hd != 64 && hd != 128) return false;
  if ((((uintptr_t)qkv | (uintptr_t)out) & 15u) || B > 65535 || (S + 127) / 128 > 65535) return false;
  if (!tg::enc_init()) return false;
  note_launch(1);
  return hd == 64 ? tg::fwd_launch<64>(qkv, out, lse, B, S, H, Hkv, s, err, scale)
                  : tg::fwd_launch<128>(qkv, out, lse, B, S, H, Hkv, s, err, scale);
}

// Returns false when the shape is outside these kernels (head dim 64 or 128, alignment, no sm_103a) or the
// grouped-head partials could not be allocated; the caller then uses the mma.sync kernels.
bool attn_bwd_tcgen05(const void* qkv, const void* out, const void* dout, const float* lse, float* D, void* dqkv,
                      int B, int S, int H, int Hkv, int hd, cudaStream_t s, cudaMemPool_t pool, unsigned* err,
                      float scale) {
  if (hd != 64 && hd != 128) return false;
  if ((((uintptr_t)qkv | (uintptr_t)out | (uintptr_t)dout | (uintptr_t)dqkv) & 15u) || B > 65535 ||
      (S + 127) / 128 > 65535)
    return false;
  if (!tg::enc_init()) return false;
  return hd == 64 ? tg::bwd_launch<64>(qkv, out, dout, lse, D, dqkv, B, S, H, Hkv, s, pool, err, scale)
                  : tg::bwd_launch<128>(qkv, out, dout, lse, D, dqkv, B, S, H, Hkv, s, pool, err, scale);
}

}  // namespace zl
