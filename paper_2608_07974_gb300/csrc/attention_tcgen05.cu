// Causal attention on the 5th-generation tensor cores (sm_103a), head dims 64 and 128: a one-pass forward
// with lazy rescaling and a two-kernel backward (dQ; dK and dV).
//
// A tile is 128 rows of one (batch, head), the longest tiles first: one CTA per tile in the forward, a deal of the
// tiles to one persistent CTA per SM in the backward. TMA brings a tile's
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

// ROWS rows x HD columns of one head from `m` (boxes of BOX rows) into a tile of HD / 64 blocks of [ROWS][64 columns].
template <int HD, int ROWS = 128, int BOX = 128>
__device__ __forceinline__ void load_tile(uint8_t* dst, const CUtensorMap* m, uint64_t* bar, int col, int row, int b) {
#pragma unroll
  for (int c = 0; c < HD / 64; ++c)
#pragma unroll
    for (int r = 0; r < ROWS; r += BOX) tma3d(dst + (c * ROWS + r) * 128, m, bar, col + 64 * c, row + r, b);
}

// D[128 x NB] = A[128 x HD] B[NB x HD]^T, both K-major tiles of load_tile.
template <int HD, int NB = 128>
__device__ __forceinline__ void mma_nt(uint32_t d, uint32_t a, uint32_t b) {
  constexpr uint32_t id = idesc_f16(128, NB, false, false);
#pragma unroll
  for (int ks = 0; ks < HD / 16; ++ks) {
    const uint32_t o = (ks % 4) * 32;
    mma_bf16(d, sdesc(a + (ks / 4) * 16384 + o, 16, 1024), sdesc(b + (ks / 4) * NB * 128 + o, 16, 1024), id,
             ks > 0 ? 1u : 0u);
  }
}

// D[128 x HD] (+)= A[128 x NB] B[NB x HD]: A in TMEM, each group of CW score columns holding its bf16
// pairs in the group's first CW / 2 columns; B a tile of load_tile read MN-major (16-row steps 2 KB apart).
template <int HD, int CW, int NB = 128>
__device__ __forceinline__ void mma_ta(uint32_t d, uint32_t a, uint32_t b, bool acc) {
  constexpr uint32_t id = idesc_f16(128, HD, false, true);
#pragma unroll
  for (int ks = 0; ks < NB / 16; ++ks)
    mma_bf16_ta(d, a + (ks * 16 / CW) * CW + (ks * 16 % CW) / 2, sdesc(b + ks * 2048, NB * 128, 1024), id,
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
// Forward, one pass with lazy rescaling. Per 64-key block j: S = Q K_j^T (TMEM), the softmax warps (a query
// row per thread) turn S into P = 2^(s - m) in place, O += P V_j. The running maximum m moves only
// when the block maximum exceeds it by more than 8 (log2 units): P then stays at most 256 (exact in fp32
// sums, the usual bf16 rounding), and O and the row sum l are rescaled (in TMEM / registers) only on such
// a move. At the end O / l is the softmax-weighted sum and m + log2 l the row's log-sum-exp.
// The first maximum is taken over two blocks, so that the largest of a row's first 128 probabilities is 1, which
// bf16 holds without rounding: the maximum of 64 keys alone makes the result's error against 64 bits 0.75% larger
// (2.045e-3 -> 2.060e-3 at B 2, S 1024, 32 heads of 128; 2.072e-3 -> 2.087e-3 at S 2048) and the forward 0.7 us
// faster at the shapes of GPT-2 (10.8 of 11.5) and 7B (20.5 of 21.2), 2.4 at B 4, S 2048 (92.3 of 94.7): the second
// block's product and reading are waited for before the first exponential. The first block kept in registers beside
// the second (168 registers) 94.9 and 21.8, K loaded a block ahead of V 94.3 and 21.2. l gathers a sum per block.
//
// Two score buffers: S of the next block is formed under this block's softmax, and two CTAs per SM (256 TMEM
// columns and at most 113 KB of shared memory each) fill each other's gaps. What bounds it: the softmax warps, two
// an SM quarter, whose block (about 1,450 cycles, of which 256 are the exponentials) is a chain of TMEM read,
// maximum, exponentials, TMEM write and hand-off. Measured against one score buffer of 128 keys and two softmax warps
// per quadrant (which fit beside it), all with the maximum of the first block alone: B 4, S 2048, 32 / 4 heads of 64
// 103 -> 92 us; B 2, S 1024, 32 heads of 128 22.7 -> 20.5 us; as it is 94.7 (726 TFLOP/s) and 21.2 (810), B 1, S 4096
// 110 us (1,245). On the same blocks: three buffers at head dim 64 93 us; two warps per quadrant, half a row each, 100 us; two groups of warps on alternate
// blocks, each with an O of its own, 98 us; one buffer and three CTAs 95 us.
// ==============================================================================================
template <int HD>
struct FCfg {
  static constexpr int KB = 64;                              // keys per block
  static constexpr int T = 128 * HD * 2, KT = KB * HD * 2;   // the Q tile, a K or V tile
  static constexpr int NST = HD == 64 ? 4 : 2;               // K and V buffers
  static constexpr int SMEM = T + NST * 2 * KT + 256 + 1024;
  static constexpr int NSW = 4;                              // softmax warps, one per TMEM lane quadrant
  static constexpr int NTHR = 64 + 32 * NSW;                 // TMA warp, MMA warp, softmax warps
  static constexpr uint32_t OCOL = 2 * KB, COLS = 256;       // two score buffers, O
  static_assert(2 * (SMEM + 1024) <= 233472, "two CTAs per SM");
  static_assert(OCOL + HD <= COLS, "TMEM columns");
};

template <int HD>
__global__ void __launch_bounds__(FCfg<HD>::NTHR, 2)
    attn_fwd_k(const __grid_constant__ CUtensorMap tqkv, const __grid_constant__ CUtensorMap tout,
               float* __restrict__ lse, int S, int H, int Hkv, float scale, unsigned* err) {
  using C_ = FCfg<HD>;
  constexpr int NST = C_::NST, KB = C_::KB;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sq = smem;                       // Q, at the end the staging of the output
  uint8_t* sk = sq + C_::T;                 // [NST] K
  uint8_t* sv = sk + NST * C_::KT;           // [NST] V
  uint64_t* kfull = (uint64_t*)(sv + NST * C_::KT);
  uint64_t* kempty = kfull + NST;
  uint64_t* vfull = kempty + NST;
  uint64_t* vempty = vfull + NST;
  uint64_t* qfull = vempty + NST;
  uint64_t* sfull = qfull + 1;    // [2], as pfull and pvdone: by block parity
  uint64_t* pfull = sfull + 2;
  uint64_t* pvdone = pfull + 2;
  uint64_t* fin = pvdone + 2;
  uint32_t* tbase = (uint32_t*)(fin + 1);
  volatile int* abort_flag = (volatile int*)(tbase + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.x, b = blockIdx.y, qb = gridDim.z - 1 - blockIdx.z;   // longest first
  const int kvh = h / (H / Hkv), q0 = qb * QB;
  const int nkb = (min(q0 + QB, S) + KB - 1) / KB;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&kfull[s], 1);
      mbar_init(&kempty[s], 1);
      mbar_init(&vfull[s], 1);
      mbar_init(&vempty[s], 1);
    }
    mbar_init(qfull, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sfull[s], 1);
      mbar_init(&pfull[s], C_::NSW);
      mbar_init(&pvdone[s], 1);
    }
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && lane < 2) prefetch_map(lane == 0 ? &tqkv : &tout);   // under the kernel before
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
      load_tile<HD, 128, KB>(sq, &tqkv, qfull, h * HD, q0, b);
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
        mbar_expect_tx(&kfull[st], C_::KT);
        load_tile<HD, KB, KB>(sk + st * C_::KT, &tqkv, &kfull[st], xk, j * KB, b);
      }
      __syncwarp();
      if (!uwait(&vempty[st], ph ^ 1u, abort_flag, err)) { ok = false; break; }
      vp[st] = (int)ph;
      if (leader) {
        mbar_expect_tx(&vfull[st], C_::KT);
        load_tile<HD, KB, KB>(sv + st * C_::KT, &tqkv, &vfull[st], xv, j * KB, b);
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
    // S of block j into its buffer, over P of block j - 2, which its P V product (issued before) reads first
    auto scores = [&](int j) {
      const int st = j % NST;
      if (!uwait(&kfull[st], (uint32_t)(j / NST) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD, KB>(tmem + (uint32_t)((j & 1) * KB), q_addr, k_addr + st * C_::KT);
        mma_commit(&sfull[j & 1]);
        mma_commit(&kempty[st]);
      }
      __syncwarp();
      return true;
    };
    ok = ok && scores(0) && (nkb == 1 || scores(1));
    for (int j = 0; ok && j < nkb; ++j) {
      const int st = j % NST;
      if (!uwait(&vfull[st], (uint32_t)(j / NST) & 1u, abort_flag, err) ||
          !uwait(&pfull[j & 1], (uint32_t)(j >> 1) & 1u, abort_flag, err)) {
        ok = false;
        break;
      }
      fence_after();
      if (leader) {
        mma_ta<HD, 32, KB>(tmem + C_::OCOL, tmem + (uint32_t)((j & 1) * KB), v_addr + st * C_::KT, j > 0);
        mma_commit(&vempty[st]);
        mma_commit(&pvdone[j & 1]);
      }
      __syncwarp();
      if (j + 2 < nkb && !scores(j + 2)) ok = false;
    }
    if (leader) mma_commit(fin);   // every MMA of the leader completes before TMEM is released
    __syncwarp();
  } else {
    // ---------------- softmax and output: a query row per thread ----------------
    const int quad = warp & 3;    // TMEM lane quadrant
    const int r = quad * 32 + lane, q = q0 + r;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    const float sl2 = scale * kL2e;
    const uint64_t SL2 = f2(sl2, sl2);
    bool ok = true;
    float m = -INFINITY;                                  // running maximum (log2 units)
    uint64_t l2 = f2(0.f, 0.f);                           // the row sum, in two parts
    for (int j = 0; j < nkb; ++j) {
      if (!uwait(&sfull[j & 1], (uint32_t)(j >> 1) & 1u, abort_flag, err)) { ok = false; break; }
      const uint32_t ts = trow + (uint32_t)((j & 1) * KB);
      uint32_t v[64];
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      fence_after();
      tmem_ld64u(ts, v);
      if (j + 2 >= nkb) {   // the diagonal blocks: keys after the query (and past the end) are masked
        const int kmax = min(q, S - 1) - j * KB;
#pragma unroll
        for (int e = 0; e < 64; ++e)
          if (e > kmax) v[e] = 0xff800000u;
      }
#pragma unroll
      for (int e = 0; e < 64; e += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) mx[u] = fmaxf(mx[u], __uint_as_float(v[e + u]));
      }
      if (j == 0 && nkb > 1) {   // the first maximum is that of 128 keys
        if (!uwait(&sfull[1], 0, abort_flag, err)) { ok = false; break; }
        fence_after();
#pragma unroll
        for (int c = 0; c < KB; c += 32) {
          uint32_t w[32];
          tmem_ld32u(ts + (uint32_t)(KB + c), w);
          if (nkb == 2) {
            const int kmax = min(q, S - 1) - KB - c;
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (e > kmax) w[e] = 0xff800000u;
          }
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) mx[u] = fmaxf(mx[u], __uint_as_float(w[e + u]));
          }
        }
      }
      const float mh = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sl2;
      const float mnew = fmaxf(m, mh);
      const bool move = mnew > m + 8.f;   // also true on the first block (m = -inf)
      if (j > 0 && __any_sync(0xffffffffu, move)) {   // rescale the O row (warp-wide TMEM access), P V of j - 1 in it
        if (!uwait(&pvdone[(j - 1) & 1], (uint32_t)((j - 1) >> 1) & 1u, abort_flag, err)) { ok = false; break; }
        fence_after();
        const float a = move ? ex2(m - mnew) : 1.f;
        l2 = mul2(l2, f2(a, a));
#pragma unroll 1
        for (int c = 0; c < HD; c += 32) {
          float o[32];
          tmem_ld32(trow + C_::OCOL + (uint32_t)c, o);
#pragma unroll
          for (int e = 0; e < 32; ++e) o[e] *= a;
          tmem_st32(trow + C_::OCOL + (uint32_t)c, o);
        }
      }
      if (move) m = mnew;
      const uint64_t NM = f2(-m, -m);
      uint64_t la = f2(0.f, 0.f), lb = la;   // the block's sum, in four parts
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
      if (lane == 0) mbar_arrive(&pfull[j & 1]);
      l2 = add2(l2, add2(la, lb));
    }
    // output: O / l, log-sum-exp m + log2 l
    const float l = uf2(l2).x + uf2(l2).y, inv = l > 0.f ? 1.f / l : 0.f;
    if (ok && uwait(&pvdone[(nkb - 1) & 1], (uint32_t)((nkb - 1) >> 1) & 1u, abort_flag, err)) {
      fence_after();
      store_rows(trow + C_::OCOL, inv, sq + quad * (HD / 64) * 4096, &tout, h * HD, q0 + quad * 32, b, S, 0, HD / 64,
                 lane);
      if (q < S) lse[((size_t)b * H + h) * S + q] = (l > 0.f ? m + log2f(l) : INFINITY) * kLn2;
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
// between the P and the dS phase of a block, and the products of the other operand run under each phase. Both
// kernels are persistent: a tile's loads and first products run under the last blocks of the one before.
// What bounds it: the P phase (about 1,100-1,400 cycles a block: TMEM reads, 512 cycles of exponentials, the
// conversion and the TMEM writes) and the hand-offs (about 280 cycles from the last warp's arrival to the next
// product, 400-550 from the last product to the warps). Measured against P and dS in shared memory (64-row
// blocks at head dim 128, one CTA per tile), both kernels together: B 2, S 1024, 32 heads of 128 127 -> 70 us; B 8,
// S 512, 12 heads of 64 46 -> 29 us; B 4, S 2048, 32 / 4 heads of 64 540 -> 280 us. One CTA per tile on the same
// blocks (each tile's loads 4,000-10,000 cycles, its output 2,500) 86, 35 and 300 us; eight elementwise warps of
// 64 columns 10-15% slower; the output by 32-byte stores from registers 2,000-4,600 cycles a tile in the dK / dV
// kernel (the dQ kernel, whose shared memory is full, keeps them: 300-1,900).
// ==============================================================================================
constexpr int NEW = 16;
constexpr int NTHR_DKV = 64 + 32 * NEW;
constexpr int NDW = 4;                        // warps of the dQ kernel that form D ahead of the tiles
constexpr int NTHR_DQ = NTHR_DKV + 32 * NDW;

template <int HD>
struct BCfg {
  static constexpr int T = 128 * HD * 2;
  // dQ kernel: K_j is held until its dQ product, V_j only until its dP product
  static constexpr int NK = HD == 64 ? 4 : 3, NV = HD == 64 ? 4 : 2;
  // Q, dO | K | V | D and -lse2 of two tiles | barriers (the tiles start at the 1024-byte aligned base)
  static constexpr int SMEM_DQ = (2 + NK + NV) * T + 4 * 128 * 4 + 320;
  // dK/dV kernel: stages of (Q_i, dO_i) with their statistics (-lse2, D), and score buffers
  static constexpr int NST = HD == 64 ? 4 : 2, NSB = HD == 64 ? 2 : 1;
  // K, V | stages | output staging, 2 KB per elementwise warp | statistics | barriers (1024-byte aligned base)
  static constexpr int SMEM_DKV = (2 + NST * 2) * T + NEW * 2048 + NST * 2 * 128 * 4 + 256;
  static_assert(SMEM_DQ <= 232448 && SMEM_DKV <= 232448, "shared memory per CTA");
  static_assert((NSB + 1) * 128 + 2 * HD <= 512, "TMEM columns");
};

// The n-th tile of CTA c among G: the tiles are sorted longest first and dealt out G at a time, the direction
// alternating between deals, so every CTA's long and short tiles even out; past the last tile it returns a
// value >= every tile count (every later deal is past it too).
__device__ __forceinline__ int snake_tile(int n, int c, int G) { return (n & 1) ? (n + 1) * G - 1 - c : n * G + c; }

// The tiles of the two kernels, longest first; at() gives tile t's head (or share), batch and 128-row block, blocks()
// its number of inner blocks. A role walks its CTA's tiles (first() / next()) and their blocks; its barrier phases
// follow its running block and tile counts.
struct QTiles {   // dQ: 128 queries of one head, key blocks 0 .. q
  int H, B, nqb;
  __device__ __forceinline__ int count() const { return H * B * nqb; }
  __device__ __forceinline__ void at(int t, int& x, int& b, int& q) const {
    const int r = t % (H * B);
    x = r % H;
    b = r / H;
    q = nqb - 1 - t / (H * B);
  }
  __device__ __forceinline__ int blocks(int t) const { return nqb - t / (H * B); }
};
struct KTiles {   // dK / dV: 128 keys of one KV head and `hpc` query heads, query blocks k .. of each
  int X, B, nqb, hpc;
  __device__ __forceinline__ int count() const { return X * B * nqb; }
  __device__ __forceinline__ void at(int t, int& x, int& b, int& k) const {
    const int r = t % (X * B);
    x = r % X;
    b = r / X;
    k = t / (X * B);
  }
  __device__ __forceinline__ int per_head(int t) const { return nqb - t / (X * B); }
};
__device__ __forceinline__ int nth_tile(int n) { return snake_tile(n, blockIdx.x, gridDim.x); }

// W bf16 of a row (packed words) to global memory; al32: 32-byte aligned rows (whole sectors per store).
template <int W>
__device__ __forceinline__ void store_words(bf16* p, const uint32_t* w, bool al32) {
#pragma unroll
  for (int e = 0; e < W; e += 8) {
    if (al32) {
      asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p + 2 * e), "r"(w[e]), "r"(w[e + 1]),
                   "r"(w[e + 2]), "r"(w[e + 3]), "r"(w[e + 4]), "r"(w[e + 5]), "r"(w[e + 6]), "r"(w[e + 7])
                   : "memory");
    } else {
      *reinterpret_cast<uint4*>(p + 2 * e) = make_uint4(w[e], w[e + 1], w[e + 2], w[e + 3]);
      *reinterpret_cast<uint4*>(p + 2 * e + 8) = make_uint4(w[e + 4], w[e + 5], w[e + 6], w[e + 7]);
    }
  }
}

// C fp32 TMEM columns at `t` (this lane's row), times f, as bf16 to `p` if `ok` (the TMEM reads are warp-wide).
template <int C>
__device__ __forceinline__ void store_cols(uint32_t t, float f, bf16* p, bool ok, bool al32) {
#pragma unroll
  for (int c = 0; c < C; c += 16) {
    float v[16];
    tmem_ld16(t + (uint32_t)c, v);
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack2(v[2 * e] * f, v[2 * e + 1] * f);
    if (ok) store_words<8>(p + c, w, al32);
  }
}

// dQ (and D) kernel, persistent. TMEM: S 0-127, dP two buffers 128-383, dQ 384 .. 384 + HD.
template <int HD>
__global__ void __launch_bounds__(NTHR_DQ, 1)
    attn_bwd_dq_k(const __grid_constant__ CUtensorMap tqkv, const __grid_constant__ CUtensorMap tdo,
                  const bf16* __restrict__ outp, const bf16* __restrict__ dout, const float* __restrict__ lse,
                  float* __restrict__ Dv, bf16* __restrict__ dqkv, int S, int B, int H, int Hkv, float scale,
                  unsigned* err) {
  using C_ = BCfg<HD>;
  constexpr int NK = C_::NK, NV = C_::NV;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* sq = smem;
  uint8_t* sdo = sq + C_::T;
  uint8_t* sk = sdo + C_::T;                      // [NK] K
  uint8_t* sv = sk + NK * C_::T;                  // [NV] V
  float* sD = (float*)(sv + NV * C_::T);          // [2][128] D, by tile parity
  float* sL = sD + 256;                           // [2][128] -lse2
  uint64_t* kfull = (uint64_t*)(sL + 256);
  uint64_t* kempty = kfull + NK;
  uint64_t* vfull = kempty + NK;
  uint64_t* vempty = vfull + NV;
  uint64_t* qfull = vempty + NV;
  uint64_t* qempty = qfull + 1;
  uint64_t* dofull = qempty + 1;
  uint64_t* doempty = dofull + 1;
  uint64_t* sfull = doempty + 1;
  uint64_t* sread = sfull + 1;                    // the elementwise warps have S in registers
  uint64_t* dpfull = sread + 1;                   // [2]
  uint64_t* dsfull = dpfull + 2;                  // [2] (the warps may be a block ahead of the MMA warp's wait)
  uint64_t* ofull = dsfull + 2;
  uint64_t* dfull = ofull + 1;                    // [2] D and -lse2 of a tile
  uint64_t* dempty = dfull + 2;                   // [2]
  uint64_t* fin = dempty + 2;
  uint32_t* tbase = (uint32_t*)(fin + 1);
  volatile int* abort_flag = (volatile int*)(tbase + 1);
  static_assert((2 * NK + 2 * NV + 16) * 8 + 8 <= 320, "barriers");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = H / Hkv;
  const QTiles tiles{H, B, (S + QB - 1) / QB};

  if (threadIdx.x == 0) {
    for (int s = 0; s < NK; ++s) { mbar_init(&kfull[s], 1); mbar_init(&kempty[s], 1); }
    for (int s = 0; s < NV; ++s) { mbar_init(&vfull[s], 1); mbar_init(&vempty[s], 1); }
    mbar_init(qfull, 1);
    mbar_init(qempty, 1);
    mbar_init(dofull, 1);
    mbar_init(doempty, 1);
    mbar_init(sfull, 1);
    mbar_init(sread, NEW);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&dpfull[s], 1);
      mbar_init(&dsfull[s], NEW);
      mbar_init(&dfull[s], NDW);
      mbar_init(&dempty[s], NEW);
    }
    mbar_init(ofull, 1);
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && lane < 2) prefetch_map(lane == 0 ? &tqkv : &tdo);   // under the kernel before
  if (warp == 1) tmem_alloc(tbase, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tbase;
  constexpr uint32_t DP = 128, DQ = 384;
  pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    const bool leader = elect_one();
    bool ok = true;
    int kp[NK], vp[NV], qp = -1, op = -1;   // parity of the last fill of each buffer, -1 if none
#pragma unroll
    for (int s = 0; s < NK; ++s) kp[s] = -1;
#pragma unroll
    for (int s = 0; s < NV; ++s) vp[s] = -1;
    int g = 0;
    for (int n = 0, t; ok && (t = nth_tile(n)) < tiles.count(); ++n) {
      int x, b, q;
      tiles.at(t, x, b, q);
      const int kvh = x / group, xk = (H + kvh) * HD, xv = (H + Hkv + kvh) * HD;
      const uint32_t nph = (uint32_t)n & 1u;
      // Q is free after the previous tile's last S product, dO after its last dP product
      if (!uwait(qempty, nph ^ 1u, abort_flag, err)) { ok = false; break; }
      qp = (int)nph;
      if (leader) {
        mbar_expect_tx(qfull, C_::T);
        load_tile<HD>(sq, &tqkv, qfull, x * HD, q * QB, b);
      }
      __syncwarp();
      for (int j = 0; j <= q; ++j, ++g) {
        const int ks = g % NK, vs = g % NV;
        const uint32_t kph = (uint32_t)(g / NK) & 1u, vph = (uint32_t)(g / NV) & 1u;
        if (!uwait(&kempty[ks], kph ^ 1u, abort_flag, err)) { ok = false; break; }
        kp[ks] = (int)kph;
        if (leader) {
          mbar_expect_tx(&kfull[ks], C_::T);
          load_tile<HD>(sk + ks * C_::T, &tqkv, &kfull[ks], xk, j * QB, b);
        }
        __syncwarp();
        if (j == 0) {
          if (!uwait(doempty, nph ^ 1u, abort_flag, err)) { ok = false; break; }
          op = (int)nph;
          if (leader) {
            mbar_expect_tx(dofull, C_::T);
            load_tile<HD>(sdo, &tdo, dofull, x * HD, q * QB, b);
          }
          __syncwarp();
        }
        if (!uwait(&vempty[vs], vph ^ 1u, abort_flag, err)) { ok = false; break; }
        vp[vs] = (int)vph;
        if (leader) {
          mbar_expect_tx(&vfull[vs], C_::T);
          load_tile<HD>(sv + vs * C_::T, &tqkv, &vfull[vs], xv, j * QB, b);
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) {   // unwinding: let the copies in flight land before the CTA exits
#pragma unroll
      for (int s = 0; s < NK; ++s) drain1(&kfull[s], kp[s]);
#pragma unroll
      for (int s = 0; s < NV; ++s) drain1(&vfull[s], vp[s]);
      drain1(qfull, qp);
      drain1(dofull, op);
    }
  } else if (warp == 1) {
    // S_{j+1} and dP_{j+1} are issued as soon as S_j has been read into registers, ahead of dQ += dS_j K_j, so they run
    // under the dS phase of block j; dP_{j+1} overwrites dS_{j-1}, whose product was issued before. The next tile's
    // first scores follow the tile's last dQ product (so that its loads hold nothing up). A tile's first dQ
    // product overwrites the accumulator: its dS phase follows the read-out of the tile before in every warp.
    const uint32_t q_addr = su32(sq), do_addr = su32(sdo), k_addr = su32(sk), v_addr = su32(sv);
    const bool leader = elect_one();   // issues every product and every commit that tracks them
    bool ok = true;
    auto scores = [&](int g, bool last) -> bool {   // S, then dP of block g; `last` of its tile
      const int ks = g % NK, vs = g % NV;
      if (!uwait(&kfull[ks], (uint32_t)(g / NK) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD>(tmem, q_addr, k_addr + ks * C_::T);
        mma_commit(sfull);
        if (last) mma_commit(qempty);
      }
      __syncwarp();
      if (!uwait(&vfull[vs], (uint32_t)(g / NV) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD>(tmem + DP + 128 * (g & 1), do_addr, v_addr + vs * C_::T);
        mma_commit(&dpfull[g & 1]);
        mma_commit(&vempty[vs]);
        if (last) mma_commit(doempty);
      }
      __syncwarp();
      return true;
    };
    int g = 0;
    for (int n = 0, t; ok && (t = nth_tile(n)) < tiles.count(); ++n) {
      const int nkb = tiles.blocks(t);
      const uint32_t nph = (uint32_t)n & 1u;
      if (!uwait(qfull, nph, abort_flag, err) || !uwait(dofull, nph, abort_flag, err) || !scores(g, nkb == 1)) {
        ok = false;
        break;
      }
      for (int j = 0; j < nkb; ++j, ++g) {
        if (j + 1 < nkb && (!uwait(sread, (uint32_t)g & 1u, abort_flag, err) || !scores(g + 1, j + 2 == nkb))) {
          ok = false;
          break;
        }
        if (!uwait(&dsfull[g & 1], (uint32_t)(g >> 1) & 1u, abort_flag, err)) { ok = false; break; }
        fence_after();
        if (leader) {
          const int ks = g % NK;
          mma_ta<HD, 32>(tmem + DQ, tmem + DP + 128 * (g & 1), k_addr + ks * C_::T, j > 0);
          mma_commit(&kempty[ks]);
          if (j == nkb - 1) mma_commit(ofull);
        }
        __syncwarp();
      }
    }
    if (leader) mma_commit(fin);
    __syncwarp();
  } else if (warp >= 2 + NEW) {
    // ---------------- D = rowsum(dO * O) and -lse2 of each tile, a tile or two ahead ----------------
    // 32 rows per warp: LR lanes per row, 16 bytes of O and dO each, four loads of each in flight
    constexpr int LR = HD / 8, RPL = 32 / LR, UN = 4;
    const int w = warp - 2 - NEW, sub = lane / LR;
    for (int n = 0, t; (t = nth_tile(n)) < tiles.count(); ++n) {
      int cx, cb, cq;
      tiles.at(t, cx, cb, cq);
      const int sb = n & 1, q0 = cq * QB;
      if (!uwait<true>(&dempty[sb], ((uint32_t)(n >> 1) & 1u) ^ 1u, abort_flag, err)) break;
      const int qr = q0 + 32 * w + lane;
      const size_t row0 = ((size_t)cb * H + cx) * S;
      sL[sb * 128 + 32 * w + lane] = qr < S ? -lse[row0 + qr] * kL2e : -INFINITY;
#pragma unroll 1
      for (int u0 = 0; u0 < 32; u0 += UN * RPL) {
        uint4 o4[UN], g4[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          const int row = min(q0 + 32 * w + u0 + u * RPL + sub, S - 1);
          const size_t o = ((size_t)cb * S + row) * ((size_t)H * HD) + (size_t)cx * HD + (lane % LR) * 8;
          o4[u] = *reinterpret_cast<const uint4*>(outp + o);
          g4[u] = *reinterpret_cast<const uint4*>(dout + o);
        }
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          const uint32_t ow[4] = {o4[u].x, o4[u].y, o4[u].z, o4[u].w}, gw[4] = {g4[u].x, g4[u].y, g4[u].z, g4[u].w};
          uint64_t acc = f2(0.f, 0.f);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc = fma2(bf2_to_f2(ow[e]), bf2_to_f2(gw[e]), acc);
          const float2 a2 = uf2(acc);
          float a = a2.x + a2.y;
#pragma unroll
          for (int x = LR / 2; x > 0; x >>= 1) a += __shfl_xor_sync(0xffffffffu, a, x);
          const int lr = 32 * w + u0 + u * RPL + sub;
          if (lane % LR == 0) {
            sD[sb * 128 + lr] = a;
            if (q0 + lr < S) Dv[row0 + q0 + lr] = a;
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&dfull[sb]);
    }
  } else {
    const int quad = warp & 3, qq = (warp - 2) >> 2;   // TMEM lane quadrant, 32-column quarter
    const int r = quad * 32 + lane;
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16), trow = tl + (uint32_t)(32 * qq);
    const uint64_t SL2 = f2(scale * kL2e, scale * kL2e);
    const int ld = (H + 2 * Hkv) * HD;
    const bool al32 = ((uintptr_t)dqkv & 31u) == 0;
    bool ok = true;
    int g = 0;
    for (int n = 0, t; ok && (t = nth_tile(n)) < tiles.count(); ++n) {
      const int nkb = tiles.blocks(t), db = n & 1;
      if (!uwait(&dfull[db], (uint32_t)(n >> 1) & 1u, abort_flag, err)) break;
      const float nl = sL[db * 128 + r], D = sD[db * 128 + r];
      const uint64_t NL = f2(nl, nl), DD = f2(D, D);
      __syncwarp();
      if (lane == 0) mbar_arrive(&dempty[db]);
      for (int j = 0; j < nkb; ++j, ++g) {
        const uint32_t gph = (uint32_t)g & 1u;
        if (!uwait(sfull, gph, abort_flag, err)) { ok = false; break; }
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
        if (!uwait(&dpfull[gph], (uint32_t)(g >> 1) & 1u, abort_flag, err)) { ok = false; break; }
        fence_after();
        const uint32_t tdp = trow + DP + 128u * gph;
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
        if (lane == 0) mbar_arrive(&dsfull[gph]);
      }
      if (!ok || !uwait(ofull, (uint32_t)n & 1u, abort_flag, err)) break;
      fence_after();
      int x, b, q;   // a quarter of dQ's columns per warp
      tiles.at(t, x, b, q);
      q = q * QB + r;
      store_cols<HD / 4>(tl + DQ + (uint32_t)(qq * (HD / 4)), scale,
                         dqkv + ((size_t)b * S + min(q, S - 1)) * ld + (size_t)x * HD + qq * (HD / 4), q < S, al32);
      fence_before();
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) tmem_release(fin, tmem, 512);
}

// dK / dV kernel, persistent. A tile is 128 keys of one KV head and `hpc` of its query heads (x = kvh * (group /
// hpc) + share): with hpc == group bf16 straight into dqkv, else fp32 partials part[2][shares of all KV
// heads][B * S][HD] (dK unscaled), summed per group afterwards. TMEM: NSB buffers of S^T / P^T, then dP^T /
// dS^T, dV, dK.
template <int HD>
__global__ void __launch_bounds__(NTHR_DKV, 1)
    attn_bwd_dkv_k(const __grid_constant__ CUtensorMap tqkv, const __grid_constant__ CUtensorMap tdo,
                   const __grid_constant__ CUtensorMap tdkv, const float* __restrict__ lse,
                   const float* __restrict__ Dv, int S, int B, int H, int Hkv, int hpc, float scale,
                   float* __restrict__ part, unsigned* err) {
  using C_ = BCfg<HD>;
  constexpr int NST = C_::NST, NSB = C_::NSB;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* sk = smem;
  uint8_t* sv = sk + C_::T;
  uint8_t* sst = sv + C_::T;                      // stage s: Q_i at s * 2 T, dO_i after it
  uint8_t* sout = sst + NST * 2 * C_::T;          // [NEW] output staging
  float* stats = (float*)(sout + NEW * 2048);     // stage s: -lse2[128], D[128]
  uint64_t* qfull = (uint64_t*)(stats + NST * 2 * 128);
  uint64_t* dofull = qfull + NST;
  uint64_t* empty = dofull + NST;
  uint64_t* kfull = empty + NST;
  uint64_t* kempty = kfull + 1;
  uint64_t* vfull = kempty + 1;
  uint64_t* vempty = vfull + 1;
  uint64_t* sfull = vempty + 1;                   // [NSB]
  uint64_t* pfull = sfull + NSB;                  // [NSB] (with two, a block ahead of the MMA warp's wait)
  uint64_t* dpfull = pfull + NSB;
  uint64_t* dsfull = dpfull + 1;
  uint64_t* ofull = dsfull + 1;
  uint64_t* fin = ofull + 1;
  uint32_t* tbase = (uint32_t*)(fin + 1);
  volatile int* abort_flag = (volatile int*)(tbase + 1);
  static_assert((3 * NST + 2 * NSB + 8) * 8 + 8 <= 256, "barriers");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int shares = H / Hkv / hpc, nqb = (S + QB - 1) / QB;
  const KTiles tiles{Hkv * shares, B, nqb, hpc};
  auto kv_head = [&](int x) { return x / shares; };
  auto q_head = [&](int x) { return x / shares * (H / Hkv) + x % shares * hpc; };   // the first of the tile's

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) { mbar_init(&qfull[s], 2); mbar_init(&dofull[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(kfull, 1);
    mbar_init(kempty, 1);
    mbar_init(vfull, 1);
    mbar_init(vempty, 1);
    for (int s = 0; s < NSB; ++s) { mbar_init(&sfull[s], 1); mbar_init(&pfull[s], NEW); }
    mbar_init(dpfull, 1);
    mbar_init(dsfull, NEW);
    mbar_init(ofull, 1);
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2 && lane < 2) prefetch_map(lane == 0 ? &tqkv : &tdo);   // under the kernel before
  if (warp == 1) tmem_alloc(tbase, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tbase;
  constexpr uint32_t DP = NSB * 128, DVC = DP + 128, DKC = DVC + HD;
  // Everything but D was complete before the dQ kernel, which this one follows, let it begin: only the warp that
  // reads D waits for that kernel to end (and with it this kernel ends after it).
  pdl_trigger();

  if (warp == 0) {
    // one elected lane: TMA of a tile's K and V and of (Q_i, dO_i) per block; every lane: four of the block's
    // -lse2 and D, loaded one block ahead
    const bool leader = elect_one();
    bool ok = true;
    int qp[NST], op[NST], kp = -1, vp = -1;   // parity of the last fill of each buffer, -1 if none
#pragma unroll
    for (int s = 0; s < NST; ++s) qp[s] = op[s] = -1;
    int st = 0;   // stage
    uint32_t ph = 0;
    int t = nth_tile(0), cx, cb, ck, h = 0, qi = 0;   // tile; the block's query head and query block
    tiles.at(t, cx, cb, ck);
    qi = ck;
    h = q_head(cx);
    float nl[4], dd[4];
    auto fetch = [&]() {
      const size_t row = ((size_t)cb * H + h) * S;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int qr = qi * QB + lane * 4 + u;
        nl[u] = qr < S ? -lse[row + qr] * kL2e : -INFINITY;
        dd[u] = qr < S ? Dv[row + qr] : 0.f;
      }
    };
    bool waited = false;
    for (int n = 0; ok && t < tiles.count(); ++n) {
      const int kvh = kv_head(cx), k0 = ck * QB, nit = hpc * (nqb - ck);
      const uint32_t nph = (uint32_t)n & 1u;
      // K is free after the previous tile's last S product, V after its last dP product
      if (!uwait(kempty, nph ^ 1u, abort_flag, err)) { ok = false; break; }
      kp = (int)nph;
      if (leader) {
        mbar_expect_tx(kfull, C_::T);
        load_tile<HD>(sk, &tqkv, kfull, (H + kvh) * HD, k0, cb);
      }
      __syncwarp();
      for (int it = 0; it < nit; ++it) {
        if (!uwait(&empty[st], ph ^ 1u, abort_flag, err)) { ok = false; break; }
        qp[st] = (int)ph;
        uint8_t* sb = sst + st * 2 * C_::T;
        if (leader) {
          mbar_expect_tx(&qfull[st], C_::T);
          load_tile<HD>(sb, &tqkv, &qfull[st], h * HD, qi * QB, cb);
        }
        __syncwarp();
        auto load_do = [&]() -> bool {   // V, then dO of the block
          if (it == 0) {
            if (!uwait(vempty, nph ^ 1u, abort_flag, err)) return false;
            vp = (int)nph;
            if (leader) {
              mbar_expect_tx(vfull, C_::T);
              load_tile<HD>(sv, &tqkv, vfull, (H + Hkv + kvh) * HD, k0, cb);
            }
            __syncwarp();
          }
          op[st] = (int)ph;
          if (leader) {
            mbar_expect_tx(&dofull[st], C_::T);
            load_tile<HD>(sb + C_::T, &tdo, &dofull[st], h * HD, qi * QB, cb);
          }
          __syncwarp();
          return true;
        };
        // D is the dQ kernel's: the first block's copies are issued (the very first V is free), then that kernel is
        // waited for; later the statistics, which complete qfull, come before the wait for V
        const bool start = !waited;
        if (start) {
          if (!load_do()) { ok = false; break; }
          pdl_wait();
          waited = true;
          fetch();
        }
        float* sl = stats + st * 256;
        *reinterpret_cast<float4*>(sl + lane * 4) = make_float4(nl[0], nl[1], nl[2], nl[3]);
        *reinterpret_cast<float4*>(sl + 128 + lane * 4) = make_float4(dd[0], dd[1], dd[2], dd[3]);
        __syncwarp();
        if (lane == 0) mbar_arrive(&qfull[st]);
        if (!start && !load_do()) { ok = false; break; }
        if (++st == NST) { st = 0; ph ^= 1u; }
        if (++qi == nqb) { qi = ck; ++h; }
        if (it + 1 < nit) fetch();
      }
      t = nth_tile(n + 1);
      if (t < tiles.count()) {
        tiles.at(t, cx, cb, ck);
        qi = ck;
        h = q_head(cx);
        if (ok) fetch();
      }
    }
    if (!waited) pdl_wait();   // (a CTA without tiles, or unwinding)
    if (!ok && lane == 0) {
#pragma unroll
      for (int s = 0; s < NST; ++s) {
        drain1(&qfull[s], qp[s]);   // (gives up after 100 ms where the statistics' arrival is missing)
        drain1(&dofull[s], op[s]);
      }
      drain1(kfull, kp);
      drain1(vfull, vp);
    }
  } else if (warp == 1) {
    // Order per block: dV += P_i dO_i, S_{i + NSB} over P_i, dK += dS_i Q_i, dP_{i+1} over dS_i. With two score buffers
    // S is always ready before its P phase begins; with one (head dim 128, where the accumulators take half of
    // TMEM) the dV product and S_{i+1} run under the dS phase. The next tile's first scores follow the tile's last
    // dK product. A tile's first dV and dK products overwrite the accumulators: its P phase follows the read-out
    // of the tile before in every warp.
    const uint32_t k_addr = su32(sk), v_addr = su32(sv), st_addr = su32(sst);
    const bool leader = elect_one();   // issues every product and every commit that tracks them
    auto scores = [&](int g, bool last) -> bool {   // S^T of block g into its buffer; `last` of its tile
      const int st = g % NST, sb = g % NSB;
      if (!uwait(&qfull[st], (uint32_t)(g / NST) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD>(tmem + 128 * sb, k_addr, st_addr + st * 2 * C_::T);
        mma_commit(&sfull[sb]);
        if (last) mma_commit(kempty);
      }
      __syncwarp();
      return true;
    };
    auto dprobs = [&](int g, bool last) -> bool {   // dP^T
      const int st = g % NST;
      if (!uwait(&dofull[st], (uint32_t)(g / NST) & 1u, abort_flag, err)) return false;
      fence_after();
      if (leader) {
        mma_nt<HD>(tmem + DP, v_addr, st_addr + st * 2 * C_::T + C_::T);
        mma_commit(dpfull);
        if (last) mma_commit(vempty);
      }
      __syncwarp();
      return true;
    };
    bool ok = true;
    int g = 0;
    for (int n = 0, t; ok && (t = nth_tile(n)) < tiles.count(); ++n) {
      const int nit = hpc * tiles.per_head(t);
      const uint32_t nph = (uint32_t)n & 1u;
      ok = uwait(kfull, nph, abort_flag, err) && scores(g, nit == 1) && uwait(vfull, nph, abort_flag, err) &&
           dprobs(g, nit == 1);
      if (NSB == 2 && ok && nit > 1) ok = scores(g + 1, nit == 2);
      for (int it = 0; ok && it < nit; ++it, ++g) {
        const int st = g % NST, sb = g % NSB;
        const uint32_t qa = st_addr + st * 2 * C_::T;
        if (!uwait(&pfull[sb], (uint32_t)(g / NSB) & 1u, abort_flag, err)) { ok = false; break; }
        fence_after();
        if (leader) mma_ta<HD, 32>(tmem + DVC, tmem + 128 * sb, qa + C_::T, it > 0);
        __syncwarp();
        if (it + NSB < nit && !scores(g + NSB, it + NSB + 1 == nit)) { ok = false; break; }
        if (!uwait(dsfull, (uint32_t)g & 1u, abort_flag, err)) { ok = false; break; }
        fence_after();
        if (leader) {
          mma_ta<HD, 32>(tmem + DKC, tmem + DP, qa, it > 0);
          mma_commit(&empty[st]);
          if (it == nit - 1) mma_commit(ofull);
        }
        __syncwarp();
        if (it + 1 < nit && !dprobs(g + 1, it + 2 == nit)) ok = false;
      }
    }
    if (leader) mma_commit(fin);
    __syncwarp();
  } else {
    const int quad = warp & 3, qq = (warp - 2) >> 2;     // TMEM lane quadrant, 32-column quarter
    const int r = quad * 32 + lane;                       // key row = TMEM lane
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16), trow = tl + (uint32_t)(32 * qq);
    const uint64_t SL2 = f2(scale * kL2e, scale * kL2e);
    // Only the causal mask is applied: queries >= S have -lse2 = -inf (P = 0) and D = 0, and rows of
    // keys >= S are never stored.
    bool ok = true;
    int g = 0, st = 0;   // running block; its stage
    uint32_t ph = 0;
    for (int n = 0, t; ok && (t = nth_tile(n)) < tiles.count(); ++n) {
      const int per_head = tiles.per_head(t), nit = hpc * per_head;
      for (int it = 0, qi = 0; it < nit; ++it, ++g) {
        const int sb = g % NSB;
        if (!uwait(&sfull[sb], (uint32_t)(g / NSB) & 1u, abort_flag, err)) { ok = false; break; }
        fence_after();
        // this stage's statistics: its qfull phase has completed (the S product waited on it); the wait orders
        // the producer's stores before these loads
        if (!uwait(&qfull[st], ph, abort_flag, err)) { ok = false; break; }
        const float4* sl4 = reinterpret_cast<const float4*>(stats + st * 256 + 32 * qq);
        const float4* sd4 = sl4 + 32;
        uint32_t p[32], pk[16];   // S, then P (fp32 bits)
        tmem_ld32u(trow + 128u * (uint32_t)sb, p);
        if (qi == 0) {   // the diagonal block: queries before the key are masked
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
        if (!uwait(dpfull, (uint32_t)g & 1u, abort_flag, err)) { ok = false; break; }
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
        if (++st == NST) { st = 0; ph ^= 1u; }
        if (++qi == per_head) qi = 0;
      }
      // half of dK's (qq 0, 1) or dV's (2, 3) columns per warp
      if (!ok || !uwait(ofull, (uint32_t)n & 1u, abort_flag, err)) break;
      fence_after();
      int cx, cb, ck;
      tiles.at(t, cx, cb, ck);
      const int which = qq >> 1, c0 = (qq & 1) * (HD / 2), key = ck * QB + r;
      const uint32_t tc = tl + (which ? DVC : DKC) + (uint32_t)c0;
      const size_t row = (size_t)cb * S + min(key, S - 1);
      if (part) {
        const size_t NS = (size_t)B * S;
        float* pr = part + ((which ? (size_t)tiles.X * NS : 0) + (size_t)cx * NS + row) * HD + c0;
#pragma unroll
        for (int e0 = 0; e0 < HD / 2; e0 += 16) {
          float v[16];
          tmem_ld16(tc + (uint32_t)e0, v);
          if (key < S) {
#pragma unroll
            for (int e = 0; e < 16; e += 4)
              *reinterpret_cast<float4*>(pr + e0 + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
          }
        }
      } else {
        const int x = ((which ? H + Hkv : H) + kv_head(cx)) * HD + c0, k0 = ck * QB + quad * 32;
        const float f = which ? 1.f : scale;
        uint8_t* box = sout + (warp - 2) * 2048;
#pragma unroll 1
        for (int e0 = 0; e0 < HD / 2; e0 += 32) {
          uint32_t u[32];
          tmem_ld32u(tc + (uint32_t)e0, u);
          if (lane == 0) bulk_wait_read0();   // this warp's last box has left the staging
          __syncwarp();
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              w[e] = pack2(__uint_as_float(u[8 * q4 + 2 * e]) * f, __uint_as_float(u[8 * q4 + 2 * e + 1]) * f);
            *reinterpret_cast<uint4*>(box + lane * 64 + ((q4 ^ ((lane >> 1) & 3)) << 4)) =
                make_uint4(w[0], w[1], w[2], w[3]);   // 64-byte swizzle
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (k0 < S) tma_store3d(&tdkv, box, x + e0, k0, cb);
            bulk_commit();
          }
        }
      }
      fence_before();
    }
    if (lane == 0) bulk_wait_read0();
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

// 3-D map over qkv viewed as [B][S][W] bf16 (W = (H + 2 Hkv) hd), box [1][rows][cols]: 64 columns in the 128-byte
// swizzle or 32 in the 64-byte one.
bool qkv_map(CUtensorMap* m, const void* qkv, int B, int S, int W, int rows, int cols = 64) {
  cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)S, (cuuint64_t)B};
  cuuint64_t strides[2] = {(cuuint64_t)W * 2, (cuuint64_t)S * W * 2};
  cuuint32_t box[3] = {(cuuint32_t)cols, (cuuint32_t)rows, 1u};
  cuuint32_t es[3] = {1, 1, 1};
  return g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(qkv), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Query heads per CTA of the dK / dV kernel, a divisor of the group: the one with the least predicted time (us). A KV
// head's whole group in one CTA needs no partials (fp32, written and read back), but its longest tile, every query
// block of every head, may outlast the SMs' mean share. A block takes about 1.2 us; the deal of shorter tiles
// ends within 3% of the mean (B 4, S 2048, 32 / 4 heads: 8 heads a CTA 324 us with the dQ kernel, 4 heads 334, one
// head 387).
int dkv_heads_per_cta(int B, int S, int Hkv, int group, int nqb, int hd) {
  const double mean = 0.5 * B * Hkv * (double)group * nqb * (nqb + 1) / g_nsm;   // blocks per SM
  int best = 1;
  double t = 1e30;
  for (int hpc = group; hpc >= 1; --hpc) {
    if (group % hpc != 0) continue;
    const double part = hpc < group ? 16.0 * Hkv * (group / hpc) * B * (double)S * hd / 6.6e6 + 2.5 : 0.0;
    const double c = 1.2 * std::max((double)hpc * nqb, 1.03 * mean) + part;
    if (c < 0.98 * t) { t = c; best = hpc; }
  }
  return best;
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
  CUtensorMap mq, mdo, mst;   // loads of 128-row boxes; stores of 32 x 32 boxes
  if (!qkv_map(&mq, qkv, B, S, W, 128) || !qkv_map(&mdo, dout, B, S, Wo, 128) || !qkv_map(&mst, dqkv, B, S, W, 32, 32))
    return false;
  const int nqb = (S + QB - 1) / QB, group = H / Hkv;
  const int hpc = dkv_heads_per_cta(B, S, Hkv, group, nqb, HD), shares = group / hpc;
  float* part = nullptr;
  if (shares > 1) {   // a KV head's query heads over several CTAs, then a fixed-order reduction
    const size_t bytes = 2ull * Hkv * shares * B * S * HD * sizeof(float);
    cudaError_t e = pool ? cudaMallocFromPoolAsync((void**)&part, bytes, pool, s) : cudaMallocAsync((void**)&part, bytes, s);
    if (e != cudaSuccess) { cudaGetLastError(); return false; }
  }
  auto grid = [&](long n) { return dim3((unsigned)std::min<long>(n, g_nsm)); };   // persistent: at most one CTA per SM
  cudaError_t e = launch_pdl(kq, grid((long)H * B * nqb), NTHR_DQ, C_::SMEM_DQ, s, mq, mdo, (const bf16*)out,
                             (const bf16*)dout, lse, D, (bf16*)dqkv, S, B, H, Hkv, scale, err);
  if (e == cudaSuccess)
    e = launch_pdl(kkv, grid((long)Hkv * shares * B * nqb), NTHR_DKV, C_::SMEM_DKV, s, mq, mdo, mst,
                   (const float*)lse, (const float*)D, S, B, H, Hkv, hpc, scale, part, err);
  if (part) {
    if (e == cudaSuccess) launch_reduce_dkv(part, dqkv, B * S, H, Hkv, shares, HD, scale, s);
    cudaFreeAsync(part, s);
  }
  if (e != cudaSuccess) return false;
  note_launch(part ? 3 : 2);
  return true;
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
  if (!qkv_map(&mq, qkv, B, S, (H + 2 * Hkv) * HD, C_::KB) || !qkv_map(&mo, out, B, S, H * HD, 32)) return false;
  if (launch_pdl(kern, dim3(H, B, (S + QB - 1) / QB), C_::NTHR, C_::SMEM, s, mq, mo, lse, S, H, Hkv, scale, err) != cudaSuccess)
    return false;
  note_launch(1);
  return true;
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
  return hd == 64 ? tg::fwd_launch<64>(qkv, out, lse, B, S, H, Hkv, s, err, scale)
                  : tg::fwd_launch<128>(qkv, out, lse, B, S, H, Hkv, s, err, scale);
}

// Returns false when the shape is outside these kernels (head dim 64 or 128, alignment, no sm_103a) or the
// grouped-head partials could not be allocated; the caller then uses the mma.sync kernels.
bool attn_bwd_tcgen05(const void* qkv, const void* out, const void* dout, const float* lse, float* D, void* dqkv,
                      int B, int S, int H, int Hkv, int hd, cudaStream_t s, cudaMemPool_t pool, unsigned* err,
                      float scale) {
  if (hd != 64 && hd != 128) return false;
  if ((((uintptr_t)qkv | (uintptr_t)out | (uintptr_t)dout | (uintptr_t)dqkv) & 15u) ||
      (long)B * H * ((S + 127) / 128) > 0x3fffffffL)   // tile numbers stay int, also past the last deal
    return false;
  if (!tg::enc_init()) return false;
  return hd == 64 ? tg::bwd_launch<64>(qkv, out, dout, lse, D, dqkv, B, S, H, Hkv, s, pool, err, scale)
                  : tg::bwd_launch<128>(qkv, out, dout, lse, D, dqkv, B, S, H, Hkv, s, pool, err, scale);
}

}  // namespace zl
