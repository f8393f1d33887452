// Causal softmax attention with grouped KV heads: the dispatch, the head padding of the tcgen05 kernels, and
// the CUDA-core version (fp32; bf16 where no tensor-core kernel takes the shape). Query head h reads KV
// head h / (H / Hkv). Scale 1/sqrt(hd). The forward saves the row log-sum-exp for the backward.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "ops.h"

namespace zl {

namespace {
// ------------------------------------------------------------------------------------------------
// CUDA-core kernels. A CTA works on 32 query (or key) rows of one head, LPR lanes per row (four; eight where a row
// would not fit four lanes' registers): lane `sub` holds the head dims 4 (LPR c + sub) .. + 3 (HDP: hd rounded up
// to 32, 64 or 128, zero padded). The other side comes in tiles of 32 rows through shared memory (read as 16-byte
// broadcasts), eight of its rows at a time (four in the backward), so that their dot products and shuffle steps are
// in flight together. A tile's rows are loaded into registers during the tile before, 16 bytes a load, because on
// small shapes the loads' latency is the kernel: with scalar loads between the barriers 4 x 64 tokens, 4 heads of
// 32 took 9.2 us forward and 14.4 us backward, with these 5.7 and 10.1 (2 x 512 tokens, 16 heads of 64 over 4: 139
// and 713, then 137 and 581: there shared-memory reads, one per four multiply-adds, are the bound).
// Masked rows of a diagonal tile (and, for dK and dV, rows past the end) are left out, not weighted with zero; the
// other tiles run a loop without masks, which gives back more than that costs: 5.8 and 9.8 us with zero weights, now
// 6.2 and 7.7 (137 and 569, now 137 and 400).
// One warp per row with one key at a time, which these replace, waited for five shuffles and a global load per
// key: 4 x 64 tokens, 4 heads of 32 (the tiny fp32 workload) is bound by that chain, not by its 17 MFLOP.
// ------------------------------------------------------------------------------------------------
constexpr int AR = 32;   // rows per CTA and per tile

template <int HDP>
constexpr int kLpr = HDP == 128 ? 8 : 4;   // lanes per row
template <int HDP>
struct RowV {
  static constexpr int L = kLpr<HDP>, NC = HDP / (4 * L), N = HDP / L;
  float v[N];
};

// This lane's part of a row of hd columns; `vec`: fp32 rows that start on 16 bytes, hd a multiple of four. All of a
// thread's loads are in flight together.
template <typename T, int HDP>
__device__ __forceinline__ void load_row(RowV<HDP>& o, const T* p, int hd, int sub, bool ok, bool vec) {
#pragma unroll
  for (int c = 0; c < RowV<HDP>::NC; ++c) {
    const int d = 4 * (RowV<HDP>::L * c + sub);
    if constexpr (std::is_same<T, float>::value) {
      if (vec) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok && d < hd) x = *reinterpret_cast<const float4*>(p + d);
        o.v[4 * c] = x.x;
        o.v[4 * c + 1] = x.y;
        o.v[4 * c + 2] = x.z;
        o.v[4 * c + 3] = x.w;
        continue;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) o.v[4 * c + q] = ok && d + q < hd ? to_f(p[d + q]) : 0.f;
  }
}
template <int HDP>
__device__ __forceinline__ void scale_row(RowV<HDP>& o, float f) {
#pragma unroll
  for (int d = 0; d < RowV<HDP>::N; ++d) o.v[d] *= f;
}
// Rotate-half RoPE of a row of HDP columns (hd = HDP), whose pairs (d, d + HDP / 2) lie in one lane: this lane's part
// of the position's (cos, sin) pairs, and the rotation as the separate pass rounds it (sg = -1: the inverse).
template <int HDP>
struct RopeV {
  float4 v[RowV<HDP>::NC];   // chunk c: pairs 4 (L c + sub) .. + 3
};
template <int HDP>
__device__ __forceinline__ void load_rope(RopeV<HDP>& t, const float2* cs, int pos, int sub) {
#pragma unroll
  for (int c = 0; c < RowV<HDP>::NC / 2; ++c) {
    const float4* p = reinterpret_cast<const float4*>(cs + (size_t)pos * (HDP / 2) + 4 * (RowV<HDP>::L * c + sub));
    t.v[2 * c] = p[0];
    t.v[2 * c + 1] = p[1];
  }
}
template <int HDP>
__device__ __forceinline__ void rotate_row(RowV<HDP>& o, const RopeV<HDP>& t, float sg) {
  constexpr int HN = RowV<HDP>::N / 2;
#pragma unroll
  for (int d = 0; d < HN; ++d) {
    const float4 p = t.v[d / 2];
    const float a = o.v[d], b = o.v[d + HN];
    rope_rot(a, b, d & 1 ? p.z : p.x, sg * (d & 1 ? p.w : p.y), o.v[d], o.v[d + HN]);
  }
}
// The row into an [AR][HDP + 4] tile.
template <int HDP>
__device__ __forceinline__ void put_row(float* tile, const RowV<HDP>& o, int row, int sub) {
#pragma unroll
  for (int c = 0; c < RowV<HDP>::NC; ++c)
    *reinterpret_cast<float4*>(tile + row * (HDP + 4) + 4 * (RowV<HDP>::L * c + sub)) =
        make_float4(o.v[4 * c], o.v[4 * c + 1], o.v[4 * c + 2], o.v[4 * c + 3]);
}
// The dot product of two rows, in each of the row's lanes.
template <int HDP>
__device__ __forceinline__ float dot_rows(const RowV<HDP>& a, const RowV<HDP>& b) {
  float x = 0.f;
#pragma unroll
  for (int d = 0; d < RowV<HDP>::N; ++d) x = fmaf(a.v[d], b.v[d], x);
#pragma unroll
  for (int m = 1; m < RowV<HDP>::L; m *= 2) x += __shfl_xor_sync(0xffffffffu, x, m);
  return x;
}
template <typename T, int HDP>
__device__ __forceinline__ void store_row(T* p, const RowV<HDP>& o, int hd, int sub, float scale) {
#pragma unroll
  for (int c = 0; c < RowV<HDP>::NC; ++c)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int d = 4 * (RowV<HDP>::L * c + sub) + q;
      if (d < hd) p[d] = from_f<T>(o.v[4 * c + q] * scale);
    }
}
constexpr int AF = 8, AB = 4;   // tile rows worked on at a time, forward and backward (eight spill there)
// The row's dot products with tile rows j .. j + U - 1, in every one of its lanes.
template <int HDP, int U>
__device__ __forceinline__ void dot_tile(float* s, const RowV<HDP>& a, const float* tile, int j, int sub) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const float* t = tile + (j + u) * (HDP + 4) + 4 * sub;
    float x = 0.f;
#pragma unroll
    for (int c = 0; c < RowV<HDP>::NC; ++c) {
      const float4 b = *reinterpret_cast<const float4*>(t + 4 * RowV<HDP>::L * c);
      x = fmaf(a.v[4 * c], b.x, x);
      x = fmaf(a.v[4 * c + 1], b.y, x);
      x = fmaf(a.v[4 * c + 2], b.z, x);
      x = fmaf(a.v[4 * c + 3], b.w, x);
    }
    s[u] = x;
  }
#pragma unroll
  for (int x = 1; x < RowV<HDP>::L; x *= 2)
#pragma unroll
    for (int u = 0; u < U; ++u) s[u] += __shfl_xor_sync(0xffffffffu, s[u], x);
}
// o += sum_u w[u] * tile row j + u. EDGE: over u from lo to hi - 1 only (a weight of zero would still turn a masked
// row's Inf or NaN into NaN).
template <int HDP, int U, bool EDGE>
__device__ __forceinline__ void axpy_tile(RowV<HDP>& o, const float* w, const float* tile, int j, int sub, int lo = 0, int hi = U) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (EDGE && (u < lo || u >= hi)) continue;
    const float* t = tile + (j + u) * (HDP + 4) + 4 * sub;
#pragma unroll
    for (int c = 0; c < RowV<HDP>::NC; ++c) {
      const float4 b = *reinterpret_cast<const float4*>(t + 4 * RowV<HDP>::L * c);
      o.v[4 * c] = fmaf(w[u], b.x, o.v[4 * c]);
      o.v[4 * c + 1] = fmaf(w[u], b.y, o.v[4 * c + 1]);
      o.v[4 * c + 2] = fmaf(w[u], b.z, o.v[4 * c + 2]);
      o.v[4 * c + 3] = fmaf(w[u], b.w, o.v[4 * c + 3]);
    }
  }
}

template <typename T, int HDP, bool ROPE>
__global__ void __launch_bounds__(AR * kLpr<HDP>) attn_fwd_k(const T* __restrict__ qkv, T* __restrict__ out, float* __restrict__ lse,
                                                  int S, int H, int Hkv, int hd, float scale, int nt, bool vec, const float2* __restrict__ cs) {
  __shared__ __align__(16) float ks[AR * (HDP + 4)], vs[AR * (HDP + 4)];
  pdl_wait();
  pdl_trigger();
  const int h = blockIdx.x / nt, b = blockIdx.y, i0 = (nt - 1 - (int)blockIdx.x % nt) * AR;   // long rows first
  const int ld = (H + 2 * Hkv) * hd, kvh = h / (H / Hkv), sub = threadIdx.x % kLpr<HDP>, row = threadIdx.x / kLpr<HDP>, i = i0 + row;
  const T* base = qkv + (size_t)b * S * ld;
  RowV<HDP> q, o, kn, vn;   // kn, vn: this thread's part of the next tile's rows, loaded during the tile before
  RopeV<HDP> tq, tn;        // and their rotations
  auto fetch = [&](int j) {
    const T* p = base + (size_t)min(j + row, S - 1) * ld + (H + kvh) * hd;
    load_row<T, HDP>(kn, p, hd, sub, j + row < S, vec);
    load_row<T, HDP>(vn, p + Hkv * hd, hd, sub, j + row < S, vec);
    if (ROPE) load_rope<HDP>(tn, cs, min(j + row, S - 1), sub);
  };
  load_row<T, HDP>(q, base + (size_t)min(i, S - 1) * ld + h * hd, hd, sub, i < S, vec);
  if (ROPE) load_rope<HDP>(tq, cs, min(i, S - 1), sub);
  fetch(0);
  if (ROPE) rotate_row<HDP>(q, tq, 1.f);
  scale_row<HDP>(q, scale);
#pragma unroll
  for (int d = 0; d < RowV<HDP>::N; ++d) o.v[d] = 0.f;
  float m = -INFINITY, l = 0.f;
  for (int j0 = 0; j0 <= i0; j0 += AR) {
    __syncthreads();
    if (ROPE) rotate_row<HDP>(kn, tn, 1.f);
    put_row<HDP>(ks, kn, row, sub);
    put_row<HDP>(vs, vn, row, sub);
    __syncthreads();
    if (j0 + AR <= i0) fetch(j0 + AR);
    auto keys = [&](auto edge) {   // the tile's keys, on the diagonal (edge) those up to the query
      constexpr bool EDGE = decltype(edge)::value;
#pragma unroll 1
      for (int j = 0; j < AR; j += AF) {
        float s[AF];
        dot_tile<HDP, AF>(s, q, ks, j, sub);
        const int n = i + 1 - j0 - j;   // visible keys from j on
        if (EDGE) {
#pragma unroll
          for (int u = 0; u < AF; ++u)
            if (u >= n) s[u] = -INFINITY;
        }
        float mn = m;
#pragma unroll
        for (int u = 0; u < AF; ++u) mn = fmaxf(mn, s[u]);
        if (!EDGE || n > 0) {   // past the row's last key a warp still runs for its other rows (a group of NaN scores has no maximum)
          const float corr = expf(m - mn);
#pragma unroll
          for (int u = 0; u < AF; ++u) s[u] = expf(s[u] - mn);
          float ls = 0.f;
#pragma unroll
          for (int u = 0; u < AF; u += 2) ls += s[u] + s[u + 1];
          l = l * corr + ls;
          scale_row<HDP>(o, corr);
          axpy_tile<HDP, AF, EDGE>(o, s, vs, j, sub, 0, n);
          m = mn;
        }
      }
    };
    if (j0 < i0) keys(std::false_type{});
    else keys(std::true_type{});
  }
  if (i >= S) return;
  store_row<T, HDP>(out + (size_t)(b * S + i) * H * hd + h * hd, o, hd, sub, 1.f / l);
  if (sub == 0) lse[((size_t)b * H + h) * S + i] = m + logf(l);
}

// Of head y's 2 nt blocks the first nt form dQ of 32 queries each, the others (y < Hkv) dK and dV of 32 keys of KV
// head y, summed over its query heads in order. D = rowsum(dO * O) is formed wherever a row needs it.
template <typename T, int HDP, bool ROPE>
__global__ void __launch_bounds__(AR * kLpr<HDP>) attn_bwd_k(const T* __restrict__ qkv, const T* __restrict__ out,
                                                  const T* __restrict__ dout, const float* __restrict__ lse,
                                                  T* __restrict__ dqkv, int S, int H, int Hkv, int hd, float scale,
                                                  int nt, bool vec, const float2* __restrict__ cs) {
  __shared__ __align__(16) float ta[AR * (HDP + 4)], tb[AR * (HDP + 4)];
  __shared__ float sl[AR], sd[AR];
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.y, sub = threadIdx.x % kLpr<HDP>, row = threadIdx.x / kLpr<HDP>;
  const int y = blockIdx.x / (2 * nt), x = blockIdx.x % (2 * nt);
  const int ld = (H + 2 * Hkv) * hd, lo = H * hd, rep = H / Hkv;
  const T* base = qkv + (size_t)b * S * ld;
  if (x < nt) {
    const int h = y, kvh = h / rep, i0 = (nt - 1 - x) * AR, i = i0 + row;
    RowV<HDP> q, g, dq, kn, vn;   // kn, vn: the next tile's rows
    RopeV<HDP> tq, tn;
    auto fetch = [&](int j) {
      const T* p = base + (size_t)min(j + row, S - 1) * ld + (H + kvh) * hd;
      load_row<T, HDP>(kn, p, hd, sub, j + row < S, vec);
      load_row<T, HDP>(vn, p + Hkv * hd, hd, sub, j + row < S, vec);
      if (ROPE) load_rope<HDP>(tn, cs, min(j + row, S - 1), sub);
    };
    const size_t io = (size_t)(b * S + min(i, S - 1)) * lo + h * hd;
    load_row<T, HDP>(q, base + (size_t)min(i, S - 1) * ld + h * hd, hd, sub, i < S, vec);
    load_row<T, HDP>(g, dout + io, hd, sub, i < S, vec);
    load_row<T, HDP>(dq, out + io, hd, sub, i < S, vec);
    const float L = lse[((size_t)b * H + h) * S + min(i, S - 1)];
    if (ROPE) load_rope<HDP>(tq, cs, min(i, S - 1), sub);
    fetch(0);
    if (ROPE) rotate_row<HDP>(q, tq, 1.f);
    scale_row<HDP>(q, scale);
    const float D = dot_rows<HDP>(dq, g);
#pragma unroll
    for (int d = 0; d < RowV<HDP>::N; ++d) dq.v[d] = 0.f;
    for (int j0 = 0; j0 <= i0; j0 += AR) {
      __syncthreads();
      if (ROPE) rotate_row<HDP>(kn, tn, 1.f);
      put_row<HDP>(ta, kn, row, sub);
      put_row<HDP>(tb, vn, row, sub);
      __syncthreads();
      if (j0 + AR <= i0) fetch(j0 + AR);
      auto keys = [&](auto edge) {   // as in the forward
        constexpr bool EDGE = decltype(edge)::value;
#pragma unroll 1
        for (int j = 0; j < AR; j += AB) {
          float s[AB], dp[AB];
          dot_tile<HDP, AB>(s, q, ta, j, sub);
          dot_tile<HDP, AB>(dp, g, tb, j, sub);
#pragma unroll
          for (int u = 0; u < AB; ++u) s[u] = expf(s[u] - L) * (dp[u] - D);
          axpy_tile<HDP, AB, EDGE>(dq, s, ta, j, sub, 0, i + 1 - j0 - j);
        }
      };
      if (j0 < i0) keys(std::false_type{});
      else keys(std::true_type{});
    }
    scale_row<HDP>(dq, scale);
    if (ROPE) rotate_row<HDP>(dq, tq, -1.f);
    if (i < S) store_row<T, HDP>(dqkv + (size_t)(b * S + i) * ld + h * hd, dq, hd, sub, 1.f);
    return;
  }
  if (y >= Hkv) return;
  const int kvh = y, j0 = (x - nt) * AR, j = j0 + row;
  RowV<HDP> k, v, dk, dv, qn, gn, on;   // qn, gn, on, ln: the next tile's query, dO and O rows and log-sum-exp
  RopeV<HDP> tk, tn;
  float ln;
  auto fetch = [&](int h, int i) {
    const bool ok = i + row < S;
    const size_t n = (size_t)min(i + row, S - 1);
    load_row<T, HDP>(qn, base + n * ld + h * hd, hd, sub, ok, vec);
    load_row<T, HDP>(gn, dout + ((size_t)b * S + n) * lo + h * hd, hd, sub, ok, vec);
    load_row<T, HDP>(on, out + ((size_t)b * S + n) * lo + h * hd, hd, sub, ok, vec);
    ln = ok ? lse[((size_t)b * H + h) * S + n] : INFINITY;
    if (ROPE) load_rope<HDP>(tn, cs, (int)n, sub);
  };
  load_row<T, HDP>(k, base + (size_t)min(j, S - 1) * ld + (H + kvh) * hd, hd, sub, j < S, vec);
  load_row<T, HDP>(v, base + (size_t)min(j, S - 1) * ld + (H + Hkv + kvh) * hd, hd, sub, j < S, vec);
  if (ROPE) load_rope<HDP>(tk, cs, min(j, S - 1), sub);
  fetch(kvh * rep, j0);
  if (ROPE) rotate_row<HDP>(k, tk, 1.f);
  scale_row<HDP>(k, scale);
#pragma unroll
  for (int d = 0; d < RowV<HDP>::N; ++d) dk.v[d] = dv.v[d] = 0.f;
  for (int hh = 0; hh < rep; ++hh) {
    const int h = kvh * rep + hh;
    for (int i0 = j0; i0 < S; i0 += AR) {
      __syncthreads();
      if (ROPE) rotate_row<HDP>(qn, tn, 1.f);
      put_row<HDP>(ta, qn, row, sub);
      put_row<HDP>(tb, gn, row, sub);
      const float D = dot_rows<HDP>(on, gn);
      if (sub == 0) {
        sd[row] = D;
        sl[row] = ln;
      }
      __syncthreads();
      if (i0 + AR < S) fetch(h, i0 + AR);
      else if (hh + 1 < rep) fetch(h + 1, j0);
      auto queries = [&](auto edge) {   // the tile's queries, on the diagonal and at the end (edge) those from the key on that exist
        constexpr bool EDGE = decltype(edge)::value;
#pragma unroll 1
        for (int i = 0; i < AR; i += AB) {
          float s[AB], dp[AB];
          dot_tile<HDP, AB>(s, k, ta, i, sub);
          dot_tile<HDP, AB>(dp, v, tb, i, sub);
#pragma unroll
          for (int u = 0; u < AB; ++u) {
            s[u] = expf(s[u] - sl[i + u]);
            dp[u] = s[u] * (dp[u] - sd[i + u]);
          }
          axpy_tile<HDP, AB, EDGE>(dv, s, tb, i, sub, j - i0 - i, S - i0 - i);
          axpy_tile<HDP, AB, EDGE>(dk, dp, ta, i, sub, j - i0 - i, S - i0 - i);
        }
      };
      if (j0 < i0 && i0 + AR <= S) queries(std::false_type{});
      else queries(std::true_type{});
    }
  }
  scale_row<HDP>(dk, scale);
  if (ROPE) rotate_row<HDP>(dk, tk, -1.f);
  if (j < S) {
    store_row<T, HDP>(dqkv + (size_t)(b * S + j) * ld + (H + kvh) * hd, dk, hd, sub, 1.f);
    store_row<T, HDP>(dqkv + (size_t)(b * S + j) * ld + (H + Hkv + kvh) * hd, dv, hd, sub, 1.f);
  }
}

template <typename T, int HDP, bool ROPE = false>
void cuda_core_fwd(const void* qkv, void* out, float* lse, int B, int S, int H, int Hkv, int hd, float scale,
                   cudaStream_t s, const float* cs = nullptr) {
  const int nt = (S + AR - 1) / AR;
  const bool vec = std::is_same<T, float>::value && hd % 4 == 0 && ((uintptr_t)qkv & 15u) == 0;
  launch_pdl(attn_fwd_k<T, HDP, ROPE>, dim3((unsigned)H * nt, B), AR * kLpr<HDP>, 0, s, (const T*)qkv, (T*)out, lse, S, H,
             Hkv, hd, scale, nt, vec, (const float2*)cs);
}
template <typename T, int HDP, bool ROPE = false>
void cuda_core_bwd(const void* qkv, const void* out, const void* dout, const float* lse, void* dqkv, int B, int S, int H,
                   int Hkv, int hd, float scale, cudaStream_t s, const float* cs = nullptr) {
  const int nt = (S + AR - 1) / AR;
  const bool vec = std::is_same<T, float>::value && hd % 4 == 0 &&
                   (((uintptr_t)qkv | (uintptr_t)out | (uintptr_t)dout) & 15u) == 0;
  launch_pdl(attn_bwd_k<T, HDP, ROPE>, dim3((unsigned)H * 2 * nt, B), AR * kLpr<HDP>, 0, s, (const T*)qkv, (const T*)out,
             (const T*)dout, lse, (T*)dqkv, S, H, Hkv, hd, scale, nt, vec, (const float2*)cs);
}

// Head padding for the tcgen05 kernels (head dims 64 and 128): dst [N, nh * hp] from src [N, nh * hd] with
// each head's columns hd .. hp - 1 zero (pad), or src [N, nh * hp] back to dst [N, nh * hd] (unpad).
// Zero query and key columns add nothing to Q K^T, zero value columns give zero output columns, and the
// gradients of the padding columns are zero, so the padded products are the unpadded ones. bf16 pairs.
__global__ void heads_pad_k(const __nv_bfloat162* __restrict__ src, __nv_bfloat162* __restrict__ dst, int N, int nh,
                            int hd, int hp, int pad) {
  pdl_wait();
  pdl_trigger();
  const int h2 = hd / 2, p2 = hp / 2;
  const int src_w = (pad ? h2 : p2) * nh, dst_w = (pad ? p2 : h2) * nh, cols = nh * (pad ? p2 : h2);
  const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
  for (int n = blockIdx.x; n < N; n += gridDim.x) {
    const __nv_bfloat162* sr = src + (size_t)n * src_w;
    __nv_bfloat162* dr = dst + (size_t)n * dst_w;
    for (int c = threadIdx.x; c < cols; c += blockDim.x) {
      if (pad) {
        const int h = c / p2, e = c - h * p2;
        dr[c] = e < h2 ? sr[h * h2 + e] : zero;
      } else {
        const int h = c / h2, e = c - h * h2;
        dr[c] = sr[h * p2 + e];
      }
    }
  }
}

void heads_pad(const void* src, void* dst, int N, int nh, int hd, int hp, bool pad, cudaStream_t s) {
  note_launch(1);
  launch_pdl(heads_pad_k, std::min(N, 152 * 16), 256, 0, s, (const __nv_bfloat162*)src, (__nv_bfloat162*)dst, N, nh, hd,
             hp, pad ? 1 : 0);
}

// The tcgen05 head dim a bf16 head of hd columns is padded to, or 0 when it runs as it is (64, 128) or
// on the mma.sync kernels (odd, or above 128).
int padded_hd(int hd) {
  if (hd == 64 || hd == 128 || hd % 2 != 0 || hd > 128) return 0;
  return hd < 64 ? 64 : 128;
}

void* scratch(size_t bytes, cudaStream_t s, cudaMemPool_t pool) {
  void* p = nullptr;
  const cudaError_t e = pool ? cudaMallocFromPoolAsync(&p, bytes, pool, s) : cudaMallocAsync(&p, bytes, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return p;
}
}  // namespace

bool attn_fwd_tc(const void* qkv, void* out, float* lse, int B, int S, int H, int Hkv, int hd, cudaStream_t s);
bool attn_fwd_tcgen05(const void* qkv, void* out, float* lse, int B, int S, int H, int Hkv, int hd, cudaStream_t s,
                      unsigned* err, float scale);
bool attn_bwd_tc(const void* qkv, const void* out, const void* dout, const float* lse, float* D, void* dqkv, int B, int S,
                 int H, int Hkv, int hd, cudaStream_t s, cudaMemPool_t pool);
bool attn_bwd_tcgen05(const void* qkv, const void* out, const void* dout, const float* lse, float* D, void* dqkv,
                      int B, int S, int H, int Hkv, int hd, cudaStream_t s, cudaMemPool_t pool, unsigned* err,
                      float scale);

namespace {
// bf16 heads of a dim the tcgen05 kernels do not take: zero-padded copies through them (padded_hd).
bool attn_fwd_padded(const void* qkv, void* out, float* lse, int B, int S, int H, int Hkv, int hd, cudaStream_t s,
                     unsigned* err, cudaMemPool_t pool) {
  const int hp = padded_hd(hd), N = B * S, nh = H + 2 * Hkv;
  if (!hp) return false;
  void* qp = scratch((size_t)N * nh * hp * 2, s, pool);
  void* op = qp ? scratch((size_t)N * H * hp * 2, s, pool) : nullptr;
  bool ok = op != nullptr;
  if (ok) {
    heads_pad(qkv, qp, N, nh, hd, hp, true, s);
    ok = attn_fwd_tcgen05(qp, op, lse, B, S, H, Hkv, hp, s, err, 1.f / sqrtf((float)hd));
    if (ok) heads_pad(op, out, N, H, hd, hp, false, s);
  }
  if (op) cudaFreeAsync(op, s);
  if (qp) cudaFreeAsync(qp, s);
  return ok;
}

bool attn_bwd_padded(const void* qkv, const void* out, const void* dout, const float* lse, float* D, void* dqkv, int B,
                     int S, int H, int Hkv, int hd, cudaStream_t s, cudaMemPool_t pool, unsigned* err) {
  const int hp = padded_hd(hd), N = B * S, nh = H + 2 * Hkv;
  if (!hp) return false;
  const size_t wq = (size_t)N * nh * hp * 2, wo = (size_t)N * H * hp * 2;
  void* buf = scratch(2 * wq + 2 * wo, s, pool);
  if (!buf) return false;
  char* qp = (char*)buf;
  char* dqp = qp + wq;
  char* op = dqp + wq;
  char* dop = op + wo;
  heads_pad(qkv, qp, N, nh, hd, hp, true, s);
  heads_pad(out, op, N, H, hd, hp, true, s);
  heads_pad(dout, dop, N, H, hd, hp, true, s);
  const bool ok = attn_bwd_tcgen05(qp, op, dop, lse, D, dqp, B, S, H, Hkv, hp, s, pool, err, 1.f / sqrtf((float)hd));
  if (ok) heads_pad(dqp, dqkv, N, nh, hd, hp, false, s);
  cudaFreeAsync(buf, s);
  return ok;
}
}  // namespace

// A rotation pass of its own is a launch forward and one backward per layer, all latency on small shapes (eight steps
// of the tiny fp32 model: 3920 us with the passes, 3810 without). Heads of 64 and 128 keep the pass: the table beside
// two rows' registers spills in the backward, 330 bytes.
bool attn_rotates(int dt, int hd) { return dt != BF16 && hd == 32; }

void attn_fwd(int dt, const void* qkv, void* out, float* lse, int B, int S, int H, int Hkv, int hd, cudaStream_t s,
              unsigned* err, cudaMemPool_t pool, const float* cs) {
  const float scale = 1.f / sqrtf((float)hd);
  if (cs) {
    note_launch(1);
    cuda_core_fwd<float, 32, true>(qkv, out, lse, B, S, H, Hkv, hd, scale, s, cs);
    return;
  }
  if (dt == BF16 && attn_fwd_tcgen05(qkv, out, lse, B, S, H, Hkv, hd, s, err, scale)) return;
  if (dt == BF16 && attn_fwd_padded(qkv, out, lse, B, S, H, Hkv, hd, s, err, pool)) return;
  note_launch(1);   // of the two kernels left
  if (dt == BF16 && attn_fwd_tc(qkv, out, lse, B, S, H, Hkv, hd, s)) return;
#define CC(T)                                                                                  \
  if (hd <= 32) cuda_core_fwd<T, 32>(qkv, out, lse, B, S, H, Hkv, hd, scale, s);               \
  else if (hd <= 64) cuda_core_fwd<T, 64>(qkv, out, lse, B, S, H, Hkv, hd, scale, s);          \
  else cuda_core_fwd<T, 128>(qkv, out, lse, B, S, H, Hkv, hd, scale, s);
  if (dt == BF16) { CC(bf16) } else { CC(float) }
#undef CC
}

void attn_bwd(int dt, const void* qkv, const void* out, const void* dout, const float* lse, float* Dbuf, void* dqkv,
              int B, int S, int H, int Hkv, int hd, cudaStream_t s, cudaMemPool_t pool, unsigned* err, const float* cs) {
  const float scale = 1.f / sqrtf((float)hd);
  if (cs) {
    note_launch(1);
    cuda_core_bwd<float, 32, true>(qkv, out, dout, lse, dqkv, B, S, H, Hkv, hd, scale, s, cs);
    return;
  }
  if (dt == BF16 && attn_bwd_tcgen05(qkv, out, dout, lse, Dbuf, dqkv, B, S, H, Hkv, hd, s, pool, err, scale)) return;
  if (dt == BF16 && attn_bwd_padded(qkv, out, dout, lse, Dbuf, dqkv, B, S, H, Hkv, hd, s, pool, err)) return;
  if (dt == BF16 && attn_bwd_tc(qkv, out, dout, lse, Dbuf, dqkv, B, S, H, Hkv, hd, s, pool)) return;
  note_launch(1);
#define CC(T)                                                                                        \
  if (hd <= 32) cuda_core_bwd<T, 32>(qkv, out, dout, lse, dqkv, B, S, H, Hkv, hd, scale, s);         \
  else if (hd <= 64) cuda_core_bwd<T, 64>(qkv, out, dout, lse, dqkv, B, S, H, Hkv, hd, scale, s);    \
  else cuda_core_bwd<T, 128>(qkv, out, dout, lse, dqkv, B, S, H, Hkv, hd, scale, s);
  if (dt == BF16) { CC(bf16) } else { CC(float) }
#undef CC
}

}  // namespace zl
