// Masked scaled dot-product attention, Eq. 1: per sequence b and head a,
//   P = softmax_j(Q K^T / sqrt(D)) over the valid keys j < len[b],
//   ctx = P V,
// and its backward (dQ, dK, dV).  All S query rows are computed; padded keys
// get probability exactly 0.
//
// bf16 (D = 64): the tensor-core kernels of attention_tc.cu, plus the
// vectorised delta = rowsum(dO * O) pre-pass here (sequences over 128; shorter
// ones form it in their one backward launch).
// fp32: blocks of query (or key) rows against tiles of the other side, exact
// fp32 arithmetic.
#include <cfloat>
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"

namespace sky {
namespace attn {

constexpr int HD = 64;

using bf16 = __nv_bfloat16;

// delta[b,a,s] = sum_d dctx[b,s,a,d] * ctx[b,s,a,d]  (equals sum_j P_sj dP_sj)
// One warp per token row; each lane takes 8 consecutive elements (16 bytes
// of bf16) per 256-column group, and the 8 lanes covering one 64-wide head
// reduce with shuffles.  NV > 0: the row has exactly NV groups, and every
// load of the row is issued before the first product (more bytes in flight
// per warp); NV == 0: any H that is a multiple of 64, one group at a time.
// Requires D == 64.
// Beside delta it writes the per-query terms the tensor-core dK/dV kernel
// adds inside its score products: xtab[(b*A + a)*2 + 0][s] = lse2 / c and
// xtab[(b*A + a)*2 + 1][s] = delta (c = log2(e)/sqrt(D)), each negated and
// split into a bf16 high and low part, as 16-byte rows [hi, lo, 0 x 6].
template <int NV>
__global__ void attn_delta_bf16(const bf16* __restrict__ ctx, const bf16* __restrict__ dctx, int S,
                                int H, int A, int64_t rows, float* __restrict__ delta,
                                const float* __restrict__ lse, uint4* __restrict__ xtab) {
  pdl_wait();
  pdl_trigger();
  const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int l = threadIdx.x & 31;
  if (row >= rows) return;
  const int64_t b = row / S, s = row % S;
  auto dot8 = [](const uint4& x, const uint4& y) {
    const __nv_bfloat162* xs = reinterpret_cast<const __nv_bfloat162*>(&x);
    const __nv_bfloat162* ys = reinterpret_cast<const __nv_bfloat162*>(&y);
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 p = __bfloat1622float2(xs[i]), q = __bfloat1622float2(ys[i]);
      acc += p.x * q.x + p.y * q.y;
    }
    return acc;
  };
  // lz: the row's lse of this lane's head, loaded beside ctx / dctx (NV > 0)
  auto finish = [&](float acc, int col, float lz) {
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    if ((l & 7) == 0 && col < H) {
      const int64_t bh = b * A + col / HD;
      delta[bh * S + s] = acc;
      auto row16 = [](float x) {  // -x as [hi, lo, 0, ...] in bf16
        const bf16 hi = __float2bfloat16_rn(-x);
        const bf16 lo = __float2bfloat16_rn(-x - __bfloat162float(hi));
        return make_uint4(static_cast<uint32_t>(__bfloat16_as_ushort(hi)) |
                              (static_cast<uint32_t>(__bfloat16_as_ushort(lo)) << 16),
                          0u, 0u, 0u);
      };
      constexpr float kC = 1.4426950408889634f * 0.125f;  // log2(e) / sqrt(64)
      xtab[(bh * 2) * S + s] = row16(__fdiv_rn(lz, kC));
      xtab[(bh * 2 + 1) * S + s] = row16(acc);
    }
  };
  if constexpr (NV > 0) {
    uint4 x[NV], y[NV];
    float lz[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      x[v] = *reinterpret_cast<const uint4*>(ctx + row * H + v * 256 + l * 8);
      y[v] = *reinterpret_cast<const uint4*>(dctx + row * H + v * 256 + l * 8);
      lz[v] = (l & 7) == 0 ? lse[(b * A + (v * 256 + l * 8) / HD) * S + s] : 0.f;
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) finish(dot8(x[v], y[v]), v * 256 + l * 8, lz[v]);
  } else {
    for (int c0 = 0; c0 < H; c0 += 256) {
      const int col = c0 + l * 8;
      float acc = 0.f, lz = 0.f;
      if (col < H) {
        acc = dot8(*reinterpret_cast<const uint4*>(ctx + row * H + col),
                   *reinterpret_cast<const uint4*>(dctx + row * H + col));
        if ((l & 7) == 0) lz = lse[(b * A + col / HD) * S + s];
      }
      finish(acc, col, lz);
    }
  }
}

// Generic form (fp32 path): one warp per (row, head).
template <typename T>
__global__ void attn_delta(const T* __restrict__ ctx, const T* __restrict__ dctx, int S, int H,
                           int A, int D, int64_t rows, float* __restrict__ delta) {
  pdl_wait();
  pdl_trigger();
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int l = threadIdx.x & 31;
  if (w >= rows * A) return;
  const int64_t row = w / A;
  const int a = (int)(w % A);
  const T* c = ctx + row * H + a * D;
  const T* dc = dctx + row * H + a * D;
  float acc = 0.f;
  for (int d = l; d < D; d += 32) acc += to_f32(c[d]) * to_f32(dc[d]);
  acc = warp_sum(acc);
  if (l == 0) {
    const int64_t b = row / S, s = row % S;
    delta[(b * A + a) * S + s] = acc;
  }
}

// ----------------------------------------------------------------- fp32 path
// Exact fp32 arithmetic, head dim up to 128.  A CTA of four warps owns 16 rows
// of one (sequence, head) and walks the other side in tiles of 64 rows staged in
// shared memory.  Half a warp owns two rows, so row maxima and sums are
// shuffles among 16 lanes and a row's probabilities go to shared memory and
// back within the half warp.  Score products: 2 rows x 4 columns a thread (six
// 16-byte shared loads for 32 FMAs); accumulating products: 2 rows x 4 dims.
// Short sequences and few heads make these latency-bound; a warp per row with
// scalar loads took 116 us forward and 182 us backward at 4 x 101 tokens, 12
// heads of 64.
constexpr int FR = 16, FC = 64, F_THR = 128;  // rows of a CTA, columns of a tile
constexpr int FP_LD = FC + 4;                 // row stride of the probability tiles
// (the backward of sequences up to 16 tokens: tiles of 16 columns, NC = 1 of 4)

// Rows are staged F_THR / G a pass, G threads a row (D <= 4 G), through registers, so
// that a tile's loads are all in flight before the first is stored.  Loading and
// storing in turn waited for each: 4 x 32 tokens, 2 heads of 64, forward 6.4 us,
// now 3.8, backward 10.7 and 7.3; 4 x 101, 12 heads 17.0 and 12.2, 39.9 and 29.4; 4 x
// 256, 24 heads of 32 52.6 and 48.7 (58.1 with 16 threads a row).
template <int G, int NC = FC / 16>
struct Stage {  // a tile's 16 NC rows: BATCHES of PASSES passes, R rows each
  static constexpr int ROWS = 16 * NC;
  static constexpr int PASSES = ROWS * G / F_THR < 8 ? ROWS * G / F_THR : 8;
  static constexpr int R = PASSES * F_THR / G, BATCHES = ROWS / R;
  static constexpr int OWN = FR * G / F_THR;  // passes of the CTA's FR rows
  static constexpr int CC = G > 16 ? G / 16 : 1;  // 64-value column groups of an output row
};
// Rows from `rows` on are zeros.  vec: D, ld and X allow 16-byte loads.
template <int G, int N>
__device__ __forceinline__ void load_rows(const float* __restrict__ X, int64_t ld, int r0, int rows, int D, bool vec,
                                          float4 (&v)[N]) {
  const int c = (threadIdx.x % G) * 4;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int r = r0 + F_THR / G * i + threadIdx.x / G;
    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < rows && c < D) {
      const float* p = X + static_cast<int64_t>(r) * ld + c;
      if (vec) {
        v[i] = *reinterpret_cast<const float4*>(p);
      } else {
        v[i].x = p[0];
        if (c + 1 < D) v[i].y = p[1];
        if (c + 2 < D) v[i].z = p[2];
        if (c + 3 < D) v[i].w = p[3];
      }
    }
  }
}
template <int G, int N>
__device__ __forceinline__ void put_rows(float* s, int LD, int D, const float4 (&v)[N]) {
  const int c = (threadIdx.x % G) * 4;
  if (c >= D) return;
#pragma unroll
  for (int i = 0; i < N; ++i)
    *reinterpret_cast<float4*>(s + (F_THR / G * i + threadIdx.x / G) * LD + c) = v[i];
}
// acc[i][c] = row (2 ty + i) . column row (tx + 16 c), over D (a multiple of 4 in shared memory)
template <int NC>
__device__ __forceinline__ void scores(const float* rows, const float* cols, int LD, int D, float (&acc)[2][NC]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[i][c] = 0.f;
  for (int d = 0; d < D; d += 4) {
    float4 r[2], k[NC];
#pragma unroll
    for (int i = 0; i < 2; ++i) r[i] = *reinterpret_cast<const float4*>(rows + (2 * ty + i) * LD + d);
#pragma unroll
    for (int c = 0; c < NC; ++c) k[c] = *reinterpret_cast<const float4*>(cols + (tx + 16 * c) * LD + d);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < NC; ++c)
        acc[i][c] = fmaf(r[i].w, k[c].w, fmaf(r[i].z, k[c].z, fmaf(r[i].y, k[c].y, fmaf(r[i].x, k[c].x, acc[i][c]))));
  }
}
// o[i][cc] += sum_j w[2 ty + i][j] cols[j][4 tx + 64 cc ..] over the tile's first n columns (n <= 64)
template <int CC, int W_LD = FP_LD>
__device__ __forceinline__ void accumulate(const float* w, const float* cols, int LD, int D, int n, float4 (&o)[2][CC]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int j = 0; j < n; j += 4) {
    float4 p[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) p[i] = *reinterpret_cast<const float4*>(w + (2 * ty + i) * W_LD + j);
#pragma unroll
    for (int cc = 0; cc < CC; ++cc) {
      const int d = 4 * tx + 64 * cc;
      if (d >= D) continue;
      float4 v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = *reinterpret_cast<const float4*>(cols + (j + e) * LD + d);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float pe[4] = {p[i].x, p[i].y, p[i].z, p[i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          o[i][cc].x = fmaf(pe[e], v[e].x, o[i][cc].x);
          o[i][cc].y = fmaf(pe[e], v[e].y, o[i][cc].y);
          o[i][cc].z = fmaf(pe[e], v[e].z, o[i][cc].z);
          o[i][cc].w = fmaf(pe[e], v[e].w, o[i][cc].w);
        }
      }
    }
  }
}
template <int CC>
__device__ __forceinline__ void store_rows(float* X, int64_t ld, int r0, int rows, int D, bool vec, float scale0,
                                           float scale1, const float4 (&o)[2][CC]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = r0 + 2 * ty + i;
    if (r >= rows) continue;
    const float sc = i ? scale1 : scale0;
#pragma unroll
    for (int cc = 0; cc < CC; ++cc) {
      const int d = 4 * tx + 64 * cc;
      if (d >= D) continue;
      const float4 v = make_float4(o[i][cc].x * sc, o[i][cc].y * sc, o[i][cc].z * sc, o[i][cc].w * sc);
      float* p = X + static_cast<int64_t>(r) * ld + d;
      if (vec) {
        *reinterpret_cast<float4*>(p) = v;
      } else {
        p[0] = v.x;
        if (d + 1 < D) p[1] = v.y;
        if (d + 2 < D) p[2] = v.z;
        if (d + 3 < D) p[3] = v.w;
      }
    }
  }
}
__device__ __forceinline__ float half_warp_max(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float half_warp_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int G>
__global__ void __launch_bounds__(F_THR) attn_fwd_f32(const float* __restrict__ qkv, const int32_t* __restrict__ lens,
                                                      int S, int H, int A, int D, int LD, bool vec,
                                                      float* __restrict__ ctx, float* __restrict__ lse,
                                                      int32_t* status) {
  using ST = Stage<G>;
  constexpr int CC = ST::CC;
  pdl_wait();
  extern __shared__ __align__(16) float sm[];
  float *sq = sm, *sk = sq + FR * LD, *sv = sk + FC * LD, *sp = sv + FC * LD;
  const int tiles = (S + FR - 1) / FR;
  const int a = static_cast<int>(blockIdx.x) / tiles, q0 = (static_cast<int>(blockIdx.x) % tiles) * FR, b = blockIdx.y;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  int len = lens[b];
  if (len < 1 || len > S) {
    if (status && threadIdx.x == 0) atomicOr(status, kStatusBadLength);
    len = len < 1 ? 1 : S;
  }
  const int64_t rs = 3 * static_cast<int64_t>(H);
  const float* q = qkv + static_cast<int64_t>(b) * S * rs + a * D;
  const float sc = 1.f / sqrtf((float)D);
  float4 own[ST::OWN];
  load_rows<G>(q, rs, q0, S, D, vec, own);
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
  float4 o[2][CC] = {};
  for (int k0 = 0; k0 < len; k0 += FC) {
    __syncthreads();
#pragma unroll
    for (int h = 0; h < ST::BATCHES; ++h) {
      constexpr int R = ST::R;
      float4 kx[ST::PASSES], vx[ST::PASSES];
      load_rows<G>(q + H, rs, k0 + R * h, len, D, vec, kx);
      load_rows<G>(q + 2 * H, rs, k0 + R * h, len, D, vec, vx);
      if (h == 0 && k0 == 0) put_rows<G>(sq, LD, D, own);
      put_rows<G>(sk + R * h * LD, LD, D, kx);
      put_rows<G>(sv + R * h * LD, LD, D, vx);
    }
    __syncthreads();
    float s[2][4];
    scores(sq, sk, LD, D, s);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        s[i][c] = k0 + tx + 16 * c < len ? s[i][c] * sc : -INFINITY;
        mx = fmaxf(mx, s[i][c]);
      }
      // (finite also while every score so far is -inf: those keys then add nothing)
      const float mn = fmaxf(fmaxf(m[i], half_warp_max(mx)), -FLT_MAX);
      const float al = expf(m[i] - mn);  // 0 in the first tile
      m[i] = mn;
      float sum = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float e = expf(s[i][c] - mn);  // masked: 0
        sp[(2 * ty + i) * FP_LD + tx + 16 * c] = e;
        sum += e;
      }
      l[i] = l[i] * al + half_warp_sum(sum);
#pragma unroll
      for (int cc = 0; cc < CC; ++cc) {
        o[i][cc].x *= al; o[i][cc].y *= al; o[i][cc].z *= al; o[i][cc].w *= al;
      }
    }
    __syncwarp();
    accumulate<CC>(sp, sv, LD, D, min(FC, len - k0), o);
    __syncwarp();
  }
  pdl_trigger();
  store_rows<CC>(ctx + static_cast<int64_t>(b) * S * H + a * D, H, q0, S, D, vec, 1.f / l[0], 1.f / l[1], o);
  if (tx == 0)
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (q0 + 2 * ty + i < S)
        lse[(static_cast<int64_t>(b) * A + a) * S + q0 + 2 * ty + i] = (m[i] + logf(l[i])) * 1.4426950408889634f;  // base 2
}

// dQ (even blockIdx.x): own rows are queries (Q, dO), columns keys (K, V).
// dK, dV (odd): own rows are keys (K, V), columns queries (Q, dO).  Either way
//   P = exp2(s log2(e)/sqrt(D) - lse_q),  dS = P (dp - delta_q),
// s and dp the products of the first and second operands; dQ or dK = dS . first
// operand of the columns / sqrt(D), dV = P . dO.  Four CTAs an SM (128 registers) are
// faster up to a head dim of 64 (29.8 us against 34.7 at 4 x 101, 12 heads), above it
// the registers are (50.6 against 57.0 at 2 x 200, 6 heads of 128).
template <int G, int NC>
__global__ void __launch_bounds__(F_THR, G > 16 ? 1 : 4) attn_bwd_f32(const float* __restrict__ qkv, const float* __restrict__ dctx,
                                                      const float* __restrict__ lse, const float* __restrict__ delta,
                                                      const int32_t* __restrict__ lens, int S, int H, int A, int D,
                                                      int LD, bool vec, float* __restrict__ dqkv) {
  using ST = Stage<G, NC>;
  constexpr int CC = ST::CC, TC = ST::ROWS, P_LD = TC + 4;
  pdl_wait();
  extern __shared__ __align__(16) float sm[];
  float *r0s = sm, *r1s = r0s + FR * LD, *c0s = r1s + FR * LD, *c1s = c0s + TC * LD;
  float *sds = c1s + TC * LD, *sp = sds + FR * P_LD, *sl = sp + FR * P_LD, *sd = sl + TC;
  const int tiles = (S + FR - 1) / FR;
  const bool keys = blockIdx.x & 1;  // own rows are keys
  const int u = static_cast<int>(blockIdx.x) >> 1;
  const int a = u / tiles, r0 = (u % tiles) * FR, b = blockIdx.y;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  int len = lens[b];
  len = len < 1 ? 1 : (len > S ? S : len);
  const int64_t rs = 3 * static_cast<int64_t>(H);
  const float* q = qkv + static_cast<int64_t>(b) * S * rs + a * D;
  const float* dO = dctx + static_cast<int64_t>(b) * S * H + a * D;
  float* out = dqkv + static_cast<int64_t>(b) * S * rs + a * D;
  const float *lse_b = lse + (static_cast<int64_t>(b) * A + a) * S, *del_b = delta + (static_cast<int64_t>(b) * A + a) * S;
  const float sc = 1.f / sqrtf((float)D), sl2 = sc * 1.4426950408889634f;
  float4 o0[2][CC] = {}, o1[2][CC] = {};
  const int cols = keys ? S : len;
  if (!keys || r0 < len) {
    float4 own0[ST::OWN], own1[ST::OWN];
    load_rows<G>(keys ? q + H : q, rs, r0, S, D, vec, own0);
    load_rows<G>(keys ? q + 2 * H : dO, keys ? rs : static_cast<int64_t>(H), r0, S, D, vec, own1);
    float lr[2], dr[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = min(r0 + 2 * ty + i, S - 1);
      lr[i] = lse_b[r];
      dr[i] = del_b[r];
    }
    for (int c0 = 0; c0 < cols; c0 += TC) {
      __syncthreads();
      // columns: queries (Q, dO; all S) or keys (K, V; the valid ones)
      const float *x0 = keys ? q : q + H, *x1 = keys ? dO : q + 2 * H;
      float lc = 0.f, dc = 0.f;
      if (keys && threadIdx.x < TC) {
        const int c = min(c0 + static_cast<int>(threadIdx.x), S - 1);
        lc = lse_b[c];
        dc = del_b[c];
      }
#pragma unroll
      for (int h = 0; h < ST::BATCHES; ++h) {
        constexpr int R = ST::R;
        float4 v0[ST::PASSES], v1[ST::PASSES];
        load_rows<G>(x0, rs, c0 + R * h, cols, D, vec, v0);
        load_rows<G>(x1, keys ? static_cast<int64_t>(H) : rs, c0 + R * h, cols, D, vec, v1);
        if (h == 0 && c0 == 0) {
          put_rows<G>(r0s, LD, D, own0);
          put_rows<G>(r1s, LD, D, own1);
        }
        put_rows<G>(c0s + R * h * LD, LD, D, v0);
        put_rows<G>(c1s + R * h * LD, LD, D, v1);
      }
      if (keys && threadIdx.x < TC) {
        sl[threadIdx.x] = lc;
        sd[threadIdx.x] = dc;
      }
      __syncthreads();
      float s[2][NC], dp[2][NC];
      scores(r0s, c0s, LD, D, s);
      scores(r1s, c1s, LD, D, dp);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int cl = tx + 16 * c;
          const bool live = c0 + cl < cols && (!keys || r0 + 2 * ty + i < len);
          const float p = live ? exp2f(fmaf(s[i][c], sl2, -(keys ? sl[cl] : lr[i]))) : 0.f;
          sds[(2 * ty + i) * P_LD + cl] = live ? p * (dp[i][c] - (keys ? sd[cl] : dr[i])) : 0.f;
          if (keys) sp[(2 * ty + i) * P_LD + cl] = p;
        }
      __syncwarp();
      const int n = min(TC, cols - c0);
      accumulate<CC, P_LD>(sds, c0s, LD, D, n, o0);
      if (keys) accumulate<CC, P_LD>(sp, c1s, LD, D, n, o1);
      __syncwarp();
    }
  }
  pdl_trigger();
  store_rows<CC>(keys ? out + H : out, rs, r0, S, D, vec, sc, sc, o0);
  if (keys) store_rows<CC>(out + 2 * H, rs, r0, S, D, vec, 1.f, 1.f, o1);
}

// Launch shape of the fp32 kernels: the shared row stride (four floats past the
// head dim, so the 16 lanes of a score product read different banks) and the
// bytes it makes, 16-row units of all heads, and whether the head rows allow
// 16-byte accesses.
constexpr int row_stride(int D) { return (D + 3) / 4 * 4 + 4; }
constexpr int fwd_smem(int D) { return ((FR + 2 * FC) * row_stride(D) + FR * FP_LD) * 4; }
constexpr int bwd_smem(int D, int NC) {
  return ((2 * FR + 32 * NC) * row_stride(D) + 2 * FR * (16 * NC + 4) + 32 * NC) * 4;
}
template <int G>
using Group = std::integral_constant<int, G>;
struct F32Shape {
  unsigned units;
  int LD;
  bool vec;
  F32Shape(int S, int H, int A, int D, const void* x, const void* y, const void* z)
      : units((unsigned)ceil_div(S, FR) * A), LD(row_stride(D)) {
    const auto a16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    vec = D % 4 == 0 && H % 4 == 0 && a16(x) && a16(y) && a16(z);
  }
};

}  // namespace attn

// ------------------------------------------------------------------- host
sky_status attention_fwd_tc(const void* qkv, const int32_t* lens, int B, int S, int H, int A,
                            void* ctx, float* lse, int32_t* status, uint64_t timeout_ns,
                            cudaStream_t stream);

sky_status attention_bwd_short_tc(const void* qkv, const void* ctx, const void* dctx, const float* lse,
                                  const int32_t* lens, int B, int S, int H, int A, void* dqkv, int32_t* status,
                                  uint64_t timeout_ns, cudaStream_t stream, float* colpart);

sky_status attention_bwd_tc(const void* qkv, const void* dctx, const float* lse, const float* delta,
                            const uint4* xtab, const int32_t* lens, int B, int S, int H, int A, void* dqkv,
                            int32_t* status, uint64_t timeout_ns, cudaStream_t stream,
                            float* colpart);

sky_status attention_fwd(const void* qkv, const int32_t* lens, int B, int S, int H, int A,
                         sky_dtype dt, void* ctx, float* lse, int32_t* status,
                         cudaStream_t stream) {
  const int D = H / A;
  if (dt == SKY_DTYPE_BF16) {
    SKY_CHECK(D == attn::HD, SKY_ERR_UNSUPPORTED, "bf16 attention needs head dim 64 (got %d)", D);
    return attention_fwd_tc(qkv, lens, B, S, H, A, ctx, lse, status, 2000000000ull, stream);
  } else {
    SKY_CHECK(D <= 128, SKY_ERR_UNSUPPORTED, "fp32 attention needs head dim <= 128");
    SKY_CHECK(S <= 3072, SKY_ERR_UNSUPPORTED, "fp32 attention: sequence too long");
    const attn::F32Shape f(S, H, A, D, qkv, ctx, nullptr);
    const auto go = [&](auto group, auto kern) {  // `group` threads a row: head dims up to four times that
      static OncePerDevice once;
      const cudaError_t e = allow_smem(once, kern, attn::fwd_smem(4 * decltype(group)::value));
      if (e != cudaSuccess) return e;
      return launch_pdl(kern, dim3(f.units, B), dim3(attn::F_THR), attn::fwd_smem(D), stream, 1,
                        static_cast<const float*>(qkv), lens, S, H, A, D, f.LD, f.vec, static_cast<float*>(ctx), lse,
                        status);
    };
    const cudaError_t le = D <= 32   ? go(attn::Group<8>{}, attn::attn_fwd_f32<8>)
                           : D <= 64 ? go(attn::Group<16>{}, attn::attn_fwd_f32<16>)
                                     : go(attn::Group<32>{}, attn::attn_fwd_f32<32>);
    if (le != cudaSuccess) return cuda_fail(le, "attention forward launch");
  }
  count_launches(1);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "attention forward launch");
}

// delta [B][A][S] floats, then (bf16 path) the dK/dV kernel's per-query rows
// [B][A][2][S] x 16 bytes, 16-byte aligned.
static size_t delta_bytes(int B, int S, int A) { return ((size_t)B * A * S * sizeof(float) + 15) & ~(size_t)15; }
size_t attention_bwd_ws(int B, int S, int A) { return delta_bytes(B, S, A) + (size_t)B * A * 2 * S * 16; }

sky_status attention_bwd(const void* qkv, const void* ctx, const void* dctx, const float* lse,
                         const int32_t* lens, int B, int S, int H, int A, sky_dtype dt, void* dqkv,
                         float* delta, int32_t* status, cudaStream_t stream, float* colpart) {
  const int D = H / A;
  const int64_t rows = (int64_t)B * S;
  const int dblocks = ceil_div(rows * A * 32, 256);
  if (dt == SKY_DTYPE_BF16) {
    SKY_CHECK(D == attn::HD, SKY_ERR_UNSUPPORTED, "bf16 attention needs head dim 64 (got %d)", D);
    // every kernel below moves 16-byte vectors of these buffers (checked
    // before the first launch)
    const auto a16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
    SKY_CHECK(a16(qkv) && a16(ctx) && a16(dctx) && a16(dqkv) && a16(delta), SKY_ERR_INVALID_ARG,
              "bf16 attention backward buffers and workspace must be 16-byte aligned");
    // one tile a sequence: everything in one launch (grid y is the batch, at most
    // 65535 as for the kernels below)
    if (S <= 128 && B <= 65535)
      return attention_bwd_short_tc(qkv, ctx, dctx, lse, lens, B, S, H, A, dqkv, status, 2000000000ull, stream,
                                    colpart);
    const auto* c = static_cast<const __nv_bfloat16*>(ctx);
    const auto* dc = static_cast<const __nv_bfloat16*>(dctx);
    const dim3 g(ceil_div(rows * 32, 256)), blk(256);
    uint4* xtab = reinterpret_cast<uint4*>(reinterpret_cast<char*>(delta) + delta_bytes(B, S, A));
    cudaError_t le;
    switch (H % 256 == 0 ? H / 256 : 0) {
      case 3: le = launch_pdl(attn::attn_delta_bf16<3>, g, blk, 0, stream, 1, c, dc, S, H, A, rows, delta, lse, xtab); break;
      case 4: le = launch_pdl(attn::attn_delta_bf16<4>, g, blk, 0, stream, 1, c, dc, S, H, A, rows, delta, lse, xtab); break;
      case 8: le = launch_pdl(attn::attn_delta_bf16<8>, g, blk, 0, stream, 1, c, dc, S, H, A, rows, delta, lse, xtab); break;
      default: le = launch_pdl(attn::attn_delta_bf16<0>, g, blk, 0, stream, 1, c, dc, S, H, A, rows, delta, lse, xtab); break;
    }
    count_launches(1);
    if (le != cudaSuccess) return cuda_fail(le, "attention delta launch");
    return attention_bwd_tc(qkv, dctx, lse, delta, xtab, lens, B, S, H, A, dqkv, status, 2000000000ull,
                            stream, colpart);
  } else {
    SKY_CHECK(D <= 128, SKY_ERR_UNSUPPORTED, "fp32 attention needs head dim <= 128");
    cudaError_t le = launch_pdl(attn::attn_delta<float>, dim3(dblocks), dim3(256), 0, stream, 1,
                                static_cast<const float*>(ctx), static_cast<const float*>(dctx), S, H, A, D, rows,
                                delta);
    const attn::F32Shape f(S, H, A, D, qkv, dctx, dqkv);
    const auto go = [&](auto group, auto nc, auto kern) {
      constexpr int G = decltype(group)::value, NC = decltype(nc)::value;
      static OncePerDevice once;
      const cudaError_t e = allow_smem(once, kern, attn::bwd_smem(4 * G, NC));
      if (e != cudaSuccess) return e;
      return launch_pdl(kern, dim3(2 * f.units, B), dim3(attn::F_THR), attn::bwd_smem(D, NC), stream, 1,
                        static_cast<const float*>(qkv), static_cast<const float*>(dctx), lse,
                        static_cast<const float*>(delta), lens, S, H, A, D, f.LD, f.vec, static_cast<float*>(dqkv));
    };
    // Up to 16 tokens a 64-column tile is mostly empty: 128 x 8 tokens, 6 heads of 128
    // 52.4 us with it, 27.8 with 16 columns (a warp a row 28.8); 12 of 64 45.2 and 25.5
    // (41.1); 64 x 16, 12 of 64 29.8 and 18.3 (70.4).
    const auto width = [&](auto group) {
      constexpr int G = decltype(group)::value;
      return S <= 16 ? go(group, std::integral_constant<int, 1>{}, attn::attn_bwd_f32<G, 1>)
                     : go(group, std::integral_constant<int, 4>{}, attn::attn_bwd_f32<G, 4>);
    };
    if (le == cudaSuccess)
      le = D <= 32 ? width(attn::Group<8>{}) : D <= 64 ? width(attn::Group<16>{}) : width(attn::Group<32>{});
    if (le != cudaSuccess) return cuda_fail(le, "attention backward launch");
  }
  count_launches(2);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "attention backward launch");
}

}  // namespace sky
