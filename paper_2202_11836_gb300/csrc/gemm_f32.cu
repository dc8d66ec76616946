// fp32 SIMT GEMM: exact fp32 FMA accumulation for the tight-tolerance fp32
// slice (tensor-core TF32 would not reach a 1e-4 relative error).  Same
// three contraction forms and epilogues as the bf16 tensor-core kernel.
//
// Bound by the FMA pipe (128 a clock and SM) where there is work enough, else by
// the latency of a slab.  A CTA of four warps computes a 64 x 64 tile, 8 x 4 a
// thread, from 32-deep slabs of A and B in shared memory (double-buffered, the
// next slab's loads in flight in registers), two adjacent columns to a packed
// FMA.  8 x 8 a thread, or 16-deep slabs, were slower: fewer warps, and less in
// flight.  The layer's products have few such tiles (404 x 768: 84 for 152 SMs,
// each SM wanting four CTAs or more), so the K range is split over a cluster of
// up to eight CTAs.  Each owns a share of the tile's rows; the others send it
// theirs through distributed shared memory, and it adds them in split order
// (reading them from the peers, behind a second barrier, cost 0.7 us a launch:
// 2-layer slice of width 128 219 -> 186 us).  Against the kernel before (64 x 64, 4 x 4 a
// thread, scalar loads, no split), alone: 404 x 768 x 3072 196 -> 52 us (37
// TFLOP/s), 1000 x 2304 x 768 -> 77 us (46 TFLOP/s);
// the error against float64 falls with the shorter sums (9.9e-7 -> 3.5e-7).
#include "common.cuh"
#include "gemm.h"
#include "ptx.cuh"

namespace sky {
namespace gemm {

namespace {
constexpr int TM = 64, TN = 64, TK = 32;
constexpr int RM = 8, RN = 4;                        // a thread's rows and columns
constexpr int F_THREADS = TM * TN / (RM * RN);
constexpr int LD4 = TK * 64 / 4 / F_THREADS;         // 16-byte groups a thread loads per slab

struct F32Params {
  int M, N, K, n_tiles, ks, k_slabs;
  const float *A, *B;
  int64_t lda, ldb;
  float* C;
  int epi;
  const float *bias, *aux;
  float* aux_out;
};

// Slab layout: element (k, i) of a TK x 64 slab at k * 64 + (i ^ swz(k)), which
// keeps 4-float groups together and spreads both kinds of store over the banks.
__device__ __forceinline__ constexpr int swz(int k) { return ((k >> 2) & 7) << 2; }

// One operand's slab: 64 rows (M or N index) from i0, k from k0.  KMAJ: element
// (i, k) at i * ld + k, else at k * ld + i.  VEC: 16-byte loads (ld % 4 == 0 and
// an aligned base, so a group of four is inside or outside as a whole).
template <bool KMAJ, bool VEC>
__device__ __forceinline__ void load_slab(const float* __restrict__ X, int64_t ld, int i0, int I, int k0,
                                          int K, float (&r)[4 * LD4]) {
  const int t = threadIdx.x;
#pragma unroll
  for (int j = 0; j < LD4; ++j) {
    const int i = i0 + (KMAJ ? t / (TK / 4) + F_THREADS / (TK / 4) * j : (t & 15) * 4);
    const int k = k0 + (KMAJ ? t % (TK / 4) * 4 : (t >> 4) + F_THREADS / 16 * j);
    const float* p = X + (KMAJ ? static_cast<int64_t>(i) * ld + k : static_cast<int64_t>(k) * ld + i);
    if constexpr (VEC) {
      const float4 v = i < I && k < K ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(0.f, 0.f, 0.f, 0.f);
      r[4 * j] = v.x; r[4 * j + 1] = v.y; r[4 * j + 2] = v.z; r[4 * j + 3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        r[4 * j + e] = (KMAJ ? i < I && k + e < K : i + e < I && k < K) ? __ldg(p + e) : 0.f;
    }
  }
}
template <bool KMAJ>
__device__ __forceinline__ void store_slab(float* s, const float (&r)[4 * LD4]) {
  const int t = threadIdx.x;
#pragma unroll
  for (int j = 0; j < LD4; ++j) {
    if constexpr (KMAJ) {
      const int i = t / (TK / 4) + F_THREADS / (TK / 4) * j, k = t % (TK / 4) * 4;
#pragma unroll
      for (int e = 0; e < 4; ++e) s[(k + e) * 64 + (i ^ swz(k))] = r[4 * j + e];
    } else {
      const int i = (t & 15) * 4, k = (t >> 4) + F_THREADS / 16 * j;
      *reinterpret_cast<float4*>(s + k * 64 + (i ^ swz(k))) =
          make_float4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
    }
  }
}

template <bool AK, bool BK, bool VEC>
__global__ void __launch_bounds__(F_THREADS) gemm_f32_kernel(const F32Params p) {
  __shared__ __align__(16) float sm[2][2][TK * 64];  // [buffer][A, B]; later, unsplit, the 64 x 64 tile
  __shared__ __align__(16) float recv[TM * TN];      // split: this CTA's rows from every split
  if (p.ks > 1) ptx::cluster_arrive();  // this CTA runs: its peers may write recv
  pdl_wait();
  const int t = threadIdx.x;
  const int split = static_cast<int>(blockIdx.x) % p.ks, tile = static_cast<int>(blockIdx.x) / p.ks;
  const int m0 = (tile / p.n_tiles) * TM, n0 = (tile % p.n_tiles) * TN;
  const int s0 = split * p.k_slabs / p.ks, s1 = (split + 1) * p.k_slabs / p.ks;
  // thread (rg, cg): rows {rg * 4 .., 32 + rg * 4 ..}, columns cg * 4 ..
  constexpr int CG = TN / RN;
  const int rg = t / CG, cg = t % CG;
  uint64_t acc[RM][RN / 2] = {};  // pairs of adjacent columns
  float ra[4 * LD4], rb[4 * LD4];
  load_slab<AK, VEC>(p.A, p.lda, m0, p.M, s0 * TK, p.K, ra);
  load_slab<BK, VEC>(p.B, p.ldb, n0, p.N, s0 * TK, p.K, rb);
  for (int s = s0; s < s1; ++s) {
    float* sa = sm[(s - s0) & 1][0];
    float* sb = sm[(s - s0) & 1][1];
    store_slab<AK>(sa, ra);
    store_slab<BK>(sb, rb);
    __syncthreads();
    if (s + 1 < s1) {
      load_slab<AK, VEC>(p.A, p.lda, m0, p.M, (s + 1) * TK, p.K, ra);
      load_slab<BK, VEC>(p.B, p.ldb, n0, p.N, (s + 1) * TK, p.K, rb);
    }
#pragma unroll
    for (int k = 0; k < TK; ++k) {
      float a[RM];
      uint64_t b[RN / 2];
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(sa + k * 64 + ((rg * 4) ^ swz(k)));
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(sa + k * 64 + ((32 + rg * 4) ^ swz(k)));
      *reinterpret_cast<ulonglong2*>(b) = *reinterpret_cast<const ulonglong2*>(sb + k * 64 + ((cg * 4) ^ swz(k)));
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        const uint64_t aa = pack2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < RN / 2; ++j) acc[i][j] = fma2(aa, b[j], acc[i][j]);
      }
    }
  }
  pdl_trigger();
  auto finish = [&](int m, int n, float v) {
    if (m >= p.M || n >= p.N) return;
    const int64_t off = static_cast<int64_t>(m) * p.N + n;
    if (p.bias) v += p.bias[n];
    if (p.epi == SKY_EPI_GELU_BWD) v *= p.aux[off];
    if (p.epi == SKY_EPI_BIAS_GELU) {
      p.aux_out[off] = gelu_grad_f(v);
      v = gelu_f(v);
    }
    p.C[off] = v;
  };
  if (p.ks == 1) {
    // through shared memory (row r at r * 64), so that a warp stores 32 consecutive
    // columns of a row
    float* st = &sm[0][0][0];
    const int c = t & 63;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RM; ++i) {
      const int r = (i < 4 ? 0 : 32) + rg * 4 + (i & 3);
      *reinterpret_cast<ulonglong2*>(st + r * 64 + cg * 4) = make_ulonglong2(acc[i][0], acc[i][1]);
    }
    __syncthreads();
#pragma unroll 4
    for (int r = t / 64; r < TM; r += F_THREADS / 64) finish(m0 + r, n0 + c, st[r * 64 + c]);
    return;
  }
  // Each CTA owns 64 / ks rows of the tile: every split sends it its partial rows,
  // half a warp a row, and it adds them in split order.
  const int own = TM / p.ks;
  ptx::cluster_wait();  // every peer runs
  const uint32_t base = ptx::smem_u32(recv);
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int r = (i < 4 ? 0 : 32) + rg * 4 + (i & 3);
    const float2 lo = unpack2(acc[i][0]), hi = unpack2(acc[i][1]);
    ptx::st_cluster_v4(ptx::mapa_shared(base, r / own) + ((split * own + r % own) * 64 + cg * 4) * 4,
                       __float_as_uint(lo.x), __float_as_uint(lo.y), __float_as_uint(hi.x), __float_as_uint(hi.y));
  }
  ptx::cluster_sync();
  for (int g = t; g < own * 16; g += F_THREADS) {
    const int r = g >> 4, c = (g & 15) * 4;
    float4 part[8];
#pragma unroll
    for (int s = 0; s < 8; ++s)
      part[s] = s < p.ks ? *reinterpret_cast<const float4*>(recv + (s * own + r) * 64 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v = part[0];
#pragma unroll
    for (int s = 1; s < 8; ++s)
      if (s < p.ks) { v.x += part[s].x; v.y += part[s].y; v.z += part[s].z; v.w += part[s].w; }
    const int m = m0 + split * own + r;
    finish(m, n0 + c, v.x);
    finish(m, n0 + c + 1, v.y);
    finish(m, n0 + c + 2, v.z);
    finish(m, n0 + c + 3, v.w);
  }
}
}  // namespace

sky_status launch_f32(sky_gemm_form form, int M, int N, int K, const float* A, const float* B,
                      float* C, int epi, const float* bias, const float* aux, float* aux_out,
                      cudaStream_t stream) {
  SKY_CHECK(epi != SKY_EPI_BIAS_GELU || (bias && aux_out), SKY_ERR_INVALID_ARG,
            "BIAS_GELU epilogue needs bias and aux_out");
  SKY_CHECK(epi == SKY_EPI_STORE || epi == SKY_EPI_BIAS_GELU || epi == SKY_EPI_GELU_BWD,
            SKY_ERR_INVALID_ARG, "unknown epilogue %d", epi);
  SKY_CHECK(epi != SKY_EPI_GELU_BWD || aux, SKY_ERR_INVALID_ARG, "GELU' epilogue needs aux");
  const bool ak = form != SKY_GEMM_XTW, bk = form == SKY_GEMM_XWT;  // K-major operands
  F32Params p{};
  p.M = M; p.N = N; p.K = K;
  p.A = A; p.B = B; p.C = C;
  p.lda = ak ? K : M;
  p.ldb = bk ? K : N;
  p.epi = epi;
  p.bias = bias; p.aux = aux; p.aux_out = aux_out;
  p.n_tiles = ceil_div(N, TN);
  p.k_slabs = ceil_div(K, TK);
  const int64_t tiles = static_cast<int64_t>(ceil_div(M, TM)) * p.n_tiles;
  const int sms = sm_count() > 0 ? sm_count() : 148;
  // Splits: a lone CTA waits for its loads, so an SM wants several.  Eight splits up
  // to eleven CTAs an SM, else four, each of two slabs or more.  Where the tiles are
  // few, one slab is enough, and eight only if every CTA has an SM to itself or that
  // halves the longest one's slabs.
  // Never two, whose pairs land on one SM.  us at 1 / 2 / 4 / 8 splits: 404 x 768 x
  // 3072 99 / - / 61 / 51, 404 x 2304 x 768 42 / - / 38 / 40, 1000 x 768 x 3072 171 / - /
  // 115 / 106, 1000 x 2304 x 768 77 / 82 / 83 / 85, 512 x 2048 x 97 9.9 / 16.1 / 13.1 / -,
  // 128 x 384 x 128 5.8 / 7.7 / 3.7 / -; 256 x 384 x 384 (12 slabs) 5.8 at four, 7.0 at
  // eight, 384 x 384 x 256 (8) 6.5 and 6.0, 150 x 448 x 448 (14) 6.8 and 6.5.
  p.ks = 1;
  const bool few = 4 * tiles <= sms;
  const bool halves = 2 * ceil_div(p.k_slabs, 8) <= ceil_div(p.k_slabs, 4);
  for (int ks = 8; ks >= 4 && p.ks == 1; ks /= 2) {
    const bool one_slab = few && p.k_slabs >= ks && (ks == 4 || 8 * tiles <= sms || halves);
    if (tiles * ks <= 11 * sms && (p.k_slabs >= 2 * ks || one_slab)) p.ks = ks;
  }
  const bool vec = p.lda % 4 == 0 && p.ldb % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  SKY_CHECK(tiles * p.ks <= 0x7fffffff, SKY_ERR_INVALID_ARG, "GEMM too large (M=%d N=%d)", M, N);
  const dim3 grid(static_cast<unsigned>(tiles * p.ks)), blk(F_THREADS);
  auto go = [&](auto kern) { return launch_pdl(kern, grid, blk, 0, stream, p.ks, p); };
  cudaError_t e;
  if (form == SKY_GEMM_XWT) e = vec ? go(gemm_f32_kernel<true, true, true>) : go(gemm_f32_kernel<true, true, false>);
  else if (form == SKY_GEMM_XW) e = vec ? go(gemm_f32_kernel<true, false, true>) : go(gemm_f32_kernel<true, false, false>);
  else e = vec ? go(gemm_f32_kernel<false, false, true>) : go(gemm_f32_kernel<false, false, false>);
  count_launches(1);
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "gemm_f32_kernel launch");
}

}  // namespace gemm
}  // namespace sky
