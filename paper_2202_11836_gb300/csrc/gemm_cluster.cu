// bf16 GEMM for products that fill the chip poorly with 256-wide tiles: small
// tiles, and the K range of a tile split over the CTAs of a cluster.
//
// The persistent kernel of gemm_tc.cu computes 256 x 256 tiles on SM pairs.
// A product of a few hundred or thousand rows has too few of those: 1024 x 768
// (a base-width layer's output at T = 1024) is 12 tiles for 76 SM pairs, each
// walking the whole K range alone.  Here a tile is 128 x BN (or 256 x BN on an
// SM pair, cta_group::2), and `ks` CTAs (pairs) of one cluster take a
// contiguous part of its k-blocks each.  When its MMAs are done a CTA puts its
// fp32 accumulator into its own shared memory (over the operand ring, which
// nothing reads any more); after a cluster barrier every CTA adds up its share
// of the tile's rows from all `ks` copies through distributed shared memory, in
// split order (deterministic), and runs the epilogue on the sums.  So a split
// product needs no workspace and no second launch, and every epilogue (bias,
// residual, GELU, GELU') can follow a split.
//
// One work unit per CTA, no persistence: with at most ~112 KiB of shared memory
// and 128 TMEM columns a CTA, two CTAs share an SM, and one's prologue and
// epilogue run under the other's main loop.  The choice between the two kernels
// and of (pair, BN, ks) is made on the host (plan_cluster).
//
//   warp 0      TMA producer, warp 1 MMA issuer (as in gemm_tc.cu)
//   warps 2..9  accumulator -> shared memory, then the reduction and epilogue
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "gemm.h"
#include "ptx.cuh"

namespace sky {
namespace gemm {
namespace {

constexpr int CBM = 128, CBK = 64;
constexpr int C_A_BYTES = CBM * CBK * 2;        // 16 KiB
constexpr int C_CHUNK_BYTES = 64 * CBK * 2;     // one 64-wide MN-major box: 8 KiB
constexpr int C_EPI = 256;                      // epilogue threads (8 warps)
constexpr int C_THREADS = 64 + C_EPI;
constexpr int C_MAX_STAGES = 8;
constexpr uint32_t kClusterHint = 2000;         // suspend hint of the epilogue's accumulator wait

struct ClusterParams {
  int M, N, bn, lg;          // bn = 4 << lg
  int n_tiles, ks, k_blocks, stages;
  int bar_off, red_off;      // shared-memory offsets of the barriers and the column-sum scratch
  int out_f32;
  void* C;
  const __nv_bfloat16* bias;
  const __half* aux;
  __half* aux_out;
  float* colpart;            // [ceil(M/32)][N] column sums of C per 32 rows, or null
  const float* resid;
  const float* ln_mean;
  const float* ln_rstd;
  const __nv_bfloat16* ln_gamma;
  const __nv_bfloat16* ln_beta;
  int32_t* status;
  uint64_t timeout_ns;
  int skip_loads;
};

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_stream_f4(const float* p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ float4 bf4(const __nv_bfloat16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&raw)[0]);
  const float2 b = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&raw)[1]);
  return make_float4(a.x, a.y, b.x, b.y);
}

// Epilogues, one instantiation each: bias only (fp32 or bf16 output), bias +
// GELU, GELU', and bias + fp32 residual or LayerNorm residual (fp32 output).
enum { E_STORE, E_GELU, E_GELU_BWD, E_RESID };

template <bool A_MN, bool B_MN, bool PAIR, int EP>
__global__ void __launch_bounds__(C_THREADS, 2)
    gemm_cluster_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const ClusterParams p) {
  constexpr int TILE_M = PAIR ? 2 * CBM : CBM;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + p.bar_off);
  uint64_t* empty = full + C_MAX_STAGES;
  uint64_t* tfull = empty + C_MAX_STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bn = p.bn;
  const int b_rows = PAIR ? bn >> 1 : bn;  // tile columns whose B operand this CTA loads
  const int sbytes = C_A_BYTES + b_rows * CBK * 2;
  const uint32_t crank = ptx::cluster_ctarank();
  const int half = PAIR ? static_cast<int>(crank & 1) : 0;  // 128-row half of the pair's tile
  const int split = static_cast<int>(PAIR ? crank >> 1 : crank);
  const uint32_t lead_rank = crank - half;
  const int tile = static_cast<int>(blockIdx.x) / (p.ks * (PAIR ? 2 : 1));
  const int m0 = (tile / p.n_tiles) * TILE_M + half * CBM;
  const int n0 = (tile % p.n_tiles) * bn;
  const int kb0 = split * p.k_blocks / p.ks, kb1 = (split + 1) * p.k_blocks / p.ks;
  const bool one_cta = p.ks * (PAIR ? 2 : 1) == 1;
  const uint64_t lim = p.timeout_ns;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(tfull, 1);
    ptx::fence_mbar_init_cluster();
    ptx::fence_proxy_async_smem();
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      ptx::tmem_alloc_pair(tmem_slot, bn);
      ptx::tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(tmem_slot, bn);
      ptx::tmem_relinquish();
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  if (PAIR) ptx::cluster_sync();  // the pair's barriers are initialised
  else __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();

  // this thread's share of the epilogue: groups of 4 columns of the rows
  // [row_lo, row_hi) of the CTA's 128-row sub-tile, C_EPI apart
  const int row_lo = CBM * split / p.ks, row_hi = CBM * (split + 1) / p.ks;
  const int groups = (row_hi - row_lo) << p.lg;
  const int et = static_cast<int>(threadIdx.x) - 64;
  constexpr int U = 4;                 // groups handled at a time
  constexpr int NB = CBM * 32 / C_EPI / U;  // batches of U at most (bn = 128, one split)
  // what the epilogue reads beside the sums, fetched under the main loop:
  // GELU' of all batches, or the fp32 residual two batches ahead
  constexpr int PB = EP == E_GELU_BWD ? NB : 2;
  float4 pre[EP == E_RESID ? PB : 1][U];
  uint2 pre_g[EP == E_GELU_BWD ? PB : 1][U];
  auto prefetch = [&](int k) {
    const int base = et + k * U * C_EPI;
#pragma unroll
    for (int u = 0; u < (EP == E_RESID || EP == E_GELU_BWD ? U : 0); ++u) {
      const int g = base + u * C_EPI;
      const int row = m0 + row_lo + (g >> p.lg), col = n0 + 4 * (g & ((1 << p.lg) - 1));
      const bool in = g < groups && row < p.M && col < p.N;
      const int64_t off = static_cast<int64_t>(row) * p.N + col;
      if constexpr (EP == E_RESID) pre[k % PB][u] = in ? ld_stream_f4(p.resid + off) : make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (EP == E_GELU_BWD)
        pre_g[k][u] = in ? __ldg(reinterpret_cast<const uint2*>(p.aux + off)) : make_uint2(0u, 0u);
    }
  };

  bool ok = true;
  if (warp == 0) {
    if (lane == 0) {
      int stage = 0, issued = 0;
      uint32_t phase = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!ptx::mbar_wait(&empty[stage], phase ^ 1u, lim, p.status)) break;
        uint8_t* sa = smem + stage * sbytes;
        uint8_t* sb = sa + C_A_BYTES;
        // a pair's leader barrier expects both CTAs' bytes
        if (half == 0) ptx::mbar_arrive_expect_tx(&full[stage], (PAIR ? 2 : 1) * sbytes);
        if (!p.skip_loads) {
          const int k0 = kb * CBK;
          auto load = [&](void* dst, const CUtensorMap* map, int c0, int c1) {
            if constexpr (PAIR)
              ptx::tma_load_2d_pair(dst, map, ptx::mapa_shared(ptx::smem_u32(&full[stage]), lead_rank),
                                    c0, c1);
            else
              ptx::tma_load_2d(dst, map, &full[stage], c0, c1);
          };
          const int nb = n0 + half * b_rows;
          if (A_MN) {
            load(sa, &tmA, m0, k0);
            load(sa + C_CHUNK_BYTES, &tmA, m0 + 64, k0);
          } else {
            load(sa, &tmA, k0, m0);
          }
          if (B_MN) {
            for (int j = 0; j < b_rows / 64; ++j) load(sb + j * C_CHUNK_BYTES, &tmB, nb + 64 * j, k0);
          } else {
            load(sb, &tmB, k0, nb);
          }
        }
        ++issued;
        if (++stage == p.stages) { stage = 0; phase ^= 1u; }
      }
      // drain (bounded): the loads still in flight, counted on the leader's barriers
      const int n_tail = half ? 0 : min(issued, p.stages);
      for (int i = 0; i < n_tail; ++i) {
        if (--stage < 0) { stage = p.stages - 1; phase ^= 1u; }
        ptx::mbar_wait(&full[stage], phase, lim, p.status);
      }
    }
  } else if (warp == 1) {
    // The whole warp walks the loop, so the descriptors stay warp-uniform, and
    // one elected lane issues.
    if (half == 0) {
      const uint32_t idesc = ptx::idesc_bf16_f32(TILE_M, bn, A_MN, B_MN);
      const uint16_t mask = static_cast<uint16_t>(3u << lead_rank);
      const bool issuer = ptx::elect_one();
      auto commit = [&](uint64_t* bar) {
        if constexpr (PAIR) ptx::tc_commit_pair(bar, mask);
        else ptx::tc_commit(bar);
      };
      const uint32_t s0 = ptx::smem_u32(smem);
      const uint64_t da = A_MN ? ptx::smem_desc_sw128(s0, C_CHUNK_BYTES, 1024) : ptx::smem_desc_sw128(s0, 16, 1024);
      const uint64_t db = B_MN ? ptx::smem_desc_sw128(s0 + C_A_BYTES, C_CHUNK_BYTES, 1024)
                               : ptx::smem_desc_sw128(s0 + C_A_BYTES, 16, 1024);
      int stage = 0;
      uint32_t phase = 0;
      bool good = true;
      for (int kb = kb0; kb < kb1; ++kb) {
        good = __all_sync(0xffffffffu, ptx::mbar_wait(&full[stage], phase, lim, p.status));
        if (!good) break;
        ptx::tc_fence_after();
        if (issuer) {
          const uint64_t off = static_cast<uint64_t>(stage * (sbytes >> 4));
#pragma unroll
          for (int kk = 0; kk < CBK / 16; ++kk) {
            const uint64_t ad = da + off + kk * (A_MN ? 128 : 2), bd = db + off + kk * (B_MN ? 128 : 2);
            const uint32_t more = (kb > kb0 || kk > 0) ? 1u : 0u;
            if constexpr (PAIR) ptx::tc_mma_f16_pair(tmem_base, ad, bd, idesc, more);
            else ptx::tc_mma_f16(tmem_base, ad, bd, idesc, more);
          }
          commit(&empty[stage]);
        }
        __syncwarp();
        if (++stage == p.stages) { stage = 0; phase ^= 1u; }
      }
      // on a timeout the issued MMAs still have to finish before TMEM is released
      if (issuer) {
        commit(tfull);
        if (!good) ptx::mbar_wait(tfull, 0, lim, p.status);
      }
    }
  } else {
    // ------------------------------------- accumulator -> shared memory
    const int q = warp & 3, hf = (warp - 2) >> 2;
#pragma unroll
    for (int k = 0; k < PB; ++k) prefetch(k);
    ok = ptx::mbar_wait(tfull, 0, lim, p.status, kClusterHint);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      ptx::tc_fence_after();
      const int r = q * 32 + lane;  // row of the sub-tile = TMEM lane
      const uint32_t srow = ptx::smem_u32(smem) + static_cast<uint32_t>(r) * bn * 4;
      const uint32_t trow = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
      for (int c = hf * (bn >> 1); c < (hf + 1) * (bn >> 1); c += 16) {
        uint32_t v[16];
        ptx::tmem_ld_32x32b_x16(trow + c, v);
        ptx::tmem_ld_wait();
        // 16-byte group j of the row at position j ^ (row & 7)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          ptx::st_shared_v4(srow + ((((c >> 2) + j) ^ (r & 7)) << 4), v[4 * j], v[4 * j + 1], v[4 * j + 2],
                            v[4 * j + 3]);
      }
    }
  }
  pdl_trigger();  // behind the main loop: see common.cuh
  ptx::tc_fence_before();
  __syncwarp();
  if (one_cta) __syncthreads();
  else ptx::cluster_sync();  // every CTA's partial accumulator is in its shared memory
  if (warp == 1) {
    ptx::tc_fence_after();
    if constexpr (PAIR) ptx::tmem_dealloc_pair(tmem_base, bn);
    else ptx::tmem_dealloc(tmem_base, bn);
  }

  if (warp >= 2) {
    // ------------------------------------- fixed-order sum and epilogue
    const uint32_t sbase = ptx::smem_u32(smem);
    float* red = reinterpret_cast<float*>(smem + p.red_off);
    const int cmask = (1 << p.lg) - 1;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const int base = et + k * U * C_EPI;
      if (base - et >= groups) break;  // uniform
      float4 v[U];
      uint32_t so[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int g = min(base + u * C_EPI, groups - 1);
        const int rl = row_lo + (g >> p.lg), c = g & cmask;
        so[u] = sbase + static_cast<uint32_t>(rl) * bn * 4 + ((c ^ (rl & 7)) << 4);
      }
      if (p.ks == 1) {
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = *reinterpret_cast<const float4*>(smem + (so[u] - sbase));
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = ld_cluster_f4(ptx::mapa_shared(so[u], half));
        for (int s = 1; s < p.ks; ++s) {
          const uint32_t rank = PAIR ? 2 * s + half : s;
          float4 w[U];
#pragma unroll
          for (int u = 0; u < U; ++u) w[u] = ld_cluster_f4(ptx::mapa_shared(so[u], rank));
#pragma unroll
          for (int u = 0; u < U; ++u) {
            v[u].x += w[u].x; v[u].y += w[u].y; v[u].z += w[u].z; v[u].w += w[u].w;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int g = base + u * C_EPI;
        const int row = m0 + row_lo + (g >> p.lg), col = n0 + 4 * (g & cmask);
        if (g >= groups || row >= p.M || col >= p.N) {
          v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          continue;
        }
        const int64_t off = static_cast<int64_t>(row) * p.N + col;
        if (EP != E_GELU_BWD && p.bias) {
          const float4 b = bf4(p.bias + col);
          v[u].x += b.x; v[u].y += b.y; v[u].z += b.z; v[u].w += b.w;
        }
        if constexpr (EP == E_GELU) {
          float gp[4];
          gelu_and_grad_as(v[u].x, v[u].x, gp[0]);
          gelu_and_grad_as(v[u].y, v[u].y, gp[1]);
          gelu_and_grad_as(v[u].z, v[u].z, gp[2]);
          gelu_and_grad_as(v[u].w, v[u].w, gp[3]);
          const __half2 h0 = __floats2half2_rn(gp[0], gp[1]), h1 = __floats2half2_rn(gp[2], gp[3]);
          __stcs(reinterpret_cast<uint2*>(p.aux_out + off),
                 make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1)));
        } else if constexpr (EP == E_GELU_BWD) {
          const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&pre_g[k][u].x));
          const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&pre_g[k][u].y));
          v[u].x *= f0.x; v[u].y *= f0.y; v[u].z *= f1.x; v[u].w *= f1.y;
        } else if constexpr (EP == E_RESID) {
          if (p.ln_mean) {  // the residual is LN(u), as the LayerNorm forward evaluates it
            const float mu = __ldg(p.ln_mean + row), rs = __ldg(p.ln_rstd + row);
            const float4 gm = bf4(p.ln_gamma + col), be = bf4(p.ln_beta + col);
            v[u].x += gm.x * ((pre[k % PB][u].x - mu) * rs) + be.x;
            v[u].y += gm.y * ((pre[k % PB][u].y - mu) * rs) + be.y;
            v[u].z += gm.z * ((pre[k % PB][u].z - mu) * rs) + be.z;
            v[u].w += gm.w * ((pre[k % PB][u].w - mu) * rs) + be.w;
          } else {
            v[u].x += pre[k % PB][u].x; v[u].y += pre[k % PB][u].y; v[u].z += pre[k % PB][u].z; v[u].w += pre[k % PB][u].w;
          }
        }
        if (!ok) continue;
        if (EP == E_RESID || (EP == E_STORE && p.out_f32))
          *reinterpret_cast<float4*>(static_cast<float*>(p.C) + off) = v[u];
        else
          *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.C) + off) =
              make_uint2(ptx::pack_bf16(v[u].x, v[u].y), ptx::pack_bf16(v[u].z, v[u].w));
      }
      if (EP == E_GELU_BWD && p.colpart) {
        // Column sums per 32 rows, before rounding.  The U groups of a thread
        // are (C_EPI >> lg) rows apart: all in one 32-row block for bn = 128,
        // two blocks of two for bn = 64.  Slot t >> lg of a block's scratch
        // takes the thread's sum; the slots are added in order.
        const int slots = C_EPI >> p.lg, slot = et >> p.lg, c = et & cmask;
        const int blocks = (U * slots) / 32;  // 1 (bn = 128) or 2 (bn = 64)
        const float4 a = make_float4(v[0].x + v[1].x, v[0].y + v[1].y, v[0].z + v[1].z, v[0].w + v[1].w);
        const float4 b = make_float4(v[2].x + v[3].x, v[2].y + v[3].y, v[2].z + v[3].z, v[2].w + v[3].w);
        float4* dst = reinterpret_cast<float4*>(red);
        if (blocks == 1) {
          dst[(slot << p.lg) + c] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
        } else {
          dst[(slot << p.lg) + c] = a;
          dst[((slots + slot) << p.lg) + c] = b;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        const int blk = et / bn, cc = et - blk * bn;
        const int row = m0 + row_lo + ((base - et) >> p.lg) + 32 * blk;
        if (blk < blocks && n0 + cc < p.N && row < m0 + row_hi && ok) {
          float t = 0.f;
          for (int s = 0; s < slots; ++s) t += red[(blk * slots + s) * bn + cc];
          p.colpart[static_cast<int64_t>(row >> 5) * p.N + n0 + cc] = t;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
      }
      if (EP == E_RESID && k + PB < NB) prefetch(k + PB);
    }
  }
  __syncwarp();
  if (!one_cta) ptx::cluster_sync();  // the peers have read this CTA's partials
}

template <bool A_MN, bool B_MN, bool PAIR, int EP>
cudaError_t launch_one(const ClusterParams& p, int tiles, int smem, const CUtensorMap& ta,
                       const CUtensorMap& tb, cudaStream_t st) {
  auto kern = gemm_cluster_kernel<A_MN, B_MN, PAIR, EP>;
  static cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
  if (attr != cudaSuccess) return attr;
  const int cl = p.ks * (PAIR ? 2 : 1);
  return launch_pdl(kern, dim3(tiles * cl), dim3(C_THREADS), smem, st, cl, ta, tb, p);
}

template <bool A_MN, bool B_MN, bool PAIR>
cudaError_t launch_epi(int epi, const ClusterParams& p, int tiles, int smem, const CUtensorMap& ta,
                       const CUtensorMap& tb, cudaStream_t st) {
  if (epi == SKY_EPI_BIAS_GELU) return launch_one<A_MN, B_MN, PAIR, E_GELU>(p, tiles, smem, ta, tb, st);
  if (epi == SKY_EPI_GELU_BWD) return launch_one<A_MN, B_MN, PAIR, E_GELU_BWD>(p, tiles, smem, ta, tb, st);
  if (p.resid) return launch_one<A_MN, B_MN, PAIR, E_RESID>(p, tiles, smem, ta, tb, st);
  return launch_one<A_MN, B_MN, PAIR, E_STORE>(p, tiles, smem, ta, tb, st);
}

}  // namespace

sky_status launch_cluster(sky_gemm_form form, const ClusterPlan& pl, int M, int N, int K, const void* A,
                          const void* B, void* C, bool out_f32, int epi, const void* bias, const void* aux,
                          void* aux_out, int32_t* status, uint64_t timeout_ns, int skip_loads,
                          cudaStream_t stream, float* colpart, const float* resid, const LnResid* ln) {
  const bool a_mn = form == SKY_GEMM_XTW, b_mn = form != SKY_GEMM_XWT;
  const int b_rows = pl.pair ? pl.bn / 2 : pl.bn;
  CUtensorMap ta, tb;
  bool ok = a_mn ? make_map(&ta, A, K, M, 64) : make_map(&ta, A, M, K, CBM);
  ok = ok && (b_mn ? make_map(&tb, B, K, N, 64) : make_map(&tb, B, N, K, b_rows));
  SKY_CHECK(ok, SKY_ERR_CUDA, "cuTensorMapEncodeTiled failed (M=%d N=%d K=%d)", M, N, K);
  ClusterParams p{};
  p.M = M; p.N = N; p.bn = pl.bn;
  p.lg = pl.bn == 64 ? 4 : 5;
  p.n_tiles = ceil_div(N, pl.bn);
  p.ks = pl.ks;
  p.k_blocks = ceil_div(K, CBK);
  p.out_f32 = out_f32;
  p.C = C;
  p.bias = static_cast<const __nv_bfloat16*>(bias);
  p.aux = epi == SKY_EPI_GELU_BWD ? static_cast<const __half*>(aux) : nullptr;
  p.aux_out = static_cast<__half*>(aux_out);
  p.colpart = colpart;
  p.resid = resid;
  if (ln) {
    p.ln_mean = ln->mean;
    p.ln_rstd = ln->rstd;
    p.ln_gamma = static_cast<const __nv_bfloat16*>(ln->gamma);
    p.ln_beta = static_cast<const __nv_bfloat16*>(ln->beta);
  }
  p.status = status;
  p.timeout_ns = timeout_ns;
  p.skip_loads = skip_loads;
  // Ring: as deep as two CTAs an SM allow, also where no SM gets a second: the
  // next kernel's CTAs then fit beside this one's (1024 x 768 x 3072 in three
  // splits of 128 x 128: 12.2 us, with the whole SM's shared memory 19.9).
  const int tiles = ceil_div(M, pl.pair ? 2 * CBM : CBM) * p.n_tiles;
  const int sbytes = C_A_BYTES + b_rows * CBK * 2;
  const int red = colpart ? 8192 : 0;
  const int tail = 256 + 1024 + red;
  const int budget = 112 * 1024 - tail;
  p.stages = std::min({budget / sbytes, C_MAX_STAGES, ceil_div(p.k_blocks, pl.ks)});
  if (p.stages < 1) p.stages = 1;
  p.bar_off = std::max(p.stages * sbytes, CBM * pl.bn * 4);
  p.red_off = p.bar_off + 256;
  const int smem = p.bar_off + tail;
  cudaError_t e;
  if (pl.pair) {
    if (form == SKY_GEMM_XWT) e = launch_epi<false, false, true>(epi, p, tiles, smem, ta, tb, stream);
    else if (form == SKY_GEMM_XW) e = launch_epi<false, true, true>(epi, p, tiles, smem, ta, tb, stream);
    else e = launch_epi<true, true, true>(epi, p, tiles, smem, ta, tb, stream);
  } else {
    if (form == SKY_GEMM_XWT) e = launch_epi<false, false, false>(epi, p, tiles, smem, ta, tb, stream);
    else if (form == SKY_GEMM_XW) e = launch_epi<false, true, false>(epi, p, tiles, smem, ta, tb, stream);
    else e = launch_epi<true, true, false>(epi, p, tiles, smem, ta, tb, stream);
  }
  count_launches(1);
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "gemm_cluster_kernel launch");
}

// Which products come here, and with which tiles.  The lines were drawn through
// a sweep of every product of a layer (three forms, all epilogues) at widths 256
// to 1280 and 16 to 6000 rows, each timed in a chain of 24 launches against the
// persistent kernel with its separate split-K reduction (the "old" times):
//   more 128 x 64 tiles than two CTAs an SM hold (304): the persistent kernel,
//     whose 256-wide tiles read half the operand bytes; 4096 x 768 x 3072
//     18.5 us against 22.8 here.  Weight gradients keep 128-wide tiles up to two
//     CTAs an SM while the K range is short (no partials to write and re-read):
//     1024 x 4096 x 1024 13.1 against 11.6, and lose from 24 k-blocks on.
//   one to two CTAs an SM: one split; from 33 k-blocks on the operand traffic
//     decides, and a 256 x 128 tile on two pairs reads the least: 2048 x 768 x
//     3072 16.3 (old) / 17.3 (one split) / 15.0 us.
//   fewer tiles than SMs: splits, as long as each keeps enough k-blocks to pay
//     for the cluster barrier and the sum: 74 x 768 x 3072 17.6 -> 6.7 us (six
//     splits), 1024 x 768 x 3072 15.5 -> 11.0 (three), 1024 x 768 x 768 8.3 ->
//     6.1 (two).  Past one CTA an SM a split has to bring more.
// Over the sweep the choice is 1.5 times as fast as before at 16 to 404 rows,
// 1.3 at 1024, 1.17 at 2048.
bool plan_cluster(sky_gemm_form form, int M, int N, int K, bool may_split, bool colpart, int sms,
                  ClusterPlan* out) {
  const int kb = ceil_div(K, CBK);
  const int64_t t64 = static_cast<int64_t>(ceil_div(M, CBM)) * ceil_div(N, 64);
  const int64_t t128 = static_cast<int64_t>(ceil_div(M, CBM)) * ceil_div(N, 128);
  if (t64 > 2 * sms) {
    *out = ClusterPlan{false, 128, 1};
    return may_split && form == SKY_GEMM_XTW && t128 <= 2 * sms && kb <= 20;
  }
  if (t64 > sms) {
    *out = kb > 32 && M >= 2 * CBM && !colpart ? ClusterPlan{true, 128, 2} : ClusterPlan{false, 64, 1};
    return true;
  }
  if (may_split && kb > 80 && 2 * t64 > sms) return false;  // long weight gradients: equal or behind
  int ks = 1;
  const auto fits = [&](int s, int kb_one, int kb_two) {  // fewest k-blocks at one / two CTAs an SM
    return s * t64 <= 2 * sms && kb >= (s * t64 <= sms ? kb_one : kb_two);
  };
  if (!colpart && fits(6, 32, 64)) ks = 6;
  else if (!colpart && fits(3, 16, 32)) ks = 3;
  else if (fits(2, 12, M > CBM ? 16 : 24)) ks = 2;
  *out = ClusterPlan{false, 64, ks};
  return true;
}

}  // namespace gemm
}  // namespace sky
