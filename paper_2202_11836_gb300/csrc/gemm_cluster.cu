// bf16 GEMM for products that fill the chip poorly with 256-wide tiles: small
// tiles, and the K range of a tile split over the CTAs of a cluster.
//
// The persistent kernel of gemm_tc.cu computes 256 x 256 tiles on SM pairs.
// A product of a few hundred or thousand rows has too few of those: 1024 x 768
// (a base-width layer's output at T = 1024) is 12 tiles for 76 SM pairs, each
// walking the whole K range alone.  Here a tile is 128 x 64 (or 256 x 128 on an
// SM pair, cta_group::2), and KS CTAs (pairs) of one cluster take a contiguous
// part of its k-blocks each.  Every CTA owns a share of the tile's rows: when
// its MMAs are done it sends the rows of its fp32 accumulator to their owners
// through distributed shared memory, and after one cluster barrier the owners
// add up their rows in split order (deterministic) and run the epilogue.  So a
// split product needs no workspace and no second launch, and every epilogue
// (bias, residual, GELU, GELU') can follow a split.
//
// One work unit per CTA, no persistence: with at most 112 KiB of shared memory
// and 128 TMEM columns a CTA, two CTAs share an SM, and one's prologue and
// epilogue run under the other's main loop.  The choice between the two kernels
// and of the tile and split is made on the host (plan_cluster).
//
// At these sizes the kernel is a chain of latencies.  For 74 x 768 x 3072 in six
// splits (globaltimer, us after the wait for the kernel before): first operands
// 0.8, accumulator 2.3.  Reading the partial rows from the peers instead (one
// split after the other, then a second barrier before anyone may leave) and
// fetching the bias behind it took 4.6 us more; sending them, all loads at once
// and everything else fetched under the main loop takes 2.1 us.
//
//   warp 0      TMA producer, warp 1 MMA issuer (as in gemm_tc.cu)
//   warps 2..9  accumulator -> owners' shared memory, then the sum and epilogue
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "gemm.h"
#include "ptx.cuh"
#include "residency.h"

namespace sky {
namespace gemm {
namespace {

constexpr int CBM = 128, CBK = 64;
constexpr int C_A_BYTES = CBM * CBK * 2;        // 16 KiB
constexpr int C_CHUNK_BYTES = 64 * CBK * 2;     // one 64-wide MN-major box: 8 KiB
constexpr int C_EPI = 256;                      // epilogue threads (8 warps)
constexpr int C_THREADS = 64 + C_EPI;
constexpr int C_MAX_STAGES = 8;
constexpr int C_SMEM = 112 * 1024;              // of a CTA: two share an SM
constexpr uint32_t kClusterHint = 2000;         // suspend hint of the epilogue's accumulator wait

struct ClusterParams {
  int M, N;
  int n_tiles, k_blocks, stages;
  int recv_off, bar_off, red_off;  // shared-memory offsets: received rows, barriers, column-sum scratch
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
  int skip_loads;  // fault injection: no TMA copies (2: only the last split's are left out)
};

// Tile and split of an instantiation, and what follows from them.
template <bool PAIR_, int BN_, int KS_>
struct Tiling {
  static constexpr bool PAIR = PAIR_;
  static constexpr int BN = BN_, KS = KS_;
  static constexpr int TILE_M = PAIR ? 2 * CBM : CBM;
  static constexpr int CL = KS * (PAIR ? 2 : 1);           // CTAs of a cluster
  static constexpr int B_ROWS = PAIR ? BN / 2 : BN;        // tile columns whose B operand a CTA loads
  static constexpr int SBYTES = C_A_BYTES + B_ROWS * CBK * 2;
  // Rows sent to their owners need room that no peer's main loop still uses.  A
  // pair's 128-wide rows would cost it half the ring: its CTAs keep their partial
  // tile over the ring, and the owners read it there.
  static constexpr bool PUSH = KS > 1 && !PAIR;
  static constexpr int ROWS = (CBM + KS - 1) / KS;         // most rows a CTA owns
  static constexpr int GPR = BN / 4;                       // 4-column groups of a row
  static constexpr int GT = (ROWS * GPR + C_EPI - 1) / C_EPI;  // groups of an epilogue thread
  // groups handled at a time: about eight partial groups in flight
  static constexpr int U = KS >= 6 ? 2 : (KS == 3 ? 3 : (GT < 4 ? GT : 4));
  static constexpr int BATCHES = (GT + U - 1) / U;
  static constexpr int RECV_BYTES = PUSH ? KS * ROWS * BN * 4 : 0;  // a multiple of 256
};

__device__ __forceinline__ float4 ld_stream_f4(const float* p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
// (also of what the kernel itself overwrites later)
__device__ __forceinline__ float4 ld_own_f4(const float* p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
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
// GELU, bias then GELU', bias + fp32 residual or LayerNorm residual (fp32 output), and
// C += product (fp32).
enum { E_STORE, E_GELU, E_GELU_BWD, E_RESID, E_ADD };

template <bool A_MN, bool B_MN, class TL, int EP>
__global__ void __launch_bounds__(C_THREADS, 2)
    gemm_cluster_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const ClusterParams p) {
  constexpr bool PAIR = TL::PAIR;
  constexpr int BN = TL::BN, KS = TL::KS, U = TL::U, GPR = TL::GPR, SBYTES = TL::SBYTES;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + p.bar_off);
  uint64_t* empty = full + C_MAX_STAGES;
  uint64_t* tfull = empty + C_MAX_STAGES;
  uint64_t* done = tfull + 1;  // after a time-out: the issued MMAs have finished
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  // Set in every CTA of the cluster by one whose accumulator did not come: no part
  // of the tile is stored then.
  const uint32_t lost = ptx::smem_u32(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t crank = ptx::cluster_ctarank();
  const int half = PAIR ? static_cast<int>(crank & 1) : 0;  // 128-row half of the pair's tile
  const int split = static_cast<int>(PAIR ? crank >> 1 : crank);
  const uint32_t lead_rank = crank - half;
  const int tile = static_cast<int>(blockIdx.x) / TL::CL;
  const int m0 = (tile / p.n_tiles) * TL::TILE_M + half * CBM;
  const int n0 = (tile % p.n_tiles) * BN;
  const int kb0 = split * p.k_blocks / KS, kb1 = (split + 1) * p.k_blocks / KS;
  const uint64_t lim = p.timeout_ns;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(tfull, 1);
    ptx::mbar_init(done, 1);
    ptx::st_shared_u32(lost, 0);
    if (TL::PUSH) ptx::fence_cluster();  // with the arrival below: before a peer writes it
    ptx::fence_mbar_init_cluster();
    ptx::fence_proxy_async_smem();
    ptx::prefetch_tensormap(&tmA);
    ptx::prefetch_tensormap(&tmB);
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      ptx::tmem_alloc_pair(tmem_slot, BN);
      ptx::tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(tmem_slot, BN);
      ptx::tmem_relinquish();
    }
  }
  ptx::tc_fence_before();
  __syncwarp();
  if constexpr (PAIR) ptx::cluster_sync();  // the pair's barriers are initialised
  else __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // this CTA runs: its peers may write its shared memory once they have seen this
  if constexpr (TL::PUSH) ptx::cluster_arrive();
  pdl_wait();

  // Rows [row_lo, row_hi) of the CTA's 128-row sub-tile are this CTA's to finish.
  // Epilogue thread et takes 4-column group et % GPR of rows et / GPR, + C_EPI / GPR, ...
  const int row_lo = CBM * split / KS, row_hi = CBM * (split + 1) / KS;
  const int et = static_cast<int>(threadIdx.x) - 64;
  constexpr int RSTEP = C_EPI / GPR;
  bool ok = true;
  // what the epilogue needs beside the sums, fetched under the main loop
  float4 bias4 = make_float4(0.f, 0.f, 0.f, 0.f), gm4 = bias4, be4 = bias4;
  float4 pre[EP == E_RESID || EP == E_ADD ? TL::GT : 1];
  float mu[EP == E_RESID ? TL::GT : 1], rs[EP == E_RESID ? TL::GT : 1];
  uint2 pre_g[EP == E_GELU_BWD ? TL::GT : 1];

  if (warp == 0) {
    const bool issuer = ptx::elect_one();
    const bool skip = p.skip_loads != 0 && (p.skip_loads != 2 || split == KS - 1);  // fault injection
    int stage = 0, issued = 0;
    uint32_t phase = 0;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(&empty[stage], phase ^ 1u, lim, p.status))) break;
      if (issuer) {
        uint8_t* sa = smem + stage * SBYTES;
        uint8_t* sb = sa + C_A_BYTES;
        // a pair's leader barrier expects both CTAs' bytes
        if (half == 0) ptx::mbar_arrive_expect_tx(&full[stage], (PAIR ? 2 : 1) * SBYTES);
        if (!skip) {
          const int k0 = kb * CBK;
          auto load = [&](void* dst, const CUtensorMap* map, int c0, int c1) {
            if constexpr (PAIR)
              ptx::tma_load_2d_pair(dst, map, ptx::mapa_shared(ptx::smem_u32(&full[stage]), lead_rank),
                                    c0, c1);
            else
              ptx::tma_load_2d(dst, map, &full[stage], c0, c1);
          };
          const int nb = n0 + half * TL::B_ROWS;
          if (A_MN) {
            load(sa, &tmA, m0, k0);
            load(sa + C_CHUNK_BYTES, &tmA, m0 + 64, k0);
          } else {
            load(sa, &tmA, k0, m0);
          }
          if (B_MN) {
#pragma unroll
            for (int j = 0; j < TL::B_ROWS / 64; ++j) load(sb + j * C_CHUNK_BYTES, &tmB, nb + 64 * j, k0);
          } else {
            load(sb, &tmB, k0, nb);
          }
        }
      }
      __syncwarp();
      ++issued;
      if (++stage == p.stages) { stage = 0; phase ^= 1u; }
    }
    // drain (bounded): the loads still in flight, counted on the leader's barriers
    const int n_tail = half ? 0 : min(issued, p.stages);
    for (int i = 0; i < n_tail; ++i) {
      if (--stage < 0) { stage = p.stages - 1; phase ^= 1u; }
      ptx::mbar_wait(&full[stage], phase, lim, p.status);
    }
  } else if (warp == 1) {
    // The whole warp walks the loop, so the descriptors stay warp-uniform, and
    // one elected lane issues.
    if (half == 0) {
      constexpr uint32_t idesc = ptx::idesc_bf16_f32(TL::TILE_M, BN, A_MN, B_MN);
      const bool issuer = ptx::elect_one();
      auto commit = [&](uint64_t* bar, uint32_t to = 3) {  // pair: bit 0 this CTA, bit 1 its peer
        if constexpr (PAIR) ptx::tc_commit_pair(bar, static_cast<uint16_t>(to << lead_rank));
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
          const uint64_t off = static_cast<uint64_t>(stage * (SBYTES >> 4));
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
      // The issued MMAs have to finish before TMEM is released.  On a timeout they
      // do so behind a barrier that no epilogue waits for.
      if (issuer) {
        if (good) commit(tfull);
        else commit(done, 1);
        ptx::mbar_wait(good ? tfull : done, 0, lim, p.status);
      }
      __syncwarp();
    }
  } else {
    const int col = n0 + 4 * (et % GPR);
    if (col < p.N) {
      if (p.bias) bias4 = bf4(p.bias + col);
      if (EP == E_RESID && p.ln_mean) {
        gm4 = bf4(p.ln_gamma + col);
        be4 = bf4(p.ln_beta + col);
      }
    }
    if constexpr (EP == E_RESID || EP == E_GELU_BWD || EP == E_ADD) {
#pragma unroll
      for (int i = 0; i < TL::GT; ++i) {
        const int rl = row_lo + et / GPR + i * RSTEP, row = m0 + rl;
        const bool in = rl < row_hi && row < p.M && col < p.N;
        const int64_t off = static_cast<int64_t>(row) * p.N + col;
        if constexpr (EP == E_RESID) {
          pre[i] = in ? ld_stream_f4(p.resid + off) : make_float4(0.f, 0.f, 0.f, 0.f);
          mu[i] = in && p.ln_mean ? __ldg(p.ln_mean + row) : 0.f;
          rs[i] = in && p.ln_mean ? __ldg(p.ln_rstd + row) : 0.f;
        } else if constexpr (EP == E_ADD) {
          pre[i] = in ? ld_own_f4(static_cast<const float*>(p.C) + off) : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
          pre_g[i] = in ? __ldg(reinterpret_cast<const uint2*>(p.aux + off)) : make_uint2(0u, 0u);
        }
      }
    }
    // ---------------------- accumulator rows -> their owners' shared memory
    const int q = warp & 3, hf = (warp - 2) >> 2;
    auto give_up = [&]() {
      if (lane < TL::CL) ptx::st_cluster_u32(ptx::mapa_shared(lost, lane), 1);
    };
    ok = ptx::mbar_wait(tfull, 0, lim, p.status, kClusterHint);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      ptx::tc_fence_after();
      const int r = q * 32 + lane;  // row of the sub-tile = TMEM lane
      const uint32_t dst = ptx::smem_u32(smem) + static_cast<uint32_t>(r) * BN * 4;
      const uint32_t trow = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll
      for (int c = 0; c < BN / 2; c += 32) {
        uint32_t v[32];
        ptx::tmem_ld_32x32b_x32(trow + hf * (BN / 2) + c, v);
        ptx::tmem_ld_wait();
        // over the ring, 16-byte group j of the row at position j ^ (row & 7)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          ptx::st_shared_v4(dst + (((hf * (BN / 8) + (c >> 2) + j) ^ (r & 7)) << 4), v[4 * j], v[4 * j + 1],
                            v[4 * j + 2], v[4 * j + 3]);
      }
    } else if (!TL::PUSH) {
      give_up();
    }
    if constexpr (TL::PUSH) {
      // rows to their owners, half a warp a row (a row a lane, straight from the
      // accumulator, took 1.3 us instead of 0.5)
      ptx::cluster_wait();  // every peer runs
      if (!ok) give_up();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      const uint32_t sm0 = ptx::smem_u32(smem);
      constexpr int N = CBM * GPR / C_EPI;
      float4 v[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int r = et / GPR + i * RSTEP;
        v[i] = ptx::ld_shared_f4(sm0 + static_cast<uint32_t>(r * BN * 4) + (((et % GPR) ^ (r & 7)) << 4));
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int r = et / GPR + i * RSTEP;
        const int owner = ((r + 1) * KS - 1) / CBM;  // the last o with CBM * o / KS <= r
        const uint32_t at = ptx::mapa_shared(sm0 + p.recv_off, owner) +
                            static_cast<uint32_t>((split * TL::ROWS + r - CBM * owner / KS) * BN * 4) +
                            (((et % GPR) ^ (r & 7)) << 4);
        ptx::st_cluster_v4(at, __float_as_uint(v[i].x), __float_as_uint(v[i].y), __float_as_uint(v[i].z),
                           __float_as_uint(v[i].w));
      }
    }
  }
  pdl_trigger();  // behind the main loop: see common.cuh
  ptx::tc_fence_before();
  __syncwarp();
  if constexpr (TL::PUSH) {
    if (warp < 2) ptx::cluster_wait();  // (the epilogue warps have)
  }
  if constexpr (TL::CL == 1) __syncthreads();
  else ptx::cluster_sync();  // every partial row is where it is read from
  if (warp == 1) {
    ptx::tc_fence_after();
    if constexpr (PAIR) ptx::tmem_dealloc_pair(tmem_base, BN);
    else ptx::tmem_dealloc(tmem_base, BN);
  }

  if (warp >= 2) {
    // ------------------------------------- fixed-order sum and epilogue
    const uint32_t sbase = ptx::smem_u32(smem) + (TL::PUSH ? p.recv_off : 0);
    float* red = reinterpret_cast<float*>(smem + p.red_off);
    const int c = et % GPR, col = n0 + 4 * c;
#pragma unroll
    for (int b = 0; b < TL::BATCHES; ++b) {
      float4 v[U], w[U][KS];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int rl = min(row_lo + et / GPR + (b * U + u) * RSTEP, row_hi - 1);
#pragma unroll
        for (int s = 0; s < KS; ++s) {
          if constexpr (TL::PUSH || KS == 1) {
            const uint32_t at = sbase + static_cast<uint32_t>((TL::PUSH ? s * TL::ROWS + rl - row_lo : rl) * BN * 4) +
                                ((c ^ (rl & 7)) << 4);
            w[u][s] = ptx::ld_shared_f4(at);
          } else {
            const uint32_t at = sbase + static_cast<uint32_t>(rl * BN * 4) + ((c ^ (rl & 7)) << 4);
            w[u][s] = ptx::ld_cluster_f4(ptx::mapa_shared(at, PAIR ? 2 * s + half : s));
          }
        }
      }
      if (b == 0) ok = ptx::ld_shared_u32(lost) == 0;  // (behind the first sums' loads)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        v[u] = w[u][0];
#pragma unroll
        for (int s = 1; s < KS; ++s) {
          v[u].x += w[u][s].x; v[u].y += w[u][s].y; v[u].z += w[u][s].z; v[u].w += w[u][s].w;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = b * U + u;
        const int rl = row_lo + et / GPR + i * RSTEP, row = m0 + rl;
        if (i >= TL::GT || rl >= row_hi || row >= p.M || col >= p.N) {
          v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          continue;
        }
        const int64_t off = static_cast<int64_t>(row) * p.N + col;
        v[u].x += bias4.x; v[u].y += bias4.y; v[u].z += bias4.z; v[u].w += bias4.w;
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
          const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&pre_g[i].x));
          const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&pre_g[i].y));
          v[u].x *= f0.x; v[u].y *= f0.y; v[u].z *= f1.x; v[u].w *= f1.y;
        } else if constexpr (EP == E_RESID) {
          if (p.ln_mean) {  // the residual is LN(u), as the LayerNorm forward evaluates it
            v[u].x += gm4.x * ((pre[i].x - mu[i]) * rs[i]) + be4.x;
            v[u].y += gm4.y * ((pre[i].y - mu[i]) * rs[i]) + be4.y;
            v[u].z += gm4.z * ((pre[i].z - mu[i]) * rs[i]) + be4.z;
            v[u].w += gm4.w * ((pre[i].w - mu[i]) * rs[i]) + be4.w;
          } else {
            v[u].x += pre[i].x; v[u].y += pre[i].y; v[u].z += pre[i].z; v[u].w += pre[i].w;
          }
        } else if constexpr (EP == E_ADD) {
          v[u].x += pre[i].x; v[u].y += pre[i].y; v[u].z += pre[i].z; v[u].w += pre[i].w;
        }
        if (!ok) continue;
        if (EP == E_RESID || EP == E_ADD || (EP == E_STORE && p.out_f32))
          *reinterpret_cast<float4*>(static_cast<float*>(p.C) + off) = v[u];
        else
          *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.C) + off) =
              make_uint2(ptx::pack_bf16(v[u].x, v[u].y), ptx::pack_bf16(v[u].z, v[u].w));
      }
      if constexpr (EP == E_GELU_BWD && BN == 64 && U == 4 && KS <= 2) {
        if (p.colpart) {
          // Column sums per 32 rows, before rounding: a thread's four groups are
          // 16 rows apart, two in each of the batch's two 32-row blocks.  A block's
          // 16 sums per column are added in order.
          float4* dst = reinterpret_cast<float4*>(red);
          dst[et] = make_float4(v[0].x + v[1].x, v[0].y + v[1].y, v[0].z + v[1].z, v[0].w + v[1].w);
          dst[C_EPI + et] = make_float4(v[2].x + v[3].x, v[2].y + v[3].y, v[2].z + v[3].z, v[2].w + v[3].w);
          asm volatile("bar.sync 1, 256;" ::: "memory");
          const int blk = et >> 6, cc = et & 63;
          const int row = m0 + row_lo + b * 64 + 32 * blk;
          if (blk < 2 && n0 + cc < p.N && ok) {
            float t = 0.f;
#pragma unroll
            for (int s = 0; s < 16; ++s) t += red[(blk * 16 + s) * 64 + cc];
            p.colpart[static_cast<int64_t>(row >> 5) * p.N + n0 + cc] = t;
          }
          asm volatile("bar.sync 1, 256;" ::: "memory");
        }
      }
    }
  }
  if constexpr (TL::CL > 1 && !TL::PUSH) {
    __syncwarp();
    ptx::cluster_sync();  // the peers have read this CTA's partial rows
  }
}

template <bool A_MN, bool B_MN, class TL, int EP>
cudaError_t launch_one(ClusterParams& p, const CUtensorMap& ta, const CUtensorMap& tb, cudaStream_t st) {
  auto kern = gemm_cluster_kernel<A_MN, B_MN, TL, EP>;
  static OncePerDevice once;
  const cudaError_t attr = allow_smem(once, kern, C_SMEM);
  if (attr != cudaSuccess) return attr;
  // Ring: as deep as two CTAs an SM allow, also where no SM gets a second: the
  // next kernel's CTAs then fit beside this one's (1024 x 768 x 3072 in three
  // splits of 128 x 128: 12.2 us, with the whole SM's shared memory 19.9).
  const int red = p.colpart ? 8192 : 0, tail = 256 + 1024 + red;
  const int room = C_SMEM - tail - TL::RECV_BYTES;
  p.stages = std::max(1, std::min({room / TL::SBYTES, C_MAX_STAGES, ceil_div(p.k_blocks, TL::KS)}));
  const int ring = std::max(p.stages * TL::SBYTES, CBM * TL::BN * 4);  // (the partial tile goes over it)
  p.recv_off = ring;
  p.bar_off = ring + TL::RECV_BYTES;
  p.red_off = p.bar_off + 256;
  const int tiles = ceil_div(p.M, TL::TILE_M) * p.n_tiles;
  static_assert(kClusterProductSmem <= C_SMEM && TL::BN <= 128, "see residency.h");
  const int smem = std::max(p.bar_off + tail, TL::CL > 1 ? kClusterProductSmem : 0);
  return launch_pdl(kern, dim3(tiles * TL::CL), dim3(C_THREADS), smem, st, TL::CL, ta, tb, p);
}

template <bool A_MN, bool B_MN, class TL>
cudaError_t launch_epi(int epi, ClusterParams& p, const CUtensorMap& ta, const CUtensorMap& tb, cudaStream_t st) {
  if (epi == SKY_EPI_BIAS_GELU) return launch_one<A_MN, B_MN, TL, E_GELU>(p, ta, tb, st);
  if (epi == SKY_EPI_GELU_BWD) return launch_one<A_MN, B_MN, TL, E_GELU_BWD>(p, ta, tb, st);
  if (p.resid) return launch_one<A_MN, B_MN, TL, A_MN ? E_ADD : E_RESID>(p, ta, tb, st);
  return launch_one<A_MN, B_MN, TL, E_STORE>(p, ta, tb, st);
}

template <bool A_MN, bool B_MN>
cudaError_t launch_plan(const ClusterPlan& pl, int epi, ClusterParams& p, const CUtensorMap& ta,
                        const CUtensorMap& tb, cudaStream_t st) {
  if (pl.pair) return launch_epi<A_MN, B_MN, Tiling<true, 128, 2>>(epi, p, ta, tb, st);
  if constexpr (A_MN) {
    if (pl.bn == 128)
      return p.resid ? launch_one<A_MN, B_MN, Tiling<false, 128, 1>, E_ADD>(p, ta, tb, st)
                     : launch_one<A_MN, B_MN, Tiling<false, 128, 1>, E_STORE>(p, ta, tb, st);
  }
  switch (pl.ks) {
    case 6: return launch_epi<A_MN, B_MN, Tiling<false, 64, 6>>(epi, p, ta, tb, st);
    case 3: return launch_epi<A_MN, B_MN, Tiling<false, 64, 3>>(epi, p, ta, tb, st);
    case 2: return launch_epi<A_MN, B_MN, Tiling<false, 64, 2>>(epi, p, ta, tb, st);
    default: return launch_epi<A_MN, B_MN, Tiling<false, 64, 1>>(epi, p, ta, tb, st);
  }
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
  p.M = M; p.N = N;
  p.n_tiles = ceil_div(N, pl.bn);
  p.k_blocks = ceil_div(K, CBK);
  p.out_f32 = out_f32;
  p.C = C;
  p.bias = static_cast<const __nv_bfloat16*>(bias);
  p.aux = static_cast<const __half*>(aux);
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
  cudaError_t e;
  if (form == SKY_GEMM_XWT) e = launch_plan<false, false>(pl, epi, p, ta, tb, stream);
  else if (form == SKY_GEMM_XW) e = launch_plan<false, true>(pl, epi, p, ta, tb, stream);
  else e = launch_plan<true, true>(pl, epi, p, ta, tb, stream);
  count_launches(1);
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "gemm_cluster_kernel launch");
}

// Which products come here, and with which tiles.  The lines were drawn through
// a sweep of every product of a layer (three forms, all epilogues) at widths 256
// to 1280 and 16 to 6000 rows, each timed in a chain of 24 launches against the
// persistent kernel with its separate split-K reduction ("old"; us below):
//   more 128 x 64 tiles than two CTAs an SM hold (304): the persistent kernel,
//     whose 256-wide tiles read half the operand bytes.  Weight gradients keep
//     128 x 128 tiles while the K range is short (no partials to write and
//     re-read), longer where 256-wide tiles fill their last wave badly: 1024 x
//     4096 x 1024 old 13.1, here 11.1; 3072 x 1024 x 1500 20.1 and 13.1.
//   one to two CTAs an SM: no split; from 40 k-blocks on the operand traffic
//     decides, and a 256 x 128 tile on two pairs reads the least.
//   half to one CTA an SM: the same from 24 k-blocks on (2048 x 768 x 3072 old
//     18.3, unsplit 15.9, here 13.2); a split of 64-wide tiles, with more CTAs
//     than SMs, loses.
//   fewer: from 12 k-blocks on two splits, and three or six while the clusters
//     fill no more than three quarters of the SMs (they have to fit the SMs'
//     groups): 64 x 768 x 3072 old 18.7, six splits 5.2; 1024 x 768 x 768 old 8.0,
//     unsplit 5.1.  Six also on all SMs from 64 k-blocks on (256 x 768 x 4096 in
//     three 7.4, six 7.5; x 6144 9.4 and 8.8), and three also with up to one and a
//     half CTAs an SM over 96 (768 x 768 x 6144 in two 14.3, three 13.7; x 8192 23.5
//     and 18.6).  Under 12 a split gains nothing (64 x 768 x 512 3.5, in two 4.0, six
//     3.8; x 640 3.9, 4.1 and 3.8).
// Long K ranges whose partial sums the workspace can take (weight gradients of
// many tokens; others have no other split and stay): few CTAs do not draw the
// operands from memory fast enough, and the persistent kernel's splits, on all SM
// pairs, are level or better.  M x N x K, old and here with the operands in L2 / in
// memory:
//   under half a CTA an SM, over 32 k-blocks a CTA and SM, or over 200: 768 x 768 x
//     4096 12.5 13.4 / 9.7 13.5, x 8192 15.1 15.9 / 17.0 19.0; 512 x 512 x 8192 12.8
//     14.1 / 11.5 17.5, x 16384 16.6 18.1 / 19.7 30.8; 128 x 768 x 12288 12.7 14.6 / 9.7
//     14.6, x 16384 14.1 16.3 / 11.7 18.3.
//   up to one CTA an SM, over 88: level or better.
//   above, over 88 where the pairs' last wave is less than a third full: 1024 x
//     1536 x 5000 18.0 19.0 / 17.8 19.2, x 8192 22.5 23.4 / 24.4 26.6; fuller ones stay:
//     768 x 2304 x 8192 27.6 28.4 / 24.9 27.6.
// Over the sweep the choice is twice as fast as before at 64 and 128 rows, 1.8
// times at 404, 1.6 at 1024, 1.34 at 2048, 1.15 at 4096.
bool plan_cluster(sky_gemm_form form, int M, int N, int K, bool may_split, bool ws_split, bool colpart, int sms,
                  ClusterPlan* out) {
  const int kb = ceil_div(K, CBK);
  const int64_t t64 = static_cast<int64_t>(ceil_div(M, CBM)) * ceil_div(N, 64);
  if (t64 > 2 * sms) {
    if (!may_split || form != SKY_GEMM_XTW || 3 * t64 > 16 * sms) return false;
    const int64_t t256 = static_cast<int64_t>(ceil_div(M, 2 * CBM)) * ceil_div(N, 256), pairs = sms / 2;
    const bool full = 4 * t256 > 3 * pairs * ceil_div(t256, pairs);
    *out = ClusterPlan{false, 128, 1};
    return kb <= (full ? 24 : 48);
  }
  const bool many = t64 > sms / 2;
  if (ws_split) {
    const int64_t pairs = std::max(1, sms / 2), units = 2 * static_cast<int64_t>(ceil_div(M, 2 * CBM)) * ceil_div(N, 128);
    if (!many && (kb * t64 > 32 * sms || kb > 200)) return false;
    if (many && kb > 88 && (t64 <= sms || 3 * units < 2 * pairs * ceil_div(units, pairs))) return false;
  }
  if (many) {
    const bool pair = M >= 2 * CBM && !colpart && kb >= (t64 <= sms ? 24 : 40);
    *out = pair ? ClusterPlan{true, 128, 2} : ClusterPlan{false, 64, 1};
    return true;
  }
  const int64_t room = 3 * sms / 4;
  int ks = 1;
  if (kb >= 12) {
    ks = 2;
    if (!colpart) {
      if (6 * t64 <= (kb >= 64 ? sms : room)) ks = 6;
      else if (3 * t64 <= room) ks = 3;
      else if (kb > 96) ks = 3;
    }
  }
  *out = ClusterPlan{false, 64, ks};
  return true;
}

}  // namespace gemm
}  // namespace sky
