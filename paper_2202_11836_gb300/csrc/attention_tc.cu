// Masked scaled dot-product attention (Eq. 1) forward and backward on the
// 5th-generation tensor cores, bf16, head dim D = 64.
//
// Forward: one CTA owns 128 query rows of one (sequence b, head a).  Per
// 64-key tile j (only tiles below len[b] are visited):
//   S_j = Q K_j^T                  tcgen05.mma M=128 N=64 K=64 -> TMEM
//   softmax (4 warps, thread = query row = TMEM lane): row max over the
//     valid keys, P_j = exp2(S_j log2(e)/sqrt(D) - m) written as bf16 pairs
//     over the scores (tcgen05.st), where the next product reads it
//   O += P_j V_j                   tcgen05.mma M=128 N=64 K=64, A = P_j from
//                                  TMEM, B = V_j from shared memory -> TMEM
// Q, K and V come straight out of the packed QKV activations by TMA (one
// tensor map, per-head column offsets), and O / l leaves by TMA from shared
// memory.  Because a thread owns a whole query row, the row max and row sum
// need no shuffles.
//
// A tile's chain (S, softmax, P V) is serial, so tiles have to overlap.  Two forms
// of the kernel, chosen by the launcher, do it:
//   two score buffers (NS = 2): S_{j+1} runs beside the softmax of tile j.  256
//     TMEM columns, so two CTAs an SM; a tile takes 0.53 us alone (S = 2048).
//   one (NS = 1): P over the only S; 128 TMEM columns, 49 KiB of shared memory and
//     80 registers a thread (half a row's scores at a time, the high half read
//     twice), so four CTAs overlap on an SM.  A tile takes 0.85 us alone, but a full
//     SM finishes more of them: 16 heads x 4 full sequences of 2048, 81 us against
//     86.  No pipe is full then (ncu: issue 46%, tensor 37%, XU 37% of the active
//     cycles); three CTAs an SM were slower.
// Where the query blocks are few, KS = 2 or 4 CTAs of a cluster share a block's keys:
// each leaves its part of O, m and l in shared memory, and each finishes 128 / KS of
// the rows from its peers' parts.  4 heads x 2048: 19.9 us before, 17.3 unsplit, 10.3
// in four; the combination costs 2 us and more with more clusters.
//
// The exponent offset m of a row is only raised when the
// tile's max exceeds it by more than 2^8 (a factor 256 in P): then O and the row
// sum are rescaled in TMEM.  Otherwise P may exceed 1 by at most that factor,
// which bf16 and the fp32 sums carry with the same relative precision; the final
// O / l and the log-sum-exp do not depend on m.  The log-sum-exp is kept in
// base-2 units, lse2 = log2 sum_j exp2(S_ij log2(e)/sqrt(D)), which is what the
// backward kernels subtract in the exponent.  All mbarrier waits are time-bounded.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cfloat>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"
#include "residency.h"

namespace sky {
namespace attn_tc {

constexpr int BQ = 128, BKV = 64, HD = 64;
constexpr int Q_BYTES = BQ * HD * 2;    // 16 KiB
constexpr int KV_BYTES = BKV * HD * 2;  // 8 KiB per K or V tile
// forward CTA: warp 0 TMA, warp 1 MMA issue, warps 2..5 softmax
constexpr int NTHR = 192;
// The backward kernels run eight softmax warps: warps w and w + 4 share TMEM
// lane quarter w % 4 and take the low / high 32 columns of each 64-wide tile.
constexpr int NSM_B = 256;              // softmax threads in the backward kernels
// Backward CTAs: warp 0 TMA, warp 1 issues the score products (S and dP),
// warps 2..9 softmax, warp 10 issues the accumulating products (dQ, or dV
// and dK), so that neither kind waits behind the other's barriers.
constexpr int NTHR_B = 352;
constexpr float LOG2E = 1.4426950408889634f;
// Suspend-time hint (ns) of every mbarrier wait: a waiting thread sleeps
// until the phase completes instead of spinning on issue slots that the
// softmax warps (the critical path) share with the producer and MMA threads.
constexpr uint32_t kWaitHint = 10000;

// Forward kernel with NS score buffers: four CTAs an SM with one, two with two.
// Shared-memory layout (offsets from a 1024-byte aligned base).  TMEM: S_0, then
// S_1, 64 columns each, of which P as bf16 pairs takes the first 32 (the A operand
// of P V, read from tensor memory); O: 64 columns behind them.
template <int NS>
struct FwdShape {
  static constexpr int CTAS = NS == 1 ? 4 : 2;  // per SM
  static constexpr int STAGES = NS + 1;         // K/V ring
  static constexpr int Q_OFF = 0;
  static constexpr int KV_OFF = Q_OFF + Q_BYTES;  // [STAGES] x {K, V}
  static constexpr int BAR_OFF = KV_OFF + STAGES * 2 * KV_BYTES;
  static constexpr int ML_OFF = BAR_OFF + 256;    // split keys: m and l of each row
  static constexpr int SMEM = ML_OFF + BQ * 8 + 1024;
  static constexpr int TMEM_COLS = 128 * NS;
};
static_assert(FwdShape<1>::CTAS * (FwdShape<1>::SMEM + 1024) <= 233472, "four forward CTAs per SM");
static_assert(FwdShape<1>::STAGES * 2 * KV_BYTES >= BQ * HD * 4, "a partial O goes over the K/V stages");
constexpr float kRescaleLog2 = 8.f;

struct FwdParams {
  int S, H, A;
  const int32_t* lens;
  __nv_bfloat16* ctx;
  float* lse;
  int32_t* status;
  uint64_t timeout_ns;
};

template <int KS, int NS>
__global__ void __launch_bounds__(NTHR, FwdShape<NS>::CTAS) attn_fwd_tc(const __grid_constant__ CUtensorMap tmQ,
                                                    const __grid_constant__ CUtensorMap tmKV,
                                                    const __grid_constant__ CUtensorMap tmOut,
                                                    const FwdParams p) {
  using SH = FwdShape<NS>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint64_t* q_full = reinterpret_cast<uint64_t*>(smem + SH::BAR_OFF);
  uint64_t* kv_full = q_full + 1;
  uint64_t* kv_empty = kv_full + SH::STAGES;
  uint64_t* s_full = kv_empty + SH::STAGES;  // [NS] S_j complete
  uint64_t* p_full = s_full + NS;            // [NS] P_j in tensor memory
  uint64_t* pv_done = p_full + NS;           // [NS] O += P_j V_j complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(pv_done + NS);

  const int qt = blockIdx.x / KS, split = blockIdx.x % KS, a = blockIdx.y, b = blockIdx.z;
  const int S = p.S, H = p.H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = b * S;  // first token row of this sequence
  const int q0 = qt * BQ;
  const uint64_t lim = p.timeout_ns;

  if (threadIdx.x == 0) {
    ptx::mbar_init(q_full, 1);
    for (int s = 0; s < SH::STAGES; ++s) {
      ptx::mbar_init(&kv_full[s], 1);
      ptx::mbar_init(&kv_empty[s], 1);
    }
    for (int s = 0; s < NS; ++s) {
      ptx::mbar_init(&s_full[s], 1);
      ptx::mbar_init(&p_full[s], 128);
      ptx::mbar_init(&pv_done[s], 1);
    }
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
    ptx::prefetch_tensormap(&tmQ);
    ptx::prefetch_tensormap(&tmKV);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, SH::TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tS0 = tmem, tO = tmem + 64 * NS;
  pdl_wait();
  int len = p.lens[b];
  if (len < 1 || len > S) {
    if (p.status && threadIdx.x == 0) atomicOr(p.status, kStatusBadLength);
    len = len < 1 ? 1 : S;
  }
  const int n_all = (len + BKV - 1) / BKV;
  const int j0 = split * n_all / KS, n_kt = (split + 1) * n_all / KS - j0;  // this CTA's key tiles
  const int last = n_kt > 0 ? n_kt - 1 : 0;

  if (warp == 0) {
    // ------------------------------------------------------------- producer
    const bool issuer = ptx::elect_one();
    if (issuer) {
      ptx::mbar_arrive_expect_tx(q_full, Q_BYTES);
      ptx::tma_load_2d(smem + SH::Q_OFF, &tmQ, q_full, a * HD, row0 + q0);
    }
    __syncwarp();
    int issued = 0;
    for (int j = 0; j < n_kt; ++j) {
      const int st = j % SH::STAGES;
      if (!__all_sync(0xffffffffu,
                      ptx::mbar_wait(&kv_empty[st], ((j / SH::STAGES) & 1) ^ 1u, lim, p.status, kWaitHint)))
        break;
      if (issuer) {
        uint8_t* kv = smem + SH::KV_OFF + st * 2 * KV_BYTES;
        ptx::mbar_arrive_expect_tx(&kv_full[st], 2 * KV_BYTES);
        ptx::tma_load_2d(kv, &tmKV, &kv_full[st], H + a * HD, row0 + (j0 + j) * BKV);
        ptx::tma_load_2d(kv + KV_BYTES, &tmKV, &kv_full[st], 2 * H + a * HD, row0 + (j0 + j) * BKV);
      }
      __syncwarp();
      ++issued;
    }
    // drain: bounded waits for the copies still in flight
    ptx::mbar_wait(q_full, 0, lim, p.status, kWaitHint);
    for (int j = issued - 1; j >= 0 && j >= issued - SH::STAGES; --j)
      ptx::mbar_wait(&kv_full[j % SH::STAGES], (j / SH::STAGES) & 1, lim, p.status, kWaitHint);
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issue
    // The whole warp walks the loop and one elected lane issues: a
    // tcgen05.mma takes its descriptors from uniform registers, and built
    // inside one lane's branch they were moved there instruction by
    // instruction, slower than the tensor pipe works on these products.
    constexpr uint32_t idS = ptx::idesc_bf16_f32(BQ, BKV, false, false);
    constexpr uint32_t idO = ptx::idesc_bf16_f32(BQ, HD, false, true);
    const bool issuer = ptx::elect_one();
    const uint64_t dq = ptx::smem_desc_sw128(ptx::smem_u32(smem + SH::Q_OFF), 16, 1024);
    const uint64_t dk0 = ptx::smem_desc_sw128(ptx::smem_u32(smem + SH::KV_OFF), 16, 1024);
    const uint64_t dv0 = ptx::smem_desc_sw128(ptx::smem_u32(smem + SH::KV_OFF + KV_BYTES), 8192, 1024);
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, lim, p.status, kWaitHint));
    };
    bool ok = wait(q_full, 0);
    auto score = [&](int j) {  // S_j into buffer j % NS
      const int st = j % SH::STAGES;
      // K_j, V_j are here, and P_{j - NS}, whose columns S_j takes, has been read
      if (!wait(&kv_full[st], (j / SH::STAGES) & 1)) return false;
      if (j >= NS && !wait(&pv_done[j % NS], (j / NS - 1) & 1)) return false;
      ptx::tc_fence_after();
      if (issuer) {
        const uint64_t dk = dk0 + static_cast<uint64_t>(st * (2 * KV_BYTES >> 4));
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk)
          ptx::tc_mma_f16(tS0 + (j % NS) * 64, dq + kk * 2, dk + kk * 2, idS, kk > 0 ? 1u : 0u);
        ptx::tc_commit(&s_full[j % NS]);
      }
      __syncwarp();
      return true;
    };
    if (NS == 2 && ok && n_kt > 0) ok = score(0);
    for (int j = 0; j < n_kt && ok; ++j) {
      if (NS == 1) ok = score(j);
      else if (j + 1 < n_kt) ok = score(j + 1);  // beside the softmax of tile j
      if (!ok || !wait(&p_full[j % NS], (j / NS) & 1)) { ok = false; break; }
      ptx::tc_fence_after();
      if (issuer) {
        const uint64_t dv = dv0 + static_cast<uint64_t>((j % SH::STAGES) * (2 * KV_BYTES >> 4));
#pragma unroll
        for (int kk = 0; kk < BKV / 16; ++kk)
          ptx::tc_mma_f16_tmem_a(tO, tS0 + (j % NS) * 64 + kk * 8, dv + kk * 128, idO, (j > 0 || kk > 0) ? 1u : 0u);
        ptx::tc_commit(&pv_done[j % NS]);
        ptx::tc_commit(&kv_empty[j % SH::STAGES]);
      }
      __syncwarp();
    }
    if (!ok && issuer) ptx::tc_commit(&pv_done[last % NS]);  // a timeout: what was issued still has to finish
    __syncwarp();
    if (n_kt > 0) ptx::mbar_wait(&pv_done[last % NS], (last / NS) & 1, lim, p.status, kWaitHint);
  } else {
    // --------------------------------------------------- softmax / epilogue
    const int q4 = warp & 3;
    const int r = q4 * 32 + lane;  // query row within the tile == TMEM lane
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    const float sl2 = LOG2E * 0.125f;  // log2(e) / sqrt(64)
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    // every lane waits (bounded); the outcome is made warp-uniform so the
    // warp-collective tcgen05 loads and votes below never see a split warp
    auto wait_all = [&](uint64_t* bar, uint32_t parity) {
      const bool mine = ptx::mbar_wait(bar, parity, lim, p.status, kWaitHint);
      return __all_sync(0xffffffffu, mine);
    };
    // two score buffers: a whole row's scores; one: half of them at a time, registers
    // for four CTAs an SM
    uint32_t vv[32 * NS];
    auto half = [&](int h) -> uint32_t(&)[32] { return *reinterpret_cast<uint32_t(*)[32]>(vv + (NS == 2 ? 32 * h : 0)); };
    for (int j = 0; j < n_kt; ++j) {
      const int left = len - (j0 + j) * BKV;  // valid keys of this tile
      const uint32_t tS = tS0 + (j % NS) * 64;
      auto load_half = [&](int h) { ptx::tmem_ld_32x32b_x32(tS + lane_base + h * 32, half(h)); };
      auto mask_half = [&](int h) {
        uint32_t(&v)[32] = half(h);
        if (left < (h + 1) * 32) {  // CTA-uniform: only the last tile holds masked keys
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (h * 32 + i >= left) v[i] = 0xff800000u;  // -inf: excluded from the max, P = 0
        }
      };
      auto half_max = [&](int h, float mx) {
        const uint32_t(&v)[32] = half(h);
        float m4[4] = {mx, __uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2])};
#pragma unroll
        for (int i = 3; i < 32; ++i) m4[i & 3] = fmaxf(m4[i & 3], __uint_as_float(v[i]));
        return fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      };
      if (!wait_all(&s_full[j % NS], (j / NS) & 1)) { ok = false; break; }
      ptx::tc_fence_after();
      // row max of the raw scores (scaling by log2(e)/sqrt(D) > 0 commutes with
      // max): the high half, then the low half, which stays in registers
      load_half(1);
      if (NS == 2) load_half(0);
      ptx::tmem_ld_wait();
      mask_half(1);
      float mx = half_max(1, -INFINITY);
      if (NS == 1) {
        load_half(0);
        ptx::tmem_ld_wait();
      }
      mask_half(0);
      mx = half_max(0, mx) * sl2;
      if (j == 0) {
        // (a split whose first keys' scores are all -inf adds nothing, as those keys
        // would behind others)
        m = KS > 1 ? fmaxf(mx, -FLT_MAX) : mx;
      } else if (__any_sync(0xffffffffu, mx > m + kRescaleLog2)) {
        // O holds P_{j-1} V_{j-1} (one buffer: S_j was issued behind it)
        if (NS == 2) {
          if (!wait_all(&pv_done[(j - 1) % NS], ((j - 1) / NS) & 1)) { ok = false; break; }
          ptx::tc_fence_after();
        }
        const float m_new = fmaxf(m, mx);
        const float alpha = exp2f(m - m_new);
#pragma unroll
        for (int c = 0; c < HD / 16; ++c) {
          uint32_t o[16];
          ptx::tmem_ld_32x32b_x16(tO + lane_base + c * 16, o);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
          ptx::tmem_st_32x32b_x16(tO + lane_base + c * 16, o);
        }
        l *= alpha;
        m = m_new;
      }
      // P = exp2(s * sl2 - m) as bf16 pairs over the scores: the low half's into
      // the columns it was read from, then the high half's behind it
      const uint64_t nm = pack2(-m, -m), sc = pack2(sl2, sl2);
      uint64_t ls[2] = {0, 0};  // pairs of zeros
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (NS == 1 && h == 1) {
          load_half(1);
          ptx::tmem_ld_wait();
          mask_half(1);
        }
        const uint32_t(&v)[32] = half(h);
        uint32_t pk[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const float2 x = unpack2(fma2(pack2(__uint_as_float(v[2 * u]), __uint_as_float(v[2 * u + 1])), sc, nm));
          const float e0 = ptx::ex2_ftz(x.x), e1 = ptx::ex2_ftz(x.y);
          ls[u & 1] = add2(ls[u & 1], pack2(e0, e1));
          pk[u] = ptx::pack_bf16(e0, e1);
        }
        ptx::tmem_st_32x32b_x16(tS + lane_base + h * 16, pk);
      }
      const float2 lsum = unpack2(add2(ls[0], ls[1]));
      l += lsum.x + lsum.y;
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      ptx::mbar_arrive(&p_full[j % NS]);
    }
    pdl_trigger();  // behind the main loop: see common.cuh
    if constexpr (KS > 1) {
      // partial O (16-byte group g of row r at group g ^ (r & 7)), m and l to shared
      // memory, over the K/V stages, which have been read
      if (n_kt > 0 && ok && wait_all(&pv_done[last % NS], (last / NS) & 1)) {
        ptx::tc_fence_after();
        const uint32_t orow = ptx::smem_u32(smem + SH::KV_OFF) + r * HD * 4;
#pragma unroll
        for (int c = 0; c < HD / 32; ++c) {
          uint32_t(&v)[32] = half(0);
          ptx::tmem_ld_32x32b_x32(tO + lane_base + c * 32, v);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int u = 0; u < 8; ++u)
            ptx::st_shared_v4(orow + (((c * 8 + u) ^ (r & 7)) << 4), v[4 * u], v[4 * u + 1], v[4 * u + 2],
                              v[4 * u + 3]);
        }
      }
      reinterpret_cast<float2*>(smem + SH::ML_OFF)[r] = make_float2(m, l);
    } else {
      // epilogue: O / l -> ctx (bf16) as 128-byte-swizzled rows over the Q
      // tile (the last S product has read it), stored by one TMA that drops the
      // rows past S; the log-sum-exp directly
      if (ok && wait_all(&pv_done[last % NS], (last / NS) & 1)) {
        ptx::tc_fence_after();
        const float inv = 1.f / l;
        const int q = q0 + r;
        const uint32_t orow = ptx::smem_u32(smem + SH::Q_OFF) + r * 128;
#pragma unroll
        for (int c = 0; c < HD / 32; ++c) {
          uint32_t(&v)[32] = half(0);
          ptx::tmem_ld_32x32b_x32(tO + lane_base + c * 32, v);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            uint32_t w[4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
              w[t] = ptx::pack_bf16(__uint_as_float(v[8 * u + 2 * t]) * inv,
                                    __uint_as_float(v[8 * u + 2 * t + 1]) * inv);
            ptx::st_shared_v4(orow + (((c * 4 + u) ^ (r & 7)) << 4), w[0], w[1], w[2], w[3]);
          }
        }
        if (q < S) p.lse[(static_cast<int64_t>(b) * p.A + a) * S + q] = m + log2f(l);
      }
      ptx::fence_proxy_async_smem();  // the staged rows -> the TMA store
      asm volatile("bar.sync 1, 128;" ::: "memory");  // the four softmax warps
      if (warp == 2 && lane == 0) {
        ptx::tma_store_3d(&tmOut, smem + SH::Q_OFF, a * HD, q0, b);
        ptx::bulk_commit_group();
        ptx::bulk_wait_group_read0();  // before the CTA's memory goes
      }
    }
  }
  if constexpr (KS > 1) {
    __syncwarp();
    ptx::cluster_sync();  // every split's part is where it is read from
    if (warp >= 2) {
      // This CTA finishes 128 / KS of the query rows, KS threads a row: the splits'
      // parts in split order, each scaled to the largest m.
      constexpr int ROWS = BQ / KS, G = HD / 4 / KS;
      const int t = static_cast<int>(threadIdx.x) - 64, lr = t / KS, sub = t % KS, row = split * ROWS + lr;
      const uint32_t part = ptx::smem_u32(smem + SH::KV_OFF) + row * HD * 4;
      const uint32_t ml = ptx::smem_u32(smem + SH::ML_OFF) + row * 8;
      float w[KS], mx = -FLT_MAX, l = 0.f;
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        const float2 x = ptx::ld_cluster_f2(ptx::mapa_shared(ml, s));
        const bool any = (s + 1) * n_all / KS > s * n_all / KS;
        w[s] = any ? x.x : -INFINITY;
        mx = fmaxf(mx, w[s]);
      }
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        w[s] = exp2f(w[s] - mx);
        l += w[s] * ptx::ld_cluster_f2(ptx::mapa_shared(ml, s)).y;
      }
      const float inv = 1.f / l;
      const uint32_t orow = ptx::smem_u32(smem + SH::Q_OFF) + lr * 128;
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const int g = sub + KS * i;
        float4 x[KS], o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < KS; ++s) x[s] = ptx::ld_cluster_f4(ptx::mapa_shared(part + ((g ^ (row & 7)) << 4), s));
#pragma unroll
        for (int s = 0; s < KS; ++s) {
          if ((s + 1) * n_all / KS == s * n_all / KS) continue;  // (nothing was written there)
          o.x += w[s] * x[s].x; o.y += w[s] * x[s].y; o.z += w[s] * x[s].z; o.w += w[s] * x[s].w;
        }
        ptx::st_shared_v2(orow + (((g >> 1) ^ (lr & 7)) << 4) + (g & 1) * 8, ptx::pack_bf16(o.x * inv, o.y * inv),
                          ptx::pack_bf16(o.z * inv, o.w * inv));
      }
      const int q = q0 + row;
      if (sub == 0 && q < S) p.lse[(static_cast<int64_t>(b) * p.A + a) * S + q] = mx + log2f(l);
      ptx::fence_proxy_async_smem();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (warp == 2 && lane == 0 && q0 + split * ROWS < S) {
        ptx::tma_store_3d(&tmOut, smem + SH::Q_OFF, a * HD, q0 + split * ROWS, b);
        ptx::bulk_commit_group();
        ptx::bulk_wait_group_read0();
      }
    }
    __syncwarp();
  }
  ptx::tc_fence_before();
  if constexpr (KS > 1) ptx::cluster_sync();  // the peers have read this CTA's part
  else __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, SH::TMEM_COLS);
  }
}

// ----------------------------------------- forward, sequences up to 128
// One 128-key tile: S = Q K^T (N = 128), one softmax pass, O = P V.  P (bf16
// pairs) goes over the scores' first 64 columns as they are consumed, O over the
// rest: 128 TMEM columns and 48 KiB, four CTAs an SM.  Latency-bound: it saves the
// second tile's round trip through the tensor pipe.
constexpr int FS_Q = 0, FS_K = Q_BYTES, FS_V = 2 * Q_BYTES, FS_BAR = 3 * Q_BYTES;
constexpr int FS_SMEM = FS_BAR + 64 + 1024;
constexpr int FS_TMEM_COLS = 128;
static_assert(4 * (FS_SMEM + 1024) <= 233472, "four forward CTAs per SM");

__global__ void __launch_bounds__(NTHR, 4) attn_fwd_short_tc(const __grid_constant__ CUtensorMap tmQKV,
                                                                  const __grid_constant__ CUtensorMap tmOut,
                                                                  const FwdParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint64_t* qk_full = reinterpret_cast<uint64_t*>(smem + FS_BAR);
  uint64_t* v_full = qk_full + 1;
  uint64_t* s_full = v_full + 1;   // S complete
  uint64_t* p_full = s_full + 1;   // P in tensor memory
  uint64_t* o_full = p_full + 1;   // O complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(o_full + 1);

  const int a = blockIdx.x, b = blockIdx.y;
  const int S = p.S, H = p.H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = b * S;
  const uint64_t lim = p.timeout_ns;
  if (threadIdx.x == 0) {
    ptx::mbar_init(qk_full, 1);
    ptx::mbar_init(v_full, 1);
    ptx::mbar_init(s_full, 1);
    ptx::mbar_init(p_full, 128);
    ptx::mbar_init(o_full, 1);
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
    ptx::prefetch_tensormap(&tmQKV);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, FS_TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tS = tmem, tO = tmem + 64;
  pdl_wait();
  int len = p.lens[b];
  if (len < 1 || len > S) {
    if (p.status && threadIdx.x == 0) atomicOr(p.status, kStatusBadLength);
    len = len < 1 ? 1 : S;
  }
  const int chunks = (len + 31) / 32;  // 32-key chunks with a valid key

  if (warp == 0) {
    if (lane == 0) {
      ptx::mbar_arrive_expect_tx(qk_full, 2 * Q_BYTES);
      ptx::tma_load_2d(smem + FS_Q, &tmQKV, qk_full, a * HD, row0);
      ptx::tma_load_2d(smem + FS_K, &tmQKV, qk_full, H + a * HD, row0);
      ptx::mbar_arrive_expect_tx(v_full, Q_BYTES);
      ptx::tma_load_2d(smem + FS_V, &tmQKV, v_full, 2 * H + a * HD, row0);
      // bounded waits for the copies before the CTA may exit
      ptx::mbar_wait(qk_full, 0, lim, p.status, kWaitHint);
      ptx::mbar_wait(v_full, 0, lim, p.status, kWaitHint);
    }
  } else if (warp == 1) {
    // (whole warp, one elected lane issuing: as above)
    constexpr uint32_t idS = ptx::idesc_bf16_f32(BQ, 128, false, false);
    constexpr uint32_t idO = ptx::idesc_bf16_f32(BQ, HD, false, true);
    const bool issuer = ptx::elect_one();
    const uint64_t dq = ptx::smem_desc_sw128(ptx::smem_u32(smem + FS_Q), 16, 1024);
    const uint64_t dk = ptx::smem_desc_sw128(ptx::smem_u32(smem + FS_K), 16, 1024);
    const uint64_t dv = ptx::smem_desc_sw128(ptx::smem_u32(smem + FS_V), 8192, 1024);
    auto wait = [&](uint64_t* bar) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, 0, lim, p.status, kWaitHint));
    };
    bool ok = wait(qk_full);
    if (ok) {
      ptx::tc_fence_after();
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk) ptx::tc_mma_f16(tS, dq + kk * 2, dk + kk * 2, idS, kk > 0 ? 1u : 0u);
        ptx::tc_commit(s_full);
      }
      __syncwarp();
      ok = wait(v_full) && wait(p_full);
    }
    if (ok) {
      ptx::tc_fence_after();
      if (issuer) {
        for (int kk = 0; kk < 2 * chunks; ++kk)
          ptx::tc_mma_f16_tmem_a(tO, tS + kk * 8, dv + kk * 128, idO, kk > 0 ? 1u : 0u);
      }
      __syncwarp();
    }
    // also on a timeout: what was issued has to finish before TMEM is released
    if (issuer) ptx::tc_commit(o_full);
    __syncwarp();
    ptx::mbar_wait(o_full, 0, lim, p.status, kWaitHint);
  } else {
    const int q4 = warp & 3;
    const int r = q4 * 32 + lane;  // query row == TMEM lane
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    const float sl2 = LOG2E * 0.125f;
    auto wait_all = [&](uint64_t* bar) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, 0, lim, p.status, kWaitHint));
    };
    float m = -INFINITY, l = 0.f;
    uint32_t v[32];
    auto load_chunk = [&](int c) {
      ptx::tmem_ld_32x32b_x32(tS + lane_base + c * 32, v);
      ptx::tmem_ld_wait();
      if (len < (c + 1) * 32) {  // CTA-uniform
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (c * 32 + i >= len) v[i] = 0xff800000u;  // -inf: excluded from the max, P = 0
      }
    };
    bool ok = wait_all(s_full);
    if (ok) {
      ptx::tc_fence_after();
      // row max, the first chunk last: it stays in registers
#pragma unroll 1
      for (int c = chunks - 1; c >= 0; --c) {
        load_chunk(c);
        float m4[4] = {m, __uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2])};
#pragma unroll
        for (int i = 3; i < 32; ++i) m4[i & 3] = fmaxf(m4[i & 3], __uint_as_float(v[i]));
        m = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      }
      m *= sl2;
      const uint64_t nm = pack2(-m, -m), sc = pack2(sl2, sl2);
      uint64_t ls[2] = {0, 0};  // pairs of zeros
#pragma unroll 1
      for (int c = 0; c < chunks; ++c) {
        if (c > 0) load_chunk(c);
        uint32_t pk[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const float2 x = unpack2(fma2(pack2(__uint_as_float(v[2 * u]), __uint_as_float(v[2 * u + 1])), sc, nm));
          const float e0 = ptx::ex2_ftz(x.x), e1 = ptx::ex2_ftz(x.y);
          ls[u & 1] = add2(ls[u & 1], pack2(e0, e1));
          pk[u] = ptx::pack_bf16(e0, e1);
        }
        ptx::tmem_st_32x32b_x16(tS + lane_base + c * 16, pk);  // over chunk c / 2, which has been read
      }
      const float2 lsum = unpack2(add2(ls[0], ls[1]));
      l = lsum.x + lsum.y;
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      ptx::mbar_arrive(p_full);
      ok = wait_all(o_full);
    }
    pdl_trigger();  // behind the products: see common.cuh
    // O / l -> ctx as in the kernel above
    if (ok) {
      ptx::tc_fence_after();
      const float inv = 1.f / l;
      const uint32_t orow = ptx::smem_u32(smem + FS_Q) + r * 128;
#pragma unroll
      for (int c = 0; c < HD / 32; ++c) {
        ptx::tmem_ld_32x32b_x32(tO + lane_base + c * 32, v);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t w[4];
#pragma unroll
          for (int t = 0; t < 4; ++t)
            w[t] = ptx::pack_bf16(__uint_as_float(v[8 * u + 2 * t]) * inv,
                                  __uint_as_float(v[8 * u + 2 * t + 1]) * inv);
          ptx::st_shared_v4(orow + (((c * 4 + u) ^ (r & 7)) << 4), w[0], w[1], w[2], w[3]);
        }
      }
      if (r < S) p.lse[(static_cast<int64_t>(b) * p.A + a) * S + r] = m + log2f(l);
    }
    ptx::fence_proxy_async_smem();  // the staged rows -> the TMA store
    asm volatile("bar.sync 1, 128;" ::: "memory");  // the four softmax warps
    if (warp == 2 && lane == 0) {
      ptx::tma_store_3d(&tmOut, smem + FS_Q, a * HD, 0, b);
      ptx::bulk_commit_group();
      ptx::bulk_wait_group_read0();  // before the CTA's memory goes
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, FS_TMEM_COLS);
  }
}

// ----------------------------------------------------------- backward, dQ
// One CTA per 128 query rows of (b, a); per 64-key tile j < len:
//   S = Q K_j^T, dP = dO V_j^T (TMEM); thread = query row:
//   P = exp2(S log2(e)/sqrt(D) - lse2), dS = P (dP - delta) -> TMEM as bf16
//   pairs, the A operand of
//   dQ += dS K_j (TMEM); finally dQ / sqrt(D) -> dQKV[:, Q block].
// Pipelining: the softmax warps release S / dP as soon as they hold them in
// registers (s_free), so S_{j+1} and dP_{j+1} run on the tensor cores while
// dS_j is formed; K / V tiles stream through a 3-stage TMA ring.
constexpr int DQ_STAGES = 3;
constexpr int DQ_QD_BYTES = 2 * Q_BYTES;  // Q and dO tiles (128 x 64 each)
constexpr int DQ_Q_OFF = 0, DQ_DO_OFF = Q_BYTES;
constexpr int DQ_KV_OFF = DQ_QD_BYTES;                           // [DQ_STAGES] x {K, V}
constexpr int DQ_BAR_OFF = DQ_KV_OFF + DQ_STAGES * 2 * KV_BYTES;
constexpr int DQ_SMEM = DQ_BAR_OFF + 256 + 1024;

struct BwdParams {
  int S, H, A;
  const int32_t* lens;
  const float* lse;
  const float* delta;
  const uint4* xtab;  // dK/dV per-query rows: [B*A][2][S] x 16 bytes (attn_delta_bf16)
  __nv_bfloat16* dqkv;
  // optional: column sums of the stored dQKV, one row per 128-row tile of a
  // sequence: colpart[b * ceil(S/128) + tile][3H]
  float* colpart;
  int32_t* status;
  uint64_t timeout_ns;
};

// v[j] of lane l -> after the call, v[0] of lane l holds the sum over the
// warp's 32 lanes of v[l]: a butterfly in which every lane keeps the half of
// its columns given by its lane bit and receives the partner's half (31
// shuffles for 32 columns).
__device__ __forceinline__ void lanes_column_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int k = 16; k >= 1; k >>= 1) {
    const bool upper = (lane & k) != 0;
#pragma unroll
    for (int j = 0; j < k; ++j) {
      const float send = upper ? v[j] : v[j + k];
      const float keep = upper ? v[j + k] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, k);
    }
  }
}
__device__ __forceinline__ float bf16_round(float x) {
  return __bfloat162float(__float2bfloat16_rn(x));
}
// The 8 softmax warps of a backward kernel (256 threads) meet here.
__device__ __forceinline__ void softmax_warps_sync() {
  asm volatile("bar.sync 1, 256;" ::: "memory");
}

__global__ void __maxnreg__(80) attn_bwd_dq_tc(const __grid_constant__ CUtensorMap tmQ,
                                                          const __grid_constant__ CUtensorMap tmKV,
                                                          const __grid_constant__ CUtensorMap tmO,
                                                          const __grid_constant__ CUtensorMap tmOut,
                                                          const BwdParams p) {
  // Launched right behind the dK/dV kernel, which it does not depend on (it
  // writes the other columns of dQKV): it starts once every dK/dV CTA has
  // started -- and so has seen the delta pre-pass complete -- runs beside it,
  // and waits for it only before exiting, so the next kernel, which waits
  // for this one, also sees dK and dV.
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint64_t* qd_full = reinterpret_cast<uint64_t*>(smem + DQ_BAR_OFF);
  uint64_t* kv_full = qd_full + 1;
  uint64_t* kv_empty = kv_full + DQ_STAGES;
  uint64_t* s_full = kv_empty + DQ_STAGES;
  uint64_t* s_free = s_full + 1;
  uint64_t* ds_full = s_free + 1;
  uint64_t* dq_done = ds_full + 1;
  uint64_t* done = dq_done + 1;  // [2], one per issuing warp
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 2);

  const int qt = blockIdx.x, a = blockIdx.y, b = blockIdx.z;
  const int S = p.S, H = p.H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int len = p.lens[b];
  if (len < 1 || len > S) {
    if (p.status && threadIdx.x == 0) atomicOr(p.status, kStatusBadLength);
    len = len < 1 ? 1 : S;
  }
  const int n_kt = (len + BKV - 1) / BKV;
  const int row0 = b * S, q0 = qt * BQ;
  const uint64_t lim = p.timeout_ns;

  if (threadIdx.x == 0) {
    ptx::mbar_init(qd_full, 1);
    for (int s = 0; s < DQ_STAGES; ++s) {
      ptx::mbar_init(&kv_full[s], 1);
      ptx::mbar_init(&kv_empty[s], 2);  // the tile's S / dP products and its dQ product
    }
    ptx::mbar_init(s_full, 1);
    ptx::mbar_init(s_free, NSM_B);
    ptx::mbar_init(ds_full, NSM_B);
    ptx::mbar_init(dq_done, 1);
    ptx::mbar_init(&done[0], 1);
    ptx::mbar_init(&done[1], 1);
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, 256);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // S: [0, 64), dP: [64, 128), dQ: [128, 192), dS as bf16 pairs (the A
  // operand of dS K, read from tensor memory): [192, 224)
  const uint32_t tS = tmem, tdP = tmem + 64, tdQ = tmem + 128, tdS = tmem + 192;

  if (warp == 0) {
    if (lane == 0) {
      ptx::prefetch_tensormap(&tmQ);
      ptx::prefetch_tensormap(&tmO);
      ptx::prefetch_tensormap(&tmKV);
      ptx::mbar_arrive_expect_tx(qd_full, DQ_QD_BYTES);
      ptx::tma_load_2d(smem + DQ_Q_OFF, &tmQ, qd_full, a * HD, row0 + q0);
      ptx::tma_load_2d(smem + DQ_DO_OFF, &tmO, qd_full, a * HD, row0 + q0);
      int issued = 0;
      for (int j = 0; j < n_kt; ++j) {
        const int st = j % DQ_STAGES;
        if (!ptx::mbar_wait(&kv_empty[st], ((j / DQ_STAGES) & 1) ^ 1u, lim, p.status, kWaitHint))
          break;
        uint8_t* kv = smem + DQ_KV_OFF + st * 2 * KV_BYTES;
        ptx::mbar_arrive_expect_tx(&kv_full[st], 2 * KV_BYTES);
        ptx::tma_load_2d(kv, &tmKV, &kv_full[st], H + a * HD, row0 + j * BKV);
        ptx::tma_load_2d(kv + KV_BYTES, &tmKV, &kv_full[st], 2 * H + a * HD, row0 + j * BKV);
        ++issued;
      }
      ptx::mbar_wait(qd_full, 0, lim, p.status, kWaitHint);
      for (int j = issued - 1; j >= 0 && j >= issued - DQ_STAGES; --j)
        ptx::mbar_wait(&kv_full[j % DQ_STAGES], (j / DQ_STAGES) & 1, lim, p.status, kWaitHint);
    }
  } else if (warp == 1) {
    constexpr uint32_t idS = ptx::idesc_bf16_f32(BQ, BKV, false, false);
    const bool issuer = ptx::elect_one();
    const uint64_t dq = ptx::smem_desc_sw128(ptx::smem_u32(smem + DQ_Q_OFF), 16, 1024);
    const uint64_t dd = ptx::smem_desc_sw128(ptx::smem_u32(smem + DQ_DO_OFF), 16, 1024);
    const uint64_t dk0 = ptx::smem_desc_sw128(ptx::smem_u32(smem + DQ_KV_OFF), 16, 1024);
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, lim, p.status, kWaitHint));
    };
    // S_j = Q K_j^T and dP_j = dO V_j^T, as soon as the softmax warps hold
    // S_{j-1} / dP_{j-1} in registers (s_free) and K_j / V_j have landed
    bool ok = wait(qd_full, 0);
    for (int j = 0; j < n_kt && ok; ++j) {
      if (j >= 1 && !wait(s_free, (j - 1) & 1)) break;
      if (!wait(&kv_full[j % DQ_STAGES], (j / DQ_STAGES) & 1)) break;
      ptx::tc_fence_after();
      if (issuer) {
        const uint64_t dk = dk0 + static_cast<uint64_t>((j % DQ_STAGES) * (2 * KV_BYTES >> 4));
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk)
          ptx::tc_mma_f16(tS, dq + kk * 2, dk + kk * 2, idS, kk > 0 ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk)
          ptx::tc_mma_f16(tdP, dd + kk * 2, dk + (KV_BYTES >> 4) + kk * 2, idS, kk > 0 ? 1u : 0u);
        ptx::tc_commit(s_full);
        ptx::tc_commit(&kv_empty[j % DQ_STAGES]);
      }
      __syncwarp();
    }
    if (issuer) ptx::tc_commit(&done[0]);
    __syncwarp();
    ptx::mbar_wait(&done[0], 0, lim, p.status, kWaitHint);
  } else if (warp == 10) {
    // dQ += dS_j K_j, in tile order, from a warp of its own, so that the dQ
    // products and the score products of the next tile go in side by side
    constexpr uint32_t idQ = ptx::idesc_bf16_f32(BQ, HD, false, true);
    const bool issuer = ptx::elect_one();
    const uint64_t dk0 = ptx::smem_desc_sw128(ptx::smem_u32(smem + DQ_KV_OFF), 8192, 1024);
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, lim, p.status, kWaitHint));
    };
    for (int j = 0; j < n_kt; ++j) {
      if (!wait(ds_full, j & 1)) break;
      if (!wait(&kv_full[j % DQ_STAGES], (j / DQ_STAGES) & 1)) break;
      ptx::tc_fence_after();
      if (issuer) {
        const uint64_t dk = dk0 + static_cast<uint64_t>((j % DQ_STAGES) * (2 * KV_BYTES >> 4));
#pragma unroll
        for (int kk = 0; kk < BKV / 16; ++kk)
          ptx::tc_mma_f16_tmem_a(tdQ, tdS + kk * 8, dk + kk * 128, idQ, (j > 0 || kk > 0) ? 1u : 0u);
        ptx::tc_commit(dq_done);
        ptx::tc_commit(&kv_empty[j % DQ_STAGES]);
      }
      __syncwarp();
    }
    if (issuer) ptx::tc_commit(&done[1]);
    __syncwarp();
    ptx::mbar_wait(&done[1], 0, lim, p.status, kWaitHint);
  } else {
    const int q4 = warp & 3;
    const int hf = (warp - 2) >> 2;  // column half: keys [32 hf, 32 hf + 32) of a tile
    const int r = q4 * 32 + lane;
    const int q = q0 + r;
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    const float sl2 = LOG2E * 0.125f;
    const int64_t sidx = (static_cast<int64_t>(b) * p.A + a) * S + (q < S ? q : 0);
    const float nlse2 = q < S ? -p.lse[sidx] : -INFINITY;  // P = 0 on rows past S
    const float dl = q < S ? p.delta[sidx] : 0.f;
    const uint64_t sc2 = pack2(sl2, sl2), nlse = pack2(nlse2, nlse2), ndl = pack2(-dl, -dl);
    bool ok = true;
    auto wait_all = [&](uint64_t* bar, uint32_t parity) {
      const bool mine = ptx::mbar_wait(bar, parity, lim, p.status, kWaitHint);
      return __all_sync(0xffffffffu, mine);
    };
    for (int j = 0; j < n_kt; ++j) {
      if (!wait_all(s_full, j & 1)) { ok = false; break; }
      ptx::tc_fence_after();
      uint32_t sv[32], dv[32];
      ptx::tmem_ld_32x32b_x32(tS + lane_base + hf * 32, sv);
      ptx::tmem_ld_32x32b_x32(tdP + lane_base + hf * 32, dv);
      ptx::tmem_ld_wait();
      ptx::tc_fence_before();
      ptx::mbar_arrive(s_free);
      const int kbase = j * BKV + hf * 32;
      uint32_t pk[16];
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const float2 x = unpack2(fma2(pack2(__uint_as_float(sv[i]), __uint_as_float(sv[i + 1])), sc2, nlse));
        const uint64_t pr = pack2(ptx::ex2_ftz(x.x), ptx::ex2_ftz(x.y));
        const float2 ds = unpack2(mul2(pr, add2(pack2(__uint_as_float(dv[i]), __uint_as_float(dv[i + 1])), ndl)));
        pk[i >> 1] = ptx::pack_bf16(ds.x, ds.y);
      }
      if (kbase + 32 > len) {  // warp-uniform: only the last tile holds masked keys
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const uint32_t lo = kbase + i < len ? 0x0000ffffu : 0u;
          const uint32_t hi = kbase + i + 1 < len ? 0xffff0000u : 0u;
          pk[i >> 1] &= lo | hi;
        }
      }
      // the dS buffer was last read by the dQ product of tile j - 1
      if (j >= 1 && !wait_all(dq_done, (j - 1) & 1)) { ok = false; break; }
      {  // this half's 32 keys = 16 columns of the row's lane
        uint32_t (&p0)[16] = *reinterpret_cast<uint32_t(*)[16]>(&pk[0]);
        ptx::tmem_st_32x32b_x16(tdS + hf * 16 + lane_base, p0);
      }
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      ptx::mbar_arrive(ds_full);
    }
    pdl_trigger();
    // epilogue: each half stages 32 of the 64 dQ columns as 128-byte-swizzled
    // bf16 rows over the Q tile (the last S product has read it); one thread
    // then stores the tile by TMA, which drops the rows past S
    float* red = reinterpret_cast<float*>(smem + DQ_KV_OFF);  // [4 row quarters][64]: ring is idle
    if (ok && wait_all(dq_done, (n_kt - 1) & 1)) {
      ptx::tc_fence_after();
      const uint32_t orow = ptx::smem_u32(smem + DQ_Q_OFF) + r * 128;
      uint32_t o[32];
      ptx::tmem_ld_32x32b_x32(tdQ + lane_base + hf * 32, o);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        uint32_t w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t)
          w[t] = ptx::pack_bf16(__uint_as_float(o[8 * u + 2 * t]) * 0.125f,
                                __uint_as_float(o[8 * u + 2 * t + 1]) * 0.125f);
        ptx::st_shared_v4(orow + (((hf * 4 + u) ^ (r & 7)) << 4), w[0], w[1], w[2], w[3]);
      }
      if (p.colpart) {  // column sums of the stored values over this warp's 32 rows
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = q < S ? bf16_round(__uint_as_float(o[j]) * 0.125f) : 0.f;
        lanes_column_sum(v, lane);
        red[q4 * 64 + hf * 32 + lane] = v[0];
      }
    } else if (p.colpart) {
      red[q4 * 64 + hf * 32 + lane] = 0.f;
    }
    ptx::fence_proxy_async_smem();  // the staged rows -> the TMA store
    softmax_warps_sync();
    if (warp == 2 && lane == 0) {
      ptx::tma_store_3d(&tmOut, smem + DQ_Q_OFF, a * HD, q0, b);
      ptx::bulk_commit_group();
    }
    if (p.colpart && q4 == 0) {  // the four row quarters, added in order, by the quarter-0 warps
      const int c = hf * 32 + lane;
      const float sum = ((red[c] + red[64 + c]) + red[128 + c]) + red[192 + c];
      p.colpart[(static_cast<int64_t>(b) * gridDim.x + qt) * (3 * H) + a * HD + c] = sum;
    }
    if (warp == 2 && lane == 0) ptx::bulk_wait_group_read0();  // before the CTA's memory goes
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, 256);
  }
  pdl_wait();
}

// --------------------------------------------------------- backward, dK dV
// One CTA per 128 keys of (b, a) (tiles at or past len[b] only write zeros);
// per 64-query tile i over all S queries:
//   S^T = K Q_i^T, dP^T = V dO_i^T (TMEM); thread = key row:
//   P^T = exp2(S^T log2(e)/sqrt(D) - lse2_q), dS^T = P^T (dP^T - delta_q),
//   written back to TMEM over the S^T / dP^T columns they came from;
//   dV += P^T dO_i, dK += dS^T Q_i with P^T, dS^T as TMEM A operands;
//   finally dK / sqrt(D), dV -> dQKV.
// Keeping P^T and dS^T in TMEM takes their 32 KiB of shared-memory stores and
// the accumulating products' 32 KiB of A-operand reads off the shared-memory
// port per tile, which the score products' operand reads otherwise saturate.
// The price is order within a CTA: S^T_{i+1} waits until dV_i has read P^T_i
// (and dP^T_{i+1} until dK_i has read dS^T_i), so the two CTAs on an SM take
// turns on the tensor pipe rather than one CTA overlapping itself.
// The Q_i / dO_i tiles serve both as K-major operands (S^T, dP^T) and as
// MN-major operands (dK, dV).
constexpr int BK2 = 128, BQ2 = 64;
constexpr int KV2_BYTES = BK2 * HD * 2;    // 16 KiB (K or V of 128 keys)
constexpr int QO2_BYTES = BQ2 * HD * 2;    // 8 KiB  (Q or dO of 64 queries)
constexpr int KV_STAGES = 3;               // Q / dO ring
constexpr int KV_K_OFF = 0, KV_V_OFF = KV2_BYTES;
constexpr int KV_Q_OFF = 2 * KV2_BYTES;
constexpr int KV_O_OFF = KV_Q_OFF + KV_STAGES * QO2_BYTES;
// The per-query terms enter the score products as one more K = 16 step:
// S^T - lse2 / c = [K | E] [Q | X_lse]^T and dP^T - delta = [V | E] [dO | X_delta]^T,
// with c = log2(e)/sqrt(D), E the 128 x 16 matrix whose first two columns are
// ones, and X the 64 x 16 per-tile matrix whose first two columns hold the
// negated term split into a bf16 high part and a bf16 low part (exact to
// about 2^-17 relative).  The softmax threads then need no per-query loads.
// E and X are K-major without swizzling, built from 8-row x 16-byte core
// matrices: a row's K columns 0..7 are 16 contiguous bytes (row groups 128
// bytes apart), and columns 8..15, all zero, come from one shared zero block
// (the descriptors' K-direction offset points there).  So an X tile is 64
// rows of 16 bytes, one bulk copy of the table the delta pre-pass writes.
constexpr int XROW_BYTES = 16;
constexpr int X_BYTES = BQ2 * XROW_BYTES;                      // 1 KiB: X of one product
constexpr int KV_E_OFF = KV_O_OFF + KV_STAGES * QO2_BYTES;     // E: 2 KiB
constexpr int KV_X_OFF = KV_E_OFF + BK2 * XROW_BYTES;          // [KV_STAGES][2 products] X
constexpr int KV_Z_OFF = KV_X_OFF + KV_STAGES * 2 * X_BYTES;   // zeros: 2 KiB
constexpr int KV_RED_OFF = KV_Z_OFF + BK2 * XROW_BYTES;  // [2 halves][4 quarters][64] floats
constexpr int KV_BAR_OFF = KV_RED_OFF + 2 * 4 * 64 * 4;
// 91 KiB: more than a third of the SM's shared memory, so at most two CTAs
// share an SM, as their 256 TMEM columns each require.
constexpr int KV_SMEM = KV_BAR_OFF + 128 + 1024;
static_assert(3 * (KV_SMEM + 1024) > 233472 && 2 * (KV_SMEM + 1024) <= 233472,
              "exactly two dK/dV CTAs per SM");

__global__ void __maxnreg__(80) attn_bwd_dkdv_tc(const __grid_constant__ CUtensorMap tmK,
                                                            const __grid_constant__ CUtensorMap tmQ,
                                                            const __grid_constant__ CUtensorMap tmO,
                                                            const __grid_constant__ CUtensorMap tmOut,
                                                            const BwdParams p) {
  // wait first, then let the dQ kernel start: once every CTA here has passed
  // the wait, the delta pre-pass (and everything before it) is complete
  pdl_wait();
  pdl_trigger();
  extern __shared__ uint8_t smem_raw[];
  const int kt = blockIdx.x, a = blockIdx.y, b = blockIdx.z;
  const int S = p.S, H = p.H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int len = p.lens[b];
  if (len < 1 || len > S) {
    if (p.status && threadIdx.x == 0) atomicOr(p.status, kStatusBadLength);
    len = len < 1 ? 1 : S;
  }
  const int row0 = b * S, k0 = kt * BK2;
  const int64_t rs = 3 * static_cast<int64_t>(H);
  if (k0 >= len) {  // keys of this tile are all padding: zero gradients
    for (int i = threadIdx.x; i < BK2 * 8; i += NTHR_B) {
      const int rr = i >> 3, c = i & 7;
      if (k0 + rr < S) {
        __nv_bfloat16* base = p.dqkv + (static_cast<int64_t>(row0) + k0 + rr) * rs + a * HD + c * 8;
        *reinterpret_cast<uint4*>(base + H) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(base + 2 * H) = make_uint4(0, 0, 0, 0);
      }
    }
    if (p.colpart && threadIdx.x < 2 * HD) {  // and zero column sums
      const int hf = threadIdx.x / HD, c = threadIdx.x % HD;
      p.colpart[(static_cast<int64_t>(b) * gridDim.x + kt) * rs + (1 + hf) * H + a * HD + c] = 0.f;
    }
    return;
  }
  const uint32_t raw_addr = ptx::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint64_t* kv_full = reinterpret_cast<uint64_t*>(smem + KV_BAR_OFF);
  uint64_t* q_full = kv_full + 1;
  uint64_t* q_empty = q_full + KV_STAGES;
  uint64_t* st_full = q_empty + KV_STAGES;  // S^T_i complete
  uint64_t* dpt_full = st_full + 1;         // dP^T_i complete
  uint64_t* pds_full = dpt_full + 1;        // P^T_i, dS^T_i stored to TMEM
  uint64_t* dv_done = pds_full + 1;         // dV += P^T_i dO_i complete: S^T columns free
  uint64_t* dk_done = dv_done + 1;          // dK += dS^T_i Q_i complete: dP^T columns free
  uint64_t* done = dk_done + 1;             // [2], one per issuing warp
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 2);
  const int n_qt = (S + BQ2 - 1) / BQ2;
  const uint64_t lim = p.timeout_ns;

  if (threadIdx.x == 0) {
    ptx::mbar_init(kv_full, 1);
    for (int s = 0; s < KV_STAGES; ++s) {
      ptx::mbar_init(&q_full[s], 1);  // lane 0's expect_tx (Q_i, dO_i, both X)
      ptx::mbar_init(&q_empty[s], 2);  // the tile's dV and dK products (each after its score product)
    }
    ptx::mbar_init(st_full, 1);
    ptx::mbar_init(dpt_full, 1);
    ptx::mbar_init(pds_full, NSM_B);
    ptx::mbar_init(dv_done, 1);
    ptx::mbar_init(dk_done, 1);
    ptx::mbar_init(&done[0], 1);
    ptx::mbar_init(&done[1], 1);
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, 256);
    ptx::tmem_relinquish();
  }
  // E: rows [1, 1, 0 x 6] (bf16); the X ring and the zero block: zeros
  for (int w = threadIdx.x; w < (KV_RED_OFF - KV_E_OFF) / 16; w += NTHR_B)
    *reinterpret_cast<uint4*>(smem + KV_E_OFF + w * 16) =
        make_uint4(w < BK2 ? 0x3F803F80u : 0u, 0u, 0u, 0u);
  ptx::fence_proxy_async_smem();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // S^T (then P^T, bf16 pairs), dP^T (then dS^T), dV, dK accumulators.  The
  // column half hf of S^T (queries 32 hf ..) holds that half's P^T in its
  // first 16 columns, so the two halves never write columns the other reads.
  const uint32_t tST = tmem, tdPT = tmem + 64, tdV = tmem + 128, tdK = tmem + 192;

  if (warp == 0) {
    // producer: K, V once; per query tile Q_i, dO_i by TMA and the tile's
    // two X matrices by bulk copy, all completing on q_full
    if (lane == 0) {
      ptx::prefetch_tensormap(&tmK);
      ptx::prefetch_tensormap(&tmQ);
      ptx::prefetch_tensormap(&tmO);
      ptx::mbar_arrive_expect_tx(kv_full, 2 * KV2_BYTES);
      ptx::tma_load_2d(smem + KV_K_OFF, &tmK, kv_full, H + a * HD, row0 + k0);
      ptx::tma_load_2d(smem + KV_V_OFF, &tmK, kv_full, 2 * H + a * HD, row0 + k0);
    }
    // this (sequence, head)'s X_lse rows, followed by its X_delta rows
    const uint4* xs_b = p.xtab + (static_cast<int64_t>(b) * p.A + a) * 2 * S;
    int issued = 0;
    for (int i = 0; i < n_qt && lane == 0; ++i) {
      const int st = i % KV_STAGES;
      if (!ptx::mbar_wait(&q_empty[st], ((i / KV_STAGES) & 1) ^ 1u, lim, p.status, kWaitHint)) break;
      const uint32_t xbytes = static_cast<uint32_t>(min(BQ2, S - i * BQ2)) * XROW_BYTES;
      ptx::mbar_arrive_expect_tx(&q_full[st], 2 * QO2_BYTES + 2 * xbytes);
      ptx::tma_load_2d(smem + KV_Q_OFF + st * QO2_BYTES, &tmQ, &q_full[st], a * HD, row0 + i * BQ2);
      ptx::tma_load_2d(smem + KV_O_OFF + st * QO2_BYTES, &tmO, &q_full[st], a * HD, row0 + i * BQ2);
      uint8_t* x = smem + KV_X_OFF + st * 2 * X_BYTES;
      ptx::bulk_load(x, xs_b + i * BQ2, xbytes, &q_full[st]);
      ptx::bulk_load(x + X_BYTES, xs_b + S + i * BQ2, xbytes, &q_full[st]);
      ++issued;
    }
    if (lane == 0) {
      ptx::mbar_wait(kv_full, 0, lim, p.status, kWaitHint);
      for (int i = issued - 1; i >= 0 && i >= issued - KV_STAGES; --i)
        ptx::mbar_wait(&q_full[i % KV_STAGES], (i / KV_STAGES) & 1, lim, p.status, kWaitHint);
    }
  } else if (warp == 1 || warp == 10) {
    // Warp 1: S^T_i = K Q_i^T, then dV += P^T_i dO_i.  Warp 10: dP^T_i =
    // V dO_i^T, then dK += dS^T_i Q_i.  Each warp's score product of tile i
    // goes in once its accumulating product of tile i - 1 has read the
    // columns it overwrites; the accumulating product once the softmax warps
    // have stored P^T_i / dS^T_i.
    // (whole warp in the loop, one elected lane issuing: as in the forward)
    const bool v_side = warp == 1;
    const bool issuer = ptx::elect_one();
    constexpr uint32_t idS = ptx::idesc_bf16_f32(BK2, BQ2, false, false);
    constexpr uint32_t idG = ptx::idesc_bf16_f32(BK2, HD, false, true);
    const uint32_t tscore = v_side ? tST : tdPT, tacc = v_side ? tdV : tdK;
    uint64_t* score_full = v_side ? st_full : dpt_full;
    uint64_t* acc_done = v_side ? dv_done : dk_done;
    // K-major operand of the score product (Q_i or dO_i) and MN-major
    // operand of the accumulating product (dO_i or Q_i)
    const int score_off = v_side ? KV_Q_OFF : KV_O_OFF, acc_off = v_side ? KV_O_OFF : KV_Q_OFF;
    const uint64_t dkv = ptx::smem_desc_sw128(ptx::smem_u32(smem + (v_side ? KV_K_OFF : KV_V_OFF)), 16, 1024);
    const uint64_t dsc = ptx::smem_desc_sw128(ptx::smem_u32(smem + score_off), 16, 1024);
    const uint64_t dac = ptx::smem_desc_sw128(ptx::smem_u32(smem + acc_off), 8192, 1024);
    const uint32_t se = ptx::smem_u32(smem + KV_E_OFF), sz = ptx::smem_u32(smem + KV_Z_OFF);
    const uint32_t sx = ptx::smem_u32(smem + KV_X_OFF + (v_side ? 0 : X_BYTES));
    const uint64_t de = ptx::smem_desc_noswizzle(se, sz - se, 128);
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, parity, lim, p.status, kWaitHint));
    };
    bool ok = wait(kv_full, 0);
    for (int i = 0; i < n_qt && ok; ++i) {
      const int st = i % KV_STAGES;
      if (i >= 1 && !wait(acc_done, (i - 1) & 1)) break;
      if (!wait(&q_full[st], (i / KV_STAGES) & 1)) break;
      ptx::tc_fence_after();
      const uint64_t soff = static_cast<uint64_t>(st * (QO2_BYTES >> 4));
      if (issuer) {
        const uint32_t sxs = sx + st * 2 * X_BYTES;
        const uint64_t dx = ptx::smem_desc_noswizzle(sxs, sz - sxs, 128);
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk)
          ptx::tc_mma_f16(tscore, dkv + kk * 2, dsc + soff + kk * 2, idS, kk > 0 ? 1u : 0u);
        ptx::tc_mma_f16(tscore, de, dx, idS, 1u);  // the per-query term: E X^T
        ptx::tc_commit(score_full);
      }
      __syncwarp();
      if (!wait(pds_full, i & 1)) break;
      ptx::tc_fence_after();
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < BQ2 / 16; ++kk)  // queries 16 kk ..: half kk / 2, packed column 8 (kk % 2)
          ptx::tc_mma_f16_tmem_a(tacc, tscore + (kk >> 1) * 32 + (kk & 1) * 8, dac + soff + kk * 128, idG,
                                 (i > 0 || kk > 0) ? 1u : 0u);
        ptx::tc_commit(acc_done);
        ptx::tc_commit(&q_empty[st]);
      }
      __syncwarp();
    }
    uint64_t* fin = &done[v_side ? 0 : 1];
    if (issuer) ptx::tc_commit(fin);
    __syncwarp();
    ptx::mbar_wait(fin, 0, lim, p.status, kWaitHint);
  } else {
    const int q4 = warp & 3;
    const int hf = (warp - 2) >> 2;  // column half: queries [32 hf, 32 hf + 32) of a tile
    const int r = q4 * 32 + lane;    // key row within the tile == TMEM lane
    const int key = k0 + r;
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    const float sl2 = LOG2E * 0.125f;
    const uint64_t sc2 = pack2(sl2, sl2);
    bool ok = true;
    auto wait_all = [&](uint64_t* bar, uint32_t parity) {
      const bool mine = ptx::mbar_wait(bar, parity, lim, p.status, kWaitHint);
      return __all_sync(0xffffffffu, mine);
    };
    for (int i = 0; i < n_qt; ++i) {
      if (!wait_all(st_full, i & 1) || !wait_all(dpt_full, i & 1)) { ok = false; break; }
      ptx::tc_fence_after();
      uint32_t sv[32], dv[32];
      ptx::tmem_ld_32x32b_x32(tST + lane_base + hf * 32, sv);
      ptx::tmem_ld_32x32b_x32(tdPT + lane_base + hf * 32, dv);
      ptx::tmem_ld_wait();
      // sv = S^T - lse2 / c and dv = dP^T - delta, the terms added by the MMAs
      uint32_t pp[16], dd[16];
#pragma unroll
      for (int t = 0; t < 32; t += 2) {
        // (a key past the valid length gets a row of its own, which the epilogue drops)
        const float2 x = unpack2(mul2(pack2(__uint_as_float(sv[t]), __uint_as_float(sv[t + 1])), sc2));
        const float2 pt = make_float2(ptx::ex2_ftz(x.x), ptx::ex2_ftz(x.y));
        const float2 ds = unpack2(mul2(pack2(pt.x, pt.y), pack2(__uint_as_float(dv[t]), __uint_as_float(dv[t + 1]))));
        pp[t >> 1] = ptx::pack_bf16(pt.x, pt.y);
        dd[t >> 1] = ptx::pack_bf16(ds.x, ds.y);
      }
      const int nq = S - i * BQ2 - hf * 32;  // queries of this half inside the sequence
      if (nq < 32) {  // warp-uniform: queries past S
#pragma unroll
        for (int t = 0; t < 32; t += 2) {
          const uint32_t keep = (t < nq ? 0x0000ffffu : 0u) | (t + 1 < nq ? 0xffff0000u : 0u);
          pp[t >> 1] &= keep;
          dd[t >> 1] &= keep;
        }
      }
      // over the columns this thread has just read: P^T_i, dS^T_i as bf16 pairs
      ptx::tmem_st_32x32b_x16(tST + lane_base + hf * 32, pp);
      ptx::tmem_st_32x32b_x16(tdPT + lane_base + hf * 32, dd);
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      ptx::mbar_arrive(pds_full);
    }
    // epilogue: the low-half warps stage dK / sqrt(D), the high-half warps dV,
    // as 128-byte-swizzled bf16 rows over the K / V tiles (the last score
    // products have read them); one thread then stores both tiles by TMA
    // through a [B][S][3H] map, which drops the rows past S.
    float* red = reinterpret_cast<float*>(smem + KV_RED_OFF);  // [2 halves][4 quarters][64]
    if (ok && wait_all(dv_done, (n_qt - 1) & 1) && wait_all(dk_done, (n_qt - 1) & 1)) {
      ptx::tc_fence_after();
      const uint32_t tacc = hf == 0 ? tdK : tdV;
      const float sc = hf == 0 ? 0.125f : 1.f;
      const uint32_t orow = ptx::smem_u32(smem + (hf == 0 ? KV_K_OFF : KV_V_OFF)) + r * 128;
      uint32_t o[2][32];
      ptx::tmem_ld_32x32b_x32(tacc + lane_base, o[0]);
      ptx::tmem_ld_32x32b_x32(tacc + lane_base + 32, o[1]);
      ptx::tmem_ld_wait();
      if (k0 + q4 * 32 + 32 > len) {  // warp-uniform: rows of keys past the valid length are zero
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int j = 0; j < 32; ++j) o[c][j] = key < len ? o[c][j] : 0u;
      }
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t w[4];
#pragma unroll
          for (int t = 0; t < 4; ++t)
            w[t] = ptx::pack_bf16(__uint_as_float(o[c][8 * u + 2 * t]) * sc,
                                  __uint_as_float(o[c][8 * u + 2 * t + 1]) * sc);
          ptx::st_shared_v4(orow + (((c * 4 + u) ^ (r & 7)) << 4), w[0], w[1], w[2], w[3]);
        }
      if (p.colpart) {  // column sums of the stored values over this warp's 32 rows
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float v[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = key < S ? bf16_round(__uint_as_float(o[c][j]) * sc) : 0.f;
          lanes_column_sum(v, lane);
          red[(hf * 4 + q4) * 64 + c * 32 + lane] = v[0];
        }
      }
    } else if (p.colpart) {
      red[(hf * 4 + q4) * 64 + lane] = 0.f;
      red[(hf * 4 + q4) * 64 + 32 + lane] = 0.f;
    }
    ptx::fence_proxy_async_smem();  // the staged rows -> the TMA store
    softmax_warps_sync();
    if (warp == 2 && lane == 0) {
      ptx::tma_store_3d(&tmOut, smem + KV_K_OFF, H + a * HD, k0, b);
      ptx::tma_store_3d(&tmOut, smem + KV_V_OFF, 2 * H + a * HD, k0, b);
      ptx::bulk_commit_group();
    }
    if (p.colpart && q4 == 0) {  // the four row quarters, added in order, by the quarter-0 warps
      const float* rh = red + hf * 4 * 64;
      float* dst = p.colpart + (static_cast<int64_t>(b) * gridDim.x + kt) * rs + (1 + hf) * H + a * HD;
#pragma unroll
      for (int c = lane; c < 64; c += 32)
        dst[c] = ((rh[c] + rh[64 + c]) + rh[128 + c]) + rh[192 + c];
    }
    if (warp == 2 && lane == 0) ptx::bulk_wait_group_read0();  // before the CTA's memory goes
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, 256);
  }
}

// ------------------------------------------- backward, sequences up to 128
// One CTA per (b, a): its 128-row tile holds every query and every key, so the
// scores, P and dS are formed once and all three gradients follow from them:
//   S = Q K^T, dP = dO V^T (M = N = 128, K = 64); thread = query row:
//   P = exp2(S log2(e)/sqrt(D) - lse2), dS = P (dP - delta), delta from the row's
//   dO and O, both as bf16 into shared memory, 128-byte-swizzled, where they are
//   read as they lie (dS K) and transposed (P^T dO, dS^T Q):
//   dV = P^T dO, dK = dS^T Q / sqrt(D), dQ = dS K / sqrt(D)  (M = 128, N = 64, K = 128).
// The dK/dV and dQ kernels above form P and dS twice, from tables of a delta
// pre-pass; at one tile a sequence each of the three is mostly prologue and
// tail.  Bound by that chain's latency: load, two products, softmax, three
// products, store.  Two CTAs share an SM, one's waits under the other's work
// (112 KiB of tiles and 256 TMEM columns each: the gradients go over the scores).
constexpr int SH_Q = 0, SH_K = Q_BYTES, SH_O = 2 * Q_BYTES, SH_V = 3 * Q_BYTES;
// P: two 64-key chunks of 128 rows, the first over V; dS: two more
constexpr int SH_P = SH_V, SH_DS = SH_P + 2 * Q_BYTES, SH_BAR = SH_DS + 2 * Q_BYTES;
constexpr int SH_SMEM = SH_BAR + 128;
constexpr int SH_THR = 320;  // warp 0 TMA, warp 1 MMA issue, warps 2..9 softmax
static_assert(2 * (SH_SMEM + 1024) <= 233472, "two CTAs per SM");

__global__ void __launch_bounds__(SH_THR, 2) attn_bwd_short_tc(const __grid_constant__ CUtensorMap tmQKV,
                                                               const __grid_constant__ CUtensorMap tmO,
                                                               const __grid_constant__ CUtensorMap tmC,
                                                               const __grid_constant__ CUtensorMap tmOut,
                                                               const BwdParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* qk_full = reinterpret_cast<uint64_t*>(smem + SH_BAR);
  uint64_t* ov_full = qk_full + 1;
  uint64_t* sc_full = ov_full + 1;   // S and dP complete
  uint64_t* pds_full = sc_full + 1;  // P and dS in shared memory
  uint64_t* g_full = pds_full + 1;   // dV, dK, dQ complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(g_full + 1);

  const int a = blockIdx.x, b = blockIdx.y;
  const int S = p.S, H = p.H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = b * S;
  const uint64_t lim = p.timeout_ns;
  if (threadIdx.x == 0) {
    ptx::mbar_init(qk_full, 1);
    ptx::mbar_init(ov_full, 1);
    ptx::mbar_init(sc_full, 1);
    ptx::mbar_init(pds_full, NSM_B);
    ptx::mbar_init(g_full, 1);
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
    ptx::prefetch_tensormap(&tmQKV);
    ptx::prefetch_tensormap(&tmO);
    ptx::prefetch_tensormap(&tmC);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, 256);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tS = tmem, tdP = tmem + 128;                      // 128 columns each
  const uint32_t tdV = tmem, tdK = tmem + 64, tdQ = tmem + 128;    // over them, 64 each
  pdl_wait();
  int len = p.lens[b];
  if (len < 1 || len > S) {
    if (p.status && threadIdx.x == 0) atomicOr(p.status, kStatusBadLength);
    len = len < 1 ? 1 : S;
  }

  if (warp == 0) {
    if (lane == 0) {
      ptx::mbar_arrive_expect_tx(qk_full, 2 * Q_BYTES);
      ptx::tma_load_2d(smem + SH_Q, &tmQKV, qk_full, a * HD, row0);
      ptx::tma_load_2d(smem + SH_K, &tmQKV, qk_full, H + a * HD, row0);
      ptx::mbar_arrive_expect_tx(ov_full, 3 * Q_BYTES);
      ptx::tma_load_2d(smem + SH_O, &tmO, ov_full, a * HD, row0);
      ptx::tma_load_2d(smem + SH_DS, &tmC, ov_full, a * HD, row0);  // ctx, until dS is formed
      ptx::tma_load_2d(smem + SH_V, &tmQKV, ov_full, 2 * H + a * HD, row0);
      // bounded waits for the copies before the CTA may exit
      ptx::mbar_wait(qk_full, 0, lim, p.status, kWaitHint);
      ptx::mbar_wait(ov_full, 0, lim, p.status, kWaitHint);
    }
  } else if (warp == 1) {
    // (whole warp, one elected lane issuing: as in the forward)
    constexpr uint32_t idS = ptx::idesc_bf16_f32(128, 128, false, false);
    constexpr uint32_t idT = ptx::idesc_bf16_f32(128, HD, true, true);   // P^T dO, dS^T Q
    constexpr uint32_t idN = ptx::idesc_bf16_f32(128, HD, false, true);  // dS K
    const bool issuer = ptx::elect_one();
    const uint32_t s0 = ptx::smem_u32(smem);
    auto kmaj = [&](int off) { return ptx::smem_desc_sw128(s0 + off, 16, 1024); };
    auto mnmaj = [&](int off) { return ptx::smem_desc_sw128(s0 + off, Q_BYTES, 1024); };
    auto wait = [&](uint64_t* bar) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, 0, lim, p.status, kWaitHint));
    };
    const uint64_t dq = kmaj(SH_Q), dk = kmaj(SH_K), dO = kmaj(SH_O), dv = kmaj(SH_V);
    bool ok = wait(qk_full);
    if (ok) {
      ptx::tc_fence_after();
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk) ptx::tc_mma_f16(tS, dq + kk * 2, dk + kk * 2, idS, kk > 0 ? 1u : 0u);
      }
      __syncwarp();
      ok = wait(ov_full);
    }
    if (ok) {
      ptx::tc_fence_after();
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk) ptx::tc_mma_f16(tdP, dO + kk * 2, dv + kk * 2, idS, kk > 0 ? 1u : 0u);
        ptx::tc_commit(sc_full);
      }
      __syncwarp();
      ok = wait(pds_full);
    }
    if (ok) {
      ptx::tc_fence_after();
      const uint64_t pt = mnmaj(SH_P), dst = mnmaj(SH_DS), ds = kmaj(SH_DS);
      const uint64_t bo = mnmaj(SH_O), bq = mnmaj(SH_Q), bk = mnmaj(SH_K);
      // Only the 16-row blocks that hold a query (of dO and Q) or a valid key (of K):
      // the rows behind are other sequences' or padding, and a zero of P or dS
      // times an infinity or NaN there would reach this sequence's gradients.
      const int nq = (S + 15) / 16, nk = (len + 15) / 16;
      if (issuer) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          if (kk < nq) ptx::tc_mma_f16(tdV, pt + kk * 128, bo + kk * 128, idT, kk > 0 ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          if (kk < nq) ptx::tc_mma_f16(tdK, dst + kk * 128, bq + kk * 128, idT, kk > 0 ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)  // keys 16 kk ..: chunk kk / 4
          if (kk < nk)
            ptx::tc_mma_f16(tdQ, ds + (kk >> 2) * (Q_BYTES >> 4) + (kk & 3) * 2, bk + kk * 128, idN, kk > 0 ? 1u : 0u);
      }
      __syncwarp();
    }
    // also on a timeout: what was issued has to finish before TMEM is released
    if (issuer) ptx::tc_commit(g_full);
    __syncwarp();
    ptx::mbar_wait(g_full, 0, lim, p.status, kWaitHint);
  } else {
    const int q4 = warp & 3, hf = (warp - 2) >> 2;  // keys [64 hf, 64 hf + 64) of the row
    const int r = q4 * 32 + lane;                   // query row = TMEM lane
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    const float sl2 = LOG2E * 0.125f;
    const bool live = r < S;
    const float nlse2 = live ? -p.lse[(static_cast<int64_t>(b) * p.A + a) * S + r] : 0.f;
    auto wait_all = [&](uint64_t* bar) {
      return __all_sync(0xffffffffu, ptx::mbar_wait(bar, 0, lim, p.status, kWaitHint));
    };
    // delta = dO . O of the row, from the swizzled tiles (loaded from global memory
    // row by row, 16 bytes a lane, this took 8 us)
    float dl = 0.f;
    bool ok = wait_all(ov_full);
    if (ok) {
      const uint32_t so = ptx::smem_u32(smem + SH_O) + r * 128, sx = ptx::smem_u32(smem + SH_DS) + r * 128;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t x[4], y[4];
        ptx::ld_shared_v4(so + ((j ^ (r & 7)) << 4), x);
        ptx::ld_shared_v4(sx + ((j ^ (r & 7)) << 4), y);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 u = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x[e]));
          const float2 w = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&y[e]));
          dl += u.x * w.x + u.y * w.y;
        }
      }
    }
    const uint64_t sc2 = pack2(sl2, sl2), nlse = pack2(nlse2, nlse2), ndl = pack2(-dl, -dl);
    softmax_warps_sync();  // every row's O is read: dS may be written
    ok = ok && wait_all(sc_full);
    if (ok) {
      ptx::tc_fence_after();
      const uint32_t sp = ptx::smem_u32(smem + SH_P) + hf * Q_BYTES + r * 128;
      const uint32_t sd = ptx::smem_u32(smem + SH_DS) + hf * Q_BYTES + r * 128;
#pragma unroll
      for (int c = 0; c < 64; c += 32) {
        uint32_t sv[32], dv[32];
        ptx::tmem_ld_32x32b_x32(tS + lane_base + hf * 64 + c, sv);
        ptx::tmem_ld_32x32b_x32(tdP + lane_base + hf * 64 + c, dv);
        ptx::tmem_ld_wait();
        const int left = live ? len - hf * 64 - c : 0;  // valid keys from this chunk's first on
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t pp[4], dd[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int i = 8 * u + 2 * e;
            const float2 x = unpack2(fma2(pack2(__uint_as_float(sv[i]), __uint_as_float(sv[i + 1])), sc2, nlse));
            const float p0 = ptx::ex2_ftz(x.x), p1 = ptx::ex2_ftz(x.y);
            const float2 ds = unpack2(
                mul2(pack2(p0, p1), add2(pack2(__uint_as_float(dv[i]), __uint_as_float(dv[i + 1])), ndl)));
            pp[e] = ptx::pack_bf16(p0, p1);
            dd[e] = ptx::pack_bf16(ds.x, ds.y);
            const uint32_t keep = (i < left ? 0x0000ffffu : 0u) | (i + 1 < left ? 0xffff0000u : 0u);
            pp[e] &= keep;
            dd[e] &= keep;
          }
          const uint32_t at = ((c / 8 + u) ^ (r & 7)) << 4;
          ptx::st_shared_v4(sp + at, pp[0], pp[1], pp[2], pp[3]);
          ptx::st_shared_v4(sd + at, dd[0], dd[1], dd[2], dd[3]);
        }
      }
      ptx::fence_proxy_async_smem();  // P, dS -> the MMAs
      ptx::tc_fence_before();
      ptx::mbar_arrive(pds_full);
      ok = wait_all(g_full);
    }
    pdl_trigger();
    // the low-half warps stage dK / sqrt(D), the high-half warps dV, and each half
    // of dQ / sqrt(D), as 128-byte-swizzled bf16 rows over tiles that the last
    // products have read; one thread stores the three by TMA, which drops the
    // rows past S
    float* red = reinterpret_cast<float*>(smem + SH_DS);  // column sums: [3][4 quarters][64]
    if (ok) {
      ptx::tc_fence_after();
      const float sc = hf == 0 ? 0.125f : 1.f;
      const int sel = hf == 0 ? 1 : 2;  // block of dqkv: 0 dQ, 1 dK, 2 dV
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const bool is_q = c == 2;
        const int col = is_q ? hf * 32 : c * 32;  // of the gradient's 64
        uint32_t o[32];
        ptx::tmem_ld_32x32b_x32((is_q ? tdQ : (hf == 0 ? tdK : tdV)) + lane_base + col, o);
        ptx::tmem_ld_wait();
        const float m = is_q ? 0.125f : sc;
        const uint32_t orow = ptx::smem_u32(smem + (is_q ? SH_Q : (hf == 0 ? SH_K : SH_V))) + r * 128;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t w[4];
#pragma unroll
          for (int t = 0; t < 4; ++t)
            w[t] = ptx::pack_bf16(__uint_as_float(o[8 * u + 2 * t]) * m, __uint_as_float(o[8 * u + 2 * t + 1]) * m);
          ptx::st_shared_v4(orow + (((col / 8 + u) ^ (r & 7)) << 4), w[0], w[1], w[2], w[3]);
        }
        if (p.colpart) {  // column sums of the stored values over this warp's 32 rows
          float v[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = live ? bf16_round(__uint_as_float(o[j]) * m) : 0.f;
          lanes_column_sum(v, lane);
          red[((is_q ? 0 : sel) * 4 + q4) * 64 + col + lane] = v[0];
        }
      }
    } else if (p.colpart) {
      red[(hf == 0 ? 1 : 2) * 256 + q4 * 64 + lane] = red[(hf == 0 ? 1 : 2) * 256 + q4 * 64 + 32 + lane] = 0.f;
      red[q4 * 64 + hf * 32 + lane] = 0.f;
    }
    ptx::fence_proxy_async_smem();  // the staged rows -> the TMA stores
    softmax_warps_sync();
    if (warp == 2 && lane == 0) {
      ptx::tma_store_3d(&tmOut, smem + SH_Q, a * HD, 0, b);
      ptx::tma_store_3d(&tmOut, smem + SH_K, H + a * HD, 0, b);
      ptx::tma_store_3d(&tmOut, smem + SH_V, 2 * H + a * HD, 0, b);
      ptx::bulk_commit_group();
    }
    const int t = static_cast<int>(threadIdx.x) - 64;
    if (p.colpart && t < 3 * HD) {  // the four row quarters, added in order
      const int g = t / HD, c = t % HD;
      const float* x = red + g * 256 + c;
      p.colpart[static_cast<int64_t>(b) * 3 * H + g * H + a * HD + c] = ((x[0] + x[64]) + x[128]) + x[192];
    }
    if (warp == 2 && lane == 0) ptx::bulk_wait_group_read0();  // before the CTA's memory goes
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, 256);
  }
}

namespace {
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  });
  return fn;
}

// [T, W] bf16 activations, box {64 columns (one head), rows}, 128B swizzle.
bool head_map(CUtensorMap* map, const void* base, int64_t T, int W, int rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(W), static_cast<cuuint64_t>(T)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(W) * 2};
  cuuint32_t box[2] = {64u, static_cast<cuuint32_t>(rows)};
  cuuint32_t estr[2] = {1u, 1u};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// dQKV as [B][S][3H] bf16 for the dK/dV tile stores: box {64 columns, 128
// rows of one sequence}, 128B swizzle; rows past S fall outside the tensor.
bool seq_map(CUtensorMap* map, void* base, int B, int S, int W, int rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(W), static_cast<cuuint64_t>(S),
                        static_cast<cuuint64_t>(B)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(W) * 2, static_cast<cuuint64_t>(W) * 2 * S};
  cuuint32_t box[3] = {64u, static_cast<cuuint32_t>(rows), 1u};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

}  // namespace attn_tc

// Forward launcher used by the bf16 attention path (D = 64).
sky_status attention_fwd_tc(const void* qkv, const int32_t* lens, int B, int S, int H, int A,
                            void* ctx, float* lse, int32_t* status, uint64_t timeout_ns,
                            cudaStream_t stream) {
  using namespace attn_tc;
  SKY_CHECK(H == A * HD, SKY_ERR_UNSUPPORTED, "tensor-core attention needs head dim 64");
  SKY_CHECK((reinterpret_cast<uintptr_t>(qkv) & 15) == 0 && (reinterpret_cast<uintptr_t>(ctx) & 15) == 0,
            SKY_ERR_UNSUPPORTED, "attention buffers must be 16-byte aligned");
  CUtensorMap tq, tkv, tout;
  const int64_t T = static_cast<int64_t>(B) * S;
  if (S <= 128 && B <= 65535) {  // one tile a sequence
    SKY_CHECK(head_map(&tq, qkv, T, 3 * H, BQ) && seq_map(&tout, ctx, B, S, H, BQ), SKY_ERR_CUDA,
              "cuTensorMapEncodeTiled failed for the attention operands");
    static OncePerDevice once;
    const cudaError_t at = allow_smem(once, attn_fwd_short_tc, FS_SMEM);
    if (at != cudaSuccess) return cuda_fail(at, "attention smem attribute");
    FwdParams p{S, H, A, lens, static_cast<__nv_bfloat16*>(ctx), lse, status, timeout_ns};
    const cudaError_t e = launch_pdl(attn_fwd_short_tc, dim3(A, B), dim3(NTHR), FS_SMEM, stream, 1, tq, tout, p);
    count_launches(1);
    return e == cudaSuccess ? SKY_OK : cuda_fail(e, "tensor-core attention forward launch");
  }
  // Which form (us; [ragged] lengths uniform in 1..S; CTAs of 128 queries, 152 SMs):
  //  two buffers up to 2.6 CTAs an SM: 2 x 1024 x 12 heads (192) 11.9 against 17.6 with
  //    one; 8 x 700 x 8 (384) 16.9 and 14.8, [8.5 and 12.8]; 6 x 700 x 12 (432) 17.8
  //    and 15.0, [12.8 and 11.2].  From 24 key tiles on, where CTAs left alone at the
  //    end take long, up to six: 4 x 2048 x 12 (768) 66 and 71; 4 x 1500 x 16 (768)
  //    [35.9 and 39.7]; 4 x 2048 x 16 (1024) 86 and 81, [64.5 and 63.4, of 512..S].
  //  else one: 16 x 512 x 16 (1024) 27.0 against 32.7, 24 x 197 x 12 (576) 9.6 and 11.6.
  //  keys in four while that leaves two CTAs an SM and each three tiles: 1024 x 9 heads
  //    (72) 8.3, unsplit 10.0; in two up to one CTA an SM and from 24 tiles on: 2048 x
  //    8 (128) 14.3 and 17.4; 800 x 12 (84, 13 tiles) 8.2 and 7.4.
  const int sms = sm_count() > 0 ? sm_count() : 148, tiles = ceil_div(S, BKV);
  const int64_t ctas = static_cast<int64_t>(ceil_div(S, BQ)) * A * B;
  const bool two = 5 * ctas <= 13 * sms || (tiles >= 24 && ctas <= 6 * sms);
  const int ks = tiles >= 12 && 2 * ctas <= sms ? 4 : tiles >= 24 && ctas <= sms ? 2 : 1;
  SKY_CHECK(head_map(&tq, qkv, T, 3 * H, BQ) && head_map(&tkv, qkv, T, 3 * H, BKV) &&
                seq_map(&tout, ctx, B, S, H, BQ / ks),
            SKY_ERR_CUDA,
            "cuTensorMapEncodeTiled failed for the attention operands");
  FwdParams p{S, H, A, lens, static_cast<__nv_bfloat16*>(ctx), lse, status, timeout_ns};
  auto go = [&](auto splits, auto bufs) {
    constexpr int KS = decltype(splits)::value, NS = decltype(bufs)::value;
    auto kern = attn_fwd_tc<KS, NS>;
    constexpr int SMEM = KS > 1 ? kSplitAttentionSmem : FwdShape<NS>::SMEM;
    static_assert(SMEM >= FwdShape<NS>::SMEM && (KS == 1 || FwdShape<NS>::TMEM_COLS <= 256), "see residency.h");
    static OncePerDevice once;
    const cudaError_t attr = allow_smem(once, kern, SMEM);
    if (attr != cudaSuccess) return attr;
    return launch_pdl(kern, dim3(ceil_div(S, BQ) * KS, A, B), dim3(NTHR), SMEM, stream, KS, tq, tkv, tout, p);
  };
  const std::integral_constant<int, 1> c1{};
  const std::integral_constant<int, 2> c2{};
  const std::integral_constant<int, 4> c4{};
  const cudaError_t e = !two ? go(c1, c1) : ks == 1 ? go(c1, c2) : ks == 2 ? go(c2, c2) : go(c4, c2);
  count_launches(1);
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "tensor-core attention forward launch");
}

// Backward of sequences up to 128 (bf16, D = 64) in one launch.
sky_status attention_bwd_short_tc(const void* qkv, const void* ctx, const void* dctx, const float* lse,
                                  const int32_t* lens, int B, int S, int H, int A, void* dqkv, int32_t* status,
                                  uint64_t timeout_ns, cudaStream_t stream, float* colpart) {
  using namespace attn_tc;
  SKY_CHECK(H == A * HD, SKY_ERR_UNSUPPORTED, "tensor-core attention needs head dim 64");
  const int64_t T = static_cast<int64_t>(B) * S;
  CUtensorMap tq, to, tc, tout;
  SKY_CHECK(head_map(&tq, qkv, T, 3 * H, BQ) && head_map(&to, dctx, T, H, BQ) && head_map(&tc, ctx, T, H, BQ) &&
                seq_map(&tout, dqkv, B, S, 3 * H, BQ),
            SKY_ERR_CUDA, "cuTensorMapEncodeTiled failed for the attention backward operands");
  static OncePerDevice once;
  const cudaError_t attr = allow_smem(once, attn_bwd_short_tc, SH_SMEM);
  if (attr != cudaSuccess) return cuda_fail(attr, "attention backward smem attribute");
  BwdParams p{S, H, A, lens, lse, nullptr, nullptr, static_cast<__nv_bfloat16*>(dqkv), colpart, status, timeout_ns};
  const cudaError_t e = launch_pdl(attn_bwd_short_tc, dim3(A, B), dim3(SH_THR), SH_SMEM, stream, 1, tq, to, tc,
                                   tout, p);
  count_launches(1);
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "tensor-core attention backward launch");
}

// Backward launchers (bf16, D = 64): delta must already hold rowsum(dO * O).
sky_status attention_bwd_tc(const void* qkv, const void* dctx, const float* lse, const float* delta,
                            const uint4* xtab, const int32_t* lens, int B, int S, int H, int A, void* dqkv,
                            int32_t* status, uint64_t timeout_ns, cudaStream_t stream,
                            float* colpart) {
  using namespace attn_tc;
  SKY_CHECK(H == A * HD, SKY_ERR_UNSUPPORTED, "tensor-core attention needs head dim 64");
  const int64_t T = static_cast<int64_t>(B) * S;
  CUtensorMap tq128, tkv64, to128, tk128, tq64, to64, tout;
  SKY_CHECK(head_map(&tq128, qkv, T, 3 * H, BQ) && head_map(&tkv64, qkv, T, 3 * H, BKV) &&
                head_map(&to128, dctx, T, H, BQ) && head_map(&tk128, qkv, T, 3 * H, BK2) &&
                head_map(&tq64, qkv, T, 3 * H, BQ2) && head_map(&to64, dctx, T, H, BQ2) &&
                seq_map(&tout, dqkv, B, S, 3 * H, BK2),
            SKY_ERR_CUDA, "cuTensorMapEncodeTiled failed for the attention backward operands");
  static OncePerDevice once1, once2;
  const cudaError_t a1 = allow_smem(once1, attn_bwd_dq_tc, DQ_SMEM), a2 = allow_smem(once2, attn_bwd_dkdv_tc, KV_SMEM);
  if (a1 != cudaSuccess) return cuda_fail(a1, "attention dQ smem attribute");
  if (a2 != cudaSuccess) return cuda_fail(a2, "attention dK/dV smem attribute");
  SKY_CHECK((reinterpret_cast<uintptr_t>(xtab) & 15) == 0, SKY_ERR_INVALID_ARG,
            "attention backward workspace must be 16-byte aligned");
  BwdParams p{S, H, A, lens, lse, delta, xtab, static_cast<__nv_bfloat16*>(dqkv), colpart, status,
              timeout_ns};
  cudaError_t e = launch_pdl(attn_bwd_dkdv_tc, dim3(ceil_div(S, BK2), A, B), dim3(NTHR_B), KV_SMEM,
                             stream, 1, tk128, tq64, to64, tout, p);
  if (e == cudaSuccess)
    e = launch_pdl(attn_bwd_dq_tc, dim3(ceil_div(S, BQ), A, B), dim3(NTHR_B), DQ_SMEM, stream, 1,
                   tq128, tkv64, to128, tout, p);
  count_launches(2);
  return e == cudaSuccess ? SKY_OK : cuda_fail(e, "tensor-core attention backward launch");
}

}  // namespace sky
