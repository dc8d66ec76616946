// Shared host/device helpers of the encoder-slice library.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <string>

#include "../../include/sky_ops.h"
#include "../../include/sky_slice.h"
#include "device_once.h"

namespace sky {

// Device status word bits (sky_ops.h: d_status).
constexpr int32_t kStatusBadLength = 1;
constexpr int32_t kStatusTimeout = 2;

// Records the thread-local error message returned by sky_last_error().
void set_error(const char* fmt, ...);
sky_status cuda_fail(cudaError_t e, const char* what);

#define SKY_CUDA(call)                                        \
  do {                                                        \
    cudaError_t e_ = (call);                                  \
    if (e_ != cudaSuccess) return ::sky::cuda_fail(e_, #call); \
  } while (0)

#define SKY_CHECK(cond, status, ...)   \
  do {                                 \
    if (!(cond)) {                     \
      ::sky::set_error(__VA_ARGS__);   \
      return (status);                 \
    }                                  \
  } while (0)

// bf16 <-> fp32 conversions usable for both storage types.
template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// GELU(h) = h * Phi(h) and its derivative Phi(h) + h * phi(h), with
// Phi(h) = (1 + erf(h / sqrt 2)) / 2 from CUDA's erff and phi from expf
// (exact-erf form, no tanh approximation).
__device__ __forceinline__ float std_normal_cdf(float h) {
  return 0.5f * (1.f + erff(h * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_f(float h) { return h * std_normal_cdf(h); }
__device__ __forceinline__ float gelu_grad_f(float h) {
  const float inv_sqrt_2pi = 0.3989422804014327f;
  return std_normal_cdf(h) + h * inv_sqrt_2pi * expf(-0.5f * h * h);
}

// GELU(h) and GELU'(h) together, for the tensor-core epilogues: Phi from the
// erf approximation of Abramowitz & Stegun, Handbook of Mathematical
// Functions, formula 7.1.25 (|erf error| <= 2.5e-5 for all x: well below the
// bf16 rounding of GELU and the fp16 rounding of GELU'), written for
// x = |h| / sqrt 2 so that Phi and phi share one exponential exp(-h^2 / 2):
//   t = 1 / (1 + p x),  Phi(-|h|) = (1/2)(a1 t + a2 t^2 + a3 t^3) exp(-h^2/2).
// The 1/2 is folded into the coefficients and 1/sqrt 2 into p; the
// reciprocal and the exponential use the hardware approximations (relative
// error of a few ulp).  The epilogue is bound by this arithmetic, so the
// three-term formula (two FMAs fewer than the five-term 7.1.26) pays.
__device__ __forceinline__ void gelu_and_grad_as(float h, float& g, float& gp) {
  float t, E;
  const float den = fmaf(fabsf(h), 0.47047f * 0.70710678118654752f, 1.f);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(den));
  const float q_poly = t * (0.5f * 0.3480242f + t * (0.5f * -0.0958798f + t * (0.5f * 0.7478556f)));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(E) : "f"((h * -0.72134752044448170f) * h));  // exp(-h^2/2)
  const float q = q_poly * E;  // Phi(-|h|)
  const float Phi = h >= 0.f ? 1.f - q : q;
  g = h * Phi;
  gp = fmaf(h * 0.3989422804014327f, E, Phi);
}

// Packed pairs of fp32: one instruction, each half rounded as its scalar form.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// gelu_and_grad_as of two values, in packed arithmetic where it pairs up, with
// the sign handled without branches: with q = Phi(-|h|),
//   GELU(h) = max(h, 0) - |h| q,   Phi(h) = 1/2 + sign(h) (1/2 - q).
// The factor of q stops at 64, where q is 0 long since, so that GELU(+inf) is +inf.
__device__ __forceinline__ void gelu_and_grad_as2(float h0, float h1, float2& g, float2& gp) {
  const auto both = [](float v) { return pack2(v, v); };
  float t0, t1, e0, e1;
  const float den0 = fmaf(fabsf(h0), 0.47047f * 0.70710678118654752f, 1.f);
  const float den1 = fmaf(fabsf(h1), 0.47047f * 0.70710678118654752f, 1.f);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t0) : "f"(den0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t1) : "f"(den1));
  const uint64_t h = pack2(h0, h1), t = pack2(t0, t1);
  const float2 x = unpack2(mul2(mul2(h, both(-0.72134752044448170f)), h));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(x.x));  // exp(-h^2/2)
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(x.y));
  const uint64_t E = pack2(e0, e1);
  uint64_t poly = fma2(t, both(0.5f * 0.7478556f), both(0.5f * -0.0958798f));
  poly = mul2(t, fma2(t, poly, both(0.5f * 0.3480242f)));
  const uint64_t q = mul2(poly, E);
  const float2 qq = unpack2(q);
  g.x = fmaf(-fabsf(fminf(h0, 64.f)), qq.x, fmaxf(h0, 0.f));
  g.y = fmaf(-fabsf(fminf(h1, 64.f)), qq.y, fmaxf(h1, 0.f));
  const uint64_t s = pack2(copysignf(1.f, h0), copysignf(1.f, h1));
  const uint64_t Phi = fma2(s, fma2(q, both(-1.f), both(0.5f)), both(0.5f));
  gp = unpack2(fma2(mul2(h, both(0.3989422804014327f)), E, Phi));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

inline int ceil_div(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

int sm_count();  // cached per device

// Number of kernels this library has launched (all threads, all devices).
void count_launches(int n);

// ---- Programmatic dependent launch ------------------------------------------
// Hot-path kernels launch with programmatic stream serialization: the next
// kernel on the stream may be scheduled once every CTA of the current one
// has called pdl_trigger() (or ended), and it runs pdl_wait() -- which returns
// when the previous grid has completed and its memory is visible -- before it
// reads anything that grid wrote or writes anything it reads.  Its launch and
// set-up then overlap the previous kernel's tail instead of following its
// completion.  SKY_PDL=0 in the environment turns the attribute off (plain
// stream order).
//
// Where a kernel triggers matters.  CTAs that wait hold registers, shared
// memory and TMEM, and they are placed where room comes free first, so a
// kernel released early starts unevenly spread.  Triggering before one's own
// wait is worst: several kernels of a chain are then resident at once.  So:
// GEMMs and the short attention kernels trigger behind their main loop, and the
// row-wise kernels, which end all at once, right after their wait.  With every
// kernel triggering first: forward of 2 base layers on 74 rows 90.1 us (now
// 79.4), FFN forward block on 4999 rows 106.0 (99.0), 4 micro-batches x 3 base
// layers 2040 (1935), LayerNorm forward + backward of 16384 rows 91.0 (82.9),
// 2-layer fp32 slice of width 128 252 (221), 4-layer base step 1096 (1083).
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

bool pdl_enabled();

// Allows a kernel `bytes` of dynamic shared memory, which is a setting of each
// device: `once` is the kernel's own, static at its launch site.
template <typename K>
cudaError_t allow_smem(OncePerDevice& once, K* kern, size_t bytes) {
  int device = -1;
  const cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  return once(device, [&] {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  });
}

// cudaLaunchKernelEx with the programmatic-serialization attribute (when
// enabled) and optionally a cluster of `cluster_x` CTAs.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                       cudaStream_t st, int cluster_x, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (pdl_enabled()) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (cluster_x > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = cluster_x;
    at[n].val.clusterDim.y = 1;
    at[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

}  // namespace sky
