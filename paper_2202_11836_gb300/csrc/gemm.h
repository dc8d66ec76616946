// Internal GEMM launchers (bf16 tensor-core and fp32 SIMT).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/sky_ops.h"

namespace sky {
namespace gemm {

// bf16 inputs on tcgen05; C is bf16 unless out_f32.
// colpart (optional, GELU_BWD epilogue): also writes partial column sums of C
// (before rounding), one row per 32 rows of C; *colpart_rows reports how many (for
// a fixed-order reduction, possibly on another stream ordered after this launch).
// resid (optional, fp32 output of the STORE epilogue, no split): C = acc +
// bias + resid[m, n], added in that order (the residual branch of Sec. II-C).
// resid == C (XTW form, no bias): C += product, which may be split.
// With `ln`, resid holds the pre-LayerNorm sum u of the previous sub-layer and
// the residual added is its LayerNorm output, recomputed in the epilogue from
// the row statistics: gamma[n] * ((u[m, n] - mean[m]) * rstd[m]) + beta[n]
// (Eq. 3; the same expression the LayerNorm forward evaluates, so the sum is
// the one an fp32 copy of the LayerNorm output would give).
struct LnResid {
  const float* mean;  // [M]
  const float* rstd;  // [M]
  const void* gamma;  // [N] bf16
  const void* beta;   // [N] bf16
};
sky_status launch_bf16(sky_gemm_form form, int M, int N, int K, const void* A, const void* B,
                       void* C, bool out_f32, int epi, const void* bias, const void* aux,
                       void* aux_out, void* ws, size_t ws_bytes, int32_t* status,
                       cudaStream_t stream, float* colpart = nullptr, size_t colpart_bytes = 0,
                       int* colpart_rows = nullptr,
                       const float* resid = nullptr, const LnResid* ln = nullptr);
// 2-D bf16 tensor map over a row-major [rows, cols] matrix, box {64, box_rows},
// 128-byte swizzle; out-of-range elements read as zero.
bool make_map(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int box_rows);

// The cluster kernel (gemm_cluster.cu): tiles of 128 x bn (pair: 256 x bn on an
// SM pair), each tile's k-blocks split over ks CTAs (pairs) of one cluster.
struct ClusterPlan {
  bool pair;
  int bn, ks;
};
// Whether a product goes to the cluster kernel, and with which tiles.
// may_split: an fp32 output without bias or residual (C += product is none); ws_split: of
// those, with a workspace that holds the persistent kernel's partial sums; colpart: column
// sums per 32 rows are wanted.
bool plan_cluster(sky_gemm_form form, int M, int N, int K, bool may_split, bool ws_split, bool colpart, int sms,
                  ClusterPlan* out);
// Arguments as launch_bf16, already checked there.
sky_status launch_cluster(sky_gemm_form form, const ClusterPlan& pl, int M, int N, int K, const void* A,
                          const void* B, void* C, bool out_f32, int epi, const void* bias,
                          const void* aux, void* aux_out, int32_t* status, uint64_t timeout_ns,
                          int skip_loads, cudaStream_t stream, float* colpart, const float* resid,
                          const LnResid* ln);

// Rows of column partials a bf16 GEMM with M rows writes (upper bound).
int colpart_rows_max(int M);
// out[n] = sum over r of part[r][n] in order r = 0, 1, ... (rowwise.cu).
cudaError_t reduce_rows_f32(const float* part, int rows, int N, float* out, cudaStream_t stream);
size_t workspace_bytes(sky_gemm_form form, int M, int N, int K, bool out_f32);
int choose_splits(int64_t mn, int tiles, int k_blocks, int sms);
// Debug controls: per-wait timeout (0 = default 2 s) and the fault-injection
// switch that makes the TMA producer skip its loads (waits then time out).
void set_debug(uint64_t timeout_ns, int skip_loads);

// fp32 SIMT path (exact fp32 FMA accumulation); same forms and epilogues.
sky_status launch_f32(sky_gemm_form form, int M, int N, int K, const float* A, const float* B,
                      float* C, int epi, const float* bias, const float* aux, float* aux_out,
                      cudaStream_t stream);

}  // namespace gemm
}  // namespace sky
