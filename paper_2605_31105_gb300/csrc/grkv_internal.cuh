// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include <utility>

#include "grkv.h"

namespace grkv {

constexpr int kD = 128;          // supported head dimension
constexpr int kMaxM = 256;       // stacked window rows g*w supported
constexpr int kMaxScoreCtas = 256;  // persistent score grid bound used to size slots
constexpr int kMaxCgIters = 4096;   // bound on the key step's conjugate-gradient iterations
constexpr int kMaxSteps = 64;       // bound on the alternating steps S

// A unit's budget when units have their own (grkv_compress_ragged): retained
// tokens, score-ranked fixed tokens, and its first row of the packed outputs.
struct UnitRow {
  int32_t B, n_fix;
  int64_t off;
};

// Validated problem sizes, derived once on the host.
struct Shape {
  int U, g, n, d, w, B, m;
  int P;          // prefix length n - w (scored, pooled, selectable)
  int pool_k, pool_type, n_sink, n_fix, causal, dtype;
  float lambda, scale;
  int lambda_inf; // lambda_v == +inf: values stay V0
  int tc;         // bf16, m <= 256, not forced portable: tensor-core scoring
  int tc_merge;   // ... and B <= 32768: tensor-core value merge
  int one_read;   // tensor-core scoring in one launch that reads K from HBM once
  int deterministic;  // Y summed in a fixed order (GRKV_DETERMINISTIC)
  int test_timeout;   // GRKV_TEST_TIMEOUT (tests of the bounded-wait exit)
  int checks;         // GRKV_CHECKS: device-side argument checks
  int update_k;   // key step after the value step (GRKV_UPDATE_K)
  int cg_iters;   // most conjugate-gradient iterations of the key step
  float cg_tol;   // ... until ||r|| <= cg_tol ||e||
  float lambda_k; // ridge weight of the key step
  int steps;      // S alternating value / key steps (Algorithm 1)
  float step_tol; // stop once max |K^(t+1) - K^(t)|, max |V^(t+1) - V^(t)| <= step_tol
  bool chained;          // select, merge: the work before is a kernel of the same call
  const UnitRow* units;  // device table [U], or null: every unit has B, n_fix and row u B
  size_t rows;           // with a table: rows of the packed outputs
};

__device__ inline UnitRow unit_row(const UnitRow* units, int u, int B, int n_fix) {
  return units ? units[u] : UnitRow{B, n_fix, (int64_t)u * B};
}

// Kernels of a call after its first are launched while the kernel before them
// drains (programmatic stream serialization): block scheduling and launch latency
// overlap its end.  chain_wait(), the first statement of every such kernel in all
// threads, then waits until that kernel has completed and its writes are visible.  No
// kernel signals earlier than its end, so only the tail of one kernel overlaps the
// start of the next, and a kernel that has ended implies that all before it have.
// (A signal at each kernel's start is slower: CTAs that only wait hold shared memory
// and block slots; 8 units n = 8192 98.5 us a compress call against 95.5, and 109 without
// chaining; one fp32 unit n = 2048 100 and 98 us against 121.)
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// chained: the work before this launch in the stream is a kernel of the same call.
template <typename... Params, typename... Args>
cudaError_t launch_kernel(bool chained, int cluster, void (*kern)(Params...), dim3 grid, int threads,
                          size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  if (chained) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// Whether the device, or the part of it that the process has, holds a cluster of that many
// such CTAs (asked after the kernel's shared-memory limit is set).  No measurable host time: a
// compress call of 8 units n = 8192 takes 18.2 to 19.0 us of it with the query and without.
template <typename... Params>
bool cluster_fits(int cluster, void (*kern)(Params...), int threads, size_t smem) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) return true;
  (void)cudaGetLastError();
  return false;
}

// Byte offsets of the workspace regions (each 256-B aligned).
struct WsLayout {
  size_t status;  // int32 device status word
  // score path (portable kernels)
  size_t pstats;  // float2 [U][nchunk][m]      per-chunk (max, sum)
  size_t ypart;   // float  [U][nchunk][m][d]   per-chunk target partials
  int chunk, nchunk;
  // score path (tensor cores)
  size_t pstats_tc;  // float2 [U][maxc][128 or 256] pass-A statistics slots
  size_t flags_tc;   // int [U] pass-A slots written per unit (one-read kernel)
  size_t lam_tc;     // float [U][128] combined log2 row normalisers (one-read scoring)
  size_t ypart_tc;   // float [U][maxc][m][128] segment Y partials (deterministic mode)
  // select
  size_t pooled;  // float [U][P]
  // merge
  size_t xbuf;    // float [U][m][B]   retained logits, then X
  size_t flags;   // uint8 [U][B]      fixed-token flags
  size_t gram;    // acc   [U][m][m]   X_G X_G^T + lambda I, then its Cholesky factor
  size_t rz;      // acc   [U][m][d]   residual R, then Z
  size_t state;   // int   [U]         outcome of the unit's solve
  size_t merge_tc;  // tensor-core merge: R/Z, Gram [U][128][128] fp32, normalisers, positions, fixed flags
  // compress intermediates
  size_t scores;  // float [U][P]
  size_t y;       // float [U][m][d]
  size_t rstats;  // float2 [U][m]
  size_t key;     // key step: CG vectors [U][C][5][m][d], X, T, T2 [U][m][B], dK [U][B][d], fixed [U][B]
  size_t total;
};

WsLayout plan_workspace(const Shape& s);

// Order-preserving map of an fp32 value to an unsigned key.
__host__ __device__ inline uint32_t order_key(float f) {
#ifdef __CUDA_ARCH__
  uint32_t b = __float_as_uint(f);
#else
  uint32_t b;
  memcpy(&b, &f, 4);
#endif
  return b ^ ((b >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}

__device__ inline void set_status(int* status, int code) { atomicCAS(status, 0, code); }

// Adds n to the process-wide count of kernels this library enqueued.
void count_launches(int n);

// Launchers (all asynchronous on `st`).
cudaError_t launch_score_simt(const Shape& s, const void* q, const void* k, const void* v,
                              float* scores, float* y, float* row_stats, char* ws,
                              const WsLayout& L, cudaStream_t st);
int score_simt_chunk(const Shape& s);   // keys per CTA of the portable scoring
cudaError_t launch_select(const Shape& s, const float* scores, int32_t* idx, char* ws,
                          const WsLayout& L, cudaStream_t st);
// Tensor-core window scoring (bf16, m <= 256 in blocks of 128 rows).  The
// default, launch_score_tc, runs two launches that each read K;
// launch_score_pipe (GRKV_ONE_READ_SCORE) reads K once per row block.
bool score_tc_supported(const Shape& s);
struct PipePlan {
  int ng, gs;   // CTA groups, CTAs per group
};
PipePlan score_pipe_plan(const Shape& s, int sms);
size_t score_pipe_slot_bytes(const Shape& s);
cudaError_t launch_score_pipe(const Shape& s, const void* q, const void* k, const void* v,
                              float* scores, float* y, float* row_stats, char* ws,
                              const WsLayout& L, cudaStream_t st);
size_t score_tc_pstats_bytes(const Shape& s, int* maxc);   // maxc: slots per unit
int sm_count();
cudaError_t launch_score_tc(const Shape& s, const void* q, const void* k, const void* v,
                            float* scores, float* y, float* row_stats, char* ws,
                            const WsLayout& L, cudaStream_t st);

// Tensor-core value merge (bf16, m <= 256 in 128-row blocks, B <= 32768).
bool merge_tc_supported(const Shape& s);
// The fp32 regression solve for m <= 256 (grkv_solve.cu): gram [U][ld][ld]
// (N with lambda when sym = 0; raw Gram blocks, symmetrised with lambda added,
// when sym = 1; the block of rows < 128, columns >= 128 is overwritten), rz
// [U][ld][128] (R in, Z out).  For m > 128, fac holds 128 columns of fac_ld
// floats per unit, units fac_unit floats apart, and fail one int per unit.
cudaError_t launch_solve(int U, int m, int ld, int sym, float lambda, int lambda_inf, float* gram,
                         float* rz, float* fac, size_t fac_unit, int fac_ld, int* fail,
                         int* status, cudaStream_t st);
size_t merge_tc_ws_bytes(const Shape& s);
// row_stats (nullable): the full-cache row statistics; with them the Gram
// needs one pass over the retained keys.
size_t key_ws_bytes(const Shape& s);
// The value step's fixed-token flags [U][B] in the workspace, on either path.
const uint8_t* merge_tc_fixed(const Shape& s, const char* ws, const WsLayout& L);
inline const uint8_t* value_step_fixed(const Shape& s, const char* ws, const WsLayout& L) {
  return s.tc_merge ? merge_tc_fixed(s, ws, L) : (const uint8_t*)(ws + L.flags);
}
// The key step (GRKV_UPDATE_K) and, for S > 1, the remaining alternating
// steps; k, v are the full caches (K0 and V0 of steps t >= 1).
cudaError_t launch_key_step(const Shape& s, const void* q, const void* k, const void* v,
                            const float* y, const float* scores, const int32_t* idx,
                            void* v_out, void* k_out, char* ws, const WsLayout& L,
                            cudaStream_t st);
cudaError_t launch_merge_tc(const Shape& s, const void* q, const void* k, const void* v,
                            const float* scores, const float* y, const float* row_stats,
                            const int32_t* idx, void* k_out, void* v_out, char* ws,
                            const WsLayout& L, cudaStream_t st);

// Selection with the pooled-score scratch [U][n-w] given directly; the
// scratch may be touched only when select_uses_pooled_buffer(s) holds (prefixes
// longer than one CTA takes: a cluster takes most of them without it).
bool select_uses_pooled_buffer(const Shape& s);
cudaError_t launch_select_pooled(const Shape& s, const float* scores, int32_t* idx,
                                 float* pooled, cudaStream_t st);
// Dispatch of the scoring step and of the value step to the kernels the
// shape selects (as every entry point runs them).
cudaError_t launch_score_any(const Shape& s, const void* q, const void* k, const void* v,
                             float* scores, float* y, float* row_stats, char* ws,
                             const WsLayout& L, cudaStream_t st);
cudaError_t launch_merge_any(const Shape& s, const void* q, const void* k, const void* v,
                             const float* scores, const float* y, const float* row_stats,
                             const int32_t* idx, void* k_out, void* v_out, char* ws,
                             const WsLayout& L, cudaStream_t st);
// GRKV_CHECKS: finite inputs (GRKV_ERR_INVALID_ARG) and the idx contract
// (GRKV_ERR_BOUNDS), written to the status word.
cudaError_t launch_check_inputs(const Shape& s, const void* q, const void* k, const void* v,
                                int* status, cudaStream_t st);
cudaError_t launch_check_idx(const Shape& s, const int32_t* idx, int* status, cudaStream_t st);
// Host-side parameter validation shared by the entry points.
int make_shape(const grkv_params* p, Shape* s);
cudaError_t launch_merge_simt(const Shape& s, const void* q, const void* k, const void* v,
                              const float* scores, const float* y, const int32_t* idx,
                              void* k_out, void* v_out, char* ws, const WsLayout& L,
                              cudaStream_t st);

}  // namespace grkv
