// Window scoring on CUDA cores (fp32 inputs, and bf16 under GRKV_FORCE_SIMT).
//
// Every logit is an fp32 FMA chain over the head dimension, probabilities use
// expf and an IEEE divide, and every reduction runs in a fixed order, so
// results are deterministic.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "simt_common.cuh"

namespace grkv {
namespace {

// ------------------------------------------------------------ logits tile --
// Both passes form S = Q K^T in tiles of MR window rows x 64 keys: 256 threads
// as 16 x 16, thread (ty, tx) rows ty MR/16 .. and keys tx, tx + 16, ...  The
// operands stay [row][t] in shared memory with rows of 132 floats, read four t
// at a time: with MR = 128, 12 16-byte loads feed 128 FMAs.  Bound by a tile's phases
// (load, products, exponentials, P) between block barriers, with two warps per scheduler to
// cover them: 8 units of n = 8192, m = 128 take 88 + 156 us, the FMA pipe busy in 38% and 41%
// of the cycles (one load per FMA, one output per thread and 64-key chunks cut into 512 CTAs
// took 355 + 603).
constexpr int kKeys = 64;        // keys per tile
constexpr int kSLD = kD + 4;     // row stride of staged operands
constexpr int kScT = 256;

// rows x 128 values into shared memory as fp32, rows of `ld` floats; rows past
// `valid` become zeros.  fp32 rows go by cp.async (committed by the caller).
template <typename T>
__device__ __forceinline__ void stage_rows(float* dst, int ld, const T* src, int rows, int valid) {
  for (int i = threadIdx.x; i < rows * (kD / 4); i += kScT) {
    const int r = i / (kD / 4), t = i % (kD / 4) * 4;
    float* d = dst + r * ld + t;
    const size_t o = (size_t)r * kD + t;
    if (r >= valid) {
      *(float4*)d = make_float4(0.f, 0.f, 0.f, 0.f);
    } else if constexpr (std::is_same<T, float>::value) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(d)),
                   "l"(src + o));
    } else {
      const uint2 w = *(const uint2*)(src + o);
      *(float4*)d = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u),
                                __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xFFFF0000u));
    }
  }
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;"); }
template <int kPending>
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}

template <int RT>
__device__ __forceinline__ void logits_tile(const float* qs, const float* ks, float (*acc)[4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) acc[i][jj] = 0.f;
#pragma unroll 2
  for (int t = 0; t < kD; t += 4) {
    float4 qv[RT], kv[4];
#pragma unroll
    for (int i = 0; i < RT; ++i) qv[i] = *(const float4*)(qs + (ty * RT + i) * kSLD + t);
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) kv[jj] = *(const float4*)(ks + (tx + 16 * jj) * kSLD + t);
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        float c = acc[i][jj];
        c = fmaf(qv[i].x, kv[jj].x, c);
        c = fmaf(qv[i].y, kv[jj].y, c);
        c = fmaf(qv[i].z, kv[jj].z, c);
        acc[i][jj] = fmaf(qv[i].w, kv[jj].w, c);
      }
  }
}

// Merges two (max, sum of exp(l - max)) row statistics.
__device__ __forceinline__ float2 stat_merge(float2 x, float2 y) {
  if (y.x == -INFINITY) return x;
  if (y.x > x.x) return make_float2(y.x, x.y * expf(x.x - y.x) + y.y);
  return make_float2(x.x, x.y + y.y * expf(y.x - x.x));
}

template <int RT>
constexpr size_t stats_smem() {
  return (size_t)(16 * RT + 2 * kKeys) * kSLD * 4;
}
template <int RT>
constexpr size_t prob_smem() {
  // Q, two K tiles (the one in use becomes P), two V tiles, row statistics, column sums
  return ((size_t)(16 * RT + 2 * kKeys) * kSLD + 2 * kKeys * kD + 2 * 16 * RT + 16 * kKeys) * 4;
}

// ---------------------------------------------------------------- pass A --
// Row statistics of one chunk of keys: (max_j l_rj, sum_j exp(l_rj - max)).
template <typename T, int RT>
__global__ void __launch_bounds__(kScT, RT == 8 ? 1 : 2)
    k_stats_chunk(const T* __restrict__ q, const T* __restrict__ k, Shape s, int chunk, int nchunk,
                  float2* __restrict__ pstats) {
  extern __shared__ __align__(16) float sm[];
  constexpr int MR = 16 * RT;
  float* qs = sm;                   // [MR][kSLD]
  float* ks = qs + MR * kSLD;       // two tiles of [kKeys][kSLD]
  const int u = blockIdx.y, c = blockIdx.x;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int j0 = c * chunk, j1 = min(s.n, j0 + chunk);
  const T* ku = k + (size_t)u * s.n * kD;
  for (int row0 = 0; row0 < s.m; row0 += MR) {
    __syncthreads();
    stage_rows(qs, kSLD, q + ((size_t)u * s.m + row0) * kD, MR, s.m - row0);
    stage_rows(ks, kSLD, ku + (size_t)j0 * kD, kKeys, j1 - j0);
    stage_commit();
    float2 st[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) st[i] = make_float2(-INFINITY, 0.f);
    for (int base = j0, b = 0; base < j1; base += kKeys, b ^= 1) {
      if (base + kKeys < j1)
        stage_rows(ks + (b ^ 1) * kKeys * kSLD, kSLD, ku + (size_t)(base + kKeys) * kD, kKeys,
                   j1 - base - kKeys);
      stage_commit();
      stage_wait<1>();
      __syncthreads();
      float acc[RT][4];
      logits_tile<RT>(qs, ks + b * kKeys * kSLD, acc);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const int r = row0 + ty * RT + i;
        float l[4], mx = -INFINITY;
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int j = base + tx + 16 * jj;
          l[jj] = (j < j1 && visible(s, r, j)) ? s.scale * acc[i][jj] : -INFINITY;
          mx = fmaxf(mx, l[jj]);
        }
        if (mx == -INFINITY) continue;
        if (mx > st[i].x) {
          st[i].y *= expf(st[i].x - mx);
          st[i].x = mx;
        }
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) st[i].y += expf(l[jj] - st[i].x);
      }
      __syncthreads();   // the other buffer is refilled next
    }
    // a row's 16 threads are half a warp
#pragma unroll
    for (int i = 0; i < RT; ++i) {
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const float2 y = make_float2(__shfl_xor_sync(0xffffffffu, st[i].x, o),
                                     __shfl_xor_sync(0xffffffffu, st[i].y, o));
        st[i] = stat_merge(st[i], y);
      }
      const int r = row0 + ty * RT + i;
      if (tx == 0 && r < s.m) pstats[((size_t)u * nchunk + c) * s.m + r] = st[i];
    }
  }
}

// ---------------------------------------------------------------- pass B --
// Probabilities of one chunk: prefix scores (column sums over the m rows) and
// the chunk's share of Y = P V.  Each CTA combines the unit's row statistics
// itself; the first chunk's also writes them out.
template <typename T, int RT>
__global__ void __launch_bounds__(kScT, 1)
    k_prob_chunk(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v, Shape s,
                 int chunk, int nchunk, const float2* __restrict__ pstats,
                 float* __restrict__ row_stats, float* __restrict__ scores,
                 float* __restrict__ ypart) {
  chain_wait();
  extern __shared__ __align__(16) float sm[];
  constexpr int MR = 16 * RT;
  float* qs = sm;                            // [MR][kSLD]
  float* ks = qs + MR * kSLD;                // two tiles of [kKeys][kSLD]; then P [key][row]
  float* vs = ks + 2 * kKeys * kSLD;         // two tiles of [kKeys][kD]
  float2* st = (float2*)(vs + 2 * kKeys * kD);   // [MR] (M_r, L_r)
  float* cs = (float*)(st + MR);             // [16][kKeys] column sums of each ty
  const int u = blockIdx.y, c = blockIdx.x, tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int j0 = c * chunk, j1 = min(s.n, j0 + chunk);
  const T* ku = k + (size_t)u * s.n * kD;
  const T* vu = v + (size_t)u * s.n * kD;
  for (int row0 = 0; row0 < s.m; row0 += MR) {
    __syncthreads();
    auto stage_tile = [&](int base, int b) {
      stage_rows(ks + b * kKeys * kSLD, kSLD, ku + (size_t)base * kD, kKeys, j1 - base);
      stage_rows(vs + b * kKeys * kD, kD, vu + (size_t)base * kD, kKeys, j1 - base);
    };
    stage_rows(qs, kSLD, q + ((size_t)u * s.m + row0) * kD, MR, s.m - row0);
    stage_tile(j0, 0);
    stage_commit();
    for (int r = tid; r < MR; r += kScT) {
      float2 x = make_float2(-INFINITY, 0.f);
      if (row0 + r < s.m) {
#pragma unroll 8
        for (int h = 0; h < nchunk; ++h)
          x = stat_merge(x, pstats[((size_t)u * nchunk + h) * s.m + row0 + r]);
        if (c == 0) *(float2*)(row_stats + ((size_t)u * s.m + row0 + r) * 2) = x;
      }
      st[r] = x;
    }
    float y[RT][8];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int e = 0; e < 8; ++e) y[i][e] = 0.f;
    for (int base = j0, b = 0; base < j1; base += kKeys, b ^= 1) {
      if (base + kKeys < j1) stage_tile(base + kKeys, b ^ 1);
      stage_commit();
      stage_wait<1>();
      __syncthreads();
      float* kt = ks + b * kKeys * kSLD;
      float acc[RT][4];
      logits_tile<RT>(qs, kt, acc);
      __syncthreads();   // K is used up: its buffer takes P
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const int r = row0 + ty * RT + i;
        const float2 ml = st[ty * RT + i];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int j = base + tx + 16 * jj;
          float p = 0.f;
          if (r < s.m && j < j1 && visible(s, r, j)) p = expf(s.scale * acc[i][jj] - ml.x) / ml.y;
          kt[(tx + 16 * jj) * kSLD + ty * RT + i] = p;
          sum[jj] += p;
        }
      }
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) cs[ty * kKeys + tx + 16 * jj] = sum[jj];
      __syncthreads();
      if (tid < kKeys && base + tid < min(j1, s.P)) {
        float t = 0.f;
#pragma unroll
        for (int g = 0; g < 16; ++g) t += cs[g * kKeys + tid];
        float* o = scores + (size_t)u * s.P + base + tid;
        *o = row0 ? *o + t : t;   // the same thread wrote the earlier rows' sum
      }
      const float* vt = vs + b * kKeys * kD;
#pragma unroll 4
      for (int jj = 0; jj < kKeys; ++jj) {
        const float4 v0 = *(const float4*)(vt + jj * kD + tx * 4);
        const float4 v1 = *(const float4*)(vt + jj * kD + 64 + tx * 4);
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const float p = kt[jj * kSLD + ty * RT + i];
          y[i][0] = fmaf(p, v0.x, y[i][0]);
          y[i][1] = fmaf(p, v0.y, y[i][1]);
          y[i][2] = fmaf(p, v0.z, y[i][2]);
          y[i][3] = fmaf(p, v0.w, y[i][3]);
          y[i][4] = fmaf(p, v1.x, y[i][4]);
          y[i][5] = fmaf(p, v1.y, y[i][5]);
          y[i][6] = fmaf(p, v1.z, y[i][6]);
          y[i][7] = fmaf(p, v1.w, y[i][7]);
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int r = row0 + ty * RT + i;
      if (r >= s.m) break;
      float* o = ypart + (((size_t)u * nchunk + c) * s.m + r) * kD + tx * 4;
      *(float4*)o = make_float4(y[i][0], y[i][1], y[i][2], y[i][3]);
      *(float4*)(o + 64) = make_float4(y[i][4], y[i][5], y[i][6], y[i][7]);
    }
  }
}

// Y = sum of the chunks' shares, in chunk order; one float4 per thread.
__global__ void __launch_bounds__(256) k_y_reduce(const float4* __restrict__ ypart, Shape s,
                                                  int nchunk, float4* __restrict__ y) {
  chain_wait();
  const int u = blockIdx.y, md = s.m * (kD / 4), i = blockIdx.x * 256 + threadIdx.x;
  if (i >= md) return;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
  for (int c = 0; c < nchunk; ++c) {
    const float4 x = ypart[((size_t)u * nchunk + c) * md + i];
    a.x += x.x;
    a.y += x.y;
    a.z += x.z;
    a.w += x.w;
  }
  y[(size_t)u * md + i] = a;
}

template <typename T, int RT>
cudaError_t score_impl(const Shape& s, const T* q, const T* k, const T* v, float* scores,
                       float* y, float* row_stats, char* ws, const WsLayout& L,
                       cudaStream_t st) {
  float2* pstats = (float2*)(ws + L.pstats);
  float* ypart = (float*)(ws + L.ypart);
  constexpr size_t smA = stats_smem<RT>(), smB = prob_smem<RT>();
  cudaError_t e = cudaFuncSetAttribute(k_stats_chunk<T, RT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smA);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_prob_chunk<T, RT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smB);
  if (e != cudaSuccess) return e;
  const dim3 grid(L.nchunk, s.U);
  k_stats_chunk<T, RT><<<grid, kScT, smA, st>>>(q, k, s, L.chunk, L.nchunk, pstats);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = launch_kernel(true, 1, k_prob_chunk<T, RT>, grid, kScT, smB, st, q, k, v, s, L.chunk, L.nchunk,
                    (const float2*)pstats, row_stats, scores, ypart);
  if (e != cudaSuccess) return e;
  e = launch_kernel(true, 1, k_y_reduce, dim3((s.m * (kD / 4) + 255) / 256, s.U), 256, 0, st,
                    (const float4*)ypart, s, L.nchunk, (float4*)y);
  count_launches(3);
  return e;
}

// The row tile follows m: 32 or 64 rows at a time waste less of it.
template <typename T>
cudaError_t score_rows(const Shape& s, const T* q, const T* k, const T* v, float* scores, float* y,
                       float* row_stats, char* ws, const WsLayout& L, cudaStream_t st) {
  if (s.m <= 32) return score_impl<T, 2>(s, q, k, v, scores, y, row_stats, ws, L, st);
  if (s.m <= 64) return score_impl<T, 4>(s, q, k, v, scores, y, row_stats, ws, L, st);
  return score_impl<T, 8>(s, q, k, v, scores, y, row_stats, ws, L, st);
}

}  // namespace

cudaError_t launch_score_simt(const Shape& s, const void* q, const void* k, const void* v,
                              float* scores, float* y, float* row_stats, char* ws,
                              const WsLayout& L, cudaStream_t st) {
  if (s.dtype == GRKV_F32)
    return score_rows<float>(s, (const float*)q, (const float*)k, (const float*)v, scores, y,
                             row_stats, ws, L, st);
  return score_rows<__nv_bfloat16>(s, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k,
                                   (const __nv_bfloat16*)v, scores, y, row_stats, ws, L, st);
}

// Keys per CTA of the portable scoring passes: whole tiles of 64, so that the
// U x chunks CTAs (one per SM at a time) finish soonest, a CTA costing its
// tiles plus about two tiles of set-up.
// One chunk count is tried per chunk size: the smallest that gives it.
int score_simt_chunk(const Shape& s) {
  const int tiles = (s.n + kKeys - 1) / kKeys, sms = 152;
  const long long U = std::max(s.U, 1);
  long long cost = -1;
  int best = 1;
  for (int chunks = 1; chunks <= std::min(tiles, 608);) {
    const int per = (tiles + chunks - 1) / chunks, used = (tiles + per - 1) / per;
    const long long c = (U * used + sms - 1) / sms * (per + 2);
    if (cost < 0 || c < cost) {
      cost = c;
      best = per;
    }
    if (per == 1) break;
    chunks = (tiles + per - 2) / (per - 1);   // the first with smaller chunks
  }
  return best * kKeys;
}

}  // namespace grkv
