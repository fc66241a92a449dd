// The value step's fp32 solve Z = (sym(G) + lambda I)^-1 R for m <= 256 (bf16
// inputs on either path; R has 128 columns).
//
// For m <= 128 one CTA holds the augmented matrix [N | R] in registers: 136
// threads own the lower triangle of N as 8 x 8 tiles, 256 own R as tiles of 8
// rows.  Step k of 16 factors the diagonal tile in the thread that owns it,
// solves the panel below it and takes the rank-8 update out of the later tiles of
// N; L goes to shared memory.  The owners of R follow behind, a step at a
// time as panels appear: W_k = L_kk^-1 R_k, then its rank-8 update; then they
// run the backward pass alone.  Bound by the chain of short steps (diagonal
// tile, panel, update; then 16 backward steps), not by its 2.3 M FMAs.  With
// few units the columns of R are split over up to four CTAs that each factor
// N again: narrower tiles of R shorten its steps, on SMs that would idle.
//
// For 128 < m <= 256 the matrix is taken in two row blocks:
// N = [A B^T; B C]: k_solve_first factors A and forms W_B = L_A^-1 B^T and
// W_0 = L_A^-1 R_0; k_solve_second factors C - W_B^T W_B, solves for Z_1, then
// Z_0 = L_A^-T (W_0 - W_B Z_1).
//
// A non-positive pivot reports GRKV_ERR_NUMERIC and gives Z = 0 (values stay V0), as does
// lambda = +inf without a report.
#include <cmath>

#include "grkv_internal.cuh"
#include "sm100.cuh"

namespace grkv {
namespace {

using namespace sm100;

// named_bar for warps whose lanes may have diverged before it
__device__ __forceinline__ void group_bar(uint32_t id, uint32_t nthreads) {
  __syncwarp();
  named_bar(id, nthreads);
}

constexpr int kSB = 128;                    // rows of a block
constexpr int kT = 8;                       // tile edge
constexpr int kNT = kSB / kT;               // tile rows
constexpr int kTri = kNT * (kNT + 1) / 2;   // threads that own a tile of N
constexpr int kNThreads = (kTri + 31) / 32 * 32;
constexpr int kRThreads = 256;              // 16 tile rows x 16 tile columns of R
constexpr int kThreads = kNThreads + kRThreads;
constexpr long long kWaitBudget = 1ll << 32;   // clock cycles of a bounded wait

struct SolveArgs {
  float* gram;        // [U][ld][ld]
  float* rz;          // [U][ld][128]  R in, Z out
  float* fac;         // m > 128: L_A by columns, fac + u fac_unit + col fac_ld + row
  size_t fac_unit;
  int fac_ld;
  int* fail;          // m > 128: [U] set when A has no factor
  int m, ld, sym, lambda_inf;
  float lambda;
  int* status;
};

// Shared memory: L by columns (the diagonal holds 1 / L_jj), two buffers for
// the rows W_k / Z_k of a step, a barrier per panel, and the failure flag.
struct alignas(16) SolveSmem {
  float L[kSB][kSB];
  float w[2][kT][kSB];
  uint64_t panel[kNT];   // panel k of L is complete
  int fail;
  int abort;
};

__device__ __forceinline__ void solve_init(SolveSmem& s, int failed) {
  if (threadIdx.x == 0) {
    for (int k = 0; k < kNT; ++k) mbar_init(&s.panel[k], 1);
    s.fail = failed;
    s.abort = 0;
    fence_mbar_init();
  }
  __syncthreads();
}

// The tile of N of thread i < kTri: by columns, so that whole warps finish early.
__device__ __forceinline__ void n_tile(int i, int& ty, int& tx) {
  int c = 0;
  while (i >= kNT - c) {
    i -= kNT - c;
    ++c;
  }
  tx = c;
  ty = c + i;
}

// kW contiguous floats.  The columns of a tile of R are split in groups of (up
// to) four, 16 groups apart, so that a warp's 16-byte accesses to a row are
// contiguous: column e of tile column tx is at 64 (e / 4) + 4 tx + e % 4.
template <int kW>
__device__ __forceinline__ void ldw(const float* p, float* v) {
  if constexpr (kW == 2) {
    const float2 a = *(const float2*)p;
    v[0] = a.x; v[1] = a.y;
  } else {
    const float4 a = *(const float4*)p;
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  }
}
template <int kW>
__device__ __forceinline__ void stw(float* p, const float* v) {
  if constexpr (kW == 2)
    *(float2*)p = make_float2(v[0], v[1]);
  else
    *(float4*)p = make_float4(v[0], v[1], v[2], v[3]);
}
template <int kTC>
struct RCols {
  static constexpr int kW = kTC < 4 ? kTC : 4, kG = kTC / kW;
  static __device__ __forceinline__ void load(const float* row, int tx, float* v) {
#pragma unroll
    for (int g = 0; g < kG; ++g) ldw<kW>(row + 16 * kW * g + kW * tx, v + kW * g);
  }
  static __device__ __forceinline__ void store(float* row, int tx, const float* v) {
#pragma unroll
    for (int g = 0; g < kG; ++g) stw<kW>(row + 16 * kW * g + kW * tx, v + kW * g);
  }
  static __device__ __forceinline__ int col(int tx, int e) { return 16 * kW * (e / kW) + kW * tx + e % kW; }
};

__device__ __forceinline__ void ld8s(const float* p, float* v) {
  ldw<4>(p, v);
  ldw<4>(p + 4, v + 4);
}
__device__ __forceinline__ void st8s(float* p, const float* v) {
  stw<4>(p, v);
  stw<4>(p + 4, v + 4);
}

// x[i][j] -= sum_c p[c ps + i] q(c)[j] over `depth` rows; q loads row c.
template <int kTC, class Q>
__device__ __forceinline__ void tile_update(float (*x)[kTC], const float* p, int ps, int depth, Q q) {
#pragma unroll 2
  for (int c = 0; c < depth; ++c) {
    float pv[kT], qv[kTC];
    ld8s(p + c * ps, pv);
    q(c, qv);
#pragma unroll
    for (int i = 0; i < kT; ++i)
#pragma unroll
      for (int j = 0; j < kTC; ++j) x[i][j] = fmaf(-pv[i], qv[j], x[i][j]);
  }
}

// Factors nb tile columns of N: the owners of N (barrier 1).
__device__ void factor(SolveSmem& s, bool mine, int ty, int tx, float (*x)[kT], int nb) {
  for (int k = 0; k < nb; ++k) {
    const int k0 = k * kT;
    if (mine && tx == k && ty == k) {
      bool bad = false;
#pragma unroll
      for (int c = 0; c < kT; ++c) {
        const float d = x[c][c];
        bad |= !(d > 0.f);
        const float inv = d > 0.f ? rsqrtf(d) : 0.f;
        x[c][c] = inv;
#pragma unroll
        for (int i = c + 1; i < kT; ++i) x[i][c] *= inv;
#pragma unroll
        for (int j = c + 1; j < kT; ++j)
#pragma unroll
          for (int i = j; i < kT; ++i) x[i][j] = fmaf(-x[i][c], x[j][c], x[i][j]);
      }
#pragma unroll
      for (int c = 0; c < kT; ++c) {
        float col[kT];
#pragma unroll
        for (int i = 0; i < kT; ++i) col[i] = i >= c ? x[i][c] : 0.f;
        st8s(&s.L[k0 + c][k0], col);
      }
      if (bad) s.fail = 1;
    }
    group_bar(1, kNThreads);
    if (mine && tx == k && ty > k) {
      // rows of the panel: L_ik = A_ik L_kk^-T
#pragma unroll
      for (int c = 0; c < kT; ++c) {
        float l[kT];
        ld8s(&s.L[k0 + c][k0], l);
#pragma unroll
        for (int i = 0; i < kT; ++i) x[i][c] *= l[c];
#pragma unroll
        for (int j = c + 1; j < kT; ++j)
#pragma unroll
          for (int i = 0; i < kT; ++i) x[i][j] = fmaf(-x[i][c], l[j], x[i][j]);
      }
#pragma unroll
      for (int c = 0; c < kT; ++c) {
        float col[kT];
#pragma unroll
        for (int i = 0; i < kT; ++i) col[i] = x[i][c];
        st8s(&s.L[k0 + c][ty * kT], col);
      }
    }
    group_bar(1, kNThreads);
    if (threadIdx.x == kNThreads - 1) mbar_arrive(&s.panel[k]);
    if (mine && tx > k)
      tile_update<kT>(x, &s.L[k0][ty * kT], kSB, kT,
                      [&](int c, float* q) { ld8s(&s.L[k0 + c][tx * kT], q); });
  }
}

// W = L^-1 R over nb tile rows: the owners of R (barrier 2), behind factor().
template <int kTC>
__device__ void forward(SolveSmem& s, int ty, int tx, float (*x)[kTC], int nb, int* status) {
  for (int k = 0; k < nb; ++k) {
    const int k0 = k * kT;
    if (!mbar_wait(&s.panel[k], 0, &s.abort, kWaitBudget)) set_status(status, GRKV_ERR_TIMEOUT);
    float(*w)[kSB] = s.w[k & 1];
    if (ty == k) {
#pragma unroll
      for (int c = 0; c < kT; ++c) {
        float l[kT];
        ld8s(&s.L[k0 + c][k0], l);
#pragma unroll
        for (int j = 0; j < kTC; ++j) x[c][j] *= l[c];
#pragma unroll
        for (int i = c + 1; i < kT; ++i)
#pragma unroll
          for (int j = 0; j < kTC; ++j) x[i][j] = fmaf(-l[i], x[c][j], x[i][j]);
      }
#pragma unroll
      for (int i = 0; i < kT; ++i) RCols<kTC>::store(w[i], tx, x[i]);
    }
    group_bar(2, kRThreads);
    if (ty > k)
      tile_update<kTC>(x, &s.L[k0][ty * kT], kSB, kT,
                       [&](int c, float* q) { RCols<kTC>::load(w[c], tx, q); });
  }
}

// W -> Z = L^-T W over nb tile rows: the owners of R.
template <int kTC>
__device__ void backward(SolveSmem& s, int ty, int tx, float (*x)[kTC], int nb) {
  group_bar(2, kRThreads);   // both w buffers are free
  for (int k = nb - 1; k >= 0; --k) {
    const int k0 = k * kT;
    float(*w)[kSB] = s.w[k & 1];
    if (ty == k) {
#pragma unroll
      for (int c = kT - 1; c >= 0; --c) {
        float l[kT];
        ld8s(&s.L[k0 + c][k0], l);   // column c: rows c + 1 .. 7 below the diagonal
#pragma unroll
        for (int i = c + 1; i < kT; ++i)
#pragma unroll
          for (int j = 0; j < kTC; ++j) x[c][j] = fmaf(-l[i], x[i][j], x[c][j]);
#pragma unroll
        for (int j = 0; j < kTC; ++j) x[c][j] *= l[c];
      }
#pragma unroll
      for (int i = 0; i < kT; ++i) RCols<kTC>::store(w[i], tx, x[i]);
    }
    group_bar(2, kRThreads);
    if (ty < k) {
      // four rows of Z_k at a time: L[k0 + r][8 ty + i] is row r of column 8 ty + i
#pragma unroll
      for (int h = 0; h < kT; h += 4) {
        float z[4][kTC];
#pragma unroll
        for (int r = 0; r < 4; ++r) RCols<kTC>::load(w[h + r], tx, z[r]);
#pragma unroll
        for (int i = 0; i < kT; ++i) {
          float l[4];
          ldw<4>(&s.L[ty * kT + i][k0 + h], l);
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < kTC; ++j) x[i][j] = fmaf(-l[r], z[r][j], x[i][j]);
        }
      }
    }
  }
}

// A tile of the diagonal block of N that starts at row r0 (identity past m).
__device__ __forceinline__ void load_n(const SolveArgs& a, const float* G, int r0, int ty, int tx,
                                       float (*x)[kT]) {
  const int i0 = r0 + ty * kT, j0 = r0 + tx * kT;
  if ((a.ld & 3) == 0 && i0 + kT <= a.m) {   // j0 <= i0: a whole tile, 16-byte rows
#pragma unroll
    for (int i = 0; i < kT; ++i) ld8s(G + (size_t)(i0 + i) * a.ld + j0, x[i]);
    if (a.sym) {
      float y[kT][kT];
#pragma unroll
      for (int j = 0; j < kT; ++j) ld8s(G + (size_t)(j0 + j) * a.ld + i0, y[j]);
#pragma unroll
      for (int i = 0; i < kT; ++i)
#pragma unroll
        for (int j = 0; j < kT; ++j)
          x[i][j] = i0 + i == j0 + j ? x[i][j] + a.lambda : 0.5f * (x[i][j] + y[j][i]);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < kT; ++i)
#pragma unroll
    for (int j = 0; j < kT; ++j) {
      const int r = i0 + i, c = j0 + j;
      float v = r == c ? 1.f : 0.f;
      if (r < a.m && c < a.m) {
        v = G[(size_t)r * a.ld + c];
        if (a.sym) v = r == c ? v + a.lambda : 0.5f * (v + G[(size_t)c * a.ld + r]);
      }
      x[i][j] = v;
    }
}

// A tile of a row-major array of `rows` x `cols` (zeros past them).
template <int kTC>
__device__ __forceinline__ void load_r(const float* src, int ld, int rows, int cols, int ty, int tx,
                                       float (*x)[kTC]) {
  using C = RCols<kTC>;
  const bool whole = (ld & 3) == 0 && cols >= 16 * kTC;
#pragma unroll
  for (int i = 0; i < kT; ++i) {
    const int r = ty * kT + i;
    const float* row = src + (size_t)r * ld;
    if (whole && r < rows) {
      C::load(row, tx, x[i]);
    } else {
#pragma unroll
      for (int e = 0; e < kTC; ++e)
        x[i][e] = r < rows && C::col(tx, e) < cols ? row[C::col(tx, e)] : 0.f;
    }
  }
}
template <int kTC>
__device__ __forceinline__ void store_r(float* dst, int ld, int rows, int cols, int ty, int tx,
                                        const float (*x)[kTC]) {
  using C = RCols<kTC>;
  const bool whole = (ld & 3) == 0 && cols >= 16 * kTC;
#pragma unroll
  for (int i = 0; i < kT; ++i) {
    const int r = ty * kT + i;
    if (r >= rows) break;
    float* row = dst + (size_t)r * ld;
    if (whole) {
      C::store(row, tx, x[i]);
    } else {
#pragma unroll
      for (int e = 0; e < kTC; ++e)
        if (C::col(tx, e) < cols) row[C::col(tx, e)] = x[i][e];
    }
  }
}
template <int kTC>
__device__ __forceinline__ void zero_tile(float (*x)[kTC]) {
#pragma unroll
  for (int i = 0; i < kT; ++i)
#pragma unroll
    for (int j = 0; j < kTC; ++j) x[i][j] = 0.f;
}

// m <= 128; kCols columns of R per CTA.
template <int kCols>
__global__ void __launch_bounds__(kThreads, 1) k_solve(SolveArgs a) {
  chain_wait();
  extern __shared__ __align__(16) float sm[];
  SolveSmem& s = *(SolveSmem*)sm;
  constexpr int kSplit = kD / kCols, kTC = kCols / 16;
  const int u = blockIdx.x / kSplit, c0 = blockIdx.x % kSplit * kCols;
  const int nb = (a.m + kT - 1) / kT;
  float* rz = a.rz + (size_t)u * a.ld * kD + c0;
  solve_init(s, 0);
  if (threadIdx.x < kNThreads) {
    if (!a.lambda_inf) {
      const bool mine = threadIdx.x < kTri;
      int ty = 0, tx = 0;
      float x[kT][kT];
      if (mine) {
        n_tile(threadIdx.x, ty, tx);
        load_n(a, a.gram + (size_t)u * a.ld * a.ld, 0, ty, tx, x);
      }
      factor(s, mine, ty, tx, x, nb);
    }
    __syncthreads();
  } else {
    const int i = threadIdx.x - kNThreads, ty = i >> 4, tx = i & 15;
    float x[kT][kTC];
    if (!a.lambda_inf) {
      load_r<kTC>(rz, kD, a.m, kCols, ty, tx, x);
      forward<kTC>(s, ty, tx, x, nb, a.status);
    }
    __syncthreads();   // s.fail settles
    if (a.lambda_inf || s.fail) {
      if (i == 0 && !a.lambda_inf) set_status(a.status, GRKV_ERR_NUMERIC);
      zero_tile<kTC>(x);
    } else {
      backward<kTC>(s, ty, tx, x, nb);
    }
    store_r<kTC>(rz, kD, a.m, kCols, ty, tx, x);
  }
}

// m > 128, first row block: four CTAs per unit, W_B = L_A^-1 B^T over the
// halves of the cross block of G and W_0 = L_A^-1 R_0 over those of R_0; the
// last also leaves L_A.
constexpr int kCols2 = 64, kTC2 = kCols2 / 16;
__global__ void __launch_bounds__(kThreads, 1) k_solve_first(SolveArgs a) {
  chain_wait();
  extern __shared__ __align__(16) float sm[];
  SolveSmem& s = *(SolveSmem*)sm;
  const int u = blockIdx.x >> 2, which = blockIdx.x & 3;
  float* G = a.gram + (size_t)u * a.ld * a.ld;
  solve_init(s, 0);
  if (threadIdx.x < kNThreads) {
    const bool mine = threadIdx.x < kTri;
    int ty = 0, tx = 0;
    float x[kT][kT];
    if (mine) {
      n_tile(threadIdx.x, ty, tx);
      load_n(a, G, 0, ty, tx, x);
    }
    factor(s, mine, ty, tx, x, kNT);
  } else {
    const int i = threadIdx.x - kNThreads, ty = i >> 4, tx = i & 15;
    const int c0 = (which & 1) * kCols2;
    float* rhs = (which & 2 ? a.rz + (size_t)u * a.ld * kD : G + kSB) + c0;
    const int ldr = which & 2 ? kD : a.ld, cols = (which & 2 ? kD : a.m - kSB) - c0;
    float x[kT][kTC2];
    load_r<kTC2>(rhs, ldr, kSB, cols, ty, tx, x);
    forward<kTC2>(s, ty, tx, x, kNT, a.status);
    store_r<kTC2>(rhs, ldr, kSB, cols, ty, tx, x);
  }
  __syncthreads();
  if (which == 3) {
    if (threadIdx.x == 0) a.fail[u] = s.fail;
    float* f = a.fac + u * a.fac_unit;
    for (int i = threadIdx.x; i < kSB * kSB; i += kThreads)   // whole tiles of the lower triangle
      if (i % kSB >= i / kSB / kT * kT) f[(size_t)(i / kSB) * a.fac_ld + i % kSB] = s.L[i / kSB][i % kSB];
  }
}

struct SecondSmem {
  SolveSmem s;
  float wb[kSB][kSB];   // W_B by rows, read 16 bytes at a time
};
static_assert(offsetof(SecondSmem, wb) % 16 == 0, "float4 rows");

// m > 128, second row block and the backward pass of the first; two CTAs per
// unit, 64 columns of R each.
__global__ void __launch_bounds__(kThreads, 1) k_solve_second(SolveArgs a) {
  chain_wait();
  extern __shared__ __align__(16) float sm[];
  SecondSmem& q = *(SecondSmem*)sm;
  SolveSmem& s = q.s;
  const int u = blockIdx.x >> 1, c0 = (blockIdx.x & 1) * kCols2;
  const int m1 = a.m - kSB, nb = (m1 + kT - 1) / kT;
  float* G = a.gram + (size_t)u * a.ld * a.ld;
  float* rz0 = a.rz + (size_t)u * a.ld * kD + c0;
  float* rz1 = rz0 + (size_t)kSB * kD;
  const bool first_failed = __ldg(a.fail + u) != 0;
  solve_init(s, first_failed);
  float* w0 = &s.L[0][0];   // W_0 [128][64], until L is written
#pragma unroll 4
  for (int i = threadIdx.x; i < kSB * kSB; i += kThreads)
    q.wb[i / kSB][i % kSB] = i % kSB < m1 ? G[(size_t)(i / kSB) * a.ld + kSB + i % kSB] : 0.f;
#pragma unroll 4
  for (int i = threadIdx.x; i < kSB * kCols2; i += kThreads)
    w0[i] = rz0[(size_t)(i / kCols2) * kD + i % kCols2];
  __syncthreads();
  const bool is_n = threadIdx.x < kNThreads, mine = threadIdx.x < kTri;
  const int i = threadIdx.x - kNThreads;
  int ty = i >> 4, tx = i & 15;
  float xr[kT][kTC2];
  if (!is_n) {
    load_r<kTC2>(rz1, kD, m1, kCols2, ty, tx, xr);
    tile_update<kTC2>(xr, &q.wb[0][ty * kT], kSB, kSB,
                      [&](int c, float* v) { RCols<kTC2>::load(w0 + c * kCols2, tx, v); });
  }
  __syncthreads();   // W_0's place is L's now
  if (is_n) {
    if (!first_failed) {
      float x[kT][kT];
      if (mine) {
        n_tile(threadIdx.x, ty, tx);
        load_n(a, G, kSB, ty, tx, x);
        tile_update<kT>(x, &q.wb[0][ty * kT], kSB, kSB,
                        [&](int c, float* v) { ld8s(&q.wb[c][tx * kT], v); });
      }
      factor(s, mine, ty, tx, x, nb);
    }
  } else if (!first_failed) {
    forward<kTC2>(s, ty, tx, xr, nb, a.status);
  }
  __syncthreads();   // s.fail settles
  const bool failed = s.fail;
  if (!is_n) {
    if (failed) {
      if (i == 0) set_status(a.status, GRKV_ERR_NUMERIC);
      zero_tile<kTC2>(xr);
    } else {
      backward<kTC2>(s, ty, tx, xr, nb);
    }
    store_r<kTC2>(rz1, kD, m1, kCols2, ty, tx, xr);
    if (failed) store_r<kTC2>(rz0, kD, kSB, kCols2, ty, tx, xr);
  }
  if (failed) return;   // the same in all threads
  __syncthreads();      // L is spent: Z_1 by rows takes its place
  float* z1 = &s.L[0][0];   // [128][64]
  if (!is_n) {
    if (ty >= nb) zero_tile<kTC2>(xr);
#pragma unroll
    for (int r = 0; r < kT; ++r) RCols<kTC2>::store(z1 + (ty * kT + r) * kCols2, tx, xr[r]);
  }
  __syncthreads();
  if (!is_n) {
    load_r<kTC2>(rz0, kD, kSB, kCols2, ty, tx, xr);
    // W_0 - W_B Z_1, four columns of W_B at a time
#pragma unroll 2
    for (int c = 0; c < nb * kT; c += 4) {
      float z[4][kTC2];
#pragma unroll
      for (int e = 0; e < 4; ++e) RCols<kTC2>::load(z1 + (c + e) * kCols2, tx, z[e]);
#pragma unroll
      for (int r = 0; r < kT; ++r) {
        float w[4];
        ldw<4>(&q.wb[ty * kT + r][c], w);
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int j = 0; j < kTC2; ++j) xr[r][j] = fmaf(-w[e], z[e][j], xr[r][j]);
      }
    }
  }
  __syncthreads();
  const float* f = a.fac + u * a.fac_unit;
#pragma unroll 4
  for (int e = threadIdx.x; e < kSB * kSB; e += kThreads)
    if (e % kSB >= e / kSB / kT * kT) s.L[e / kSB][e % kSB] = __ldg(f + (size_t)(e / kSB) * a.fac_ld + e % kSB);
  __syncthreads();
  if (!is_n) {
    backward<kTC2>(s, ty, tx, xr, kNT);
    store_r<kTC2>(rz0, kD, kSB, kCols2, ty, tx, xr);
  }
}

__global__ void k_zero_rows(float4* __restrict__ p, size_t count) {
  chain_wait();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (size_t)gridDim.x * blockDim.x)
    p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

template <typename K>
cudaError_t run(K kern, unsigned grid, size_t smem, const SolveArgs& a, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  count_launches(1);
  return launch_kernel(true, 1, kern, dim3(grid), kThreads, smem, st, a);
}

}  // namespace

// The columns of R are split while that leaves one CTA per SM of a GB300.
cudaError_t launch_solve(int U, int m, int ld, int sym, float lambda, int lambda_inf, float* gram,
                         float* rz, float* fac, size_t fac_unit, int fac_ld, int* fail,
                         int* status, cudaStream_t st) {
  SolveArgs a{gram, rz, fac, fac_unit, fac_ld, fail, m, ld, sym, lambda_inf, lambda, status};
  if (m > kMaxM || ld < m) return cudaErrorInvalidValue;
  const unsigned n = (unsigned)U;
  if (m <= kSB) {
    if (U <= 38) return run(k_solve<32>, n * 4, sizeof(SolveSmem), a, st);
    if (U <= 76) return run(k_solve<64>, n * 2, sizeof(SolveSmem), a, st);
    return run(k_solve<128>, n, sizeof(SolveSmem), a, st);
  }
  if (lambda_inf) {
    count_launches(1);
    return launch_kernel(true, 1, k_zero_rows, dim3(608), 256, 0, st, (float4*)rz,
                         (size_t)U * ld * (kD / 4));
  }
  cudaError_t e = run(k_solve_first, n * 4, sizeof(SolveSmem), a, st);
  if (e != cudaSuccess) return e;
  return run(k_solve_second, n * 2, sizeof(SecondSmem), a, st);
}

}  // namespace grkv
