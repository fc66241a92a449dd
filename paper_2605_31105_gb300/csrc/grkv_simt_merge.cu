// The value step on CUDA cores: fp32 inputs, and bf16 inputs under
// GRKV_FORCE_SIMT (m <= 256, any B).
//
// For fp32 inputs the regression (R, the Gram, the Cholesky factor, Z and the
// update) carries about twice fp32's precision.  GB300 issues 2 fp64 FMAs per
// SM and clock against 128 in fp32, so the products run as pairs of floats
// (Df): each product is exact (two_prod), sums keep their rounding errors
// (two_sum), 10 to 12 fp32 instructions per multiply-add, about 2^-46 relative.  A
// unit that needs more (a pivot far below its diagonal, residuals or a Z near the ends of
// fp32's range) is solved again in fp64 (k_simt_solve64).
//
// One CTA per unit and fp64 took 19.3 ms for 8 units of m = 128, B = 512 and
// 1.78 ms for one unit of m = 32, B = 256; the work is now cut into tiles over
// the whole GPU:
//   k_simt_logits   s Q K0^T in 32 x 32 tiles, K_out = K0, and in one more CTA
//                   per unit the fixed set
//   k_simt_softmax  row softmax over the retained keys, one warp per row
//   k_simt_regr     R = Y - X V0 and N = X_G X_G^T + lambda I, 8 x 32 tiles
//   k_simt_chol     Cholesky of N, one CTA per unit, diagonal blocks inverted
//   k_simt_subst    Z = N^-1 R, 8 columns per CTA
//   k_simt_solve64  units left to fp64
//   k_simt_update   V_out = V0 + X_G^T Z in 32 x 32 tiles
// bf16 inputs run the same tiles with plain fp32 sums and the blocked fp32
// solve (grkv_solve.cu).
#include <cmath>
#include <type_traits>

#include "block_select.cuh"
#include "simt_common.cuh"

namespace grkv {
namespace {

// ---------------------------------------------------- pairs of floats --
// Knuth's two-sum and the FMA two-product; the intrinsics keep the compiler
// from contracting them.
struct alignas(8) Df {
  float hi, lo;
};

__device__ __forceinline__ Df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ Df quick_two_sum(float a, float b) {   // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
// acc += a b, the low part left unnormalised
__device__ __forceinline__ void df_mac(Df& acc, float a, float b) {
  const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
  const Df t = two_sum(acc.hi, p);
  acc.hi = t.hi;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(t.lo, e));
}
__device__ __forceinline__ void df_mac(Df& acc, float a, Df b) {
  const float p = __fmul_rn(a, b.hi), e = __fmaf_rn(a, b.lo, __fmaf_rn(a, b.hi, -p));
  const Df t = two_sum(acc.hi, p);
  acc.hi = t.hi;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(t.lo, e));
}
__device__ __forceinline__ void df_mac(Df& acc, Df a, Df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -p)));
  const Df t = two_sum(acc.hi, p);
  acc.hi = t.hi;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(t.lo, e));
}
__device__ __forceinline__ Df df_norm(Df a) { return quick_two_sum(a.hi, a.lo); }
__device__ __forceinline__ Df df_neg(Df a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ Df df_mul(Df a, Df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -p)));
  return quick_two_sum(p, e);
}
// Square root and reciprocal: the fp32 value and one Newton step on it.
__device__ __forceinline__ Df df_sqrt(Df d) {
  const float x = sqrtf(d.hi);
  const float r = __fadd_rn(__fmaf_rn(-x, x, d.hi), d.lo);
  return quick_two_sum(x, r / (2.f * x));
}
__device__ __forceinline__ Df df_rcp(Df d) {
  const float x = 1.f / d.hi;
  const float r = __fmaf_rn(-x, d.lo, __fmaf_rn(-x, d.hi, 1.f));
  return quick_two_sum(x, __fmul_rn(x, r));
}

// Accumulator policies: Df for fp32 inputs, float for bf16.
__device__ __forceinline__ void mac(Df& a, float x, float y) { df_mac(a, x, y); }
__device__ __forceinline__ void mac(float& a, float x, float y) { a = fmaf(x, y, a); }
__device__ __forceinline__ void mac(Df& a, float x, Df y) { df_mac(a, x, y); }
__device__ __forceinline__ void zero(Df& a) { a = {0.f, 0.f}; }
__device__ __forceinline__ void zero(float& a) { a = 0.f; }
__device__ __forceinline__ Df minus(float y, Df a) {   // y - a
  Df t = two_sum(y, -a.hi);
  return df_norm({t.hi, __fsub_rn(t.lo, a.lo)});
}
__device__ __forceinline__ float minus(float y, float a) { return y - a; }
__device__ __forceinline__ Df plus(Df a, float y) {
  Df t = two_sum(a.hi, y);
  return df_norm({t.hi, __fadd_rn(t.lo, a.lo)});
}
__device__ __forceinline__ float plus(float a, float y) { return a + y; }
__device__ __forceinline__ float value(Df a) { return a.hi; }
__device__ __forceinline__ float value(float a) { return a; }

__device__ __forceinline__ void stv(float* p, size_t i, float x) { p[i] = x; }
__device__ __forceinline__ void stv(__nv_bfloat16* p, size_t i, float x) {
  p[i] = __float2bfloat16_rn(x);
}

// State of a unit's solve (workspace): Z is valid, left to fp64, the dual system has no
// Cholesky factor (V_out = V0), or Z is valid and in fp64.
enum { kSolved = 0, kNeeds64 = 1, kSingular = 2, kSolved64 = 3 };

// The range of residuals and of Z that pairs of floats hold: products of values below kSmall
// have rounding errors below fp32's smallest, and sums of 256 values of kLarge stay far below
// its largest.
constexpr float kSmall = 0x1p-100f, kLarge = 0x1p100f;

struct SArgs {
  Shape s;
  int tiles;       // CTAs per unit of the launch: CTA x is tile x % tiles of unit x / tiles
  const int32_t* idx;
  const float* scores;
  const float* y;
  float* x;        // [U][m][B] logits, then X
  uint8_t* flags;  // [U][B]
  int* state;      // [U]
  int* status;
};

// Retained position of slot i; an entry outside [0, n) is reported by
// k_simt_logits and read as 0.
__device__ __forceinline__ int rpos(const SArgs& a, int u, int i) {
  const int j = a.idx[(size_t)u * a.s.B + i];
  return (unsigned)j < (unsigned)a.s.n ? j : 0;
}

// ------------------------------------------------- logits, K_out, fixed set --
constexpr int kLP = kD + 1;        // padded row stride of the staged tiles
constexpr int kFixKeys = 8192;     // candidate keys the fixed-set CTA holds in shared memory
constexpr size_t kLogitsSmem = (size_t)64 * kLP * 4;
static_assert(kFixKeys * 4 <= kLogitsSmem, "keys fit the tile buffers");

// Fixed set of unit u: retained sinks, the window, and the n_fix best-scored
// retained prefix non-sink tokens (ties to the smaller position).  Lists past
// kFixKeys re-read their scores in each radix pass.
__device__ void fixed_set(const SArgs& a, int u, uint32_t* keys, int* hist, int* sh) {
  const Shape& s = a.s;
  const float* cu = a.scores + (size_t)u * s.P;
  uint8_t* F = a.flags + (size_t)u * s.B;
  const bool held = s.B <= kFixKeys;
  // 0 marks a slot that is no candidate (no finite or infinite score maps to 0)
  auto key_of = [&](int i) {
    const int j = rpos(a, u, i);
    return (j >= s.n_sink && j < s.P) ? max(order_key(cu[j]), 1u) : 0u;
  };
  int nc = 0;
  for (int i = threadIdx.x; i < s.B; i += blockDim.x) {
    if ((unsigned)a.idx[(size_t)u * s.B + i] >= (unsigned)s.n)
      set_status(a.status, GRKV_ERR_INVALID_ARG);
    const uint32_t key = key_of(i);
    if (held) keys[i] = key;
    F[i] = key ? 0 : 1;
    nc += key != 0u;
  }
  int ncand;
  (void)block_exclusive_scan(nc, sh + 8, &ncand);
  const int nf = min(s.n_fix, ncand);
  if (nf <= 0) return;
  auto get = [&](int i, uint32_t* key) {
    *key = held ? keys[i] : key_of(i);
    return *key != 0u;
  };
  block_topk_mark(get, [&](int i, int) { F[i] = 1; }, s.B, nf, hist, sh);
}

// 1 + ceil(B / 32) * ceil(m / 32) CTAs per unit: the first takes the fixed
// set, the others one 32 x 32 tile of logits each.  The tiles of the first 32
// rows also copy their K0 rows to K_out.
template <typename T>
__global__ void __launch_bounds__(256) k_simt_logits(const T* __restrict__ q,
                                                     const T* __restrict__ k,
                                                     T* __restrict__ k_out, SArgs a) {
  chain_wait();
  extern __shared__ __align__(16) float sm[];
  __shared__ int hist[256];
  __shared__ int sh[48];
  const Shape& s = a.s;
  const int u = blockIdx.x / a.tiles, tile = blockIdx.x % a.tiles;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tile == 0) {
    if (tid == 0) a.state[u] = kSolved;
    fixed_set(a, u, (uint32_t*)sm, hist, sh);
    return;
  }
  const int nb = (s.B + 31) / 32, t = tile - 1;
  const int r0 = t / nb * 32, b0 = t % nb * 32;
  float* qs = sm;               // [32][kLP]
  float* ks = sm + 32 * kLP;    // [32][kLP]
  const T* qu = q + ((size_t)u * s.m + r0) * kD;
  const T* ku = k + (size_t)u * s.n * kD;
  T* ko = k_out + ((size_t)u * s.B + b0) * kD;
  for (int jj = warp; jj < 32; jj += 8) {
    const int i = b0 + jj;
    const size_t row = i < s.B ? (size_t)rpos(a, u, i) * kD : 0;
#pragma unroll
    for (int e = 0; e < kD / 32; ++e) {
      const int c = e * 32 + lane;
      const T raw = ku[row + c];
      ks[jj * kLP + c] = ldv(&raw, 0);
      if (r0 == 0 && i < s.B) ko[(size_t)jj * kD + c] = raw;
      qs[jj * kLP + c] = r0 + jj < s.m ? ldv(qu, (size_t)jj * kD + c) : 0.f;
    }
  }
  __syncthreads();
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
  for (int e = 0; e < kD; ++e) {
    const float kv = ks[lane * kLP + e];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = fmaf(qs[(warp + 8 * i) * kLP + e], kv, acc[i]);
  }
  const int slot = b0 + lane;
  if (slot >= s.B) return;
  const int j = rpos(a, u, slot);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + warp + 8 * i;
    if (r < s.m)
      a.x[((size_t)u * s.m + r) * s.B + slot] = visible(s, r, j) ? s.scale * acc[i] : -INFINITY;
  }
}

// X = row softmax over the retained keys; one warp per row of the unit.
__global__ void __launch_bounds__(256) k_simt_softmax(SArgs a) {
  chain_wait();
  const int lane = threadIdx.x & 31, B = a.s.B;
  const int u = blockIdx.x / a.tiles, r = blockIdx.x % a.tiles * 8 + (threadIdx.x >> 5);
  if (r >= a.s.m) return;
  float* xr = a.x + ((size_t)u * a.s.m + r) * B;
  float M = -INFINITY;
#pragma unroll 4
  for (int i = lane; i < B; i += 32) M = fmaxf(M, xr[i]);
  for (int o = 16; o; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  float L = 0.f;
#pragma unroll 4
  for (int i = lane; i < B; i += 32) L += expf(xr[i] - M);
  for (int o = 16; o; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
#pragma unroll 4
  for (int i = lane; i < B; i += 32) xr[i] = expf(xr[i] - M) / L;
}

// ----------------------------------------------------------- R and N --
// Output tiles of 8 rows x 32 columns, one output per thread: at 10 to 12
// instructions per multiply-add two shared loads each cost nothing, and small
// tiles spread one unit over many SMs.  Tiles 0 .. ceil(m/8) * 4 - 1 are R's,
// the rest cover the lower triangle of N by blocks of 32 columns.
constexpr int kRS = 64;   // retained slots per slab

__host__ __device__ constexpr int regr_r_tiles(int m) { return (m + 7) / 8 * (kD / 32); }
// N's tiles: row block rb (8 rows) meets column blocks 0 .. rb / 4
__host__ __device__ constexpr int regr_n_tiles(int m) {
  const int rb = (m + 7) / 8, full = rb / 4, rest = rb % 4;
  return 4 * full * (full + 1) / 2 + rest * (full + 1);
}

template <typename T, typename A>
__global__ void __launch_bounds__(256) k_simt_regr(const T* __restrict__ v, SArgs a,
                                                   A* __restrict__ gram, A* __restrict__ rz) {
  chain_wait();
  __shared__ float as[8][kRS + 1];
  __shared__ float bs[kRS][33];
  const Shape& s = a.s;
  const int u = blockIdx.x / a.tiles, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = s.m, B = s.B;
  int t = blockIdx.x % a.tiles, r0, c0;
  const bool is_r = t < regr_r_tiles(m);
  if (is_r) {
    r0 = t / (kD / 32) * 8;
    c0 = t % (kD / 32) * 32;
  } else {
    t -= regr_r_tiles(m);
    int rb = 0;
    while (t >= rb / 4 + 1) {
      t -= rb / 4 + 1;
      ++rb;
    }
    r0 = rb * 8;
    c0 = t * 32;
  }
  const float* X = a.x + (size_t)u * m * B;
  const uint8_t* F = a.flags + (size_t)u * B;
  const T* vu = v + (size_t)u * s.n * kD;
  // N's operands leave out the fixed slots; fetch() loads the slab at `base`
  float ra[2], rb8[8];
  auto fetch = [&](int base) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = base + e * 32 + lane, r = r0 + warp;
      ra[e] = (i < B && r < m && (is_r || !F[i])) ? X[(size_t)r * B + i] : 0.f;
    }
    if (is_r) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int i = base + warp + e * 8;
        rb8[e] = i < B ? ldv(vu, (size_t)rpos(a, u, i) * kD + c0 + lane) : 0.f;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int i = base + (e & 1) * 32 + lane, r = c0 + warp + (e >> 1) * 8;
        rb8[e] = (i < B && r < m && !F[i]) ? X[(size_t)r * B + i] : 0.f;
      }
    }
  };
  A acc;
  zero(acc);
  fetch(0);
  for (int base = 0; base < B; base += kRS) {
    as[warp][lane] = ra[0];
    as[warp][32 + lane] = ra[1];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (is_r)
        bs[warp + e * 8][lane] = rb8[e];
      else
        bs[(e & 1) * 32 + lane][warp + (e >> 1) * 8] = rb8[e];
    }
    __syncthreads();
    if (base + kRS < B) fetch(base + kRS);
#pragma unroll 8
    for (int kk = 0; kk < kRS; ++kk) mac(acc, as[warp][kk], bs[kk][lane]);
    __syncthreads();
  }
  const int r = r0 + warp, c = c0 + lane;
  if (r >= m) return;
  if (is_r) {
    const size_t o = ((size_t)u * m + r) * kD + c;
    rz[o] = minus(a.y[o], acc);
  } else if (c <= r) {
    const A n = r == c ? plus(acc, s.lambda) : plus(acc, 0.f);
    gram[((size_t)u * m + r) * m + c] = n;
    gram[((size_t)u * m + c) * m + r] = n;
  }
}

// ------------------------------------------------------------- the solve --
constexpr int kChT = 512;
constexpr int kCLD = 129;          // row stride (pairs) of N in k_simt_chol
constexpr int kBLD = 33;           // row stride (pairs) of a 32 x 32 block
constexpr size_t kCholSmem = (size_t)(128 * kCLD + 4 * 32 * kBLD + 2 * 128) * sizeof(Df);

// N = L L^T for m <= 128, one CTA per unit, N in shared memory: panels of 32
// columns, right-looking inside the panel, then the trailing triangle; last the
// diagonal blocks are inverted, one warp each.  Writes L's blocks below the
// diagonal and the inverted diagonal blocks over N.  A pivot below 2^-20 of
// its diagonal entry or below 2^-60, where pairs of floats leave too few
// digits, sends the unit to fp64.  Bound by the chain of columns, two block barriers, a root and
// a division each: 8 units of m = 128 take 114 us, one of m = 32 29 us.
__global__ void __launch_bounds__(kChT, 1) k_simt_chol(SArgs a, Df* __restrict__ gram) {
  chain_wait();
  extern __shared__ __align__(16) float sm[];
  Df* N = (Df*)sm;                      // [128][kCLD]
  Df* inv = N + 128 * kCLD;             // [4][32][kBLD]
  Df* col = inv + 4 * 32 * kBLD;        // [128] the current column of L below the diagonal
  Df* dinv = col + 128;                 // [128] 1 / L_jj
  const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = a.s.m, mp = (m + 31) / 32 * 32;
  Df* G = gram + (size_t)u * m * m;
  for (int i = warp; i < mp; i += kChT / 32)
    for (int j = lane; j < mp; j += 32)
      N[i * kCLD + j] = (i < m && j < m) ? G[(size_t)i * m + j] : Df{i == j ? 1.f : 0.f, 0.f};
  for (int i = tid; i < mp; i += kChT)
    dinv[i].hi = i < m ? G[(size_t)i * m + i].hi : 1.f;   // N_jj until the column is done
  for (int j0 = 0; j0 < mp; j0 += 32) {
    for (int j = j0; j < j0 + 32; ++j) {
      __syncthreads();
      const Df d = N[j * kCLD + j];
      if (!(d.hi > 0x1p-60f) || !(d.hi > 0x1p-20f * dinv[j].hi)) {   // same answer in all threads
        if (tid == 0) a.state[u] = kNeeds64;
        return;
      }
      // the pivot stays as it is: other warps may not have read it yet, and L_jj is only
      // used through its reciprocal
      const Df rinv = df_rcp(df_sqrt(d));
      if (tid > 0 && tid < mp - j) {
        const Df l = df_mul(N[(j + tid) * kCLD + j], rinv);
        N[(j + tid) * kCLD + j] = l;
        col[j + tid] = l;
      }
      __syncthreads();
      if (tid == 0) dinv[j] = rinv;
      for (int c = j + 1 + warp; c < j0 + 32; c += kChT / 32) {
        const Df lc = df_neg(col[c]);
        for (int i = c + lane; i < mp; i += 32) {
          Df x = N[i * kCLD + c];
          df_mac(x, col[i], lc);
          N[i * kCLD + c] = df_norm(x);
        }
      }
    }
    __syncthreads();
    // trailing triangle: rows i >= c >= j0 + 32
    for (int c = j0 + 32 + warp; c < mp; c += kChT / 32)
      for (int i = c + lane; i < mp; i += 32) {
        Df x = N[i * kCLD + c];
#pragma unroll 8
        for (int e = 0; e < 32; ++e) df_mac(x, df_neg(N[i * kCLD + j0 + e]), N[c * kCLD + j0 + e]);
        N[i * kCLD + c] = df_norm(x);
      }
  }
  __syncthreads();
  if (warp * 32 < mp) {
    // lane c: column c of the inverse of diagonal block `warp`
    Df* I = inv + warp * 32 * kBLD;
    const int o = warp * 32;
    for (int i = 0; i < 32; ++i) {
      Df x{i == lane ? 1.f : 0.f, 0.f};
      for (int e = 0; e < i; ++e) df_mac(x, df_neg(N[(o + i) * kCLD + o + e]), I[e * kBLD + lane]);
      I[i * kBLD + lane] = i < lane ? Df{0.f, 0.f} : df_mul(df_norm(x), dinv[o + i]);
    }
  }
  __syncthreads();
  for (int i = warp; i < m; i += kChT / 32)
    for (int j = lane; j < m; j += 32) {
      if (j / 32 > i / 32) continue;
      G[(size_t)i * m + j] = j / 32 == i / 32 ? inv[(i / 32 * 32 + i % 32) * kBLD + j % 32]
                                              : N[i * kCLD + j];
    }
}

// Z = L^-T L^-1 R by 32-row blocks, 8 columns per CTA; thread (row, column).
// The factor's blocks are all staged first.
constexpr size_t kSubstSmem =
    (size_t)(10 * 32 * kBLD + 128 * 9 + 32 * 9) * sizeof(Df) + 256;

__global__ void __launch_bounds__(256) k_simt_subst(SArgs a, const Df* __restrict__ gram,
                                                    Df* __restrict__ rz) {
  chain_wait();
  extern __shared__ __align__(16) float sm[];
  Df* Lb = (Df*)sm;                     // block (i, j), j <= i, at i (i + 1) / 2 + j
  Df* W = Lb + 10 * 32 * kBLD;          // [128][9]
  Df* tmp = W + 128 * 9;                // [32][9]
  uint8_t* seen = (uint8_t*)(tmp + 32 * 9);   // [32][8] of a thread's residuals: 1 nonzero, 2 not small
  const int u = blockIdx.x / (kD / 8), tid = threadIdx.x, r = tid >> 3, c = tid & 7;
  const int m = a.s.m, nb = (m + 31) / 32;
  const int state = a.state[u];
  const Df* G = gram + (size_t)u * m * m;
  Df* Z = rz + (size_t)u * m * kD + blockIdx.x % (kD / 8) * 8;
  for (int i = tid >> 5; i < nb * 32; i += 8)
    for (int j = tid & 31; j < (i / 32 + 1) * 32; j += 32) {
      const int bi = i / 32, bj = j / 32;
      const Df pad{i == j ? 1.f : 0.f, 0.f};
      Lb[((bi * (bi + 1) / 2 + bj) * 32 + i % 32) * kBLD + j % 32] =
          (i < m && j < m) ? G[(size_t)i * m + j] : pad;
    }
  int size = 0;
  for (int b = 0; b < nb; ++b) {
    const int i = b * 32 + r;
    const Df x = i < m ? Z[(size_t)i * kD + c] : Df{0.f, 0.f};
    W[i * 9 + c] = x;
    size |= (x.hi != 0.f ? 1 : 0) | (fabsf(x.hi) >= kSmall ? 2 : 0);
  }
  seen[tid] = (uint8_t)size;
  // another CTA of the unit may have given it to fp64 between two reads: one answer for the block
  if (__syncthreads_or(state != kSolved)) return;
  bool fits = true;
  if (tid < 8) {
    for (int e = tid; e < 256; e += 8) size |= seen[e];
    fits = size != 1;
  }
  auto solve_block = [&](int b, Df acc, bool back) {
    tmp[r * 9 + c] = df_norm(acc);
    __syncthreads();
    const Df* I = Lb + (size_t)(b * (b + 1) / 2 + b) * 32 * kBLD;
    Df z{0.f, 0.f};
#pragma unroll 8
    for (int e = 0; e < 32; ++e) df_mac(z, back ? I[e * kBLD + r] : I[r * kBLD + e], tmp[e * 9 + c]);
    z = df_norm(z);
    W[(b * 32 + r) * 9 + c] = z;
    if (back) fits = fits && fabsf(z.hi) < kLarge;   // false for NaN
    __syncthreads();
  };
  for (int b = 0; b < nb; ++b) {   // L W = R
    Df acc = W[(b * 32 + r) * 9 + c];
    for (int p = 0; p < b; ++p) {
      const Df* L = Lb + (size_t)(b * (b + 1) / 2 + p) * 32 * kBLD;
#pragma unroll 8
      for (int e = 0; e < 32; ++e) df_mac(acc, df_neg(L[r * kBLD + e]), W[(p * 32 + e) * 9 + c]);
    }
    solve_block(b, acc, false);
  }
  for (int b = nb - 1; b >= 0; --b) {   // L^T Z = W
    Df acc = W[(b * 32 + r) * 9 + c];
    for (int p = b + 1; p < nb; ++p) {
      const Df* L = Lb + (size_t)(p * (p + 1) / 2 + b) * 32 * kBLD;
#pragma unroll 8
      for (int e = 0; e < 32; ++e) df_mac(acc, df_neg(L[e * kBLD + r]), W[(p * 32 + e) * 9 + c]);
    }
    solve_block(b, acc, true);
  }
  // outside the range of pairs: R is needed again, so Z is only written when it holds
  if (__syncthreads_or(!fits)) {
    if (tid == 0) a.state[u] = kNeeds64;
    return;
  }
  for (int b = 0; b < nb; ++b) {
    const int i = b * 32 + r;
    if (i < m) Z[(size_t)i * kD + c] = W[i * 9 + c];
  }
}

// Units left to fp64 (and every unit with m > 128), one CTA each: right-looking
// Cholesky in global memory, substitution with one column per thread.  With m > 128 it starts
// from the R and N formed in pairs, under the rules of k_simt_chol and k_simt_subst: a pivot or
// a residual that pairs cannot hold starts the unit over.  Such units have R and N formed again
// in fp64.  Z goes back as pairs, or stays in fp64 where a column is outside their range.  A
// non-positive pivot is then GRKV_ERR_NUMERIC and leaves V0 in place.
template <typename T>
__global__ void __launch_bounds__(512) k_simt_solve64(const T* __restrict__ v, SArgs a, int all,
                                                      Df* __restrict__ gram,
                                                      Df* __restrict__ rz) {
  chain_wait();
  __shared__ double diag[kMaxM];
  __shared__ uint8_t seen[512];
  enum { kGood, kLost, kNotPositive };
  __shared__ int pivot;
  const Shape& s = a.s;
  const int u = blockIdx.x, tid = threadIdx.x, m = s.m, B = s.B, nthr = blockDim.x;
  if (!all && a.state[u] != kNeeds64) return;
  const float* X = a.x + (size_t)u * m * B;
  const uint8_t* F = a.flags + (size_t)u * B;
  const T* vu = v + (size_t)u * s.n * kD;
  Df* Gd = gram + (size_t)u * m * m;
  Df* Rd = rz + (size_t)u * m * kD;
  double* N = (double*)Gd;
  double* R = (double*)Rd;
  for (bool pairs = all;; pairs = false) {
    if (pairs) {
      for (int p = tid; p < m * m; p += nthr) {
        const Df g = Gd[p];
        N[p] = (double)g.hi + (double)g.lo;
      }
      // thread (phase, column): kD divides the block's threads
      bool finite = true, nonzero = false, fits = false;
      for (int p = tid; p < m * kD; p += nthr) {
        const Df g = Rd[p];
        R[p] = (double)g.hi + (double)g.lo;
        finite = finite && isfinite(R[p]);
        nonzero |= g.hi != 0.f;
        fits |= fabsf(g.hi) >= kSmall;
      }
      seen[tid] = (nonzero ? 1 : 0) | (fits ? 2 : 0);
      __syncthreads();
      int size = 0;
      for (int h = tid % kD; h < nthr; h += kD) size |= seen[h];
      if (__syncthreads_or(!finite || size == 1)) continue;
    } else {
      for (int p = tid / 32; p < m * m; p += nthr / 32) {   // a warp per entry on or below the diagonal
        const int r1 = p / m, r2 = p % m;
        if (r2 > r1) continue;
        double g = 0.0;
        for (int i = tid % 32; i < B; i += 32)
          if (!F[i]) g += (double)X[(size_t)r1 * B + i] * (double)X[(size_t)r2 * B + i];
        for (int o = 16; o; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if (tid % 32 == 0) N[p] = r1 == r2 ? g + (double)s.lambda : g;
      }
      for (int p = tid; p < m * kD; p += nthr) {
        const int r = p / kD, c = p % kD;
        double g = 0.0;
        for (int i = 0; i < B; ++i)
          g += (double)X[(size_t)r * B + i] * (double)ldv(vu, (size_t)rpos(a, u, i) * kD + c);
        R[p] = (double)a.y[(size_t)u * m * kD + p] - g;
      }
      __syncthreads();
    }
    if (tid < m) diag[tid] = N[(size_t)tid * m + tid];
    __syncthreads();
    int now = kGood;
    for (int c = 0; c < m; ++c) {
      if (tid == 0) {
        const double d = N[(size_t)c * m + c];
        pivot = pairs && !(d > 0x1p-60 && d > 0x1p-20 * diag[c]) ? kLost
                : !(d > 0.0)                                     ? kNotPositive
                                                                 : kGood;
        if (pivot == kGood) N[(size_t)c * m + c] = sqrt(d);
      }
      __syncthreads();
      if ((now = pivot) != kGood) break;
      const double piv = N[(size_t)c * m + c];
      for (int i = c + 1 + tid; i < m; i += nthr) N[(size_t)i * m + c] /= piv;
      __syncthreads();
      const int rest = m - c - 1;
      for (int p = tid; p < rest * rest; p += nthr) {
        const int i = c + 1 + p / rest, j = c + 1 + p % rest;
        if (j <= i) N[(size_t)i * m + j] -= N[(size_t)i * m + c] * N[(size_t)j * m + c];
      }
      __syncthreads();
    }
    if (now == kGood) break;
    if (now == kNotPositive) {
      if (tid == 0) {
        a.state[u] = kSingular;
        set_status(a.status, GRKV_ERR_NUMERIC);
      }
      return;
    }
  }
  bool wide = false;   // the thread's column of Z does not fit pairs
  if (tid < kD) {
    double largest = 0.0;
    for (int i = 0; i < m; ++i) {
      double z = R[(size_t)i * kD + tid];
      for (int c = 0; c < i; ++c) z -= N[(size_t)i * m + c] * R[(size_t)c * kD + tid];
      R[(size_t)i * kD + tid] = z / N[(size_t)i * m + i];
    }
    for (int i = m - 1; i >= 0; --i) {
      double z = R[(size_t)i * kD + tid];
      for (int c = i + 1; c < m; ++c) z -= N[(size_t)c * m + i] * R[(size_t)c * kD + tid];
      z /= N[(size_t)i * m + i];
      R[(size_t)i * kD + tid] = z;
      largest = fmax(largest, fabs(z));
      wide |= !(fabs(z) < (double)kLarge);   // NaN too
    }
    wide |= largest > 0.0 && largest < (double)kSmall;
  }
  wide = __syncthreads_or(wide);
  if (tid == 0) a.state[u] = wide ? kSolved64 : kSolved;
  if (wide || tid >= kD) return;
  for (int i = 0; i < m; ++i) {
    const double z = R[(size_t)i * kD + tid];
    const float hi = (float)z;
    Rd[(size_t)i * kD + tid] = {hi, (float)(z - (double)hi)};
  }
}

// One output in fp64: a column x [m] of X, a column z [m] of Z, in fp64 if wide.
__device__ __noinline__ float update64(const float* x, int B, const Df* z, int m, bool wide,
                                       float v0) {
  double g = 0.0;
  for (int r = 0; r < m; ++r) {
    const Df p = z[(size_t)r * kD];
    const double zr = wide ? ((const double*)z)[(size_t)r * kD] : (double)p.hi + (double)p.lo;
    g += (double)x[(size_t)r * B] * zr;
  }
  return (float)((double)v0 + g);
}

// V_out[G] = V0[G] + X_G^T Z, V_out[F] = V0[F]: 32 slots x 32 columns per CTA,
// four outputs per thread.  Outputs that pairs cannot hold are formed in fp64.
template <typename T, typename A>
__global__ void __launch_bounds__(256) k_simt_update(const T* __restrict__ v,
                                                     T* __restrict__ v_out, SArgs a,
                                                     const A* __restrict__ rz) {
  chain_wait();
  __shared__ float xs[32][33];
  __shared__ A zs[32][32];
  const Shape& s = a.s;
  const int u = blockIdx.x / a.tiles, tile = blockIdx.x % a.tiles;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = s.m, B = s.B, b0 = tile / (kD / 32) * 32, c0 = tile % (kD / 32) * 32;
  const float* X = a.x + (size_t)u * m * B;
  const A* Z = rz + (size_t)u * m * kD;
  const T* vu = v + (size_t)u * s.n * kD;
  A acc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) zero(acc[i]);
  const bool keep = s.lambda_inf || a.state[u] == kSingular;   // V_out = V0
  const bool wide = !s.lambda_inf && a.state[u] == kSolved64;
  for (int r0 = 0; r0 < m && !keep && !wide; r0 += 32) {
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = r0 + warp + e * 8;
      xs[warp + e * 8][lane] = (r < m && b0 + lane < B) ? X[(size_t)r * B + b0 + lane] : 0.f;
      if (r < m)
        zs[warp + e * 8][lane] = Z[(size_t)r * kD + c0 + lane];
      else
        zero(zs[warp + e * 8][lane]);
    }
    __syncthreads();
#pragma unroll 8
    for (int r = 0; r < 32; ++r) {
      const A z = zs[r][lane];
#pragma unroll
      for (int i = 0; i < 4; ++i) mac(acc[i], xs[r][warp + 8 * i], z);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int slot = b0 + warp + 8 * i;
    if (slot >= B) break;
    const size_t o = ((size_t)u * B + slot) * kD + c0 + lane;
    const T v0 = vu[(size_t)rpos(a, u, slot) * kD + c0 + lane];
    if (keep || a.flags[(size_t)u * B + slot]) {
      v_out[o] = v0;
      continue;
    }
    float x = value(plus(acc[i], ldv(&v0, 0)));
    if constexpr (std::is_same<A, Df>::value)
      if (wide || !isfinite(x)) x = update64(X + slot, B, Z + c0 + lane, m, wide, ldv(&v0, 0));
    stv(v_out, o, x);
  }
}

template <typename T, typename A>
cudaError_t merge_impl(const Shape& s, const T* q, const T* k, const T* v, const float* scores,
                       const float* y, const int32_t* idx, T* k_out, T* v_out, char* ws,
                       const WsLayout& L, cudaStream_t st) {
  SArgs a{s, 0, idx, scores, y, (float*)(ws + L.xbuf), (uint8_t*)(ws + L.flags),
          (int*)(ws + L.state), (int*)(ws + L.status)};
  A* gram = (A*)(ws + L.gram);
  A* rz = (A*)(ws + L.rz);
  const unsigned U = (unsigned)s.U, nb = (unsigned)(s.B + 31) / 32, nr = (unsigned)(s.m + 31) / 32;
  a.tiles = (int)(1 + nb * nr);
  cudaError_t e = launch_kernel(s.chained, 1, k_simt_logits<T>, dim3(U * a.tiles), 256, kLogitsSmem, st, q,
                                k, k_out, a);
  count_launches(1);
  if (e == cudaSuccess && !s.lambda_inf) {
    a.tiles = (s.m + 7) / 8;
    e = launch_kernel(true, 1, k_simt_softmax, dim3(U * a.tiles), 256, 0, st, a);
    if (e != cudaSuccess) return e;
    a.tiles = regr_r_tiles(s.m) + regr_n_tiles(s.m);
    e = launch_kernel(true, 1, k_simt_regr<T, A>, dim3(U * a.tiles), 256, 0, st, v, a, gram, rz);
    count_launches(2);
    if (e != cudaSuccess) return e;
    if constexpr (std::is_same<A, Df>::value) {
      // the factor of m <= 128 fits shared memory as pairs; more rows take fp64
      const bool pairs = s.m <= 128;
      if (pairs) {
        e = cudaFuncSetAttribute(k_simt_chol, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kCholSmem);
        if (e == cudaSuccess)
          e = cudaFuncSetAttribute(k_simt_subst, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)kSubstSmem);
        if (e != cudaSuccess) return e;
        e = launch_kernel(true, 1, k_simt_chol, dim3(U), kChT, kCholSmem, st, a, gram);
        if (e == cudaSuccess)
          e = launch_kernel(true, 1, k_simt_subst, dim3(U * (kD / 8)), 256, kSubstSmem, st, a,
                            (const Df*)gram, rz);
        if (e != cudaSuccess) return e;
        count_launches(2);
      }
      e = launch_kernel(true, 1, k_simt_solve64<T>, dim3(U), 512, 0, st, v, a, pairs ? 0 : 1, gram, rz);
      count_launches(1);
    } else {
      // gram's region holds 8 bytes per entry: the second half takes the factor
      // of the first 128 rows (m^2 >= 128^2 floats a unit where it is used)
      e = launch_solve(s.U, s.m, s.m, 0, 0.f, 0, (float*)gram, (float*)rz,
                       (float*)gram + (size_t)s.U * s.m * s.m, (size_t)s.m * s.m, 128, a.state,
                       a.status, st);
    }
  }
  if (e != cudaSuccess) return e;
  a.tiles = (int)nb * (kD / 32);
  count_launches(1);
  return launch_kernel(true, 1, k_simt_update<T, A>, dim3(U * a.tiles), 256, 0, st, v, v_out, a,
                       (const A*)rz);
}

}  // namespace

cudaError_t launch_merge_simt(const Shape& s, const void* q, const void* k, const void* v,
                              const float* scores, const float* y, const int32_t* idx,
                              void* k_out, void* v_out, char* ws, const WsLayout& L,
                              cudaStream_t st) {
  if (s.dtype == GRKV_F32)
    return merge_impl<float, Df>(s, (const float*)q, (const float*)k, (const float*)v, scores, y,
                                 idx, (float*)k_out, (float*)v_out, ws, L, st);
  return merge_impl<__nv_bfloat16, float>(
      s, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, scores, y,
      idx, (__nv_bfloat16*)k_out, (__nv_bfloat16*)v_out, ws, L, st);
}

}  // namespace grkv
