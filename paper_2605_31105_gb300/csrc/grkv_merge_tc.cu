// GRKV value step on the tensor cores (bf16, d = 128, m <= 256, B <= 32768).
//
// Algorithm 1's value step in dual form (Sec. 3.4, App. D.1) with the fixed
// tokens of App. D.3:
//   k_merge_fixed   the fixed set (retained sinks, the window, and the n_fix
//                   retained prefix tokens with the largest scores), a flag per
//                   slot, and a stable partition of the B retained slots into
//                   "positions": the n_G non-fixed slots first, then the fixed
//                   ones, each in slot order.  The window stays last in both
//                   orders, so slot or position p is visible to window row r
//                   exactly when p <= B - w + r % w.
//   k_merge_gram    a cluster of CTAs per unit: phase 0 over the slots: row max /
//                   sum of l = s Q K0^T; phase 1 over the positions:
//                   X = softmax, R~ += Xh V0 and the Gram G += Xh XGh^T +
//                   (2 Xl) XGh^T on tcgen05 (Xh, Xl the bf16 high / low parts
//                   of X; XGh is Xh with the fixed columns zeroed, which removes
//                   them from both terms; N = (G + G^T) / 2 restores the cross
//                   terms).  Writes R = Y - R~, G and the row normalisers to the
//                   workspace.  With the full-cache row statistics only phase 1
//                   runs, unless they lie far above the retained ones.
//   launch_solve    N = sym(G) + lambda I, Z = N^-1 R in fp32 (grkv_solve.cu).
//   k_merge_update  over the slots: S^T = K0 Q^T (one TMEM lane per token),
//                   X_G^T (zero for fixed slots) as bf16 high / low parts back
//                   into TMEM, dV = XGh^T Zh + XGh^T Zl + XGl^T Zh with X_G^T
//                   as the TMEM A operand, V_out = V0 + dV in the gathered V0
//                   tile, and K_out = K0, V_out by TMA tile stores.
//
// The kernels rely on the idx contract of grkv.h: ascending, with the window
// n-w..n-1 in the last w slots.
#include <algorithm>
#include <cmath>

#include "block_select.cuh"
#include "grkv_internal.cuh"
#include "sm100.cuh"
#include "tmap.cuh"

namespace grkv {
namespace {

using namespace sm100;

constexpr int kTile = 128;
constexpr int kRows = 128;
constexpr int kThreads = 384;    // k_merge_cross
constexpr int kThreadsG = 640;   // k_merge_gram
constexpr int kThreadsU = 736;   // k_merge_update
constexpr uint32_t kTileBytes = kTile * kD * 2;   // 32 KB
constexpr int kMaxB = 32768;
constexpr int kSms = 152;        // SMs of a GB300
constexpr int kClusterSms = 128; // SMs that clusters of up to 8 CTAs (one per SM) can be counted on to fill
constexpr long long kBudget = 1ll << 32;

// Shared memory (offsets from a 1024-byte aligned base).  k_merge_gram: Q, a
// ring of four gathered tiles, two XGh tiles.  k_merge_update: Q, two K0
// tiles, two V0 / V_out tiles, Zh, Zl.  Both continue with the barriers.
constexpr int kRingG = 4;
constexpr uint32_t kOffQ = 0;
constexpr uint32_t kOffRing = kTileBytes;
constexpr uint32_t kOffXG = kOffRing + kRingG * kTileBytes;   // gram: 2 tiles
constexpr uint32_t kOffBar = 7 * kTileBytes;
static_assert(kOffXG + 2 * kTileBytes == kOffBar, "shared-memory layout");
constexpr uint32_t kSmemBytes = kOffBar + 256 + 1024;

// TMEM columns.  gram: S[2] 0..255, R~ 256..383, Gram 384..511.
// update: S^T[2] (then X_G^T) 0..255, D[2] 256..511.
constexpr uint32_t kColS = 0;
constexpr uint32_t kColR = 256;
constexpr uint32_t kColG = 384;
constexpr uint32_t kColD = 256;

struct MArgs {
  int U, n, w, m, P, B, causal, n_sink, n_fix;
  float sl2;
  const int32_t* idx;        // [U][B]
  const float* scores;       // [U][P]
  const float* y;            // [U][m][128]
  const __nv_bfloat16* k;    // [U][n][128]
  const __nv_bfloat16* v;
  __nv_bfloat16* k_out;      // [U][B][128]
  __nv_bfloat16* v_out;
  const float* rstats;       // [U][m][2] full-cache row max / sum (natural units) or null
  float* rz;                 // [U][128][128]  R (gram) -> Z (solve)
  float* gram;               // [U][128][128]  raw Gram
  float* lam;                // [U][128]       log2 normaliser of each window row
  int32_t* src;              // [U][B]         K / V row of each position
  int32_t* ng;               // [U]            number of non-fixed slots
  uint8_t* fixed;            // [U][B]         1 for a fixed slot
  int ranks;                 // k_merge_gram: CTAs per unit and row block
  // Row blocks (nrb of them): an update launch takes the 128 window rows row0 .. row0+127;
  // the per-unit arrays hold ldr rows (128 or 256):
  // rz [U][ldr][128], gram [U][ldr][ldr], lam [U][ldr].
  int row0, nrb, ldr;
  int upd_mode;              // update: 0 V_out = V0 + dV; 1 vpart = V0 + dV; 2 V_out = vpart + dV
  float* vpart;              // [U][B][128] fp32, between the update's two row blocks
  int* status;
  const UnitRow* units;      // budgets of the units, or null (B each)
  int split;                 // update: CTAs per unit
};

__device__ __forceinline__ float lo_half(uint32_t h) { return __uint_as_float(h << 16); }
__device__ __forceinline__ float hi_half(uint32_t h) { return __uint_as_float(h & 0xFFFF0000u); }

// TMEM column, within a 128-column buffer, of the packed high (lo = 0) or low
// (lo = 1) parts of K rows 16kk .. 16kk+15 of an A operand written back in
// place over 32-column chunks (chunk c: high parts in 32c .. 32c+15, low parts
// in 32c+16 .. 32c+31).
__device__ __forceinline__ uint32_t xt_col(int kk, int lo) {
  return (kk >> 1) * 32 + lo * 16 + (kk & 1) * 8;
}

// The wait for copies or MMAs in flight at the end of a CTA: bounded, whether or not another
// wait has given up.
__device__ __noinline__ void mbar_drain_wait(uint64_t* bar, uint32_t parity) {
  volatile int no_abort = 0;
  mbar_wait(bar, parity, &no_abort, kBudget);
}
__device__ __forceinline__ void mbar_drain(uint64_t* bar, uint32_t parity) {
  if (!mbar_try_wait(bar, parity)) mbar_drain_wait(bar, parity);
}
// mbar_wait for all lanes of a warp with one answer, so that warp-collective
// instructions after a wait are reached by all lanes or by none.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort, kBudget));
}

// Four rows (64 columns each) of a 2-D tensor map into consecutive 128-byte rows.
__device__ __forceinline__ void tma_gather4(void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int r0, int r1, int r2, int r3) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
      : "memory");
}

// Producer side of a ring of R gathered tiles, run by W warps: warp pw
// (0 <= pw < W) gathers its share of the tile's 32 four-row groups (the rows
// rows_u[t*128 + row], clamped to B-1; a row outside [0, n) reads row 0) with
// TMA gather4 into the 128-byte-swizzled tile and arrives on the slot's full
// barrier (initialised with W arrivals) with its share of the transaction
// bytes, so a slot is full once every share has landed.  The issue cost of
// gather4 is paid by the issuing warp, so more warps fill a tile faster.  The
// row indices are fetched by rows() one tile ahead of load(), so their
// latency overlaps the wait for a free slot, and one fetch can serve the K and
// V tiles of the same rows.
template <int R, int W>
struct Gatherer {
  // warp pw takes the four-row groups g0(pw) .. g0(pw + 1) - 1 of the 32 in a tile
  static constexpr int g0(int pw) { return pw * (kTile / 4) / W; }
  static_assert(kTile / 4 / W <= 32 && W >= 1, "gather split");
  uint8_t* ring;
  uint64_t* full;
  uint64_t* empty;
  uint32_t use = 0;
  // lanes < the warp's group count: the four rows of group g0(pw) + lane of tile t, as map rows
  __device__ __forceinline__ void rows(const int32_t* rows_u, int B, int n, int row0, int t,
                                       int pw, int lane, int* j) const {
    if (lane < g0(pw + 1) - g0(pw)) {
      const int r = 4 * (g0(pw) + lane);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int jj = __ldg(rows_u + min(t * kTile + r + e, B - 1));
        j[e] = row0 + ((unsigned)jj < (unsigned)n ? jj : 0);
      }
    }
  }
  __device__ __forceinline__ bool load(const CUtensorMap* map, const int* j, int pw, int lane,
                                       volatile int* abort_flag) {
    const uint32_t slot = use % R;
    bool ok = true;
    if (use >= R) ok = mbar_wait(&empty[slot], (use / R - 1) & 1, abort_flag, kBudget);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) return false;
    uint8_t* dst = ring + slot * kTileBytes;
    uint64_t* bar = &full[slot];
    const int ng = g0(pw + 1) - g0(pw);
    if (lane == 0) mbar_expect_tx(bar, ng * 4 * kD * 2);
    __syncwarp();
    if (lane < ng) {
      const int r = 4 * (g0(pw) + lane);
      tma_gather4(dst + r * 128, map, bar, 0, j[0], j[1], j[2], j[3]);
      tma_gather4(dst + kTileBytes / 2 + r * 128, map, bar, 64, j[0], j[1], j[2], j[3]);
    }
    ++use;
    return true;
  }
  // every issued gather lands before the CTA can exit
  __device__ __forceinline__ void drain() {
    for (uint32_t i = use > R ? use - R : 0; i < use; ++i) mbar_drain(&full[i % R], (i / R) & 1);
  }
};

// The same tile layout by 16-byte asynchronous copies, half a warp per 256-byte row: rows
// r0 .. r0 + 32 kN - 1 of the tile at shared address `tile`, row r0 + 32 h + l from row j[h] of
// lane l.  A gather4 tile takes 8 K cycles from issue to arrival beside another tile in flight
// and the TMA stores, these copies about 3.5 K; the issuing warp has to see its copies land
// before the tensor cores may read them, though.  256 units B = 2048: k_merge_gram 97 us with
// gather4 and 88 with these; k_merge_update 102 us with gather4 for K0 and these for V0 (which only
// threads read), 103 with these for both and 106 with gather4 for both.
template <int kN>
__device__ __forceinline__ void gather_async(uint32_t tile, int r0, const __nv_bfloat16* base,
                                             const int* j, int lane) {
  const int c = lane & 15;
  const uint32_t dst = tile + (c >> 3) * (kTileBytes / 2);
#pragma unroll
  for (int i = 0; i < 16 * kN; ++i) {
    const int r = 2 * i + (lane >> 4);
    const int row = __shfl_sync(0xffffffffu, j[i / 16], r & 31);
    cp_async16(dst + sw128_offset(r0 + r, c & 7), base + (size_t)row * kD + c * 8);
  }
}
// Lane l's rows of gather_async: rows_u[first + 32 h + l], clamped to the last of `count`; an
// entry outside [0, n) reads row 0.
template <int kN>
__device__ __forceinline__ void gather_index(const int32_t* rows_u, int first, int count, int n,
                                             int lane, int* j) {
#pragma unroll
  for (int h = 0; h < kN; ++h) {
    const int x = __ldg(rows_u + min(first + 32 * h + lane, count - 1));
    j[h] = (unsigned)x < (unsigned)n ? x : 0;
  }
}
// The warp's copies have landed and are visible to the tensor cores and TMA.
__device__ __forceinline__ void gather_arrive(uint64_t* full, int lane) {
  cp_async_wait_all();
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) mbar_arrive(full);
}

// S = Q K0^T for one gathered tile into TMEM columns s_col (issued by one thread).
__device__ __forceinline__ void issue_s(uint32_t s_tmem, uint32_t qa, uint32_t ka) {
  const uint32_t id_s = idesc_bf16(kRows, kTile, 0, 0);
#pragma unroll
  for (int kk = 0; kk < kD / 16; ++kk) {
    const uint32_t off = (kk >> 2) * (kTileBytes / 2) + (kk & 3) * 32;
    mma_bf16(s_tmem, sw128_desc(qa + off, 16, 1024), sw128_desc(ka + off, 16, 1024), id_s, kk > 0);
  }
}

__device__ __forceinline__ void store_row_chunk(uint8_t* tile, int row, int C, const uint32_t* w) {
  // row `row`, tokens 32C..32C+31 of a SW128 tile of 128-byte rows: token
  // block C/2, 16-byte chunks (C&1)*4 .. +3
#pragma unroll
  for (int qq = 0; qq < 4; ++qq)
    *(uint4*)(tile + (C >> 1) * (kTileBytes / 2) + sw128_offset(row, (C & 1) * 4 + qq)) =
        make_uint4(w[4 * qq], w[4 * qq + 1], w[4 * qq + 2], w[4 * qq + 3]);
}

// One 32-position chunk of a row of a gram tile: Xh (packed bf16, the A operand of
// R~ and of the Gram's first term) and 2 (X - Xh), X = exp2(l - lam); X = 0 past
// position vl of the chunk when kMasked.  Pairs of floats as in the scoring kernel.
template <bool kMasked>
__device__ __forceinline__ void gram_chunk(float* v, int vl, float sl2, float lam, uint32_t* hi,
                                           uint32_t* lo, float& vmax, float& xsum) {
  if (kMasked) {
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (e > vl) v[e] = -INFINITY;
  }
#pragma unroll
  for (int e = 0; e < 32; e += 2) vmax = fmaxf(vmax, fmaxf(v[e], v[e + 1]));
  const uint64_t s2 = pack2(sl2, sl2), l2 = pack2(-lam, -lam), minus2 = pack2(-2.f, -2.f);
  uint64_t sum = 0;   // a pair of zeros
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    float x0, x1;
    unpack2(fma2(pack2(v[2 * e], v[2 * e + 1]), s2, l2), x0, x1);
    x0 = fast_exp2(x0);
    x1 = fast_exp2(x1);
    const uint64_t x = pack2(x0, x1);
    sum = add2(sum, x);
    const uint32_t h = pack_bf16(x0, x1);
    hi[e] = h;
    unpack2(fma2(pack2(lo_half(h), hi_half(h)), minus2, add2(x, x)), x0, x1);   // exact
    lo[e] = pack_bf16(x0, x1);
  }
  float s0, s1;
  unpack2(sum, s0, s1);
  xsum += s0 + s1;
}

// Online max / sum of exp2 over one 32-column chunk (log2 units); positions
// past vlim are skipped when kMasked.
template <bool kMasked>
__device__ __forceinline__ void stats32(float* v, int p0, int vlim, float sl2, float& M, float& L) {
  if (kMasked) {
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (p0 + e > vlim) v[e] = -INFINITY;
  }
  float m16[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) m16[e] = fmaxf(v[e], v[e + 16]);
#pragma unroll
  for (int h = 8; h >= 1; h >>= 1)
#pragma unroll
    for (int e = 0; e < h; ++e) m16[e] = fmaxf(m16[e], m16[e + h]);
  if (kMasked && m16[0] == -INFINITY) return;
  const float cm = m16[0] * sl2;
  if (cm > M) {
    L *= fast_exp2(M - cm);
    M = cm;
  }
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int e = 0; e < 32; ++e) s[e & 3] += fast_exp2(fmaf(v[e], sl2, -M));
  L += (s[0] + s[1]) + (s[2] + s[3]);
}

// ======================================================== k_merge_fixed
// One CTA (256 threads) per unit; shared memory holds one key per slot.
__global__ void __launch_bounds__(256) k_merge_fixed(MArgs a) {
  chain_wait();
  extern __shared__ uint32_t fkey[];   // [B] candidate keys, 0 = not a candidate
  __shared__ int hist[256], sh[64];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int u = blockIdx.x;
  const UnitRow ur = unit_row(a.units, u, a.B, a.n_fix);
  const int B = ur.B;
  const int32_t* idx_u = a.idx + ur.off;
  const float* sc_u = a.scores + (size_t)u * a.P;
  // Candidates for the score-ranked part: retained prefix tokens past the sinks.
  // Their scores are non-negative, so every key is above 0.
  // An idx entry outside [0, n) is reported and read as position 0.
  auto pos = [&](int i) {
    const int j = __ldg(idx_u + i);
    return (unsigned)j < (unsigned)a.n ? j : 0;
  };
  int nc = 0;
  for (int i = tid; i < B; i += nt) {
    if ((unsigned)__ldg(idx_u + i) >= (unsigned)a.n) set_status(a.status, GRKV_ERR_INVALID_ARG);
    const int j = pos(i);
    const bool cand = j >= a.n_sink && j < a.P;
    fkey[i] = cand ? max(order_key(__ldg(sc_u + j)), 1u) : 0u;
    nc += cand;
  }
  __syncthreads();
  int ncand;
  (void)block_exclusive_scan(nc, sh + 8, &ncand);
  const int nf = min(ur.n_fix, ncand);
  uint32_t tau = 0xFFFFFFFFu;
  int need_eq = 0;
  if (nf > 0) {
    auto get = [&](int i, uint32_t* key) {
      *key = fkey[i];
      return *key != 0u;
    };
    block_kth_largest(get, B, nf, hist, sh, &tau, &need_eq);
  }
  // fixed: not a candidate, above tau, or among the first need_eq ties
  const int seg = (B + nt - 1) / nt;
  const int lo = min(B, tid * seg), hi = min(B, lo + seg);
  int eq = 0;
  for (int i = lo; i < hi; ++i) eq += (fkey[i] == tau);
  int tot;
  int er = block_exclusive_scan(eq, sh + 8, &tot);
  int keep = 0;
  for (int i = lo; i < hi; ++i) {
    const uint32_t kx = fkey[i];
    bool fixed = kx == 0u || kx > tau;
    if (kx == tau) fixed = er++ < need_eq;
    fkey[i] = fixed ? 1u : 0u;   // each thread rewrites only its own segment
    a.fixed[ur.off + i] = fixed ? 1 : 0;
    keep += !fixed;
  }
  int ng;
  const int gpos = block_exclusive_scan(keep, sh + 8, &ng);
  int g = gpos;
  for (int i = lo; i < hi; ++i) {
    const int at = fkey[i] ? ng + (i - g) : g;
    g += !fkey[i];
    a.src[ur.off + at] = pos(i);
  }
  if (tid == 0) a.ng[u] = ng;
}

// ======================================================== k_merge_gram
// A cluster of a.ranks CTAs (a power of two) per unit and row block, each on a contiguous
// share of the unit's tiles; the shares of R~ and of the Gram meet in distributed shared
// memory, where rank r adds rows [128 r / ranks, 128 (r + 1) / ranks) of all shares
// in rank order and writes them.
//
// With the full-cache row statistics (always in grkv_compress) one phase: X against
// the full row maximum M_r, X' = exp2(l - M_r) = X L'_r with L'_r = sum of X' over the
// visible retained keys, so R = Y - R~'/L'_r and G_ij = G'_ij/(L'_i L'_j).  The
// retained maximum is at most M_r; if it is more than 64 (log2 units) below it for
// some row, or L' underflows, the cluster starts over with two phases, which is
// also the path without statistics: row statistics over the slots, then R~ and
// the Gram over the positions with X itself.
//
// Roles (640 threads): warp 0 the Q load; warps 0, 2, 3 the gathers; warp 1 MMA
// issue; warps 4-19 four compute groups of 128 threads, 32 positions of every
// tile each, one thread per window row (TMEM lane).  A thread copies its 32 logits
// to registers and writes Xh and 2 (X - Xh) over them (TMEM A operands) and XGh =
// Xh of the non-fixed positions to shared memory (the Gram's B operand).
//
// Bound by the gathers (4.4 K cycles per tile of K0 and V0 rows) where a rank has many
// tiles, by latency where it has one.  The shares leave through
// shared memory: stored from TMEM row by row, each instruction touched 32 lines
// and the rows took 16 K cycles of 48 K.
//
// Measured, against one CTA per unit and block, two 128-thread groups on alternate
// tiles, and a second launch for units that start over: 8 units B = 512 44 -> 15 us,
// 64 units with budgets 200 .. 1536 88 -> 26 us, 32 units B = 1024 m = 256 103 -> 22 us,
// 256 units B = 2048 129 -> 99 us (two waves), 84 with the asynchronous gathers.
struct GBars {
  uint64_t ring_full[kRingG], ring_empty[kRingG];
  uint64_t q_full;
  uint64_t s_full[2], x_full[2];   // S written; statistics taken or X written
  uint64_t acc_done, drain;
  uint32_t tmem;
  int abort;
};
static_assert(sizeof(GBars) <= 256, "barrier block");
constexpr int kGroupsG = 4, kWarpsG = 20;

// Float offset of 4-float chunk c of row r in a 128 x 128 fp32 tile whose chunks
// are permuted so that threads on consecutive rows meet different banks.
__device__ __forceinline__ int dump_at(int r, int c) { return r * kD + ((c ^ (r & 31)) << 2); }

__device__ __forceinline__ uint32_t peer_addr(uint32_t saddr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 peer_load4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ float2 peer_load2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];"
               : "=f"(v.x), "=f"(v.y)
               : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ void cluster_bar() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

__global__ void __launch_bounds__(kThreadsG, 1)
    k_merge_gram(const __grid_constant__ CUtensorMap tmQ, MArgs a) {
  chain_wait();
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  GBars* bars = (GBars*)(sm + kOffBar);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler
  const int C = a.ranks, rank = blockIdx.x % C, ub = blockIdx.x / C;
  const int u = ub / a.nrb, row0 = (ub % a.nrb) * kRows;   // window rows row0 .. row0 + 127
  const UnitRow ur = unit_row(a.units, u, a.B, a.n_fix);
  const int B = ur.B, T = (B + kTile - 1) / kTile;
  // A unit is split as launch_gram splits a call at its own budget, so that its sums, and
  // with them its results' last bits, do not follow the largest budget of the call.
  const int lg = min(31 - __clz(C), 31 - __clz(T));        // 2^lg ranks hold tiles
  const int ta = min(T, (T * rank) >> lg), tb = min(T, (T * (rank + 1)) >> lg);   // this rank's
  const int ng = __ldg(a.ng + u);
  if (tid == 0) {
    for (int i = 0; i < kRingG; ++i) {
      mbar_init(&bars->ring_full[i], 1);   // the gathering warp
      mbar_init(&bars->ring_empty[i], 1);
    }
    mbar_init(&bars->q_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->s_full[i], 1);
      mbar_init(&bars->x_full[i], 4 * kGroupsG);
    }
    mbar_init(&bars->acc_done, 1);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem, 512);
    tmem_relinquish();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem;
  volatile int* abort_flag = &bars->abort;
  float* dump_r = (float*)(sm + kOffRing);                     // [128][128] (dump_at)
  float* dump_g = (float*)(sm + kOffRing + 2 * kTileBytes);
  float2* stat = (float2*)(sm + kOffXG);                       // [kGroupsG][128]
  float* cs = (float*)(sm + kOffXG) + 2 * kGroupsG * kRows;    // [128] 1 / L'_r
  const uint32_t stat_a = smem_u32(stat);

  const bool gathers = warp == 0 || warp == 2 || warp == 3, computes = warp >= 4;
  const int g = (warp - 4) >> 2, q = warp & 3, row = q * 32 + lane, grow = row0 + row;
  const int pw = warp == 0 ? 0 : warp - 1;
  const bool row_ok = grow < a.m;
  // slots / positions past vlim are invisible to this row (and so are those >= B)
  const int vlim = a.causal ? B - a.w + grow % a.w : B - 1;
  const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
  uint32_t use = 0, job = 0;   // ring loads (gathers, MMA warp) and S tiles (MMA warp, compute) so far
  bool single = a.rstats != nullptr, ok = true;
  float lam = INFINITY;
  if (single && computes && row_ok)
    lam = __ldg(a.rstats + ((size_t)u * a.m + grow) * 2) * 1.4426950408889634f;
  if (warp == 0 && lane == 0) {
    prefetch_tensormap(&tmQ);
    mbar_expect_tx(&bars->q_full, kTileBytes);
    const uint64_t pol = l2_evict_last();
    tma_load_3d(sm + kOffQ, &tmQ, &bars->q_full, 0, row0, u, pol);
    tma_load_3d(sm + kOffQ + kTileBytes / 2, &tmQ, &bars->q_full, 64, row0, u, pol);
  }

  // phase 0: statistics over the slots (K0); phase 1: R~ and the Gram over the
  // positions (K0 and V0)
  for (int ph = single ? 1 : 0, acc_use = 0;;) {
    float M = -INFINITY, L = 0.f;   // phase 0: row statistics; phase 1: largest logit, sum of X
    if (gathers) {
      // the phase's loads in turn to the three warps, a whole tile each
      __syncwarp();
      const int32_t* rows_u = (ph ? a.src : a.idx) + ur.off;
      const int per = ph + 1, loads = (tb - ta) * per;   // K0 of a tile, in phase 1 then its V0
      int next[4];
      if (pw < loads) gather_index<4>(rows_u, (ta + pw / per) * kTile, B, a.n, lane, next);
      for (int i = pw; i < loads; i += 3) {
        const int j[4] = {next[0], next[1], next[2], next[3]};
        if (i + 3 < loads) gather_index<4>(rows_u, (ta + (i + 3) / per) * kTile, B, a.n, lane, next);
        const uint32_t n = use + i, slot = n % kRingG;
        if (n >= kRingG) ok = ok && mbar_wait_warp(&bars->ring_empty[slot], (n / kRingG - 1) & 1, abort_flag);
        if (!ok) break;
        gather_async<4>(smem_u32(sm + kOffRing + slot * kTileBytes), 0,
                        (ph && (i & 1) ? a.v : a.k) + (size_t)u * a.n * kD, j, lane);
        gather_arrive(&bars->ring_full[slot], lane);
      }
      use += loads;
    } else if (warp == 1) {
      constexpr uint32_t id_s = idesc_bf16(kRows, kTile, 0, 0);   // S = Q K0^T
      constexpr uint32_t id_r = idesc_bf16(kRows, kD, 0, 1);      // R~ += Xh V0 (V0 MN-major)
      constexpr uint32_t id_g = idesc_bf16(kRows, kRows, 0, 0);   // G += A XGh^T
      constexpr uint32_t kTileDesc = kTileBytes >> 4;             // in descriptor units
      const uint64_t q_desc = sw128_desc(smem_u32(sm + kOffQ), 16, 1024);
      const uint64_t k_desc = sw128_desc(smem_u32(sm + kOffRing), 16, 1024);
      const uint64_t v_desc = sw128_desc(smem_u32(sm + kOffRing), kTileBytes / 2, 1024);
      const uint64_t x_desc = sw128_desc(smem_u32(sm + kOffXG), 16, 1024);
      ok = ok && mbar_wait_warp(&bars->q_full, 0, abort_flag);
      // after the next tile's S: the job's X is there (phase 0: its logits are read)
      auto finish = [&](int t, uint32_t jb, uint32_t vuse) -> bool {
        const uint32_t b = jb & 1;
        if (!mbar_wait_warp(&bars->x_full[b], (jb >> 1) & 1, abort_flag)) return false;
        if (!ph) return true;
        const uint32_t vs = vuse % kRingG;
        if (!mbar_wait_warp(&bars->ring_full[vs], (vuse / kRingG) & 1, abort_flag)) return false;
        tc_fence_after();
        const uint32_t hi = tmem + kColS + b * kTile;
        mma8_ts<id_r, false>(tmem + kColR, hi, v_desc + vs * kTileDesc, t > ta);
        if (t * kTile < ng) {   // the tile has non-fixed positions
          mma8_ts<id_g, true>(tmem + kColG, hi, x_desc + b * kTileDesc, t > ta);
          mma8_ts<id_g, true>(tmem + kColG, hi + 16, x_desc + b * kTileDesc, true);
        }
        mma_commit_elect(&bars->ring_empty[vs]);
        return true;
      };
      uint32_t pv = 0;
      for (int t = ta; t < tb && ok; ++t, ++job) {
        const uint32_t b = job & 1, ks = use % kRingG;
        ok = mbar_wait_warp(&bars->ring_full[ks], (use / kRingG) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        // the buffer's last X was read by MMAs issued before, its last logits by finish()
        mma8_ss<id_s>(tmem + kColS + b * kTile, q_desc, k_desc + ks * kTileDesc);
        mma_commit_elect(&bars->ring_empty[ks]);
        mma_commit_elect(&bars->s_full[b]);
        if (t > ta) ok = finish(t - 1, job - 1, pv);
        pv = use + 1;
        use += ph ? 2 : 1;
      }
      if (ok && tb > ta) ok = finish(tb - 1, job - 1, pv);
      if (ph) mma_commit_elect(&bars->acc_done);
    } else {
      for (int t = ta; t < tb && ok; ++t, ++job) {
        const uint32_t b = job & 1;
        const int p0 = t * kTile + 32 * g;
        // s_full also says that the MMAs that read this buffer's XGh have completed
        ok = mbar_wait_warp(&bars->s_full[b], (job >> 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t sbase = lane_addr + kColS + b * kTile + 32 * g;
        float v[32];
        tmem_ld32f(sbase, v);
        tmem_wait32(v);
        const bool full = __all_sync(0xffffffffu, p0 + 31 <= vlim);
        if (!ph) {
          if (full)
            stats32<false>(v, p0, vlim, a.sl2, M, L);
          else
            stats32<true>(v, p0, vlim, a.sl2, M, L);
          __syncwarp();
        } else {
          uint32_t hi[16], lo[16];
          if (full)
            gram_chunk<false>(v, 0, a.sl2, lam, hi, lo, M, L);
          else
            gram_chunk<true>(v, vlim - p0, a.sl2, lam, hi, lo, M, L);
          tmem_st16(sbase, hi);
          tmem_st16(sbase + 16, lo);
          if (t * kTile < ng) {
            const int gn = ng - p0;   // the chunk's non-fixed positions
            if (gn < 32) {
#pragma unroll
              for (int e = 0; e < 16; ++e)
                hi[e] &= (2 * e < gn ? 0xFFFFu : 0u) | (2 * e + 1 < gn ? 0xFFFF0000u : 0u);
            }
            store_row_chunk(sm + kOffXG + b * kTileBytes, row, g, hi);
          }
          tmem_st_wait();
          fence_proxy_async_smem();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->x_full[b]);
      }
    }

    if (ph == 0) {
      // every rank's and group's statistics of the rows give the normalisers
      if (computes) stat[g * kRows + row] = make_float2(M, L);
      cluster_bar();
      if (computes) {
        M = -INFINITY;
        L = 0.f;
        for (int r = 0; r < C; ++r)
          for (int h = 0; h < kGroupsG; ++h) {
            const float2 o = peer_load2(peer_addr(stat_a + (h * kRows + row) * 8, r));
            if (o.x == -INFINITY) continue;
            if (o.x > M) {
              L = L * fast_exp2(M - o.x) + o.y;
              M = o.x;
            } else {
              L += o.y * fast_exp2(o.x - M);
            }
          }
        lam = (row_ok && L > 0.f) ? M + __log2f(L) : INFINITY;
        if (rank == 0 && g == 0) a.lam[(size_t)u * a.ldr + grow] = lam;
      }
      cluster_bar();   // the peers have read: the XGh tiles may be written
      ph = 1;
      continue;
    }

    // the rank's shares to shared memory: every gathered tile has been multiplied
    if (computes) {
      ok = ok && mbar_wait_warp(&bars->acc_done, acc_use & 1, abort_flag);
      tc_fence_after();
      stat[g * kRows + row] = make_float2(M, L);
      const bool any = ok && tb > ta, any_g = any && ta * kTile < ng;   // MMAs that ran
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        float v[32];
        tmem_ld32f(lane_addr + (h ? kColG : kColR) + 32 * g, v);
        tmem_wait32(v);
        const bool have = h ? any_g : any;
        float* d = h ? dump_g : dump_r;
#pragma unroll
        for (int c = 0; c < 8; ++c)
          *(float4*)(d + dump_at(row, 8 * g + c)) =
              have ? make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3])
                   : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      tc_fence_before();
    }
    ++acc_use;
    fence_proxy_async_smem();   // a second attempt gathers over the shares
    cluster_bar();
    bool bad = false;
    if (single && tid < kRows) {
      const int gr = row0 + tid;
      float vm = -INFINITY, ls = 0.f;
      for (int r = 0; r < C; ++r)
        for (int h = 0; h < kGroupsG; ++h) {
          const float2 o = peer_load2(peer_addr(stat_a + (h * kRows + tid) * 8, r));
          vm = fmaxf(vm, o.x);
          ls += o.y;
        }
      const bool in = gr < a.m;
      const float full = in ? __ldg(a.rstats + ((size_t)u * a.m + gr) * 2) * 1.4426950408889634f : 0.f;
      bad = in && !(ls > 0.f && full - vm * a.sl2 <= 64.f);
      cs[tid] = in && ls > 0.f ? 1.f / ls : 0.f;
      if (rank == 0) a.lam[(size_t)u * a.ldr + gr] = in && ls > 0.f ? full + __log2f(ls) : INFINITY;
    }
    if (__syncthreads_or(bad)) {   // the same answer in every rank
      single = false;
      ph = 0;
      cluster_bar();   // the peers have read the statistics
      continue;
    }
    // rows r0 .. r1 - 1 of R and of the Gram block: a warp per row, a lane per four columns
    const int r0 = kRows * rank / C, r1 = kRows * (rank + 1) / C;
    const uint32_t ra = smem_u32(dump_r), ga = smem_u32(dump_g);
    for (int r = r0 + warp; r < r1; r += kWarpsG) {
      const int gr = row0 + r, c = 4 * lane;
      const uint32_t off = dump_at(r, lane) * 4;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f), z = x, o = x, y = x;
      if (gr < a.m) y = __ldg((const float4*)(a.y + ((size_t)u * a.m + gr) * kD + c));
      for (int p = 0; p < C; ++p) {
        const float4 xr = peer_load4(peer_addr(ra + off, p)), zr = peer_load4(peer_addr(ga + off, p));
        x = make_float4(x.x + xr.x, x.y + xr.y, x.z + xr.z, x.w + xr.w);
        z = make_float4(z.x + zr.x, z.y + zr.y, z.z + zr.z, z.w + zr.w);
      }
      const float ci = single ? cs[r] : 1.f;
      const float4 cj = single ? *(const float4*)(cs + c) : make_float4(1.f, 1.f, 1.f, 1.f);
      const bool in = gr < a.m;
      if (!ok) continue;
      *(float4*)(a.rz + ((size_t)u * a.ldr + gr) * kD + c) =
          in ? make_float4(y.x - ci * x.x, y.y - ci * x.y, y.z - ci * x.z, y.w - ci * x.w) : o;
      const int gc = row0 + c;
      if (in)
        o = make_float4(gc < a.m ? z.x * (ci * cj.x) : 0.f, gc + 1 < a.m ? z.y * (ci * cj.y) : 0.f,
                        gc + 2 < a.m ? z.z * (ci * cj.z) : 0.f,
                        gc + 3 < a.m ? z.w * (ci * cj.w) : 0.f);
      *(float4*)(a.gram + ((size_t)u * a.ldr + gr) * a.ldr + gc) = o;
    }
    cluster_bar();   // no rank leaves while a peer reads its shares
    break;
  }
  if (warp == 0 && lane == 0) mbar_drain(&bars->q_full, 0);
  if (warp == 1) {
    // every MMA issued completes before TMEM is released
    mma_commit_elect(&bars->drain);
    mbar_drain(&bars->drain, 0);
  }
  if (!ok && lane == 0) set_status(a.status, GRKV_ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// ======================================================== k_merge_cross
// The off-diagonal Gram block of a unit with two row blocks (128 < m <= 256):
// G01 = X_G0 X_G1^T over the non-fixed positions, as the split products
// Xh0 Xh1^T + Xl0 Xh1^T + Xh0 Xl1^T (the low-low term dropped, as in the
// diagonal blocks).  X uses the final row normalisers of both blocks (from
// the diagonal launches), so nothing is rescaled afterwards.  G01 goes to
// gram[u][r0][128 + r1].  Roles
// (384 threads): warp 0 the Q loads; warps 0, 2, 3 the K0 gathers; warp 1 MMA
// issue; warps 4-7 the rows of block 0 (X_0 high / low parts written back
// over S_0 in TMEM, the A operands); warps 8-11 the rows of block 1 (XGh_1,
// XGl_1 in shared memory, the B operands).  One tile in flight: the S MMAs of
// a tile are issued after the Gram MMAs of the previous one, so s_full also
// tells both groups that their buffers are free.
struct CBars {
  uint64_t ring_full[2], ring_empty[2];
  uint64_t q_full, s_full, x0_full, x1_full, acc_done, drain;
  uint32_t tmem;
  int abort;
};
static_assert(sizeof(CBars) <= 256, "barrier block");
constexpr uint32_t kOffQ1C = kTileBytes, kOffRingC = 2 * kTileBytes, kOffXhC = 4 * kTileBytes,
                   kOffXlC = 5 * kTileBytes, kOffBarC = 6 * kTileBytes;
constexpr uint32_t kSmemBytesC = kOffBarC + 256 + 1024;

__global__ void __launch_bounds__(kThreads, 1)
    k_merge_cross(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                  MArgs a) {
  chain_wait();
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  CBars* bars = (CBars*)(sm + kOffBarC);
  uint8_t* xgh = sm + kOffXhC;
  uint8_t* xgl = sm + kOffXlC;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int u = blockIdx.x;
  const UnitRow ur = unit_row(a.units, u, a.B, a.n_fix);
  const int B = ur.B;
  const int ng = __ldg(a.ng + u), TG = (ng + kTile - 1) / kTile;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->ring_full[i], 3);   // one expect_tx arrival per gathering warp
      mbar_init(&bars->ring_empty[i], 1);
    }
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->s_full, 1);
    mbar_init(&bars->x0_full, 128);
    mbar_init(&bars->x1_full, 128);
    mbar_init(&bars->acc_done, 1);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem, 512);
    tmem_relinquish();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem;
  volatile int* abort_flag = &bars->abort;
  constexpr uint32_t kColS0 = 0, kColS1 = 128, kColGC = 256;

  if (warp == 0 || warp == 2 || warp == 3) {
    if (warp == 0 && lane == 0) {
      prefetch_tensormap(&tmQ);
      mbar_expect_tx(&bars->q_full, 2 * kTileBytes);
      const uint64_t pol = l2_evict_last();
      for (int h = 0; h < 2; ++h) {
        tma_load_3d(sm + h * kTileBytes, &tmQ, &bars->q_full, 0, h * kRows, u, pol);
        tma_load_3d(sm + h * kTileBytes + kTileBytes / 2, &tmQ, &bars->q_full, 64, h * kRows, u, pol);
      }
    }
    __syncwarp();
    const int32_t* src_u = a.src + ur.off;
    const int pw = warp == 0 ? 0 : warp - 1;
    Gatherer<2, 3> gt{sm + kOffRingC, bars->ring_full, bars->ring_empty};
    int jn[4];
    if (TG > 0) gt.rows(src_u, B, a.n, u * a.n, 0, pw, lane, jn);
    bool ok = true;
    for (int t = 0; t < TG && ok; ++t) {
      const int j[4] = {jn[0], jn[1], jn[2], jn[3]};
      if (t + 1 < TG) gt.rows(src_u, B, a.n, u * a.n, t + 1, pw, lane, jn);
      ok = gt.load(&tmK, j, pw, lane, abort_flag);
    }
    gt.drain();
    if (warp == 0 && lane == 0) mbar_drain(&bars->q_full, 0);
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t id_g = idesc_bf16(kRows, kRows, 0, 0);   // G01 += A XG1^T
      bool ok = mbar_wait(&bars->q_full, 0, abort_flag, kBudget);
      const uint32_t qa0 = smem_u32(sm), qa1 = smem_u32(sm + kOffQ1C);
      const uint32_t ha = smem_u32(xgh), la = smem_u32(xgl);
      for (int t = 0; t < TG && ok; ++t) {
        ok = mbar_wait(&bars->ring_full[t & 1], (t >> 1) & 1, abort_flag, kBudget);
        if (!ok) break;
        tc_fence_after();
        const uint32_t ka = smem_u32(sm + kOffRingC + (t & 1) * kTileBytes);
        issue_s(tmem + kColS0, qa0, ka);
        issue_s(tmem + kColS1, qa1, ka);
        mma_commit(&bars->ring_empty[t & 1]);
        mma_commit(&bars->s_full);
        ok = mbar_wait(&bars->x0_full, t & 1, abort_flag, kBudget);
        if (ok) ok = mbar_wait(&bars->x1_full, t & 1, abort_flag, kBudget);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk) {
          const uint32_t off = (kk >> 2) * (kTileBytes / 2) + (kk & 3) * 32;
          mma_bf16_ts(tmem + kColGC, tmem + kColS0 + xt_col(kk, 0), sw128_desc(ha + off, 16, 1024),
                      id_g, (t > 0 || kk > 0));
        }
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk) {
          const uint32_t off = (kk >> 2) * (kTileBytes / 2) + (kk & 3) * 32;
          mma_bf16_ts(tmem + kColGC, tmem + kColS0 + xt_col(kk, 1), sw128_desc(ha + off, 16, 1024),
                      id_g, 1);
        }
#pragma unroll
        for (int kk = 0; kk < kTile / 16; ++kk) {
          const uint32_t off = (kk >> 2) * (kTileBytes / 2) + (kk & 3) * 32;
          mma_bf16_ts(tmem + kColGC, tmem + kColS0 + xt_col(kk, 0), sw128_desc(la + off, 16, 1024),
                      id_g, 1);
        }
      }
      mma_commit(&bars->acc_done);
      mma_commit(&bars->drain);
      mbar_drain(&bars->drain, 0);
    }
  } else {
    const int grp = (warp - 4) >> 2, q = warp & 3, row = q * 32 + lane;
    const int grow = grp * kRows + row;
    const float lam = grow < a.m ? a.lam[(size_t)u * a.ldr + grow] : INFINITY;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const uint32_t sbase = lane_addr + (grp ? kColS1 : kColS0);
    bool ok = true;
    for (int t = 0; t < TG && ok; ++t) {
      ok = mbar_wait_warp(&bars->s_full, t & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      float v[32];
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        tmem_ld32f(sbase + 32 * c, v);
        tmem_wait32(v);
        uint32_t hi[16], lo[16];
        const int p0 = t * kTile + 32 * c;
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          const float x0 = p0 + e < ng ? fast_exp2(fmaf(v[e], a.sl2, -lam)) : 0.f;
          const float x1 = p0 + e + 1 < ng ? fast_exp2(fmaf(v[e + 1], a.sl2, -lam)) : 0.f;
          const uint32_t h = pack_bf16(x0, x1);
          hi[e / 2] = h;
          lo[e / 2] = pack_bf16(x0 - lo_half(h), x1 - hi_half(h));
        }
        if (grp == 0) {
          tmem_st16(sbase + 32 * c, hi);
          tmem_st16(sbase + 32 * c + 16, lo);
        } else {
          store_row_chunk(xgh, row, c, hi);
          store_row_chunk(xgl, row, c, lo);
        }
      }
      if (grp == 0) {
        tmem_st_wait();
      } else {
        fence_proxy_async_smem();
      }
      tc_fence_before();
      mbar_arrive(grp == 0 ? &bars->x0_full : &bars->x1_full);
    }
    if (grp == 0) {
      if (ok) ok = mbar_wait_warp(&bars->acc_done, 0, abort_flag);
      tc_fence_after();
      if (ok) {
        float* up = a.gram + ((size_t)u * a.ldr + row) * a.ldr + kRows;   // row r0, columns 128 + r1
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float g[32];
          tmem_ld32f(lane_addr + kColGC + 32 * c, g);
          tmem_wait32(g);
#pragma unroll
          for (int e = 0; e < 32; e += 4)
            *(float4*)(up + 32 * c + e) = TG > 0 ? make_float4(g[e], g[e + 1], g[e + 2], g[e + 3])
                                                 : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
    if (!ok && row == 0) set_status(a.status, GRKV_ERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// ======================================================== k_merge_update
// Slot order, a unit's tiles over `split` CTAs, 736 threads.  Roles: warp 0 the Q load and
// the K_out tile stores, warp 22 the V_out tile stores; warp 1 MMA issue;
// warps 2, 3, 16, 17 the K0 gathers (TMA) and 18-21 the V0 gathers (cp.async; two-slot rings
// each, on all four SM sub-partitions); warps 4-7 and 8-11
// two compute groups taking alternate tiles (one thread per token = TMEM lane
// of S^T): X_G^T from S^T, zero for fixed slots, written back over S^T as
// packed bf16 (rows 32c .. 32c+31 of chunk c: high parts to columns 32c ..
// 32c+15, low parts to 32c+16 .. 32c+31, each chunk read before it is
// overwritten); warps 12-15 the epilogue (thread = token): V_out = V0 + dV in
// the V0 tile, which warp 22 then stores.  A fixed slot has X = 0 and so
// dV = 0: its row is left as V0.
struct UBars {
  uint64_t k_full[2], k_empty[2], v_full[2], v_empty[2];
  uint64_t q_full;
  uint64_t s_full[2], x_full[2], d_full[2], d_empty[2], vo_full[2];
  uint64_t drain;
  uint32_t tmem;
  int abort;
};
static_assert(sizeof(UBars) <= 256, "barrier block");
constexpr uint32_t kOffKU = kTileBytes;                    // K0 ring, 2 tiles
constexpr uint32_t kOffVU = kOffKU + 2 * kTileBytes;       // V0 / V_out ring, 2 tiles
constexpr uint32_t kOffZU = kOffVU + 2 * kTileBytes;       // Zh, Zl
constexpr uint32_t kOffLamU = kOffBar + 256;               // [128] row normalisers
static_assert(kOffZU + 2 * kTileBytes == kOffBar, "update shared-memory layout");
constexpr uint32_t kSmemBytesU = kOffLamU + kRows * 4 + 1024;

// The first `rows` rows of a swizzled tile to consecutive rows of an output, by one warp.
__device__ __forceinline__ void copy_rows(__nv_bfloat16* dst, const uint8_t* tile, int rows, int lane) {
#pragma unroll 4
  for (int i = lane; i < rows * 16; i += 32) {
    const int r = i >> 4, c = i & 15;
    *(uint4*)(dst + (size_t)r * kD + c * 8) =
        *(const uint4*)(tile + (c >> 3) * (kTileBytes / 2) + sw128_offset(r, c & 7));
  }
}

__global__ void __launch_bounds__(kThreadsU, 1)
    k_merge_update(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmKo, const __grid_constant__ CUtensorMap tmVo,
                   MArgs a) {
  chain_wait();
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  UBars* bars = (UBars*)(sm + kOffBar);
  float* lam_s = (float*)(sm + kOffLamU);
  uint8_t* zh = sm + kOffZU;
  uint8_t* zl = zh + kTileBytes;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler
  // the CTA's tiles T0 .. T0 + T - 1 of the unit (`split` CTAs per unit)
  const int u = blockIdx.x / a.split, part = blockIdx.x - u * a.split;
  const UnitRow ur = unit_row(a.units, u, a.B, a.n_fix);
  const int B = ur.B, Tu = (B + kTile - 1) / kTile;
  const int T0 = (int)((long long)part * Tu / a.split);
  const int T = (int)((long long)(part + 1) * Tu / a.split) - T0, S0 = T0 * kTile;
  const int32_t* idx_u = a.idx + ur.off;
  // packed outputs (budgets of their own): tiles are addressed by row, and a unit's last,
  // partial tile is copied by a warp so that it ends where the next unit's rows begin
  const bool packed = a.units != nullptr;
  const int out_y = packed ? (int)ur.off + S0 : S0, out_z = packed ? 0 : u;
  const int t_part = packed && S0 + T * kTile > B ? T - 1 : -1;   // the partial tile, if any
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->k_full[i], 4);    // one expect_tx arrival per gathering warp
      mbar_init(&bars->v_full[i], 128);  // every gathering thread, once its copies have landed
      mbar_init(&bars->k_empty[i], 2);   // the S^T MMA and the K_out store
      mbar_init(&bars->v_empty[i], 1);   // the V_out store
      mbar_init(&bars->s_full[i], 1);
      mbar_init(&bars->x_full[i], 128);
      mbar_init(&bars->d_full[i], 1);
      mbar_init(&bars->d_empty[i], 128);
      mbar_init(&bars->vo_full[i], 128);
    }
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem, 512);
    tmem_relinquish();
  }
  // rows past m have lam = +inf and give X = 0
  if (tid < kRows) lam_s[tid] = a.lam[(size_t)u * a.ldr + a.row0 + tid];
  // Z (fp32 [row][d]) to the bf16 B operands Zh, Zl: MN-major tiles of
  // 128-byte rows (d contiguous), two blocks of 64 columns
  {
    const float* Z = a.rz + ((size_t)u * a.ldr + a.row0) * kD;
    for (int i = tid; i < kRows * (kD / 8); i += kThreadsU) {
      const int r = i >> 4, d8 = i & 15;
      const float4 z0 = __ldg((const float4*)(Z + r * kD + d8 * 8));
      const float4 z1 = __ldg((const float4*)(Z + r * kD + d8 * 8 + 4));
      const float zz[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
      uint32_t h[4], l[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h[j] = pack_bf16(zz[2 * j], zz[2 * j + 1]);
        l[j] = pack_bf16(zz[2 * j] - lo_half(h[j]), zz[2 * j + 1] - hi_half(h[j]));
      }
      const uint32_t off = (d8 >> 3) * (kTileBytes / 2) + sw128_offset(r, d8 & 7);
      *(uint4*)(zh + off) = make_uint4(h[0], h[1], h[2], h[3]);
      *(uint4*)(zl + off) = make_uint4(l[0], l[1], l[2], l[3]);
    }
    fence_proxy_async_smem();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem;
  volatile int* abort_flag = &bars->abort;

  if (warp == 0) {
    if (lane == 0) {
      prefetch_tensormap(&tmQ);
      prefetch_tensormap(&tmKo);
      mbar_expect_tx(&bars->q_full, kTileBytes);
      const uint64_t pol = l2_evict_last();
      tma_load_3d(sm + kOffQ, &tmQ, &bars->q_full, 0, a.row0, u, pol);
      tma_load_3d(sm + kOffQ + kTileBytes / 2, &tmQ, &bars->q_full, 64, a.row0, u, pol);
      // K_out = K0 tile by tile (the map clips the rows past B)
      bool ok = true;
      for (int t = 0; t < T && ok; ++t) {
        const int sl = t & 1;
        ok = mbar_wait(&bars->k_full[sl], (t >> 1) & 1, abort_flag, kBudget);
        if (!ok) break;
        if (a.upd_mode != 2 && t != t_part) {   // the second row block's K_out is the first's
          const uint8_t* kt = sm + kOffKU + sl * kTileBytes;
          tma_store_3d(&tmKo, kt, 0, out_y + t * kTile, out_z);
          tma_store_3d(&tmKo, kt + kTileBytes / 2, 64, out_y + t * kTile, out_z);
          bulk_commit();
          bulk_wait_read<0>();
        }
        mbar_arrive(&bars->k_empty[sl]);
      }
      bulk_wait_all();
      mbar_drain(&bars->q_full, 0);
      if (!ok) set_status(a.status, GRKV_ERR_TIMEOUT);
    }
    __syncwarp();
    if (t_part >= 0 && a.upd_mode != 2 &&
        mbar_wait_warp(&bars->k_full[t_part & 1], (t_part >> 1) & 1, abort_flag))
      copy_rows(a.k_out + (ur.off + S0 + (size_t)t_part * kTile) * kD,
                sm + kOffKU + (t_part & 1) * kTileBytes, B - S0 - t_part * kTile, lane);
  } else if (warp == 22) {
    if (lane == 0) {
      prefetch_tensormap(&tmVo);
      // V_out tile by tile, once the epilogue has written it
      bool ok = true;
      for (int t = 0; t < T && ok; ++t) {
        const int sl = t & 1;
        ok = mbar_wait(&bars->vo_full[sl], (t >> 1) & 1, abort_flag, kBudget);
        if (!ok) break;
        if (a.upd_mode != 1 && t != t_part) {   // mode 1 leaves its result in vpart
          const uint8_t* vt = sm + kOffVU + sl * kTileBytes;
          tma_store_3d(&tmVo, vt, 0, out_y + t * kTile, out_z);
          tma_store_3d(&tmVo, vt + kTileBytes / 2, 64, out_y + t * kTile, out_z);
          bulk_commit();
          bulk_wait_read<0>();
        }
        mbar_arrive(&bars->v_empty[sl]);
      }
      bulk_wait_all();
      if (!ok) set_status(a.status, GRKV_ERR_TIMEOUT);
    }
    __syncwarp();
    if (t_part >= 0 && a.upd_mode != 1 &&
        mbar_wait_warp(&bars->vo_full[t_part & 1], (t_part >> 1) & 1, abort_flag))
      copy_rows(a.v_out + (ur.off + S0 + (size_t)t_part * kTile) * kD,
                sm + kOffVU + (t_part & 1) * kTileBytes, B - S0 - t_part * kTile, lane);
  } else if (warp == 2 || warp == 3 || warp == 16 || warp == 17) {
    // K0 gathers
    const int pw = warp < 4 ? warp - 2 : warp - 14, row0 = u * a.n;
    Gatherer<2, 4> g{sm + kOffKU, bars->k_full, bars->k_empty};
    int jn[4];
    if (T > 0) g.rows(idx_u, B, a.n, row0, T0, pw, lane, jn);
    bool ok = true;
    for (int t = 0; t < T && ok; ++t) {
      const int j[4] = {jn[0], jn[1], jn[2], jn[3]};
      if (t + 1 < T) g.rows(idx_u, B, a.n, row0, T0 + t + 1, pw, lane, jn);
      ok = g.load(&tmK, j, pw, lane, abort_flag);
    }
    g.drain();
  } else if (warp >= 18 && warp < 22) {
    // V0 gathers: a quarter of every tile each (own ring, so that a K tile never waits
    // for a V slot); only threads read a V0 tile, so the copies themselves arrive
    const int r0 = 32 * (warp - 18);
    const __nv_bfloat16* v0 = a.v + (size_t)u * a.n * kD;
    // mode 2 builds V_out from vpart: no V0 tiles
    const int TG = a.upd_mode == 2 ? 0 : T;
    int next[1];
    if (TG > 0) gather_index<1>(idx_u, T0 * kTile + r0, B, a.n, lane, next);
    for (int t = 0; t < TG; ++t) {
      const int j[1] = {next[0]}, sl = t & 1;
      if (t + 1 < TG) gather_index<1>(idx_u, (T0 + t + 1) * kTile + r0, B, a.n, lane, next);
      if (t >= 2 && !mbar_wait_warp(&bars->v_empty[sl], ((t >> 1) - 1) & 1, abort_flag)) break;
      gather_async<1>(smem_u32(sm + kOffVU + sl * kTileBytes), r0, v0, j, lane);
      cp_async_arrive(&bars->v_full[sl]);
    }
    cp_async_wait_all();
  } else if (warp == 1) {
    // the whole warp walks the tiles, an elected lane issues (as in the scoring kernel)
    constexpr uint32_t id_s = idesc_bf16(kTile, kRows, 0, 0);   // S^T = K0 Q^T
    constexpr uint32_t id_d = idesc_bf16(kTile, kD, 0, 1);      // dV = X_G^T Z (Z MN-major)
    const uint64_t q_desc = sw128_desc(smem_u32(sm + kOffQ), 16, 1024);
    const uint64_t k_desc = sw128_desc(smem_u32(sm + kOffKU), 16, 1024);
    const uint64_t zh_desc = sw128_desc(smem_u32(zh), kTileBytes / 2, 1024);
    const uint64_t zl_desc = sw128_desc(smem_u32(zl), kTileBytes / 2, 1024);
    bool ok = mbar_wait_warp(&bars->q_full, 0, abort_flag);
    auto issue_d = [&](int t) -> bool {
      const uint32_t d = tmem + kColD + (t & 1) * kD, x = tmem + kColS + (t & 1) * kTile;
      if (!mbar_wait_warp(&bars->x_full[t & 1], (t >> 1) & 1, abort_flag)) return false;
      if (t >= 2 && !mbar_wait_warp(&bars->d_empty[t & 1], ((t >> 1) - 1) & 1, abort_flag)) return false;
      tc_fence_after();
      mma8_ts<id_d, false>(d, x, zh_desc, false);
      mma8_ts<id_d, false>(d, x, zl_desc, true);
      mma8_ts<id_d, false>(d, x + 16, zh_desc, true);
      mma_commit_elect(&bars->d_full[t & 1]);
      return true;
    };
    for (int t = 0; t < T && ok; ++t) {
      const int sl = t & 1;
      ok = mbar_wait_warp(&bars->k_full[sl], (t >> 1) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      // S^T into buffer sl: its previous contents (X_G^T of tile t - 2) were
      // read by the dV MMAs issued before this one
      mma8_ss<id_s>(tmem + kColS + sl * kTile, k_desc + sl * (kTileBytes >> 4), q_desc);
      mma_commit_elect(&bars->k_empty[sl]);
      mma_commit_elect(&bars->s_full[sl]);
      if (t >= 1) ok = issue_d(t - 1);
    }
    if (ok && T > 0) ok = issue_d(T - 1);
    mma_commit_elect(&bars->drain);
    mbar_drain(&bars->drain, 0);
  } else if (warp >= 4 && warp < 12) {
    // compute groups: group cg takes the tiles t with t % 2 == cg
    const int cg = (warp - 4) >> 2, q = warp & 3, tok = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    bool ok = true;
    for (int t = cg; t < T && ok; t += 2) {
      const int sl = t & 1, slot = S0 + t * kTile + tok;
      const bool zero = slot >= B || __ldg(a.fixed + ur.off + min(slot, B - 1)) != 0;
      ok = mbar_wait_warp(&bars->s_full[sl], (t >> 1) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t sbase = lane_addr + kColS + sl * kTile;
      float v[32];
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        tmem_ld32f(sbase + 32 * c, v);
        tmem_wait32(v);
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          const float4 l4 = *(const float4*)(lam_s + 32 * c + (e & ~3));
          const float la = (e & 2) ? l4.z : l4.x, lb = (e & 2) ? l4.w : l4.y;
          float x0 = fast_exp2(fmaf(v[e], a.sl2, -la)), x1 = fast_exp2(fmaf(v[e + 1], a.sl2, -lb));
          if (zero) x0 = x1 = 0.f;
          const uint32_t h = pack_bf16(x0, x1);
          hi[e / 2] = h;
          lo[e / 2] = pack_bf16(x0 - lo_half(h), x1 - hi_half(h));
        }
        tmem_st16(sbase + 32 * c, hi);
        tmem_st16(sbase + 32 * c + 16, lo);
      }
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(&bars->x_full[sl]);
    }
    if (!ok && tok == 0 && cg == 0) set_status(a.status, GRKV_ERR_TIMEOUT);
  } else if (warp >= 12 && warp < 16) {
    // epilogue: thread = token (TMEM lane of D).  Mode 0: V_out = V0 + dV in
    // the V tile; mode 1: vpart = V0 + dV (fp32, every retained slot); mode 2:
    // V_out = vpart + dV into the V tile slot (no V0 there)
    const int q = warp & 3, tok = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const int mode = a.upd_mode;
    bool ok = true;
    for (int t = 0; t < T && ok; ++t) {
      const int sl = t & 1, slot = S0 + t * kTile + tok;
      const bool in = slot < B;
      const bool live = in && (mode != 0 || __ldg(a.fixed + ur.off + min(slot, B - 1)) == 0);
      ok = mbar_wait_warp(&bars->d_full[sl], (t >> 1) & 1, abort_flag);
      if (ok && mode != 2) ok = mbar_wait_warp(&bars->v_full[sl], (t >> 1) & 1, abort_flag);
      if (ok && mode == 2 && t >= 2)
        ok = mbar_wait_warp(&bars->v_empty[sl], ((t >> 1) - 1) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      uint8_t* vt = sm + kOffVU + sl * kTileBytes;
      const uint32_t dcol = lane_addr + kColD + sl * kD;
      float* vp = mode != 0 ? a.vpart + (ur.off + min(slot, B - 1)) * kD : nullptr;
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        float dv[32];
        tmem_ld32f(dcol + c * 32, dv);
        tmem_wait32(dv);
        if (c == 3) {
          tc_fence_before();
          mbar_arrive(&bars->d_empty[sl]);
        }
        if (live) {
          // columns 32c .. 32c+31: half c/2, 16-byte chunks (c%2)*4 .. +3
          uint8_t* row = vt + (c >> 1) * (kTileBytes / 2);
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            uint4* p = (uint4*)(row + sw128_offset(tok, (c & 1) * 4 + h));
            float x[8];
            if (mode == 2) {
              const float4 p0 = *(const float4*)(vp + 32 * c + 8 * h);
              const float4 p1 = *(const float4*)(vp + 32 * c + 8 * h + 4);
              x[0] = p0.x; x[1] = p0.y; x[2] = p0.z; x[3] = p0.w;
              x[4] = p1.x; x[5] = p1.y; x[6] = p1.z; x[7] = p1.w;
            } else {
              const uint4 v0 = *p;
              const uint32_t w[4] = {v0.x, v0.y, v0.z, v0.w};
#pragma unroll
              for (int z = 0; z < 4; ++z) {
                x[2 * z] = lo_half(w[z]);
                x[2 * z + 1] = hi_half(w[z]);
              }
            }
#pragma unroll
            for (int z = 0; z < 8; ++z) x[z] += dv[8 * h + z];
            if (mode == 1) {
              *(float4*)(vp + 32 * c + 8 * h) = make_float4(x[0], x[1], x[2], x[3]);
              *(float4*)(vp + 32 * c + 8 * h + 4) = make_float4(x[4], x[5], x[6], x[7]);
            } else {
              *p = make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]),
                              pack_bf16(x[6], x[7]));
            }
          }
        }
      }
      fence_proxy_async_smem();
      mbar_arrive(&bars->vo_full[sl]);
    }
    if (!ok && tok == 0) set_status(a.status, GRKV_ERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

}  // namespace

bool merge_tc_supported(const Shape& s) {
  return s.dtype == GRKV_BF16 && s.m <= 2 * kRows && s.B <= kMaxB && s.B >= 1;
}

// Workspace of the tensor-core merge: rz [U][ldr][128], gram [U][ldr][ldr],
// lam [U][ldr] (fp32), src [U][B], ng [U], fail [U] (int32), fixed [U][B]
// (bytes), and for two row blocks vpart [U][B][128] (fp32).
struct MergeWs {
  int ldr, nrb;
  size_t rz, gram, lam, src, ng, fail, fixed, vpart, total;
};
MergeWs merge_ws(const Shape& s) {
  MergeWs w;
  const size_t U = (size_t)s.U, B = (size_t)s.B;
  w.nrb = s.m > kRows ? 2 : 1;
  w.ldr = w.nrb * kRows;
  const size_t ldr = (size_t)w.ldr;
  w.rz = 0;
  w.gram = w.rz + U * ldr * kD * 4;
  w.lam = w.gram + U * ldr * ldr * 4;
  w.src = w.lam + U * ldr * 4;
  w.ng = w.src + U * B * 4;
  w.fail = w.ng + U * 4;
  w.fixed = w.fail + U * 4;
  w.vpart = (w.fixed + U * B + 15) & ~(size_t)15;
  w.total = w.vpart + (w.nrb > 1 ? U * B * kD * 4 : 0);
  return w;
}

// As many ranks as leave every cluster room on the SMs at once: 8 units of B = 512
// take 15 us with four ranks, one tile each.  With budgets per unit B is the largest; the
// kernel leaves ranks of units with fewer tiles idle.
cudaError_t launch_gram(const CUtensorMap& mq, MArgs a, cudaStream_t st) {
  const int tiles = (a.B + kTile - 1) / kTile, blocks = a.U * a.nrb;
  a.ranks = 1;
  while (a.ranks < 8 && 2 * a.ranks <= tiles && blocks * 2 * a.ranks <= kClusterSms) a.ranks *= 2;
  while (a.ranks > 1 && !cluster_fits(a.ranks, k_merge_gram, kThreadsG, kSmemBytes)) a.ranks /= 2;
  return launch_kernel(true, a.ranks, k_merge_gram, dim3(blocks * a.ranks), kThreadsG, kSmemBytes, st,
                       mq, a);
}

size_t merge_tc_ws_bytes(const Shape& s) { return merge_ws(s).total; }

const uint8_t* merge_tc_fixed(const Shape& s, const char* ws, const WsLayout& L) {
  return (const uint8_t*)(ws + L.merge_tc + merge_ws(s).fixed);
}

cudaError_t launch_merge_tc(const Shape& s, const void* q, const void* k, const void* v,
                            const float* scores, const float* y, const float* row_stats,
                            const int32_t* idx, void* k_out, void* v_out, char* ws,
                            const WsLayout& L, cudaStream_t st) {
  CUtensorMap mq, mk, mko, mvo;
  if (!encode_bf16_3d(&mq, q, kD, s.m, s.U, 64, kRows) ||
      !encode_bf16_2d_rows(&mk, k, kD, (uint64_t)s.U * s.n) ||
      !encode_bf16_3d(&mko, k_out, kD, s.units ? s.rows : s.B, s.units ? 1 : s.U, 64, kTile) ||
      !encode_bf16_3d(&mvo, v_out, kD, s.units ? s.rows : s.B, s.units ? 1 : s.U, 64, kTile))
    return cudaErrorInvalidValue;
  MArgs a{};
  a.U = s.U;
  a.n = s.n;
  a.w = s.w;
  a.m = s.m;
  a.P = s.P;
  a.B = s.B;
  a.causal = s.causal;
  a.n_sink = s.n_sink;
  a.n_fix = s.n_fix;
  a.sl2 = (float)((double)s.scale * 1.4426950408889634);
  a.idx = idx;
  a.scores = scores;
  a.y = y;
  a.k = (const __nv_bfloat16*)k;
  a.v = (const __nv_bfloat16*)v;
  a.k_out = (__nv_bfloat16*)k_out;
  a.v_out = (__nv_bfloat16*)v_out;
  a.rstats = row_stats;
  const MergeWs W = merge_ws(s);
  char* mw = ws + L.merge_tc;
  a.rz = (float*)(mw + W.rz);
  a.gram = (float*)(mw + W.gram);
  a.lam = (float*)(mw + W.lam);
  a.src = (int32_t*)(mw + W.src);
  a.ng = (int32_t*)(mw + W.ng);
  int32_t* fail = (int32_t*)(mw + W.fail);
  a.fixed = (uint8_t*)(mw + W.fixed);
  a.vpart = W.nrb > 1 ? (float*)(mw + W.vpart) : nullptr;
  a.ldr = W.ldr;
  a.nrb = W.nrb;
  a.status = (int*)(ws + L.status);
  a.units = s.units;
  // a unit's update tiles are independent: few units spread over the SMs
  a.split = std::max(1, std::min(kSms / std::max(s.U, 1), (s.B + kTile - 1) / kTile));
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_merge_gram, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kSmemBytes)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_merge_update, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kSmemBytesU)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_merge_fixed, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                s.B * 4)) != cudaSuccess)
    return e;
  if (W.nrb > 1 && (e = cudaFuncSetAttribute(k_merge_cross, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kSmemBytesC)) != cudaSuccess)
    return e;
  if ((e = launch_kernel(s.chained, 1, k_merge_fixed, dim3(s.U), 256, s.B * 4, st, a)) != cudaSuccess)
    return e;
  // the retained statistics, R and the diagonal Gram block of every row block
  if ((e = launch_gram(mq, a, st)) != cudaSuccess) return e;
  int launches = 2;
  if (W.nrb > 1) {
    if ((e = launch_kernel(true, 1, k_merge_cross, dim3(s.U), kThreads, kSmemBytesC, st, mq, mk, a)) !=
        cudaSuccess)
      return e;
    launches += 1;
  }
  count_launches(launches);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // with two row blocks the solve keeps its first factor where the transpose of
  // the cross block would be
  if ((e = launch_solve(s.U, s.m, W.ldr, 1, s.lambda, s.lambda_inf, a.gram, a.rz,
                        a.gram + (size_t)kRows * W.ldr, (size_t)W.ldr * W.ldr, W.ldr, fail,
                        a.status, st)) != cudaSuccess)
    return e;
  if (W.nrb == 1) {
    a.row0 = 0;
    a.upd_mode = 0;
    if ((e = launch_kernel(true, 1, k_merge_update, dim3(s.U * a.split), kThreadsU, kSmemBytesU, st, mq,
                           mk, mko, mvo, a)) != cudaSuccess)
      return e;
    launches = 1;
  } else {
    // the value update of each row block (the first leaves V0 + dV_0 in vpart)
    launches = 0;
    for (int rb = 0; rb < 2; ++rb) {
      a.row0 = rb * kRows;
      a.upd_mode = rb == 0 ? 1 : 2;
      if ((e = launch_kernel(true, 1, k_merge_update, dim3(s.U * a.split), kThreadsU, kSmemBytesU, st, mq,
                           mk, mko, mvo, a)) != cudaSuccess)
      return e;
      launches += 1;
    }
  }
  count_launches(launches);
  return cudaGetLastError();
}

}  // namespace grkv
