// Window scoring on the 5th-generation tensor cores in two launches (bf16,
// d = 128, m <= 256 as one or two blocks of 128 window rows), the default
// scoring path.  The one-read path of GRKV_ONE_READ_SCORE is in
// grkv_score_pipe.cu.
//
// For every unit the path needs, over all n keys, the row statistics of the
// window logits (pass A: M_r, L_r) and then, with those, the probabilities,
// the per-key prefix scores c_j = sum_r P_rj and the target Y = P V (pass B);
// Eq. 4 and Algorithm 1 of the paper.  The row normaliser depends on every
// key, so this path reads the keys twice: pass A and pass B are two persistent
// launches over all units (one CTA per SM), each CTA on a contiguous range of
// the units' tiles.  A tile of 128 tokens is one job per row block: both row
// blocks of m > 128 use the K and V tile that one load brought, so the caches
// are read 2x / 1x whatever m is (a pair of launches per row block read them
// 4x / 2x).
//
// Roles.  Warp 0 issues TMA loads (the unit's Q, then K and V tiles through the
// ring); warp 1 issues tcgen05 MMAs (S = Q K^T into TMEM; Y += P V with P read
// from TMEM); warps 4-19 are four compute groups of 128 threads that share
// every job, 32 tokens each.  A compute thread owns one window row (one TMEM
// lane) and one 32-logit chunk of a job, which it copies to registers at once, so
// that the next S MMA runs under this job's exponentials.  Pass A keeps the row's
// running max / sum in registers; pass B writes exp2(l - Lambda_r) as bf16 over the
// S columns it came from (the A operand of the Y MMA) and sums probabilities
// over rows with a warp transpose-reduction.
//   pass A: warp 2 merges the groups' statistics of each segment (the CTA's
//           tiles of one unit) into the segment's global slot; warp 3 zeroes Y.
//   pass B: warp 2 adds the row quarters' sums of every tile and writes the
//           scores.  One row block: warps 20-23 combine a unit's slots into log2
//           normalisers one segment ahead and add each segment's Y partial to the
//           unit's Y.  Two: the compute threads do both at a segment's ends, and
//           keep the first block's probabilities in registers until the second's
//           are there, so that one transpose-reduction serves both.
//
// Sixteen compute warps of 32 logits, rather than eight of 64: with two warps per
// scheduler the chain max -> exponential -> sum was exposed.  Logits are scaled
// and summed in pairs (fma / add.f32x2), half the issue slots of those steps.
//
// The MMA warp walks its jobs as a whole and an elected lane issues: with one lane
// alone, its address arithmetic (it shares a scheduler with four busy warps) took
// 2.7 K cycles a job and bound both passes of m > 128.
//
// Measured, 256 units (eight compute warps and a pair of launches per row block before).
// m = 128, n = 32768: pass A 0.30 ms, pass B 0.61 ms, at 7.1 TB/s of HBM traffic, their
// bound (1.116 ms together before).  m = 256, n = 131072: pass A 1.72 ms (4.9 TB/s), pass B
// 3.17 ms (5.4 TB/s), bound by the latency chains of the compute groups (exponential unit
// 49% and 27% busy, issue slots 57% and 51%; 8.6 ms together before).
#include <algorithm>
#include <cmath>

#include "grkv_internal.cuh"
#include "sm100.cuh"
#include "tmap.cuh"

namespace grkv {
namespace {

using namespace sm100;

constexpr int kTile = 128;            // tokens per tile
constexpr int kRows = 128;            // window rows per block
constexpr int kGroups = 4;            // compute groups, kTile / kGroups = 32 tokens each
constexpr int kCompWarps = 4 * kGroups;
constexpr uint32_t kTileBytes = kTile * kD * 2;   // 32 KB
constexpr long long kWaitBudget = 1ll << 32;      // cycles (~2 s) before a wait gives up
constexpr long long kTestWaitBudget = 1ll << 22;  // ~2 ms: the budget of GRKV_TEST_TIMEOUT

// Pass B over two row blocks: the compute threads, which then have registers for both
// blocks' probabilities, fetch their own normalisers and add their own Y.
constexpr int score_threads(int pass, int rb) { return pass == 0 || rb == 2 ? 640 : 768; }
// K / V tiles in flight.  More is not better: with five, pass B over 256 units n = 32768
// takes 0.62-0.64 ms instead of 0.61 (HBM serves 152 streams that run further ahead less
// well); three cost 1%.
constexpr int kRingSlots = 4;

// Shared-memory layout (offsets from a 1024-byte aligned base): Q, the K / V
// ring, then one region for pass A's statistics or pass B's sums and normalisers.
template <int RB>
struct Layout {
  static constexpr int kRing = kRingSlots;
  static constexpr uint32_t kOffQ = 0;                                // RB x 32 KB
  static constexpr uint32_t kOffRing = kOffQ + RB * kTileBytes;       // kRing x 32 KB
  static constexpr uint32_t kOffAux = kOffRing + kRing * kTileBytes;
  // pass A: [2 buf][kGroups][RB][128] float2
  static constexpr uint32_t kAstatBytes = 2 * kGroups * RB * kRows * 8;
  // pass B: [2 buf][4 row quarters][128] float, then the normalisers, [2 buf][128]
  // float (RB = 1), or the groups' shares of the statistics, [kGroups][256] float2
  static constexpr uint32_t kRedBytes = 2 * 4 * kTile * 4;
  static constexpr uint32_t kLamBytes = RB == 1 ? 2 * kRows * 4 : kGroups * RB * kRows * 8;
  static constexpr uint32_t kAuxBytes =
      kAstatBytes > kRedBytes + kLamBytes ? kAstatBytes : kRedBytes + kLamBytes;
  static constexpr uint32_t kOffBar = kOffAux + kAuxBytes;
  static constexpr uint32_t kSmemBytes = kOffBar + 512 + 1024;        // + alignment slack
};
static_assert(Layout<1>::kSmemBytes <= 227 * 1024 && Layout<2>::kSmemBytes <= 227 * 1024, "smem");

// TMEM columns.  Pass A: four S buffers.  Pass B: two S buffers and two Y
// accumulators (alternate segments of one row block, or the two row blocks); a
// compute thread writes its 32 probabilities as bf16 pairs over the first 16 of the 32
// S columns that it has copied to registers.
constexpr uint32_t kColY = 256;
constexpr int s_bufs(int pass) { return pass == 0 ? 4 : 2; }

struct Args {
  int U, n, w, m, P, causal;
  int tpu;        // tiles per unit
  int maxc;       // statistics slots per unit
  int keep_keys;  // pass A leaves its keys in L2 for pass B's reverse sweep
  float sl2;      // scale * log2(e)
  float* scores;   // [U][P]
  float* y;        // [U][m][128], zeroed by pass A
  float* row_stats;  // [U][m][2]
  float2* pstats;    // [U][maxc][RB * 128]  (max in log2 units, sum)
  int* status;
  float* ypart;      // [U][maxc][m][128] segment Y partials (deterministic mode) or null
  long long wait_budget;   // cycles before a bounded wait gives up
  int test_withhold;       // GRKV_TEST_TIMEOUT: CTA 0 withholds one arrive
};

// The partition of the U tpu tiles over the CTAs.
struct Sched {
  int U, tpu, G;
  __device__ long long tiles() const { return (long long)U * tpu; }
  __device__ long long start(int c) const { return tiles() * c / G; }
  // CTA whose range holds tile t.
  __device__ int owner(long long t) const {
    return (int)(((t + 1) * G + tiles() - 1) / tiles()) - 1;
  }
  __device__ int first_cta(int u) const { return owner((long long)u * tpu); }
  __device__ int nslots(int u) const {
    return owner((long long)u * tpu + tpu - 1) - first_cta(u) + 1;
  }
  // True if CTA c holds no tile (only when there are fewer tiles than CTAs).
  __device__ bool empty(int c) const { return tiles() < G && start(c) == start(c + 1); }
};

// A CTA's tiles in order, backwards in pass B (kRev; what pass A read last is read
// first).  A segment is the CTA's run of tiles of one unit.
template <bool kRev>
struct TileIter {
  int tpu, u, ti, left;
  bool begin;
  __device__ TileIter(const Sched& sc, int c) {
    const long long t0 = sc.start(c), t1 = sc.start(c + 1), t = kRev ? t1 - 1 : t0;
    tpu = sc.tpu;
    left = (int)(t1 - t0);
    u = (int)(t / tpu);
    ti = (int)(t - (long long)u * tpu);
    begin = true;
  }
  __device__ bool more() const { return left > 0; }
  __device__ bool seg_first() const { return begin || ti == (kRev ? tpu - 1 : 0); }
  __device__ bool seg_last() const { return left == 1 || ti == (kRev ? 0 : tpu - 1); }
  __device__ int j0() const { return ti * kTile; }
  __device__ void advance() {
    begin = false;
    --left;
    if (kRev) {
      if (--ti < 0) {
        ti = tpu - 1;
        --u;
      }
    } else if (++ti == tpu) {
      ti = 0;
      ++u;
    }
  }
};

// Position in a ring: slot and the parity of its current use.
struct RingPos {
  uint32_t slot, phase;
  __device__ void add(uint32_t k, uint32_t ring) {
    slot += k;
    if (slot >= ring) {
      slot -= ring;
      phase ^= 1;
    }
  }
};

// Three-operand maximum (one instruction on sm_100 and later).
__device__ __forceinline__ float fmax3f(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float max32(const float* v) {
  float m[11];
#pragma unroll
  for (int e = 0; e < 10; ++e) m[e] = fmax3f(v[3 * e], v[3 * e + 1], v[3 * e + 2]);
  m[10] = fmaxf(v[30], v[31]);
  const float x0 = fmax3f(m[0], m[1], m[2]), x1 = fmax3f(m[3], m[4], m[5]),
              x2 = fmax3f(m[6], m[7], m[8]), x3 = fmaxf(m[9], m[10]);
  return fmaxf(fmax3f(x0, x1, x2), x3);
}

// Pass A on 32 logits: online row max / sum of exp2 in log2 units.
__device__ __forceinline__ void stats_chunk(float* v, bool full, int j0, int lim, int n, float sl2,
                                            float& M, float& L) {
  if (!full) {
#pragma unroll
    for (int e = 0; e < 32; ++e)
      if (j0 + e > lim || j0 + e >= n) v[e] = -INFINITY;
  }
  // no branch on the maximum: a row that has seen nothing visible yet keeps
  // M = -inf, L = 0 against the reference 0
  const float top = fmaxf(M, max32(v) * sl2);
  const float ref = top == -INFINITY ? 0.f : top;
  L *= fast_exp2(M - ref);
  M = top;
  const uint64_t s2 = pack2(sl2, sl2), m2 = pack2(-ref, -ref);
  uint64_t acc[2] = {0, 0};   // two pairs of zeros
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    float a, b;
    unpack2(fma2(pack2(v[2 * e], v[2 * e + 1]), s2, m2), a, b);
    acc[e & 1] = add2(acc[e & 1], pack2(fast_exp2(a), fast_exp2(b)));
  }
  float a, b;
  unpack2(add2(acc[0], acc[1]), a, b);
  L += a + b;
}

// mbar_wait for all lanes of a warp with one answer, so that warp-collective
// instructions after a wait are reached by all lanes or by none.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort,
                                               long long budget) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort, budget));
}
// One arrive for the whole warp, after all its lanes' reads and writes.
__device__ __forceinline__ void mbar_arrive_warp(uint64_t* bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

template <int kRing>
struct Bars {
  uint64_t ring_full[kRing], ring_empty[kRing];
  uint64_t q_full, q_empty;
  uint64_t s_full[4], s_done[4];            // S written / (pass A) copied to registers
  uint64_t p_full[2];                       // pass B: P written
  uint64_t y_full[2], y_empty[2];
  uint64_t astat_full[2], astat_empty[2];   // compute groups -> statistics publisher
  uint64_t red_full[2], red_empty[2];       // compute groups -> score writer
  uint64_t lam_full[2], lam_empty[2];       // statistics fetcher -> compute groups
  uint64_t drain;
  uint32_t tmem;
  int abort;
};
static_assert(sizeof(Bars<kRingSlots>) <= 512, "barrier block");

// Merges two (max, sum) row statistics in log2 units.
__device__ __forceinline__ float2 stat_merge(float2 x, float2 y) {
  if (x.x == -INFINITY) return y;
  if (y.x == -INFINITY) return x;
  const float M = fmaxf(x.x, y.x);
  return make_float2(M, x.y * fast_exp2(x.x - M) + y.y * fast_exp2(y.x - M));
}

// log2 normaliser of a row from its combined statistics (infinite past row m: p = 0).
__device__ __forceinline__ float log2_norm(float2 st, bool row_ok) {
  return row_ok && st.y > 0.f ? st.x + __log2f(st.y) : INFINITY;
}
__device__ __forceinline__ void write_stats(float* out, float2 st) {
  out[0] = st.x * 0.69314718055994531f;
  out[1] = st.y;
}
// Where CTA `cta` adds row r of unit u's Y partial; in deterministic mode the
// partial goes to a slot of its own, summed in slot order later.
__device__ __forceinline__ float* y_row(const Args& a, const Sched& sc, int u, int cta, int r) {
  return a.ypart ? a.ypart + (((size_t)u * a.maxc + (cta - sc.first_cta(u))) * a.m + r) * kD
                 : a.y + ((size_t)u * a.m + r) * kD;
}
// 32 columns of this thread's Y row from TMEM, stored or added (all lanes of the warp).
__device__ __forceinline__ void add_y32(uint32_t taddr, float* dst, bool row_ok, bool store) {
  float v[32];
  tmem_ld32f(taddr, v);
  tmem_wait32(v);
  if (!row_ok) return;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const float4 x = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
    if (store)
      ((float4*)dst)[e] = x;
    else
      atomicAdd((float4*)dst + e, x);
  }
}

// kPass 0: pass A, 1: pass B.  RB: row blocks.
template <int kPass, int RB>
__global__ void __launch_bounds__(score_threads(kPass, RB), 1)
    k_score_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
               const __grid_constant__ CUtensorMap tmV, Args a) {
  using Lay = Layout<RB>;
  constexpr int kRing = Lay::kRing, kS = s_bufs(kPass);
  if (kPass == 1) chain_wait();
  // One row block: each V is loaded one tile after its K, as it stays in the
  // ring through the tile's compute.  Two: its first use is half a tile after its K's.
  constexpr bool kLateV = RB == 1;
  constexpr bool kOwn = kPass == 1 && RB == 2;   // see score_threads
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  Bars<kRing>* bars = (Bars<kRing>*)(sm + Lay::kOffBar);
  float2* astat = (float2*)(sm + Lay::kOffAux);                  // pass A
  float* red = (float*)(sm + Lay::kOffAux);                      // pass B
  float* lam_s = (float*)(sm + Lay::kOffAux + Lay::kRedBytes);   // pass B, RB = 1
  float2* stat_s = (float2*)lam_s;                               // pass B, RB = 2
  const int tid = threadIdx.x, lane = tid & 31, cta = blockIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform for the compiler
  const Sched sc{a.U, a.tpu, (int)gridDim.x};

  if (tid == 0) {
    for (int i = 0; i < kRing; ++i) {
      mbar_init(&bars->ring_full[i], 1);
      mbar_init(&bars->ring_empty[i], 1);
    }
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->q_empty, 1);
    for (int i = 0; i < 4; ++i) {
      mbar_init(&bars->s_full[i], 1);
      mbar_init(&bars->s_done[i], kCompWarps);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->p_full[i], kCompWarps);
      mbar_init(&bars->y_full[i], 1);
      mbar_init(&bars->y_empty[i], kOwn ? kCompWarps : 4);
      mbar_init(&bars->astat_full[i], kCompWarps);
      mbar_init(&bars->astat_empty[i], 1);
      mbar_init(&bars->red_full[i], kCompWarps);
      mbar_init(&bars->red_empty[i], 1);
      mbar_init(&bars->lam_full[i], kOwn ? kCompWarps : 4);
      mbar_init(&bars->lam_empty[i], kCompWarps);
    }
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

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      prefetch_tensormap(&tmQ);
      prefetch_tensormap(&tmK);
      if (kPass == 1) prefetch_tensormap(&tmV);
      const uint64_t keep = l2_evict_last();
      const uint64_t stream = kPass == 0 && a.keep_keys ? l2_evict_normal() : l2_evict_first();
      uint32_t idx = 0;   // loads issued through the ring
      int seg = 0;
      bool ok = true, late = false;
      int v_j0 = 0, v_u = 0;
      auto load = [&](const CUtensorMap* map, int j0, int u) -> bool {
        const uint32_t slot = idx % kRing;
        if (idx >= kRing && !mbar_wait(&bars->ring_empty[slot], (idx / kRing - 1) & 1, abort_flag,
                                       a.wait_budget))
          return false;
        uint8_t* dst = sm + Lay::kOffRing + slot * kTileBytes;
        mbar_expect_tx(&bars->ring_full[slot], kTileBytes);
        tma_load_3d(dst, map, &bars->ring_full[slot], 0, j0, u, stream);
        tma_load_3d(dst + kTileBytes / 2, map, &bars->ring_full[slot], 64, j0, u, stream);
        ++idx;
        return true;
      };
      for (TileIter<kPass == 1> it(sc, cta); ok && it.more(); it.advance()) {
        if (it.seg_first()) {
          if (seg >= 1) ok = mbar_wait(&bars->q_empty, (seg - 1) & 1, abort_flag, a.wait_budget);
          if (!ok) break;
          ++seg;
          mbar_expect_tx(&bars->q_full, RB * kTileBytes);
          for (int rb = 0; rb < RB; ++rb) {
            uint8_t* dq = sm + Lay::kOffQ + rb * kTileBytes;
            tma_load_3d(dq, &tmQ, &bars->q_full, 0, rb * kRows, it.u, keep);
            tma_load_3d(dq + kTileBytes / 2, &tmQ, &bars->q_full, 64, rb * kRows, it.u, keep);
          }
        }
        ok = load(&tmK, it.j0(), it.u);
        if (kPass == 1) {
          if (!kLateV) {
            if (ok) ok = load(&tmV, it.j0(), it.u);
          } else {
            if (ok && late) ok = load(&tmV, v_j0, v_u);
            late = true;
            v_j0 = it.j0();
            v_u = it.u;
          }
        }
      }
      if (kPass == 1 && kLateV && ok && late) load(&tmV, v_j0, v_u);
      // let every issued load land before the CTA can exit (these waits
      // ignore the abort flag, and are bounded)
      volatile int no_abort = 0;
      for (uint32_t i = idx > kRing ? idx - kRing : 0; i < idx; ++i)
        mbar_wait(&bars->ring_full[i % kRing], (i / kRing) & 1, &no_abort, a.wait_budget);
      if (seg > 0) mbar_wait(&bars->q_full, (seg - 1) & 1, &no_abort, a.wait_budget);
    }
  } else if (warp == 1) {
    // ----------------------------------------------------------- MMA issuer
    // The whole warp walks the jobs (uniform control flow and descriptors; one
    // elected lane issues): the issuer shares its scheduler with four compute warps,
    // and one lane's address arithmetic was what bound pass B (2.7 K cycles a job).
    constexpr uint32_t id_s = idesc_bf16(kRows, kTile, 0, 0);   // S = Q K^T, both K-major
    constexpr uint32_t id_y = idesc_bf16(kRows, kD, 0, 1);      // Y += P V, V MN-major
    const uint64_t q_desc = sw128_desc(smem_u32(sm + Lay::kOffQ), 16, 1024);
    const uint64_t k_desc = sw128_desc(smem_u32(sm + Lay::kOffRing), 16, 1024);
    const uint64_t v_desc = sw128_desc(smem_u32(sm + Lay::kOffRing), kTileBytes / 2, 1024);
    constexpr uint32_t kTileDesc = kTileBytes >> 4;   // a tile's bytes in descriptor units
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      return mbar_wait_warp(bar, parity, abort_flag, a.wait_budget);
    };
    TileIter<kPass == 1> it(sc, cta);
    // ring slot and phase of the next K and V: with kLateV the loads are K0, K1, V0,
    // K2, V1, ..., V(last - 1), V(last), else K0, V0, K1, V1, ...
    RingPos kp{0, 0}, vp{0, 0};
    vp.add(kLateV && it.left > 1 ? 2 : 1, kRing);
    uint32_t i = 0, t = 0;
    int seg = 0, y_seg = 0;
    bool ok = true;
    // The Y MMA of the job before: issued after this job's S MMA.
    bool y_first = false, y_last = false;
    int y_left = it.left;   // tiles whose Y MMAs are still to come
    auto issue_y = [&](uint32_t yi, int rb) -> bool {
      const uint32_t pb = yi & 1;
      const uint32_t yb = RB == 1 ? y_seg & 1 : rb, yuse = RB == 1 ? y_seg >> 1 : y_seg;
      if (y_first && yuse >= 1 && !wait(&bars->y_empty[yb], (yuse - 1) & 1)) return false;
      if (!wait(&bars->p_full[pb], (yi >> 1) & 1)) return false;
      if (rb == 0 && !wait(&bars->ring_full[vp.slot], vp.phase)) return false;
      tc_fence_after();
      mma8_ts<id_y, false>(tmem + kColY + yb * kD, tmem + pb * kTile,
                                          v_desc + vp.slot * kTileDesc, !y_first);
      if (rb == RB - 1) {
        mma_commit_elect(&bars->ring_empty[vp.slot]);
        // the last V follows its predecessor directly
        --y_left;
        vp.add(kLateV && y_left == 1 ? 1 : 2, kRing);
      }
      if (y_last) {
        mma_commit_elect(&bars->y_full[yb]);
        if (rb == RB - 1) ++y_seg;
      }
      return true;
    };
    for (; ok && it.more(); it.advance(), ++t) {
      const bool first = it.seg_first(), last = it.seg_last();
      if (first) ok = wait(&bars->q_full, seg & 1);
      if (ok) ok = wait(&bars->ring_full[kp.slot], kp.phase);
#pragma unroll
      for (int rb = 0; rb < RB; ++rb, ++i) {
        // Pass A: the buffer's last logits are in registers.  Pass B: the Y MMA that
        // reads the buffer's last probabilities was issued before this S MMA; a
        // tile's S also says that its score sums (tile t - 2's) have been read.
        const uint32_t sb = i % kS, use = i / kS;
        if (kPass == 0 && ok && use >= 1) ok = wait(&bars->s_done[sb], (use - 1) & 1);
        if (kPass == 1 && rb == 0 && ok && t >= 2)
          ok = wait(&bars->red_empty[t & 1], ((t >> 1) - 1) & 1);
        if (!ok) break;
        tc_fence_after();
        mma8_ss<id_s>(tmem + sb * kTile, q_desc + rb * kTileDesc, k_desc + kp.slot * kTileDesc);
        mma_commit_elect(&bars->s_full[sb]);
        if (rb == RB - 1) {
          mma_commit_elect(&bars->ring_empty[kp.slot]);
          if (last) mma_commit_elect(&bars->q_empty);
        }
        if (kPass == 1) {
          if (i > 0) ok = issue_y(i - 1, RB == 1 ? 0 : 1 - rb);
          if (!ok) break;
          if (rb == 0) {
            y_first = first;
            y_last = last;
          }
        }
      }
      kp.add(kPass == 0 || (kLateV && t == 0) ? 1 : 2, kRing);
      if (last) ++seg;
    }
    if (kPass == 1 && ok && i > 0) issue_y(i - 1, RB - 1);
    // every MMA issued so far completes before TMEM can be released (this
    // wait ignores the abort flag, and is bounded)
    mma_commit_elect(&bars->drain);
    volatile int no_abort = 0;
    mbar_wait(&bars->drain, 0, &no_abort, a.wait_budget);
    __syncwarp();
  } else if (kPass == 0 && warp == 2) {
    // ----------------------------------------------- statistics publisher
    // Merges the compute groups' row statistics of each segment into the
    // segment's global slot.
    int aseg = 0;
    bool ok = true;
    for (TileIter<kPass == 1> it(sc, cta); ok && it.more(); it.advance()) {
      if (!it.seg_last()) continue;
      const int ab = aseg & 1;
      ok = mbar_wait_warp(&bars->astat_full[ab], (aseg >> 1) & 1, abort_flag, a.wait_budget);
      if (!ok) break;
      const int k = cta - sc.first_cta(it.u);
      // k < maxc always holds (the host sizes maxc from the same partition)
      if (k >= 0 && k < a.maxc) {
        float2* slot = a.pstats + ((size_t)it.u * a.maxc + k) * (RB * kRows);
        const float2* as = astat + ab * kGroups * RB * kRows;
#pragma unroll
        for (int t = 0; t < RB * 4; ++t) {
          const int r = t * 32 + lane;
          slot[r] = stat_merge(stat_merge(as[r], as[RB * kRows + r]),
                               stat_merge(as[2 * RB * kRows + r], as[3 * RB * kRows + r]));
        }
      }
      mbar_arrive_warp(&bars->astat_empty[ab], lane);
      ++aseg;
    }
  } else if (kPass == 0 && warp == 3) {
    // Y starts at zero: pass B adds to it.
    if (a.y) {
      const size_t n4 = (size_t)a.U * a.m * kD / 4;
      for (size_t i = (size_t)cta * 32 + lane; i < n4; i += (size_t)gridDim.x * 32)
        ((float4*)a.y)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  } else if (kPass == 1 && warp == 2) {
    // ------------------------------------------------------- score writer
    // Adds the four row quarters' sums of every tile and writes the prefix scores.
    uint32_t t = 0;
    bool ok = true;
    for (TileIter<kPass == 1> it(sc, cta); ok && it.more(); it.advance(), ++t) {
      const uint32_t tb = t & 1;
      ok = mbar_wait_warp(&bars->red_full[tb], (t >> 1) & 1, abort_flag, a.wait_budget);
      if (!ok) break;
      const float* rt = red + tb * 4 * kTile;
      float* out = a.scores + (size_t)it.u * a.P;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j = c * 32 + lane;
        const float cs = ((rt[j] + rt[kTile + j]) + rt[2 * kTile + j]) + rt[3 * kTile + j];
        if (it.j0() + j < a.P) out[it.j0() + j] = cs;
      }
      mbar_arrive_warp(&bars->red_empty[tb], lane);
    }
  } else if (kPass == 1 && RB == 1 && warp >= 4 + kCompWarps) {
    // ------------------------------------- statistics fetcher, Y flusher
    // Segment s + 1's normalisers are combined before segment s's Y partial is
    // added.  One thread owns one row (TMEM lane); the CTA that holds the unit's first
    // tile also writes the unit's row statistics.
    const int q = warp & 3, row = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    const long long t0 = sc.start(cta), t1 = sc.start(cta + 1);
    // segments from the CTA's last unit down, as its tiles
    const int u0 = (int)((t1 - 1) / a.tpu), nseg = t1 > t0 ? u0 - (int)(t0 / a.tpu) + 1 : 0;
    bool ok = true;
    for (int s = 0; ok && s <= nseg && nseg > 0; ++s) {
      if (s < nseg) {
        const int u = u0 - s, lb = s & 1;
        if (s >= 2)
          ok = mbar_wait_warp(&bars->lam_empty[lb], ((s >> 1) - 1) & 1, abort_flag, a.wait_budget);
        if (!ok) break;
        const int ns = sc.nslots(u), c0 = sc.first_cta(u);
        const bool dense = sc.tiles() >= sc.G;   // every CTA holds tiles
        float2 st = make_float2(-INFINITY, 0.f);
        // sixteen slots per round trip
        for (int k0 = 0; k0 < ns; k0 += 16) {
          float2 pr[16];
#pragma unroll
          for (int kk = 0; kk < 16; ++kk) {
            const bool use = k0 + kk < ns && (dense || !sc.empty(c0 + k0 + kk));
            pr[kk] = use ? __ldg(a.pstats + ((size_t)u * a.maxc + k0 + kk) * kRows + row)
                         : make_float2(-INFINITY, 0.f);
          }
#pragma unroll
          for (int kk = 0; kk < 16; ++kk) st = stat_merge(st, pr[kk]);
        }
        lam_s[lb * kRows + row] = log2_norm(st, row < a.m);
        if (cta == c0 && row < a.m) write_stats(a.row_stats + ((size_t)u * a.m + row) * 2, st);
        // GRKV_TEST_TIMEOUT: CTA 0 never announces its first normalisers, so
        // its compute groups' bounded wait expires
        __syncwarp();
        if (lane == 0 && !(a.test_withhold && cta == 0 && s == 0 && q == 0))
          mbar_arrive(&bars->lam_full[lb]);
      }
      if (s == 0) continue;
      const int fs = s - 1, u = u0 - fs, yb = fs & 1;
      ok = mbar_wait_warp(&bars->y_full[yb], (fs >> 1) & 1, abort_flag, a.wait_budget);
      if (!ok) break;
      tc_fence_after();
      float* dst = y_row(a, sc, u, cta, row);
#pragma unroll 1
      for (int c = 0; c < 4; ++c)
        add_y32(lane_addr + kColY + yb * kD + c * 32, dst + c * 32, row < a.m, a.ypart != nullptr);
      tc_fence_before();
      mbar_arrive_warp(&bars->y_empty[yb], lane);
    }
    if (!ok && row == 0) set_status(a.status, GRKV_ERR_TIMEOUT);
  } else if (warp >= 4 && warp < 4 + kCompWarps) {
    // ------------------------------------------------------- compute groups
    const int g = (warp - 4) >> 2, q = warp & 3, row = q * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    // last position each of the thread's rows sees
    int lim[RB];
#pragma unroll
    for (int rb = 0; rb < RB; ++rb)
      lim[rb] = a.causal ? a.n - a.w + (rb * kRows + row) % a.w : a.n - 1;
    float M[RB], L[RB];      // pass A: running stats (log2 units)
    float lam[RB];           // pass B: log2 normalisers (infinite past row m: p = 0)
    uint32_t i = 0, t = 0;
    int seg = 0;
    bool ok = true;
    for (TileIter<kPass == 1> it(sc, cta); ok && it.more(); it.advance(), ++t) {
      const int t0 = it.j0() + 32 * g;   // this group's first token
      const bool in = t0 + 32 <= a.n;
      if (it.seg_first()) {
        if (kPass == 0) {
#pragma unroll
          for (int rb = 0; rb < RB; ++rb) {
            M[rb] = -INFINITY;
            L[rb] = 0.f;
          }
        } else if (!kOwn) {
          const int lb = seg & 1;
          ok = mbar_wait_warp(&bars->lam_full[lb], (seg >> 1) & 1, abort_flag, a.wait_budget);
          if (!ok) break;
          lam[0] = lam_s[lb * kRows + row];
          mbar_arrive_warp(&bars->lam_empty[lb], lane);
        } else {
          // Each group combines a quarter of the unit's slots.  No warp still reads the last
          // segment's shares: this warp has waited for that segment's y_full, which follows Y MMAs
          // that waited for p_full of every warp, and a warp arrives there after it has read them.
          const int ns = sc.nslots(it.u), c0 = sc.first_cta(it.u);
          const bool dense = sc.tiles() >= sc.G;   // every CTA holds tiles
          float2 st[RB];
#pragma unroll
          for (int rb = 0; rb < RB; ++rb) {
            st[rb] = make_float2(-INFINITY, 0.f);
            for (int k0 = g; k0 < ns; k0 += 8 * kGroups) {   // eight slots per round trip
              float2 pr[8];
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) {
                const int k = k0 + kk * kGroups;
                const bool use = k < ns && (dense || !sc.empty(c0 + k));
                pr[kk] = use ? __ldg(a.pstats + ((size_t)it.u * a.maxc + k) * (RB * kRows) +
                                     rb * kRows + row)
                             : make_float2(-INFINITY, 0.f);
              }
#pragma unroll
              for (int kk = 0; kk < 8; ++kk) st[rb] = stat_merge(st[rb], pr[kk]);
            }
            stat_s[(g * RB + rb) * kRows + row] = st[rb];
          }
          __syncwarp();
          // GRKV_TEST_TIMEOUT: CTA 0 never completes its first normalisers
          if (lane == 0 && !(a.test_withhold && cta == 0 && seg == 0 && warp == 4))
            mbar_arrive(&bars->lam_full[0]);
          ok = mbar_wait_warp(&bars->lam_full[0], seg & 1, abort_flag, a.wait_budget);
          if (!ok) break;
#pragma unroll
          for (int rb = 0; rb < RB; ++rb) {
            const int r = rb * kRows + row;
            float2 x = stat_s[r];
#pragma unroll
            for (int h = 1; h < kGroups; ++h) x = stat_merge(x, stat_s[h * RB * kRows + r]);
            lam[rb] = log2_norm(x, r < a.m);
            if (g == 0 && cta == c0 && r < a.m)
              write_stats(a.row_stats + ((size_t)it.u * a.m + r) * 2, x);
          }
        }
      }
      float both[RB == 2 ? 32 : 1];   // pass B: the first row block's probabilities
#pragma unroll
      for (int rb = 0; rb < RB; ++rb, ++i) {
        const uint32_t sb = i % kS;
        // one answer per warp; rows past the abort are left unprocessed
        if (ok) ok = mbar_wait_warp(&bars->s_full[sb], (i / kS) & 1, abort_flag, a.wait_budget);
        if (!ok) break;
        tc_fence_after();
        float v[32];
        tmem_ld32f(lane_addr + sb * kTile + 32 * g, v);
        tmem_wait32(v);
        if (kPass == 0) {
          tc_fence_before();
          mbar_arrive_warp(&bars->s_done[sb], lane);
        }
        // chunks away from the window and the end of the unit need no mask
        const bool full = in && t0 + 31 <= lim[rb];
        if (kPass == 0) {
          stats_chunk(v, full, t0, lim[rb], a.n, a.sl2, M[rb], L[rb]);
          continue;
        }
        const uint64_t s2 = pack2(a.sl2, a.sl2), m2 = pack2(-lam[rb], -lam[rb]);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          float x, y;
          unpack2(fma2(pack2(v[2 * e], v[2 * e + 1]), s2, m2), x, y);
          v[2 * e] = fast_exp2(x);
          v[2 * e + 1] = fast_exp2(y);
        }
        if (!full) {
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (t0 + e > lim[rb] || t0 + e >= a.n) v[e] = 0.f;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t pk[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) pk[e] = pack_bf16(v[16 * h + 2 * e], v[16 * h + 2 * e + 1]);
          tmem_st8(lane_addr + sb * kTile + 32 * g + 8 * h, pk);
        }
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive_warp(&bars->p_full[sb], lane);
        if (RB == 2 && rb == 0) {
#pragma unroll
          for (int e = 0; e < 32; ++e) both[e % (RB == 2 ? 32 : 1)] = v[e];
          continue;
        }
        if (RB == 2) {
          // one reduction for both row blocks
#pragma unroll
          for (int e = 0; e < 16; ++e)
            unpack2(add2(pack2(both[(2 * e) % (RB == 2 ? 32 : 1)], both[(2 * e + 1) % (RB == 2 ? 32 : 1)]),
                         pack2(v[2 * e], v[2 * e + 1])),
                    v[2 * e], v[2 * e + 1]);
        }
        // transpose-reduce: lane t ends with the warp's sum for token t
#pragma unroll
        for (int hh = 16; hh >= 1; hh >>= 1) {
          const bool up = (lane & hh) != 0;
#pragma unroll
          for (int e = 0; e < hh; ++e) {
            const float send = up ? v[e] : v[e + hh];
            const float keep = up ? v[e + hh] : v[e];
            v[e] = keep + __shfl_xor_sync(0xffffffffu, send, hh);
          }
        }
        const uint32_t tb = t & 1;
        red[(tb * 4 + q) * kTile + 32 * g + lane] = v[0];
        mbar_arrive_warp(&bars->red_full[tb], lane);
      }
      if (!ok) break;
      if (it.seg_last()) {
        if (kPass == 0) {
          const int ab = seg & 1;
          if (seg >= 2)
            ok = mbar_wait_warp(&bars->astat_empty[ab], ((seg >> 1) - 1) & 1, abort_flag,
                                a.wait_budget);
          if (!ok) break;
#pragma unroll
          for (int rb = 0; rb < RB; ++rb)
            astat[((ab * kGroups + g) * RB + rb) * kRows + row] = make_float2(M[rb], L[rb]);
          mbar_arrive_warp(&bars->astat_full[ab], lane);
        } else if (kOwn) {
#pragma unroll
          for (int rb = 0; rb < RB; ++rb) {
            const int r = rb * kRows + row;
            ok = ok && mbar_wait_warp(&bars->y_full[rb], seg & 1, abort_flag, a.wait_budget);
            if (!ok) break;
            tc_fence_after();
            add_y32(lane_addr + kColY + rb * kD + 32 * g, y_row(a, sc, it.u, cta, r) + 32 * g,
                    r < a.m, a.ypart != nullptr);
            tc_fence_before();
            mbar_arrive_warp(&bars->y_empty[rb], lane);
          }
          if (!ok) break;
        }
        ++seg;
      }
    }
    if (!ok && row == 0) set_status(a.status, GRKV_ERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// Deterministic mode: Y[u] = the unit's segment partials added in slot order.
__global__ void k_y_sum_slots(const float4* __restrict__ part, float4* __restrict__ y, Sched sc,
                              int m, int maxc) {
  chain_wait();
  const size_t per_unit = (size_t)m * kD / 4;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < (size_t)sc.U * per_unit;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t u = i / per_unit, r = i - u * per_unit;
    const int ns = sc.nslots((int)u), c0 = sc.first_cta((int)u);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < ns; ++k) {
      if (sc.empty(c0 + k)) continue;
      const float4 x = __ldg(part + (u * maxc + k) * per_unit + r);
      acc.x += x.x;
      acc.y += x.y;
      acc.z += x.z;
      acc.w += x.w;
    }
    y[i] = acc;
  }
}

int g_num_sms[64] = {};

template <int kPass, int RB>
cudaError_t launch_pass(int G, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                        const Args& a, cudaStream_t st) {
  auto kern = k_score_tc<kPass, RB>;
  const uint32_t smem = Layout<RB>::kSmemBytes;
  const cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  count_launches(1);
  return launch_kernel(kPass == 1, 1, kern, dim3(G), score_threads(kPass, RB), smem, st, mq, mk, mv, a);
}

// CTAs that can share one unit's tiles when U units are split evenly over
// `sms` CTAs: the unit's share, and a partial one at each end.
int score_tc_slots(int U, int sms) { return std::min(sms, (sms + U - 1) / std::max(U, 1) + 2); }

}  // namespace

bool score_tc_supported(const Shape& s) { return s.dtype == GRKV_BF16 && s.m <= 2 * kRows; }

size_t score_tc_pstats_bytes(const Shape& s, int* maxc) {
  *maxc = score_tc_slots(s.U, kMaxScoreCtas);
  const size_t rows = (size_t)(s.m > kRows ? 2 : 1) * kRows;
  return (size_t)s.U * *maxc * rows * sizeof(float2);
}

int sm_count() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!g_num_sms[dev] &&
      cudaDeviceGetAttribute(&g_num_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    g_num_sms[dev] = 0;
  return g_num_sms[dev];
}

cudaError_t launch_score_tc(const Shape& s, const void* q, const void* k, const void* v,
                            float* scores, float* y, float* row_stats, char* ws,
                            const WsLayout& L, cudaStream_t st) {
  CUtensorMap mq, mk, mv;
  if (!encode_bf16_3d(&mq, q, kD, s.m, s.U, 64, kRows) ||
      !encode_bf16_3d(&mk, k, kD, s.n, s.U, 64, kTile) ||
      !encode_bf16_3d(&mv, v, kD, s.n, s.U, 64, kTile))
    return cudaErrorInvalidValue;
  const int G = sm_count();
  if (G <= 0 || G > kMaxScoreCtas) return cudaErrorInvalidDevice;
  Args a{};
  a.U = s.U;
  a.n = s.n;
  a.w = s.w;
  a.m = s.m;
  a.P = s.P;
  a.causal = s.causal;
  a.tpu = (s.n + kTile - 1) / kTile;
  a.maxc = score_tc_slots(s.U, G);
  // Pass B walks each CTA's tiles backwards, so the keys that pass A read last may
  // still be in L2.  They are kept there (evict-normal loads) when the cache is many
  // times L2: 2.1 GB of keys, 256 units n = 32768, 1325 -> 1298 us a compress call.  With
  // 134 MB of keys (32 units n = 16384) that costs 184 -> 193 us, as the merge then finds
  // fewer of its rows in L2; 268 MB of keys lose 1%.
  a.keep_keys = (size_t)s.U * s.n * kD * 2 > ((size_t)512 << 20);
  a.sl2 = (float)((double)s.scale * 1.4426950408889634);
  a.scores = scores;
  a.y = s.deterministic ? nullptr : y;
  a.row_stats = row_stats;
  a.pstats = (float2*)(ws + L.pstats_tc);
  a.status = (int*)(ws + L.status);
  a.ypart = s.deterministic ? (float*)(ws + L.ypart_tc) : nullptr;
  a.test_withhold = s.test_timeout;
  a.wait_budget = s.test_timeout ? kTestWaitBudget : kWaitBudget;
  cudaError_t e;
  if (s.m <= kRows) {
    e = launch_pass<0, 1>(G, mq, mk, mv, a, st);
    if (e == cudaSuccess) e = launch_pass<1, 1>(G, mq, mk, mv, a, st);
  } else {
    e = launch_pass<0, 2>(G, mq, mk, mv, a, st);
    if (e == cudaSuccess) e = launch_pass<1, 2>(G, mq, mk, mv, a, st);
  }
  if (e == cudaSuccess && a.ypart) {
    const size_t n4 = (size_t)s.U * s.m * kD / 4;
    const int blocks = (int)std::min<size_t>((n4 + 255) / 256, (size_t)G * 8);
    e = launch_kernel(true, 1, k_y_sum_slots, dim3(blocks), 256, 0, st, (const float4*)a.ypart,
                      (float4*)y, Sched{s.U, a.tpu, G}, s.m, a.maxc);
    count_launches(1);
  }
  return e;
}

}  // namespace grkv
