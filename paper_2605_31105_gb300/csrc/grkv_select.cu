// Selection (every path): pooled prefix scores, the B - w best positions
// (ties to the smaller one) in ascending order, then the window.
//
// k_select_reg holds a unit's pooled scores as order-preserving keys in
// registers, kPer consecutive positions per thread, over one CTA of 1024 threads
// (n - w <= 32768) or a cluster of 8 (up to 262144).  The cut is the kk-th
// largest key, found among the few keys above a sampled bound where that pays, else
// over all keys: its sign and exponent by nine counting steps (a ballot of the
// whole block each, no histogram: almost every key shares a few exponents,
// which serialises shared atomics), its mantissa by three histogram passes
// over the keys that share them; one scan of (above, equal) counts places the
// positions.  Bound by the latency of its ~20 block-wide steps; with a fixed 32
// positions per thread, four full histogram passes and two scans it took 33 us
// for n - w = 8160 (255 threads at work) and 317 us for 131,008 (one CTA
// re-reading a pooled copy from global memory).
// Longer prefixes, pooling wider than 129, and devices that hold no cluster of 8 take
// k_select (a pooled copy in the workspace).
#include <algorithm>
#include <cmath>

#include "block_select.cuh"
#include "grkv_internal.cuh"

namespace grkv {
namespace {

// One CTA per unit over the pooled copy [U][n-w].
__global__ void __launch_bounds__(1024) k_select(const float* __restrict__ scores, Shape s,
                                                 float* __restrict__ pooled,
                                                 int32_t* __restrict__ idx) {
  chain_wait();
  __shared__ int hist[256];
  __shared__ int sh[48];
  const int u = blockIdx.x, tid = threadIdx.x, P = s.P, h = s.pool_k / 2;
  const float* c = scores + (size_t)u * P;
  float* pl = pooled + (size_t)u * P;
  const UnitRow ur = unit_row(s.units, u, s.B, s.n_fix);
  const int kk_u = ur.B - s.w;
  int32_t* out = idx + ur.off;
  // four positions per step, the neighbour offset outermost, so that each
  // step's loads are independent of one another
  for (int j0 = tid; j0 < P; j0 += 4 * blockDim.x) {
    int j[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) j[q] = j0 + q * blockDim.x;
    if (s.pool_type == GRKV_POOL_MAX) {
      float mx[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) mx[q] = j[q] < P ? c[j[q]] : 0.f;
      for (int t = 1; t <= h; ++t) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (j[q] >= P) continue;
          if (j[q] - t >= 0) mx[q] = fmaxf(mx[q], c[j[q] - t]);
          if (j[q] + t < P) mx[q] = fmaxf(mx[q], c[j[q] + t]);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (j[q] < P) pl[j[q]] = mx[q];
    } else {
      double a[4] = {0.0, 0.0, 0.0, 0.0};   // left to right, zero padding, divisor k
      for (int t = -h; t <= h; ++t) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (j[q] < P && j[q] + t >= 0 && j[q] + t < P) a[q] += (double)c[j[q] + t];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (j[q] < P) pl[j[q]] = (float)(a[q] / (double)s.pool_k);
    }
  }
  __syncthreads();
  if (kk_u >= P) {
    for (int j = tid; j < P; j += blockDim.x) out[j] = j;
  } else if (kk_u > 0) {
    auto get = [&](int i, uint32_t* key) {
      *key = order_key(pl[i]);
      return true;
    };
    // positions: count the marks of earlier segments first
    const int seg = (P + blockDim.x - 1) / blockDim.x;
    const int lo = min(P, tid * seg), hi = min(P, lo + seg);
    uint32_t tau;
    int need_eq;
    block_kth_largest(get, P, kk_u, hist, sh, &tau, &need_eq);
    // the segment's keys in chunks of eight loaded together
    auto seg_keys = [&](int i0, uint32_t* kk) {
#pragma unroll
      for (int q = 0; q < 8; ++q) kk[q] = i0 + q < hi ? order_key(pl[i0 + q]) : 0u;
    };
    int eq = 0;
    for (int i0 = lo; i0 < hi; i0 += 8) {
      uint32_t kk[8];
      seg_keys(i0, kk);
#pragma unroll
      for (int q = 0; q < 8; ++q) eq += (i0 + q < hi && kk[q] == tau);
    }
    int tot;
    const int er0 = block_exclusive_scan(eq, sh + 8, &tot);
    int sel = 0, er = er0;
    for (int i0 = lo; i0 < hi; i0 += 8) {
      uint32_t kk[8];
      seg_keys(i0, kk);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (i0 + q >= hi) continue;
        if (kk[q] > tau) {
          ++sel;
        } else if (kk[q] == tau) {
          if (er < need_eq) ++sel;
          ++er;
        }
      }
    }
    int pos = block_exclusive_scan(sel, sh + 8, &tot);
    er = er0;
    for (int i0 = lo; i0 < hi; i0 += 8) {
      uint32_t kk[8];
      seg_keys(i0, kk);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (i0 + q >= hi) continue;
        if (kk[q] > tau) {
          out[pos++] = i0 + q;
        } else if (kk[q] == tau) {
          if (er < need_eq) out[pos++] = i0 + q;
          ++er;
        }
      }
    }
  }
  for (int a = tid; a < s.w; a += blockDim.x) out[kk_u + a] = P + a;
}


// ------------------------------------------------- keys in registers --
constexpr int kThr = 1024, kWarps = kThr / 32, kReps = 8;
constexpr int kCluster = 8;
constexpr int kMaxP = kThr * 32;                   // one CTA
constexpr int kMaxHalo = 64;                       // pooling radius of a cluster's CTAs
constexpr int kMaxClusterP = kCluster * kThr * 32;

__host__ __device__ constexpr int pad_at(int j) { return j + (j >> 5); }   // conflict-free segments

size_t reg_smem_bytes(int per, int halo) { return (size_t)(pad_at(kThr * per + 2 * halo) + 4) * 4; }

__device__ __forceinline__ uint32_t peer_addr(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(r)
      : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void peer_store(uint32_t a, int v) {
  asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ int peer_load(uint32_t a) {
  int v;
  asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_bar() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

constexpr int kSamples = 256;   // keys that place the candidates' bound

struct SelSmem {
  int hist[kReps][256];
  int sum[3][256];        // a pass's histogram (read by the peers of a cluster)
  int cnt[2][kWarps];     // per-warp counts of a counting step
  int tot[2][kCluster];   // per-CTA counts
  int scan[kWarps];
  int scan_tot[2][kCluster];   // keys above the cut and equal to it, per CTA
  int digit, left;
  uint32_t samp[kSamples];
  uint32_t bound;
  int cand_tot[kCluster];   // candidates per CTA
};

template <int kPer, int kCs>
__global__ void __launch_bounds__(kThr, 1) k_select_reg(const float* __restrict__ scores, Shape s,
                                                        int32_t* __restrict__ idx) {
  extern __shared__ float sc[];
  __shared__ SelSmem sh;
  chain_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int u = blockIdx.x / kCs, rank = blockIdx.x % kCs;
  const int P = s.P, h = s.pool_k / 2;
  const UnitRow ur = unit_row(s.units, u, s.B, s.n_fix);
  const int kk = ur.B - s.w;
  const float* c = scores + (size_t)u * P;
  int32_t* out = idx + ur.off;
  for (int a = rank * kThr + tid; a < s.w; a += kCs * kThr) out[kk + a] = P + a;
  if (kk <= 0) return;   // the same in every CTA of the cluster
  if (kk >= P) {
    for (int j = rank * kThr + tid; j < P; j += kCs * kThr) out[j] = j;
    return;
  }
  // the scores of the CTA's positions and, in a cluster, their neighbours
  const int first = rank * kThr * kPer, halo = kCs > 1 ? h : 0, s0 = first - halo;
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    const int i = e * kThr + tid, j = s0 + i;
    if (j >= 0 && j < P) sc[pad_at(i)] = __ldg(c + j);
  }
  if (kCs > 1 && tid < 2 * halo) {
    const int i = kPer * kThr + tid, j = s0 + i;
    if (j >= 0 && j < P) sc[pad_at(i)] = __ldg(c + j);
  }
  if (kCs > 1)
    cluster_bar();   // also: every peer runs before the first store into it
  else
    __syncthreads();
  auto at = [&](int j) { return sc[pad_at(j - s0)]; };
  const int lo = first + tid * kPer;
  uint32_t kr[kPer];
  if (s.pool_type == GRKV_POOL_MAX && h == 3) {
    // window max over w[e .. e + 6] from pairs and quadruples (cells outside [0, P) ignored)
    float w[kPer + 6];
    if (lo >= 3 && lo + kPer + 3 <= P) {
#pragma unroll
      for (int i = 0; i < kPer + 6; ++i) w[i] = at(lo - 3 + i);
    } else {
#pragma unroll
      for (int i = 0; i < kPer + 6; ++i) {
        const int j = lo - 3 + i;
        w[i] = (j >= 0 && j < P) ? at(j) : -INFINITY;
      }
    }
    float m2[kPer + 5], m4[kPer + 3];
#pragma unroll
    for (int i = 0; i < kPer + 5; ++i) m2[i] = fmaxf(w[i], w[i + 1]);
#pragma unroll
    for (int i = 0; i < kPer + 3; ++i) m4[i] = fmaxf(m2[i], m2[i + 2]);
#pragma unroll
    for (int e = 0; e < kPer; ++e)
      kr[e] = lo + e < P ? order_key(fmaxf(fmaxf(m4[e], m2[e + 4]), w[e + 6])) : 0u;
  } else {
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int j = lo + e;
      kr[e] = 0u;
      if (j < P) {
        float pv;
        if (s.pool_type == GRKV_POOL_MAX) {
          pv = at(j);
          for (int t = 1; t <= h; ++t) {
            if (j - t >= 0) pv = fmaxf(pv, at(j - t));
            if (j + t < P) pv = fmaxf(pv, at(j + t));
          }
        } else {
          double acc = 0.0;   // left to right, zero padding, divisor k
          for (int t = -h; t <= h; ++t)
            if (j + t >= 0 && j + t < P) acc += (double)at(j + t);
          pv = (float)(acc / (double)s.pool_k);
        }
        kr[e] = order_key(pv);
      }
    }
  }
  const int valid = max(0, min(kPer, P - lo));   // positions of this thread inside the prefix
  // Candidates: the keys at or above a bound that kSamples evenly spaced keys place a little
  // below the cut (three standard deviations of the sample's count, so the cut is nearly
  // always among them).  They are a few times kk keys, written in order of position to
  // shared memory (of the cluster's first CTA), and the exact cut is found among them.
  // Too few or too many (an unlucky sample, ties) leave it to the steps below, over all keys.
  // Only where a thread has 32 keys or every step spans a cluster: 256 units n - w = 32736
  // 51 -> 36 us, 32 of 131,008 95 -> 51 us; with 16 or fewer keys a thread in one CTA the
  // steps over all keys are as fast or faster (n - w = 16352 18.2 us either way, 8160 13 against 15).
  constexpr bool kCandidates = kPer * kCs >= 32;
  constexpr int kCap = kThr * kPer / 2;   // key and position per candidate, over the scores
  if (kCandidates && kk < kCap) {
    constexpr int kOwn = kSamples / kCs, kStride = kThr / kOwn;   // one sample every kStride threads
    if (tid % kStride == 0) {
      const uint32_t x = valid > 0 ? kr[0] : 0u;
      const int at_s = rank * kOwn + tid / kStride;
      if (kCs > 1) {
#pragma unroll
        for (int q = 0; q < kCs; ++q) peer_store(peer_addr(&sh.samp[at_s], q), (int)x);
      } else {
        sh.samp[at_s] = x;
      }
    }
    if (kCs > 1)
      cluster_bar();
    else
      __syncthreads();
    if (warp == 0) {
      const int nv = min(kSamples, (P + kStride * kPer - 1) / (kStride * kPer));   // inside the prefix
      const float q = (float)kk * (float)nv / (float)P;   // samples above the cut, on average
      const int r = (int)(q + 3.f * sqrtf(q) + 5.f);
      uint32_t x[kSamples / 32], bound = 0;
#pragma unroll
      for (int i = 0; i < kSamples / 32; ++i) x[i] = sh.samp[i * 32 + lane];
      if (r < nv) {
        // the r-th largest sample to its 18 leading bits
        for (int bit = 31; bit >= 14; --bit) {
          const uint32_t cand = bound | 1u << bit;
          int n = 0;
#pragma unroll
          for (int i = 0; i < kSamples / 32; ++i) n += x[i] >= cand;
          if (__reduce_add_sync(0xffffffffu, n) >= r) bound = cand;
        }
      }
      if (lane == 0) sh.bound = bound;
    }
    __syncthreads();
    const uint32_t bound = sh.bound;
    int mine = 0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) mine += e < valid && kr[e] >= bound;
    int total;
    int at_c = block_exclusive_scan(mine, sh.scan, &total);
    if (kCs > 1) {
      if (tid < kCs) peer_store(peer_addr(&sh.cand_tot[rank], tid), total);
      cluster_bar();
      total = 0;
#pragma unroll
      for (int q = 0; q < kCs; ++q) {
        if (q < rank) at_c += sh.cand_tot[q];
        total += sh.cand_tot[q];
      }
    }
    if (total >= kk && total <= kCap) {   // the same answer in every CTA of the cluster
      uint32_t* ck = (uint32_t*)sc;       // keys, then positions: the scores are spent
      uint32_t* cp = ck + kCap;
      const uint32_t k_at = peer_addr(ck, 0), p_at = peer_addr(cp, 0);
#pragma unroll
      for (int e = 0; e < kPer; ++e) {
        if (e < valid && kr[e] >= bound) {
          if (kCs > 1) {
            peer_store(k_at + 4 * at_c, (int)kr[e]);
            peer_store(p_at + 4 * at_c, lo + e);
          } else {
            ck[at_c] = kr[e];
            cp[at_c] = (uint32_t)(lo + e);
          }
          ++at_c;
        }
      }
      if (kCs > 1) {
        cluster_bar();
        if (rank != 0) return;
      } else {
        __syncthreads();
      }
      uint32_t tau;
      int need_eq;
      block_kth_largest(
          [&](int i, uint32_t* key) {
            *key = ck[i];
            return true;
          },
          total, kk, sh.hist[0], sh.scan, &tau, &need_eq);
      const int seg = (total + kThr - 1) / kThr;
      const int i0 = min(total, tid * seg), i1 = min(total, i0 + seg);
      int cnt = 0;   // above the cut (low half), equal to it
      for (int i = i0; i < i1; ++i) cnt += ck[i] > tau ? 1 : ck[i] == tau ? 1 << 16 : 0;
      int all;
      const int pre = block_exclusive_scan(cnt, sh.scan, &all);
      int gt = pre & 0xFFFF, eq = pre >> 16;
      for (int i = i0; i < i1; ++i) {
        const uint32_t x = ck[i];
        if (x > tau || (x == tau && eq < need_eq)) out[gt + min(eq, need_eq)] = (int)cp[i];
        gt += x > tau;
        eq += x == tau;
      }
      return;
    }
  }
  // sign and exponent: the largest prefix with at least kk keys at or above it
  uint32_t prefix = 0;
  int above = 0;   // keys at or past the upper end of the prefix's range
#pragma unroll 1
  for (int bit = 31; bit >= 23; --bit) {
    const uint32_t cand = prefix | 1u << bit;
    int n = 0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) n += kr[e] >= cand;   // padding keys are 0
    n = __reduce_add_sync(0xffffffffu, n);
    int* cnt = sh.cnt[bit & 1];
    if (lane == 0) cnt[warp] = n;
    __syncthreads();
    n = __reduce_add_sync(0xffffffffu, cnt[lane]);
    if (kCs > 1) {
      int* tot = sh.tot[bit & 1];
      if (tid < kCs) peer_store(peer_addr(&tot[rank], tid), n);
      cluster_bar();
      n = 0;
#pragma unroll
      for (int q = 0; q < kCs; ++q) n += tot[q];
    }
    if (n >= kk)
      prefix = cand;
    else
      above = n;
  }
  // mantissa: 8, 8 and 7 bits
  uint32_t mask = 0xFF800000u;
  int rem = kk - above;
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    const int shift = pass == 0 ? 15 : pass == 1 ? 7 : 0;
    const uint32_t dmask = pass == 2 ? 127u : 255u;
    for (int i = tid; i < kReps * 256; i += kThr) (&sh.hist[0][0])[i] = 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < kPer; ++e)
      if (e < valid && (kr[e] & mask) == prefix)
        atomicAdd(&sh.hist[warp % kReps][(kr[e] >> shift) & dmask], 1);
    __syncthreads();
    if (tid < 256) {
      int t = 0;
#pragma unroll
      for (int q = 0; q < kReps; ++q) t += sh.hist[q][tid];
      sh.sum[pass][tid] = t;
    }
    if (kCs > 1)
      cluster_bar();
    else
      __syncthreads();
    if (warp == 0) {
      // digit search from 255 down: lane l owns bins 8l .. 8l + 7
      int n[8], own = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        n[q] = 0;
        if (kCs > 1) {
#pragma unroll
          for (int r = 0; r < kCs; ++r) n[q] += peer_load(peer_addr(&sh.sum[pass][8 * lane + q], r));
        } else {
          n[q] = sh.sum[pass][8 * lane + q];
        }
        own += n[q];
      }
      int suf = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf += y;
      }
      int up = suf - own, dg = -1, left = 0;
#pragma unroll
      for (int q = 7; q >= 0; --q) {
        if (dg < 0 && (up + n[q] >= rem || (lane == 0 && q == 0))) {
          dg = 8 * lane + q;
          left = rem - up;
        }
        up += n[q];
      }
      const unsigned found = __ballot_sync(0xffffffffu, dg >= 0);
      const int src = 31 - __clz(found);
      const int dsel = __shfl_sync(0xffffffffu, dg, src), lsel = __shfl_sync(0xffffffffu, left, src);
      if (lane == 0) {
        sh.digit = dsel;
        sh.left = lsel;
      }
    }
    __syncthreads();
    prefix |= (uint32_t)sh.digit << shift;
    mask |= dmask << shift;
    rem = sh.left;
  }
  // positions: a scan of the counts above the cut (low half) and equal to it
  uint32_t mine = 0;
#pragma unroll
  for (int e = 0; e < kPer; ++e)
    if (e < valid) mine += kr[e] > prefix ? 1u : kr[e] == prefix ? 1u << 16 : 0u;
  uint32_t inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sh.scan[warp] = (int)inc;
  __syncthreads();
  uint32_t wt = (uint32_t)sh.scan[lane];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, wt, o);
    if (lane >= o) wt += y;
  }
  const uint32_t total = __shfl_sync(0xffffffffu, wt, 31);
  const uint32_t before_warp = __shfl_sync(0xffffffffu, wt, warp == 0 ? 0 : warp - 1);
  const uint32_t pre = (warp == 0 ? 0u : before_warp) + inc - mine;
  int gt = (int)(pre & 0xFFFFu), eq = (int)(pre >> 16);
  if (kCs > 1) {
    if (tid < kCs) {
      peer_store(peer_addr(&sh.scan_tot[0][rank], tid), (int)(total & 0xFFFFu));
      peer_store(peer_addr(&sh.scan_tot[1][rank], tid), (int)(total >> 16));
    }
    cluster_bar();
    for (int q = 0; q < rank; ++q) {
      gt += sh.scan_tot[0][q];
      eq += sh.scan_tot[1][q];
    }
  }
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    if (e >= valid) break;
    const bool is_eq = kr[e] == prefix;
    if (kr[e] > prefix || (is_eq && eq < rem)) out[gt + min(eq, rem)] = lo + e;
    gt += kr[e] > prefix;
    eq += is_eq;
  }
  if (kCs > 1) cluster_bar();   // no CTA leaves while a peer may read its histograms
}

template <int kPer, int kCs>
cudaError_t launch_reg(const Shape& s, const float* scores, int32_t* idx, cudaStream_t st) {
  auto kern = k_select_reg<kPer, kCs>;
  const size_t bytes = reg_smem_bytes(kPer, kCs > 1 ? kMaxHalo : 0);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  if (kCs > 1 && !cluster_fits(kCs, kern, kThr, bytes)) return cudaErrorInvalidClusterSize;
  return launch_kernel(s.chained, kCs, kern, dim3((unsigned)s.U * kCs), kThr, bytes, st, scores, s, idx);
}

}  // namespace

bool select_uses_pooled_buffer(const Shape& s) { return s.P > kMaxP; }

cudaError_t launch_select_pooled(const Shape& s, const float* scores, int32_t* idx,
                                 float* pooled, cudaStream_t st) {
  count_launches(1);
  const int per = (s.P + kThr - 1) / kThr;
  if (per <= 2) return launch_reg<2, 1>(s, scores, idx, st);
  if (per <= 4) return launch_reg<4, 1>(s, scores, idx, st);
  if (per <= 8) return launch_reg<8, 1>(s, scores, idx, st);
  if (per <= 16) return launch_reg<16, 1>(s, scores, idx, st);
  if (per <= 32) return launch_reg<32, 1>(s, scores, idx, st);
  cudaError_t e = cudaErrorInvalidClusterSize;   // until a cluster takes it
  if (s.pool_k / 2 <= kMaxHalo) {
    if (per <= 8 * kCluster)
      e = launch_reg<8, kCluster>(s, scores, idx, st);
    else if (per <= 16 * kCluster)
      e = launch_reg<16, kCluster>(s, scores, idx, st);
    else if (s.P <= kMaxClusterP)
      e = launch_reg<32, kCluster>(s, scores, idx, st);
  }
  if (e != cudaErrorInvalidClusterSize) return e;
  return launch_kernel(s.chained, 1, k_select, dim3(s.U), 1024, 0, st, scores, s, pooled, idx);
}

cudaError_t launch_select(const Shape& s, const float* scores, int32_t* idx, char* ws,
                          const WsLayout& L, cudaStream_t st) {
  return launch_select_pooled(s, scores, idx, (float*)(ws + L.pooled), st);
}

}  // namespace grkv
