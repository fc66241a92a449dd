// The key step (Sec. 3.4 "Key step", App. D.2) for m <= 128 and at most 64 retained
// columns per CTA: one cluster of kC CTAs per unit, everything between the
// inputs and K* on chip.  The mathematics is grkv_key.cu's: with X the retained attention
// at K0 and V* the merged values,
//   e = Y - X V*,  (J_G J_G^T + lambda_k I) alpha = e by conjugate gradients,
//   J_G J_G^T p = (X o (T2 - rho2)) V*,  rho2 = rowsum(X o T2),
//   T2 = s^2 Q Q^T (X o (p V*^T - rho1)) on the free columns (0 on fixed ones),
//   rho1 = rowsum(p o X V*),  K*_G = K0_G + s (X o (alpha V*^T - rho1))^T Q.
//
// Rank c carries retained columns [c Bc, c Bc + nc) of the three products and
// d-columns [c W, c W + W), W = 128 / kC, of the CG vectors.  Products run on
// tcgen05 with fp32 operands as three bf16 parts (the six part products of
// combined order <= 2): V* and s^2 Q Q^T stay in shared memory, p and dS2 are A operands
// in TMEM, X is held in registers (thread = window row x 32 columns).  Partial
// results cross the cluster by st.async into the owner's shared memory, each
// exchange completing one mbarrier: rho2; the product's slices to their
// owners; p . Ap; ||r||^2; p's slices and rho1 to everyone.  Every rank adds in rank
// order, so all hold the same scalars and take the same branches.
//
// Bound by latency: three dependent products and five exchanges an iteration, 37 K cycles
// (17.7 us; 8 units of m = 128, B = 512), the tensor pipe busy in 13% of them.  The split
// through global memory that this replaces staged every operand in each iteration and met
// at two global barriers: 95 us an iteration.
#include <cmath>
#include <type_traits>

#include "grkv_internal.cuh"
#include "key_args.cuh"
#include "sm100.cuh"

namespace grkv {
namespace {

using namespace sm100;

constexpr int kThr = 256;
constexpr int kNc = 64;                        // retained columns per CTA at most
constexpr long long kWaitBudget = 1ll << 32;   // clock cycles of a bounded wait

constexpr uint32_t kQPart = 128 * 128 * 2;     // one part of Q or of s^2 Q Q^T
constexpr uint32_t kVPart = kNc * 128 * 2;     // one part of the CTA's K0 or V*
constexpr uint32_t kSPart = 128 * kNc * 2;     // one part of dS
constexpr uint32_t kDBytes = 128 * 128 * 4;    // dS parts, or the exchanged m x d values

// TMEM columns: parts of p (or alpha; Q Q^T at first), parts of dS2 (or X), then
// T, the three orders of T2, or the product with V*.
constexpr uint32_t kColP = 0, kColX = 192, kColT = 288, kColO = kColT;

template <int kC>
struct alignas(16) Misc {
  float rho1[2 * kC][128];    // partial row sums by (rank, half of its slice)
  float rho2[kC][128];        // partial row sums by rank
  float half[2][128];         // the two column halves of a row within the CTA
  float red[2][kThr / 32];
  float scal[2][kC];
  uint64_t mma, ex_rho2, ex_out, ex_pap, ex_rn, ex_p;
  uint32_t tmem;
  int abort;
};

template <typename T, int kC>
struct Smem {
  static constexpr int kParts = std::is_same<T, float>::value ? 3 : 1;   // of Q, K0 and V*
  static constexpr uint32_t kOffV = 3 * kQPart, kOffD = kOffV + kParts * kVPart,
                            kOffMisc = kOffD + kDBytes,
                            kBytes = kOffMisc + sizeof(Misc<kC>) + 1024;
};
static_assert(Smem<float, 8>::kBytes <= 232448, "shared memory of one CTA");
static_assert(3 * kSPart <= kDBytes, "dS shares its place with the exchanges");

__device__ __forceinline__ uint32_t peer(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_async(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                   addr),
               "r"(__float_as_uint(v)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async4(uint32_t addr, const float* v, uint32_t bar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::
          "r"(addr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
      "r"(__float_as_uint(v[3])), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// mbar_wait for a barrier that peers complete: acquires at cluster scope.
__device__ __forceinline__ bool peer_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
  long long t0 = 0;
  while (true) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n"
        " mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (*abort) return false;
    if (t0 == 0) t0 = clock64();
    if (clock64() - t0 > kWaitBudget) {
      *abort = 1;
      return false;
    }
  }
}

__device__ __forceinline__ float lo16(uint32_t h) { return __uint_as_float(h << 16); }
__device__ __forceinline__ float hi16(uint32_t h) { return __uint_as_float(h & 0xFFFF0000u); }

// A pair of values into its three bf16 parts, packed.
__device__ __forceinline__ void split_pair(float a, float b, uint32_t* p) {
  p[0] = pack_bf16(a, b);
  const float a1 = a - lo16(p[0]), b1 = b - hi16(p[0]);
  p[1] = pack_bf16(a1, b1);
  p[2] = pack_bf16(a1 - lo16(p[1]), b1 - hi16(p[1]));
}

// Eight contiguous elements into kParts swizzled 16-byte chunks.
__device__ __forceinline__ void stage8(const __nv_bfloat16* src, bool in, uint8_t* dst, uint32_t) {
  *(uint4*)dst = in ? __ldg((const uint4*)src) : make_uint4(0, 0, 0, 0);
}
__device__ __forceinline__ void stage8(const float* src, bool in, uint8_t* dst, uint32_t part) {
  uint32_t p[4][3] = {};
  if (in) {
    const float4 a = __ldg((const float4*)src), b = __ldg((const float4*)src + 1);
    split_pair(a.x, a.y, p[0]);
    split_pair(a.z, a.w, p[1]);
    split_pair(b.x, b.y, p[2]);
    split_pair(b.z, b.w, p[3]);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q)
    *(uint4*)(dst + q * part) = make_uint4(p[0][q], p[1][q], p[2][q], p[3][q]);
}
// rows x 128 values as two halves of 64 columns, 128-byte swizzled rows (the
// K-major image of the rows and the MN-major one of their transpose)
template <typename T>
__device__ __forceinline__ void stage_tile(const T* src, int rows, int valid, uint8_t* dst,
                                           uint32_t part) {
  for (int i = threadIdx.x; i < rows * 16; i += kThr) {
    const int r = i >> 4, c = i & 15;
    stage8(src + (size_t)r * kD + c * 8, r < valid,
           dst + (c >> 3) * (rows * 128) + sw128_offset(r, c & 7), part);
  }
}

__device__ __forceinline__ float elem(const float* p, size_t i) { return p[i]; }
__device__ __forceinline__ float elem(const __nv_bfloat16* p, size_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void put(float* p, size_t i, float v) { p[i] = v; }
__device__ __forceinline__ void put(__nv_bfloat16* p, size_t i, float v) { p[i] = __float2bfloat16_rn(v); }

template <typename T, int kC>
__global__ void __launch_bounds__(kThr, 1) k_key_cluster(KeyClusterArgs a) {
  using S = Smem<T, kC>;
  constexpr int kParts = S::kParts;
  constexpr int kW = 128 / kC, kH = kW / 2, kCh = kH / 4;   // slice, columns of it per thread, in fours
  extern __shared__ uint8_t raw[];
  uint8_t* sm = (uint8_t*)(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
  uint8_t *gq = sm, *vt = sm + S::kOffV, *dt = sm + S::kOffD;
  Misc<kC>& x = *(Misc<kC>*)(sm + S::kOffMisc);
  float4* dbuf = (float4*)dt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = (warp & 3) * 32 + lane, half = warp >> 2;
  const int u = blockIdx.x / kC, rank = blockIdx.x % kC;
  const int m = a.m, B = a.B;
  const int Bc = ((B + kC - 1) / kC + 7) / 8 * 8;
  const int c0 = min(B, rank * Bc), nc = min(B, c0 + Bc) - c0;
  const int nn = max(16, (Bc + 15) / 16 * 16);     // columns of the MMAs
  const size_t kv = ((size_t)u * B + c0) * kD;
  const T* q = (const T*)a.q + (size_t)u * m * kD;
  const T* vs = (const T*)a.v_out + kv;
  T* ko = (T*)a.k_out + kv;

  if (tid == 0) {
    for (uint64_t* bar : {&x.mma, &x.ex_rho2, &x.ex_out, &x.ex_pap, &x.ex_rn, &x.ex_p}) mbar_init(bar, 1);
    x.abort = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&x.tmem, 512);
    tmem_relinquish();
  }
  stage_tile(q, 128, m, gq, kQPart);
  stage_tile((const T*)ko, kNc, nc, vt, kVPart);
  fence_proxy_async_smem();
  __syncthreads();
  cluster_sync();   // every rank's barriers are initialised
  tc_fence_after();
  const uint32_t tm = x.tmem, lane_tm = tm + ((uint32_t)((warp & 3) * 32) << 16);
  const uint32_t gqa = smem_u32(gq), vta = smem_u32(vt), dta = smem_u32(dt);
  uint32_t ph_mma = 0, ph_rho2 = 0, ph_out = 0, ph_pap = 0, ph_rn = 0, ph_p = 0;
  bool live = true;

  auto wait = [&](uint64_t* bar, uint32_t& ph) {
    const bool ok = peer_wait(bar, ph, &x.abort);
    __syncwarp();   // tcgen05 loads and stores follow, warp by warp
    ph ^= 1;
    return ok;
  };
  // every earlier write of the CTA is visible to the MMAs issued next by thread 0
  auto ready = [&](bool ok) {
    tc_fence_before();
    live = __syncthreads_and(ok) && live;
    if (tid == 0) tc_fence_after();
    return live;
  };
  auto mma_done = [&]() {
    const bool ok = wait(&x.mma, ph_mma);
    tc_fence_after();
    return ok;
  };
  // the part products of combined order <= 2
  auto products = [&](int pa_n, int pb_n, auto issue) {
    uint32_t acc = 0;
    for (int pa = 0; pa < pa_n; ++pa)
      for (int pb = 0; pb < pb_n; ++pb)
        if (pa + pb <= 2) {
          issue(pa, pb, acc);
          acc = 1;
        }
    mma_commit(&x.mma);
  };
  // The once-per-unit products, as exact as fp32 multiply-add chains: parts of combined order
  // <= 3, the leading one alone in the first accumulator (low = 0), the others in the second.
  // With one accumulator for the six parts of order <= 2 the update's error after one iteration
  // (fp32 inputs, of |K* - K0|) is 1.4 to 3.0e-5, with two 0.2 to 0.5e-5, in plain fp32 0.7 to
  // 1.4e-5: the residual Y - X V* is a small difference.  2 us more a call for 8 units.
  auto products2 = [&](int pa_n, int pb_n, auto issue) {
    uint32_t acc = 0;
    for (int pa = 0; pa < pa_n; ++pa)
      for (int pb = 0; pb < pb_n; ++pb) {
        if (pa + pb > 3) continue;
        const int low = pa + pb > 0;
        issue(pa, pb, low, low ? acc : 0u);
        acc |= low;
      }
    mma_commit(&x.mma);
  };
  // the sum of two accumulators' 32 columns
  auto load2 = [&](uint32_t col, uint32_t col_low, float* v) {
    float l[32];
    tmem_ld32f(lane_tm + col_low, l);
    tmem_ld32f(lane_tm + col, v);
    tmem_wait32(l);
    tmem_wait32(v);
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] += l[e];
  };
  auto split_store_tmem = [&](const float* v, uint32_t col, uint32_t part_cols) {   // 32 values
    uint32_t w[3][16];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      uint32_t p[3];
      split_pair(v[2 * e], v[2 * e + 1], p);
      w[0][e] = p[0];
      w[1][e] = p[1];
      w[2][e] = p[2];
    }
#pragma unroll
    for (int q3 = 0; q3 < 3; ++q3) tmem_st16(lane_tm + col + q3 * part_cols, w[q3]);
  };
  auto block_sum = [&](float v, float* red) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < kThr / 32; ++i) t += red[i];
    return t;
  };
  // a scalar summed over the ranks
  auto all_sum = [&](float v, int which, uint64_t* bar, uint32_t& ph) {
    v = block_sum(v, x.red[which]);
    if (tid < kC) st_async(peer(smem_u32(&x.scal[which][rank]), tid), v, peer(smem_u32(bar), tid));
    if (tid == 0) mbar_expect_tx(bar, kC * 4);
    live = __syncthreads_and(wait(bar, ph)) && live;
    float t = 0.f;
#pragma unroll
    for (int c = 0; c < kC; ++c) t += x.scal[which][c];
    return t;
  };
  // the CTA's per-row value (both halves combined by `op`) to every rank's dst[rank][row]
  auto send_row = [&](float v, float* dst, uint64_t* bar, auto op) {
    x.half[half][row] = v;
    __syncthreads();
    v = op(x.half[0][row], x.half[1][row]);
    const uint32_t at = smem_u32(dst + rank * 128 + row), b = smem_u32(bar);
#pragma unroll
    for (int c = 0; c < kC / 2; ++c) st_async(peer(at, half * (kC / 2) + c), v, peer(b, half * (kC / 2) + c));
    if (tid == 0) mbar_expect_tx(bar, kC * 128 * 4);
  };
  auto sum2 = [](float p, float r) { return p + r; };
  // the rows' partial product (64 columns of kColO per thread; two: its second accumulator
  // in kColP) to the slices' owners
  auto send_out = [&](auto two) {
    const uint32_t at = smem_u32(dbuf), b = smem_u32(&x.ex_out);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float v[32];
      const uint32_t c = 64 * half + 32 * h;
      if constexpr (decltype(two)::value) {
        load2(kColO + c, kColP + c, v);
      } else {
        tmem_ld32f(lane_tm + kColO + c, v);
        tmem_wait32(v);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int col4 = 16 * half + 8 * h + e, owner = col4 / (kW / 4), ch = col4 % (kW / 4);
        st_async4(peer(at + ((rank * (kW / 4) + ch) * 128 + row) * 16, owner), v + 4 * e, peer(b, owner));
      }
    }
    if (tid == 0) mbar_expect_tx(&x.ex_out, kDBytes);
  };
  // ... and the owner's sum over the ranks
  auto recv_out = [&](float* o) {
#pragma unroll
    for (int e = 0; e < kCh; ++e) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int c = 0; c < kC; ++c) {
        const float4 t = dbuf[(c * (kW / 4) + half * kCh + e) * 128 + row];
        s.x += t.x;
        s.y += t.y;
        s.z += t.z;
        s.w += t.w;
      }
      o[4 * e] = s.x;
      o[4 * e + 1] = s.y;
      o[4 * e + 2] = s.z;
      o[4 * e + 3] = s.w;
    }
  };

  // ---- S = Q K0^T and Q Q^T
  if (tid == 0) {
    products2(kParts, kParts, [&](int pa, int pb, int low, uint32_t acc) {
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        mma_bf16(tm + kColT + 64 * low, sw128_desc(gqa + pa * kQPart + (kk >> 2) * (kQPart / 2) + (kk & 3) * 32, 16, 1024),
                 sw128_desc(vta + pb * kVPart + (kk >> 2) * (kVPart / 2) + (kk & 3) * 32, 16, 1024),
                 idesc_bf16(128, nn, 0, 0), acc | (kk > 0));
    });
  }
  live = __syncthreads_and(mma_done()) && live;
  if (tid == 0) {
    products2(kParts, kParts, [&](int pa, int pb, int low, uint32_t acc) {
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
        mma_bf16(tm + kColP + 128 * low, sw128_desc(gqa + pa * kQPart + (kk >> 2) * (kQPart / 2) + (kk & 3) * 32, 16, 1024),
                 sw128_desc(gqa + pb * kQPart + (kk >> 2) * (kQPart / 2) + (kk & 3) * 32, 16, 1024),
                 idesc_bf16(128, 128, 0, 0), acc | (kk > 0));
    });
  }
  float X[32];
  uint32_t vis = 0, fixed = 0;   // bit e: column 32 half + e
  if constexpr (kParts > 1) {
    load2(kColT + 32 * half, kColT + 64 + 32 * half, X);
  } else {
    tmem_ld32f(lane_tm + kColT + 32 * half, X);
    tmem_wait32(X);
  }
  {
    const int lim = a.causal ? a.n - a.w + row % a.w : a.n - 1;
    const int32_t* idx = a.idx + (size_t)u * B + c0;
    const uint8_t* fx = a.fixed + (size_t)u * B + c0;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      const int j = 32 * half + e;
      if (j >= nc) continue;
      const int pos = __ldg(idx + j);
      if (row < m && ((unsigned)pos < (unsigned)a.n ? pos : 0) <= lim) vis |= 1u << e;
      if (__ldg(fx + j)) fixed |= 1u << e;
    }
  }
  float mx = -INFINITY;
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    X[e] *= a.scale;
    if (vis >> e & 1) mx = fmaxf(mx, X[e]);
  }
  send_row(mx, &x.rho2[0][0], &x.ex_rho2, [](float p, float r) { return fmaxf(p, r); });
  live = __syncthreads_and(wait(&x.ex_rho2, ph_rho2)) && live;
  mx = x.rho2[0][row];
#pragma unroll
  for (int c = 1; c < kC; ++c) mx = fmaxf(mx, x.rho2[c][row]);
  float sum = 0.f;
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    X[e] = (vis >> e & 1) ? expf(X[e] - mx) : 0.f;
    sum += X[e];
  }
  // (rho1 and its barrier: the maxima may still be being read elsewhere)
  send_row(sum, &x.rho1[0][0], &x.ex_p, sum2);
  // s^2 Q Q^T: three parts over Q, which its product has read
  bool ok = mma_done();
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    float v[32];
    const uint32_t c = 64 * half + 32 * h;
    if constexpr (kParts > 1) {
      load2(kColP + c, kColP + 128 + c, v);
    } else {
      tmem_ld32f(lane_tm + kColP + c, v);
      tmem_wait32(v);
    }
    const float s2 = a.scale * a.scale;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      uint32_t p[4][3];
#pragma unroll
      for (int z = 0; z < 4; ++z) split_pair(s2 * v[8 * e + 2 * z], s2 * v[8 * e + 2 * z + 1], p[z]);
#pragma unroll
      for (int q3 = 0; q3 < 3; ++q3)
        *(uint4*)(gq + q3 * kQPart + half * (kQPart / 2) + sw128_offset(row, 4 * h + e)) =
            make_uint4(p[0][q3], p[1][q3], p[2][q3], p[3][q3]);
    }
  }
  stage_tile(vs, kNc, nc, vt, kVPart);   // V* over K0
  ok = wait(&x.ex_p, ph_p) && ok;
  sum = 0.f;
#pragma unroll
  for (int c = 0; c < kC; ++c) sum += (&x.rho1[0][0])[c * 128 + row];
  const float inv = sum > 0.f ? 1.f / sum : 0.f;
#pragma unroll
  for (int e = 0; e < 32; ++e) X[e] *= inv;

  // ---- products of the CG
  auto issue_out = [&](uint32_t col, int pa, int pb, uint32_t acc) {   // (parts at kColX) V*
    for (int kk = 0; kk < nn / 16; ++kk)
      mma_bf16_ts(tm + col, tm + kColX + pa * 32 + kk * 8,
                  sw128_desc(vta + pb * kVPart + kk * 2048, kVPart / 2, 1024),
                  idesc_bf16(128, 128, 0, 1), acc | (kk > 0));
  };
  auto out_product = [&]() {
    if (tid == 0)
      products(3, kParts, [&](int pa, int pb, uint32_t acc) { issue_out(kColO, pa, pb, acc); });
  };
  if (kParts > 1) {   // Q Q^T's second accumulator has been read by all: X's parts overlap it
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  split_store_tmem(X, kColX + 16 * half, 32);
  tmem_st_wait();
  fence_proxy_async_smem();
  float xv[kH], r[kH], p[kH], al[kH];
#pragma unroll
  for (int e = 0; e < kH; ++e) xv[e] = r[e] = p[e] = al[e] = 0.f;
  float rs = 0.f, stop = 0.f;
  if (ready(ok)) {
    if (tid == 0)
      products2(3, kParts, [&](int pa, int pb, int low, uint32_t acc) {
        issue_out(low ? kColP : kColO, pa, pb, acc);
      });
    ok = mma_done();
    send_out(std::true_type());
    tc_fence_before();
    live = __syncthreads_and(wait(&x.ex_out, ph_out) && ok) && live;
    tc_fence_after();   // the second accumulator's columns take p next
    recv_out(xv);
    const float* y = a.y + ((size_t)u * m + min(row, m - 1)) * kD + rank * kW + half * kH;
#pragma unroll
    for (int e = 0; e < kH; ++e) {
      r[e] = row < m ? __ldg(y + e) - xv[e] : 0.f;
      p[e] = r[e];
      rs = fmaf(r[e], r[e], rs);
    }
    rs = all_sum(rs, 1, &x.ex_rn, ph_rn);
    stop = a.tol * a.tol * rs;
  }

  // T = v V*^T for the slices v of every rank (p or alpha) in kColT, and rho1 = rowsum(v o X V*)
  float rho1 = 0.f;
  auto t_product = [&](const float* v) {
    float part = 0.f;
#pragma unroll
    for (int e = 0; e < kH; ++e) part = fmaf(v[e], xv[e], part);
    const uint32_t at = smem_u32(dbuf + (rank * (kW / 4) + half * kCh) * 128 + row);
    const uint32_t ar = smem_u32(&x.rho1[2 * rank + half][row]), b = smem_u32(&x.ex_p);
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      const uint32_t bc = peer(b, c), atc = peer(at, c);
#pragma unroll
      for (int e = 0; e < kCh; ++e) st_async4(atc + e * 2048, v + 4 * e, bc);
      st_async(peer(ar, c), part, bc);
    }
    if (tid == 0) mbar_expect_tx(&x.ex_p, kDBytes + 2 * kC * 128 * 4);
    bool w = wait(&x.ex_p, ph_p);
    rho1 = 0.f;
#pragma unroll
    for (int c = 0; c < 2 * kC; ++c) rho1 += x.rho1[c][row];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float f[32];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float4 t = dbuf[(16 * half + 8 * h + e) * 128 + row];
        f[4 * e] = t.x;
        f[4 * e + 1] = t.y;
        f[4 * e + 2] = t.z;
        f[4 * e + 3] = t.w;
      }
      split_store_tmem(f, kColP + 32 * half + 16 * h, 64);
    }
    tmem_st_wait();
    if (!ready(w)) return;
    if (tid == 0)
      products(3, kParts, [&](int pa, int pb, uint32_t acc) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_bf16_ts(tm + kColT, tm + kColP + pa * 64 + kk * 8,
                      sw128_desc(vta + pb * kVPart + (kk >> 2) * (kVPart / 2) + (kk & 3) * 32, 16, 1024),
                      idesc_bf16(128, nn, 0, 0), acc | (kk > 0));
      });
  };
  // dS = X o (T - rho1) as three parts in shared memory, [row][64 columns]
  auto stage_ds = [&]() {
    float t[32];
    tmem_ld32f(lane_tm + kColT + 32 * half, t);
    tmem_wait32(t);
#pragma unroll
    for (int e = 0; e < 32; ++e) t[e] = 32 * half + e < nc ? X[e] * (t[e] - rho1) : 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      uint32_t w[4][3];
#pragma unroll
      for (int z = 0; z < 4; ++z) split_pair(t[8 * e + 2 * z], t[8 * e + 2 * z + 1], w[z]);
#pragma unroll
      for (int q3 = 0; q3 < 3; ++q3)
        *(uint4*)(dt + q3 * kSPart + sw128_offset(row, 4 * half + e)) =
            make_uint4(w[0][q3], w[1][q3], w[2][q3], w[3][q3]);
    }
    fence_proxy_async_smem();
  };

  for (int it = 0; it < a.iters && live; ++it) {
    if (!(rs > stop) || !(rs > 0.f)) break;
    t_product(p);
    if (!live) break;
    ok = mma_done();
    stage_ds();
    if (!ready(ok)) break;
    if (tid == 0)
      products(3, 1, [&](int pa, int, uint32_t acc) {
        // T2 = (s^2 Q Q^T) dS: part pa meets parts 0 .. 2 - pa of dS side by side (64
        // columns each), so that order o = pa + pb gathers at columns 64 o; one part pair at
        // a time, each MMA would read A again for half the columns (3.7 K cycles against 1.9 K)
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_bf16(tm + kColT + 64 * pa,
                   sw128_desc(gqa + pa * kQPart + (kk >> 2) * (kQPart / 2) + (kk & 3) * 32, 16, 1024),
                   sw128_desc(dta + kk * 2048, kSPart, 1024),
                   idesc_bf16(128, 64 * (3 - pa), 0, 1), acc | (kk > 0));
      });
    ok = mma_done();
    float t[32], t1[32];
    tmem_ld32f(lane_tm + kColT + 64 + 32 * half, t1);
    tmem_wait32(t1);
    tmem_ld32f(lane_tm + kColT + 128 + 32 * half, t);
    tmem_wait32(t);
#pragma unroll
    for (int e = 0; e < 32; ++e) t1[e] += t[e];
    tmem_ld32f(lane_tm + kColT + 32 * half, t);
    tmem_wait32(t);
    float rho2 = 0.f;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      t[e] = (fixed >> e & 1) || 32 * half + e >= nc ? 0.f : t[e] + t1[e];
      rho2 = fmaf(X[e], t[e], rho2);
    }
    send_row(rho2, &x.rho2[0][0], &x.ex_rho2, sum2);
    ok = wait(&x.ex_rho2, ph_rho2) && ok;
    rho2 = 0.f;
#pragma unroll
    for (int c = 0; c < kC; ++c) rho2 += x.rho2[c][row];
#pragma unroll
    for (int e = 0; e < 32; ++e) t[e] = X[e] * (t[e] - rho2);
    split_store_tmem(t, kColX + 16 * half, 32);
    tmem_st_wait();
    if (!ready(ok)) break;
    out_product();
    ok = mma_done();
    send_out(std::false_type());
    live = __syncthreads_and(wait(&x.ex_out, ph_out) && ok) && live;
    float ap[kH], pap = 0.f;
    recv_out(ap);
#pragma unroll
    for (int e = 0; e < kH; ++e) {
      ap[e] = fmaf(a.lambda_k, p[e], ap[e]);
      pap = fmaf(p[e], ap[e], pap);
    }
    pap = all_sum(pap, 0, &x.ex_pap, ph_pap);
    if (!live || !(pap > 0.f)) break;   // the direction has vanished
    const float step = rs / pap;
    float rn = 0.f;
#pragma unroll
    for (int e = 0; e < kH; ++e) {
      al[e] = fmaf(step, p[e], al[e]);
      r[e] = fmaf(-step, ap[e], r[e]);
      rn = fmaf(r[e], r[e], rn);
    }
    rn = all_sum(rn, 1, &x.ex_rn, ph_rn);
    const float beta = rn / rs;
#pragma unroll
    for (int e = 0; e < kH; ++e) p[e] = fmaf(beta, p[e], r[e]);
    rs = rn;
  }

  // ---- K*_G = K0_G + s dS^T Q with dS at alpha: as (s Q^T dS), d on the lanes
  if (live) t_product(al);
  if (live) {
    ok = mma_done();
    stage_tile(q, 128, m, gq, kQPart);
    stage_ds();
    if (ready(ok)) {
      if (tid == 0)
        products2(kParts, 3, [&](int pa, int pb, int low, uint32_t acc) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_bf16(tm + kColT + 64 * low, sw128_desc(gqa + pa * kQPart + kk * 2048, kQPart / 2, 1024),
                     sw128_desc(dta + pb * kSPart + kk * 2048, kSPart, 1024),
                     idesc_bf16(128, nn, 1, 1), acc | (kk > 0));
        });
      live = __syncthreads_and(mma_done()) && live;
      float dk[32];
      load2(kColT + 32 * half, kColT + 64 + 32 * half, dk);
      const int d = row;
      if (live)
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          const int j = 32 * half + e;
          if (j >= nc) continue;
          const size_t o = (size_t)j * kD + d;
          const float k0 = elem(ko, o);
          const bool keep = fixed >> e & 1;
          const float v = keep ? k0 : fmaf(a.scale, dk[e], k0);
          if (a.Kt) a.Kt[kv + o] = v;
          if (!keep) put(ko, o, v);
        }
    }
  }
  if (!live && tid == 0) set_status(a.status, GRKV_ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // no peer still writes here
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tm, 512);
}

template <typename T, int kC>
cudaError_t launch(const KeyClusterArgs& a, int U, cudaStream_t st, bool* done) {
  auto kern = k_key_cluster<T, kC>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)Smem<T, kC>::kBytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kC;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)U * kC);
  cfg.blockDim = dim3(kThr);
  cfg.dynamicSmemBytes = Smem<T, kC>::kBytes;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int nclusters = 0;
  if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) != cudaSuccess || nclusters < 1) {
    (void)cudaGetLastError();
    return cudaSuccess;   // not on this device: the caller takes the other path
  }
  *done = true;
  count_launches(1);
  return cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace

// A rank holds at most 64 columns.  Few units take the widest cluster (an
// iteration's elementwise work shrinks with the columns of a rank); more
// units than that fills take the smallest one that holds B.
cudaError_t launch_key_cluster(const Shape& s, const KeyClusterArgs& a, cudaStream_t st, bool* done) {
  *done = false;
  if (s.m > 128 || s.B > 8 * kNc) return cudaSuccess;
  const bool f32 = s.dtype == GRKV_F32;
  int c = 8;
  while (c > 2 && s.U * c > 152 && s.B <= c / 2 * kNc) c /= 2;
  if (c == 8) return f32 ? launch<float, 8>(a, s.U, st, done) : launch<__nv_bfloat16, 8>(a, s.U, st, done);
  if (c == 4) return f32 ? launch<float, 4>(a, s.U, st, done) : launch<__nv_bfloat16, 4>(a, s.U, st, done);
  return f32 ? launch<float, 2>(a, s.U, st, done) : launch<__nv_bfloat16, 2>(a, s.U, st, done);
}

}  // namespace grkv
