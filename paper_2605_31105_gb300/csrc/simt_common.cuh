// Pieces shared by the portable CUDA-core kernels (window scoring in
// grkv_simt.cu, the value step in grkv_simt_merge.cu).
#pragma once

#include "grkv_internal.cuh"

namespace grkv {
namespace {

__device__ __forceinline__ float ldv(const float* p, size_t i) { return p[i]; }
__device__ __forceinline__ float ldv(const __nv_bfloat16* p, size_t i) {
  return __bfloat162float(p[i]);
}

// Window slot a = r mod w sits at position n - w + a and sees keys j <= n - w + a.
__device__ __forceinline__ bool visible(const Shape& s, int r, int j) {
  return !s.causal || j <= s.n - s.w + (r % s.w);
}

}  // namespace
}  // namespace grkv
