// Arguments of the on-chip key step (grkv_key_cluster.cu), filled by the key
// step's launcher (grkv_key.cu).
#pragma once

#include "grkv_internal.cuh"

namespace grkv {

struct KeyClusterArgs {
  int n, w, m, B, causal, iters;
  float scale, lambda_k, tol;
  const void* q;          // [U][m][d]
  const float* y;         // [U][m][d]
  const int32_t* idx;     // [U][B]
  const uint8_t* fixed;   // [U][B] the value step's fixed set
  const void* v_out;      // [U][B][d] merged values V*
  void* k_out;            // [U][B][d] K0 on entry, K* on exit
  float* Kt;              // [U][B][d] K* in fp32 for the alternation, or null
  int* status;
};

// Sets *done when it launched; otherwise the shape or the device is not
// served and nothing was enqueued.
cudaError_t launch_key_cluster(const Shape& s, const KeyClusterArgs& a, cudaStream_t st, bool* done);

}  // namespace grkv
