// The mixture denoiser's tensor-core form (k_gmm_tc.cu), as k_gmm.cu uses it.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace pa {

// Where its scratch lies in the handle's workspace: partial dot products of
// every CTA, responsibilities, the rows' scalars.
struct GmmTcLayout {
  size_t part, resp, rcoef, total;  // byte offsets, total bytes
  int slots;                        // partial sums kept per row: one per CTA of its block
};
GmmTcLayout gmm_tc_layout(int K, int64_t D, int max_rows);

// The shared memory of its kernels fits the current device (and is granted).
cudaError_t gmm_tc_setup(int K, bool* ok);

struct GmmTcArgs {
  const float* X;             // [max_rows][D], rows < *n_rows
  const float* mu;            // [K][D]
  const float* coef;          // [3][T]: sqrt(a), 1 / (2 v), sqrt(1 - a) / v
  const float* mnorm;         // [K]
  const int32_t* miss_bt;     // [.][2]
  const int32_t* n_rows;      // device
  float* eps;                 // [.][D]
  char* ws;                   // scratch of gmm_tc_layout
  int32_t* status;
  int K, T, max_rows;
  int64_t D;
};
// Three kernels on st: dot products, responsibilities, output.
cudaError_t gmm_tc_launch(const GmmTcArgs& a, cudaStream_t st);
constexpr int kGmmTcLaunches = 3;

}  // namespace pa
