// history_fx.h -- FP64 contractions on the tensor cores (history_fx.cu).
#pragma once

#include "fx_common.cuh"
#include "kbe_internal.h"

namespace kbe {

// Whether an FP64 slice is better there than on the FP64 pipe: from (n + 1)^2 M^3 =
// 5e6 on, and never for the rows that kbe_run_steps takes in its cooperative
// kernel.  Below that the FP64 pipe is as fast or faster, above it falls behind
// with the cube of M (slices on the FP64 pipe against the tensor cores, us: M = 5,
// n = 163 95 / 87; M = 8, n = 64 89 / 66, n = 1023 7080 / 905; M = 12, n = 29 63 / 91,
// n = 50 107 / 130; M = 16, n = 16 55 / 84, n = 30 102 / 89; M = 24, n = 10 68 / 100,
// n = 20 159 / 138; M = 32, n = 16 249 / 140).
__host__ __device__ inline bool fx_takes(int M, int n) {
  const double N = n + 1.0, m = M;
  return N * m * m > kRunMaxRow && N * N * m * m * m >= 5e6;
}
// The same for KBE_DF64 slices against their own kernel (history_df.cu): from
// 8e6 on (us, double-float / tensor cores: M = 8, n = 100 111 / 77; M = 16, n = 30 74 /
// 89, n = 511 4620 / 1350; M = 24, n = 20 114 / 138; M = 32, n = 16 168 / 140).
__host__ __device__ inline bool fx_takes_df(int M, int n) {
  const double N = n + 1.0, m = M;
  return N * m * m > kRunMaxRow && N * N * m * m * m >= 8e6;
}
// Workspace of one system's contractions up to row n_max - 1.
size_t fx_workspace_bytes(int M, int n_max);
cudaError_t fx_prepare();  // one-time kernel attributes of the current device
// The FP64 history slice (the sums of launch_history_f64 over all stored rows).
cudaError_t launch_history_fx(const HistoryArgs& a, void* work, size_t work_bytes, cudaStream_t s, int* launches);
// The slices of the systems in a device table (all with part_rows(M) == NA; quad:
// all M multiples of 4), bases and totals set, on one CTA per SM.
cudaError_t launch_fx_table(int NA, bool quad, const fx::Sys* table, const fx::Head* head, cudaStream_t s, int* launches);
// The cotangents of the Sigma row in the slice's adjoint (a.dSl, a.dSg).
cudaError_t launch_adjoint_fx(const AdjHistArgs& a, void* work, size_t work_bytes, int* status, cudaStream_t s,
                              int* launches);

}  // namespace kbe
