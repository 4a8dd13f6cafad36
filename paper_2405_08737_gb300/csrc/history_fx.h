// history_fx.h -- FP64 contractions on the tensor cores (history_fx.cu).
#pragma once

#include "fx_common.cuh"
#include "kbe_internal.h"

namespace kbe {

// Whether an FP64 slice goes there instead of the FP64 pipe: from (n + 1)^2 M^3 =
// 5e6 on, and never for the rows that kbe_run_steps takes in its cooperative
// kernel.  Above the line the tensor cores are faster at every M (FP64 pipe / tensor cores,
// us: M = 3, n = 456 127 / 70; M = 5, n = 200 119 / 64; M = 8, n = 98 108 / 64, n = 1023 7050 / 835;
// M = 9, n = 85 156 / 82; M = 13, n = 47 135 / 92; M = 16, n = 34 129 / 82; M = 24, n = 19 156 / 84;
// M = 33, n = 11 163 / 86; M = 64, n = 4 222 / 84).  They cross below it, between 1.5e6
// and 3e6 (M = 8, n = 65 92 / 56; M = 12, n = 30 62 / 69, n = 40 88 / 79; M = 16, n = 17 56 / 69,
// n = 24 78 / 70; M = 24, n = 10 68 / 72): the line was measured with an earlier form
// of these kernels, and rows in between pay up to two thirds more than they had to.
// The adjoint's line is the slice's (n at 5e6: M = 5 170 / 92, M = 8 131 / 82, M = 16 184 /
// 117, M = 33 277 / 163; crossing near 2e6: M = 12, n = 30 102 / 104, M = 24, n = 10 111 / 120).
__host__ __device__ inline bool fx_takes(int M, int n) {
  const double N = n + 1.0, m = M;
  return N * m * m > kRunMaxRow && N * N * m * m * m >= 5e6;
}
// The same for KBE_DF64 slices against their own kernel (history_df.cu): from
// 8e6 on (us, double-float / tensor cores: M = 5, n = 260 152 / 73; M = 8, n = 130 132 / 68;
// M = 13, n = 60 115 / 99; M = 16, n = 50 127 / 84; M = 33, n = 18 218 / 122).  They cross between
// 2e6 and 6e6 (M = 8, n = 65 72 / 56; M = 9, n = 60 68 / 78, n = 85 99 / 82; M = 13, n = 47 81 / 92;
// M = 16, n = 30 68 / 76, n = 34 90 / 82; M = 24, n = 14 72 / 80, n = 19 99 / 84).
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
