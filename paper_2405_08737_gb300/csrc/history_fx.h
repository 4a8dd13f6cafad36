// history_fx.h -- FP64 contractions on the tensor cores (history_fx.cu).
#pragma once

#include "fx_common.cuh"
#include "kbe_internal.h"

namespace kbe {

// Workspace of one system's contractions up to row n_max - 1.
size_t fx_workspace_bytes(int M, int n_max);
cudaError_t fx_prepare();  // one-time kernel attributes of the current device
// The FP64 history slice (the sums of launch_history_f64 over all stored rows).
cudaError_t launch_history_fx(const HistoryArgs& a, void* work, size_t work_bytes, cudaStream_t s, int* launches);
// The cotangents of the Sigma row in the slice's adjoint (a.dSl, a.dSg).
cudaError_t launch_adjoint_fx(const AdjHistArgs& a, void* work, size_t work_bytes, int* status, cudaStream_t s,
                              int* launches);

}  // namespace kbe
