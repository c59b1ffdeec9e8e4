// Tensor-core (tcgen05 / TMEM) backward path: interface to the rest of the library.
#pragma once
#include "sa_common.cuh"

namespace sa {

// True when the bf16 tensor-core kernels can run this backward problem.
bool tc_backward_supported(const BwdArgs& a, int dtype);
// Workspace of launch_bwd_tc (0: it does not serve this head dimension).
size_t tc_backward_ws_bytes(int B, int Hq, int Hkv, int n, int d, int w);
// dq, dk, dv of every branch, and the partial sums of the gate gradients (a.partials, a.chunks).
cudaError_t launch_bwd_tc(BwdArgs& a, cudaStream_t st);

}  // namespace sa
