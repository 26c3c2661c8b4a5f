// Dense block of a small batch: factorisation and substitutions of each instance
// by a cluster of CTAs that holds its whole block in shared memory
// (dense_cluster.cu).
#pragma once
#include <cuda_runtime.h>

#include "device.h"
#include "recorder.h"

namespace nrpf {

// Whether the plan's block fits and the batch is small enough for it to pay.
bool dense_cluster_fits(const DevPlan& P, const DevState& S, size_t width);

// S.x rows s .. s+nde-1 <- the dense block's share of the solution, between the
// sparse forward and backward levels.  S.lu is left as the Schur tasks wrote it.
template <typename T>
void launch_dense_cluster(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                          Recorder* rec = nullptr);

}  // namespace nrpf
