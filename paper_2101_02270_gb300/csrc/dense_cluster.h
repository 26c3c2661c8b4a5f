// Dense block of a small batch: factorisation and substitutions of each instance
// by a cluster of CTAs that holds its whole block in shared memory
// (dense_cluster.cu).
#pragma once
#include <cuda_runtime.h>

#include "device.h"
#include "recorder.h"

namespace nrpf {

// Clusters that the device can hold at once, 0 where the plan's block does not fit
// one (width: bytes of a value).
int dense_cluster_resident(const DevPlan& P, size_t width);

// Whether a batch of B instances of the plan is small enough for the clusters to pay.
bool dense_cluster_pays(const DevPlan& P, int B, size_t width);

// S.x rows s .. s+nde-1 <- the dense block's share of the solution, between the
// sparse forward and backward levels.  S.lu is left as the Schur tasks wrote it.
template <typename T>
void launch_dense_cluster(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                          Recorder* rec = nullptr);

}  // namespace nrpf
