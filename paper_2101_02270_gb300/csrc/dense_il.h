// LU of the interleaved FP32 dense block by outer panels of 64 columns
// (dense_il.cu).
#pragma once
#include <cuda_runtime.h>

#include "device.h"
#include "recorder.h"

namespace nrpf {

// Factorises columns 0 .. P.nde-1 (a multiple of 16) of every active tile's block.
void launch_dense_il_factor(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                            Recorder* rec = nullptr);

}  // namespace nrpf
