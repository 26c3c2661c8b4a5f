// The linear solve of a Newton step for small plans: refactorisation and both
// substitutions of several instances in one CTA's shared memory (small_solve.cu).
#pragma once
#include <cstddef>

#include <cuda_runtime.h>

#include "device.h"
#include "plan.h"
#include "recorder.h"

namespace nrpf {

// Whether the plan has the whole-solve schedule and some batch of it, in a
// precision of `width` bytes, would take this kernel.
bool small_solve_fits(const HostPlan& h, size_t width);

// Instances per CTA for a batch padded to Bp, or 0: the level kernels serve it.
int small_solve_instances(const DevPlan& P, int Bp, size_t width);

// S.x <- J^-1 S.x for every active tile, from the Jacobian values in S.lu (the
// whole LU array zeroed before they were filled in); S.lu is left as it is.
template <typename T>
void launch_small_solve(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                        Recorder* rec = nullptr);

}  // namespace nrpf
