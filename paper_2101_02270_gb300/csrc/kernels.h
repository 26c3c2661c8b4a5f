// Launchers of the batched Newton-Raphson kernels (kernels.cu).
#pragma once
#include <cstddef>
#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "device.h"
#include "recorder.h"

#define NRPF_CONVERGED_CODE 0
#define NRPF_MAXIT_CODE 1
#define NRPF_FAILED_CODE 2

// S.active of an instance that is still iterating: far from its solution, or
// near it (max |F| of at most kNearMismatch).  The instance-major dense block
// is updated on the tensor cores while an instance is far (dense_im.cu), and by
// FP32 FMAs in pivot order when it is near.  The tensor-core form is the faster
// one (9,000 buses x 1,000, per refactorisation: 36 against 105 ms) and the more
// exact one; the line is there because the step from a mismatch of 1e-3 p.u. or
// less is, by quadratic convergence, the last or the last but one, and an FP32
// factor's own error is what it leaves in the voltages (3.5e-9 on the 9,000-bus
// grid, at a mismatch of 2e-9).  Taking that step with the same roundings as
// ever keeps converged voltages where they were, to 9e-10 on that grid and 1e-10
// or less on smaller or more lightly loaded ones; with the tensor cores in every
// step they move by 3.2e-9 (to 3.2e-10 from the exact root).
constexpr int kActiveFar = 1, kActiveNear = 2;
constexpr double kNearMismatch = 1e-3;

namespace nrpf {

void launch_load(const DevPlan& P, const DevState& S, int B, const double* sbus, const double* v0,
                 cudaStream_t st, Recorder* rec = nullptr);
void launch_store(const DevPlan& P, const DevState& S, int B, double* v_out, int32_t* iters,
                  uint8_t* status, cudaStream_t st, Recorder* rec = nullptr);
// gates of the Newton loop (addresses inside the device control block)
inline const int32_t* ctl_prev(const DevState& S) {
  return reinterpret_cast<const int32_t*>(reinterpret_cast<const char*>(S.ctl) + offsetof(SolveCtl, prev));
}
inline const int32_t* ctl_cur(const DevState& S) {
  return reinterpret_cast<const int32_t*>(reinterpret_cast<const char*>(S.ctl) + offsetof(SolveCtl, cur));
}

// Per-instance Ybus values [B, nnzY] complex into S.yv (interleaved).
void launch_load_y(const DevPlan& P, const DevState& S, int B, const double* y, cudaStream_t st,
                   Recorder* rec = nullptr);

// Per-instance Ybus values of outage cases into S.yv: the plan's base values
// minus the stamps of each instance's outaged branches (outages [B, k]).
void launch_outage_y(const DevPlan& P, const DevState& S, int B, const int32_t* outages, int k, const int4* bpos,
                     const double* bval, int nbr, cudaStream_t st, Recorder* rec = nullptr);

// Reset the loop control (prev = 1, cur = 0, it = 0) with the tolerance and
// iteration limit of this solve.
void launch_ctl_init(const DevState& S, int maxit, double tol, cudaStream_t st, Recorder* rec = nullptr);
// Convergence test of iteration ctl->it: counts the instances still active
// into ctl->cur.
void launch_check(const DevState& S, cudaStream_t st, Recorder* rec = nullptr);
// End of one iteration: prev = cur, cur = 0, it += 1; with a graph handle
// (graph != 0), also sets the loop's condition to (cur > 0 && it < maxit).
// graph: 0, or 1 + the loop graph's slot in SolveCtl::graph_iters
void launch_iter_tail(const DevState& S, cudaGraphConditionalHandle cond, int graph, cudaStream_t st,
                      Recorder* rec = nullptr);

template <typename T>
void launch_mismatch(const DevPlan& P, const DevState& S, int jac, const int32_t* gate, cudaStream_t st,
                     Recorder* rec = nullptr);
// What of the LU workspace is zeroed before a refactorisation: everything, the
// sparse segments (the Schur tasks then write every position of the dense
// block), or what the small plans' kernel reads (the sparse segments and the
// dense block's columns without its padding).  Except for the last the identity
// padding of the dense block is set too.
enum class LuPrep { kWhole, kSparse, kColumns };
template <typename T>
void launch_prepare_lu(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                       Recorder* rec = nullptr, LuPrep prep = LuPrep::kWhole);
// Tiles up to which an FP64 refactorisation goes by entries (FP32: any number)
constexpr int kEntryTiles64 = 152;

// Bytes of S.limb, the fixed-point operands of the FP64 trailing update, for a
// workspace of Bp instances.
size_t dense_limb_bytes(const DevPlan& P, int Bp);
// dense = false: the sparse part and the Schur tasks only.
template <typename T>
void launch_factor(const DevPlan& P, const DevState& S, const std::vector<int32_t>& lvl_ptr,
                   const int32_t* gate, cudaStream_t st, Recorder* rec = nullptr, bool dense = true);
// dense = false: the dense block is factorised and solved between the levels, by
// a cluster of CTAs per instance (dense_cluster.h).
template <typename T>
void launch_solve(const DevPlan& P, const DevState& S, const std::vector<int32_t>& fw_lvl,
                  const std::vector<int32_t>& bw_lvl, const int32_t* gate, cudaStream_t st,
                  Recorder* rec = nullptr, bool dense = true);
template <typename T>
void launch_update(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                   Recorder* rec = nullptr);
template <typename T>
void launch_rhs_in(const DevPlan& P, const DevState& S, int B, const double* rhs, cudaStream_t st);
template <typename T>
void launch_rhs_out(const DevPlan& P, const DevState& S, int B, double* dx, cudaStream_t st);
template <typename T>
void launch_f_out(const DevPlan& P, const DevState& S, int B, double* F, double* norm, cudaStream_t st);
template <typename T>
void launch_lu_out(const DevPlan& P, const DevState& S, int B, const int64_t* map, int64_t nnz, double* out,
                   cudaStream_t st);

}  // namespace nrpf
