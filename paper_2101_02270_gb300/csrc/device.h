// Device-side plan and per-solve state shared by the kernels and the C ABI.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace nrpf {

// Instances are interleaved in tiles of kTile (Sec. 3.1, Fig. 1d: element-major,
// batch contiguous): element e of instance b lives at
//   ((b / kTile) * E + e) * kTile + (b % kTile)
// for an array holding E elements per instance.  A warp of 32 lanes covers one
// tile, so every per-element access of a warp is one contiguous 256-byte
// (float64) or 128-byte (float32) segment.
constexpr int kTile = 32;

// Layout of the dense block inside a tile's LU array.  FP64: element (r, c)
// of the ndp x ndp block at (c * ndp + r) * 32 + lane.  FP32: four
// consecutive rows of a column stay together per lane,
// (c * ndp + (r & ~3)) * 32 + lane * 4 + (r & 3), so a lane reads rows
// r..r+3 (r % 4 == 0) as one 16-byte vector and a warp's access is still one
// contiguous 512-byte segment.  ndp is a multiple of the panel width (>= 4).
template <typename T>
struct DenseGroup {
  static constexpr int G = sizeof(T) == 4 ? 4 : 1;
};

struct DevUpd {
  int32_t ukj, lsrc, llen, dst_off;
};

// Read-only plan arrays on the device (copied once by pf_plan_create).
struct DevPlan {
  int n, m, s, nd, ndp, kb, mp;  // mp = s + ndp (rhs length incl. padding)
  // columns of the dense block that are worked on, ndp its leading dimension: nd
  // rounded up to the 16 of the FP32 kernels' steps where ndp is rounded further
  // (their outer panels), ndp otherwise
  int nde;
  int sms;  // of the plan's device
  int clusters;  // of dense_cluster.cu that the device holds at once, 0: the block does not fit one
  int dim;  // 1: instance-major dense block (FP32 LU; see dense_im.h), 0: interleaved
  int64_t NS, NLU;
  int nnzY;
  const int32_t* rowptr;   // [n+1]
  const int32_t* colidx;   // [nnzY]
  const double* yre;       // [nnzY]
  const double* yim;       // [nnzY]
  const int32_t* ydiag;    // [n] index of the diagonal entry in row i
  const int8_t* bus_type;  // [n]
  const int32_t* jmap;     // [nnzY*4]
  const int32_t* rhs_p;    // [n] A row of the P equation (-1 for slack)
  const int32_t* rhs_q;    // [n] A row of the Q equation (-1 unless PQ)
  const int32_t* one_pos;  // [ndp-nd]
  int n_one;
  // sparse refactor
  const int32_t* lu_cols;      // columns grouped by level
  const int32_t* col_upd_ptr;  // [m+1]
  const DevUpd* upd;
  const int32_t* dst;
  const int32_t* dp;           // [m] diagonal position (-1 for dense columns)
  const int64_t* ce;           // [m] segment end
  // the same by entries (plan.h); n_fac_lvl = 0: by columns
  const int32_t* fac_lvl_ptr;
  const int32_t* fac_task;
  const int2* fac_op;
  int n_fac_lvl, n_fac_task;
  // Schur complement of the sparse columns into the dense block
  const int4* schur_task;     // {dense column, 32-row chunk, first entry, end}
  const int32_t* schur_ent;   // (L(i, k) position << 5) | row in chunk
  const int32_t* schur_u;     // U(k, j) position of the entry
  const uint32_t* schur_jmask; // rows of the chunk holding a Jacobian entry
  int n_schur;
  // the whole linear solve of a small plan (plan.h; n_sm_lvl = 0: not small)
  const int32_t* sm_lvl_ptr;
  const int32_t* sm_task;
  const int2* sm_op;
  int n_sm_lvl, n_sm_task, n_sm_op;
  // FS/BS
  const int32_t* fw_rows; const int32_t* fw_ptr; const int32_t* fw_pos; const int32_t* fw_col;
  const int32_t* bw_rows; const int32_t* bw_ptr; const int32_t* bw_pos; const int32_t* bw_col;
  const int32_t* unk_pos;  // [m]
  // level boundaries of the schedules (device copies, for fused kernels)
  const int32_t* lu_lvl_ptr; int n_lu_lvl;
  const int32_t* fw_lvl_ptr; int n_fw_lvl;
  const int32_t* bw_lvl_ptr; int n_bw_lvl;
};

// Per-solve workspace (capacity Bp instances, a multiple of kTile).
// Device-resident control of the Newton loop, so that one iteration can run
// unchanged from a graph: every kernel of an iteration reads its gate and the
// iteration number here.
constexpr int kLoopSlots = 64;  // loop graphs kept per workspace, one per padded batch size and set of kernels
struct SolveCtl {
  int32_t prev;     // instances active after the previous check: gate of the
                    // LU preparation and mismatch (nonzero before the first)
  int32_t cur;      // instances active after this iteration's check: gate of
                    // factorisation, FS/BS and update
  int32_t it;       // Newton iteration of the check
  int32_t maxit;
  double tol;
  long long graph_iters[kLoopSlots];  // loop bodies run by each loop graph since the last reset
};

struct DevState {
  int Bp;
  double* vm;    // [n] magnitudes
  double* va;    // [n] angles
  double* ve;    // [n] real part
  double* vf;    // [n] imaginary part
  double* vinv;  // [n] 1/|V|
  double* psp;   // [n] specified P
  double* qsp;   // [n] specified Q
  void* x;       // [mp] right-hand side / solution (LU precision)
  void* lu;      // [NLU] LU values (LU precision)
  void* inv;     // [kb] inverse pivots of the current dense diagonal block
  void* dinv;    // [s] inverse pivots of the sparse columns (LU precision), or null
  void* limb;    // operands of the FP64 trailing update in fixed point (kernels.cu), or null
  unsigned long long* norm;  // [Bp] max |F| as float64 bits
  int32_t* iters;   // [Bp]
  int32_t* status;  // [Bp]
  int32_t* active;  // [Bp] 0: finished; kActiveFar / kActiveNear (kernels.h)
  int32_t* bad;     // [Bp] non-finite step detected
  SolveCtl* ctl;  // Newton loop control (one per workspace)
  const double2* yv;  // [nnzY] per-instance Ybus values (re, im), or null: the plan's shared values
  const void* im_maps;  // host pointer to the workspace's DenseImMaps (instance-major plans), never read on the device
};

// offset of LU position p of lane `lane` within its tile's array (positions
// >= NS are in the dense block: interleaved, grouped by four rows in FP32, or
// instance-major when P.dim is set, lane l's block then at NS * 32 + l * ndp^2)
template <typename T>
__device__ __forceinline__ size_t lu_off(const DevPlan& P, int64_t p, int lane) {
  constexpr int G = DenseGroup<T>::G;
  const int64_t NS = P.NS;
  if (p < NS) return (size_t)p * kTile + lane;
  const int64_t q = p - NS;
  if (P.dim) return (size_t)NS * kTile + (size_t)lane * (size_t)P.ndp * (size_t)P.ndp + (size_t)q;
  if (G == 1) return (size_t)p * kTile + lane;
  return (size_t)NS * kTile + (size_t)(q & ~(int64_t)(G - 1)) * kTile + (size_t)lane * G + (size_t)(q & (G - 1));
}

}  // namespace nrpf
