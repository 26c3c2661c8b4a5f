// Batched Newton-Raphson kernels (sm_103a).  Every kernel works on tiles of
// kTile = 32 interleaved instances: lane = instance within the tile, so all
// plan indices are warp-uniform (broadcast loads) and all value accesses are
// contiguous across the warp.
#include <algorithm>
#include <cfloat>
#include <cstdint>
#include <vector>

#include "dense_cluster.h"
#include "dense_il.h"
#include "dense_im.h"
#include "device.h"
#include "kernels.h"

namespace nrpf {

namespace {

__device__ __forceinline__ size_t sidx(int tile, int64_t E, int64_t e, int lane) {
  return ((size_t)tile * (size_t)E + (size_t)e) * kTile + lane;
}

__device__ __forceinline__ bool tile_active(const DevState& S, int tile, int lane) {
  return __any_sync(0xffffffffu, S.active[tile * kTile + lane] != 0);
}

template <typename T>
__device__ __forceinline__ size_t dense_off(int r, int c, int ld, int lane) {
  constexpr int G = DenseGroup<T>::G;
  return ((size_t)c * ld + (r & ~(G - 1))) * kTile + (size_t)lane * G + (r & (G - 1));
}

// ---------------------------------------------------------------------------
// Input / output transposes: user [B, n] complex128 <-> interleaved tiles
// (the paper's "transpose to batch" step on the device, Sec. 3.2).
// Block (32, 8): a 32-bus x 32-instance tile through shared memory.
// ---------------------------------------------------------------------------
__global__ void k_load(DevPlan P, DevState S, int B, const double2* __restrict__ sbus,
                       const double2* __restrict__ v0) {
  __shared__ double2 ss[32][33];
  __shared__ double2 sv[32][33];
  const int tile = blockIdx.y;
  const int i0 = blockIdx.x * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int r = ty; r < 32; r += 8) {
    int b = tile * kTile + r;
    int i = i0 + tx;
    double2 s = make_double2(0.0, 0.0), v = make_double2(1.0, 0.0);
    if (b < B && i < P.n) {
      s = sbus[(size_t)b * P.n + i];
      v = v0[(size_t)b * P.n + i];
    }
    ss[r][tx] = s;
    sv[r][tx] = v;
  }
  __syncthreads();
  for (int c = ty; c < 32; c += 8) {
    int i = i0 + c;
    if (i >= P.n) continue;
    double2 s = ss[tx][c], v = sv[tx][c];
    size_t o = sidx(tile, P.n, i, tx);
    // a start on the positive real axis (flat start) needs no FP64 sqrt or
    // atan2: |V| is the real part itself and the angle 0
    const bool real = v.y == 0.0 && v.x > 0.0;
    double vm = real ? v.x : sqrt(v.x * v.x + v.y * v.y);
    S.psp[o] = s.x;
    S.qsp[o] = s.y;
    S.vm[o] = vm;
    S.va[o] = real ? 0.0 : atan2(v.y, v.x);
    S.ve[o] = v.x;
    S.vf[o] = v.y;
    S.vinv[o] = 1.0 / vm;
  }
  if (blockIdx.x == 0 && ty == 0) {
    int b = tile * kTile + tx;
    S.iters[b] = 0;
    S.status[b] = NRPF_MAXIT_CODE;
    S.active[b] = b < B ? 1 : 0;
    S.bad[b] = 0;
    S.norm[b] = 0ull;
  }
}

__global__ void k_store(DevPlan P, DevState S, int B, double2* __restrict__ v_out,
                        int32_t* __restrict__ iters, uint8_t* __restrict__ status) {
  __shared__ double2 sv[32][33];
  const int tile = blockIdx.y;
  const int i0 = blockIdx.x * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int c = ty; c < 32; c += 8) {
    int i = i0 + c;
    if (i >= P.n) continue;
    size_t o = sidx(tile, P.n, i, tx);
    sv[tx][c] = make_double2(S.ve[o], S.vf[o]);
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    int b = tile * kTile + r;
    int i = i0 + tx;
    if (b < B && i < P.n) v_out[(size_t)b * P.n + i] = sv[r][tx];
  }
  if (blockIdx.x == 0 && ty == 0) {
    int b = tile * kTile + tx;
    if (b < B) {
      iters[b] = S.iters[b];
      status[b] = (uint8_t)S.status[b];
    }
  }
}

// ---------------------------------------------------------------------------
// Nodal power mismatch (Eq. 1, Alg. 1) fused with the Jacobian refill straight
// into the permuted LU workspace (Sec. 3.1.2, static lookup jmap).
// Rectangular voltages e + jf avoid a sine/cosine per admittance entry:
//   I_i = sum_k Y_ik V_k,  S_i = V_i conj(I_i)
//   W_ik = V_i conj(Y_ik V_k)          (k != i)
//   dP_i/dth_k = Im W_ik, dQ_i/dth_k = -Re W_ik,
//   dP_i/d|V_k| = Re W_ik / |V_k|, dQ_i/d|V_k| = Im W_ik / |V_k|
//   dP_i/dth_i = -Q_i - B_ii |V_i|^2,  dQ_i/dth_i = P_i - G_ii |V_i|^2
//   dP_i/d|V_i| = P_i/|V_i| + G_ii |V_i|, dQ_i/d|V_i| = Q_i/|V_i| - B_ii |V_i|
// Block: 32 lanes x kWarps warps; each warp walks `per` buses, eight, which
// amortises the block's reduction, or fewer while that fills the GPU: a bus is a
// chain of index, value and FP64 arithmetic, 4 us of it, so that eight in a row
// took 33 us on 30 buses and 66 us on one tile of 2,000 (now 11 and 18 us).
// The right-hand side receives -F at the permuted row of each equation.
// ---------------------------------------------------------------------------
constexpr int kMWarps = 8;

template <typename T>
__global__ void __launch_bounds__(32 * kMWarps) k_mismatch_jac(DevPlan P, DevState S, int jac, int per,
                                                               const int32_t* __restrict__ gate) {
  __shared__ double red[kMWarps][32];
  const int lane = threadIdx.x, warp = threadIdx.y;
  const int tile = blockIdx.y;
  if (gate && *gate == 0) return;
  T* __restrict__ LU = reinterpret_cast<T*>(S.lu) + (size_t)tile * P.NLU * kTile;
  T* __restrict__ X = reinterpret_cast<T*>(S.x) + (size_t)tile * P.mp * kTile;
  const double* __restrict__ ve = S.ve + (size_t)tile * P.n * kTile;
  const double* __restrict__ vf = S.vf + (size_t)tile * P.n * kTile;
  const double* __restrict__ vinv = S.vinv + (size_t)tile * P.n * kTile;
  // per-instance admittances (interleaved like every per-instance array) or
  // the plan's shared ones; the choice is uniform over the launch
  const double2* __restrict__ Yv = S.yv ? S.yv + (size_t)tile * P.nnzY * kTile + lane : nullptr;
  auto yval = [&](int d, double& G, double& Bv) {
    if (Yv) {
      const double2 y = Yv[(size_t)d * kTile];
      G = y.x;
      Bv = y.y;
    } else {
      G = P.yre[d];
      Bv = P.yim[d];
    }
  };
  double nrm = 0.0;
  const int ibeg = (blockIdx.x * kMWarps + warp) * per;
  for (int ii = 0; ii < per; ++ii) {
    const int i = ibeg + ii;
    if (i >= P.n) break;
    const int bt = P.bus_type[i];
    if (bt == 3) continue;
    const double ei = ve[i * kTile + lane], fi = vf[i * kTile + lane];
    double Ir = 0.0, Ii = 0.0;
    const int d0 = P.rowptr[i], d1 = P.rowptr[i + 1];
    for (int d = d0; d < d1; ++d) {
      const int k = P.colidx[d];
      double G, Bv;
      yval(d, G, Bv);
      const double ek = ve[k * kTile + lane], fk = vf[k * kTile + lane];
      const double yr = G * ek - Bv * fk;
      const double yi = G * fk + Bv * ek;
      Ir += yr;
      Ii += yi;
      if (jac && k != i) {
        const int4 jm = reinterpret_cast<const int4*>(P.jmap)[d];
        if (jm.x >= 0) {
          // off-diagonal Jacobian entries, formed in the LU precision (they
          // are stored in it; the mismatch above stays FP64)
          const T Wr = (T)ei * (T)yr + (T)fi * (T)yi;
          const T Wi = (T)fi * (T)yr - (T)ei * (T)yi;
          const T ik = (T)vinv[k * kTile + lane];
          LU[lu_off<T>(P, jm.x, lane)] = Wi;
          if (jm.y >= 0) LU[lu_off<T>(P, jm.y, lane)] = Wr * ik;
          if (jm.z >= 0) LU[lu_off<T>(P, jm.z, lane)] = -Wr;
          if (jm.w >= 0) LU[lu_off<T>(P, jm.w, lane)] = Wi * ik;
        }
      }
    }
    const double Pc = ei * Ir + fi * Ii;
    const double Qc = fi * Ir - ei * Ii;
    const size_t o = (size_t)i * kTile + lane;
    const size_t so = (size_t)tile * P.n * kTile + o;
    const double dP = Pc - S.psp[so];
    double a = fabs(dP);
    X[(size_t)P.rhs_p[i] * kTile + lane] = (T)(-dP);
    if (bt == 1) {
      const double dQ = Qc - S.qsp[so];
      X[(size_t)P.rhs_q[i] * kTile + lane] = (T)(-dQ);
      const double q = fabs(dQ);
      a = (q > a || q != q) ? q : a;
    }
    nrm = (a > nrm || a != a) ? a : nrm;
    if (jac) {
      const int dd = P.ydiag[i];
      const int4 jm = reinterpret_cast<const int4*>(P.jmap)[dd];
      double G, Bv;
      yval(dd, G, Bv);
      const double vm2 = ei * ei + fi * fi;
      const double ivm = vinv[o];
      const double vm = vm2 * ivm;
      LU[lu_off<T>(P, jm.x, lane)] = (T)(-Qc - Bv * vm2);
      if (jm.y >= 0) LU[lu_off<T>(P, jm.y, lane)] = (T)(Pc * ivm + G * vm);
      if (jm.z >= 0) LU[lu_off<T>(P, jm.z, lane)] = (T)(Pc - G * vm2);
      if (jm.w >= 0) LU[lu_off<T>(P, jm.w, lane)] = (T)(Qc * ivm - Bv * vm);
    }
  }
  // NaN -> +inf so that the unsigned-integer max keeps it
  if (!(nrm <= DBL_MAX)) nrm = __longlong_as_double(0x7ff0000000000000ll);
  red[warp][lane] = nrm;
  __syncthreads();
  if (warp == 0) {
    double r = red[0][lane];
    for (int w = 1; w < kMWarps; ++w) r = fmax(r, red[w][lane]);
    atomicMax(&S.norm[tile * kTile + lane], (unsigned long long)__double_as_longlong(r));
  }
}

// Per-instance Ybus values: user [B, nnzY] complex -> interleaved tiles,
// through a 32-entry x 32-instance tile in shared memory (block (32, 8)).
__global__ void k_load_y(int nnzY, int B, const double2* __restrict__ y, double2* __restrict__ yv) {
  __shared__ double2 t[32][33];
  const int d0 = blockIdx.x * 32, tile = blockIdx.y;
  for (int r = threadIdx.y; r < 32; r += 8) {  // r = instance within the tile
    const int b = tile * kTile + r, d = d0 + threadIdx.x;
    t[r][threadIdx.x] = (b < B && d < nnzY) ? y[(size_t)b * nnzY + d] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int c = threadIdx.y; c < 32; c += 8) {  // c = entry within the block
    const int d = d0 + c;
    if (d < nnzY) yv[((size_t)tile * nnzY + d) * kTile + threadIdx.x] = t[threadIdx.x][c];
  }
}

// Outage cases built on the device: every instance starts from the plan's
// base admittances (interleaved layout), then loses the stamps of its outaged
// branches (repeated indices of one instance count once).
__global__ void k_base_y(DevPlan P, double2* __restrict__ yv, int tiles) {
  const int lane = threadIdx.x;
  const int64_t q = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;  // (tile, entry)
  if (q >= (int64_t)tiles * P.nnzY) return;
  const int d = (int)(q % P.nnzY);
  yv[q * kTile + lane] = make_double2(P.yre[d], P.yim[d]);
}

__global__ void k_outage_y(int nnzY, int B, int k, const int32_t* __restrict__ outages,
                           const int4* __restrict__ bpos, const double* __restrict__ bval, int nbr,
                           double2* __restrict__ yv) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  double2* y = yv + (size_t)(b / kTile) * nnzY * kTile + (b % kTile);
  for (int a = 0; a < k; ++a) {
    const int e = outages[(size_t)b * k + a];
    if (e < 0 || e >= nbr) continue;
    bool seen = false;
    for (int c = 0; c < a; ++c) seen = seen || outages[(size_t)b * k + c] == e;
    if (seen) continue;
    const int4 ps = bpos[e];
    const double gs = bval[3 * e], bs = bval[3 * e + 1], bh = bval[3 * e + 2];
    y[(size_t)ps.x * kTile].x -= gs;
    y[(size_t)ps.x * kTile].y -= bs + bh;
    y[(size_t)ps.y * kTile].x -= gs;
    y[(size_t)ps.y * kTile].y -= bs + bh;
    y[(size_t)ps.z * kTile].x += gs;
    y[(size_t)ps.z * kTile].y += bs;
    y[(size_t)ps.w * kTile].x += gs;
    y[(size_t)ps.w * kTile].y += bs;
  }
}

// Convergence test and per-instance bookkeeping, one thread per instance.
// it = number of updates performed so far.
__global__ void k_check(DevState S, int Bp) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= Bp) return;
  const int it = S.ctl->it, maxit = S.ctl->maxit;
  const double tol = S.ctl->tol;
  int32_t* counter = &S.ctl->cur;
  const double nrm = __longlong_as_double((long long)S.norm[b]);
  S.norm[b] = 0ull;
  if (!S.active[b]) return;
  int keep = 0;
  if (S.bad[b]) {  // the previous step was not finite: it does not count
    S.status[b] = NRPF_FAILED_CODE;
    S.iters[b] = it - 1;
  } else if (!(nrm <= DBL_MAX)) {
    S.status[b] = NRPF_FAILED_CODE;
    S.iters[b] = it;
  } else if (nrm < tol) {
    S.status[b] = NRPF_CONVERGED_CODE;
    S.iters[b] = it;
  } else if (it >= maxit) {
    S.status[b] = NRPF_MAXIT_CODE;
    S.iters[b] = it;
  } else {
    keep = 1;
    S.iters[b] = it + 1;
  }
  S.active[b] = !keep ? 0 : nrm > kNearMismatch ? kActiveFar : kActiveNear;
  const unsigned mask = __ballot_sync(__activemask(), keep);
  if (keep && (threadIdx.x & 31) == __ffs(mask) - 1) atomicAdd(counter, __popc(mask));
}

__global__ void k_ctl_init(SolveCtl* c, int maxit, double tol) {
  c->prev = 1;
  c->cur = 0;
  c->it = 0;
  c->maxit = maxit;
  c->tol = tol;
}

// One thread.  The check of this iteration has finished (stream order), so
// cur is final.
__global__ void k_iter_tail(SolveCtl* c, cudaGraphConditionalHandle cond, int graph) {
  const int cur = c->cur;
  c->prev = cur;
  c->cur = 0;
  c->it += 1;
  if (graph) {
    c->graph_iters[graph - 1] += 1;
    cudaGraphSetConditional(cond, (cur > 0 && c->it < c->maxit) ? 1u : 0u);
  }
}

// Zero a buffer (16-byte stores, grid-stride), skipped once no instance is
// active.
// Zero the first n16 16-byte words of each of `tiles` arrays spaced stride16
// words apart (the LU arrays of the tiles: whole, or their sparse segments).
__global__ void k_zero16(uint4* __restrict__ p, size_t n16, size_t stride16, int tiles,
                         const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
  const size_t total = n16 * (size_t)tiles;
  if (n16 == stride16) {  // the whole per-tile arrays: one contiguous range
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
      p[i] = z;
    return;
  }
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
    p[(i / n16) * stride16 + i % n16] = z;
}

// Identity on the padding of the dense block, and zero right-hand side on
// its padding rows (m .. s+nde-1): no other kernel writes those rows, and a
// stale non-finite value there would leak into real rows as 0 * NaN during
// the backward substitution.
template <typename T>
__global__ void k_set_ones(DevPlan P, DevState S, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int tile = blockIdx.y, lane = threadIdx.x;
  T* LU = reinterpret_cast<T*>(S.lu) + (size_t)tile * P.NLU * kTile;
  T* X = reinterpret_cast<T*>(S.x) + (size_t)tile * P.mp * kTile;
  // padding columns nd .. nde-1 of the dense block: whole identity columns
  // (the refactorisation does not zero the dense block)
  const int t = blockIdx.x;  // a block per padding column
  for (int r = threadIdx.y; r < P.nde; r += blockDim.y)
    LU[lu_off<T>(P, P.NS + (int64_t)(P.nd + t) * P.ndp + r, lane)] = (T)(r == P.nd + t ? 1 : 0);
  if (threadIdx.y == 0) X[(size_t)(P.m + t) * kTile + lane] = (T)0;
}

// ---------------------------------------------------------------------------
// Sparse left-looking refactorisation, one level of the column schedule
// (Alg. 2 / Alg. 3 stage 1: every column of a level in parallel, one lane per
// instance).  Column j: for each finished column k with U(k,j) != 0, in
// ascending k:  col_j[rows of L(:,k)] -= U(k,j) * L(:,k);  then, for a sparse
// column, L(:,j) /= U(j,j).  Dense-block columns only receive the updates of
// the sparse columns (their Schur complement), and are finished later.
// ---------------------------------------------------------------------------
constexpr int kLWarps = 4;

template <typename T>
__global__ void __launch_bounds__(32 * kLWarps) k_lu_sparse_level(DevPlan P, DevState S, int c0, int c1,
                                                                  const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x;
  const int ci = c0 + blockIdx.x * kLWarps + threadIdx.y;
  const int tile = blockIdx.y;
  if (ci >= c1) return;
  if (!tile_active(S, tile, lane)) return;
  T* __restrict__ LUb = reinterpret_cast<T*>(S.lu) + (size_t)tile * P.NLU * kTile;  // tile base
  T* __restrict__ LU = LUb + lane;  // sparse positions (< NS): p * 32
  const int j = P.lu_cols[ci];
  const int u0 = P.col_upd_ptr[j], u1 = P.col_upd_ptr[j + 1];
  for (int u = u0; u < u1; ++u) {
    const DevUpd up = P.upd[u];
    const T x = LU[(size_t)up.ukj * kTile];
    const int32_t* __restrict__ dst = P.dst + up.dst_off;
    const T* __restrict__ src = LU + (size_t)up.lsrc * kTile;
    int q = 0;
    for (; q + 4 <= up.llen; q += 4) {
      const size_t o0 = lu_off<T>(P, dst[q], lane), o1 = lu_off<T>(P, dst[q + 1], lane);
      const size_t o2 = lu_off<T>(P, dst[q + 2], lane), o3 = lu_off<T>(P, dst[q + 3], lane);
      const T s0 = src[(size_t)q * kTile], s1 = src[(size_t)(q + 1) * kTile];
      const T s2 = src[(size_t)(q + 2) * kTile], s3 = src[(size_t)(q + 3) * kTile];
      const T a0 = LUb[o0], a1 = LUb[o1];
      const T a2 = LUb[o2], a3 = LUb[o3];
      LUb[o0] = a0 - x * s0;
      LUb[o1] = a1 - x * s1;
      LUb[o2] = a2 - x * s2;
      LUb[o3] = a3 - x * s3;
    }
    for (; q < up.llen; ++q) LUb[lu_off<T>(P, dst[q], lane)] -= x * src[(size_t)q * kTile];
  }
  const int dpj = P.dp[j];
  if (dpj >= 0) {
    const T inv = (T)1 / LU[(size_t)dpj * kTile];
    const int64_t e = P.ce[j];
    for (int64_t p = dpj + 1; p < e; ++p) LU[(size_t)p * kTile] *= inv;
  }
}

// ---------------------------------------------------------------------------
// The level schedules in one launch each.  A tile belongs to a cluster of C
// CTAs, whose warps share the tasks of a level and meet at the cluster's barrier
// (C = 1: the CTA's) before the next: one launch per level costs 3 to 4 us, most
// of it the launch and the chain of gate, schedule and value loads, and the
// 2,000-bus FP64 plan has 31 + 31 + 30 levels per iteration.
// C: as many CTAs (a power of two, at most 8, of 1,024 threads) as the tiles leave
// SMs for and a level has tasks for, 32 to a CTA: within one CTA the values stay
// in L1 and the barrier is cheap.  With more tiles than SMs one smaller CTA each,
// so that all are resident at once (64 registers: 2, 3, 4 CTAs of 512, 320, 256
// threads per SM).
// ---------------------------------------------------------------------------
struct LevelShape {
  int cluster, threads;
};
inline LevelShape level_shape(int tiles, int tasks, int levels) {
  if (tiles > 456) return {1, 256};
  if (tiles > 304) return {1, 320};
  if (tiles > 152) return {1, 512};
  int c = 8;
  while (c > 1 && (c * tiles > 152 || (int64_t)16 * c * levels >= tasks)) c /= 2;
  return {c, 1024};
}

__device__ __forceinline__ void level_barrier(int cluster) {
  if (cluster > 1)
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
  else
    __syncthreads();
}

// Sparse refactorisation by entries (plan.h: fac_*), every level.  A warp takes a
// task of up to 16 operations (or one longer entry): 32 operations come with one
// coalesced load and are handed out by shuffles, and the values of eight are in
// flight together; the entry being formed stays in a register and takes its
// subtractions in ascending k, exactly as the left-looking columns do.  The
// operations of a warp's next task are loaded ahead, across the barrier too, so
// that a level's chain is value, arithmetic, store, barrier.  By columns
// (k_lu_sparse_level, a launch per level) a task reads, changes and writes the
// whole column once per k, each waiting for the one before.  Per refactorisation
// of the 2,000-bus plans, by columns and by entries:
//   FP64: 1 tile 2.68, 0.65 ms; 60 tiles 4.24, 1.74 ms; 313 tiles 7.57, 8.9 ms
//   FP32: 11 tiles 0.86, 0.22 ms; 313 tiles 2.60, 2.41 ms
// so FP64 with more tiles than SMs keeps the columns.
template <typename T>
__global__ void __launch_bounds__(1024) k_sparse_factor(DevPlan P, DevState S, int cluster,
                                                        const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x & 31;
  const int tile = blockIdx.x / cluster;
  if (!tile_active(S, tile, lane)) return;  // uniform over the cluster
  const int W = cluster * (blockDim.x >> 5);
  const int w = (blockIdx.x % cluster) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  T* LU = reinterpret_cast<T*>(S.lu) + (size_t)tile * P.NLU * kTile + lane;
  T* DI = reinterpret_cast<T*>(S.dinv) + (size_t)tile * P.s * kTile + lane;
  const int32_t* __restrict__ lvl = P.fac_lvl_ptr;
  const int total = lvl[P.n_fac_lvl];
  int nt = w, nq0 = 0, nq1 = 0;  // the task loaded ahead: its operations, 32 of them in nop
  int2 nop = make_int2(0, 0);
  auto fetch = [&](int t) {
    nt = t;
    if (t < total) {
      nq0 = P.fac_task[t];
      nq1 = P.fac_task[t + 1];
      nop = P.fac_op[min(nq0 + lane, nq1 - 1)];
    }
  };
  fetch(w);
  int t1 = lvl[1], t2 = P.n_fac_lvl > 1 ? lvl[2] : t1;
  for (int l = 0, t0 = 0; l < P.n_fac_lvl; ++l) {
    int t = t0 + w;
    if (t >= t1) fetch(t1 + w);
    while (t < t1) {
      if (nt != t) fetch(t);
      const int q0 = nq0, q1 = nq1;
      int2 op = nop;
      t += W;
      fetch(t < t1 ? t : t1 + w);
      T acc = (T)0, scale = (T)0;
      int pos = 0, kind = 0, col = 0;
      auto finish = [&] {
        if (kind == 2) acc *= scale;
        if (kind == 3) DI[(size_t)col * kTile] = (T)1 / acc;
        if (kind) LU[(size_t)pos * kTile] = acc;
      };
      for (int qb = q0; qb < q1; qb += 32) {
        const int cnt = min(32, q1 - qb);
        if (qb > q0) op = P.fac_op[min(qb + lane, q1 - 1)];
        for (int i = 0; i < cnt; i += 8) {
          T a[8], b[8];
          int x[8], y[8];
#pragma unroll
          for (int z = 0; z < 8; ++z) {
            x[z] = __shfl_sync(0xffffffffu, op.x, i + z);
            y[z] = __shfl_sync(0xffffffffu, op.y, i + z);
            if (i + z < cnt) {
              a[z] = LU[(size_t)(x[z] >> 2) * kTile];
              const int k = x[z] & 3;
              if (k == 0) b[z] = LU[(size_t)y[z] * kTile];
              else if (k == 2) b[z] = DI[(size_t)y[z] * kTile];
            }
          }
#pragma unroll
          for (int z = 0; z < 8; ++z) {
            if (i + z < cnt) {
              const int k = x[z] & 3;
              if (k == 0) {
                acc -= a[z] * b[z];
              } else {
                finish();
                acc = a[z];
                scale = b[z];
                pos = x[z] >> 2;
                kind = k;
                col = y[z];
              }
            }
          }
        }
      }
      finish();
    }
    t0 = t1;
    t1 = t2;
    if (l + 3 <= P.n_fac_lvl) t2 = lvl[l + 3];
    level_barrier(cluster);
  }
}

// Schur complement of the sparse columns into the dense block, after the
// sparse levels (every U(k, j) is then final).  A warp per (dense column j,
// chunk of 32 dense rows) and tile: the rows live in shared memory (one
// column of 32 rows per lane) while the products L(i, k) U(k, j) of all
// sparse columns k are applied, then go back once.  The warp reads 32 entries
// with one coalesced load and hands them out by shuffles, so the L and U loads
// of eight entries are in flight together.
//   FP64 (bound by the FP64 pipe): each row starts from A(i, j) and takes the
//   subtractions, in the order of the sparse columns as a left-looking
//   column does; no separate subtraction pass.  At most 72 registers: 7 CTAs
//   per SM, the shared-memory limit.
//   FP32 (bound by load latency): each row starts from 0, sums the products
//   and is subtracted from A(i, j) at the end, which keeps the register count
//   and so the warps per SM up (at most 48 registers: ten CTAs per SM).
constexpr int kSchurWarps = 4;

template <typename T>
__global__ void __launch_bounds__(32 * kSchurWarps, sizeof(T) == 8 ? 7 : 10) k_schur(DevPlan P, DevState S, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  __shared__ T acc[kSchurWarps][32][33];  // [row of the chunk][lane], padded: a row of one lane is read across the warp
  const int lane = threadIdx.x, w = threadIdx.y;
  const int t = blockIdx.x * kSchurWarps + w;
  const int tile = blockIdx.y;
  if (t >= P.n_schur) return;
  if (!tile_active(S, tile, lane)) return;
  T* __restrict__ LUb = reinterpret_cast<T*>(S.lu) + (size_t)tile * P.NLU * kTile;
  const T* __restrict__ LU = LUb + lane;  // sparse positions (< NS): p * 32
  T(*a)[33] = acc[w];
  const int4 task = P.schur_task[t];
  // A(i, j) = J(i, j) where J has an entry, else 0: the block is not zeroed
  // before the refactorisation; the Jacobian fill has written its entries
  const uint32_t jm = P.schur_jmask[t];
  constexpr bool kSeeded = DenseGroup<T>::G != 4;
  if constexpr (kSeeded) {
    const int64_t col = P.NS + (int64_t)task.x * P.ndp + 32 * task.y;
    const int nr = min(32, P.ndp - 32 * task.y);
#pragma unroll 4
    for (int r = 0; r < 32; ++r)
      a[r][lane] = (r < nr && (jm >> r & 1u)) ? LUb[lu_off<T>(P, col + r, lane)] : (T)0;
  } else {
#pragma unroll
    for (int r = 0; r < 32; ++r) a[r][lane] = (T)0;
  }
  for (int eb = task.z; eb < task.w; eb += 32) {
    const int cnt = min(32, task.w - eb);
    const int32_t xl = lane < cnt ? P.schur_ent[eb + lane] : 0;
    const int32_t ul = lane < cnt ? P.schur_u[eb + lane] : 0;
    for (int i = 0; i < cnt; i += 8) {
      T l[8], u[8];
      int r[8];
#pragma unroll
      for (int z = 0; z < 8; ++z) {
        const int32_t x = __shfl_sync(0xffffffffu, xl, i + z);
        const int32_t up = __shfl_sync(0xffffffffu, ul, i + z);
        r[z] = x & 31;
        const bool ok = i + z < cnt;
        l[z] = ok ? LU[(size_t)(x >> 5) * kTile] : (T)0;
        u[z] = ok ? LU[(size_t)up * kTile] : (T)0;
      }
      // entries of one task keep their order (the sparse columns ascending)
#pragma unroll
      for (int z = 0; z < 8; ++z)
        if (i + z < cnt) {
          if constexpr (kSeeded) a[r[z]][lane] -= l[z] * u[z];
          else a[r[z]][lane] += l[z] * u[z];
        }
    }
  }
  // every row of the chunk below the padded size is written back
  if constexpr (!kSeeded) {
    if (P.dim) {
      // instance-major block: instance l's 32 rows of column task.x are one
      // contiguous 128-byte line, written by the whole warp (lane = row)
      __syncwarp();
      const int nr = min(32, P.ndp - 32 * task.y);
      const bool jrow = (jm >> lane) & 1u;
      float* __restrict__ col = LUb + (size_t)P.NS * kTile + (size_t)task.x * P.ndp + 32 * task.y + lane;
      const size_t bstride = (size_t)P.ndp * (size_t)P.ndp;
      if (lane < nr) {
#pragma unroll 4
        for (int l = 0; l < 32; ++l) {
          float* q = col + (size_t)l * bstride;
          const float sum = a[lane][l];
          *q = jrow ? *q - sum : -sum;
        }
      }
      return;
    }
    // FP32 grouped interleaved block: rows 4g .. 4g+3 of the chunk are one
    // 16-byte word per lane; A(i, j) minus the sum
    float4* __restrict__ A4 = reinterpret_cast<float4*>(LUb + (size_t)P.NS * kTile);
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const int r0 = 32 * task.y + 4 * g;
      if (r0 >= P.nde) break;
      float4* q = A4 + ((size_t)task.x * P.ndp + r0) * 8 + lane;
      const uint32_t jb = jm >> (4 * g) & 0xFu;
      float4 v = jb ? *q : make_float4(0.f, 0.f, 0.f, 0.f);
      v.x = (jb & 1u) ? v.x - a[4 * g][lane] : -a[4 * g][lane];
      v.y = (jb & 2u) ? v.y - a[4 * g + 1][lane] : -a[4 * g + 1][lane];
      v.z = (jb & 4u) ? v.z - a[4 * g + 2][lane] : -a[4 * g + 2][lane];
      v.w = (jb & 8u) ? v.w - a[4 * g + 3][lane] : -a[4 * g + 3][lane];
      *q = v;
    }
  } else {
    const int64_t col = P.NS + (int64_t)task.x * P.ndp + 32 * task.y;
    const int nr = min(32, P.ndp - 32 * task.y);
#pragma unroll 4
    for (int r = 0; r < nr; ++r) LUb[lu_off<T>(P, col + r, lane)] = a[r][lane];
  }
}

// ---------------------------------------------------------------------------
// Dense trailing block: right-looking blocked LU without pivoting, panel width
// kb, on every instance's ndp x ndp column-major block (Sec. 4.3: the serial
// tail of the column DAG, where few columns remain per level, is handled as
// one dense matrix whose updates are independent multiply-adds).
//   (a) k_dense_diag   : factor the kb x kb diagonal block, store 1/pivots
//   (b) k_dense_panel  : L21 = A21 U11^-1 (rows) and U12 = L11^-1 A12 (cols),
//                        four rows or four columns per thread
//   (c) k_dense_update : A22 -= L21 U12, a register tile per thread (4x4 FP64, 8x8 FP32)
// ---------------------------------------------------------------------------
template <typename T, int KB>
__global__ void k_dense_diag(DevPlan P, DevState S, int k, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x;
  const int tile = blockIdx.x * blockDim.y + threadIdx.y;
  if (tile * kTile >= S.Bp) return;
  if (!tile_active(S, tile, lane)) return;
  T* __restrict__ A = reinterpret_cast<T*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile;  // dense block
  T* __restrict__ inv = reinterpret_cast<T*>(S.inv) + (size_t)tile * KB * kTile + lane;
  const int ld = P.ndp;
  T D[KB][KB];
#pragma unroll
  for (int c = 0; c < KB; ++c)
#pragma unroll
    for (int r = 0; r < KB; ++r) D[r][c] = A[dense_off<T>(k + r, k + c, ld, lane)];
#pragma unroll
  for (int c = 0; c < KB; ++c) {
    const T ip = (T)1 / D[c][c];
    inv[c * kTile] = ip;
#pragma unroll
    for (int r = c + 1; r < KB; ++r) D[r][c] *= ip;
#pragma unroll
    for (int cc = c + 1; cc < KB; ++cc)
#pragma unroll
      for (int r = c + 1; r < KB; ++r) D[r][cc] -= D[r][c] * D[c][cc];
  }
#pragma unroll
  for (int c = 0; c < KB; ++c)
#pragma unroll
    for (int r = 0; r < KB; ++r) A[dense_off<T>(k + r, k + c, ld, lane)] = D[r][c];
}

// The 16 x 16 block does not fit a thread's registers: one CTA per tile, eight warps
// with two rows each, r = w and w + 8, in registers, the pivot row published in shared
// memory, one barrier per pivot.
constexpr int kDiagWarps = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kDiagWarps) k_dense_diag16(DevPlan P, DevState S, int k,
                                                                  const int32_t* __restrict__ gate) {
  constexpr int KB = 16;
  __shared__ T prow[2][KB][kTile];
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x, w = threadIdx.y, tile = blockIdx.x;
  if (!tile_active(S, tile, lane)) return;  // uniform over the CTA
  T* __restrict__ A = reinterpret_cast<T*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile;  // dense block
  T* __restrict__ inv = reinterpret_cast<T*>(S.inv) + (size_t)tile * KB * kTile + lane;
  const int ld = P.ndp;
  T d[2][KB];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < KB; ++c) d[h][c] = A[dense_off<T>(k + w + 8 * h, k + c, ld, lane)];
#pragma unroll
  for (int c = 0; c < KB; ++c) {
    if (w == (c & 7)) {
#pragma unroll
      for (int cc = c; cc < KB; ++cc) prow[c & 1][cc][lane] = d[c >> 3][cc];
    }
    __syncthreads();
    const T ip = (T)1 / prow[c & 1][c][lane];
    if (w == (c & 7)) inv[c * kTile] = ip;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (w + 8 * h > c) {
        const T l = d[h][c] * ip;
        d[h][c] = l;
#pragma unroll
        for (int cc = c + 1; cc < KB; ++cc) d[h][cc] -= l * prow[c & 1][cc][lane];
      }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < KB; ++c) A[dense_off<T>(k + w + 8 * h, k + c, ld, lane)] = d[h][c];
}

// four consecutive rows r .. r+3 (r a multiple of 4) of dense column c for
// this lane: one 16-byte load in the grouped FP32 layout, four loads in FP64
template <typename T>
__device__ __forceinline__ void ld4(const T* __restrict__ A, int r, int c, int ld, int lane, T (&v)[4]) {
  if constexpr (DenseGroup<T>::G == 4) {
    const float4 q = reinterpret_cast<const float4*>(A)[((size_t)c * ld + r) * 8 + lane];
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = A[dense_off<T>(r + i, c, ld, lane)];
  }
}

template <typename T>
__device__ __forceinline__ void st4(T* __restrict__ A, int r, int c, int ld, int lane, const T (&v)[4]) {
  if constexpr (DenseGroup<T>::G == 4) {
    reinterpret_cast<float4*>(A)[((size_t)c * ld + r) * 8 + lane] = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) A[dense_off<T>(r + i, c, ld, lane)] = v[i];
  }
}

// y <- L^-1 y for NC columns held in registers, L the NR x NR unit-lower
// block at dense (k, k): column-oriented forward elimination, the
// subtractions into each y[c] in ascending p
template <typename T, int NR, int NC>
__device__ __forceinline__ void unit_lower_solve(const T* __restrict__ A, int k, int ld, int lane, T (&y)[NC][NR]) {
#pragma unroll
  for (int p = 0; p < NR - 1; ++p)
#pragma unroll
    for (int q = (p + 1) / 4; q < NR / 4; ++q) {
      T l[4];
      ld4(A, k + 4 * q, k + p, ld, lane, l);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (4 * q + i > p) {
#pragma unroll
          for (int t = 0; t < NC; ++t) y[t][4 * q + i] -= l[i] * y[t][p];
        }
    }
}

template <typename T, int KB>
__global__ void k_dense_panel(DevPlan P, DevState S, int k, int cend, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x;
  const int tile = blockIdx.y;
  if (!tile_active(S, tile, lane)) return;
  const int ld = P.ndp;
  const int r0 = k + KB;              // first trailing row/column
  const int ngrp = (ld - r0) / 4;     // groups of four rows (down to ld)
  const int ngc = (cend - r0) / 4;    // groups of four columns (up to cend)
  const int g = blockIdx.x * blockDim.y + threadIdx.y;
  if (g >= ngrp + ngc) return;
  T* __restrict__ A = reinterpret_cast<T*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile;  // dense block
  const T* __restrict__ inv = reinterpret_cast<const T*>(S.inv) + (size_t)tile * KB * kTile + lane;
  if (g < ngrp) {
    // rows i0..i0+3: x U11 = a  (U11 upper, pivots inverted), column by
    // column; the subtractions into x[c] in ascending p
    const int i0 = r0 + 4 * g;
    T x[KB][4];
#pragma unroll
    for (int c = 0; c < KB; ++c) ld4(A, i0, k + c, ld, lane, x[c]);
#pragma unroll
    for (int c = 0; c < KB; ++c) {
#pragma unroll
      for (int q = 0; q < KB / 4; ++q) {
        if (4 * q >= c) break;
        T u[4];
        ld4(A, k + 4 * q, k + c, ld, lane, u);  // U(k+4q .. k+4q+3, k+c)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (4 * q + i < c) {
#pragma unroll
            for (int t = 0; t < 4; ++t) x[c][t] -= x[4 * q + i][t] * u[i];
          }
      }
      const T ip = inv[c * kTile];
#pragma unroll
      for (int t = 0; t < 4; ++t) x[c][t] *= ip;
    }
#pragma unroll
    for (int c = 0; c < KB; ++c) st4(A, i0, k + c, ld, lane, x[c]);
  } else {
    // columns j0..j0+3: L11 y = a  (L11 unit lower)
    const int j0 = r0 + 4 * (g - ngrp);
    T y[4][KB];
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int q = 0; q < KB / 4; ++q) {
        T v[4];
        ld4(A, k + 4 * q, j0 + t, ld, lane, v);
#pragma unroll
        for (int i = 0; i < 4; ++i) y[t][4 * q + i] = v[i];
      }
    unit_lower_solve<T, KB, 4>(A, k, ld, lane, y);
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int q = 0; q < KB / 4; ++q) {
        const T v[4] = {y[t][4 * q], y[t][4 * q + 1], y[t][4 * q + 2], y[t][4 * q + 3]};
        st4(A, k + 4 * q, j0 + t, ld, lane, v);
      }
  }
}

// occupancy hint: 128-thread CTAs, at least kUpdMinBlocks resident per SM
// (the 8x8 FP32 tile is latency-bound when registers limit residency)
template <typename T, int TS>
struct UpdOcc {
  static constexpr int value = (sizeof(T) == 4 && TS == 8) ? 2 : 6;
};

// The updated region is the trailing block [r0, ld) x [r0, ld) without its
// part [kend, ld) x [kend, ld): kend = ld for a one-level panel (the whole
// trailing block); kend = the end of the outer panel for an inner step of a
// two-level panel (the outer panel's own columns, and its rows to the right).
template <typename T, int KB, int TS>
__global__ void __launch_bounds__(128, UpdOcc<T, TS>::value) k_dense_update(DevPlan P, DevState S, int k, int kend,
                                                                           int cend, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x;
  const int tile = blockIdx.y;
  if (!tile_active(S, tile, lane)) return;
  const int ld = P.ndp;
  const int r0 = k + KB;
  const int nbr = (ld - r0) / TS, nbk = (kend - r0) / TS, nbx = (cend - kend) / TS;
  const int n1 = nbr * nbk;  // columns [r0, kend), all rows
  const int t = blockIdx.x * blockDim.y + threadIdx.y;
  if (t >= n1 + nbk * nbx) return;
  int i0, j0;
  if (t < n1) {
    i0 = r0 + TS * (t % nbr);
    j0 = r0 + TS * (t / nbr);
  } else {  // rows [r0, kend), columns [kend, ld)
    i0 = r0 + TS * ((t - n1) % nbk);
    j0 = kend + TS * ((t - n1) / nbk);
  }
  T* __restrict__ Ab = reinterpret_cast<T*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile;  // dense block
  T acc[TS][TS];
  if constexpr (DenseGroup<T>::G == 4 && TS == 8) {
    // FP32, grouped rows: rows r..r+3 of column c for this lane are the
    // float4 at index (c * ld + r) * 8 + lane.  acc2[p][c] holds rows 2p,
    // 2p+1 of column c: one packed two-wide FMA (fma.rn.f32x2) per pair, with
    // -b, which rounds as acc - a b in one step
    float4* __restrict__ A4 = reinterpret_cast<float4*>(Ab);
    float2 acc2[4][TS];
#pragma unroll
    for (int c = 0; c < TS; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = A4[((size_t)(j0 + c) * ld + i0 + 4 * h) * 8 + lane];
        acc2[2 * h][c] = make_float2(v.x, v.y);
        acc2[2 * h + 1][c] = make_float2(v.z, v.w);
      }
#pragma unroll
    for (int pp = 0; pp < KB / 4; ++pp) {
      float4 bq[TS];  // rows k+4pp .. k+4pp+3 of columns j0 .. j0+7 (U12)
#pragma unroll
      for (int c = 0; c < TS; ++c) bq[c] = A4[((size_t)(j0 + c) * ld + k + 4 * pp) * 8 + lane];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int p = 4 * pp + q;
        const float4 a0 = A4[((size_t)(k + p) * ld + i0) * 8 + lane];  // rows i0..i0+7 of column k+p (L21)
        const float4 a1 = A4[((size_t)(k + p) * ld + i0 + 4) * 8 + lane];
        const float2 ap[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y),
                              make_float2(a1.z, a1.w)};
#pragma unroll
        for (int c = 0; c < TS; ++c) {
          const float nb = -(q == 0 ? bq[c].x : q == 1 ? bq[c].y : q == 2 ? bq[c].z : bq[c].w);
          const float2 b2 = make_float2(nb, nb);
#pragma unroll
          for (int r = 0; r < 4; ++r) acc2[r][c] = __ffma2_rn(ap[r], b2, acc2[r][c]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < TS; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        A4[((size_t)(j0 + c) * ld + i0 + 4 * h) * 8 + lane] =
            make_float4(acc2[2 * h][c].x, acc2[2 * h][c].y, acc2[2 * h + 1][c].x, acc2[2 * h + 1][c].y);
  } else if constexpr (DenseGroup<T>::G == 1) {
    // element (r, c) is Ab[(c * ld + r) * 32 + lane]: a column pointer plus a
    // compile-time offset for every access
    T* __restrict__ A = Ab + lane;
    const size_t cstride = (size_t)ld * kTile;
    T* __restrict__ cj = A + (size_t)j0 * cstride + (size_t)i0 * kTile;      // (i0, j0)
    const T* __restrict__ pa = A + (size_t)k * cstride + (size_t)i0 * kTile;  // (i0, k)
    const T* __restrict__ pb = A + (size_t)j0 * cstride + (size_t)k * kTile;  // (k, j0)
#pragma unroll
    for (int c = 0; c < TS; ++c)
#pragma unroll
      for (int r = 0; r < TS; ++r) acc[r][c] = cj[c * cstride + r * kTile];
#pragma unroll(KB > 16 ? 8 : KB)
    for (int p = 0; p < KB; ++p) {
      T a[TS], b[TS];
#pragma unroll
      for (int r = 0; r < TS; ++r) a[r] = pa[p * cstride + r * kTile];
#pragma unroll
      for (int c = 0; c < TS; ++c) b[c] = pb[c * cstride + p * kTile];
#pragma unroll
      for (int c = 0; c < TS; ++c)
#pragma unroll
        for (int r = 0; r < TS; ++r) acc[r][c] -= a[r] * b[c];
    }
#pragma unroll
    for (int c = 0; c < TS; ++c)
#pragma unroll
      for (int r = 0; r < TS; ++r) cj[c * cstride + r * kTile] = acc[r][c];
  } else {
    // grouped layout with a 4x4 tile (FP32 with panel 4): element by element
#pragma unroll
    for (int c = 0; c < TS; ++c)
#pragma unroll
      for (int r = 0; r < TS; ++r) acc[r][c] = Ab[dense_off<T>(i0 + r, j0 + c, ld, lane)];
#pragma unroll(KB > 16 ? 8 : KB)
    for (int p = 0; p < KB; ++p) {
      T a[TS], b[TS];
#pragma unroll
      for (int r = 0; r < TS; ++r) a[r] = Ab[dense_off<T>(i0 + r, k + p, ld, lane)];
#pragma unroll
      for (int c = 0; c < TS; ++c) b[c] = Ab[dense_off<T>(k + p, j0 + c, ld, lane)];
#pragma unroll
      for (int c = 0; c < TS; ++c)
#pragma unroll
        for (int r = 0; r < TS; ++r) acc[r][c] -= a[r] * b[c];
    }
#pragma unroll
    for (int c = 0; c < TS; ++c)
#pragma unroll
      for (int r = 0; r < TS; ++r) Ab[dense_off<T>(i0 + r, j0 + c, ld, lane)] = acc[r][c];
  }
}

// ---------------------------------------------------------------------------
// FP64 trailing update of depth 16 in integer arithmetic.  An FP64 multiply-add
// of a warp holds its quarter of the SM for 64 cycles; a 32 x 32 + 64-bit integer
// one (mad.wide) four.  The update is therefore made in fixed point:
//  * k_dense_limbs: with h_p half the exponent of pivot p, the 16 entries
//    l_p 2^h_p of each row of L21 become integers of 55 bits and sign,
//    X = x 2^(1077 - E), E the largest (biased) exponent among them, rounded to
//    nearest; likewise u_p 2^-h_p of each column of U12.  X = hi 2^28 + lo, both
//    signed 28 bits.  The factors h_p leave the products as they are and take a
//    scaling of the unknowns (a bus with a very short line) out of the rows' and
//    columns' ranges.
//  * k_dense_update_fixed: sum of hi hi and of hi lo + lo hi over the 16 products
//    in two 64-bit integers, exactly (lo lo, 2^54 of 2^110, is left out);
//    then hh + hl / 2^28, rounded, is converted and subtracted once, C <- C - T s
//    with the power of two s = 2^(Ea + Eb - 1075 - 1023).
// Error of an entry (i, j), in units of R_i C_j, the largest |l_p 2^h_p| of its row
// times the largest |u_p 2^-h_p| of its column, which need not meet in a product:
// rounding the operands 16 (2^-55 + 2^-55), the products lo lo 16 2^-54, at most
// 2^-49.4 together, typically 2^-54.  By multiply-adds it is 16 roundings of 2^-53 of
// the entry's partial sums.  The first is the smaller one as long as R_i C_j is near
// the entries that matter in row i; where the exponents of the 16 pivots lie further
// apart, R_i and C_j come from pivots of different size.  So an instance whose pivots
// span more than kFixSpread binary orders, or whose operands hold an infinity, a NaN,
// a subnormal, or scales beyond the exponent range, takes multiply-adds in pivot order,
// lane by lane.  On meshed grids of 100 to 3,000 buses the pivots of 16 columns span 1 to
// 3 orders.
// Component-wise backward error of solves with the dense block, max_i |S y - c|_i /
// (|S| |y| + |c|)_i, over that of multiply-adds, geometric mean and worst of 33 draws each
// of 420, 700 and 1,300 buses, emulated: plain impedances 0.72 to 0.83 (1.4); impedances
// spread over 10^6 or 10^8, or 3 % of the lines shorter by 10^2 to 10^8, 0.78 to 1.00
// (4.0; multiply-adds in reversed order 5.4).  Without the limit 0.74 to 10^4 (6 10^4),
// without h_p either to 5 10^5 (2 10^6).
// Backward error of staged FP64 solves, max norm |J x - b| / (|J| |x| + |b|),
// median of 16 instances, by multiply-adds and in this form (meshed grids):
//   buses (dense)  700 (136)  1,300 (240)  2,000 (272)  2,000 (448)  3,000 (544)
//   multiply-adds  5.3e-17    6.4e-17      8.1e-17      1.7e-16      1.4e-16
//   this form      4.0e-17    5.1e-17      6.2e-17      1.1e-16      9.1e-17
// Bounds: 48 mad.wide per entry and 16 products, four cycles each on the pipe that
// makes them (79 ms for four refactorisations of 10,000 272-wide blocks), and two
// FP64 instructions, conversion and subtraction (53 ms); measured 121 ms, where
// multiply-adds took 397. Loading the operands through registers instead of one
// bulk copy per side took 138 ms; more warps per CTA were no faster.
// ---------------------------------------------------------------------------
constexpr int kFixK = 16;
constexpr int kFixBad = 0x4000;  // exponent of a row that fixed point cannot hold
constexpr int kFixSpread = 4;

// S.limb, per tile and in groups of four rows of L21 (then of four columns of
// U12): int4 [2][ndp/4][kFixK][2][32], a lane's int4 = (hi, lo) of two rows, so
// that a group's operands are one run at constant offsets; then int4
// [2][ndp/4][32], the four exponents (L21's with the bias of the product taken
// off); then int32 [32], whether the instance's pivots are too far apart.
__host__ __device__ __forceinline__ size_t limb_flags(int ndp) {
  return (size_t)(ndp / 4) * 2 * kTile * (2 * kFixK + 1);
}
__host__ __device__ __forceinline__ size_t limb_vecs(int ndp) {  // int4 per tile
  return limb_flags(ndp) + kTile * sizeof(int32_t) / sizeof(int4);
}

// A warp takes two rows of L21 or two columns of U12, which share a lane's int4.
__global__ void __launch_bounds__(128) k_dense_limbs(DevPlan P, DevState S, int k, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x, tile = blockIdx.y, ld = P.ndp;
  if (!tile_active(S, tile, lane)) return;
  const int r0 = k + kFixK, n = ld - r0;
  const int t = 2 * (blockIdx.x * blockDim.y + threadIdx.y);
  if (t >= 2 * n) return;
  const bool row = t < n;
  const int i = r0 + (row ? t : t - n), g = (row ? 0 : ld / 4) + i / 4;
  const double* __restrict__ A = reinterpret_cast<const double*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile + lane;
  int4* base = reinterpret_cast<int4*>(S.limb) + (size_t)tile * limb_vecs(ld);
  int4* out = base + ((size_t)g * kFixK * 2 + (i & 2) / 2) * kTile + lane;
  int2* eo = reinterpret_cast<int2*>(base + ((size_t)(ld / 4) * 2 * kFixK * 2 + g) * kTile + lane) + (i & 2) / 2;
  long long x[2][kFixK];
#pragma unroll
  for (int p = 0; p < kFixK; ++p)
#pragma unroll
    for (int z = 0; z < 2; ++z)
      x[z][p] = __double_as_longlong(A[(row ? (size_t)(k + p) * ld + i + z : (size_t)(i + z) * ld + k + p) * kTile]);
  int h[kFixK], pmin = 0x7ff, pmax = 0;
#pragma unroll
  for (int p = 0; p < kFixK; ++p) {
    const int e = (__double2hiint(A[((size_t)(k + p) * ld + k + p) * kTile]) >> 20) & 0x7ff;
    pmin = min(pmin, e);
    pmax = max(pmax, e);
    h[p] = (e - 1023) >> 1;
    if (!row) h[p] = -h[p];
  }
  if (t == 0) reinterpret_cast<int32_t*>(base + limb_flags(ld))[lane] = pmax - pmin > kFixSpread;
  constexpr int kNone = -0x4000;
  int em[2] = {kNone, kNone};
  bool bad[2] = {false, false};
#pragma unroll
  for (int p = 0; p < kFixK; ++p)
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      const int ex = (int)(x[z][p] >> 52) & 0x7ff;
      bad[z] |= ex == 0x7ff || (ex == 0 && (x[z][p] << 1) != 0);
      if (ex) em[z] = max(em[z], ex + h[p]);
    }
#pragma unroll
  for (int p = 0; p < kFixK; ++p) {
    int w[2][2];
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      const long long q = x[z][p];
      const int ex = (int)(q >> 52) & 0x7ff, d = min(em[z] - (ex + h[p]), 60);
      const long long m = ((q & 0xfffffffffffffll) | 0x10000000000000ll) << 2;
      long long v = d <= 0 ? m : (m + (1ll << (d - 1))) >> d;
      if (ex == 0) v = 0;
      if ((q < 0) != row) v = -v;  // the rows of L21 negated: the sums are subtracted
      w[z][1] = (int)((unsigned)v << 4) >> 4;
      w[z][0] = (int)((v - w[z][1]) >> 28);
    }
    out[(size_t)p * 2 * kTile] = make_int4(w[0][0], w[0][1], w[1][0], w[1][1]);
  }
  int e[2];
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    // an all-zero row: any exponent that keeps the scale of a zero sum normal
    e[z] = bad[z] ? kFixBad : em[z] == kNone ? 1075 : em[z];
    if (row) e[z] -= 1075;
  }
  *eo = make_int2(e[0], e[1]);
}

__device__ __forceinline__ void mad_wide(long long& c, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
}

// A warp per 4 x 4 entries, 2 x 2 warps per CTA.  The CTA's operands, two groups of
// rows and two of columns with all their 16 depths, are two runs of 32 KB: two bulk
// copies bring them to shared memory, and three CTAs per SM cover each other's
// copies, integer work and conversions.
constexpr int kFixWR = 2, kFixWC = 2;  // warps (groups of four rows, of four columns) per CTA
constexpr size_t kFixGroup = (size_t)kFixK * 2 * kTile * sizeof(int4);  // 16 KB
constexpr size_t kFixSmem = (kFixWR + kFixWC) * kFixGroup;
constexpr uint32_t kFixSpinLimit = 1u << 20;

__global__ void __launch_bounds__(32 * kFixWR * kFixWC, 3) k_dense_update_fixed(DevPlan P, DevState S, int k,
                                                               const int32_t* __restrict__ gate) {
  extern __shared__ __align__(128) unsigned char fix_smem[];
  __shared__ __align__(8) uint64_t bar;
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x, w = threadIdx.y, tile = blockIdx.y, ld = P.ndp;
  if (!tile_active(S, tile, lane)) return;  // uniform over the CTA
  const int ng = (ld - k - kFixK) / 4, nb = (ng + kFixWR - 1) / kFixWR;  // groups of rows (and of columns)
  const int gi0 = kFixWR * (int)(blockIdx.x % nb), gj0 = kFixWC * (int)(blockIdx.x / nb);
  const int gi = gi0 + w % kFixWR, gj = gj0 + w / kFixWR;
  const int g0 = (k + kFixK) / 4, G = ld / 4;
  const int4* base = reinterpret_cast<const int4*>(S.limb) + (size_t)tile * limb_vecs(ld);
  const uint32_t sb = static_cast<uint32_t>(__cvta_generic_to_shared(&bar));
  const uint32_t sm = static_cast<uint32_t>(__cvta_generic_to_shared(fix_smem));
  if (lane == 0 && w == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sb) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const uint32_t na = (uint32_t)(min(kFixWR, ng - gi0) * kFixGroup), nbt = (uint32_t)(min(kFixWC, ng - gj0) * kFixGroup);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sb), "r"(na + nbt) : "memory");
    auto copy = [&](uint32_t dst, const int4* src, uint32_t bytes) {
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                   "l"(src), "r"(bytes), "r"(sb)
                   : "memory");
    };
    copy(sm, base + (size_t)(g0 + gi0) * kFixK * 2 * kTile, na);
    copy(sm + kFixWR * (uint32_t)kFixGroup, base + (size_t)(G + g0 + gj0) * kFixK * 2 * kTile, nbt);
  }
  const bool mine = gi < ng && gj < ng;
  int4 ea = make_int4(0, 0, 0, 0), eb = ea;
  double* __restrict__ A = reinterpret_cast<double*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile + lane;
  double* __restrict__ C = A + ((size_t)(4 * (g0 + gj)) * ld + 4 * (g0 + gi)) * kTile;
  bool wide = false;
  if (mine) {
    ea = base[((size_t)2 * G * kFixK * 2 + g0 + gi) * kTile + lane];
    eb = base[((size_t)2 * G * kFixK * 2 + G + g0 + gj) * kTile + lane];
    wide = reinterpret_cast<const int32_t*>(base + limb_flags(ld))[lane] != 0;
  }
  long long hh[4][4], hl[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      hh[r][q] = 0;
      hl[r][q] = 1ll << 27;  // rounds hl / 2^28
    }
  __syncthreads();  // the barrier is initialised
  auto wait = [&] {
    uint32_t ok = 0;
    for (uint32_t spins = 0; !ok && spins < kFixSpinLimit; ++spins)
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(sb)
          : "memory");
    return ok != 0;
  };
  if (__syncthreads_or(!wait())) {  // a copy did not land in time: the step is discarded
    wait();  // no copy of this CTA's may land after it
    S.bad[tile * kTile + lane] = 1;
    return;
  }
  if (!mine) return;
  const int er[4] = {ea.x, ea.y, ea.z, ea.w}, ec[4] = {eb.x, eb.y, eb.z, eb.w};
  const int lo = min(min(er[0], er[1]), min(er[2], er[3])) + min(min(ec[0], ec[1]), min(ec[2], ec[3]));
  const int hi = max(max(er[0], er[1]), max(er[2], er[3])) + max(max(ec[0], ec[1]), max(ec[2], ec[3]));
  double c[4][4];
  if (wide || lo <= 0 || hi >= 2047) {  // the scales are not normal numbers, or kFixBad
    const double* __restrict__ L = A + ((size_t)k * ld + 4 * (g0 + gi)) * kTile;
    const double* __restrict__ U = A + ((size_t)(4 * (g0 + gj)) * ld + k) * kTile;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 4; ++r) c[r][q] = C[((size_t)q * ld + r) * kTile];
#pragma unroll 2
    for (int p = 0; p < kFixK; ++p) {
      double l[4], u[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        l[r] = L[((size_t)p * ld + r) * kTile];
        u[r] = U[((size_t)r * ld + p) * kTile];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) c[r][q] -= l[r] * u[q];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 4; ++r) C[((size_t)q * ld + r) * kTile] = c[r][q];
    return;
  }
  const int4* la = reinterpret_cast<const int4*>(fix_smem + (w % kFixWR) * kFixGroup) + lane;
  const int4* lb = reinterpret_cast<const int4*>(fix_smem + (kFixWR + w / kFixWR) * kFixGroup) + lane;
#pragma unroll
  for (int p = 0; p < kFixK; ++p) {
    const int4 a[2] = {la[(2 * p) * kTile], la[(2 * p + 1) * kTile]};
    const int4 b[2] = {lb[(2 * p) * kTile], lb[(2 * p + 1) * kTile]};
    const int ah[4] = {a[0].x, a[0].z, a[1].x, a[1].z}, al[4] = {a[0].y, a[0].w, a[1].y, a[1].w};
    const int bh[4] = {b[0].x, b[0].z, b[1].x, b[1].z}, bl[4] = {b[0].y, b[0].w, b[1].y, b[1].w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        mad_wide(hh[r][q], ah[r], bh[q]);
        mad_wide(hl[r][q], ah[r], bl[q]);
      }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) mad_wide(hl[r][q], al[r], bh[q]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) c[r][q] = C[((size_t)q * ld + r) * kTile];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const long long t = hh[r][q] + (hl[r][q] >> 28);
      C[((size_t)q * ld + r) * kTile] = fma((double)t, __hiloint2double((er[r] + ec[q]) << 20, 0), c[r][q]);
    }
}

// ---------------------------------------------------------------------------
// Forward / backward substitution (Sec. 4.3.3).  Row-oriented gathers per
// level instead of the paper's atomicAdd scatter: every row writes only its
// own entry, so the result is deterministic.
// ---------------------------------------------------------------------------
// All levels of the forward (BWD: backward) schedule in one launch (see
// k_sparse_factor): a warp per row, its entries in the order of the list, four
// products' loads in flight; the warp's next row and that row's first four
// entries are loaded ahead, across the barrier too.
template <typename T, bool BWD>
__global__ void __launch_bounds__(1024) k_subst(DevPlan P, DevState S, int cluster, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x & 31;
  const int tile = blockIdx.x / cluster;
  if (!tile_active(S, tile, lane)) return;  // uniform over the cluster
  const int W = cluster * (blockDim.x >> 5);
  const int w = (blockIdx.x % cluster) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const T* __restrict__ LU = reinterpret_cast<const T*>(S.lu) + (size_t)tile * P.NLU * kTile + lane;
  T* X = reinterpret_cast<T*>(S.x) + (size_t)tile * P.mp * kTile + lane;
  const int nl = BWD ? P.n_bw_lvl : P.n_fw_lvl;
  const int32_t* __restrict__ lvl = BWD ? P.bw_lvl_ptr : P.fw_lvl_ptr;
  const int32_t* __restrict__ rows = BWD ? P.bw_rows : P.fw_rows;
  const int32_t* __restrict__ ptr = BWD ? P.bw_ptr : P.fw_ptr;
  const int32_t* __restrict__ pos = BWD ? P.bw_pos : P.fw_pos;
  const int32_t* __restrict__ col = BWD ? P.bw_col : P.fw_col;
  const int total = lvl[nl];
  int nr = 0, ni = 0, ne0 = 0, ne1 = 0, np[4], nc[4];  // the row loaded ahead
  auto fetch = [&](int r) {
    nr = r;
    if (r < total) {
      ni = rows[r];
      ne0 = ptr[r];
      ne1 = ptr[r + 1];
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (ne0 + z < ne1) {
          np[z] = pos[ne0 + z];
          nc[z] = col[ne0 + z];
        }
    }
  };
  fetch(w);
  int r1 = lvl[1], r2 = nl > 1 ? lvl[2] : r1;
  for (int l = 0, r0 = 0; l < nl; ++l) {
    int r = r0 + w;
    if (r >= r1) fetch(r1 + w);
    while (r < r1) {
      if (nr != r) fetch(r);
      const int i = ni, e1 = ne1;
      int e = ne0;
      T acc = X[(size_t)i * kTile], a[4], b[4];
      const T d = BWD ? LU[(size_t)P.dp[i] * kTile] : (T)1;
      const int n0 = min(e1 - e, 4);
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (z < n0) {
          a[z] = LU[(size_t)np[z] * kTile];
          b[z] = X[(size_t)nc[z] * kTile];
        }
      r += W;
      fetch(r < r1 ? r : r1 + w);
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (z < n0) acc -= a[z] * b[z];
      for (e += n0; e + 4 <= e1; e += 4) {
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          a[z] = LU[(size_t)pos[e + z] * kTile];
          b[z] = X[(size_t)col[e + z] * kTile];
        }
#pragma unroll
        for (int z = 0; z < 4; ++z) acc -= a[z] * b[z];
      }
      for (; e < e1; ++e) acc -= LU[(size_t)pos[e] * kTile] * X[(size_t)col[e] * kTile];
      X[(size_t)i * kTile] = BWD ? acc / d : acc;
    }
    r0 = r1;
    r1 = r2;
    if (l + 3 <= nl) r2 = lvl[l + 3];
    level_barrier(cluster);
  }
}

// Dense block solves, one CTA of NW warps per tile (32 instances), the tile's
// right-hand side in shared memory when it fits.  Forward (unit lower) and
// backward (upper) substitution by blocks of SB columns: as soon as a block of
// x is known, warp 0 updates the next block's SB rows and solves them against
// their SB x SB diagonal block, in registers, while the other warps update the
// rows beyond (independent multiply-adds), so that the serial part of a block
// hides behind the rest of it and one barrier per block suffices.  Backward, the
// last warp has the reciprocals of the pivots ready two blocks ahead: an FP64
// division on the serial part costs as much as ten of its multiply-adds.
// Reads the block once (592 KB per instance of the 2,000-bus FP64 plan) and is
// bound by latency and barriers: what matters is loads in flight.  A warp takes
// four rows of a column in FP32 (one 16-byte load per lane), two in FP64, for
// all SB columns at once.  NW: 32 while every tile can have an SM of its own
// (one CTA of 1,024 threads per SM), else 16 (FP64: 10, for its registers) and
// three CTAs per SM.  Measured per
// solve with 8 warps, a row at a time, the diagonal block in between (two
// barriers per block), and in this form:
//   FP64, 272 wide:  1 tile 1.07 -> 0.76 ms, 60 tiles 1.95 -> 0.90 ms, 313 tiles 2.44 -> 2.01 ms
//   FP32, 320 wide: 11 tiles 1.26 -> 0.31 ms, 313 tiles 1.36 -> 0.87 ms
// (FP64: the pipe takes 16 cycles per multiply-add of a warp, 0.6 ms per tile and
// SM.)
template <typename T, int SB, bool SMEM, int NW>
__global__ void __launch_bounds__(32 * NW, NW == 32 ? 1 : 3) k_dense_solve_smem(DevPlan P, DevState S,
                                                                               const int32_t* __restrict__ gate) {
  constexpr int U = DenseGroup<T>::G == 4 ? 4 : 2;  // rows per step of a warp
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T rec[2][SB][kTile];  // reciprocal pivots of two blocks
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x, warp = threadIdx.y;
  const int tile = blockIdx.x;
  if (!__syncthreads_or(S.active[tile * kTile + lane])) return;
  const T* __restrict__ Ab = reinterpret_cast<const T*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile;
  T* __restrict__ X = reinterpret_cast<T*>(S.x) + ((size_t)tile * P.mp + P.s) * kTile + lane;
  const int ld = P.ndp, n = P.nde;
  // rows r .. r+U-1 of column c (r a multiple of U)
  auto ldu = [&](int r, int c, T(&v)[U]) {
    if constexpr (U == 4) {
      ld4(Ab, r, c, ld, lane, v);
    } else {
#pragma unroll
      for (int i = 0; i < U; ++i) v[i] = Ab[dense_off<T>(r + i, c, ld, lane)];
    }
  };
  // the tile's right-hand side: in shared memory when it fits, else in place
  // in global memory (same blocked algorithm, L2-resident per tile)
  T* xs = SMEM ? reinterpret_cast<T*>(smem_raw) : X - lane;  // xs[r * 32 + lane]
  if (SMEM)
    for (int r = warp; r < n; r += NW) xs[r * kTile + lane] = X[(size_t)r * kTile];
  // rows r .. r+U-1 minus the block's columns k0 .. k0+SB-1 times xb
  auto update = [&](int r, int k0, const T(&xb)[SB], T(&acc)[U]) {
#pragma unroll
    for (int i = 0; i < U; ++i) acc[i] = xs[(r + i) * kTile + lane];
#pragma unroll
    for (int c = 0; c < SB; ++c) {
      T v[U];
      ldu(r, k0 + c, v);
#pragma unroll
      for (int i = 0; i < U; ++i) acc[i] -= v[i] * xb[c];
    }
  };
  // warp 0: rows k .. k+SB-1 of the block before (columns k0 .., or none when
  // k0 < 0), then their own diagonal block
  auto head = [&](int k, int k0, const T(&xb)[SB], bool upper) {
    T x[SB];
#pragma unroll
    for (int g = 0; g < SB / U; ++g) {
      T acc[U];
      if (k0 >= 0) {
        update(k + U * g, k0, xb, acc);
      } else {
#pragma unroll
        for (int i = 0; i < U; ++i) acc[i] = xs[(k + U * g + i) * kTile + lane];
      }
#pragma unroll
      for (int i = 0; i < U; ++i) x[U * g + i] = acc[i];
    }
    if (!upper) {
#pragma unroll
      for (int c = 0; c < SB - 1; ++c)
#pragma unroll
        for (int g = (c + 1) / U; g < SB / U; ++g) {
          T v[U];
          ldu(k + U * g, k + c, v);
#pragma unroll
          for (int i = 0; i < U; ++i)
            if (U * g + i > c) x[U * g + i] -= v[i] * x[c];
        }
    } else {
#pragma unroll
      for (int c = SB - 1; c >= 0; --c)
#pragma unroll
        for (int g = c / U; g >= 0; --g) {
          T v[U];
          ldu(k + U * g, k + c, v);
#pragma unroll
          for (int i = U - 1; i >= 0; --i) {
            if (U * g + i == c) x[c] *= rec[(k / SB) & 1][c][lane];
            if (U * g + i < c) x[U * g + i] -= v[i] * x[c];
          }
        }
    }
#pragma unroll
    for (int r = 0; r < SB; ++r) xs[(k + r) * kTile + lane] = x[r];
  };
  auto reciprocals = [&](int k) {
    T d[SB];
#pragma unroll
    for (int c = 0; c < SB; ++c) d[c] = Ab[dense_off<T>(k + c, k + c, ld, lane)];
#pragma unroll
    for (int c = 0; c < SB; ++c) rec[(k / SB) & 1][c][lane] = (T)1 / d[c];
  };
  if (warp == NW - 1) reciprocals(n - SB);
  if (warp == NW - 2 && n > SB) reciprocals(n - 2 * SB);
  T xb[SB];
#pragma unroll
  for (int c = 0; c < SB; ++c) xb[c] = (T)0;
  __syncthreads();
  if (warp == 0) head(0, -1, xb, false);
  __syncthreads();
  for (int k0 = 0; k0 + SB < n; k0 += SB) {
#pragma unroll
    for (int c = 0; c < SB; ++c) xb[c] = xs[(k0 + c) * kTile + lane];
    if (warp == 0) {
      head(k0 + SB, k0, xb, false);
    } else {
      for (int r = k0 + 2 * SB + U * (warp - 1); r < n; r += U * (NW - 1)) {
        T acc[U];
        update(r, k0, xb, acc);
#pragma unroll
        for (int i = 0; i < U; ++i) xs[(r + i) * kTile + lane] = acc[i];
      }
    }
    __syncthreads();
  }
  if (warp == 0) head(n - SB, -1, xb, true);
  __syncthreads();
  for (int k0 = n - SB; k0 > 0; k0 -= SB) {
#pragma unroll
    for (int c = 0; c < SB; ++c) xb[c] = xs[(k0 + c) * kTile + lane];
    if (warp == 0) {
      head(k0 - SB, k0, xb, true);
    } else {
      // block k0's have been used, and block k0 - 2 SB takes their place
      if (warp == NW - 1 && k0 >= 2 * SB) reciprocals(k0 - 2 * SB);
      for (int r = U * (warp - 1); r < k0 - SB; r += U * (NW - 1)) {
        T acc[U];
        update(r, k0, xb, acc);
#pragma unroll
        for (int i = 0; i < U; ++i) xs[(r + i) * kTile + lane] = acc[i];
      }
    }
    __syncthreads();
  }
  if (SMEM)
    for (int r = warp; r < n; r += NW) X[(size_t)r * kTile] = xs[r * kTile + lane];
}

// ---------------------------------------------------------------------------
// Voltage update (Sec. 3, step 4): th[PV+PQ] += dx, |V|[PQ] += dx, then the
// rectangular form and 1/|V| for the next mismatch.  Inactive instances keep
// their voltages.  A non-finite step marks the instance failed.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_update(DevPlan P, DevState S, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x;
  const int tile = blockIdx.y;
  const int i = blockIdx.x * blockDim.y + threadIdx.y;
  if (i >= P.n) return;
  const int b = tile * kTile + lane;
  if (!S.active[b]) return;
  const int bt = P.bus_type[i];
  if (bt == 3) return;
  const T* __restrict__ X = reinterpret_cast<const T*>(S.x) + (size_t)tile * P.mp * kTile + lane;
  const size_t o = sidx(tile, P.n, i, lane);
  const double dth = (double)X[(size_t)P.rhs_p[i] * kTile];
  double va = S.va[o] + dth;
  double vm = S.vm[o];
  bool ok = fabs(dth) <= DBL_MAX;
  if (bt == 1) {
    const double dvm = (double)X[(size_t)P.rhs_q[i] * kTile];
    ok = ok && fabs(dvm) <= DBL_MAX;
    vm += dvm;
  }
  if (!ok) {
    S.bad[b] = 1;
    return;
  }
  double sn, cs;
  sincos(va, &sn, &cs);
  S.va[o] = va;
  S.vm[o] = vm;
  S.ve[o] = vm * cs;
  S.vf[o] = vm * sn;
  S.vinv[o] = 1.0 / vm;
}

// Scatter a user right-hand side [B, m] (J row order) into the permuted rhs,
// and gather the solution back into J column order.
template <typename T>
__global__ void k_rhs_in(DevPlan P, DevState S, int B, const double* __restrict__ rhs) {
  const int lane = threadIdx.x, tile = blockIdx.y;
  const int u = blockIdx.x * blockDim.y + threadIdx.y;
  if (u >= P.m) return;
  const int b = tile * kTile + lane;
  T* X = reinterpret_cast<T*>(S.x) + (size_t)tile * P.mp * kTile + lane;
  X[(size_t)P.unk_pos[u] * kTile] = b < B ? (T)rhs[(size_t)b * P.m + u] : (T)0;
}

template <typename T>
__global__ void k_rhs_out(DevPlan P, DevState S, int B, double* __restrict__ dx) {
  const int lane = threadIdx.x, tile = blockIdx.y;
  const int u = blockIdx.x * blockDim.y + threadIdx.y;
  if (u >= P.m) return;
  const int b = tile * kTile + lane;
  const T* X = reinterpret_cast<const T*>(S.x) + (size_t)tile * P.mp * kTile + lane;
  if (b < B) dx[(size_t)b * P.m + u] = (double)X[(size_t)P.unk_pos[u] * kTile];
}

// F in J row order and the norm, for the mismatch stage entry point.
template <typename T>
__global__ void k_f_out(DevPlan P, DevState S, int B, double* __restrict__ F, double* __restrict__ norm) {
  const int lane = threadIdx.x, tile = blockIdx.y;
  const int u = blockIdx.x * blockDim.y + threadIdx.y;
  const int b = tile * kTile + lane;
  if (b >= B) return;
  if (u < P.m) {
    const T* X = reinterpret_cast<const T*>(S.x) + (size_t)tile * P.mp * kTile + lane;
    F[(size_t)b * P.m + u] = -(double)X[(size_t)P.unk_pos[u] * kTile];
  }
  if (u == 0) norm[b] = __longlong_as_double((long long)S.norm[b]);
}

// LU values of the pattern (CCS order of pf_plan_get_pattern) out to [B, nnz].
template <typename T>
__global__ void k_lu_out(DevPlan P, DevState S, int B, const int64_t* __restrict__ map, int64_t nnz,
                         double* __restrict__ out) {
  const int lane = threadIdx.x, tile = blockIdx.y;
  const int64_t q = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
  if (q >= nnz) return;
  const int b = tile * kTile + lane;
  if (b >= B) return;
  const T* LU = reinterpret_cast<const T*>(S.lu) + (size_t)tile * P.NLU * kTile;
  out[(size_t)b * nnz + q] = (double)LU[lu_off<T>(P, map[q], lane)];
}

}  // namespace

// ---------------------------------------------------------------------------
// Host-side launchers (every launch goes through NRPF_LAUNCH for counting and
// optional per-class CUDA-event timing)
// ---------------------------------------------------------------------------
static inline dim3 grid2(int64_t items, int per_block, int tiles) {
  return dim3((unsigned)((items + per_block - 1) / per_block), (unsigned)tiles);
}

void launch_load(const DevPlan& P, const DevState& S, int B, const double* sbus, const double* v0,
                 cudaStream_t st, Recorder* rec) {
  dim3 g((P.n + 31) / 32, S.Bp / kTile);
  NRPF_LAUNCH(rec, K_LOAD, st,
              k_load<<<g, dim3(32, 8), 0, st>>>(P, S, B, reinterpret_cast<const double2*>(sbus),
                                                reinterpret_cast<const double2*>(v0)));
}

void launch_store(const DevPlan& P, const DevState& S, int B, double* v_out, int32_t* iters,
                  uint8_t* status, cudaStream_t st, Recorder* rec) {
  dim3 g((P.n + 31) / 32, S.Bp / kTile);
  NRPF_LAUNCH(rec, K_STORE, st,
              k_store<<<g, dim3(32, 8), 0, st>>>(P, S, B, reinterpret_cast<double2*>(v_out), iters, status));
}

template <typename T>
void launch_mismatch(const DevPlan& P, const DevState& S, int jac, const int32_t* gate, cudaStream_t st,
                     Recorder* rec) {
  const int tiles = S.Bp / kTile;
  auto blocks = [&](int per) { return (P.n + kMWarps * per - 1) / (kMWarps * per); };
  int per = 8;
  while (per > 1 && (int64_t)blocks(per) * tiles < 4 * 152) per /= 2;
  NRPF_LAUNCH(rec, K_MISMATCH, st,
              k_mismatch_jac<T><<<dim3(blocks(per), tiles), dim3(32, kMWarps), 0, st>>>(P, S, jac, per, gate));
}

void launch_load_y(const DevPlan& P, const DevState& S, int B, const double* y, cudaStream_t st, Recorder* rec) {
  dim3 g((P.nnzY + 31) / 32, S.Bp / kTile);
  NRPF_LAUNCH(rec, K_LOAD, st,
              k_load_y<<<g, dim3(32, 8), 0, st>>>(P.nnzY, B, reinterpret_cast<const double2*>(y),
                                                  const_cast<double2*>(S.yv)));
}

void launch_outage_y(const DevPlan& P, const DevState& S, int B, const int32_t* outages, int k, const int4* bpos,
                     const double* bval, int nbr, cudaStream_t st, Recorder* rec) {
  const int tiles = S.Bp / kTile;
  double2* yv = const_cast<double2*>(S.yv);
  NRPF_LAUNCH(rec, K_LOAD, st,
              k_base_y<<<grid2((int64_t)tiles * P.nnzY, 8, 1), dim3(32, 8), 0, st>>>(P, yv, tiles));
  if (k > 0)
    NRPF_LAUNCH(rec, K_LOAD, st,
                k_outage_y<<<(B + 127) / 128, 128, 0, st>>>(P.nnzY, B, k, outages, bpos, bval, nbr, yv));
}

void launch_ctl_init(const DevState& S, int maxit, double tol, cudaStream_t st, Recorder* rec) {
  NRPF_LAUNCH(rec, K_AUX, st, k_ctl_init<<<1, 1, 0, st>>>(S.ctl, maxit, tol));
}

void launch_check(const DevState& S, cudaStream_t st, Recorder* rec) {
  NRPF_LAUNCH(rec, K_CHECK, st, k_check<<<(S.Bp + 255) / 256, 256, 0, st>>>(S, S.Bp));
}

void launch_iter_tail(const DevState& S, cudaGraphConditionalHandle cond, int graph, cudaStream_t st,
                      Recorder* rec) {
  NRPF_LAUNCH(rec, K_AUX, st, k_iter_tail<<<1, 1, 0, st>>>(S.ctl, cond, graph));
}

template <typename T>
void launch_prepare_lu(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                       Recorder* rec, LuPrep prep) {
  // per tile, NLU * 32 values; the sparse segments are the first NS * 32
  // (both multiples of 128 bytes), the dense block's nd columns follow.
  const size_t stride16 = (size_t)P.NLU * kTile * sizeof(T) / 16;
  const size_t values = prep == LuPrep::kWhole ? (size_t)P.NLU
                        : prep == LuPrep::kSparse  ? (size_t)P.NS
                        : P.dim ? (size_t)P.NLU : (size_t)(P.NS + (int64_t)P.nd * P.ndp);
  const size_t n16 = P.nd == 0 ? stride16 : values * kTile * sizeof(T) / 16;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  NRPF_LAUNCH(rec, K_ZERO, st,
              k_zero16<<<sms * 8, 256, 0, st>>>(reinterpret_cast<uint4*>(S.lu), n16, stride16, S.Bp / kTile, gate));
  if (P.n_one > 0 && prep != LuPrep::kColumns) {
    if (sizeof(T) == 4 && P.dim)
      launch_dense_im_set_ones(P, S, gate, st, rec);
    else if (P.nde > P.nd)
      NRPF_LAUNCH(rec, K_ONES, st, k_set_ones<T><<<dim3(P.nde - P.nd, S.Bp / kTile), dim3(32, 8), 0, st>>>(P, S, gate));
  }
}

// one panel step of width KB at column k.  The column part of the panel
// covers columns < cend; the update covers the trailing block's columns
// [r0, kend) and, for rows [r0, kend), columns [kend, cend)
// (kend = cend = ld: the whole trailing block).
template <typename T, int KB>
static void launch_dense_step(const DevPlan& P, const DevState& S, int k, int kend, int cend, const int32_t* gate,
                              cudaStream_t st, Recorder* rec) {
  const int tiles = S.Bp / kTile;
  const int rows = P.ndp - k - KB;
  if constexpr (KB == 16)
    NRPF_LAUNCH(rec, K_DENSE_DIAG, st, k_dense_diag16<T><<<tiles, dim3(32, kDiagWarps), 0, st>>>(P, S, k, gate));
  else
    NRPF_LAUNCH(rec, K_DENSE_DIAG, st,
                k_dense_diag<T, KB><<<(tiles + 3) / 4, dim3(32, 4), 0, st>>>(P, S, k, gate));
  if (rows > 0) {
    const int cols = cend - k - KB;
    NRPF_LAUNCH(rec, K_DENSE_PANEL, st,
                k_dense_panel<T, KB><<<grid2(rows / 4 + cols / 4, 4, tiles), dim3(32, 4), 0, st>>>(P, S, k, cend,
                                                                                                  gate));
    // register tile: 4 x 4 for FP64 (the FP64 pipe is the bound), 8 x 8 for
    // FP32 (halves the loads per multiply-add; FP32 is load-bound)
    constexpr int TS = (sizeof(T) == 4 && KB >= 8) ? 8 : 4;
    const int64_t nk = (kend - k - KB) / TS;
    const int64_t ntiles = (rows / TS) * nk + nk * ((cend - kend) / TS);
    if (ntiles > 0) {
      NRPF_LAUNCH(rec, K_DENSE_UPDATE, st,
                  k_dense_update<T, KB, TS><<<grid2(ntiles, 4, tiles), dim3(32, 4), 0, st>>>(P, S, k, kend, cend,
                                                                                            gate));
    }
  }
}

// FP64, outer panel of width KBO (two-level blocking): 16-wide steps factorise the
// outer panel's columns and its rows to the right (U12), each step updating
// only that L-shaped region; then one trailing update of depth KBO (one pass
// over the trailing block per KBO columns instead of per 16).
template <typename T, int KBO>
static void launch_dense_outer(const DevPlan& P, const DevState& S, int k, const int32_t* gate, cudaStream_t st,
                               Recorder* rec) {
  const int tiles = S.Bp / kTile;
  for (int ki = k; ki < k + KBO; ki += 16) launch_dense_step<T, 16>(P, S, ki, k + KBO, P.ndp, gate, st, rec);
  const int rest = P.ndp - k - KBO;
  if (rest > 0) {
    constexpr int TS = 4;
    NRPF_LAUNCH(rec, K_DENSE_UPDATE, st,
                k_dense_update<T, KBO, TS><<<grid2((int64_t)(rest / TS) * (rest / TS), 4, tiles), dim3(32, 4), 0,
                                             st>>>(P, S, k, P.ndp, P.ndp, gate));
  }
}

// one of the level kernels, a cluster per tile
template <typename K>
static void launch_levels(K kernel, int cls, const DevPlan& P, const DevState& S, int tasks, int levels,
                          const int32_t* gate, cudaStream_t st, Recorder* rec) {
  const int tiles = S.Bp / kTile;
  const LevelShape sh = level_shape(tiles, tasks, levels);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * sh.cluster));
  cfg.blockDim = dim3((unsigned)sh.threads);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)sh.cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = sh.cluster > 1 ? 1 : 0;
  NRPF_LAUNCH(rec, cls, st, cudaLaunchKernelEx(&cfg, kernel, P, S, sh.cluster, gate));
}

template <typename T>
void launch_factor(const DevPlan& P, const DevState& S, const std::vector<int32_t>& lvl_ptr,
                   const int32_t* gate, cudaStream_t st, Recorder* rec, bool dense) {
  const int tiles = S.Bp / kTile;
  if (P.n_fac_lvl > 0 && S.dinv && (sizeof(T) == 4 || tiles <= kEntryTiles64))
    launch_levels(k_sparse_factor<T>, K_LU_SPARSE, P, S, P.n_fac_task, P.n_fac_lvl, gate, st, rec);
  else for (size_t l = 0; l + 1 < lvl_ptr.size(); ++l) {
    int c0 = lvl_ptr[l], c1 = lvl_ptr[l + 1];
    if (c1 <= c0) continue;
    NRPF_LAUNCH(rec, K_LU_SPARSE, st,
                k_lu_sparse_level<T><<<grid2(c1 - c0, kLWarps, tiles), dim3(32, kLWarps), 0, st>>>(P, S, c0, c1,
                                                                                                  gate));
  }
  if (P.n_schur > 0)
    NRPF_LAUNCH(rec, K_SCHUR, st,
                k_schur<T><<<grid2(P.n_schur, kSchurWarps, tiles), dim3(32, kSchurWarps), 0, st>>>(P, S, gate));
  if (!dense) return;
  if constexpr (sizeof(T) == 4) {
    if (P.dim) {
      if (P.ndp > 0) launch_dense_im_factor(P, S, *reinterpret_cast<const DenseImMaps*>(S.im_maps), gate, st, rec);
      return;
    }
    if (P.kb >= 16) {  // narrower panels only where a plan asks for them
      launch_dense_il_factor(P, S, gate, st, rec);
      return;
    }
  }
  if constexpr (sizeof(T) == 8) {
    if (S.limb && P.kb == 8) {
      // two panels of eight, then one trailing update of depth 16
      static bool configured[64] = {};
      int dev = 0;
      cudaGetDevice(&dev);
      if (dev < 0 || dev >= 64 || !configured[dev]) {
        cudaFuncSetAttribute(k_dense_update_fixed, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFixSmem);
        if (dev >= 0 && dev < 64) configured[dev] = true;
      }
      for (int k = 0; k < P.ndp; k += kFixK) {
        const int rest = P.ndp - k - kFixK, kend = std::min(k + kFixK, P.ndp);
        for (int ki = k; ki < kend; ki += 8) launch_dense_step<T, 8>(P, S, ki, kend, P.ndp, gate, st, rec);
        if (rest <= 0) continue;
        NRPF_LAUNCH(rec, K_DENSE_UPDATE, st,
                    k_dense_limbs<<<grid2(rest, 4, tiles), dim3(32, 4), 0, st>>>(P, S, k, gate));
        NRPF_LAUNCH(rec, K_DENSE_UPDATE, st,
                    k_dense_update_fixed<<<dim3((unsigned)(((rest / 4 + kFixWR - 1) / kFixWR) *
                                                           ((rest / 4 + kFixWC - 1) / kFixWC)),
                                                (unsigned)tiles),
                                           dim3(32, kFixWR * kFixWC), kFixSmem, st>>>(P, S, k, gate));
      }
      return;
    }
  }
  for (int k = 0; k < P.ndp; k += P.kb) {
    if (P.kb == 4) launch_dense_step<T, 4>(P, S, k, P.ndp, P.ndp, gate, st, rec);
    else if (P.kb == 8) launch_dense_step<T, 8>(P, S, k, P.ndp, P.ndp, gate, st, rec);
    if constexpr (sizeof(T) == 8) {
      if (P.kb == 16) launch_dense_step<T, 16>(P, S, k, P.ndp, P.ndp, gate, st, rec);
      else if (P.kb == 32) launch_dense_outer<T, 32>(P, S, k, gate, st, rec);
      else if (P.kb == 64) launch_dense_outer<T, 64>(P, S, k, gate, st, rec);
    }
  }
}

size_t dense_limb_bytes(const DevPlan& P, int Bp) { return limb_vecs(P.ndp) * sizeof(int4) * (size_t)(Bp / kTile); }

// Dense solve with the tile's right-hand side in shared memory, when it fits.
constexpr size_t kSolveSmemMax = 200 * 1024;

template <typename T, int SB, int NW>
static void launch_dense_solve_nw(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                                  Recorder* rec, size_t smem) {
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_dense_solve_smem<T, SB, true, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)kSolveSmemMax);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  if (smem <= kSolveSmemMax)
    NRPF_LAUNCH(rec, K_DENSE_SOLVE, st,
                k_dense_solve_smem<T, SB, true, NW><<<S.Bp / kTile, dim3(32, NW), smem, st>>>(P, S, gate));
  else
    NRPF_LAUNCH(rec, K_DENSE_SOLVE, st,
                k_dense_solve_smem<T, SB, false, NW><<<S.Bp / kTile, dim3(32, NW), 0, st>>>(P, S, gate));
}

template <typename T, int SB>
static void launch_dense_solve_smem(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                                    Recorder* rec, size_t smem) {
  if (S.Bp / kTile <= 152)
    launch_dense_solve_nw<T, SB, 32>(P, S, gate, st, rec, smem);
  else
    launch_dense_solve_nw<T, SB, (sizeof(T) == 8 ? 10 : 16)>(P, S, gate, st, rec, smem);
}

template <typename T>
void launch_solve(const DevPlan& P, const DevState& S, const std::vector<int32_t>& fw_lvl,
                  const std::vector<int32_t>& bw_lvl, const int32_t* gate, cudaStream_t st, Recorder* rec,
                  bool dense) {
  if (P.n_fw_lvl > 0) launch_levels(k_subst<T, false>, K_FWD, P, S, fw_lvl.back(), P.n_fw_lvl, gate, st, rec);
  if (!dense) {
    launch_dense_cluster<T>(P, S, gate, st, rec);
  } else if (sizeof(T) == 4 && P.dim) {
    if (P.ndp > 0) launch_dense_im_solve(P, S, gate, st, rec);
  } else if (P.ndp > 0) {
    const size_t smem = (size_t)P.nde * kTile * sizeof(T);
    if (P.nde % 8 == 0)
      launch_dense_solve_smem<T, 8>(P, S, gate, st, rec, smem);
    else
      launch_dense_solve_smem<T, 4>(P, S, gate, st, rec, smem);
  }
  if (P.n_bw_lvl > 0) launch_levels(k_subst<T, true>, K_BWD, P, S, bw_lvl.back(), P.n_bw_lvl, gate, st, rec);
}

template <typename T>
void launch_update(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st, Recorder* rec) {
  NRPF_LAUNCH(rec, K_UPDATE, st, k_update<T><<<grid2(P.n, 8, S.Bp / kTile), dim3(32, 8), 0, st>>>(P, S, gate));
}

template <typename T>
void launch_rhs_in(const DevPlan& P, const DevState& S, int B, const double* rhs, cudaStream_t st) {
  cudaMemsetAsync(S.x, 0, (size_t)P.mp * S.Bp * sizeof(T), st);
  if (P.m > 0) k_rhs_in<T><<<grid2(P.m, 8, S.Bp / kTile), dim3(32, 8), 0, st>>>(P, S, B, rhs);
}

template <typename T>
void launch_rhs_out(const DevPlan& P, const DevState& S, int B, double* dx, cudaStream_t st) {
  if (P.m > 0) k_rhs_out<T><<<grid2(P.m, 8, S.Bp / kTile), dim3(32, 8), 0, st>>>(P, S, B, dx);
}

template <typename T>
void launch_f_out(const DevPlan& P, const DevState& S, int B, double* F, double* norm, cudaStream_t st) {
  k_f_out<T><<<grid2(P.m > 0 ? P.m : 1, 8, S.Bp / kTile), dim3(32, 8), 0, st>>>(P, S, B, F, norm);
}

template <typename T>
void launch_lu_out(const DevPlan& P, const DevState& S, int B, const int64_t* map, int64_t nnz, double* out,
                   cudaStream_t st) {
  if (nnz > 0) k_lu_out<T><<<grid2(nnz, 8, S.Bp / kTile), dim3(32, 8), 0, st>>>(P, S, B, map, nnz, out);
}

#define NRPF_INST(T)                                                                                          \
  template void launch_mismatch<T>(const DevPlan&, const DevState&, int, const int32_t*, cudaStream_t,       \
                                   Recorder*);                                                               \
  template void launch_prepare_lu<T>(const DevPlan&, const DevState&, const int32_t*, cudaStream_t,          \
                                     Recorder*, LuPrep);                                                     \
  template void launch_factor<T>(const DevPlan&, const DevState&, const std::vector<int32_t>&,               \
                                 const int32_t*, cudaStream_t, Recorder*, bool);                             \
  template void launch_solve<T>(const DevPlan&, const DevState&, const std::vector<int32_t>&,                \
                                const std::vector<int32_t>&, const int32_t*, cudaStream_t, Recorder*, bool); \
  template void launch_update<T>(const DevPlan&, const DevState&, const int32_t*, cudaStream_t, Recorder*);  \
  template void launch_rhs_in<T>(const DevPlan&, const DevState&, int, const double*, cudaStream_t);         \
  template void launch_rhs_out<T>(const DevPlan&, const DevState&, int, double*, cudaStream_t);              \
  template void launch_f_out<T>(const DevPlan&, const DevState&, int, double*, double*, cudaStream_t);       \
  template void launch_lu_out<T>(const DevPlan&, const DevState&, int, const int64_t*, int64_t, double*,     \
                                 cudaStream_t);

NRPF_INST(double)
NRPF_INST(float)

}  // namespace nrpf
