// One CTA solves J dx = -F for a few instances of a small plan, start to end, in
// shared memory: the LU of all columns (sparse and dense alike), the forward
// substitution, which is the LU's schedule with the right-hand side as one more
// column, and the backward substitution (Sec. 4.3; plan.h: sm_*).
//
// On a 30-bus grid the work of a step is a few thousand multiply-adds, but its
// schedules are 17 + 17 + 16 dependent levels and a dense tail: as launches 60
// per iteration, as kernels that walk the levels over global memory still about
// 2 us a level (the chain of an L2 round trip, a store and a barrier).  Here a
// level costs a shared-memory read, a chain of FMAs and __syncthreads: 30 buses x
// 64 in FP64, LU, dense tail and substitutions of an iteration 163 -> 75 us (65
// levels; an FP64 multiply-add of a warp holds its quarter of the SM for 64
// cycles, a division for 350).
//
// When: batches whose CTAs, one per SM, are one wave, and plans and precisions for
// which this then is the faster form.  A second wave takes as long as the first, where
// the level kernels' time grows by a quarter; only FP64 plans of few values and many
// levels are the faster ones still in the second: 45 to 50 buses x 3,200, level kernels /
// this kernel, us: 1,001 values, 19 levels 1,069 / 911; 1,092, 25: 1,242 / 1,101; but 1,049,
// 12: 866 / 922; 940, 12: 923 / 925.  Solves by the level kernels / by this kernel, us
// (buses, values, dense columns: instances):
//   FP64  30, 675, 12:     64: 695 / 391   1,216: 810 / 401     2,432: 851 / 458
//   FP64  40, 918, 12:     4,864: 1,143 / 1,066 (two waves)   8,000: 1,486 / 1,982
//   FP64  100, 2,424, 23:  64: 811 / 760   1,216: 1,054 / 856   2,432: 1,188 / 1,567   10,000: 2,843 / 6,742
//   FP32  40, 1,062, 20:   64: 603 / 502   2,432: 708 / 579     10,000: 1,262 / 1,889
//   FP32  55, 1,576, 25:   64: 483 / 632   1,216: 544 / 670     10,000: 1,215 / 2,451
// In FP32 the level kernels are the faster ones beyond 1,200 values, and where the
// dense tail, a chain of levels per column here, has more than 20 columns (30 buses,
// 929 values, 22: 64 instances 409 / 486).
// The smallest plans (30 buses: 675 values in FP64, 771 in FP32) keep to this kernel in
// every batch, so that their results do not depend on it, bit for bit: of the sizes up
// to 10,000 all are at least as fast as with a launch per level (10,000: 1,442 us FP64,
// 2,435 FP32), where the level kernels take 1,225 / 1,432 and 932 / 1,472.
//
// Layout: value v of instance i of the CTA at v * S + i, S = 8, 16 or 32 instances
// per CTA: the fewest with which the batch's CTAs are one wave (2,432 instances, 30
// buses: 16 of them 458 us in one wave).  A warp is
// 32 / S workers of S lanes (lane = instance); a worker takes a task, one entry:
// its operations come with coalesced loads of S at a time, ahead of the barrier,
// and are handed out by shuffles; the entry stays in a register and takes its
// products in ascending k, as in the other kernels.
#include "small_solve.h"

#include "kernels.h"

namespace nrpf {

namespace {

constexpr size_t kSmallSmem = 200 * 1024;
constexpr size_t kSmallValuesFp32 = 1200;
constexpr int kSmallDenseFp32 = 20;
// values per level of the sparse LU up to which a plan keeps to the kernel in a second
// wave, and values up to which it always does
constexpr size_t kSmallPerLevel64 = 60;
constexpr size_t kSmallAlways64 = 700, kSmallAlways32 = 800;
constexpr int kSmallThreads = 512;

template <typename T, int S, bool OPS>
__global__ void __launch_bounds__(kSmallThreads) k_small_solve(DevPlan P, DevState st, int nval,
                                                               const int32_t* __restrict__ gate) {
  extern __shared__ __align__(16) unsigned char small_smem[];
  if (gate && *gate == 0) return;
  T* val = reinterpret_cast<T*>(small_smem);
  constexpr int kParts = kTile / S;
  const int tile = blockIdx.x / kParts, first = (blockIdx.x % kParts) * S;  // first lane of the tile served here
  const int lane = threadIdx.x & 31, i = lane & (S - 1);
  const int W = (kSmallThreads / 32) * kParts;
  const int w = (threadIdx.x >> 5) * kParts + lane / S;
  if (!__syncthreads_or(st.active[tile * kTile + first + i])) return;
  const T* __restrict__ LU = reinterpret_cast<const T*>(st.lu) + (size_t)tile * P.NLU * kTile;
  T* __restrict__ X = reinterpret_cast<T*>(st.x) + (size_t)tile * P.mp * kTile + first + i;
  const int NS = (int)P.NS, nd = P.nd, vx = nval - 2 * P.m;
  for (int v = w; v < NS; v += W) val[v * S + i] = LU[(size_t)v * kTile + first + i];
  for (int q = w; q < nd * nd; q += W)
    val[(NS + q) * S + i] = LU[lu_off<T>(P, (int64_t)NS + (q / nd) * P.ndp + q % nd, first + i)];
  for (int v = w; v < P.m; v += W) val[(vx + v) * S + i] = X[(size_t)v * kTile];
  const int32_t* __restrict__ lvl = P.sm_lvl_ptr;
  const int total = lvl[P.n_sm_lvl];
  const int32_t* __restrict__ task = P.sm_task;
  const int2* __restrict__ ops = P.sm_op;
  if (OPS) {
    // the schedule too
    int2* so = reinterpret_cast<int2*>(val + (size_t)nval * S);
    const int nops = P.n_sm_op;
    int32_t* ts = reinterpret_cast<int32_t*>(so + nops);
    for (int q = threadIdx.x; q < nops; q += kSmallThreads) so[q] = P.sm_op[q];
    for (int q = threadIdx.x; q <= total; q += kSmallThreads) ts[q] = P.sm_task[q];
    task = ts;
    ops = so;
    __syncthreads();
  }
  int nq0 = 0, nq1 = 0;  // the task loaded ahead: its operations, S of them in nop
  int2 nop = make_int2(0, 0);
  auto fetch = [&](int t) {
    if (t < total) {
      nq0 = task[t];
      nq1 = task[t + 1];
      nop = ops[min(nq0 + i, nq1 - 1)];
    } else {
      nq0 = nq1 = 0;
    }
  };
  // every lane of the warp runs the same rounds (the shuffles need them all):
  // workers without a task in a round have no operations
  fetch(w);
  int t1 = lvl[1], t2 = P.n_sm_lvl > 1 ? lvl[2] : t1;
  __syncthreads();
  for (int l = 0, t0 = 0; l < P.n_sm_lvl; ++l) {
    for (int t = t0 + w, tw = t0 + w - lane / S; tw < t1; t += W, tw += W) {
      const bool mine = t < t1;
      const int q0 = nq0, cnt = mine ? nq1 - nq0 : 0;
      int2 op = nop;
      if (mine) fetch(t + W < t1 ? t + W : t1 + w);
      T acc = (T)0, b0 = (T)0;
      int head = 0, col = 0;
      for (int c = 0; __any_sync(0xffffffffu, c < cnt); c += 8) {
        if (c > 0 && c % S == 0) op = c < cnt ? ops[q0 + min(c + i, cnt - 1)] : op;
        T a[8], b[8];
#pragma unroll
        for (int z = 0; z < 8; ++z) {
          const int x = __shfl_sync(0xffffffffu, op.x, (c + z) % S, S), y = __shfl_sync(0xffffffffu, op.y, (c + z) % S, S);
          const bool on = c + z < cnt;
          if (z == 0 && c == 0) {
            head = x;
            col = y;
          }
          a[z] = on ? val[(x >> 2) * S + i] : (T)0;
          // the entry's own value first (for an L entry or a backward row with
          // the inverse pivot that scales it at the end), then its products
          b[z] = on && ((x & 3) == 0 || (x & 3) == 2) ? val[y * S + i] : (T)0;
        }
#pragma unroll
        for (int z = 0; z < 8; ++z) {
          if (z == 0 && c == 0) {
            acc = a[0];
            b0 = b[0];
          } else {
            acc -= a[z] * b[z];
          }
        }
      }
      if (cnt > 0) {
        const int kind = head & 3;
        if (kind == 2) acc *= b0;
        if (kind == 3) val[col * S + i] = (T)1 / acc;
        val[(head >> 2) * S + i] = acc;
      }
    }
    if (t0 + w >= t1) fetch(t1 + w);
    t0 = t1;
    t1 = t2;
    if (l + 3 <= P.n_sm_lvl) t2 = lvl[l + 3];
    __syncthreads();
  }
  for (int v = w; v < P.m; v += W) X[(size_t)v * kTile] = val[(vx + v) * S + i];
}

template <typename T, int S, bool OPS>
void launch(const DevPlan& P, const DevState& st, int nval, size_t smem, const int32_t* gate, cudaStream_t s,
            Recorder* rec) {
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_small_solve<T, S, OPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  NRPF_LAUNCH(rec, K_LU_SPARSE, s,
              k_small_solve<T, S, OPS><<<(unsigned)(st.Bp / S), kSmallThreads, smem, s>>>(P, st, nval, gate));
}

template <typename T, int S>
void launch_for(const DevPlan& P, const DevState& st, int nval, const int32_t* gate, cudaStream_t s, Recorder* rec) {
  const size_t values = (size_t)nval * S * sizeof(T);
  const size_t ops = (size_t)P.n_sm_op * sizeof(int2) + ((size_t)P.n_sm_task + 1) * sizeof(int32_t);
  if (values + ops <= kSmallSmem) launch<T, S, true>(P, st, nval, values + ops, gate, s, rec);
  else launch<T, S, false>(P, st, nval, values, gate, s, rec);
}

static_assert(kSmallAlways64 * 32 * 8 <= kSmallSmem && kSmallAlways32 * 32 * 4 <= kSmallSmem, "32 instances fit");

}  // namespace

bool small_solve_fits(const HostPlan& h, size_t width) {
  const size_t nval = (size_t)(h.NS + (int64_t)h.nd * h.nd + 2 * (int64_t)h.m);
  return h.sm_lvl_ptr.size() > 1 && nval * 8 * width <= kSmallSmem &&
         (width == 8 || (nval <= kSmallValuesFp32 && h.nd <= kSmallDenseFp32));
}

int small_solve_instances(const DevPlan& P, int Bp, size_t width) {
  if (P.n_sm_lvl == 0) return 0;
  const size_t nval = (size_t)(P.NS + (int64_t)P.nd * P.nd) + 2 * (size_t)P.m;
  int s = 4;
  while (s < 32 && nval * 2 * s * width <= kSmallSmem) {
    s *= 2;
    if (Bp / s <= P.sms) return s;
  }
  // s: the most that fit
  if (width == 8 && nval <= kSmallPerLevel64 * P.n_lu_lvl && Bp / s <= 2 * P.sms) return s;
  return nval <= (width == 8 ? kSmallAlways64 : kSmallAlways32) ? s : 0;
}

template <typename T>
void launch_small_solve(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st, Recorder* rec) {
  const int nval = (int)(P.NS + (int64_t)P.nd * P.nd) + 2 * P.m;
  const int s = small_solve_instances(P, S.Bp, sizeof(T));
  if (s == 32) launch_for<T, 32>(P, S, nval, gate, st, rec);
  else if (s == 16) launch_for<T, 16>(P, S, nval, gate, st, rec);
  else if (s == 8) launch_for<T, 8>(P, S, nval, gate, st, rec);
}

template void launch_small_solve<float>(const DevPlan&, const DevState&, const int32_t*, cudaStream_t, Recorder*);
template void launch_small_solve<double>(const DevPlan&, const DevState&, const int32_t*, cudaStream_t, Recorder*);

}  // namespace nrpf
