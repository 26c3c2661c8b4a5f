// Branch power flows after a solve (pf_branch_flows): the power entering each
// branch at its two ends, from the solved bus voltages.
#include <cuda_runtime.h>

#include "../../include/nrpf.h"

namespace {

// A thread owns one branch and walks over a group of instances: the branch's
// admittance (two FP64 divisions, each about ten FMAs of an FP64 pipe that runs
// at two per SM and clock) is formed once and kept in registers.  The threads are
// numbered through the branches of the first group, then of the next, so that no
// lane is idle whatever the number of branches (an FP64 instruction takes the same
// time with one lane as with 32), at the price of one integer division per thread.
// Branches are fastest, so the flow writes are coalesced; the two voltage reads are
// gathers from the instance's row, which stays in L1/L2 while its branches read it.
// pi model: ys = 1/(r + jx), half the charging b at each end;
// I_f = ys (V_f - V_t) + j b/2 V_f, S_f = V_f conj(I_f), and symmetrically at t.
// Bound: 18 FP64 operations per branch and instance (0.74 ms for 2,600 branches
// x 10,000 instances at the FP64 peak; the bytes alone take 0.17 ms): measured
// 0.88 ms there.  With one thread per (branch, instance), which divided for
// each, it took 1.73 ms; 1,000 buses x 10,000 0.91, now 0.48.  A block of 256
// threads along the branches, of which only 41 exist on a 30-bus grid, took 22.6 us
// on 5,000 instances of it and 36.3 on 10,000; a thread per branch and instance 19.9
// and 33.5, this form 19.8 and 24.8.
constexpr int kThreads = 256;

__global__ void __launch_bounds__(kThreads) k_branch_flows(
    int n, int nbr, const int32_t* __restrict__ f, const int32_t* __restrict__ t, const double* __restrict__ r,
    const double* __restrict__ x, const double* __restrict__ b, int B, int per, unsigned long long total,
    const uint8_t* __restrict__ in_service, const double2* __restrict__ v, double2* __restrict__ sf,
    double2* __restrict__ st) {
  const unsigned long long idx = (unsigned long long)blockIdx.x * kThreads + threadIdx.x;
  if (idx >= total) return;  // total: branches x groups
  const long long g = total >> 32 ? (long long)(idx / (unsigned)nbr) : (long long)((unsigned)idx / (unsigned)nbr);
  const int e = (int)(idx - (unsigned long long)g * (unsigned)nbr);
  const int ef = f[e], et = t[e];
  const double den = r[e] * r[e] + x[e] * x[e];
  const double gs = r[e] / den, bs = -x[e] / den, bh = 0.5 * b[e];
  const int i0 = (int)(g * per), i1 = B - i0 < per ? B : i0 + per;
#pragma unroll 4
  for (int i = i0; i < i1; ++i) {
    const size_t q = (size_t)i * nbr + e;
    if (in_service && !in_service[q]) {
      sf[q] = make_double2(0.0, 0.0);
      st[q] = make_double2(0.0, 0.0);
      continue;
    }
    const double2 vf = v[(size_t)i * n + ef], vt = v[(size_t)i * n + et];
    const double dr = vf.x - vt.x, di = vf.y - vt.y;
    // I_f = ys (V_f - V_t) + j bh V_f
    const double ifr = gs * dr - bs * di - bh * vf.y;
    const double ifi = gs * di + bs * dr + bh * vf.x;
    // I_t = -ys (V_f - V_t) + j bh V_t
    const double itr = -(gs * dr - bs * di) - bh * vt.y;
    const double iti = -(gs * di + bs * dr) + bh * vt.x;
    // S = V conj(I)
    sf[q] = make_double2(vf.x * ifr + vf.y * ifi, vf.y * ifr - vf.x * ifi);
    st[q] = make_double2(vt.x * itr + vt.y * iti, vt.y * itr - vt.x * iti);
  }
}

// Instances per group, up to 16.  A thread's FP64 work is that of two divisions, 37
// operations, and 18 per instance, and the SM with the most blocks ends last: the
// group that makes this least, with at least three blocks per SM, which covers the
// latency of the gathers, or single instances.
constexpr int kPerGroup = 16;
constexpr long long kSms = 152;

int instances_per_group(int B, int nbr) {
  int best = 1;
  long long least = 0;
  for (int per = 1; per <= kPerGroup; ++per) {
    const long long blocks = (((long long)B + per - 1) / per * nbr + kThreads - 1) / kThreads;
    if (per > 1 && blocks < 3 * kSms) break;
    const long long cost = (blocks + kSms - 1) / kSms * (37 + 18 * per);
    if (per == 1 || cost < least) {
      best = per;
      least = cost;
    }
  }
  return best;
}

}  // namespace

extern "C" int pf_branch_flows(int n, int nbr, const int32_t* f, const int32_t* t, const double* r,
                               const double* x, const double* b, int B, const uint8_t* in_service,
                               const double* v, double* sf, double* st, void* stream) {
  if (n <= 0 || nbr < 0 || B < 0) return NRPF_ERR_ARG;
  if ((long long)B * nbr == 0) return NRPF_OK;
  if (!f || !t || !r || !x || !b || !v || !sf || !st) return NRPF_ERR_ARG;
  if (((long long)B * nbr + kThreads - 1) / kThreads > 0x7fffffffLL) return NRPF_ERR_ARG;
  const int per = instances_per_group(B, nbr);
  const unsigned long long total = (unsigned long long)(((long long)B + per - 1) / per) * (unsigned)nbr;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  k_branch_flows<<<(unsigned)((total + kThreads - 1) / kThreads), kThreads, 0, s>>>(
      n, nbr, f, t, r, x, b, B, per, total, in_service, reinterpret_cast<const double2*>(v),
      reinterpret_cast<double2*>(sf), reinterpret_cast<double2*>(st));
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}
