// LU and substitutions of one instance's dense block by one cluster of CTAs, the
// block in their shared memory throughout (Sec. 4.3's dense tail, for small
// batches).
//
// The tile-wide kernels give every lane of a warp an instance.  With one instance
// 31 lanes work for nothing, which an FP64 instruction (64 cycles of a quarter SM,
// whatever its lanes do) makes expensive, and the block's 34 panels are 102
// launches.  Here the lanes are rows and the instance has eight SMs:
//  * blocks of eight columns are dealt to the CTAs in turn; CTA 0 also keeps the
//    right-hand side, which takes the same operations as a column;
//  * per block: its CTA factorises the panel (8 x 8 in one warp, then a row per
//    thread), the cluster's barrier, every CTA copies the panel from that CTA's
//    shared memory and updates its own columns to the right (a row and eight
//    columns per thread);
//  * backward: the right-hand side travels with the blocks, last to first: a
//    block's CTA takes it from the one before, solves its eight unknowns and
//    updates the rows above.
// The 272-wide FP64 block of the 2,000-bus grid, one instance, LU and solves of an
// iteration: 2.3 ms by the tile-wide kernels, 0.6 here; bound by the FP64 pipe of
// the eight SMs (0.22 ms), the serial panels and 68 cluster barriers.
#include "dense_cluster.h"

namespace nrpf {

namespace {

constexpr int kClu = 8;         // CTAs per cluster (the portable maximum)
constexpr int kCluThreads = 512;
constexpr int kCluNb = 8;       // columns per block
constexpr size_t kCluSmem = 220 * 1024;
// When: a block of an instance takes its time in every round of resident clusters, the
// tile-wide kernels theirs per tile, and clusters that share an SM slow each other.  So
// FP64 up to 64 instances and two rounds (a cluster's FP64 work alone is far less than
// a tile's), FP32 up to one round and 32 instances, or 64 of blocks up to 192 wide.
// Solves, tile-wide kernels / clusters, ms (width of the block: instances):
//   FP64  400:  1: 20.0 / 12.6   16: 20.0 / 17.7   32: 20.0 / 23.1   64: 23.1 / 35.6
//         280:  1: 11.3 / 6.76   32: 11.3 / 7.64   64: 12.3 / 11.3
//   FP32  576:  8: 4.99 / 4.58   16: 5.11 / 6.66   32: 5.27 / 8.75   64: 6.78 / 13.9
//         448:  8: 3.68 / 3.10   16: 3.72 / 4.41   32: 3.79 / 5.74   64: 4.24 / 8.63
//         320:  1: 2.80 / 2.32   32: 2.85 / 2.44   48: 2.98 / 3.24   64: 3.00 / 3.39
//         176:  1: 2.03 / 1.63   32: 2.03 / 1.66   64: 2.06 / 2.04
constexpr int kCluInstances = 64, kCluRounds64 = 2;
constexpr int kCluInstances32Wide = 32, kCluWide32 = 192;

// dynamic shared memory of a CTA: its columns, the current panel, the right-hand
// side, the inverse pivots of its columns
size_t clu_smem(int ld, size_t w) {
  const int nblk = ld / kCluNb, nl = (nblk + kClu - 1) / kClu;
  return ((size_t)nl * kCluNb * ld + (size_t)kCluNb * ld + ld + (size_t)nl * kCluNb) * w;
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// value at `p` (an address in this CTA's shared memory) of the cluster's CTA `rank`
__device__ __forceinline__ float remote(const float* p, uint32_t rank) {
  uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p)), r;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(r) : "memory");
  return v;
}
__device__ __forceinline__ double remote(const double* p, uint32_t rank) {
  uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p)), r;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
  return v;
}

template <typename T>
__global__ void __launch_bounds__(kCluThreads) k_dense_cluster(DevPlan P, DevState S,
                                                               const int32_t* __restrict__ gate) {
  extern __shared__ __align__(16) unsigned char clu_raw[];
  if (gate && *gate == 0) return;
  const int b = blockIdx.x / kClu, rank = blockIdx.x % kClu;
  if (!S.active[b]) return;  // uniform over the cluster
  const int ld = P.nde, nblk = ld / kCluNb, nl = (nblk + kClu - 1) / kClu;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int W = kCluThreads / 32;
  T* A = reinterpret_cast<T*>(clu_raw);            // [nl * 8 columns][ld]
  T* Lp = A + (size_t)nl * kCluNb * ld;            // [8][ld] the current panel
  T* y = Lp + (size_t)kCluNb * ld;                 // [ld] the right-hand side
  T* inv = y + ld;                                 // [nl * 8] inverse pivots of this CTA's columns
  const T* __restrict__ G = reinterpret_cast<const T*>(S.lu) + (size_t)(b >> 5) * P.NLU * kTile;
  T* __restrict__ X = reinterpret_cast<T*>(S.x) + ((size_t)(b >> 5) * P.mp + P.s) * kTile + (b & 31);
  for (int lb = 0; lb * kClu + rank < nblk; ++lb)
    for (int q = tid; q < kCluNb * ld; q += kCluThreads) {
      const int c = (lb * kClu + rank) * kCluNb + q / ld, r = q % ld;
      A[(size_t)lb * kCluNb * ld + q] = G[lu_off<T>(P, P.NS + (int64_t)c * P.ndp + r, b & 31)];
    }
  if (rank == 0)
    for (int r = tid; r < ld; r += kCluThreads) y[r] = X[(size_t)r * kTile];
  __syncthreads();
  for (int kb = 0; kb < nblk; ++kb) {
    const int k0 = kb * kCluNb, r0 = k0 + kCluNb, own = kb % kClu;
    T* pan = A + (size_t)(kb / kClu) * kCluNb * ld;  // in CTA own
    if (rank == own) {
      if (warp == 0) {
        // lane = row r (8) x column group q (4): columns q and q + 4
        const int r = lane & 7, q = lane >> 3;
        T v[2] = {pan[(size_t)q * ld + k0 + r], pan[(size_t)(q + 4) * ld + k0 + r]};
#pragma unroll
        for (int c = 0; c < kCluNb; ++c) {
          const T piv = __shfl_sync(0xffffffffu, v[c >> 2], c + 8 * (c & 3));
          const T lraw = __shfl_sync(0xffffffffu, v[c >> 2], r + 8 * (c & 3));
          const T ip = (T)1 / piv;
          const T l = lraw * ip;
          if (lane == 0) inv[(kb / kClu) * kCluNb + c] = ip;
          if (q == (c & 3) && r > c) v[c >> 2] = l;
#pragma unroll
          for (int h = c >> 2; h < 2; ++h) {
            const T u = __shfl_sync(0xffffffffu, v[h], c + 8 * q);
            if (q + 4 * h > c && r > c) v[h] -= l * u;
          }
        }
        pan[(size_t)q * ld + k0 + r] = v[0];
        pan[(size_t)(q + 4) * ld + k0 + r] = v[1];
      }
      __syncthreads();
      for (int i = r0 + tid; i < ld; i += kCluThreads) {
        T x[kCluNb];
#pragma unroll
        for (int c = 0; c < kCluNb; ++c) {
          T acc = pan[(size_t)c * ld + i];
#pragma unroll
          for (int p = 0; p < c; ++p) acc -= x[p] * pan[(size_t)c * ld + k0 + p];
          x[c] = acc * inv[(kb / kClu) * kCluNb + c];
        }
#pragma unroll
        for (int c = 0; c < kCluNb; ++c) pan[(size_t)c * ld + i] = x[c];
      }
    }
    cluster_barrier();
    for (int q = tid; q < kCluNb * (ld - k0); q += kCluThreads) {
      const size_t o = (size_t)(q / (ld - k0)) * ld + k0 + q % (ld - k0);
      Lp[o] = rank == own ? pan[o] : remote(pan + o, own);
    }
    __syncthreads();
    // this CTA's blocks to the right of kb, and on CTA 0 the right-hand side
    const int lb0 = kb < rank ? 0 : (kb - rank) / kClu + 1;
    const int nc = ((nblk - rank + kClu - 1) / kClu - lb0) * kCluNb;
    // rows k0 .. k0+7 of each column: L11 v = a, a column per thread
    for (int t = tid; t < nc + (rank == 0 ? 1 : 0); t += kCluThreads) {
      T* col = t < nc ? A + ((size_t)lb0 * kCluNb + t) * ld : y;
      T v[kCluNb];
#pragma unroll
      for (int r = 0; r < kCluNb; ++r) v[r] = col[k0 + r];
#pragma unroll
      for (int p = 0; p < kCluNb; ++p)
#pragma unroll
        for (int r = p + 1; r < kCluNb; ++r) v[r] -= Lp[(size_t)p * ld + k0 + r] * v[p];
#pragma unroll
      for (int r = 0; r < kCluNb; ++r) col[k0 + r] = v[r];
    }
    __syncthreads();
    // rows below: 32 rows (a row per lane) x one block of columns per warp
    const int nch = (ld - r0 + 31) / 32, nt = nch * (nc / kCluNb);
    for (int t = warp; t < nt + (rank == 0 ? nch : 0); t += W) {
      const int i = r0 + 32 * (t % nch) + lane;
      if (i >= ld) continue;
      T l[kCluNb];
#pragma unroll
      for (int p = 0; p < kCluNb; ++p) l[p] = Lp[(size_t)p * ld + i];
      if (t < nt) {
        T* blk = A + (size_t)(lb0 + t / nch) * kCluNb * ld;
#pragma unroll
        for (int c = 0; c < kCluNb; ++c) {
          T acc = blk[(size_t)c * ld + i];
#pragma unroll
          for (int p = 0; p < kCluNb; ++p) acc -= l[p] * blk[(size_t)c * ld + k0 + p];
          blk[(size_t)c * ld + i] = acc;
        }
      } else {
        T acc = y[i];
#pragma unroll
        for (int p = 0; p < kCluNb; ++p) acc -= l[p] * y[k0 + p];
        y[i] = acc;
      }
    }
    __syncthreads();
  }
  for (int kb = nblk - 1; kb >= 0; --kb) {
    const int k0 = kb * kCluNb, own = kb % kClu;
    cluster_barrier();  // the right-hand side's last holder is done with it
    if (rank != own) continue;
    const int src = kb == nblk - 1 ? 0 : (kb + 1) % kClu;
    if (src != rank) {
      for (int r = tid; r < k0 + kCluNb; r += kCluThreads) y[r] = remote(y + r, src);
      __syncthreads();
    }
    const T* pan = A + (size_t)(kb / kClu) * kCluNb * ld;
    if (warp == 0) {
      const int r = lane & 7;
      T v = y[k0 + r];
#pragma unroll
      for (int c = kCluNb - 1; c >= 0; --c) {
        const T x = __shfl_sync(0xffffffffu, v, c) * inv[(kb / kClu) * kCluNb + c];
        if (r == c) v = x;
        if (r < c) v -= pan[(size_t)c * ld + k0 + r] * x;
      }
      if (lane < kCluNb) {
        y[k0 + r] = v;
        X[(size_t)(k0 + r) * kTile] = v;
      }
    }
    __syncthreads();
    for (int i = tid; i < k0; i += kCluThreads) {
      T acc = y[i];
#pragma unroll
      for (int c = kCluNb - 1; c >= 0; --c) acc -= pan[(size_t)c * ld + i] * y[k0 + c];
      y[i] = acc;
    }
  }
  cluster_barrier();  // no CTA leaves while another reads its shared memory
}

}  // namespace

namespace {

void configure(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, unsigned instances, size_t smem, cudaStream_t st) {
  cfg.gridDim = dim3(instances * kClu);
  cfg.blockDim = dim3(kCluThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kClu;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
}

template <typename T>
int resident(const DevPlan& P) {
  cudaFuncSetAttribute(k_dense_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCluSmem);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  configure(cfg, at, 1, clu_smem(P.nde, sizeof(T)), nullptr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_dense_cluster<T>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace

int dense_cluster_resident(const DevPlan& P, size_t width) {
  if (P.nde < 2 * kCluNb || P.nde % kCluNb != 0 || clu_smem(P.nde, width) > kCluSmem) return 0;
  return width == 8 ? resident<double>(P) : resident<float>(P);
}

bool dense_cluster_pays(const DevPlan& P, int B, size_t width) {
  if (width == 8) return B <= kCluInstances && B <= kCluRounds64 * P.clusters;
  if (P.nde <= kCluWide32) return P.clusters > 0 && B <= kCluInstances;
  return B <= kCluInstances32Wide && B <= P.clusters;
}

template <typename T>
void launch_dense_cluster(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st, Recorder* rec) {
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_dense_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCluSmem);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  configure(cfg, at, (unsigned)S.Bp, clu_smem(P.nde, sizeof(T)), st);
  NRPF_LAUNCH(rec, K_DENSE_SOLVE, st, cudaLaunchKernelEx(&cfg, k_dense_cluster<T>, P, S, gate));
}

template void launch_dense_cluster<float>(const DevPlan&, const DevState&, const int32_t*, cudaStream_t, Recorder*);
template void launch_dense_cluster<double>(const DevPlan&, const DevState&, const int32_t*, cudaStream_t, Recorder*);

}  // namespace nrpf
