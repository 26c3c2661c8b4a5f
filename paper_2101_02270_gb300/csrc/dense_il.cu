// Dense block of the FP32 LU in the interleaved layout (Sec. 4.3: the serial tail of
// the column DAG, factorised as one dense matrix per instance, a lane each).  Rows
// r .. r + 3 of column c (r a multiple of 4) for a lane are one 16-byte word,
//   float4 (c * ndp + r) * 8 + lane,
// so a warp reads four entries of all its instances in 512 contiguous bytes.
//
// Blocked LU without pivoting, in outer panels of 64 columns, steps of 16:
//   k_il_gemm  (strip) : the step's 16 columns and 16 rows minus the products of the
//                        panel's earlier steps (depth 16, 32, 48)
//   k_il_diag          : LU of the 16 x 16 diagonal block, its inverse pivots
//   k_il_panel         : L21 = A21 U11^-1 below, U12 = L11^-1 A12 to the right
//   k_il_gemm          : after the four steps, A22 -= L21 U12 at depth 64
// Every entry takes its subtractions in ascending pivot order, each one fused
// multiply-add, whatever the blocking.  Within a panel the steps look left, so that an
// entry is read and written once per panel; looking right, each step updating the rest
// of the panel's columns and rows, made three more passes over them.  Work stops at
// P.nde, nd rounded up to 16, where the leading dimension is rounded up to 64.
//
// What bounds it is the traffic between L2 and shared memory: 10,000 blocks of 320, five
// factorisations, 14.5 ms of multiply-adds, 54 GB of operands and 20 GB of entries per
// factorisation, in 26.1 ms; a thread per 8 x 8 entries that loaded its operands
// through L1, looking right in the panel, took 32.8 ms.  (8 x 8 entries per warp from
// the same stages, twice the warps: 26.7 ms.)
#include "dense_il.h"
#include "kernels.h"

namespace nrpf {

namespace {

constexpr int kIlB = 16;       // step
constexpr int kIlOuter = 64;   // outer panel
constexpr int kIlDiagWarps = 8;
constexpr int kIlPanelWarps = 4;

__device__ __forceinline__ bool il_active(const DevState& S, int tile, int lane) {
  return __any_sync(0xffffffffu, S.active[tile * kTile + lane]);
}

__device__ __forceinline__ float4* il_block(const DevPlan& P, const DevState& S, int tile, int lane) {
  return reinterpret_cast<float4*>(reinterpret_cast<float*>(S.lu) + ((size_t)tile * P.NLU + P.NS) * kTile) + lane;
}

// the word of rows r .. r + 3 (r a multiple of 4) of column c
__device__ __forceinline__ size_t il_at(int r, int c, int ld) { return ((size_t)c * ld + r) * 8; }

__device__ __forceinline__ float comp(const float4& v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

__device__ __forceinline__ float2 neg2(float v) { return make_float2(-v, -v); }

// Step at ki: one CTA per tile, eight warps with rows w and w + 8 in registers, the
// pivot row published in shared memory, one barrier per pivot.  (As one warp per tile with the block in 256 registers, mostly spilled, the
// elimination took 18 us on 11 tiles, against 4.)
__global__ void __launch_bounds__(32 * kIlDiagWarps) k_il_diag(DevPlan P, DevState S, int ki,
                                                               const int32_t* __restrict__ gate) {
  __shared__ float prow[2][kIlB][kTile];
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x, w = threadIdx.y, tile = blockIdx.x;
  if (!il_active(S, tile, lane)) return;  // uniform over the CTA
  float4* __restrict__ A4 = il_block(P, S, tile, lane);
  // element (r, c) of this lane: A[il_at(r & ~3, c) * 4 + (r & 3)]
  float* __restrict__ A = reinterpret_cast<float*>(A4);
  float* __restrict__ inv = reinterpret_cast<float*>(S.inv) + (size_t)tile * kIlB * kTile + lane;
  const int ld = P.ndp;
  auto at = [&](int r, int c) -> float& { return A[il_at(r & ~3, c, ld) * 4 + (r & 3)]; };
  float d[2][kIlB];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < kIlB; ++c) d[h][c] = at(ki + w + 8 * h, ki + c);
#pragma unroll
  for (int c = 0; c < kIlB; ++c) {
    if (w == (c & 7)) {
#pragma unroll
      for (int cc = c; cc < kIlB; ++cc) prow[c & 1][cc][lane] = d[c >> 3][cc];
    }
    __syncthreads();
    const float ip = 1.f / prow[c & 1][c][lane];
    if (w == (c & 7)) inv[c * kTile] = ip;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (w + 8 * h > c) {
        const float l = d[h][c] * ip;
        d[h][c] = l;
#pragma unroll
        for (int cc = c + 1; cc < kIlB; ++cc) d[h][cc] = fmaf(-l, prow[c & 1][cc][lane], d[h][cc]);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < kIlB; ++c) at(ki + w + 8 * h, ki + c) = d[h][c];
}

// The step's rows below and columns to the right, four rows or four columns per
// thread, 16 x 4 entries in 64 registers, pairs of rows packed for the two-wide
// multiply-add.  Bound by memory: 16 x 4 entries in and out per thread for 136 packed
// multiply-adds; the diagonal block's factors come through L1.
__global__ void __launch_bounds__(32 * kIlPanelWarps, 3) k_il_panel(DevPlan P, DevState S, int ki,
                                                                    const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x, tile = blockIdx.y;
  if (!il_active(S, tile, lane)) return;
  const int ld = P.ndp, r0 = ki + kIlB;
  const int ng = (P.nde - r0) / 4;  // groups of four rows, as many of columns
  const int g = blockIdx.x * kIlPanelWarps + threadIdx.y;
  if (g >= 2 * ng) return;
  float4* __restrict__ A4 = il_block(P, S, tile, lane);
  if (g < ng) {
    // rows i0 .. i0 + 3: x U11 = a, x[c] rows (0, 1) and (2, 3)
    const int i0 = r0 + 4 * g;
    const float* __restrict__ inv = reinterpret_cast<const float*>(S.inv) + (size_t)tile * kIlB * kTile + lane;
    float2 x[kIlB][2];
#pragma unroll
    for (int c = 0; c < kIlB; ++c) {
      const float4 v = A4[il_at(i0, ki + c, ld)];
      x[c][0] = make_float2(v.x, v.y);
      x[c][1] = make_float2(v.z, v.w);
    }
#pragma unroll
    for (int c = 0; c < kIlB; ++c) {
#pragma unroll
      for (int q = 0; 4 * q < c; ++q) {
        const float4 u = A4[il_at(ki + 4 * q, ki + c, ld)];
#pragma unroll
        for (int z = 0; z < 4; ++z)
          if (4 * q + z < c) {
            const float2 nu = neg2(comp(u, z));
            x[c][0] = __ffma2_rn(x[4 * q + z][0], nu, x[c][0]);
            x[c][1] = __ffma2_rn(x[4 * q + z][1], nu, x[c][1]);
          }
      }
      const float ip = inv[c * kTile];
      x[c][0] = make_float2(x[c][0].x * ip, x[c][0].y * ip);
      x[c][1] = make_float2(x[c][1].x * ip, x[c][1].y * ip);
    }
#pragma unroll
    for (int c = 0; c < kIlB; ++c)
      A4[il_at(i0, ki + c, ld)] = make_float4(x[c][0].x, x[c][0].y, x[c][1].x, x[c][1].y);
  } else {
    // columns j0 .. j0 + 3: L11 y = a, y[t][r / 2] rows (r, r + 1) of column t
    const int j0 = r0 + 4 * (g - ng);
    float2 y[4][kIlB / 2];
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int q = 0; q < kIlB / 4; ++q) {
        const float4 v = A4[il_at(ki + 4 * q, j0 + t, ld)];
        y[t][2 * q] = make_float2(v.x, v.y);
        y[t][2 * q + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
    for (int p = 0; p < kIlB - 1; ++p)
#pragma unroll
      for (int q = (p + 1) / 4; q < kIlB / 4; ++q) {
        const float4 l = A4[il_at(ki + 4 * q, ki + p, ld)];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 lh = h ? make_float2(l.z, l.w) : make_float2(l.x, l.y);
          const int r = 4 * q + 2 * h;  // rows r, r + 1
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const float yp = p & 1 ? y[t][p / 2].y : y[t][p / 2].x;
            if (r > p)
              y[t][r / 2] = __ffma2_rn(lh, neg2(yp), y[t][r / 2]);
            else if (r == p)
              y[t][r / 2].y = fmaf(-lh.y, yp, y[t][r / 2].y);
          }
        }
      }
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int q = 0; q < kIlB / 4; ++q)
        A4[il_at(ki + 4 * q, j0 + t, ld)] =
            make_float4(y[t][2 * q].x, y[t][2 * q].y, y[t][2 * q + 1].x, y[t][2 * q + 1].y);
  }
}

// C minus the products of the depth pivots k .. k + depth - 1 (a multiple of 16), with
// strip = 0 for rows and columns r0 .. nde - 1, with strip = 1 for columns r0 .. r0 + 15
// of these rows and then rows r0 .. r0 + 15 of columns r0 + 16 .. nde - 1.
//
// A warp takes 8 rows and 16 columns, lane by lane: 128 accumulators for 24 words of
// shared memory per four pivots and 16 x 8 x 4 multiply-adds.  Four warps make a CTA's
// tile, 32 rows x 16 columns (row strips: 16 x 32).  Its operands come eight pivots at
// a time by bulk copies, runs of 4 (2) KB of a column of L and of 1 KB of a column of
// U, through a ring of two stages; two CTAs per SM.
constexpr int kIlTC = 16;  // columns of a warp
constexpr int kIlGemmWarps = 512 / (8 * kIlTC);
constexpr int kIlKc = 8;
constexpr uint32_t kIlStage = 48 * kIlKc * kTile * 4;  // 48 KB
constexpr size_t kIlSmem = 2 * kIlStage;
constexpr uint32_t kIlSpinLimit = 1u << 20;

__global__ void __launch_bounds__(32 * kIlGemmWarps, 2) k_il_gemm(DevPlan P, DevState S, int k, int depth, int r0, int strip,
                                                    const int32_t* __restrict__ gate) {
  extern __shared__ __align__(128) unsigned char il_smem[];
  __shared__ __align__(8) uint64_t bars[2];
  if (gate && *gate == 0) return;
  const int lane = threadIdx.x, w = threadIdx.y, tile = blockIdx.y;
  if (!il_active(S, tile, lane)) return;  // uniform over the CTA
  const int ld = P.ndp, n = P.nde, nbr = (n - r0 + 31) / 32;
  int i0, j0;
  bool wide = false;  // 16 rows x 32 columns
  if (!strip) {
    i0 = r0 + 32 * (int)(blockIdx.x % nbr);
    j0 = r0 + 16 * (int)(blockIdx.x / nbr);
  } else if ((int)blockIdx.x < nbr) {
    i0 = r0 + 32 * (int)blockIdx.x;
    j0 = r0;
  } else {
    wide = true;
    i0 = r0;
    j0 = r0 + 16 + 32 * ((int)blockIdx.x - nbr);
  }
  const int nr = wide ? 16 : min(32, n - i0), nc = wide ? min(32, n - j0) : 16;  // multiples of 16
  const uint32_t apitch = wide ? 2048 : 4096;       // bytes of a column of L in a stage
  const uint32_t uoff = kIlKc * apitch;             // the columns of U follow, 1 KB each
  const float4* __restrict__ A0 = il_block(P, S, tile, 0);
  const uint32_t sm = static_cast<uint32_t>(__cvta_generic_to_shared(il_smem));
  const uint32_t sb = static_cast<uint32_t>(__cvta_generic_to_shared(bars));
  // chunk c (pivots k + 8 c ..) into stage c % 2, by the first warp
  auto fetch = [&](int c) {
    const uint32_t st = sm + (c & 1) * kIlStage, bar = sb + 8 * (c & 1);
    const int p0 = k + kIlKc * c;
    if (lane == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                   "r"((uint32_t)((nr + nc) * kIlKc * 128))
                   : "memory");
    __syncwarp();
    auto copy = [&](uint32_t dst, const float4* src, uint32_t bytes) {
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                   "l"(src), "r"(bytes), "r"(bar)
                   : "memory");
    };
    if (lane < kIlKc) copy(st + lane * apitch, A0 + il_at(i0, p0 + lane, ld), (uint32_t)nr * 128);
    if (lane < nc) copy(st + uoff + lane * 1024, A0 + il_at(p0, j0 + lane, ld), 1024);
  };
  const int chunks = depth / kIlKc;  // at least two
  if (w == 0) {
    if (lane == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sb) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sb + 8) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    fetch(0);
    fetch(1);
  }
  const int wr = wide ? 8 * (w & 1) : 8 * (w & 3), wc = kIlTC * (wide ? w >> 1 : w >> 2);
  const bool mine = wr < nr && wc < nc;
  float4* __restrict__ C = il_block(P, S, tile, lane) + il_at(i0 + wr, j0 + wc, ld);
  float2 acc[4][kIlTC];  // rows 2p, 2p + 1 of column c
  if (mine) {
#pragma unroll
    for (int c = 0; c < kIlTC; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = C[il_at(4 * h, c, ld)];
        acc[2 * h][c] = make_float2(v.x, v.y);
        acc[2 * h + 1][c] = make_float2(v.z, v.w);
      }
  }
  __syncthreads();  // the barriers are initialised
  auto wait = [&](int c) {
    uint32_t ok = 0;
    for (uint32_t spins = 0; !ok && spins < kIlSpinLimit; ++spins)
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(sb + 8 * (c & 1)), "r"((uint32_t)(c >> 1 & 1))
          : "memory");
    return ok != 0;
  };
#pragma unroll 1
  for (int ch = 0; ch < chunks; ++ch) {
    const bool ok = wait(ch);
    if (ok && mine) {
      const unsigned char* st = il_smem + (ch & 1) * kIlStage;
      const float4* la = reinterpret_cast<const float4*>(st + wr * 128) + lane;
      const float4* lu = reinterpret_cast<const float4*>(st + uoff + wc * 1024) + lane;
#pragma unroll
      for (int pp = 0; pp < kIlKc / 4; ++pp) {
        float4 a[4][2];
#pragma unroll
        for (int z = 0; z < 4; ++z)
#pragma unroll
          for (int h = 0; h < 2; ++h) a[z][h] = la[(4 * pp + z) * (apitch / 16) + h * 32];
#pragma unroll
        for (int c = 0; c < kIlTC; ++c) {
          const float4 u = lu[c * 64 + pp * 32];
#pragma unroll
          for (int z = 0; z < 4; ++z) {
            const float2 nu = neg2(comp(u, z));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              acc[2 * h][c] = __ffma2_rn(make_float2(a[z][h].x, a[z][h].y), nu, acc[2 * h][c]);
              acc[2 * h + 1][c] = __ffma2_rn(make_float2(a[z][h].z, a[z][h].w), nu, acc[2 * h + 1][c]);
            }
          }
        }
      }
    }
    if (__syncthreads_or(!ok)) {  // a copy did not land in time: the step is discarded
      wait(ch);  // no copy of this CTA's may land after it
      if (ch + 1 < chunks) wait(ch + 1);
      S.bad[tile * kTile + lane] = 1;
      return;
    }
    if (w == 0 && ch + 2 < chunks) fetch(ch + 2);
  }
  if (!mine) return;
#pragma unroll
  for (int c = 0; c < kIlTC; ++c)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      C[il_at(4 * h, c, ld)] = make_float4(acc[2 * h][c].x, acc[2 * h][c].y, acc[2 * h + 1][c].x, acc[2 * h + 1][c].y);
}

}  // namespace

void launch_dense_il_factor(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st, Recorder* rec) {
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_il_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIlSmem);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const unsigned tiles = (unsigned)(S.Bp / kTile);
  auto gemm = [&](int k, int depth, int r0, bool strip) {
    const int n = P.nde - r0;
    const int rows = (n + 31) / 32, blocks = strip ? rows + (n - 16 + 31) / 32 : rows * (n / 16);
    NRPF_LAUNCH(rec, K_DENSE_UPDATE, st,
                k_il_gemm<<<dim3((unsigned)blocks, tiles), dim3(32, kIlGemmWarps), kIlSmem, st>>>(P, S, k, depth, r0, strip,
                                                                                      gate));
  };
  for (int k = 0; k < P.nde; k += kIlOuter) {
    for (int ki = k; ki < P.nde && ki < k + kIlOuter; ki += kIlB) {
      if (ki > k) gemm(k, ki - k, ki, true);
      NRPF_LAUNCH(rec, K_DENSE_DIAG, st, k_il_diag<<<tiles, dim3(32, kIlDiagWarps), 0, st>>>(P, S, ki, gate));
      const int groups = (P.nde - ki - kIlB) / 4 * 2;
      if (groups > 0)
        NRPF_LAUNCH(rec, K_DENSE_PANEL, st,
                    k_il_panel<<<dim3((unsigned)((groups + kIlPanelWarps - 1) / kIlPanelWarps), tiles),
                                 dim3(32, kIlPanelWarps), 0, st>>>(P, S, ki, gate));
    }
    if (k + kIlOuter < P.nde) gemm(k, kIlOuter, k + kIlOuter, false);
  }
}

}  // namespace nrpf
