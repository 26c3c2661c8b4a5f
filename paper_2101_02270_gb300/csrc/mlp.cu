// Learned warm start: a small MLP that maps per-bus injections (P, Q) to an
// initial voltage guess (|V|, angle of the non-slack buses), trained on the
// solver's own solutions; Newton-Raphson always runs from its guess to the
// same tolerance.  All GEMMs (forward and backward) run on the tcgen05 tensor
// cores with BF16 operands and FP32 accumulation (gemm_tc.cuh), with bias, GELU,
// loss and GELU' in their epilogues; AdamW is a CUDA kernel; master weights and
// optimiser state are FP32.
//   h1 = GELU(x W1^T + b1), h2 = GELU(h1 W2^T + b2), y = h2 W3^T + b3
// with W_l stored [out][in] (row-major), exact erf-GELU, loss = mean (y - t)^2
// on standardised inputs and targets.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <new>
#include <random>
#include <vector>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/nrpf.h"
#include "gemm_tc.cuh"
#include "handle.h"

namespace nrpf {
namespace {

using bf16 = __nv_bfloat16;

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * __expf(-0.5f * z * z);
}

// ---- GEMM epilogues (gemm_tc.cuh: one element each, rows contiguous over a warp) ----
struct EpiF32 {  // C = acc, [nrows][ncols] (the padding of the product is dropped)
  static constexpr bool kSum = false;
  float* C;
  int nrows, ncols;
  __device__ float operator()(int r, int c, float v) const {
    if (r < nrows && c < ncols) C[(int64_t)r * ncols + c] = v;
    return 0.f;
  }
};
struct EpiBiasGelu {  // Z = acc + b (FP32, kept for the backward pass unless null), H = GELU(Z) (BF16); padding columns -> 0
  static constexpr bool kSum = false;
  const float* b;
  float* Z;
  bf16* H;
  int ld, nvalid;
  __device__ float operator()(int r, int c, float v) const {
    const float z = c < nvalid ? v + b[c] : 0.f;
    if (Z) Z[(int64_t)r * ld + c] = z;
    H[(int64_t)r * ld + c] = __float2bfloat16(c < nvalid ? gelu_f(z) : 0.f);
    return 0.f;
  }
};
struct EpiUnstd {  // y = (acc + b) sd + mu: the prediction in physical units, [B][nvalid]
  static constexpr bool kSum = false;
  const float *b, *mu, *sd;
  float* y;
  int nrows, nvalid;
  __device__ float operator()(int r, int c, float v) const {
    if (r < nrows && c < nvalid) y[(int64_t)r * nvalid + c] = (v + b[c]) * sd[c] + mu[c];
    return 0.f;
  }
};
struct EpiLoss {  // y = acc + b, dY = 2 (y - t) / (B nout) (BF16; padding -> 0); summand (y - t)^2
  static constexpr bool kSum = true;
  const float *b, *t, *mu, *sd;
  bf16* dY;
  double* sum;
  int nrows, nvalid, ld;
  __device__ float operator()(int r, int c, float v) const {
    float l = 0.f, g = 0.f;
    if (r < nrows && c < nvalid) {
      const float d = (v + b[c]) - (t[(int64_t)r * nvalid + c] - mu[c]) / sd[c];
      l = d * d;
      g = 2.f * d / ((float)nrows * (float)nvalid);
    }
    dY[(int64_t)r * ld + c] = __float2bfloat16(g);
    return l;
  }
};
struct EpiGeluBack {  // dZ = acc * GELU'(Z) (BF16); rows >= nrows and columns >= nvalid -> 0
  static constexpr bool kSum = false;
  const float* Z;
  bf16* dZ;
  int nrows, nvalid, ld;
  __device__ float operator()(int r, int c, float v) const {
    const int64_t i = (int64_t)r * ld + c;
    dZ[i] = __float2bfloat16((r < nrows && c < nvalid) ? v * gelu_grad_f(Z[i]) : 0.f);
    return 0.f;
  }
};

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// 2-D map of a row-major BF16 matrix [rows][K]: boxes of 64 (K) x `box_rows`
// rows, 128-byte swizzle (the layout the UMMA descriptors expect)
bool make_tmap(CUtensorMap* m, const bf16* ptr, int rows, int K, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kGemmBK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(ptr), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// variant: 0 = copy-then-MMA kernel, 1 = TMA pipeline (falls back to 0 when
// the tensor-map encoder is unavailable)
int g_gemm_variant = 1;

template <class Epi, int BN, bool AT, bool BT>
bool launch_gemm_tma(const bf16* A, const bf16* B, int M, int N, int K, Epi epi, int* err, cudaStream_t st) {
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_gemm_tma<Epi, CUtensorMap, BN, AT, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)GemmTile<BN>::kSmem);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  CUtensorMap ta, tb;
  if (!(AT ? make_tmap(&ta, A, K, M, kGemmBK) : make_tmap(&ta, A, M, K, kGemmBM)) ||
      !(BT ? make_tmap(&tb, B, K, N, kGemmBK) : make_tmap(&tb, B, N, K, BN)))
    return false;
  k_gemm_tma<Epi, CUtensorMap, BN, AT, BT>
      <<<dim3(N / BN, M / kGemmBM), kGemmTmaThreads, GemmTile<BN>::kSmem, st>>>(ta, tb, M, N, K, epi, err);
  return true;
}

// Tile width of the pipelined kernel: 64 while 128-wide tiles would leave some
// of the 152 SMs without one.  On a minibatch of 1,024 rows the products with
// 1,024 columns have 64 tiles of 128 x 128.
inline bool narrow_tiles(int M, int N) { return (int64_t)(M / kGemmBM) * (N / 128) < 152; }

// C[M][N] = A B^T, A [M][K] (AT: stored [K][M]), B [N][K] (BT: stored [K][N])
template <bool AT = false, bool BT = false, class Epi>
int gemm(const bf16* A, const bf16* B, int M, int N, int K, Epi epi, int* err, cudaStream_t st,
         int variant = -1) {
  if (M % kGemmBM || N % kGemmBN || K % kGemmBK || M <= 0 || N <= 0 || K <= 0) return NRPF_ERR_ARG;
  if (variant < 0) variant = g_gemm_variant;
  bool done = false;
  if (variant == 1)
    done = narrow_tiles(M, N) ? launch_gemm_tma<Epi, 64, AT, BT>(A, B, M, N, K, epi, err, st)
                              : launch_gemm_tma<Epi, 128, AT, BT>(A, B, M, N, K, epi, err, st);
  if (!done) {
    static bool configured[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !configured[dev]) {
      cudaFuncSetAttribute(k_gemm_tc<Epi, AT, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
      if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    k_gemm_tc<Epi, AT, BT><<<dim3(N / kGemmBN, M / kGemmBM), kGemmThreads, kGemmSmem, st>>>(A, B, M, N, K, epi, err);
  }
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

// ---- elementwise / layout kernels ----
// x (FP32 [B][nin]) -> standardised BF16 [Bp][nin_p], zero padding.  A thread
// keeps two columns' mean and deviation and walks over the rows of its block:
// no index is divided, and with V2 (rows of x 8-byte aligned) a warp reads 256
// bytes and writes 128 per row.
constexpr int kPrepRows = 16;
template <bool V2>
__global__ void __launch_bounds__(256) k_prep_x(const float* __restrict__ x, const float* __restrict__ mu,
                                                const float* __restrict__ sd, bf16* __restrict__ xb, int B, int Bp,
                                                int nin, int nin_p) {
  const int c = 2 * (blockIdx.x * 256 + threadIdx.x);
  if (c >= nin_p) return;
  const bool v0 = c < nin, v1 = c + 1 < nin;
  const float m0 = v0 ? mu[c] : 0.f, m1 = v1 ? mu[c + 1] : 0.f;
  const float s0 = v0 ? sd[c] : 1.f, s1 = v1 ? sd[c + 1] : 1.f;
  // Bp is a multiple of 128 and so of kPrepRows
  for (int64_t r0 = (int64_t)blockIdx.y * kPrepRows; r0 < Bp; r0 += (int64_t)gridDim.y * kPrepRows) {
#pragma unroll 4
    for (int64_t r = r0; r < r0 + kPrepRows; ++r) {
      float2 v = make_float2(0.f, 0.f);
      if (r < B) {
        const float* q = x + r * nin + c;
        if (V2) {
          if (v0) v = *reinterpret_cast<const float2*>(q);
        } else {
          if (v0) v.x = q[0];
          if (v1) v.y = q[1];
        }
        v = make_float2(v0 ? (v.x - m0) / s0 : 0.f, v1 ? (v.y - m1) / s1 : 0.f);
      }
      *reinterpret_cast<__nv_bfloat162*>(xb + r * nin_p + c) = __floats2bfloat162_rn(v.x, v.y);
    }
  }
}

// Column sums of a BF16 [Bp][ld] matrix into FP32 g[n] (bias gradients), each
// column added in the order of its rows.  That chain, one FADD per row, is the
// floor (1,024 rows: 2 us); the loads are taken off it: a CTA takes 64 columns,
// its eight warps bring 128 rows at a time into shared memory (a 128-byte line
// per warp and row, all in flight), and a ninth adds the chunk before while the
// next one arrives.  One thread per column, at most 16 CTAs and every load on
// the chain, took 101 us for the three biases of a step of 1,024 rows.
constexpr int kColRows = 128;
__global__ void __launch_bounds__(288) k_colsum(const bf16* __restrict__ D, float* __restrict__ g, int Bp, int ld,
                                                int n) {
  __shared__ __nv_bfloat162 buf[2][kColRows][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;  // warps 0 .. 7 load, warp 8 adds
  const int c = blockIdx.x * 64 + 2 * lane;                 // ld is a multiple of 128
  const __nv_bfloat162* __restrict__ src = reinterpret_cast<const __nv_bfloat162*>(D + c);
  const int nch = Bp / kColRows;
  float2 s = make_float2(0.f, 0.f);
  for (int k = 0; k <= nch; ++k) {
    if (w < 8 && k < nch) {
#pragma unroll
      for (int j = 0; j < kColRows / 8; ++j)
        buf[k & 1][8 * j + w][lane] = src[((int64_t)k * kColRows + 8 * j + w) * (ld / 2)];
    } else if (w == 8 && k > 0) {
#pragma unroll 16
      for (int r = 0; r < kColRows; ++r) {
        const float2 v = __bfloat1622float2(buf[(k - 1) & 1][r][lane]);
        s.x += v.x;
        s.y += v.y;
      }
    }
    __syncthreads();
  }
  if (w == 8) {
    if (c < n) g[c] = s.x;
    if (c + 1 < n) g[c + 1] = s.y;
  }
}

// AdamW on the six FP32 tensors of the network, refreshing the padded BF16
// copies of the weights: 30 bytes per parameter and no reuse, so HBM is the
// bound (9.2 M parameters: 41 us at the measured copy rate).  A thread takes
// four consecutive parameters with 16-byte accesses, and one launch covers all
// tensors: as six launches of one parameter per thread, each dividing its
// 64-bit index, a step took 63 us.
struct AdamSet {
  float* p[6];
  const float* g[6];
  float *m[6], *v[6];
  bf16* pb[6];      // null: no BF16 copy
  int64_t n[6];
  int cols[6], ld[6];  // of the tensor, of its BF16 copy
  float wd[6];
  unsigned first[7];  // first CTA of each tensor
};

__global__ void __launch_bounds__(256) k_adamw(AdamSet a, float lr, float b1, float b2, float eps, float c1, float c2) {
  int k = 0;
#pragma unroll
  for (int q = 1; q < 6; ++q) k += blockIdx.x >= a.first[q];
  const int64_t i = 4 * ((int64_t)(blockIdx.x - a.first[k]) * 256 + threadIdx.x);
  const int64_t n = a.n[k];
  if (i >= n) return;
  const float wd = a.wd[k];
  auto step = [&](float& p, float g, float& m, float& v) {
    float pi = p * (1.f - lr * wd);
    // the roundings are pinned: weights repeat bit for bit over the steps
    m = __fmaf_rn(1.f - b1, g, __fmul_rn(b1, m));
    v = __fmaf_rn(__fmul_rn(1.f - b2, g), g, __fmul_rn(b2, v));
    pi -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    p = pi;
  };
  bf16* pb = a.pb[k];
  const int64_t r = i / a.cols[k];
  int c = (int)(i - r * a.cols[k]);
  if (i + 4 <= n) {
    float4 p = *reinterpret_cast<const float4*>(a.p[k] + i), m = *reinterpret_cast<const float4*>(a.m[k] + i);
    float4 v = *reinterpret_cast<const float4*>(a.v[k] + i);
    const float4 g = *reinterpret_cast<const float4*>(a.g[k] + i);
    step(p.x, g.x, m.x, v.x);
    step(p.y, g.y, m.y, v.y);
    step(p.z, g.z, m.z, v.z);
    step(p.w, g.w, m.w, v.w);
    *reinterpret_cast<float4*>(a.p[k] + i) = p;
    *reinterpret_cast<float4*>(a.m[k] + i) = m;
    *reinterpret_cast<float4*>(a.v[k] + i) = v;
    if (pb && c + 4 <= a.cols[k] && c % 4 == 0) {  // ld is a multiple of 128
      __nv_bfloat162* q = reinterpret_cast<__nv_bfloat162*>(pb + r * a.ld[k] + c);
      q[0] = __floats2bfloat162_rn(p.x, p.y);
      q[1] = __floats2bfloat162_rn(p.z, p.w);
    } else if (pb) {
      const float e[4] = {p.x, p.y, p.z, p.w};
      int64_t row = r;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        while (c >= a.cols[k]) {
          c -= a.cols[k];
          ++row;
        }
        pb[row * a.ld[k] + c++] = __float2bfloat16(e[j]);
      }
    }
  } else {
    for (int64_t j = i; j < n; ++j) {
      step(a.p[k][j], a.g[k][j], a.m[k][j], a.v[k][j]);
      if (pb) pb[(j / a.cols[k]) * a.ld[k] + j % a.cols[k]] = __float2bfloat16(a.p[k][j]);
    }
  }
}

// the loss from the FP64 sum of the squares
__global__ void k_loss_out(const double* __restrict__ sum, double count, float* __restrict__ loss) {
  *loss = (float)(*sum / count);
}

// FP32 [rows][cols] -> BF16 [rows][ld] (padding untouched)
__global__ void k_to_bf16(const float* __restrict__ a, bf16* __restrict__ b, int64_t n, int cols, int ld) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  b[(i / cols) * ld + i % cols] = __float2bfloat16(a[i]);
}

inline unsigned nb(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }
inline int rup(int x, int m) { return (x + m - 1) / m * m; }

}  // namespace
}  // namespace nrpf

using nrpf::bf16;

struct pf_mlp {
  int nin, nh1, nh2, nout, bmax;
  int nin_p, nout_p, bp;  // padded sizes
  int64_t step = 0;
  // parameters (FP32 master, dense [out][in]) and their BF16 padded copies
  float *W[3], *b[3], *mW[3], *vW[3], *mb[3], *vb[3], *gW[3], *gb[3];
  bf16* Wb[3];
  int fin[3], fout[3], fin_p[3], fout_p[3];
  // activations
  bf16 *xb, *h1, *h2, *dy, *dz2, *dz1;
  float *z1, *z2;
  float *mux, *sdx, *muy, *sdy;
  double* loss;  // sum of the squares of the last step
  int* err;
  std::vector<void*> allocs;
};

namespace {

int alloc_into(pf_mlp* p, size_t bytes, void** out) {
  void* d = nullptr;
  cudaError_t e = cudaMalloc(&d, std::max<size_t>(bytes, 256));
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? NRPF_ERR_NOMEM : NRPF_ERR_CUDA;
  p->allocs.push_back(d);
  cudaMemset(d, 0, std::max<size_t>(bytes, 256));
  *out = d;
  return NRPF_OK;
}

template <class T>
int al(pf_mlp* p, size_t count, T** out) {
  void* d = nullptr;
  int rc = alloc_into(p, count * sizeof(T), &d);
  *out = reinterpret_cast<T*>(d);
  return rc;
}

// refresh the padded BF16 copies of every weight
void refresh_bf16(pf_mlp* p, cudaStream_t st) {
  for (int l = 0; l < 3; ++l) {
    const int64_t n = (int64_t)p->fout[l] * p->fin[l];
    nrpf::k_to_bf16<<<nrpf::nb(n), 256, 0, st>>>(p->W[l], p->Wb[l], n, p->fin[l], p->fin_p[l]);
  }
}

// The hidden layers: h1, h2 (BF16) of Bp rows, and z1, z2 for a backward pass
int forward_hidden(pf_mlp* p, int B, const float* x, bool backward, cudaStream_t st) {
  using namespace nrpf;
  const int Bp = rup(B, kGemmBM);
  const dim3 g(nb(p->nin_p / 2), std::min(nb(Bp, kPrepRows), 65535u));
  if (p->nin % 2 == 0 && reinterpret_cast<uintptr_t>(x) % 8 == 0)
    k_prep_x<true><<<g, 256, 0, st>>>(x, p->mux, p->sdx, p->xb, B, Bp, p->nin, p->nin_p);
  else
    k_prep_x<false><<<g, 256, 0, st>>>(x, p->mux, p->sdx, p->xb, B, Bp, p->nin, p->nin_p);
  int rc;
  if ((rc = gemm(p->xb, p->Wb[0], Bp, p->fout_p[0], p->nin_p, EpiBiasGelu{p->b[0], backward ? p->z1 : nullptr, p->h1, p->fout_p[0], p->nh1},
                 p->err, st)))
    return rc;
  return gemm(p->h1, p->Wb[1], Bp, p->fout_p[1], p->fin_p[1], EpiBiasGelu{p->b[1], backward ? p->z2 : nullptr, p->h2, p->fout_p[1], p->nh2},
              p->err, st);
}

}  // namespace

extern "C" {

int pf_mlp_create(int nin, int nh1, int nh2, int nout, int bmax, uint64_t seed, pf_mlp** out) {
  if (!out || nin <= 0 || nh1 <= 0 || nh2 <= 0 || nout <= 0 || bmax <= 0) return NRPF_ERR_ARG;
  *out = nullptr;
  if (nh1 % nrpf::kGemmBN || nh2 % nrpf::kGemmBN) return NRPF_ERR_ARG;  // hidden widths: multiples of 128
  pf_mlp* p = new (std::nothrow) pf_mlp();
  if (!p) return NRPF_ERR_NOMEM;
  p->nin = nin; p->nh1 = nh1; p->nh2 = nh2; p->nout = nout; p->bmax = bmax;
  p->nin_p = nrpf::rup(nin, nrpf::kGemmBN);  // also the N of the first weight gradient
  p->nout_p = nrpf::rup(nout, nrpf::kGemmBN);
  p->bp = nrpf::rup(bmax, nrpf::kGemmBM);
  const int fin[3] = {nin, nh1, nh2}, fout[3] = {nh1, nh2, nout};
  const int fin_p[3] = {p->nin_p, nh1, nh2}, fout_p[3] = {nh1, nh2, p->nout_p};
  int rc = NRPF_OK;
  std::mt19937_64 rng(seed);
  for (int l = 0; l < 3 && !rc; ++l) {
    p->fin[l] = fin[l]; p->fout[l] = fout[l]; p->fin_p[l] = fin_p[l]; p->fout_p[l] = fout_p[l];
    const size_t nw = (size_t)fout[l] * fin[l];
    if ((rc = al(p, nw, &p->W[l])) || (rc = al(p, fout[l], &p->b[l])) || (rc = al(p, nw, &p->mW[l])) ||
        (rc = al(p, nw, &p->vW[l])) || (rc = al(p, fout[l], &p->mb[l])) || (rc = al(p, fout[l], &p->vb[l])) ||
        (rc = al(p, nw, &p->gW[l])) || (rc = al(p, fout[l], &p->gb[l])) ||
        (rc = al(p, (size_t)fout_p[l] * fin_p[l], &p->Wb[l])))
      break;
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases
    std::vector<float> w(nw);
    const double a = 1.0 / std::sqrt((double)fin[l]);
    std::uniform_real_distribution<double> U(-a, a);
    for (auto& x : w) x = (float)U(rng);
    cudaMemcpy(p->W[l], w.data(), nw * 4, cudaMemcpyHostToDevice);
  }
  const size_t bp = p->bp;
  if (!rc)
    if ((rc = al(p, bp * p->nin_p, &p->xb)) || (rc = al(p, bp * nh1, &p->h1)) || (rc = al(p, bp * nh2, &p->h2)) ||
        (rc = al(p, bp * p->nout_p, &p->dy)) || (rc = al(p, bp * nh2, &p->dz2)) || (rc = al(p, bp * nh1, &p->dz1)) ||
        (rc = al(p, bp * nh1, &p->z1)) || (rc = al(p, bp * nh2, &p->z2)) ||
        (rc = al(p, (size_t)nin, &p->mux)) || (rc = al(p, (size_t)nin, &p->sdx)) || (rc = al(p, (size_t)nout, &p->muy)) ||
        (rc = al(p, (size_t)nout, &p->sdy)) || (rc = al(p, 1, &p->loss)) || (rc = al(p, 1, &p->err))) {
    }
  if (rc) {
    pf_mlp_destroy(p);
    return rc;
  }
  // identity standardisation until pf_mlp_set_norm is called
  std::vector<float> zeros(std::max(nin, nout), 0.f), ones(std::max(nin, nout), 1.f);
  cudaMemcpy(p->mux, zeros.data(), nin * 4, cudaMemcpyHostToDevice);
  cudaMemcpy(p->sdx, ones.data(), nin * 4, cudaMemcpyHostToDevice);
  cudaMemcpy(p->muy, zeros.data(), nout * 4, cudaMemcpyHostToDevice);
  cudaMemcpy(p->sdy, ones.data(), nout * 4, cudaMemcpyHostToDevice);
  refresh_bf16(p, nullptr);
  if (cudaDeviceSynchronize() != cudaSuccess) {
    pf_mlp_destroy(p);
    return NRPF_ERR_CUDA;
  }
  *out = p;
  return NRPF_OK;
}

int pf_mlp_set_norm(pf_mlp* p, const float* mux, const float* sdx, const float* muy, const float* sdy) {
  if (!p || !mux || !sdx || !muy || !sdy) return NRPF_ERR_ARG;
  cudaMemcpy(p->mux, mux, p->nin * 4, cudaMemcpyHostToDevice);
  cudaMemcpy(p->sdx, sdx, p->nin * 4, cudaMemcpyHostToDevice);
  cudaMemcpy(p->muy, muy, p->nout * 4, cudaMemcpyHostToDevice);
  cudaMemcpy(p->sdy, sdy, p->nout * 4, cudaMemcpyHostToDevice);
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

int pf_mlp_params(pf_mlp* p, int set, float* const* host) {
  if (!p || !host) return NRPF_ERR_ARG;
  cudaDeviceSynchronize();
  for (int l = 0; l < 3; ++l) {
    const size_t nw = (size_t)p->fout[l] * p->fin[l];
    if (!host[2 * l] || !host[2 * l + 1]) return NRPF_ERR_ARG;
    if (set) {
      cudaMemcpy(p->W[l], host[2 * l], nw * 4, cudaMemcpyHostToDevice);
      cudaMemcpy(p->b[l], host[2 * l + 1], p->fout[l] * 4, cudaMemcpyHostToDevice);
    } else {
      cudaMemcpy(host[2 * l], p->W[l], nw * 4, cudaMemcpyDeviceToHost);
      cudaMemcpy(host[2 * l + 1], p->b[l], p->fout[l] * 4, cudaMemcpyDeviceToHost);
    }
  }
  if (set) {
    refresh_bf16(p, nullptr);
    p->step = 0;
    for (int l = 0; l < 3; ++l) {
      cudaMemset(p->mW[l], 0, (size_t)p->fout[l] * p->fin[l] * 4);
      cudaMemset(p->vW[l], 0, (size_t)p->fout[l] * p->fin[l] * 4);
      cudaMemset(p->mb[l], 0, p->fout[l] * 4);
      cudaMemset(p->vb[l], 0, p->fout[l] * 4);
    }
  }
  return cudaDeviceSynchronize() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

int pf_mlp_grads(pf_mlp* p, float* const* host) {
  if (!p || !host) return NRPF_ERR_ARG;
  cudaDeviceSynchronize();
  for (int l = 0; l < 3; ++l) {
    cudaMemcpy(host[2 * l], p->gW[l], (size_t)p->fout[l] * p->fin[l] * 4, cudaMemcpyDeviceToHost);
    cudaMemcpy(host[2 * l + 1], p->gb[l], p->fout[l] * 4, cudaMemcpyDeviceToHost);
  }
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

int pf_mlp_predict(pf_mlp* p, int B, const float* x, float* y, void* stream) {
  if (!p || B < 0 || B > p->bmax) return B > 0 && p && B > p->bmax ? NRPF_ERR_CAPACITY : NRPF_ERR_ARG;
  if (B == 0) return NRPF_OK;
  if (!x || !y) return NRPF_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int rc = forward_hidden(p, B, x, false, st);
  if (rc) return rc;
  return nrpf::gemm(p->h2, p->Wb[2], nrpf::rup(B, nrpf::kGemmBM), p->nout_p, p->fin_p[2],
                    nrpf::EpiUnstd{p->b[2], p->muy, p->sdy, y, B, p->nout}, p->err, st);
}

int pf_mlp_train_step(pf_mlp* p, int B, const float* x, const float* t, float lr, float wd, int update,
                      float* loss_out, void* stream) {
  using namespace nrpf;
  if (!p || B <= 0 || B > p->bmax || !x || !t) return p && B > p->bmax ? NRPF_ERR_CAPACITY : NRPF_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int Bp = rup(B, kGemmBM);
  int rc = forward_hidden(p, B, x, true, st);
  if (rc) return rc;
  // Every product of the backward pass reads its operands as they are stored
  // (the tensor core takes either order), writes what the next one reads, and
  // no padded gradient is copied: with transposed copies of all activations,
  // gradients and weights, and separate passes for the loss, GELU' and the
  // gradients' padding, a step of 1,024 rows took 34 launches and 610 us.
  cudaMemsetAsync(p->loss, 0, sizeof(double), st);
  if ((rc = gemm(p->h2, p->Wb[2], Bp, p->nout_p, p->nh2,
                 EpiLoss{p->b[2], t, p->muy, p->sdy, p->dy, p->loss, B, p->nout, p->nout_p}, p->err, st)))
    return rc;
  // layer 3: dW3 = dY^T H2, dZ2 = (dY W3) GELU'(Z2)
  if ((rc = gemm<true, true>(p->dy, p->h2, p->nout_p, p->nh2, Bp, EpiF32{p->gW[2], p->nout, p->nh2}, p->err, st)))
    return rc;
  k_colsum<<<p->nout_p / 64, 288, 0, st>>>(p->dy, p->gb[2], Bp, p->nout_p, p->nout);
  if ((rc = gemm<false, true>(p->dy, p->Wb[2], Bp, p->nh2, p->nout_p, EpiGeluBack{p->z2, p->dz2, B, p->nh2, p->nh2},
                              p->err, st)))
    return rc;
  // layer 2
  if ((rc = gemm<true, true>(p->dz2, p->h1, p->nh2, p->nh1, Bp, EpiF32{p->gW[1], p->nh2, p->nh1}, p->err, st)))
    return rc;
  k_colsum<<<p->nh2 / 64, 288, 0, st>>>(p->dz2, p->gb[1], Bp, p->nh2, p->nh2);
  if ((rc = gemm<false, true>(p->dz2, p->Wb[1], Bp, p->nh1, p->nh2, EpiGeluBack{p->z1, p->dz1, B, p->nh1, p->nh1},
                              p->err, st)))
    return rc;
  // layer 1
  if ((rc = gemm<true, true>(p->dz1, p->xb, p->nh1, p->nin_p, Bp, EpiF32{p->gW[0], p->nh1, p->nin}, p->err, st)))
    return rc;
  k_colsum<<<p->nh1 / 64, 288, 0, st>>>(p->dz1, p->gb[0], Bp, p->nh1, p->nh1);
  if (update) {
    p->step += 1;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - (float)std::pow(b1, (double)p->step), c2 = 1.f - (float)std::pow(b2, (double)p->step);
    AdamSet a{};
    for (int l = 0; l < 3; ++l) {
      const int w = 2 * l, bi = 2 * l + 1;
      a.p[w] = p->W[l]; a.g[w] = p->gW[l]; a.m[w] = p->mW[l]; a.v[w] = p->vW[l]; a.pb[w] = p->Wb[l];
      a.n[w] = (int64_t)p->fout[l] * p->fin[l]; a.cols[w] = p->fin[l]; a.ld[w] = p->fin_p[l]; a.wd[w] = wd;
      a.p[bi] = p->b[l]; a.g[bi] = p->gb[l]; a.m[bi] = p->mb[l]; a.v[bi] = p->vb[l]; a.pb[bi] = nullptr;
      a.n[bi] = p->fout[l]; a.cols[bi] = 1; a.ld[bi] = 1; a.wd[bi] = 0.f;
    }
    for (int k = 0; k < 6; ++k) a.first[k + 1] = a.first[k] + nb(a.n[k], 1024);
    k_adamw<<<a.first[6], 256, 0, st>>>(a, lr, b1, b2, eps, c1, c2);
  }
  if (loss_out) k_loss_out<<<1, 1, 0, st>>>(p->loss, (double)B * (double)p->nout, loss_out);
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

}  // extern "C"

namespace {
// per-column mean and standard deviation of a [B][n] FP32 matrix (FP64 sums)
__global__ void k_colstats(const float* __restrict__ X, int64_t B, int n, float* __restrict__ mu,
                           float* __restrict__ sd) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  double s = 0.0;
  for (int64_t r = 0; r < B; ++r) s += X[r * n + c];
  const double m = s / (double)B;
  double q = 0.0;
  for (int64_t r = 0; r < B; ++r) {
    const double d = X[r * n + c] - m;
    q += d * d;
  }
  const double v = q / (double)B;
  mu[c] = (float)m;
  sd[c] = v > 1e-24 ? (float)sqrt(v) : 1.0f;  // constant features keep unit scale
}
}  // namespace

extern "C" {

int pf_mlp_fit_norm(pf_mlp* p, int64_t B, const float* X, const float* T, void* stream) {
  if (!p || B <= 0 || !X || !T) return NRPF_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  k_colstats<<<nrpf::nb(p->nin), 256, 0, st>>>(X, B, p->nin, p->mux, p->sdx);
  k_colstats<<<nrpf::nb(p->nout), 256, 0, st>>>(T, B, p->nout, p->muy, p->sdy);
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

int pf_mlp_error(pf_mlp* p) {
  if (!p) return NRPF_ERR_ARG;
  int e = 0;
  cudaMemcpy(&e, p->err, 4, cudaMemcpyDeviceToHost);
  return e;
}

void pf_mlp_destroy(pf_mlp* p) {
  if (!p) return;
  cudaDeviceSynchronize();
  for (void* a : p->allocs) cudaFree(a);
  delete p;
}

// ---- warm-start glue between the solver's layouts and the network's ----
}  // extern "C"

namespace {
// features: X[b] = [P_0 .. P_{n-1}, Q_0 .. Q_{n-1}] from sbus [B, n] complex
__global__ void k_ws_features(int n, int B, const double2* __restrict__ sbus, float* __restrict__ X) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * n) return;
  const int64_t b = i / n;
  const int k = (int)(i % n);
  const double2 s = sbus[i];
  X[b * 2 * n + k] = (float)s.x;
  X[b * 2 * n + n + k] = (float)s.y;
}
// targets: T[b] = [|V| of non-slack buses, angles of non-slack buses] (ascending bus order)
__global__ void k_ws_targets(int n, int B, const int32_t* __restrict__ nsidx, const double2* __restrict__ V,
                             float* __restrict__ T, int nns) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * n) return;
  const int64_t b = i / n;
  const int k = (int)(i % n);
  const int q = nsidx[k];
  if (q < 0) return;
  const double2 v = V[i];
  T[b * 2 * nns + q] = (float)sqrt(v.x * v.x + v.y * v.y);
  T[b * 2 * nns + nns + q] = (float)atan2(v.y, v.x);
}
// V0 from a prediction: slack keeps v_flat, PV keeps |v_flat| with the
// predicted angle, PQ takes the predicted magnitude and angle
__global__ void k_ws_v0(int n, int B, const int32_t* __restrict__ nsidx, const int8_t* __restrict__ bt,
                        const float* __restrict__ Y, const double2* __restrict__ vflat, double2* __restrict__ v0,
                        int nns) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * n) return;
  const int64_t b = i / n;
  const int k = (int)(i % n);
  const double2 vf = vflat[i];
  const int q = nsidx[k];
  if (q < 0 || bt[k] == 3) {
    v0[i] = vf;
    return;
  }
  double mag = bt[k] == 2 ? sqrt(vf.x * vf.x + vf.y * vf.y) : (double)Y[b * 2 * nns + q];
  if (!(mag > 0.0) || !(mag < 10.0)) mag = sqrt(vf.x * vf.x + vf.y * vf.y);  // keep the guess sane
  double ang = (double)Y[b * 2 * nns + nns + q];
  if (!(fabs(ang) < 10.0)) ang = 0.0;
  double sn, cs;
  sincos(ang, &sn, &cs);
  v0[i] = make_double2(mag * cs, mag * sn);
}

// Screen of warm-started results: one warp per instance takes min |V|^2 over
// its buses; the instance is redone from flat start when it did not converge,
// or when some magnitude is below vmin (a low-voltage root of the power-flow
// equations, reached from a guess far from the operating point) or not finite.
__global__ void k_ws_screen(int n, int B, const double2* __restrict__ v, const uint8_t* __restrict__ status,
                            double vmin2, uint8_t* __restrict__ redo) {
  const int b = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (b >= B) return;
  const double2* vb = v + (size_t)b * n;
  double lo = INFINITY;
  bool finite = true;
  for (int k = lane; k < n; k += 32) {
    const double2 x = vb[k];
    const double m2 = x.x * x.x + x.y * x.y;
    finite = finite && isfinite(m2);
    lo = fmin(lo, m2);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
  finite = __all_sync(0xffffffffu, finite);
  if (lane == 0) redo[b] = (status[b] != 0 || !finite || lo < vmin2) ? 1 : 0;
}
}  // namespace

extern "C" {

int pf_warmstart_features(int n, int B, const double* sbus, float* X, void* stream) {
  if (n <= 0 || B < 0 || (B > 0 && (!sbus || !X))) return NRPF_ERR_ARG;
  if (B == 0) return NRPF_OK;
  k_ws_features<<<nrpf::nb((int64_t)B * n), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      n, B, reinterpret_cast<const double2*>(sbus), X);
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

int pf_warmstart_targets(int n, int B, const int32_t* nsidx, int nns, const double* v, float* T, void* stream) {
  if (n <= 0 || B < 0 || nns <= 0 || (B > 0 && (!nsidx || !v || !T))) return NRPF_ERR_ARG;
  if (B == 0) return NRPF_OK;
  k_ws_targets<<<nrpf::nb((int64_t)B * n), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      n, B, nsidx, reinterpret_cast<const double2*>(v), T, nns);
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

int pf_warmstart_v0(int n, int B, const int32_t* nsidx, const int8_t* bus_type, int nns, const float* Y,
                    const double* v_flat, double* v0, void* stream) {
  if (n <= 0 || B < 0 || nns <= 0 || (B > 0 && (!nsidx || !bus_type || !Y || !v_flat || !v0))) return NRPF_ERR_ARG;
  if (B == 0) return NRPF_OK;
  k_ws_v0<<<nrpf::nb((int64_t)B * n), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      n, B, nsidx, bus_type, Y, reinterpret_cast<const double2*>(v_flat), reinterpret_cast<double2*>(v0), nns);
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

int pf_warmstart_screen(int n, int B, const double* v, const uint8_t* status, double vmin, uint8_t* redo,
                        void* stream) {
  if (n <= 0 || B < 0 || !(vmin >= 0.0) || (B > 0 && (!v || !status || !redo))) return NRPF_ERR_ARG;
  if (B == 0) return NRPF_OK;
  k_ws_screen<<<(B + 7) / 8, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      n, B, reinterpret_cast<const double2*>(v), status, vmin * vmin, redo);
  return cudaGetLastError() == cudaSuccess ? NRPF_OK : NRPF_ERR_CUDA;
}

// Standalone tensor-core GEMM: C[M,N] (FP32) = A[M,K] B[N,K]^T (BF16, row-major).
int pf_gemm_bf16(const void* A, const void* B, float* C, int M, int N, int K, int variant, int* err,
                 void* stream) {
  if (!A || !B || !C || !err || variant < 0 || variant > 1) return NRPF_ERR_ARG;
  return nrpf::gemm(reinterpret_cast<const bf16*>(A), reinterpret_cast<const bf16*>(B), M, N, K, nrpf::EpiF32{C, M, N},
                    err, reinterpret_cast<cudaStream_t>(stream), variant);
}

int pf_gemm_set_variant(int variant) {
  if (variant < 0 || variant > 1) return NRPF_ERR_ARG;
  nrpf::g_gemm_variant = variant;
  return NRPF_OK;
}

}  // extern "C"
