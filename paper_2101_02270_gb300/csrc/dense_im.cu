// Instance-major dense block for the FP32 LU (Sec. 4.3: the serial tail of the
// column DAG, factorised as one dense matrix per instance).
//
// In the interleaved layout every lane of a warp is its own instance, so the
// 32 threads of a warp never share an operand and the trailing update can
// only reuse data through a per-thread register tile.  Here instance b's
// dense block is its own column-major ndp x ndp matrix,
//   element (r, c) at lu + ((b / 32) * NLU + NS) * 32 + (b % 32) * ndp^2 + c * ndp + r,
// inside the same per-tile LU array (only the order of the dense part
// changes; ndp is a multiple of 64).  The factorisation is blocked, without
// pivoting, and left-looking by outer panels (blocked Crout).  Outer panel j
// at column kj = 128 j, of width 128 (64 for the last one when ndp % 128 ==
// 64):
//   k_im_gemm          : (j > 0) its block column and row, rows [kj, ndp) x
//                        columns [kj, kj+128) and rows [kj, kj+128) x columns
//                        [kj+128, ndp), minus the products of all earlier
//                        panels in one pass of depth kj, one 128 x 128 tile
//                        of C per CTA: on the tensor cores, from operands
//                        split into three BF16 parts each, or near the
//                        solution by packed two-wide FP32 FMAs (an 8 x 8
//                        register tile per thread, operand chunks of depth 32
//                        loaded by TMA into a two-stage ring);
//   k_im_diag  (step 0): LU of the 64 x 64 diagonal block at (kj, kj), and the
//                        inverses U11^-1, L11^-1 of its factors;
//   k_im_panel (step 0): L21 = A21 U11^-1 for the rows below and
//                        U12 = L11^-1 A12 for the columns to the right, as
//                        register-tiled products on 128 x 64 tiles;
//   k_im_diag  (step 1): block (kj+64, kj+64) minus L(., kj:kj+64) U(kj:kj+64, .),
//                        then its LU and inverses;
//   k_im_panel (step 1): rows below / columns right of kj+128, each first minus
//                        its product with step 0's L or U, then multiplied by
//                        the inverse.
// Every entry of the block is read and written by k_im_gemm once per
// refactorisation (a right-looking order would rewrite the trailing block
// after every outer panel), and each entry still takes its subtractions in
// ascending pivot order, as the interleaved kernels do.  The panel multiplies
// by the explicit inverses of the 64 x 64 diagonal factors (the LU is the
// FP32 inner solve of an inexact Newton step whose mismatch and update stay
// FP64).
#include <cfloat>
#include <cstdint>

#include "dense_im.h"
#include "gemm_tc.cuh"
#include "kernels.h"

namespace nrpf {

namespace {

constexpr int kImOuter = 128;               // outer panel width
constexpr int kImTile = 128;                // GEMM tile (rows and columns of C)
constexpr int kImKc = 32;                   // GEMM depth per stage
constexpr int kImStages = 2;
// column groups of 32 per warp in the block update (four columns of each per
// thread): 2 (an 8 x 8 register tile, 8 warps per CTA) or 4 (8 x 16, 4 warps).
// The wider tile needs fewer shared-memory wavefronts per FMA but leaves half
// the warps; measured on the 9,000-bus update it is 1 % slower, so the 8 x 8
// tile is used.
constexpr int kImGC = 2;
// packed two-wide FP32 FMA (fma.rn.f32x2) in the trailing update: each
// instruction updates two rows of a column; the B chunk is negated while it is
// transposed, so acc + a (-b) rounds exactly as fmaf(-a, b, acc)
constexpr bool kImPacked = true;
constexpr int kImGemmThreads = 32 * 4 * (4 / kImGC);
static_assert(kImGemmThreads == 256, "the tensor-core form splits its work over eight warps");
constexpr uint32_t kImABytes = kImKc * kImTile * 4;  // 16 KB: [32 columns][128 rows]
constexpr uint32_t kImBBytes = kImTile * kImKc * 4;  // 16 KB: [128 columns][32 rows], swizzled
constexpr uint32_t kImStageBytes = kImABytes + kImBBytes;
// two TMA stages, the double-buffered transposed B chunk, 1024-byte alignment slack
constexpr size_t kImGemmSmem = (size_t)kImStages * kImStageBytes + 2 * (size_t)kImKc * kImTile * 4 + 1024;
// bounded wait on the TMA completion barriers (each try_wait also suspends
// for a hardware-defined time window)
constexpr uint32_t kImSpinLimit = 1u << 20;

constexpr int kImDiagThreads = 128;
constexpr int kImSolveThreads = 256;
constexpr int kPitch = 68;  // shared row pitch (floats) of 64-wide blocks: rows stay 16-byte aligned

__device__ __forceinline__ float* im_block(const DevPlan& P, const DevState& S, int b) {
  return reinterpret_cast<float*>(S.lu) + ((size_t)(b >> 5) * (size_t)P.NLU + (size_t)P.NS) * kTile +
         (size_t)(b & 31) * (size_t)P.ndp * (size_t)P.ndp;
}

__device__ __forceinline__ uint32_t su32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte asynchronous copy global -> shared (no register staging)
__device__ __forceinline__ void cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(su32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp16_wait_all() {
  asm volatile("cp.async.commit_group;\n cp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void bar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void bar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t spins = 0; spins < kImSpinLimit; ++spins) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ void tma_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                       uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(su32(bar))
      : "memory");
}

__device__ __forceinline__ float comp(const float4& v, int q) {
  return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w;
}

// ---------------------------------------------------------------------------
// Update C -= A B of one 128 x 128 tile of one instance, over the depth of the
// pivot columns k .. k + 32 nkc - 1, the tile held in registers throughout.
// Per chunk of depth 32, TMA lands the A chunk (As[kk][i] = A(i0 + i, k + 32 kc
// + kk), 512 bytes per kk) and the B chunk as 128 rows of 128 bytes (row j =
// B(k + 32 kc + 0..31, j0 + j), 16-byte chunk q stored at chunk q ^ (j % 8):
// TMA 128-byte swizzle) in a two-stage ring.  The CTA first transposes the B
// chunk into Bt[kk][j] (double-buffered, so one barrier per chunk suffices),
// then every thread runs the register-tiled product: per kk two 16-byte loads
// of A and two of B feed 64 FMAs, the next kk's fragments loaded while the
// current ones are used.
// Warp w = (wy, wx), wy = w % 4, wx = w / 4, owns the 32 x (32 kImGC) block at
// rows 32 wy, columns 32 kImGC wx of the tile; its lane (lx, ly), lx = lane % 8,
// ly = lane / 8, owns rows 32 wy + ly*4 + 16h + q and columns 32 kImGC wx +
// lx*4 + 32g + r (h < 2, g < kImGC; q, r < 4).  Every shared load of a warp then touches four
// (A) or eight (B) distinct 16-byte words of one 128-byte row: one wavefront.
// A tile whose rows (columns) run past ndp has 64 of them; the warps outside
// skip the arithmetic (the TMA box past ndp is filled with zeros, unused).
// Returns the chunk whose wait ran out, or -1.
// ---------------------------------------------------------------------------

// TMA copies of GEMM chunk kc (A: 128 rows x 32 columns, B: 32 rows x 128
// columns of instance (tile_b, lane_b)) into stage kc % kImStages
__device__ __forceinline__ void issue_chunk(uint8_t* sm, uint64_t* full, const CUtensorMap* tmA,
                                            const CUtensorMap* tmB, int kc, int i0, int j0, int k, int lane_b,
                                            int tile_b) {
  const int s = kc % kImStages;
  const uint32_t sa = su32(sm) + (uint32_t)s * kImStageBytes;
  // order the generic-proxy reads of this stage before the async-proxy writes
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  bar_expect_tx(&full[s], kImStageBytes);
  tma_4d(sa, tmA, i0, k + kc * kImKc, lane_b, tile_b, &full[s]);
  tma_4d(sa + kImABytes, tmB, k + kc * kImKc, j0, lane_b, tile_b, &full[s]);
}

__device__ __forceinline__ void fma_kk(float (&acc)[2][kImGC][4][4], const float4 (&a)[2],
                                       const float4 (&b)[kImGC]) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int g = 0; g < kImGC; ++g)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float bv = comp(b[g], r);
        float* d = acc[h][g][r];
        d[0] = fmaf(-a[h].x, bv, d[0]);
        d[1] = fmaf(-a[h].y, bv, d[1]);
        d[2] = fmaf(-a[h].z, bv, d[2]);
        d[3] = fmaf(-a[h].w, bv, d[3]);
      }
}

// the same update on packed pairs: acc2[h][g][r][p] = rows 2p, 2p+1 of the
// thread's 4-row group h, column g, r; b holds -B
__device__ __forceinline__ void fma_kk2(float2 (&acc)[2][kImGC][4][2], const float4 (&a)[2],
                                        const float4 (&b)[kImGC]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 a01 = make_float2(a[h].x, a[h].y), a23 = make_float2(a[h].z, a[h].w);
#pragma unroll
    for (int g = 0; g < kImGC; ++g)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float bv = comp(b[g], r);
        const float2 b2 = make_float2(bv, bv);
        acc[h][g][r][0] = __ffma2_rn(a01, b2, acc[h][g][r][0]);
        acc[h][g][r][1] = __ffma2_rn(a23, b2, acc[h][g][r][1]);
      }
  }
}

__device__ __forceinline__ int gemm_tile(float* __restrict__ C, int ld, int i0, int j0, int k, int nkc, uint8_t* sm,
                                         uint64_t* full, const CUtensorMap* tmA, const CUtensorMap* tmB, int lane_b,
                                         int tile_b, bool active, int rw, int cw, int lx, int ly) {
  // acc[h][g][r][q] (acc2: the same as pairs of q): row rw + ly*4 + 16h + q,
  // column cw + lx*4 + 32g + r
  float acc[2][kImGC][4][4];
  float2 acc2[2][kImGC][4][2];
  const size_t cstride = (size_t)ld;
  if (active) {
    const float* __restrict__ Ct = C + (size_t)(j0 + cw + lx * 4) * ld + i0 + rw + ly * 4;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int g = 0; g < kImGC; ++g)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float4 v = *reinterpret_cast<const float4*>(Ct + (size_t)(32 * g + r) * cstride + 16 * h);
          if constexpr (kImPacked) {
            acc2[h][g][r][0] = make_float2(v.x, v.y);
            acc2[h][g][r][1] = make_float2(v.z, v.w);
          } else {
            acc[h][g][r][0] = v.x;
            acc[h][g][r][1] = v.y;
            acc[h][g][r][2] = v.z;
            acc[h][g][r][3] = v.w;
          }
        }
  }
  float* Bt0 = reinterpret_cast<float*>(sm + (size_t)kImStages * kImStageBytes);
  const int tid = threadIdx.x;
#pragma unroll 1
  for (int kc = 0; kc < nkc; ++kc) {
    const int s = kc % kImStages;
    const bool ok = bar_wait(&full[s], (uint32_t)(kc / kImStages) & 1u);
    // transpose the B chunk: thread tid takes column j = tid % 128 and the
    // 16-byte words q = tid / 128, tid / 128 + 2, ... of its row
    float* Bt = Bt0 + (kc & 1) * (kImKc * kImTile);
    {
      const uint8_t* Bs = sm + (size_t)s * kImStageBytes + kImABytes;
      const int j = tid & (kImTile - 1);
#pragma unroll
      for (int q = tid >> 7; q < kImKc / 4; q += kImGemmThreads / kImTile) {
        const float4 v = *reinterpret_cast<const float4*>(Bs + j * 128 + ((q ^ (j & 7)) << 4));
        const float sg = kImPacked ? -1.f : 1.f;
        Bt[(4 * q) * kImTile + j] = sg * v.x;
        Bt[(4 * q + 1) * kImTile + j] = sg * v.y;
        Bt[(4 * q + 2) * kImTile + j] = sg * v.z;
        Bt[(4 * q + 3) * kImTile + j] = sg * v.w;
      }
    }
    // one barrier: the chunk has landed for everyone, Bt is complete, and
    // every warp is done with chunk kc - 1 (its stage may be refilled)
    if (__syncthreads_or(!ok)) return kc;
    if (kc >= 1 && kc + 1 < nkc && tid == 0)
      issue_chunk(sm, full, tmA, tmB, kc + 1, i0, j0, k, lane_b, tile_b);
    if (active) {
      const float* As = reinterpret_cast<const float*>(sm + (size_t)s * kImStageBytes) + rw + ly * 4;
      const float* Bq = Bt + cw + lx * 4;
      float4 a[2], b[kImGC];
      a[0] = *reinterpret_cast<const float4*>(As);
      a[1] = *reinterpret_cast<const float4*>(As + 16);
#pragma unroll
      for (int g = 0; g < kImGC; ++g) b[g] = *reinterpret_cast<const float4*>(Bq + 32 * g);
#pragma unroll 8
      for (int kk = 0; kk < kImKc - 1; ++kk) {
        float4 an[2], bn[kImGC];
        an[0] = *reinterpret_cast<const float4*>(As + (kk + 1) * kImTile);
        an[1] = *reinterpret_cast<const float4*>(As + (kk + 1) * kImTile + 16);
#pragma unroll
        for (int g = 0; g < kImGC; ++g) bn[g] = *reinterpret_cast<const float4*>(Bq + (kk + 1) * kImTile + 32 * g);
        if constexpr (kImPacked) fma_kk2(acc2, a, b);
        else fma_kk(acc, a, b);
        a[0] = an[0];
        a[1] = an[1];
#pragma unroll
        for (int g = 0; g < kImGC; ++g) b[g] = bn[g];
      }
      if constexpr (kImPacked) fma_kk2(acc2, a, b);
      else fma_kk(acc, a, b);
    }
  }
  if (active) {
    float* __restrict__ Ct = C + (size_t)(j0 + cw + lx * 4) * ld + i0 + rw + ly * 4;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int g = 0; g < kImGC; ++g)
#pragma unroll
        for (int r = 0; r < 4; ++r)
          *reinterpret_cast<float4*>(Ct + (size_t)(32 * g + r) * cstride + 16 * h) =
              kImPacked ? make_float4(acc2[h][g][r][0].x, acc2[h][g][r][0].y, acc2[h][g][r][1].x, acc2[h][g][r][1].y)
                        : make_float4(acc[h][g][r][0], acc[h][g][r][1], acc[h][g][r][2], acc[h][g][r][3]);
  }
  return -1;
}

__device__ __forceinline__ void update_fma(float* __restrict__ A, int ld, int i0, int j0, int nkc, uint8_t* sm,
                                           uint64_t* full, const CUtensorMap* tmA, const CUtensorMap* tmB, int lane_b,
                                           int tile_b, int32_t* bad) {
  const int k = 0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rw = (warp & 3) * 32, cw = (warp >> 2) * 32 * kImGC;
  if (tid == 0) {
    for (int s = 0; s < kImStages; ++s) bar_init(&full[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (tid == 0)
    for (int kc = 0; kc < kImStages && kc < nkc; ++kc)
      issue_chunk(sm, full, tmA, tmB, kc, i0, j0, k, lane_b, tile_b);
  // rows (columns) of this tile inside the block: 128, or 64 at the edge
  const int mrows = ld - i0 < kImTile ? ld - i0 : kImTile;
  const int ncols = ld - j0 < kImTile ? ld - j0 : kImTile;
  const bool active = rw < mrows && cw < ncols;
  const int fail = gemm_tile(A, ld, i0, j0, k, nkc, sm, full, tmA, tmB, lane_b, tile_b, active, rw, cw,
                             lane & 7, lane >> 3);
  if (fail >= 0 && tid == 0) {
    // a copy did not land in time: the instance is marked failed (its step
    // is discarded) and the CTA waits, bounded, for the copies it issued
    // (chunks up to fail + 1: one chunk ahead of the one consumed)
    *bad = 1;
    const int issued = fail + 2 < nkc ? fail + 2 : nkc;
    for (int kc = fail; kc < issued; ++kc) bar_wait(&full[kc % kImStages], (uint32_t)(kc / kImStages) & 1u);
  }
}

// ---------------------------------------------------------------------------
// Update C -= A B of one 128 x 128 tile of one instance over the pivot columns
// 0 .. r0-1, as an FP32 product on the BF16 tensor cores.
//
// Each operand is split into three BF16 parts, x = h + m + l with h = bf16(x),
// m = bf16(x - h), l = bf16(x - h - m): 24 bits, the whole FP32 significand
// (the method of Henry, Tang & Heinecke, "Leveraging the bfloat16 Artificial
// Intelligence Datatype for Higher-Precision Computations", ARITH 2019).  Of
// the nine partial products the six above 2^-24 are taken, smallest first:
//   Ah Bl + Al Bh + Am Bm + Am Bh + Ah Bm + Ah Bh   (Am Bl, Al Bm: <= 2^-25)
// each exact in the FP32 accumulator's inputs.  The accumulator holds the sum of
// one chunk of depth 32 only; the chunk's sum is then added to C in FP32 with
// rounding to nearest, so the tensor core's own rounding acts on sums of 32
// products and C is rounded once per chunk instead of once per product.
// Error of J^-1 F against FP64 with all updates in this form, and by FP32 FMAs
// (meshed grids, 32 instances, the first Newton step; median of |dx - dx64| /
// |dx64|):
//   buses         700      2,000    4,000    9,000
//   dense block   192      320      768      2,176
//   this form     5.6e-7   1.6e-6   4.3e-6   6.6e-5
//   FP32 FMAs     2.1e-6   1.9e-6   8.5e-6   4.9e-4
//
// Data flow per chunk of depth 32 (256 threads, eight warps):
//  * A (columns of L, rows contiguous): warp w reads its 32 rows (w % 4), one
//    128-byte line per column, 16 columns (w / 4), a chunk ahead into
//    registers; a thread holds a row, so pairs of its columns are what a TMEM
//    operand's 32-bit columns take: the parts go to TMEM (tcgen05.st), and the
//    MMA reads A from there, which leaves shared memory to B;
//  * B (columns of U, depth contiguous): 16 bytes of depth per thread and column,
//    eight threads a line; the parts go to shared memory as 64-byte rows with
//    64-byte swizzle (K-major; the 8-byte stores of a half warp cover all banks);
//  * thread 0 issues 2 x 6 MMAs of 128 x 128 x 16 and commits them; meanwhile
//    the next chunk is split into the other buffer, then all warps add the
//    finished chunk to C in registers (one row, 64 columns per thread).
// Two CTAs run on an SM (128 registers, 256 of 512 TMEM columns each): the MMAs
// of one cover the conversion, the barrier and the read-back of the other.
//
// Bounds, per instance and refactorisation of the 2,176-wide block: 37.6 GFLOP
// of BF16 products (20 us at the measured cuBLAS rate), 140.5 MB of DRAM (21 us)
// and 196 MB through L2.  Measured, 1,000 instances: 36.6 us each (171 TFLOP/s
// of FP32 products); by FP32 FMAs 104.8 us (60 TFLOP/s, 0.77 of the FMA peak).
// ---------------------------------------------------------------------------
constexpr uint32_t kImAccCols = 128;                  // TMEM columns of the accumulator
constexpr uint32_t kImACols = 3 * kImKc / 2;          // ... of one A buffer (three parts, two values a column)
constexpr uint32_t kImTmemCols = 256;                 // allocated: 128 + 2 * 48, rounded up to a power of two
constexpr uint32_t kImBPart = kImTile * kImKc * 2;    // 8 KB: one part of a B chunk
constexpr uint32_t kImBBuf = 3 * kImBPart;
constexpr size_t kImGemmTcSmem = 2 * (size_t)kImBBuf + 1024;

// the three BF16 parts of two FP32 values, packed (x0 in the low half)
__device__ __forceinline__ void split3(float x0, float x1, uint32_t& h, uint32_t& m, uint32_t& l) {
  const float2 minus1 = make_float2(-1.f, -1.f);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(x1), "f"(x0));
  // x - part is exact in FP32
  float2 r = __ffma2_rn(make_float2(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u)), minus1,
                        make_float2(x0, x1));
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(r.y), "f"(r.x));
  r = __ffma2_rn(make_float2(__uint_as_float(m << 16), __uint_as_float(m & 0xffff0000u)), minus1, r);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(r.y), "f"(r.x));
}

// Shared-memory descriptor, K-major rows of 64 bytes with 64-byte swizzle:
// 8-row atoms of 512 B (stride byte offset), layout type 4.
__device__ __forceinline__ uint64_t make_sdesc_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// D (+)= A B with A in TMEM (a row per lane, two BF16 per column)
__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3])
               : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void update_tc(float* __restrict__ A, int ld, int i0, int j0, int nkc, uint8_t* sm,
                                          uint64_t* done, uint32_t* tmem_holder, int32_t* bad) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) tmem_alloc(tmem_holder, kImTmemCols);
  if (tid == 0) {
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // this thread's row of A and C, its half of the columns of C and of A's depth
  const int rg = warp & 3, half = warp >> 2;
  const int row = i0 + rg * 32 + lane;
  const bool rok = row < ld;             // uniform over a warp: ld % 64 == 0
  const bool cok = j0 + half * 64 < ld;  // the half's 64 columns of C
  const float* __restrict__ Ap = A + (size_t)(half * 16) * ld + row;
  // its four columns of B, four of depth in each
  const int bq = tid & 7, bj = tid >> 3;
  const float* __restrict__ Bp = A + (size_t)(j0 + bj) * ld + 4 * bq;
  const uint32_t boff = (uint32_t)bj * 64u + ((((uint32_t)bq >> 1) ^ (((uint32_t)bj >> 1) & 3u)) << 4) +
                        ((uint32_t)bq & 1u) * 8u;
  float a[16];
  float4 bv[4];
  auto load = [&](int kc) {
    const size_t k = (size_t)kc * kImKc;
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] = rok ? Ap[(k + q) * ld] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      bv[i] = j0 + bj + 32 * i < ld ? *reinterpret_cast<const float4*>(Bp + (size_t)(32 * i) * ld + k)
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  load(0);
  float c[64];
  float* __restrict__ C = A + (size_t)(j0 + half * 64) * ld + row;
  if (rok && cok) {
#pragma unroll
    for (int q = 0; q < 64; ++q) c[q] = C[(size_t)q * ld];
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_holder;
  const uint32_t lane_base = tmem + ((uint32_t)(rg * 32) << 16);
  // negate A (bit 13): the accumulator holds minus the chunk's product
  constexpr uint32_t idesc = make_idesc_bf16(kImTile, kImTile) | (1u << 13);
  bool ok = true;
  // chunk kc's accumulator into C, once its MMAs have completed
  auto add_chunk = [&](int kc) {
    ok = mbar_wait(done, (uint32_t)kc & 1u);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      float v[16];
      tmem_ld16(lane_base + (uint32_t)(half * 64 + g * 16), v);
#pragma unroll
      for (int q = 0; q < 16; ++q) c[16 * g + q] += v[q];
    }
  };
  int issued = 0;
#pragma unroll 1
  for (int kc = 0; kc < nkc; ++kc) {
    // split chunk kc into buffer kc % 2: the MMAs that read it (chunk kc - 2)
    // were waited for before chunk kc - 1 was issued
    uint8_t* Bs = sm + (kc & 1) * kImBBuf;
    const uint32_t at = lane_base + kImAccCols + (uint32_t)(kc & 1) * kImACols + (uint32_t)half * 8u;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      uint32_t h[4], m[4], l[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) split3(a[8 * g + 2 * q], a[8 * g + 2 * q + 1], h[q], m[q], l[q]);
      tmem_st4(at + 4 * g, h);
      tmem_st4(at + 16 + 4 * g, m);
      tmem_st4(at + 32 + 4 * g, l);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint2 h, m, l;
      split3(bv[i].x, bv[i].y, h.x, m.x, l.x);
      split3(bv[i].z, bv[i].w, h.y, m.y, l.y);
      uint8_t* q = Bs + boff + i * (32 * 64);
      *reinterpret_cast<uint2*>(q) = h;
      *reinterpret_cast<uint2*>(q + kImBPart) = m;
      *reinterpret_cast<uint2*>(q + 2 * kImBPart) = l;
    }
    if (kc + 1 < nkc) load(kc + 1);
    if (kc > 0) add_chunk(kc - 1);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    // both operands are in place and every warp has read the accumulator
    if (__syncthreads_or(!ok)) break;
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t ta = tmem + kImAccCols + (uint32_t)(kc & 1) * kImACols;
      const uint32_t sb = su32(Bs);
      constexpr int pa[6] = {0, 2, 1, 1, 0, 0}, pb[6] = {2, 0, 1, 0, 1, 0};
#pragma unroll
      for (int p = 0; p < 6; ++p)
#pragma unroll
        for (int ks = 0; ks < kImKc / 16; ++ks)
          umma_bf16_ts(tmem, ta + 16 * pa[p] + 8 * ks, make_sdesc_sw64(sb + pb[p] * kImBPart + 32 * ks), idesc,
                       p + ks > 0 ? 1u : 0u);
      umma_commit(done);
    }
    issued = kc + 1;
  }
  if (ok && issued == nkc) add_chunk(nkc - 1);
  if (__syncthreads_or(!ok || issued != nkc)) {
    // the MMAs did not complete in time: the instance is marked failed (its
    // step is discarded), after a second bounded wait before TMEM is freed
    if (tid == 0) *bad = 1;
    if (issued > 0) mbar_wait(done, (uint32_t)(issued - 1) & 1u);
  } else if (rok && cok) {
#pragma unroll
    for (int q = 0; q < 64; ++q) C[(size_t)q * ld] = c[q];
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tmem_dealloc(tmem, kImTmemCols);
  }
}

// The block column and row of the outer panel at r0: tiles of 128 over rows
// [r0, ld) x columns [r0, r0+128) and rows [r0, r0+128) x columns [r0+128,
// ld), 2 ntc - 1 of them (ntc = tiles across [r0, ld)), each minus the
// products over pivot columns 0 .. r0-1 (r0 / 32 chunks).  grid: Bp * (2 ntc
// - 1) CTAs, tile-fastest within an instance, so that the CTAs resident at
// one time share their instance's operand panels in L2.  An instance far from
// its solution takes the tensor cores, one near it the FMA pipe (kActiveNear,
// kernels.h, says why the line lies there): two kernels, whose CTAs leave at once
// where the instance is the other's.  In one kernel the FMA form's 97 KB of shared
// memory per CTA left the tensor-core form, whose operands come through L1, 34 KB
// of it: 49 ms per refactorisation of 1,000 instances of the 9,000-bus grid, 37
// alone.
struct ImTile {
  float* A;
  int b, i0, j0;
};

__device__ __forceinline__ ImTile im_tile(const DevPlan& P, const DevState& S, int r0, int ntc) {
  const int ntile = 2 * ntc - 1;
  const int b = (int)(blockIdx.x / (unsigned)ntile);
  const int t = (int)(blockIdx.x - (unsigned)b * (unsigned)ntile);
  return {im_block(P, S, b), b, r0 + (t < ntc ? t : 0) * kImTile, r0 + (t < ntc ? 0 : t - ntc + 1) * kImTile};
}

// 1024-byte alignment for the swizzled chunks (offset arithmetic on the shared
// array keeps the pointer in the shared address space)
__device__ __forceinline__ uint8_t* align1024(uint8_t* p) { return p + ((1024u - (su32(p) & 1023u)) & 1023u); }

__global__ void __launch_bounds__(kImGemmThreads, 2) k_im_gemm(const __grid_constant__ CUtensorMap tmA,
                                                               const __grid_constant__ CUtensorMap tmB, DevPlan P,
                                                               DevState S, int r0, int ntc,
                                                               const int32_t* __restrict__ gate) {
  extern __shared__ uint8_t im_smem_raw[];
  __shared__ __align__(8) uint64_t bars[kImStages];
  if (gate && *gate == 0) return;
  const ImTile t = im_tile(P, S, r0, ntc);
  if (S.active[t.b] != kActiveNear) return;
  update_fma(t.A, P.ndp, t.i0, t.j0, r0 / kImKc, align1024(im_smem_raw), bars, &tmA, &tmB, t.b & 31, t.b >> 5,
             &S.bad[t.b]);
}

__global__ void __launch_bounds__(kImGemmThreads, 2) k_im_gemm_tc(DevPlan P, DevState S, int r0, int ntc,
                                                                  const int32_t* __restrict__ gate) {
  extern __shared__ uint8_t im_smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_holder;
  if (gate && *gate == 0) return;
  const ImTile t = im_tile(P, S, r0, ntc);
  if (S.active[t.b] != kActiveFar) return;
  update_tc(t.A, P.ndp, t.i0, t.j0, r0 / kImKc, align1024(im_smem_raw), &bar, &tmem_holder, &S.bad[t.b]);
}

// ---------------------------------------------------------------------------
// LU of the 64 x 64 diagonal block at (ki, ki), one CTA of 128 threads per
// instance, and the inverses of its factors.  With PRE, the block first receives
// the product L(ki:ki+64, k:k+64) U(k:k+64, ki:ki+64) of the outer panel's first
// step.  Unblocked elimination in the order of right-looking LU (every entry takes
// its products in ascending pivot order), then
//   ui[q * 64 + c] = U11^-1(q, c),  li[q * 64 + r] = L11^-1(r, q)
// (zero outside the triangles) to the instance's slot of S.inv, the operands the
// panel kernel multiplies by.
//
// Thread (ti, tj) = (tid % 16, tid / 16) holds rows 4 ti .. 4 ti + 3 of columns
// 8 tj .. 8 tj + 7 in registers.  A block of eight pivots is then one tj, half a
// warp, which factorises its 64 x 8 panel by shuffles alone; the two row groups of
// the block finish their rows of U likewise; and a rank-8 update in registers
// takes the rest: two barriers per eight pivots.  The inverses go column by column,
// a thread each (64 for L11^-1, 64 for U11^-1), eight rows at a time: the columns
// are independent and need no barrier.  Both share one 64 x 64 array, one its lower
// and one its upper triangle; 42 KB and 20 warps on an SM.
// What bounds it is issue and latency within a CTA, so small CTAs, five per SM.  With
// 512 threads, eight per row, two barriers per pivot (one for each of the sweeps)
// and two CTAs per SM 200,000 blocks took 24.7 ms; now 14.0 ms (15.1 ms before the
// two products went to packed FMAs, pairs of rows in a register pair; the factors are
// kept negated in shared memory so that those need no negation), every rounding the
// same.
// ---------------------------------------------------------------------------
constexpr int kXPitch = 65;
constexpr size_t kImDiagSmem = (64 * kPitch + 64 * kXPitch + 4 * 8 * 64 + 64) * sizeof(float);
static_assert(2 * 64 * kPitch <= 64 * kPitch + 64 * kXPitch + 4 * 8 * 64, "PRE operands fit before the rest");

template <bool PRE>
__global__ void __launch_bounds__(kImDiagThreads, 5) k_im_diag(DevPlan P, DevState S, int k, int ki,
                                                               const int32_t* __restrict__ gate) {
  extern __shared__ __align__(16) float diag_smem[];
  float(*M)[kPitch] = reinterpret_cast<float(*)[kPitch]>(diag_smem);                    // M[c][r]: minus L, minus U / pivots
  float(*X)[kXPitch] = reinterpret_cast<float(*)[kXPitch]>(diag_smem + 64 * kPitch);    // X[r][c]: the inverses
  float(*Lp)[8][64] = reinterpret_cast<float(*)[8][64]>(diag_smem + 64 * kPitch + 64 * kXPitch);  // [2]: L(r, p)
  float(*Up)[8][64] = Lp + 2;                                                           // [2]: U(p, c)
  float* invd = diag_smem + 64 * kPitch + 64 * kXPitch + 4 * 8 * 64;
  if (gate && *gate == 0) return;
  const int b = blockIdx.x;
  if (!S.active[b]) return;
  const int ld = P.ndp, tid = threadIdx.x, ti = tid & 15, tj = tid >> 4;
  float* __restrict__ A = im_block(P, S, b);
  float2 w2[2][8];  // row 4 ti + a, column 8 tj + c at w2[a / 2][c], pairs of rows packed
#define v(a, c) ((a) & 1 ? w2[(a) >> 1][c].y : w2[(a) >> 1][c].x)
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float4 q = *reinterpret_cast<const float4*>(A + (size_t)(ki + 8 * tj + c) * ld + ki + 4 * ti);
    v(0, c) = q.x;
    v(1, c) = q.y;
    v(2, c) = q.z;
    v(3, c) = q.w;
  }
  if (PRE) {
    float(*W1)[kPitch] = reinterpret_cast<float(*)[kPitch]>(diag_smem);                 // W1[q][r] = L(ki + r, k + q)
    float(*W2)[kPitch] = reinterpret_cast<float(*)[kPitch]>(diag_smem + 64 * kPitch);   // W2[c][q] = U(k + q, ki + c)
#pragma unroll
    for (int j = 0; j < 64 * 16 / kImDiagThreads; ++j) {
      const int e = tid + j * kImDiagThreads, c = e >> 4, r4 = 4 * (e & 15);
      cp16(&W1[c][r4], A + (size_t)(k + c) * ld + ki + r4);
      cp16(&W2[c][r4], A + (size_t)(ki + c) * ld + k + r4);
    }
    cp16_wait_all();
    __syncthreads();
#pragma unroll 1
    for (int q = 0; q < 64; q += 4) {
      float4 l[4];
#pragma unroll
      for (int z = 0; z < 4; ++z) l[z] = *reinterpret_cast<const float4*>(&W1[q + z][4 * ti]);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float4 u = *reinterpret_cast<const float4*>(&W2[8 * tj + c][q]);
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const float2 nu = make_float2(-comp(u, z), -comp(u, z));
          w2[0][c] = __ffma2_rn(make_float2(l[z].x, l[z].y), nu, w2[0][c]);
          w2[1][c] = __ffma2_rn(make_float2(l[z].z, l[z].w), nu, w2[1][c]);
        }
      }
    }
    __syncthreads();  // M, X and the rest overwrite the operands
  }
#pragma unroll 1
  for (int kb = 0; kb < 8; ++kb) {
    float(*L)[64] = Lp[kb & 1], (*U)[64] = Up[kb & 1];
    if (tj >> 1 == kb >> 1) {  // the warp whose half holds the panel
      // pivot p: row 8 kb + p, held by row group 2 kb + p / 4 of this half warp
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        float row[8];
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (c >= p) row[c] = __shfl_sync(0xffffffffu, v(p & 3, c), 2 * kb + (p >> 2), 16);
        if (tj == kb) {
          const float inv = 1.f / row[p];
          if (ti == 0) invd[8 * kb + p] = inv;
#pragma unroll
          for (int a = 0; a < 4; ++a)
            if (4 * ti + a > 8 * kb + p) {
              const float l = v(a, p) * inv;
              v(a, p) = l;
#pragma unroll
              for (int c = p + 1; c < 8; ++c) v(a, c) = fmaf(-l, row[c], v(a, c));
            }
        }
      }
      if (tj == kb) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
          *reinterpret_cast<float4*>(&L[c][4 * ti]) = make_float4(v(0, c), v(1, c), v(2, c), v(3, c));
      }
    }
    __syncthreads();
    if ((tj | 1) > kb) {  // a warp with columns to the right
      // rows of U: row p to the rows of its block below it
#pragma unroll
      for (int p = 0; p < 7; ++p) {
        float u[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) u[c] = __shfl_sync(0xffffffffu, v(p & 3, c), 2 * kb + (p >> 2), 16);
        if (tj > kb && ti >> 1 == kb) {
#pragma unroll
          for (int a = 0; a < 4; ++a)
            if (4 * (ti & 1) + a > p) {
              const float l = L[p][4 * ti + a];
#pragma unroll
              for (int c = 0; c < 8; ++c) v(a, c) = fmaf(-l, u[c], v(a, c));
            }
        }
      }
      if (tj > kb && ti >> 1 == kb) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          float4* o = reinterpret_cast<float4*>(&U[4 * (ti & 1) + a][8 * tj]);
          o[0] = make_float4(v(a, 0), v(a, 1), v(a, 2), v(a, 3));
          o[1] = make_float4(v(a, 4), v(a, 5), v(a, 6), v(a, 7));
        }
      }
    }
    __syncthreads();
    if (tj > kb && ti >> 1 > kb) {
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        const float4 l = *reinterpret_cast<const float4*>(&L[p][4 * ti]);
        const float4 u0 = *reinterpret_cast<const float4*>(&U[p][8 * tj]);
        const float4 u1 = *reinterpret_cast<const float4*>(&U[p][8 * tj + 4]);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float u = -(c < 4 ? comp(u0, c) : comp(u1, c - 4));
          const float2 nu = make_float2(u, u);
          w2[0][c] = __ffma2_rn(make_float2(l.x, l.y), nu, w2[0][c]);
          w2[1][c] = __ffma2_rn(make_float2(l.z, l.w), nu, w2[1][c]);
        }
      }
    }
  }
  // the factors out; in M, negated, with U's column c over pivot c
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int col = 8 * tj + c;
    *reinterpret_cast<float4*>(A + (size_t)(ki + col) * ld + ki + 4 * ti) =
        make_float4(v(0, c), v(1, c), v(2, c), v(3, c));
    const float inv = invd[col];
#pragma unroll
    for (int a = 0; a < 4; ++a) M[col][4 * ti + a] = -(4 * ti + a < col ? v(a, c) * inv : v(a, c));
  }
#undef v
  for (int e = tid; e < 64 * kXPitch; e += kImDiagThreads) X[0][e] = 0.f;
  __syncthreads();
  // Column c of L11^-1: x_i -= L(i, p) x_p, p ascending; of U11^-1, not yet scaled by
  // the pivots of its rows: x_i -= (U(i, p) / pivot p) x_p, p descending.
  {
    const bool low = tid < 64;
    const int c = tid & 63;
    auto get = [&](int r) { return r == c ? 1.f : (low ? r > c : r < c) ? X[r][c] : 0.f; };
    auto put = [&](int r, float x) {
      if (low ? r > c : r < c) X[r][c] = x;
    };
#pragma unroll 1
    for (int z = 0; z < 8; ++z) {
      const int pb = 8 * (low ? z : 7 - z);  // this block's first row
      float x[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) x[r] = get(pb + r);
      if (low) {
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
          for (int r = p + 1; r < 8; ++r) x[r] = fmaf(M[pb + p][pb + r], x[p], x[r]);
      } else {
#pragma unroll
        for (int p = 7; p >= 0; --p)
#pragma unroll
          for (int r = 0; r < p; ++r) x[r] = fmaf(M[pb + p][pb + r], x[p], x[r]);
      }
#pragma unroll
      for (int r = 0; r < 8; ++r) put(pb + r, x[r]);
#pragma unroll 1
      for (int y = z + 1; y < 8; ++y) {
        const int ib = 8 * (low ? y : 7 - y);
        float2 w[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) w[r] = make_float2(get(ib + 2 * r), get(ib + 2 * r + 1));
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          // p ascending (descending) with q; the block's column p of M, rows ib ..
          const float xp = low ? x[q] : x[7 - q];
          const float* m = &M[pb + (low ? q : 7 - q)][ib];
          const float4 m0 = *reinterpret_cast<const float4*>(m), m1 = *reinterpret_cast<const float4*>(m + 4);
          const float2 x2 = make_float2(xp, xp);
          w[0] = __ffma2_rn(make_float2(m0.x, m0.y), x2, w[0]);
          w[1] = __ffma2_rn(make_float2(m0.z, m0.w), x2, w[1]);
          w[2] = __ffma2_rn(make_float2(m1.x, m1.y), x2, w[2]);
          w[3] = __ffma2_rn(make_float2(m1.z, m1.w), x2, w[3]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          put(ib + 2 * r, w[r].x);
          put(ib + 2 * r + 1, w[r].y);
        }
      }
    }
  }
  __syncthreads();
  float* __restrict__ inv_out = reinterpret_cast<float*>(S.inv) + (size_t)b * 8192;
  for (int e = tid; e < 4096; e += kImDiagThreads) {
    const int q = e >> 6, c = e & 63;
    inv_out[e] = c > q ? X[q][c] * invd[q] : c == q ? invd[q] : 0.f;     // U11^-1(q, c)
    inv_out[4096 + e] = c > q ? X[c][q] : c == q ? 1.f : 0.f;            // L11^-1(c, q)
  }
}

// ---------------------------------------------------------------------------
// Panel of the step at ki (the diagonal block factorised, its inverses in
// S.inv): tasks 0 .. nch-1 take 128 rows each of L21 (rows ki+64 ..), tasks
// nch .. 2nch-1 128 columns each of U12 (columns ki+64 ..).  Both are products
// on a 128 x 64 tile T whose long side m runs over the task's rows (columns)
// and whose short side n over the 64 columns (rows) of the step:
//   rows   : T(m, n) = A(i, ki + n),  L21(i, .) = [T - L(i, k:k+64) U(k:k+64, ki:ki+64)] U11^-1
//   columns: T(m, n) = A(ki + n, j),  U12(., j) = L11^-1 [T - L(ki:ki+64, k:k+64) U(k:k+64, j)]
// (the bracketed product only with PRE, the second step of an outer panel).
// All operands sit in shared memory k-major: P[q][m], Q[q][n].  Warp w =
// (wm, wn), wm = w % 2, wn = w / 2, owns m in [64 wm, 64 wm + 64) and n in
// [32 wn, 32 wn + 32); lane (lx, ly), lx = lane % 4, ly = lane / 4, owns m =
// 64 wm + ly*4 + 32h + q and n = 32 wn + lx*4 + 16g + r (h, g < 2; q, r < 4):
// per q two 16-byte loads of P and two of Q feed 64 FMAs (packed in pairs of
// m).  The inverse is triangular, so the second product stops at q < 32 (wn +
// 1).
// ---------------------------------------------------------------------------
constexpr int kImPanelThreads2 = 128;
// row pitches (floats) of Pk / T2 and of Qk: with 132 and 68 the stores that
// transpose (a quarter warp's 16-byte stores of four rows n = no + 16g + r of
// T2; scalar stores of four rows 4 q4 + c of Pk or Qk) meet 2-way bank
// conflicts instead of 4-way
constexpr int kT2Pitch = 132;
constexpr int kQkPitch = 68;
// Pk (reused for T2 once the left-looking product is done), Q2, Qk
constexpr size_t kImPanelSmemPre = (size_t)(64 * kT2Pitch + 64 * 64 + 64 * kQkPitch) * sizeof(float);
constexpr size_t kImPanelSmem = (size_t)(64 * kT2Pitch + 64 * 64) * sizeof(float);


// acc[h][g][r][p] holds rows (2p, 2p+1) of the thread's 4-row group h,
// column (g, r); one packed two-wide FMA per pair (same rounding as fmaf)
__device__ __forceinline__ void fma_q(float2 (&acc)[2][2][4][2], const float4 (&a)[2], const float4 (&b)[2],
                                      float sign) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 a01 = make_float2(a[h].x, a[h].y), a23 = make_float2(a[h].z, a[h].w);
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float bv = sign * comp(b[g], r);
        const float2 b2 = make_float2(bv, bv);
        acc[h][g][r][0] = __ffma2_rn(a01, b2, acc[h][g][r][0]);
        acc[h][g][r][1] = __ffma2_rn(a23, b2, acc[h][g][r][1]);
      }
  }
}

__device__ __forceinline__ float& el(float2 (&acc)[2][2][4][2], int h, int g, int r, int q) {
  return (q & 1) ? acc[h][g][r][q >> 1].y : acc[h][g][r][q >> 1].x;
}

template <bool PRE>
__global__ void __launch_bounds__(kImPanelThreads2, 3) k_im_panel(DevPlan P, DevState S, int k, int ki, int nch,
                                                               const int32_t* __restrict__ gate) {
  extern __shared__ __align__(16) float pan_smem[];
  float* Pk = pan_smem;                           // PRE: [64 q][kT2Pitch]
  float* T2 = pan_smem;                           // [64 n][kT2Pitch]: the first result, k-major (over Pk)
  float* Q2 = pan_smem + 64 * kT2Pitch;           // [64 q][64 n]: the inverse factor
  float* Qk = Q2 + 64 * 64;                       // PRE: [64 q][kQkPitch]
  if (gate && *gate == 0) return;
  const int per = 2 * nch;
  const int b = (int)(blockIdx.x / (unsigned)per);
  const int task = (int)(blockIdx.x - (unsigned)b * (unsigned)per);
  if (!S.active[b]) return;
  const int ld = P.ndp, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wm = warp & 1, wn = warp >> 1, lx = lane & 3, ly = lane >> 2;
  const int mo = wm * 64 + ly * 4, no = wn * 32 + lx * 4;
  float* __restrict__ A = im_block(P, S, b);
  const bool rows = task < nch;
  const int base = ki + 64 + (rows ? task : task - nch) * 128;  // first row (rows) or column (columns)
  const int mvalid = min(128, ld - base);
  const bool active = wm * 64 < mvalid;
  // operands: contiguous 16-byte words by asynchronous copies, all in flight
  // together; the transposed ones through registers, fully unrolled
  {
    const float* src = reinterpret_cast<const float*>(S.inv) + (size_t)b * 8192 + (rows ? 0 : 4096);
#pragma unroll
    for (int j = 0; j < 64 * 16 / kImPanelThreads2; ++j) {
      const int e = tid + j * kImPanelThreads2;
      cp16(Q2 + 4 * e, src + 4 * e);
    }
  }
  // The transposed operands are read four 16-byte words of one column per
  // four lanes (64-byte segments): lanes (c4 = lane % 4, the column from the
  // rest), word q4 = c4 + 4 (j % 4).
  if (PRE) {
    if (rows) {
      // Pk[q][m] = L(base + m, k + q); Qk[q][n] = U(k + q, ki + n)
#pragma unroll
      for (int j = 0; j < 64 * 32 / kImPanelThreads2; ++j) {
        const int e = tid + j * kImPanelThreads2, q = e >> 5, m4 = e & 31;
        if (4 * m4 < mvalid) cp16(Pk + q * kT2Pitch + 4 * m4, A + (size_t)(k + q) * ld + base + 4 * m4);
      }
#pragma unroll
      for (int j = 0; j < 64 * 16 / kImPanelThreads2; ++j) {
        const int n = (tid >> 2) + 32 * (j >> 2), q4 = (tid & 3) + 4 * (j & 3);
        const float4 v = *reinterpret_cast<const float4*>(A + (size_t)(ki + n) * ld + k + 4 * q4);
        Qk[(4 * q4) * kQkPitch + n] = v.x;
        Qk[(4 * q4 + 1) * kQkPitch + n] = v.y;
        Qk[(4 * q4 + 2) * kQkPitch + n] = v.z;
        Qk[(4 * q4 + 3) * kQkPitch + n] = v.w;
      }
    } else {
      // Pk[q][m] = U(k + q, base + m); Qk[q][n] = L(ki + n, k + q)
#pragma unroll
      for (int j = 0; j < 64 * 16 / kImPanelThreads2; ++j) {
        const int e = tid + j * kImPanelThreads2, q = e >> 4, n4 = e & 15;
        cp16(Qk + q * kQkPitch + 4 * n4, A + (size_t)(k + q) * ld + ki + 4 * n4);
      }
#pragma unroll
      for (int j = 0; j < 128 * 16 / kImPanelThreads2; ++j) {
        const int m = (tid >> 2) + 32 * (j >> 2), q4 = (tid & 3) + 4 * (j & 3);
        if (m < mvalid) {
          const float4 v = *reinterpret_cast<const float4*>(A + (size_t)(base + m) * ld + k + 4 * q4);
          Pk[(4 * q4) * kT2Pitch + m] = v.x;
          Pk[(4 * q4 + 1) * kT2Pitch + m] = v.y;
          Pk[(4 * q4 + 2) * kT2Pitch + m] = v.z;
          Pk[(4 * q4 + 3) * kT2Pitch + m] = v.w;
        }
      }
    }
  }
  // el(acc, h, g, r, q) = T(m = mo + 32h + q, n = no + 16g + r); pairs of q packed
  float2 acc[2][2][4][2];
  if (active) {
    if (rows) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int g = 0; g < 2; ++g)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float4 v =
                *reinterpret_cast<const float4*>(A + (size_t)(ki + no + 16 * g + r) * ld + base + mo + 32 * h);
            acc[h][g][r][0] = make_float2(v.x, v.y);
            acc[h][g][r][1] = make_float2(v.z, v.w);
          }
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const float4 v =
                *reinterpret_cast<const float4*>(A + (size_t)(base + mo + 32 * h + q) * ld + ki + no + 16 * g);
            el(acc, h, g, 0, q) = v.x;
            el(acc, h, g, 1, q) = v.y;
            el(acc, h, g, 2, q) = v.z;
            el(acc, h, g, 3, q) = v.w;
          }
    }
  }
  cp16_wait_all();
  __syncthreads();
  if (PRE && active) {
#pragma unroll 4
    for (int q = 0; q < 64; ++q) {
      const float4 a[2] = {*reinterpret_cast<const float4*>(Pk + q * kT2Pitch + mo),
                           *reinterpret_cast<const float4*>(Pk + q * kT2Pitch + mo + 32)};
      const float4 bq[2] = {*reinterpret_cast<const float4*>(Qk + q * kQkPitch + no),
                            *reinterpret_cast<const float4*>(Qk + q * kQkPitch + no + 16)};
      fma_q(acc, a, bq, -1.f);
    }
  }
  if (PRE) __syncthreads();  // T2 overwrites Pk
  if (active) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int g = 0; g < 2; ++g)
#pragma unroll
        for (int r = 0; r < 4; ++r)
          *reinterpret_cast<float4*>(T2 + (no + 16 * g + r) * kT2Pitch + mo + 32 * h) =
              make_float4(acc[h][g][r][0].x, acc[h][g][r][0].y, acc[h][g][r][1].x, acc[h][g][r][1].y);
  }
  __syncthreads();
  if (!active) return;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        acc[h][g][r][0] = make_float2(0.f, 0.f);
        acc[h][g][r][1] = make_float2(0.f, 0.f);
      }
  const int qend = 32 * (wn + 1);
#pragma unroll 4
  for (int q = 0; q < qend; ++q) {
    const float4 a[2] = {*reinterpret_cast<const float4*>(T2 + q * kT2Pitch + mo),
                         *reinterpret_cast<const float4*>(T2 + q * kT2Pitch + mo + 32)};
    const float4 bq[2] = {*reinterpret_cast<const float4*>(Q2 + q * 64 + no),
                          *reinterpret_cast<const float4*>(Q2 + q * 64 + no + 16)};
    fma_q(acc, a, bq, 1.f);
  }
  if (rows) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int g = 0; g < 2; ++g)
#pragma unroll
        for (int r = 0; r < 4; ++r)
          *reinterpret_cast<float4*>(A + (size_t)(ki + no + 16 * g + r) * ld + base + mo + 32 * h) =
              make_float4(acc[h][g][r][0].x, acc[h][g][r][0].y, acc[h][g][r][1].x, acc[h][g][r][1].y);
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int g = 0; g < 2; ++g)
          *reinterpret_cast<float4*>(A + (size_t)(base + mo + 32 * h + q) * ld + ki + no + 16 * g) =
              make_float4(el(acc, h, g, 0, q), el(acc, h, g, 1, q), el(acc, h, g, 2, q), el(acc, h, g, 3, q));
  }
}

// ---------------------------------------------------------------------------
// Dense forward (unit lower L) and backward (upper U) substitution, one CTA
// per instance, the right-hand side in shared memory.  Per block of 64
// columns: the 64 x 64 triangle is copied to shared memory and solved by one
// warp (two rows per lane, the solved entry broadcast by a shuffle); then every
// thread updates its rows below (above) the block with the block's 64
// entries, reading the matrix columns contiguously across the CTA.  The solve
// reads each instance's block once and is bound by how many loads are in
// flight, and by the last wave: at most 32 registers per thread let eight CTAs (eight
// instances) run on an SM.  On 1,000 blocks of 2,176 (18.9 GB per solve) six CTAs of 40
// registers took 4.7 ms, two waves, the second nearly empty; eight take 3.2 ms
// (5.9 TB/s).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kImSolveThreads, 8) k_im_dsolve(DevPlan P, DevState S,
                                                              const int32_t* __restrict__ gate) {
  extern __shared__ float xs[];                  // [ndp]
  __shared__ float T[64][65];                    // T[c][r]
  if (gate && *gate == 0) return;
  const int b = blockIdx.x;
  if (!S.active[b]) return;
  const int ld = P.ndp, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* __restrict__ A = im_block(P, S, b);
  float* __restrict__ X = reinterpret_cast<float*>(S.x) + ((size_t)(b >> 5) * P.mp + P.s) * kTile + (b & 31);
  for (int r = tid; r < ld; r += kImSolveThreads) xs[r] = X[(size_t)r * kTile];
  __syncthreads();
  for (int kb = 0; kb < ld; kb += 64) {
    for (int e = tid; e < 64 * 64; e += kImSolveThreads) {
      const int c = e >> 6, r = e & 63;
      T[c][r] = A[(size_t)(kb + c) * ld + kb + r];
    }
    __syncthreads();
    if (warp == 0) {
      float v0 = xs[kb + lane], v1 = xs[kb + 32 + lane];
#pragma unroll 8
      for (int c = 0; c < 64; ++c) {
        const float xc = __shfl_sync(0xffffffffu, c < 32 ? v0 : v1, c & 31);
        if (lane > c) v0 = fmaf(-T[c][lane], xc, v0);
        if (32 + lane > c) v1 = fmaf(-T[c][32 + lane], xc, v1);
      }
      xs[kb + lane] = v0;
      xs[kb + 32 + lane] = v1;
    }
    __syncthreads();
    for (int r = kb + 64 + tid; r < ld; r += kImSolveThreads) {
      float acc = xs[r];
#pragma unroll 8
      for (int c = 0; c < 64; ++c) acc = fmaf(-A[(size_t)(kb + c) * ld + r], xs[kb + c], acc);
      xs[r] = acc;
    }
    __syncthreads();
  }
  for (int kb = ld - 64; kb >= 0; kb -= 64) {
    for (int e = tid; e < 64 * 64; e += kImSolveThreads) {
      const int c = e >> 6, r = e & 63;
      T[c][r] = A[(size_t)(kb + c) * ld + kb + r];
    }
    __syncthreads();
    if (warp == 0) {
      float v0 = xs[kb + lane], v1 = xs[kb + 32 + lane];
#pragma unroll 8
      for (int c = 63; c >= 0; --c) {
        if (c >= 32) {
          if (lane == c - 32) v1 = v1 * (1.f / T[c][c]);
        } else if (lane == c) {
          v0 = v0 * (1.f / T[c][c]);
        }
        const float xc = __shfl_sync(0xffffffffu, c < 32 ? v0 : v1, c & 31);
        if (lane < c) v0 = fmaf(-T[c][lane], xc, v0);
        if (32 + lane < c) v1 = fmaf(-T[c][32 + lane], xc, v1);
      }
      xs[kb + lane] = v0;
      xs[kb + 32 + lane] = v1;
    }
    __syncthreads();
    for (int r = tid; r < kb; r += kImSolveThreads) {
      float acc = xs[r];
#pragma unroll 8
      for (int c = 0; c < 64; ++c) acc = fmaf(-A[(size_t)(kb + c) * ld + r], xs[kb + c], acc);
      xs[r] = acc;
    }
    __syncthreads();
  }
  for (int r = tid; r < ld; r += kImSolveThreads) X[(size_t)r * kTile] = xs[r];
}

// Padding of the dense block, one CTA per instance: columns nd .. ndp-1 are
// identity columns (contiguous in the instance-major layout), and the
// right-hand side's padding rows m .. m+n_one-1 are zero, so that no stale
// value leaks into real rows during the substitutions.
__global__ void __launch_bounds__(256) k_im_set_ones(DevPlan P, DevState S, const int32_t* __restrict__ gate) {
  if (gate && *gate == 0) return;
  const int b = blockIdx.x;
  const int ld = P.ndp;
  float* __restrict__ A = im_block(P, S, b) + (size_t)P.nd * ld;
  const int n = P.n_one * ld;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const int c = e / ld, r = e - c * ld;
    A[e] = r == P.nd + c ? 1.f : 0.f;
  }
  float* __restrict__ X = reinterpret_cast<float*>(S.x) + (size_t)(b >> 5) * P.mp * kTile + (b & 31);
  for (int t = threadIdx.x; t < P.n_one; t += blockDim.x) X[(size_t)(P.m + t) * kTile] = 0.f;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn im_encode_fn() {
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

}  // namespace

bool make_dense_im_maps(const DevPlan& P, void* lu, int Bp, DenseImMaps* out) {
  EncodeTiledFn fn = im_encode_fn();
  if (!fn || !lu || Bp <= 0 || Bp % kTile || P.ndp <= 0 || P.ndp % 64) return false;
  const cuuint64_t ld = (cuuint64_t)P.ndp;
  void* base = reinterpret_cast<float*>(lu) + (size_t)P.NS * kTile;
  const cuuint64_t dims[4] = {ld, ld, (cuuint64_t)kTile, (cuuint64_t)(Bp / kTile)};
  const cuuint64_t strides[3] = {ld * 4, ld * ld * 4, (cuuint64_t)P.NLU * kTile * 4};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  const cuuint32_t box_a[4] = {(cuuint32_t)kImTile, (cuuint32_t)kImKc, 1, 1};
  const cuuint32_t box_b[4] = {(cuuint32_t)kImKc, (cuuint32_t)kImTile, 1, 1};
  if (fn(&out->a, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box_a, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
         CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  return fn(&out->b, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box_b, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

void launch_dense_im_factor(const DevPlan& P, const DevState& S, const DenseImMaps& maps, const int32_t* gate,
                            cudaStream_t st, Recorder* rec) {
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_im_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kImGemmSmem);
    cudaFuncSetAttribute(k_im_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kImGemmTcSmem);
    cudaFuncSetAttribute(k_im_diag<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kImDiagSmem);
    cudaFuncSetAttribute(k_im_diag<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kImDiagSmem);
    cudaFuncSetAttribute(k_im_panel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kImPanelSmem);
    cudaFuncSetAttribute(k_im_panel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kImPanelSmemPre);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const unsigned Bp = (unsigned)S.Bp;
  const int ld = P.ndp;
  // the two 64-wide steps of the outer panel at k
  auto outer = [&](int k) {
    NRPF_LAUNCH(rec, K_DENSE_DIAG, st,
                k_im_diag<false><<<Bp, kImDiagThreads, kImDiagSmem, st>>>(P, S, k, k, gate));
    int nr = ld - k - 64;
    if (nr > 0) {
      const int nch = (nr + 127) / 128;
      NRPF_LAUNCH(rec, K_DENSE_PANEL, st,
                  k_im_panel<false><<<Bp * 2 * nch, kImPanelThreads2, kImPanelSmem, st>>>(P, S, k, k, nch, gate));
    }
    if (ld - k < kImOuter) return;  // a last outer panel of 64
    NRPF_LAUNCH(rec, K_DENSE_DIAG, st,
                k_im_diag<true><<<Bp, kImDiagThreads, kImDiagSmem, st>>>(P, S, k, k + 64, gate));
    nr = ld - k - kImOuter;
    if (nr > 0) {
      const int nch = (nr + 127) / 128;
      NRPF_LAUNCH(rec, K_DENSE_PANEL, st,
                  k_im_panel<true><<<Bp * 2 * nch, kImPanelThreads2, kImPanelSmemPre, st>>>(P, S, k, k + 64, nch,
                                                                                          gate));
    }
  };
  // block column and row of the outer panel at r0 minus the products of the
  // panels before it
  auto gemm = [&](int r0) {
    const int ntc = (ld - r0 + kImTile - 1) / kImTile;
    const unsigned grid = Bp * (unsigned)(2 * ntc - 1);
    NRPF_LAUNCH(rec, K_DENSE_UPDATE, st,
                k_im_gemm_tc<<<grid, kImGemmThreads, kImGemmTcSmem, st>>>(P, S, r0, ntc, gate));
    NRPF_LAUNCH(rec, K_DENSE_UPDATE, st,
                k_im_gemm<<<grid, kImGemmThreads, kImGemmSmem, st>>>(maps.a, maps.b, P, S, r0, ntc, gate));
  };
  // Left-looking by outer panels: panel j's block column and row first take
  // the products of panels 0 .. j-1 (depth kj, each entry's subtractions in
  // ascending pivot order, as in the right-looking form), then it is factorised.
  for (int kj = 0; kj < ld; kj += kImOuter) {
    if (kj > 0) gemm(kj);
    outer(kj);
  }
}

void launch_dense_im_set_ones(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                              Recorder* rec) {
  NRPF_LAUNCH(rec, K_ONES, st, k_im_set_ones<<<(unsigned)S.Bp, 256, 0, st>>>(P, S, gate));
}

void launch_dense_im_solve(const DevPlan& P, const DevState& S, const int32_t* gate, cudaStream_t st,
                           Recorder* rec) {
  const size_t smem = (size_t)P.ndp * sizeof(float);
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    cudaFuncSetAttribute(k_im_dsolve, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  NRPF_LAUNCH(rec, K_DENSE_SOLVE, st,
              k_im_dsolve<<<(unsigned)S.Bp, kImSolveThreads, smem, st>>>(P, S, gate));
}

}  // namespace nrpf
