// FP32 CUDA-core GEMM C = A B^T with both operands K-major (rows of length p).
// The correlations D^T Y (Algorithm 1 step 1) and, in the same launch, the Gram
// matrix G = D^T D (Batch-OMP, [RZE08] as cited in Section 4) of the shapes that the
// tensor-core kernel does not take (p > 64, p % 4 != 0), and the FP32 reference path.
//
// Bound by the FP32 pipes: 2 m n p FLOP, 3.1 GFLOP at p = 100, n = 512, m = 30,000,
// 42 us at the measured 75 TFLOP/s.  128 x 128 tiles, 8 x 8 results per thread as
// packed FP32x2 multiply-adds (half the issue slots of scalar ones), two CTAs per
// SM.  Tiles of 32 columns of A and B come in by 4-byte cp.async (no alignment
// or length rule for the rows), two in flight, stored transposed: element (k, r) at
// k 128 + (r ^ 4 (k mod 8)), so that the eight k x four r of a warp's copies and the
// 16-byte reads of four consecutive r each fall on distinct banks.  Each result is
// one FP32 multiply-add chain over k = 0, 1, ..., as it always was: the same bits.
// Measured with the Gram matrix: 78 us, 144 for the earlier kernel (scalar
// loads through registers, padded tiles, scalar multiply-adds: 101 with those here) and
// its separate 16-CTA Gram launch.
#include "dl_internal.cuh"

namespace dlk {
namespace {

constexpr int TM = 128, TN = 128, TK = 32, NTHR = 256;
constexpr int kTileFloats = TK * TM;  // one operand of one stage
constexpr size_t kSimtSmem = (size_t)2 * 2 * kTileFloats * sizeof(float);

// Position of element (k, r) of a tile.
__device__ __forceinline__ int tile_at(int k, int r) { return k * TM + (r ^ ((k & 7) << 2)); }

__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  const int bytes = valid ? 4 : 0;  // 0: the destination is filled with zero, src is not read
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

// Columns k0 .. k0+31 of 128 rows of A (row i0 first): the eight warps take 16 rows
// each, 4 rows x 8 columns per instruction.
__device__ __forceinline__ void load_tile(float* dst, const float* __restrict__ A, int64_t rows, int64_t i0,
                                          int p, int k0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rl = lane >> 3, kl = lane & 7;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int r = 16 * warp + 4 * h + rl;
    const bool row = i0 + r < rows;
    const float* src = A + (row ? i0 + r : 0) * p;
#pragma unroll
    for (int q = 0; q < TK / 8; ++q) {
      const int k = 8 * q + kl;
      const bool ok = row && k0 + k < p;
      cp_async4(dst + tile_at(k, r), src + (ok ? k0 + k : 0), ok);
    }
  }
}

struct SimtProblem {
  const float* A;
  int64_t rows;
  float* C;
  int64_t ldc;
};

// C = A B^T of two problems with the same B: row tiles [0, tiles0) are P0's.
__global__ void __launch_bounds__(NTHR, 2) gemm_nt_kernel(const SimtProblem P0, const SimtProblem P1,
                                                          int64_t tiles0, const float* __restrict__ B,
                                                          int rows_b, int p, int* __restrict__ zero) {
  if (zero && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *zero = 0;
  extern __shared__ __align__(16) float sm[];
  const bool second = (int64_t)blockIdx.x >= tiles0;
  const SimtProblem P = second ? P1 : P0;
  const int64_t i0 = ((int64_t)blockIdx.x - (second ? tiles0 : 0)) * TM;
  const int j0 = blockIdx.y * TN;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // columns 4tx.. and 64+4tx.., rows 8ty..
  float2 acc[8][4];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = make_float2(0.f, 0.f);
  const int nk = (p + TK - 1) / TK;
  auto fetch = [&](int c) {
    float* st = sm + (c & 1) * 2 * kTileFloats;
    load_tile(st, P.A, P.rows, i0, p, c * TK);
    load_tile(st + kTileFloats, B, rows_b, j0, p, c * TK);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0);
  for (int c = 0; c < nk; ++c) {
    if (c + 1 < nk) {
      fetch(c + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float* As = sm + (c & 1) * 2 * kTileFloats;
    const float* Bs = As + kTileFloats;
    const int kn = p - c * TK < TK ? p - c * TK : TK;
#pragma unroll 8
    for (int k = 0; k < kn; ++k) {
      const int sw = (k & 7) << 2;
      const float4 a0 = *(const float4*)(As + k * TM + ((8 * ty) ^ sw));
      const float4 a1 = *(const float4*)(As + k * TM + ((8 * ty + 4) ^ sw));
      const float4 b0 = *(const float4*)(Bs + k * TN + ((4 * tx) ^ sw));
      const float4 b1 = *(const float4*)(Bs + k * TN + ((64 + 4 * tx) ^ sw));
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                           make_float2(b1.z, b1.w)};
#pragma unroll
      for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = __ffma2_rn(make_float2(a[x], a[x]), b[y], acc[x][y]);
    }
    __syncthreads();
  }
  const bool vec = (P.ldc & 3) == 0 && ((uintptr_t)P.C & 15) == 0;
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int64_t gi = i0 + 8 * ty + x;
    if (gi >= P.rows) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gj = j0 + 64 * h + 4 * tx;
      float* out = P.C + gi * P.ldc + gj;
      const float v[4] = {acc[x][2 * h].x, acc[x][2 * h].y, acc[x][2 * h + 1].x, acc[x][2 * h + 1].y};
      if (vec && gj + 4 <= rows_b) {
        *(float4*)out = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (gj + q < rows_b) out[q] = v[q];
      }
    }
  }
}

}  // namespace

cudaError_t gemm_nt_simt_pair(const float* A0, int64_t rows0, float* C0, int64_t ldc0, const float* A1,
                              int64_t rows1, float* C1, int64_t ldc1, const float* B, int rows_b, int p,
                              cudaStream_t st, int* zero) {
  if (rows0 < 0) rows0 = 0;
  if (rows1 < 0 || !A1) rows1 = 0;
  const int64_t t0 = (rows0 + TM - 1) / TM, t1 = (rows1 + TM - 1) / TM;
  if (t0 + t1 == 0 || rows_b <= 0) return cudaSuccess;
  cudaError_t e =
      cudaFuncSetAttribute(gemm_nt_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSimtSmem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)(t0 + t1), (unsigned)((rows_b + TN - 1) / TN));
  gemm_nt_kernel<<<grid, NTHR, kSimtSmem, st>>>(SimtProblem{A0, rows0, C0, ldc0},
                                                SimtProblem{A1, rows1, C1, ldc1}, t0, B, rows_b, p,
                                                zero);
  return cudaGetLastError();
}

cudaError_t gemm_nt_simt(const float* A, int64_t rows_a, const float* B, int rows_b, int p, float* C,
                         int64_t ldc, cudaStream_t st) {
  return gemm_nt_simt_pair(A, rows_a, C, ldc, nullptr, 0, nullptr, 0, B, rows_b, p, st);
}

}  // namespace dlk

// ---- Gram matrix G = D D^T (n x n, row-major; D n x p row-major) ----------------
// The Gram matrix of Batch-OMP and of the residual-form OMP's Cholesky rows, as
// one short launch: a CTA per 32 x 32 block of the upper triangle (136 CTAs at
// n = 512, one SM each), 256 threads of 2 x 2 entries, the two 32-atom row
// blocks in shared memory (odd pitch: no bank conflicts), FP32 sums in row
// order; each block is written with its mirror, so G is exactly symmetric.
namespace dlk {
namespace {

constexpr int GT = 32, GK = 64;

__global__ void __launch_bounds__(256) gram_kernel(const float* __restrict__ D, int n, int p,
                                                   float* __restrict__ G, int tiles,
                                                   int* __restrict__ zero) {
  if (zero && blockIdx.x == 0 && threadIdx.x == 0) *zero = 0;
  __shared__ float Dj[GT][GK + 1];
  __shared__ float Dk[GT][GK + 1];
  // block b -> (jt, kt) with jt <= kt, row by row of the upper triangle
  int b = blockIdx.x, jt = 0;
  while (b >= tiles - jt) {
    b -= tiles - jt;
    ++jt;
  }
  const int kt = jt + b;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  for (int k0 = 0; k0 < p; k0 += GK) {
    __syncthreads();
    for (int e = tid; e < GT * GK; e += 256) {
      const int r = e / GK, c = e % GK;
      const int j = jt * GT + r, k = kt * GT + r;
      Dj[r][c] = (j < n && k0 + c < p) ? __ldg(D + (size_t)j * p + k0 + c) : 0.f;
      Dk[r][c] = (k < n && k0 + c < p) ? __ldg(D + (size_t)k * p + k0 + c) : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < GK; ++c) {
      const float a0 = Dj[2 * ty][c], a1 = Dj[2 * ty + 1][c];
      const float b0 = Dk[2 * tx][c], b1 = Dk[2 * tx + 1][c];
      acc[0][0] = fmaf(a0, b0, acc[0][0]);
      acc[0][1] = fmaf(a0, b1, acc[0][1]);
      acc[1][0] = fmaf(a1, b0, acc[1][0]);
      acc[1][1] = fmaf(a1, b1, acc[1][1]);
    }
  }
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int j = jt * GT + 2 * ty + a, k = kt * GT + 2 * tx + c;
      if (j < n && k < n) {
        G[(size_t)j * n + k] = acc[a][c];
        G[(size_t)k * n + j] = acc[a][c];
      }
    }
}

}  // namespace

cudaError_t gram_simt(const float* D, int n, int p, float* G, cudaStream_t st, int* zero) {
  if (n <= 0) return cudaSuccess;
  const int tiles = (n + GT - 1) / GT;
  gram_kernel<<<tiles * (tiles + 1) / 2, 256, 0, st>>>(D, n, p, G, tiles, zero);
  return cudaGetLastError();
}

}  // namespace dlk
