// Batch-OMP sparse coding of several signals per warp, for small dictionaries and
// short supports (Algorithm 1 step 1; n <= 128 and s <= 8, n <= 256 and s <= 6; the
// arithmetic of omp_warp_kernel, see k_omp.cu, operation by operation, so the results are the
// same bits).
//
// With n = 128 a warp per signal leaves each lane four correlations, and most of
// its instructions are the per-signal part of a step -- reductions, broadcasts, the
// Cholesky row, the pivot -- that all 32 lanes repeat: about 600 per signal and step
// issued, at 0.56 per cycle and scheduler.  Here SW lanes (8 for n <= 128, 16
// for n <= 256) take a signal, so that a warp runs 4 or 2 signals in step and each
// lane works on up to 16 correlations as four 16-byte vectors: lane l holds atoms
// 4 (l + SW v) + e.  A signal's correlations, its vectors u_q and its Cholesky rows
// lie in shared memory, where the entry of the selected atom is one load instead of an
// indexed register; for n <= 128 with many signals the Gram matrix lies there too,
// else its rows come from L2.  Signals that stop early idle until their
// warp's others end.
//
// The argmax compares |alpha| truncated as omp_warp_kernel truncates it for this n
// (the low tbits() mantissa bits, which there carry the 32-atom block), with the
// vector number in those bits: the largest key is the largest truncated value and
// among equal ones the lowest vector, then the lowest lane wins, then the lowest
// e -- the lowest atom, as there.
//
// Measured (us, omp_warp_kernel's in brackets): n = 128, s = 4, m = 60,000 36.5 (59.1);
// n = 256, s = 6, m = 20,000 35.2 (47.2); n = 200, s = 5, m = 15,001 25.5 (34.2); what is left
// is the latency of a step's chain with 17 to 20 warps per SM, which shared memory sets.
#include "dl_internal.cuh"
#include "omp_common.cuh"
#include "omp_sub.cuh"

#include <math.h>

#include <algorithm>

namespace dlk {
namespace {

using namespace omp;

constexpr int SUB_WARPS = 24;                // most warps per CTA (one CTA per SM)
constexpr size_t kSubSmem = 220 * 1024;      // dynamic shared memory of a CTA

__device__ __forceinline__ float4 ld_stream4(const float* p) {
  float4 v;
  asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p));
  return v;
}
// Rows of G in shared memory (pitch NP, zero past n), or in global memory (VEC: n % 4
// == 0, as float4).
template <int NP, bool GSH, bool VEC>
struct SubGram {
  const float* G;
  int n;
  __device__ __forceinline__ float diag(int j) const {
    return GSH ? G[j * NP + j] : __ldg(G + (size_t)j * n + j);
  }
  __device__ __forceinline__ float4 vec(int row, int j) const {
    if (GSH) return *(const float4*)(G + row * NP + j);
    const float* Gr = G + (size_t)row * n;
    if (VEC) return j < n ? __ldg((const float4*)(Gr + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
    return make_float4(j < n ? __ldg(Gr + j) : 0.f, j + 1 < n ? __ldg(Gr + j + 1) : 0.f,
                       j + 2 < n ? __ldg(Gr + j + 2) : 0.f, j + 3 < n ? __ldg(Gr + j + 3) : 0.f);
  }
};

// TB: truncated mantissa bits; GSH: G in shared memory (pitch NP); VEC: rows of G
// in global memory as float4 (n % 4 == 0).
template <int SW, int V, int TB, bool GSH, bool VEC>
__global__ void __launch_bounds__(SUB_WARPS * 32, 1) omp_sub_kernel(
    const float* __restrict__ A0, int64_t lda, const float* __restrict__ G, int n,
    const float* __restrict__ Y, int p, int64_t m, int s, int32_t* __restrict__ oidx,
    float* __restrict__ oval, int32_t* __restrict__ ocnt, float* __restrict__ ores,
    int* __restrict__ err, int* __restrict__ rs_list, int* __restrict__ rs_count, int rs_cap) {
  constexpr int SPW = 32 / SW, NP = 4 * SW * V;
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int sub = lane / SW, l = lane % SW;
  const SubGram<NP, GSH, VEC> gram{GSH ? sm : G, n};
  float* base = sm + (GSH ? n * NP : 0) + (warp * SPW + sub) * sub_signal_floats<SW, V>(s);
  const float qnan = __int_as_float(0x7fc00000);
  if (GSH) {
#pragma unroll 4
    for (int q = threadIdx.x; q < n * (NP / 4); q += blockDim.x) {
      const int j = q / (NP / 4), k = 4 * (q % (NP / 4));
      const float* Gr = G + (size_t)j * n;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (VEC) {
        if (k < n) v = __ldg((const float4*)(Gr + k));
      } else {
        v.x = k < n ? __ldg(Gr + k) : 0.f;
        v.y = k + 1 < n ? __ldg(Gr + k + 1) : 0.f;
        v.z = k + 2 < n ? __ldg(Gr + k + 2) : 0.f;
        v.w = k + 3 < n ? __ldg(Gr + k + 3) : 0.f;
      }
      ((float4*)sm)[q] = v;
    }
    __syncthreads();
  }
  const int64_t stride = (int64_t)gridDim.x * W * SPW;
  for (int64_t i0 = ((int64_t)blockIdx.x * W + warp) * SPW; i0 < m; i0 += stride) {
    const int64_t i = i0 + sub;
    const bool live = i < m;
    {  // warm L2 with the warp's next signals
      const int64_t in = i + stride;
      if (in < m) {
        if (32 * l < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(A0 + in * lda + 32 * l));
        if (32 * l < p) asm volatile("prefetch.global.L2 [%0];" ::"l"(Y + in * p + 32 * l));
      }
    }
    const float* y = Y + (live ? i : 0) * p;
    const float* a0 = A0 + (live ? i : 0) * lda;
    // correlations; atoms past n never win
    float4 a[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int j = 4 * (l + SW * v);
      a[v] = j < n ? ld_stream4(a0 + j) : make_float4(qnan, qnan, qnan, qnan);
      if (j + 1 >= n) a[v].y = qnan;
      if (j + 2 >= n) a[v].z = qnan;
      if (j + 3 >= n) a[v].w = qnan;
    }
    float yy;  // ||y||^2
    {
      float t[32 / SW];
#pragma unroll
      for (int h = 0; h < 32 / SW; ++h) {
        t[h] = 0.f;
        for (int r = l + SW * h; r < p; r += 32) {
          const float v = ld_stream(y + r);
          t[h] = fmaf(v, v, t[h]);
        }
      }
      yy = sub_norm2<SW>(t);
    }
    omp_sub_core<SW, V, TB>(i, live, a, yy, gram, base, s, oidx, oval, ocnt, ores, err, rs_list, rs_count,
                            rs_cap);
  }
}

template <int SW, int V, int TB>
cudaError_t launch_sub(const float* A0, int64_t lda, const float* G, int n, const float* Y, int p,
                       int64_t m, int s, int32_t* idx, float* val, int32_t* cnt, float* ores, int* err,
                       int* rl, int* rc, int rcap, cudaStream_t st) {
  constexpr int SPW = 32 / SW, NP = 4 * SW * V;
  const size_t per = (size_t)SPW * sub_signal_floats<SW, V>(s) * sizeof(float);
  const size_t gbytes = (size_t)n * NP * sizeof(float);
  // warps per CTA: enough for the signals of one round, as many as fit
  const int64_t need = (m + (int64_t)num_sms() * SPW - 1) / ((int64_t)num_sms() * SPW);
  auto fit = [&](size_t g) { return (int64_t)((kSubSmem - g) / per); };
  const bool gsh = NP <= 128 && need >= 8 && fit(gbytes) >= 8;
  int64_t W = std::min<int64_t>(SUB_WARPS, fit(gsh ? gbytes : 0));
  if (need < W) W = need;
  const size_t smem = (gsh ? gbytes : 0) + (size_t)W * per;
  const bool vec = n % 4 == 0 && ((uintptr_t)G & 15) == 0;
  constexpr bool kCanShare = NP <= 128;
  auto kern = gsh ? (vec ? omp_sub_kernel<SW, V, TB, kCanShare, true> : omp_sub_kernel<SW, V, TB, kCanShare, false>)
                  : (vec ? omp_sub_kernel<SW, V, TB, false, true> : omp_sub_kernel<SW, V, TB, false, false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t blocks = (m + W * SPW - 1) / (W * SPW);
  kern<<<(unsigned)(blocks < num_sms() ? blocks : num_sms()), (unsigned)(W * 32), smem, st>>>(
      A0, lda, G, n, Y, p, m, s, idx, val, cnt, ores, err, rl, rc, rcap);
  return cudaGetLastError();
}

}  // namespace

// Taken where it is the faster one (us, omp_warp_kernel's in brackets).  n <= 128: from
// eight warps of signals per SM on, when the Gram matrix pays in shared memory
// (s = 4, n = 128: m = 10,000 10.0 (12.7), m = 1000 5.8 (3.8)).  n <= 256: s <= 6 (n = 256,
// m = 20,000: s = 2 12.3 (17.4), s = 6 35.2 (47.2), s = 8 60.6 (58.8); m = 3000, s = 6 8.0 (9.7)).
bool omp_sub_supported(int n, int s, int64_t m) {
  if (n < 1 || n > 256 || s < 1 || s > SUB_SMAX) return false;
  return n <= 128 ? m >= 32 * (int64_t)num_sms() : s <= 6 && m >= 16 * (int64_t)num_sms();
}

cudaError_t omp_sub(const float* A0, int64_t lda, const float* G, int n, const float* Y, int p, int64_t m,
                    int s, int32_t* idx, float* val, int32_t* cnt, float* ores, int* err, int* rl, int* rc,
                    int rcap, cudaStream_t st) {
  if (!omp_sub_supported(n, s, m)) return cudaErrorInvalidValue;
  // tbits of the 32-atom blocks omp_warp_kernel has for this n
  if (n <= 64)
    return launch_sub<8, 2, tbits<2>()>(A0, lda, G, n, Y, p, m, s, idx, val, cnt, ores, err, rl, rc, rcap, st);
  if (n <= 128)
    return launch_sub<8, 4, tbits<4>()>(A0, lda, G, n, Y, p, m, s, idx, val, cnt, ores, err, rl, rc, rcap, st);
  return launch_sub<16, 4, tbits<8>()>(A0, lda, G, n, Y, p, m, s, idx, val, cnt, ores, err, rl, rc, rcap, st);
}

}  // namespace dlk
