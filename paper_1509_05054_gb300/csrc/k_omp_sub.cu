// Batch-OMP sparse coding of several signals per warp, for small dictionaries and
// short supports (Algorithm 1 step 1; n <= 256, s <= 8; the arithmetic of
// omp_warp_kernel, see k_omp.cu, operation by operation, so the results are the
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

#include <math.h>

#include <algorithm>

namespace dlk {
namespace {

using namespace omp;

constexpr int SUB_SMAX = 8;
constexpr int SUB_WARPS = 24;                // most warps per CTA (one CTA per SM)
constexpr size_t kSubSmem = 220 * 1024;      // dynamic shared memory of a CTA

__device__ __forceinline__ float4 ld_stream4(const float* p) {
  float4 v;
  asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p));
  return v;
}
__device__ __forceinline__ float4 f4_fma2(float2 a, float4 b, float4 c) {
  const float2 lo = __ffma2_rn(a, make_float2(b.x, b.y), make_float2(c.x, c.y));
  const float2 hi = __ffma2_rn(a, make_float2(b.z, b.w), make_float2(c.z, c.w));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Floats of one signal: alpha and u_q (q < s - 1) of NP = 4 SW V each, s x s Cholesky rows.
template <int SW, int V>
__host__ __device__ constexpr int sub_signal_floats(int s) {
  return s * 4 * SW * V + (s * s + 3) / 4 * 4;
}

// TB: truncated mantissa bits; GSH: G in shared memory (pitch NP); VEC: rows of G
// in global memory as float4 (n % 4 == 0).
template <int SW, int V, int TB, bool GSH, bool VEC>
__global__ void __launch_bounds__(SUB_WARPS * 32, 1) omp_sub_kernel(
    const float* __restrict__ A0, int64_t lda, const float* __restrict__ G, int n,
    const float* __restrict__ Y, int p, int64_t m, int s, int32_t* __restrict__ oidx,
    float* __restrict__ oval, int32_t* __restrict__ ocnt, float* __restrict__ ores,
    int* __restrict__ err, int* __restrict__ rs_list, int* __restrict__ rs_count, int rs_cap) {
  constexpr int SPW = 32 / SW, NP = 4 * SW * V;
  constexpr unsigned VMASK = 0x7FFFFFFFu & ~((1u << TB) - 1u);
  static_assert(V <= (1 << TB), "vector number in the truncated bits");
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int sub = lane / SW, l = lane % SW;
  const float* Gs = sm;
  float* base = sm + (GSH ? n * NP : 0) + (warp * SPW + sub) * sub_signal_floats<SW, V>(s);
  float* L = base + s * NP;
  float4* al = (float4*)base + l;                    // alpha: vector v at al[SW v]
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
    // ||y||^2, summed as a warp sums it (element r on lane r mod 32, then a tree by halves)
    float yy;
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
      if constexpr (SW == 8) yy = (t[0] + t[2]) + (t[1] + t[3]);
      else yy = t[0] + t[1];
#pragma unroll
      for (int o = SW / 2; o > 0; o >>= 1) yy += __shfl_xor_sync(FULL, yy, o);
    }
    bool act = live && isfinite(yy);
    if (live && !isfinite(yy) && l == 0) atomicOr(err, ERR_NONFINITE);
    float myc = 0.f, myz = 0.f;  // lane q: c_q = 1 / L_qq, z_q
    int myI = -1;                // lane q: I_q
    float rr = yy;
    int k = 0;
    float kmax = 0.f;
    auto keys = [&]() {  // this lane's largest key
      kmax = 0.f;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        auto key = [&](float x) {
          return __uint_as_float((__float_as_uint(x) & VMASK) | (uint32_t)(V - 1 - v));
        };
        kmax = fmax3(kmax, fmaxf(key(a[v].x), key(a[v].y)), fmaxf(key(a[v].z), key(a[v].w)));
      }
    };
#pragma unroll
    for (int v = 0; v < V; ++v) al[SW * v] = a[v];
    keys();
    __syncwarp();
#pragma unroll 1
    for (int step = 0; step < s; ++step) {
      // ---- argmax over the signal's lanes
      float km = kmax;
#pragma unroll
      for (int o = SW / 2; o > 0; o >>= 1) km = fmaxf(km, __shfl_xor_sync(FULL, km, o));
      const unsigned kb = __float_as_uint(km);
      if ((kb & VMASK) == 0u) act = false;  // max |alpha| = 0
      if (!__any_sync(FULL, act)) break;
      const unsigned ball = __ballot_sync(FULL, __float_as_uint(kmax) == kb) >> (sub * SW);
      const int lsel = __ffs(ball) - 1;
      const int vsel = lsel + SW * (V - 1 - (int)(kb & ((1u << TB) - 1u)) % V);
      const int vs = act ? vsel : 0;  // (in range also for a signal that has stopped)
      const float4 q4 = ((const float4*)base)[vs];
      int e = 3;
      float asel = q4.w;
      if ((__float_as_uint(q4.z) & VMASK) == (kb & VMASK)) e = 2, asel = q4.z;
      if ((__float_as_uint(q4.y) & VMASK) == (kb & VMASK)) e = 1, asel = q4.y;
      if ((__float_as_uint(q4.x) & VMASK) == (kb & VMASK)) e = 0, asel = q4.x;
      const int sel = act ? 4 * vs + e : 0;
      // ---- the Gram loads: diagonal and row
      const bool need_u = step + 1 < s;
      const float gss = GSH ? Gs[sel * NP + sel] : __ldg(G + (size_t)sel * n + sel);
      float4 g[V];
      if (need_u) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int j = 4 * (l + SW * v);
          if (GSH) {
            g[v] = *(const float4*)(Gs + sel * NP + j);
          } else if (VEC) {
            g[v] = j < n ? __ldg((const float4*)(G + (size_t)sel * n + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
          } else {
            const float* Gr = G + (size_t)sel * n;
            g[v].x = j < n ? __ldg(Gr + j) : 0.f;
            g[v].y = j + 1 < n ? __ldg(Gr + j + 1) : 0.f;
            g[v].z = j + 2 < n ? __ldg(Gr + j + 2) : 0.f;
            g[v].w = j + 3 < n ? __ldg(Gr + j + 3) : 0.f;
          }
        }
      }
      // ---- Cholesky row: lane q < step: w_q = c_q u_q[sel]
      const float ul = l < step ? base[(1 + l) * NP + sel] : 0.f;
      const float w = ul * myc, negaw = -w * myc;
      float wsq = 0.f;
      for (int q = 0; q < step; ++q) {
        const float wq = __shfl_sync(FULL, w, q, SW);
        wsq = fmaf(wq, wq, wsq);
      }
      if (l < step) L[step * s + l] = w;
      const float delta = gss - wsq;
      if (act && !(delta > kPivotMin)) {
        if (l == 0) {
          if (!isfinite(delta)) atomicOr(err, ERR_NONFINITE);
          if (rs_count) {  // rounding dominates this pivot: redo the signal in FP64
            const int pos = atomicAdd(rs_count, 1);
            if (pos < rs_cap) rs_list[pos] = (int)i;
          }
        }
        act = false;
      }
      // c_k = 1 / L_kk: rsqrtf refined by one Newton-Raphson step, y + y (1 - d y^2) / 2
      float ck = rsqrtf(delta);
      ck = fmaf(0.5f * ck, fmaf(-delta * ck, ck, 1.0f), ck);
      const float zk = asel * ck;
      if (act) {
        if (l == step) {
          myc = ck;
          myz = zk;
          myI = sel;
        }
        rr = fmaf(-zk, zk, rr);
        k = step + 1;
        if (l == 0) base[sel] = qnan;  // selected: masked from now on
      }
      __syncwarp();
      // ---- u_step = G[:, sel] + sum_q negaw_q u_q;  alpha -= (z_k c_k) u_step
      if (need_u) {
#pragma unroll
        for (int v = 0; v < V; ++v) a[v] = al[SW * v];
#pragma unroll 2
        for (int q = 0; q < step; ++q) {
          const float nq = __shfl_sync(FULL, negaw, q, SW);
          const float2 n2 = make_float2(nq, nq);
          const float4* uq = al + (1 + q) * (NP / 4);
#pragma unroll
          for (int v = 0; v < V; ++v) g[v] = f4_fma2(n2, uq[SW * v], g[v]);
        }
        const float nz = -zk * ck;
        const float2 nz2 = make_float2(nz, nz);
        float4* us = al + (1 + step) * (NP / 4);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          us[SW * v] = g[v];
          a[v] = f4_fma2(nz2, g[v], a[v]);
          al[SW * v] = a[v];
        }
        keys();
      }
      if (rr <= kResidRel * yy) act = false;
      __syncwarp();
    }
    // ---- back substitution L^T gamma = z
    float gam = 0.f, acc2 = 0.f;
    for (int q = s - 1; q >= 0; --q) {
      const float gl = (myz - acc2) * myc;  // valid on lane q
      const float gq = __shfl_sync(FULL, gl, q, SW);
      if (q < k) {
        if (l == q) gam = gq;
        if (l < q) acc2 = fmaf(L[q * s + l], gq, acc2);
      }
    }
    // ---- the support in ascending atom order
    int rank = 0;
    for (int q = 0; q < s; ++q) {
      const int Iq = __shfl_sync(FULL, myI, q, SW);
      rank += q < k && Iq < myI ? 1 : 0;
    }
    if (live) {
      const int64_t o = i * s;
      if (l < k) {
        oidx[o + rank] = myI;
        oval[o + rank] = gam;
      } else if (l < s) {
        oidx[o + l] = -1;
        oval[o + l] = 0.f;
      }
      if (l == 0) {
        ocnt[i] = k;
        if (ores) ores[i] = rr;
      }
    }
    __syncwarp();
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
