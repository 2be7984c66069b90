// Batch-OMP of several signals per warp, in step: the loop shared by the kernel for
// small dictionaries (k_omp_sub.cu, where the layout is described) and the kernel for
// whole small problems (k_small.cu).  Internal to the library.
#pragma once

#include "dl_internal.cuh"
#include "omp_common.cuh"

#include <math.h>

namespace dlk {
namespace {

using namespace omp;

constexpr int SUB_SMAX = 8;

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

// ||y||^2 of a signal by its SW lanes, summed as a warp sums it: t[h] is the sum
// of squares of the elements l + SW h + 32 k, then a tree by halves.
template <int SW>
__device__ __forceinline__ float sub_norm2(const float (&t)[32 / SW]) {
  float yy;
  if constexpr (SW == 8) yy = (t[0] + t[2]) + (t[1] + t[3]);
  else yy = t[0] + t[1];
#pragma unroll
  for (int o = SW / 2; o > 0; o >>= 1) yy += __shfl_xor_sync(FULL, yy, o);
  return yy;
}

// The OMP of the signal i of each group of SW lanes (live: there is one), from its
// correlations a (vector v of lane l: atoms 4 (l + SW v) .., NaN past n) and yy =
// ||y||^2.  base: the signal's shared memory, sub_signal_floats(s) floats.  TB:
// truncated mantissa bits of the argmax.  gram: diag(j) and vec(row, j) (four entries).
// Writes the slots, the count and (when given) the residual-energy estimate.
template <int SW, int V, int TB, class Gram>
__device__ __forceinline__ void omp_sub_core(int64_t i, bool live, float4 (&a)[V], float yy, const Gram& gram,
                                             float* base, int s, int32_t* __restrict__ oidx,
                                             float* __restrict__ oval, int32_t* __restrict__ ocnt,
                                             float* __restrict__ ores, int* __restrict__ err,
                                             int* __restrict__ rs_list, int* __restrict__ rs_count,
                                             int rs_cap) {
  constexpr int NP = 4 * SW * V;
  constexpr unsigned VMASK = 0x7FFFFFFFu & ~((1u << TB) - 1u);
  static_assert(V <= (1 << TB), "vector number in the truncated bits");
  const int lane = threadIdx.x & 31, sub = lane / SW, l = lane % SW;
  float* L = base + s * NP;
  float4* al = (float4*)base + l;  // alpha: vector v at al[SW v]
  const float qnan = __int_as_float(0x7fc00000);
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
    const float gss = gram.diag(sel);
    float4 g[V];
    if (need_u) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int j = 4 * (l + SW * v);
        g[v] = gram.vec(sel, j);
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
    __syncwarp();  // every lane has read the selected atom's four correlations
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

}  // namespace
}  // namespace dlk
