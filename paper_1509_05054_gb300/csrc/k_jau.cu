// Jacobi atom update in the AK-SVD form with full parallelism (PAK-SVD,
// group size n; Section 3, Eq. 3 and Eq. 5; Algorithm 2 with step 4 replaced
// by Eq. 5).  With E = Y - D X formed once:
//   F_j x_j^T = E_{I_j} x_{j,I_j}^T + ||x_{j,I_j}||^2 d_j  =  U_j + r_j d_j
//   d_j'      = (U_j + r_j d_j) / ||U_j + r_j d_j||
//   x_{j,i}'  = F^T d_j' = e_i^T d_j' + (d_j^T d_j') x_{j,i}      for i in I_j
// U = E X^T (p x n) and r_j = ||x_j||^2 are accumulated signal by signal (the
// support sets I_j are never materialised), then every atom is updated by one
// warp, then every signal recomputes its error and its coefficients.
//
// The passes over the signals give each signal eight lanes (four signals per
// warp).  With enough signals the plain case (all atoms at once, AK-SVD or SGK) runs
// as three passes: errors stored, sums of the pairs sorted by atom, rows (see
// errors_kernel).  Otherwise, with p % 4 == 0 and 16-byte aligned Y and D, pass A
// adds x e_i into 16 copies of U with vector reductions in L2 (red.v4.f32); else it
// keeps per-CTA copies of U (shared memory when they fit).  The copies are summed in
// a fixed order, and so are the energy partial sums.
#include "dl_internal.cuh"
#include "tc_ptx.cuh"

#include <math.h>

namespace dlk {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int ACC_THREADS = 1024;
constexpr int ROW_THREADS = 256;
constexpr int ACC4_THREADS = 256;
constexpr int kMaxAtoms = 1024;  // largest n the library accepts

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// Sum of the warp's 32 non-negative FP32 values in FP64: integers in units of 2^-56
// of the largest value's binade (24 bits and 33 more), added exactly by three integer
// reductions of 27, 27 and 3 bits each.  What is cut off and the conversion are below
// 2^-51 of the sum, as the roundings of five FP64 additions are, over the whole range.
__device__ __forceinline__ double warp_sum_fixed(float v) {
  const unsigned b = __float_as_uint(v) & 0x7fffffffu;
  const int top = (int)(__reduce_max_sync(FULL, b) >> 23);
  if (top == 255) return (double)warp_sum(v);  // infinite or NaN, as the plain sum
  const int ex = (int)(b >> 23), e = ex > 0 ? ex : 1, et = top > 0 ? top : 1;  // (subnormals: no leading one)
  const unsigned long long mant = (unsigned long long)((b & 0x7fffffu) | (ex > 0 ? 0x800000u : 0u)) << 33;
  const unsigned long long q = et - e < 57 ? mant >> (et - e) : 0ull;
  const unsigned long long s0 = __reduce_add_sync(FULL, (unsigned)q & 0x7ffffffu);
  const unsigned long long s1 = __reduce_add_sync(FULL, (unsigned)(q >> 27) & 0x7ffffffu);
  const unsigned long long s2 = __reduce_add_sync(FULL, (unsigned)(q >> 54));
  return (double)(s0 + (s1 << 27) + (s2 << 54)) * __hiloint2double((et + 840) << 20, 0);  // 2^(et - 183)
}

// Block-wide sum of the threads' FP32 partial sums (not negative); result valid on
// thread 0.  FP64 instructions run at 1/64 of the FP32 rate, and a kernel's last CTAs
// all sum at once (two FP64 sums of every thread cost the errors pass 3.5 us of
// 16.5), so a warp's sum is taken in integers and only one value per warp is FP64.
__device__ double block_sum_f(float v, double* scratch) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const double s = warp_sum_fixed(v);
  __syncthreads();
  if (lane == 0) scratch[w] = s;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < nw; ++q) r += scratch[q];
  return r;
}

// Pass A: e_i = y_i - D x_i; U[:, j] += x_{j,i} e_i; r_j += x_{j,i}^2;
// partial ||E||^2 and ||Y||^2.  Eight lanes per signal (four signals per warp):
// lane g of group q holds rows g + 8((t + q) mod RL), t < RL (p <= 8*RL); the
// rotation by q puts the four groups' shared-memory atomics on distinct banks.
// Support slots t and t + 8 live on group lane t % 8.
template <int RL, bool SMEM>
__global__ void __launch_bounds__(ACC_THREADS, 1) accum_kernel(
    const float* __restrict__ Y, int p, int64_t m, const float* __restrict__ D, int n, int s,
    const int32_t* __restrict__ idx, const float* __restrict__ val, const int32_t* __restrict__ cnt,
    float* __restrict__ Upart, double* __restrict__ epart, int* __restrict__ err) {
  extern __shared__ float sh[];
  __shared__ double red[ACC_THREADS / 32];
  const int lane = threadIdx.x & 31;
  const int g = lane & 7, gbase = lane & ~7;
  const int q = (threadIdx.x >> 3) & 3;
  int row[RL];
#pragma unroll
  for (int t = 0; t < RL; ++t) row[t] = g + 8 * ((t + q) % RL);
  const int np = n * p;
  float* U = SMEM ? sh : Upart;  // atom-major: U[j*p + r]; then r_j at U[np + j]
  if (SMEM) {
    for (int q = threadIdx.x; q < np + n; q += blockDim.x) U[q] = 0.f;
    __syncthreads();
  }
  float ee = 0.f, yy = 0.f;
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x >> 3);
  const int64_t g0 = (int64_t)blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 3);
  // every lane of a warp loops the same number of times (shuffles stay converged)
  const int64_t trips = (m + groups - 1) / groups;
  for (int64_t k = 0; k < trips; ++k) {
    const int64_t i = g0 + k * groups;
    const bool live = i < m;
    float e[RL];
#pragma unroll
    for (int t = 0; t < RL; ++t) {
      const int r = row[t];
      e[t] = (live && r < p) ? Y[i * p + r] : 0.f;
      yy = fmaf(e[t], e[t], yy);
    }
    const int c = live ? cnt[i] : 0;
    const int j0 = (g < c) ? idx[i * s + g] : 0;
    const float x0 = (g < c) ? val[i * s + g] : 0.f;
    const int j1 = (g + 8 < c) ? idx[i * s + g + 8] : 0;
    const float x1 = (g + 8 < c) ? val[i * s + g + 8] : 0.f;
    const int cmax = __reduce_max_sync(0xffffffffu, (unsigned)c);
    for (int t = 0; t < cmax; ++t) {
      const int jj = __shfl_sync(0xffffffffu, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(0xffffffffu, t < 8 ? x0 : x1, gbase + (t & 7));
      if (t < c) {
#pragma unroll
        for (int u = 0; u < RL; ++u) {
          const int r = row[u];
          if (r < p) e[u] = fmaf(-xx, __ldg(D + (size_t)jj * p + r), e[u]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < RL; ++u) ee = fmaf(e[u], e[u], ee);
    for (int t = 0; t < cmax; ++t) {
      const int jj = __shfl_sync(0xffffffffu, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(0xffffffffu, t < 8 ? x0 : x1, gbase + (t & 7));
      if (t < c) {
#pragma unroll
        for (int u = 0; u < RL; ++u) {
          const int r = row[u];
          if (r < p) atomicAdd(&U[(size_t)jj * p + r], xx * e[u]);
        }
        if (g == 0) atomicAdd(&U[np + jj], xx * xx);
      }
    }
  }
  if (!isfinite(ee) || !isfinite(yy)) atomicOr(err, ERR_NONFINITE);
  if (SMEM) {
    __syncthreads();
    float* out = Upart + (size_t)blockIdx.x * (np + n);
    for (int q = threadIdx.x; q < np + n; q += blockDim.x) out[q] = U[q];
  }
  const double see = block_sum_f(ee, red);
  const double syy = block_sum_f(yy, red);
  if (threadIdx.x == 0) {
    epart[2 * blockIdx.x] = see;
    epart[2 * blockIdx.x + 1] = syy;
  }
}

// ---- float4 forms (p % 4 == 0, Y and D 16-byte aligned) ----
// Eight lanes per signal; lane g holds the float4 vectors v = g + 8k (rows
// 4v..4v+3), k < RV, p <= 32 RV.  The support loops are unrolled to SMAX.

__device__ __forceinline__ void red_add_v4(float* addr, float4 v) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ float4 f4_fma(float a, float4 b, float4 c) {
  return make_float4(fmaf(a, b.x, c.x), fmaf(a, b.y, c.y), fmaf(a, b.z, c.z), fmaf(a, b.w, c.w));
}
__device__ __forceinline__ float f4_dot(float4 a, float4 b, float acc) {
  return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, acc))));
}

// Pass A, float4 form: CTA b adds x_{j,i} e_i into copy b mod kUCopies of U
// (zeroed, p x n atom-major, then r at + n p) by vector reductions in L2
// (native FP32 adds); r_j is summed per CTA in shared memory and added once per
// CTA.  Spreading the reductions over several copies keeps the L2 lines of
// frequently used atoms from serialising them; the copies are then summed in a
// fixed order.
// NS (P-NSGK, Eq. 7): the error is that of Z = Y + D0 Xp - D0 X against the
// current atoms and the previous representations Xp, e = y - D0 x + (D0 - D) xp
// (D0: the dictionary the iteration started from; equal to D before any group
// has moved), and U, r are accumulated over Xp's supports and values.  *pvalid
// == 0 means there are no previous representations yet: Xp = X.
template <int RV, int SMAX, bool NS>
__global__ void __launch_bounds__(ACC4_THREADS, 4) accum4_kernel(
    const float* __restrict__ Y, int p, int64_t m, const float* __restrict__ D, int n, int s,
    const int32_t* __restrict__ idx, const float* __restrict__ val, const int32_t* __restrict__ cnt,
    float* __restrict__ U, double* __restrict__ epart, int* __restrict__ err, int a0, int a1,
    int energies, const float* __restrict__ D0, const int32_t* __restrict__ pidx,
    const float* __restrict__ pval, const int32_t* __restrict__ pcnt,
    const int* __restrict__ pvalid, int moved) {
  __shared__ float rsh[kMaxAtoms];
  __shared__ double red[ACC4_THREADS / 32];
  for (int j = threadIdx.x; j < n; j += blockDim.x) rsh[j] = 0.f;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int g = lane & 7, gbase = lane & ~7;
  const int pv = p >> 2;
  const float4* __restrict__ Y4 = (const float4*)Y;
  const float4* __restrict__ D4 = (const float4*)(NS ? D0 : D);
  const float4* __restrict__ Dc4 = (const float4*)D;
  const bool have_prev = NS && *pvalid != 0;
  const int32_t* __restrict__ sidx = have_prev ? pidx : idx;
  const float* __restrict__ sval = have_prev ? pval : val;
  const int32_t* __restrict__ scnt = have_prev ? pcnt : cnt;
  float* __restrict__ Uc = U + (size_t)(blockIdx.x % kUCopies) * jau_ulen(p, n);
  float ee = 0.f, yy = 0.f;
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x >> 3);
  const int64_t g0 = (int64_t)blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 3);
  const int64_t trips = (m + groups - 1) / groups;
  for (int64_t k = 0; k < trips; ++k) {
    const int64_t i = g0 + k * groups;
    const bool live = i < m;
    float4 e[RV];
#pragma unroll
    for (int q = 0; q < RV; ++q) {
      const int v = g + 8 * q;
      e[q] = (live && v < pv) ? Y4[i * pv + v] : make_float4(0.f, 0.f, 0.f, 0.f);
      yy = f4_dot(e[q], e[q], yy);
    }
    const int c = live ? cnt[i] : 0;
    const int j0 = (g < c) ? idx[i * s + g] : 0;
    const float x0 = (g < c) ? val[i * s + g] : 0.f;
    const int j1 = (SMAX > 8 && g + 8 < c) ? idx[i * s + g + 8] : 0;
    const float x1 = (SMAX > 8 && g + 8 < c) ? val[i * s + g + 8] : 0.f;
    const int cmax = __reduce_max_sync(FULL, (unsigned)c);
#pragma unroll
    for (int t = 0; t < SMAX; ++t) {
      if (t >= cmax) break;
      const int jj = __shfl_sync(FULL, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(FULL, t < 8 ? x0 : x1, gbase + (t & 7));
      if (t < c) {
#pragma unroll
        for (int q = 0; q < RV; ++q) {
          const int v = g + 8 * q;
          if (v < pv) e[q] = f4_fma(-xx, __ldg(D4 + (size_t)jj * pv + v), e[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < RV; ++q) ee = f4_dot(e[q], e[q], ee);
    // the slots whose contributions are accumulated: X, or Xp for P-NSGK
    int sc = c, sj0 = j0, sj1 = j1, scmax = cmax;
    float sx0 = x0, sx1 = x1;
    if (NS) {
      sc = live ? scnt[i] : 0;
      sj0 = (g < sc) ? sidx[i * s + g] : 0;
      sx0 = (g < sc) ? sval[i * s + g] : 0.f;
      sj1 = (SMAX > 8 && g + 8 < sc) ? sidx[i * s + g + 8] : 0;
      sx1 = (SMAX > 8 && g + 8 < sc) ? sval[i * s + g + 8] : 0.f;
      scmax = __reduce_max_sync(FULL, (unsigned)sc);
      if (moved) {  // e += (D0 - D) xp for the atoms earlier groups have moved
#pragma unroll
        for (int t = 0; t < SMAX; ++t) {
          if (t >= scmax) break;
          const int jj = __shfl_sync(FULL, t < 8 ? sj0 : sj1, gbase + (t & 7));
          const float xx = __shfl_sync(FULL, t < 8 ? sx0 : sx1, gbase + (t & 7));
          if (t < sc) {
#pragma unroll
            for (int q = 0; q < RV; ++q) {
              const int v = g + 8 * q;
              if (v < pv) {
                e[q] = f4_fma(xx, __ldg(D4 + (size_t)jj * pv + v), e[q]);
                e[q] = f4_fma(-xx, __ldg(Dc4 + (size_t)jj * pv + v), e[q]);
              }
            }
          }
        }
      }
    }
#pragma unroll
    for (int t = 0; t < SMAX; ++t) {
      if (t >= scmax) break;
      const int jj = __shfl_sync(FULL, t < 8 ? sj0 : sj1, gbase + (t & 7));
      const float xx = __shfl_sync(FULL, t < 8 ? sx0 : sx1, gbase + (t & 7));
      if (t < sc && jj >= a0 && jj < a1) {
#pragma unroll
        for (int q = 0; q < RV; ++q) {
          const int v = g + 8 * q;
          if (v < pv)
            red_add_v4(Uc + ((size_t)jj * pv + v) * 4,
                       make_float4(xx * e[q].x, xx * e[q].y, xx * e[q].z, xx * e[q].w));
        }
        if (g == 0) atomicAdd(&rsh[jj], xx * xx);
      }
    }
  }
  if (!isfinite(ee) || !isfinite(yy)) atomicOr(err, ERR_NONFINITE);
  __syncthreads();
  const size_t np = (size_t)n * p;
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    if (rsh[j] != 0.f) atomicAdd(Uc + np + j, rsh[j]);
  const double see = block_sum_f(ee, red);
  const double syy = block_sum_f(yy, red);
  if (threadIdx.x == 0 && energies) {
    epart[2 * blockIdx.x] = see;
    epart[2 * blockIdx.x + 1] = syy;
  }
}

// ---- The plain case: errors, bucketed sums, rows -------------------------------
// All atoms at once (no groups, no P-NSGK).  Rows whose length is no multiple of
// four floats, or that do not start on 16 bytes, are read float by float from Y; the
// atoms are then padded once per update (Dp), and E, U and D' have padded rows (p4).
// What bounds accum4_kernel
// is the L2's reduction rate: s rows of p floats per signal, 205 MB of vector
// reductions at p = 64, n = 512, s = 8, m = 1e5 (44.9 us), and what bounds
// rows4_kernel is issuing about 1,000 instructions per four signals (33.7 us).
// Three passes instead:
//   errors_kernel  E = Y - D X, stored; no shared memory, so that L1 holds the
//                  atoms (gathered from L2 they cost twice as much);
//   sums_kernel    U = E X^T and r: a CTA takes a tile of E into shared memory,
//                  buckets the tile's (signal, x) pairs by atom (a counting sort: the
//                  shared-memory counter of the atom gives the pair's rank), and
//                  sums runs of equal atoms in registers; U in L2 gets one row
//                  per atom and tile (plus one per share of the pairs);
//   rows_kernel    x' and the final error from E and the rows of D'.
// The eight lanes of a signal take four slots at a time without branches, so that
// eight 16-byte gathers per lane are in flight; the four dot products of a group
// are summed together by halving exchanges (4 shuffles instead of 12).
// Measured at the size above: 15.7, 17.4 and 18.1 us.
constexpr int EP_THREADS = 256;

// Two packed multiply-adds: c + a b.
__device__ __forceinline__ float4 f4_fma2(float a, float4 b, float4 c) {
  const float2 lo = __ffma2_rn(make_float2(a, a), make_float2(b.x, b.y), make_float2(c.x, c.y));
  const float2 hi = __ffma2_rn(make_float2(a, a), make_float2(b.z, b.w), make_float2(c.z, c.w));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ float f4_sum(float4 v) { return (v.x + v.y) + (v.z + v.w); }

// Lane g's vector q of a row of pv vectors at base (valid when g + 8 q < pv).
template <int RV, bool FULLP>
__device__ __forceinline__ void load_row(float4 (&r)[RV], const float4* base, int g, int pv, bool on) {
#pragma unroll
  for (int q = 0; q < RV; ++q)
    r[q] = on && (FULLP || g + 8 * q < pv) ? __ldg(base + g + 8 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// The same of a row that is read once: not kept in L1, which is left to the atoms.
__device__ __forceinline__ float4 ld_once(const float4* a) {
  float4 v;
  asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(a));
  return v;
}
template <int RV, bool FULLP>
__device__ __forceinline__ void load_once(float4 (&r)[RV], const float4* base, int g, int pv, bool on) {
#pragma unroll
  for (int q = 0; q < RV; ++q)
    r[q] = on && (FULLP || g + 8 * q < pv) ? ld_once(base + g + 8 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// Lane g's vectors of the signal at y (p floats): as float4 (YV), or float by float.
template <int RV, bool FULLP, bool YV>
__device__ __forceinline__ void load_signal(float4 (&r)[RV], const float* __restrict__ y, int p, int g, int pv,
                                            bool on) {
  if constexpr (YV) {
    load_once<RV, FULLP>(r, (const float4*)y, g, pv, on);
  } else {
#pragma unroll
    for (int q = 0; q < RV; ++q) {
      const int c = 4 * (g + 8 * q);
      r[q].x = on && c < p ? __ldg(y + c) : 0.f;
      r[q].y = on && c + 1 < p ? __ldg(y + c + 1) : 0.f;
      r[q].z = on && c + 2 < p ? __ldg(y + c + 2) : 0.f;
      r[q].w = on && c + 3 < p ? __ldg(y + c + 3) : 0.f;
    }
  }
}

// The atoms with rows padded by zeros to p4 floats.
__global__ void pad_atoms_kernel(const float* __restrict__ D, int p, int n, int p4, float* __restrict__ Dp) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n * p4) return;
  const int j = q / p4, r = q - j * p4;
  Dp[q] = r < p ? D[(size_t)j * p + r] : 0.f;
}

// A signal's slots over its eight lanes: lane g holds slots g and g + 8.
struct Slots {
  int c, j0, j1;
  float x0, x1;
};
__device__ __forceinline__ Slots load_slots(int64_t i, bool live, int g, int s, const int32_t* __restrict__ idx,
                                            const float* __restrict__ val, const int32_t* __restrict__ cnt) {
  Slots q;
  q.c = live ? cnt[i] : 0;
  const bool a = live && g < s, b = live && g + 8 < s;  // (unused slots: atom -1, masked by the count)
  q.j0 = a ? idx[i * s + g] : -1;
  q.x0 = a ? val[i * s + g] : 0.f;
  q.j1 = b ? idx[i * s + g + 8] : -1;
  q.x1 = b ? val[i * s + g + 8] : 0.f;
  return q;
}

// D and E have rows of p4 floats.
template <int RV, bool FULLP, bool YV>
__global__ void __launch_bounds__(EP_THREADS, RV <= 2 ? 4 : 3) errors_kernel(
    const float* __restrict__ Y, int p, int p4, int64_t m, const float* __restrict__ D, int s,
    const int32_t* __restrict__ idx, const float* __restrict__ val, const int32_t* __restrict__ cnt,
    float* __restrict__ E, double* __restrict__ epart, int* __restrict__ err, float4* __restrict__ Uc,
    int ulen4) {
  __shared__ double red[EP_THREADS / 32];
  // the copies of U that sums_kernel adds to
  for (int q = blockIdx.x * EP_THREADS + threadIdx.x; q < ulen4; q += gridDim.x * EP_THREADS)
    Uc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int lane = threadIdx.x & 31, g = lane & 7, gbase = lane & ~7;
  const int pv = p4 >> 2;
  const float4* __restrict__ D4 = (const float4*)D;
  float ee = 0.f, yy = 0.f;
  const int64_t groups = (int64_t)gridDim.x * (EP_THREADS / 8);
  const int64_t trips = (m + groups - 1) / groups;
  int64_t i = (int64_t)blockIdx.x * (EP_THREADS / 8) + (threadIdx.x >> 3);
  Slots next = load_slots(i, i < m, g, s, idx, val, cnt);
  for (int64_t k = 0; k < trips; ++k, i += groups) {
    const bool live = i < m;
    const Slots sl = next;  // (loaded a trip ahead: the gathers start at once)
    float4 e[RV];
    load_signal<RV, FULLP, YV>(e, Y + (live ? i : 0) * p, p, g, pv, live);
    next = load_slots(i + groups, i + groups < m, g, s, idx, val, cnt);
    const int c = sl.c, o0 = sl.j0 * pv, o1 = sl.j1 * pv;  // row offsets in vectors
    const float x0 = sl.x0, x1 = sl.x1;
    const int cmax = __reduce_max_sync(FULL, (unsigned)c);
    for (int t0 = 0; t0 < cmax; t0 += 4) {
      float4 d[4][RV];
      float x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int src = gbase + ((t0 + u) & 7);
        const int o = __shfl_sync(FULL, t0 < 8 ? o0 : o1, src);
        x[u] = __shfl_sync(FULL, t0 < 8 ? x0 : x1, src);
        load_row<RV, FULLP>(d[u], D4 + o, g, pv, t0 + u < c);
      }
      if (t0 == 0) {
#pragma unroll
        for (int q = 0; q < RV; ++q) yy = f4_dot(e[q], e[q], yy);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < RV; ++q) e[q] = f4_fma2(t0 + u < c ? -x[u] : 0.f, d[u][q], e[q]);
    }
    if (cmax == 0) {
#pragma unroll
      for (int q = 0; q < RV; ++q) yy = f4_dot(e[q], e[q], yy);
    }
#pragma unroll
    for (int q = 0; q < RV; ++q) {
      ee = f4_dot(e[q], e[q], ee);
      if (live && (FULLP || g + 8 * q < pv)) ((float4*)E)[i * pv + g + 8 * q] = e[q];
    }
  }
  if (!isfinite(ee) || !isfinite(yy)) atomicOr(err, ERR_NONFINITE);
  const double see = block_sum_f(ee, red);
  const double syy = block_sum_f(yy, red);
  if (threadIdx.x == 0) {
    epart[2 * blockIdx.x] = see;
    epart[2 * blockIdx.x + 1] = syy;
  }
}

constexpr int SUM_THREADS = 512;
constexpr int SUM_SHARES = SUM_THREADS / 16;     // half warps
constexpr int SUM_KEEP = 6;                      // pairs a thread keeps in registers
constexpr size_t SUM_SMEM = 113 * 1024;          // dynamic, two CTAs per SM
struct SumSmem {  // byte offsets, T signals per tile (T % 4 == 0)
  int np, sk, sx, off, rank, total;
  __host__ __device__ SumSmem(int p, int n, int s, int T) {
    np = (T * s + 4 * SUM_SHARES - 1) / (4 * SUM_SHARES) * (4 * SUM_SHARES);  // padded pairs
    sk = T * p * 4;         // after the errors [T][p]: sorted pairs, atom << 16 | signal
    sx = sk + np * 4;       // their x
    off = sx + np * 4;      // pairs per atom, then bucket starts
    rank = off + n * 4;     // rank of each pair in its bucket (u16; unsorted)
    total = rank + (T * s * 2 + 15) / 16 * 16;
  }
};
// Signals per tile: equal tiles for two CTAs per SM, as few per CTA as fit; at
// least 64 where there are few signals.  0: none fits.
int sum_tile(int64_t m, int p, int n, int s) {
  const int64_t g = 2 * num_sms();
  for (int64_t k = 1;; ++k) {
    int64_t T = (m + g * k - 1) / (g * k);
    if (T < 64) T = 64;
    T = (T + 3) / 4 * 4;
    if (T * s < 65536 && T < 65536 && (size_t)SumSmem(p, n, s, (int)T).total <= SUM_SMEM) return (int)T;
    if (T == 64) return 0;
  }
}

__global__ void __launch_bounds__(SUM_THREADS, 2) sums_kernel(
    const float* __restrict__ E, int p, int64_t m, int T, int n, int s, const int32_t* __restrict__ idx,
    const float* __restrict__ val, float* __restrict__ U, int* __restrict__ err) {
  extern __shared__ __align__(128) uint8_t ssh[];
  __shared__ int wsum[SUM_THREADS / 32];
  __shared__ uint64_t bar;
  const SumSmem lay(p, n, s, T);
  const float* Es = (const float*)ssh;
  uint32_t* sk = (uint32_t*)(ssh + lay.sk);
  float* sx = (float*)(ssh + lay.sx);
  int* off = (int*)(ssh + lay.off);
  uint16_t* rank = (uint16_t*)(ssh + lay.rank);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pv = p >> 2;
  float* __restrict__ Uc = U + (size_t)(blockIdx.x % kUCopies) * jau_ulen(p, n);
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int64_t ntiles = (m + T - 1) / T;
  uint32_t phase = 0;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, phase ^= 1) {
    const int64_t lo = tile * T;
    const int nr = (int)(m - lo < T ? m - lo : T);
    const int npair = nr * s;
    __syncthreads();  // the previous tile has been summed
    if (threadIdx.x == 0) {  // the tile's errors, one bulk copy (rows are contiguous; p % 4 == 0)
      const uint32_t bytes = (uint32_t)nr * (uint32_t)p * 4u;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc::mbar_expect_tx(&bar, bytes);
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
              tc::smem_u32(ssh)),
          "l"(E + lo * p), "r"(bytes), "r"(tc::smem_u32(&bar))
          : "memory");
    }
    for (int a = threadIdx.x; a < n; a += SUM_THREADS) off[a] = 0;
    __syncthreads();
    // ---- each pair's rank in its atom's bucket (unused slots hold atom -1); a thread's
    // first pairs stay in registers
    int ka[SUM_KEEP], kr[SUM_KEEP];
    float kx[SUM_KEEP];
#pragma unroll
    for (int u = 0; u < SUM_KEEP; ++u) {
      const int k = threadIdx.x + u * SUM_THREADS;
      ka[u] = k < npair ? idx[lo * s + k] : -1;
      kx[u] = k < npair ? val[lo * s + k] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < SUM_KEEP; ++u) kr[u] = ka[u] >= 0 ? atomicAdd(&off[ka[u]], 1) : 0;
    for (int k = threadIdx.x + SUM_KEEP * SUM_THREADS; k < npair; k += SUM_THREADS) {
      const int a = idx[lo * s + k];
      if (a >= 0) rank[k] = (uint16_t)atomicAdd(&off[a], 1);
    }
    __syncthreads();
    // ---- bucket starts: exclusive scan of the counts in place, two atoms per thread (n <= 1024)
    int np = 0;
    {
      const int a = 2 * threadIdx.x;
      const int v0 = a < n ? off[a] : 0, v1 = a + 1 < n ? off[a + 1] : 0;
      int inc = v0 + v1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += x;
      }
      if (lane == 31) wsum[warp] = inc;
      __syncthreads();
      int before = 0;
#pragma unroll
      for (int w = 0; w < SUM_THREADS / 32; ++w) {
        const int x = wsum[w];
        if (w < warp) before += x;
        np += x;
      }
      const int ex = before + inc - v0 - v1;
      if (a < n) off[a] = ex;
      if (a + 1 < n) off[a + 1] = ex + v0;
    }
    const int share = (np + 4 * SUM_SHARES - 1) / (4 * SUM_SHARES) * 4;  // pairs per half warp
    __syncthreads();
#pragma unroll
    for (int u = 0; u < SUM_KEEP; ++u)
      if (ka[u] >= 0) {
        const int pos = off[ka[u]] + kr[u];
        sk[pos] = (uint32_t)ka[u] << 16 | (uint32_t)((threadIdx.x + u * SUM_THREADS) / s);
        sx[pos] = kx[u];
      }
    for (int k = threadIdx.x + SUM_KEEP * SUM_THREADS; k < npair; k += SUM_THREADS) {
      const int a = idx[lo * s + k];
      if (a >= 0) {
        const int pos = off[a] + rank[k];
        sk[pos] = (uint32_t)a << 16 | (uint32_t)(k / s);
        sx[pos] = val[lo * s + k];
      }
    }
    for (int k = np + threadIdx.x; k < share * SUM_SHARES; k += SUM_THREADS) {  // no atom
      sk[k] = 0xffff0000u;
      sx[k] = 0.f;
    }
    const bool ok = tc::mbar_wait(&bar, phase);
    if (!ok && threadIdx.x == 0) atomicOr(err, ERR_TIMEOUT);
    if (!__syncthreads_and(ok)) break;
    // ---- sums over runs of equal atoms: half a warp takes an equal share of the pairs, 16 lanes a row
    const int hw = threadIdx.x >> 4, l16 = threadIdx.x & 15;
    const int k1 = (hw + 1) * share;
    for (int q0 = 0; q0 < pv; q0 += 16) {  // (a second round of vectors for p > 64)
      const bool on = q0 + l16 < pv;
      const float* col = Es + 4 * (on ? q0 + l16 : 0);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float rx = 0.f;
      for (int k = hw * share; k < k1; k += 4) {
        const uint4 K = *(const uint4*)(sk + k);
        const float4 X = *(const float4*)(sx + k);
        const uint32_t next = k + 4 < k1 ? sk[k + 4] >> 16 : ~0u;
        const uint32_t at[5] = {K.x >> 16, K.y >> 16, K.z >> 16, K.w >> 16, next};
        const float x[4] = {X.x, X.y, X.z, X.w};
        float4 r[4];
        r[0] = *(const float4*)(col + (K.x & 0xffffu) * p);
        r[1] = *(const float4*)(col + (K.y & 0xffffu) * p);
        r[2] = *(const float4*)(col + (K.z & 0xffffu) * p);
        r[3] = *(const float4*)(col + (K.w & 0xffffu) * p);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          acc = f4_fma2(x[h], r[h], acc);
          rx = fmaf(x[h], x[h], rx);
          if (at[h] != at[h + 1]) {  // the run ends
            if (at[h] != 0xffffu) {
              if (on) red_add_v4(Uc + ((size_t)at[h] * pv + q0 + l16) * 4, acc);
              if (l16 == 0 && q0 == 0) atomicAdd(Uc + (size_t)n * p + at[h], rx);
            }
            acc = make_float4(0.f, 0.f, 0.f, 0.f);
            rx = 0.f;
          }
        }
      }
    }
  }
}

// Pass B of the plain case: x_t' = e.d'_{j_t} + c_{j_t} x_t (sgk: x_t) into the CSC
// values, and ||y - D' x'||^2.
template <int RV, bool FULLP, bool YV>
__global__ void __launch_bounds__(EP_THREADS, RV <= 1 ? 4 : RV == 2 ? 3 : 2) rows_plain_kernel(
    const float* __restrict__ Y, const float* __restrict__ E, int p, int p4, int64_t m,
    const float* __restrict__ Dn, const float* __restrict__ C, int s, const int32_t* __restrict__ idx,
    const float* __restrict__ val, const int32_t* __restrict__ cnt, const int64_t* __restrict__ colptr,
    float* __restrict__ csc_val, double* __restrict__ epart, int sgk) {
  __shared__ double red[EP_THREADS / 32];
  const int lane = threadIdx.x & 31, g = lane & 7, gbase = lane & ~7;
  const int b2 = g >> 2 & 1, b1 = g >> 1 & 1, tau = 2 * b2 + b1;  // the slot of four this lane sums
  const int pv = p4 >> 2;
  const float4* __restrict__ N4 = (const float4*)Dn;
  float e2 = 0.f;
  const int64_t groups = (int64_t)gridDim.x * (EP_THREADS / 8);
  const int64_t trips = (m + groups - 1) / groups;
  int64_t i = (int64_t)blockIdx.x * (EP_THREADS / 8) + (threadIdx.x >> 3);
  Slots next = load_slots(i, i < m, g, s, idx, val, cnt);
  for (int64_t k = 0; k < trips; ++k, i += groups) {
    const bool live = i < m;
    const Slots sl = next;
    float4 y[RV], e[RV];
    load_signal<RV, FULLP, YV>(y, Y + (live ? i : 0) * p, p, g, pv, live);
    load_once<RV, FULLP>(e, (const float4*)E + (live ? i : 0) * pv, g, pv, live);
    next = load_slots(i + groups, i + groups < m, g, s, idx, val, cnt);
    const int c = sl.c, j0 = sl.j0, j1 = sl.j1;
    const float x0 = sl.x0, x1 = sl.x1;
    const float c0 = g < c ? __ldg(C + j0) : 0.f, c1 = g + 8 < c ? __ldg(C + j1) : 0.f;
    const int64_t o = live ? colptr[i] : 0;
    const int cmax = __reduce_max_sync(FULL, (unsigned)c);
    for (int t0 = 0; t0 < cmax; t0 += 4) {
      float4 d[4][RV];
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int jj = __shfl_sync(FULL, t0 < 8 ? j0 : j1, gbase + ((t0 + u) & 7));
        load_row<RV, FULLP>(d[u], N4 + jj * pv, g, pv, t0 + u < c);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float2 a = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < RV; ++q) {
          a = __ffma2_rn(make_float2(e[q].x, e[q].y), make_float2(d[u][q].x, d[u][q].y), a);
          a = __ffma2_rn(make_float2(e[q].z, e[q].w), make_float2(d[u][q].z, d[u][q].w), a);
        }
        v[u] = a.x + a.y;
      }
      // four sums over eight lanes: lanes with bit 2 set keep slots 2 and 3, then bit 1 picks one
      const float w0 = (b2 ? v[2] : v[0]) + __shfl_xor_sync(FULL, b2 ? v[0] : v[2], 4);
      const float w1 = (b2 ? v[3] : v[1]) + __shfl_xor_sync(FULL, b2 ? v[1] : v[3], 4);
      float dot = (b1 ? w1 : w0) + __shfl_xor_sync(FULL, b1 ? w0 : w1, 2);
      dot += __shfl_xor_sync(FULL, dot, 1);
      const int src = gbase + ((t0 + tau) & 7);
      const float xo = __shfl_sync(FULL, t0 < 8 ? x0 : x1, src);
      const float co = __shfl_sync(FULL, t0 < 8 ? c0 : c1, src);
      const float xn = sgk ? xo : fmaf(co, xo, dot);
      if (!(g & 1) && t0 + tau < c && csc_val) csc_val[o + t0 + tau] = xn;
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // y - D' x' from the same rows (zero past the count)
        float xu = __shfl_sync(FULL, xn, gbase + 4 * (u >> 1) + 2 * (u & 1));
        if (t0 + u >= c) xu = 0.f;
#pragma unroll
        for (int q = 0; q < RV; ++q) y[q] = f4_fma2(-xu, d[u][q], y[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < RV; ++q) e2 = f4_dot(y[q], y[q], e2);
  }
  const double se = block_sum_f(e2, red);
  if (threadIdx.x == 0) epart[blockIdx.x] = se;
}

// ---- Pass A, deterministic form ---------------------------------------------
// U_j = sum_{i in I_j} x_{j,i} e_i and r_j = sum x_{j,i}^2 summed in an order
// fixed by the signal and slot indices, so that every run gives the same bits
// (float4 rows, p <= 128, n <= 1024, s <= 16).  CTA b owns a contiguous range
// of signals (at most DET_R):
//   1. eight lanes per signal form e_i into shared memory (as accum4_kernel),
//      and the (atom, x) pair of every accumulated slot, numbered k = signal x
//      s + slot within the range; counts per atom;
//   2. the pairs are bucketed by atom (exclusive scan of the counts, then
//      positions inside each bucket from shared-memory counters);
//   3. each bucket is put in ascending k order (ranks by comparison, one warp
//      per bucket), which fixes the order whatever the counters handed out;
//   4. one warp per atom sums x e_i and x^2 over its bucket in that order and
//      writes the range's U_j and r_j as slice b (zeros for atoms the range
//      does not use).
// The slices are then summed in slice order (reduce4_kernel).
constexpr int DET_THREADS = 1024;

int det_range(int p, int n, int s) {  // signals per CTA within 200 KB of shared memory
  const size_t per = sizeof(float) * (size_t)p + (size_t)s * (4 + 4 + 4 + 4);
  const size_t fixed = sizeof(int) * (3 * (size_t)n + 1) + 64;
  const size_t cap = 200u * 1024u;
  return fixed >= cap ? 0 : (int)((cap - fixed) / per);
}
size_t det_smem_bytes(int p, int n, int s, int R) {
  return sizeof(float) * (size_t)R * p + (size_t)R * s * (4 + 4 + 4 + 4) +
         sizeof(int) * (3 * (size_t)n + 1) + 64;
}

template <int RV, int SMAX, bool NS>
__global__ void __launch_bounds__(DET_THREADS, 1) accum_det_kernel(
    const float* __restrict__ Y, int p, int64_t m, int64_t R, const float* __restrict__ D, int n,
    int s, const int32_t* __restrict__ idx, const float* __restrict__ val,
    const int32_t* __restrict__ cnt, float* __restrict__ Upart, size_t len,
    double* __restrict__ epart, int* __restrict__ err, int a0, int a1, int energies,
    const float* __restrict__ D0, const int32_t* __restrict__ pidx, const float* __restrict__ pval,
    const int32_t* __restrict__ pcnt, const int* __restrict__ pvalid, int moved) {
  extern __shared__ float dsh[];
  __shared__ double red[DET_THREADS / 32];
  const int64_t lo = (int64_t)blockIdx.x * R;
  const int64_t hi = lo + R < m ? lo + R : m;
  const int nr = (int)(hi > lo ? hi - lo : 0);  // signals of this range
  const int npair = nr * s;
  float* Es = dsh;                                   // [R][p]
  int* pa = (int*)(Es + (size_t)R * p);              // [R s] atom of pair k (-1: none)
  float* px = (float*)(pa + (size_t)R * s);          // [R s] x of pair k
  int* bk = (int*)(px + (size_t)R * s);              // [R s] bucketed: k
  float* bx = (float*)(bk + (size_t)R * s);          // [R s] bucketed: x
  int* cntA = (int*)(bx + (size_t)R * s);            // [n] pairs per atom
  int* off = cntA + n;                               // [n + 1] bucket starts
  int* fill = off + n + 1;                           // [n]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane & 7, gbase = lane & ~7;
  const int pv = p >> 2;
  for (int a = threadIdx.x; a < n; a += DET_THREADS) {
    cntA[a] = 0;
    fill[a] = 0;
  }
  __syncthreads();
  const float4* __restrict__ Y4 = (const float4*)Y;
  const float4* __restrict__ D4 = (const float4*)(NS ? D0 : D);
  const float4* __restrict__ Dc4 = (const float4*)D;
  const bool have_prev = NS && *pvalid != 0;
  const int32_t* __restrict__ sidx = have_prev ? pidx : idx;
  const float* __restrict__ sval = have_prev ? pval : val;
  const int32_t* __restrict__ scnt = have_prev ? pcnt : cnt;
  float ee = 0.f, yy = 0.f;
  // ---- 1. errors and pairs
  for (int sl = threadIdx.x >> 3; sl < ((nr + 3) & ~3); sl += DET_THREADS / 8) {
    const int64_t i = lo + sl;
    const bool live = sl < nr;
    float4 e[RV];
#pragma unroll
    for (int q = 0; q < RV; ++q) {
      const int v = g + 8 * q;
      e[q] = (live && v < pv) ? Y4[i * pv + v] : make_float4(0.f, 0.f, 0.f, 0.f);
      yy = f4_dot(e[q], e[q], yy);
    }
    const int c = live ? cnt[i] : 0;
    const int j0 = (g < c) ? idx[i * s + g] : 0;
    const float x0 = (g < c) ? val[i * s + g] : 0.f;
    const int j1 = (SMAX > 8 && g + 8 < c) ? idx[i * s + g + 8] : 0;
    const float x1 = (SMAX > 8 && g + 8 < c) ? val[i * s + g + 8] : 0.f;
    const int cmax = __reduce_max_sync(FULL, (unsigned)c);
#pragma unroll
    for (int t = 0; t < SMAX; ++t) {
      if (t >= cmax) break;
      const int jj = __shfl_sync(FULL, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(FULL, t < 8 ? x0 : x1, gbase + (t & 7));
      if (t < c) {
#pragma unroll
        for (int q = 0; q < RV; ++q) {
          const int v = g + 8 * q;
          if (v < pv) e[q] = f4_fma(-xx, __ldg(D4 + (size_t)jj * pv + v), e[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < RV; ++q) ee = f4_dot(e[q], e[q], ee);
    int sc = c, sj0 = j0, sj1 = j1;
    float sx0 = x0, sx1 = x1;
    if (NS) {
      sc = live ? scnt[i] : 0;
      sj0 = (g < sc) ? sidx[i * s + g] : 0;
      sx0 = (g < sc) ? sval[i * s + g] : 0.f;
      sj1 = (SMAX > 8 && g + 8 < sc) ? sidx[i * s + g + 8] : 0;
      sx1 = (SMAX > 8 && g + 8 < sc) ? sval[i * s + g + 8] : 0.f;
      const int scmax = __reduce_max_sync(FULL, (unsigned)sc);
      if (moved) {  // e += (D0 - D) xp for the atoms earlier groups have moved
#pragma unroll
        for (int t = 0; t < SMAX; ++t) {
          if (t >= scmax) break;
          const int jj = __shfl_sync(FULL, t < 8 ? sj0 : sj1, gbase + (t & 7));
          const float xx = __shfl_sync(FULL, t < 8 ? sx0 : sx1, gbase + (t & 7));
          if (t < sc) {
#pragma unroll
            for (int q = 0; q < RV; ++q) {
              const int v = g + 8 * q;
              if (v < pv) {
                e[q] = f4_fma(xx, __ldg(D4 + (size_t)jj * pv + v), e[q]);
                e[q] = f4_fma(-xx, __ldg(Dc4 + (size_t)jj * pv + v), e[q]);
              }
            }
          }
        }
      }
    }
    if (live) {
#pragma unroll
      for (int q = 0; q < RV; ++q) {
        const int v = g + 8 * q;
        if (v < pv) *(float4*)(Es + (size_t)sl * p + 4 * v) = e[q];
      }
      if (g < s) {
        const bool ok = g < sc && sj0 >= a0 && sj0 < a1;
        pa[sl * s + g] = ok ? sj0 : -1;
        px[sl * s + g] = sx0;
        if (ok) atomicAdd(&cntA[sj0], 1);
      }
      if (SMAX > 8 && g + 8 < s) {
        const bool ok = g + 8 < sc && sj1 >= a0 && sj1 < a1;
        pa[sl * s + g + 8] = ok ? sj1 : -1;
        px[sl * s + g + 8] = sx1;
        if (ok) atomicAdd(&cntA[sj1], 1);
      }
    }
  }
  if (!isfinite(ee) || !isfinite(yy)) atomicOr(err, ERR_NONFINITE);
  __syncthreads();
  // ---- 2. buckets: exclusive scan of the counts (n <= 1024), then positions
  {
    const int a = threadIdx.x;
    const int v = a < n ? cntA[a] : 0;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    __shared__ int wsum[32];
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      int x = wsum[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += t;
      }
      wsum[lane] = x;
    }
    __syncthreads();
    const int ex = (warp > 0 ? wsum[warp - 1] : 0) + inc - v;
    if (a < n) off[a] = ex;
    if (a == n - 1) off[n] = ex + v;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < npair; k += DET_THREADS) {
    const int a = pa[k];
    if (a >= 0) {
      const int pos = off[a] + atomicAdd(&fill[a], 1);
      bk[pos] = k;
      bx[pos] = px[k];
    }
  }
  __syncthreads();
  // ---- 3. and 4. one warp per atom: order the bucket by k, then sum over it
  float* out = Upart + (size_t)blockIdx.x * len;
  const size_t np = (size_t)n * p;
  for (int a = warp; a < n; a += DET_THREADS / 32) {
    const int b0 = off[a], L = off[a + 1] - b0;
    for (int q0 = 0; q0 < L; q0 += 32) {  // rank of each pair by k among the bucket's pairs
      const int q = q0 + lane;
      const int kq = q < L ? bk[b0 + q] : 0x7fffffff;
      const float xq = q < L ? bx[b0 + q] : 0.f;
      int rank = 0;
      for (int r0 = 0; r0 < L; r0 += 32) {
        const int kr = r0 + lane < L ? bk[b0 + r0 + lane] : 0x7fffffff;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) rank += __shfl_sync(FULL, kr, j) < kq ? 1 : 0;
      }
      __syncwarp();
      if (q < L) {  // park at the final position in the pair arrays (free after step 2)
        pa[b0 + rank] = kq;
        px[b0 + rank] = xq;
      }
      __syncwarp();
    }
    __syncwarp();
    constexpr int RU = RV;  // rows lane + 32 u of U_j, u < ceil(p / 32) <= RV
    float ac[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) ac[u] = 0.f;
    float rx = 0.f;
    for (int q = 0; q < L; ++q) {
      const int k = pa[b0 + q];
      const float xx = px[b0 + q];
      const float* er = Es + (size_t)(k / s) * p;
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const int r = lane + 32 * u;
        if (r < p) ac[u] = fmaf(xx, er[r], ac[u]);
      }
      rx = fmaf(xx, xx, rx);
    }
#pragma unroll
    for (int u = 0; u < RU; ++u) {
      const int r = lane + 32 * u;
      if (r < p) out[(size_t)a * p + r] = ac[u];
    }
    if (lane == 0) out[np + a] = rx;
  }
  for (size_t q = np + n + threadIdx.x; q < len; q += DET_THREADS) out[q] = 0.f;
  const double see = block_sum_f(ee, red);
  const double syy = block_sum_f(yy, red);
  if (threadIdx.x == 0 && energies) {
    epart[2 * blockIdx.x] = see;
    epart[2 * blockIdx.x + 1] = syy;
  }
}

// Pass B, float4 form: e = y - D x; x_t' = e.d'_{j_t} + c_{j_t} x_t for all t
// (independent dot products), then y - D' x'.  GROUP: only slots whose atom is
// in [a0, a1) are updated; the others keep x_t and their current atom in the
// residual.  sgk: the coefficients stay (x' = x; SGK rule, Eq. 6).
template <int RV, int SMAX, bool GROUP>
__global__ void __launch_bounds__(ROW_THREADS, 4) rows4_kernel(
    const float* __restrict__ Y, int p, int64_t m, const float* __restrict__ D,
    const float* __restrict__ Dn, const float* __restrict__ C, int s,
    const int32_t* __restrict__ idx, float* __restrict__ val, const int32_t* __restrict__ cnt,
    const int64_t* __restrict__ colptr, int32_t* __restrict__ csc_rowidx,
    float* __restrict__ csc_val, double* __restrict__ epart, int a0, int a1, int sgk) {
  __shared__ double red[ROW_THREADS / 32];
  const int lane = threadIdx.x & 31;
  const int g = lane & 7, gbase = lane & ~7;
  const int pv = p >> 2;
  const float4* __restrict__ Y4 = (const float4*)Y;
  const float4* __restrict__ D4 = (const float4*)D;
  const float4* __restrict__ N4 = (const float4*)Dn;
  (void)a0;
  (void)a1;
  float e2 = 0.f;
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x >> 3);
  const int64_t g0 = (int64_t)blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 3);
  const int64_t trips = (m + groups - 1) / groups;
  for (int64_t k = 0; k < trips; ++k) {
    const int64_t i = g0 + k * groups;
    const bool live = i < m;
    {  // warm L2 with the next trip's signal: its samples, slots, count and column start
      const int64_t inx = i + groups;
      if (inx < m) {
        const char* a = nullptr;
        if (g < 2 * RV && 128 * g < 4 * p) a = (const char*)(Y + inx * p) + 128 * g;
        else if (g == 6) a = (const char*)(idx + inx * s);
        else if (g == 7) a = (const char*)(val + inx * s);
        if (a) asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
      }
    }
    float4 y[RV], e[RV];
#pragma unroll
    for (int q = 0; q < RV; ++q) {
      const int v = g + 8 * q;
      y[q] = (live && v < pv) ? Y4[i * pv + v] : make_float4(0.f, 0.f, 0.f, 0.f);
      e[q] = y[q];
    }
    const int c = live ? cnt[i] : 0;
    const int j0 = (g < c) ? idx[i * s + g] : 0;
    const float x0 = (g < c) ? val[i * s + g] : 0.f;
    const int j1 = (SMAX > 8 && g + 8 < c) ? idx[i * s + g + 8] : 0;
    const float x1 = (SMAX > 8 && g + 8 < c) ? val[i * s + g + 8] : 0.f;
    const int cmax = __reduce_max_sync(FULL, (unsigned)c);
#pragma unroll
    for (int t = 0; t < SMAX; ++t) {
      if (t >= cmax) break;
      const int jj = __shfl_sync(FULL, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(FULL, t < 8 ? x0 : x1, gbase + (t & 7));
      if (t < c) {
        const bool other = GROUP && (jj < a0 || jj >= a1);  // stays: also in the final residual
#pragma unroll
        for (int q = 0; q < RV; ++q) {
          const int v = g + 8 * q;
          if (v < pv) {
            const float4 d = __ldg(D4 + (size_t)jj * pv + v);
            e[q] = f4_fma(-xx, d, e[q]);
            if (other) y[q] = f4_fma(-xx, d, y[q]);
          }
        }
      }
    }
    float xn[SMAX];
#pragma unroll
    for (int t = 0; t < SMAX; ++t) {
      xn[t] = 0.f;
      if (t >= cmax) break;
      const int jj = __shfl_sync(FULL, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(FULL, t < 8 ? x0 : x1, gbase + (t & 7));
      const bool upd = t < c && (!GROUP || (jj >= a0 && jj < a1));
      float dot = 0.f;
      float4 dn[RV];
#pragma unroll
      for (int q = 0; q < RV; ++q) {
        const int v = g + 8 * q;
        dn[q] = (upd && v < pv) ? __ldg(N4 + (size_t)jj * pv + v) : make_float4(0.f, 0.f, 0.f, 0.f);
        dot = f4_dot(e[q], dn[q], dot);
      }
      dot += __shfl_xor_sync(FULL, dot, 4);
      dot += __shfl_xor_sync(FULL, dot, 2);
      dot += __shfl_xor_sync(FULL, dot, 1);
      xn[t] = upd && !sgk ? fmaf(__ldg(C + jj), xx, dot) : (t < c ? xx : 0.f);
      // residual with the updated atoms, y - D' x', from the same rows of D'
#pragma unroll
      for (int q = 0; q < RV; ++q) y[q] = f4_fma(upd ? -xn[t] : 0.f, dn[q], y[q]);
    }
#pragma unroll
    for (int q = 0; q < RV; ++q) e2 = f4_dot(y[q], y[q], e2);
    // lane g writes slots g and g + 8
    float nx0 = 0.f, nx1 = 0.f;
#pragma unroll
    for (int t = 0; t < SMAX; ++t) {
      if (t == g) nx0 = xn[t];
      if (t == g + 8) nx1 = xn[t];
    }
    if (g < c) {
      val[i * s + g] = nx0;
      if (csc_val) {
        const int64_t o = colptr[i] + g;
        if (csc_rowidx) csc_rowidx[o] = j0;
        csc_val[o] = nx0;
      }
    }
    if (SMAX > 8 && g + 8 < c) {
      val[i * s + g + 8] = nx1;
      if (csc_val) {
        const int64_t o = colptr[i] + g + 8;
        if (csc_rowidx) csc_rowidx[o] = j1;
        csc_val[o] = nx1;
      }
    }
  }
  const double se = block_sum_f(e2, red);
  if (threadIdx.x == 0) epart[blockIdx.x] = se;
}

// U = sum of the partial slices, float4 columns (len % 4 == 0): 8 slice
// groups per column in a CTA of 256 threads, then the 8 group sums in order
// (deterministic).
__global__ void __launch_bounds__(256) reduce4_kernel(const float4* __restrict__ Upart, int nslices,
                                                      int len4, float4* __restrict__ U) {
  __shared__ float4 part[8][32];
  const int tx = threadIdx.x & 31, gs = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + tx;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c < len4) {
#pragma unroll 4
    for (int b = gs; b < nslices; b += 8) {
      const float4 v = Upart[(size_t)b * len4 + c];
      acc.x += v.x;
      acc.y += v.y;
      acc.z += v.z;
      acc.w += v.w;
    }
  }
  part[gs][tx] = acc;
  __syncthreads();
  if (gs == 0 && c < len4) {
    float4 t = part[0][tx];
#pragma unroll
    for (int q = 1; q < 8; ++q) {
      t.x += part[q][tx].x;
      t.y += part[q][tx].y;
      t.z += part[q][tx].z;
      t.w += part[q][tx].w;
    }
    U[c] = t;
  }
}

// U[q] = sum over partial slices in slice order (deterministic).
__global__ void reduce_kernel(const float* __restrict__ Upart, int nslices, int len,
                              float* __restrict__ U) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= len) return;
  float acc = 0.f;
  for (int b = 0; b < nslices; ++b) acc += Upart[(size_t)b * len + q];
  U[q] = acc;
}

// One warp per atom: v = U_j + r_j d_j; d' = v/||v|| (d kept if v = 0); c = d^T d'.
template <int PL>
// Atoms a0 <= j < a1.
__global__ void atoms_kernel(const float* __restrict__ D, int p, int n, const float* __restrict__ U,
                             float* __restrict__ Dn, float* __restrict__ C, int a0, int a1) {
  const int lane = threadIdx.x & 31;
  const int j = a0 + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (j >= a1) return;
  const float rj = U[(size_t)n * p + j];
  float d[PL], v[PL];
  float vv = 0.f;
#pragma unroll
  for (int u = 0; u < PL; ++u) {
    const int r = lane + 32 * u;
    d[u] = (r < p) ? D[(size_t)j * p + r] : 0.f;
    v[u] = (r < p) ? fmaf(rj, d[u], U[(size_t)j * p + r]) : 0.f;
    vv = fmaf(v[u], v[u], vv);
  }
  vv = warp_sum(vv);
  if (vv > 0.f) {
    const float inv = 1.0f / sqrtf(vv);
    float c = 0.f;
#pragma unroll
    for (int u = 0; u < PL; ++u) {
      const int r = lane + 32 * u;
      v[u] *= inv;
      c = fmaf(d[u], v[u], c);
      if (r < p) Dn[(size_t)j * p + r] = v[u];
    }
    c = warp_sum(c);
    if (lane == 0) C[j] = c;
  } else {
#pragma unroll
    for (int u = 0; u < PL; ++u) {
      const int r = lane + 32 * u;
      if (r < p) Dn[(size_t)j * p + r] = d[u];
    }
    if (lane == 0) C[j] = 1.f;
  }
}

// The same for float4 rows, from the kUCopies copies of U and r that pass A added
// to: one CTA per atom sums its rows of the copies in a fixed order and forms the
// atom (a reduction and an atom kernel took 2.4 + 1.8 us; 2.5 us).  Clearing the
// copies here as well cost 25 us: their lines have just been read from both dies.
__global__ void __launch_bounds__(256) atoms4_kernel(const float* __restrict__ D, int p, int n,
                                                     const float* __restrict__ Uc,
                                                     float* __restrict__ Dn, float* __restrict__ C, int a0) {
  __shared__ float4 part[8][32];
  __shared__ float rpart[8];
  static_assert(kUCopies == 16, "two copies per warp");
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j = a0 + blockIdx.x, pv = p >> 2;
  const size_t len = jau_ulen(p, n);
  const float* u0 = Uc + (size_t)w * len;
  const float* u1 = Uc + (size_t)(w + 8) * len;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  if (lane < pv) {
    const float4 a = __ldg((const float4*)(u0 + (size_t)j * p) + lane);
    const float4 b = __ldg((const float4*)(u1 + (size_t)j * p) + lane);
    part[w][lane] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
  }
  if (lane == 0) rpart[w] = __ldg(u0 + (size_t)n * p + j) + __ldg(u1 + (size_t)n * p + j);
  const float4 d = w == 0 && lane < pv ? __ldg((const float4*)(D + (size_t)j * p) + lane) : zero;
  __syncthreads();
  if (w > 0) return;
  float4 v = zero;
  float rj = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if (lane < pv) {
      const float4 x = part[q][lane];
      v = make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
    }
    rj += rpart[q];
  }
  v = make_float4(fmaf(rj, d.x, v.x), fmaf(rj, d.y, v.y), fmaf(rj, d.z, v.z), fmaf(rj, d.w, v.w));
  const float vv = warp_sum(f4_dot(v, v, 0.f));
  float c = 1.f;
  if (vv > 0.f) {
    const float inv = 1.0f / sqrtf(vv);
    v = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
    c = warp_sum(f4_dot(d, v, 0.f));
  } else {
    v = d;  // unused atom (or F x^T = 0): kept
  }
  if (lane < pv) *((float4*)(Dn + (size_t)j * p) + lane) = v;
  if (lane == 0) C[j] = c;
}

// Pass B: per signal, e = y - D x (old atoms), x_t' = e.d'_{j_t} + c_{j_t} x_t,
// then ||y - D' x'||^2.  Writes the slots and, optionally, the CSC arrays.
// Eight lanes per signal (four signals per warp), as in pass A.
template <int RL>
__global__ void __launch_bounds__(ROW_THREADS) rows_kernel(
    const float* __restrict__ Y, int p, int64_t m, const float* __restrict__ D,
    const float* __restrict__ Dn, const float* __restrict__ C, int s,
    const int32_t* __restrict__ idx, float* __restrict__ val, const int32_t* __restrict__ cnt,
    const int64_t* __restrict__ colptr, int32_t* __restrict__ csc_rowidx,
    float* __restrict__ csc_val, double* __restrict__ epart, int sgk) {
  __shared__ double red[ROW_THREADS / 32];
  const int lane = threadIdx.x & 31;
  const int g = lane & 7, gbase = lane & ~7;
  float e2 = 0.f;
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x >> 3);
  const int64_t g0 = (int64_t)blockIdx.x * (blockDim.x >> 3) + (threadIdx.x >> 3);
  const int64_t trips = (m + groups - 1) / groups;
  for (int64_t k = 0; k < trips; ++k) {
    const int64_t i = g0 + k * groups;
    const bool live = i < m;
    float y[RL], e[RL];
#pragma unroll
    for (int u = 0; u < RL; ++u) {
      const int r = g + 8 * u;
      y[u] = (live && r < p) ? Y[i * p + r] : 0.f;
      e[u] = y[u];
    }
    const int c = live ? cnt[i] : 0;
    const int j0 = (g < c) ? idx[i * s + g] : 0;
    const float x0 = (g < c) ? val[i * s + g] : 0.f;
    const int j1 = (g + 8 < c) ? idx[i * s + g + 8] : 0;
    const float x1 = (g + 8 < c) ? val[i * s + g + 8] : 0.f;
    const int cmax = __reduce_max_sync(0xffffffffu, (unsigned)c);
    for (int t = 0; t < cmax; ++t) {
      const int jj = __shfl_sync(0xffffffffu, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(0xffffffffu, t < 8 ? x0 : x1, gbase + (t & 7));
      if (t < c) {
#pragma unroll
        for (int u = 0; u < RL; ++u) {
          const int r = g + 8 * u;
          if (r < p) e[u] = fmaf(-xx, __ldg(D + (size_t)jj * p + r), e[u]);
        }
      }
    }
    float nx0 = 0.f, nx1 = 0.f;  // x_t' for the slots held by this lane
    for (int t = 0; t < cmax; ++t) {
      const int jj = __shfl_sync(0xffffffffu, t < 8 ? j0 : j1, gbase + (t & 7));
      const float xx = __shfl_sync(0xffffffffu, t < 8 ? x0 : x1, gbase + (t & 7));
      float dot = 0.f;
      if (t < c) {
#pragma unroll
        for (int u = 0; u < RL; ++u) {
          const int r = g + 8 * u;
          if (r < p) dot = fmaf(e[u], __ldg(Dn + (size_t)jj * p + r), dot);
        }
      }
      dot += __shfl_xor_sync(0xffffffffu, dot, 4);
      dot += __shfl_xor_sync(0xffffffffu, dot, 2);
      dot += __shfl_xor_sync(0xffffffffu, dot, 1);
      if (t < c) {
        const float xn = sgk ? xx : fmaf(__ldg(C + jj), xx, dot);
        if (g == (t & 7)) {
          if (t < 8) nx0 = xn;
          else nx1 = xn;
        }
        // residual with the updated atoms: y - D' x'
#pragma unroll
        for (int u = 0; u < RL; ++u) {
          const int r = g + 8 * u;
          if (r < p) y[u] = fmaf(-xn, __ldg(Dn + (size_t)jj * p + r), y[u]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < RL; ++u) e2 = fmaf(y[u], y[u], e2);
    if (g < c) {
      val[i * s + g] = nx0;
      if (csc_val) {
        const int64_t o = colptr[i] + g;
        if (csc_rowidx) csc_rowidx[o] = j0;
        csc_val[o] = nx0;
      }
    }
    if (g + 8 < c) {
      val[i * s + g + 8] = nx1;
      if (csc_val) {
        const int64_t o = colptr[i] + g + 8;
        if (csc_rowidx) csc_rowidx[o] = j1;
        csc_val[o] = nx1;
      }
    }
  }
  const double se = block_sum_f(e2, red);
  if (threadIdx.x == 0) epart[blockIdx.x] = se;
}

// Block 0: the RMSE before and after the update from the partial sums (a fixed
// order); the other blocks copy the updated atoms Dn into D.  One CTA's FP64
// instructions are the whole cost (1/64 of the FP32 rate): four warps, the three
// sums side by side, and the two quotients and square roots in two lanes at once
// (7.4 us with 256 threads, three block sums after one another and one thread at the
// end, 7.9 with 1024 threads; 4.6 to 5.8 us).
constexpr int FIN_THREADS = 128;
__global__ void __launch_bounds__(FIN_THREADS) finalize_kernel(
    const double* __restrict__ epa, int na, const double* __restrict__ epb, int nb,
    double* __restrict__ rmse, int* __restrict__ iter, const float* __restrict__ Dn,
    float* __restrict__ D, int64_t np, int p, int pitch) {
  __shared__ double red[FIN_THREADS / 32][3];
  if (blockIdx.x > 0) {
    const int64_t stride = (int64_t)(gridDim.x - 1) * blockDim.x;
    for (int64_t q = (int64_t)(blockIdx.x - 1) * blockDim.x + threadIdx.x; q < np; q += stride)
      D[q] = Dn[p == pitch ? q : q / p * pitch + q % p];
    return;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double ee = 0.0, yy = 0.0, e2 = 0.0;
  for (int b = threadIdx.x; b < na; b += FIN_THREADS) {
    const double2 v = *(const double2*)(epa + 2 * b);
    ee += v.x;
    yy += v.y;
  }
  for (int b = threadIdx.x; b < nb; b += FIN_THREADS) e2 += epb[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ee += __shfl_xor_sync(FULL, ee, o);
    yy += __shfl_xor_sync(FULL, yy, o);
    e2 += __shfl_xor_sync(FULL, e2, o);
  }
  if (lane == 0) {
    red[w][0] = ee;
    red[w][1] = yy;
    red[w][2] = e2;
  }
  __syncthreads();
  if (w > 0) return;
  ee = yy = e2 = 0.0;
#pragma unroll
  for (int q = 0; q < FIN_THREADS / 32; ++q) {
    ee += red[q][0];
    yy += red[q][1];
    e2 += red[q][2];
  }
  // (one lane reads and advances the counter: the other lanes never see it move)
  const int it = __shfl_sync(FULL, lane == 0 ? *iter : 0, 0);
  if (lane < 2) {
    const double num = lane == 0 ? ee : e2;
    rmse[2 * it + lane] = yy > 0.0 ? sqrt(num / yy) : 0.0;
  }
  if (lane == 0) *iter = it + 1;
}

// ---- CSC helpers ------------------------------------------------------------------
// The slots as CSC: colptr is the exclusive scan of the counts.  CTA b owns `rounds`
// x 256 signals; the first kernel sums the counts of each CTA's signals, the second
// adds up the sums before its own, scans its counts and writes colptr and the
// column entries of its signals.  (A scan over 4096 signals per CTA with FP64
// block sums, a serial sum over the earlier CTAs and a separate entry kernel took
// 4.5 + 4.5 + 2.7 us at m = 60,000, s = 4; 1.9 + 4.3 us.)
constexpr int CSC_THREADS = 256;
int csc_rounds(int64_t m) {
  const int64_t most = (int64_t)CSC_THREADS * kCscBlocks;
  return (int)((m + most - 1) / most);
}

__global__ void __launch_bounds__(CSC_THREADS) count_sum_kernel(const int32_t* __restrict__ cnt, int64_t m,
                                                                int rounds, int64_t* __restrict__ bsum) {
  __shared__ long long wsum[CSC_THREADS / 32];
  const int64_t base = (int64_t)blockIdx.x * rounds * CSC_THREADS + threadIdx.x;
  long long s = 0;
  for (int u = 0; u < rounds; ++u) {
    const int64_t i = base + (int64_t)u * CSC_THREADS;
    s += __reduce_add_sync(FULL, i < m ? cnt[i] : 0);
  }
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    s = 0;
#pragma unroll
    for (int w = 0; w < CSC_THREADS / 32; ++w) s += wsum[w];
    bsum[blockIdx.x] = s;
  }
}

// rowidx and cval: null to leave them.
__global__ void __launch_bounds__(CSC_THREADS) csc_write_kernel(
    const int32_t* __restrict__ cnt, const int32_t* __restrict__ idx, const float* __restrict__ val,
    int64_t m, int s, int rounds, const int64_t* __restrict__ bsum, int64_t* __restrict__ colptr,
    int32_t* __restrict__ rowidx, float* __restrict__ cval) {
  __shared__ long long psum[CSC_THREADS / 32];
  __shared__ int wsum[CSC_THREADS / 32];
  __shared__ int off[CSC_THREADS + 1];  // starts relative to the round's first entry
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t i0 = (int64_t)blockIdx.x * rounds * CSC_THREADS;
  int c = i0 + threadIdx.x < m ? cnt[i0 + threadIdx.x] : 0;
  long long before = 0;
  for (int b = threadIdx.x; b < (int)blockIdx.x; b += CSC_THREADS) before += bsum[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(FULL, before, o);
  if (lane == 0) psum[w] = before;
  __syncthreads();
  before = 0;
#pragma unroll
  for (int q = 0; q < CSC_THREADS / 32; ++q) before += psum[q];
  for (int u = 0; u < rounds && i0 < m; ++u, i0 += CSC_THREADS) {
    const int nr = (int)(m - i0 < CSC_THREADS ? m - i0 : CSC_THREADS);
    int inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    int ex = inc - c, all = 0;
#pragma unroll
    for (int q = 0; q < CSC_THREADS / 32; ++q) {
      if (q < w) ex += wsum[q];
      all += wsum[q];
    }
    off[threadIdx.x] = ex;
    if (threadIdx.x == 0) off[CSC_THREADS] = all;
    if ((int)threadIdx.x < nr) colptr[i0 + threadIdx.x] = before + ex;
    if (i0 + nr == m && threadIdx.x == 0) colptr[m] = before + all;
    __syncthreads();
    if (rowidx) {
#pragma unroll 4
      for (int k = threadIdx.x; k < nr * s; k += CSC_THREADS) {
        const int j = idx[i0 * s + k];
        const int q = k / s, t = k - q * s, o = off[q];
        if (t < off[q + 1] - o) {
          rowidx[before + o + t] = j;
          if (cval) cval[before + o + t] = val[i0 * s + k];
        }
      }
    }
    before += all;
    const int64_t in = i0 + CSC_THREADS + threadIdx.x;
    c = u + 1 < rounds && in < m ? cnt[in] : 0;
    __syncthreads();
  }
}

// The caller's CSC columns into slots; a column with too many entries, out of order
// or out of range is flagged and left empty.  W lanes (a power of two >= s) per
// column: the entries are read as they lie (one thread per column, a chain of s
// dependent comparisons, took 10.6 us at m = 1e5, s = 8; 5.1 us).
template <int W>
__global__ void __launch_bounds__(256) csc_to_slots_kernel(
    const int64_t* __restrict__ colptr, const int32_t* __restrict__ rowidx, const float* __restrict__ cval,
    int64_t m, int n, int s, int32_t* __restrict__ idx, float* __restrict__ val, int32_t* __restrict__ cnt,
    int* __restrict__ err) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t i = g / W;
  const int t = (int)(g & (W - 1)), lane = threadIdx.x & 31;
  const bool live = i < m;
  const int64_t a = live ? colptr[i] : 0, b = live ? colptr[i + 1] : 0;
  const bool span = b >= a && b - a <= s && a >= 0 && b <= m * (int64_t)s;
  const int c = span ? (int)(b - a) : 0;
  const int j = t < c ? rowidx[a + t] : -1;
  const float x = t < c ? cval[a + t] : 0.f;
  const int left = __shfl_up_sync(FULL, j, 1, W);
  const bool bad = !span || (t < c && (j < 0 || j >= n || (t > 0 && j <= left)));
  const unsigned ball = __ballot_sync(FULL, bad);
  const unsigned mine = (W == 32 ? ~0u : ((1u << W) - 1u) << (lane & ~(W - 1)));
  const bool ok = (ball & mine) == 0u;
  if (!live) return;
  if (t < s) {
    idx[i * s + t] = ok ? j : -1;
    val[i * s + t] = ok ? x : 0.f;
  }
  if (t == 0) {
    cnt[i] = ok ? c : 0;
    if (!ok) atomicOr(err, ERR_CSC);
  }
}

cudaError_t reduce_slices(float* Upart, int nslices, int len, float* U, cudaStream_t st) {
  if (len % 4 == 0)
    reduce4_kernel<<<(len / 4 + 31) / 32, 256, 0, st>>>((const float4*)Upart, nslices, len / 4,
                                                         (float4*)U);
  else
    reduce_kernel<<<(len + 255) / 256, 256, 0, st>>>(Upart, nslices, len, U);
  return cudaGetLastError();
}

template <int PL>
cudaError_t accum_t(const float* Y, int p, int64_t m, const float* D, int n, int s,
                    const int32_t* idx, const float* val, const int32_t* cnt, const JauWork& w,
                    int* err, cudaStream_t st) {
  const size_t smem = jau_accum_smem(p, n);
  if (smem > 0) {
    cudaFuncSetAttribute(accum_kernel<PL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    accum_kernel<PL, true><<<w.nb_accum, ACC_THREADS, smem, st>>>(Y, p, m, D, n, s, idx, val, cnt,
                                                                  w.Upart, w.epart_a, err);
  } else {
    cudaMemsetAsync(w.Upart, 0, sizeof(float) * ((size_t)n * p + n), st);
    accum_kernel<PL, false><<<w.nb_accum, ACC_THREADS, 0, st>>>(Y, p, m, D, n, s, idx, val, cnt,
                                                                w.Upart, w.epart_a, err);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return reduce_slices(w.Upart, smem > 0 ? w.nb_accum : 1, n * p + n, w.U, st);
}

}  // namespace

int num_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return sms;
}

size_t jau_accum_smem(int p, int n) {
  const size_t bytes = sizeof(float) * ((size_t)n * p + n);
  return bytes <= 200u * 1024u ? bytes : 0;
}
int jau_accum_blocks(int p, int n, int mult) {
  // float4 form: 4 (8) CTAs of 256 threads per SM
  if (p % 4 == 0) return (mult >= 2 ? 8 : 4) * num_sms();
  // the shared-memory form runs 1 CTA per SM unless two partial slices fit on one SM
  if (jau_accum_smem(p, n) > 0)
    return (mult >= 2 && jau_accum_smem(p, n) <= 100u * 1024u) ? 2 * num_sms() : num_sms();
  return (mult >= 2 ? 8 : 4) * num_sms();
}
int jau_accum_blocks_max(int p, int n) {
  return (p % 4 != 0 && jau_accum_smem(p, n) > 0) ? 2 * num_sms() : 8 * num_sms();
}
size_t jau_slices(int64_t m, int p, int n, int s) {
  if (p % 4 != 0) return jau_accum_smem(p, n) > 0 ? 2 * (size_t)num_sms() : 1;
  return jau_det_supported(p, n, s, nullptr, nullptr) ? (size_t)jau_det_ranges(m, p, n, s) : 1;
}
bool jau_vec4(int p, const float* Y, const float* D) {
  return p % 4 == 0 && ((uintptr_t)Y % 16) == 0 && ((uintptr_t)D % 16) == 0;
}
int jau_launches(const JauWork& w) {
  // errors and sums, or one accumulation pass; atoms (after a reduction of the
  // slices where there are no copies); rows; finalize
  return (w.E ? 2 : 1) + (w.padded ? 1 : 0) + (w.copies ? 1 : 2) + 2;
}
int jau_row_blocks(int per_sm) { return (per_sm == 2 || per_sm == 8 ? per_sm : 4) * num_sms(); }
int jau_row_blocks_max() { return 8 * num_sms(); }

// From one signal per resident eight lanes of the errors pass on: with fewer, all
// passes are bound by launches, and accum4_kernel has one launch less (one
// iteration at p = 16, n = 32, s = 3, m = 1000: 97.4 us against 99.2; p = 64,
// n = 256, s = 6, m = 20,000: 77.5 against 75.8).
bool jau_plain_supported(int64_t m, int p, int n, int s) {
  return m >= jau_plain_min() && p <= 128 && n <= 1024 && s <= 16 && sum_tile(m, jau_p4(p), n, s) > 0;
}
int jau_plain_min() { return 32 * num_sms(); }
// one full round of resident CTAs each (see the kernels' launch bounds)
int jau_plain_blocks(int p) { return (p <= 64 ? 4 : 3) * num_sms(); }
int jau_plain_row_blocks(int p) { return (p <= 32 ? 4 : p <= 64 ? 3 : 2) * num_sms(); }

bool jau_det_supported(int p, int n, int s, const float* Y, const float* D) {
  return (Y || D ? jau_vec4(p, Y, D) : p % 4 == 0) && p <= 128 && n <= 1024 && s <= 16 &&
         det_range(p, n, s) >= 64;
}
// CTAs of the deterministic pass A for m signals: at least one per SM, each range
// within the shared-memory budget
int64_t jau_det_ranges(int64_t m, int p, int n, int s) {
  const int64_t R = det_range(p, n, s);
  int64_t nb = R > 0 ? (m + R - 1) / R : 1;
  const int64_t floor_nb = 2 * (int64_t)num_sms();
  if (nb < floor_nb) nb = floor_nb;
  return nb;
}

cudaError_t jau_accumulate_det(const float* Y, int p, int64_t m, const float* D, int n, int s,
                               const int32_t* idx, const float* val, const int32_t* cnt,
                               const JauWork& w, int* err, cudaStream_t st) {
  const int nb = w.nb_accum;
  const int64_t R = (m + nb - 1) / nb;
  const size_t len = jau_ulen(p, n);
  const size_t smem = det_smem_bytes(p, n, s, (int)R);
  const int a0 = w.a0, a1 = w.a1 > 0 ? w.a1 : n;
  cudaError_t e = cudaSuccess;
#define DL_ACCD(RV, SM)                                                                        \
  do {                                                                                         \
    if (w.nsgk) {                                                                              \
      e = cudaFuncSetAttribute(accum_det_kernel<RV, SM, true>,                                 \
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);        \
      if (e == cudaSuccess)                                                                    \
        accum_det_kernel<RV, SM, true><<<nb, DET_THREADS, smem, st>>>(                         \
            Y, p, m, R, D, n, s, idx, val, cnt, w.Upart, len, w.epart_a, err, a0, a1,          \
            (int)w.energies, w.D0, w.pidx, w.pval, w.pcnt, w.pvalid, w.a0 > 0 ? 1 : 0);        \
    } else {                                                                                   \
      e = cudaFuncSetAttribute(accum_det_kernel<RV, SM, false>,                                \
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);        \
      if (e == cudaSuccess)                                                                    \
        accum_det_kernel<RV, SM, false><<<nb, DET_THREADS, smem, st>>>(                        \
            Y, p, m, R, D, n, s, idx, val, cnt, w.Upart, len, w.epart_a, err, a0, a1,          \
            (int)w.energies, D, idx, val, cnt, nullptr, 0);                                    \
    }                                                                                          \
  } while (0)
#define DL_ACCD_S(RV) \
  if (s <= 8) DL_ACCD(RV, 8); else DL_ACCD(RV, 16)
  if (p <= 32) { DL_ACCD_S(1); }
  else if (p <= 64) { DL_ACCD_S(2); }
  else if (p <= 96) { DL_ACCD_S(3); }
  else { DL_ACCD_S(4); }
#undef DL_ACCD_S
#undef DL_ACCD
  if (e != cudaSuccess) return e;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return reduce_slices(w.Upart, nb, (int)len, w.U, st);
}

cudaError_t jau_accumulate(const float* Y, int p, int64_t m, const float* D, int n, int s,
                           const int32_t* idx, const float* val, const int32_t* cnt,
                           const JauWork& w, int* err, cudaStream_t st) {
  if (w.det && jau_det_supported(p, n, s, Y, D))
    return jau_accumulate_det(Y, p, m, D, n, s, idx, val, cnt, w, err, st);
  if (w.E) {  // the plain case
    const int p4 = jau_p4(p);
    const size_t len = jau_ulen(p4, n);
    const bool vec = jau_vec4(p, Y, D);
    cudaError_t e;
    if (!vec) {
      pad_atoms_kernel<<<(n * p4 + 255) / 256, 256, 0, st>>>(D, p, n, p4, w.Dp);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
#define DL_ERRS(RV)                                                                                  \
  do {                                                                                               \
    auto kern = !vec ? errors_kernel<RV, false, false>                                               \
                     : p == 32 * RV ? errors_kernel<RV, true, true> : errors_kernel<RV, false, true>; \
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,                       \
                         cudaSharedmemCarveoutMaxL1);                                                \
    kern<<<w.nb_accum, EP_THREADS, 0, st>>>(Y, p, p4, m, vec ? D : w.Dp, s, idx, val, cnt, w.E,      \
                                            w.epart_a, err, (float4*)w.Ucopy,                        \
                                            (int)(len * kUCopies / 4));                              \
  } while (0)
    if (p <= 32) DL_ERRS(1);
    else if (p <= 64) DL_ERRS(2);
    else if (p <= 96) DL_ERRS(3);
    else DL_ERRS(4);
#undef DL_ERRS
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int T = sum_tile(m, p4, n, s);
    const size_t smem = (size_t)SumSmem(p4, n, s, T).total;
    if ((e = cudaFuncSetAttribute(sums_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
        cudaSuccess)
      return e;
    const int64_t nt = (m + T - 1) / T;
    sums_kernel<<<(unsigned)(nt < 2 * num_sms() ? nt : 2 * num_sms()), SUM_THREADS, smem, st>>>(
        w.E, p4, m, T, n, s, idx, val, w.Ucopy, err);
    return cudaGetLastError();
  }
  if (jau_vec4(p, Y, D)) {
    const size_t len = jau_ulen(p, n);
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.Ucopy, 0, sizeof(float) * len * kUCopies, st)) != cudaSuccess) return e;
#define DL_ACC4(RV, SM)                                                                  \
  do {                                                                                       \
    if (w.nsgk)                                                                              \
      accum4_kernel<RV, SM, true><<<w.nb_accum, ACC4_THREADS, 0, st>>>(                     \
          Y, p, m, D, n, s, idx, val, cnt, w.Ucopy, w.epart_a, err, w.a0, w.a1 > 0 ? w.a1 : n, \
          (int)w.energies, w.D0, w.pidx, w.pval, w.pcnt, w.pvalid, w.a0 > 0 ? 1 : 0);         \
    else                                                                                     \
      accum4_kernel<RV, SM, false><<<w.nb_accum, ACC4_THREADS, 0, st>>>(                    \
          Y, p, m, D, n, s, idx, val, cnt, w.Ucopy, w.epart_a, err, w.a0, w.a1 > 0 ? w.a1 : n, \
          (int)w.energies, D, idx, val, cnt, nullptr, 0);                                     \
  } while (0)
#define DL_ACC4_S(RV) \
  if (s <= 8) DL_ACC4(RV, 8); else DL_ACC4(RV, 16)
    if (p <= 32) { DL_ACC4_S(1); }
    else if (p <= 64) { DL_ACC4_S(2); }
    else if (p <= 96) { DL_ACC4_S(3); }
    else { DL_ACC4_S(4); }
#undef DL_ACC4_S
#undef DL_ACC4
    return cudaGetLastError();
  }
  if (p % 4 == 0) {
    // unaligned operands: scalar form with global atomics and w.nb_accum CTAs
    cudaError_t e = cudaMemsetAsync(w.Upart, 0, sizeof(float) * ((size_t)n * p + n), st);
    if (e != cudaSuccess) return e;
#define DL_ACCG(PL)                                                                          \
  accum_kernel<PL, false><<<w.nb_accum, ACC_THREADS, 0, st>>>(Y, p, m, D, n, s, idx, val, cnt, \
                                                              w.Upart, w.epart_a, err)
    if (p <= 32) DL_ACCG(4);
    else if (p <= 64) DL_ACCG(8);
    else if (p <= 96) DL_ACCG(12);
    else DL_ACCG(16);
#undef DL_ACCG
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int len = n * p + n;
    reduce_kernel<<<(len + 255) / 256, 256, 0, st>>>(w.Upart, 1, len, w.U);
    return cudaGetLastError();
  }
  if (p <= 32) return accum_t<4>(Y, p, m, D, n, s, idx, val, cnt, w, err, st);
  if (p <= 64) return accum_t<8>(Y, p, m, D, n, s, idx, val, cnt, w, err, st);
  if (p <= 96) return accum_t<12>(Y, p, m, D, n, s, idx, val, cnt, w, err, st);
  return accum_t<16>(Y, p, m, D, n, s, idx, val, cnt, w, err, st);
}

cudaError_t jau_atoms(const float* D, int p, int n, const JauWork& w, cudaStream_t st) {
  const int a0 = w.a0, a1 = w.a1 > 0 ? w.a1 : n;
  if (w.copies) {
    if (a1 > a0)
      atoms4_kernel<<<a1 - a0, 256, 0, st>>>(w.padded ? w.Dp : D, jau_p4(p), n, w.Ucopy, w.Dn, w.C, a0);
    return cudaGetLastError();
  }
  const int blocks = (a1 - a0 + 7) / 8;
  if (blocks <= 0) return cudaSuccess;
  if (p <= 32) atoms_kernel<1><<<blocks, 256, 0, st>>>(D, p, n, w.U, w.Dn, w.C, a0, a1);
  else if (p <= 64) atoms_kernel<2><<<blocks, 256, 0, st>>>(D, p, n, w.U, w.Dn, w.C, a0, a1);
  else if (p <= 96) atoms_kernel<3><<<blocks, 256, 0, st>>>(D, p, n, w.U, w.Dn, w.C, a0, a1);
  else atoms_kernel<4><<<blocks, 256, 0, st>>>(D, p, n, w.U, w.Dn, w.C, a0, a1);
  return cudaGetLastError();
}

cudaError_t jau_rows(const float* Y, int p, int64_t m, const float* D, int n, int s,
                     const int32_t* idx, float* val, const int32_t* cnt, const JauWork& w,
                     const int64_t* colptr, int32_t* csc_rowidx, float* csc_val, cudaStream_t st) {
  const int nb = w.nb_row;
  const int a1 = w.a1 > 0 ? w.a1 : n;
  const bool grouped = w.a0 > 0 || a1 < n;
#define DL_ROWS(PL)                                                                              \
  rows_kernel<PL><<<nb, ROW_THREADS, 0, st>>>(Y, p, m, D, w.Dn, w.C, s, idx, val, cnt, colptr, \
                                              csc_rowidx, csc_val, w.epart_b, (int)w.sgk)
  if (w.E) {  // the plain case (the row indices are the coding pass's: csc_rowidx is null)
    const int p4 = jau_p4(p);
    const bool vec = jau_vec4(p, Y, D);
#define DL_ROWSP(RV)                                                                              \
  do {                                                                                            \
    auto kern = !vec ? rows_plain_kernel<RV, false, false>                                        \
                     : p == 32 * RV ? rows_plain_kernel<RV, true, true>                           \
                                    : rows_plain_kernel<RV, false, true>;                         \
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,                    \
                         cudaSharedmemCarveoutMaxL1);                                             \
    kern<<<nb, EP_THREADS, 0, st>>>(Y, w.E, p, p4, m, w.Dn, w.C, s, idx, val, cnt, colptr, csc_val, \
                                    w.epart_b, (int)w.sgk);                                       \
  } while (0)
    if (p <= 32) DL_ROWSP(1);
    else if (p <= 64) DL_ROWSP(2);
    else if (p <= 96) DL_ROWSP(3);
    else DL_ROWSP(4);
#undef DL_ROWSP
    return cudaGetLastError();
  }
  if (jau_vec4(p, Y, D)) {
#define DL_ROWS4(RV, SM)                                                                         \
  do {                                                                                         \
    if (grouped)                                                                               \
      rows4_kernel<RV, SM, true><<<nb, ROW_THREADS, 0, st>>>(Y, p, m, D, w.Dn, w.C, s, idx, val, \
                                                             cnt, colptr, csc_rowidx, csc_val,  \
                                                             w.epart_b, w.a0, a1, (int)w.sgk);  \
    else                                                                                       \
      rows4_kernel<RV, SM, false><<<nb, ROW_THREADS, 0, st>>>(Y, p, m, D, w.Dn, w.C, s, idx,    \
                                                              val, cnt, colptr, csc_rowidx,     \
                                                              csc_val, w.epart_b, 0, n,         \
                                                              (int)w.sgk);                      \
  } while (0)
#define DL_ROWS4_S(RV) \
  if (s <= 8) DL_ROWS4(RV, 8); else DL_ROWS4(RV, 16)
    if (p <= 32) { DL_ROWS4_S(1); }
    else if (p <= 64) { DL_ROWS4_S(2); }
    else if (p <= 96) { DL_ROWS4_S(3); }
    else { DL_ROWS4_S(4); }
#undef DL_ROWS4_S
#undef DL_ROWS4
    return cudaGetLastError();
  }
  if (p <= 32) DL_ROWS(4);
  else if (p <= 64) DL_ROWS(8);
  else if (p <= 96) DL_ROWS(12);
  else DL_ROWS(16);
#undef DL_ROWS
  return cudaGetLastError();
}

cudaError_t jau_finalize(const JauWork& w, double* rmse_out, int* iter, float* D, int n, int p,
                         cudaStream_t st) {
  const int64_t np = (int64_t)n * p;
  int64_t cb = (np + FIN_THREADS - 1) / FIN_THREADS;
  if (cb > 256) cb = 256;
  finalize_kernel<<<(unsigned)(1 + cb), FIN_THREADS, 0, st>>>(w.epart_a, w.nb_accum, w.epart_b,
                                                              w.nb_row, rmse_out, iter, w.Dn, D, np, p,
                                                              w.E ? jau_p4(p) : p);
  return cudaGetLastError();
}

cudaError_t slots_to_csc(const int32_t* idx, const float* val, const int32_t* cnt, int64_t m, int s,
                         int64_t* bsum, int64_t* colptr, int32_t* rowidx, float* cval, cudaStream_t st) {
  if (m <= 0) return cudaMemsetAsync(colptr, 0, sizeof(int64_t), st);
  const int rounds = csc_rounds(m);
  const int64_t per = (int64_t)rounds * CSC_THREADS;
  const unsigned nb = (unsigned)((m + per - 1) / per);
  count_sum_kernel<<<nb, CSC_THREADS, 0, st>>>(cnt, m, rounds, bsum);
  csc_write_kernel<<<nb, CSC_THREADS, 0, st>>>(cnt, idx, val, m, s, rounds, bsum, colptr, rowidx, cval);
  return cudaGetLastError();
}

cudaError_t csc_to_slots(const int64_t* colptr, const int32_t* rowidx, const float* cval,
                         int64_t m, int n, int s, int32_t* idx, float* val, int32_t* cnt,
                         int* err, cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
#define DL_SLOTS(W)                                                                                    \
  csc_to_slots_kernel<W><<<(unsigned)((m * W + 255) / 256), 256, 0, st>>>(colptr, rowidx, cval, m, n, s, \
                                                                          idx, val, cnt, err)
  if (s <= 4) DL_SLOTS(4);
  else if (s <= 8) DL_SLOTS(8);
  else DL_SLOTS(16);
#undef DL_SLOTS
  return cudaGetLastError();
}

}  // namespace dlk
