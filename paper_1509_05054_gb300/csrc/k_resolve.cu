// Re-solve of the signals the FP32 OMP cannot decide: a Cholesky pivot below
// 1e-6 (dominated by FP32 rounding), or, for long supports, a step whose top
// two |correlations| lie inside the FP32 error of alpha.  One CTA of four warps
// per listed signal redoes its whole OMP (Algorithm 1 step 1) so that every
// decision and the coefficients are those of the FP64 Batch-OMP:
//
//   * the residual r = y - D_I gamma is kept in FP64 (p values), with gamma from
//     the FP64 Cholesky factor L of G[I,I] (entries d_q^T d_sel taken in FP64 from
//     the FP32 atoms, which FP64 holds exactly) by triangular solves, L z = D_I^T y
//     and L^T gamma = z.  (Kept as an inverse factor, gamma += z B_k, the
//     coefficients of eight near-dependent atoms with a pivot of 2e-9 were off by 1e-4
//     of the largest; solves leave 5e-7, the error of FP64 Cholesky itself.)
//   * each step's correlations alpha = alpha0 - G[:, I] gamma are taken in
//     FP32, fresh every step (no rounding carries over from step to step), from
//     alpha0 (the FP32 product of the coding pass, or, after reduced-precision
//     correlations, D^T y taken here in FP32), the FP32 Gram rows of the
//     selected atoms (copied to shared memory as atoms are selected) and gamma
//     rounded to FP32.  With alpha0 within c ||y|| dmax and the Gram entries
//     within c dmax^2 of exact, c = max(4.5e-6, (p + 2) 2^-24) (split-TF32
//     products: three 2^-22 terms and FP32 sums; or FP32 sums of p products;
//     measured 2.2e-7 and 4.7e-7 at p = 64), alpha is within
//     E = (c + 1.5e-6) dmax (||y|| + dmax sum |gamma_q|) of exact, so
//     the exact argmax lies among the atoms within 2E of the FP32 maximum; each
//     one's correlation d_j^T r is recomputed in FP64 and the largest is taken
//     (lowest index on ties), as the FP64 oracle decides;
//   * the stop rules are the FP64 ones: pivot <= 1e-12, residual energy
//     <= 1e-14 ||y||^2, max |alpha| = 0.
//
// FP64 runs at a small fraction of the FP32 rate on this GPU, so the FP64 work
// is kept to O(k p) per step (the Gram entries of the new atom, the residual and
// the few candidates); the O(n p) and O(n k) products stay FP32.
//
// Few signals are listed (tens to hundreds of 1e5), so the pass takes as long as
// one signal's chain of FP64 latencies, while the rest of the GPU waits.  One
// warp per signal, with a division and a sum over shared memory for every entry of the
// solves, took 209 us at p = 64, n = 1024, s = 10 and 243 us at p = 100, n = 512,
// s = 12.  Here the rows of L are kept divided by their diagonal, so that an entry of
// a solve costs a shuffle and one multiply-add, with the sums on as many lanes as there
// are entries left; eight lanes per dot product take all of a step's Gram entries (or
// candidates) at once, and four warps share the correlations: 55 and 72 us
// (53 and 66 with the inverse factor).
#include "dl_internal.cuh"

#include <math.h>

namespace dlk {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int RS_PMAX = 128;     // largest p (one row per thread)
constexpr int RS_THREADS = 128;
constexpr int RS_GROUPS = RS_THREADS / 8;  // dot products at once, eight lanes each
constexpr int RS_NT = 1024 / RS_THREADS;   // atoms per thread
constexpr int RS_PITCH = RS_PMAX + 8;      // row pitch of Ds: the groups of a warp on distinct banks

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}
// Sum over the eight lanes of a group (all eight call it).
__device__ __forceinline__ double group_sum_d(double v, unsigned mask) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  return v;
}

// Dynamic shared memory: the Gram rows of the selected atoms (s x n floats),
// alpha0 (n, NaN once selected), the candidates of the step (n ints).
__global__ void __launch_bounds__(RS_THREADS) resolve_kernel(
    const float* __restrict__ Y, int p, const float* __restrict__ D, const float* __restrict__ G,
    const float* __restrict__ A0, int64_t lda, int n, int s, const int* __restrict__ list,
    const int* __restrict__ count, int cap, int32_t* __restrict__ oidx, float* __restrict__ oval,
    int32_t* __restrict__ ocnt) {
  __shared__ double Lr[DL_RESOLVE_SMAX][DL_RESOLVE_SMAX + 1];  // L_qt / L_qq, t < q
  __shared__ double Lc[DL_RESOLVE_SMAX][DL_RESOLVE_SMAX + 1];  // L_qt / L_tt, t < q
  __shared__ double gd[DL_RESOLVE_SMAX + 2];                   // d_q^T d_sel, q <= k; then d_sel^T r, d_sel^T y
  __shared__ double Ds[DL_RESOLVE_SMAX][RS_PITCH];            // selected atoms
  __shared__ double Gm[DL_RESOLVE_SMAX];                      // gamma
  __shared__ double rs[RS_PMAX], yd[RS_PMAX];                 // residual; y
  __shared__ double gv[RS_GROUPS], wred[RS_THREADS / 32];
  __shared__ double sh_rr, sh_gsum;
  __shared__ float ys[RS_PMAX], g32[DL_RESOLVE_SMAX];
  __shared__ float fred[RS_THREADS / 32];
  __shared__ int I[DL_RESOLVE_SMAX], gj[RS_GROUPS], ncand, sh_stop;
  extern __shared__ float sh[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = tid >> 3, l8 = tid & 7;
  const unsigned gmask = 0xffu << (lane & 24);
  float* Gs = sh;                      // row q: G[I_q][:]
  float* a0 = sh + (size_t)s * n;      // alpha0
  int* cand = (int*)(a0 + n);
  int total = *count;
  if (total > cap) total = cap;
  if ((int)blockIdx.x >= total) return;  // nothing listed for this CTA (the usual case)

  // largest atom norm (the error bound scales with it)
  float dmax2 = 0.f;
  for (int j = tid; j < n; j += RS_THREADS) dmax2 = fmaxf(dmax2, __ldg(G + (size_t)j * n + j));
  dmax2 = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(dmax2)));
  if (lane == 0) fred[warp] = dmax2;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < RS_THREADS / 32; ++w) dmax2 = fmaxf(dmax2, fred[w]);
  const double dmax = sqrt((double)dmax2 * 1.0001);
  // relative error of alpha0 and of the Gram entries (split TF32, or FP32 sums of p
  // products), plus the FP32 sums over the selected atoms
  const double cerr = fmax(4.5e-6, (p + 2) * 0x1p-24) + 1.5e-6;

  for (int e = blockIdx.x; e < total; e += gridDim.x) {
    const int64_t i = list[e];
    __syncthreads();  // the previous signal's shared values have been read
    const float yt = tid < p ? Y[i * p + tid] : 0.f;
    if (tid < p) {
      ys[tid] = yt;
      rs[tid] = yd[tid] = (double)yt;
    }
    {
      const double t = warp_sum_d((double)yt * (double)yt);
      if (lane == 0) wred[warp] = t;
    }
    __syncthreads();
    double yy = 0.0;
#pragma unroll
    for (int w = 0; w < RS_THREADS / 32; ++w) yy += wred[w];
    if (A0) {  // FP32 correlations of the coding pass
      for (int j = tid; j < n; j += RS_THREADS) a0[j] = __ldg(A0 + i * lda + j);
    } else {   // alpha0 = D^T y in FP32, eight lanes per atom
      for (int j0 = 0; j0 < n; j0 += RS_GROUPS) {
        const int j = j0 + grp;
        float a = 0.f;
        if (j < n) {
#pragma unroll 8
          for (int r = l8; r < p; r += 8) a = fmaf(__ldg(D + (size_t)j * p + r), ys[r], a);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
        if (j < n && l8 == 0) a0[j] = a;
      }
    }
    const double ynorm = sqrt(yy);
    double rr = yy;
    double gsum = 0.0;  // sum |gamma_q|
    double linv = 0.0, z = 0.0;  // warp 0, lane q: 1 / L_qq, z_q
    int k = 0;
    for (int step = 0; step < s; ++step) {
      if (tid == 0) ncand = 0;
      __syncthreads();  // alpha0, g32, the Gram row and the residual of the last step
      // ---- FP32 correlations alpha = alpha0 - G[:, I] gamma (selected: NaN)
      float av[RS_NT];
      float best = 0.f;
#pragma unroll
      for (int t = 0; t < RS_NT; ++t) {
        const int j = tid + RS_THREADS * t;
        av[t] = j < n ? a0[j] : 0.f;
      }
      for (int q = 0; q < k; ++q) {
        const float* Gq = Gs + (size_t)q * n + tid;
        const float gq = g32[q];
#pragma unroll
        for (int t = 0; t < RS_NT; ++t)
          if (tid + RS_THREADS * t < n) av[t] = fmaf(-Gq[RS_THREADS * t], gq, av[t]);
      }
#pragma unroll
      for (int t = 0; t < RS_NT; ++t) {
        av[t] = fabsf(av[t]);
        best = fmaxf(best, av[t]);  // NaN ignored
      }
      best = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(best)));
      if (lane == 0) fred[warp] = best;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < RS_THREADS / 32; ++w) best = fmaxf(best, fred[w]);
      if (!(best > 0.f)) break;
      // ---- the exact argmax among the atoms within 2E of the FP32 maximum
      const double E = cerr * dmax * (ynorm + dmax * gsum);
      const float lo = (float)((double)best - 2.0 * E) * (1.f - 0x1p-22f);
#pragma unroll
      for (int t = 0; t < RS_NT; ++t) {
        const int j = tid + RS_THREADS * t;
        if (j < n && av[t] >= lo) cand[atomicAdd(&ncand, 1)] = j;
      }
      __syncthreads();
      const int nc = ncand;
      int sel = nc > 0 ? cand[0] : n;
      if (nc > 1) {
        double bv = 0.0;  // the group's best candidate
        int bj = n;
        for (int c = grp; c < nc; c += RS_GROUPS) {
          const int j = cand[c];
          double v = 0.0;
#pragma unroll 4
          for (int r = l8; r < p; r += 8) v = fma((double)__ldg(D + (size_t)j * p + r), rs[r], v);
          v = fabs(group_sum_d(v, gmask));
          if (v > bv || (v == bv && v > 0.0 && j < bj)) {
            bv = v;
            bj = j;
          }
        }
        if (l8 == 0) {
          gv[grp] = bv;
          gj[grp] = bj;
        }
        __syncthreads();
        double bestv = 0.0;
        sel = n;
        for (int q = 0; q < RS_GROUPS && q < nc; ++q)
          if (gv[q] > bestv || (gv[q] == bestv && gv[q] > 0.0 && gj[q] < sel)) {
            bestv = gv[q];
            sel = gj[q];
          }
      }
      if (sel >= n) break;
      // ---- the new atom (FP64) and its Gram row to shared memory
      if (tid < p) Ds[k][tid] = (double)__ldg(D + (size_t)sel * p + tid);
#pragma unroll
      for (int t = 0; t < RS_NT; ++t)
        if (tid + RS_THREADS * t < n)
          Gs[(size_t)k * n + tid + RS_THREADS * t] = __ldg(G + (size_t)sel * n + tid + RS_THREADS * t);
      __syncthreads();
      // ---- FP64 Gram entries of the new atom, d_sel^T r and d_sel^T y
      for (int q = grp; q <= k + 2; q += RS_GROUPS) {
        const double* x = q <= k ? Ds[q] : q == k + 1 ? rs : yd;
        double v = 0.0, v2 = 0.0;
#pragma unroll 4
        for (int r = l8; r < p; r += 16) {
          v = fma(x[r], Ds[k][r], v);
          if (r + 8 < p) v2 = fma(x[r + 8], Ds[k][r + 8], v2);
        }
        v = group_sum_d(v + v2, gmask);
        if (l8 == 0) gd[q] = v;
      }
      __syncthreads();
      if (!(fabs(gd[k + 1]) > 0.0)) break;
      // ---- L w = g, delta = G[sel, sel] - w.w, z_k, L^T gamma = z
      if (warp == 0) {
        double w = lane < k ? gd[lane] * linv : 0.0;
        for (int q = 0; q + 1 < k; ++q) {
          const double wq = __shfl_sync(FULL, w, q);
          if (lane > q && lane < k) w = fma(-Lr[lane][q], wq, w);
        }
        const double delta = gd[k] - warp_sum_d(w * w);
        const double zw = gd[k + 2] - warp_sum_d(w * z);
        const bool stop = delta <= 1e-12;
        if (!stop) {
          const double inv = rsqrt(delta), zk = zw * inv;
          if (lane < k) {
            Lr[k][lane] = w * inv;
            Lc[k][lane] = w * linv;
          }
          if (lane == k) {
            linv = inv;
            z = zk;
          }
          __syncwarp();
          double gm = z * linv;  // (zero past lane k)
          for (int q = k; q > 0; --q) {
            const double gq = __shfl_sync(FULL, gm, q);
            if (lane < q) gm = fma(-Lc[q][lane], gq, gm);
          }
          if (lane <= k) {
            Gm[lane] = gm;
            g32[lane] = (float)gm;
          }
          const double gs = warp_sum_d(fabs(gm));
          if (lane == 0) {
            I[k] = sel;
            a0[sel] = __int_as_float(0x7fc00000);  // masked from now on
            sh_rr = rr - zk * zk;
            sh_gsum = gs;
          }
        }
        if (lane == 0) sh_stop = stop ? 1 : 0;
      }
      __syncthreads();
      if (sh_stop) break;
      rr = sh_rr;
      gsum = sh_gsum;
      k = step + 1;
      // ---- r = y - D_I gamma
      if (tid < p) {
        double v = (double)yt;
        for (int q = 0; q < k; ++q) v = fma(-Ds[q][tid], Gm[q], v);
        rs[tid] = v;
      }
      if (rr <= 1e-14 * yy) break;
    }
    // ---- write the support in ascending atom order with gamma
    if (tid < k) {
      int rank = 0;
      for (int q = 0; q < k; ++q) rank += I[q] < I[tid] ? 1 : 0;
      oidx[i * s + rank] = I[tid];
      oval[i * s + rank] = (float)Gm[tid];
    } else if (tid < s) {
      oidx[i * s + tid] = -1;
      oval[i * s + tid] = 0.f;
    }
    if (tid == 0) ocnt[i] = k;
  }
}

}  // namespace

cudaError_t omp_resolve64(const float* Y, int p, const float* D, const float* G, const float* A0,
                          int64_t lda, int n, int s, const int* list, const int* count, int cap,
                          int32_t* idx, float* val, int32_t* cnt, cudaStream_t st) {
  if (p < 1 || p > RS_PMAX || n > RS_NT * RS_THREADS || s < 1 || s > DL_RESOLVE_SMAX)
    return cudaErrorInvalidValue;
  const size_t smem = ((size_t)s + 2) * n * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(resolve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  resolve_kernel<<<2 * num_sms(), RS_THREADS, smem, st>>>(Y, p, D, G, A0, lda, n, s, list, count, cap,
                                                     idx, val, cnt);
  return cudaGetLastError();
}

}  // namespace dlk
