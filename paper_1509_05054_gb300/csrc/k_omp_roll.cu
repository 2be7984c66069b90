// Batch-OMP sparse coding with the vectors of the progressive Cholesky in
// tensor memory and shared memory, rolled loops (Algorithm 1 step 1; the
// arithmetic of omp_warp_kernel, see k_omp.cu, operation by operation, so the
// results are the same bits).
//
// What bounds the coding of wide dictionaries and long supports is how many
// signals an SM holds at once: a signal's vectors u_q (q < s - 1) take
// (s - 1) n floats -- 36 KB at n = 1024, s = 10 -- and each step is a chain of
// dependent latencies (argmax, Gram row from L2, Cholesky row).  With the
// vectors in shared memory alone omp_warp_kernel held four signals per SM there
// (one warp per scheduler, 0.11 instructions per cycle).  Here a persistent CTA
// of 4Q warps per SM keeps COLS / NT vectors of each warp's signal in TMEM
// (256 KB per SM; warp w owns 512/Q columns of its lane quadrant, u_q[32t + l]
// in lane l, column NT q + t) and the rest in shared memory: 16 signals per SM
// at s <= 8, 12 at s <= 10, 8 up to s = 15 and 4 at s = 16 for n = 1024.  Because every vector
// then has an address, the loops over steps and vectors are rolled and w, c and
// the back substitution live one entry per lane: the code is a few KB, while the
// unrolled form with register vectors (NT (s - 1) floats per lane) is tens of KB.
// Measured at p = 64, n = 1024, s = 10, m = 46,000: 430 us for 1,655 before, at
// 0.54 instructions per scheduler and cycle with three warps each: about half of
// the time is issue, the rest the latency of each step's chain.
#include "dl_internal.cuh"
#include "omp_common.cuh"
#include "tc_ptx.cuh"

#include <math.h>

namespace dlk {
namespace {

using namespace omp;

// ---- TMEM access (32 lanes x 32-bit columns, this warp's quadrant); loads are
// complete after tm_wait, and tie keeps the uses of their registers behind it
__device__ __forceinline__ void tm_ld(uint32_t a, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(a));
}
__device__ __forceinline__ void tm_ld(uint32_t a, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(a));
}
__device__ __forceinline__ uint32_t tm_ld1(uint32_t a) {
  uint32_t r;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(a));
  return r;
}
__device__ __forceinline__ void tm_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void tie(uint32_t (&r)[N]) {
#pragma unroll
  for (int t = 0; t < N; ++t) asm volatile("" : "+r"(r[t]));
}
__device__ __forceinline__ void tm_st(uint32_t a, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(a),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tm_st(uint32_t a, const uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(a), "r"(r[0]),
      "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
__device__ __forceinline__ void tm_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// alpha[tsel] on the owning lane, masked to NaN (selected); an indexed branch
// executed by one lane.
template <int NT>
__device__ __forceinline__ float take_alpha(float2 (&alpha)[NT / 2], int tsel, float qnan) {
  float out = 0.f;
#define DL_TAKE_CASE(T)                  \
  case T:                                \
    if constexpr (T < NT) {              \
      constexpr int TT = T < NT ? T : 0; \
      if constexpr (TT & 1) {            \
        out = alpha[TT >> 1].y;          \
        alpha[TT >> 1].y = qnan;         \
      } else {                           \
        out = alpha[TT >> 1].x;          \
        alpha[TT >> 1].x = qnan;         \
      }                                  \
    }                                    \
    break;
#define DL_TAKE_4(T) DL_TAKE_CASE(T) DL_TAKE_CASE(T + 1) DL_TAKE_CASE(T + 2) DL_TAKE_CASE(T + 3)
  switch (tsel) {
    DL_TAKE_4(0) DL_TAKE_4(4) DL_TAKE_4(8) DL_TAKE_4(12)
    DL_TAKE_4(16) DL_TAKE_4(20) DL_TAKE_4(24) DL_TAKE_4(28)
    default: break;
  }
#undef DL_TAKE_4
#undef DL_TAKE_CASE
  return out;
}

// Columns of TMEM and vectors in TMEM of each of 4Q warps (TM; none otherwise).
template <int NT, int Q, bool TM>
struct Shape {
  static constexpr int W = 4 * Q;
  static constexpr int NTM = !TM ? 0 : (512 / Q) / NT < DL_RESOLVE_SMAX - 1 ? (512 / Q) / NT : DL_RESOLVE_SMAX - 1;
  static constexpr int COLS = NTM * NT;
  // registers for two vectors of TMEM loads in flight (65536 / threads, less the rest)
  static constexpr bool TWO = 512 / Q - 64 >= 3 * NT;
  static_assert(COLS * Q <= 512 && (NTM >= 1 || !TM), "TMEM columns");
  // dynamic shared memory of `warps` warps for supports of s: vectors past NTM, and the Cholesky rows
  static size_t smem(int s, int warps = W) {
    const int nsh = s - 1 > NTM ? s - 1 - NTM : 0;
    return (size_t)warps * ((size_t)nsh * NT * 32 * sizeof(float) + (size_t)s * s * sizeof(float));
  }
};

// The OMP of signal i by one warp; see omp_one (omp_one.cuh) for the steps.
// tcol: TMEM address of this warp's first column; u_q for q < NTM at tcol +
// NT q, the others in u_s (shared memory, [q - NTM][pair][lane]); L: s x s.
template <int NT, int NTM, bool FULLN, bool TWO>
__device__ __forceinline__ void omp_one_roll(
    int64_t i, const float* __restrict__ G, int n, float* L, float2* u_s, uint32_t tcol,
    const float* __restrict__ a0row, const float* __restrict__ y, int p, int s,
    int32_t* __restrict__ oidx, float* __restrict__ oval, int32_t* __restrict__ ocnt,
    float* __restrict__ ores, int* __restrict__ err, int* __restrict__ rs_list,
    int* __restrict__ rs_count, int rs_cap, float gap_tol) {
  constexpr int NV = NT / 2;
  constexpr int C = NT < 16 ? NT : 16;  // columns per TMEM access
  constexpr int TB = tbits<NT>();
  constexpr unsigned TMASK = (1u << TB) - 1u;
  constexpr unsigned VMASK = 0x7FFFFFFFu & ~TMASK;
  const int lane = threadIdx.x & 31;

  float yy = 0.f;
  for (int r = lane; r < p; r += 32) {
    const float v = ld_stream(y + r);
    yy = fmaf(v, v, yy);
  }
  yy = warp_sum(yy);
  const bool finite_in = isfinite(yy);
  if (!finite_in && lane == 0) atomicOr(err, ERR_NONFINITE);

  const float qnan = __int_as_float(0x7fc00000);
  float2 alpha[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int j0 = 64 * v + lane, j1 = j0 + 32;
    alpha[v].x = (FULLN || j0 < n) ? ld_stream(a0row + j0) : qnan;
    alpha[v].y = (FULLN || j1 < n) ? ld_stream(a0row + j1) : qnan;
  }

  float myc = 0.f;  // lane j: c_j = 1 / L_jj
  float myz = 0.f;  // lane j: z_j
  int myI = -1;     // lane j: I_j
  float rr = yy;
  int k = 0;

#pragma unroll 1
  for (int step = 0; step < s; ++step) {
    if (!finite_in) break;
    const float kmax = keys_max<NT>(alpha, VMASK);
    const unsigned kbits = __reduce_max_sync(FULL, __float_as_uint(kmax));
    if ((kbits & VMASK) == 0u) break;  // max |alpha| = 0
    const unsigned ball = __ballot_sync(FULL, __float_as_uint(kmax) == kbits);
    const int lsel = __ffs(ball) - 1;
    const int tsel = NT - 1 - (int)(kbits & TMASK);
    const int sel = 32 * tsel + lsel;
    // the Gram loads early: the diagonal (for the pivot), then the row
    const bool need_u = step + 1 < s;
    const float* __restrict__ Gr = G + (size_t)sel * n;
    const float gss = __ldg(Gr + sel);
    float2 g[NV];
    if (need_u) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int j0 = 64 * v + lane, j1 = j0 + 32;
        g[v].x = (FULLN || j0 < n) ? __ldg(Gr + j0) : 0.f;
        g[v].y = (FULLN || j1 < n) ? __ldg(Gr + j1) : 0.f;
      }
    }
    // u_q[sel] to lane q, q < step: single TMEM columns and a shuffle from the
    // owning lane, or the owning lane's entry in shared memory
    float ul = 0.f;
    {
      if constexpr (NTM > 0) {
        uint32_t tv[NTM];
        if (step > 0) tm_wait_st();  // u_{step-1} was just stored
#pragma unroll
        for (int q = 0; q < NTM; ++q) tv[q] = q < step ? tm_ld1(tcol + NT * q + tsel) : 0u;
        tm_wait();
        tie(tv);
#pragma unroll
        for (int q = 0; q < NTM; ++q) {
          if (q >= step) break;
          const float v = __shfl_sync(FULL, __uint_as_float(tv[q]), lsel);
          if (lane == q) ul = v;
        }
      }
      if (lane >= NTM && lane < step) {
        const float2 pr = u_s[((lane - NTM) * NV + (tsel >> 1)) * 32 + lsel];
        ul = (tsel & 1) ? pr.y : pr.x;
      }
    }
    float amine = 0.f;
    if (lane == lsel) amine = take_alpha<NT>(alpha, tsel, qnan);
    const float asel = __shfl_sync(FULL, amine, lsel);
    if (s > 8 && gap_tol > 0.f && rs_count) {
      // second largest |alpha| (the winner is masked now), full precision
      float top2 = 0.f;
#pragma unroll
      for (int v = 0; v < NV; ++v) top2 = fmaxf(top2, fmaxf(fabsf(alpha[v].x), fabsf(alpha[v].y)));
      top2 = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(top2)));
      if (fabsf(asel) - top2 < gap_tol * sqrtf(yy)) {
        if (lane == 0) {
          const int pos = atomicAdd(rs_count, 1);
          if (pos < rs_cap) rs_list[pos] = (int)i;
        }
        break;
      }
    }
    const float w = ul * myc;  // lane q < step: w_q = c_q u_q[sel]
    const float negaw = -w * myc;
    float wsq = 0.f;
    for (int q = 0; q < step; ++q) {
      const float wq = __shfl_sync(FULL, w, q);
      wsq = fmaf(wq, wq, wsq);
    }
    if (lane < step) L[step * s + lane] = w;
    const float delta = gss - wsq;
    if (!(delta > kPivotMin)) {
      if (lane == 0) {
        if (!isfinite(delta)) atomicOr(err, ERR_NONFINITE);
        if (rs_count) {  // rounding dominates this pivot: redo the signal in FP64
          const int pos = atomicAdd(rs_count, 1);
          if (pos < rs_cap) rs_list[pos] = (int)i;
        }
      }
      break;
    }
    // c_k = 1 / L_kk: rsqrtf refined by one Newton-Raphson step, y + y (1 - d y^2) / 2
    float ck = rsqrtf(delta);
    ck = fmaf(0.5f * ck, fmaf(-delta * ck, ck, 1.0f), ck);
    const float zk = asel * ck;
    if (lane == step) {
      myc = ck;
      myz = zk;
      myI = sel;
    }
    rr = fmaf(-zk, zk, rr);
    k = step + 1;

    if (need_u) {  // u_step = G[:, sel] + sum_q negaw_q u_q;  alpha -= (z_k c_k) u_step
      const int nt = step < NTM ? step : NTM;
      auto add = [&](float nq, uint32_t (&r)[NT / C][C]) {
        const float2 nw = make_float2(nq, nq);
#pragma unroll
        for (int h = 0; h < NT / C; ++h) {
          tie(r[h]);
#pragma unroll
          for (int v = 0; v < C / 2; ++v) {
            float2& gv = g[h * (C / 2) + v];
            gv = __ffma2_rn(nw, make_float2(__uint_as_float(r[h][2 * v]), __uint_as_float(r[h][2 * v + 1])), gv);
          }
        }
      };
      int q0 = 0;
      if constexpr (TWO) {  // two vectors per wait, while the registers allow it
#pragma unroll 1
        for (; q0 + 1 < nt; q0 += 2) {
          uint32_t r0[NT / C][C], r1[NT / C][C];
#pragma unroll
          for (int h = 0; h < NT / C; ++h) tm_ld(tcol + NT * q0 + C * h, r0[h]);
#pragma unroll
          for (int h = 0; h < NT / C; ++h) tm_ld(tcol + NT * (q0 + 1) + C * h, r1[h]);
          const float n0 = __shfl_sync(FULL, negaw, q0), n1 = __shfl_sync(FULL, negaw, q0 + 1);
          tm_wait();
          add(n0, r0);
          add(n1, r1);
        }
      }
#pragma unroll 1
      for (int q = q0; q < nt; ++q) {
        uint32_t r[NT / C][C];
#pragma unroll
        for (int h = 0; h < NT / C; ++h) tm_ld(tcol + NT * q + C * h, r[h]);
        const float nq = __shfl_sync(FULL, negaw, q);
        tm_wait();
        add(nq, r);
      }
#pragma unroll 2
      for (int q = NTM; q < step; ++q) {
        const float nq = __shfl_sync(FULL, negaw, q);
        const float2 nw = make_float2(nq, nq);
        const float2* uq = u_s + (q - NTM) * NV * 32 + lane;
#pragma unroll
        for (int v = 0; v < NV; ++v) g[v] = __ffma2_rn(nw, uq[v * 32], g[v]);
      }
      if (step < NTM) {
#pragma unroll
        for (int h = 0; h < NT / C; ++h) {
          uint32_t r[C];
#pragma unroll
          for (int v = 0; v < C / 2; ++v) {
            r[2 * v] = __float_as_uint(g[h * (C / 2) + v].x);
            r[2 * v + 1] = __float_as_uint(g[h * (C / 2) + v].y);
          }
          tm_st(tcol + NT * step + C * h, r);
        }
      } else {
        float2* uq = u_s + (step - NTM) * NV * 32 + lane;
#pragma unroll
        for (int v = 0; v < NV; ++v) uq[v * 32] = g[v];
      }
      const float nz = -zk * ck;
      const float2 nz2 = make_float2(nz, nz);
#pragma unroll
      for (int v = 0; v < NV; ++v) alpha[v] = __ffma2_rn(nz2, g[v], alpha[v]);
    }
    __syncwarp();  // row `step` of L and a shared u_step are read later
    if (rr <= kResidRel * yy) break;
  }
  if constexpr (NTM > 0) tm_wait_st();
  __syncwarp();

  // ---- back substitution L^T gamma = z
  float gam = 0.f, acc2 = 0.f;
  for (int q = k - 1; q >= 0; --q) {
    const float gl = (myz - acc2) * myc;  // valid on lane q
    const float gq = __shfl_sync(FULL, gl, q);
    if (lane == q) gam = gq;
    if (lane < q) acc2 = fmaf(L[q * s + lane], gq, acc2);
  }
  // ---- the support in ascending atom order
  int rank = 0;
  for (int q = 0; q < k; ++q) rank += __shfl_sync(FULL, myI, q) < myI ? 1 : 0;
  const int64_t base = i * s;
  if (lane < k) {
    oidx[base + rank] = myI;
    oval[base + rank] = gam;
  } else if (lane < s) {
    oidx[base + lane] = -1;
    oval[base + lane] = 0.f;
  }
  if (lane == 0) {
    ocnt[i] = k;
    if (ores) ores[i] = rr;
  }
  __syncwarp();
}

// Persistent: one CTA of W <= 4Q warps per SM; warp w of CTA b codes signals
// b * W + w + t * gridDim.x * W.
template <int NT, int Q, bool TM, bool FULLN>
__global__ void __launch_bounds__(Q * 128, 1) omp_roll_kernel(
    const float* __restrict__ A0, int64_t lda, const float* __restrict__ G, int n,
    const float* __restrict__ Y, int p, int64_t m, int s, int32_t* __restrict__ oidx,
    float* __restrict__ oval, int32_t* __restrict__ ocnt, float* __restrict__ ores,
    int* __restrict__ err, int* __restrict__ rs_list, int* __restrict__ rs_count, int rs_cap,
    float gap_tol) {
  using S = Shape<NT, Q, TM>;
  const int W = blockDim.x >> 5;
  extern __shared__ float2 smem_u[];
  __shared__ uint32_t tbase_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (TM && warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     tc::smem_u32(&tbase_sh)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  uint32_t tbase = 0;
  if (TM) {
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    tbase = tbase_sh;
  }
  const uint32_t tcol = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * S::COLS);
  const int nsh = s - 1 > S::NTM ? s - 1 - S::NTM : 0;
  float2* u_s = smem_u + (size_t)warp * nsh * (NT / 2) * 32;
  float* L = (float*)(smem_u + (size_t)W * nsh * (NT / 2) * 32) + warp * s * s;
  const int64_t stride = (int64_t)gridDim.x * W;
  for (int64_t i = (int64_t)blockIdx.x * W + warp; i < m; i += stride) {
    const int64_t ip = i + stride;
    if (ip < m) {  // warm L2 with the warp's next signal: correlations and samples
      if (lane * 32 < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(A0 + ip * lda + lane * 32));
      if (lane * 32 < p) asm volatile("prefetch.global.L2 [%0];" ::"l"(Y + ip * p + lane * 32));
    }
    omp_one_roll<NT, S::NTM, FULLN, S::TWO>(i, G, n, L, u_s, tcol, A0 + i * lda, Y + i * p, p, s, oidx, oval,
                                    ocnt, ores, err, rs_list, rs_count, rs_cap, gap_tol);
  }
  if (!TM) return;
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(512)
                 : "memory");
}

constexpr size_t kRollSmem = 226 * 1024;  // dynamic shared memory one CTA may ask for

template <int NT, int Q, bool TM>
cudaError_t launch_q(const float* A0, int64_t lda, const float* G, int n, const float* Y, int p,
                     int64_t m, int s, int32_t* idx, float* val, int32_t* cnt, float* ores,
                     int* err, int* rl, int* rc, int rcap, float gt, cudaStream_t st) {
  // the rounds that 4Q warps per SM need, with the signals spread evenly over them:
  // no warp more than that
  const int64_t round = (int64_t)num_sms() * Shape<NT, Q, TM>::W;
  const int64_t slots = (m + round - 1) / round * num_sms();
  const int W = (int)((m + slots - 1) / slots);
  const size_t smem = Shape<NT, Q, TM>::smem(s, W);
  auto kern = n == 32 * NT ? omp_roll_kernel<NT, Q, TM, true> : omp_roll_kernel<NT, Q, TM, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t need = (m + W - 1) / W;
  const int grid = (int)(need < num_sms() ? need : num_sms());
  kern<<<grid, W * 32, smem, st>>>(A0, lda, G, n, Y, p, m, s, idx, val, cnt, ores, err, rl, rc, rcap, gt);
  return cudaGetLastError();
}

}  // namespace

// Taken where it is the faster one: wide dictionaries from s = 5 (p = 64,
// n = 1024, m = 20,000: s = 6 94 us against 386 of omp_warp_kernel, s = 10 185
// against 728, s = 16 891 against 1,639; at s = 4, where that kernel's vectors fit
// in registers, 62 against 49), and supports past 8 (m = 40,000: n = 512, s = 9
// 177 against 215 us, s = 16 577 against 821; n = 256, s = 10 165 against 235).
// With s <= 8 and n <= 512 the unrolled kernels are as fast or faster.
//
// A call of few signals is one round of at most a few warps per SM, and its time is
// one signal's chain of steps, of which TMEM's latency is a large part: while
// the vectors of the warps of that one round fit in shared memory, they all lie there
// and no TMEM is allocated.  n = 256, s = 10, m = 300 9.2 us (in TMEM with the
// signals on as few SMs as hold them 20.8, spread over all SMs 12.6; omp_warp_kernel
// 7.9); n = 512, s = 12, m = 600 12.9 (23.2, 16.5; 13.4); n = 1024, s = 10, m = 600
// 13.0 (19.4, 14.9; 27).
bool omp_roll_supported(int n, int s) {
  return n > 128 && n <= 1024 && s <= DL_RESOLVE_SMAX && (s > 8 || (n > 512 && s > 4));
}

cudaError_t omp_roll(const float* A0, int64_t lda, const float* G, int n, const float* Y, int p,
                     int64_t m, int s, int32_t* idx, float* val, int32_t* cnt, float* ores,
                     int* err, int* rl, int* rc, int rcap, float gt, cudaStream_t st) {
  if (!omp_roll_supported(n, s)) return cudaErrorInvalidValue;
  if (m <= 0) return cudaSuccess;
  // one round with every vector in shared memory, else the most warps whose vectors fit
#define DL_ROLL_SH(NT, Q)                                                                 \
  if (m <= 4 * Q * (int64_t)num_sms() &&                                                  \
      Shape<NT, Q, false>::smem(s, (int)((m + num_sms() - 1) / num_sms())) <= kRollSmem)  \
  return launch_q<NT, Q, false>(A0, lda, G, n, Y, p, m, s, idx, val, cnt, ores, err, rl, rc, rcap, gt, st)
#define DL_ROLL(NT, Q)                          \
  if (Shape<NT, Q, true>::smem(s) <= kRollSmem) \
  return launch_q<NT, Q, true>(A0, lda, G, n, Y, p, m, s, idx, val, cnt, ores, err, rl, rc, rcap, gt, st)
  if (n > 512) {
    DL_ROLL_SH(32, 2);
    DL_ROLL(32, 4);
    DL_ROLL(32, 3);
    DL_ROLL(32, 2);
    DL_ROLL(32, 1);
  } else if (n > 256) {
    DL_ROLL_SH(16, 4);
    DL_ROLL(16, 6);
    DL_ROLL(16, 5);
    DL_ROLL(16, 4);
    DL_ROLL(16, 3);
  } else {
    DL_ROLL_SH(8, 4);
    DL_ROLL(8, 8);
    DL_ROLL(8, 6);
  }
#undef DL_ROLL
#undef DL_ROLL_SH
  return cudaErrorInvalidValue;
}

}  // namespace dlk
