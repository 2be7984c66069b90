// The learned support proposer: a BF16 MLP p -> hidden -> hidden -> n (GELU, sigmoid
// outputs) trained with binary cross-entropy on multi-hot OMP supports, and its
// inference (top-2s candidates per signal).  All products run on one tcgen05
// GEMM kernel with FP32 accumulation in TMEM and fused epilogues (bias, GELU,
// GELU derivative, the cross-entropy's gradient and loss, bias gradients).
// Operands are BF16, row-major; either may be contracted along its rows
// (K-major tiles) or along its columns (MN-major tiles), so the backward
// products read the forward pass's arrays as they are.
//
// What bounds a training step of 4096 rows at hidden = n = 512 (13 GFLOP, 7 us of
// tensor time) is everything around the MMAs.  Measured before (us per step):
// products 258 (64 CTAs of 128 threads, a row per thread in the epilogue, scalar
// atomics for the split sums), the loss and its gradient as a kernel with
// FP64 arithmetic per element 68, explicit transposes 37, column sums 29, six
// memsets 8; with the gaps 460.  Now 77: seven launches that overlap each other's
// start, 128 x 128 tiles with sixteen warps and coalesced rows in the epilogue, the
// loss, its gradient and the bias gradients in the epilogues, vector reductions for
// the split sums, and a layer's two backward products in one launch.  What is left is
// mostly each launch's chain of load, MMA and epilogue latencies (about 10 us).
#include "dl_internal.cuh"
#include "sum2.cuh"
#include "tc_ptx.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <stdint.h>

namespace dlk {
namespace {

using namespace tc;

constexpr int GM_THREADS = 512;  // sixteen warps: four per TMEM lane quadrant in the epilogue
constexpr int GM_TILE = 128;     // rows and columns of a CTA's output tile
constexpr int GM_BK = 64;        // contraction elements per stage (128 bytes of BF16)
constexpr int GM_WC = GM_TILE / (GM_THREADS / 128);  // columns a warp takes in the epilogue (of 32 rows)
constexpr int GM_WU = GM_WC / 4;                     // as 16-byte units
// Three stages of 32 KB: two CTAs per SM, so that one's epilogue overlaps the
// other's loads and MMAs.
constexpr int GM_STAGES = 3;
constexpr uint32_t GM_OP_BYTES = GM_TILE * GM_BK * 2;  // one operand of a stage, 16 KB
constexpr size_t GM_SMEM = 1024 + (size_t)GM_STAGES * 2 * GM_OP_BYTES + 256;
static_assert((size_t)GM_STAGES * 2 * GM_OP_BYTES >= GM_TILE * GM_TILE * sizeof(float), "epilogue staging");
// kind::f16: D F32, A and B BF16, M = N = 128; bits 15 and 16: A, B MN-major
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GM_TILE >> 3) << 17) |
                            ((uint32_t)(GM_TILE >> 4) << 24);

__device__ __forceinline__ float gelu_f(float a) { return 0.5f * a * (1.f + erff(a * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float a) {
  return 0.5f * (1.f + erff(a * 0.70710678118654752f)) +
         a * 0.39894228040143268f * expf(-0.5f * a * a);
}

// Descriptor of an operand tile: K-major (128 rows of 128 bytes), or MN-major
// (two blocks of 64 columns, 8 KB apart, each 64 contraction rows of 128 bytes),
// both with the 128-byte swizzle and 8-row groups of 1024 bytes.
template <bool MN>
__device__ __forceinline__ uint64_t tile_desc(const void* base) {
  uint64_t d = sw128_desc(base);
  if (MN) d += (uint64_t)((8192 >> 4) - 1) << 16;  // leading byte offset
  return d;
}
// 16 contraction elements further (descriptor units of 16 bytes).
template <bool MN>
constexpr uint64_t kstep() { return MN ? (16 * 128) >> 4 : 32 >> 4; }

template <bool MN>
__device__ __forceinline__ void load_tile(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int k0,
                                          int mn0) {
  if (MN) {
    tma_load_2d(dst, map, bar, mn0, k0);
    tma_load_2d(dst + 8192, map, bar, mn0 + 64, k0);
  } else {
    tma_load_2d(dst, map, bar, k0, mn0);
  }
}

__device__ __forceinline__ uint2 pack_bf16x4(float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*(const uint32_t*)&a, *(const uint32_t*)&b);
}

// C[M x N] = A B, contraction length K: A is M x K (AMN: stored K x M), B is N x K
// (BMN: stored K x N), row-major BF16; M or N or K need not fill the tiles (TMA
// fills with zeros), N % 64 == 0, K % 64 == 0.  One CTA per 128 x 128 tile and
// slice bz of the contraction.  Warp 0 issues the TMA loads, warp 1 the
// MMAs; then all sixteen warps take 32 rows x 32 columns each through shared memory
// (16-byte units XORed with the row: no bank conflicts either way) so that every
// global access is whole 128-byte lines (FP32) and a lane keeps the same four
// columns throughout.
struct Job {
  CUtensorMap A, B;
  int64_t M;
  int N, K;
  int gx, gy, gz;  // row tiles, column tiles, slices of the contraction
  MlpEpi epi;
};

template <bool AMN, bool BMN, int OP>
__device__ __forceinline__ void gemm_tile(const Job& job, int bx, int by, int bz, int* __restrict__ err) {
  const CUtensorMap& tmA = job.A;
  const CUtensorMap& tmB = job.B;
  const int64_t M = job.M;
  const int N = job.N, K = job.K;
  const MlpEpi& epi = job.epi;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* As = base;
  uint8_t* Bs = base + GM_STAGES * GM_OP_BYTES;
  uint64_t* full = (uint64_t*)(Bs + GM_STAGES * GM_OP_BYTES);
  uint64_t* empty = full + GM_STAGES;
  uint64_t* done = empty + GM_STAGES;
  uint32_t* tmem_slot = (uint32_t*)(done + 1);
  __shared__ int s_fail;
  __shared__ double s_loss[GM_THREADS / 32];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t m0 = (int64_t)bx * GM_TILE;
  const int n0 = by * GM_TILE;
  const int nk = K / GM_BK;
  const int per = (nk + job.gz - 1) / job.gz;
  const int kbeg = bz * per;
  const int cnt = (kbeg + per < nk ? kbeg + per : nk) - kbeg;
  if (cnt <= 0) return;  // no share of the contraction (uniform in the CTA)

  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int q = 0; q < GM_STAGES; ++q) {
      mbar_init(&full[q], 1);
      mbar_init(&empty[q], 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"((uint32_t)GM_TILE)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // The setup above overlaps the end of the previous kernel (launch_gemm): the
  // next one may start its own, and nothing before this wait reads or writes
  // global memory.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (threadIdx.x == 0) {
    for (int j = 0; j < cnt; ++j) {
      const int st = j % GM_STAGES;
      if (j >= GM_STAGES && !mbar_wait(&empty[st], (uint32_t)((j / GM_STAGES - 1) & 1))) {
        s_fail = 1;
        break;
      }
      mbar_expect_tx(&full[st], 2 * GM_OP_BYTES);
      load_tile<AMN>(As + st * GM_OP_BYTES, &tmA, &full[st], (kbeg + j) * GM_BK, (int)m0);
      load_tile<BMN>(Bs + st * GM_OP_BYTES, &tmB, &full[st], (kbeg + j) * GM_BK, n0);
    }
  } else if (threadIdx.x == 32) {
    bool ok = true;
    for (int j = 0; j < cnt; ++j) {
      const int st = j % GM_STAGES;
      if (!(ok = mbar_wait(&full[st], (uint32_t)((j / GM_STAGES) & 1)))) break;
      tc_fence_after();
      const uint64_t ad = tile_desc<AMN>(As + st * GM_OP_BYTES);
      const uint64_t bd = tile_desc<BMN>(Bs + st * GM_OP_BYTES);
#pragma unroll
      for (int k = 0; k < GM_BK / 16; ++k)
        mma_f16(tmem, ad + k * kstep<AMN>(), bd + k * kstep<BMN>(),
                kIdesc | (AMN ? 1u << 15 : 0u) | (BMN ? 1u << 16 : 0u), (j > 0 || k > 0) ? 1u : 0u);
      mma_commit(&empty[st]);
    }
    if (ok) {
      mma_commit(done);
      ok = mbar_wait(done, 0);
    }
    if (!ok) s_fail = 1;
  }
  __syncthreads();
  tc_fence_after();
  double loss = 0.0;
  const int col0 = n0 + GM_WC * (warp >> 2);
  if (!s_fail && col0 < N) {
    const int quad = warp & 3;
    float4* stage = (float4*)base + warp * (32 * GM_WU);
#pragma unroll
    for (int c = 0; c < GM_WC / 16; ++c) {
      uint32_t r[16];
      tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(GM_WC * (warp >> 2) + 16 * c), r);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        stage[lane * GM_WU + ((4 * c + q) ^ (lane & (GM_WU - 1)))] =
            make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                        __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
    }
    const int64_t row0 = m0 + quad * 32;
    const int u = lane & (GM_WU - 1), rl = lane / GM_WU, col = col0 + 4 * u;
    uint32_t target = 0;  // BCE: lane = row, its support inside these 32 columns
    if (OP == MLP_EPI_BCE && row0 + lane < M) {
      static_assert(GM_WC == 32, "target bits");
      const int4* sp = (const int4*)(epi.sup + (row0 + lane) * 16);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int4 v = __ldg(sp + q);
        if ((unsigned)(v.x - col0) < 32u) target |= 1u << (v.x - col0);
        if ((unsigned)(v.y - col0) < 32u) target |= 1u << (v.y - col0);
        if ((unsigned)(v.z - col0) < 32u) target |= 1u << (v.z - col0);
        if ((unsigned)(v.w - col0) < 32u) target |= 1u << (v.w - col0);
      }
    }
    const float4 bias = epi.bias ? __ldg((const float4*)(epi.bias + col)) : make_float4(0.f, 0.f, 0.f, 0.f);
    const float fm = (float)M, im = 1.f / fm;
    const bool pow2 = (M & (M - 1)) == 0;  // then the product with 1/M is the quotient, exactly
    float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);  // column sums of the BF16 output
    Sum2 ls;
    __syncwarp();
#pragma unroll 2
    for (int it = 0; it < GM_WU; ++it) {
      const int rr = (32 / GM_WU) * it + rl;
      const int64_t row = row0 + rr;
      const uint32_t tg = OP == MLP_EPI_BCE ? __shfl_sync(0xffffffffu, target, rr) >> (4 * u) : 0;
      if (row >= M) continue;
      float4 a = stage[rr * GM_WU + (u ^ (rr & (GM_WU - 1)))];
      const int64_t o = row * epi.ldc + col;
      if (OP == MLP_EPI_RED) {
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(epi.out_f32 + o), "f"(a.x),
                     "f"(a.y), "f"(a.z), "f"(a.w)
                     : "memory");
        continue;
      }
      a.x += bias.x;
      a.y += bias.y;
      a.z += bias.z;
      a.w += bias.w;
      if (OP == MLP_EPI_LOGITS || OP == MLP_EPI_GELU_FWD)
        if (epi.out_f32) *(float4*)(epi.out_f32 + o) = a;
      if (OP == MLP_EPI_GELU_FWD) {
        a = make_float4(gelu_f(a.x), gelu_f(a.y), gelu_f(a.z), gelu_f(a.w));
      } else if (OP == MLP_EPI_GELU_BWD) {
        const float4 x = __ldg((const float4*)(epi.aux + o));
        a = make_float4(a.x * gelu_grad_f(x.x), a.y * gelu_grad_f(x.y), a.z * gelu_grad_f(x.z),
                        a.w * gelu_grad_f(x.w));
      } else if (OP == MLP_EPI_BCE) {
        // dz = (sigmoid(z) - t) / B, and the loss sum(softplus(z) - t z) / B
        float* v = &a.x;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float z = v[q], t = (tg >> q & 1) ? 1.f : 0.f;
          const float sg = 1.f / (1.f + expf(-z));
          const float sp = fmaxf(z, 0.f) + log1pf(expf(-fabsf(z)));
          ls.add(sp - t * z);
          v[q] = pow2 ? (sg - t) * im : (sg - t) / fm;
        }
      }
      if (OP != MLP_EPI_LOGITS || epi.out_bf16) {
        const uint2 h = pack_bf16x4(a);
        *(uint2*)(epi.out_bf16 + o) = h;
        if (OP == MLP_EPI_GELU_BWD || OP == MLP_EPI_BCE) {
          cs.x += __uint_as_float(h.x << 16);
          cs.y += __uint_as_float(h.x & 0xffff0000u);
          cs.z += __uint_as_float(h.y << 16);
          cs.w += __uint_as_float(h.y & 0xffff0000u);
        }
      }
    }
    if (OP == MLP_EPI_GELU_BWD || OP == MLP_EPI_BCE) {
#pragma unroll
      for (int o = GM_WU; o < 32; o <<= 1) {
        cs.x += __shfl_xor_sync(0xffffffffu, cs.x, o);
        cs.y += __shfl_xor_sync(0xffffffffu, cs.y, o);
        cs.z += __shfl_xor_sync(0xffffffffu, cs.z, o);
        cs.w += __shfl_xor_sync(0xffffffffu, cs.w, o);
      }
      if (lane < GM_WU)
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(epi.colsum + col), "f"(cs.x),
                     "f"(cs.y), "f"(cs.z), "f"(cs.w)
                     : "memory");
    }
    if (OP == MLP_EPI_BCE) loss = ls.value();
  }
  if (OP == MLP_EPI_BCE) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) s_loss[warp] = loss;
  }
  if (s_fail && threadIdx.x == 0) atomicOr(err, ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (OP == MLP_EPI_BCE && threadIdx.x == 0) {
    for (int w = 1; w < GM_THREADS / 32; ++w) loss += s_loss[w];
    atomicAdd(epi.loss, loss / (double)M);
  }
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)GM_TILE)
                 : "memory");
}

template <bool AMN, bool BMN, int OP>
__global__ void __launch_bounds__(GM_THREADS, 2)
    gemm_bf16_kernel(const __grid_constant__ Job job, int* __restrict__ err) {
  const int t = (int)blockIdx.x % (job.gx * job.gy);
  gemm_tile<AMN, BMN, OP>(job, t % job.gx, t / job.gx, (int)blockIdx.x / (job.gx * job.gy), err);
}

// A layer's two backward products, which read the same dY, in one launch: the
// input gradient dY W (with the GELU derivative), then the weight gradient
// dY^T X.  Either alone leaves a good part of the two CTAs per SM idle (128 and
// 144 CTAs of 304 at batch 4096 and width 512).
__global__ void __launch_bounds__(GM_THREADS, 2)
    gemm_backward_kernel(const __grid_constant__ Job data, const __grid_constant__ Job weight,
                         int* __restrict__ err) {
  const int nd = data.gx * data.gy, b = (int)blockIdx.x;
  if (b < nd) {
    gemm_tile<false, true, MLP_EPI_GELU_BWD>(data, b % data.gx, b / data.gx, 0, err);
  } else {
    const int t = (b - nd) % (weight.gx * weight.gy);
    gemm_tile<true, true, MLP_EPI_RED>(weight, t % weight.gx, t / weight.gx,
                                       (b - nd) / (weight.gx * weight.gy), err);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

// rows x cols BF16, row-major; boxes of 64 columns (128 bytes) x box_rows.
bool map_bf16(CUtensorMap* map, const void* ptr, int64_t rows, int64_t cols, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)GM_BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)ptr, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_job(Job& j, bool amn, const void* A, int64_t M, bool bmn, const void* B, int N, int64_t K,
              int slices, const MlpEpi& epi) {
  if (K <= 0 || K % GM_BK != 0 || N % 64 != 0) return false;
  j.M = M;
  j.N = N;
  j.K = (int)K;
  j.gx = (int)((M + GM_TILE - 1) / GM_TILE);
  j.gy = (N + GM_TILE - 1) / GM_TILE;
  j.gz = slices;
  j.epi = epi;
  return (amn ? map_bf16(&j.A, A, K, M, GM_BK) : map_bf16(&j.A, A, M, K, GM_TILE)) &&
         (bmn ? map_bf16(&j.B, B, K, N, GM_BK) : map_bf16(&j.B, B, N, K, GM_TILE));
}

// Programmatic dependent launch: the kernel's barriers, TMEM and launch latency
// overlap the previous kernel of the stream; it waits for that one's results
// (griddepcontrol.wait) before it touches global memory.
template <typename... Args>
cudaError_t launch_dependent(void (*kern)(Args...), unsigned grid, unsigned threads, size_t smem,
                             cudaStream_t st, Args... args) {
  if (smem > 0) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <bool AMN, bool BMN, int OP>
cudaError_t launch_gemm(const void* A, int64_t M, const void* B, int N, int64_t K, int slices,
                        const MlpEpi& epi, int* err, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  Job j;
  if (!make_job(j, AMN, A, M, BMN, B, N, K, slices, epi)) return cudaErrorInvalidValue;
  return launch_dependent(gemm_bf16_kernel<AMN, BMN, OP>, (unsigned)(j.gx * j.gy * j.gz), GM_THREADS,
                          GM_SMEM, st, j, err);
}

// Slices of a weight gradient's contraction: few output tiles, a long contraction,
// so split it until the tiles fill `ctas`, at least two stages per slice.
int weight_slices(int64_t B, int Nout, int Nin, int ctas) {
  const int64_t tiles = (int64_t)((Nout + GM_TILE - 1) / GM_TILE) * ((Nin + GM_TILE - 1) / GM_TILE);
  const int64_t nk = B / GM_BK;
  int64_t per = (tiles * nk + ctas - 1) / ctas;
  if (per < 2) per = 2;
  return (int)((nk + per - 1) / per);
}

// rows of Y (FP32, p wide; selected by idx when given) -> BF16 rows pk wide, and
// their support slots (-1 padded to 16) when sup is given; and clears zero_len
// floats at zero (the gradients of the step).
__global__ void gather_rows_kernel(const float* __restrict__ Y, int p, int pk,
                                   const int64_t* __restrict__ idx, int64_t B,
                                   const int32_t* __restrict__ sup_in, int s,
                                   __nv_bfloat16* __restrict__ X, int32_t* __restrict__ sup_out,
                                   float4* __restrict__ zero, int64_t zero_len4) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t q = e; q < zero_len4; q += (int64_t)gridDim.x * blockDim.x)
    zero[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (e >= B * pk) return;
  const int64_t b = e / pk;
  const int c = (int)(e - b * pk);
  const int64_t r = idx ? idx[b] : b;
  X[e] = __float2bfloat16_rn(c < p ? Y[r * p + c] : 0.f);
  if (sup_in && c < 16) sup_out[b * 16 + c] = c < s ? sup_in[r * s + c] : -1;
}

__global__ void f32_to_bf16_kernel(const float* __restrict__ in, int64_t count,
                                   __nv_bfloat16* __restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < count) out[e] = __float2bfloat16_rn(in[e]);
}

// Adam (Kingma & Ba) on FP32 master weights; refreshes the BF16 copy.
__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t count, float lr, float b1, float b2,
                            float eps, float c1, float c2, __nv_bfloat16* __restrict__ wbf) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= count) return;
  const float gg = g[e];
  const float mm = b1 * m[e] + (1.f - b1) * gg;
  const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
  m[e] = mm;
  v[e] = vv;
  const float ww = w[e] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  w[e] = ww;
  if (wbf) wbf[e] = __float2bfloat16_rn(ww);
}

__device__ __forceinline__ float topk_value(const __nv_bfloat16* z, int64_t o) {
  return __bfloat162float(z[o]);
}
__device__ __forceinline__ float topk_value(const float* z, int64_t o) { return fabsf(z[o]); }

// Top-K of each row of n values (one warp per row, row i at z + i * ld), indices
// ascending: the proposer's logits (BF16), or |correlations| (FP32 rows of
// D^T y, the network-free proposer).
template <int NT, typename T>
__global__ void topk_kernel(const T* __restrict__ z, int64_t ld, int64_t m, int n, int K,
                            int32_t* __restrict__ cand) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= m) return;
  float v[NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    const int j = 32 * t + lane;
    v[t] = j < n ? topk_value(z, i * ld + j) : -INFINITY;
  }
  int mine = -1;  // lane k < K: the k-th pick
  for (int k = 0; k < K; ++k) {
    float bv = -INFINITY;
    int bt = 0;
#pragma unroll
    for (int t = 0; t < NT; ++t)
      if (v[t] > bv) {
        bv = v[t];
        bt = t;
      }
    int bj = 32 * bt + lane;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
      if (ov > bv || (ov == bv && oj < bj)) {
        bv = ov;
        bj = oj;
      }
    }
    if (lane == k) mine = bj;
    if ((bj & 31) == lane) {
#pragma unroll
      for (int t = 0; t < NT; ++t)
        if (t == (bj >> 5)) v[t] = -INFINITY;
    }
  }
  // ascending order of the K picks
  int rank = 0;
  for (int q = 0; q < K; ++q) {
    const int o = __shfl_sync(0xffffffffu, mine, q);
    if (lane < K && o < mine) ++rank;
  }
  if (lane < K) cand[i * K + rank] = mine;
}

}  // namespace

bool mlp_gemm_supported() { return encode_fn() != nullptr; }

cudaError_t mlp_forward(const void* A, int64_t M, const void* W, int N, int K, int op,
                        const MlpEpi& epi, int* err, cudaStream_t st) {
  switch (op) {
    case MLP_EPI_GELU_FWD: return launch_gemm<false, false, MLP_EPI_GELU_FWD>(A, M, W, N, K, 1, epi, err, st);
    case MLP_EPI_LOGITS: return launch_gemm<false, false, MLP_EPI_LOGITS>(A, M, W, N, K, 1, epi, err, st);
    case MLP_EPI_BCE: return launch_gemm<false, false, MLP_EPI_BCE>(A, M, W, N, K, 1, epi, err, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t mlp_backward(const void* dY, int64_t B, const void* W, int Nout, int Nin, const MlpEpi& epi,
                         const void* X, float* dW, int* err, cudaStream_t st) {
  Job d, w;
  MlpEpi ew{};
  ew.out_f32 = dW;
  ew.ldc = Nin;
  if (!make_job(d, false, dY, B, true, W, Nin, Nout, 1, epi)) return cudaErrorInvalidValue;
  int room = 2 * num_sms() - d.gx * d.gy;  // CTAs beside the input gradient's (at least one per SM)
  if (room < num_sms()) room = num_sms();
  if (!make_job(w, true, dY, Nout, true, X, Nin, B, weight_slices(B, Nout, Nin, room), ew))
    return cudaErrorInvalidValue;
  return launch_dependent(gemm_backward_kernel, (unsigned)(d.gx * d.gy + w.gx * w.gy * w.gz), GM_THREADS,
                          GM_SMEM, st, d, w, err);
}

cudaError_t mlp_backward_weight(const void* dY, const void* X, int64_t B, int Nout, int Nin, float* dW,
                                int* err, cudaStream_t st) {
  MlpEpi epi{};
  epi.out_f32 = dW;
  epi.ldc = Nin;
  return launch_gemm<true, true, MLP_EPI_RED>(dY, Nout, X, Nin, B,
                                              weight_slices(B, Nout, Nin, num_sms()), epi, err, st);
}

cudaError_t mlp_gather(const float* Y, int p, int pk, const int64_t* idx, int64_t B, const int32_t* sup_in,
                       int s, void* X, int32_t* sup_out, float* zero, int64_t zero_len, cudaStream_t st) {
  const int64_t tot = B * pk;
  return launch_dependent(gather_rows_kernel, (unsigned)((tot + 255) / 256), 256u, (size_t)0, st, Y, p, pk,
                          idx, B, sup_in, s, (__nv_bfloat16*)X, sup_out, (float4*)zero, zero_len / 4);
}

cudaError_t mlp_to_bf16(const float* in, int64_t count, void* out, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  f32_to_bf16_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(in, count, (__nv_bfloat16*)out);
  return cudaGetLastError();
}

cudaError_t mlp_adam(float* w, const float* g, float* m, float* v, int64_t count, float lr, int t,
                     void* wbf, cudaStream_t st) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  adam_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(w, g, m, v, count, lr, b1, b2, 1e-8f,
                                                               c1, c2, (__nv_bfloat16*)wbf);
  return cudaGetLastError();
}

cudaError_t mlp_topk(const void* z, int64_t m, int n, int K, int32_t* cand, cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((m + 7) / 8);
  const __nv_bfloat16* zz = (const __nv_bfloat16*)z;
  if (n <= 128) topk_kernel<4><<<blocks, 256, 0, st>>>(zz, n, m, n, K, cand);
  else if (n <= 256) topk_kernel<8><<<blocks, 256, 0, st>>>(zz, n, m, n, K, cand);
  else if (n <= 512) topk_kernel<16><<<blocks, 256, 0, st>>>(zz, n, m, n, K, cand);
  else topk_kernel<32><<<blocks, 256, 0, st>>>(zz, n, m, n, K, cand);
  return cudaGetLastError();
}

cudaError_t topk_abs(const float* A, int64_t lda, int64_t m, int n, int K, int32_t* cand,
                     cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((m + 7) / 8);
  if (n <= 128) topk_kernel<4><<<blocks, 256, 0, st>>>(A, lda, m, n, K, cand);
  else if (n <= 256) topk_kernel<8><<<blocks, 256, 0, st>>>(A, lda, m, n, K, cand);
  else if (n <= 512) topk_kernel<16><<<blocks, 256, 0, st>>>(A, lda, m, n, K, cand);
  else topk_kernel<32><<<blocks, 256, 0, st>>>(A, lda, m, n, K, cand);
  return cudaGetLastError();
}

}  // namespace dlk
