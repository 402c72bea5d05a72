// kuramoto_general.cu -- Eq. 2 with a general coupling matrix K_ij.
//
// The coupling sum is rewritten with sin(x_j - x_i) = sin x_j cos x_i -
// cos x_j sin x_i (the identity behind Eq. 3, applied row by row):
//
//   sum_j K_ij sin(x_j - x_i) = cos x_i P_s[i] - sin x_i P_c[i],
//   P_s = K sin(x),  P_c = K cos(x),
//
// so one SRK2 stage of all R replicas is one GEMM of K (N x N) with the
// 2R columns [sin x_r | cos x_r] plus an elementwise sub-step.  Two forms:
//   SDE_KURAMOTO_GENERAL      BF16 operands on tcgen05, FP32 accumulation in
//                             tensor memory (tc_gemm.cuh)
//   SDE_KURAMOTO_GENERAL_FP32 FP32 operands, FP32 CUDA-core GEMM (the
//                             baseline the tensor-core form is set against)
// Phases are 32-bit fixed-point turns as in kuramoto.cu; the receiving
// oscillator's own sin/cos are always evaluated in FP32 from its phase.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <utility>

#include "kuramoto.h"
#include "kuramoto_internal.h"
#include "philox.cuh"
#include "tc_gemm.cuh"
#include "tc_gemm_sk.cuh"
#include "tma_map.h"

namespace sde {

namespace {

template <typename T>
__device__ __forceinline__ T to_op(float v);
template <>
__device__ __forceinline__ float to_op<float>(float v) {
  return v;
}
template <>
__device__ __forceinline__ __nv_bfloat16 to_op<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// Operand rows [2r] = sin, [2r+1] = cos of every phase.  Grid: (N / 256, R).
template <typename T>
__global__ void kg_operand_kernel(const uint32_t *theta, T *op, int64_t N) {
  const int64_t r = blockIdx.y;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  float s, c;
  sincos_turns(theta[r * N + i], s, c);
  op[(2 * r) * N + i] = to_op<T>(s);
  op[(2 * r + 1) * N + i] = to_op<T>(c);
}

// One SRK2 stage for every (replica, oscillator) from the GEMM output Dt
// (the forms without the fused epilogue): the same per-element update as the
// tensor-core epilogue (tc::stage_group), the next operand written as T.
// Grid: (N / 256, R).
// kStageIlp elements per thread (i, i + 256, ...): every input of the group is
// loaded before any arithmetic, so each thread keeps several loads in flight.
constexpr int kStageIlp = 4;

// The GEMM output at idx: the sum of its `planes` partial sums, plane stride
// `stride` (one plane unless the FP32 GEMM split K).
__device__ __forceinline__ float plane_sum(const float *__restrict__ Dt, int64_t idx, int planes, int64_t stride) {
  float s = Dt[idx];
  for (int p = 1; p < planes; ++p) s += Dt[p * stride + idx];
  return s;
}

template <int STAGE, typename T>
__global__ void __launch_bounds__(256) kg_stage_kernel(const float *__restrict__ Dt, int planes,
                                                       const tc::StageArgs a, T *op_next) {
  const int64_t r = blockIdx.y;
  const int64_t N = a.N;
  const int64_t i0 = (int64_t)blockIdx.x * (256 * kStageIlp) + threadIdx.x;
  const uint2 key = seed_to_key(a.seed);
  uint32_t th[kStageIlp], th_s[kStageIlp];
  float ps[kStageIlp], pc[kStageIlp], om[kStageIlp], psi[kStageIlp], g1[kStageIlp];
  bool ok[kStageIlp];
#pragma unroll
  for (int u = 0; u < kStageIlp; ++u) {
    const int64_t i = i0 + u * 256;
    ok[u] = i < N;
    const int64_t ii = ok[u] ? i : 0;
    const int64_t idx = r * N + ii;
    ps[u] = Dt[(2 * r) * N + ii];
    pc[u] = Dt[(2 * r + 1) * N + ii];
    th[u] = a.theta[idx];
    th_s[u] = STAGE == 0 ? th[u] : a.theta_t[idx];
    om[u] = a.omega[idx];
    g1[u] = STAGE == 1 ? a.g1[idx] : 0.0f;
    psi[u] = (STAGE == 0 && a.fresh) ? 0.0f : tc::psi_plane(a, a.n >> 2, (int)(a.n & 3))[idx];
  }
  // the other planes of the FP32 GEMM's K shares; a loop among the loads above would
  // keep them apart (BF16, 1024 x 64: 0.5 us per stage)
  if (std::is_same<T, float>::value) {
#pragma unroll 4
    for (int p = 1; p < planes; ++p) {
      const float *D = Dt + p * 2 * a.NR;
#pragma unroll
      for (int u = 0; u < kStageIlp; ++u) {
        const int64_t ii = ok[u] ? i0 + u * 256 : 0;
        ps[u] += D[(2 * r) * N + ii];
        pc[u] += D[(2 * r + 1) * N + ii];
      }
    }
  }
#pragma unroll
  for (int u = 0; u < kStageIlp; ++u) {
    if (!ok[u]) continue;
    const int64_t i = i0 + u * 256;
    const int64_t idx = r * N + i;
    if (STAGE == 0 && a.fresh) psi[u] = tc::stage_noise<STAGE>(a, r, i, idx, key);
    const tc::StageOut o = tc::stage_math<STAGE>(a, th_s[u], th[u], om[u], psi[u], g1[u], ps[u], pc[u]);
    tc::stage_store<STAGE>(a, op_next, r, i, idx, o);
  }
}

// Coupling sums alone: out[r][i] = cos x_i Dt[2r][i] - sin x_i Dt[2r+1][i].
__global__ void kg_coupling_kernel(const float *__restrict__ Dt, int planes, const uint32_t *theta, float *out,
                                   int64_t N) {
  const int64_t r = blockIdx.y;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  float s, c;
  sincos_turns(theta[r * N + i], s, c);
  const int64_t stride = 2 * N * gridDim.y;
  out[r * N + i] = c * plane_sum(Dt, (2 * r) * N + i, planes, stride) -
                   s * plane_sum(Dt, (2 * r + 1) * N + i, planes, stride);
}

__global__ void kg_to_bf16_kernel(const float *src, __nv_bfloat16 *dst, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = __float2bfloat16_rn(src[i]);
}

// ---- FP32 CUDA-core GEMM (baseline): Dt[c][i] = sum_j K[i][j] B[c][j] ----
//
// One CTA of 128 threads: 256 rows x 8 TN columns of D over a share of K, 16 x
// TN outputs per thread as packed FP32 pairs along the rows.  K slices of 16
// come into shared memory transposed, by 4-byte asynchronous copies three slices
// deep: no registers hold them on the way, and each copy instruction of a warp
// reads four whole 32-byte sectors.  Each k's fragments are read while the
// previous k is multiplied.  Partial sums of a K split go to planes of Dt and are
// added by the kernel that reads them.
// What bounds it: shared memory returns 128 bytes per cycle to the SM's four
// schedulers, 4 (16 + TN) cycles per k against 16 TN cycles of packed FMAs, so
// the FMA pipe is the limit from TN = 6 up; and how evenly the tiles fill the
// GPU (sgemm_shape).  M x columns x K, us per step of two GEMMs and sub-steps,
// against slices of 8 held in registers on the way (16-byte loads, a row per
// lane): 4000 x 256 x 4000 395 and 488 (44 TFLOP/s), 3992 x 32 x 3992 91 and 138,
// 1000 x 128 x 1000 38 and 56, 1000 x 14 x 1000 27 and 48, 3000 x 200 x 3000 194
// and 210 (8192 x 512 x 8192 1510 us per GEMM, 46 TFLOP/s; 538 us for one GEMM with 128 x 128 tiles of scalar FMAs, which gave 48
// CTAs).  With the columns stored as (b, b) pairs in shared memory its return
// path is at 130 % of the FMA time; slices of 16 through registers spilled.
constexpr int SG_BM = 256, SG_BK = 16, SG_THREADS = 128, SG_TM = 16, SG_STAGES = 3;

struct SgemmShape {
  int tn = 0;     // columns per thread
  int split = 1;  // K shares (planes of Dt)
  int kshare = 0; // K per share, a multiple of SG_BK
};

// Columns of a B slice in shared memory: the swizzle stays within 32.
__host__ __device__ constexpr int sg_cols(int tn) { return (8 * tn + 31) / 32 * 32; }
constexpr int sg_smem_bytes(int tn) { return SG_STAGES * SG_BK * (SG_BM + sg_cols(tn)) * 4; }

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Four bytes, zero where `bytes` is 0.
__device__ __forceinline__ void copy4_async(uint32_t dst, const float *src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

template <int TN>
__global__ void __launch_bounds__(SG_THREADS, TN <= 7 ? 2 : 1)
    sgemm_nt_kernel(const float *__restrict__ A, const float *__restrict__ B, float *__restrict__ Dt, int M, int Ncols,
                    int Kdim, int kshare) {
  constexpr int BN = 8 * TN;
  constexpr int BS = sg_cols(TN);
  constexpr int NA = SG_BM / 16, NB = (BN + 15) / 16;  // rows (columns) per thread, 16 apart
  extern __shared__ __align__(16) float sg_smem[];
  auto As = reinterpret_cast<float (*)[SG_BK][SG_BM]>(sg_smem);
  auto Bs = reinterpret_cast<float (*)[SG_BK][BS]>(sg_smem + SG_STAGES * SG_BK * SG_BM);
  const int tid = threadIdx.x;
  const int tx = tid & 7, ty = tid >> 3;  // columns tx + 8 j; rows 64 i + 4 ty .. + 3, i = 0 .. 3
  const int m0 = blockIdx.x * SG_BM, n0 = blockIdx.y * BN;
  const int kb = blockIdx.z * kshare, ke = min(kb + kshare, Kdim);
  // A copy instruction of a warp: a 32-byte sector of each of four rows.  Element
  // (k, r) lies at [k][r ^ 4 (k mod 8)]: the 32 words on 32 banks, and four rows
  // of one k still together.  Rows past the end repeat the last one (their
  // outputs are not stored).
  const int lk = tid & 7, lr = tid >> 3;
  const float *Ab = A + (size_t)m0 * Kdim + lk, *Bb = B + (size_t)n0 * Kdim + lk;
  uint32_t oa[NA], ob[NB];
#pragma unroll
  for (int q = 0; q < NA; ++q) oa[q] = (uint32_t)min(lr + 16 * q, M - 1 - m0) * (uint32_t)Kdim;
#pragma unroll
  for (int q = 0; q < NB; ++q) ob[q] = (uint32_t)min(lr + 16 * q, Ncols - 1 - n0) * (uint32_t)Kdim;
  // lr ^ 4 lk, its bit 4 (of lk alone) applied to 16 q
  const int low = (lr ^ (4 * lk)) & 15, high = lk >> 2;
  const uint32_t da = smem_addr(&As[0][lk][low]), db = smem_addr(&Bs[0][lk][low]);
  // Kdim and kshare are multiples of 8: eight k's lie wholly inside the share or
  // are zero
  auto load = [&](int k0, int stage) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = k0 + 8 * h, bytes = k < ke ? 4 : 0;
      const int ks = k < ke ? k : kb;
      const uint32_t sa = da + (uint32_t)(stage * SG_BK + 8 * h) * (SG_BM * 4);
      const uint32_t sb = db + (uint32_t)(stage * SG_BK + 8 * h) * (BS * 4);
#pragma unroll
      for (int q = 0; q < NA; ++q) copy4_async(sa + 64u * (uint32_t)(q ^ high), Ab + ks + oa[q], bytes);
#pragma unroll
      for (int q = 0; q < NB; ++q)
        if (BN % 16 == 0 || lr + 16 * q < BN) copy4_async(sb + 64u * (uint32_t)(q ^ high), Bb + ks + ob[q], bytes);
    }
  };
  float2 acc[SG_TM / 2][TN];
#pragma unroll
  for (int i = 0; i < SG_TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int q = 0; q + 1 < SG_STAGES; ++q) {
    if (kb + q * SG_BK < ke) load(kb + q * SG_BK, q);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int stage = 0;
  for (int k0 = kb; k0 < ke; k0 += SG_BK) {
    asm volatile("cp.async.wait_group %0;" ::"n"(SG_STAGES - 2) : "memory");
    __syncthreads();  // this slice is there, and nobody reads the one before it any more
    const int next = k0 + (SG_STAGES - 1) * SG_BK;
    if (next < ke) load(next, stage == 0 ? SG_STAGES - 1 : stage - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    float4 fa[2][4];
    float fb[2][TN];
    auto frag = [&](int q, int kk) {
      const int r = (4 * ty) ^ (4 * (kk & 7));
#pragma unroll
      for (int i = 0; i < 4; ++i) fa[q][i] = *(const float4 *)&As[stage][kk][64 * i + r];
#pragma unroll
      for (int j = 0; j < TN; ++j) fb[q][j] = Bs[stage][kk][(tx ^ (4 * (kk & 1))) + 8 * (j ^ ((kk & 7) >> 1))];
    };
    frag(0, 0);
#pragma unroll
    for (int kk = 0; kk < SG_BK; ++kk) {
      if (kk + 1 < SG_BK) frag((kk + 1) & 1, kk + 1);
      const float4 (&a)[4] = fa[kk & 1];
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const float2 b = make_float2(fb[kk & 1][j], fb[kk & 1][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[2 * i][j] = __ffma2_rn(make_float2(a[i].x, a[i].y), b, acc[2 * i][j]);
          acc[2 * i + 1][j] = __ffma2_rn(make_float2(a[i].z, a[i].w), b, acc[2 * i + 1][j]);
        }
      }
    }
    stage = stage + 1 == SG_STAGES ? 0 : stage + 1;
  }
  float *D = Dt + (size_t)blockIdx.z * Ncols * M;
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int col = n0 + tx + 8 * j;
    if (col >= Ncols) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + 64 * i + 4 * ty;  // M is a multiple of 8
      if (m < M)
        *(float4 *)(D + (size_t)col * M + m) =
            make_float4(acc[2 * i][j].x, acc[2 * i][j].y, acc[2 * i + 1][j].x, acc[2 * i + 1][j].y);
    }
  }
}

constexpr int kSgemmTn[] = {1, 2, 3, 5, 7, 8};
constexpr int kSgemmMaxSplit = 16;

// Columns per thread and K shares of the FP32 GEMM for M x Ncols outputs, by
// the cycles of the busiest SM: its tile shares times the cycles per k (the
// larger of 16 TN of packed FMAs and 4 (16 + TN) of shared-memory return, and
// a sixth more where a single share leaves one warp per scheduler); a share
// costs about 24 more k's for its prologue and epilogue, and every plane of
// partial sums its write and read (8 bytes per output at 24 bytes per cycle
// and SM).
SgemmShape sgemm_shape(int64_t M, int64_t Ncols, int64_t Kdim, int sm_count) {
  SgemmShape best;
  double t_best = 0.0;
  for (int tn : kSgemmTn) {
    const int64_t tiles = ((M + SG_BM - 1) / SG_BM) * ((Ncols + 8 * tn - 1) / (8 * tn));
    for (int s = 1; s <= kSgemmMaxSplit; ++s) {
      const int64_t share = ((Kdim + s - 1) / s + SG_BK - 1) / SG_BK * SG_BK;
      if (s > 1 && (share < 64 || share * (s - 1) >= Kdim || (s - 1) * M * Ncols * 4 > (256ll << 20))) break;
      const double per_sm = (double)((tiles * s + sm_count - 1) / sm_count);
      const double cyc = std::max(16.0 * tn, 4.0 * (SG_TM + tn)) * (tiles * s <= sm_count ? 1.17 : 1.0);
      const double t = per_sm * cyc * (double)(share + 24) +
                       (double)s * (double)M * (double)Ncols * 8.0 / (24.0 * sm_count);
      if (best.tn == 0 || t < t_best) {
        best.tn = tn;
        best.split = s;
        best.kshare = (int)share;
        t_best = t;
      }
    }
  }
  return best;
}

template <int TN>
cudaError_t launch_sgemm_tn(const SgemmShape &p, const float *A, const float *B, float *Dt, int M, int Ncols, int Kdim,
                            bool configure, cudaStream_t s) {
  if (configure)
    return cudaFuncSetAttribute(sgemm_nt_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, sg_smem_bytes(TN));
  const dim3 grid((M + SG_BM - 1) / SG_BM, (Ncols + 8 * TN - 1) / (8 * TN), p.split);
  sgemm_nt_kernel<TN><<<grid, SG_THREADS, sg_smem_bytes(TN), s>>>(A, B, Dt, M, Ncols, Kdim, p.kshare);
  return cudaGetLastError();
}

// configure: the kernel's shared memory instead of a launch.
cudaError_t launch_sgemm(const SgemmShape &p, const float *A, const float *B, float *Dt, int M, int Ncols, int Kdim,
                         cudaStream_t s, bool configure = false) {
  switch (p.tn) {
    case 1: return launch_sgemm_tn<1>(p, A, B, Dt, M, Ncols, Kdim, configure, s);
    case 2: return launch_sgemm_tn<2>(p, A, B, Dt, M, Ncols, Kdim, configure, s);
    case 3: return launch_sgemm_tn<3>(p, A, B, Dt, M, Ncols, Kdim, configure, s);
    case 5: return launch_sgemm_tn<5>(p, A, B, Dt, M, Ncols, Kdim, configure, s);
    case 7: return launch_sgemm_tn<7>(p, A, B, Dt, M, Ncols, Kdim, configure, s);
    case 8: return launch_sgemm_tn<8>(p, A, B, Dt, M, Ncols, Kdim, configure, s);
    default: return cudaErrorInvalidValue;
  }
}

constexpr int64_t kTimedStepStride = 8;

int grid_for(int64_t n, int sm_count) {
  const int64_t b = (n + 255) / 256;
  return (int)std::min<int64_t>(b, (int64_t)sm_count * 16);
}

// 2D BF16 tensor map: rows x cols (cols contiguous), box of box_rows x 64.
sde_status make_map(CUtensorMap *map, const void *base, int64_t rows, int64_t cols, int box_rows) {
  return make_map_bf16(map, base, rows, cols, box_rows);
}

struct GemmPlan {
  CUtensorMap mapK;
  CUtensorMap mapOp[2];  // box of bn rows (one CTA's tile)
  CUtensorMap mapOpHalf[2];  // box of 128 rows (one CTA's half of a pair tile)
  SgemmShape sg;      // FP32 GEMM
  int bn = 0;
  bool pair = false;  // CTA-pair GEMM (tc_gemm2_bf16_kernel)
  tc::EpiMaps em;     // pair GEMM: the SRK2 state its fused epilogue loads by TMA
  float *omega_copy = nullptr;  // [R][N] the run's omega (a fixed address for em.omega)
  // stream-K GEMM (tc_gemm_sk_bf16_kernel): sk_P CTAs, 0 = whole tiles
  int sk_P = 0;
  float *ws = nullptr;        // [sk_P][256][128] partial sums
  uint32_t *flags = nullptr;  // [sk_P] epoch of the partial in each slot
  uint32_t epoch = 0;
};

bool is_tc(const KuramotoCtx *k) { return k->model == SDE_KURAMOTO_GENERAL; }

void *op_buf(KuramotoCtx *k, int which) {
  if (is_tc(k)) return (void *)(k->Bt + (size_t)which * 2 * k->R * k->N);
  return (void *)(k->Bt32 + (size_t)which * 2 * k->R * k->N);
}

tc::StageArgs stage_args(KuramotoCtx *k, int next, const float *omega, int64_t n, int64_t run_begin) {
  const double inv2pi = 0.15915494309189533577;
  tc::StageArgs a{};
  a.theta = k->theta;
  a.theta_t = k->theta_t;
  a.g1 = k->g1;
  a.psi4 = k->psi4;
  a.omega = omega;
  a.op_next = (next >= 0 && is_tc(k)) ? (__nv_bfloat16 *)op_buf(k, next) : nullptr;
  a.N = k->N;
  a.NR = k->N * k->R;
  a.n = n;
  a.fresh = ((n & 3) == 0 || n == run_begin) ? 1 : 0;
  a.pre_slice = -1;
  a.wscale = (float)(k->dt * inv2pi);
  a.kc = (float)(k->dt * inv2pi);
  a.kh = (float)(0.5 * k->dt * inv2pi);
  a.sc = (float)(sqrt(2.0 * k->D * k->dt) * inv2pi);
  a.seed = k->seed;
  return a;
}

// Launch with programmatic stream serialization: the GEMM's prologue
// (barrier set-up, tensor-memory allocation) may start while the previous
// kernel of the stream finishes; the kernel waits (griddepcontrol.wait)
// before it reads anything that kernel wrote.
template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                             Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <int BN, int EPI>
cudaError_t launch_tc(KuramotoCtx *k, int which, const tc::StageArgs &sa, cudaStream_t s) {
  GemmPlan *g = (GemmPlan *)k->gemm_plan;
  const int M = (int)k->N, Ncols = (int)(2 * k->R), Kdim = (int)k->N;
  return launch_dependent(tc::tc_gemm_bf16_kernel<BN, EPI>, dim3(M / tc::BM, Ncols / BN), tc::EpiThreads<EPI>::value,
                          tc::Shape<BN>::SMEM_BYTES, s, g->mapK, g->mapOp[which], k->P, M, Kdim, k->err, sa,
                          k->wait_ns);
}

template <int EPI>
cudaError_t launch_tc2(KuramotoCtx *k, int which, const tc::StageArgs &sa, cudaStream_t s) {
  GemmPlan *g = (GemmPlan *)k->gemm_plan;
  const int M = (int)k->N, Ncols = (int)(2 * k->R), Kdim = (int)k->N;
  // clusters of two CTAs along x (the kernel's compile-time cluster shape)
  return launch_dependent(tc::tc_gemm2_bf16_kernel<EPI>, dim3(M / tc::BM, Ncols / tc::BN2),
                          tc::EpiThreads<EPI>::value, tc::SMEM2_BYTES, s, g->mapK, g->mapOpHalf[which], g->em, k->P,
                          M, Kdim, k->err, sa, k->wait_ns);
}

template <int EPI>
cudaError_t launch_sk(KuramotoCtx *k, int which, const tc::StageArgs &sa, cudaStream_t s) {
  GemmPlan *g = (GemmPlan *)k->gemm_plan;
  const int M = (int)k->N, Ncols = (int)(2 * k->R), Kdim = (int)k->N;
  const int tiles_n = Ncols / tc::SK_BN;
  const int64_t T = (int64_t)(M / tc::BM) * tiles_n * (Kdim / tc::BK);
  if (++g->epoch == 0) g->epoch = 1;  // flags start at 0: epoch 0 never marks a partial
  return launch_dependent(tc::tc_gemm_sk_bf16_kernel<EPI>, dim3((unsigned)g->sk_P), tc::SK_THREADS,
                          tc::SK_SMEM_BYTES, s, g->mapK, g->mapOp[which], k->P, M, Kdim, tiles_n, T, g->ws,
                          g->flags, g->epoch, k->err, sa, k->wait_ns);
}

// GEMM reading operand buffer `which`; epi = EPI_STORE_D writes Dt, the stage
// epilogues apply the SRK2 sub-step and write operand buffer 1 - which.
cudaError_t launch_gemm(KuramotoCtx *k, int which, cudaStream_t s, int epi = tc::EPI_STORE_D,
                        const float *omega = nullptr, int64_t n = 0, int64_t run_begin = 0) {
  const int M = (int)k->N, Ncols = (int)(2 * k->R), Kdim = (int)k->N;
  if (is_tc(k)) {
    GemmPlan *g = (GemmPlan *)k->gemm_plan;
    tc::StageArgs sa = stage_args(k, epi == tc::EPI_STORE_D ? -1 : 1 - which, omega, n, run_begin);
    if (g->pair && g->sk_P == 0 && epi != tc::EPI_STORE_D) {
      // the fused CTA-pair GEMMs of a Philox block draw the next block ahead,
      // a slice per launch; a block whose predecessor lay wholly in this run
      // is not drawn again at its first step
      const int64_t block = n >> 2;
      if (4 * block >= run_begin) sa.pre_slice = (int32_t)(2 * (n & 3) + (epi == tc::EPI_STAGE1 ? 1 : 0));
      if (block >= 1 && 4 * (block - 1) >= run_begin && n != run_begin) sa.fresh = 0;
    }
    if (g->sk_P > 0) {
      if (epi == tc::EPI_STAGE0) return launch_sk<tc::EPI_STAGE0>(k, which, sa, s);
      if (epi == tc::EPI_STAGE1) return launch_sk<tc::EPI_STAGE1>(k, which, sa, s);
      return launch_sk<tc::EPI_STORE_D>(k, which, sa, s);
    }
    if (g->pair) {
      if (epi == tc::EPI_STAGE0) return launch_tc2<tc::EPI_STAGE0>(k, which, sa, s);
      if (epi == tc::EPI_STAGE1) return launch_tc2<tc::EPI_STAGE1>(k, which, sa, s);
      return launch_tc2<tc::EPI_STORE_D>(k, which, sa, s);
    }
    if (g->bn == 256) {
      if (epi == tc::EPI_STAGE0) return launch_tc<256, tc::EPI_STAGE0>(k, which, sa, s);
      if (epi == tc::EPI_STAGE1) return launch_tc<256, tc::EPI_STAGE1>(k, which, sa, s);
      return launch_tc<256, tc::EPI_STORE_D>(k, which, sa, s);
    }
    if (epi == tc::EPI_STAGE0) return launch_tc<128, tc::EPI_STAGE0>(k, which, sa, s);
    if (epi == tc::EPI_STAGE1) return launch_tc<128, tc::EPI_STAGE1>(k, which, sa, s);
    return launch_tc<128, tc::EPI_STORE_D>(k, which, sa, s);
  } else {
    return launch_sgemm(((GemmPlan *)k->gemm_plan)->sg, k->Kf32, (const float *)op_buf(k, which), k->P, M, Ncols, Kdim,
                        s);
  }
}

dim3 grid_nr(const KuramotoCtx *k) { return dim3((unsigned)((k->N + 255) / 256), (unsigned)k->R); }
dim3 grid_stage(const KuramotoCtx *k) {
  return dim3((unsigned)((k->N + 256 * kStageIlp - 1) / (256 * kStageIlp)), (unsigned)k->R);
}

cudaError_t launch_operand(KuramotoCtx *k, int which, cudaStream_t s) {
  if (is_tc(k))
    kg_operand_kernel<__nv_bfloat16><<<grid_nr(k), 256, 0, s>>>(k->theta, (__nv_bfloat16 *)op_buf(k, which),
                                                                 k->N);
  else
    kg_operand_kernel<float><<<grid_nr(k), 256, 0, s>>>(k->theta, (float *)op_buf(k, which), k->N);
  return cudaGetLastError();
}

template <int STAGE>
cudaError_t launch_stage(KuramotoCtx *k, int next, const float *omega, int64_t n, int64_t run_begin,
                         cudaStream_t s) {
  const tc::StageArgs a = stage_args(k, next, omega, n, run_begin);
  if (is_tc(k))
    kg_stage_kernel<STAGE, __nv_bfloat16>
        <<<grid_stage(k), 256, 0, s>>>(k->P, 1, a, (__nv_bfloat16 *)op_buf(k, next));
  else
    kg_stage_kernel<STAGE, float><<<grid_stage(k), 256, 0, s>>>(k->P, ((GemmPlan *)k->gemm_plan)->sg.split, a,
                                                               (float *)op_buf(k, next));
  return cudaGetLastError();
}

}  // namespace

sde_status kuramoto_general_alloc(KuramotoCtx *k) {
  const size_t NR = (size_t)k->N * (size_t)k->R;
  const size_t NN = (size_t)k->N * (size_t)k->N;
  if (is_tc(k)) {
    if (k->N % tc::BM != 0 || (2 * k->R) % 128 != 0) {
      set_error("invalid argument: the tensor-core form needs n_osc % 128 == 0 and n_replicas % 64 == 0 "
                "(use SDE_KURAMOTO_GENERAL_FP32 for other sizes)");
      return SDE_ERR_INVALID_ARG;
    }
  }
  if (!is_tc(k) && k->N % 8 != 0) {
    set_error("invalid argument: the FP32 general-coupling form needs n_osc % 8 == 0");
    return SDE_ERR_INVALID_ARG;
  }
  cudaError_t e;
  if ((e = device_alloc((void **)&k->theta_t, NR * 4)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if ((e = device_alloc((void **)&k->g1, NR * 4)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  GemmPlan *g = new GemmPlan();
  k->gemm_plan = g;
  if (!is_tc(k)) g->sg = sgemm_shape(k->N, 2 * k->R, k->N, k->sm_count);
  if ((e = device_alloc((void **)&k->P, NR * 2 * 4 * g->sg.split)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if ((e = device_alloc((void **)&k->psi4, NR * 8 * sizeof(float))) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if (is_tc(k)) {
    if ((e = device_alloc((void **)&k->Kbf16, NN * 2)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
    if ((e = device_alloc((void **)&k->Bt, NR * 2 * 2 * 2)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
    g->bn = (2 * k->R) % 256 == 0 ? 256 : 128;
    g->pair = k->N % 256 == 0 && (2 * k->R) % tc::BN2 == 0 && !(k->flags & SDE_FLAG_GEMM_SINGLE_CTA);
    sde_status st = make_map(&g->mapK, k->Kbf16, k->N, k->N, tc::BM);
    if (st != SDE_OK) return st;
    for (int w = 0; w < 2; ++w) {
      st = make_map(&g->mapOp[w], op_buf(k, w), 2 * k->R, k->N, g->bn);
      if (st != SDE_OK) return st;
      st = make_map(&g->mapOpHalf[w], op_buf(k, w), 2 * k->R, k->N, tc::BH2);
      if (st != SDE_OK) return st;
    }
    if (g->pair) {
      if ((e = device_alloc((void **)&g->omega_copy, NR * 4)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
      const struct {
        CUtensorMap *map;
        const void *base;
        int64_t planes;
      } arrays[] = {{&g->em.theta, k->theta, 1},   {&g->em.theta_t, k->theta_t, 1}, {&g->em.g1, k->g1, 1},
                    {&g->em.omega, g->omega_copy, 1}, {&g->em.psi, k->psi4, 8}};
      for (const auto &a : arrays) {
        st = make_map_w32(a.map, a.base, a.planes, k->R, k->N, tc::EQ_REPS, tc::BM);
        if (st != SDE_OK) return st;
      }
    }
    const void *kernels[] = {
        (const void *)tc::tc_gemm_bf16_kernel<256, tc::EPI_STORE_D>,
        (const void *)tc::tc_gemm_bf16_kernel<256, tc::EPI_STAGE0>,
        (const void *)tc::tc_gemm_bf16_kernel<256, tc::EPI_STAGE1>,
        (const void *)tc::tc_gemm_bf16_kernel<128, tc::EPI_STORE_D>,
        (const void *)tc::tc_gemm_bf16_kernel<128, tc::EPI_STAGE0>,
        (const void *)tc::tc_gemm_bf16_kernel<128, tc::EPI_STAGE1>};
    for (int q = 0; q < 6; ++q)
      if ((e = cudaFuncSetAttribute(kernels[q], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    q < 3 ? tc::Shape<256>::SMEM_BYTES : tc::Shape<128>::SMEM_BYTES)) !=
          cudaSuccess)
        return cuda_fail(e, "cudaFuncSetAttribute");
    const void *kernels2[] = {(const void *)tc::tc_gemm2_bf16_kernel<tc::EPI_STORE_D>,
                              (const void *)tc::tc_gemm2_bf16_kernel<tc::EPI_STAGE0>,
                              (const void *)tc::tc_gemm2_bf16_kernel<tc::EPI_STAGE1>};
    for (int q = 0; q < 3; ++q)
      if ((e = cudaFuncSetAttribute(kernels2[q], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    tc::SMEM2_BYTES)) != cudaSuccess)
        return cuda_fail(e, "cudaFuncSetAttribute");
    // Stream-K on request (SDE_FLAG_GEMM_STREAM_K): as many CTAs as can be
    // resident at once (every CTA must be, for the heads' waits to end), each
    // with at least SK_MIN_UNITS K slices, where that is more CTAs than tiles.
    if (g->bn == 256 && (k->flags & SDE_FLAG_GEMM_STREAM_K)) {
      const void *kernels3[] = {(const void *)tc::tc_gemm_sk_bf16_kernel<tc::EPI_STORE_D>,
                                (const void *)tc::tc_gemm_sk_bf16_kernel<tc::EPI_STAGE0>,
                                (const void *)tc::tc_gemm_sk_bf16_kernel<tc::EPI_STAGE1>};
      int resident = 1 << 30;
      for (int q = 0; q < 3; ++q) {
        if ((e = cudaFuncSetAttribute(kernels3[q], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      tc::SK_SMEM_BYTES)) != cudaSuccess)
          return cuda_fail(e, "cudaFuncSetAttribute");
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernels3[q], tc::SK_THREADS,
                                                               tc::SK_SMEM_BYTES)) != cudaSuccess)
          return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
        resident = std::min(resident, per_sm * k->sm_count);
      }
      const int64_t tiles = (k->N / tc::BM) * (2 * k->R / tc::SK_BN);
      const int64_t T = tiles * (k->N / tc::BK);
      const int64_t P = std::min<int64_t>(resident, T / tc::SK_MIN_UNITS);
      if (P > tiles) {
        g->sk_P = (int)P;
        if ((e = device_alloc((void **)&g->ws, (size_t)P * tc::SK_BN * tc::BM * sizeof(float))) != cudaSuccess)
          return cuda_fail(e, "cudaMalloc");
        if ((e = device_alloc((void **)&g->flags, (size_t)P * sizeof(uint32_t))) != cudaSuccess)
          return cuda_fail(e, "cudaMalloc");
        if ((e = cudaMemset(g->flags, 0, (size_t)P * sizeof(uint32_t))) != cudaSuccess)
          return cuda_fail(e, "cudaMemset");
      }
    }
  } else {
    if ((e = launch_sgemm(g->sg, nullptr, nullptr, nullptr, 0, 0, 0, nullptr, true)) != cudaSuccess)
      return cuda_fail(e, "cudaFuncSetAttribute(sgemm_nt_kernel)");
    if ((e = device_alloc((void **)&k->Kf32, NN * 4)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
    if ((e = device_alloc((void **)&k->Bt32, NR * 2 * 4 * 2)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  }
  k->block = is_tc(k) ? tc::THREADS : SG_THREADS;
  k->opt = is_tc(k) ? g->bn : 8 * g->sg.tn;
  if (is_tc(k)) {
    const GemmPlan *g = (const GemmPlan *)k->gemm_plan;
    // CTAs per GEMM tile (0: stream-K, the split grid's CTA count in opt)
    k->cs = g->sk_P > 0 ? 0 : (g->pair ? 2 : 1);
    if (g->sk_P > 0) k->opt = g->sk_P;
  } else {
    k->cs = 1;
  }
  return SDE_OK;
}

void kuramoto_general_free(KuramotoCtx *k) {
  cudaFree(k->Kf32);
  cudaFree(k->Kbf16);
  cudaFree(k->Bt);
  cudaFree(k->Bt32);
  cudaFree(k->P);
  cudaFree(k->psi4);
  if (k->gemm_plan) {
    cudaFree(((GemmPlan *)k->gemm_plan)->ws);
    cudaFree(((GemmPlan *)k->gemm_plan)->flags);
    cudaFree(((GemmPlan *)k->gemm_plan)->omega_copy);
  }
  delete (GemmPlan *)k->gemm_plan;
  k->gemm_plan = nullptr;
}

sde_status kuramoto_set_coupling(KuramotoCtx *k, const float *K_dev, cudaStream_t s) {
  if (!(k->model == SDE_KURAMOTO_GENERAL || k->model == SDE_KURAMOTO_GENERAL_FP32)) {
    set_error("invalid argument: sde_set_coupling applies to the general-coupling models only");
    return SDE_ERR_INVALID_ARG;
  }
  SDE_CHECK_ARG(K_dev != nullptr, "K is NULL");
  const int64_t NN = k->N * k->N;
  if (is_tc(k)) {
    kg_to_bf16_kernel<<<grid_for(NN, k->sm_count), 256, 0, s>>>(K_dev, k->Kbf16, NN);
    SDE_CUDA_TRY(cudaGetLastError());
  } else {
    SDE_CUDA_TRY(cudaMemcpyAsync(k->Kf32, K_dev, sizeof(float) * NN, cudaMemcpyDeviceToDevice, s));
  }
  k->have_K = true;
  return SDE_OK;
}

sde_status kuramoto_general_run(KuramotoCtx *k, const sde_run_desc *r, cudaStream_t s, double *rbuf) {
  if (!k->have_K) {
    set_error("invalid argument: set the coupling matrix with sde_set_coupling before running");
    return SDE_ERR_INVALID_ARG;
  }
  SDE_CUDA_TRY(launch_operand(k, 0, s));
  // SDE_FLAG_TIME_KERNELS: an event between two GEMMs keeps the second one's
  // prologue from overlapping the first one's end, so the fused form (back
  // to back GEMMs, > 99 % of the loop) is timed as one block over all its
  // launches (the r(t) samples in between included), and the separate form
  // per GEMM launch on every kTimedStepStride-th step
  const bool fused = is_tc(k) && (k->flags & SDE_FLAG_FUSED);
  if (fused && ((GemmPlan *)k->gemm_plan)->pair && r->n_end > r->n_begin)
    SDE_CUDA_TRY(cudaMemcpyAsync(((GemmPlan *)k->gemm_plan)->omega_copy, r->omega_dev,
                                 sizeof(float) * (size_t)k->N * (size_t)k->R, cudaMemcpyDeviceToDevice, s));
  if (fused && r->n_end > r->n_begin) SDE_CUDA_TRY(ktime_begin(k, s));
  int64_t sample = 0;
  for (int64_t n = r->n_begin; n < r->n_end; ++n) {
    if (k->M > 0 && (n - r->n_begin) % k->M == 0) {
      SDE_CUDA_TRY(kur_order_launch(k->theta, k->N, k->R, rbuf + sample * k->R, s));
      ++sample;
    }
    if (fused) {
      // the SRK2 sub-steps run in the GEMM epilogues
      SDE_CUDA_TRY(launch_gemm(k, 0, s, tc::EPI_STAGE0, r->omega_dev, n, r->n_begin));
      SDE_CUDA_TRY(launch_gemm(k, 1, s, tc::EPI_STAGE1, r->omega_dev, n, r->n_begin));
      continue;
    }
    const bool timed = (n - r->n_begin) % kTimedStepStride == 0;
    if (timed) SDE_CUDA_TRY(ktime_begin(k, s));
    SDE_CUDA_TRY(launch_gemm(k, 0, s));
    if (timed) SDE_CUDA_TRY(ktime_end(k, s));
    SDE_CUDA_TRY(launch_stage<0>(k, 1, r->omega_dev, n, r->n_begin, s));
    if (timed) SDE_CUDA_TRY(ktime_begin(k, s));
    SDE_CUDA_TRY(launch_gemm(k, 1, s));
    if (timed) SDE_CUDA_TRY(ktime_end(k, s));
    SDE_CUDA_TRY(launch_stage<1>(k, 0, r->omega_dev, n, r->n_begin, s));
  }
  if (fused && r->n_end > r->n_begin) SDE_CUDA_TRY(ktime_end(k, s, 2 * (r->n_end - r->n_begin)));
  if (k->M > 0) SDE_CUDA_TRY(kur_order_launch(k->theta, k->N, k->R, rbuf + sample * k->R, s));
  return SDE_OK;
}

sde_status kuramoto_general_coupling(KuramotoCtx *k, float *out, cudaStream_t s) {
  if (!k->have_K) {
    set_error("invalid argument: set the coupling matrix with sde_set_coupling first");
    return SDE_ERR_INVALID_ARG;
  }
  SDE_CUDA_TRY(launch_operand(k, 0, s));
  SDE_CUDA_TRY(launch_gemm(k, 0, s));
  kg_coupling_kernel<<<grid_nr(k), 256, 0, s>>>(k->P, ((GemmPlan *)k->gemm_plan)->sg.split, k->theta, out, k->N);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}

}  // namespace sde
