// mlp.cu -- the learned surrogate of <<v>>: an ensemble of multilayer
// perceptrons trained and evaluated by the library's own kernels.
//
// Layer l computes z = h W_l^T + b_l; hidden layers apply SiLU, z / (1 +
// e^-z).  Loss: mean over the batch of (out - y)^2.  Backward: dW_l =
// dZ_l^T h_l, db_l = column sums of dZ_l, dH_{l-1} = dZ_l W_l, dZ_{l-1} =
// dH_{l-1} * SiLU'(z_{l-1}).  Adam (Kingma & Ba, Algorithm 1) on FP32 master
// weights.  Every GEMM reads BF16 operands (weights and activations rounded
// from FP32) and accumulates in FP32; pre-activations are kept in FP32.
//
// Inference (sde_mlp_forward) of width-256 networks with at least two hidden
// layers runs the fused tensor-core kernel of mlp_tc.cuh: the square hidden
// layers as tcgen05 MMAs (M = 128 points, N = 256, K = 256) with the bias,
// SiLU and the output layer in their epilogues.  The training path (forward
// with stored pre-activations, backward, Adam) runs on the CUDA cores, every
// sum over k in ascending order with one FMA per term: about a dozen launches
// per step for all members together (members are a grid dimension):
// 155 us for 4 members of 1024 points, 1.70 ms when each member's layers were
// launched by themselves.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "fp64_math.cuh"
#include "mlp_tc.cuh"
#include "philox.cuh"
#include "tma_map.h"

using sde::cuda_fail;
using sde::set_error;

namespace sde {
namespace {

constexpr uint32_t kTagInit = 6u;  // Philox stream tag of the initial weights

__device__ __forceinline__ float sigmoidf_(float z) { return 1.0f / (1.0f + expf(-z)); }

__device__ __forceinline__ float silu_grad(float acc, float z) {
  const float s = sigmoidf_(z);
  return acc * (s * (1.0f + z * (1.0f - s)));
}

__device__ __forceinline__ float bf16_round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// ---- square layers: C[m][n] = sum_k A(m, k) B(n, k), members along z -------
//
// 64 x 64 outputs per CTA of 128 threads, 8 x 4 per thread as packed FP32
// pairs along m (a packed FMA rounds each half like fmaf, so every output is
// the same chain of FMAs over ascending k as a scalar loop).  K slices of 32
// are staged as FP32 in shared memory, the next slice's global loads (16
// bytes each) in flight during the current slice's FMAs.
// What bounds it: shared memory returns 128 bytes per cycle to the SM's four
// schedulers, 48 cycles per k against 32 of packed FMAs, and its latency with
// one or two warps per scheduler, so the fragments of kF k's are read ahead.
// The members and, for the weight gradients, the layers share a launch
// (grid.z): one member's GEMM fills a tenth of the GPU.  4 members, 1024 points
// each, 256 wide: 22 us a layer forward, 26 us backward, 34 us for the weight
// gradients of both square layers (one member's layer at a time: 17, 27 and 84
// us each).  Measured beside it: 4 x 4 outputs in 256 threads (23, 26, 37 us);
// 8 x 8 (gradients 8 x 4) in 64 threads from BF16 in shared memory, half the
// shared traffic but one warp per scheduler (28, 32, 59 us); these tiles from
// BF16 in shared memory (a step of all launches 8 us longer: the conversions cost
// more than the loads).  Matrix instructions would take 94 us per step, but another
// order of summation flips BF16 roundings of activations and moves the parameters
// by 4e-5 within eight steps.
enum Epi { EPI_FWD = 0, EPI_DSILU = 1, EPI_DW = 2 };

constexpr int TM = 64, TN = 64, TK = 32, GT = 128, TPAD = 4, kF = 2;
constexpr int kMaxLayers = 9;  // n_hidden <= 8

struct GemmArgs {
  int64_t B;        // rows of a member's batch
  int32_t H;        // width of the square layers
  int32_t n_layers; // EPI_DW: layers along z (member-major)
  int64_t rows;     // row stride between members in the activation buffers (= B)
  const void *a[kMaxLayers];             // FWD: h_l; DSILU, DW: dZ_l (FP32 holding BF16 values)
  const __nv_bfloat16 *b[kMaxLayers];    // FWD, DSILU: W_l of the first member; DW: h_l
  int64_t b_member;                      // member stride of b
  const float *bias;                     // FWD, first member
  int64_t p_member;                      // member stride of bias / gradients (parameters per member)
  float *z;                              // FWD: pre-activation out; DSILU: in, overwritten by dZ_{l-1}
  __nv_bfloat16 *h;                      // FWD: SiLU(z) out
  float *grad[kMaxLayers];               // DW: gradient of W_l, first member
};

__device__ __forceinline__ void unpack(const uint4 &v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ void unpack(const uint4 &v, float (&f)[4]) {
  f[0] = __uint_as_float(v.x);
  f[1] = __uint_as_float(v.y);
  f[2] = __uint_as_float(v.z);
  f[3] = __uint_as_float(v.w);
}

// One operand's 64 x 32 slice: TRANS false: rows of `ld` elements with k
// contiguous; true: rows of k with the 64 outputs contiguous.  `limit` bounds
// the row index of the source (batch rows), zero beyond it.
template <typename T, bool TRANS>
struct Slice {
  static constexpr int EV = 16 / (int)sizeof(T);            // elements per 16-byte load
  static constexpr int NV = TM * TK / EV / GT;              // loads per thread
  uint4 v[NV];
  __device__ __forceinline__ void load(const T *src, int64_t ld, int64_t o0, int64_t k0, int64_t limit) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = threadIdx.x + i * GT;
      const int64_t row = TRANS ? k0 + c / (TM / EV) : o0 + (c & (TM - 1));
      const int64_t col = TRANS ? o0 + (c % (TM / EV)) * EV : k0 + (c / TM) * EV;
      v[i] = row < limit ? *reinterpret_cast<const uint4 *>(src + row * ld + col) : make_uint4(0u, 0u, 0u, 0u);
    }
  }
  __device__ __forceinline__ void store(float (*S)[TM + TPAD]) const {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = threadIdx.x + i * GT;
      float f[EV];
      unpack(v[i], f);
      if (TRANS) {
        float *d = &S[c / (TM / EV)][(c % (TM / EV)) * EV];
#pragma unroll
        for (int e = 0; e < EV; e += 4) *reinterpret_cast<float4 *>(d + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
      } else {
#pragma unroll
        for (int e = 0; e < EV; ++e) S[(c / TM) * EV + e][c & (TM - 1)] = f[e];
      }
    }
  }
};

template <int EPI>
__global__ void __launch_bounds__(GT) mlp_gemm_kernel(const GemmArgs g) {
  using TA = typename std::conditional<EPI == EPI_FWD, __nv_bfloat16, float>::type;
  constexpr bool A_T = EPI == EPI_DW, B_T = EPI != EPI_FWD;
  __shared__ __align__(16) float As[2][TK][TM + TPAD];
  __shared__ __align__(16) float Bs[2][TK][TN + TPAD];
  // the small gradients, which need nothing from this launch, may start
  if (EPI == EPI_DW) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int layer = EPI == EPI_DW ? (int)(blockIdx.z % g.n_layers) : 0;
  const int64_t member = EPI == EPI_DW ? blockIdx.z / g.n_layers : blockIdx.z;
  const int64_t m0 = (int64_t)blockIdx.x * TM;
  const int n0 = blockIdx.y * TN;
  const int64_t H = g.H, B = g.B;
  const TA *A = (const TA *)g.a[layer] + member * g.rows * H;
  const __nv_bfloat16 *Bm = g.b[layer] + member * g.b_member;
  const int64_t K = EPI == EPI_DW ? B : H;
  const int64_t a_limit = B, b_limit = EPI == EPI_DW ? B : H;  // both operands of DW run over batch rows
  Slice<TA, A_T> sa;
  Slice<__nv_bfloat16, B_T> sb;
  sa.load(A, H, m0, 0, a_limit);
  sb.load(Bm, H, n0, 0, b_limit);
  sa.store(As[0]);
  sb.store(Bs[0]);
  __syncthreads();
  float4 zv[8];  // EPI_DSILU: the pre-activations, in flight during the slices
  if (EPI == EPI_DSILU) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int64_t m = m0 + (i < 4 ? 0 : 32) + ty * 4 + (i & 3);
      zv[i] = m < B ? *reinterpret_cast<const float4 *>(g.z + (member * g.rows + m) * H + n0 + tx * 4)
                    : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
  }
  float2 acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.0f, 0.0f);
  int buf = 0;
  for (int64_t k0 = 0; k0 < K; k0 += TK) {
    const bool more = k0 + TK < K;
    if (more) {
      sa.load(A, H, m0, k0 + TK, a_limit);
      sb.load(Bm, H, n0, k0 + TK, b_limit);
    }
    // kF k's fragments at a time, read while the previous ones are multiplied
    float4 a0[2][kF], a1[2][kF], b[2][kF];
    auto frag = [&](int q, int k) {
#pragma unroll
      for (int u = 0; u < kF; ++u) {
        a0[q][u] = *reinterpret_cast<const float4 *>(&As[buf][k + u][ty * 4]);
        a1[q][u] = *reinterpret_cast<const float4 *>(&As[buf][k + u][32 + ty * 4]);
        b[q][u] = *reinterpret_cast<const float4 *>(&Bs[buf][k + u][tx * 4]);
      }
    };
    frag(0, 0);
#pragma unroll
    for (int kg = 0; kg < TK / kF; ++kg) {
      const int q = kg & 1;
      if (kg + 1 < TK / kF) frag(q ^ 1, (kg + 1) * kF);
#pragma unroll
      for (int u = 0; u < kF; ++u) {
        const float2 ap[4] = {make_float2(a0[q][u].x, a0[q][u].y), make_float2(a0[q][u].z, a0[q][u].w),
                              make_float2(a1[q][u].x, a1[q][u].y), make_float2(a1[q][u].z, a1[q][u].w)};
        const float bv[4] = {b[q][u].x, b[q][u].y, b[q][u].z, b[q][u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[i][j] = __ffma2_rn(ap[i], make_float2(bv[j], bv[j]), acc[i][j]);
      }
    }
    if (more) {
      buf ^= 1;
      sa.store(As[buf]);
      sb.store(Bs[buf]);
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t m = m0 + (i < 4 ? 0 : 32) + ty * 4 + (i & 3);
    const int n = n0 + tx * 4;
    float c[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) c[j] = (i & 1) ? acc[i / 2][j].y : acc[i / 2][j].x;
    if (EPI == EPI_DW) {
      float *o = g.grad[layer] + member * g.p_member + m * H + n;  // FP32 parameters: 4-byte aligned only
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = c[j];
    } else if (m < B) {
      const int64_t o = (member * g.rows + m) * H + n;
      if (EPI == EPI_FWD) {
        const float *bias = g.bias + member * g.p_member + n;
        __nv_bfloat16 hv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          c[j] += bias[j];
          hv[j] = __float2bfloat16_rn(c[j] * sigmoidf_(c[j]));
        }
        *reinterpret_cast<float4 *>(g.z + o) = make_float4(c[0], c[1], c[2], c[3]);
        *reinterpret_cast<uint2 *>(g.h + o) = *reinterpret_cast<const uint2 *>(hv);
      } else {
        const float4 z = zv[i];
        *reinterpret_cast<float4 *>(g.z + o) =
            make_float4(bf16_round(silu_grad(c[0], z.x)), bf16_round(silu_grad(c[1], z.y)),
                        bf16_round(silu_grad(c[2], z.z)), bf16_round(silu_grad(c[3], z.w)));
      }
    }
  }
}

// ---- layer 0, and the BF16 copies of the parameters ------------------------
//
// The first blocks of each member compute layer 0 (n_in <= 8 inputs: one
// thread per column, kRows0 batch rows per block), the others round the
// member's FP32 parameters to the BF16 operands of the square layers; the two
// do not depend on each other.
constexpr int kRows0 = 16;

struct Layer0Args {
  const float *X;        // [members or 1][B][n_in]
  int64_t x_member;      // member stride of X (0: one batch for all members)
  const float *params;   // first member
  int64_t P, P_bf16;     // parameters per member and the member stride of wbf (a multiple of 8)
  int64_t w0, b0;        // offsets of W_0, b_0
  int64_t B, rows;
  int32_t n_in, H, blocks0;
  float *z;
  __nv_bfloat16 *h, *wbf;
};

__global__ void __launch_bounds__(256) mlp_layer0_kernel(const Layer0Args a) {
  __shared__ float xs[kRows0][8];
  const int64_t member = blockIdx.y;
  const float *pm = a.params + member * a.P;
  if ((int)blockIdx.x >= a.blocks0) {
    const int64_t stride = (int64_t)(gridDim.x - a.blocks0) * 256;
    for (int64_t i = (int64_t)(blockIdx.x - a.blocks0) * 256 + threadIdx.x; i < a.P; i += stride)
      a.wbf[member * a.P_bf16 + i] = __float2bfloat16_rn(pm[i]);
    return;
  }
  const int64_t r0 = (int64_t)blockIdx.x * kRows0;
  const int nr = (int)(a.B - r0 < kRows0 ? a.B - r0 : kRows0);
  for (int i = threadIdx.x; i < nr * a.n_in; i += 256)
    xs[i / a.n_in][i % a.n_in] = bf16_round(a.X[member * a.x_member + r0 * a.n_in + i]);
  __syncthreads();
  for (int n = threadIdx.x; n < a.H; n += 256) {
    float w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = k < a.n_in ? bf16_round(pm[a.w0 + (int64_t)n * a.n_in + k]) : 0.0f;
    const float bias = pm[a.b0 + n];
    for (int r = 0; r < nr; ++r) {
      float acc = 0.0f;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < a.n_in) acc = fmaf(xs[r][k], w[k], acc);
      const float z = acc + bias;
      const int64_t o = (member * a.rows + r0 + r) * a.H + n;
      a.z[o] = z;
      a.h[o] = __float2bfloat16_rn(z * sigmoidf_(z));
    }
  }
}

// ---- output layer, its gradient and the last hidden layer's dZ -------------
//
// 32 batch rows per block: each row's dot product with w_out is one lane's
// chain over ascending k (rows staged in shared memory); training goes on to
// g = 2/B (pred - y) and dZ = g w_out SiLU'(z), which overwrites z.
constexpr int kRowsOut = 32, kOutChunk = 256;

struct OutArgs {
  const __nv_bfloat16 *h;  // last hidden activations
  float *z;                // last hidden pre-activations, replaced by dZ
  const float *params;     // first member
  int64_t P, wo, bo;
  int64_t B, rows;
  int32_t H;
  const float *y;          // [members or 1][B]; NULL: forward only
  int64_t y_member;
  float *pred;             // first member
  int64_t pred_member;
  float *g;                // [members][rows]
};

__global__ void __launch_bounds__(256) mlp_out_kernel(const OutArgs a) {
  __shared__ __align__(16) __nv_bfloat16 hs[kRowsOut][kOutChunk + 8];
  __shared__ float ws[kOutChunk];
  __shared__ float gs[kRowsOut];
  const int64_t member = blockIdx.y;
  const int64_t r0 = (int64_t)blockIdx.x * kRowsOut;
  const int nr = (int)(a.B - r0 < kRowsOut ? a.B - r0 : kRowsOut);
  const float *pm = a.params + member * a.P;
  const __nv_bfloat16 *h = a.h + (member * a.rows + r0) * a.H;
  float acc = 0.0f;
  for (int c0 = 0; c0 < a.H; c0 += kOutChunk) {
    const int cn = a.H - c0 < kOutChunk ? a.H - c0 : kOutChunk;  // a multiple of 64
    for (int i = threadIdx.x; i < nr * (cn / 8); i += 256) {
      const int r = i / (cn / 8), c = (i % (cn / 8)) * 8;
      *reinterpret_cast<uint4 *>(&hs[r][c]) = *reinterpret_cast<const uint4 *>(h + (int64_t)r * a.H + c0 + c);
    }
    for (int i = threadIdx.x; i < cn; i += 256) ws[i] = bf16_round(pm[a.wo + c0 + i]);
    __syncthreads();
    if ((int)threadIdx.x < nr) {
      for (int c = 0; c < cn; c += 8) {
        float f[8];
        unpack(*reinterpret_cast<const uint4 *>(&hs[threadIdx.x][c]), f);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc = fmaf(f[e], ws[c + e], acc);
      }
    }
    __syncthreads();
  }
  if ((int)threadIdx.x < nr) {
    const int64_t b = r0 + threadIdx.x;
    const float pred = acc + pm[a.bo];
    a.pred[member * a.pred_member + b] = pred;
    if (a.y) {
      const float d = pred - a.y[member * a.y_member + b];
      const float gv = 2.0f * d / (float)a.B;
      a.g[member * a.rows + b] = gv;
      gs[threadIdx.x] = gv;
    }
  }
  if (!a.y) return;
  __syncthreads();
  // eight float4 of z per thread at a time, loaded before any of them is replaced
  float4 *z = reinterpret_cast<float4 *>(a.z + (member * a.rows + r0) * a.H);
  const int q4 = a.H / 4, total = nr * q4;
  for (int i0 = threadIdx.x; i0 < total; i0 += 8 * 256) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + u * 256 < total) v[u] = z[i0 + u * 256];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 + u * 256;
      if (i >= total) break;
      const float gv = gs[i / q4];
      const float *w = pm + a.wo + (i % q4) * 4;
      v[u].x = bf16_round(silu_grad(gv * bf16_round(w[0]), v[u].x));
      v[u].y = bf16_round(silu_grad(gv * bf16_round(w[1]), v[u].y));
      v[u].z = bf16_round(silu_grad(gv * bf16_round(w[2]), v[u].z));
      v[u].w = bf16_round(silu_grad(gv * bf16_round(w[3]), v[u].w));
      z[i] = v[u];
    }
  }
}

// ---- the small gradients and the loss --------------------------------------
//
// One launch, the blocks of a member in four roles: (0) W_out and (1) W_0, 64
// columns per block, each output one chain of FMAs over the batch; (2) bias
// gradients, eight columns per block; (3) the output bias and the loss.  A
// chain over the batch is serial, so the rows are staged 128 at a time in
// shared memory by all threads, the next rows' loads in flight meanwhile.
struct SmallArgs {
  const __nv_bfloat16 *h_last;
  const float *dz[kMaxLayers];  // hidden layers' dZ
  const float *X;
  int64_t x_member;
  const float *g, *pred, *y;
  int64_t pred_member, y_member;
  int64_t B, rows, P;
  int32_t H, n_in, n_hidden;
  int64_t w0, wo, bo;
  int64_t b[kMaxLayers];        // hidden layers' bias offsets
  float *grad;                  // first member
  float *loss;                  // [members] or NULL
};

__device__ __forceinline__ float block_sum(float s, float *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  s = threadIdx.x < 8 ? red[threadIdx.x] : 0.0f;
  if (threadIdx.x < 32) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  __syncthreads();
  return s;  // valid in thread 0
}

constexpr int kChainRows = 128;

// out[n * nk + k] = sum_b D[b][n] F[b][k], n0 .. n0 + 63, k < nk <= 8: 64
// threads per pair of k's, a column each, two chains side by side (one warp's
// instructions per row are what a tile waits for: all eight k's in one thread
// took 27 us for the launch instead of 24).  NK = 1: one k, g in FP32;
// NK = 8: X, a BF16 operand.
template <typename T, int NK>
__device__ __forceinline__ void chain_grad(const T *D, int64_t ldd, const float *F, int nk, int64_t B, int n0,
                                           float *out, float (*Ds)[64], float (*Fs)[8]) {
  constexpr int EV = 16 / (int)sizeof(T), NV = kChainRows * 64 / EV / 256;
  uint4 v[NV];
  float f[4];
  auto load = [&](int64_t b0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = threadIdx.x + i * 256;
      const int64_t b = b0 + c / (64 / EV);
      v[i] = b < B ? *reinterpret_cast<const uint4 *>(D + b * ldd + n0 + (c % (64 / EV)) * EV)
                   : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = threadIdx.x + i * 256;  // row e / 8, k = e % 8
      const int64_t b = b0 + e / 8;
      f[i] = (b < B && e % 8 < nk) ? F[b * nk + e % 8] : 0.0f;
    }
  };
  load(0);
  constexpr int KT = NK == 1 ? 1 : 2;  // chains per thread
  const int col = threadIdx.x & 63, kq = (threadIdx.x >> 6) * KT;
  const bool active = kq < nk;
  float acc[KT] = {};
  for (int64_t b0 = 0; b0 < B; b0 += kChainRows) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = threadIdx.x + i * 256;
      float e[EV];
      unpack(v[i], e);
      float *d = &Ds[c / (64 / EV)][(c % (64 / EV)) * EV];
#pragma unroll
      for (int q = 0; q < EV; q += 4) *reinterpret_cast<float4 *>(d + q) = make_float4(e[q], e[q + 1], e[q + 2], e[q + 3]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = threadIdx.x + i * 256;
      Fs[e / 8][e % 8] = NK > 1 ? bf16_round(f[i]) : f[i];
    }
    __syncthreads();
    if (b0 + kChainRows < B) load(b0 + kChainRows);
    if (active) {
      // eight rows' values are read before their FMAs: a chain waits for its
      // FMAs only, not for shared memory row by row
#pragma unroll 2
      for (int r0 = 0; r0 < kChainRows; r0 += 8) {
        float d[8], fr[8][KT];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          d[r] = Ds[r0 + r][col];
#pragma unroll
          for (int k = 0; k < KT; ++k) fr[r][k] = Fs[r0 + r][kq + k];
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int k = 0; k < KT; ++k) acc[k] = fmaf(d[r], fr[r][k], acc[k]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < KT; ++k)
    if (kq + k < nk) out[(int64_t)(n0 + col) * nk + kq + k] = acc[k];
}

__device__ __forceinline__ void small_grad(const SmallArgs &a) {
  __shared__ __align__(16) float Ds[kChainRows][64];
  __shared__ __align__(16) float Fs[kChainRows][8];
  __shared__ float red[32];
  const int64_t member = blockIdx.y;
  float *grad = a.grad + member * a.P;
  const float *g = a.g + member * a.rows;
  const int nc = a.H / 64;
  int j = blockIdx.x;
  if (j < nc) {
    chain_grad<__nv_bfloat16, 1>(a.h_last + member * a.rows * a.H, a.H, g, 1, a.B, j * 64, grad + a.wo, Ds, Fs);
    return;
  }
  j -= nc;
  if (j < nc) {
    chain_grad<float, 8>(a.dz[0] + member * a.rows * a.H, a.H, a.X + member * a.x_member, a.n_in, a.B, j * 64,
                            grad + a.w0, Ds, Fs);
    return;
  }
  j -= nc;
  if (j < a.n_hidden * (a.H / 8)) {
    const int l = j / (a.H / 8), n0 = (j % (a.H / 8)) * 8;
    const float *dz = a.dz[l] + member * a.rows * a.H + n0;
    float s[8] = {};
    for (int64_t b = threadIdx.x; b < a.B; b += 256) {
      const float4 u = *reinterpret_cast<const float4 *>(dz + b * a.H);
      const float4 w = *reinterpret_cast<const float4 *>(dz + b * a.H + 4);
      const float e[8] = {u.x, u.y, u.z, u.w, w.x, w.y, w.z, w.w};
#pragma unroll
      for (int q = 0; q < 8; ++q) s[q] += e[q];
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float t = block_sum(s[q], red);
      if (threadIdx.x == 0) grad[a.b[l] + n0 + q] = t;
    }
    return;
  }
  float s = 0.0f, sq = 0.0f;
  for (int64_t b = threadIdx.x; b < a.B; b += 256) {
    s += g[b];
    const float d = a.pred[member * a.pred_member + b] - a.y[member * a.y_member + b];
    sq += d * d;
  }
  s = block_sum(s, red);
  sq = block_sum(sq, red);
  if (threadIdx.x == 0) {
    grad[a.bo] = s;
    if (a.loss) a.loss[member] = sq / (float)a.B;
  }
}

// Launched so that it runs beside the square layers' weight gradients, which
// leave most of an SM's warps free: its inputs were complete before that launch
// began.  The wait at its end makes it end after them.  4 members x 1024 points:
// 172.6 us per step with the two launches one after the other, 155.5 together;
// 20,000 points 2.19 and 1.94 ms.
__global__ void __launch_bounds__(256) mlp_small_grad_kernel(const SmallArgs a) {
  small_grad(a);
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) for weights and biases.
__global__ void init_kernel(float *params, const int64_t *off, const int *fin, int L, int64_t P, int member,
                            uint64_t seed) {
  const uint2 key = seed_to_key(seed);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
    int l = 0;
    while (l + 1 < L && i >= off[l + 1]) ++l;
    const float bound = rsqrtf((float)fin[l]);
    const uint4 r = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(i >> 32), (uint32_t)member, kTagInit), key);
    params[(int64_t)member * P + i] = (2.0f * uniform24(r.x) - 1.0f) * bound;
  }
}

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int64_t n, float lr_t, float b1,
                            float b2, float eps_t) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr_t * mi / (sqrtf(vi) + eps_t);
  }
}

__global__ void features_kernel(const sde_jj_point *pts, int64_t n, float *X, const float *lo_hi) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const sde_jj_point p = pts[i];
    const double raw[5] = {p.a, p.omega, p.f, p.gamma, log10(p.D)};
#pragma unroll
    for (int k = 0; k < 5; ++k)
      X[i * 5 + k] = (float)(2.0 * (raw[k] - (double)lo_hi[k]) / ((double)lo_hi[5 + k] - (double)lo_hi[k]) - 1.0);
  }
}

// Mean and standard deviation over the members' outputs (rows `stride` apart)
// in FP64.  The FP64 pipe bounds it (one warp instruction per 16 cycles and SM):
// the divisions by the member counts are products with their reciprocals, the
// square root is Goldschmidt's.
__global__ void ensemble_stats_kernel(const float *out, int members, int64_t stride, int64_t B, double inv_n,
                                      double inv_n1, float *mean, float *spread) {
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < B; b += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int q = 0; q < members; ++q) s += out[(int64_t)q * stride + b];
    const double mu = s * inv_n;
    mean[b] = (float)mu;
    if (!spread) continue;
    double m2 = 0.0;
    for (int q = 0; q < members; ++q) {
      const double d = out[(int64_t)q * stride + b] - mu;
      m2 = fma(d, d, m2);
    }
    spread[b] = members > 1 ? (float)sqrt_goldschmidt(m2 * inv_n1) : 0.0f;
  }
}

int grid1(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 4096); }

// BF16 copies of the square hidden layers' weights for the tensor-core
// forward: whh[member][l][n][k] = W_{l+1}[n][k] of that member.
struct SquareOffsets {
  int64_t w[mlptc::MAX_HH];
};

// Grid: (HH / 1024, square layers, members), four elements per thread.
__global__ void __launch_bounds__(256) square_weights_kernel(const float *params, int64_t P, SquareOffsets off,
                                                             __nv_bfloat16 *whh) {
  constexpr int HH = mlptc::H * mlptc::H;
  const float *w = params + blockIdx.z * P + off.w[blockIdx.y];
  __nv_bfloat16 *d = whh + ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * HH;
  const int i = (int)blockIdx.x * 1024 + threadIdx.x;
  float v[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) v[u] = w[i + 256 * u];
#pragma unroll
  for (int u = 0; u < 4; ++u) d[i + 256 * u] = __float2bfloat16_rn(v[u]);
}

}  // namespace
}  // namespace sde

struct sde_mlp {
  sde_mlp_config cfg{};
  int L = 0;                    // linear layers
  std::vector<int> fin, fout;   // per layer
  std::vector<int64_t> woff, boff;
  int64_t P = 0;                // parameters per member
  float *params = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;  // [members][P]
  int64_t P_bf16 = 0;              // P rounded up to 8: the BF16 copies' rows stay 16-byte aligned
  int64_t rows = 0;                // batch rows of the activation buffers (members share them)
  __nv_bfloat16 *wbf = nullptr;    // [members][P_bf16]
  std::vector<__nv_bfloat16 *> h;  // L entries: layer inputs (bf16), h[0] unused (layer 0 reads X)
  std::vector<float *> z;          // L - 1 hidden pre-activations; the backward leaves dZ in their place
  float *out = nullptr;            // [members][max_batch]
  float *gout = nullptr;           // [rows] output-layer gradient
  float *lo_hi = nullptr;          // [10]
  int64_t *off_dev = nullptr;
  int *fin_dev = nullptr;
  int64_t step = 0;
  // tensor-core forward (width 256, at least two hidden layers)
  bool tc = false;                 // the shape has the tensor-core path
  bool use_tc = true;              // sde_mlp_use_tensor_cores
  __nv_bfloat16 *whh = nullptr;    // [members][n_hidden - 1][256][256]
  CUtensorMap map_whh;
  uint32_t *err = nullptr;         // latched kErrTimeout of the tensor-core kernel
  int sm_count = 1;
};

namespace {

using namespace sde;

// Members whose batches of B rows fit in the activation buffers together.
int64_t member_group(const sde_mlp *q, int64_t B) {
  return std::max<int64_t>(1, std::min<int64_t>(q->cfg.n_members, q->rows / B));
}

// Forward pass of members m0 .. m0 + G - 1, each over its own B rows of X
// (x_member apart; 0: the same rows); with y also the output gradient and the
// last hidden layer's dZ.  Predictions -> q->out.
sde_status mlp_forward_members(sde_mlp *q, int64_t m0, int64_t G, const float *X, int64_t x_member, int64_t B,
                               const float *y, int64_t y_member, cudaStream_t s) {
  SDE_CUDA_TRY(cudaGetLastError());
  const int H = q->cfg.hidden;
  const float *pm = q->params + m0 * q->P;
  Layer0Args a0{};
  a0.X = X;
  a0.x_member = x_member;
  a0.params = pm;
  a0.P = q->P;
  a0.P_bf16 = q->P_bf16;
  a0.w0 = q->woff[0];
  a0.b0 = q->boff[0];
  a0.B = B;
  a0.rows = B;
  a0.n_in = q->cfg.n_in;
  a0.H = H;
  a0.blocks0 = (int)((B + kRows0 - 1) / kRows0);
  a0.z = q->z[0];
  a0.h = q->h[1];
  a0.wbf = q->wbf;
  mlp_layer0_kernel<<<dim3((unsigned)(a0.blocks0 + 128), (unsigned)G), 256, 0, s>>>(a0);
  SDE_CUDA_TRY(cudaGetLastError());
  for (int l = 1; l < q->L - 1; ++l) {
    GemmArgs g{};
    g.B = B;
    g.H = H;
    g.n_layers = 1;
    g.rows = B;
    g.a[0] = q->h[l];
    g.b[0] = q->wbf + q->woff[l];
    g.b_member = q->P_bf16;
    g.bias = pm + q->boff[l];
    g.p_member = q->P;
    g.z = q->z[l];
    g.h = q->h[l + 1];
    mlp_gemm_kernel<EPI_FWD><<<dim3((unsigned)((B + TM - 1) / TM), H / TN, (unsigned)G), GT, 0, s>>>(g);
    SDE_CUDA_TRY(cudaGetLastError());
  }
  OutArgs o{};
  o.h = q->h[q->L - 1];
  o.z = q->z[q->L - 2];
  o.params = pm;
  o.P = q->P;
  o.wo = q->woff[q->L - 1];
  o.bo = q->boff[q->L - 1];
  o.B = B;
  o.rows = B;
  o.H = H;
  o.y = y;
  o.y_member = y_member;
  o.pred = q->out + m0 * q->cfg.max_batch;
  o.pred_member = q->cfg.max_batch;
  o.g = q->gout;
  mlp_out_kernel<<<dim3((unsigned)((B + kRowsOut - 1) / kRowsOut), (unsigned)G), 256, 0, s>>>(o);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}

// Gradients of the MSE of members m0 .. m0 + G - 1 -> grad (q->P apart), their
// losses -> loss (NULL allowed).
sde_status mlp_grad_members(sde_mlp *q, int64_t m0, int64_t G, const float *X, int64_t x_member, const float *y,
                            int64_t y_member, int64_t B, float *grad, float *loss, cudaStream_t s) {
  sde_status st = mlp_forward_members(q, m0, G, X, x_member, B, y, y_member, s);
  if (st != SDE_OK) return st;
  const int H = q->cfg.hidden, nh = q->cfg.n_hidden;
  for (int l = nh - 1; l >= 1; --l) {  // dZ_{l-1} = (dZ_l W_l) SiLU'(z_{l-1})
    GemmArgs g{};
    g.B = B;
    g.H = H;
    g.n_layers = 1;
    g.rows = B;
    g.a[0] = q->z[l];
    g.b[0] = q->wbf + q->woff[l];
    g.b_member = q->P_bf16;
    g.z = q->z[l - 1];
    mlp_gemm_kernel<EPI_DSILU><<<dim3((unsigned)((B + TM - 1) / TM), H / TN, (unsigned)G), GT, 0, s>>>(g);
    SDE_CUDA_TRY(cudaGetLastError());
  }
  if (nh > 1) {  // dW_l = dZ_l^T h_l of every square layer
    GemmArgs g{};
    g.B = B;
    g.H = H;
    g.n_layers = nh - 1;
    g.rows = B;
    g.b_member = B * H;
    g.p_member = q->P;
    for (int l = 1; l < nh; ++l) {
      g.a[l - 1] = q->z[l];
      g.b[l - 1] = q->h[l];
      g.grad[l - 1] = grad + q->woff[l];
    }
    mlp_gemm_kernel<EPI_DW><<<dim3(H / TM, H / TN, (unsigned)(G * (nh - 1))), GT, 0, s>>>(g);
    SDE_CUDA_TRY(cudaGetLastError());
  }
  SmallArgs a{};
  a.h_last = q->h[nh];
  for (int l = 0; l < nh; ++l) {
    a.dz[l] = q->z[l];
    a.b[l] = q->boff[l];
  }
  a.X = X;
  a.x_member = x_member;
  a.g = q->gout;
  a.pred = q->out + m0 * q->cfg.max_batch;
  a.pred_member = q->cfg.max_batch;
  a.y = y;
  a.y_member = y_member;
  a.B = B;
  a.rows = B;
  a.P = q->P;
  a.H = H;
  a.n_in = q->cfg.n_in;
  a.n_hidden = nh;
  a.w0 = q->woff[0];
  a.wo = q->woff[nh];
  a.bo = q->boff[nh];
  a.grad = grad;
  a.loss = loss;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * (H / 64) + nh * (H / 8) + 1), (unsigned)G);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = nh > 1 ? 1 : 0;  // only behind the weight-gradient launch
  SDE_CUDA_TRY(cudaLaunchKernelEx(&cfg, mlp_small_grad_kernel, a));
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}

void mlp_free(sde_mlp *q) {
  if (!q) return;
  cudaDeviceSynchronize();
  cudaFree(q->params);
  cudaFree(q->m);
  cudaFree(q->v);
  cudaFree(q->grad);
  cudaFree(q->wbf);
  for (auto p : q->h) cudaFree(p);
  for (auto p : q->z) cudaFree(p);
  cudaFree(q->out);
  cudaFree(q->gout);
  cudaFree(q->lo_hi);
  cudaFree(q->off_dev);
  cudaFree(q->fin_dev);
  cudaFree(q->whh);
  cudaFree(q->err);
  delete q;
}

}  // namespace

using namespace sde;

extern "C" {

sde_status sde_mlp_create(const sde_mlp_config *cfg, sde_mlp **out) {
  clear_error();
  SDE_CHECK_ARG(out != nullptr, "out is NULL");
  *out = nullptr;
  SDE_CHECK_ARG(cfg != nullptr, "cfg is NULL");
  SDE_CHECK_ARG(cfg->n_in >= 1 && cfg->n_in <= 8, "n_in must be in [1, 8]");
  SDE_CHECK_ARG(cfg->hidden >= 64 && cfg->hidden <= 1024 && cfg->hidden % 64 == 0,
                "hidden must be a multiple of 64 in [64, 1024]");
  SDE_CHECK_ARG(cfg->n_hidden >= 1 && cfg->n_hidden <= 8, "n_hidden must be in [1, 8]");
  SDE_CHECK_ARG(cfg->n_members >= 1 && cfg->n_members <= 16, "n_members must be in [1, 16]");
  SDE_CHECK_ARG(cfg->max_batch >= 1 && cfg->max_batch <= (1ll << 24), "max_batch must be in [1, 2^24]");
  SDE_CHECK_ARG(cfg->lr > 0.0f && cfg->beta1 >= 0.0f && cfg->beta1 < 1.0f && cfg->beta2 >= 0.0f &&
                    cfg->beta2 < 1.0f && cfg->eps > 0.0f,
                "Adam hyper-parameters out of range");
  for (int k = 0; k < 5; ++k) SDE_CHECK_ARG(cfg->hi[k] > cfg->lo[k], "feature box needs hi > lo");
  sde_mlp *q = new (std::nothrow) sde_mlp();
  if (!q) {
    set_error("host allocation failed");
    return SDE_ERR_NO_MEMORY;
  }
  q->cfg = *cfg;
  q->L = cfg->n_hidden + 1;
  int64_t off = 0;
  for (int l = 0; l < q->L; ++l) {
    const int fi = l == 0 ? cfg->n_in : cfg->hidden;
    const int fo = l == q->L - 1 ? 1 : cfg->hidden;
    q->fin.push_back(fi);
    q->fout.push_back(fo);
    q->woff.push_back(off);
    off += (int64_t)fi * fo;
    q->boff.push_back(off);
    off += fo;
  }
  q->P = off;
  const int64_t M = cfg->n_members, B = cfg->max_batch, H = cfg->hidden;
  sde_status st = SDE_OK;
  auto alloc = [&](void **p, size_t bytes) {
    if (st != SDE_OK) return;
    cudaError_t e = device_alloc(p, bytes ? bytes : 1);
    if (e != cudaSuccess) st = cuda_fail(e, "cudaMalloc");
  };
  alloc((void **)&q->params, sizeof(float) * M * q->P);
  alloc((void **)&q->m, sizeof(float) * M * q->P);
  alloc((void **)&q->v, sizeof(float) * M * q->P);
  alloc((void **)&q->grad, sizeof(float) * M * q->P);
  // the members' batches share the activation rows: at least one member's
  // largest batch, and up to 32 MB more of pre-activations per layer so that
  // small networks' members train together at their largest batch too
  q->rows = std::max<int64_t>(B, std::min<int64_t>(M * B, (32ll << 20) / (4 * H)));
  q->P_bf16 = (q->P + 7) & ~7ll;
  const int64_t rows = q->rows;
  alloc((void **)&q->wbf, sizeof(__nv_bfloat16) * M * q->P_bf16);
  q->h.assign(q->L, nullptr);
  q->z.assign(q->L - 1, nullptr);
  for (int l = 1; l < q->L; ++l) alloc((void **)&q->h[l], sizeof(__nv_bfloat16) * rows * H);
  for (int l = 0; l < q->L - 1; ++l) alloc((void **)&q->z[l], sizeof(float) * rows * H);
  alloc((void **)&q->out, sizeof(float) * M * B);
  alloc((void **)&q->gout, sizeof(float) * rows);
  alloc((void **)&q->lo_hi, sizeof(float) * 10);
  alloc((void **)&q->off_dev, sizeof(int64_t) * (q->L + 1));
  alloc((void **)&q->fin_dev, sizeof(int) * q->L);
  alloc((void **)&q->err, sizeof(uint32_t));
  q->tc = cfg->hidden == mlptc::H && cfg->n_hidden >= 2 && cfg->n_hidden - 1 <= mlptc::MAX_HH &&
          cfg->n_in <= mlptc::MAX_IN;
  if (q->tc) alloc((void **)&q->whh, sizeof(__nv_bfloat16) * M * (cfg->n_hidden - 1) * H * H);
  alloc_injection_disarm();
  if (st == SDE_OK && q->tc) {
    st = make_map_bf16(&q->map_whh, q->whh, M * (cfg->n_hidden - 1) * H, H, mlptc::H);
    if (st == SDE_OK) {
      int dev = 0;
      cudaError_t e = cudaGetDevice(&dev);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&q->sm_count, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) st = cuda_fail(e, "cudaDeviceGetAttribute");
    }
    if (st == SDE_OK) {
      cudaError_t e = cudaFuncSetAttribute(mlptc::mlp_fwd_tc_kernel<false>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, mlptc::SMEM_BYTES);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlptc::mlp_fwd_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 mlptc::SMEM_BYTES);
      if (e != cudaSuccess) st = cuda_fail(e, "cudaFuncSetAttribute(mlp_fwd_tc_kernel)");
    }
  }
  if (st == SDE_OK) {
    float lh[10];
    for (int k = 0; k < 5; ++k) {
      lh[k] = cfg->lo[k];
      lh[5 + k] = cfg->hi[k];
    }
    std::vector<int64_t> offs(q->woff.begin(), q->woff.end());
    offs.push_back(q->P);
    cudaError_t e = cudaMemcpy(q->lo_hi, lh, sizeof lh, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(q->off_dev, offs.data(), sizeof(int64_t) * offs.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(q->fin_dev, q->fin.data(), sizeof(int) * q->L, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(q->m, 0, sizeof(float) * M * q->P);
    if (e == cudaSuccess) e = cudaMemset(q->err, 0, sizeof(uint32_t));
    if (e == cudaSuccess) e = cudaMemset(q->v, 0, sizeof(float) * M * q->P);
    for (int mm = 0; mm < M && e == cudaSuccess; ++mm) {
      init_kernel<<<grid1(q->P), 256>>>(q->params, q->off_dev, q->fin_dev, q->L, q->P, mm, cfg->seed);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) st = cuda_fail(e, "sde_mlp_create");
  }
  if (st != SDE_OK) {
    std::string msg = sde_last_error();
    mlp_free(q);
    set_error(msg);
    return st;
  }
  *out = q;
  return SDE_OK;
}

void sde_mlp_destroy(sde_mlp *q) { mlp_free(q); }

int64_t sde_mlp_num_params(const sde_mlp *q) { return q ? q->P : -1; }

sde_status sde_mlp_set_params(sde_mlp *q, int32_t member, const float *p, void *stream) {
  clear_error();
  SDE_CHECK_ARG(q && p, "mlp and params must be non-NULL");
  SDE_CHECK_ARG(member >= 0 && member < q->cfg.n_members, "member out of range");
  SDE_CUDA_TRY(cudaMemcpyAsync(q->params + (int64_t)member * q->P, p, sizeof(float) * q->P,
                               cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
  return SDE_OK;
}

sde_status sde_mlp_get_params(sde_mlp *q, int32_t member, float *p, void *stream) {
  clear_error();
  SDE_CHECK_ARG(q && p, "mlp and params must be non-NULL");
  SDE_CHECK_ARG(member >= 0 && member < q->cfg.n_members, "member out of range");
  SDE_CUDA_TRY(cudaMemcpyAsync(p, q->params + (int64_t)member * q->P, sizeof(float) * q->P,
                               cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
  return SDE_OK;
}

sde_status sde_mlp_features(sde_mlp *q, const sde_jj_point *pts, int64_t n, float *X, void *stream) {
  clear_error();
  SDE_CHECK_ARG(q != nullptr && n >= 0, "mlp is NULL or n < 0");
  SDE_CHECK_ARG(q->cfg.n_in == 5, "the parameter features need n_in == 5");
  if (n == 0) return SDE_OK;
  SDE_CHECK_ARG(pts && X, "points and X must be non-NULL");
  features_kernel<<<grid1(n), 256, 0, (cudaStream_t)stream>>>(pts, n, X, q->lo_hi);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}

sde_status sde_mlp_forward(sde_mlp *q, const float *X, int64_t B, float *mean, float *spread, void *stream) {
  clear_error();
  SDE_CHECK_ARG(q != nullptr, "mlp is NULL");
  SDE_CHECK_ARG(B >= 0 && B <= q->cfg.max_batch, "batch exceeds max_batch");
  if (B == 0) return SDE_OK;
  SDE_CHECK_ARG(X && mean, "X and mean must be non-NULL");
  cudaStream_t s = (cudaStream_t)stream;
  if (q->tc && q->use_tc) {
    const int n_hh = q->cfg.n_hidden - 1;
    SquareOffsets so{};
    mlptc::Args a{};
    for (int l = 0; l < n_hh; ++l) {
      so.w[l] = q->woff[l + 1];
      a.off_bh[l] = q->boff[l + 1];
    }
    square_weights_kernel<<<dim3(mlptc::H * mlptc::H / 1024, (unsigned)n_hh, (unsigned)q->cfg.n_members), 256, 0, s>>>(
        q->params, q->P, so, q->whh);
    SDE_CUDA_TRY(cudaGetLastError());
    a.X = X;
    a.params = q->params;
    a.P = q->P;
    a.B = B;
    a.n_in = q->cfg.n_in;
    a.n_hh = n_hh;
    a.off_w0 = q->woff[0];
    a.off_b0 = q->boff[0];
    a.off_wo = q->woff[q->L - 1];
    a.off_bo = q->boff[q->L - 1];
    a.out = q->out;
    a.out_stride = q->cfg.max_batch;
    a.err = q->err;
    // One CTA per SM, shared evenly among the members.  Where that leaves each
    // CTA one tile, all its warps share it (129 points of 2 members: 25 us per call
    // instead of 29).
    const int64_t tiles = (B + mlptc::BM - 1) / mlptc::BM;
    const int64_t per_member = std::max<int64_t>(1, q->sm_count / q->cfg.n_members);
    const dim3 grid((unsigned)std::min(tiles, per_member), (unsigned)q->cfg.n_members);
    if (tiles <= per_member)
      mlptc::mlp_fwd_tc_kernel<true><<<grid, mlptc::THREADS, mlptc::SMEM_BYTES, s>>>(q->map_whh, a);
    else
      mlptc::mlp_fwd_tc_kernel<false><<<grid, mlptc::THREADS, mlptc::SMEM_BYTES, s>>>(q->map_whh, a);
    SDE_CUDA_TRY(cudaGetLastError());
  } else {
    const int64_t G = member_group(q, B);
    for (int64_t mm = 0; mm < q->cfg.n_members; mm += G) {
      sde_status st =
          mlp_forward_members(q, mm, std::min<int64_t>(G, q->cfg.n_members - mm), X, 0, B, nullptr, 0, s);
      if (st != SDE_OK) return st;
    }
  }
  ensemble_stats_kernel<<<grid1(B), 256, 0, s>>>(q->out, q->cfg.n_members, q->cfg.max_batch, B,
                                                 1.0 / q->cfg.n_members, 1.0 / (q->cfg.n_members - 1.0), mean,
                                                 spread);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}

sde_status sde_mlp_grad(sde_mlp *q, int32_t member, const float *X, const float *y, int64_t B, float *grad,
                        float *loss, void *stream) {
  clear_error();
  SDE_CHECK_ARG(q != nullptr, "mlp is NULL");
  SDE_CHECK_ARG(member >= 0 && member < q->cfg.n_members, "member out of range");
  SDE_CHECK_ARG(B >= 1 && B <= q->cfg.max_batch, "batch must be in [1, max_batch]");
  SDE_CHECK_ARG(X && y && grad, "X, y and grad must be non-NULL");
  return mlp_grad_members(q, member, 1, X, 0, y, 0, B, grad, loss, (cudaStream_t)stream);
}

sde_status sde_mlp_use_tensor_cores(sde_mlp *q, int32_t enable) {
  clear_error();
  SDE_CHECK_ARG(q != nullptr, "mlp is NULL");
  if (enable && !q->tc) {
    set_error("the tensor-core forward needs hidden == 256, 2..8 hidden layers and n_in <= 8");
    return SDE_ERR_UNSUPPORTED;
  }
  q->use_tc = enable != 0;
  return SDE_OK;
}

sde_status sde_mlp_check(sde_mlp *q) {
  clear_error();
  SDE_CHECK_ARG(q != nullptr, "mlp is NULL");
  SDE_CUDA_TRY(cudaDeviceSynchronize());
  uint32_t err = 0;
  SDE_CUDA_TRY(cudaMemcpy(&err, q->err, sizeof(uint32_t), cudaMemcpyDeviceToHost));
  if (err) SDE_CUDA_TRY(cudaMemset(q->err, 0, sizeof(uint32_t)));
  if (err & kErrTimeout) {
    set_error("a bounded device wait of the tensor-core forward expired");
    return SDE_ERR_TIMEOUT;
  }
  return SDE_OK;
}

sde_status sde_mlp_set_lr(sde_mlp *q, float lr) {
  clear_error();
  SDE_CHECK_ARG(q != nullptr && lr > 0.0f, "mlp must be non-NULL and lr > 0");
  q->cfg.lr = lr;
  return SDE_OK;
}

static sde_status mlp_train(sde_mlp *q, const float *X, const float *y, int64_t B, float *loss, void *stream,
                            bool per_member) {
  clear_error();
  SDE_CHECK_ARG(q != nullptr, "mlp is NULL");
  SDE_CHECK_ARG(B >= 1 && B <= q->cfg.max_batch, "batch must be in [1, max_batch]");
  SDE_CHECK_ARG(X && y, "X and y must be non-NULL");
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t G = member_group(q, B), x_member = per_member ? B * q->cfg.n_in : 0, y_member = per_member ? B : 0;
  for (int64_t mm = 0; mm < q->cfg.n_members; mm += G) {
    sde_status st = mlp_grad_members(q, mm, std::min<int64_t>(G, q->cfg.n_members - mm), X + mm * x_member, x_member,
                                     y + mm * y_member, y_member, B, q->grad + mm * q->P, loss ? loss + mm : nullptr, s);
    if (st != SDE_OK) return st;
  }
  q->step += 1;
  const double b1 = q->cfg.beta1, b2 = q->cfg.beta2;
  const double c1 = 1.0 - pow(b1, (double)q->step), c2 = 1.0 - pow(b2, (double)q->step);
  // Adam with the bias corrections folded into the step size and epsilon:
  // p -= lr * (m / c1) / (sqrt(v / c2) + eps) = (lr sqrt(c2) / c1) m / (sqrt(v) + eps sqrt(c2))
  const float lr_t = (float)(q->cfg.lr * sqrt(c2) / c1);
  const float eps_t = (float)(q->cfg.eps * sqrt(c2));
  const int64_t n = q->P * q->cfg.n_members;
  adam_kernel<<<grid1(n), 256, 0, s>>>(q->params, q->grad, q->m, q->v, n, lr_t, (float)b1, (float)b2, eps_t);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}

sde_status sde_mlp_train_step(sde_mlp *q, const float *X, const float *y, int64_t B, float *loss, void *stream) {
  return mlp_train(q, X, y, B, loss, stream, false);
}

sde_status sde_mlp_train_step_members(sde_mlp *q, const float *X, const float *y, int64_t B, float *loss,
                                      void *stream) {
  return mlp_train(q, X, y, B, loss, stream, true);
}

}  // extern "C"
