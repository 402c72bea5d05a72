// josephson.cu -- per-path SRK2 integration of Eq. 1 on the GPU.
//
// Each path lives in registers for the whole launch (Alg. 1: load x, v and
// the parameters, loop over m steps, store back; Sec. 4.1).  One Philox
// block gives the Gaussians of four consecutive steps (Sec. 4.1 draws two
// uniforms per step; here one Gaussian per step suffices since Eq. 1 has one
// noise component).  The step is Alg. 2 applied to y = (x, v):
//
//   F1 = -gamma v - 2 pi cos(2 pi x) + a cos(omega t_n) + f
//   x~ = x + dt v,          v~ = v + dt F1 + s psi
//   F2 = -gamma v~ - 2 pi cos(2 pi x~) + a cos(omega t_{n+1}) + f
//   x' = x + dt/2 (v + v~), v' = v + dt/2 (F1 + F2) + s psi,   s = sqrt(2 gamma D dt)
//
// Time is kept modulo the drive period as the integer k = n mod P (Sec. 5),
// so cos(omega t_n) = cos(2 pi k / P) comes from a P-entry table in shared
// memory.  Position is kept as x in [0, 1) plus an integer winding count
// (folded once per group of four steps), so FP32 resolution does not degrade
// as paths run away.  cos(2 pi x) is a branch-free minimax polynomial
// (jj_force below).
//
// The window average of v (the time-averaged velocity <<v>> of Sec. 5) is
// summed in FP32 over blocks of 64 steps (aligned to absolute step indices)
// and flushed into an FP64 per-path accumulator; per-warp moments of the
// per-path averages are FP64.
//
// A thread advances one, two or four paths; with two or four, pairs of paths
// share Blackwell's packed FP32x2 FMA, add and multiply (jj_step2,
// box_muller_tab2), which round exactly like the scalar instructions, so
// every launch variant produces the same bits.
#include <cuda_runtime.h>
#include <math.h>

#include <mutex>
#include <string>

#include "fp64_math.cuh"
#include "internal.h"
#include "philox.cuh"

namespace sde {
namespace {

// A - 2 pi cos(2 pi x) for |x| < 2^22 without branches: with r = x - rint(x)
// in [-1/2, 1/2] and b = 1/4 - |r| in [-1/4, 1/4], cos(2 pi x) = sin(2 pi b),
// and sin(2 pi b) = b P(b^2) with P a degree-4 polynomial whose coefficients
// minimise the largest absolute error on [0, 1/4] (Lawson's iteratively
// reweighted least squares, about 3e-9 in exact arithmetic).  The factor
// -2 pi of Eq. 1's force is folded into P, so the force term and the addend
// A = a cos(omega t) + f - gamma v cost one FMA.  In FP32 the error of
// cos(2 pi x) is at most 1.7e-7 (RMS 3.7e-8).
__device__ __forceinline__ float jj_force(float x, float A) {
  const float b = 0.25f - fabsf(x - rintf(x));
  const float s = b * b;
  float p = -2.484164429e+02f;  // -2 pi x (39.536705, -76.5497818, 81.6010056, -41.3416557, 6.28318501)
  p = fmaf(p, s, 4.809764709e+02f);
  p = fmaf(p, s, -5.127142334e+02f);
  p = fmaf(p, s, 2.597572937e+02f);
  p = fmaf(p, s, -3.947841644e+01f);
  return fmaf(b, p, A);
}

// One SRK2 step (Alg. 2), or with EM one Euler-Maruyama step (the
// first-order scheme of PROG2, Sec. 4.2).  x is kept in [0, 1) up to the
// drift of the steps since the last wrap (at most four steps, see
// jj_segment).  e0, e1: the drive and bias a cos(omega t) + f at t_n and
// t_{n+1}.
template <bool ACC, bool EM>
__device__ __forceinline__ void jj_step(float &x, float &v, float &acc, float z, const JJConsts &c, float e0,
                                        float e1) {
  const float vn = fmaf(c.s, z, v);  // v plus the noise increment, used by both stages
  const float F1 = jj_force(x, fmaf(-c.gamma, v, e0));
  if (EM) {
    x = fmaf(c.dt, v, x);
    v = fmaf(c.dt, F1, vn);
    if (ACC) acc += v;
    return;
  }
  const float xt = fmaf(c.dt, v, x);
  const float vt = fmaf(c.dt, F1, vn);
  const float F2 = jj_force(xt, fmaf(-c.gamma, vt, e1));
  x = fmaf(c.h, v + vt, x);
  v = fmaf(c.h, F1 + F2, vn);
  if (ACC) acc += v;
}

// The same step for two paths at once on packed FP32 pairs (Blackwell's
// two-wide FMA, add and multiply, rounded like fmaf and +), so one
// instruction advances both paths of a thread.  Same operations in the same
// order as jj_force / jj_step: the results are bit-identical.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

__device__ __forceinline__ float2 jj_force2(float2 x, float2 A) {
  // -|r| by setting the sign bit; rint is symmetric, so -rint(x) = rint(-x)
  const float2 r = __fadd2_rn(x, make_float2(rintf(-x.x), rintf(-x.y)));
  const float2 nr = make_float2(__int_as_float(__float_as_int(r.x) | 0x80000000),
                                __int_as_float(__float_as_int(r.y) | 0x80000000));
  const float2 b = __fadd2_rn(f2(0.25f), nr);
  const float2 s = __fmul2_rn(b, b);
  float2 p = __ffma2_rn(f2(-2.484164429e+02f), s, f2(4.809764709e+02f));
  p = __ffma2_rn(p, s, f2(-5.127142334e+02f));
  p = __ffma2_rn(p, s, f2(2.597572937e+02f));
  p = __ffma2_rn(p, s, f2(-3.947841644e+01f));
  return __ffma2_rn(b, p, A);
}

template <bool ACC, bool EM>
__device__ __forceinline__ void jj_step2(float2 &x, float2 &v, float2 &acc, float2 z, const JJConsts &c, float e0,
                                         float e1) {
  const float2 vn = __ffma2_rn(f2(c.s), z, v);
  const float2 F1 = jj_force2(x, __ffma2_rn(f2(-c.gamma), v, f2(e0)));
  if (EM) {
    x = __ffma2_rn(f2(c.dt), v, x);
    v = __ffma2_rn(f2(c.dt), F1, vn);
    if (ACC) acc = __fadd2_rn(acc, v);
    return;
  }
  const float2 xt = __ffma2_rn(f2(c.dt), v, x);
  const float2 vt = __ffma2_rn(f2(c.dt), F1, vn);
  const float2 F2 = jj_force2(xt, __ffma2_rn(f2(-c.gamma), vt, f2(e1)));
  x = __ffma2_rn(f2(c.h), __fadd2_rn(v, vt), x);
  v = __ffma2_rn(f2(c.h), __fadd2_rn(F1, F2), vn);
  if (ACC) acc = __fadd2_rn(acc, v);
}

// Steps s of a group for all ILP paths (packed pairs where ILP is even).
template <int ILP, bool ACC, bool EM>
__device__ __forceinline__ void jj_steps(float (&x)[ILP], float (&v)[ILP], float (&acc)[ILP],
                                         const float (&z)[ILP][4], int s, const JJConsts &c, float e0, float e1) {
  if constexpr (ILP % 2 == 0) {
#pragma unroll
    for (int i = 0; i < ILP; i += 2) {
      float2 X = make_float2(x[i], x[i + 1]), V = make_float2(v[i], v[i + 1]);
      float2 S = make_float2(acc[i], acc[i + 1]);
      jj_step2<ACC, EM>(X, V, S, make_float2(z[i][s], z[i + 1][s]), c, e0, e1);
      x[i] = X.x;
      x[i + 1] = X.y;
      v[i] = V.x;
      v[i + 1] = V.y;
      acc[i] = S.x;
      acc[i + 1] = S.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < ILP; ++i) jj_step<ACC, EM>(x[i], v[i], acc[i], z[i][s], c, e0, e1);
  }
}

// Fold x back into [0, 1), counting whole turns in w.
__device__ __forceinline__ void jj_wrap(float &x, int &w) {
  const float fl = floorf(x);
  x -= fl;
  w += (int)fl;
}

// Drive tables: the shared cos(2 pi k / P) table (P + 4 entries) and, for
// P <= kWarpTableMaxP, one table of a cos + f per warp, each padded to a
// multiple of 4 floats.
constexpr int kWarpTableMaxP = 1020;
constexpr int kJJMaxBlock = 512;  // the largest block any Josephson launch uses

__host__ __device__ inline int jj_table_stride(int P) { return (P + 4 + 3) & ~3; }

__host__ inline size_t jj_smem_bytes(int P, int block) {
  const int pp = jj_table_stride(P);
  return sizeof(float) * (size_t)pp * (P <= kWarpTableMaxP ? 1 + block / 32 : 1);
}

// The Box-Muller transforms of the Philox blocks r[i] of ILP paths into their
// four Gaussians z[i][0..3]: pairs of paths together on packed FP32 pairs
// (the same roundings as one path at a time), so each packed pair of paths
// gets its Gaussians already paired for jj_step2.
template <int ILP>
__device__ __forceinline__ void jj_transform(const uint4 (&r)[ILP], const float *bm_tab, float (&z)[ILP][4]) {
  if constexpr (ILP % 2 == 0) {
#pragma unroll
    for (int i = 0; i < ILP; i += 2) {
      float2 Z0, Z1, Z2, Z3;
      box_muller_tab2(r[i].x, r[i].y, r[i + 1].x, r[i + 1].y, bm_tab, Z0, Z1);
      box_muller_tab2(r[i].z, r[i].w, r[i + 1].z, r[i + 1].w, bm_tab, Z2, Z3);
      z[i][0] = Z0.x;
      z[i + 1][0] = Z0.y;
      z[i][1] = Z1.x;
      z[i + 1][1] = Z1.y;
      z[i][2] = Z2.x;
      z[i + 1][2] = Z2.y;
      z[i][3] = Z3.x;
      z[i + 1][3] = Z3.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < ILP; ++i) {
      box_muller_tab(r[i].x, r[i].y, bm_tab, z[i][0], z[i][1]);
      box_muller_tab(r[i].z, r[i].w, bm_tab, z[i][2], z[i][3]);
    }
  }
}

// Advance ILP paths over the steps [n0, n1).  `k` is the drive-table index
// of step n0 (n0 mod P) and is updated.
// SCALED: `drive` holds a cos(2 pi k / P) + f for this point (a per-warp or
// per-point table), else cos(2 pi k / P) and the drive term is formed here.
template <int ILP, bool ACC, bool EM = false, bool SCALED = false, bool ONEBB = false>
__device__ __forceinline__ void jj_segment(float (&x)[ILP], int (&w)[ILP], float (&v)[ILP],
                                           double (&vs)[ILP], const JJConsts &c,
                                           const float *__restrict__ drive, int P, int &k,
                                           int64_t n0, int64_t n1, const PhiloxKeys &key,
                                           const uint32_t (&pid)[ILP], uint32_t point,
                                           const float *bm_tab) {
  if (n0 >= n1) return;
  float acc[ILP];
#pragma unroll
  for (int i = 0; i < ILP; ++i) acc[i] = 0.0f;
  // group indices fit in 32 bits: steps are at most 2^33
  const uint32_t g0 = (uint32_t)(n0 >> 2), g1 = (uint32_t)((n1 - 1) >> 2);
  // Blocks of 16 groups (64 steps) aligned to absolute step indices; the
  // FP32 partial sums are flushed after each block, outside the group loop,
  // so the FP64 adds run once per 64 steps.
  // PIPE (four or more paths per thread): the Gaussians of group g + 1 are
  // drawn while group g is stepped, in one basic block, so the integer Philox
  // work interleaves with the FP32 steps (16 more live registers; with fewer
  // paths per thread the lost occupancy costs more than the overlap gains).
  constexpr bool PIPE = ILP >= 4;  // with ONEBB (the four-path kernels): see the group loop
  float z[ILP][4];
  if constexpr (PIPE) {
    uint4 r0[ILP];
#pragma unroll
    for (int i = 0; i < ILP; ++i) r0[i] = philox4x32_10(make_uint4(g0, pid[i], point, kTagJosephson), key);
    jj_transform<ILP>(r0, bm_tab, z);
  }
  for (uint32_t gb = g0; gb <= g1; gb = (gb | 15u) + 1u) {
    const uint32_t ge = (gb | 15u) < g1 ? (gb | 15u) : g1;
    for (uint32_t g = gb; g <= ge; ++g) {
      if constexpr (PIPE && ONEBB) {
        // ONEBB: a whole group with P a multiple of 4 as one basic block --
        // the next group's Philox words, the four steps, the position fold
        // and the next group's Box-Muller transform -- so that the compiler
        // can interleave the integer, special-function and FP32 work of
        // all three (the same operations as below, in the same order per
        // value: bit-identical).
        const int64_t base = (int64_t)g << 2;
        if ((P & 3) == 0 && base >= n0 && base + 4 <= n1) {
          uint4 rn[ILP];
#pragma unroll
          for (int i = 0; i < ILP; ++i)
            rn[i] = philox4x32_10(make_uint4(g + 1, pid[i], point, kTagJosephson), key);
          const float4 d = *reinterpret_cast<const float4 *>(drive + k);
          const float d4 = drive[k + 4];
          float e[5];
          e[0] = SCALED ? d.x : fmaf(c.a, d.x, c.f);
          e[1] = SCALED ? d.y : fmaf(c.a, d.y, c.f);
          e[2] = SCALED ? d.z : fmaf(c.a, d.z, c.f);
          e[3] = SCALED ? d.w : fmaf(c.a, d.w, c.f);
          e[4] = SCALED ? d4 : fmaf(c.a, d4, c.f);
          k = (k + 4 == P) ? 0 : k + 4;
#pragma unroll
          for (int s = 0; s < 4; ++s) jj_steps<ILP, ACC, EM>(x, v, acc, z, s, c, e[s], e[s + 1]);
#pragma unroll
          for (int i = 0; i < ILP; ++i) jj_wrap(x[i], w[i]);
          jj_transform<ILP>(rn, bm_tab, z);
          continue;
        }
      }
      // PIPE: the Philox words of group g + 1 now, their Box-Muller
      // transform into z once this group's steps have read it
      uint4 rn[ILP];
#pragma unroll
      for (int i = 0; i < ILP; ++i)
        rn[i] = philox4x32_10(make_uint4(PIPE ? g + 1 : g, pid[i], point, kTagJosephson), key);
      if constexpr (!PIPE) jj_transform<ILP>(rn, bm_tab, z);
      const int64_t base = (int64_t)g << 2;
      if (base >= n0 && base + 4 <= n1) {
        // full group: drive values at t_{4g} .. t_{4g+4}
        float e[5];
        if ((P & 3) == 0) {
          // k is a multiple of 4 here; the table is padded by 4 entries
          const float4 d = *reinterpret_cast<const float4 *>(drive + k);
          e[0] = SCALED ? d.x : fmaf(c.a, d.x, c.f);
          e[1] = SCALED ? d.y : fmaf(c.a, d.y, c.f);
          e[2] = SCALED ? d.z : fmaf(c.a, d.z, c.f);
          e[3] = SCALED ? d.w : fmaf(c.a, d.w, c.f);
          e[4] = SCALED ? drive[k + 4] : fmaf(c.a, drive[k + 4], c.f);
          k += 4;
          if (k == P) k = 0;
        } else {
#pragma unroll
          for (int s = 0; s < 5; ++s) {
            e[s] = SCALED ? drive[k] : fmaf(c.a, drive[k], c.f);
            if (s < 4) k = (k + 1 == P) ? 0 : k + 1;
          }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) jj_steps<ILP, ACC, EM>(x, v, acc, z, s, c, e[s], e[s + 1]);
      } else {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int64_t n = base + s;
          if (n >= n0 && n < n1) {
            const float e0 = SCALED ? drive[k] : fmaf(c.a, drive[k], c.f);
            k = (k + 1 == P) ? 0 : k + 1;
            const float e1 = SCALED ? drive[k] : fmaf(c.a, drive[k], c.f);
            jj_steps<ILP, ACC, EM>(x, v, acc, z, s, c, e0, e1);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < ILP; ++i) jj_wrap(x[i], w[i]);
      if constexpr (PIPE) jj_transform<ILP>(rn, bm_tab, z);
    }
    // Flush the FP32 partial sums at absolute 64-step boundaries, so that a
    // run split at any multiple of 64 steps reproduces the unsplit sums.
    if (ACC && ((ge + 1) & 15) == 0) {
#pragma unroll
      for (int i = 0; i < ILP; ++i) {
        vs[i] += (double)acc[i];
        acc[i] = 0.0f;
      }
    }
  }
  if (ACC) {
#pragma unroll
    for (int i = 0; i < ILP; ++i) vs[i] += (double)acc[i];
  }
}

__device__ __forceinline__ double warp_sum(double a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// Moments of the per-path window averages of a unit, after step n_end.
template <int ILP>
__device__ __forceinline__ void jj_unit_moments(Moments *out, int64_t n_end, const JJConsts &c,
                                                const double (&vs)[ILP], const bool (&valid)[ILP], int lane) {
  const int64_t reach = n_end < c.steps ? n_end : c.steps;
  const int64_t wcount = reach > c.wstart ? reach - c.wstart : 0;
  double cnt = 0.0, sum = 0.0;
  if (wcount > 0) {
#pragma unroll
    for (int i = 0; i < ILP; ++i)
      if (valid[i]) {
        cnt += 1.0;
        sum += vs[i] / (double)wcount;
      }
  }
  cnt = warp_sum(cnt);
  sum = warp_sum(sum);
  const double mean = cnt > 0.0 ? sum / cnt : 0.0;
  double m2 = 0.0;
  if (wcount > 0) {
#pragma unroll
    for (int i = 0; i < ILP; ++i)
      if (valid[i]) {
        const double d = vs[i] / (double)wcount - mean;
        m2 += d * d;
      }
  }
  m2 = warp_sum(m2);
  if (lane == 0) *out = Moments{cnt, mean, m2};
}

template <int ILP, bool EM, bool ONEBB = false>
__device__ __forceinline__ void jj_unit(const JJLaunchArgs &A, int u, const float *drive, float *wtab,
                                        const float *bm_tab, int lane) {
  const JJUnit un = A.units[u];
  const JJConsts c = A.consts[un.point];
  const PhiloxKeys &key = A.keys;
  float x[ILP], v[ILP];
  int w[ILP];
  double vs[ILP];
  uint32_t pid[ILP];
  bool valid[ILP];
  int64_t gi[ILP];
#pragma unroll
  for (int i = 0; i < ILP; ++i) {
    const int j = lane + 32 * i;
    valid[i] = j < un.n_paths;
    pid[i] = (uint32_t)(un.path_begin + j);
    gi[i] = c.path_offset + un.path_begin + j;
    x[i] = 0.0f;
    v[i] = 0.0f;
    w[i] = 0;
    vs[i] = 0.0;
    if (valid[i]) {
      x[i] = A.st.x_in[gi[i]];
      v[i] = A.st.v_in[gi[i]];
      if (A.st.w_in) w[i] = A.st.w_in[gi[i]];
      if (A.st.vsum_in) vs[i] = A.st.vsum_in[gi[i]];
    }
    const float fl = floorf(x[i]);
    x[i] -= fl;
    w[i] += (int)fl;
  }
  const int64_t nb = A.n_begin;
  const int64_t ne = A.n_end < c.steps ? A.n_end : c.steps;
  if (nb < ne) {
    int k = (int)(nb % A.P);
    const int64_t split = ne < c.wstart ? ne : c.wstart;
    const int64_t w0 = nb > c.wstart ? nb : c.wstart;
    if (wtab) {
      // this warp's copy of the drive term a cos(2 pi k / P) + f of the unit's point
      for (int q = lane; q < A.P + 4; q += 32) wtab[q] = fmaf(c.a, drive[q], c.f);
      __syncwarp();
      jj_segment<ILP, false, EM, true, ONEBB>(x, w, v, vs, c, wtab, A.P, k, nb, split, key, pid,
                                              (uint32_t)un.point, bm_tab);
      jj_segment<ILP, true, EM, true, ONEBB>(x, w, v, vs, c, wtab, A.P, k, w0, ne, key, pid, (uint32_t)un.point,
                                             bm_tab);
      __syncwarp();  // the table is rewritten for the warp's next unit
    } else {
      jj_segment<ILP, false, EM, false, ONEBB>(x, w, v, vs, c, drive, A.P, k, nb, split, key, pid,
                                               (uint32_t)un.point, bm_tab);
      jj_segment<ILP, true, EM, false, ONEBB>(x, w, v, vs, c, drive, A.P, k, w0, ne, key, pid, (uint32_t)un.point,
                                              bm_tab);
    }
  }
  bool bad = false;
#pragma unroll
  for (int i = 0; i < ILP; ++i) {
    if (valid[i]) {
      A.st.x_out[gi[i]] = x[i];
      A.st.v_out[gi[i]] = v[i];
      A.st.w_out[gi[i]] = w[i];
      A.st.vsum_out[gi[i]] = vs[i];
      bad |= !(isfinite(x[i]) && isfinite(v[i]));
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(A.err, kErrNonFinite);

  jj_unit_moments<ILP>(A.partials + u, A.n_end, c, vs, valid, lane);
}

template <int ILP, bool EM, bool ONEBB = false>
__device__ __forceinline__ void jj_kernel_body(const JJLaunchArgs &A) {
  // drive table cos(2 pi k / P), k = 0 .. P + 3 (four entries of padding
  // repeat the start of the period), 16-byte aligned
  extern __shared__ float4 drive_s4[];
  __shared__ float bm_tab[2 * kBmTable];  // Box-Muller angle table
  float *drive_s = reinterpret_cast<float *>(drive_s4);
  for (int i = threadIdx.x; i < A.P + 4; i += blockDim.x) drive_s[i] = A.drive[i % A.P];
  fill_bm_table(bm_tab);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int warps = blockDim.x >> 5;
  // per-warp tables of the drive term (P <= kWarpTableMaxP), 16-byte aligned
  const int pp = jj_table_stride(A.P);
  float *wtab = A.P <= kWarpTableMaxP ? drive_s + pp * (1 + (threadIdx.x >> 5)) : nullptr;
  if (A.queue) {
    // Persistent: warps pull units from the longest-first work list.
    for (;;) {
      int u = 0;
      if (lane == 0) u = (int)atomicAdd(A.queue, 1u) + A.unit_begin;
      u = __shfl_sync(0xffffffffu, u, 0);
      if (u >= A.unit_end) break;
      jj_unit<ILP, EM, ONEBB>(A, u, drive_s, wtab, bm_tab, lane);
    }
  } else {
    const int u = A.unit_begin + blockIdx.x * warps + (threadIdx.x >> 5);
    if (u < A.unit_end) jj_unit<ILP, EM, ONEBB>(A, u, drive_s, wtab, bm_tab, lane);
  }
}

template <int ILP, bool EM = false>
__global__ void __launch_bounds__(512) jj_kernel(const JJLaunchArgs A) {
  jj_kernel_body<ILP, EM>(A);
}

// The same kernel with registers capped at 64 per thread (blocks of up to 512
// threads, two per SM): more resident warps for more spills; the autotuner
// picks.
template <int ILP, bool EM = false>
__global__ void __launch_bounds__(512, 2) jj_kernel_cap64(const JJLaunchArgs A) {
  jj_kernel_body<ILP, EM>(A);
}

// Packed-pair kernels (2 or 4 paths per thread) at the fewest registers that
// hold them without spills: 72 for one pair (28 warps per SM in blocks of
// 128), 128 for two pairs with the noise of the next group in flight (16
// warps, each with two independent pairs and the Philox work to overlap).
template <int ILP, bool EM = false>
__global__ void __maxnreg__(ILP == 2 ? 72 : 128) jj_kernel_packed(const JJLaunchArgs A) {
  jj_kernel_body<ILP, EM, ILP >= 4>(A);
}

// Four paths per thread held to 96 registers (20 warps per SM in blocks of
// 128): the autotuner weighs the extra warps against the compiler's freedom
// to overlap.
template <bool EM = false>
__global__ void __maxnreg__(96) jj_kernel_packed4_cap96(const JJLaunchArgs A) {
  jj_kernel_body<4, EM, true>(A);
}

// ---- small ensembles: steps and noise in different warps -------------------
//
// With fewer warps than schedulers a launch lasts as long as one path's chain
// of dependent operations, and there the noise, which depends on no state, is
// better drawn elsewhere: a CTA holds kPairs pairs of warps, one stepping 32
// paths, the other drawing their Gaussians ahead into a ring of two blocks of
// 64 steps (named barriers hand the blocks over; blocks of 32 steps: 197 us
// where 64 take 164).  Four warps per CTA, so that each has a scheduler to
// itself.  The chain of a step is 13 FP32 operations (x -> force -> v~ -> x'), 52
// cycles at 4 each; rint(x) on it is taken as (x + 1.5 2^23) - 1.5 2^23, the same
// value for |x| < 2^22 in two additions where the conversion unit takes longer,
// and a group's floor(x) from two comparisons.  The steps' values and roundings
// are those of the one-path kernel: bit-identical.
// 1024 paths, 20,000 steps: 0.80 ms (83 cycles per step: the chain, x's fold after
// every fourth step, and the step's other operations issued in between) against
// 2.19 ms for the fastest kernel that draws and steps in one warp.
constexpr int kPairs = 2;               // stepping warps per CTA
constexpr int kWsBlock = 64 * kPairs;
constexpr uint32_t kRingGroups = 16;    // groups of 4 steps per ring block (aligned to 64 steps)
constexpr float kRoundMagic = 12582912.0f;
// Largest |v| at a group's start for which x moves by less than one period in
// the group's steps and predictors, so that floor(x) is -1, 0 or 1 (and |x|
// far below 2^22): over four steps |v| grows to at most q^4 (|v| + 4 kick), q =
// 1 + 2 gamma dt, kick = twice a step's largest force and noise (a 24-bit
// uniform's Gaussian is below 5.8).
__host__ __device__ inline double jj_ws_vmax(double gamma, double a, double f, double dt, double s) {
  const double q = 1.0 + 2.0 * gamma * dt, q4 = q * q * q * q;
  const double kick = 2.0 * (dt * (6.2832 + fabs(a) + fabs(f)) + 5.8 * s);
  return 0.98 / (5.0 * dt * q4) - 4.0 * kick;
}

__device__ __forceinline__ float jj_force_lat(float x, float A) {
  const float b = 0.25f - fabsf(x - __fsub_rn(__fadd_rn(x, kRoundMagic), kRoundMagic));
  const float s = b * b;
  float p = -2.484164429e+02f;  // as in jj_force
  p = fmaf(p, s, 4.809764709e+02f);
  p = fmaf(p, s, -5.127142334e+02f);
  p = fmaf(p, s, 2.597572937e+02f);
  p = fmaf(p, s, -3.947841644e+01f);
  return fmaf(b, p, A);
}

template <bool ACC, bool EM>
__device__ __forceinline__ void jj_step_lat(float &x, float &v, float &acc, float z, const JJConsts &c, float e0,
                                            float e1) {
  const float vn = fmaf(c.s, z, v);
  const float F1 = jj_force_lat(x, fmaf(-c.gamma, v, e0));
  if (EM) {
    x = fmaf(c.dt, v, x);
    v = fmaf(c.dt, F1, vn);
    if (ACC) acc += v;
    return;
  }
  const float xt = fmaf(c.dt, v, x);
  const float vt = fmaf(c.dt, F1, vn);
  const float F2 = jj_force_lat(xt, fmaf(-c.gamma, vt, e1));
  x = fmaf(c.h, v + vt, x);
  v = fmaf(c.h, F1 + F2, vn);
  if (ACC) acc += v;
}

__device__ __forceinline__ void pair_bar_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_bar_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// A whole group: four steps, then x back into [0, 1) knowing that it moved by
// less than one period (the same x and w as jj_wrap).
template <bool ACC, bool EM>
__device__ __forceinline__ void jj_ws_group(float &x, int &w, float &v, float &acc, const float4 &z, const JJConsts &c,
                                            const float4 &d, float d4) {
  jj_step_lat<ACC, EM>(x, v, acc, z.x, c, d.x, d.y);
  jj_step_lat<ACC, EM>(x, v, acc, z.y, c, d.y, d.z);
  jj_step_lat<ACC, EM>(x, v, acc, z.z, c, d.z, d.w);
  jj_step_lat<ACC, EM>(x, v, acc, z.w, c, d.w, d4);
  const float up = __fsub_rn(x, 1.0f), dn = __fadd_rn(x, 1.0f);
  const bool hi = x >= 1.0f, lo = x < 0.0f;
  w += (hi ? 1 : 0) - (lo ? 1 : 0);
  x = hi ? up : (lo ? dn : x);
}

// A whole ring block on one side of the window's start.  Returns
// whether every group started with |v| <= vmax (warp-uniform); if not the
// caller repeats the block group by group.
template <bool ACC, bool EM>
__device__ __forceinline__ bool jj_ws_block_steps(float &x, int &w, float &v, float &acc, const float4 *zr,
                                                  const JJConsts &c, const float *tab, int P, int &k, float vmax) {
  bool bad = false;
  float4 z = zr[0], d = *reinterpret_cast<const float4 *>(tab + k);
  float d4 = tab[k + 4];
#pragma unroll 4
  for (uint32_t g = 0; g < kRingGroups; ++g) {
    // the next group's noise and drive, read during this group's steps
    k = k + 4 == P ? 0 : k + 4;
    const float4 zn = zr[((g + 1) & (kRingGroups - 1)) * 32], dn = *reinterpret_cast<const float4 *>(tab + k);
    const float d4n = tab[k + 4];
    bad |= !(fabsf(v) <= vmax);
    jj_ws_group<ACC, EM>(x, w, v, acc, z, c, d, d4);
    z = zn;
    d = dn;
    d4 = d4n;
  }
  return !__any_sync(0xffffffffu, bad);
}

// The steps of one group at its ends: those in [n0, n1), then those in [m0,
// m1) with the window sum, x folded after each part (as two jj_segment calls
// meeting inside the group do).
template <bool EM>
__device__ __forceinline__ void jj_ws_partial(float &x, int &w, float &v, float &acc, const float4 &z4,
                                              const JJConsts &c, const float *drive, int P, int &k, int64_t base,
                                              int64_t n0, int64_t n1, int64_t m0, int64_t m1) {
  const float z[4] = {z4.x, z4.y, z4.z, z4.w};
  bool any0 = false, any1 = false;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int64_t n = base + s;
    if (n >= n0 && n < n1) {
      const int kn = k + 1 == P ? 0 : k + 1;
      jj_step<false, EM>(x, v, acc, z[s], c, drive[k], drive[kn]);
      k = kn;
      any0 = true;
    }
  }
  if (any0) jj_wrap(x, w);
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int64_t n = base + s;
    if (n >= m0 && n < m1) {
      const int kn = k + 1 == P ? 0 : k + 1;
      jj_step<true, EM>(x, v, acc, z[s], c, drive[k], drive[kn]);
      k = kn;
      any1 = true;
    }
  }
  if (any1) jj_wrap(x, w);
}

// The unit of a pair of warps and the run's steps.
struct JJWsUnit {
  int32_t path_begin, n_paths;  // within the point
  uint32_t point;
  int64_t offset;               // of its first path in the state arrays
  int64_t n_begin, n_end;
};

// One warp of a pair (`steps`: the stepping one) over its unit; tab holds the
// point's drive table, ring the pair's Gaussians.
template <bool EM>
__device__ __forceinline__ void jj_ws_pair(const JJWsUnit &r, const JJConsts &c, const JJState &st,
                                           const PhiloxKeys &keys, int P, const float *tab, const float *bm_tab,
                                           float4 (*ring)[kRingGroups][32], int pair, bool steps, uint32_t *err,
                                           Moments *out) {
  const int lane = threadIdx.x & 31;
  const int64_t nb = r.n_begin, ne = r.n_end < c.steps ? r.n_end : c.steps;
  const uint32_t g0 = (uint32_t)(nb >> 2), g1 = ne > nb ? (uint32_t)((ne - 1) >> 2) : g0;
  const uint32_t nblk = ne > nb ? g1 / kRingGroups - g0 / kRingGroups + 1u : 0u;
  const int bar_full = 1 + 4 * pair, bar_empty = 3 + 4 * pair;
  if (!steps) {
    // ---- noise ----
    const uint32_t pid = (uint32_t)(r.path_begin + lane);
    for (uint32_t i = 0; i < nblk; ++i) {
      const int b = (int)(i & 1u);
      const uint32_t lo = i == 0 ? g0 : (g0 / kRingGroups + i) * kRingGroups;
      const uint32_t hi = i + 1 == nblk ? g1 : (lo | (kRingGroups - 1u));
      if (i >= 2) pair_bar_sync(bar_empty + b);
#pragma unroll 2
      for (uint32_t g = lo; g <= hi; ++g) {
        const uint4 wd = philox4x32_10(make_uint4(g, pid, r.point, kTagJosephson), keys);
        float2 z02, z13;
        box_muller_tab2(wd.x, wd.y, wd.z, wd.w, bm_tab, z02, z13);
        ring[b][g % kRingGroups][lane] = make_float4(z02.x, z13.x, z02.y, z13.y);
      }
      pair_bar_arrive(bar_full + b);
    }
    return;
  }
  // ---- steps ----
  const bool valid[1] = {lane < r.n_paths};
  const int64_t gi = r.offset + lane;
  float x = 0.0f, v = 0.0f;
  int w = 0;
  double vs[1] = {0.0};
  if (valid[0]) {
    x = st.x_in[gi];
    v = st.v_in[gi];
    if (st.w_in) w = st.w_in[gi];
    if (st.vsum_in) vs[0] = st.vsum_in[gi];
  }
  jj_wrap(x, w);
  float acc = 0.0f;
  int k = (int)(nb % P);
  const int64_t ws = c.wstart;
  const float vmax = (float)jj_ws_vmax(c.gamma, c.a, c.f, c.dt64, c.s);
  for (uint32_t i = 0; i < nblk; ++i) {
    const int b = (int)(i & 1u);
    const uint32_t lo = i == 0 ? g0 : (g0 / kRingGroups + i) * kRingGroups;
    const uint32_t hi = i + 1 == nblk ? g1 : (lo | (kRingGroups - 1u));
    const float4 *zr = &ring[b][0][lane];
    pair_bar_sync(bar_full + b);
    const int64_t n0 = (int64_t)lo << 2, n1 = ((int64_t)hi + 1) << 2;
    bool done = false;
    if (n0 >= nb && n1 <= ne && lo % kRingGroups == 0u && hi % kRingGroups == kRingGroups - 1u && (ws <= n0 || ws >= n1)) {
      const float x0 = x, v0 = v, acc0 = acc;
      const int w0 = w, k0 = k;
      done = ws <= n0 ? jj_ws_block_steps<true, EM>(x, w, v, acc, zr, c, tab, P, k, vmax)
                      : jj_ws_block_steps<false, EM>(x, w, v, acc, zr, c, tab, P, k, vmax);
      if (!done) {
        x = x0;
        v = v0;
        acc = acc0;
        w = w0;
        k = k0;
      }
    }
    if (!done) {
      for (uint32_t g = lo; g <= hi; ++g) {
        const int64_t m0 = (int64_t)g << 2, m1 = m0 + 4;
        const float4 z = zr[(g % kRingGroups) * 32];
        if (m0 >= nb && m1 <= ne && (ws <= m0 || ws >= m1) && !__any_sync(0xffffffffu, !(fabsf(v) <= vmax))) {
          const float4 d = *reinterpret_cast<const float4 *>(tab + k);
          if (ws <= m0)
            jj_ws_group<true, EM>(x, w, v, acc, z, c, d, tab[k + 4]);
          else
            jj_ws_group<false, EM>(x, w, v, acc, z, c, d, tab[k + 4]);
          k = k + 4 == P ? 0 : k + 4;
        } else {
          jj_ws_partial<EM>(x, w, v, acc, z, c, tab, P, k, m0, nb, ne < ws ? ne : ws, nb > ws ? nb : ws, ne);
        }
      }
    }
    if (i + 2 < nblk) pair_bar_arrive(bar_empty + b);
    if (((hi + 1u) & 15u) == 0u) {  // flush at absolute 64-step boundaries, as jj_segment
      vs[0] += (double)acc;
      acc = 0.0f;
    }
  }
  vs[0] += (double)acc;
  if (valid[0]) {
    st.x_out[gi] = x;
    st.v_out[gi] = v;
    st.w_out[gi] = w;
    st.vsum_out[gi] = vs[0];
  }
  if (err && __any_sync(0xffffffffu, valid[0] && !(isfinite(x) && isfinite(v))) && lane == 0)
    atomicOr(err, kErrNonFinite);
  jj_unit_moments<1>(out, r.n_end, c, vs, valid, lane);
}

template <bool EM>
__global__ void __launch_bounds__(kWsBlock) jj_ws_kernel(const JJLaunchArgs A) {
  extern __shared__ float4 drive_s4[];  // per pair: a cos(2 pi k / P) + f, k = 0 .. P + 3
  __shared__ float bm_tab[2 * kBmTable];
  __shared__ float4 ring[kPairs][2][kRingGroups][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pair = warp % kPairs;
  const bool steps = warp < kPairs;
  const int u = A.unit_begin + (int)blockIdx.x * kPairs + pair;
  const bool have = u < A.unit_end;
  const JJUnit un = A.units[have ? u : A.unit_begin];
  const JJConsts c = A.consts[un.point];
  float *tab = reinterpret_cast<float *>(drive_s4) + jj_table_stride(A.P) * pair;
  if (steps)
    for (int q = lane; q < A.P + 4; q += 32) tab[q] = fmaf(c.a, A.drive[q < A.P ? q : q % A.P], c.f);
  fill_bm_table(bm_tab);
  __syncthreads();
  if (!have) return;
  const JJWsUnit r{un.path_begin, un.n_paths, (uint32_t)un.point, c.path_offset + un.path_begin, A.n_begin, A.n_end};
  jj_ws_pair<EM>(r, c, A.st, A.keys, A.P, tab, bm_tab, ring[pair], pair, steps, A.err, A.partials + u);
}

__global__ void jj_prepare_kernel(const sde_jj_point *pts, int n_points, int P,
                                  const int64_t *steps, const int64_t *offsets,
                                  const int64_t *paths, JJConsts *out, float *drive) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n_points) {
    const sde_jj_point p = pts[t];
    const double dt = 2.0 * 3.14159265358979323846 / (p.omega * (double)P);
    JJConsts c;
    c.gamma = (float)p.gamma;
    c.a = (float)p.a;
    c.f = (float)p.f;
    c.dt = (float)dt;
    c.h = (float)(0.5 * dt);
    c.s = (float)sqrt(2.0 * p.gamma * p.D * dt);
    c.paths = (int32_t)paths[t];
    c.pad = 0;
    c.steps = steps[t];
    c.wstart = steps[t] - steps[t] / 2;
    c.path_offset = offsets[t];
    c.dt64 = dt;
    out[t] = c;
  }
  if (t < P) drive[t] = (float)cospi(2.0 * (double)t / (double)P);
}

// FP64 sum over the block in a fixed order; every thread receives it.
__device__ __forceinline__ double block_sum64(double a, double *red) {
  a = warp_sum(a);
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  if (warps == 1) return a;
  __syncthreads();
  if (lane == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  return warp_sum(lane < warps ? red[lane] : 0.0);
}

// The observables of one point from the moments of its units [u0, u1), by one
// block: mean = sum n_i mean_i / n, then M2 = sum m2_i + n_i (mean_i - mean)^2
// (deterministic: fixed strides and tree).  Two passes with one division
// instead of a pairwise merge per unit, whose two FP64 divisions took ~1.2 us
// each on one lane's chain: 1,000,000 paths through the allocation-free entry
// point, 1000 steps, 2.99 -> 1.59 ms together with its packed kernels.
__device__ __forceinline__ void jj_point_row(const Moments *partials, int u0, int u1, int64_t steps, double dt,
                                             int64_t n_end, sde_obs_row *out, double *red) {
  double n = 0.0, sum = 0.0;
  for (int u = u0 + (int)threadIdx.x; u < u1; u += blockDim.x) {
    const Moments m = partials[u];
    n += m.n;
    sum = fma(m.n, m.mean, sum);
  }
  n = block_sum64(n, red);
  sum = block_sum64(sum, red);
  const double mean = n > 0.0 ? sum / n : 0.0;
  double m2 = 0.0;
  for (int u = u0 + (int)threadIdx.x; u < u1; u += blockDim.x) {
    const Moments m = partials[u];
    const double d = m.mean - mean;
    m2 += fma(m.n * d, d, m.m2);
  }
  m2 = block_sum64(m2, red);
  if (threadIdx.x == 0) {
    const int64_t reach = n_end < steps ? n_end : steps;
    sde_obs_row row;
    row.count = n;
    row.mean = mean;
    row.var = n > 1.0 ? m2 / (n - 1.0) : 0.0;
    row.se = n > 0.0 ? sqrt(row.var / n) : 0.0;
    row.t = (double)reach * dt;
    *out = row;
  }
}

// Threads of a block over n_units units: a warp for a few, more where the
// strided loop would be long.
int jj_row_threads(int n_units) { return n_units <= 64 ? 32 : (n_units <= 1024 ? 256 : 1024); }

__global__ void jj_finalize_kernel(const JJConsts *consts, const int2 *range, const Moments *partials, int64_t n_end,
                                   sde_obs_row *obs) {
  __shared__ double red[32];
  const int p = blockIdx.x;
  jj_point_row(partials, range[p].x, range[p].y, consts[p].steps, consts[p].dt64, n_end, obs + p, red);
}

__global__ void philox_fill_kernel(const uint4 *ctr, uint2 key, uint4 *out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = philox4x32_10(ctr[i], key);
}

__global__ void box_muller_fill_kernel(const uint4 *ctr, uint2 key, float4 *z, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint4 r = philox4x32_10(ctr[i], key);
    float4 o;
    box_muller(r.x, r.y, o.x, o.y);
    box_muller(r.z, r.w, o.z, o.w);
    z[i] = o;
  }
}

// Box-Muller of given word pairs (w0, w1) -> (z0, z1): variant 0 the
// library's default transform, 1 the Josephson kernels' (table angle,
// hardware logarithm).
__global__ void box_muller_words_kernel(const uint2 *w, int64_t n, int variant, float2 *z) {
  __shared__ float tab[2 * kBmTable];
  fill_bm_table(tab);
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint2 p = w[i];
    float2 o;
    if (variant == 1)
      box_muller_tab(p.x, p.y, tab, o.x, o.y);
    else
      box_muller(p.x, p.y, o.x, o.y);
    z[i] = o;
  }
}

size_t jj_ws_smem(int P) { return sizeof(float) * (size_t)jj_table_stride(P) * kPairs; }

void *jj_kernel_ptr(int variant) {
  switch (variant) {
    case 1: return (void *)jj_kernel<1>;
    case 2: return (void *)jj_kernel_packed<2>;
    case 4: return (void *)jj_kernel_packed<4>;
    case 14: return (void *)jj_kernel_packed4_cap96<>;
    case 11: return (void *)jj_kernel_cap64<1>;
    case 12: return (void *)jj_kernel_cap64<2>;
    case 101: return (void *)jj_kernel<1, true>;
    case 102: return (void *)jj_kernel_packed<2, true>;
    case 104: return (void *)jj_kernel_packed<4, true>;
    case 111: return (void *)jj_kernel_cap64<1, true>;
    case 112: return (void *)jj_kernel_cap64<2, true>;
    case 114: return (void *)jj_kernel_packed4_cap96<true>;
    case kJJWarpPairs: return (void *)jj_ws_kernel<false>;
    case 100 + kJJWarpPairs: return (void *)jj_ws_kernel<true>;
  }
  return nullptr;
}

}  // namespace

cudaError_t jj_prepare(const sde_jj_point *points_dev, int n_points, int P, const int64_t *steps_dev,
                       const int64_t *offsets_dev, const int64_t *paths_dev, JJConsts *consts_dev,
                       float *drive_dev, cudaStream_t s) {
  const int n = n_points > P ? n_points : P;
  jj_prepare_kernel<<<(n + 255) / 256, 256, 0, s>>>(points_dev, n_points, P, steps_dev, offsets_dev,
                                                    paths_dev, consts_dev, drive_dev);
  return cudaGetLastError();
}

int jj_ws_grid(int n_units) { return (n_units + kPairs - 1) / kPairs; }
int jj_ws_block() { return kWsBlock; }

// The warp-pair kernel takes drive tables of whole groups that fit a warp's
// table, and points whose velocities leave the block path (jj_ws_vmax) rarely:
// the driven velocity is of the order of a / omega + f / gamma and the noise's
// sqrt(D), a few of each.
bool jj_ws_eligible(const sde_jj_point *pts, int n_points, int P) {
  if (P % 4 != 0 || P > kWarpTableMaxP) return false;
  for (int i = 0; i < n_points; ++i) {
    const sde_jj_point &p = pts[i];
    const double dt = 2.0 * 3.14159265358979323846 / (p.omega * (double)P);
    const double vmax = jj_ws_vmax(p.gamma, p.a, p.f, dt, sqrt(2.0 * p.gamma * p.D * dt));
    if (!(vmax >= 2.0 * (fabs(p.a) / p.omega + fabs(p.f) / p.gamma + 6.0 * sqrt(p.D)) + 3.0)) return false;
  }
  return true;
}

// `ilp` encodes the variant: 1, 2, 4 = paths per thread; +10 = fewer registers
// (64 for 1 and 2 paths per thread, 96 for 4); kJJWarpPairs = one path per
// thread, the noise drawn by a second warp; +100 = Euler-Maruyama.
cudaError_t jj_launch(const JJLaunchArgs &a, int ilp, int block, int grid, cudaStream_t s) {
  const size_t smem = jj_smem_bytes(a.P, block);
  switch (ilp) {
    case 1: jj_kernel<1><<<grid, block, smem, s>>>(a); break;
    case 2: jj_kernel_packed<2><<<grid, block, smem, s>>>(a); break;
    case 4: jj_kernel_packed<4><<<grid, block, smem, s>>>(a); break;
    case 14: jj_kernel_packed4_cap96<><<<grid, block, smem, s>>>(a); break;
    case 11: jj_kernel_cap64<1><<<grid, block, smem, s>>>(a); break;
    case 12: jj_kernel_cap64<2><<<grid, block, smem, s>>>(a); break;
    // Euler-Maruyama variants: the code + 100
    case 101: jj_kernel<1, true><<<grid, block, smem, s>>>(a); break;
    case 102: jj_kernel_packed<2, true><<<grid, block, smem, s>>>(a); break;
    case 104: jj_kernel_packed<4, true><<<grid, block, smem, s>>>(a); break;
    case 111: jj_kernel_cap64<1, true><<<grid, block, smem, s>>>(a); break;
    case 112: jj_kernel_cap64<2, true><<<grid, block, smem, s>>>(a); break;
    case 114: jj_kernel_packed4_cap96<true><<<grid, block, smem, s>>>(a); break;
    case kJJWarpPairs: jj_ws_kernel<false><<<grid, kWsBlock, jj_ws_smem(a.P), s>>>(a); break;
    case 100 + kJJWarpPairs: jj_ws_kernel<true><<<grid, kWsBlock, jj_ws_smem(a.P), s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

int jj_max_blocks_per_sm(int ilp, int block, int P) {
  int nb = 0;
  void *k = jj_kernel_ptr(ilp);
  if (!k) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, block, jj_smem_bytes(P, block)) != cudaSuccess)
    return 0;
  return nb;
}

// The dynamic shared memory limit is a per-function maximum shared by every
// launch in the process, so it is raised once, to what the largest table
// layout (P = kWarpTableMaxP, kJJMaxBlock threads) needs, and never lowered.
cudaError_t jj_configure() {
  static const cudaError_t status = [] {
    const int smem = (int)jj_smem_bytes(kWarpTableMaxP, kJJMaxBlock);
    const int variants[] = {1, 2, 4, 11, 12, 14, 101, 102, 104, 111, 112, 114};
    for (int v : variants) {
      const cudaError_t e = cudaFuncSetAttribute(jj_kernel_ptr(v), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }();
  return status;
}

cudaError_t jj_finalize(const JJConsts *consts, const int2 *point_range, int n_points, int max_units,
                        const Moments *partials, int64_t n_end, sde_obs_row *obs, cudaStream_t s) {
  jj_finalize_kernel<<<n_points, jj_row_threads(max_units), 0, s>>>(consts, point_range, partials, n_end, obs);
  return cudaGetLastError();
}

cudaError_t philox_fill(const uint32_t *ctr, uint64_t seed, uint32_t *out, int64_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t blocks = (n + 255) / 256;
  philox_fill_kernel<<<(int)(blocks < 65535 ? blocks : 65535), 256, 0, s>>>(
      (const uint4 *)ctr, make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)), (uint4 *)out, n);
  return cudaGetLastError();
}

cudaError_t box_muller_fill(const uint32_t *ctr, uint64_t seed, float *z, int64_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t blocks = (n + 255) / 256;
  box_muller_fill_kernel<<<(int)(blocks < 65535 ? blocks : 65535), 256, 0, s>>>(
      (const uint4 *)ctr, make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)), (float4 *)z, n);
  return cudaGetLastError();
}

cudaError_t box_muller_words(const uint32_t *w, int64_t n, int variant, float *z, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t blocks = (n + 255) / 256;
  box_muller_words_kernel<<<(int)(blocks < 4096 ? blocks : 4096), 256, 0, s>>>((const uint2 *)w, n, variant,
                                                                               (float2 *)z);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the per-path kernel (sde_josephson_run_noalloc).
//
// Some callers cannot call cudaMalloc: code that runs inside another
// framework's memory pool or arena (which forbids allocations behind its
// back), code that is itself being captured into a CUDA graph by a host
// program, or embedded/real-time hosts that pre-reserve all device memory at
// start-up.  For them this entry point keeps its only scratch -- one
// reduction partial per warp of 32 paths -- in a fixed array in the
// library's static device memory instead of a workspace allocated by
// sde_create.  Every GPU that loads the library holds this array until the
// process exits.
// ---------------------------------------------------------------------------

#define SDE_NOALLOC_UNITS (SDE_NOALLOC_MAX_PATHS / 32)

namespace {

// 32768 partials x 24 bytes = 768 KiB.  Shared by every call on a device;
// it keeps the previous call's contents.  Each call writes every slot it
// later reads, so nothing has to be cleared first.
static __device__ __align__(256) Moments g_noalloc_partials[SDE_NOALLOC_UNITS];

struct NoallocArgs {
  JJConsts c;
  double inv4P;  // 1 / (4 P)
  int32_t P;
  int32_t n_paths;
  int64_t n_begin, n_end;
  PhiloxKeys keys;
  JJState st;
  Moments *partials;  // device address of g_noalloc_partials
};

// cos(2 pi k / P) rounded to FP32, k in [0, P].
__device__ __forceinline__ float drive_entry(int k, int P, double inv4P) { return (float)cos_ratio64(k, P, inv4P); }

// ILP paths per thread (2 or 4, packed pairs as in the persistent kernels), the moments taken per 32 paths as with one path per thread: the
// same arithmetic and unit decomposition as the plain schedule with one path
// per thread whatever ILP.
template <int ILP>
__device__ __forceinline__ void jj_noalloc_body(const NoallocArgs &A) {
  extern __shared__ float4 drive_s4[];  // a cos(2 pi k / P) + f, k = 0 .. P + 3
  __shared__ float bm_tab[2 * kBmTable];
  float *drive_s = reinterpret_cast<float *>(drive_s4);
  const JJConsts &c = A.c;
  for (int i = threadIdx.x; i < A.P + 4; i += blockDim.x)
    drive_s[i] = fmaf(c.a, drive_entry(i % A.P, A.P, A.inv4P), c.f);
  fill_bm_table(bm_tab);
  __syncthreads();
  const int u = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * ILP;  // first unit of 32 paths
  const int n_units = (A.n_paths + 31) / 32;
  if (u >= n_units) return;
  const int lane = threadIdx.x & 31;
  float x[ILP], v[ILP];
  int w[ILP];
  double vs[ILP];
  uint32_t pid[ILP];
  bool valid[ILP];
#pragma unroll
  for (int i = 0; i < ILP; ++i) {
    const int j = (u + i) * 32 + lane;
    valid[i] = j < A.n_paths;
    pid[i] = (uint32_t)j;
    x[i] = v[i] = 0.0f;
    w[i] = 0;
    vs[i] = 0.0;
    if (valid[i]) {
      x[i] = A.st.x_in[j];
      v[i] = A.st.v_in[j];
      if (A.st.w_in) w[i] = A.st.w_in[j];
      if (A.st.vsum_in) vs[i] = A.st.vsum_in[j];
    }
    jj_wrap(x[i], w[i]);
  }
  const int64_t ne = A.n_end < c.steps ? A.n_end : c.steps;
  if (A.n_begin < ne) {
    int k = (int)(A.n_begin % A.P);
    const int64_t split = ne < c.wstart ? ne : c.wstart;
    jj_segment<ILP, false, false, true, ILP >= 4>(x, w, v, vs, c, drive_s, A.P, k, A.n_begin, split, A.keys, pid, 0u,
                                                  bm_tab);
    jj_segment<ILP, true, false, true, ILP >= 4>(x, w, v, vs, c, drive_s, A.P, k,
                                                 A.n_begin > c.wstart ? A.n_begin : c.wstart, ne, A.keys, pid, 0u,
                                                 bm_tab);
  }
#pragma unroll
  for (int i = 0; i < ILP; ++i) {
    if (valid[i]) {
      const int j = (u + i) * 32 + lane;
      A.st.x_out[j] = x[i];
      A.st.v_out[j] = v[i];
      A.st.w_out[j] = w[i];
      A.st.vsum_out[j] = vs[i];
    }
    if (u + i < n_units) {
      const double vsi[1] = {vs[i]};
      const bool vi[1] = {valid[i]};
      jj_unit_moments<1>(A.partials + u + i, A.n_end, c, vsi, vi, lane);
    }
  }
}

__global__ void __maxnreg__(72) jj_noalloc_packed2_kernel(const NoallocArgs A) { jj_noalloc_body<2>(A); }
__global__ void __maxnreg__(96) jj_noalloc_packed4_kernel(const NoallocArgs A) { jj_noalloc_body<4>(A); }

// Small ensembles: a pair of warps per 32 paths (jj_ws_pair).
__global__ void __launch_bounds__(kWsBlock) jj_noalloc_ws_kernel(const NoallocArgs A) {
  extern __shared__ float4 drive_s4[];
  __shared__ float bm_tab[2 * kBmTable];
  __shared__ float4 ring[kPairs][2][kRingGroups][32];
  float *tab = reinterpret_cast<float *>(drive_s4);
  const int pair = (threadIdx.x >> 5) % kPairs;
  const bool steps = threadIdx.x < 32 * kPairs;
  const JJConsts &c = A.c;
  for (int i = threadIdx.x; i < A.P + 4; i += kWsBlock)
    tab[i] = fmaf(c.a, drive_entry(i % A.P, A.P, A.inv4P), c.f);
  fill_bm_table(bm_tab);
  __syncthreads();
  const int u = (int)blockIdx.x * kPairs + pair;
  if (u >= (A.n_paths + 31) / 32) return;
  const JJWsUnit r{u * 32, A.n_paths - u * 32 < 32 ? A.n_paths - u * 32 : 32, 0u, (int64_t)u * 32, A.n_begin, A.n_end};
  jj_ws_pair<false>(r, c, A.st, A.keys, A.P, tab, bm_tab, ring[pair], pair, steps, nullptr, A.partials + u);
}

__global__ void jj_noalloc_finalize(const Moments *partials, int n_units, int64_t steps, double dt,
                                    int64_t n_end, sde_obs_row *obs) {
  __shared__ double red[32];
  jj_point_row(partials, 0, n_units, steps, dt, n_end, obs, red);
}

}  // namespace

namespace {
// Device address of g_noalloc_partials, resolved once per device.
constexpr int kMaxDevices = 64;
Moments *g_noalloc_ptr[kMaxDevices] = {};
std::mutex g_noalloc_mutex;
}  // namespace

}  // namespace sde

extern "C" sde_status sde_josephson_run_noalloc(const sde_jj_point *point, int32_t steps_per_period,
                                                int64_t n_paths, int64_t total_steps, uint64_t seed,
                                                int64_t n_begin, int64_t n_end, const float *x_in_dev,
                                                const float *v_in_dev, const int32_t *w_in_dev,
                                                const double *vsum_in_dev, float *x_out_dev,
                                                float *v_out_dev, int32_t *w_out_dev,
                                                double *vsum_out_dev, sde_obs_row *obs_dev,
                                                void *stream) {
  using namespace sde;
  clear_error();
  SDE_CHECK_ARG(point != nullptr, "point is NULL");
  SDE_CHECK_ARG(n_paths >= 0, "n_paths must be >= 0");
  if (n_paths > SDE_NOALLOC_MAX_PATHS) {
    set_error("invalid argument: sde_josephson_run_noalloc handles at most " +
              std::to_string(SDE_NOALLOC_MAX_PATHS) + " paths per call (got " +
              std::to_string(n_paths) + "); use sde_create/sde_run_ensemble for larger ensembles");
    return SDE_ERR_INVALID_ARG;
  }
  SDE_CHECK_ARG(steps_per_period >= 1 && steps_per_period <= 4096, "steps_per_period must be in [1, 4096]");
  SDE_CHECK_ARG(total_steps >= 0 && total_steps <= (1ll << 33), "total_steps out of range");
  SDE_CHECK_ARG(n_begin >= 0 && n_end >= n_begin && n_end <= (1ll << 33), "need 0 <= n_begin <= n_end");
  SDE_CHECK_ARG(isfinite(point->gamma) && isfinite(point->a) && isfinite(point->omega) &&
                    isfinite(point->f) && isfinite(point->D),
                "point parameters must be finite");
  SDE_CHECK_ARG(point->omega > 0.0 && point->gamma > 0.0 && point->D >= 0.0,
                "need omega > 0, gamma > 0, D >= 0");
  SDE_CHECK_ARG(obs_dev != nullptr, "obs_dev is NULL");
  if (n_paths > 0)
    SDE_CHECK_ARG(x_in_dev && v_in_dev && x_out_dev && v_out_dev && w_out_dev && vsum_out_dev,
                  "x_in, v_in, x_out, v_out, w_out and vsum_out must be non-NULL");
  int dev = 0;
  SDE_CUDA_TRY(cudaGetDevice(&dev));
  SDE_CHECK_ARG(dev >= 0 && dev < kMaxDevices, "device index out of range");
  Moments *partials = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
      void *p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_partials);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_partials)");
      g_noalloc_ptr[dev] = (Moments *)p;
    }
    partials = g_noalloc_ptr[dev];
  }
  cudaStream_t s = (cudaStream_t)stream;
  NoallocArgs a{};
  // the same FP64 expressions, rounded once, as jj_prepare_kernel
  const double dt = 2.0 * 3.14159265358979323846 / (point->omega * (double)steps_per_period);
  a.c.gamma = (float)point->gamma;
  a.c.a = (float)point->a;
  a.c.f = (float)point->f;
  a.c.dt = (float)dt;
  a.c.h = (float)(0.5 * dt);
  a.c.s = (float)sqrt(2.0 * point->gamma * point->D * dt);
  a.c.paths = (int32_t)n_paths;
  a.c.steps = total_steps;
  a.c.wstart = total_steps - total_steps / 2;
  a.c.dt64 = dt;
  a.inv4P = 1.0 / (4.0 * (double)steps_per_period);
  a.P = steps_per_period;
  a.n_paths = (int32_t)n_paths;
  a.n_begin = n_begin;
  a.n_end = n_end;
  a.keys = philox_round_keys(seed);
  a.st = JJState{x_in_dev, v_in_dev, w_in_dev, vsum_in_dev, x_out_dev, v_out_dev, w_out_dev, vsum_out_dev};
  a.partials = partials;
  const int n_units = (int)((n_paths + 31) / 32);
  if (n_units > 0) {
    // Pairs of warps up to kWsUnitsPerSm units per SM as in the persistent
    // schedule; then two paths per thread, and four where they still give each
    // SM 20 warps (what 96 registers allow).  1000 steps against the scalar
    // one-path kernel (both with the same reduction): 1000 paths 62 vs 101 us,
    // 38,000 122 vs 150, 50,000 171 vs 210, 500,000 0.88 vs 1.15 ms.
    int sms = 0;
    SDE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = sizeof(float) * (size_t)(steps_per_period + 4);
    if (n_units <= kWsUnitsPerSm * sms && jj_ws_eligible(point, 1, steps_per_period))
      jj_noalloc_ws_kernel<<<jj_ws_grid(n_units), kWsBlock, smem, s>>>(a);
    else if (n_units >= 4 * 20 * sms)
      jj_noalloc_packed4_kernel<<<(n_units + 15) / 16, 128, smem, s>>>(a);
    else
      jj_noalloc_packed2_kernel<<<(n_units + 7) / 8, 128, smem, s>>>(a);
    SDE_CUDA_TRY(cudaGetLastError());
  }
  jj_noalloc_finalize<<<1, jj_row_threads(n_units), 0, s>>>(partials, n_units, total_steps, dt, n_end, obs_dev);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}
