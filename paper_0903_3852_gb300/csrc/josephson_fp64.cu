// josephson_fp64.cu -- Eq. 1 advanced by Alg. 2 in double precision on the
// GPU, the counterpart of the paper's double-precision run of Fig. 2 (its
// FP32 and FP64 ensembles agree to within the statistical error of the
// histogram, Sec. 5).  It exists to measure the FP32 path's error on the GPU
// itself: same noise stream as the FP32 kernels (Philox4x32-10 block n / 4 of
// counter (path, point, tag 1), identical 24-bit uniforms), with the
// Box-Muller transform, the potential force and the drive evaluated in FP64.
//
// One thread per path, one launch per point; positions are plain FP64 values
// (53 bits hold the fractional part to 1e-12 of a period out to 10^4 periods,
// so no winding count is kept).
//
// What bounds it: the FP64 pipe, one warp instruction per 16 cycles and SM.  So
// the transcendental functions are written in as few FP64 operations as their
// arguments allow (ranges known, no special cases): 14 for a force, 16 for a
// Gaussian, 8 for the rest of a step, 52 per step against 86 with the
// library's cospi, log, sqrt and sincospi; the drive term, the tables of the
// logarithm and of the angle's sine and cosine are formed once per block, and
// integers become doubles through their bit patterns.  Blocks are sized so that
// every SM holds the same number of paths.  65536 paths, 400 steps: 4.96 -> 2.64
// ms (9.9e9 path-steps/s); 3000 paths 2.48 -> 0.69 ms.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "fp64_math.cuh"
#include "philox.cuh"

namespace sde {
namespace {

struct JJ64Args {
  double gamma, a, f;
  double dt, h, s;  // dt, dt / 2, sqrt(2 gamma D dt)
  int32_t P;
  uint32_t point;   // noise counter word c2
  int64_t n_paths;
  int64_t n_begin, n_end;
  int64_t wstart;   // the window holds state indices (wstart, S]
  const double *x_in, *v_in, *vsum_in;
  double *x_out, *v_out, *vsum_out;
  uint32_t *err;
  PhiloxKeys keys;
};

// Tables of a block (shared memory).
constexpr int kLogTable = 128;   // leading 7 bits of a mantissa
constexpr int kAngleTable = 64;  // sixty-fourths of a turn
struct Tables64 {
  double inv[kLogTable];     // c_i ~ 1 / (1 + (i + 1/2) / 128), at most 14 bits; c_0 = 1, c_127 = 1/2
  double two_log[kLogTable]; // 2 ln c_i
  double exponent[25];       // -2 (e - 24) ln 2
  double cs[kAngleTable], sn[kAngleTable];
};

__device__ __forceinline__ void fill_tables64(Tables64 &t) {
  for (int i = threadIdx.x; i < kLogTable; i += blockDim.x) {
    const double c = i == 0 ? 1.0 : (i == kLogTable - 1 ? 0.5 : rint(8192.0 / (1.0 + (i + 0.5) / kLogTable)) / 8192.0);
    t.inv[i] = c;
    t.two_log[i] = 2.0 * log(c);
  }
  for (int i = threadIdx.x; i < 25; i += blockDim.x) t.exponent[i] = (24 - i) * (2.0 * log(2.0));
  for (int i = threadIdx.x; i < kAngleTable; i += blockDim.x) sincospi(i / 32.0, &t.sn[i], &t.cs[i]);
}

// -2 ln(m 2^-24) for m in [1, 2^24].  m = 2^e f, f in [1, 2); with c_i from the
// leading bits of f, z = f c_i - 1 is exact and in (-0.004, 1/128], and
// -2 ln u = -2 (e - 24) ln 2 + 2 ln c_i - 2 ln(1 + z), the last as z times a
// degree-6 polynomial (interpolation at the Chebyshev nodes of the interval,
// within 1e-20).  c_0 = 1 and c_127 = 1/2 make the table terms cancel for u
// near 1, so the result keeps its relative accuracy there; u = 1 gives 0.
__device__ __forceinline__ double minus2_log24(uint32_t m, const Tables64 &t) {
  const uint32_t bits = __float_as_uint((float)m);  // exact: 24 bits
  const uint32_t mant = bits & 0x7FFFFFu;
  const int e = (int)(bits >> 23) - 127, i = (int)(mant >> 16);
  const double f = __hiloint2double((int)(0x3FF00000u | (mant >> 3)), (int)(mant << 29));
  const double z = fma(f, t.inv[i], -1.0);
  double q = -0.2828473837233479;
  q = fma(q, z, 0.3333355763843714);
  q = fma(q, z, -0.4000000966277093);
  q = fma(q, z, 0.5000000000732646);
  q = fma(q, z, -0.6666666666658018);
  q = fma(q, z, 0.9999999999999994);
  q = fma(q, z, -2.0);
  return fma(z, q, t.exponent[e] + t.two_log[i]);
}

// Box-Muller in FP64 from the same 24-bit uniforms as the FP32 path.  The
// angle 2 pi (j + 1) 2^-24 is the nearest sixty-fourth of a turn plus b, |b| <=
// pi / 64: sin b and cos b from short polynomials (interpolation at the
// Chebyshev nodes, within 3e-17), combined with the table by angle addition.
__device__ __forceinline__ void box_muller64(uint32_t w0, uint32_t w1, const Tables64 &t, double &z0, double &z1) {
  const double rho = sqrt_goldschmidt(minus2_log24((w0 >> 8) + 1u, t));
  const int j = (int)(w1 >> 8) + 1;
  const int q = (j + (1 << 17)) >> 18;
  const int rem = j - (q << 18);
  // 1.5 2^52 + rem by its bits, less 1.5 2^52: rem exactly; times 2 pi 2^-24
  const double b = (__longlong_as_double(0x4338000000000000ll + (long long)rem) - 6755399441055744.0) *
                   3.7450702829239286e-07;
  const double b2 = b * b;
  double ps = fma(b2, -0.00019840273845896154, 0.008333333324333688);
  ps = fma(b2, ps, -0.16666666666666546);
  const double sb = fma(b, b2 * ps, b);
  double pc = fma(b2, -0.001388799249796147, 0.041666666585670434);
  pc = fma(b2, pc, -0.4999999999999892);
  const double cm1 = b2 * pc;  // cos b - 1
  const double C = t.cs[q & (kAngleTable - 1)], S = t.sn[q & (kAngleTable - 1)];
  z0 = rho * fma(C, cm1, fma(-S, sb, C));
  z1 = rho * fma(S, cm1, fma(C, sb, S));
}

// A - 2 pi cos(2 pi x).
__device__ __forceinline__ double jj_force64(double x, double A) {
  const double b = 0.25 - fabs(x - rint(x));
  const double s = b * b;
  double p = -0.6339542652986321;  // -2 pi times the coefficients of sin2pi64_poly
  p = fma(p, s, 4.509654417248789);
  p = fma(p, s, -24.00131607613064);
  p = fma(p, s, 94.84243079652464);
  p = fma(p, s, -264.2625677114168);
  p = fma(p, s, 481.9571309735275);
  p = fma(p, s, -512.7409032401533);
  p = fma(p, s, 259.7575760906731);
  p = fma(p, s, -39.47841760435743);
  return fma(b, p, A);
}

__global__ void __launch_bounds__(512) jj64_kernel(const JJ64Args A) {
  extern __shared__ double drive_s[];  // [P]: a cos(2 pi k / P) + f
  __shared__ Tables64 tab;
  for (int k = threadIdx.x; k < A.P; k += blockDim.x)
    drive_s[k] = fma(A.a, cos2pi64((double)k / (double)A.P), A.f);
  fill_tables64(tab);
  __syncthreads();
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= A.n_paths) return;
  double x = A.x_in[j], v = A.v_in[j];
  double vs = A.vsum_in ? A.vsum_in[j] : 0.0;
  int32_t k = (int32_t)(A.n_begin % A.P);
  // Alg. 2: predictor with F(y_n, t_n), corrector with the mean of the two
  // stages; the same Gaussian in both
  auto step = [&](double psi, bool sum) {
    const int32_t k1 = k + 1 == A.P ? 0 : k + 1;
    const double vn = fma(A.s, psi, v);
    const double F1 = jj_force64(x, fma(-A.gamma, v, drive_s[k]));
    const double xt = fma(A.dt, v, x);
    const double vt = fma(A.dt, F1, vn);
    const double F2 = jj_force64(xt, fma(-A.gamma, vt, drive_s[k1]));
    x = fma(A.h, v + vt, x);
    v = fma(A.h, F1 + F2, vn);
    if (sum) vs += v;
    k = k1;
  };
  for (int64_t n = A.n_begin; n < A.n_end;) {
    const int64_t g = n >> 2;
    const uint4 w = philox4x32_10(make_uint4((uint32_t)g, (uint32_t)j, A.point, kTagJosephson), A.keys);
    double z[4];
    box_muller64(w.x, w.y, tab, z[0], z[1]);
    box_muller64(w.z, w.w, tab, z[2], z[3]);
    const int64_t base = g << 2;
    const bool whole = n == base && base + 4 <= A.n_end;
    if (whole && base + 1 > A.wstart) {
#pragma unroll
      for (int q = 0; q < 4; ++q) step(z[q], true);
    } else if (whole && base + 4 <= A.wstart) {
#pragma unroll
      for (int q = 0; q < 4; ++q) step(z[q], false);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (base + q >= n && base + q < A.n_end) step(z[q], base + q + 1 > A.wstart);
    }
    n = base + 4;
  }
  if (A.err && !(isfinite(x) && isfinite(v))) atomicOr(A.err, kErrNonFinite);
  A.x_out[j] = x;
  A.v_out[j] = v;
  if (A.vsum_out) A.vsum_out[j] = vs;
}

// Threads per block for n paths: the SMs' shares of the paths rounded up to
// whole warps, in as few blocks per SM as hold them (the busiest SM has at most
// 32 paths per block more than its share: 65536 paths in blocks of 256 left
// some SMs with two blocks and some with one).
int jj64_block(int64_t n, int sms) {
  const int64_t share = (n + sms - 1) / sms;
  const int64_t per_sm = (share + 511) / 512;
  const int64_t block = ((share + per_sm - 1) / per_sm + 31) / 32 * 32;
  return (int)std::min<int64_t>(512, std::max<int64_t>(32, block));
}

}  // namespace
}  // namespace sde

extern "C" sde_status sde_josephson_run_fp64(const sde_jj_point *point, int32_t steps_per_period,
                                             int64_t n_paths, int64_t total_steps, uint64_t seed,
                                             uint32_t point_index, int64_t n_begin, int64_t n_end,
                                             const double *x_in_dev, const double *v_in_dev,
                                             const double *vsum_in_dev, double *x_out_dev,
                                             double *v_out_dev, double *vsum_out_dev, uint32_t *err_dev,
                                             void *stream) {
  using namespace sde;
  SDE_CHECK_ARG(point != nullptr, "point is NULL");
  SDE_CHECK_ARG(n_paths >= 0 && n_paths < (1ll << 31), "n_paths must be in [0, 2^31)");
  SDE_CHECK_ARG(steps_per_period >= 1 && steps_per_period <= 4096, "steps_per_period must be in [1, 4096]");
  SDE_CHECK_ARG(total_steps >= 0 && total_steps <= (1ll << 33), "total_steps out of range");
  SDE_CHECK_ARG(n_begin >= 0 && n_end >= n_begin && n_end <= (1ll << 33), "need 0 <= n_begin <= n_end");
  SDE_CHECK_ARG(isfinite(point->gamma) && isfinite(point->a) && isfinite(point->omega) && isfinite(point->f) &&
                    isfinite(point->D),
                "point parameters must be finite");
  SDE_CHECK_ARG(point->omega > 0.0 && point->gamma > 0.0 && point->D >= 0.0,
                "need omega > 0, gamma > 0, D >= 0");
  if (n_paths == 0) return SDE_OK;
  SDE_CHECK_ARG(x_in_dev && v_in_dev && x_out_dev && v_out_dev, "x/v buffers must be non-NULL");
  JJ64Args a{};
  a.gamma = point->gamma;
  a.a = point->a;
  a.f = point->f;
  a.dt = 2.0 * 3.14159265358979323846 / (point->omega * (double)steps_per_period);
  a.h = 0.5 * a.dt;
  a.s = sqrt(2.0 * point->gamma * point->D * a.dt);
  a.P = steps_per_period;
  a.point = point_index;
  a.n_paths = n_paths;
  a.n_begin = n_begin;
  a.n_end = n_end < total_steps ? n_end : total_steps;  // a point stops at its S
  if (a.n_end < a.n_begin) a.n_end = a.n_begin;
  a.wstart = total_steps - total_steps / 2;
  a.x_in = x_in_dev;
  a.v_in = v_in_dev;
  a.vsum_in = vsum_in_dev;
  a.x_out = x_out_dev;
  a.v_out = v_out_dev;
  a.vsum_out = vsum_out_dev;
  a.err = err_dev;
  a.keys = philox_round_keys(seed);
  int dev = 0, sms = 0;
  SDE_CUDA_TRY(cudaGetDevice(&dev));
  SDE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int block = jj64_block(n_paths, sms);
  const size_t smem = sizeof(double) * (size_t)steps_per_period;
  const unsigned grid = (unsigned)((n_paths + block - 1) / block);
  jj64_kernel<<<grid, block, smem, (cudaStream_t)stream>>>(a);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}
