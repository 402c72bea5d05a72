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
// arguments allow (ranges known, no special cases) without losing accuracy to the
// library's: 11 for a force, 18 for a Gaussian, 9 for the rest of a step, 49 per
// step against 86 with the library's cospi, log, sqrt and sincospi; the drive
// term and the tables are put into shared memory once per block, integers become
// doubles through their bit patterns, comparisons are made on high words.
// Blocks are sized so that every SM holds the same number of paths.  65536 paths,
// 400 steps: 4.96 -> 2.54 ms (1.03e10 path-steps/s).
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "fp64_math.cuh"
#include "philox.cuh"

namespace sde {
namespace {

// Threads of a block at least: a warp alone would take longer over the tables than
// over a few steps.
constexpr int kMinThreads64 = 128;

struct JJ64Args {
  double gamma, a, f;
  double dt, h, s;  // dt, dt / 2, sqrt(2 gamma D dt)
  double inv4P;     // 1 / (4 P)
  int32_t P;
  uint32_t point;   // noise counter word c2
  int32_t block_paths;  // paths per block, one per thread; the other threads help with the tables
  int64_t n_paths;
  int64_t n_begin, n_end;
  int64_t wstart;   // the window holds state indices (wstart, S]
  const double *x_in, *v_in, *vsum_in;
  double *x_out, *v_out, *vsum_out;
  uint32_t *err;
  PhiloxKeys keys;
};

// Tables, each value as a sum hi + lo: hi rounded to a multiple of 2^-43 (2^-52
// for the angles), lo the rest.  Formed by the compiler in integers, as
// multiples of 2^-96 and 2^-62, so they are the same wherever it runs.
constexpr int kLogTable = 128;   // leading 7 bits of a mantissa
constexpr int kAngleTable = 64;  // sixty-fourths of a turn
struct Tables64 {
  double inv[kLogTable];        // c_i ~ 1 / (1 + (i + 1/2) / 128), at most 14 bits; c_0 = 1, c_127 = 1/2
  double2 two_log[kLogTable];   // 2 ln c_i
  double2 exponent[26];         // -2 (e - 24) ln 2 (the last is padding)
  double2 cs[kAngleTable], sn[kAngleTable];
};

// c_i in units of 2^-13.
constexpr int log_scale(int i) {
  return i == 0 ? 8192 : (i == kLogTable - 1 ? 4096 : (8192 * 512 + 257 + 2 * i) / (2 * (257 + 2 * i)));
}

struct HiLo {
  double hi, lo;
};

// 2 ln(k / 8192), k <= 8192: -4 atanh(y), y = (8192 - k) / (8192 + k) <= 1/3, by its series.
constexpr HiLo two_log_of(int k) {
  const unsigned __int128 num = 8192 - k, den = 8192 + k;
  unsigned __int128 term = (num << 98) / den, sum = 0;  // 4 y^(2 q + 1) 2^96
  for (int q = 0; term != 0; ++q) {
    sum += term / (2 * q + 1);
    term = (term * num / den) * num / den;
  }
  const long long hi = (long long)((sum + ((unsigned __int128)1 << 52)) >> 53);
  const long long lo = (long long)((__int128)sum - ((__int128)hi << 53));
  return {-(double)hi / (double)(1ll << 43), -(double)lo / (double)(1ll << 48) / (double)(1ll << 48)};
}

// cos(2 pi i / 64) 2^62, i in [0, 16], by half angles: cos^2(x / 2) = (1 + cos x) / 2.
constexpr long long cos64_of(int i) {
  if (i == 0) return 1ll << 62;
  if (i == 16) return 0;
  const long long c = 2 * i <= 16 ? cos64_of(2 * i) : -cos64_of(32 - 2 * i);
  const unsigned __int128 sq = (unsigned __int128)((unsigned long long)((1ll << 62) + c)) << 61;
  unsigned long long r = 0;
  for (int bit = 62; bit >= 0; --bit) {
    const unsigned long long t = r | (1ull << bit);
    if ((unsigned __int128)t * t <= sq) r = t;
  }
  return (long long)r;
}

constexpr HiLo split62(long long v) {
  const long long hi = (v + 512) >> 10;
  return {(double)hi / (double)(1ll << 52), (double)(v - hi * 1024) / (double)(1ll << 62)};
}

struct TableData {
  double inv[kLogTable], log_hi[kLogTable], log_lo[kLogTable];
  double cos_hi[kAngleTable / 4 + 1], cos_lo[kAngleTable / 4 + 1];  // a quarter turn
};

constexpr TableData make_tables() {
  TableData t{};
  for (int i = 0; i < kLogTable; ++i) {
    t.inv[i] = log_scale(i) / 8192.0;
    const HiLo v = two_log_of(log_scale(i));
    t.log_hi[i] = v.hi;
    t.log_lo[i] = v.lo;
  }
  for (int i = 0; i <= kAngleTable / 4; ++i) {
    const HiLo v = split62(cos64_of(i));
    t.cos_hi[i] = v.hi;
    t.cos_lo[i] = v.lo;
  }
  return t;
}

__device__ constexpr TableData kTables = make_tables();

// cos(2 pi i / 64) of a whole turn from the quarter.
__device__ __forceinline__ double2 cos_entry(int i) {
  const int h = i & 31, q = h <= 16 ? h : 32 - h;
  const bool neg = (h > 16) != ((i & 32) != 0);
  const double hi = kTables.cos_hi[q], lo = kTables.cos_lo[q];
  return neg ? make_double2(-hi, -lo) : make_double2(hi, lo);
}

__device__ __forceinline__ void fill_tables64(Tables64 &t) {
  for (int i = threadIdx.x; i < kLogTable; i += blockDim.x) {
    t.inv[i] = kTables.inv[i];
    t.two_log[i] = make_double2(kTables.log_hi[i], kTables.log_lo[i]);
  }
  // from -2 ln(1/2) = -two_log[127]; 24 times a multiple of 2^-43 below 2 is exact
  for (int i = threadIdx.x; i < 25; i += blockDim.x)
    t.exponent[i] = make_double2((i - 24) * kTables.log_hi[kLogTable - 1], (i - 24) * kTables.log_lo[kLogTable - 1]);
  for (int i = threadIdx.x; i < kAngleTable; i += blockDim.x) {
    t.cs[i] = cos_entry(i);
    t.sn[i] = cos_entry((i + 48) & (kAngleTable - 1));
  }
}

// -2 ln(m 2^-24) for m in [1, 2^24].  m = 2^e f, f in [1, 2); with c_i from the
// leading bits of f, z = f c_i - 1 is exact and in (-0.004, 1/128], and
// -2 ln u = -2 (e - 24) ln 2 + 2 ln c_i - 2 z + z^2 r(z), r of degree 5
// (interpolation at the Chebyshev nodes of the interval, within 1e-20).  The
// first three terms are multiples of 2^-43 (z of 2^-36) and their sum is exact;
// the rest is small, so the result is rounded once: within 0.54 ulp over all m
// (0.52 for a correctly rounded logarithm doubled; 25 without the low parts).
// c_0 = 1 and c_127 = 1/2 make the table terms cancel for u near 1; u = 1 gives 0.
__device__ __forceinline__ double minus2_log24(uint32_t m, const Tables64 &t) {
  const uint32_t bits = __float_as_uint((float)m);  // exact: 24 bits
  const uint32_t mant = bits & 0x7FFFFFu;
  const int e = (int)(bits >> 23) - 127, i = (int)(mant >> 16);
  const double f = __hiloint2double((int)(0x3FF00000u | (mant >> 3)), (int)(mant << 29));
  const double z = fma(f, t.inv[i], -1.0);
  const double2 te = t.exponent[e], tl = t.two_log[i];
  double r = -0.2828473837233479;
  r = fma(r, z, 0.3333355763843714);
  r = fma(r, z, -0.4000000966277093);
  r = fma(r, z, 0.5000000000732646);
  r = fma(r, z, -0.6666666666658018);
  r = fma(r, z, 0.9999999999999994);
  return fma(-2.0, z, te.x + tl.x) + fma(z * z, r, te.y + tl.y);
}

// Box-Muller in FP64 from the same 24-bit uniforms as the FP32 path.  The
// angle 2 pi (j + 1) 2^-24 is the nearest sixty-fourth of a turn plus b, |b| <=
// pi / 64: sin b and cos b from short polynomials (interpolation at the
// Chebyshev nodes, within 3e-17), combined with the table by angle addition,
// the largest term last: sine and cosine within 8.3e-17.
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
  const double2 C = t.cs[q & (kAngleTable - 1)], S = t.sn[q & (kAngleTable - 1)];
  z0 = rho * (C.x + fma(C.x, cm1, fma(-S.x, sb, C.y)));
  z1 = rho * (S.x + fma(S.x, cm1, fma(C.x, sb, S.y)));
}

// A - 2 pi cos(2 pi x).  With d = |x - rint(x)|, the cosine is an even polynomial
// of d (d < 1/8) or of 1/2 - d (d >= 3/8, with the other sign), or an odd one of
// 1/4 - d; each of these differences is exact.  Coefficients: least squares over
// [0, 1/8] of the function less its leading FP64 constant.  Without A within
// 9.6e-16 (RMS 2.8e-16; 2 pi times a correctly rounded cosine 1.04e-15, 3.2e-16).
// The selections between the polynomials cost no FP64 issue.
__device__ __forceinline__ double jj_force64(double x, double A) {
  const double d = fabs(x - rint(x));
  const int hi = __double2hiint(d);  // compared as an integer: 1/8 and 3/8 have no low bits
  const bool far = hi >= 0x3FD80000, odd = hi >= 0x3FC00000 && !far;
  const double t = (odd ? 0.25 : (far ? 0.5 : 0.0)) - d;
  const double s = t * t;
  double p = odd ? -23.72575465200541 : -49.07454462882556;
  p = fma(p, s, odd ? 94.8355962158329 : 166.02855703122987);
  p = fma(p, s, odd ? -264.2624799289404 : -378.52811281837717);
  p = fma(p, s, odd ? 481.95713035499193 : 536.9410175504025);
  p = fma(p, s, odd ? -512.7409032378275 : -408.02624637851824);
  p = fma(p, s, odd ? 259.75757609066903 : 124.02510672119752);
  p = fma(p, s, odd ? -39.47841760435743 : -6.283185307179586);
  return fma(odd ? t : (far ? -1.0 : 1.0), p, A);
}

__global__ void __launch_bounds__(512) jj64_kernel(const JJ64Args A) {
  extern __shared__ double drive_s[];  // [P]: a cos(2 pi k / P) + f
  __shared__ Tables64 tab;
  for (int k = threadIdx.x; k < A.P; k += blockDim.x)
    drive_s[k] = fma(A.a, cos_ratio64(k, A.P, A.inv4P), A.f);
  fill_tables64(tab);
  __syncthreads();
  const int64_t j = (int64_t)blockIdx.x * A.block_paths + threadIdx.x;
  if ((int)threadIdx.x >= A.block_paths || j >= A.n_paths) return;
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

// Paths per block for n paths: the SMs' shares of the paths rounded up to
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
  a.block_paths = jj64_block(n_paths, sms);
  a.inv4P = 1.0 / (4.0 * (double)steps_per_period);
  const size_t smem = sizeof(double) * (size_t)steps_per_period;
  const unsigned grid = (unsigned)((n_paths + a.block_paths - 1) / a.block_paths);
  jj64_kernel<<<grid, std::max(a.block_paths, kMinThreads64), smem, (cudaStream_t)stream>>>(a);
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}
