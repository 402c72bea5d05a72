// kuramoto.cu -- SRK2 integration of the noisy Kuramoto model (Eq. 2,
// gamma = 1) on the GPU, in three forms of the coupling sum:
//
//  * mean field (Eq. 3): sum_j sin(x_j - x_i) = cos x_i S - sin x_i C with
//    S = sum_j sin x_j, C = sum_j cos x_j.  One CTA owns one replica for the
//    whole run: its phases stay in registers, S and C come from a block
//    reduction per stage (two per step), r(t) = sqrt(S^2 + C^2) / N is read
//    off the first-stage sums.  No grid-wide synchronisation.
//  * mean field over the whole grid (Eq. 3 for replicas too large for a CTA
//    or a cluster, such as the 2^24 oscillators of Fig. 4): two launches
//    per step, each reducing its partial sums of sin/cos through the last
//    block to finish (fixed-order FP64 sum of the per-block partials, no
//    waiting between blocks).
//  * pairwise (Alg. 3 / Fig. 3): the direct all-pairs sum, tiles of source
//    sines and cosines staged in shared memory; one launch per SRK2 stage with
//    the sub-step fused into the epilogue (Sec. 4.2 splits it into UpdateRHS and
//    AdvanceSystem; higher order by interleaving stages), or, for small
//    populations, all steps in one launch with a replica per cluster.
//  * general K_ij: the sum as a GEMM against [sin x | cos x] (see
//    kuramoto_general.cu).
//
// Phases are kept as 32-bit fixed-point turns (2^32 units per 2 pi): the
// wrap modulo 2 pi is exact integer overflow and the resolution (1.5e-9
// rad) does not depend on the phase, in the spirit of keeping time modulo
// the period (Sec. 5).  Drift increments are computed in FP32 and rounded to
// the fixed-point grid once per stage (the predictor phase too), and sin/cos
// of a phase come from its fixed-point value directly (turns.cuh).
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include <cooperative_groups.h>

#include "kuramoto.h"
#include "kuramoto_internal.h"
#include "philox.cuh"
#include "turns.cuh"

namespace sde {

namespace {

__device__ __forceinline__ float2 warp_sum2(float a, float b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  return make_float2(a, b);
}

// Sum of (a, b) over the block; every thread receives the totals.  `red`
// alternates between two slots so one barrier per reduction suffices.
__device__ __forceinline__ float2 block_sum2(float a, float b, float2 *red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2 v = warp_sum2(a, b);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  const int nw = blockDim.x >> 5;
  v = lane < nw ? red[lane] : make_float2(0.0f, 0.0f);
  return warp_sum2(v.x, v.y);
}

// Partial sums of sin and cos in fixed point, units of 2^-17 (the replica
// forms that keep a replica in one CTA or cluster, n_osc <= 8192): integer
// sums are exact and associative, so the totals are the same however the
// oscillators are split over threads, warps and CTAs, and a warp adds 32
// values in one redux instruction.  |sum| <= 8192 x 2^17 = 2^30.  The
// quantisation (<= 2^-18 per value) moves S and C by ~1e-5 at N = 4096,
// which reaches a phase only through K dt / (2 pi N).
constexpr float kQuant = 131072.0f;
constexpr float kInvQuant = 1.0f / 131072.0f;

// round(v 2^17) to the nearest integer (ties to even) for |v| <= 1, on the FMA
// pipe: v 2^17 + 1.5 2^23 lies in [2^23, 2^24), where the FP32 spacing is 1,
// so the one rounding of the FMA is the rounding to an integer, read off the
// mantissa bits.  The same integer as __float2int_rn(v * 2^17), without the
// conversion unit.
__device__ __forceinline__ int quant(float v) {
  return __float_as_int(fmaf(v, kQuant, 12582912.0f)) - 0x4B400000;
}

__device__ __forceinline__ int2 warp_qsum(int a, int b) {
  return make_int2(__reduce_add_sync(0xffffffffu, a), __reduce_add_sync(0xffffffffu, b));
}

__device__ __forceinline__ float2 unquant(int2 v) { return make_float2((float)v.x * kInvQuant, (float)v.y * kInvQuant); }

// Block total of the fixed-point pair; every thread receives it.  `red`
// alternates between two slots so one barrier per reduction suffices.
__device__ __forceinline__ float2 block_qsum(int a, int b, int2 *red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int2 v = warp_qsum(a, b);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  const int nw = blockDim.x >> 5;
  v = lane < nw ? red[lane] : make_int2(0, 0);
  return unquant(warp_qsum(v.x, v.y));
}

// Blocks of up to 1024 threads hold 1-2 oscillators per thread; larger
// per-thread counts run in blocks of at most 512 threads (128 registers).
template <int OPT, bool FULL>
__global__ void __launch_bounds__(OPT <= 2 ? 1024 : 512, 1) kur_meanfield_kernel(const KurArgs A) {
  __shared__ int2 red[2][32];
  const int rep = blockIdx.x;
  const int64_t N = A.N;
  const int64_t base = (int64_t)rep * N;
  const PhiloxKeys &key = A.keys;
  uint32_t th[OPT];
  float wdt[OPT];
  bool valid[OPT];
#pragma unroll
  for (int k = 0; k < OPT; ++k) {
    const int64_t i = threadIdx.x + (int64_t)k * blockDim.x;
    valid[k] = i < N;
    th[k] = valid[k] ? A.theta_in[base + i] : 0u;
    wdt[k] = valid[k] ? A.omega[base + i] * A.wscale : 0.0f;
  }
  int slot = 0;
  int64_t sample_ctr = 0;  // (n - n_begin) mod M
  int64_t sample_idx = 0;
  const float invN = 1.0f / (float)N;
  for (int64_t n = A.n_begin; n < A.n_end;) {
    const int64_t g = n >> 2;
    float z[OPT][4];
    uint32_t oid[OPT];
#pragma unroll
    for (int k = 0; k < OPT; ++k) oid[k] = threadIdx.x + k * blockDim.x;
    gauss4_n<OPT>((uint32_t)g, oid, (uint32_t)rep, kTagKuramoto, key, z);
    const int s0 = (int)(n & 3);
    const int64_t rem = A.n_end - (g << 2);
    const int s1 = rem < 4 ? (int)rem : 4;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (s < s0 || s >= s1) continue;
      float sn[OPT], cs[OPT];
      int S = 0, C = 0;
      sincos_turns_n<OPT>(th, sn, cs);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        if (!FULL && !valid[k]) sn[k] = cs[k] = 0.0f;
        S += quant(sn[k]);
        C += quant(cs[k]);
      }
      float2 sc = block_qsum(S, C, red[slot]);
      slot ^= 1;
      if (A.M > 0 && sample_ctr == 0) {
        if (threadIdx.x == 0 && A.r_out) {
          const double Sd = sc.x, Cd = sc.y;
          A.r_out[sample_idx * A.R + rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
        }
        ++sample_idx;
      }
      if (A.M > 0 && ++sample_ctr == A.M) sample_ctr = 0;
      float g1[OPT], sn2[OPT], cs2[OPT];
      int S2 = 0, C2 = 0;
      uint32_t tp[OPT];
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        g1[k] = cs[k] * sc.x - sn[k] * sc.y;
        const float d1 = fmaf(A.sc, z[k][s], fmaf(A.kc, g1[k], wdt[k]));
        tp[k] = th[k] + (uint32_t)__float2int_rn(d1 * 4294967296.0f);
      }
      sincos_turns_n<OPT>(tp, sn2, cs2);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        if (!FULL && !valid[k]) sn2[k] = cs2[k] = 0.0f;
        S2 += quant(sn2[k]);
        C2 += quant(cs2[k]);
      }
      sc = block_qsum(S2, C2, red[slot]);
      slot ^= 1;
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        const float g2 = cs2[k] * sc.x - sn2[k] * sc.y;
        const float d = fmaf(A.sc, z[k][s], fmaf(A.kh, g1[k] + g2, wdt[k]));
        th[k] += (uint32_t)__float2int_rn(d * 4294967296.0f);
      }
    }
    n = (g + 1) << 2;
  }
  // Final sample at n_end.
  if (A.M > 0) {
    int S = 0, C = 0;
#pragma unroll
    for (int k = 0; k < OPT; ++k) {
      float sn, cs;
      sincos_turns(th[k], sn, cs);
      if (valid[k]) {
        S += quant(sn);
        C += quant(cs);
      }
    }
    const float2 sc = block_qsum(S, C, red[slot]);
    if (threadIdx.x == 0 && A.r_out) {
      const double Sd = sc.x, Cd = sc.y;
      A.r_out[sample_idx * A.R + rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
    }
  }
  (void)invN;
#pragma unroll
  for (int k = 0; k < OPT; ++k) {
    const int64_t i = threadIdx.x + (int64_t)k * blockDim.x;
    if (valid[k]) A.theta_out[base + i] = th[k];
  }
}

// Mean field with one replica spread over a thread-block cluster of CS CTAs
// (CS from the launch): each CTA holds N / CS oscillators in registers.  Per
// stage every warp reduces its (S, C) with shuffles and stores the pair into
// its slot of every CTA of the cluster (distributed shared memory); one
// cluster barrier later each warp of each CTA sums the CS x warps slots in
// the same fixed order, so all CTAs of a replica use identical sums.  Slots
// are double-buffered across stages, so one barrier per stage suffices.
template <int OPT, bool FULL>
__global__ void __launch_bounds__(512, 1) kur_meanfield_cluster_kernel(const KurArgs A) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ int2 slots[2][32];  // [buffer][cluster rank * warps + warp]
  const int cs = (int)cluster.num_blocks();
  const int crank = (int)cluster.block_rank();
  const int nwarps = blockDim.x >> 5;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nslots = cs * nwarps;  // <= 32, checked by the host
  const int rep = blockIdx.x / cs;
  const int64_t N = A.N;
  const int64_t chunk = (N + cs - 1) / cs;
  const int64_t i0 = (int64_t)crank * chunk;
  const int64_t base = (int64_t)rep * N;
  const PhiloxKeys &key = A.keys;
  uint32_t th[OPT];
  float wdt[OPT];
  bool valid[OPT];
  uint32_t oid[OPT];
#pragma unroll
  for (int k = 0; k < OPT; ++k) {
    const int64_t li = threadIdx.x + (int64_t)k * blockDim.x;
    const int64_t i = i0 + li;
    valid[k] = li < chunk && i < N;
    oid[k] = (uint32_t)i;
    th[k] = valid[k] ? A.theta_in[base + i] : 0u;
    wdt[k] = valid[k] ? A.omega[base + i] * A.wscale : 0.0f;
  }
  cluster.sync();  // every CTA of the cluster runs before the first remote store into it
  int buf = 0;
  int64_t sample_ctr = 0, sample_idx = 0;
  // cluster-wide (S, C)
  auto cluster_sum = [&](int S, int C) -> float2 {
    const int2 part = warp_qsum(S, C);
    if (lane < cs) {
      int2 *dst = cluster.map_shared_rank(&slots[buf][crank * nwarps + warp], lane);
      *dst = part;
    }
    cluster.sync();
    const int2 v = lane < nslots ? slots[buf][lane] : make_int2(0, 0);
    buf ^= 1;
    return unquant(warp_qsum(v.x, v.y));
  };
  for (int64_t n = A.n_begin; n < A.n_end;) {
    const int64_t g = n >> 2;
    float z[OPT][4];
    gauss4_n<OPT>((uint32_t)g, oid, (uint32_t)rep, kTagKuramoto, key, z);
    const int s0 = (int)(n & 3);
    const int64_t rem = A.n_end - (g << 2);
    const int s1 = rem < 4 ? (int)rem : 4;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (s < s0 || s >= s1) continue;
      float sn[OPT], cs_[OPT];
      int S = 0, C = 0;
      sincos_turns_n<OPT>(th, sn, cs_);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        if (!FULL && !valid[k]) sn[k] = cs_[k] = 0.0f;
        S += quant(sn[k]);
        C += quant(cs_[k]);
      }
      float2 sc = cluster_sum(S, C);
      if (A.M > 0 && sample_ctr == 0) {
        if (threadIdx.x == 0 && crank == 0 && A.r_out) {
          const double Sd = sc.x, Cd = sc.y;
          A.r_out[sample_idx * A.R + rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
        }
        ++sample_idx;
      }
      if (A.M > 0 && ++sample_ctr == A.M) sample_ctr = 0;
      float g1[OPT], sn2[OPT], cs2[OPT];
      int S2 = 0, C2 = 0;
      uint32_t tp[OPT];
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        g1[k] = cs_[k] * sc.x - sn[k] * sc.y;
        const float d1 = fmaf(A.sc, z[k][s], fmaf(A.kc, g1[k], wdt[k]));
        tp[k] = th[k] + (uint32_t)__float2int_rn(d1 * 4294967296.0f);
      }
      sincos_turns_n<OPT>(tp, sn2, cs2);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        if (!FULL && !valid[k]) sn2[k] = cs2[k] = 0.0f;
        S2 += quant(sn2[k]);
        C2 += quant(cs2[k]);
      }
      sc = cluster_sum(S2, C2);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        const float g2 = cs2[k] * sc.x - sn2[k] * sc.y;
        const float d = fmaf(A.sc, z[k][s], fmaf(A.kh, g1[k] + g2, wdt[k]));
        th[k] += (uint32_t)__float2int_rn(d * 4294967296.0f);
      }
    }
    n = (g + 1) << 2;
  }
  if (A.M > 0) {
    int S = 0, C = 0;
#pragma unroll
    for (int k = 0; k < OPT; ++k) {
      float sn, c;
      sincos_turns(th[k], sn, c);
      if (valid[k]) {
        S += quant(sn);
        C += quant(c);
      }
    }
    const float2 sc = cluster_sum(S, C);
    if (threadIdx.x == 0 && crank == 0 && A.r_out) {
      const double Sd = sc.x, Cd = sc.y;
      A.r_out[sample_idx * A.R + rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
    }
  }
#pragma unroll
  for (int k = 0; k < OPT; ++k)
    if (valid[k]) A.theta_out[base + oid[k]] = th[k];
  cluster.sync();  // no CTA leaves while others may still read its exchange slots
}

// ---- cluster exchange by asynchronous remote stores ----------------------

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait (at most limit_ns) for the phase `parity` of an mbarrier; false on
// expiry.  try_wait may suspend the thread for a while before it answers
// (longer than a short limit: the hardware takes the suspend-time hint as a
// hint only), so limits under a millisecond poll with the non-blocking
// test_wait instead.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  const uint64_t t0 = now_ns();
  const bool poll = limit_ns < 1000000ull;
  for (;;) {
    uint32_t done;
    if (poll)
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(done)
          : "r"(bar), "r"(parity)
          : "memory");
    else
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(done)
          : "r"(bar), "r"(parity)
          : "memory");
    if (done) return true;
    if (now_ns() - t0 > limit_ns) return false;
  }
}

// The end of a cluster kernel whose CTAs send one another a stage's data
// asynchronously, counted by two alternating mbarriers of the receiver (bar0
// and the next; stage s on barrier s & 1), when a wait may have expired.  A CTA
// barrier of the cluster orders threads, not the copies they issued, and a CTA
// that ends while a copy still reads or writes its shared memory is a fault;
// so if any CTA of the cluster gave up, every CTA stays until all that was sent
// to it has arrived.  Both open phases of its barriers (stages got and got + 1:
// nobody sends a later one before this CTA has sent stage got + 1) are credited
// with what was never sent, `missing(stage)` bytes, so they complete when the
// last copy in flight lands; the wait for that is bounded by a second whatever
// the context's limit.  Nothing is waited for when no wait expired: then every
// stage was received by everyone before this.
//
// late: this thread's wait expired (any thread of the CTA may say so); got:
// stages that thread 0 received; flag: a word of shared memory, zero since
// before the kernel's first cluster barrier.  All threads of the cluster call it.
template <typename Missing>
__device__ __forceinline__ void cluster_drain(bool late, uint32_t got, uint32_t bar0, int *flag, int cs,
                                              Missing missing) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  late = __syncthreads_or(late);
  if (late && (int)threadIdx.x < cs)  // their CTAs are still there: they have not passed the barrier below
    *(volatile int *)cluster.map_shared_rank(flag, threadIdx.x) = 1;
  cluster.sync();  // every copy that ever will be is issued, every count of them written
  if (*(volatile int *)flag == 0) return;
  if (threadIdx.x == 0) {
#pragma unroll
    for (uint32_t s = got; s < got + 2u; ++s) {
      const uint32_t bytes = missing(s);
      if (bytes > 0)
        asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar0 + 8u * (s & 1u)), "r"(bytes)
                     : "memory");
    }
    for (uint32_t s = got; s < got + 2u; ++s) mbar_wait_bounded(bar0 + 8u * (s & 1u), (s >> 1) & 1u, 1000000000ull);
  }
  cluster.sync();  // everything sent has arrived everywhere: no CTA's memory is in use any more
}

// The cluster mean field with the exchange done by st.async: every warp
// sends its (S, C) pair into its slot of every CTA of the cluster with an
// asynchronous remote store that completes on the receiving CTA's mbarrier
// (transaction bytes), and each CTA waits on its own mbarrier for the
// cs x warps pairs of the stage instead of a cluster-wide barrier (whose
// release/acquire fence is what the plain cluster kernel waits on).  Two
// slot buffers and two mbarriers alternate by stage: a CTA can only send
// stage s + 2 after receiving everyone's stage s + 1 pairs, each sent after
// its sender had read the stage s slots, so a buffer is never overwritten
// while it is read, and the receiver has re-armed the buffer's mbarrier
// (after its own stage s wait, before its stage s + 1 sends) before any
// stage s + 2 store can arrive.  Waits are bounded (A.wait_ns, one second by
// default): on expiry the kernel records kErrTimeout, leaves the step loop
// (warp-uniformly) and meets the others in cluster_drain.
template <int OPT, bool FULL>
__global__ void __launch_bounds__(512, 1) kur_meanfield_async_kernel(const KurArgs A) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ int2 slots[2][32];
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ int gave_up;           // some CTA of the cluster did
  __shared__ uint32_t sent_s[16];   // stages each warp sent
  const int cs = (int)cluster.num_blocks();
  const int crank = (int)cluster.block_rank();
  const int nwarps = blockDim.x >> 5;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nslots = cs * nwarps;  // <= 32, checked by the host
  const uint32_t bytes = (uint32_t)nslots * 8u;
  if (threadIdx.x == 0) {
    gave_up = 0;
    // each phase is armed (arrival + expected bytes) before any store of it can
    // arrive: stages 0 and 1 here, stage s + 2 right after stage s completes
    // (no sender reaches stage s + 2 before this CTA has sent stage s + 1)
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[0])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[1])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&mbar[0])), "r"(bytes)
                 : "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&mbar[1])), "r"(bytes)
                 : "memory");
  }
  cluster.sync();  // every CTA's barriers exist and are armed before the first remote store
  const int rep = blockIdx.x / cs;
  const int64_t N = A.N;
  const int64_t chunk = (N + cs - 1) / cs;
  const int64_t i0 = (int64_t)crank * chunk;
  const int64_t base = (int64_t)rep * N;
  const PhiloxKeys &key = A.keys;
  uint32_t th[OPT];
  float wdt[OPT];
  bool valid[OPT];
  uint32_t oid[OPT];
#pragma unroll
  for (int k = 0; k < OPT; ++k) {
    const int64_t li = threadIdx.x + (int64_t)k * blockDim.x;
    const int64_t i = i0 + li;
    valid[k] = li < chunk && i < N;
    oid[k] = (uint32_t)i;
    th[k] = valid[k] ? A.theta_in[base + i] : 0u;
    wdt[k] = valid[k] ? A.omega[base + i] * A.wscale : 0.0f;
  }
  // remote addresses of this warp's slot and of the mbarriers, in CTA `lane`
  const uint32_t my_slot0 = smem_u32(&slots[0][crank * nwarps + warp]);
  const uint32_t my_slot1 = smem_u32(&slots[1][crank * nwarps + warp]);
  const uint32_t rslot0 = lane < cs ? cluster_map(my_slot0, (uint32_t)lane) : 0u;
  const uint32_t rslot1 = lane < cs ? cluster_map(my_slot1, (uint32_t)lane) : 0u;
  const uint32_t rbar0 = lane < cs ? cluster_map(smem_u32(&mbar[0]), (uint32_t)lane) : 0u;
  const uint32_t rbar1 = lane < cs ? cluster_map(smem_u32(&mbar[1]), (uint32_t)lane) : 0u;
  uint32_t stage = 0;    // stages sent by this warp
  bool failed = false;   // a wait of the last of them expired (warp-uniform)
  bool mine_ok = true;   // not this thread's
  auto cluster_sum = [&](int S, int C) -> float2 {
    const int2 part = warp_qsum(S, C);
    const int b = (int)(stage & 1u);
    const uint32_t parity = (stage >> 1) & 1u;
    const uint32_t bar = smem_u32(&mbar[b]);
    if (lane < cs)
      asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.s32 [%0], {%1, %2}, [%3];" ::"r"(
                       b ? rslot1 : rslot0),
                   "r"(part.x), "r"(part.y), "r"(b ? rbar1 : rbar0)
                   : "memory");
    const bool ok = mbar_wait_bounded(bar, parity, A.wait_ns);
    if (__any_sync(0xffffffffu, !ok)) {
      failed = true;
      mine_ok = ok;
      if (lane == 0) atomicOr(A.err, kErrTimeout);
    }
    if (threadIdx.x == 0 && ok)  // arm this buffer's next phase (stage + 2)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    const int2 v = lane < nslots ? slots[b][lane] : make_int2(0, 0);
    ++stage;
    return unquant(warp_qsum(v.x, v.y));
  };
  int64_t sample_ctr = 0, sample_idx = 0;
  for (int64_t n = A.n_begin; n < A.n_end && !failed;) {
    const int64_t g = n >> 2;
    float z[OPT][4];
    gauss4_n<OPT>((uint32_t)g, oid, (uint32_t)rep, kTagKuramoto, key, z);
    const int s0 = (int)(n & 3);
    const int64_t rem = A.n_end - (g << 2);
    const int s1 = rem < 4 ? (int)rem : 4;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (s < s0 || s >= s1 || failed) continue;
      float sn[OPT], cs_[OPT];
      int S = 0, C = 0;
      sincos_turns_n<OPT>(th, sn, cs_);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        if (!FULL && !valid[k]) sn[k] = cs_[k] = 0.0f;
        S += quant(sn[k]);
        C += quant(cs_[k]);
      }
      float2 sc = cluster_sum(S, C);
      if (failed) continue;  // a stage is sent only after the one before it was received
      if (A.M > 0 && sample_ctr == 0) {
        if (threadIdx.x == 0 && crank == 0 && A.r_out) {
          const double Sd = sc.x, Cd = sc.y;
          A.r_out[sample_idx * A.R + rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
        }
        ++sample_idx;
      }
      if (A.M > 0 && ++sample_ctr == A.M) sample_ctr = 0;
      float g1[OPT], sn2[OPT], cs2[OPT];
      int S2 = 0, C2 = 0;
      uint32_t tp[OPT];
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        g1[k] = cs_[k] * sc.x - sn[k] * sc.y;
        const float d1 = fmaf(A.sc, z[k][s], fmaf(A.kc, g1[k], wdt[k]));
        tp[k] = th[k] + (uint32_t)__float2int_rn(d1 * 4294967296.0f);
      }
      sincos_turns_n<OPT>(tp, sn2, cs2);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        if (!FULL && !valid[k]) sn2[k] = cs2[k] = 0.0f;
        S2 += quant(sn2[k]);
        C2 += quant(cs2[k]);
      }
      sc = cluster_sum(S2, C2);
#pragma unroll
      for (int k = 0; k < OPT; ++k) {
        const float g2 = cs2[k] * sc.x - sn2[k] * sc.y;
        const float d = fmaf(A.sc, z[k][s], fmaf(A.kh, g1[k] + g2, wdt[k]));
        th[k] += (uint32_t)__float2int_rn(d * 4294967296.0f);
      }
    }
    n = (g + 1) << 2;
  }
  if (A.M > 0 && !failed) {
    int S = 0, C = 0;
#pragma unroll
    for (int k = 0; k < OPT; ++k) {
      float sn, c;
      sincos_turns(th[k], sn, c);
      if (valid[k]) {
        S += quant(sn);
        C += quant(c);
      }
    }
    const float2 sc = cluster_sum(S, C);
    if (threadIdx.x == 0 && crank == 0 && A.r_out) {
      const double Sd = sc.x, Cd = sc.y;
      A.r_out[sample_idx * A.R + rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
    }
  }
#pragma unroll
  for (int k = 0; k < OPT; ++k)
    if (valid[k]) A.theta_out[base + oid[k]] = th[k];
  if (lane == 0) sent_s[warp] = stage;
  const uint32_t got = failed && !mine_ok ? stage - 1 : stage;  // stages thread 0 received
  cluster_drain(failed, got, smem_u32(&mbar[0]), &gave_up, cs, [&](uint32_t s) {
    uint32_t miss = 0;
    for (int q = 0; q < cs; ++q) {
      const volatile uint32_t *sent = cluster.map_shared_rank(sent_s, q);
      for (int w = 0; w < nwarps; ++w) miss += sent[w] <= s ? 8u : 0u;
    }
    return miss;
  });
}

// ---- mean field over the whole grid ------------------------------------

// The launches of a step follow one another closely: each starts while the one
// before it ends (its blocks take the places as they become free) and waits here
// until that one's results are all there.  It lets the next one do the same; a
// grid that waits has started all its blocks, so nothing it needs is kept out.
// Per step, against plain launches: 16.7 -> 13.0 us for 3 replicas of 20,000
// oscillators, 21.1 -> 17.0 for 8 of 91,126, 118.5 -> 115.4 for one of 2^24.  The
// pairwise stages are not launched so: their blocks are few and long, and started
// early they land unevenly on the SMs (6000 x 1: 18 -> 32 us).
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int kMfgThreads = 256;
constexpr int kMfgIlp = 4;  // oscillators per thread per iteration: one 16-byte access per array

// Four consecutive elements from index i0 of a replica's array in one access;
// those outside [0, n) are not touched (zero) where the chunk is not whole.
// STREAM marks what the next launch does not find in L2 anyway as first to be
// evicted.
template <bool STREAM, typename T>
__device__ __forceinline__ void mfg_load4(const T *p, uint32_t i0, uint32_t n, bool vec, T (&v)[4]) {
  if (vec) {
    const uint4 *q = reinterpret_cast<const uint4 *>(p + i0);
    const uint4 u = STREAM ? __ldcs(q) : *q;
    memcpy(v, &u, 16);
  } else {
#pragma unroll
    for (uint32_t e = 0; e < 4; ++e) v[e] = i0 + e < n ? p[i0 + e] : T(0);
  }
}

template <bool STREAM, typename T>
__device__ __forceinline__ void mfg_store4(T *p, uint32_t i0, uint32_t n, bool vec, const T (&v)[4]) {
  if (vec) {
    uint4 u;
    memcpy(&u, v, 16);
    uint4 *q = reinterpret_cast<uint4 *>(p + i0);
    if (STREAM)
      __stcs(q, u);
    else
      *q = u;
  } else {
#pragma unroll
    for (uint32_t e = 0; e < 4; ++e)
      if (i0 + e < n) p[i0 + e] = v[e];
  }
}

int64_t mfg_plane(int64_t NR) { return (NR + 3) & ~3ll; }

struct MfgArgs {
  uint32_t *theta;    // [R][N] theta_n; the corrector overwrites it with theta_{n+1}
  uint32_t *theta_t;  // [R][N] predictor phases theta~_n
  float *y;           // [R][N] first-stage part of the step: wdt + kh g1 + sc psi
  float *psi;         // [3][plane] Gaussians of steps 4g+1..4g+3 of the current Philox block
  int64_t plane;      // R N rounded up to a multiple of 4
  bool omega_vec;     // omega starts on a 16-byte boundary, as the library's arrays do
  bool reverse;       // from the last oscillator to the first
  const float *omega;
  float2 *partials;   // [R][gridDim.x] per-block sums
  double *tot;        // [R][4]: (S, C) of theta_n, then (S, C) of theta~_n
  uint32_t *count;    // [R] blocks finished in this launch (the last one resets it)
  double *r_out;      // [rows][R]
  int64_t N, R;
  int64_t n;           // step index (noise counter)
  int64_t sample_row;  // r row written from this launch's totals, -1 = none
  float wscale, kc, kh, sc;
  PhiloxKeys keys;
};

// MODE 2: sums of (sin, cos) of theta_n.  MODE 0 and 3 (predictor): g1 from the
// totals of theta_n, theta~ = theta + d1, sums over theta~.  MODE 1
// (corrector): g2 from the totals of theta~, theta_{n+1} = theta + y + kh g2,
// sums over theta_{n+1} (the next step's first-stage sums).  The Gaussian of
// step n is element n mod 4 of the Philox block n / 4 of the oscillator (as
// in the other forms): the predictor draws the block at its first step, or
// at the first step of a run (MODE 3), and keeps the later elements in `psi`
// for the next three steps (MODE 0 reads them).  Each thread
// strides over the replica; the block's FP32 sums go to `partials`, and the
// block that finishes last adds all partials of the replica in block order
// in FP64, so the totals do not depend on which block that is.
//
// What bounds it: HBM (16 B per oscillator for the corrector, 20 for the
// predictor, 28 where it draws), then the noise of the drawing launch.  A thread
// takes four consecutive oscillators in one 16-byte access per array: with four
// 4-byte accesses the launches were bound by issue (153.7 us per step of 2^24
// oscillators, 127.9 with 16-byte ones).  theta is the one array both launches
// of a step use; the others are marked as first to leave L2 (120.2 us), and the
// corrector runs from the last oscillator to the first, so that it starts with
// what the predictor left there (2 us of it).  1,000,003 x 7, no row of which
// but the first starts on a 16-byte boundary: 80.4 -> 66.5 us.
template <int MODE>
__global__ void __launch_bounds__(kMfgThreads, MODE == 3 ? 4 : (MODE == 2 ? 8 : 5)) kur_mfg_kernel(const MfgArgs A) {
  chain_begin();
  constexpr bool kPred = MODE == 0 || MODE == 3;
  constexpr bool kGen = MODE == 3;
  __shared__ float2 red[32];
  __shared__ double2 red64[32];
  __shared__ bool is_last;
  const int rep = A.reverse ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
  const int64_t N = A.N;
  const int64_t base = (int64_t)rep * N;
  double *tot = A.tot + 4 * rep;
  float S = 0.0f, C = 0.0f;
  if (kPred) {
    S = (float)tot[0];
    C = (float)tot[1];
  } else if (MODE == 1) {
    S = (float)tot[2];
    C = (float)tot[3];
  }
  const int j = (int)(A.n & 3);
  float ps = 0.0f, pc = 0.0f;
  // per-replica base pointers, 32-bit oscillator indices: a chunk is four
  // oscillators on a 16-byte boundary of the [R][N] arrays, so its first index
  // is -lead (as an unsigned number) in a replica's first chunk.  N < 2^31: no
  // sum below wraps onto a valid index.
  const uint32_t Nu = (uint32_t)N;
  const uint32_t lead = (uint32_t)(base & 3);
  uint32_t *th_r = A.theta + base;
  uint32_t *tt_r = A.theta_t + base;
  float *y_r = A.y + base;
  const float *om_r = A.omega + base;
  const float *psi_in = (kPred && !kGen && j > 0) ? A.psi + (int64_t)(j - 1) * A.plane + base : nullptr;
  float *psi_out = A.psi + base;  // plane k - 1 at + (k - 1) A.plane
  const uint32_t chunks = (lead + Nu + 3u) >> 2, stride = gridDim.x * (uint32_t)kMfgThreads;
  for (uint32_t q = blockIdx.x * (uint32_t)kMfgThreads + threadIdx.x; q < chunks; q += stride) {
    const uint32_t i0 = 4u * (A.reverse ? chunks - 1u - q : q) - lead;
    const bool full = i0 < Nu && Nu - i0 >= 4u;
    uint32_t t0[4], tt[4];
    float a1[4], a2[4];
    mfg_load4<false>(th_r, i0, Nu, full, t0);
    if (kPred) {
      mfg_load4<true>(om_r, i0, Nu, full && A.omega_vec, a1);
      if (!kGen) mfg_load4<true>(psi_in, i0, Nu, full, a2);
    } else if (MODE == 1) {
      mfg_load4<true>(tt_r, i0, Nu, full, tt);
      mfg_load4<true>(y_r, i0, Nu, full, a1);
    }
    float z[4][4];
    if (kGen) {
      const uint32_t ids[4] = {i0, i0 + 1, i0 + 2, i0 + 3};
      gauss4_n<4>((uint32_t)(A.n >> 2), ids, (uint32_t)rep, kTagKuramoto, A.keys, z);
#pragma unroll
      for (int e = 0; e < 4; ++e) a2[e] = pick4(z[e], j);
#pragma unroll
      for (int k = 1; k < 4; ++k)
        if (k > j) {
          const float zk[4] = {z[0][k], z[1][k], z[2][k], z[3][k]};
          mfg_store4<true>(psi_out + (int64_t)(k - 1) * A.plane, i0, Nu, full, zk);
        }
    }
    // the sin/cos polynomials of two oscillators at a time on packed FP32 pairs
    float sn[4], cs[4];
    if (MODE == 2) {
      sincos_turns_n<4>(t0, sn, cs);
    } else if (kPred) {
      float s0[4], c0[4], y[4];
      uint32_t tp[4];
      sincos_turns_n<4>(t0, s0, c0);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float g1 = c0[e] * S - s0[e] * C;
        const float wdt = a1[e] * A.wscale;
        const float d1 = fmaf(A.sc, a2[e], fmaf(A.kc, g1, wdt));
        tp[e] = t0[e] + (uint32_t)__float2int_rn(d1 * 4294967296.0f);
        y[e] = fmaf(A.sc, a2[e], fmaf(A.kh, g1, wdt));
      }
      mfg_store4<true>(tt_r, i0, Nu, full, tp);
      mfg_store4<true>(y_r, i0, Nu, full, y);
      sincos_turns_n<4>(tp, sn, cs);
    } else {
      float s2[4], c2[4];
      uint32_t t1[4];
      sincos_turns_n<4>(tt, s2, c2);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float g2 = c2[e] * S - s2[e] * C;
        t1[e] = t0[e] + (uint32_t)__float2int_rn(fmaf(A.kh, g2, a1[e]) * 4294967296.0f);
      }
      mfg_store4<false>(th_r, i0, Nu, full, t1);
      sincos_turns_n<4>(t1, sn, cs);
    }
    if (!full) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (i0 + e >= Nu) sn[e] = cs[e] = 0.0f;
    }
    ps += (sn[0] + sn[1]) + (sn[2] + sn[3]);
    pc += (cs[0] + cs[1]) + (cs[2] + cs[3]);
  }
  const float2 b = block_sum2(ps, pc, red);
  if (threadIdx.x == 0) {
    A.partials[(int64_t)rep * gridDim.x + blockIdx.x] = b;
    __threadfence();
    is_last = atomicAdd(&A.count[rep], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  double s = 0.0, c = 0.0;
  for (int q = threadIdx.x; q < (int)gridDim.x; q += kMfgThreads) {
    const float2 p = __ldcg(&A.partials[(int64_t)rep * gridDim.x + q]);
    s += p.x;
    c += p.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red64[warp] = make_double2(s, c);
  __syncthreads();
  if (threadIdx.x == 0) {
    double S64 = 0.0, C64 = 0.0;
    for (int w = 0; w < kMfgThreads / 32; ++w) {
      S64 += red64[w].x;
      C64 += red64[w].y;
    }
    if (kPred) {
      tot[2] = S64;
      tot[3] = C64;
    } else {
      tot[0] = S64;
      tot[1] = C64;
      if (A.sample_row >= 0 && A.r_out)
        A.r_out[A.sample_row * A.R + rep] = sqrt(S64 * S64 + C64 * C64) / (double)N;
    }
    A.count[rep] = 0u;
  }
}

// ---- pairwise form (Alg. 3) --------------------------------------------

// Every pair term is sin(x_j - x_i) = sin x_j cos x_i - cos x_j sin x_i, two
// FMAs on the sines and cosines of the two phases (each within 7e-8, from the
// fixed-point phases; the kernel that writes a phase writes its pair too).
// Both products of a term enter the receiver's running sum one after the
// other, and in between the sum carries s_j c_i, which rounds at 6e-8 s_j c_i
// however small the term.  So the phases are taken relative to one near
// oscillator 0's: the frame drops out of every difference, and in a population
// that is nearly in step the sines are as small as the terms (spread 1e-3 rad:
// 1e-9 per source, 4e-8 in a fixed frame).  Where the phases are spread the terms
// themselves are of order 1.  The frame of a stage's phases is oscillator 0's phase
// one stage earlier, which every block can read while they are written, moved on
// by its own frequency where the stage is a whole step.
//
// What bounds it: the FMA pipe, once the shared loads are kept below it.  Two
// sources share a packed FP32 FMA (a receiver's sums over even and odd sources
// are added at the end), so one 128-bit load (s0, s1, -c0, -c1), the same for
// all lanes, brings two terms' operands already paired for RPT receivers per
// lane: 2 RPT packed FMAs of 2 cycles on the scheduler's FMA pipe against 4
// cycles of the SM's shared-memory return path, which four schedulers share.
// N = 4096, 64 replicas: 76 us per stage launch to launch (54 us of packed FMAs)
// against 342 us for a polynomial sine per term (9 packed instructions per two
// terms); N = 1000, 3 replicas: 4.3 us against 23 us.
//
// RPT receivers per thread; S slices (warps) of a block take disjoint parts
// of the sources and their partial sums are added in slice order.
struct PairShape {
  int rpt, s;
  int receivers() const { return rpt * 32; }
  int threads() const { return 32 * s; }
};

// A step at oscillator 0's own frequency, in units of the phases.
__device__ __forceinline__ uint32_t frame_step(float omega0, float wscale) {
  return (uint32_t)__float2int_rn(omega0 * wscale * 4294967296.0f);
}

template <int RPT>
__device__ __forceinline__ void pair_terms(const float4 &src, const float (&si)[RPT], const float (&ci)[RPT],
                                           float2 (&acc)[RPT]) {
#pragma unroll
  for (int k = 0; k < RPT; ++k) acc[k] = __ffma2_rn(make_float2(src.x, src.y), make_float2(ci[k], ci[k]), acc[k]);
#pragma unroll
  for (int k = 0; k < RPT; ++k) acc[k] = __ffma2_rn(make_float2(src.z, src.w), make_float2(si[k], si[k]), acc[k]);
}

// One SRK2 stage: receivers i of one replica in this CTA, all sources j
// streamed through shared memory in tiles.  STAGE 0 (predictor) reads the
// phases theta, writes theta~ and the first-stage coupling sum g1; STAGE 1
// (corrector) takes the sums over theta~ and writes the new theta.  STAGE 2
// is PROG2's UpdateRHS: the sums over theta, stored in g1 for the
// AdvanceSystem kernel of the Euler-Maruyama scheme, and that kernel's frame in
// theta~'s first place.
template <int STAGE, int RPT, int S>
__global__ void __launch_bounds__(32 * S) kur_pairwise_stage(const KurPairArgs A) {
  constexpr int THREADS = 32 * S, RPC = RPT * 32;
  constexpr int TILE = S == 1 ? 64 : 1024;  // sources
  constexpr int NP = TILE / 2 / THREADS;
  __shared__ float4 src_s[TILE / 2];
  __shared__ float red[S * RPC];
  const int rep = blockIdx.y;
  const uint32_t N = (uint32_t)A.N;  // < 2^31
  const int64_t base = (int64_t)rep * A.N;
  const float2 *src = (STAGE == 1 ? A.sc_t : A.sc) + base;  // corrector: sums over theta~
  const int t = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * RPC;
  float si[RPT], ci[RPT];
  float2 acc[RPT];
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    const int64_t i = i0 + t + 32 * k;
    const float2 a = i < N ? src[i] : make_float2(0.0f, 0.0f);
    si[k] = a.x;
    ci[k] = a.y;
    acc[k] = make_float2(0.0f, 0.0f);
  }
  // the next tile's sources are in flight during the current tile's terms;
  // sources beyond N are zero terms
  float2 pa[NP], pb[NP];
  auto load = [&](uint32_t j0) {
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const uint32_t j = j0 + 2 * (threadIdx.x + u * THREADS);
      pa[u] = j < N ? src[j] : make_float2(0.0f, 0.0f);
      pb[u] = j + 1 < N ? src[j + 1] : make_float2(0.0f, 0.0f);
    }
  };
  load(0);
  for (uint32_t j0 = 0; j0 < N; j0 += TILE) {
#pragma unroll
    for (int u = 0; u < NP; ++u)
      src_s[threadIdx.x + u * THREADS] = make_float4(pa[u].x, pb[u].x, -pa[u].y, -pb[u].y);
    __syncthreads();
    if (N - j0 > TILE) load(j0 + TILE);
    const int cnt = N - j0 < TILE ? (int)(N - j0) : TILE;
    const int pairs = ((cnt + 7) & ~7) >> 1;
    const int per = ((pairs + S - 1) / S + 3) & ~3;
    const int pe = min((q + 1) * per, pairs);
    for (int p = q * per; p < pe; p += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) pair_terms<RPT>(src_s[p + u], si, ci, acc);
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < RPT; ++k) red[q * RPC + t + 32 * k] = acc[k].x + acc[k].y;
  __syncthreads();
  const uint2 key = seed_to_key(A.seed);
  const int64_t n = A.n;
  if (STAGE == 2 && blockIdx.x == 0 && threadIdx.x == 0) A.theta_t[base] = A.theta[base] + frame_step(A.omega[base], A.wscale);
  for (int rl = threadIdx.x; rl < RPC; rl += THREADS) {
    const int64_t i = i0 + rl;
    if (i >= N) break;
    float g = red[rl];
#pragma unroll
    for (int w = 1; w < S; ++w) g += red[w * RPC + rl];
    const int64_t gi = base + i;
    if (STAGE == 2) {
      A.g1[gi] = g;
      continue;
    }
    float z[4];
    gauss4((uint32_t)(n >> 2), (uint32_t)i, (uint32_t)rep, kTagKuramoto, key, z);
    const float psi = pick4(z, (int)(n & 3));
    const float wdt = A.omega[gi] * A.wscale;
    uint32_t th = A.theta[gi];
    const uint32_t frame = STAGE == 0 ? A.theta[base] + frame_step(A.omega[base], A.wscale) : A.theta_t[base];
    float sn, cs;
    if (STAGE == 0) {
      const float d1 = fmaf(A.sc_noise, psi, fmaf(A.kc, g, wdt));
      th += (uint32_t)__float2int_rn(d1 * 4294967296.0f);
      A.theta_t[gi] = th;
      A.g1[gi] = g;
      sincos_turns(th - frame, sn, cs);
      A.sc_t[gi] = make_float2(sn, cs);
    } else {
      const float d = fmaf(A.sc_noise, psi, fmaf(A.kh, A.g1[gi] + g, wdt));
      th += (uint32_t)__float2int_rn(d * 4294967296.0f);
      A.theta[gi] = th;
      sincos_turns(th - frame, sn, cs);
      A.sc[gi] = make_float2(sn, cs);
    }
  }
}

// sin and cos of every phase, the sources of the first pairwise stage.
__global__ void kur_sincos_kernel(const uint32_t *theta, float2 *sc, int64_t N, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float sn, cs;
    sincos_turns(theta[i] - theta[i / N * N], sn, cs);
    sc[i] = make_float2(sn, cs);
  }
}

// The shape of the pairwise launches.  Eight receivers per thread keep the
// shared loads well below the FMA pipe's time; four slices give each of an
// SM's schedulers one warp of every block (with two, 1024 blocks on 152 SMs
// left 3 warps on one scheduler and 4 on another: 92 us per stage at N = 4096,
// 64 replicas, against 76 us).  Below about twelve warps per SM more slices
// take the place of receivers per thread.  A replica of at most 32 oscillators is
// a single warp's, in a block of little shared memory: with many of them a stage
// lasts as long as its blocks take to come and go (N = 2, 30,000 replicas: 53 us per
// stage with {8, 4}, 19 so; N = 33, 30,000: 69 with {8, 4}).
PairShape pair_shape(int64_t N, int64_t R, int sm_count) {
  if (N <= 32) return {1, 1};
  const int64_t want = (int64_t)sm_count * 12;
  if ((N + 255) / 256 * R * 4 >= want) return {8, 4};
  if ((N + 127) / 128 * R * 8 >= want) return {4, 8};
  return {2, 16};
}

template <int STAGE>
cudaError_t launch_pairwise(const KurPairArgs &a, int64_t R, const PairShape &p, cudaStream_t s) {
  const dim3 grid((unsigned)((a.N + p.receivers() - 1) / p.receivers()), (unsigned)R);
  if (p.s == 4)
    kur_pairwise_stage<STAGE, 8, 4><<<grid, p.threads(), 0, s>>>(a);
  else if (p.s == 8)
    kur_pairwise_stage<STAGE, 4, 8><<<grid, p.threads(), 0, s>>>(a);
  else if (p.s == 1)
    kur_pairwise_stage<STAGE, 1, 1><<<grid, p.threads(), 0, s>>>(a);
  else
    kur_pairwise_stage<STAGE, 2, 16><<<grid, p.threads(), 0, s>>>(a);
  return cudaGetLastError();
}

// ---- pairwise form, a replica per cluster --------------------------------
//
// All steps in one launch, for populations whose stages are shorter than a
// launch: a cluster of CS CTAs holds a replica, every CTA the sines and cosines
// of all its N oscillators in shared memory (twice: theta, theta~) and the
// state of its own share of the receivers in registers.  A stage is the sums
// over one buffer, the sub-step of the own receivers, and their new sines and
// cosines copied into the other buffer of every CTA of the cluster (one bulk
// copy each, counted by the receiver's mbarrier; two alternate).  Nobody still
// reads the buffer being written, or copies from it: a CTA sends stage s + 1
// after it has received stage s from everyone, and each sent that after its
// sums over the buffer that stage s + 1 replaces.  For the same reason a
// receiver has armed a mbarrier again before the next data for it can arrive.
//
// Each warp takes every 16th group of four source pairs for all receivers of
// the CTA, 64 at a time: eight lanes hold eight receivers each, and the four
// groups of eight lanes take different pairs, so that one 16-byte load still
// feeds sixteen packed FMAs (kur_pairwise_stage) however few receivers a CTA
// has, and no warp has more to do than another.
//
// What bounds it: the latency of a stage's steps one after the other (1.5 us at
// 100 oscillators), then the FMA pipe at about half its rate.  1000 oscillators,
// 3 replicas: 4.3 us per step of two stages against 8.6 with a launch per stage;
// with ordinary remote stores and a cluster barrier for the exchange 5.4.
constexpr int kPcThreads = 512, kPcWarps = kPcThreads / 32;
constexpr int kPcGroup = 64;  // receivers taken together

struct PairClusterArgs {
  uint32_t *theta;
  const float *omega;
  double *r_out;  // [samples][R]
  int64_t N, R;
  int64_t n_begin, n_end;
  int32_t M;
  int32_t chunk;   // receivers per CTA, even, <= kPcThreads
  int32_t npairs;  // source pairs, a multiple of 64
  float wscale, kc, kh, sc_noise;
  PhiloxKeys keys;
  uint32_t *err;
  uint64_t wait_ns;  // limit of each wait for the other CTAs' stage
};

constexpr size_t kPcMaxSmem = 200 * 1024;

// Receivers per CTA (whole source pairs) and source pairs (whole rounds of the warps).
__host__ __device__ inline int64_t pair_cluster_chunk(int64_t N, int cs) { return ((N + cs - 1) / cs + 1) & ~1ll; }
__host__ __device__ inline int64_t pair_cluster_pairs(int64_t N) { return ((N + 1) / 2 + 63) / 64 * 64; }
size_t pair_cluster_smem(int64_t chunk, int64_t npairs) {
  const size_t groups = (size_t)((chunk + kPcGroup - 1) / kPcGroup);
  return 2 * sizeof(float4) * (size_t)npairs + sizeof(float) * groups * kPcGroup * kPcWarps;
}

template <bool EULER>
__global__ void __launch_bounds__(kPcThreads, 1) kur_pair_cluster_kernel(const PairClusterArgs A) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ float4 pc_smem[];  // [2][npairs] (s0, s1, -c0, -c1), then the warps' partial sums
  __shared__ float2 red_r[32];
  __shared__ __align__(8) uint64_t mbar[2];
  __shared__ int gave_up;       // some CTA of the cluster did
  __shared__ int late_s;        // a thread of this CTA did
  __shared__ uint32_t sent_s;   // stages this CTA sent
  const int cs = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int rep = blockIdx.x / cs;
  const int N = (int)A.N, chunk = A.chunk, npairs = A.npairs;
  const int groups = (chunk + kPcGroup - 1) / kPcGroup;
  const int64_t base = (int64_t)rep * A.N;
  float *part = reinterpret_cast<float *>(pc_smem + 2 * npairs);  // [warp][groups * 64]
  const int i = crank * chunk + t;  // this thread's receiver
  const bool own = t < chunk && i < N;
  const bool active = (t & ~31) < chunk;  // this warp has receivers
  uint32_t frame = A.theta[base];  // of the sines and cosines sent next (see pair_terms)
  const uint32_t step0 = frame_step(A.omega[base], A.wscale);
  // all sources of theta; pairs beyond N stay zero in both buffers
  for (int p = t; p < npairs; p += kPcThreads) {
    float s0 = 0.0f, c0 = 0.0f, s1 = 0.0f, c1 = 0.0f;
    if (2 * p < N) sincos_turns(A.theta[base + 2 * p] - frame, s0, c0);
    if (2 * p + 1 < N) sincos_turns(A.theta[base + 2 * p + 1] - frame, s1, c1);
    pc_smem[p] = make_float4(s0, s1, -c0, -c1);
    pc_smem[npairs + p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  // the others' copies overwrite these through the asynchronous proxy: ordered after them
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  uint32_t th = own ? A.theta[base + i] : 0u;
  const float wdt = own ? A.omega[base + i] * A.wscale : 0.0f;
  // this CTA's pairs in a buffer, and the bytes a stage brings from the others
  const int first = crank * chunk / 2, mine = max(0, min(chunk / 2, npairs - first));
  const uint32_t bytes = 16u * (uint32_t)(min(npairs, cs * chunk / 2) - mine);
  const uint32_t bar0 = smem_u32(&mbar[0]);
  if (t == 0) {
    gave_up = late_s = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8 * q) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 2; ++q)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar0 + 8 * q), "r"(bytes) : "memory");
  }
  cluster.sync();  // every CTA's buffers and barriers are there before the first copy into them
  uint32_t stage = 0, got = 0;  // stages sent; received, as thread 0 counts them
  bool stop = false;                      // a wait of this CTA expired, as all its threads see it

  // sum_j sin(x_j - x_i) over the sources of buffer b for this thread's receiver
  auto sums = [&](int b) -> float {
    const float4 *src = pc_smem + b * npairs;
    const int l = lane & 7;
    // The next frame: oscillator 0's phase in this buffer, to a first order that
    // follows it within a few stages, and a step on if the phases sent next are.
    // Every CTA holds the same bits of its sine.
    const float s0 = src[0].x;
    frame += (uint32_t)__float2int_rn(683565276.0f * (src[0].z < 0.0f ? s0 : copysignf(1.0f, s0)));  // 2^32 / (2 pi)
    if (EULER || b == 0) frame += step0;
    for (int g = 0; g < groups; ++g) {
      float si[8], ci[8];
      float2 acc[8];
      const int p0 = (crank * chunk + g * kPcGroup) / 2 + l * 4;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 v = p0 + k < npairs ? src[p0 + k] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        si[2 * k] = v.x;
        si[2 * k + 1] = v.y;
        ci[2 * k] = -v.z;
        ci[2 * k + 1] = -v.w;
        acc[2 * k] = acc[2 * k + 1] = make_float2(0.0f, 0.0f);
      }
#pragma unroll 2
      for (int p = warp * 4 + (lane >> 3); p < npairs; p += 4 * kPcWarps) pair_terms<8>(src[p], si, ci, acc);
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        v[k] = acc[k].x + acc[k].y;
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 8);
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 16);
      }
      if (lane < 8) {
        float4 *o = reinterpret_cast<float4 *>(part + (warp * groups + g) * kPcGroup + l * 8);
        o[0] = make_float4(v[0], v[1], v[2], v[3]);
        o[1] = make_float4(v[4], v[5], v[6], v[7]);
      }
    }
    __syncthreads();
    stop = *(volatile int *)&late_s != 0;  // written before this barrier or after publish's
    float sum = 0.0f;
    if (t < chunk) {
#pragma unroll
      for (int w = 0; w < kPcWarps; ++w) sum += part[w * groups * kPcGroup + t];
    }
    return sum;
  };
  // the new sine and cosine of the own receiver into buffer b of every CTA; not
  // called once a wait of this CTA has expired (the others' waits expire too)
  auto publish = [&](uint32_t phase, int b) {
    float4 *dst = pc_smem + b * npairs;
    if (active) {
      float sn, cs_;
      sincos_turns(phase - frame, sn, cs_);
      if (!own) sn = cs_ = 0.0f;
      const float s1 = __shfl_xor_sync(0xffffffffu, sn, 1), c1 = __shfl_xor_sync(0xffffffffu, cs_, 1);
      if ((t & 1) == 0 && t / 2 < mine) {
        dst[first + t / 2] = make_float4(sn, s1, -cs_, -c1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
    }
    __syncthreads();
    if (lane == 0 && warp < cs && warp != crank && mine > 0) {
      const uint32_t from = smem_u32(dst + first);
      asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       cluster_map(from, (uint32_t)warp)),
                   "r"(from), "r"(16u * (uint32_t)mine), "r"(cluster_map(bar0 + 8 * (stage & 1u), (uint32_t)warp))
                   : "memory");
    }
  };
  // the other CTAs' part of the stage
  auto receive = [&]() {
    if (bytes > 0) {
      const uint32_t bar = bar0 + 8 * (stage & 1u), parity = (stage >> 1) & 1u;
      if (!mbar_wait_bounded(bar, parity, A.wait_ns)) {
        *(volatile int *)&late_s = 1;
        atomicOr(A.err, kErrTimeout);
      } else if (t == 0) {
        ++got;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      }
    }
    ++stage;
  };
  auto order = [&](int b, int64_t row) {  // r(t) of the replica, by the CTA of rank 0
    float S = 0.0f, C = 0.0f;
    for (int p = t; p < npairs; p += kPcThreads) {
      const float4 v = pc_smem[b * npairs + p];
      S += v.x + v.y;
      C -= v.z + v.w;
    }
    const float2 sc = block_sum2(S, C, red_r);
    if (t == 0) {
      const double Sd = sc.x, Cd = sc.y;
      A.r_out[row * A.R + rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
    }
    __syncthreads();
  };

  int b = 0;  // the buffer of theta_n
  int64_t row = 0;
  int m = 0;  // (n - n_begin) mod M
  float z[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  auto draw = [&](int64_t n) {
    if (active) gauss4((uint32_t)(n >> 2), (uint32_t)i, (uint32_t)rep, kTagKuramoto, A.keys, z);
  };
  if (A.n_begin < A.n_end) draw(A.n_begin);
  for (int64_t n = A.n_begin; n < A.n_end; ++n) {
    if (A.M > 0) {
      if (m == 0) {
        if (crank == 0) order(b, row);
        ++row;
      }
      if (++m == A.M) m = 0;
    }
    const float psi = pick4(z, (int)(n & 3));
    const float g1 = sums(b);
    if (stop) break;
    const float d1 = fmaf(A.sc_noise, psi, fmaf(A.kc, g1, wdt));
    const uint32_t tp = th + (uint32_t)__float2int_rn(d1 * 4294967296.0f);
    if (EULER) {
      th = tp;
      b ^= 1;
    } else {
      publish(tp, 1);
      receive();
      const float g2 = sums(1);
      if (stop) break;
      const float d = fmaf(A.sc_noise, psi, fmaf(A.kh, g1 + g2, wdt));
      th += (uint32_t)__float2int_rn(d * 4294967296.0f);
    }
    publish(th, b);
    if (((n + 1) & 3) == 0) draw(n + 1);  // while the others' data arrives
    receive();
  }
  if (A.M > 0 && crank == 0 && !stop) order(b, row);  // meaningless after an expired wait, like theta
  if (own) A.theta[base + i] = th;
  if (cs == 1) return;
  if (t == 0) sent_s = stage;
  __syncthreads();
  cluster_drain(*(volatile int *)&late_s != 0, got, bar0, &gave_up, cs, [&](uint32_t s) {
    uint32_t miss = 0;
    for (int q = 0; q < cs; ++q)
      if (q != crank && *(volatile uint32_t *)cluster.map_shared_rank(&sent_s, q) <= s)
        miss += 16u * (uint32_t)max(0, min(chunk / 2, npairs - q * chunk / 2));
    return miss;
  });
}

// Shared memory and cluster size of the kernel's launches (not under capture).
cudaError_t pair_cluster_configure() {
  for (const void *fn : {(const void *)kur_pair_cluster_kernel<false>, (const void *)kur_pair_cluster_kernel<true>}) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPcMaxSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaLaunchConfig_t pair_cluster_config(int64_t N, int64_t R, int cs, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(R * cs));
  cfg.blockDim = dim3(kPcThreads);
  cfg.dynamicSmemBytes = pair_cluster_smem(pair_cluster_chunk(N, cs), pair_cluster_pairs(N));
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)cs;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

cudaError_t launch_pair_cluster(const PairClusterArgs &a, int cs, bool euler, cudaStream_t s) {
  cudaLaunchAttribute attr;
  cudaLaunchConfig_t cfg = pair_cluster_config(a.N, a.R, cs, &attr);
  cfg.stream = s;
  if (euler) return cudaLaunchKernelEx(&cfg, kur_pair_cluster_kernel<true>, a);
  return cudaLaunchKernelEx(&cfg, kur_pair_cluster_kernel<false>, a);
}

// CTAs per replica of the cluster form, or 0 where a launch per stage is the
// faster one, from a model of both in ns per stage.  A launch: 3.6 us and the
// busiest SM's blocks at the rate that their receivers per thread reach; a
// cluster stage: 1.3 us of sums, sub-step and exchange, and per 64 receivers 0.33
// us and 1.17 ns per source pair, times the waves of clusters.  Both sides
// measured, us per stage, launch and cluster: 1000 oscillators x 3 replicas 4.3
// and 2.2, x 19 6.4 and 5.2, x 40 8.4 and 8.9; 2000 x 1 6.4 and 4.5, x 9 8.4 and
// 7.5, x 18 10.5 and 13.0; 3000 x 2 6.4 and 7.8; 4096 x 1 8.4 and 12; 900 x 64
// 10.5 and 8.9; 300 x 200 6.4 and 9.1.
int pair_cluster_size(int64_t N, int64_t R, bool euler, int sm_count) {
  const double terms_per_ns = 128.0 / 2 * 1.9;  // of an SM: two FMAs per term
  const PairShape shape = pair_shape(N, R, sm_count);
  const int64_t blocks = (N + shape.receivers() - 1) / shape.receivers() * R;
  const double slack = shape.rpt == 8 ? 1.25 : (shape.rpt == 4 ? 1.6 : 2.2);  // shared loads per FMA
  const double busiest = (double)((blocks + sm_count - 1) / sm_count) * shape.receivers() * (double)N;
  double best = 3600.0 + slack * busiest / terms_per_ns + (euler ? 3000.0 : 0.0);  // PROG2's second launch
  int best_cs = 0;
  for (int cs = 16; cs >= 1; cs >>= 1) {
    const int64_t chunk = pair_cluster_chunk(N, cs), npairs = pair_cluster_pairs(N);
    if (chunk > kPcThreads || R * cs > 1 << 20 || pair_cluster_smem(chunk, npairs) > kPcMaxSmem) continue;
    const double groups = (double)((chunk + kPcGroup - 1) / kPcGroup);
    const double stage = 1300.0 + groups * (330.0 + 1.17 * (double)npairs);
    if (stage * (double)((R * cs + sm_count - 1) / sm_count) >= best) continue;  // without asking the driver
    if (pair_cluster_configure() != cudaSuccess) break;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = pair_cluster_config(N, R, cs, &attr);
    int resident = 0;
    if (cudaOccupancyMaxActiveClusters(&resident, (const void *)kur_pair_cluster_kernel<false>, &cfg) != cudaSuccess ||
        resident < 1)
      continue;
    const double ns = stage * (double)((R + resident - 1) / resident);
    if (ns < best) {
      best = ns;
      best_cs = cs;
    }
  }
  cudaGetLastError();  // a form that the device does not take is no error
  return best_cs;
}

// PROG2's AdvanceSystem with Euler-Maruyama: theta += wdt + kc g + sc psi
// for every oscillator of every replica, g the stored coupling sums.
__global__ void kur_advance_euler_kernel(const KurPairArgs A, int64_t R) {
  const uint2 key = seed_to_key(A.seed);
  const int64_t NR = A.N * R;
  for (int64_t gi = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; gi < NR;
       gi += (int64_t)gridDim.x * blockDim.x) {
    const int64_t rep = gi / A.N, i = gi - rep * A.N;
    float z[4];
    gauss4((uint32_t)(A.n >> 2), (uint32_t)i, (uint32_t)rep, kTagKuramoto, key, z);
    const float d = fmaf(A.sc_noise, pick4(z, (int)(A.n & 3)), fmaf(A.kc, A.g1[gi], A.omega[gi] * A.wscale));
    const uint32_t th = A.theta[gi] + (uint32_t)__float2int_rn(d * 4294967296.0f);
    A.theta[gi] = th;
    float sn, cs;
    sincos_turns(th - A.theta_t[rep * A.N], sn, cs);
    A.sc[gi] = make_float2(sn, cs);
  }
}

// r(t) of every replica from fixed-point phases (one CTA per replica).
__global__ void kur_order_kernel(const uint32_t *theta, int64_t N, int64_t R, double *r_out) {
  __shared__ float2 red[32];
  const int rep = blockIdx.x;
  float S = 0.0f, C = 0.0f;
  for (int64_t i = threadIdx.x; i < N; i += blockDim.x) {
    float sn, cs;
    sincos_turns(theta[(int64_t)rep * N + i], sn, cs);
    S += sn;
    C += cs;
  }
  const float2 sc = block_sum2(S, C, red);
  if (threadIdx.x == 0) {
    const double Sd = sc.x, Cd = sc.y;
    r_out[rep] = sqrt(Sd * Sd + Cd * Cd) / (double)N;
  }
}

// Radians (any range) <-> fixed-point turns.  Phases in [0, 8) -- every phase a
// run returns -- go through 64-bit integers: phi 2^61 (exact down to 2^-38)
// times 2^66 / (2 pi) has turns 2^63 in its high word, within 2^-60 of the exact
// product, closer than FP64's 53 bits; other values take the FP64 path.  FP64
// multiplies on this GPU made the two kernels 189 and 125 us for 2^24 phases;
// with integers both take 50 us together.
__device__ __forceinline__ uint32_t phase_to_turns(float phi) {
  const uint32_t bits = __float_as_uint(phi);
  if (bits >= 0x41000000u) {  // negative, >= 8, or not finite
    double t = (double)phi * 0.15915494309189533577;  // 1 / (2 pi)
    t -= floor(t);
    return (uint32_t)(uint64_t)llrint(t * 4294967296.0);
  }
  const int e = (int)(bits >> 23) - 127 + 38;  // shift of the 24-bit mantissa
  if (e < 0) return 0u;                        // below 2^-38: far less than half a unit
  const uint64_t u = (uint64_t)((bits & 0x7FFFFFu) | 0x800000u) << e;
  return (uint32_t)((__umul64hi(u, 0xA2F9836E4E441529ull) + (1ull << 30)) >> 31);  // 2^66 / (2 pi)
}

__device__ __forceinline__ float turns_to_phase(uint32_t th) {
  const uint64_t p = __umul64hi((uint64_t)th << 32, 0xC90FDAA22168C234ull);  // 2 pi 2^61: th 2 pi 2^29
  return __ull2float_rn(p) * 4.3368086899420177e-19f;                         // 2^-61
}

// Four phases per thread in 16-byte accesses where both arrays allow it.
__global__ void kur_to_fixed(const float *phi, uint32_t *theta, int64_t n) {
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  int64_t done = 0;
  if ((((uintptr_t)phi | (uintptr_t)theta) & 15u) == 0u) {
    done = n & ~3ll;
    for (int64_t i = t0; i < n / 4; i += stride) {
      const float4 v = reinterpret_cast<const float4 *>(phi)[i];
      reinterpret_cast<uint4 *>(theta)[i] =
          make_uint4(phase_to_turns(v.x), phase_to_turns(v.y), phase_to_turns(v.z), phase_to_turns(v.w));
    }
  }
  for (int64_t i = done + t0; i < n; i += stride) theta[i] = phase_to_turns(phi[i]);
}

__global__ void kur_from_fixed(const uint32_t *theta, float *phi, int64_t n) {
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  int64_t done = 0;
  if ((((uintptr_t)phi | (uintptr_t)theta) & 15u) == 0u) {
    done = n & ~3ll;
    for (int64_t i = t0; i < n / 4; i += stride) {
      const uint4 v = reinterpret_cast<const uint4 *>(theta)[i];
      reinterpret_cast<float4 *>(phi)[i] =
          make_float4(turns_to_phase(v.x), turns_to_phase(v.y), turns_to_phase(v.z), turns_to_phase(v.w));
    }
  }
  for (int64_t i = done + t0; i < n; i += stride) phi[i] = turns_to_phase(theta[i]);
}

// Observables: mean, variance and standard error of r over replicas for
// each sample row (one warp per row, fixed summation order).
__global__ void kur_obs_kernel(const double *r, int64_t rows, int64_t R, int64_t n_begin, int64_t n_end,
                               int M, double dt, sde_obs_row *obs) {
  const int64_t row = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  double s = 0.0;
  for (int64_t q = lane; q < R; q += 32) s += r[row * R + q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const double mean = s / (double)R;
  double m2 = 0.0;
  for (int64_t q = lane; q < R; q += 32) {
    const double d = r[row * R + q] - mean;
    m2 += d * d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
  if (lane == 0) {
    sde_obs_row o;
    o.mean = mean;
    o.count = (double)R;
    o.var = R > 1 ? m2 / (double)(R - 1) : 0.0;
    o.se = sqrt(o.var / (double)R);
    const int64_t n = row == rows - 1 ? n_end : n_begin + row * (int64_t)M;
    o.t = (double)n * dt;
    obs[row] = o;
  }
}

// Direct coupling sums for the uniform models: out[r][i] = (K/N) sum_j
// sin(x_j - x_i), accurate sinpif per pair (inspection path, not the
// integrator).
__global__ void kur_coupling_uniform_kernel(const uint32_t *theta, float *out, int64_t N, float KoverN) {
  __shared__ float src_s[256];
  const int rep = blockIdx.y;
  const int64_t base = (int64_t)rep * N;
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const float ti = i < N ? (float)(int32_t)theta[base + i] * 2.3283064365386963e-10f : 0.0f;
  float acc = 0.0f;
  for (int64_t j0 = 0; j0 < N; j0 += 256) {
    const int cnt = (N - j0) < 256 ? (int)(N - j0) : 256;
    if (threadIdx.x < cnt) src_s[threadIdx.x] = (float)(int32_t)theta[base + j0 + threadIdx.x] * 2.3283064365386963e-10f;
    __syncthreads();
    for (int jj = 0; jj < cnt; ++jj) {
      float d = src_s[jj] - ti;
      d -= rintf(d);
      acc += sinpif(2.0f * d);
    }
    __syncthreads();
  }
  if (i < N) out[base + i] = KoverN * acc;
}

// FULL: every thread holds OPT oscillators of its replica, so none is masked.
template <int OPT, bool FULL>
cudaError_t launch_mf_cluster(const KurArgs &a, int block, int cs, bool async, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.R * cs));
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (async) return cudaLaunchKernelEx(&cfg, kur_meanfield_async_kernel<OPT, FULL>, a);
  return cudaLaunchKernelEx(&cfg, kur_meanfield_cluster_kernel<OPT, FULL>, a);
}

// cs > 1: one replica per cluster of cs CTAs (opt oscillators per thread of
// each CTA); cs == 1: one CTA per replica.
template <int OPT>
cudaError_t launch_mf(const KurArgs &a, int block, int cs, bool async, cudaStream_t s) {
  constexpr bool kPow2 = (OPT & (OPT - 1)) == 0;  // the unmasked form is built for these only
  const bool full = kPow2 && a.N == (int64_t)cs * block * OPT;
  if (cs > 1) {
    if constexpr (OPT <= 8) {
      if (full) return launch_mf_cluster<OPT, kPow2>(a, block, cs, async, s);
      return launch_mf_cluster<OPT, false>(a, block, cs, async, s);
    }
    return cudaErrorInvalidValue;
  }
  if (full)
    kur_meanfield_kernel<OPT, kPow2><<<(unsigned)a.R, block, 0, s>>>(a);
  else
    kur_meanfield_kernel<OPT, false><<<(unsigned)a.R, block, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_meanfield(const KurArgs &a, int block, int opt, int cs, bool async, cudaStream_t s) {
  switch (opt) {
    case 1: return launch_mf<1>(a, block, cs, async, s);
    case 2: return launch_mf<2>(a, block, cs, async, s);
    case 3: return launch_mf<3>(a, block, cs, async, s);
    case 4: return launch_mf<4>(a, block, cs, async, s);
    case 5: return launch_mf<5>(a, block, cs, async, s);
    case 6: return launch_mf<6>(a, block, cs, async, s);
    case 8: return launch_mf<8>(a, block, cs, async, s);
    case 16: return launch_mf<16>(a, block, cs, async, s);
    default: return cudaErrorInvalidValue;
  }
}

// Blocks per replica of the grid-wide mean field, enough oscillators per
// thread to amortise the reduction: one full wave of each kernel (resident blocks per SM from the occupancy
// calculator x SMs, shared among the replicas), at most one block per
// kMfgThreads x kMfgIlp oscillators.
void mfg_grid_for(int64_t N, int64_t R, int sm_count, int grid[4]) {
  const void *fn[4] = {(const void *)kur_mfg_kernel<0>, (const void *)kur_mfg_kernel<1>,
                       (const void *)kur_mfg_kernel<2>, (const void *)kur_mfg_kernel<3>};
  const int64_t need = (N + kMfgThreads * kMfgIlp - 1) / (kMfgThreads * kMfgIlp);
  for (int m = 0; m < 4; ++m) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn[m], kMfgThreads, 0) != cudaSuccess)
      per_sm = 4;
    const int64_t fill = std::max<int64_t>(1, ((int64_t)std::max(1, per_sm) * sm_count + R - 1) / R);
    grid[m] = (int)std::max<int64_t>(1, std::min<int64_t>(need, fill));
  }
}

cudaError_t launch_mfg(const MfgArgs &a, int mode, int blocks, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks, (unsigned)a.R);
  cfg.blockDim = dim3(kMfgThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;  // chain_begin
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  switch (mode) {
    case 0: return cudaLaunchKernelEx(&cfg, kur_mfg_kernel<0>, a);
    case 1: return cudaLaunchKernelEx(&cfg, kur_mfg_kernel<1>, a);
    case 3: return cudaLaunchKernelEx(&cfg, kur_mfg_kernel<3>, a);
    default: return cudaLaunchKernelEx(&cfg, kur_mfg_kernel<2>, a);
  }
}

// Oscillators per thread the replica kernels are built for, the smallest that
// holds x (17 if none does): with powers of two alone N = 5000 ran at 8 per
// thread where 5 hold it (2.1 instead of 1.4 us per step for 20 replicas).
int opt_at_least(int64_t x) {
  for (int o : {1, 2, 3, 4, 5, 6, 8, 16})
    if (o >= x) return o;
  return 17;
}

}  // namespace

// ---------------------------------------------------------------------------

namespace {

struct MfShape {
  int cs, block, opt;
  bool async;  // cluster exchange by st.async + mbarrier instead of a cluster barrier
};

// Candidate shapes for the mean-field kernel: one CTA per replica, or a
// cluster of 2, 4 or 8 CTAs per replica (distributed shared memory
// reductions; more, smaller CTAs let co-resident replicas overlap each
// other's barrier latency).
std::vector<MfShape> meanfield_candidates(int64_t N) {
  std::vector<MfShape> out;
  for (int cs : {1, 2, 4, 8}) {
    const int64_t chunk = (N + cs - 1) / cs;
    for (int block : {128, 256, 512, 1024}) {
      if (block == 128 && cs < 8) continue;
      if (cs > 1 && cs * (block / 32) > 32) continue;  // one exchange slot per warp of the cluster
      if (block > ((chunk + 31) / 32) * 32 && block > 256) continue;  // mostly idle threads
      const int opt = opt_at_least((chunk + block - 1) / block);
      const int max_opt = cs > 1 ? 8 : 16;
      const int max_block = cs > 1 ? 512 : (opt <= 2 ? 1024 : 512);
      if (opt > max_opt || block > max_block) continue;
      out.push_back({cs, block, opt, false});
      if (cs > 1) out.push_back({cs, block, opt, true});
    }
  }
  return out;
}

}  // namespace

MfgArgs mfg_args(KuramotoCtx *k, const float *omega, double *rbuf) {
  const double inv2pi = 0.15915494309189533577;
  MfgArgs a{};
  a.theta = k->theta;
  a.theta_t = k->theta_t;
  a.y = k->g1;
  a.psi = k->psi4;
  a.plane = mfg_plane(k->N * k->R);
  a.omega = omega;
  a.omega_vec = ((uintptr_t)omega & 15u) == 0u;
  a.partials = k->mfg_partials;
  a.tot = k->mfg_tot;
  a.count = k->mfg_count;
  a.r_out = rbuf;
  a.N = k->N;
  a.R = k->R;
  a.wscale = (float)(k->dt * inv2pi);
  a.kc = (float)(k->K / (double)k->N * k->dt * inv2pi);
  a.kh = (float)(0.5 * k->K / (double)k->N * k->dt * inv2pi);
  a.sc = (float)(sqrt(2.0 * k->D * k->dt) * inv2pi);
  a.keys = philox_round_keys(k->seed);
  return a;
}

// Steps [n_begin, n_end) of the grid-wide mean field: the sums of theta at
// n_begin, then predictor and corrector launches per step.  r(t) rows as in
// the single-CTA form: every M steps from n_begin, plus n_end as the last row.
sde_status run_meanfield_grid(KuramotoCtx *k, int64_t n_begin, int64_t n_end, const float *omega,
                              double *rbuf, int64_t n_rows, cudaStream_t s) {
  MfgArgs a = mfg_args(k, omega, rbuf);
  const int *grid = k->mfg_grid;
  a.n = n_begin;
  a.sample_row = n_rows > 0 ? 0 : -1;
  a.reverse = true;
  SDE_CUDA_TRY(launch_mfg(a, 2, grid[2], s));
  for (int64_t n = n_begin; n < n_end; ++n) {
    a.n = n;
    const int pred = (n == n_begin || (n & 3) == 0) ? 3 : 0;
    a.sample_row = -1;
    a.reverse = false;
    SDE_CUDA_TRY(ktime_begin(k, s));
    SDE_CUDA_TRY(launch_mfg(a, pred, grid[pred], s));
    SDE_CUDA_TRY(ktime_end(k, s));
    const int64_t m = n + 1;
    if (n_rows > 0) {
      if (m == n_end)
        a.sample_row = n_rows - 1;
      else if ((m - n_begin) % k->M == 0)
        a.sample_row = (m - n_begin) / k->M;
    }
    a.reverse = true;
    SDE_CUDA_TRY(ktime_begin(k, s));
    SDE_CUDA_TRY(launch_mfg(a, 1, grid[1], s));
    SDE_CUDA_TRY(ktime_end(k, s));
  }
  return SDE_OK;
}

// Time a short run of every candidate shape on scratch phases and keep the
// fastest.
sde_status meanfield_autotune(KuramotoCtx *k, int only_cs, bool with_grid) {
  auto cands = meanfield_candidates(k->N);
  if (k->flags & SDE_FLAG_ASYNC_EXCHANGE) {
    std::vector<MfShape> keep;
    for (const auto &c : cands)
      if (c.async) keep.push_back(c);
    cands.swap(keep);
  } else if (with_grid && only_cs == 0) {
    cands.push_back({0, kMfgThreads, 0, false});
  }
  if (only_cs > 0) {
    std::vector<MfShape> keep;
    for (const auto &c : cands)
      if (c.cs == only_cs) keep.push_back(c);
    cands.swap(keep);
  }
  if (cands.empty()) {
    set_error("invalid argument: no mean-field launch shape holds n_osc = " + std::to_string(k->N));
    return SDE_ERR_INVALID_ARG;
  }
  const size_t NR = (size_t)k->N * (size_t)k->R;
  float *omega = nullptr;
  cudaStream_t s = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  sde_status st = SDE_OK;
  cudaError_t e;
  if ((e = device_alloc((void **)&omega, NR * 4)) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
  if ((e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking)) != cudaSuccess) st = cuda_fail(e, "stream");
  if (st == SDE_OK && (e = cudaEventCreate(&e0)) != cudaSuccess) st = cuda_fail(e, "event");
  if (st == SDE_OK && (e = cudaEventCreate(&e1)) != cudaSuccess) st = cuda_fail(e, "event");
  if (st == SDE_OK) {
    cudaMemsetAsync(omega, 0, NR * 4, s);
    cudaMemsetAsync(k->theta, 0, NR * 4, s);
    KurArgs a{};
    a.theta_in = k->theta;
    a.theta_out = k->theta;
    a.omega = omega;
    a.r_out = nullptr;
    a.N = k->N;
    a.R = k->R;
    a.n_begin = 0;
    a.n_end = 64;
    a.M = 0;
    a.wscale = 1e-3f;
    a.kc = 1e-4f;
    a.kh = 5e-5f;
    a.sc = 1e-3f;
    a.keys = philox_round_keys(0);
    a.err = k->err;
    a.wait_ns = k->wait_ns;
    float best = 1e30f;
    for (const MfShape &c : cands) {
      float tmin = 1e30f;
      for (int rep = 0; rep < 3 && st == SDE_OK; ++rep) {
        cudaEventRecord(e0, s);
        if (c.cs == 0) {
          const uint32_t flags = k->flags;
          k->flags &= ~SDE_FLAG_TIME_KERNELS;
          st = run_meanfield_grid(k, a.n_begin, a.n_end, omega, nullptr, 0, s);
          k->flags = flags;
          if (st != SDE_OK) break;
        } else if ((e = launch_meanfield(a, c.block, c.opt, c.cs, c.async, s)) != cudaSuccess) {
          st = cuda_fail(e, "mean-field autotune launch");
          break;
        }
        cudaEventRecord(e1, s);
        if ((e = cudaEventSynchronize(e1)) != cudaSuccess) {
          st = cuda_fail(e, "mean-field autotune");
          break;
        }
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0) tmin = std::min(tmin, ms);
      }
      if (st != SDE_OK) break;
      if (tmin < best) {
        best = tmin;
        k->cs = c.cs;
        k->mf_async = c.async;
        k->block = c.block;
        k->opt = c.opt;
      }
    }
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (s) cudaStreamDestroy(s);
  cudaFree(omega);
  if (st == SDE_OK) cudaMemset(k->err, 0, sizeof(uint32_t));  // scratch runs report nothing
  return st;
}

sde_status kuramoto_validate(const sde_config *cfg) {
  SDE_CHECK_ARG(cfg->n_osc >= 1, "n_osc must be >= 1");
  SDE_CHECK_ARG(cfg->n_replicas >= 1 && cfg->n_replicas <= 65535, "n_replicas must be in [1, 65535]");
  SDE_CHECK_ARG(isfinite(cfg->K) && isfinite(cfg->D) && isfinite(cfg->dt), "K, D, dt must be finite");
  SDE_CHECK_ARG(cfg->D >= 0.0, "D must be >= 0");
  SDE_CHECK_ARG(cfg->dt > 0.0, "dt must be > 0");
  SDE_CHECK_ARG(cfg->sample_every >= 0, "sample_every must be >= 0");
  SDE_CHECK_ARG(cfg->n_osc < (1ll << 31), "n_osc too large");
  if (cfg->flags & SDE_FLAG_EULER) {
    if (cfg->model != SDE_KURAMOTO_PAIRWISE) {
      set_error("unsupported: Euler-Maruyama (SDE_FLAG_EULER) is built for the Josephson and the "
                "pairwise Kuramoto models");
      return SDE_ERR_UNSUPPORTED;
    }
  }
  const bool mf = cfg->model == SDE_KURAMOTO_MEANFIELD;
  if (mf)
    SDE_CHECK_ARG(cfg->schedule == SDE_SCHED_PERSISTENT || cfg->schedule == SDE_SCHED_GRID,
                  "mean-field schedule must be SDE_SCHED_PERSISTENT (choose the form) or SDE_SCHED_GRID");
  else
    SDE_CHECK_ARG(cfg->schedule == SDE_SCHED_PERSISTENT, "schedule must be 0 for this Kuramoto model");
  // Forms of the mean field: a replica per CTA or cluster (n_osc <= 8192), or
  // spread over the whole grid (any n_osc; forced by SDE_SCHED_GRID).
  const bool grid_forced = mf && (cfg->schedule == SDE_SCHED_GRID || cfg->n_osc > 8192);
  if (grid_forced)
    SDE_CHECK_ARG(cfg->cluster_ctas == 0 && cfg->block_threads == 0,
                  "the grid-wide mean field takes cluster_ctas = 0 and block_threads = 0");
  return SDE_OK;
}

sde_status kuramoto_create(const sde_config *cfg, int sm_count, uint32_t *err, KuramotoCtx **out) {
  *out = nullptr;
  const sde_status vs = kuramoto_validate(cfg);
  if (vs != SDE_OK) return vs;
  const bool mf = cfg->model == SDE_KURAMOTO_MEANFIELD;
  const bool grid_forced = mf && (cfg->schedule == SDE_SCHED_GRID || cfg->n_osc > 8192);
  KuramotoCtx *k = new (std::nothrow) KuramotoCtx();
  if (!k) {
    set_error("host allocation failed");
    return SDE_ERR_NO_MEMORY;
  }
  k->model = cfg->model;
  k->N = cfg->n_osc;
  k->R = cfg->n_replicas;
  k->K = cfg->K;
  k->D = cfg->D;
  k->dt = cfg->dt;
  k->M = cfg->sample_every;
  k->seed = cfg->seed;
  k->sm_count = sm_count;
  k->err = err;
  k->flags = cfg->flags;
  const size_t NR = (size_t)k->N * (size_t)k->R;
  sde_status st = SDE_OK;
  cudaError_t e;
  auto alloc = [&](void **p, size_t bytes) {
    if (st != SDE_OK) return;
    if ((e = device_alloc(p, bytes ? bytes : 1)) != cudaSuccess) st = cuda_fail(e, "cudaMalloc");
  };
  alloc((void **)&k->theta, NR * 4);
  // the grid-wide form is a candidate when few replicas leave SMs idle
  const bool grid_possible =
      mf && (grid_forced || (cfg->cluster_ctas == 0 && cfg->block_threads == 0 && cfg->n_replicas * 4 < sm_count));
  const bool pairwise = cfg->model == SDE_KURAMOTO_PAIRWISE;
  if (pairwise)
    k->pair_cs = pair_cluster_size(k->N, k->R, (cfg->flags & SDE_FLAG_EULER) != 0, sm_count);
  if ((pairwise && k->pair_cs == 0) || grid_possible) {
    alloc((void **)&k->theta_t, NR * 4);
    alloc((void **)&k->g1, NR * 4);
  }
  if (pairwise && k->pair_cs == 0) alloc((void **)&k->pair_sc, NR * 2 * sizeof(float2));
  if (grid_possible) {
    mfg_grid_for(k->N, k->R, sm_count, k->mfg_grid);
    k->mfg_blocks = *std::max_element(k->mfg_grid, k->mfg_grid + 4);
    alloc((void **)&k->mfg_partials, sizeof(float2) * (size_t)k->mfg_blocks * (size_t)k->R);
    alloc((void **)&k->mfg_tot, sizeof(double) * 4 * (size_t)k->R);
    alloc((void **)&k->mfg_count, sizeof(uint32_t) * (size_t)k->R);
    alloc((void **)&k->psi4, sizeof(float) * 3 * (size_t)mfg_plane((int64_t)NR));
    if (st == SDE_OK && (e = cudaMemset(k->mfg_count, 0, sizeof(uint32_t) * (size_t)k->R)) != cudaSuccess)
      st = cuda_fail(e, "cudaMemset");
  }
  if (st == SDE_OK && (cfg->model == SDE_KURAMOTO_GENERAL || cfg->model == SDE_KURAMOTO_GENERAL_FP32))
    st = kuramoto_general_alloc(k);
  if (st != SDE_OK) {
    kuramoto_destroy(k);
    return st;
  }
  // Launch shape.
  SDE_CHECK_ARG(cfg->cluster_ctas == 0 || cfg->cluster_ctas == 1 || cfg->cluster_ctas == 2 ||
                    cfg->cluster_ctas == 4 || cfg->cluster_ctas == 8,
                "cluster_ctas must be 0, 1, 2, 4 or 8");
  if (grid_forced) {
    k->cs = 0;
    k->block = kMfgThreads;
  } else if (cfg->model == SDE_KURAMOTO_MEANFIELD && cfg->block_threads == 0) {
    st = meanfield_autotune(k, cfg->cluster_ctas, grid_possible);
    if (st != SDE_OK) {
      kuramoto_destroy(k);
      return st;
    }
  } else if (cfg->model == SDE_KURAMOTO_MEANFIELD && cfg->cluster_ctas > 1) {
    // a fixed cluster shape: cs CTAs of block threads per replica
    const int cs = cfg->cluster_ctas, block = cfg->block_threads;
    const int64_t chunk = (k->N + cs - 1) / cs;
    const int opt = opt_at_least((chunk + block - 1) / block);
    if (block < 32 || block % 32 != 0 || block > 512 || cs * (block / 32) > 32 || opt > 8) {
      kuramoto_destroy(k);
      set_error("invalid argument: with cluster_ctas > 1, block_threads must be a multiple of 32, at most "
                "512 and at most 32 warps per cluster, with at most 8 oscillators per thread");
      return SDE_ERR_INVALID_ARG;
    }
    k->cs = cs;
    k->block = block;
    k->opt = opt;
    k->mf_async = (cfg->flags & SDE_FLAG_ASYNC_EXCHANGE) != 0;
  } else if (cfg->model == SDE_KURAMOTO_MEANFIELD) {
    int block = cfg->block_threads;
    int opt = opt_at_least((k->N + block - 1) / block);
    if (block < 32 || block % 32 != 0 || block > (opt <= 2 ? 1024 : 512) || opt > 16) {
      kuramoto_destroy(k);
      set_error("invalid argument: block_threads must be a multiple of 32, at most 1024 for <= 2 "
                "oscillators per thread and 512 above, with at most 16 oscillators per thread");
      return SDE_ERR_INVALID_ARG;
    }
    k->block = block;
    k->opt = opt;
  } else if (pairwise && k->pair_cs > 0) {
    k->cs = k->pair_cs;
    k->block = kPcThreads;
    k->opt = 1;
  } else if (pairwise) {
    const PairShape p = pair_shape(k->N, k->R, sm_count);
    k->block = p.threads();
    k->opt = p.rpt;
  }
  *out = k;
  return SDE_OK;
}

void kuramoto_tuning(const KuramotoCtx *k, int32_t *block, int32_t *per_thread, int32_t *cluster) {
  if (block) *block = k->block;
  if (per_thread)
    *per_thread = (k->model == SDE_KURAMOTO_MEANFIELD && k->cs == 0)
                      ? (int32_t)((k->N + (int64_t)k->mfg_grid[0] * kMfgThreads - 1) /
                                  ((int64_t)k->mfg_grid[0] * kMfgThreads))
                      : k->opt;
  if (cluster) *cluster = k->cs;
}

cudaError_t ktime_begin(KuramotoCtx *k, cudaStream_t s) {
  if (!(k->flags & SDE_FLAG_TIME_KERNELS)) return cudaSuccess;
  while ((int64_t)k->kev.size() < 2 * (k->kev_used + 1)) {
    cudaEvent_t e;
    const cudaError_t err = cudaEventCreate(&e);
    if (err != cudaSuccess) return err;
    k->kev.push_back(e);
  }
  return cudaEventRecord(k->kev[2 * k->kev_used], s);
}

cudaError_t ktime_end(KuramotoCtx *k, cudaStream_t s, int64_t launches) {
  if (!(k->flags & SDE_FLAG_TIME_KERNELS)) return cudaSuccess;
  const cudaError_t err = cudaEventRecord(k->kev[2 * k->kev_used + 1], s);
  ++k->kev_used;
  k->kev_launches += launches;
  return err;
}

bool kuramoto_kernel_stats(KuramotoCtx *k, float *mean_ms, float *total_ms, int64_t *launches) {
  if (k->kev_used == 0) return false;
  if (cudaEventSynchronize(k->kev[2 * k->kev_used - 1]) != cudaSuccess) return false;
  double tot = 0.0;
  for (int64_t i = 0; i < k->kev_used; ++i) {
    float ms = 0.0f;
    if (cudaEventElapsedTime(&ms, k->kev[2 * i], k->kev[2 * i + 1]) != cudaSuccess) return false;
    tot += ms;
  }
  if (total_ms) *total_ms = (float)tot;
  if (k->kev_launches == 0) return false;
  if (mean_ms) *mean_ms = (float)(tot / (double)k->kev_launches);
  if (launches) *launches = k->kev_launches;
  return true;
}

void kuramoto_set_wait_limit(KuramotoCtx *k, uint64_t ns) {
  if (k) k->wait_ns = ns;
}

void kuramoto_destroy(KuramotoCtx *k) {
  if (!k) return;
  cudaDeviceSynchronize();
  for (cudaEvent_t e : k->kev) cudaEventDestroy(e);
  cudaFree(k->theta);
  cudaFree(k->theta_t);
  cudaFree(k->g1);
  cudaFree(k->pair_sc);
  cudaFree(k->r_scratch);
  cudaFree(k->mfg_partials);
  cudaFree(k->mfg_tot);
  cudaFree(k->mfg_count);
  kuramoto_general_free(k);
  delete k;
}

sde_status kuramoto_run(KuramotoCtx *k, const sde_run_desc *r, cudaStream_t s, cudaEvent_t ev0,
                        cudaEvent_t ev1, sde_obs_row *obs_in, sde_obs_row **obs, int64_t *max_rows,
                        int64_t *rows) {
  SDE_CHECK_ARG(r->phi_in_dev && r->phi_out_dev && r->omega_dev,
                "Kuramoto run needs phi_in, phi_out and omega");
  const int64_t L = r->n_end - r->n_begin;
  const int64_t n_rows = k->M > 0 ? (L + k->M - 1) / k->M + 1 : 0;
  // Observable and sample buffers.
  if (n_rows > *max_rows) {
    cudaFree(obs_in);
    *obs = nullptr;
    *max_rows = 0;
    SDE_CUDA_TRY(device_alloc((void **)obs, sizeof(sde_obs_row) * n_rows));
    *max_rows = n_rows;
  }
  double *rbuf = r->r_out_dev;
  if (!rbuf && n_rows > 0) {
    if (k->r_scratch_rows < n_rows) {
      cudaFree(k->r_scratch);
      k->r_scratch = nullptr;
      k->r_scratch_rows = 0;
      SDE_CUDA_TRY(device_alloc((void **)&k->r_scratch, sizeof(double) * n_rows * k->R));
      k->r_scratch_rows = n_rows;
    }
    rbuf = k->r_scratch;
  }
  const int64_t NR = k->N * k->R;
  const int cvt_grid = (int)std::min<int64_t>((NR + 255) / 256, 4096);
  kur_to_fixed<<<cvt_grid, 256, 0, s>>>(r->phi_in_dev, k->theta, NR);
  SDE_CUDA_TRY(cudaGetLastError());
  const double inv2pi = 0.15915494309189533577;
  k->kev_used = 0;
  k->kev_launches = 0;
  SDE_CUDA_TRY(cudaEventRecord(ev0, s));
  if (k->model == SDE_KURAMOTO_MEANFIELD && k->cs == 0) {
    sde_status st = run_meanfield_grid(k, r->n_begin, r->n_end, r->omega_dev, rbuf, n_rows, s);
    if (st != SDE_OK) return st;
  } else if (k->model == SDE_KURAMOTO_MEANFIELD) {
    KurArgs a{};
    a.theta_in = k->theta;
    a.theta_out = k->theta;
    a.omega = r->omega_dev;
    a.r_out = rbuf;
    a.N = k->N;
    a.R = k->R;
    a.n_begin = r->n_begin;
    a.n_end = r->n_end;
    a.M = k->M;
    a.wscale = (float)(k->dt * inv2pi);
    a.kc = (float)(k->K / (double)k->N * k->dt * inv2pi);
    a.kh = (float)(0.5 * k->K / (double)k->N * k->dt * inv2pi);
    a.sc = (float)(sqrt(2.0 * k->D * k->dt) * inv2pi);
    a.keys = philox_round_keys(k->seed);
    a.err = k->err;
    a.wait_ns = k->wait_ns;
    SDE_CUDA_TRY(launch_meanfield(a, k->block, k->opt, k->cs, k->mf_async, s));
  } else if (k->model == SDE_KURAMOTO_PAIRWISE && k->pair_cs > 0) {
    PairClusterArgs a{};
    a.theta = k->theta;
    a.omega = r->omega_dev;
    a.r_out = rbuf;
    a.N = k->N;
    a.R = k->R;
    a.n_begin = r->n_begin;
    a.n_end = r->n_end;
    a.M = k->M;
    a.chunk = (int32_t)pair_cluster_chunk(k->N, k->pair_cs);
    a.npairs = (int32_t)pair_cluster_pairs(k->N);
    a.wscale = (float)(k->dt * inv2pi);
    a.kc = (float)(k->K / (double)k->N * k->dt * inv2pi);
    a.kh = (float)(0.5 * k->K / (double)k->N * k->dt * inv2pi);
    a.sc_noise = (float)(sqrt(2.0 * k->D * k->dt) * inv2pi);
    a.keys = philox_round_keys(k->seed);
    a.err = k->err;
    a.wait_ns = k->wait_ns;
    const bool euler = (k->flags & SDE_FLAG_EULER) != 0;
    SDE_CUDA_TRY(ktime_begin(k, s));
    SDE_CUDA_TRY(launch_pair_cluster(a, k->pair_cs, euler, s));
    SDE_CUDA_TRY(ktime_end(k, s, (euler ? 1 : 2) * (r->n_end - r->n_begin)));  // per stage
  } else if (k->model == SDE_KURAMOTO_PAIRWISE) {
    KurPairArgs a{};
    a.theta = k->theta;
    a.theta_t = k->theta_t;
    a.g1 = k->g1;
    a.sc = k->pair_sc;
    a.sc_t = k->pair_sc + NR;
    a.omega = r->omega_dev;
    a.N = k->N;
    a.wscale = (float)(k->dt * inv2pi);
    a.kc = (float)(k->K / (double)k->N * k->dt * inv2pi);
    a.kh = (float)(0.5 * k->K / (double)k->N * k->dt * inv2pi);
    a.sc_noise = (float)(sqrt(2.0 * k->D * k->dt) * inv2pi);
    a.seed = k->seed;
    const PairShape shape = pair_shape(k->N, k->R, k->sm_count);
    if (r->n_end > r->n_begin) {
      kur_sincos_kernel<<<cvt_grid, 256, 0, s>>>(k->theta, k->pair_sc, k->N, NR);
      SDE_CUDA_TRY(cudaGetLastError());
    }
    int64_t sample = 0;
    const bool euler = (k->flags & SDE_FLAG_EULER) != 0;
    const unsigned adv_grid = (unsigned)std::min<int64_t>((NR + 255) / 256, (int64_t)k->sm_count * 8);
    for (int64_t n = r->n_begin; n < r->n_end; ++n) {
      if (k->M > 0 && (n - r->n_begin) % k->M == 0) {
        kur_order_kernel<<<(unsigned)k->R, 256, 0, s>>>(k->theta, k->N, k->R, rbuf + sample * k->R);
        ++sample;
      }
      a.n = n;
      if (euler) {
        // PROG2: UpdateRHS, then AdvanceSystem
        SDE_CUDA_TRY(ktime_begin(k, s));
        SDE_CUDA_TRY(launch_pairwise<2>(a, k->R, shape, s));
        SDE_CUDA_TRY(ktime_end(k, s));
        kur_advance_euler_kernel<<<adv_grid, 256, 0, s>>>(a, k->R);
        continue;
      }
      SDE_CUDA_TRY(ktime_begin(k, s));
      SDE_CUDA_TRY(launch_pairwise<0>(a, k->R, shape, s));
      SDE_CUDA_TRY(ktime_end(k, s));
      SDE_CUDA_TRY(ktime_begin(k, s));
      SDE_CUDA_TRY(launch_pairwise<1>(a, k->R, shape, s));
      SDE_CUDA_TRY(ktime_end(k, s));
    }
    SDE_CUDA_TRY(cudaGetLastError());
    if (k->M > 0) kur_order_kernel<<<(unsigned)k->R, 256, 0, s>>>(k->theta, k->N, k->R, rbuf + sample * k->R);
  } else {
    sde_status st = kuramoto_general_run(k, r, s, rbuf);
    if (st != SDE_OK) return st;
  }
  SDE_CUDA_TRY(cudaGetLastError());
  SDE_CUDA_TRY(cudaEventRecord(ev1, s));
  kur_from_fixed<<<cvt_grid, 256, 0, s>>>(k->theta, r->phi_out_dev, NR);
  SDE_CUDA_TRY(cudaGetLastError());
  if (n_rows > 0) {
    kur_obs_kernel<<<(unsigned)((n_rows + 7) / 8), 256, 0, s>>>(rbuf, n_rows, k->R, r->n_begin, r->n_end,
                                                                 k->M, k->dt, *obs);
    SDE_CUDA_TRY(cudaGetLastError());
  }
  *rows = n_rows;
  return SDE_OK;
}

sde_status kuramoto_coupling(KuramotoCtx *k, const float *phi_dev, float *out_dev, cudaStream_t s) {
  SDE_CHECK_ARG(phi_dev != nullptr && out_dev != nullptr, "phi and out must be non-NULL");
  const int64_t NR = k->N * k->R;
  const int cvt_grid = (int)std::min<int64_t>((NR + 255) / 256, 4096);
  kur_to_fixed<<<cvt_grid, 256, 0, s>>>(phi_dev, k->theta, NR);
  SDE_CUDA_TRY(cudaGetLastError());
  if (k->model == SDE_KURAMOTO_GENERAL || k->model == SDE_KURAMOTO_GENERAL_FP32)
    return kuramoto_general_coupling(k, out_dev, s);
  const dim3 grid((unsigned)((k->N + 255) / 256), (unsigned)k->R);
  kur_coupling_uniform_kernel<<<grid, 256, 0, s>>>(k->theta, out_dev, k->N, (float)(k->K / (double)k->N));
  SDE_CUDA_TRY(cudaGetLastError());
  return SDE_OK;
}

cudaError_t kur_order_launch(const uint32_t *theta, int64_t N, int64_t R, double *r_out, cudaStream_t s) {
  kur_order_kernel<<<(unsigned)R, 256, 0, s>>>(theta, N, R, r_out);
  return cudaGetLastError();
}

}  // namespace sde
