// Scalar finalisation of a solve: the passes leave block sums and the pass that
// needs the scalars adds them up in a fixed order (from r = 256 on the forward's go
// to FP64 accumulators instead, whose additions are exact); the backward z pass ends
// with its last block doing so.
//
// The sums run in float-float arithmetic: a value is an FP32 pair (hi, lo)
// whose exact sum carries it, combined with error-free transformations
// (Knuth's TwoSum, Dekker's Fast2Sum), about 44 significant bits. This
// GPU's FP64 pipe issues roughly one warp instruction per ~18 SM cycles, so
// FP64 shuffle trees and long FP64 reductions on the critical path cost
// several microseconds; FP32 pairs do the same job on the FP32 pipe, in a
// fixed order (deterministic run to run). Only the few scalar formulas of
// Eq. 4, once per solve in one thread, stay in FP64.
#pragma once

#include "dpsr_dev.cuh"

namespace dpsr {

struct FF {
  float hi, lo;
};

// a + b = s + e exactly (TwoSum; no ordering condition on a and b).
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  const float e = (a - (s - bb)) + (b - bb);
  return {s, e};
}

__device__ __forceinline__ FF ff_add(FF x, FF y) {
  const FF s = ff_two_sum(x.hi, y.hi);
  const float e = s.lo + (x.lo + y.lo);
  const float hi = s.hi + e;  // Fast2Sum: |s.hi| >= |e|
  return {hi, e - (hi - s.hi)};
}

__device__ __forceinline__ FF ff_add(FF x, float y) {
  const FF s = ff_two_sum(x.hi, y);
  const float e = s.lo + x.lo;
  const float hi = s.hi + e;
  return {hi, e - (hi - s.hi)};
}

__device__ __forceinline__ FF ff_shfl_xor(FF x, int m) {
  return {__shfl_xor_sync(0xffffffffu, x.hi, m), __shfl_xor_sync(0xffffffffu, x.lo, m)};
}

__device__ __forceinline__ double ff_to_double(FF x) { return (double)x.hi + (double)x.lo; }

// Block sums of two per-thread values in a fixed order (lane butterfly, then
// the warps in index order); the result is valid in thread 0. Every thread
// of the block calls it (it synchronises the block).
template <int NT>
__device__ __forceinline__ void block_sum_ff(FF& a, FF& b) {
  static_assert(NT % 32 == 0, "whole warps");
  __shared__ FF red[2][NT / 32];
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    a = ff_add(a, ff_shfl_xor(a, m));
    b = ff_add(b, ff_shfl_xor(b, m));
  }
  const int tid = threadIdx.x;
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = a;
    red[1][tid >> 5] = b;
  }
  __syncthreads();
  if (tid == 0) {
    a = red[0][0];
    b = red[1][0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) {
      a = ff_add(a, red[0][w]);
      b = ff_add(b, red[1][w]);
    }
  }
}

// Sums in no fixed order with one result: lane 0's v in pieces, a lane of the warp
// and a bin for each: the bits of v from a bin's unit 2^(90 - 40 b) up to the next
// bin's. Less than 2^40 units each, so that 2^13 pieces add up exactly in FP64, in
// any order. Float pairs are multiples of 2^-149 below 2^130: seven bins hold all of
// v. A value that is not finite goes to bin 0 as it is. `slot`: the first bin, the
// others two doubles apart. (The inverse y pass at r = 512: 240 us with plain
// additions, 242 so; 252 with the pieces taken off one after the other.)
__device__ __forceinline__ void add_exact(double* slot, double v, int lane) {
  v = __shfl_sync(0xffffffffu, v, 0);
  auto above = [v](int unit) {  // v without the bits below 2^unit
    const long long bits = __double_as_longlong(v);
    const int keep = (int)((bits >> 52) & 0x7ff) - 1023 - unit;  // of the 52 behind the leading one
    return keep < 0 ? 0.0 : (keep >= 52 ? v : __longlong_as_double(bits & (-1ll << (52 - keep))));
  };
  const bool finite = isfinite(v);
  if (lane >= kMuBins || (!finite && lane > 0)) return;
  const int unit = 90 - 40 * lane;
  const double p = finite ? above(unit) - (lane > 0 ? above(unit + 40) : 0.0) : v;
  if (p != 0.0) atomicAdd(slot + 2 * lane, p);
}

// A warp: the sums of the bins, in lane 0 (copies, then bins from the smallest, in
// that order).
__device__ __forceinline__ double2 sum_bins(const double2* slots, int lane) {
  const double2 own = lane < kMuCopies * kMuBins ? __ldcg(slots + lane) : make_double2(0.0, 0.0);
  double2 v = own;
#pragma unroll
  for (int c = 1; c < kMuCopies; ++c) {
    v.x += __shfl_down_sync(0xffffffffu, own.x, c * kMuBins);
    v.y += __shfl_down_sync(0xffffffffu, own.y, c * kMuBins);
  }
  double2 s = make_double2(0.0, 0.0);
#pragma unroll
  for (int b = kMuBins - 1; b >= 0; --b) {
    s.x += __shfl_sync(0xffffffffu, v.x, b);
    s.y += __shfl_sync(0xffffffffu, v.y, b);
  }
  return s;
}

// The scalars of Eq. 4 from the forward's reduced sums:
// mu = <W, chi'> / N, chi'(0) = sum_k chi~ / n, s = chi'(0) - mu.
struct FwdScalars {
  double mu, s, alpha;
  float a_chi, b_chi;
  bool bad;
};
__device__ __forceinline__ FwdScalars fwd_scalars(const Solve& S, double a, double b) {
  FwdScalars q;
  // r^3 is a power of two: its reciprocal is exact in FP32
  const double inv_n = (double)__frcp_rn((float)S.r * (float)S.r * (float)S.r);
  q.mu = a * inv_n * S.inv_N;
  const double chi0 = b * inv_n;
  q.s = chi0 - q.mu;
  q.bad = !isfinite(q.s) || !(fabs(q.s) > 1e-7 * (fabs(chi0) + fabs(q.mu)) + 1e-37);
  q.alpha = q.bad ? 0.0 : (double)kM / fabs(q.s);
  q.a_chi = (float)(q.alpha * inv_n);
  q.b_chi = (float)(-q.alpha * q.mu);
  return q;
}

// Those of its adjoint: a = sum dchi, b = sum dchi * chi = alpha * sum dchi (chi' - mu);
// with alpha = m / |s|: D = b / alpha = b |s| / m and
// s_bar = -m sign(s) D / s^2 = -sign(s) D alpha^2 / m.
struct BwdScalars {
  double D, s_bar, mu_bar;
  float g_a, g_s, g_w;
};
__device__ __forceinline__ BwdScalars bwd_scalars(const Solve& S, double a, double b) {
  BwdScalars q;
  const double inv_n = (double)__frcp_rn((float)S.r * (float)S.r * (float)S.r);
  const double alpha = S.sc->alpha, s = S.sc->s;
  q.D = alpha > 0 ? b * fabs(s) * (1.0 / (double)kM) : 0.0;
  q.s_bar = -(s > 0 ? 1.0 : -1.0) * q.D * alpha * alpha * (1.0 / (double)kM);
  q.mu_bar = -alpha * a - q.s_bar;
  q.g_a = (float)(alpha * inv_n);
  q.g_s = (float)(q.s_bar * inv_n);
  q.g_w = (float)(q.mu_bar * inv_n * S.inv_N);
  return q;
}

// Thread 0: the scalars from the reduced sums.
__device__ inline void finalize_scalars(const Solve& S, double a, double b, bool bwd) {
  Scalars* sc = S.sc;
  if (!bwd) {
    const FwdScalars q = fwd_scalars(S, a, b);
    sc->acc_mu = a;
    sc->acc_s0 = b;
    sc->mu = q.mu;
    sc->s = q.s;
    sc->alpha = q.alpha;
    sc->a_chi = q.a_chi;
    sc->b_chi = q.b_chi;
    if (q.bad) atomicOr(S.status, kStDegenerate);
  } else {
    const BwdScalars q = bwd_scalars(S, a, b);
    sc->S = a;
    sc->D = q.D;
    sc->s_bar = q.s_bar;
    sc->mu_bar = q.mu_bar;
    sc->g_a = q.g_a;
    sc->g_s = q.g_s;
    sc->g_w = q.g_w;
    sc->c_mu = q.g_w;
  }
}

// The `n` block partials of S.part summed by every thread of a block (each a
// strided subset, loads in flight together, then the block tree: a fixed
// order); the sums are valid in thread 0.
template <int NT>
__device__ __forceinline__ void sum_partials(const Solve& S, int n, FF& x, FF& y) {
  x = y = FF{0.f, 0.f};
#pragma unroll 8
  for (int i = threadIdx.x; i < n; i += NT) {
    const float4 p = __ldcg(S.part + i);
    x = ff_add(x, FF{p.x, p.y});
    y = ff_add(y, FF{p.z, p.w});
  }
  block_sum_ff<NT>(x, y);
}

// Every thread of the block calls this after the block sums (a, b) are in
// thread 0 (block_sum_ff). Thread 0 publishes them as the block's partial
// S.part[bid]; the last of the `nblocks` blocks of the solve to arrive sums
// all partials (each thread a strided subset, loads in flight together, then
// the block tree: a fixed order) and writes the scalars. Only thread 0
// fences, on both sides of its ticket; the block barrier orders the other
// threads' accesses around it (the pattern of a cooperative grid barrier).
template <int NT>
__device__ inline void last_block_finalize(const Solve& S, int ticket, int nblocks, int bid, FF a,
                                           FF b, bool bwd) {
  __shared__ unsigned last;
  const int tid = threadIdx.x;
  if (tid == 0) {
    S.part[bid] = make_float4(a.hi, a.lo, b.hi, b.lo);
    __threadfence();  // this block's partials before its arrival
    last = atomicAdd(&S.sc->ticket[ticket], 1u) == (unsigned)nblocks - 1u ? 1u : 0u;
    if (last) __threadfence();  // every arrival before the reads below
  }
  __syncthreads();
  if (!last) return;
  FF x, y;
  sum_partials<NT>(S, nblocks, x, y);
  if (tid == 0) {
    finalize_scalars(S, ff_to_double(x), ff_to_double(y), bwd);
    S.sc->ticket[ticket] = 0;
    if (bwd) S.sc->bparts = 0;
  }
}

}  // namespace dpsr
