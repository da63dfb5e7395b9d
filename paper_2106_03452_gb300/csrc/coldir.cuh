// Column transforms straight from global memory (r >= 64): the values that a
// thread transforms come by coalesced loads and leave by coalesced stores, and
// shared memory carries only the exchange between the two FFT stages.
//
// A block takes C consecutive kz columns: thread (t, c) of 128 holds elements
// t + T j of column c, so that C lanes read one contiguous run of a row (128
// bytes up to r = 128, 64 above). Moving tiles by TMA instead costs each value
// a shared-memory write by the copy and a read on the way in, the same on the
// way out, and two more where a second field waits: over a third of the
// passes' shared-memory traffic, their busiest unit, for no reuse.
#pragma once

#include "dpsr_dev.cuh"

namespace dpsr {

template <int L>
struct ColDir {
  static constexpr int R1 = Shape<L>::R1, T = Shape<L>::T;
  static constexpr int NT = 128, C = NT / T;       // threads; columns (8 or 16)
  // Exchange row k1 T + n, columns contiguous: a warp writes 32 consecutive
  // values and reads C-value runs of rows T apart. With 8 columns two such
  // runs of a half-warp would share banks: each k1 is padded by half a line.
  static constexpr int KS = T * C + (C == 8 ? 8 : 0);
  static constexpr int XCH = R1 * KS;              // float2 of one exchange buffer
  // Two buffers, used in turn, save the barrier that keeps a transform's
  // writes behind the last one's reads; at r = 512 they would cost a block per SM.
  static constexpr int NBUF = L >= 512 ? 1 : 2;
};

// Group FFT of the block's columns in registers (distribution as fft_r). All
// threads of the block call it; `turn` counts the calls.
template <int L, int DIR>
__device__ __forceinline__ void fft_d(float2 (&v)[Shape<L>::R1], int t, int c, const TwTab<L>& tw, float2* xch,
                                      int turn) {
  using P = ColDir<L>;
  constexpr int R1 = P::R1, T = P::T, M = R1 / T;
  Dft<R1, DIR>::run(v);
#pragma unroll
  for (int k1 = 1; k1 < R1; ++k1) {
    float2 w = tw(k1);
    if (DIR > 0) w.y = -w.y;
    v[k1] = cmul(v[k1], w);
  }
  float2* x = xch + (P::NBUF == 2 ? (turn & 1) * P::XCH : 0);
  if (P::NBUF == 1 && turn > 0) __syncthreads();  // the last transform's reads
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) x[k1 * P::KS + t * P::C + c] = v[k1];
  __syncthreads();
#pragma unroll
  for (int m = 0; m < M; ++m) {
    float2 u[T];
#pragma unroll
    for (int n2 = 0; n2 < T; ++n2) u[n2] = x[(t + T * m) * P::KS + n2 * P::C + c];
    Dft<T, DIR>::run(u);
#pragma unroll
    for (int k2 = 0; k2 < T; ++k2) v[m + M * k2] = u[k2];
  }
}

// A spectral value that is read once: not kept in L1.
__device__ __forceinline__ float2 ld_once(const float2* p) {
  float2 v;
  asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
  return v;
}

}  // namespace dpsr
