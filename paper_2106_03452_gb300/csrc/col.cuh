// A column of a swizzled TMA box (see bxl) as one thread of its FFT group sees
// it: its own elements t + T j, and the group FFT's exchange in place.
//
// An exchange index is k1 T + (t ^ k1 mod T), and the swizzle XORs a row's low
// bits into its address as well, so the address of exchange step k1 is the
// thread's own (row t) XOR a constant, plus a constant: one logic operation an
// access where the general index arithmetic takes four or five. The column
// passes issue some 100 such accesses per transform next to 400 FP32
// operations, and are bound by issue slots as much as by HBM.
#pragma once

#include "dpsr_dev.cuh"
#include "tma.cuh"

namespace dpsr {

// Alignment of the boxes: the bits that the XOR touches (T rows) must be the
// box offset's own.
template <int L>
constexpr int box_align() {
  return Shape<L>::T * tile_cols(L) * 8 > 1024 ? Shape<L>::T * tile_cols(L) * 8 : 1024;
}

template <int L, bool FAST = (Shape<L>::T >= 8)>
struct Col {  // T a multiple of the swizzle's 8 rows: rows t + T j share row t's pattern
  static constexpr int T = Shape<L>::T, RB = tile_cols(L) * 8;  // row bytes
  uint32_t p, px;  // row t; exchange row t T + t
  __device__ __forceinline__ Col(const float2* box, int t, int c) {
    p = smem_u32(box) + (uint32_t)bxl<L>(t, c) * 8u;
    px = p + (uint32_t)t * (T * RB);
  }
  // XOR of rows s and s ^ k (k < T): the row's offset and its swizzled chunk
  static __device__ __forceinline__ constexpr uint32_t flip(int k) {
    return (uint32_t)(k * RB | (RB == 128 ? (k & 7) << 4 : ((k >> 1) & 3) << 4));
  }
  static __device__ __forceinline__ float2 ld(uint32_t a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
  }
  static __device__ __forceinline__ void st(uint32_t a, float2 v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
  }
  __device__ __forceinline__ float2 get(int j) const { return ld(p + j * (T * RB)); }
  __device__ __forceinline__ void put(int j, float2 v) const { st(p + j * (T * RB), v); }
  __device__ __forceinline__ void xput(int k1, float2 v) const { st((p ^ flip(k1 % T)) + k1 * (T * RB), v); }
  __device__ __forceinline__ float2 xget(int m, int n2) const { return ld((px ^ flip(n2)) + m * (T * T * RB)); }
};

template <int L>
struct Col<L, false> {
  static constexpr int T = Shape<L>::T;
  float2* b;
  int t, c;
  __device__ __forceinline__ Col(float2* box, int t_, int c_) : b(box), t(t_), c(c_) {}
  __device__ __forceinline__ float2 get(int j) const { return b[bxl<L>(t + T * j, c)]; }
  __device__ __forceinline__ void put(int j, float2 v) const { b[bxl<L>(t + T * j, c)] = v; }
  __device__ __forceinline__ void xput(int k1, float2 v) const { b[bxl<L>(k1 * T + (t ^ (k1 % T)), c)] = v; }
  __device__ __forceinline__ float2 xget(int m, int n2) const { return b[bxl<L>((t + T * m) * T + (n2 ^ t), c)]; }
};

// The group FFT of fft_r with its exchange in a box column.
template <int L, int DIR, bool IL>
__device__ __forceinline__ void fft_c(float2 (&v)[Shape<L>::R1], const Col<L>& col, const TwTab<L>& tw) {
  constexpr int R1 = Shape<L>::R1, T = Shape<L>::T, M = R1 / T;
  if constexpr (T == 1) {
    Dft<L, DIR>::run(v);
  } else {
    Dft<R1, DIR>::run(v);
#pragma unroll
    for (int k1 = 1; k1 < R1; ++k1) {
      float2 w = tw(k1);
      if (DIR > 0) w.y = -w.y;
      v[k1] = cmul(v[k1], w);
    }
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) col.xput(k1, v[k1]);
    group_sync<T, IL>();
#pragma unroll
    for (int m = 0; m < M; ++m) {
      float2 u[T];
#pragma unroll
      for (int n2 = 0; n2 < T; ++n2) u[n2] = col.xget(m, n2);
      Dft<T, DIR>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < T; ++k2) v[m + M * k2] = u[k2];
    }
    group_sync<T, IL>();
  }
}

// The same for a 512-point column of an 8-column tile by 32 threads of 16 values
// instead of 16 of 32: half the registers a thread, twice the warps on an SM, which
// the column passes have the shared memory for (three CTAs either way). x pass:
// forward 487 -> 431 us, backward 567 -> 434 (168 -> 80 registers); y passes:
// forward 398 -> 382, inverse 257 -> 234, backward 211 either way. (Not below: at r =
// 128 and 256 an SM has 20 and 24 warps already, and the shuffles cost more than
// the rest gives: forward x pass of a training batch 71 -> 79 us, of r = 256 52 -> 60.)
// 512 = 16 x 2 x 16:
// radix 16 in registers, the exchange, then each 32-point DFT by a pair of lanes,
// which halve it by a decimation in frequency (lane b takes the outputs 2 q + b)
// and trade eight values by shuffles. Two adjacent columns take two warps: thread
// t of a column is lane (t >> 4) 16 + (t & 7) 2 + column of warp (t >> 3) & 1, so
// that a half-warp reaches 8 rows of two columns, all 32 banks, and the two lanes
// of a pair (t, t ^ 16) share a warp.
struct Wide512 {
  static constexpr int R1 = 16, T = 32;
  static constexpr int TWP = 33, TWN = 16 * TWP;  // twiddle W^(t k1) at k1 TWP + t
  static __device__ __forceinline__ int group(int tid) { return 2 * (tid >> 6) + (tid & 1); }
  static __device__ __forceinline__ int lane(int tid) {
    return ((tid & 16) | ((tid >> 2) & 8)) + ((tid >> 1) & 7);
  }
  // the two warps of two columns: all 64 threads
  static __device__ __forceinline__ void sync() {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (int)(threadIdx.x >> 6)) : "memory");
  }
};

struct ColWide {
  static constexpr int RB = 64;
  uint32_t p, px;  // row t; exchange row (t & 15) 32 + (t & 16) / 2 + (t & 7)
  __device__ __forceinline__ ColWide(const float2* box, int t, int c) {
    p = smem_u32(box) + (uint32_t)bxl<512>(t, c) * 8u;
    px = smem_u32(box) + (uint32_t)bxl<512>((t & 15) * 32 + ((t & 16) >> 1) + (t & 7), c) * 8u;
  }
  __device__ __forceinline__ float2 get(int j) const { return Col<512>::ld(p + j * (32 * RB)); }
  __device__ __forceinline__ void put(int j, float2 v) const { Col<512>::st(p + j * (32 * RB), v); }
  // exchange value (k1, n) at row k1 32 + (n ^ (k1 & 7))
  __device__ __forceinline__ void xput(int k1, float2 v) const {
    Col<512>::st((p ^ Col<512>::flip(k1 & 7)) + k1 * (32 * RB), v);
  }
  // value (t & 15, 8 (t >> 4) + i + 16 h)
  __device__ __forceinline__ float2 xget(int i, int h) const {
    return Col<512>::ld((px ^ Col<512>::flip(i)) + h * (16 * RB));
  }
};

template <int DIR>
__device__ __forceinline__ void fft_wide(float2 (&v)[16], const ColWide& col, const float2* tw, int t) {
  Dft<16, DIR>::run(v);
#pragma unroll
  for (int k1 = 1; k1 < 16; ++k1) {
    float2 w = tw[k1 * Wide512::TWP + t];
    if (DIR > 0) w.y = -w.y;
    v[k1] = cmul(v[k1], w);
  }
  Wide512::sync();  // both warps have read the column
#pragma unroll
  for (int k1 = 0; k1 < 16; ++k1) col.xput(k1, v[k1]);
  Wide512::sync();
  const bool b = t >= 16;
  sfor<0, 8>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    const float2 y0 = col.xget(i, 0), y1 = col.xget(i, 1);
    const float2 s = cadd(y0, y1);
    float2 d = twc32<i, DIR>(csub(y0, y1));  // W32^i; the other lane's n = 8 + i takes W4 more
    if (b) d = DIR < 0 ? make_float2(d.y, -d.x) : make_float2(-d.y, d.x);
    const float2 give = b ? s : d, keep = b ? d : s;
    const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, 16), __shfl_xor_sync(0xffffffffu, give.y, 16));
    v[i] = b ? got : keep;
    v[8 + i] = b ? keep : got;
  });
  Dft<16, DIR>::run(v);
  Wide512::sync();  // both warps have read the exchange
}

// How a column of a tile is transformed, by size: its threads, their share of the
// values (t + T j), its shared-memory view, and the place of entry i of Solve::tw.
template <int L>
struct ColFft {
  static constexpr bool WIDE = false;
  static constexpr int R1 = Shape<L>::R1, T = Shape<L>::T, TWN = L;
  static constexpr bool IL = T == 16;  // interleaved groups: conflict-free column accesses
  using LN = Lanes<T, IL>;
  using CL = Col<L>;
  static __device__ __forceinline__ int tw_at(int i) { return i; }
  template <int DIR>
  static __device__ __forceinline__ void run(float2 (&v)[R1], const CL& c, const float2* tw, int t) {
    fft_c<L, DIR, IL>(v, c, TwTab<L>{tw, t});
  }
  static __device__ __forceinline__ void sync() { group_sync<T, IL>(); }
};
template <>
struct ColFft<512> : Wide512 {
  static constexpr bool WIDE = true;
  using LN = Wide512;
  using CL = ColWide;
  static __device__ __forceinline__ int tw_at(int i) { return (i & 15) * TWP + (i >> 4); }  // W^(t k1) at 16 t + k1
  template <int DIR>
  static __device__ __forceinline__ void run(float2 (&v)[R1], const CL& c, const float2* tw, int t) {
    fft_wide<DIR>(v, c, tw, t);
  }
};

}  // namespace dpsr
