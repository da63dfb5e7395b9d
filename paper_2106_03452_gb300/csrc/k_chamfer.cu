// Bi-directional L2 Chamfer distance with exact nearest neighbours from a
// shallow box tree, for callers that bring a workspace (dpsr_chamfer_tree).
//
// Per set: a counting sort along a Morton curve of 2^B slabs per axis, leaves
// of 32 consecutive points with their boxes, and boxes over 32 leaves each. A
// query only scans the leaves whose box is not farther than its best point so
// far. Box distances are computed with the point distance's operations in the
// same order, and rounding is monotonic, so a pruned leaf never holds a point
// that the brute force search would have returned: indices (ties to the lowest)
// and distances are bit for bit its.
//
// The slabs have equal widths over the range of a sample of 512 points, unless
// that leaves the cells crowded (a far outlier in the sample, a cluster in a
// large box): a query would open nearly every leaf of a cell that holds most
// points in no order. The sort then starts again with slabs that hold equally
// many points of the sample, narrow wherever the points are dense. 20 000 x
// 20 000, with equal widths over the whole set's box before and now (brute force
// 618 us): a surface 56.5 and 56.4 us, the same with one point 10^6 away 1 074 and
// 60, a cluster in a box a thousand times its size 850 and 69, scales from 10^-4
// to 10^3 1 059 and 79, all points of a set equal 1 407 and 129.
//
// Bound: 2 na nb distances by brute force (577 us for 20 000 x 20 000, one
// thread per query and 79 blocks on 152 SMs). Here a query on points of a
// surface scans four leaves, and what is left is the latency of the sort's
// phases and of the descent. A cell of c points costs its queries c / 32 leaves
// each; where coordinates differ a cell of the second kind holds about a
// slab's points (n / 16) at most, and in that worst case the scans cost half
// the brute force.
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "dpsr.h"
#include "dpsr_dev.cuh"
#include "finalize.cuh"
#include "launch.h"

namespace dpsr {

constexpr int kCs = 8;         // CTAs (one cluster) that sort one set
constexpr int kSortNT = 512;   // threads of each
constexpr int kLeaf = 32;
constexpr int kQNT = 128;      // threads of a query block
constexpr int kQW = 4;         // consecutive sorted queries of a warp
constexpr int kQB = kQW * kQNT / 32;  // and of a block

// Slabs per axis 2^B: 16 up to 32 768 points (about 13 a cell on a surface),
// 32 above, where 16 would leave several leaves to a cell.
__host__ __device__ constexpr int cell_bits(int64_t n) { return n <= 32768 ? 4 : 5; }

struct NnSet {
  const float* p;     // n x 3
  int n, nl1, nl2;    // points, leaves, boxes of 32 leaves
  float4* sorted;     // nl1 * 32: x, y, z, original index (padding: NaN)
  float4* box1;       // nl1 x (lo, hi); lo.w: the lowest index inside
  float4* box2;       // nl2 x (lo, hi)
  int* start;         // first sorted position of each cell
  float* slab;        // 3 x 32: lower bounds of an axis' slabs 1 .. 2^B - 1
};
struct NnPair {
  NnSet s[2];
  float* grad;        // na x 3
  double* loss;
  float* loss32;
  float4* part;       // partial sums of the query blocks
  unsigned* ticket;
};

__device__ __forceinline__ unsigned morton3(unsigned x, unsigned y, unsigned z) {
  auto spread = [](unsigned v) {  // bits of v (at most 10) to every third place
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    return (v | (v << 2)) & 0x09249249u;
  };
  return spread(x) | (spread(y) << 1) | (spread(z) << 2);
}

// Slab of a coordinate: the number of bounds that do not exceed it (they
// ascend): first of those between the quarters, which every point is compared
// with, then of the few in its quarter, read together. A NaN is in the first
// slab: the order of the points only decides how tight the boxes are.
template <int BITS>
__device__ __forceinline__ unsigned slab_of(const float* bound, float v) {
  constexpr unsigned Q = 1u << (BITS - 2);
  const unsigned k = (v >= bound[Q - 1]) + (v >= bound[2 * Q - 1]) + (v >= bound[3 * Q - 1]);
  unsigned n = k * Q;
#pragma unroll
  for (unsigned j = 0; j < Q; j += 4) {
    const float4 b = *reinterpret_cast<const float4*>(bound + k * Q + j);
    n += (v >= b.x) + (v >= b.y) + (v >= b.z) + (j + 4 < Q ? v >= b.w : 0);
  }
  return n;
}
template <int BITS>
__device__ __forceinline__ unsigned cell_of(const float (&bound)[3][32], float x, float y, float z) {
  return morton3(slab_of<BITS>(bound[0], x), slab_of<BITS>(bound[1], y), slab_of<BITS>(bound[2], z));
}

__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, d));
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, d));
  return v;
}

// Box of the 32 points (or boxes) of a warp's lanes; `low` (their lowest index) goes along.
__device__ __forceinline__ void warp_box(float3 lo, float3 hi, int low, float4* out, int lane) {
  lo.x = warp_min(lo.x);
  lo.y = warp_min(lo.y);
  lo.z = warp_min(lo.z);
  hi.x = warp_max(hi.x);
  hi.y = warp_max(hi.y);
  hi.z = warp_max(hi.z);
  low = __reduce_min_sync(0xffffffffu, low);
  if (lane == 0) {
    out[0] = make_float4(lo.x, lo.y, lo.z, __int_as_float(low));
    out[1] = make_float4(hi.x, hi.y, hi.z, 0.f);
  }
}

// A point of the sample that places the slabs: one from each 512th of the set, at
// a hashed place in it, so that no regularity of the input's order meets the
// step. Every CTA of the cluster takes the same ones.
__device__ __forceinline__ int64_t sample_index(int n) {
  const int64_t i0 = (int64_t)threadIdx.x * n / kSortNT, i1 = (int64_t)(threadIdx.x + 1) * n / kSortNT;
  return i0 + (int64_t)(((uint64_t)(threadIdx.x * 2654435769u) * (uint64_t)(i1 - i0)) >> 32);
}

// Bounds of slabs that hold equally many points of the sample: a bitonic sort
// along each axis, an element a thread (45 steps, the ten that cross warps
// through shared memory), the finite ones split evenly.
__device__ void even_slabs(const float (&p)[3], int bits, float (&bound)[3][32]) {
  __shared__ float sh[2][3][kSortNT];
  const int tid = threadIdx.x;
  float v[3];
  int finite[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    finite[d] = __syncthreads_count(isfinite(p[d]));
    v[d] = isfinite(p[d]) ? p[d] : INFINITY;  // behind the others
  }
  int turn = 0;
#pragma unroll
  for (int k = 2; k <= kSortNT; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const bool low = ((tid & k) == 0) == ((tid & j) == 0);
      if (j >= 32) {
#pragma unroll
        for (int d = 0; d < 3; ++d) sh[turn][d][tid] = v[d];
        __syncthreads();
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float o = j >= 32 ? sh[turn][d][tid ^ j] : __shfl_xor_sync(0xffffffffu, v[d], j);
        v[d] = low ? fminf(v[d], o) : fmaxf(v[d], o);
      }
      if (j >= 32) turn ^= 1;
    }
  }
  __syncthreads();
#pragma unroll
  for (int d = 0; d < 3; ++d) sh[0][d][tid] = v[d];
  __syncthreads();
  if (tid < 32) {
    const int q = tid + 1;  // the last entries stay infinite
#pragma unroll
    for (int d = 0; d < 3; ++d)
      bound[d][tid] = q < (1 << bits) && finite[d] > 0 ? sh[0][d][q * finite[d] >> bits] : INFINITY;
  }
}

// One cluster of 8 CTAs per set sorts it and builds its boxes: the slabs,
// per-CTA histograms in shared memory, exclusive offsets per cell and CTA
// through distributed shared memory (each CTA owns an eighth of the cells),
// scatter, boxes. The phases are separated by cluster barriers, so one launch
// does what would take five; 20 000 points are five per thread. Cluster 0 also
// clears the gradient and the arrival counter of the query kernel.
template <int BITS>
__device__ void nn_sort(const NnSet& S, int* hist, float (&bound)[3][32]) {
  constexpr int NC = 1 << (3 * BITS), SL = NC / kCs, PT = SL / kSortNT;  // cells, per CTA, per thread
  static_assert(PT >= 1, "a cell per thread at least");
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  __shared__ float red[6][kSortNT / 32];
  __shared__ float g[6];  // equal slabs: lower end[3], slabs per unit length[3]
  __shared__ int wsum[kSortNT / 32];
  __shared__ float wsq[kSortNT / 32];
  __shared__ int slice_total;
  __shared__ float slice_sq;
  const int n = S.n, first = rank * kSortNT + tid;
  constexpr int STEP = kCs * kSortNT;
  float p[3];
  {
    const int64_t i = sample_index(n);
#pragma unroll
    for (int d = 0; d < 3; ++d) p[d] = S.p[3 * i + d];
  }
  // its range (upper ends negated: minima throughout)
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float v = warp_min(isfinite(p[k % 3]) ? (k < 3 ? p[k] : -p[k - 3]) : INFINITY);
    if (lane == 0) red[k][w] = v;
  }
  __syncthreads();
  if (w < 3) {
    const float lo = warp_min(lane < kSortNT / 32 ? red[w][lane] : INFINITY);
    const float hi = -warp_min(lane < kSortNT / 32 ? red[w + 3][lane] : INFINITY);
    const float sc = (float)(1 << BITS) / (hi - lo);
    const bool ok = hi > lo && isfinite(sc);
    if (lane == 0) {
      g[w] = isfinite(lo) ? lo : 0.f;
      g[w + 3] = ok ? sc : 0.f;
    }
    bound[w][lane] = ok && lane + 1 < (1 << BITS) ? lo + (float)(lane + 1) * ((hi - lo) / (float)(1 << BITS)) : INFINITY;
  }
  bool even = false;
  // Points off the range, infinite or NaN go to an edge cell: the order of the
  // points only decides how tight the boxes are.
  auto cell = [&](float x, float y, float z) {
    if (even) return cell_of<BITS>(bound, x, y, z);
    auto q = [](float v) { return (unsigned)min(max((int)v, 0), (1 << BITS) - 1); };
    return morton3(q((x - g[0]) * g[3]), q((y - g[1]) * g[4]), q((z - g[2]) * g[5]));
  };
  const int c0 = rank * SL + tid * PT;
  int pos, tot[PT];
  for (;;) {
    for (int i = tid; i < NC; i += kSortNT) hist[i] = 0;
    __syncthreads();
#pragma unroll 4
    for (int64_t i = first; i < n; i += STEP) atomicAdd(&hist[cell(S.p[3 * i], S.p[3 * i + 1], S.p[3 * i + 2])], 1);
    cl.sync();
    // this CTA's cells: counts over the CTAs, their exclusive scan and their squares
    int run = 0;
    float sq = 0.f;
#pragma unroll
    for (int j = 0; j < PT; ++j) {
      tot[j] = 0;
#pragma unroll
      for (int r = 0; r < kCs; ++r) tot[j] += cl.map_shared_rank(hist, r)[c0 + j];
      run += tot[j];
      sq = fmaf((float)tot[j], (float)tot[j], sq);
    }
    int incl = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += v;
      sq += __shfl_xor_sync(0xffffffffu, sq, d);
    }
    if (lane == 31) {
      wsum[w] = incl;
      wsq[w] = sq;
    }
    __syncthreads();
    pos = incl - run;
    int total = 0;
    sq = 0.f;
#pragma unroll
    for (int k = 0; k < kSortNT / 32; ++k) {
      pos += k < w ? wsum[k] : 0;
      total += wsum[k];
      sq += wsq[k];
    }
    if (tid == 0) {
      slice_total = total;
      slice_sq = sq;
    }
    cl.sync();
    if (even) break;
    // Crowded: a point shares its cell with more than four times as many as in a
    // plane across the cells (on a sphere it is a sixth of the plane's). The same
    // sum, and answer, in every CTA.
    sq = 0.f;
#pragma unroll
    for (int r = 0; r < kCs; ++r) sq += *cl.map_shared_rank(&slice_sq, r);
    if (sq <= (float)n * (64.f + (float)n * (4.f / (float)(1 << (2 * BITS))))) break;
    even = true;
    even_slabs(p, BITS, bound);
  }
  if (rank == 0 && tid < 3 * 32) S.slab[tid] = bound[tid >> 5][tid & 31];
  for (int r = 0; r < rank; ++r) pos += *cl.map_shared_rank(&slice_total, r);
  // every CTA's first position of each cell, written back to its histogram
#pragma unroll
  for (int j = 0; j < PT; ++j) {
    S.start[c0 + j] = pos;
#pragma unroll
    for (int r = 0; r < kCs; ++r) {
      int* h = cl.map_shared_rank(hist, r) + c0 + j;
      const int c = *h;
      *h = pos;
      pos += c;
    }
  }
  cl.sync();
#pragma unroll 4
  for (int64_t i = first; i < n; i += STEP) {
    const float x = S.p[3 * i], y = S.p[3 * i + 1], z = S.p[3 * i + 2];
    const int at = atomicAdd(&hist[cell(x, y, z)], 1);
    S.sorted[at] = make_float4(x, y, z, __int_as_float((int)i));
  }
  const float nan = __int_as_float(0x7fffffff);
  for (int64_t i = (int64_t)n + first; i < (int64_t)S.nl1 * kLeaf; i += STEP) S.sorted[i] = make_float4(nan, nan, nan, nan);
  __threadfence();
  cl.sync();
  // boxes: a warp per leaf, then a warp per 32 leaves
  constexpr int NW = STEP / 32;
  for (int l = rank * (kSortNT / 32) + w; l < S.nl1; l += NW) {
    const float4 p = __ldcg(S.sorted + (int64_t)l * kLeaf + lane);
    const bool bad = isnan(p.x) || isnan(p.y) || isnan(p.z);  // never anybody's neighbour
    const float3 v = make_float3(p.x, p.y, p.z);
    const float inf = INFINITY;
    warp_box(bad ? make_float3(inf, inf, inf) : v, bad ? make_float3(-inf, -inf, -inf) : v,
             bad ? INT_MAX : __float_as_int(p.w), S.box1 + 2 * (int64_t)l, lane);
  }
  __threadfence();
  cl.sync();
  for (int l = rank * (kSortNT / 32) + w; l < S.nl2; l += NW) {
    const int64_t own = (int64_t)l * 32 + lane, c = min(own, (int64_t)S.nl1 - 1);
    float4 lo = __ldcg(S.box1 + 2 * c), hi = __ldcg(S.box1 + 2 * c + 1);
    // Of leaves whose points are all equal, and equal to one another's, the one
    // with the lowest index answers for all: the others' boxes are closed.
    // Otherwise each of them is as far as the best point, and is opened.
    const bool one = own < S.nl1 && lo.x == hi.x && lo.y == hi.y && lo.z == hi.z;
    const unsigned ones = __ballot_sync(0xffffffffu, one);
    if (ones & (ones - 1u)) {
      bool closed = false;
      for (unsigned m = ones; m; m &= m - 1u) {
        const int src = __ffs(m) - 1;
        const float x = __shfl_sync(0xffffffffu, lo.x, src), y = __shfl_sync(0xffffffffu, lo.y, src),
                    z = __shfl_sync(0xffffffffu, lo.z, src);
        const int low = __shfl_sync(0xffffffffu, __float_as_int(lo.w), src);
        closed = closed || (one && x == lo.x && y == lo.y && z == lo.z && low < __float_as_int(lo.w));
      }
      if (closed) {
        const float inf = INFINITY;
        lo = make_float4(inf, inf, inf, lo.w);
        hi = make_float4(-inf, -inf, -inf, 0.f);
        S.box1[2 * own] = lo;
        S.box1[2 * own + 1] = hi;
      }
    }
    warp_box(make_float3(lo.x, lo.y, lo.z), make_float3(hi.x, hi.y, hi.z), 0, S.box2 + 2 * (int64_t)l, lane);
  }
}

__global__ void __launch_bounds__(kSortNT) k_nn_sort(const __grid_constant__ NnPair P) {
  extern __shared__ int hist[];
  __shared__ __align__(16) float bound[3][32];
  const int set = blockIdx.x / kCs;
  pdl_trigger();
  pdl_wait();
  if (set == 0) {
    for (int64_t i = blockIdx.x * kSortNT + threadIdx.x; i < (int64_t)P.s[0].n * 3; i += kCs * kSortNT) P.grad[i] = 0.f;
    if (blockIdx.x == 0 && threadIdx.x == 0) *P.ticket = 0u;
  }
  const NnSet& S = P.s[set];
  if (cell_bits(S.n) == 4) nn_sort<4>(S, hist, bound);
  else nn_sort<5>(S, hist, bound);
}

// Squared distance between a query and a box: the operations of the point
// distance below, on the gap between the two along each axis.
__device__ __forceinline__ float box_d2(float4 lo, float4 hi, float4 q) {
  const float dx = fmaxf(fmaxf(lo.x - q.x, q.x - hi.x), 0.f), dy = fmaxf(fmaxf(lo.y - q.y, q.y - hi.y), 0.f),
              dz = fmaxf(fmaxf(lo.z - q.z, q.z - hi.z), 0.f);
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Nearest neighbours, a warp per query: its lanes test 32 boxes, or the 32
// points of a leaf, in one step, and of the boxes in reach the nearest is
// opened first. Both directions in one launch, with the gradient and the loss
// in the same pass. A warp takes four queries next to each other on the curve
// and starts each with the point that the one before found, so that most
// descents open two or three leaves. (Packets of 16 queries that descend
// together, two lanes each, took 75 us for 20 000 x 20 000: the few packets
// that straddle a jump of the curve reach every box.)
__global__ void __launch_bounds__(kQNT) k_nn_query(const __grid_constant__ NnPair P) {
  constexpr unsigned ALL = 0xffffffffu;
  pdl_trigger();
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int nb0 = (P.s[0].n + kQB - 1) / kQB;  // blocks of the first direction
  const int dir = (int)blockIdx.x < nb0 ? 0 : 1;
  const NnSet &Q = P.s[dir], &T = P.s[1 - dir];
  const int64_t first = ((int64_t)blockIdx.x - (dir ? nb0 : 0)) * kQB + (threadIdx.x >> 5) * kQW;
  const float cw = 2.f / (float)Q.n;
  FF sum = {0.f, 0.f};
  int bi = -1;
  float3 bp = make_float3(0.f, 0.f, 0.f);  // the point found last: -1 none
  for (int64_t qi = first; qi < first + kQW && qi < Q.n; ++qi) {
    const float4 q = Q.sorted[qi];
    float best = INFINITY;
    // no point is at a finite distance from a query that is not finite
    const bool live = isfinite(q.x) && isfinite(q.y) && isfinite(q.z);
    if (!live) bi = -1;
    if (live) {
      auto dist = [&](float3 p) {
        const float dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
        return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      };
      auto scan = [&](int leaf) {  // ties to the lowest index
        const float4 p = T.sorted[(int64_t)leaf * kLeaf + lane];
        const float d = dist(make_float3(p.x, p.y, p.z));
        const bool hit = d <= best && d < INFINITY;  // false for a NaN
        if (!__any_sync(ALL, hit)) return;
        const float m = __uint_as_float(__reduce_min_sync(ALL, hit ? __float_as_uint(d) : 0xffffffffu));
        const int id = __float_as_int(p.w);
        const int low = (int)__reduce_min_sync(ALL, hit && d == m ? (unsigned)id : 0xffffffffu);
        if (m < best || low < bi) {
          const int src = __ffs(__ballot_sync(ALL, hit && d == m && id == low)) - 1;
          best = m;
          bi = low;
          bp = make_float3(__shfl_sync(ALL, p.x, src), __shfl_sync(ALL, p.y, src), __shfl_sync(ALL, p.z, src));
        }
      };
      int seed = -1;
      if (bi >= 0) {
        best = dist(bp);
        if (!(best < INFINITY)) bi = -1;
      }
      if (bi < 0) {  // the leaf at the query's own cell
        best = INFINITY;
        // slabs of the query, a lane per bound (those past the last are infinite, as q is not)
        auto slab = [&](int d, float v) { return (unsigned)__popc(__ballot_sync(ALL, v >= T.slab[32 * d + lane])); };
        const unsigned cell = morton3(slab(0, q.x), slab(1, q.y), slab(2, q.z));
        seed = min(T.start[cell] / kLeaf, T.nl1 - 1);
        scan(seed);
      }
      // the lane with the smallest distance among `mask`
      auto nearest = [&](unsigned mask, float d) {
        const unsigned u = (mask >> lane) & 1u ? __float_as_uint(d) : 0xffffffffu;
        return __ffs(__ballot_sync(ALL, u == __reduce_min_sync(ALL, u)) & mask) - 1;
      };
      for (int c2 = 0; c2 < T.nl2; c2 += 32) {
        const int b2 = min(c2 + lane, T.nl2 - 1);
        const float d2 = box_d2(T.box2[2 * (int64_t)b2], T.box2[2 * (int64_t)b2 + 1], q);
        unsigned m2 = __ballot_sync(ALL, c2 + lane < T.nl2 && d2 <= best);
        while (m2) {
          const int j2 = nearest(m2, d2);
          m2 &= ~(1u << j2);
          const int c1 = (c2 + j2) * 32;
          const int b1 = min(c1 + lane, T.nl1 - 1);  // nl1 <= 2^26: no overflow
          const float d1 = box_d2(T.box1[2 * (int64_t)b1], T.box1[2 * (int64_t)b1 + 1], q);
          unsigned m1 = __ballot_sync(ALL, c1 + lane < T.nl1 && c1 + lane != seed && d1 <= best);
          while (m1) {
            const int j1 = nearest(m1, d1);
            m1 &= ~(1u << j1);
            scan(c1 + j1);
            m1 &= __ballot_sync(ALL, d1 <= best);
          }
          m2 &= __ballot_sync(ALL, d2 <= best);
        }
      }
    }
    // loss and its gradient with respect to a: each a is pulled by its
    // neighbour in b, and each b pulls its neighbour in a
    sum = ff_add(sum, bi >= 0 ? best : INFINITY);
    const int id = __float_as_int(q.w);
    if (lane < 3) {
      const float qv = lane == 0 ? q.x : (lane == 1 ? q.y : q.z), bv = lane == 0 ? bp.x : (lane == 1 ? bp.y : bp.z);
      if (dir == 0) atomicAdd(P.grad + 3 * (int64_t)id + lane, bi >= 0 ? cw * (qv - bv) : __int_as_float(0x7fffffff));
      else if (bi >= 0) atomicAdd(P.grad + 3 * (int64_t)bi + lane, cw * (bv - qv));
    }
  }
  // every lane of a warp holds its sum: lane 0's counts
  FF zero = {0.f, 0.f};
  FF sum_a = lane == 0 && dir == 0 ? sum : zero, sum_b = lane == 0 && dir == 1 ? sum : zero;
  block_sum_ff<kQNT>(sum_a, sum_b);
  __shared__ unsigned last;
  if (threadIdx.x == 0) {
    P.part[blockIdx.x] = make_float4(sum_a.hi, sum_a.lo, sum_b.hi, sum_b.lo);
    __threadfence();
    last = atomicAdd(P.ticket, 1u) == gridDim.x - 1u ? 1u : 0u;
    if (last) __threadfence();
  }
  __syncthreads();
  if (!last) return;
  FF x = {0.f, 0.f}, y = {0.f, 0.f};
#pragma unroll 4
  for (unsigned i = threadIdx.x; i < gridDim.x; i += kQNT) {
    const float4 p = __ldcg(P.part + i);
    x = ff_add(x, FF{p.x, p.y});
    y = ff_add(y, FF{p.z, p.w});
  }
  block_sum_ff<kQNT>(x, y);
  if (threadIdx.x == 0) {
    const double v = ff_to_double(x) / (double)P.s[0].n + ff_to_double(y) / (double)P.s[1].n;
    *P.loss = v;
    if (P.loss32) *P.loss32 = (float)v;
  }
}

// The workspace's parts for sets of na and nb points from `base` on (null:
// sizes only); the bytes that they take.
static size_t nn_layout(NnPair& P, int64_t na, int64_t nb, char* base) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* q = base + off;
    off += (bytes + 255) & ~(size_t)255;
    return q;
  };
  int64_t blocks = 0;
  for (int k = 0; k < 2; ++k) {
    NnSet& S = P.s[k];
    const int64_t n = k ? nb : na, nl1 = (n + kLeaf - 1) / kLeaf, nl2 = (nl1 + 31) / 32;
    S.n = (int)n;
    S.nl1 = (int)nl1;
    S.nl2 = (int)nl2;
    S.sorted = (float4*)take(sizeof(float4) * kLeaf * nl1);
    S.box1 = (float4*)take(sizeof(float4) * 2 * nl1);
    S.box2 = (float4*)take(sizeof(float4) * 2 * nl2);
    S.start = (int*)take(sizeof(int) << (3 * cell_bits(n)));
    S.slab = (float*)take(sizeof(float) * 3 * 32);
    blocks += (n + kQB - 1) / kQB;
  }
  P.part = (float4*)take(sizeof(float4) * blocks);
  P.ticket = (unsigned*)take(sizeof(unsigned));
  return off;
}

}  // namespace dpsr

extern "C" {

size_t dpsr_chamfer_ws_bytes(int64_t na, int64_t nb) {
  if (na < 1 || nb < 1 || na > INT32_MAX || nb > INT32_MAX) return 0;
  dpsr::NnPair P = {};
  return dpsr::nn_layout(P, na, nb, nullptr);
}

int dpsr_chamfer_tree(const float* a, int64_t na, const float* b, int64_t nb, void* ws, size_t ws_bytes,
                      float* grad_a, double* loss, float* loss32, void* stream) {
  const size_t need = dpsr_chamfer_ws_bytes(na, nb);
  if (!a || !b || !ws || !grad_a || !loss || need == 0 || ws_bytes < need || ((uintptr_t)ws & 15)) return DPSR_EINVAL;
  dpsr::NnPair P = {};
  dpsr::nn_layout(P, na, nb, (char*)ws);
  P.s[0].p = a;
  P.s[1].p = b;
  P.grad = grad_a;
  P.loss = loss;
  P.loss32 = loss32;
  cudaStream_t st = (cudaStream_t)stream;
  const int bits = std::max(dpsr::cell_bits(na), dpsr::cell_bits(nb));
  const size_t smem = sizeof(int) << (3 * bits);
  // per call: the attribute belongs to the current device, and costs nothing next to the launch
  if (smem > 48 * 1024 && cudaFuncSetAttribute(dpsr::k_nn_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return DPSR_ECUDA;
  }
  const int64_t blocks = (na + dpsr::kQB - 1) / dpsr::kQB + (nb + dpsr::kQB - 1) / dpsr::kQB;
  cudaError_t e = dpsr::launch_k(dpsr::k_nn_sort, dim3(2 * dpsr::kCs), dim3(dpsr::kSortNT), smem, st, dpsr::kCs, P);
  if (e == cudaSuccess)
    e = dpsr::launch_k(dpsr::k_nn_query, dim3((unsigned)blocks),
                       dim3(dpsr::kQNT), 0, st, 0, P);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess ? DPSR_OK : DPSR_ECUDA;
}

}  // extern "C"
