// Bi-directional L2 Chamfer distance with exact nearest neighbours from a
// shallow box tree, for callers that bring a workspace (dpsr_chamfer_tree).
//
// Per set: a counting sort along a Morton curve of 2^B cells per axis over the
// set's bounding box, leaves of 32 consecutive points with their boxes, and
// boxes over 32 leaves each. A query only scans the leaves whose box is not
// farther than its best point so far. Box distances are computed with the
// point distance's operations in the same order, and rounding is monotonic, so
// a pruned leaf never holds a point that the brute force search would have
// returned: indices (ties to the lowest) and distances are bit for bit its.
//
// Bound: 2 na nb distances by brute force (577 us for 20 000 x 20 000, one
// thread per query and 79 blocks on 152 SMs) against a few hundred per query
// here; what is left is the latency of the sort's phases and of the descent.
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

// Cells per axis 2^B: 16 up to 32 768 points (about 13 a cell on a surface),
// 32 above, where 16 would leave several leaves to a cell.
__host__ __device__ constexpr int cell_bits(int64_t n) { return n <= 32768 ? 4 : 5; }

struct NnSet {
  const float* p;     // n x 3
  int n, nl1, nl2;    // points, leaves, boxes of 32 leaves
  float4* sorted;     // nl1 * 32: x, y, z, original index (padding: NaN)
  float4* box1;       // nl1 x (lo, hi)
  float4* box2;       // nl2 x (lo, hi)
  int* start;         // first sorted position of each cell
  float* grid;        // lo[3], cells per unit length[3] of the cell grid
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

// Cell of a point on a set's grid. Coordinates off the grid, infinite or NaN
// go to an edge cell: the order of the points only decides how tight the
// boxes are.
__device__ __forceinline__ unsigned cell_of(const float* g, float x, float y, float z, int bits) {
  const int m = (1 << bits) - 1;
  auto q = [m](float v) { return (unsigned)min(max((int)v, 0), m); };
  return morton3(q((x - g[0]) * g[3]), q((y - g[1]) * g[4]), q((z - g[2]) * g[5]));
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

// Box of the 32 points (or boxes) of a warp's lanes: lo in the low values.
__device__ __forceinline__ void warp_box(float3 lo, float3 hi, float4* out, int lane) {
  lo.x = warp_min(lo.x);
  lo.y = warp_min(lo.y);
  lo.z = warp_min(lo.z);
  hi.x = warp_max(hi.x);
  hi.y = warp_max(hi.y);
  hi.z = warp_max(hi.z);
  if (lane == 0) {
    out[0] = make_float4(lo.x, lo.y, lo.z, 0.f);
    out[1] = make_float4(hi.x, hi.y, hi.z, 0.f);
  }
}

// One cluster of 8 CTAs per set sorts it and builds its boxes: bounding box,
// per-CTA histograms in shared memory, exclusive offsets per cell and CTA
// through distributed shared memory (each CTA owns an eighth of the cells),
// scatter, boxes. The phases are separated by cluster barriers, so one launch
// does what would take five; 20 000 points are five per thread. Cluster 0 also
// clears the gradient and the arrival counter of the query kernel.
template <int BITS>
__device__ void nn_sort(const NnSet& S, int* hist) {
  constexpr int NC = 1 << (3 * BITS), SL = NC / kCs, PT = SL / kSortNT;  // cells, per CTA, per thread
  static_assert(PT >= 1, "a cell per thread at least");
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  __shared__ float red[6][kSortNT / 32];
  __shared__ float bb[6];      // this CTA's bounding box: lo, -hi
  __shared__ float g[6];
  __shared__ int wsum[kSortNT / 32];
  __shared__ int slice_total;
  const int n = S.n, first = rank * kSortNT + tid;
  constexpr int STEP = kCs * kSortNT;
  // bounding box of the finite coordinates (hi negated: minima throughout)
  float m[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) m[k] = INFINITY;
#pragma unroll 4
  for (int64_t i = first; i < n; i += STEP) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float v = S.p[3 * i + d];
      if (isfinite(v)) {
        m[d] = fminf(m[d], v);
        m[3 + d] = fminf(m[3 + d], -v);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    m[k] = warp_min(m[k]);
    if (lane == 0) red[k][w] = m[k];
  }
  for (int i = tid; i < NC; i += kSortNT) hist[i] = 0;
  __syncthreads();
  if (w < 6) {
    const float v = warp_min(lane < kSortNT / 32 ? red[w][lane] : INFINITY);
    if (lane == 0) bb[w] = v;
  }
  cl.sync();
  if (tid < 6) {
    float v = INFINITY;
    for (int r = 0; r < kCs; ++r) v = fminf(v, cl.map_shared_rank(bb, r)[tid]);
    const float lo = __shfl_sync(0x3fu, v, tid % 3), hi = -__shfl_sync(0x3fu, v, tid % 3 + 3);
    const float sc = (float)(1 << BITS) / (hi - lo);
    const bool ok = hi > lo && isfinite(sc);
    g[tid] = tid < 3 ? (isfinite(lo) ? lo : 0.f) : (ok ? sc : 0.f);
    if (rank == 0) S.grid[tid] = g[tid];
  }
  __syncthreads();
#pragma unroll 4
  for (int64_t i = first; i < n; i += STEP)
    atomicAdd(&hist[cell_of(g, S.p[3 * i], S.p[3 * i + 1], S.p[3 * i + 2], BITS)], 1);
  cl.sync();
  // this CTA's cells: counts over the CTAs, their exclusive scan, then every
  // CTA's first position of each cell written back to its histogram
  const int c0 = rank * SL + tid * PT;
  int run = 0, tot[PT];
#pragma unroll
  for (int j = 0; j < PT; ++j) {
    tot[j] = 0;
#pragma unroll
    for (int r = 0; r < kCs; ++r) tot[j] += cl.map_shared_rank(hist, r)[c0 + j];
    run += tot[j];
  }
  int incl = run;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  int pos = incl - run, total = 0;
#pragma unroll
  for (int k = 0; k < kSortNT / 32; ++k) {
    pos += k < w ? wsum[k] : 0;
    total += wsum[k];
  }
  if (tid == 0) slice_total = total;
  cl.sync();
  for (int r = 0; r < rank; ++r) pos += *cl.map_shared_rank(&slice_total, r);
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
    const int at = atomicAdd(&hist[cell_of(g, x, y, z, BITS)], 1);
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
    warp_box(bad ? make_float3(inf, inf, inf) : v, bad ? make_float3(-inf, -inf, -inf) : v, S.box1 + 2 * (int64_t)l, lane);
  }
  __threadfence();
  cl.sync();
  for (int l = rank * (kSortNT / 32) + w; l < S.nl2; l += NW) {
    const int64_t c = min((int64_t)l * 32 + lane, (int64_t)S.nl1 - 1);
    const float4 lo = __ldcg(S.box1 + 2 * c), hi = __ldcg(S.box1 + 2 * c + 1);
    warp_box(make_float3(lo.x, lo.y, lo.z), make_float3(hi.x, hi.y, hi.z), S.box2 + 2 * (int64_t)l, lane);
  }
}

__global__ void __launch_bounds__(kSortNT) k_nn_sort(const __grid_constant__ NnPair P) {
  extern __shared__ int hist[];
  const int set = blockIdx.x / kCs;
  pdl_trigger();
  pdl_wait();
  if (set == 0) {
    for (int64_t i = blockIdx.x * kSortNT + threadIdx.x; i < (int64_t)P.s[0].n * 3; i += kCs * kSortNT) P.grad[i] = 0.f;
    if (blockIdx.x == 0 && threadIdx.x == 0) *P.ticket = 0u;
  }
  const NnSet& S = P.s[set];
  if (cell_bits(S.n) == 4) nn_sort<4>(S, hist);
  else nn_sort<5>(S, hist);
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
        seed = min(T.start[cell_of(T.grid, q.x, q.y, q.z, cell_bits(T.n))] / kLeaf, T.nl1 - 1);
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
    S.grid = (float*)take(sizeof(float) * 6);
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
