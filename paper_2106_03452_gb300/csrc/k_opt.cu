// Kernels of the optimisation setting (Sec. 3.2; supplementary Sec. B)
// around the DPSR layer: the bi-directional L2 Chamfer distance between
// points sampled on the mesh and the input cloud (with its gradient with
// respect to the mesh points), the largest component of the mesh for the
// resampling step, and area-weighted sampling of points on the mesh.
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "dpsr.h"
#include "dpsr_dev.cuh"
#include "finalize.cuh"
#include "launch.h"

namespace dpsr {

// ---------------------------------------------------------------------------
// Nearest neighbour by brute force: for every query q_i, the index of the
// closest target (ties: the lowest index) and the squared distance. Targets
// pass through shared memory in tiles of 1024.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_nearest(const float* __restrict__ q, int64_t nq,
                                                 const float* __restrict__ t, int64_t nt,
                                                 int* __restrict__ idx, float* __restrict__ d2) {
  constexpr int TILE = 1024;
  __shared__ float4 sh[TILE];
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  float qx = 0.f, qy = 0.f, qz = 0.f;
  if (i < nq) {
    qx = q[3 * i];
    qy = q[3 * i + 1];
    qz = q[3 * i + 2];
  }
  float best = INFINITY;
  int bi = -1;
  for (int64_t base = 0; base < nt; base += TILE) {
    const int n = (int)std::min<int64_t>(TILE, nt - base);
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const int64_t j = base + k;
      sh[k] = make_float4(t[3 * j], t[3 * j + 1], t[3 * j + 2], 0.f);
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
      const float4 p = sh[k];
      const float dx = p.x - qx, dy = p.y - qy, dz = p.z - qz;
      const float d = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      if (d < best) {
        best = d;
        bi = (int)(base + k);
      }
    }
  }
  if (i < nq) {
    idx[i] = bi;
    d2[i] = best;
  }
}

// dL/da for L = mean_a min_b |a-b|^2 + mean_b min_a |a-b|^2 with respect to
// the points a (the second term scatters: each b pulls its nearest a). A point
// without a neighbour (index -1: no finite distance) pulls nobody, and one of a
// gets a NaN gradient.
__global__ void __launch_bounds__(256) k_chamfer_grad(const float* __restrict__ a, int64_t na,
                                                      const float* __restrict__ b, int64_t nb,
                                                      const int* __restrict__ ab, const int* __restrict__ ba,
                                                      float* __restrict__ ga) {
  const float ca = 2.f / (float)na, cb = 2.f / (float)nb;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < na + nb;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i < na) {
      const int j = ab[i];
#pragma unroll
      for (int d = 0; d < 3; ++d)
        atomicAdd(&ga[3 * i + d], j >= 0 ? ca * (a[3 * i + d] - b[3 * (int64_t)j + d]) : __int_as_float(0x7fffffff));
    } else {
      const int64_t k = i - na;
      const int j = ba[k];
      if (j < 0) continue;
#pragma unroll
      for (int d = 0; d < 3; ++d) atomicAdd(&ga[3 * (int64_t)j + d], cb * (a[3 * (int64_t)j + d] - b[3 * k + d]));
    }
  }
}

// Sum of n values in float-float, in one block (a small reduction per call).
__global__ void __launch_bounds__(256) k_sum2(const float* __restrict__ x, int64_t nx, const float* __restrict__ y,
                                              int64_t ny, double* __restrict__ out) {
  FF sx = {0.f, 0.f}, sy = {0.f, 0.f};
  for (int64_t i = threadIdx.x; i < nx; i += blockDim.x) sx = ff_add(sx, x[i]);
  for (int64_t i = threadIdx.x; i < ny; i += blockDim.x) sy = ff_add(sy, y[i]);
  block_sum_ff<256>(sx, sy);
  if (threadIdx.x == 0) *out = ff_to_double(sx) / (double)nx + ff_to_double(sy) / (double)ny;
}

// ---------------------------------------------------------------------------
// Components of the inside region {chi < level} of the periodic grid, with
// voxels joined along the edge directions of the mesh's tetrahedra (x, y, z,
// x+y, x+z, y+z, x+y+z), so that the negative corners of a tetrahedron are
// always in one component and every mesh triangle belongs to exactly one.
// Lock-free union-find: parent[v] = v for inside voxels, -1 outside; a union
// hangs the larger root under the smaller one with compare-and-swap. Every
// loop is bounded (a count far above any path length); running out sets
// *err.
// ---------------------------------------------------------------------------
constexpr int kFindLimit = 1 << 22;

// Parents are read at L2 (another SM may have just changed them through an
// atomic; a stale L1 copy would only make the CAS below fail again).
__device__ __forceinline__ int uf_find(int* parent, int v, unsigned* err) {
  for (int it = 0; it < kFindLimit; ++it) {
    const int p = __ldcg(parent + v);
    if (p == v) return v;
    const int gp = __ldcg(parent + p);
    if (gp != p) atomicCAS(&parent[v], p, gp);  // path halving
    v = gp;
  }
  atomicOr(err, 1u);
  return v;
}

__global__ void k_cc_init(const float* __restrict__ chi, int64_t n, float level, int* __restrict__ parent) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    parent[v] = chi[v] < level ? (int)v : -1;
}

__global__ void k_cc_union(int r, int* __restrict__ parent, unsigned* __restrict__ err) {
  const int64_t n = (int64_t)r * r * r;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    if (__ldcg(parent + v) < 0) continue;
    const int i = (int)(v / ((int64_t)r * r)), j = (int)((v / r) % r), k = (int)(v % r);
#pragma unroll
    for (int d = 1; d < 8; ++d) {  // the seven monotone offsets (dx, dy, dz) in {0,1}^3 \ 0
      const int64_t w = ((int64_t)((i + (d & 1)) & (r - 1)) * r + ((j + ((d >> 1) & 1)) & (r - 1))) * r +
                        ((k + ((d >> 2) & 1)) & (r - 1));
      if (__ldcg(parent + w) < 0) continue;
      int a = (int)v, b = (int)w;
      for (int it = 0; it < kFindLimit; ++it) {
        a = uf_find(parent, a, err);
        b = uf_find(parent, b, err);
        if (a == b) break;
        if (a < b) {
          const int s = a;
          a = b;
          b = s;
        }
        if (atomicCAS(&parent[a], a, b) == a) break;
        if (it == kFindLimit - 1) atomicOr(err, 1u);
      }
    }
  }
}

// Flatten to roots and count voxels per root.
__global__ void k_cc_flatten(int64_t n, int* __restrict__ parent, int* __restrict__ size, unsigned* __restrict__ err) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    if (__ldcg(parent + v) < 0) continue;
    const int root = uf_find(parent, (int)v, err);
    atomicAdd(&size[root], 1);
  }
}
__global__ void k_cc_relabel(int64_t n, int* __restrict__ parent, unsigned* __restrict__ err) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (__ldcg(parent + v) >= 0) parent[v] = uf_find(parent, (int)v, err);
}

// The root with the most voxels (ties: the lowest root), as
// (size << 32) | (0xffffffff - root) maxima.
__global__ void k_cc_largest(int64_t n, const int* __restrict__ size, unsigned long long* __restrict__ best) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int s = size[v];
    if (s > 0) atomicMax(best, ((unsigned long long)s << 32) | (0xffffffffull - (unsigned long long)v));
  }
}

// ---------------------------------------------------------------------------
// Area-weighted sampling of points on a triangle soup: areas, their prefix
// sums (per block, then the block totals by one block, then the offsets), a
// counter-based uniform per sample (a 64-bit integer hash of seed and index,
// SplitMix64's finaliser), a binary search, and uniform barycentric
// coordinates (the reflection of the unit square onto the triangle).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ double u01(uint64_t seed, uint64_t i) {
  return (double)(mix64(seed + 0x9e3779b97f4a7c15ull * (i + 1)) >> 11) * (1.0 / 9007199254740992.0);
}

constexpr int kScanBlock = 1024;  // triangles per block of the scan
constexpr int kScanNT = 256;      // its threads, four consecutive triangles each

// b - a in FP32, and whether that is exact and a normal number or zero (TwoSum's
// error term; close coordinates, the usual case, leave none; NaN is not).
__device__ __forceinline__ float diff32(float b, float a, bool& ok) {
  const float d = b - a, bb = d + a;
  const float e = (b - bb) + ((bb - d) - a);
  ok = ok && e == 0.f && (d == 0.f || fabsf(d) >= 1.17549435e-38f);
  return d;
}
// A normal FP32 number or zero in FP64, on the integer pipe: conversions share
// the narrow FP64 pipe's rate.
__device__ __forceinline__ double widen(float v) {
  const unsigned u = __float_as_uint(v);
  const unsigned hi = ((u & 0x7fffffffu) >> 3) + 0x38000000u;
  return __hiloint2double((int)((v == 0.f ? 0u : hi) | (u & 0x80000000u)), (int)(u << 29));
}

// Area of the triangle of nine coordinates, times two, squared, in FP64.
__device__ __forceinline__ double cross2(const float* c) {
  bool ok = true;
  const float fx = diff32(c[3], c[0], ok), fy = diff32(c[4], c[1], ok), fz = diff32(c[5], c[2], ok);
  const float gx = diff32(c[6], c[0], ok), gy = diff32(c[7], c[1], ok), gz = diff32(c[8], c[2], ok);
  double ux, uy, uz, vx, vy, vz;
  if (ok) {
    ux = widen(fx), uy = widen(fy), uz = widen(fz);
    vx = widen(gx), vy = widen(gy), vz = widen(gz);
  } else {
    ux = (double)c[3] - c[0], uy = (double)c[4] - c[1], uz = (double)c[5] - c[2];
    vx = (double)c[6] - c[0], vy = (double)c[7] - c[1], vz = (double)c[8] - c[2];
  }
  const double cx = uy * vz - uz * vy, cy = uz * vx - ux * vz, cz = ux * vy - uy * vx;
  return cx * cx + cy * cy + cz * cz;
}

// Areas and their prefix sums within blocks of 1 024 triangles, in FP64. The
// bound is the FP64 pipe (a warp instruction per 15 SM cycles): exact FP32
// differences instead of FP64 ones, and a scan of thread totals (four triangles
// a thread) instead of ten rounds over every triangle. The triangles pass
// through shared memory: whole lines from HBM, and nine conflict-free 16-byte
// reads a thread. (A Newton root from an FP32 seed in place of sqrt() had the
// last bit wrong in one area of some 2^14, and sampling 20 000 points on 150 001
// triangles took 22.5 us with it, 20.5 with sqrt().)
__global__ void __launch_bounds__(kScanNT) k_area_scan(const float* __restrict__ tris, int64_t T,
                                                       double* __restrict__ cum, double* __restrict__ block_tot) {
  constexpr int PT = kScanBlock / kScanNT;
  __shared__ float4 st4[kScanBlock * 9 / 4];
  __shared__ double wtot[kScanNT / 32];
  float* st = reinterpret_cast<float*>(st4);
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t t0 = (int64_t)blockIdx.x * kScanBlock;
  const int n = (int)std::min<int64_t>(kScanBlock, T - t0);
  const float* src = tris + 9 * t0;
  if (n == kScanBlock && ((uintptr_t)src & 15) == 0) {
#pragma unroll
    for (int i = 0; i < kScanBlock * 9 / 4 / kScanNT; ++i)
      st4[tid + i * kScanNT] = __ldg(reinterpret_cast<const float4*>(src) + tid + i * kScanNT);
  } else {
    for (int i = tid; i < 9 * n; i += kScanNT) st[i] = __ldg(src + i);
    for (int i = 9 * n + tid; i < 9 * kScanBlock; i += kScanNT) st[i] = 0.f;  // no area
  }
  __syncthreads();
  float t[9 * PT];
#pragma unroll
  for (int q = 0; q < 9 * PT / 4; ++q) *reinterpret_cast<float4*>(t + 4 * q) = st4[tid * (9 * PT / 4) + q];
  double a[PT];
#pragma unroll
  for (int q = 0; q < PT; ++q) {
    a[q] = fma(0.5, sqrt(cross2(t + 9 * q)), q ? a[q - 1] : 0.0);
  }
  double incl = a[PT - 1];
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) wtot[w] = incl;
  double before = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) before = 0.0;
  __syncthreads();
  for (int k = 0; k < w; ++k) before += wtot[k];
#pragma unroll
  for (int q = 0; q < PT; ++q)
    if (tid * PT + q < n) cum[t0 + tid * PT + q] = before + a[q];
  if (tid == kScanNT - 1) block_tot[blockIdx.x] = before + a[PT - 1];
}

// One block: exclusive prefix of the block totals in place, and the total
// (16 us by one thread for 147 blocks, 2.3 by 256).
__global__ void __launch_bounds__(kScanNT) k_block_offsets(double* __restrict__ tot, int nblocks) {
  __shared__ double wtot[kScanNT / 32];
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (nblocks + kScanNT - 1) / kScanNT;
  const int b0 = std::min(tid * per, nblocks), b1 = std::min(b0 + per, nblocks);
  double run = 0.0;
  for (int b = b0; b < b1; ++b) run += tot[b];
  double incl = run;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) wtot[w] = incl;
  double acc = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) acc = 0.0;
  __syncthreads();
  for (int k = 0; k < w; ++k) acc += wtot[k];
  for (int b = b0; b < b1; ++b) {
    const double v = tot[b];
    tot[b] = acc;
    acc += v;
  }
  if (tid == kScanNT - 1) tot[nblocks] = acc;
}

// A sample's triangle by two searches: the last block whose offset does not
// exceed its draw, then the first triangle of the block whose sum does. No pass
// adds the offsets to the sums first. Up to 2 048 blocks (two million
// triangles) every CTA adds the block totals up in shared memory itself;
// beyond that k_block_offsets has. The second search takes three pivots a step:
// five dependent reads of a 1 024-triangle block instead of ten. The searches
// live in L1, and the grid is small: launched early it would crowd onto the SMs
// that the scan leaves free, so it waits (20 000 points on 150 001 triangles,
// both kernels: 40 us early with the offsets in a launch of their own, 20.5).
//
// The searches compare bits (non-negative doubles are ordered as their bits are):
// the narrow FP64 pipe, which many samples keep busy, has the coordinates to do.
// And half of an SM's memory stays L1, for both kernels alike (a change between
// them empties the SM): the offsets of 13 blocks would take all of it, and the
// searches' reads miss. A million samples of 150 000 triangles: 176 us without
// either, 140 with the comparisons, 103 with both; 20 000: 25.4, 23.5 and 23.5.
constexpr int kOffShared = 2048;
constexpr int kSampleCarve = 50;  // per cent of shared memory: seven blocks
// Threads of a block: 64 up to what the GPU holds of those at a time (20 000 samples:
// 313 blocks, two per SM), 128 beyond.
constexpr int kSampleBlocks = 152 * 7, kSampleFew = 64, kSampleMany = 128;

// The bits of a non-negative sum; a NaN (areas that are not finite) above all.
__device__ __forceinline__ long long sum_bits(double v) {
  const long long k = __double_as_longlong(v);
  return (k & LLONG_MAX) > 0x7ff0000000000000ll ? LLONG_MAX : k;
}

template <int NT>
__global__ void __launch_bounds__(NT) k_sample(const float* __restrict__ tris, const float* __restrict__ nrm,
                                               int64_t T, const double* __restrict__ cum,
                                               const double* __restrict__ tot, int nblocks, int64_t M, uint64_t seed,
                                               float* __restrict__ p, float* __restrict__ n) {
  __shared__ double sh[kOffShared];
  __shared__ double wtot[NT / 32];
  pdl_trigger();
  pdl_wait();
  const double* off = tot;
  const long long* sums = reinterpret_cast<const long long*>(cum);
  double A;
  if (nblocks <= kOffShared) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int i = tid; i < nblocks; i += NT) sh[i] = tot[i];
    __syncthreads();
    const int per = (nblocks + NT - 1) / NT;
    const int b0 = std::min(tid * per, nblocks), b1 = std::min(b0 + per, nblocks);
    double run = 0.0;
    for (int b = b0; b < b1; ++b) run += sh[b];
    double incl = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const double v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += v;
    }
    if (lane == 31) wtot[w] = incl;
    double acc = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) acc = 0.0;
    __syncthreads();
    A = 0.0;
    for (int k = 0; k < NT / 32; ++k) {
      if (k == w) acc += A;
      A += wtot[k];
    }
    for (int b = b0; b < b1; ++b) {
      const double v = sh[b];
      sh[b] = acc;
      acc += v;
    }
    __syncthreads();
    off = sh;
  } else {
    A = tot[nblocks];
  }
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < M; s += (int64_t)gridDim.x * blockDim.x) {
    int64_t lo = 0;
    if (T > 1) {
      const double x = u01(seed, 3 * s) * A;
      const long long xk = sum_bits(x);
      int b = 0, e = nblocks;  // off[b] <= x (off[0] = 0), off[e] > x or e the end
      while (e - b > 1) {
        const int mid = (b + e) >> 1;
        if (__double_as_longlong(off[mid]) > xk) e = mid;
        else b = mid;  // NaN areas too: the last triangle answers, as in the second search
      }
      const long long yk = sum_bits(x - off[b]);
      lo = (int64_t)b * kScanBlock;
      int64_t hi = std::min<int64_t>(lo + kScanBlock, T) - 1;
      while (lo < hi) {
        const int len = (int)(hi - lo);
        const int64_t m1 = lo + len / 4, m2 = lo + len / 2, m3 = lo + 3 * len / 4;  // lo <= m1 <= m2 <= m3 < hi
        const long long c1 = sums[m1], c2 = sums[m2], c3 = sums[m3];
        if (c2 > yk) {
          hi = m2;
          if (c1 > yk) hi = m1;
          else lo = m1 + 1;
        } else {
          lo = m2 + 1;
          if (c3 > yk) hi = m3;
          else lo = m3 + 1;
        }
      }
    }
    double u = u01(seed, 3 * s + 1), v = u01(seed, 3 * s + 2);
    if (u + v > 1.0) {
      u = 1.0 - u;
      v = 1.0 - v;
    }
    const float* t = tris + 9 * lo;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      p[3 * s + d] = (float)(t[d] + u * (t[3 + d] - t[d]) + v * (t[6 + d] - t[d]));
      n[3 * s + d] = nrm[3 * lo + d];
    }
  }
}

// The share of shared memory of the sampling kernels, once per device.
static cudaError_t sample_carve() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || (dev < 64 && (done.load() >> dev) & 1u)) return e;
  const auto share = cudaFuncAttributePreferredSharedMemoryCarveout;
  e = cudaFuncSetAttribute(k_area_scan, share, kSampleCarve);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sample<kSampleFew>, share, kSampleCarve);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sample<kSampleMany>, share, kSampleCarve);
  if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev);
  return e;
}

}  // namespace dpsr

extern "C" {

int dpsr_chamfer(const float* a, int64_t na, const float* b, int64_t nb, int* ws_idx, float* ws_d2, float* grad_a,
                 double* loss, void* stream) {
  if (!a || !b || !ws_idx || !ws_d2 || !grad_a || !loss || na < 1 || nb < 1 || na > INT32_MAX || nb > INT32_MAX)
    return DPSR_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int* ab = ws_idx;
  int* ba = ws_idx + na;
  float* dab = ws_d2;
  float* dba = ws_d2 + na;
  if (cudaMemsetAsync(grad_a, 0, sizeof(float) * 3 * na, st) != cudaSuccess) return DPSR_ECUDA;
  dpsr::k_nearest<<<(unsigned)((na + 255) / 256), 256, 0, st>>>(a, na, b, nb, ab, dab);
  dpsr::k_nearest<<<(unsigned)((nb + 255) / 256), 256, 0, st>>>(b, nb, a, na, ba, dba);
  const int blocks = (int)std::min<int64_t>((na + nb + 255) / 256, 4736);
  dpsr::k_chamfer_grad<<<blocks, 256, 0, st>>>(a, na, b, nb, ab, ba, grad_a);
  dpsr::k_sum2<<<1, 256, 0, st>>>(dab, na, dba, nb, loss);
  return cudaGetLastError() == cudaSuccess ? DPSR_OK : DPSR_ECUDA;
}

int dpsr_largest_region(const float* chi, int r, float level, int* labels, int* ws, unsigned long long* best,
                        unsigned* err, void* stream) {
  if (!chi || !labels || !ws || !best || !err || r < 2 || r > 512 || (r & (r - 1))) return DPSR_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t n = (int64_t)r * r * r;
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, 152 * 32);
  if (cudaMemsetAsync(ws, 0, sizeof(int) * n, st) != cudaSuccess ||
      cudaMemsetAsync(best, 0, sizeof(unsigned long long), st) != cudaSuccess ||
      cudaMemsetAsync(err, 0, sizeof(unsigned), st) != cudaSuccess)
    return DPSR_ECUDA;
  dpsr::k_cc_init<<<blocks, 256, 0, st>>>(chi, n, level, labels);
  dpsr::k_cc_union<<<blocks, 256, 0, st>>>(r, labels, err);
  dpsr::k_cc_flatten<<<blocks, 256, 0, st>>>(n, labels, ws, err);
  dpsr::k_cc_relabel<<<blocks, 256, 0, st>>>(n, labels, err);
  dpsr::k_cc_largest<<<blocks, 256, 0, st>>>(n, ws, best);
  return cudaGetLastError() == cudaSuccess ? DPSR_OK : DPSR_ECUDA;
}

int dpsr_mesh_sample(const float* tris, const float* normals, int64_t T, int64_t M, uint64_t seed, double* ws,
                     float* points, float* pnormals, void* stream) {
  if (!tris || !normals || !ws || !points || !pnormals || T < 1 || M < 0) return DPSR_EINVAL;
  if (M == 0) return DPSR_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const int nblk = (int)((T + dpsr::kScanBlock - 1) / dpsr::kScanBlock);
  double* cum = ws;
  double* tot = ws + T;  // nblk + 1 entries
  cudaError_t e = dpsr::sample_carve();
  if (e == cudaSuccess)
    e = dpsr::launch_k(dpsr::k_area_scan, dim3(nblk), dim3(dpsr::kScanNT), 0, st, 0, tris, T, cum, tot);
  if (e == cudaSuccess && nblk > dpsr::kOffShared)
    e = dpsr::launch_k(dpsr::k_block_offsets, dim3(1), dim3(dpsr::kScanNT), 0, st, 0, tot, nblk);
  auto sample = [&](auto fn, int nt) {
    const unsigned blocks = (unsigned)std::min<int64_t>((M + nt - 1) / nt, dpsr::kSampleBlocks);
    return dpsr::launch_after(fn, dim3(blocks), dim3(nt), 0, st, 0, tris, normals, T, (const double*)cum,
                              (const double*)tot, nblk, M, seed, points, pnormals);
  };
  if (e == cudaSuccess)
    e = M <= (int64_t)dpsr::kSampleBlocks * dpsr::kSampleFew ? sample(dpsr::k_sample<dpsr::kSampleFew>, dpsr::kSampleFew)
                                                            : sample(dpsr::k_sample<dpsr::kSampleMany>, dpsr::kSampleMany);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess ? DPSR_OK : DPSR_ECUDA;
}

}  // extern "C"
