// Mesh extraction on the indicator grid and the surrogate gradient through
// it: the optimisation setting of Sec. 3.2 turns chi into a mesh at level 0
// and back-propagates a loss on points of that mesh through the inverse
// surface normal (Eq. 6: d p_mesh / d chi = -n_mesh).
//
// Extraction: a marching-cubes variant without case tables. Each cube of the
// periodic grid is split into Kuhn's six tetrahedra (the monotone paths from
// corner (0,0,0) to (1,1,1) along the three axes in every order); the level
// set is linear inside each tetrahedron: one triangle where one corner's sign
// differs from the other three, two (a quad) where two and two differ. The
// split puts on every face of a cube the diagonal from its lowest to its
// highest corner, the same diagonal the neighbouring cube puts there, and a
// vertex on an edge is computed from the edge's lower endpoint in both cubes,
// so neighbouring cubes produce bit-identical shared vertices: the surface is
// closed (watertight) wherever it stays away from the wrap-around of the
// periodic domain. Output: a triangle soup in unit-cube coordinates
// (unwrapped: a cube at index r - 1 reaches 1.0), each triangle with its unit
// normal pointing towards increasing chi (outwards for outward point
// normals, reading 8), its corners wound counter-clockwise about it.
#include <math.h>

#include <algorithm>

#include "dpsr.h"
#include "dpsr_dev.cuh"
#include "launch.h"

namespace dpsr {

// The six Kuhn tetrahedra: corners 0, kuhn1(t), kuhn2(t), 7 of the cube (bits x, y, z).
__host__ __device__ constexpr int kuhn1(int t) { return 1 << (t >> 1); }
__host__ __device__ constexpr int kuhn2(int t) { return (0x656353 >> (4 * t)) & 7; }

// Corner signs of tetrahedron t from the 8 corner bits of a cube.
__host__ __device__ constexpr unsigned tet_mask(unsigned neg, int t) {
  return (neg & 1u) | (((neg >> kuhn1(t)) & 1u) << 1) | (((neg >> kuhn2(t)) & 1u) << 2) | (((neg >> 7) & 1u) << 3);
}
// Triangles of a sign mask of 4 corners: one where one corner differs, two where two do.
__host__ __device__ constexpr int tet_tris(unsigned m) { return (0x0112122112212110ull >> (4 * m)) & 3; }

__device__ __forceinline__ float3 f3sub(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 f3cross(float3 a, float3 b) {
  return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float f3dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

// Emit triangle (p0, p1, p2) oriented towards `up` (a vector from the
// tetrahedron's negative corners to its positive ones).
__device__ __forceinline__ void emit(float* tris, float* nrm, unsigned long long k, unsigned long long cap,
                                     float3 p0, float3 p1, float3 p2, float3 up) {
  if (k >= cap) return;
  float3 n = f3cross(f3sub(p1, p0), f3sub(p2, p0));
  if (f3dot(n, up) < 0.f) {
    const float3 q = p1;
    p1 = p2;
    p2 = q;
    n = make_float3(-n.x, -n.y, -n.z);
  }
  const float len = sqrtf(f3dot(n, n));
  const float s = len > 0.f ? 1.f / len : 0.f;
  float* t = tris + 9 * k;
  t[0] = p0.x; t[1] = p0.y; t[2] = p0.z;
  t[3] = p1.x; t[4] = p1.y; t[5] = p1.z;
  t[6] = p2.x; t[7] = p2.y; t[8] = p2.z;
  nrm[3 * k] = n.x * s;
  nrm[3 * k + 1] = n.y * s;
  nrm[3 * k + 2] = n.z * s;
}

// One tetrahedron: its corners' ids, values (chi - level) and cube.
struct Tet {
  int q[4];
  float f[4];
  float3 o;  // unwrapped grid coordinates of the cube's corner 0
  __device__ __forceinline__ int id(int a) const { return a & 2 ? (a & 1 ? q[3] : q[2]) : (a & 1 ? q[1] : q[0]); }
  __device__ __forceinline__ float val(int a) const { return a & 2 ? (a & 1 ? f[3] : f[2]) : (a & 1 ? f[1] : f[0]); }
  // Vertex on the edge between corners a and b, from its lower endpoint
  // (corner ids increase along a tetrahedron), in unit-cube coordinates.
  __device__ __forceinline__ float3 cut(int a, int b, float inv_r) const {
    const int lo = min(a, b), hi = max(a, b), u = id(lo), v = id(hi);
    const float fu = val(lo), fv = val(hi);
    const float t = fu / (fu - fv);
    const float ux = o.x + (u & 1), uy = o.y + ((u >> 1) & 1), uz = o.z + ((u >> 2) & 1);
    const float dx = (float)((v & 1) - (u & 1)), dy = (float)(((v >> 1) & 1) - ((u >> 1) & 1)),
                dz = (float)(((v >> 2) & 1) - ((u >> 2) & 1));
    return make_float3((ux + t * dx) * inv_r, (uy + t * dy) * inv_r, (uz + t * dz) * inv_r);
  }
};

constexpr int kMeshNT = 256;

// Cubes are classified V = 4 consecutive ones along z to a thread (vector
// loads of the four grid rows they touch; V = 1 below r = 64 and for grids off a
// 16-byte boundary), the few that the level set crosses (1 in 70 at r = 128)
// are compacted into a list in shared memory, and the block then works through
// (cube, tetrahedron) pairs, a thread each, at output places known from one
// block scan and one atomic per block. Before, a thread did all of a cube: one
// lane in a warp emitting up to twelve triangles, and an atomic on the one
// counter per crossed cube (125 us at r = 128; now 15.5, against 2.5 for one
// read of the grid at the copy rate: the list phase's uneven blocks are left).
//
// LABELS: a component label per voxel (dpsr_largest_region); then only the
// tetrahedra whose negative corners carry label `keep` emit (their negative
// corners are always in one component).
template <bool LABELS, int V>
__global__ void __launch_bounds__(kMeshNT) k_mesh_extract(const float* __restrict__ chi, int r, int lg, float level,
                                                          float* __restrict__ tris, float* __restrict__ nrm,
                                                          unsigned long long* __restrict__ count,
                                                          unsigned long long cap, const int* __restrict__ labels,
                                                          int keep) {
  __shared__ unsigned list[kMeshNT * V];   // cube within the block | neg << 10 | other << 18
  __shared__ unsigned place[kMeshNT * V];  // first triangle of the cube within the block
  __shared__ unsigned wsum[kMeshNT / 32];
  __shared__ unsigned long long base;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, mask = r - 1;
  const int64_t cell0 = ((int64_t)blockIdx.x * kMeshNT + tid) * V, ncell = (int64_t)1 << (3 * lg);
  const bool in = cell0 < ncell;
  const int i = (int)(cell0 >> (2 * lg)), j = (int)(cell0 >> lg) & mask, k = (int)cell0 & mask;
  unsigned info[V], ntri[V], mine = 0;  // mine: crossed cubes << 16 | triangles
#pragma unroll
  for (int c = 0; c < V; ++c) info[c] = ntri[c] = 0;
  if (in) {
    unsigned s[4];  // per row (x + 2 y): sign bits of z = k .. k + V
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float* row = chi + ((((int64_t)((i + (q & 1)) & mask)) << lg) + ((j + (q >> 1)) & mask) << lg);
      s[q] = 0;
      if constexpr (V == 4) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(row + k));
        s[q] = (f.x - level < 0.f ? 1u : 0u) | (f.y - level < 0.f ? 2u : 0u) | (f.z - level < 0.f ? 4u : 0u) |
               (f.w - level < 0.f ? 8u : 0u);
      } else {
        s[q] = __ldg(row + k) - level < 0.f ? 1u : 0u;
      }
      s[q] |= (__ldg(row + ((k + V) & mask)) - level < 0.f ? 1u : 0u) << V;
    }
#pragma unroll
    for (int c = 0; c < V; ++c) {
      unsigned neg = 0, other = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) neg |= ((s[q] >> c) & 1u) << q | ((s[q] >> (c + 1)) & 1u) << (4 + q);
      if (neg == 0u || neg == 255u) continue;
      if constexpr (LABELS) {  // negative corners that belong to other components
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (!((neg >> q) & 1u)) continue;
          const int ii = (i + (q & 1)) & mask, jj = (j + ((q >> 1) & 1)) & mask, kk = (k + c + (q >> 2)) & mask;
          if (__ldg(labels + ((((int64_t)ii << lg) + jj) << lg) + kk) != keep) other |= 1u << q;
        }
      }
      unsigned n = 0;
#pragma unroll
      for (int t = 0; t < 6; ++t)
        if (!LABELS || tet_mask(other, t) == 0u) n += tet_tris(tet_mask(neg, t));
      if (n == 0) continue;
      info[c] = (unsigned)(tid * V + c) | neg << 10 | other << 18;
      ntri[c] = n;
      mine += 1u << 16 | n;
    }
  }
  if (!__syncthreads_or(mine != 0u)) return;
  // block scan of (crossed cubes, triangles), at most 1 024 and 12 288
  unsigned incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  unsigned at = incl - mine, total = 0;
#pragma unroll
  for (int q = 0; q < kMeshNT / 32; ++q) {
    at += q < w ? wsum[q] : 0u;
    total += wsum[q];
  }
  if (tid == 0) base = atomicAdd(count, (unsigned long long)(total & 0xffffu));
#pragma unroll
  for (int c = 0; c < V; ++c) {
    if (!ntri[c]) continue;
    list[at >> 16] = info[c];
    place[at >> 16] = at & 0xffffu;
    at += 1u << 16 | ntri[c];
  }
  __syncthreads();
  const float inv_r = 1.f / (float)r;  // r is a power of two: exact
  const int items = (int)(total >> 16) * 6;
  for (int it = tid; it < items; it += kMeshNT) {
    const int cube = it / 6, t = it % 6;
    const unsigned e = list[cube], neg = (e >> 10) & 255u, other = (e >> 18) & 255u;
    const unsigned m = tet_mask(neg, t);
    if (tet_tris(m) == 0 || (LABELS && tet_mask(other, t) != 0u)) continue;
    unsigned long long out = base + place[cube];
    for (int u = 0; u < t; ++u)
      if (!LABELS || tet_mask(other, u) == 0u) out += tet_tris(tet_mask(neg, u));
    const int64_t cell = (int64_t)blockIdx.x * (kMeshNT * V) + (e & 1023u);
    const int ci = (int)(cell >> (2 * lg)), cj = (int)(cell >> lg) & mask, ck = (int)cell & mask;
    Tet T;
    T.q[0] = 0;
    T.q[1] = kuhn1(t);
    T.q[2] = kuhn2(t);
    T.q[3] = 7;
    T.o = make_float3((float)ci, (float)cj, (float)ck);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int q = T.q[a];
      const int ii = (ci + (q & 1)) & mask, jj = (cj + ((q >> 1) & 1)) & mask, kk = (ck + (q >> 2)) & mask;
      T.f[a] = __ldg(chi + ((((int64_t)ii << lg) + jj) << lg) + kk) - level;
    }
    const int cnt = __popc(m);
    // up: from the centroid of the negative corners to that of the positive ones
    float3 pn = make_float3(0.f, 0.f, 0.f), pp = pn;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float3 g = make_float3((float)(T.q[a] & 1), (float)((T.q[a] >> 1) & 1), (float)((T.q[a] >> 2) & 1));
      if ((m >> a) & 1u) pn = make_float3(pn.x + g.x, pn.y + g.y, pn.z + g.z);
      else pp = make_float3(pp.x + g.x, pp.y + g.y, pp.z + g.z);
    }
    const float wn = 1.f / (float)cnt, wp = 1.f / (float)(4 - cnt);
    const float3 up = make_float3(pp.x * wp - pn.x * wn, pp.y * wp - pn.y * wn, pp.z * wp - pn.z * wn);
    if (cnt != 2) {
      const unsigned one = cnt == 1 ? m : ~m & 15u;
      const int odd = __ffs(one) - 1;
      unsigned rest = 15u ^ one;
      const int o0 = __ffs(rest) - 1;
      rest &= rest - 1;
      const int o1 = __ffs(rest) - 1, o2 = 31 - __clz(rest);
      emit(tris, nrm, out, cap, T.cut(odd, o0, inv_r), T.cut(odd, o1, inv_r), T.cut(odd, o2, inv_r), up);
    } else {
      const unsigned pos = ~m & 15u;
      const int n0 = __ffs(m) - 1, n1 = 31 - __clz(m), p0 = __ffs(pos) - 1, p1 = 31 - __clz(pos);
      // the quad n0-p0, n0-p1, n1-p1, n1-p0 in cyclic order
      const float3 v0 = T.cut(n0, p0, inv_r), v1 = T.cut(n0, p1, inv_r), v2 = T.cut(n1, p1, inv_r),
                   v3 = T.cut(n1, p0, inv_r);
      emit(tris, nrm, out, cap, v0, v1, v2, up);
      emit(tris, nrm, out + 1, cap, v0, v2, v3, up);
    }
  }
}

static int launch_mesh_extract(const float* chi, int r, float level, float* tris, float* nrm,
                               unsigned long long* count, int64_t cap, const int* labels, int keep,
                               cudaStream_t st) {
  if (cudaMemsetAsync(count, 0, sizeof(unsigned long long), st) != cudaSuccess) return DPSR_ECUDA;
  int lg = 0;
  while ((1 << lg) < r) ++lg;
  // Four cubes a thread from r = 64 on: below, a block of 1 024 cubes leaves SMs idle
  // (32 blocks at r = 32: a sphere 12.5 us, noise 58.1; by single cubes 9.8 and 21.7).
  const int v = r >= 64 && ((uintptr_t)chi & 15) == 0 ? 4 : 1;
  const int64_t n = (int64_t)r * r * r;
  const unsigned blocks = (unsigned)((n + kMeshNT * v - 1) / (kMeshNT * v));
  auto go = [&](auto fn) {
    fn<<<blocks, kMeshNT, 0, st>>>(chi, r, lg, level, tris, nrm, count, (unsigned long long)cap, labels, keep);
  };
  if (labels) v == 4 ? go(k_mesh_extract<true, 4>) : go(k_mesh_extract<true, 1>);
  else v == 4 ? go(k_mesh_extract<false, 4>) : go(k_mesh_extract<false, 1>);
  return cudaGetLastError() == cudaSuccess ? DPSR_OK : DPSR_ECUDA;
}

// Surrogate gradient of Eq. 6 at M mesh points: the loss gradient dL/dp_i
// reaches chi as dL/dchi(p_i) = dL/dp_i . (-n_i), and that value goes onto
// the grid by the adjoint of the trilinear lookup at p_i (the rasterization
// of Eq. A2 with scalar values).
__global__ void __launch_bounds__(256) k_mesh_surrogate(float* __restrict__ grid, int r,
                                                        const float* __restrict__ p, const float* __restrict__ n,
                                                        const float* __restrict__ g, int64_t M) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
    const float v = -(g[3 * i] * n[3 * i] + g[3 * i + 1] * n[3 * i + 1] + g[3 * i + 2] * n[3 * i + 2]);
    const Axis ax = axis_of(p[3 * i], r), ay = axis_of(p[3 * i + 1], r), az = axis_of(p[3 * i + 2], r);
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const int dx = d >> 2, dy = (d >> 1) & 1, dz = d & 1;
      const float w = (dx ? ax.t : 1.f - ax.t) * (dy ? ay.t : 1.f - ay.t) * (dz ? az.t : 1.f - az.t);
      const size_t j = ((size_t)(dx ? ax.i1 : ax.i0) * r + (dy ? ay.i1 : ay.i0)) * r + (dz ? az.i1 : az.i0);
      atomicAdd(&grid[j], w * v);
    }
  }
}

}  // namespace dpsr

extern "C" {

int dpsr_mesh_extract(const float* chi, int r, float level, float* tris, float* normals, int64_t max_tris,
                      unsigned long long* count, void* stream) {
  if (!chi || !count || r < 2 || r > 512 || (r & (r - 1)) || max_tris < 0 || !isfinite(level))
    return DPSR_EINVAL;
  if (max_tris > 0 && (!tris || !normals)) return DPSR_EINVAL;
  return dpsr::launch_mesh_extract(chi, r, level, tris, normals, count, max_tris, nullptr, 0, (cudaStream_t)stream);
}

int dpsr_mesh_extract_region(const float* chi, int r, float level, const int* labels, int keep, float* tris,
                             float* normals, int64_t max_tris, unsigned long long* count, void* stream) {
  if (!chi || !labels || !count || r < 2 || r > 512 || (r & (r - 1)) || max_tris < 0 || !isfinite(level))
    return DPSR_EINVAL;
  if (max_tris > 0 && (!tris || !normals)) return DPSR_EINVAL;
  return dpsr::launch_mesh_extract(chi, r, level, tris, normals, count, max_tris, labels, keep, (cudaStream_t)stream);
}

int dpsr_mesh_surrogate_splat(float* dchi, int r, const float* points, const float* normals, const float* dldp,
                              int64_t M, int accumulate, void* stream) {
  if (!dchi || r < 2 || r > 512 || (r & (r - 1)) || M < 0) return DPSR_EINVAL;
  if (M > 0 && (!points || !normals || !dldp)) return DPSR_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (!accumulate && cudaMemsetAsync(dchi, 0, sizeof(float) * (size_t)r * r * r, st) != cudaSuccess)
    return DPSR_ECUDA;
  if (M == 0) return DPSR_OK;
  const int blocks = (int)std::min<int64_t>((M + 255) / 256, 4736);
  dpsr::k_mesh_surrogate<<<blocks, 256, 0, st>>>(dchi, r, points, normals, dldp, M);
  return cudaGetLastError() == cudaSuccess ? DPSR_OK : DPSR_ECUDA;
}

}  // extern "C"
