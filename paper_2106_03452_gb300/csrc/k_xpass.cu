// x-axis pass: FFT along x of the partially transformed fields, the spectral
// solve of Eq. 3 (forward) or its adjoint (backward), and the inverse FFT
// along x, for a tile of 16 (8) consecutive kz columns at one ky, moved between
// HBM and shared memory by TMA.
//
// Forward:  chi~ = G(k) (D + i u_x C),  G = g(u) / (-2 pi |u|^2),
//           g = exp(-2 sigma^2 |u|^2 / r^2)                        (Eq. 3, A7)
//           with the spectral sums for the mean and the value at x = 0 of
//           Eq. 4 (Parseval over the half spectrum, and along x) up to r = 128.
// Backward: F = G(k) (g_a FFT(dchi) + g_s + g_w W~), the bracket formed here up
//           to r = 128 and by the y pass above (kHalfW);  Q1 = IFFT_x(F),
//           Q2 = IFFT_x(-i u_x F)  (the adjoint of Eq. 3, conj(H_a) = -H_a).
// Three FFTs of length r per column in each direction.
#include <atomic>

#include "col.cuh"
#include "dpsr_dev.cuh"
#include "launch.h"
#include "finalize.cuh"
#include "tma.cuh"

namespace dpsr {

template <int L>
struct XGeo {
  using F = ColFft<L>;
  static constexpr int R1 = F::R1, T = F::T;
  static constexpr int KC = tile_cols(L);                   // kz columns per CTA (one TMA box row)
  static constexpr int NG = KC * T >= 32 ? KC : 32 / T;     // groups (at least one warp)
  static constexpr int NT = NG * T;                         // threads
  static constexpr int H = L / 2;
  static constexpr int NCHUNK = x_tiles(L) / L;
  static constexpr int BOX = L * KC;                        // float2 per box
  static constexpr int KP = kpitch(L);                      // row pitch of the spectral buffers
  // Two tiles per CTA in both directions. Up to r = 128 the forward needs W~
  // for its spectral sums, after the transforms of C: it reads W~'s column
  // straight from L2 (the spectra stay resident there), and the backward reads
  // W~'s tile. From r = 256 on W~ has no part in the x passes (kHalfW).
  static constexpr bool HW = kHalfW<L>;
  static constexpr bool TIGHT = L == 256;
  static constexpr int NCH = 2;
};

// G(k) = g(k) / (-2 pi |u|^2) with g separable: g1[kx] * (g1[ky] g1[kz]);
// gyz and u2yz are the per-thread (ky, kz) factors. Zero at k = 0.
__device__ __forceinline__ float spectral_G(int kx, float gyz, float u2yz, const float* g1,
                                            const float* u2) {
  const float s = u2[kx] + u2yz;
  if (s == 0.f) return 0.f;
  return __fdividef(g1[kx] * gyz, -6.28318530717958647692f * s);
}

template <int L, bool BWD>
constexpr size_t xpass_smem() {
  using P = XGeo<L>;
  constexpr int NCH = P::NCH;
  // r = 256: the boxes at the start of an allocation aligned for them, and no
  // static shared memory (the barriers lie in the twiddles of k1 = 0, which are
  // one and not read): six CTAs an SM to the byte instead of five, forward 52.4 ->
  // 49.2 us, backward 49.0 -> 46.0
  return (P::TIGHT ? 0 : box_align<L>()) + sizeof(float2) * ((size_t)NCH * P::BOX + P::F::TWN) + 3 * sizeof(float) * L;
}

// One CTA per (kz tile, ky): TMA loads the tiles [x][16 or 8 kz] of the
// input channels (128B-swizzled boxes), each group of T threads transforms
// one kz column along x in registers (the box column doubles as its exchange
// buffer), and TMA stores the results.
template <int L, bool BWD>
__global__ void __launch_bounds__(XGeo<L>::NT, L >= 512 ? 3 : (L >= 256 ? 6 : 5))
    k_xpass(const __grid_constant__ Solve s0, const Solve* __restrict__ tab) {
  using P = XGeo<L>;
  constexpr int NCH = P::NCH;
  const Solve& S = tab ? tab[blockIdx.z] : s0;
  const int kz0 = blockIdx.x * P::KC, ky = blockIdx.y;
  using F = ColFft<L>;
  const int tid = threadIdx.x, g = F::LN::group(tid), t = F::LN::lane(tid);
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  constexpr uint32_t AL = box_align<L>();
  const uint32_t pad = P::TIGHT ? 0u : (AL - (smem_u32(smem_raw) & (AL - 1u))) & (AL - 1u);
  float2* box = reinterpret_cast<float2*>(smem_raw + pad);  // NCH boxes
  float2* tw = box + NCH * P::BOX;
  float* g1 = reinterpret_cast<float*>(tw + P::F::TWN);
  float* u2 = g1 + L;
  float* iu = u2 + L;
  // One barrier per box: the forward transforms D while C still lands.
  uint64_t* bar;
  if constexpr (P::TIGHT) {
    static_assert(box_align<256>() == 1024, "the declared alignment");
    bar = reinterpret_cast<uint64_t*>(tw);
  } else {
    __shared__ uint64_t bars[NCH];
    bar = bars;
  }
  // inputs: forward D, C; backward FFT_zy(dchi) and, without kHalfW, W~
  const int src0 = kSpD, src1 = BWD ? kSpW : kSpC;
  pdl_trigger();
  pdl_wait();
  // the binning of this forward pass is done: its counters start the next one at zero
  if constexpr (!BWD) clear_bin_counters(S, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
  if constexpr (!BWD && P::HW) {
    if (blockIdx.x == 0 && blockIdx.y == 0 && tid < kMuCopies * kMuBins)
      reinterpret_cast<double2*>(S.part)[tid] = make_double2(0.0, 0.0);
  }
  // From r = 64 on the splat's spectra (D, C, W~) are only loaded for the
  // x-chunks that points touch, a lane of warp 0 per chunk; the rest is zero.
  constexpr bool TWO = !(BWD && P::HW);  // two input tiles
  const unsigned chunks = kSkip<L> && TWO ? chunk_mask(S, L) : 0xffu;
  constexpr int XC = L / kXChunks;
  auto has = [chunks](int j) { return !kSkip<L> || ((chunks >> (P::T * j / XC)) & 1u); };  // x = t + T j, t < T
  auto load_chunks = [&](int buf, int c) {  // warp 0
    if (tid == 0) mbar_expect_tx(&bar[c], __popc(chunks) * XC * P::KC * (uint32_t)sizeof(float2));
    __syncwarp();
    if (tid < kXChunks && ((chunks >> tid) & 1u))
      tma_load_3d(box + c * P::BOX + tid * XC * P::KC, &S.tmc[buf], kz0, ky, tid * XC, &bar[c]);
  };
  auto load_all = [&](int buf, int c) {  // thread 0
    mbar_expect_tx(&bar[c], P::BOX * (uint32_t)sizeof(float2));
    for (int x = 0; x < L; x += tma_rows(L))
      tma_load_3d(box + c * P::BOX + x * P::KC, &S.tmx[buf], kz0, ky, x, &bar[c]);
  };
  if (tid < 32) {
    if (tid == 0) {
#pragma unroll
      for (int c = 0; c < NCH; ++c) mbar_init(&bar[c], 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if constexpr (kSkip<L>) {
      if (!BWD) load_chunks(src0, 0);
      else if (tid == 0) load_all(src0, 0);
      if constexpr (TWO) load_chunks(src1, 1);
    } else if (tid == 0) {
      load_all(src0, 0);
      load_all(src1, 1);
    }
  }
  for (int i = tid; i < L; i += P::NT) {
    if (!P::TIGHT || i >= P::T) tw[F::tw_at(i)] = S.tw[i];
    g1[i] = S.g1[i];
    u2[i] = S.u2[i];  // x axis
    iu[i] = S.iu[i];
  }
  __syncthreads();
  // Each thread records its own bounded waits; the block votes before any
  // store, so that a timeout leaves uniformly (the transforms of a lane whose
  // wait ran out compute on stale data, which is never stored).
  bool ok = true;
  auto box_wait = [&](int c, uint32_t phase = 0u) {
    if (ok) ok = mbar_wait(&bar[c], phase);
  };
  auto leave = [&]() {  // after a failed vote
    if (tid == 0) {
      atomicOr(S.status, kStTimeout);
#pragma unroll
      for (int c = 0; c < (TWO ? 2 : 1); ++c) mbar_wait(&bar[c], 0);  // copies in flight: a last bounded chance
    }
  };
  const int gc = g < P::KC ? g : P::KC - 1;  // extra groups (tiny r) shadow the last column
  const bool own = g < P::KC;
  const int kz = min(kz0 + gc, P::H);
  // (a column next to a valid one is transformed with it: they share barriers)
  const bool valid = own && kz0 + (F::WIDE ? g & ~1 : g) <= P::H;
  // shared-memory twiddles and one live column array
  // u2 in shared memory is the x axis' table; the y and z axes' come from global memory
  const float gyz = g1[ky] * g1[kz], u2yz = __ldg(S.u2 + L + ky) + __ldg(S.u2 + 2 * L + kz);
  const typename F::CL c0(box, t, gc), c1(box + P::BOX, t, gc);
  float2 a[P::R1];
  if constexpr (!BWD) {
    // Columns past Nyquist (the last kz tile) hold zeros and are not stored:
    // their groups skip the transforms.
    float am = 0.f, as = 0.f, wz = 0.f;
    if (valid) {
      // chi~ = G (FFT_x(D) + i u_x FFT_x(C)); one column array live at a time:
      // FFT_x(D) goes back to its column, FFT_x(C) meets it there.
      box_wait(0);
#pragma unroll
      for (int j = 0; j < P::R1; ++j) a[j] = has(j) ? c0.get(j) : czero();
      F::template run<-1>(a, c0, tw, t);
      if (own) {  // groups past the last column (tiny r) only shadow it
#pragma unroll
        for (int j = 0; j < P::R1; ++j) c0.put(j, a[j]);
      }
      box_wait(1);
#pragma unroll
      for (int j = 0; j < P::R1; ++j) a[j] = has(j) ? c1.get(j) : czero();
      F::template run<-1>(a, c1, tw, t);
#pragma unroll
      for (int j = 0; j < P::R1; ++j) {
        const int kx = t + P::T * j;  // this lane wrote c0(kx) above
        const float G = spectral_G(kx, gyz, u2yz, g1, u2);
        a[j] = cscale(cadd(c0.get(j), cmul_iu(a[j], iu[kx])), G);
      }
    }
    if (valid) {
      F::template run<+1>(a, c0, tw, t);  // P = unnormalised IFFT_x(chi~)
      if constexpr (!P::HW) {
        // Spectral sums of Eq. 4, by Parseval along x against the x-domain W~
        // (its column straight from L2):
        // sum_kx conj(W~(kx)) chi~(kx) = sum_x conj(W~_x(x)) P(x),
        // sum_kx chi~(kx) = P(x = 0).
        const float2* wc = S.spec[kSpW] + (size_t)ky * P::KP + kz;
#pragma unroll
        for (int j = 0; j < P::R1; ++j) {
          const float2 w = has(j) ? __ldcg(wc + (size_t)(t + P::T * j) * L * P::KP) : czero();
          am += w.x * a[j].x + w.y * a[j].y;
        }
        if (t == 0) as = a[0].x;
        wz = (kz == 0 || kz == P::H) ? 1.f : 2.f;
      }
      if (own) {
#pragma unroll
        for (int j = 0; j < P::R1; ++j) c0.put(j, a[j]);
      }
    }
    FF fm = {am * wz, 0.f}, fs = {as * wz, 0.f};  // wz in {1, 2}: exact
    fence_async_smem();
    if (!__syncthreads_and(ok)) {  // the tile is complete
      leave();
      return;
    }
    if (tid == 0) {
      for (int x = 0; x < L; x += tma_rows(L)) tma_store_3d(&S.tmx[kSpChi], kz0, ky, x, box + x * P::KC);
      tma_store_commit();
    }
    // Summed by the inverse plane kind, which runs before anything reads the
    // scalars. A last-block ticket here (a fence and an atomic on one address
    // per CTA, its place on the SM held for the round trip) cost more than the
    // transforms: 75 -> 63 us at r = 256 without it, 807 -> 552 at r = 512.
    if constexpr (!P::HW) {
      block_sum_ff<P::NT>(fm, fs);
      if (tid == 0) S.part[blockIdx.y * gridDim.x + blockIdx.x] = make_float4(fm.hi, fm.lo, fs.hi, fs.lo);
    }
    if (tid == 0) tma_store_wait_read();
  } else {
    // FFT_x of (g_a FFT_zy(dchi) + g_w W~ + g_s delta_{x=0}): the three terms
    // of the adjoint spectrum combined before the transform (it is linear); from
    // r = 256 on the y pass has combined them.
    float* coef = nullptr;
    if constexpr (!P::HW) {
      __shared__ float coef_[3];
      coef = coef_;
      const Scalars* sc = S.sc;
      const int np = sc->bparts;
      if (np > 0) {  // the plane pass left its partial sums: every CTA adds them up, the first one publishes
        FF x, y;
        sum_partials<P::NT>(S, np, x, y);
        if (tid == 0) {
          const BwdScalars q = bwd_scalars(S, ff_to_double(x), ff_to_double(y));
          coef[0] = q.g_a;
          coef[1] = q.g_s;
          coef[2] = q.g_w;
          if (blockIdx.x == 0 && blockIdx.y == 0) finalize_scalars(S, ff_to_double(x), ff_to_double(y), true);
        }
      } else if (tid == 0) {
        coef[0] = sc->g_a;
        coef[1] = sc->g_s;
        coef[2] = sc->g_w;
      }
    }
    box_wait(0);
    if constexpr (TWO) box_wait(1);
    if (!__syncthreads_and(ok)) {  // both tiles are needed from the start
      leave();
      return;
    }
    if constexpr (P::HW) {
#pragma unroll
      for (int j = 0; j < P::R1; ++j) a[j] = c0.get(j);
    } else {
      const float ga = coef[0], gs = coef[1], gw = coef[2];
#pragma unroll
      for (int j = 0; j < P::R1; ++j) {
        const int x = t + P::T * j;
        a[j] = cadd(cscale(c0.get(j), ga), has(j) ? cscale(c1.get(j), gw) : czero());
        if (x == 0) a[j].x += gs;
      }
    }
    F::template run<-1>(a, c0, tw, t);
    {
      // F = G (.); Q2's input -i u_x F goes to the column of W~ (read above by
      // this group), Q1 = IFFT_x(F) is transformed from registers first
#pragma unroll
      for (int j = 0; j < P::R1; ++j) {
        const int kx = t + P::T * j;
        a[j] = cscale(a[j], spectral_G(kx, gyz, u2yz, g1, u2));
        if (own) c1.put(j, cmul_iu(a[j], -iu[kx]));
      }
      F::template run<+1>(a, c0, tw, t);
      if (own) {
#pragma unroll
        for (int j = 0; j < P::R1; ++j) c0.put(j, a[j]);
      }
      fence_async_smem();
      __syncthreads();
      if (tid == 0) {  // Q1 leaves while Q2 is transformed: 61.7 -> 60.4 us at r = 256, 635 -> 615 us at r = 512
        for (int x = 0; x < L; x += tma_rows(L)) tma_store_3d(&S.tmx[kSpD], kz0, ky, x, box + x * P::KC);
        tma_store_commit();
      }
#pragma unroll
      for (int j = 0; j < P::R1; ++j) a[j] = c1.get(j);
      F::template run<+1>(a, c1, tw, t);
      if (own) {
#pragma unroll
        for (int j = 0; j < P::R1; ++j) c1.put(j, a[j]);
      }
    }
    fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      for (int x = 0; x < L; x += tma_rows(L))
        tma_store_3d(&S.tmx[kSpChi], kz0, ky, x, box + P::BOX + x * P::KC);  // Q2
      tma_store_commit();
      tma_store_wait_read();
    }
  }
}

template <int L, bool BWD>
static cudaError_t launch_xpass_t(const Solve& s, const Solve* tab, int count, cudaStream_t st) {
  using P = XGeo<L>;
  constexpr size_t smem = xpass_smem<L, BWD>();
  static std::atomic<bool> attr_set{false};
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_xpass<L, BWD>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  return launch_k(k_xpass<L, BWD>, dim3(P::NCHUNK, L, count), dim3(P::NT), smem, st, 0, s, tab);
}

cudaError_t launch_xpass(bool bwd, int r, const Solve& s, const Solve* tab, int count,
                         cudaStream_t st) {
  switch (r) {
    case 8: return bwd ? launch_xpass_t<8, true>(s, tab, count, st) : launch_xpass_t<8, false>(s, tab, count, st);
    case 16: return bwd ? launch_xpass_t<16, true>(s, tab, count, st) : launch_xpass_t<16, false>(s, tab, count, st);
    case 32: return bwd ? launch_xpass_t<32, true>(s, tab, count, st) : launch_xpass_t<32, false>(s, tab, count, st);
    case 64: return bwd ? launch_xpass_t<64, true>(s, tab, count, st) : launch_xpass_t<64, false>(s, tab, count, st);
    case 128: return bwd ? launch_xpass_t<128, true>(s, tab, count, st) : launch_xpass_t<128, false>(s, tab, count, st);
    case 256: return bwd ? launch_xpass_t<256, true>(s, tab, count, st) : launch_xpass_t<256, false>(s, tab, count, st);
    case 512: return bwd ? launch_xpass_t<512, true>(s, tab, count, st) : launch_xpass_t<512, false>(s, tab, count, st);
    default: return cudaErrorInvalidValue;
  }
}

int xpass_blocks(int r) { return x_tiles(r); }

}  // namespace dpsr
