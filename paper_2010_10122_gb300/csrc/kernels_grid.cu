// Degridding (Eq. R3) and gridding (Eq. Rad2) kernels of the w-gridder.
//
// Work decomposition (GPU counterpart of Secs. 4.3-4.4):
//  * the uv grid is cut into T x T tiles; visibilities are binned by (tile of their first
//    cell, first w-plane c0) — the device index;
//  * a group of G lanes (G = 4, 8 or 16 >= alpha) handles one visibility: lane j evaluates
//    the j-th kernel piece in u, v and w by Horner (Sec. 4.2) and owns column j of the
//    alpha x alpha footprint;
//  * degrid: one CTA per (tile, sub-batch of planes) stages tile + (alpha - 1) halo of those
//    planes in shared memory; each visibility of the tile sums its footprint over the staged
//    planes, lanes reduce by shuffles, and the partial sum goes to a fixed slot; a finalize
//    pass adds the slots in order (deterministic, no atomics);
//  * grid: one CTA per (tile, sub-batch of planes) owns the T x T cells of those planes and
//    accumulates contributions of visibilities from its own tile and the three tiles whose
//    footprints reach into it, then writes every cell exactly once (no global atomics, no
//    separate zeroing pass; empty tiles write zeros).  Accumulation schemes: FP32 on the tensor
//    cores, products of bf16 slices that lose nothing (k_grid_mma, the automatic choice with 32-cell
//    tiles), or shared-memory atomics (k_grid_atomic); FP64 planes by warps that each own whole
//    planes (k_grid_owner: shared-memory double atomics occupy the FP64 pipe);
//  * FP64 plans with the double-float FFT keep the planes as double-float pairs: k_degrid_dd, and
//    k_grid_cells_dd with the cells' sums in registers, in pair arithmetic on the FP32 pipes
//    (df64.cuh).
#include <cmath>
#include <type_traits>

#include "df64.cuh"
#include "fft_engine.cuh"
#include "wgrid_internal.h"

namespace wg {

constexpr int kThreads = 256;


// asynchronous 8- or 16-byte global -> shared copy (cp.async) of one plane cell; completed by
// stage_wait() before the block's barrier
template <typename CT>
__device__ __forceinline__ void stage_copy(CT* d, const CT* g) {
  static_assert(sizeof(CT) == 8 || sizeof(CT) == 16, "plane cell size");
  const unsigned sa = (unsigned)__cvta_generic_to_shared(d);
  if (sizeof(CT) == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(g) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(g) : "memory");
}
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

template <typename R>
__device__ __forceinline__ R horner(const R* __restrict__ sc, int deg, int j, R z) {
  R r = sc[deg * kMaxG + j];
  for (int d = deg - 1; d >= 0; --d) r = fma(r, z, sc[d * kMaxG + j]);
  return r;
}

// piece j of direction d (0 u, 1 v, 2 w) of indexed visibility vi: from the per-call table when
// present, else by Horner from the shared-memory coefficients
template <typename R>
__device__ __forceinline__ R kernel_value(const IndexView<R>& ix, const R* __restrict__ sc,
                                          int deg, uint32_t vi, int d, int j, R z) {
  if (ix.wts != nullptr) return ix.wts[(int64_t)vi * (3 * kMaxG) + d * kMaxG + j];
  return horner(sc, deg, j, z);
}

// The coefficients of one kernel piece held in a lane's registers (FP32 kernels, where a lane
// evaluates the same piece for every visibility it handles): zero-padded up to degree G + 3
// (alpha <= G), so Horner runs a fixed number of steps with no shared-memory loads.
template <typename R, int G>
struct LanePiece {
  static constexpr int kDeg = G + 3;
  R c[kDeg + 1];
  __device__ __forceinline__ void load(const R* __restrict__ sc, int deg, int j) {
#pragma unroll
    for (int d = 0; d <= kDeg; ++d) c[d] = d <= deg ? sc[d * kMaxG + j] : (R)0;
  }
  __device__ __forceinline__ R eval(R z) const {
    R r = c[kDeg];
#pragma unroll
    for (int d = kDeg - 1; d >= 0; --d) r = fma(r, z, c[d]);
    return r;
  }
};
// register pieces for FP32 only (an FP64 piece would take 40 registers; FP64 plans read the
// per-call or plan-resident value table, or Horner from shared memory)
template <typename R, int G>
using LanePieceOf = LanePiece<R, sizeof(R) == 4 ? G : 0>;

template <typename R, int G>
__device__ __forceinline__ R kernel_value(const IndexView<R>& ix, const LanePieceOf<R, G>& pc,
                                          const R* __restrict__ sc, int deg, uint32_t vi, int d,
                                          int j, R z) {
  if (ix.wts != nullptr) return ix.wts[(int64_t)vi * (3 * kMaxG) + d * kMaxG + j];
  if (sizeof(R) == 4) return pc.eval(z);
  return horner(sc, deg, j, z);
}

template <int G>
__device__ __forceinline__ unsigned group_mask() {
  const int lane = threadIdx.x & 31;
  return G == 32 ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
}

// The visibilities of tile t that meet each of the planes s0 .. s0 + sb - 1 (at most 32): lane pl
// holds plane s0 + pl's index range, so that all are known after one load.
struct DegridRange {
  uint32_t first, end;   // of this lane's plane
  unsigned used;         // planes some visibility meets
  uint32_t lo, hi;       // this CTA's visibilities (share)
  __device__ __forceinline__ DegridRange(const uint32_t* __restrict__ offt, int nw, int aw, int s0, int sb) {
    const int lane = threadIdx.x & 31, p = s0 + min(lane, sb - 1);
    first = offt[max(0, p - aw + 1)];
    end = offt[min(p + 1, nw)];
    used = __ballot_sync(0xffffffffu, lane < sb && first != end);
  }
  // blockIdx.z's share among gridDim.z CTAs, of at least `least` visibilities (a multiple of 64, so
  // that shares are whole passes of a CTA): only tiles with more are taken by several
  __device__ __forceinline__ void share(int sb, uint32_t least) {
    lo = __shfl_sync(0xffffffffu, first, 0);
    hi = __shfl_sync(0xffffffffu, end, sb - 1);
    if (gridDim.z == 1) return;
    const uint32_t n = max(least, ((hi - lo + gridDim.z - 1) / gridDim.z + 63) & ~63u);
    lo = min(hi, lo + blockIdx.z * n);
    hi = min(hi, lo + n);
  }
};
// f(cell of the buffer, cell of the plane) for the tile and its halo in the used planes: a warp
// takes whole rows, so a cell costs an addition
template <typename F>
__device__ __forceinline__ void degrid_rows(const Geom& g, int tu, int tv, int p0, int sb, unsigned used, F f) {
  const int T = g.tile, TH = T + g.alpha - 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t pstride = (int64_t)g.nu * g.nv;
  for (int c = lane; c < TH; c += 32) {
    int gv = tv * T + c; if (gv >= g.nv) gv -= g.nv;
    for (int pl = 0; pl < sb; ++pl) {
      if (!((used >> pl) & 1)) continue;
      for (int r = warp; r < TH; r += kThreads / 32) {
        int gu = tu * T + r; if (gu >= g.nu) gu -= g.nu;
        f((pl * TH + r) * TH + c, (p0 + pl) * pstride + (int64_t)gu * g.nv + gv);
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// degrid
//
// CTA = (uv tile, sub-batch of bs planes).  The CTA stages tile + (alpha - 1) halo of each plane
// of its sub-batch that some visibility of the tile needs, then every visibility of the tile
// whose planes meet the sub-batch computes its partial sum over those planes and stores it, as
// is, in slot (sub-batch id - first sub-batch id of the visibility) of a partial-sum array
// indexed by the visibility's position in the index.  Sub-batches are aligned to multiples of
// bs over the whole plane range, so a visibility meets at most `nslot` of them; a finalize pass
// adds its slots in slot order (deterministic, no atomics) and applies the w-reference phase,
// the Hermitian fold and the weight.
//
// Bound by the staged bytes from L2 (half of the time of double-float planes on 16-cell tiles, where
// the halo makes 3.6 times the tile's cells) and then by the latency of the footprint sums.  So the
// index ranges of all planes come in one load, rows are copied without a division per cell, the
// next visibility's index entry is loaded ahead, and dense tiles go to several CTAs (see degrid_shares).
// Measured before and after, FP32: 1e6 visibilities on a 2048^2 image, alpha = 8, 0.69 -> 0.62 ms; 1e7
// on 4096^2 4.10 -> 3.90; with a tenth of 8e5 visibilities in one tile, alpha = 6, 3.15 -> 0.63.  (Real
// and imaginary part packed in one FMA: 0.74 / 0.66 / 0.74 ms with one / two / four planes at once.)
// ---------------------------------------------------------------------------------------
template <typename R, int G>
__global__ void __launch_bounds__(kThreads)
k_degrid(const Geom g, const __grid_constant__ Coef<R> coef, const IndexView<R> ix,
         const typename C2<R>::T* __restrict__ planes, int b0, int nb, int bs,
         typename C2<R>::T* __restrict__ partial, int64_t nvis_idx, uint32_t least) {
  using CT = typename C2<R>::T;
  extern __shared__ __align__(16) unsigned char smem[];
  R* sc = reinterpret_cast<R*>(smem);
  CT* st = reinterpret_cast<CT*>(smem + (kMaxDeg + 1) * kMaxG * sizeof(R));
  const int T = g.tile, alpha = g.alpha, aw = g.alpha_w;
  const int TH = T + alpha - 1;
  const int t = blockIdx.x;
  const int tu = t / g.ntv, tv = t - tu * g.ntv;
  const int s0 = b0 + blockIdx.y * bs;
  const int sb = min(bs, b0 + nb - s0);
  const int sbid = s0 / bs;                       // global sub-batch id (s0 is a multiple of bs)
  DegridRange range(ix.off + (int64_t)t * g.nw, g.nw, aw, s0, sb);
  if (range.used == 0) return;                    // no visibility of this tile meets these planes
  range.share(sb, least);
  const uint32_t lo = range.lo, hi = range.hi;
  if (lo == hi) return;
  degrid_rows(g, tu, tv, s0 - b0, sb, range.used,
              [&](int e, int64_t cell) { stage_copy(st + e, planes + cell); });
  for (int i = threadIdx.x; i < (g.deg + 1) * kMaxG; i += blockDim.x) sc[i] = coef.c[i];
  // the index entries of a group's next visibility are loaded while the current one is summed,
  // the first one's while the planes are staged
  const uint32_t gofs = (threadIdx.x / G) % (32 / G);
  uint32_t v0 = lo + (threadIdx.x >> 5) * (32 / G), mt_n = 0;
  Z4<R> zz_n;
  zz_n.u = zz_n.v = zz_n.w = zz_n.pad = (R)0;
  if (v0 + gofs < hi) { mt_n = ix.meta[v0 + gofs]; zz_n = ix.z[v0 + gofs]; }
  stage_wait();
  __syncthreads();
  // G lanes per visibility (lane j = piece / footprint column j).  Visibilities of a tile are
  // sorted by first plane, so the groups of a warp have nearly the same plane range: the plane
  // loop runs over the union of the warp's ranges (warp-uniform bounds, per-group predicate)
  // instead of all G candidate planes.
  const int j = threadIdx.x & (G - 1);
  LanePieceOf<R, G> pc;
  if (sizeof(R) == 4) pc.load(sc, g.deg, j);
  const int grp = threadIdx.x / G, ngrp = blockDim.x / G;
  const unsigned gmask = group_mask<G>();
  for (; v0 < hi; v0 += ngrp) {
    const uint32_t vi = v0 + gofs;
    const bool act = vi < hi;
    const uint32_t mt = act ? mt_n : 0u;
    const Z4<R> zz = zz_n;
    if (vi + ngrp < hi) { mt_n = ix.meta[vi + ngrp]; zz_n = ix.z[vi + ngrp]; }
    const int du = mt & 255, dv = (mt >> 8) & 255, c0 = (int)(mt >> 16);
    const bool lj = act && j < alpha;
    R pu = lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, 0, j, zz.u) : (R)0;
    R pv = lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, 1, j, zz.v) : (R)0;
    R pw = g.do_w ? (lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, 2, j, zz.w) : (R)0)
                  : (j == 0 ? (R)1 : (R)0);
    R wu[G];
#pragma unroll
    for (int i = 0; i < G; ++i) wu[i] = __shfl_sync(0xffffffffu, pu, i, G);
    const int qlo = act ? max(0, s0 - c0) : G, qhi = act ? min(aw, s0 + sb - c0) : 0;
    const int wlo = __reduce_min_sync(0xffffffffu, (unsigned)qlo);
    const int whi = __reduce_max_sync(0xffffffffu, (unsigned)qhi);
    R ar = (R)0, ai = (R)0;
    for (int q = wlo; q < whi; ++q) {
      const R wq = __shfl_sync(0xffffffffu, pw, q, G);
      if (lj && q >= qlo && q < qhi) {
        const CT* row = st + (c0 + q - s0) * TH * TH + du * TH + dv + j;
        R sr = (R)0, si = (R)0;
#pragma unroll
        for (int i = 0; i < G; ++i) {
          if (i < alpha) {
            CT gv = row[i * TH];
            sr = fma(wu[i], gv.x, sr);
            si = fma(wu[i], gv.y, si);
          }
        }
        ar = fma(wq, sr, ar);
        ai = fma(wq, si, ai);
      }
    }
    ar *= pv;
    ai *= pv;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      ar += __shfl_xor_sync(0xffffffffu, ar, o, G);
      ai += __shfl_xor_sync(0xffffffffu, ai, o, G);
    }
    if (act && j == 0) {
      const int slot = sbid - c0 / bs;
      CT o; o.x = ar; o.y = ai;
      partial[(int64_t)slot * nvis_idx + vi] = o;
    }
  }
}

// ---------------------------------------------------------------------------------------
// degrid of double-float planes (FP64 plans with the double-float FFT)
//
// The same decomposition as k_degrid, on planes whose cells are double-float pairs (float4:
// re hi, re lo, im hi, im lo): kernel values come as pairs (the kernel-value table stores them split), and the
// footprint sum runs in pair arithmetic on the FP32 pipes (15 instructions for an FP64 FMA, which GB300
// issues at 1/64 of the FP32 rate).  Two forms:
//  * packed (supports above 8, with w): real and imaginary part in one packed instruction, the staged cells
//    reordered in place to (re hi, im hi, re lo, im lo); each lane sums its column over rows, four planes
//    at once (independent chains; two: 8.5 against 8.3 ms), the u weights from shared memory (in
//    registers they leave room for two planes only: 9.9 ms).  1e6 visibilities on a 3456^2 grid, alpha = 15:
//    10.1 -> 8.6 ms, 4.2 of them with the sums left out.
//  * one plane at a time, unpacked, u weights in registers: without w there is one plane (1e6 visibilities on
//    1024 x 768, alpha = 14: 0.54 ms, packed 0.72), and 32-cell tiles leave two or three planes to a CTA, which
//    a group of four fills badly, and room for four CTAs per SM where the packed form's registers take three
//    (alpha = 7, 1e6 visibilities on 3072^2: 2.42 ms, packed 3.18).
// The lanes' sums are reduced by shuffles in pair arithmetic, and the partial sum is stored in FP64 as
// in k_degrid.
// ---------------------------------------------------------------------------------------
// piece j of direction d of indexed visibility vi as a double-float pair
__device__ __forceinline__ dd kernel_value_dd(const IndexView<double>& ix, const double* __restrict__ sc,
                                              int deg, uint32_t vi, int d, int j, double z) {
  if (ix.wts != nullptr) {
    const float2 p = reinterpret_cast<const float2*>(ix.wts)[(int64_t)vi * (3 * kMaxG) + d * kMaxG + j];
    return dd_make(p.x, p.y);
  }
  return split_double(horner(sc, deg, j, z));
}

__device__ __forceinline__ dd shfl_dd(dd x, int src, int width) {
  return dd_make(__shfl_sync(0xffffffffu, x.h, src, width), __shfl_sync(0xffffffffu, x.l, src, width));
}

// w d + c for a weight w given as (wh, wh), (-wh, -wh), (-wl, -wl): dd_fma(w, d, c) on packed values
__device__ __forceinline__ d2 d2_fma_weight(f2 wh, f2 nwh, f2 nwl, d2 d, d2 c) {
  const f2 p = s_mul(wh, d.h);
  f2 e = s_fma(nwh, d.h, p);   // minus all of the product below p
  e = s_fma(nwh, d.l, e);
  e = s_fma(nwl, d.h, e);
  const d2 s = d2_two_sum(c.h, p);
  return d2_fast_two_sum(s.h, s_add(s.l, s_sub(c.l, e)));
}

constexpr size_t kDegridWeights = kThreads * (sizeof(float4) + sizeof(float2));
// shared memory of k_degrid_dd beside the planes.  With a kernel-value table at most 76 KB in all for every
// support, so that an SM holds three CTAs
__host__ __device__ constexpr size_t degrid_dd_fixed(bool packed, bool table) {
  return (packed ? kDegridWeights : 0) + (packed && table ? 0 : (kMaxDeg + 1) * kMaxG * sizeof(double));
}

template <int G, bool kPacked>
__global__ void __launch_bounds__(kThreads, G == 16 ? 3 : 4)
k_degrid_dd(const Geom g, const __grid_constant__ Coef<double> coef, const IndexView<double> ix,
            const double2* __restrict__ planes, int b0, int nb, int bs,
            double2* __restrict__ partial, int64_t nvis_idx, uint32_t least) {
  extern __shared__ __align__(16) unsigned char smem[];
  // the coefficients where there is no kernel-value table, the planes, the groups' u weights (packed form)
  double* sc = reinterpret_cast<double*>(smem);
  double2* st = reinterpret_cast<double2*>(smem + degrid_dd_fixed(kPacked, ix.wts != nullptr) - (kPacked ? kDegridWeights : 0));
  const int T = g.tile, alpha = g.alpha, aw = g.alpha_w;
  const int TH = T + alpha - 1;
  const int t = blockIdx.x;
  const int tu = t / g.ntv, tv = t - tu * g.ntv;
  const int s0 = b0 + blockIdx.y * bs;
  const int sb = min(bs, b0 + nb - s0);
  const int sbid = s0 / bs;                       // global sub-batch id (s0 is a multiple of bs)
  DegridRange range(ix.off + (int64_t)t * g.nw, g.nw, aw, s0, sb);
  if (range.used == 0) return;                    // no visibility of this tile meets these planes
  range.share(sb, least);
  const uint32_t lo = range.lo, hi = range.hi;
  if (lo == hi) return;
  const int j = threadIdx.x & (G - 1);
  const int grp = threadIdx.x / G, ngrp = blockDim.x / G;
  const dd zero = dd_make(0.f, 0.f);
  [[maybe_unused]] float4* wt = reinterpret_cast<float4*>(st + (size_t)min(bs, nb) * TH * TH) + grp * G;
  [[maybe_unused]] float2* wt2 = reinterpret_cast<float2*>(wt + (ngrp - grp) * G) + grp * G;
  // with a kernel-value table, the group's next visibility's index entry and table values are
  // loaded while the current one is summed (the loads' latency is otherwise exposed), and the
  // first one's while the planes are staged
  const float2* tw = reinterpret_cast<const float2*>(ix.wts);
  const uint32_t gofs = grp % (32 / G);
  uint32_t mt_n = 0;
  float2 pu_n = make_float2(0.f, 0.f), pv_n = pu_n, pw_n = pu_n;
  auto prefetch = [&](uint32_t vi) {
    if (vi < hi) {
      mt_n = ix.meta[vi];
      if (tw != nullptr && j < alpha) {
        const int64_t b = (int64_t)vi * (3 * kMaxG) + j;
        pu_n = tw[b]; pv_n = tw[b + kMaxG]; pw_n = tw[b + 2 * kMaxG];
      }
    }
  };
  uint32_t v0 = lo + (threadIdx.x >> 5) * (32 / G);
  prefetch(v0 + gofs);
  if (tw == nullptr)
    for (int i = threadIdx.x; i < (g.deg + 1) * kMaxG; i += blockDim.x) sc[i] = coef.c[i];
  degrid_rows(g, tu, tv, s0 - b0, sb, range.used,
              [&](int e, int64_t cell) { stage_copy(st + e, planes + cell); });
  stage_wait();
  if constexpr (kPacked) {
    // (re hi, re lo, im hi, im lo) to (re hi, im hi, re lo, im lo): each thread the cells it copied
    degrid_rows(g, tu, tv, s0 - b0, sb, range.used, [&](int e, int64_t) {
      float4* v = reinterpret_cast<float4*>(st) + e;
      const float2 m = make_float2(v->y, v->z);
      v->y = m.y;
      v->z = m.x;
    });
  }
  __syncthreads();
  for (; v0 < hi; v0 += ngrp) {
    const uint32_t vi = v0 + gofs;
    const bool act = vi < hi;
    const uint32_t mt = act ? mt_n : 0u;
    const float2 tu = pu_n, tv = pv_n, tww = pw_n;
    prefetch(v0 + ngrp + gofs);
    Z4<double> zz;
    zz.u = zz.v = zz.w = zz.pad = 0.0;
    if (act && tw == nullptr) zz = ix.z[vi];
    const int du = mt & 255, dv = (mt >> 8) & 255, c0 = (int)(mt >> 16);
    const bool lj = act && j < alpha;
    dd pu = zero, pv = zero, pw = zero;
    if (lj) {
      if (tw != nullptr) {
        pu = dd_make(tu.x, tu.y); pv = dd_make(tv.x, tv.y); pw = dd_make(tww.x, tww.y);
      } else {
        pu = kernel_value_dd(ix, sc, g.deg, vi, 0, j, zz.u);
        pv = kernel_value_dd(ix, sc, g.deg, vi, 1, j, zz.v);
        pw = kernel_value_dd(ix, sc, g.deg, vi, 2, j, zz.w);
      }
    }
    if (!g.do_w) pw = j == 0 ? dd_make(1.f, 0.f) : zero;
    const int qlo = act ? max(0, s0 - c0) : G, qhi = act ? min(aw, s0 + sb - c0) : 0;
    const int wlo = __reduce_min_sync(0xffffffffu, (unsigned)qlo);
    const int whi = __reduce_max_sync(0xffffffffu, (unsigned)qhi);
    dd ar = zero, ai = zero;
    if constexpr (kPacked) {
      __syncwarp();   // the previous visibility's weights are consumed
      wt[j] = make_float4(-pu.h, -pu.h, -pu.l, -pu.l);
      wt2[j] = make_float2(pu.h, pu.h);
      __syncwarp();
      const int cell = du * TH + dv + (lj ? j : 0);
      d2 acc{f2_make(0.f, 0.f), f2_make(0.f, 0.f)};   // (re, im)
      // NP planes from q on at once: their column sums are independent chains
      auto planes_sum = [&](int q, auto np) {
        constexpr int NP = decltype(np)::value;
        const ulonglong2* row[NP];
        bool on[NP];
        d2 sum[NP];
#pragma unroll
        for (int n = 0; n < NP; ++n) {
          on[n] = lj && q + n >= qlo && q + n < qhi;
          const int pl = on[n] ? c0 + q + n - s0 : 0;
          row[n] = reinterpret_cast<const ulonglong2*>(st) + pl * TH * TH + cell;
          sum[n].h = sum[n].l = f2_make(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
          if (i < alpha) {
            const ulonglong2 nw = *reinterpret_cast<const ulonglong2*>(&wt[i]);
            const f2 wh{*reinterpret_cast<const pk64*>(&wt2[i])}, nwh{nw.x}, nwl{nw.y};
#pragma unroll
            for (int n = 0; n < NP; ++n) {
              const ulonglong2 v = row[n][i * TH];
              sum[n] = d2_fma_weight(wh, nwh, nwl, d2{f2{v.x}, f2{v.y}}, sum[n]);
            }
          }
        }
#pragma unroll
        for (int n = 0; n < NP; ++n) {
          const dd wq = shfl_dd(pw, q + n, G);
          // a plane the visibility does not meet (or a lane past its columns) gave what it read
          if (!on[n]) sum[n].h = sum[n].l = f2_make(0.f, 0.f);
          acc = d2_fma_weight(f2_make(wq.h, wq.h), f2_make(-wq.h, -wq.h), f2_make(-wq.l, -wq.l), sum[n], acc);
        }
      };
      int q = wlo;
      for (; q + 2 < whi; q += 4) planes_sum(q, std::integral_constant<int, 4>());
      if (q < whi) planes_sum(q, std::integral_constant<int, 2>());
      const float2 ach = f2_split(acc.h), acl = f2_split(acc.l);
      ar = dd_make(ach.x, acl.x);
      ai = dd_make(ach.y, acl.y);
    } else {
      dd wu[G];
#pragma unroll
      for (int i = 0; i < G; ++i) wu[i] = shfl_dd(pu, i, G);
      for (int q = wlo; q < whi; ++q) {
        const dd wq = shfl_dd(pw, q, G);
        if (lj && q >= qlo && q < qhi) {
          const float4* row = reinterpret_cast<const float4*>(st + (c0 + q - s0) * TH * TH + du * TH + dv + j);
          dd sr = zero, si = zero;
#pragma unroll
          for (int i = 0; i < G; ++i) {
            if (i < alpha) {
              const float4 gv = row[i * TH];
              sr = dd_fma(wu[i], dd_make(gv.x, gv.y), sr);
              si = dd_fma(wu[i], dd_make(gv.z, gv.w), si);
            }
          }
          ar = dd_fma(wq, sr, ar);
          ai = dd_fma(wq, si, ai);
        }
      }
    }
    ar = dd_mul(ar, pv);
    ai = dd_mul(ai, pv);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      ar = dd_add(ar, dd_make(__shfl_xor_sync(0xffffffffu, ar.h, o, G), __shfl_xor_sync(0xffffffffu, ar.l, o, G)));
      ai = dd_add(ai, dd_make(__shfl_xor_sync(0xffffffffu, ai.h, o, G), __shfl_xor_sync(0xffffffffu, ai.l, o, G)));
    }
    if (act && j == 0) {
      const int slot = sbid - c0 / bs;
      partial[(int64_t)slot * nvis_idx + vi] = make_double2(join_double(ar), join_double(ai));
    }
  }
}

// vis[k] = wgt_k * fold(e^{2 pi i w_k nshift} * sum of the visibility's partial-sum slots)
template <typename R>
__global__ void k_degrid_finalize(const Geom g, const IndexView<R> ix,
                                  const typename C2<R>::T* __restrict__ partial, int64_t nvis_idx,
                                  int bs, const R* __restrict__ wgt,
                                  typename C2<R>::T* __restrict__ vis) {
  using CT = typename C2<R>::T;
  const int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (pos >= nvis_idx) return;
  const uint32_t id = ix.idx[pos];
  const int c0 = (int)(ix.meta[pos] >> 16);
  const int nsl = (c0 + g.alpha_w - 1) / bs - c0 / bs + 1;
  R ar = (R)0, ai = (R)0;
  for (int sl = 0; sl < nsl; ++sl) {
    CT v = partial[(int64_t)sl * nvis_idx + pos];
    ar += v.x; ai += v.y;
  }
  if (ix.ph != nullptr) {  // exp(2 pi i w nshift) times the gridded sum
    CT ph = ix.ph[pos];
    R r = ar * ph.x - ai * ph.y;
    ai = ar * ph.y + ai * ph.x;
    ar = r;
  }
  if (id & kFoldBit) ai = -ai;  // Hermitian fold undone: d = conj(d')
  const int64_t k = id & ~kFoldBit;
  if (wgt != nullptr) { R w = wgt[k]; ar *= w; ai *= w; }
  CT o; o.x = ar; o.y = ai;
  vis[k] = o;
}

// ---------------------------------------------------------------------------------------
// grid, plane-owner variant (FP64 planes of plans with cuFFT; FP32 on request)
//
// CTA = (uv tile, sub-batch of bs planes).  Warp w owns planes w, w + 8, ... of the
// sub-batch: it alone updates their T x T accumulators, so the updates are plain shared-memory
// read-modify-writes (no atomics, deterministic order).  Visibilities are handled in chunks:
// first a group of G lanes per visibility stages its kernel values in u and v (Sec. 4.2) and
// its data times the w kernel value of each of its planes; then each warp walks the chunk and,
// for every visibility touching one of its planes, spreads the 32 lanes over the cells of the
// footprint that fall inside the tile (the clipped footprint, row-major) and adds their
// staged 2-D weights wu * wv times the visibility's plane-weighted data into each of its planes
// the visibility touches.  The 2-D weights are formed once per visibility in phase 1 (by the
// visibility's lane group, exchanging its u and v values by shuffles), not once per warp.
// ---------------------------------------------------------------------------------------
// visibilities staged per chunk: the staged 2-D weights of a chunk take kChunk x G^2 values
template <int G>
struct OwnerChunk {
  static constexpr int value = G > 8 ? 12 : 48;
};
// plane-owner gridding CTA: 8 warps (4 warps with 4 planes each measured 10 % slower: fewer
// warps to hide the shared-memory latency of the updates)
constexpr int kOwnerThreads = 256;
constexpr int kOwnerWarps = kOwnerThreads / 32;   // warp w owns planes w, w + kOwnerWarps, ...

template <typename R, int G>
struct GridStage {
  static constexpr int kChunk = OwnerChunk<G>::value;
  R wt[kChunk][G * G];                  // wu_i * wv_j of the clipped footprint cells, row-major
  typename C2<R>::T dq[kChunk][G];      // data x w kernel value of plane q of the visibility
  int ru[kChunk], rv[kChunk], c0[kChunk];
};

// The part of a visibility's footprint inside the tile: rows i0.., columns j0..j0 + w - 1 of
// the footprint, `cells` cells in all, footprint origin at tile cell (ru, rv).
struct OwnerFootprint {
  int i0, j0, w, cells, ru, rv;
};

// Add visibility v of the chunk into the warp's planes p1, p1 + kOwnerWarps, .. < phi: lane
// takes cells lane + 32 m (m < MC) of the clipped footprint in row-major order, loads their
// staged 2-D weights and updates each plane (plane pl uses the staged data x w value of the
// visibility's plane pl + qoff).  Lanes past the last cell update a private cell of the row
// padding (columns T, T + 1) with weight 0, so every update is unconditional.
template <typename R, int G, int MC>
__device__ __forceinline__ void owner_add(const GridStage<R, G>* __restrict__ stg, int v,
                                          const OwnerFootprint& fp, int lane, int T, int pitch,
                                          int p1, int phi, int qoff,
                                          typename C2<R>::T* __restrict__ acc, int plane_elems) {
  using CT = typename C2<R>::T;
  const float rw = 1.0f / (float)fp.w;
  const int dummy = (lane >> 1) * pitch + T + (lane & 1);
  R wt[MC];
  int off[MC];
#pragma unroll
  for (int m = 0; m < MC; ++m) {
    const int c = lane + 32 * m;
    // c = ii * w + jj; exact in float: c < 256 and w <= 16 keep (c + 0.5) / w at least 1 / 32
    // away from an integer
    const int ii = (int)(((float)c + 0.5f) * rw), jj = c - ii * fp.w;
    const bool ok = c < fp.cells;
    const int i = fp.i0 + (ok ? ii : 0), j = fp.j0 + (ok ? jj : 0);
    wt[m] = ok ? stg->wt[v][c] : (R)0;
    off[m] = ok ? (fp.ru + i) * pitch + fp.rv + j : dummy;
  }
  // loads, arithmetic and stores in separate sweeps: the cells of one lane are distinct, but the compiler
  // cannot see that, and interleaved loads and stores would serialise the MC update chains
  for (int pl = p1; pl < phi; pl += kOwnerWarps) {
    const CT dq = stg->dq[v][pl + qoff];
    CT* base = acc + pl * plane_elems;
    CT a[MC];
#pragma unroll
    for (int m = 0; m < MC; ++m) a[m] = base[off[m]];
#pragma unroll
    for (int m = 0; m < MC; ++m) {
      a[m].x = fma(dq.x, wt[m], a[m].x);
      a[m].y = fma(dq.y, wt[m], a[m].y);
    }
#pragma unroll
    for (int m = 0; m < MC; ++m) base[off[m]] = a[m];
  }
}

template <typename R, int G>
__global__ void __launch_bounds__(kOwnerThreads)
k_grid_owner(const Geom g, const __grid_constant__ Coef<R> coef, const IndexView<R> ix,
       const typename C2<R>::T* __restrict__ vis, const R* __restrict__ wgt,
       typename C2<R>::T* __restrict__ planes, int b0, int nb, int bs, int pitch) {
  using CT = typename C2<R>::T;
  extern __shared__ __align__(16) unsigned char smem[];
  R* sc = reinterpret_cast<R*>(smem);
  using Stage = GridStage<R, G>;
  constexpr int kChunk = Stage::kChunk;
  Stage* stg = reinterpret_cast<Stage*>(smem + (kMaxDeg + 1) * kMaxG * sizeof(R));
  CT* acc = reinterpret_cast<CT*>(reinterpret_cast<unsigned char*>(stg) + sizeof(Stage));
  const int T = g.tile, alpha = g.alpha, aw = g.alpha_w;
  const int t = blockIdx.x;
  const int tu = t / g.ntv, tv = t - tu * g.ntv;
  const int s0 = b0 + blockIdx.y * bs;
  const int sb = min(bs, b0 + nb - s0);
  const int plane_elems = T * pitch;
  for (int i = threadIdx.x; i < (g.deg + 1) * kMaxG; i += blockDim.x) sc[i] = coef.c[i];
  for (int e = threadIdx.x; e < sb * plane_elems; e += blockDim.x) {
    CT z; z.x = (R)0; z.y = (R)0;
    acc[e] = z;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // phase-1 mapping: groups of G lanes, one visibility each
  const int j1 = threadIdx.x & (G - 1), grp = threadIdx.x / G, ngrp = blockDim.x / G;
  const unsigned gmask = group_mask<G>();
  __syncthreads();   // coefficients staged
  LanePieceOf<R, G> pc;
  if (sizeof(R) == 4) pc.load(sc, g.deg, j1);

  for (int src = 0; src < 4; ++src) {
    const int ou = (src & 1) ? -1 : 0, ov = (src & 2) ? -1 : 0;
    int stu = tu + ou; if (stu < 0) stu += g.ntu;
    int stv = tv + ov; if (stv < 0) stv += g.ntv;
    const uint32_t* offs = ix.off + ((int64_t)stu * g.ntv + stv) * g.nw;
    const uint32_t lo = offs[max(0, s0 - aw + 1)], hi = offs[min(g.nw, s0 + sb)];
    for (uint32_t cs = lo; cs < hi; cs += kChunk) {
      const int nch = (int)min((uint32_t)kChunk, hi - cs);
      __syncthreads();  // previous chunk consumed (and accumulators zeroed)
      // ---- phase 1: kernel values and plane-weighted data of the chunk ----
      for (int v = grp; v < nch; v += ngrp) {
        const uint32_t vi = cs + v;
        const uint32_t mt = ix.meta[vi];
        const int ru = (int)(mt & 255) + ou * T, rv = (int)((mt >> 8) & 255) + ov * T;
        const bool hit = (ru + alpha > 0) && (rv + alpha > 0);
        if (j1 == 0) {
          stg->ru[v] = ru; stg->rv[v] = rv;
          stg->c0[v] = hit ? (int)(mt >> 16) : -(1 << 20);
        }
        if (!hit) continue;   // uniform within the group
        const Z4<R> zz = ix.z[vi];
        const bool lj = j1 < alpha;
        const R pu = lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, 0, j1, zz.u) : (R)0;
        const R pv = lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, 1, j1, zz.v) : (R)0;
        // 2-D weights of the footprint cells inside the tile (rows i0.., columns j0..j0+w-1),
        // row-major: lane j1 forms cells j1, j1 + G, ... from the group's u and v values
        {
          const int i0 = max(0, -ru), i1 = min(alpha, T - ru);
          const int j0 = max(0, -rv), w = min(alpha, T - rv) - j0;
          const int cells = (i1 - i0) * w;
          const float rw = 1.0f / (float)w;
          const int nt = (cells + G - 1) / G;   // same trip count for the whole group
          for (int tq = 0; tq < nt; ++tq) {
            const int c = j1 + G * tq;
            // exact in float: c < 256 and w <= 16 keep (c + 0.5) / w at least 1 / 32 away
            // from an integer
            const int ii = (int)(((float)c + 0.5f) * rw), jj = c - ii * w;
            const bool ok = c < cells;
            const R a = __shfl_sync(gmask, pu, ok ? i0 + ii : 0, G);
            const R b = __shfl_sync(gmask, pv, ok ? j0 + jj : 0, G);
            if (ok) stg->wt[v][c] = a * b;
          }
        }
        const R wwj = g.do_w ? (lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, 2, j1, zz.w) : (R)0)
                             : (j1 == 0 ? (R)1 : (R)0);
        R dr = (R)0, di = (R)0;
        if (j1 == 0) {
          const uint32_t id = ix.idx[vi];
          const int64_t k = id & ~kFoldBit;
          CT d = vis[k];
          dr = d.x; di = d.y;
          if (wgt != nullptr) { R w = wgt[k]; dr *= w; di *= w; }
          if (id & kFoldBit) di = -di;      // grid conj(d) at the folded coordinates
          if (ix.ph != nullptr) {           // times conj(exp(2 pi i w nshift))
            CT ph = ix.ph[vi];
            R r = dr * ph.x + di * ph.y;
            di = di * ph.x - dr * ph.y;
            dr = r;
          }
        }
        dr = __shfl_sync(gmask, dr, 0, G);
        di = __shfl_sync(gmask, di, 0, G);
        CT o; o.x = dr * wwj; o.y = di * wwj;
        stg->dq[v][j1] = o;
      }
      __syncthreads();
      // ---- phase 2: each warp adds the chunk into its own planes ----
      for (int v = 0; v < nch; ++v) {
        const int c0 = stg->c0[v];
        if (c0 < -1000) continue;
        // this warp's planes among the visibility's planes c0 .. c0 + aw - 1
        const int plo = max(0, c0 - s0), phi = min(sb, c0 - s0 + aw);
        const int p1 = plo + ((warp - plo) & (kOwnerWarps - 1));
        if (p1 >= phi) continue;
        const int ru = stg->ru[v], rv = stg->rv[v];
        // footprint rows i0..i1-1 and columns j0..j1-1 inside the tile
        const int i0 = max(0, -ru), i1 = min(alpha, T - ru);
        const int j0 = max(0, -rv), j1c = min(alpha, T - rv);
        const int w = j1c - j0, cells = (i1 - i0) * w;
        // dispatch on the warp-uniform number of cells per lane, so that each case runs
        // exactly its updates (no predicated-off FP64 instructions)
        const OwnerFootprint fp{i0, j0, w, cells, ru, rv};
        switch ((cells + 31) >> 5) {
          case 1: owner_add<R, G, 1>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
          case 2: owner_add<R, G, 2>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
          case 3: owner_add<R, G, (G > 8 ? 3 : 1)>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
          case 4: owner_add<R, G, (G > 8 ? 4 : 1)>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
          case 5: owner_add<R, G, (G > 8 ? 5 : 1)>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
          case 6: owner_add<R, G, (G > 8 ? 6 : 1)>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
          case 7: owner_add<R, G, (G > 8 ? 7 : 1)>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
          default: owner_add<R, G, (G > 8 ? 8 : 1)>(stg, v, fp, lane, T, pitch, p1, phi, s0 - c0, acc, plane_elems); break;
        }
      }
    }
  }
  __syncthreads();
  const int64_t pstride = (int64_t)g.nu * g.nv;
  for (int e = threadIdx.x; e < sb * T * T; e += blockDim.x) {
    const int pl = e / (T * T), rem = e - pl * T * T;
    const int r = rem / T, c = rem - r * T;
    planes[(int64_t)(s0 - b0 + pl) * pstride + (int64_t)(tu * T + r) * g.nv + tv * T + c] =
        acc[pl * plane_elems + r * pitch + c];
  }
}

// ---------------------------------------------------------------------------------------
// per-call visibility data for the pair-arithmetic gridding: position pos of the index gets
// wgt_k * d_k, conjugated where the visibility was folded (Hermitian symmetry), times
// conj(e^{2 pi i w nshift}) (the w reference shift), as double-float pairs -- the FP64 work that
// the gridding kernel would otherwise repeat on every (tile, sub-batch) visit
// ---------------------------------------------------------------------------------------
__global__ void k_grid_vis_dd(const IndexView<double> ix, const double2* __restrict__ vis,
                              const double* __restrict__ wgt, int64_t nvis_idx,
                              float4* __restrict__ out) {
  const int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (pos >= nvis_idx) return;
  const uint32_t id = ix.idx[pos];
  const int64_t k = id & ~kFoldBit;
  const double2 d = vis[k];
  double xr = d.x, xi = d.y;
  if (wgt != nullptr) { const double w = wgt[k]; xr *= w; xi *= w; }
  if (id & kFoldBit) xi = -xi;      // grid conj(d) at the folded coordinates
  if (ix.ph != nullptr) {           // times conj(exp(2 pi i w nshift))
    const double2 ph = ix.ph[pos];
    const double r = xr * ph.x + xi * ph.y;
    xi = xi * ph.x - xr * ph.y;
    xr = r;
  }
  const dd a = split_double(xr), b = split_double(xi);
  out[pos] = make_float4(a.h, a.l, b.h, b.l);
}

cudaError_t launch_grid_vis_dd(const IndexView<double>& ix, const double2* vis, const double* wgt,
                               int64_t nvis_idx, float4* out, cudaStream_t s) {
  if (nvis_idx == 0) return cudaSuccess;
  k_grid_vis_dd<<<(unsigned)((nvis_idx + 255) / 256), 256, 0, s>>>(ix, vis, wgt, nvis_idx, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// grid of double-float planes (FP64 plans with the double-float FFT): accumulators in registers
//
// CTA = (rows x cols cells of a uv tile, 8 planes).  A half-warp owns 4 x 4 cells and a lane one
// cell in all 8 planes, its sums in registers as double-float pairs with the real and the imaginary
// part packed: a cell's update in pair arithmetic is 15 packed FP32 instructions, with nothing
// read from or written to shared memory but the staged visibility (the plane-owner scheme with
// pairs in shared memory spent half its issue slots on those).  Visibilities of the tile, and of
// the tiles whose footprints reach into the cells, form one list, staged in chunks: kernel values
// in u and v, and data times w kernel value by plane (zero in the planes a visibility does not
// meet).  Each half-warp walks its own bit mask of the chunk's visibilities that meet its 4 x 4
// cells (alpha = 15: 69 % of its lanes are inside the footprint, against 57 % for 4 x 8 cells of a
// whole warp), updating planes two at a time where a visibility of either half meets them.
// Cells are updated in index order: deterministic.
//
// Bound by the FP32 pipe (53 % active) and, of the rest, by warps waiting for the one with the most
// visibilities of a chunk.  16 planes per lane (118 registers, 2 CTAs per SM) measured 13.3 ms where
// 8 planes take 11.4, and whole-warp 4 x 8 cells 11.4 where half-warps take 10.6 (3456^2 grid, 1e6
// visibilities, alpha = 15; the plane-owner kernel 19.6).
//
// Shapes, by template (W warps x SPLIT, PG planes):
//  * <8, 1, 8>: 16 x 16 cells, every warp walks the whole chunk.
//  * <2, 4, 8>: 8 x 8 cells, four sets of two warps, each taking every fourth visibility, their sums
//    added in order at the end: for plans whose densest tile would be the run time.
//  * <8, 1, 2>: the first with two planes, for grids without w: 40 registers, six CTAs per SM (2560^2, 20 000
//    visibilities, alpha = 6: 104 us with eight planes, 78 with two, the plane-owner kernel 82).
constexpr int kCellsPlanes = 8;
template <int W>
struct CellsTile {   // cells and visibilities per set of a CTA
  static constexpr int rows = W == 8 ? 16 : 8, cols = W >= 4 ? 16 : 8;
  static constexpr int vis = W == 8 ? 64 : 32;
};
template <int W, int SPLIT, int PG>
struct CellsStage {
  static constexpr int kChunk = CellsTile<W>::vis * SPLIT;
  // row kChunk: no visibility
  float2 wu[kChunk + 1][kMaxG], wv[kChunk + 1][kMaxG];   // kernel values as pairs
  float4 dq[kChunk + 1][PG + 1];   // data x w kernel value by plane: re hi, im hi, re lo, im lo
  int head[kChunk + 1];   // footprint origin (row + 64, column + 64 << 8), plane pairs met << 16; or 0
  int cum[4], first[4];   // visibilities before each source tile; index position minus that
};

template <int W, int SPLIT, int PG>
__global__ void __launch_bounds__(32 * W * SPLIT, (PG == 2 ? 48 : 32) / (W * SPLIT))
k_grid_cells_dd(const Geom g, const __grid_constant__ Coef<double> coef, const IndexView<double> ix,
                const float4* __restrict__ vis, float4* __restrict__ planes, int b0, int nb) {
  extern __shared__ __align__(16) unsigned char smem[];
  double* sc = reinterpret_cast<double*>(smem);
  using Stage = CellsStage<W, SPLIT, PG>;
  Stage& sm = *reinterpret_cast<Stage*>(smem + (kMaxDeg + 1) * kMaxG * sizeof(double));
  constexpr int TR = CellsTile<W>::rows, TC = CellsTile<W>::cols, G = 16, N = 32 * W;
  const int alpha = g.alpha, aw = g.alpha_w;
  const int nqv = g.nv / TC, nqu = g.nu / TR, peru = g.tile / TR, perv = g.tile / TC;
  const int tr = blockIdx.x / nqv, qv = blockIdx.x - tr * nqv;
  // rows from both ends of the grid towards its middle: short baselines, the densest rows, lie at
  // the ends (row 0 and, wrapped, the last) and start first
  const int qu = (tr & 1) ? nqu - 1 - tr / 2 : tr / 2;
  const int tu = qu / peru, tv = qv / perv, su = (qu - tu * peru) * TR, sv = (qv - tv * perv) * TC;
  const int s0 = b0 + blockIdx.y * PG;
  const int sb = min(PG, b0 + nb - s0);
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) % W;
  const int set = SPLIT > 1 ? threadIdx.x / N : 0;   // takes every SPLIT-th visibility from here
  const int row0 = warp / (TC / 8) * 4, col0 = warp % (TC / 8) * 8;
  const int row = row0 + ((lane >> 2) & 3), col = col0 + ((lane >> 4) << 2) + (lane & 3);
  if (ix.wts == nullptr)
    for (int i = threadIdx.x; i < (g.deg + 1) * kMaxG; i += blockDim.x) sc[i] = coef.c[i];
  if (threadIdx.x < 32) {
    // the square's tile and, where the square lies on its edge, the three whose footprints reach in
    const int ou = lane & 1, ov = (lane >> 1) & 1;
    uint32_t lo = 0, n = 0;
    if (lane < 4 && !(ou && su >= alpha) && !(ov && sv >= alpha)) {
      int stu = tu - ou; if (stu < 0) stu += g.ntu;
      int stv = tv - ov; if (stv < 0) stv += g.ntv;
      const uint32_t* offs = ix.off + ((int64_t)stu * g.ntv + stv) * g.nw;
      lo = offs[max(0, s0 - aw + 1)];
      n = offs[min(g.nw, s0 + sb)] - lo;
    }
    uint32_t c = n;
    for (int o = 1; o < 4; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, c, o);
      if (lane >= o) c += up;
    }
    if (lane < 4) { sm.cum[lane] = (int)c; sm.first[lane] = (int)(lo - (c - n)); }
  }
  if (threadIdx.x < PG) sm.dq[Stage::kChunk][threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (threadIdx.x == 0) sm.head[Stage::kChunk] = 0;
  f2 ah[PG], al[PG];   // this lane's cell: (re, im) high parts, low parts
#pragma unroll
  for (int p = 0; p < PG; ++p) ah[p] = al[p] = f2_make(0.f, 0.f);
  __syncthreads();
  const int total = sm.cum[3];

  for (int cs = 0; cs < total; cs += Stage::kChunk) {
    if (cs) __syncthreads();   // previous chunk consumed
    {
      const int j1 = threadIdx.x & (G - 1);
      const unsigned gmask = group_mask<G>();
      const int nch = min(Stage::kChunk, total - cs);
      for (int v = threadIdx.x / G; v < nch; v += N * SPLIT / G) {
        const int k = cs + v;
        const int src = (k >= sm.cum[0]) + (k >= sm.cum[1]) + (k >= sm.cum[2]);
        const uint32_t vi = (uint32_t)sm.first[src] + (uint32_t)k;
        const uint32_t mt = ix.meta[vi];
        const float2* tw = reinterpret_cast<const float2*>(ix.wts);
        float2 pu = make_float2(0.f, 0.f), pv = pu, pw = pu;
        if (tw != nullptr) {   // the table holds zeros beyond alpha
          const int64_t b = (int64_t)vi * (3 * kMaxG) + j1;
          pu = tw[b]; pv = tw[b + kMaxG]; pw = tw[b + 2 * kMaxG];
        }
        const float4 d = vis[vi];
        const int ru = (int)(mt & 255) - (src & 1) * g.tile - su;
        const int rv = (int)((mt >> 8) & 255) - (src >> 1) * g.tile - sv;
        const bool hit = ru < TR && ru + alpha > 0 && rv < TC && rv + alpha > 0;
        const int plo = (int)(mt >> 16) - s0;   // first plane of the visibility, in the CTA's
        if (j1 == 0) {
          int m = 0;
#pragma unroll
          for (int q = 0; q < PG / 2; ++q)
            if (2 * q + 2 > plo && 2 * q < plo + aw) m |= 1 << q;
          sm.head[v] = hit ? (ru + 64) | (rv + 64) << 8 | m << 16 : 0;
        }
        if (!hit) continue;   // uniform within the group
        if (tw == nullptr && j1 < alpha) {
          const Z4<double> zz = ix.z[vi];
          const dd a = split_double(horner(sc, g.deg, j1, zz.u)), b = split_double(horner(sc, g.deg, j1, zz.v));
          const dd c = split_double(horner(sc, g.deg, j1, zz.w));
          pu = make_float2(a.h, a.l); pv = make_float2(b.h, b.l); pw = make_float2(c.h, c.l);
        }
        sm.wu[v][j1] = pu;
        sm.wv[v][j1] = pv;
        if (!g.do_w) pw = j1 == 0 ? make_float2(1.f, 0.f) : make_float2(0.f, 0.f);
        // lane p of the group takes plane s0 + p, the visibility's plane q = p - plo
        const int q = j1 - plo;
        const dd w = dd_make(__shfl_sync(gmask, pw.x, q & (G - 1), G), __shfl_sync(gmask, pw.y, q & (G - 1), G));
        if (j1 < PG) {
          const bool on = q >= 0 && q < aw;
          const dd qr = dd_mul(dd_make(d.x, d.y), w), qi = dd_mul(dd_make(d.z, d.w), w);
          sm.dq[v][j1] = on ? make_float4(qr.h, qi.h, qr.l, qi.l) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
    __syncthreads();
    // the visibilities whose footprints meet each half-warp's cells, as bit masks
    uint64_t mA = 0, mB = 0;
#pragma unroll
    for (int r = 0; r < CellsTile<W>::vis / 32; ++r) {
      const int v = SPLIT * (32 * r + lane) + set;
      const int h = cs + v < total ? sm.head[v] : 0;
      const int ru = (h & 255) - 64, rv = ((h >> 8) & 255) - 64;
      const bool rows = ru < row0 + 4 && ru + alpha > row0;
      const bool a = rows && rv < col0 + 4 && rv + alpha > col0;
      const bool b = rows && rv < col0 + 8 && rv + alpha > col0 + 4;
      mA |= (uint64_t)__ballot_sync(0xffffffffu, a) << (32 * r);
      mB |= (uint64_t)__ballot_sync(0xffffffffu, b) << (32 * r);
    }
    const int n = max(__popcll(mA), __popcll(mB));
    uint64_t m = lane < 16 ? mA : mB;
    for (int k = 0; k < n; ++k) {
      const int v = m ? SPLIT * (__ffsll((long long)m) - 1) + set : Stage::kChunk;
      m &= m - 1;
      const int h = sm.head[v];
      const int i = row + 64 - (h & 255), j = col + 64 - ((h >> 8) & 255);
      const bool in = (unsigned)i < (unsigned)alpha && (unsigned)j < (unsigned)alpha;
      const float2 a = sm.wu[v][in ? i : 0], b = sm.wv[v][in ? j : 0];
      const dd w = dd_mul(dd_make(a.x, a.y), dd_make(b.x, b.y));
      const float wh = in ? w.h : 0.f, wl = in ? w.l : 0.f;
      const f2 wh2 = f2_make(wh, wh), nwh = f2_make(-wh, -wh), nwl = f2_make(-wl, -wl);
      const unsigned met = __reduce_or_sync(0xffffffffu, (unsigned)h >> 16);
#pragma unroll
      for (int q = 0; q < PG / 2; ++q) {
        if (!(met & (1u << q))) continue;
#pragma unroll
        for (int p = 2 * q; p < 2 * q + 2; ++p) {
          const ulonglong2 dv = *reinterpret_cast<const ulonglong2*>(&sm.dq[v][p]);
          const f2 dh{dv.x}, dl{dv.y};
          // ah + al += d w: pr the rounded product of the high parts, e minus all below it
          const f2 pr = s_mul(dh, wh2);
          f2 e = s_fma(dh, nwh, pr);
          e = s_fma(dh, nwl, e);
          e = s_fma(dl, nwh, e);
          const d2 s = d2_two_sum(ah[p], pr);
          const d2 r = d2_fast_two_sum(s.h, s_add(s.l, s_sub(al[p], e)));
          ah[p] = r.h;
          al[p] = r.l;
        }
      }
    }
  }
  if constexpr (SPLIT > 1) {   // the sets' sums, in order
    __syncthreads();
    static_assert(sizeof(Stage) >= (SPLIT - 1) * PG * N * sizeof(ulonglong2), "partial sums fit the stage");
    ulonglong2* part = reinterpret_cast<ulonglong2*>(&sm);
    const int c = threadIdx.x % N;
    if (set)
#pragma unroll
      for (int p = 0; p < PG; ++p) part[((set - 1) * PG + p) * N + c] = make_ulonglong2(ah[p].v, al[p].v);
    __syncthreads();
    if (set) return;
    for (int o = 0; o < SPLIT - 1; ++o)
#pragma unroll
      for (int p = 0; p < PG; ++p) {
        const ulonglong2 x = part[(o * PG + p) * N + c];
        const d2 r = s_add(d2{ah[p], al[p]}, d2{f2{x.x}, f2{x.y}});
        ah[p] = r.h;
        al[p] = r.l;
      }
  }
  const int64_t pstride = (int64_t)g.nu * g.nv;
  float4* out = planes + (int64_t)(s0 - b0) * pstride + (int64_t)(qu * TR + row) * g.nv + qv * TC + col;
#pragma unroll
  for (int p = 0; p < PG; ++p) {
    if (p >= sb) break;
    const float2 h = f2_split(ah[p]), l = f2_split(al[p]);
    out[p * pstride] = make_float4(h.x, l.x, h.y, l.y);
  }
}

// ---------------------------------------------------------------------------------------
// grid, shared-atomic variant (FP32 plans that do not take the tensor cores, see grid_variant_of)
//
// CTA = (uv tile, sub-batch of planes), owning the T x T cells of those planes as separate real
// and imaginary accumulators in shared memory.  A warp handles one visibility at a time: lane
// (j, rg) = (lane mod G, lane / G) takes footprint column j and rows rg, rg + 32 / G, ...;
// with the accumulator row pitch = G (mod 32), the 32 lanes of every atomic add hit 32
// different banks.  Kernel values (Sec. 4.2): each lane evaluates piece j in u (rg = 0) or v
// (rg > 0) and in w, and the warp exchanges them by shuffles.  Warps run concurrently, so cells
// shared by overlapping footprints are combined by the atomics (summation order not fixed).
// ---------------------------------------------------------------------------------------
// Shared memory per gridding CTA, 54 KB: four gridding CTAs per SM (with the kernel held to 64 registers).  The kernel is
// latency-bound (the atomics' read-modify-write); measured on the 1e8-visibility FP32 workload:
// two CTAs per SM (110 KB) 244 ms, three (72 KB) 197-263 ms, four 175 ms
constexpr size_t kGridAtomicSmemBudget = 54 * 1024;
constexpr int kGridAtomicMinBlocks = 4;

// shared-memory atomic add without a returned value (PTX red; 2 % faster than atomicAdd on the
// 1e8-visibility FP32 gridding)
__device__ __forceinline__ void red_add(float* p, float v) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("red.shared.add.f32 [%0], %1;" :: "r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void red_add(double* p, double v) { atomicAdd(p, v); }

template <int G>
struct AtomicLayout {
  static constexpr int kRowGroups = 32 / G;                      // rows handled at once
  static constexpr int kRowsPerLane = G * G / 32 > 0 ? G * G / 32 : 1;   // ceil(G / kRowGroups)
};

template <typename R, int G>
__global__ void __launch_bounds__(kThreads, kGridAtomicMinBlocks)
k_grid_atomic(const Geom g, const __grid_constant__ Coef<R> coef, const IndexView<R> ix,
              const typename C2<R>::T* __restrict__ vis, const R* __restrict__ wgt,
              typename C2<R>::T* __restrict__ planes, int b0, int nb, int bs, int pitch) {
  using CT = typename C2<R>::T;
  constexpr int RG = AtomicLayout<G>::kRowGroups;
  constexpr int KR = AtomicLayout<G>::kRowsPerLane;
  extern __shared__ __align__(16) unsigned char smem[];
  R* sc = reinterpret_cast<R*>(smem);
  R* acc = reinterpret_cast<R*>(smem + (kMaxDeg + 1) * kMaxG * sizeof(R));
  const int T = g.tile, alpha = g.alpha, aw = g.alpha_w;
  const int t = blockIdx.x;
  const int tu = t / g.ntv, tv = t - tu * g.ntv;
  const int s0 = b0 + blockIdx.y * bs;
  const int sb = min(bs, b0 + nb - s0);
  const int plane_elems = T * pitch;
  R* acc_im = acc + sb * plane_elems;   // real parts of the sb planes, then imaginary parts
  for (int i = threadIdx.x; i < (g.deg + 1) * kMaxG; i += blockDim.x) sc[i] = coef.c[i];
  for (int e = threadIdx.x; e < 2 * sb * plane_elems; e += blockDim.x) acc[e] = (R)0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int j = lane & (G - 1), rg = lane / G;
  LanePieceOf<R, G> pc;
  if (sizeof(R) == 4) pc.load(sc, g.deg, j);
  const bool lj = j < alpha;

  // sources: this tile and the tiles one to the left / above / both, whose visibilities'
  // alpha x alpha footprints can reach into this tile (alpha - 1 <= T)
  for (int src = 0; src < 4; ++src) {
    const int ou = (src & 1) ? -1 : 0, ov = (src & 2) ? -1 : 0;
    int stu = tu + ou; if (stu < 0) stu += g.ntu;
    int stv = tv + ov; if (stv < 0) stv += g.ntv;
    const uint32_t* offs = ix.off + ((int64_t)stu * g.ntv + stv) * g.nw;
    const uint32_t lo = offs[max(0, s0 - aw + 1)], hi = offs[min(g.nw, s0 + sb)];
    // blocks of 32 visibilities per warp, interleaved over the warps (visibility vb + l nwarps
    // of block vb goes to lane l): each lane loads the coordinates and data of its visibility
    // (one round trip for 32), then the warp takes the block's visibilities whose footprint
    // meets the tile one at a time, broadcast by shuffles
    for (uint32_t vb = lo + warp; vb < hi; vb += 32 * nwarps) {
      const uint32_t vl = vb + lane * nwarps;
      uint32_t mtl = 0;
      Z4<R> zl;
      zl.u = zl.v = zl.w = zl.pad = (R)0;
      R drl = (R)0, dil = (R)0;
      bool hitl = false;
      if (vl < hi) {
        mtl = ix.meta[vl];
        const int ru = (int)(mtl & 255) + ou * T, rv = (int)((mtl >> 8) & 255) + ov * T;
        hitl = ru + alpha > 0 && rv + alpha > 0;   // footprint meets this tile
        if (hitl) {
          zl = ix.z[vl];
          const uint32_t id = ix.idx[vl];
          const int64_t k = id & ~kFoldBit;
          const CT d = vis[k];
          drl = d.x; dil = d.y;
          if (wgt != nullptr) { const R w = wgt[k]; drl *= w; dil *= w; }
          if (id & kFoldBit) dil = -dil;    // grid conj(d) at the folded coordinates
          if (ix.ph != nullptr) {           // times conj(exp(2 pi i w nshift))
            const CT ph = ix.ph[vl];
            const R r = drl * ph.x + dil * ph.y;
            dil = dil * ph.x - drl * ph.y;
            drl = r;
          }
        }
      }
      unsigned hits = __ballot_sync(0xffffffffu, hitl);
      while (hits != 0u) {
        const int v = __ffs(hits) - 1;
        hits &= hits - 1u;
        const uint32_t vi = vb + v * nwarps;
        const uint32_t mt = __shfl_sync(0xffffffffu, mtl, v);
        const int ru = (int)(mt & 255) + ou * T, rv = (int)((mt >> 8) & 255) + ov * T;
        const int c0 = (int)(mt >> 16);
        const R zu = __shfl_sync(0xffffffffu, zl.u, v), zv = __shfl_sync(0xffffffffu, zl.v, v);
        const R zw = __shfl_sync(0xffffffffu, zl.w, v);
        const R dr = __shfl_sync(0xffffffffu, drl, v), di = __shfl_sync(0xffffffffu, dil, v);
        // piece j in u (row group 0) or v (the others), and in w
        const R puv = lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, rg == 0 ? 0 : 1, j,
                                              rg == 0 ? zu : zv) : (R)0;
        const R pw = g.do_w ? (lj ? kernel_value<R, G>(ix, pc, sc, g.deg, vi, 2, j, zw) : (R)0)
                            : (j == 0 ? (R)1 : (R)0);
        // this lane's column weight and the 2-D weights of its rows, clipped to the tile
        const R pv = __shfl_sync(0xffffffffu, puv, G + j);   // lane G + j holds v piece j
        const int col = rv + j;
        const bool colok = lj && col >= 0 && col < T;
        R cw[KR];
        int off[KR];
#pragma unroll
        for (int k = 0; k < KR; ++k) {
          const int i = rg + k * RG;
          const R pu = __shfl_sync(0xffffffffu, puv, i < G ? i : 0);   // lane i holds u piece i
          const int row = ru + i;
          const bool ok = colok && i < alpha && row >= 0 && row < T;
          cw[k] = ok ? pu * pv : (R)0;
          off[k] = ok ? row * pitch + col : -1;
        }
        const int qlo = max(0, s0 - c0), qhi = min(aw, s0 + sb - c0);
        for (int q = qlo; q < qhi; ++q) {
          const R wq = __shfl_sync(0xffffffffu, pw, q);
          const R qr = dr * wq, qi = di * wq;
          R* bre = acc + (c0 + q - s0) * plane_elems;
          R* bim = acc_im + (c0 + q - s0) * plane_elems;
#pragma unroll
          for (int k = 0; k < KR; ++k) {
            if (off[k] >= 0) {
              red_add(bre + off[k], qr * cw[k]);
              red_add(bim + off[k], qi * cw[k]);
            }
          }
        }
      }
    }
  }
  __syncthreads();
  const int64_t pstride = (int64_t)g.nu * g.nv;
  for (int e = threadIdx.x; e < sb * T * T; e += blockDim.x) {
    const int pl = e / (T * T), rem = e - pl * T * T;
    const int r = rem / T, c = rem - r * T;
    CT o;
    o.x = acc[pl * plane_elems + r * pitch + c];
    o.y = acc_im[pl * plane_elems + r * pitch + c];
    planes[(int64_t)(s0 - b0 + pl) * pstride + (int64_t)(tu * T + r) * g.nv + tv * T + c] = o;
  }
}

// ---------------------------------------------------------------------------------------
// grid on the tensor cores (automatic for most FP32 plans with 32-cell tiles, see grid_variant_of)
//
// Gridding visibilities onto 16 x 16 cells of a plane is a matrix product over the visibilities k:
// cells[i][j] += sum_k wu_k[i] (wv_k[j] ww_k d_k), 16 rows against 16 columns x (re, im), and one
// mma.m16n8k16 adds 16 visibilities to 16 x 8 cells.  (mma.sync, not tcgen05: the operands are
// made in registers, 16 visibilities at a time for 16 x 16 cells, and the tensor pipe is active 16 % of the
// time with alpha 6, 26 % with alpha 8.)  The shared-memory atomics of k_grid_atomic execute as
// compare-and-swap loops: about 1050 warp instructions per visibility (alpha 6, 1.6e6 visibilities on 42 planes of
// 2048^2) against 430 here; 616 with alpha 8 (5e5 visibilities on 33 planes of 1408^2).
//
// FP32 accuracy is kept: each factor is cut exactly into three bf16 parts (8 + 8 + 8 significant bits; planes
// of 16 visibilities whose data times w kernel all lie below 2^-63 are summed in FP32 instead, because the parts
// would reach into the bf16 subnormals), and all products of parts down to 2^-24 are summed, the leading ones
// 8 visibilities at a time and the other seven over 16, each from zero, and added to FP32 accumulators with
// round-to-nearest (the tensor core drops what lies 24 bits below its largest addend and rounds towards
// zero, so nothing is carried on in it).  Rounding error of the gridded image against an FP64 plan with
// the same kernel and grid, ten plans of 200^2 - 1024^2 and both narrow and wide (e^(3 N(0,1))) data: 2.0 -
// 5.2e-7, 0.85 - 0.99 times the atomics'; on dense cells, where the atomics add more often, less (see
// kMmaMaxGain).
//
// Warps work alone, without barriers: warp = (16 x 16 quarter of a 32 x 32 tile, kMmaPlanes planes),
// accumulators in registers, each cell written once; a CTA holds the four quarters.  A warp looks
// through the visibilities of the tile and of the three tiles whose footprints reach into it, 64
// at a time, and puts those that meet its cells and planes into a queue in shared memory;
// whenever the queue holds 16 it evaluates their kernels (8 or 16 lanes per visibility, lane =
// piece, Horner from registers) into rows padded with zeros on both sides and adds them.  The
// result does not depend on timing: a plan grids bitwise reproducibly.
//
// Bound: latency at about one group of 16 per warp (a warp's candidates, their data and one group
// take 9 us at 16 warps per SM), then issue.  Planes per warp: two instead of four measured 1.3
// times slower (more visits), 96 and 168 registers 1.15 and 1.0 times.  Stage times before and after,
// GB300: 2048^2, 1e6 visibilities, 55 planes of 2816^2 2.46 -> 1.56 ms; 4096^2, 1e7 visibilities 15.0
// -> 10.7 ms; 8192^2, 5e7 visibilities 117 -> 74 ms; 512^2, 1.2e5 visibilities 0.66 -> 0.17 ms.
//
// On small grids the few dense tiles at the grid's origin would be the whole run time: there SPLIT = 4 warps
// share each quarter, taking turns at the candidates, and their sums are added in a fixed order (512^2, 1.2e5
// visibilities: 0.34 -> 0.17 ms), for every tile or in a launch of its own for the dense ones: see mma_launches.
// ---------------------------------------------------------------------------------------
constexpr int kMmaTile = 32, kMmaPlanes = 4, kMmaQueue = 256, kMmaPad = 16;
constexpr int kMmaRow = 48;   // kMmaPad zeros, up to 16 kernel values, zeros
constexpr int kMmaBlocks = 2;   // blocks of 32 candidates looked at together

// an index entry: position in the index, visibility and fold bit, ru + 32 | (rv + 32) << 8 | c0 << 16
struct MmaEntry { uint32_t at, id, pos; };
struct alignas(16) MmaWarp {
  float wu[16][kMmaRow], wv[16][kMmaRow];
  float2 dw[16][kMmaPlanes];   // data x w kernel value of the warp's planes
  float zu[16], zv[16], zw[16];
  float2 d[16];
  int ru[16], rv[16], c0[16];
  MmaEntry queue[kMmaQueue];
};

__device__ __forceinline__ void mma_bf16(float* d, const unsigned* a, const unsigned* b) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// the same over 8 visibilities: one register of two rows' fragments, one of the columns'
__device__ __forceinline__ void mma_bf16_k8(float* d, unsigned a0, unsigned a1, unsigned b) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(b));
}
// the bf16 parts (upper halves) of two values as one register each: x = p0 + p1 + p2 exactly
__device__ __forceinline__ void split_bf16(float x, float y, unsigned& p0, unsigned& p1, unsigned& p2) {
  auto top = [](float v) { return __uint_as_float(__float_as_uint(v) & 0xffff0000u); };
  auto pack = [](float a, float b) { return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632); };
  p0 = pack(x, y);
  x -= top(x); y -= top(y);
  p1 = pack(x, y);
  x -= top(x); y -= top(y);
  p2 = pack(x, y);
}

template <int G, int SPLIT>
__global__ void __launch_bounds__(128 * SPLIT, SPLIT == 1 ? 4 : 1)
k_grid_mma(const Geom g, const __grid_constant__ Coef<float> coef, const IndexView<float> ix,
           const float2* __restrict__ vis, const float* __restrict__ wgt,
           float2* __restrict__ planes, int b0, int nb, uint32_t dense) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int T = kMmaTile;
  const int alpha = g.alpha, aw = g.alpha_w;
  // tile rows from both ends of the grid towards its middle: short baselines, the densest rows,
  // lie at the ends (row 0 and, wrapped, the last) and start first
  const int tr = blockIdx.x / g.ntv, tv = blockIdx.x - tr * g.ntv;
  const int tu = (tr & 1) ? g.ntu - 1 - tr / 2 : tr / 2;
  const int s0 = b0 + blockIdx.y * kMmaPlanes;
  const int sb = min(kMmaPlanes, b0 + nb - s0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  MmaWarp& sm = reinterpret_cast<MmaWarp*>(smem)[warp];
  const int quarter = warp / SPLIT, part = warp - quarter * SPLIT;
  const int sr0 = (quarter & 2) ? 16 : 0, sc0 = (quarter & 1) ? 16 : 0;
  const int gid = lane >> 2, tig = lane & 3;
  // the four sources' ranges of visibilities whose planes meet this warp's (lane: source and end)
  uint32_t lo[4], before[4], total = 0;
  {
    const int src = (lane >> 1) & 3;
    int stu = tu - (src & 1); if (stu < 0) stu += g.ntu;
    int stv = tv - (src >> 1); if (stv < 0) stv += g.ntv;
    const uint32_t at = ix.off[((int64_t)stu * g.ntv + stv) * g.nw +
                               ((lane & 1) ? min(g.nw, s0 + sb) : max(0, s0 - aw + 1))];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      lo[s] = __shfl_sync(0xffffffffu, at, 2 * s);
      before[s] = total;
      total += __shfl_sync(0xffffffffu, at, 2 * s + 1) - lo[s];
    }
  }
  // tiles of up to `dense` candidates are the SPLIT = 1 launch's, the others the SPLIT = 4 launch's
  if (__any_sync(0xffffffffu, SPLIT == 1 ? total > dense : total < dense)) return;
  const int64_t pstride = (int64_t)g.nu * g.nv;
  float2* out = planes + (int64_t)(s0 - b0) * pstride + (int64_t)(tu * T + sr0 + gid) * g.nv +
                tv * T + sc0 + 2 * tig;
  // the accumulators never live across the end of a branch that may diverge (they would be
  // spilled): an empty warp stores its zeros here, and the loops below end on votes
  if (!__any_sync(0xffffffffu, total > 0)) {
    for (int pl = part; pl < sb; pl += SPLIT)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        *reinterpret_cast<float4*>(out + pl * pstride + (int64_t)(8 * (c >> 1)) * g.nv + 8 * (c & 1)) =
            make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  float acc[kMmaPlanes][4][4];   // plane, (columns 0-7 re, im, columns 8-15 re, im), fragment
#pragma unroll
  for (int a = 0; a < kMmaPlanes * 16; ++a) (&acc[0][0][0])[a] = 0.f;

  {
    uint32_t mt[kMmaBlocks], id[kMmaBlocks], at[kMmaBlocks];
    auto entries = [&](uint32_t e0) {   // index entries of the next candidates
#pragma unroll
      for (int b = 0; b < kMmaBlocks; ++b) {
        const uint32_t e = e0 + 32 * b + lane;
        mt[b] = id[b] = at[b] = 0;
        if (e < total) {
          const int src = (e >= before[1]) + (e >= before[2]) + (e >= before[3]);
          at[b] = e + (src == 0 ? lo[0] : src == 1 ? lo[1] - before[1]
                       : src == 2 ? lo[2] - before[2] : lo[3] - before[3]);
          mt[b] = ix.meta[at[b]];
          id[b] = ix.idx[at[b]];
        }
      }
    };
    entries(32 * kMmaBlocks * part);
    float4* z4 = reinterpret_cast<float4*>(&sm.wu[0][0]);
    for (int i = lane; i < 2 * 16 * kMmaRow / 4; i += 32) z4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (lane < 16) {
      sm.ru[lane] = sm.rv[lane] = sm.c0[lane] = 0;
      sm.zu[lane] = sm.zv[lane] = sm.zw[lane] = 0.f;
      sm.d[lane] = make_float2(0.f, 0.f);
    }
    // this lane's kernel piece: coefficients in registers, zeros up to degree G + 3
    const int j = lane & (G - 1);
    float pc[G + 4];
#pragma unroll
    for (int d = 0; d <= G + 3; ++d) pc[d] = d <= g.deg ? coef.c[d * kMaxG + j] : 0.f;
    auto piece = [&](float z) {
      float r = pc[G + 3];
#pragma unroll
      for (int d = G + 2; d >= 0; --d) r = fmaf(r, z, pc[d]);
      return r;
    };
    int head = 0, cnt = 0;
    constexpr uint32_t kStep = 32 * kMmaBlocks * SPLIT;   // the parts take turns
    for (uint32_t e0 = 32 * kMmaBlocks * part;; e0 += kStep) {
      // the test against the warp's cells and planes; hits go to the queue in index order
#pragma unroll
      for (int b = 0; b < kMmaBlocks; ++b) {
        const uint32_t e = e0 + 32 * b + lane;
        const int src = (e >= before[1]) + (e >= before[2]) + (e >= before[3]);
        const int ru = (int)(mt[b] & 255) - (src & 1) * T, rv = (int)((mt[b] >> 8) & 255) - (src >> 1) * T;
        const int c0 = (int)(mt[b] >> 16);
        const bool hit = e < total && ru < sr0 + 16 && ru + alpha > sr0 && rv < sc0 + 16 &&
                         rv + alpha > sc0 && c0 < s0 + sb && c0 + aw > s0;
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (hit) {
          MmaEntry& q = sm.queue[(head + cnt + __popc(m & ((1u << lane) - 1u))) & (kMmaQueue - 1)];
          q.at = at[b]; q.id = id[b];
          q.pos = (uint32_t)((ru + 32) | (rv + 32) << 8 | c0 << 16);
        }
        cnt += __popc(m);
      }
      const bool done = __any_sync(0xffffffffu, e0 + kStep >= total);
      if (!done) entries(e0 + kStep);
      __syncwarp();
      while (cnt >= 16 || (done && cnt > 0)) {
        const int nv = min(cnt, 16);
        // 16 visibilities: lanes 0-15 their coordinates, lanes 16-31 their data
        {
          const int v = lane & 15;
          const MmaEntry q = sm.queue[(head + v) & (kMmaQueue - 1)];
          if (v < nv) {
            if (lane < 16) {
              const Z4<float> z = ix.z[q.at];
              sm.zu[v] = z.u; sm.zv[v] = z.v; sm.zw[v] = z.w;
              sm.ru[v] = (int)(q.pos & 255) - 32; sm.rv[v] = (int)((q.pos >> 8) & 255) - 32;
              sm.c0[v] = (int)(q.pos >> 16);
            } else {
              const int64_t k = q.id & ~kFoldBit;
              float2 d = vis[k];
              if (wgt != nullptr) { const float w = wgt[k]; d.x *= w; d.y *= w; }
              if (q.id & kFoldBit) d.y = -d.y;    // grid conj(d) at the folded coordinates
              if (ix.ph != nullptr) {             // times conj(exp(2 pi i w nshift))
                const float2 ph = ix.ph[q.at];
                const float r = d.x * ph.x + d.y * ph.y;
                d.y = d.y * ph.x - d.x * ph.y;
                d.x = r;
              }
              sm.d[v] = d;
            }
          }
          head = (head + nv) & (kMmaQueue - 1);
          cnt -= nv;
        }
        __syncwarp();
#pragma unroll
        for (int v0 = 0; v0 < 16; v0 += 32 / G) {
          // (slots beyond the last visibility hold an older one, or zeros: their data count as zero)
          const int v = v0 + lane / G, c0 = sm.c0[v];
          const float pu = piece(sm.zu[v]), pv = piece(sm.zv[v]), pw = piece(sm.zw[v]);
          sm.wu[v][kMmaPad + j] = j < alpha ? pu : 0.f;
          sm.wv[v][kMmaPad + j] = j < alpha ? pv : 0.f;
          const float ww = g.do_w ? (j < alpha ? pw : 0.f) : (j == 0 ? 1.f : 0.f);
          // lane pl of the group takes plane s0 + pl, the visibility's plane q = s0 + pl - c0
          const int q = s0 + j - c0;
          const float wq = __shfl_sync(0xffffffffu, ww, q & (G - 1), G);
          if (j < kMmaPlanes) {
            const bool on = v < nv && q >= 0 && q < aw;
            const float2 d = sm.d[v];
            sm.dw[v][j] = on ? make_float2(d.x * wq, d.y * wq) : make_float2(0.f, 0.f);
          }
        }
        __syncwarp();
        // this lane's four visibilities: k = 2 tig, 2 tig + 1, 2 tig + 8, 2 tig + 9
        float x[4][2], y[4][2];   // wu at rows gid, gid + 8; wv at columns gid, gid + 8
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int v = 2 * tig + (q & 1) + (q & 2) * 4;
          const float* u = &sm.wu[v][kMmaPad + sr0 + gid - sm.ru[v]];
          const float* w = &sm.wv[v][kMmaPad + sc0 + gid - sm.rv[v]];
          x[q][0] = u[0]; x[q][1] = u[8];
          y[q][0] = w[0]; y[q][1] = w[8];
        }
        unsigned A[3][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)   // rows gid, gid + 8 at k 0-7, then at k 8-15
          split_bf16(x[(r >> 1) * 2][r & 1], x[(r >> 1) * 2 + 1][r & 1], A[0][r], A[1][r], A[2][r]);
#pragma unroll
        for (int pl = 0; pl < kMmaPlanes; ++pl) {
          float2 d[4];
          float most = 0.f;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            d[q] = sm.dw[2 * tig + (q & 1) + (q & 2) * 4][pl];
            most = fmaxf(most, fmaxf(fabsf(d[q].x), fabsf(d[q].y)));
          }
          if (!__any_sync(0xffffffffu, most >= 0x1p-63f)) {
            bool any = false;   // (a NaN counts)
#pragma unroll
            for (int q = 0; q < 4; ++q) any = any || d[q].x != 0.f || d[q].y != 0.f;
            if (!__any_sync(0xffffffffu, any)) continue;
            // the slices of such data would reach into the bf16 subnormals, which end at 2^-133: in FP32
            // as they are, each lane the cells of its fragments
#pragma unroll 1
            for (int v = 0; v < nv; ++v) {
              const float* u = &sm.wu[v][kMmaPad + sr0 + gid - sm.ru[v]];
              const float* w = &sm.wv[v][kMmaPad + sc0 + 2 * tig - sm.rv[v]];
              const float2 e = sm.dw[v][pl];
#pragma unroll
              for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                  const float wc = w[(c & 1) + 4 * (c & 2)], ur = u[8 * r];
                  float &re = acc[pl][c & 2][2 * r + (c & 1)], &im = acc[pl][(c & 2) + 1][2 * r + (c & 1)];
                  re = __fmaf_rn(ur, wc * e.x, re);
                  im = __fmaf_rn(ur, wc * e.y, im);
                }
            }
            continue;
          }
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            float b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) b[q] = y[q][nt >> 1] * ((nt & 1) ? d[q].y : d[q].x);
            unsigned B[3][2];
            split_bf16(b[0], b[1], B[0][0], B[1][0], B[2][0]);
            split_bf16(b[2], b[3], B[0][1], B[1][1], B[2][1]);
            float s[4], m[4], m8[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] = m[i] = m8[i] = 0.f;
            mma_bf16_k8(m, A[0][0], A[0][1], B[0][0]);
            mma_bf16_k8(m8, A[0][2], A[0][3], B[0][1]);
            mma_bf16(s, A[2], B[1]);
            mma_bf16(s, A[1], B[2]);
            mma_bf16(s, A[2], B[0]);
            mma_bf16(s, A[0], B[2]);
            mma_bf16(s, A[1], B[1]);
            mma_bf16(s, A[1], B[0]);
            mma_bf16(s, A[0], B[1]);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[pl][nt][i] += (m[i] + m8[i]) + s[i];
          }
        }
        __syncwarp();   // the staged visibilities have been used
      }
      if (done) break;
    }
  }
  if constexpr (SPLIT > 1) {
    // the parts' sums through their own shared memory, added in a fixed order
    static_assert(sizeof(MmaWarp) >= kMmaPlanes * 16 * 32 * sizeof(float), "room for a part's sums");
    float* mine = reinterpret_cast<float*>(&sm);
    if (part > 0) {
#pragma unroll
      for (int i = 0; i < kMmaPlanes * 16; ++i) mine[32 * i + lane] = (&acc[0][0][0])[i];
    }
    asm volatile("bar.sync %0, %1;" ::"r"(quarter + 1), "r"(32 * SPLIT) : "memory");
    if (part > 0) return;
#pragma unroll 1
    for (int o = 1; o < SPLIT; ++o) {
      const float* other = mine + o * (sizeof(MmaWarp) / sizeof(float));
#pragma unroll
      for (int i = 0; i < kMmaPlanes * 16; ++i) (&acc[0][0][0])[i] += other[32 * i + lane];
    }
  }
#pragma unroll
  for (int pl = 0; pl < kMmaPlanes; ++pl) {
    if (pl >= sb) break;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int r = 0; r < 2; ++r)   // two adjacent cells, 16-byte aligned (nv is a multiple of 32)
        *reinterpret_cast<float4*>(out + pl * pstride + (int64_t)(8 * r) * g.nv + 8 * h) =
            make_float4(acc[pl][2 * h][2 * r], acc[pl][2 * h + 1][2 * r], acc[pl][2 * h][2 * r + 1],
                        acc[pl][2 * h + 1][2 * r + 1]);
  }
}

// ---------------------------------------------------------------------------------------
// grid, row-band owner variant (FP32, alpha <= 8, 32-cell tiles; deterministic)
//
// CTA = (32 x 32 uv tile, sub-batch of up to kBandPlanes planes), accumulators in shared memory
// as (re, im) float pairs with a row pitch of kBandPitch pairs.  Warp w owns tile rows 4w ..
// 4w + 3 of every plane of the sub-batch, so its updates are plain read-modify-writes (no
// atomics, each cell updated in index order: deterministic) and the 32 lanes of an update --
// (row r, footprint column j) = (lane / 8, lane mod 8) -- touch 32 distinct cells in two
// shared-memory wavefronts (pitch = 8 mod 16 pairs).  Visibilities of the tile and of the three
// tiles whose footprints reach into it are taken in chunks of kBandChunk:
//  1a. each visibility's footprint is tested against the tile (a bit of a 64-bit hit mask);
//  1b. the hits are staged in index order (slot = hits before it): kernel values in u and v,
//      and the data times the w kernel value of each of its planes (a group of 8 lanes per
//      visibility, lane j evaluating piece j by Horner from registers, Sec. 4.2); each staged
//      visibility sets its bit in the 64-bit masks of the row bands its footprint meets;
//  2.  each warp walks the set bits of its band's mask and adds those visibilities into its
//      rows, with the loop over the visibility's planes in the sub-batch unrolled per count.
// ---------------------------------------------------------------------------------------
constexpr int kBandTile = 32, kBandRows = 4, kBandPitch = 40, kBandChunk = 64, kBandPlanes = 8;
constexpr int kBandWarps = kBandTile / kBandRows;
static_assert(kBandRows * 8 == 32 && kBandWarps * 32 == 256, "band layout");
static_assert(kBandPitch % 16 == 8 && kBandPitch >= kBandTile + 8, "band pitch");

struct BandStage {
  float wu[kBandChunk][8], wv[kBandChunk][8];
  float2 dq[kBandChunk][8];   // data x w kernel value of plane q of the visibility
  int ru[kBandChunk], rv[kBandChunk], c0[kBandChunk];
  unsigned long long hits;                 // chunk positions whose footprint meets the tile
  unsigned long long band[kBandWarps];     // staged slots whose footprint meets band w
};

// add staged visibility v into planes pl0 .. pl0 + NQ - 1 of this lane's cell
template <int NQ>
__device__ __forceinline__ void band_add(float2* __restrict__ base, const float2* __restrict__ dq,
                                         float w2) {
  constexpr int kPlane = kBandTile * kBandPitch;
  float2 a[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) a[q] = base[q * kPlane];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const float2 d = dq[q];
    a[q].x = fmaf(d.x, w2, a[q].x);
    a[q].y = fmaf(d.y, w2, a[q].y);
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) base[q * kPlane] = a[q];
}

__global__ void __launch_bounds__(256, 2)
k_grid_band(const Geom g, const __grid_constant__ Coef<float> coef, const IndexView<float> ix,
            const float2* __restrict__ vis, const float* __restrict__ wgt,
            float2* __restrict__ planes, int b0, int nb, int bs) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* sc = reinterpret_cast<float*>(smem);
  BandStage* stg = reinterpret_cast<BandStage*>(smem + (kMaxDeg + 1) * kMaxG * sizeof(float));
  float2* acc = reinterpret_cast<float2*>(reinterpret_cast<unsigned char*>(stg) + sizeof(BandStage));
  constexpr int T = kBandTile, kPlane = kBandTile * kBandPitch;
  const int alpha = g.alpha, aw = g.alpha_w;
  const int t = blockIdx.x;
  const int tu = t / g.ntv, tv = t - tu * g.ntv;
  const int s0 = b0 + blockIdx.y * bs;
  const int sb = min(bs, b0 + nb - s0);
  for (int i = threadIdx.x; i < (g.deg + 1) * kMaxG; i += blockDim.x) sc[i] = coef.c[i];
  for (int e = threadIdx.x; e < sb * kPlane; e += blockDim.x) acc[e] = make_float2(0.f, 0.f);
  if (threadIdx.x <= kBandWarps) {
    if (threadIdx.x == kBandWarps) stg->hits = 0ull;
    else stg->band[threadIdx.x] = 0ull;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // phase 1: groups of 8 lanes, one visibility each, lane j1 = kernel piece j1
  const int j1 = threadIdx.x & 7, grp = threadIdx.x >> 3;
  constexpr int kGroups = 256 / 8;
  const unsigned gmask = 0xffu << (lane & 24);
  LanePiece<float, 8> pc;
  pc.load(sc, g.deg, j1);
  // phase 2: this warp's rows band0 .. band0 + 3; lane (r, j)
  const int band0 = warp * kBandRows;
  const int row = band0 + (lane >> 3), j = lane & 7;
  for (int src = 0; src < 4; ++src) {
    // sources: this tile and the tiles one to the left / above / both, whose visibilities'
    // footprints can reach into this tile (alpha - 1 <= T)
    const int ou = (src & 1) ? -1 : 0, ov = (src & 2) ? -1 : 0;
    int stu = tu + ou; if (stu < 0) stu += g.ntu;
    int stv = tv + ov; if (stv < 0) stv += g.ntv;
    const uint32_t* offs = ix.off + ((int64_t)stu * g.ntv + stv) * g.nw;
    const uint32_t lo = offs[max(0, s0 - aw + 1)], hi = offs[min(g.nw, s0 + sb)];
    for (uint32_t cs = lo; cs < hi; cs += kBandChunk) {
      const int nch = (int)min((uint32_t)kBandChunk, hi - cs);
      // 1a: hit test (each group keeps its visibilities' index entries for 1b)
      uint32_t mt[kBandChunk / kGroups];
#pragma unroll
      for (int pass = 0; pass < kBandChunk / kGroups; ++pass) {
        const int v = grp + pass * kGroups;
        mt[pass] = 0u;
        if (v < nch) {
          mt[pass] = ix.meta[cs + v];
          const int ru = (int)(mt[pass] & 255) + ou * T, rv = (int)((mt[pass] >> 8) & 255) + ov * T;
          if (j1 == 0 && ru + alpha > 0 && rv + alpha > 0) atomicOr(&stg->hits, 1ull << v);
        }
      }
      __syncthreads();
      const unsigned long long hits = stg->hits;
      // 1b: stage the hits in index order
#pragma unroll
      for (int pass = 0; pass < kBandChunk / kGroups; ++pass) {
        const int v = grp + pass * kGroups;
        if (v >= nch || !((hits >> v) & 1ull)) continue;   // uniform within the group
        const int slot = __popcll(hits & ((1ull << v) - 1ull));
        const uint32_t vi = cs + v;
        const int ru = (int)(mt[pass] & 255) + ou * T, rv = (int)((mt[pass] >> 8) & 255) + ov * T;
        const Z4<float> zz = ix.z[vi];
        const bool lj = j1 < alpha;
        stg->wu[slot][j1] = lj ? pc.eval(zz.u) : 0.f;
        stg->wv[slot][j1] = lj ? pc.eval(zz.v) : 0.f;
        const float ww = g.do_w ? (lj ? pc.eval(zz.w) : 0.f) : (j1 == 0 ? 1.f : 0.f);
        float dr = 0.f, di = 0.f;
        if (j1 == 0) {
          const uint32_t id = ix.idx[vi];
          const int64_t k = id & ~kFoldBit;
          const float2 d = vis[k];
          dr = d.x; di = d.y;
          if (wgt != nullptr) { const float w = wgt[k]; dr *= w; di *= w; }
          if (id & kFoldBit) di = -di;      // grid conj(d) at the folded coordinates
          if (ix.ph != nullptr) {           // times conj(exp(2 pi i w nshift))
            const float2 ph = ix.ph[vi];
            const float rr = dr * ph.x + di * ph.y;
            di = di * ph.x - dr * ph.y;
            dr = rr;
          }
          stg->ru[slot] = ru; stg->rv[slot] = rv; stg->c0[slot] = (int)(mt[pass] >> 16);
        }
        // the row bands the footprint meets (lanes 1 .. : one band each)
        const int blo = max(ru, 0) / kBandRows, bhi = min(ru + alpha - 1, T - 1) / kBandRows;
        if (j1 >= 1 && blo + j1 - 1 <= bhi) atomicOr(&stg->band[blo + j1 - 1], 1ull << slot);
        dr = __shfl_sync(gmask, dr, 0, 8);
        di = __shfl_sync(gmask, di, 0, 8);
        stg->dq[slot][j1] = make_float2(dr * ww, di * ww);
      }
      __syncthreads();
      if (threadIdx.x == 0) stg->hits = 0ull;   // read again only after the next barrier
      // 2: this warp's visibilities
      unsigned long long m = stg->band[warp];
      __syncwarp();
      if (lane == 0) stg->band[warp] = 0ull;
      while (m != 0ull) {
        const int v = __ffsll((long long)m) - 1;
        m &= m - 1ull;
        const int c0 = stg->c0[v], ru = stg->ru[v], rv = stg->rv[v];
        const int qlo = max(0, s0 - c0), qhi = min(aw, s0 + sb - c0);
        const int i = row - ru, col = rv + j;
        const bool ok = i >= 0 && i < alpha && j < alpha && col >= 0 && col < T;
        const float w2 = ok ? stg->wu[v][ok ? i : 0] * stg->wv[v][j] : 0.f;
        // idle lanes update a private padding cell of their row with weight 0
        float2* base = acc + (c0 + qlo - s0) * kPlane + row * kBandPitch + (ok ? col : T + j);
        const float2* dqv = stg->dq[v] + qlo;
        switch (qhi - qlo) {
          case 1: band_add<1>(base, dqv, w2); break;
          case 2: band_add<2>(base, dqv, w2); break;
          case 3: band_add<3>(base, dqv, w2); break;
          case 4: band_add<4>(base, dqv, w2); break;
          case 5: band_add<5>(base, dqv, w2); break;
          case 6: band_add<6>(base, dqv, w2); break;
          case 7: band_add<7>(base, dqv, w2); break;
          case 8: band_add<8>(base, dqv, w2); break;
          default: break;
        }
      }
      __syncthreads();   // the staged chunk has been consumed
    }
  }
  const int64_t pstride = (int64_t)g.nu * g.nv;
  for (int e = threadIdx.x; e < sb * T * T; e += blockDim.x) {
    const int pl = e / (T * T), rem = e - pl * T * T;
    const int r = rem / T, c = rem - r * T;
    planes[(int64_t)(s0 - b0 + pl) * pstride + (int64_t)(tu * T + r) * g.nv + tv * T + c] =
        acc[pl * kPlane + r * kBandPitch + c];
  }
}

// ---------------------------------------------------------------------------------------
// per-call kernel values: one thread per (visibility, direction, piece), Horner (Sec. 4.2)
// ---------------------------------------------------------------------------------------
template <typename R>
__global__ void k_weights(const Geom g, const __grid_constant__ Coef<R> coef, const IndexView<R> ix,
                          int64_t nvis_idx, R* __restrict__ wts) {
  __shared__ R sc[(kMaxDeg + 1) * kMaxG];
  for (int i = threadIdx.x; i < (g.deg + 1) * kMaxG; i += blockDim.x) sc[i] = coef.c[i];
  __syncthreads();
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nvis_idx * 3 * kMaxG) return;
  const int64_t pos = e / (3 * kMaxG);
  const int r = (int)(e - pos * 3 * kMaxG), d = r / kMaxG, j = r - d * kMaxG;
  const Z4<R> zz = ix.z[pos];
  R v = (R)0;
  if (j < g.alpha) v = horner(sc, g.deg, j, d == 0 ? zz.u : (d == 1 ? zz.v : zz.w));
  if (sizeof(R) == 8 && g.df64_planes) {
    // the pair-arithmetic kernels read the value as a double-float pair (same 8 bytes)
    const dd p = split_double((double)v);
    reinterpret_cast<float2*>(wts)[e] = make_float2(p.h, p.l);
  } else {
    wts[e] = v;
  }
}

template <typename R>
cudaError_t launch_weights(const Geom& g, const Coef<R>& coef, const IndexView<R>& ix,
                           int64_t nvis_idx, R* wts, cudaStream_t s) {
  if (nvis_idx == 0) return cudaSuccess;
  const int64_t n = nvis_idx * 3 * kMaxG;
  k_weights<R><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(g, coef, ix, nvis_idx, wts);
  return cudaGetLastError();
}
template cudaError_t launch_weights<float>(const Geom&, const Coef<float>&, const IndexView<float>&,
                                           int64_t, float*, cudaStream_t);
template cudaError_t launch_weights<double>(const Geom&, const Coef<double>&,
                                            const IndexView<double>&, int64_t, double*,
                                            cudaStream_t);

// ---------------------------------------------------------------------------------------
// launchers: sub-batch sizes from a shared-memory budget per CTA
// ---------------------------------------------------------------------------------------
// degridding CTA shared memory: FP32 54 KB, four CTAs per SM (measured on the 1e8-visibility
// workload: 72 KB 71.9 ms, 54 KB 61.3 ms, 44 KB 66.8 ms -- fewer planes per CTA against more
// warps to hide the staging loads); FP64 72 KB (FP64-pipe bound: more planes per CTA, fewer
// visits per visibility)
template <typename R>
constexpr size_t degrid_smem_budget() { return sizeof(R) == 4 ? 54 * 1024 : 72 * 1024; }
constexpr size_t kGridSmemBudget = 110 * 1024;

template <typename R>
static size_t coef_bytes() { return (kMaxDeg + 1) * kMaxG * sizeof(R); }

template <typename R>
static size_t degrid_plane_bytes(const Geom& g) {
  const int TH = g.tile + g.alpha - 1;
  return (size_t)TH * TH * sizeof(typename C2<R>::T);
}

template <typename R>
int degrid_subbatch(const Geom& g) {
  return (int)std::max<size_t>(1, (degrid_smem_budget<R>() - coef_bytes<R>()) / degrid_plane_bytes<R>(g));
}

// Allows a kernel all the dynamic shared memory of a CTA (227 KB).  Every launch sets the same value: host
// threads that launch a kernel with different sizes at the same time would otherwise lower each other's
// limit between setting it and the launch.
template <typename K>
static cudaError_t allow_shared(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

template <typename R, int G>
static cudaError_t degrid_g(const Geom& g, const Coef<R>& coef, const IndexView<R>& ix,
                            const typename C2<R>::T* planes, int b0, int nb, int bs,
                            typename C2<R>::T* partial, int64_t nvis_idx, cudaStream_t s) {
  size_t smem = coef_bytes<R>() + (size_t)std::min(bs, nb) * degrid_plane_bytes<R>(g);
  int64_t ntiles = (int64_t)g.ntu * g.ntv;
  // several CTAs for the densest tiles, where one would be the run time (they stage the same planes
  // and sum different visibilities; the sums are the same): see degrid_shares
  const int64_t nsub = (nb + bs - 1) / bs;
  const double meets = g.alpha_w + bs - 1.0;
  const double densest = g.max_tile * std::min(1.0, meets / g.nw);
  const double mean = g.nvis * meets / bs / (152.0 * 4.0);
  const uint32_t least = (uint32_t)std::max(128.0, 0.5 * mean) / 64 * 64;
  const int Z = degrid_shares(densest, mean, least, (double)(ntiles * nsub), sizeof(R) == 4);
  dim3 grid((unsigned)ntiles, (unsigned)nsub, (unsigned)Z);
  if constexpr (sizeof(R) == 8) {
    if (g.df64_planes) {
      auto launch = [&](auto kernel, bool packed) {
        const size_t bytes = smem - coef_bytes<R>() + degrid_dd_fixed(packed, ix.wts != nullptr);
        cudaError_t e = allow_shared(kernel);
        if (e != cudaSuccess) return e;
        kernel<<<grid, kThreads, bytes, s>>>(g, coef, ix, planes, b0, nb, bs, partial, nvis_idx, least);
        return cudaGetLastError();
      };
      if constexpr (G == 16)
        if (g.do_w) return launch(k_degrid_dd<G, true>, true);
      return launch(k_degrid_dd<G, false>, false);
    }
  }
  cudaError_t e = allow_shared(k_degrid<R, G>);
  if (e != cudaSuccess) return e;
  k_degrid<R, G><<<grid, kThreads, smem, s>>>(g, coef, ix, planes, b0, nb, bs, partial, nvis_idx, least);
  return cudaGetLastError();
}

template <int W, int SPLIT, int PG>
static cudaError_t grid_cells_split(const Geom& g, const Coef<double>& coef, const IndexView<double>& ix,
                                    const float4* vis, float4* planes, int b0, int nb, cudaStream_t s) {
  const size_t smem = coef_bytes<double>() + sizeof(CellsStage<W, SPLIT, PG>);
  cudaError_t e = allow_shared(k_grid_cells_dd<W, SPLIT, PG>);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)((int64_t)(g.nu / CellsTile<W>::rows) * (g.nv / CellsTile<W>::cols)),
            (unsigned)((nb + PG - 1) / PG));
  k_grid_cells_dd<W, SPLIT, PG><<<grid, 32 * W * SPLIT, smem, s>>>(g, coef, ix, vis, planes, b0, nb);
  return cudaGetLastError();
}

static cudaError_t grid_cells_dd(const Geom& g, const Coef<double>& coef, const IndexView<double>& ix,
                                 const float4* vis, float4* planes, int b0, int nb, cudaStream_t s) {
  // visibilities that a warp of the densest tile walks, against the mean over the warps the GPU
  // holds at once (32 on each SM; a visibility meets (alpha + 3)(alpha + 7) / 32 warps' 4 x 8 cells
  // and (alpha_w + 7) / 8 plane groups).  Measured <8, 1> against <2, 4>: 0.57 / 0.29 ms at 379
  // against a mean of 163 (27 000 visibilities, alpha 14), 80 / 29 ms at 150 000 against 2 400;
  // 10.6 / 16.1 ms at 169 against 7 000, 0.07 / 0.12 ms at 26 against 43 (1e4 visibilities)
  const double reach = (g.alpha + 3.0) * (g.alpha + 7.0), groups = g.alpha_w + kCellsPlanes - 1.0;
  const double densest = g.max_tile * std::min(1.0, groups / g.nw) *
                         std::min(1.0, reach / ((double)g.tile * g.tile));
  const double mean = g.nvis * groups / kCellsPlanes * reach / 32 / (152.0 * 32.0);
  if (densest > 1.2 * mean + 32.0) return grid_cells_split<2, 4, kCellsPlanes>(g, coef, ix, vis, planes, b0, nb, s);
  if (g.nw <= 2) return grid_cells_split<8, 1, 2>(g, coef, ix, vis, planes, b0, nb, s);
  return grid_cells_split<8, 1, kCellsPlanes>(g, coef, ix, vis, planes, b0, nb, s);
}

template <typename R, int G>
static cudaError_t grid_owner_g(const Geom& g, const Coef<R>& coef, const IndexView<R>& ix,
                                const typename C2<R>::T* vis, const R* wgt,
                                typename C2<R>::T* planes, int b0, int nb, cudaStream_t s) {
  // accumulator rows padded by two cells: rows of a clipped footprint start on different
  // banks, and the 2 x T padding cells of a plane give each lane of its owner warp a private
  // cell for idle updates
  const int pitch = g.tile + 2;
  const size_t per = (size_t)g.tile * pitch * sizeof(typename C2<R>::T);
  const size_t fixed = coef_bytes<R>() + sizeof(GridStage<R, G>);
  const int nwarps = kOwnerWarps;
  int bs = (int)std::max<size_t>(1, (kGridSmemBudget - fixed) / per);
  if (bs > nwarps) bs -= bs % nwarps;  // equal planes per warp
  bs = std::min(bs, nb);
  size_t smem = fixed + (size_t)bs * per;
  int64_t ntiles = (int64_t)g.ntu * g.ntv;
  dim3 grid((unsigned)ntiles, (unsigned)((nb + bs - 1) / bs));
  if constexpr (sizeof(R) == 8) {
    if (g.df64_planes)
      return grid_cells_dd(g, coef, ix, reinterpret_cast<const float4*>(vis),
                           reinterpret_cast<float4*>(planes), b0, nb, s);
  }
  cudaError_t e = allow_shared(k_grid_owner<R, G>);
  if (e != cudaSuccess) return e;
  k_grid_owner<R, G><<<grid, kOwnerThreads, smem, s>>>(g, coef, ix, vis, wgt, planes, b0, nb, bs, pitch);
  return cudaGetLastError();
}

template <typename R, int G>
static cudaError_t grid_atomic_g(const Geom& g, const Coef<R>& coef, const IndexView<R>& ix,
                                 const typename C2<R>::T* vis, const R* wgt,
                                 typename C2<R>::T* planes, int b0, int nb, cudaStream_t s) {
  // row pitch = G (mod 32) words: the 32 lanes of an atomic add (G columns x 32 / G rows)
  // fall in 32 different banks
  int pitch = g.tile;
  while (pitch % 32 != G % 32) ++pitch;
  const size_t per = (size_t)g.tile * pitch * sizeof(typename C2<R>::T);
  int bs = (int)std::max<size_t>(1, (kGridAtomicSmemBudget - coef_bytes<R>()) / per);
  bs = std::min(bs, nb);
  size_t smem = coef_bytes<R>() + (size_t)bs * per;
  cudaError_t e = allow_shared(k_grid_atomic<R, G>);
  if (e != cudaSuccess) return e;
  int64_t ntiles = (int64_t)g.ntu * g.ntv;
  dim3 grid((unsigned)ntiles, (unsigned)((nb + bs - 1) / bs));
  k_grid_atomic<R, G><<<grid, kThreads, smem, s>>>(g, coef, ix, vis, wgt, planes, b0, nb, bs, pitch);
  return cudaGetLastError();
}

template <int G, int SPLIT>
static cudaError_t grid_mma_split(const Geom& g, const Coef<float>& coef, const IndexView<float>& ix,
                                  const float2* vis, const float* wgt, float2* planes, int b0,
                                  int nb, uint32_t dense, cudaStream_t s) {
  const size_t smem = 4 * SPLIT * sizeof(MmaWarp);
  cudaError_t e = allow_shared(k_grid_mma<G, SPLIT>);
  if (e != cudaSuccess) return e;
  int64_t ntiles = (int64_t)g.ntu * g.ntv;
  dim3 grid((unsigned)ntiles, (unsigned)((nb + kMmaPlanes - 1) / kMmaPlanes));
  k_grid_mma<G, SPLIT><<<grid, 128 * SPLIT, smem, s>>>(g, coef, ix, vis, wgt, planes, b0, nb, dense);
  return cudaGetLastError();
}

// hits of the densest quarter (about half of its tile's visibilities, those whose planes meet the warp's)
// and their mean over the warps the GPU holds at once (16 on each SM; a visibility meets 2.1 quarters
// and (alpha + 3) / 4 plane groups)
static double mma_mean(const Geom& g) {
  return 2.1 * (double)g.nvis * (g.alpha_w + kMmaPlanes - 1) / kMmaPlanes / (152.0 * 16.0);
}
static MmaLaunches mma_form(const Geom& g, int nb) {
  const double window = std::min(1.0, (double)(g.alpha_w + kMmaPlanes - 1) / g.nw);
  return mma_launches(0.5 * (double)g.max_tile * window, mma_mean(g),
                      (double)g.ntu * g.ntv * ((nb + kMmaPlanes - 1) / kMmaPlanes));
}

template <int G>
static cudaError_t grid_mma(const Geom& g, const Coef<float>& coef, const IndexView<float>& ix,
                            const float2* vis, const float* wgt, float2* planes, int b0, int nb,
                            cudaStream_t s) {
  switch (mma_form(g, nb)) {
    case kMmaEven: return grid_mma_split<G, 1>(g, coef, ix, vis, wgt, planes, b0, nb, 0xffffffffu, s);
    case kMmaDense: return grid_mma_split<G, 4>(g, coef, ix, vis, wgt, planes, b0, nb, 0, s);
    default: break;
  }
  // the dense tiles first; candidates: those of a tile and its three sources, four times the hits of a quarter
  const uint32_t dense = (uint32_t)(0.25 * (2.0 * mma_mean(g) + 64.0));
  const cudaError_t e = grid_mma_split<G, 4>(g, coef, ix, vis, wgt, planes, b0, nb, dense + 1, s);
  return e != cudaSuccess ? e : grid_mma_split<G, 1>(g, coef, ix, vis, wgt, planes, b0, nb, dense, s);
}

static cudaError_t grid_band(const Geom& g, const Coef<float>& coef, const IndexView<float>& ix,
                             const float2* vis, const float* wgt, float2* planes, int b0, int nb,
                             cudaStream_t s) {
  const int bs = std::min(kBandPlanes, nb);
  const size_t smem = coef_bytes<float>() + sizeof(BandStage) +
                      (size_t)bs * kBandTile * kBandPitch * sizeof(float2);
  cudaError_t e = allow_shared(k_grid_band);
  if (e != cudaSuccess) return e;
  int64_t ntiles = (int64_t)g.ntu * g.ntv;
  dim3 grid((unsigned)ntiles, (unsigned)((nb + bs - 1) / bs));
  k_grid_band<<<grid, 256, smem, s>>>(g, coef, ix, vis, wgt, planes, b0, nb, bs);
  return cudaGetLastError();
}

// the gridding variant a plan uses (Geom::grid_variant 0 = automatic).  Automatic FP32 takes the
// tensor cores, which need 32-cell tiles, else the shared-memory atomics (on the 1e8-visibility
// workload the row-band owners measured 289 ms, the atomics 171 ms, the tensor cores 121 ms)
constexpr int kVariantMma = 4;   // tensor cores: automatic choice only
// ... and only up to this rounding gain of the plan.  The two kernels round differently, and the image
// correction amplifies the planes' rounding by the gain: their images lie 1 - 4e-7 x gain of the norm apart
// (3.3 - 5.0e-6 at a gain of 22, 1.8 - 2.7e-5 at about 110, 1.6 - 2.7e-4 at about 800).  Plans of a larger gain
// than those of 1e-5 (coarse accuracies, low oversampling) keep the atomics, so that an image changes by no
// more than 1e-5 of its norm with the kernel.  That is the only reason: array observations of 256^2 - 2048^2
// against an FP64 plan at 1e-9, tensor cores / atomics: gain 110 1.42 - 1.46e-4 / 1.42 - 1.47e-4, 200 2.8 - 3.3e-5 /
// 3.3 - 5.0e-5, 800 1.4 - 1.6e-4 / 1.4 - 2.7e-4, and the stage 277 / 1161 us (512^2), 1.26 / 1.98 ms (2048^2).
constexpr double kMmaMaxGain = 40.0;
template <typename R>
static int grid_variant_of(const Geom& g) {
  if (g.df64_planes) return 2;   // k_grid_cells_dd, see grid_owner_g
  const bool band_ok = sizeof(R) == 4 && g.alpha <= 8 && g.tile == kBandTile;
  if (g.grid_variant == 3) return band_ok ? 3 : 1;
  if (g.grid_variant != 0) return g.grid_variant;
  if (sizeof(R) == 8) return 2;
  // the narrowest kernels on a single plane with many visibilities and no dominating tile: half of a group's
  // lanes and three of a warp's four planes idle (1e6 visibilities on 1024 x 768, alpha = 4: 257 us by atomics,
  // 296 by the tensor cores; on 2816^2 219 and 236; 2e6 on 2048^2 356 and 399, on 1024^2 442 and 427; on 672 x
  // 512, where the densest tile is the run time, 405 and 224; 2e4 on 1024 x 768 23 and 19)
  const bool thin = g.alpha <= 4 && g.nw == 1 && mma_mean(g) > 400.0 && mma_form(g, 1) == kMmaEven;
  return g.tile == kMmaTile && g.gain <= kMmaMaxGain && !thin ? kVariantMma : 1;
}

// kernels that one launch_grid starts
template <typename R>
int grid_kernels(const Geom& g, int nb) {
  return sizeof(R) == 4 && grid_variant_of<R>(g) == kVariantMma && mma_form(g, nb) == kMmaBoth ? 2 : 1;
}
template int grid_kernels<float>(const Geom&, int);
template int grid_kernels<double>(const Geom&, int);

template <typename R, int G>
static cudaError_t grid_g(const Geom& g, const Coef<R>& coef, const IndexView<R>& ix,
                          const typename C2<R>::T* vis, const R* wgt,
                          typename C2<R>::T* planes, int b0, int nb, cudaStream_t s) {
  const int variant = grid_variant_of<R>(g);
  if (variant == 2) return grid_owner_g<R, G>(g, coef, ix, vis, wgt, planes, b0, nb, s);
  if constexpr (sizeof(R) == 4 && G <= 8) {
    if (variant == 3)
      return grid_band(g, coef, ix, (const float2*)vis, (const float*)wgt, (float2*)planes, b0,
                       nb, s);
  }
  if constexpr (sizeof(R) == 4) {
    if (variant == kVariantMma)   // groups of at least 8 lanes, one per plane of a CTA
      return grid_mma<(G < 8 ? 8 : G)>(g, coef, ix, (const float2*)vis, (const float*)wgt,
                                       (float2*)planes, b0, nb, s);
  }
  return grid_atomic_g<R, G>(g, coef, ix, vis, wgt, planes, b0, nb, s);
}

template <typename R>
cudaError_t launch_degrid(const Geom& g, const Coef<R>& coef, const IndexView<R>& ix,
                          const typename C2<R>::T* planes, int b0, int nb, int bs,
                          typename C2<R>::T* partial, int64_t nvis_idx, cudaStream_t s) {
  if (g.alpha <= 4) return degrid_g<R, 4>(g, coef, ix, planes, b0, nb, bs, partial, nvis_idx, s);
  if (g.alpha <= 8) return degrid_g<R, 8>(g, coef, ix, planes, b0, nb, bs, partial, nvis_idx, s);
  return degrid_g<R, 16>(g, coef, ix, planes, b0, nb, bs, partial, nvis_idx, s);
}

template <typename R>
cudaError_t launch_degrid_finalize(const Geom& g, const IndexView<R>& ix,
                                   const typename C2<R>::T* partial, int64_t nvis_idx, int bs,
                                   const R* wgt, typename C2<R>::T* vis, cudaStream_t s) {
  if (nvis_idx == 0) return cudaSuccess;
  k_degrid_finalize<R><<<(unsigned)((nvis_idx + 255) / 256), 256, 0, s>>>(g, ix, partial, nvis_idx,
                                                                          bs, wgt, vis);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_grid(const Geom& g, const Coef<R>& coef, const IndexView<R>& ix,
                        const typename C2<R>::T* vis, const R* wgt, typename C2<R>::T* planes,
                        int b0, int nb, cudaStream_t s) {
  if (g.alpha <= 4) return grid_g<R, 4>(g, coef, ix, vis, wgt, planes, b0, nb, s);
  if (g.alpha <= 8) return grid_g<R, 8>(g, coef, ix, vis, wgt, planes, b0, nb, s);
  return grid_g<R, 16>(g, coef, ix, vis, wgt, planes, b0, nb, s);
}

template cudaError_t launch_degrid<float>(const Geom&, const Coef<float>&, const IndexView<float>&,
                                          const float2*, int, int, int, float2*, int64_t,
                                          cudaStream_t);
template cudaError_t launch_degrid<double>(const Geom&, const Coef<double>&,
                                           const IndexView<double>&, const double2*, int, int, int,
                                           double2*, int64_t, cudaStream_t);
template cudaError_t launch_degrid_finalize<float>(const Geom&, const IndexView<float>&,
                                                   const float2*, int64_t, int, const float*,
                                                   float2*, cudaStream_t);
template cudaError_t launch_degrid_finalize<double>(const Geom&, const IndexView<double>&,
                                                    const double2*, int64_t, int, const double*,
                                                    double2*, cudaStream_t);
template int degrid_subbatch<float>(const Geom&);
template int degrid_subbatch<double>(const Geom&);
template cudaError_t launch_grid<float>(const Geom&, const Coef<float>&, const IndexView<float>&,
                                        const float2*, const float*, float2*, int, int,
                                        cudaStream_t);
template cudaError_t launch_grid<double>(const Geom&, const Coef<double>&,
                                         const IndexView<double>&, const double2*,
                                         const double*, double2*, int, int, cudaStream_t);

}  // namespace wg
