// 2-D complex FFT of FP64 planes computed in double-float ("df64") arithmetic on the FP32 pipes.
//
// GB300 executes FP64 FMAs at 1/64 of its FP32 rate, which makes cuFFT's double-precision
// transforms the dominant cost of the FP64 (eps ~ 1e-12) mode.  Here every value is carried as
// an unevaluated sum hi + lo of two floats (48-bit significand); additions use the two-sum and
// products the fma-based two-product error-free transformations, so a radix-8 butterfly costs a
// few hundred FP32 operations instead of FP64 ones.  Normwise accuracy of a 3200 x 3200
// transform is ~5e-15 relative (vs ~2e-16 for FP64); the planner accounts for it (its
// rounding is amplified by the 1 / psi correction, see plane_rounding / rounding_gain).
//
// Algorithm: each 1-D transform is a mixed-radix Stockham autosort FFT.  Nearly every side runs on
// PAIRS of lines packed into the FP32 x2 instructions (k_fft_pairs: radices up to 12, one
// shared-memory buffer, one CTA for up to two thousand points and clusters of 2, 4 or 8 CTAs above;
// see there).  The kernels of one line per CTA (k_fft_lines: radices 8 and 4 for the power of two, 5, 3,
// the symmetric 7 and 11, 2 only for n = 2 * odd; about n / 8 threads, two ping-pong buffers;
// k_fft_lines_cluster: split lines on 2 or 4 CTAs) remain for the sides where they are as fast or
// faster: see pair_plan and make_side.  The 2-D plane transform is a pass over rows (contiguous)
// and a pass over columns.  On the image side planes are complex128 (converted around the pairs'
// passes; the line kernels split and join on load and store); on the uv side they are complex128
// or, for the (de)gridding kernels in pair arithmetic, float pairs.
// Transforms are unnormalised, forward = e^{-2 pi i}, like cuFFT's.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "df64.cuh"
#include "fft_engine.cuh"
#include "host_math.h"
#include "wgrid_internal.h"

namespace wg {

// df64 constants of the small DFT kernels
struct DftConst {
  dd c31;            // sin(2 pi / 3)
  dd c51, c52;       // cos(2 pi / 5), cos(4 pi / 5)
  dd s51, s52;       // sin(2 pi / 5), sin(4 pi / 5)
  dd r2;             // sqrt(2) / 2
  dd c7[3], s7[3];   // cos, sin (2 pi k / 7), k = 1 .. 3
  dd c11[5], s11[5]; // cos, sin (2 pi k / 11), k = 1 .. 5
};

constexpr int kMaxStages = 24;
struct FftLine {
  int n;                     // transform length held by one CTA (half the line when split)
  int nst;                   // number of radix stages
  int threads;               // CTA size of the line kernel (about n / 8)
  int radix[kMaxStages];
  const float4* tw;          // e^{-2 pi i t / n}, t = 0 .. n - 1, df64
  // split lines (length S n, S = split = 2 or 4, too long for one CTA's shared memory): CTA h
  // (h < S) of a line transforms y_h[j] = e^{-/+ 2 pi i j h / (S n)} sum_{r < S} x[j + r n]
  // e^{-/+ 2 pi i r h / S}, one radix-S decimation-in-frequency step applied while loading,
  // and its n outputs are the line's outputs S k + h.  split = 1: one CTA per line.
  int split;
  const float4* tw2;         // e^{-2 pi i t / (S n)}, t = 0 .. S n - 1, df64 (split lines only)
  DftConst k;
};

// W^(t) for the transform direction: table entry (forward) or its conjugate (inverse)
__device__ __forceinline__ cdd twiddle(const float4* __restrict__ tw, int t, bool fwd) {
  float4 v = __ldg(&tw[t]);
  cdd w = load_cdd(v);
  if (!fwd) w.i = dd_neg(w.i);
  return w;
}

__device__ __forceinline__ void dft2(cdd* x) {
  cdd a = c_add(x[0], x[1]), b = c_sub(x[0], x[1]);
  x[0] = a; x[1] = b;
}
__device__ __forceinline__ void dft4(cdd* x, bool fwd) {
  cdd t0 = c_add(x[0], x[2]), t1 = c_sub(x[0], x[2]);
  cdd t2 = c_add(x[1], x[3]), t3 = c_mul_mi(c_sub(x[1], x[3]), fwd);
  x[0] = c_add(t0, t2); x[2] = c_sub(t0, t2);
  x[1] = c_add(t1, t3); x[3] = c_sub(t1, t3);
}
__device__ __forceinline__ void dft8(cdd* x, bool fwd, const DftConst& k) {
  cdd e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
  dft4(e, fwd);
  dft4(o, fwd);
  // o_k *= W8^k, W8 = e^{-/+ 2 pi i / 8}
  {
    // k = 1: (1 -/+ i) / sqrt2
    cdd a = o[1], r;
    if (fwd) { r.r = dd_add(a.r, a.i); r.i = dd_sub(a.i, a.r); }
    else { r.r = dd_sub(a.r, a.i); r.i = dd_add(a.i, a.r); }
    o[1] = c_scale(r, k.r2);
    o[2] = c_mul_mi(o[2], fwd);
    // k = 3: (-1 -/+ i) / sqrt2
    a = o[3];
    if (fwd) { r.r = dd_sub(a.i, a.r); r.i = dd_neg(dd_add(a.r, a.i)); }
    else { r.r = dd_neg(dd_add(a.r, a.i)); r.i = dd_sub(a.r, a.i); }
    o[3] = c_scale(r, k.r2);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    x[q] = c_add(e[q], o[q]);
    x[q + 4] = c_sub(e[q], o[q]);
  }
}
__device__ __forceinline__ void dft3(cdd* x, bool fwd, const DftConst& k) {
  cdd t1 = c_add(x[1], x[2]);
  cdd y0 = c_add(x[0], t1);
  dd half = dd_make(0.5f, 0.f);
  cdd t2 = c_sub(x[0], c_scale(t1, half));
  cdd t3 = c_mul_mi(c_scale(c_sub(x[1], x[2]), k.c31), fwd);   // -/+ i s (x1 - x2)
  x[0] = y0;
  x[1] = c_add(t2, t3);
  x[2] = c_sub(t2, t3);
}
__device__ __forceinline__ void dft5(cdd* x, bool fwd, const DftConst& k) {
  cdd t1 = c_add(x[1], x[4]), t2 = c_add(x[2], x[3]);
  cdd t3 = c_sub(x[1], x[4]), t4 = c_sub(x[2], x[3]);
  cdd y0 = c_add(x[0], c_add(t1, t2));
  cdd a1 = c_add(x[0], c_add(c_scale(t1, k.c51), c_scale(t2, k.c52)));
  cdd a2 = c_add(x[0], c_add(c_scale(t1, k.c52), c_scale(t2, k.c51)));
  cdd b1 = c_add(c_scale(t3, k.s51), c_scale(t4, k.s52));
  cdd b2 = c_sub(c_scale(t3, k.s52), c_scale(t4, k.s51));
  cdd ib1 = c_mul_mi(b1, fwd), ib2 = c_mul_mi(b2, fwd);   // -/+ i b
  x[0] = y0;
  x[1] = c_add(a1, ib1);
  x[4] = c_sub(a1, ib1);
  x[2] = c_add(a2, ib2);
  x[3] = c_sub(a2, ib2);
}
// odd radix R (7, 11): with a_k = x_k + x_{R-k} and b_k = x_k - x_{R-k} (k = 1 .. P = (R - 1) / 2),
//   y_q = x_0 + sum_k a_k cos(2 pi k q / R) -/+ i sum_k b_k sin(2 pi k q / R),
// and y_{R-q} the same with the other sign of the sine sum (forward: minus for y_q); the sums
// are chains of dd_fma against the pair constants (4 P^2 of them instead of the (R - 1)^2
// complex products of a plain DFT)
template <int R>
__device__ __forceinline__ void dft_odd(cdd* x, bool fwd, const dd* cs, const dd* sn) {
  constexpr int P = (R - 1) / 2;
  cdd a[P], b[P];
#pragma unroll
  for (int k = 1; k <= P; ++k) {
    a[k - 1] = c_add(x[k], x[R - k]);
    b[k - 1] = c_sub(x[k], x[R - k]);
  }
  cdd y0 = x[0];
#pragma unroll
  for (int k = 0; k < P; ++k) y0 = c_add(y0, a[k]);
#pragma unroll
  for (int q = 1; q <= P; ++q) {
    cdd re = x[0], im;
    im.r = dd_make(0.f, 0.f);
    im.i = im.r;
#pragma unroll
    for (int k = 1; k <= P; ++k) {
      const int m = (k * q) % R;
      const int mm = m <= P ? m : R - m;
      const dd c = cs[mm - 1];
      const dd sv = m <= P ? sn[mm - 1] : dd_neg(sn[mm - 1]);
      re.r = dd_fma(a[k - 1].r, c, re.r);
      re.i = dd_fma(a[k - 1].i, c, re.i);
      im.r = dd_fma(b[k - 1].r, sv, im.r);
      im.i = dd_fma(b[k - 1].i, sv, im.i);
    }
    const cdd mi = c_mul_mi(im, true);   // -i im
    x[q] = fwd ? c_add(re, mi) : c_sub(re, mi);
    x[R - q] = fwd ? c_sub(re, mi) : c_add(re, mi);
  }
  x[0] = y0;
}

template <int R>
__device__ __forceinline__ void butterfly(cdd* x, bool fwd, const FftLine& L) {
  if constexpr (R == 2) dft2(x);
  else if constexpr (R == 3) dft3(x, fwd, L.k);
  else if constexpr (R == 4) dft4(x, fwd);
  else if constexpr (R == 5) dft5(x, fwd, L.k);
  else if constexpr (R == 8) dft8(x, fwd, L.k);
  else if constexpr (R == 7) dft_odd<7>(x, fwd, L.k.c7, L.k.s7);
  else dft_odd<11>(x, fwd, L.k.c11, L.k.s11);
}


// One radix-R Stockham stage of a length-n line: butterfly j (j = tid, tid + T, ...) reads
// src[j + kk M], twiddles, transforms and writes dst[(j / Ns) Ns R + j mod Ns + q Ns].
// Shared-memory position of line element e: the low three bits of e are XORed with the next
// three (swz = 7, lines whose length is a multiple of 8), so that the stride-R writes of the
// first stages spread over the banks; a permutation within aligned groups of 8 elements.
__device__ __forceinline__ int swizzle(int e, int swz) { return e ^ ((e >> 3) & swz); }

template <int R>
__device__ __forceinline__ void stage(const float4* __restrict__ src, float4* __restrict__ dst,
                                      int n, int Ns, bool fwd, const FftLine& L, int swz) {
  const int M = n / R;
  const int tstep = n / (Ns * R);
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    const int jq = j / Ns, jm = j - jq * Ns;
    cdd x[R];
#pragma unroll
    for (int kk = 0; kk < R; ++kk) x[kk] = load_cdd(src[swizzle(j + kk * M, swz)]);
    if (Ns > 1) {
      // jm * kk * tstep < Ns * R * tstep = n: no reduction needed
#pragma unroll
      for (int kk = 1; kk < R; ++kk) x[kk] = c_mul(x[kk], twiddle(L.tw, jm * kk * tstep, fwd));
    }
    butterfly<R>(x, fwd, L);
    const int idx = jq * Ns * R + jm;
#pragma unroll
    for (int q = 0; q < R; ++q) dst[swizzle(idx + q * Ns, swz)] = store_cdd(x[q]);
  }
}

constexpr int kLoadBatch = 4;   // doubles a thread loads at once (mode 0)

// 16-byte asynchronous global -> shared copies (cp.async): a line's load is issued before the
// previous line's store, so the two overlap
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Transform lines g = blockIdx.x, blockIdx.x + gridDim.x, ... < nlines (a persistent CTA): line
// g is line g mod lines_per_plane of plane g / lines_per_plane, element i at global offset
// plane * plane_elems + line * line_stride + i * elem_stride (complex elements).  The plane's
// lines from `split` on are shifted by `skip` (a pass over the first and last rows of a plane
// only, skipping the middle).  mode 0: load doubles, store df64; mode 1: load df64, store
// doubles; mode 2: load and store df64.  Elements lhalf .. n - lhalf - 1 are known zeros and not
// loaded, elements shalf .. n - shalf - 1 are not stored (lhalf = shalf = n: everything).  Two
// n-element shared-memory buffers (ping-pong); with kAsync, after the last stage the buffer the
// stages no longer read receives the next line (asynchronous copies) while the result is stored
// (a line loaded through registers, kAsync false, gains nothing from it: those launches run one
// line per CTA).  kAll
// adds the rare radices 2, 7 and 11, kept out of the common instance so that its register
// allocation is not burdened with them.
template <int TMAX, int MINB, bool kAll, bool kAsync, bool kSplit>
__global__ void __launch_bounds__(TMAX, MINB)
k_fft_lines(const __grid_constant__ FftLine L, void* __restrict__ data, int64_t plane_elems,
            int lines_per_plane, int64_t line_stride, int64_t elem_stride, int mode, int fwd,
            int split, int skip, int lhalf, int shalf, int64_t nlines) {
  extern __shared__ __align__(16) float4 fsm[];
  const int n = L.n;
  const int S = kSplit ? L.split : 1;      // CTAs per line
  const int nfull = S * n;                 // elements of the whole line
  const int T = blockDim.x;
  const int swz = (n & 7) == 0 ? 7 : 0;
  float4* src = fsm;
  float4* dst = fsm + n;
  auto line_base = [&](int64_t gl) -> int64_t {
    gl /= S;                               // S CTAs per line, h = gl mod S
    const int64_t plane = gl / lines_per_plane;
    int line = (int)(gl - plane * lines_per_plane);
    if (line >= split) line += skip;
    return plane * plane_elems + (int64_t)line * line_stride;
  };
  // line gl into buffer b, each thread its elements i = tid, tid + T, ...; known zeros are
  // written directly.  kAsync (pairs, modes 1 and 2): asynchronous copies, completed by the
  // thread's cp_async_wait_all.  Otherwise loaded kLoadBatch at a time through registers, doubles
  // (mode 0) split into float pairs on the way.
  // element i of the whole line as a df64 complex value (0 in the known-zero range)
  auto load_elem = [&](const float4* g4, int64_t base, int i) -> cdd {
    if (i >= lhalf && i < nfull - lhalf) {
      cdd z; z.r = dd_make(0.f, 0.f); z.i = z.r;
      return z;
    }
    const float4 v = g4[base + (int64_t)i * elem_stride];
    if (mode == 0) {
      const double2 d = make_double2(__hiloint2double(__float_as_int(v.y), __float_as_int(v.x)),
                                     __hiloint2double(__float_as_int(v.w), __float_as_int(v.z)));
      cdd x; x.r = split_double(d.x); x.i = split_double(d.y);
      return x;
    }
    return load_cdd(v);
  };
  auto issue = [&](int64_t gl, float4* b) {
    const int64_t base = line_base(gl);
    const float4* g4 = reinterpret_cast<const float4*>(data);
    if constexpr (kSplit) {   // the decimation step of this CTA's part (see FftLine)
      const int h = (int)(gl % S);
      const bool f = fwd != 0;
#pragma unroll 2
      for (int j = threadIdx.x; j < n; j += T) {
        // output h of the radix-S DFT only (h is the same for the whole CTA)
        cdd y;
        if (S == 2) {
          const cdd x0 = load_elem(g4, base, j), x1 = load_elem(g4, base, j + n);
          y = h == 0 ? c_add(x0, x1) : c_sub(x0, x1);
        } else {
          cdd x4[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) x4[r] = load_elem(g4, base, j + r * n);
          if ((h & 1) == 0) {
            const cdd t0 = c_add(x4[0], x4[2]), t2 = c_add(x4[1], x4[3]);
            y = h == 0 ? c_add(t0, t2) : c_sub(t0, t2);
          } else {
            const cdd t1 = c_sub(x4[0], x4[2]), t3 = c_mul_mi(c_sub(x4[1], x4[3]), f);
            y = h == 1 ? c_add(t1, t3) : c_sub(t1, t3);
          }
        }
        if (h > 0) y = c_mul(y, twiddle(L.tw2, j * h, f));
        b[swizzle(j, swz)] = store_cdd(y);
      }
      return;
    }
    if (kAsync) {
      for (int i = threadIdx.x; i < n; i += T) {
        float4* d = b + swizzle(i, swz);
        if (i < lhalf || i >= n - lhalf) cp_async16(d, g4 + base + i * elem_stride);
        else *d = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      cp_async_commit();
      return;
    }
    for (int i0 = threadIdx.x; i0 < n; i0 += kLoadBatch * T) {
      float4 v[kLoadBatch];
#pragma unroll
      for (int k = 0; k < kLoadBatch; ++k) {
        const int i = i0 + k * T;
        if (i < n) v[k] = (i < lhalf || i >= n - lhalf) ? g4[base + i * elem_stride]
                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < kLoadBatch; ++k) {
        const int i = i0 + k * T;
        if (i < n) {
          if (mode == 0) {
            const double2 d = make_double2(__hiloint2double(__float_as_int(v[k].y), __float_as_int(v[k].x)),
                                           __hiloint2double(__float_as_int(v[k].w), __float_as_int(v[k].z)));
            cdd x; x.r = split_double(d.x); x.i = split_double(d.y);
            b[swizzle(i, swz)] = store_cdd(x);
          } else {
            b[swizzle(i, swz)] = v[k];
          }
        }
      }
    }
  };
  const bool f = fwd != 0;
  // the radix stages in the two buffers; the result ends in src
  auto run_stages = [&]() {
    int Ns = 1;
    for (int s = 0; s < L.nst; ++s) {
      const int R = L.radix[s];
      switch (R) {
        case 3: stage<3>(src, dst, n, Ns, f, L, swz); break;
        case 4: stage<4>(src, dst, n, Ns, f, L, swz); break;
        case 5: stage<5>(src, dst, n, Ns, f, L, swz); break;
        case 8: stage<8>(src, dst, n, Ns, f, L, swz); break;
        default:
          if (kAll) {
            if (R == 2) stage<2>(src, dst, n, Ns, f, L, swz);
            else if (R == 7) stage<7>(src, dst, n, Ns, f, L, swz);
            else stage<11>(src, dst, n, Ns, f, L, swz);
          }
          break;
      }
      __syncthreads();
      float4* t = src; src = dst; dst = t;
      Ns *= R;
    }
  };
  // result element i of this CTA is element i (or, split, 2 i + h) of the line
  auto store_line = [&](int64_t gl) {
    const int64_t base = line_base(gl);
    const int h = (int)(gl % S), st = S;
    if (mode != 1) {
      float4* out = reinterpret_cast<float4*>(data) + base;
      for (int i = threadIdx.x; i < n; i += T) {
        const int o = st * i + h;
        if (o < shalf || o >= nfull - shalf) out[(int64_t)o * elem_stride] = src[swizzle(i, swz)];
      }
    } else {
      double2* out = reinterpret_cast<double2*>(data) + base;
      for (int i = threadIdx.x; i < n; i += T) {
        const int o = st * i + h;
        if (o >= shalf && o < nfull - shalf) continue;   // not needed downstream
        cdd x = load_cdd(src[swizzle(i, swz)]);
        double2 v; v.x = join_double(x.r); v.y = join_double(x.i);
        out[(int64_t)o * elem_stride] = v;
      }
    }
  };
  int64_t gl = blockIdx.x;
  if (gl >= nlines) return;
  if constexpr (!kAsync) {   // one line (or half line) per CTA
    issue(gl, src);
    __syncthreads();
    run_stages();
    store_line(gl);
    return;
  }
  issue(gl, src);
  cp_async_wait_all();
  __syncthreads();
  for (;;) {
    run_stages();
    // the result is in src; dst is no longer read: the next line's copies go there while the
    // result is stored
    const int64_t gn = gl + gridDim.x;
    const bool more = gn < nlines;
    if (more) issue(gn, dst);
    store_line(gl);
    if (!more) break;
    cp_async_wait_all();
    __syncthreads();   // the next line is in place everywhere, and src is no longer read
    float4* t = src; src = dst; dst = t;
    gl = gn;
  }
}

// Split lines on a thread-block cluster of S = L.split CTAs (2 or 4): CTA h copies points
// [h n, h n + n) of its line into shared memory with asynchronous 16-byte copies (all of them
// in flight at once; known zeros written directly, doubles split into float pairs in place),
// the cluster exchanges the parts through distributed shared memory for the radix-S
// decimation-in-frequency step (CTA h forms only its own y_h, see FftLine), and each CTA then
// transforms its n points like a one-CTA line and stores the line's outputs S k + h.  The
// register-path split of k_fft_lines reads all S n points of the line in every CTA with few
// loads in flight; it remains the fallback when a cluster cannot be launched.
template <int TMAX, int MINB, bool kAll>
__global__ void __launch_bounds__(TMAX, MINB)
k_fft_lines_cluster(const __grid_constant__ FftLine L, void* __restrict__ data, int64_t plane_elems,
                    int lines_per_plane, int64_t line_stride, int64_t elem_stride, int mode,
                    int fwd, int split, int skip, int lhalf, int shalf) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) float4 fsm[];
  cg::cluster_group cl = cg::this_cluster();
  const int n = L.n, S = L.split, nfull = S * n, T = blockDim.x;
  const int swz = (n & 7) == 0 ? 7 : 0;
  const bool f = fwd != 0;
  const int h = (int)cl.block_rank();           // cluster dims (S, 1, 1): blockIdx.x mod S
  const int64_t lid = blockIdx.x / (unsigned)S;
  const int64_t plane = lid / lines_per_plane;
  int line = (int)(lid - plane * lines_per_plane);
  if (line >= split) line += skip;
  const int64_t base = plane * plane_elems + (int64_t)line * line_stride;
  float4* A = fsm;
  float4* B = fsm + n;
  const float4* g4 = reinterpret_cast<const float4*>(data);
  const int i0 = h * n;
  for (int j = threadIdx.x; j < n; j += T) {
    const int i = i0 + j;
    float4* d = A + swizzle(j, swz);
    if (i < lhalf || i >= nfull - lhalf) cp_async16(d, g4 + base + (int64_t)i * elem_stride);
    else *d = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  cp_async_commit();
  cp_async_wait_all();
  if (mode == 0) {   // doubles in: each split into a float pair in place (the same 16 bytes)
    for (int j = threadIdx.x; j < n; j += T) {
      const int i = i0 + j;
      if (i >= lhalf && i < nfull - lhalf) continue;
      float4* d = A + swizzle(j, swz);
      const float4 v = *d;
      const double2 dv = make_double2(__hiloint2double(__float_as_int(v.y), __float_as_int(v.x)),
                                      __hiloint2double(__float_as_int(v.w), __float_as_int(v.z)));
      cdd x; x.r = split_double(dv.x); x.i = split_double(dv.y);
      *d = store_cdd(x);
    }
  }
  cl.sync();         // every part is in place
  const float4* P[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) P[r] = cl.map_shared_rank(A, (unsigned)(r < S ? r : 0));
  for (int j = threadIdx.x; j < n; j += T) {
    const int off = swizzle(j, swz);
    cdd y;
    if (S == 2) {
      const cdd x0 = load_cdd(P[0][off]), x1 = load_cdd(P[1][off]);
      y = h == 0 ? c_add(x0, x1) : c_sub(x0, x1);
    } else {
      cdd x4[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) x4[r] = load_cdd(P[r][off]);
      if ((h & 1) == 0) {
        const cdd t0 = c_add(x4[0], x4[2]), t2 = c_add(x4[1], x4[3]);
        y = h == 0 ? c_add(t0, t2) : c_sub(t0, t2);
      } else {
        const cdd t1 = c_sub(x4[0], x4[2]), t3 = c_mul_mi(c_sub(x4[1], x4[3]), f);
        y = h == 1 ? c_add(t1, t3) : c_sub(t1, t3);
      }
    }
    if (h > 0) y = c_mul(y, twiddle(L.tw2, j * h, f));
    B[off] = store_cdd(y);
  }
  cl.sync();         // the other CTAs have read this CTA's part: A is free for the stages
  float4* src = B;
  float4* dst = A;
  int Ns = 1;
  for (int st = 0; st < L.nst; ++st) {
    const int R = L.radix[st];
    switch (R) {
      case 3: stage<3>(src, dst, n, Ns, f, L, swz); break;
      case 4: stage<4>(src, dst, n, Ns, f, L, swz); break;
      case 5: stage<5>(src, dst, n, Ns, f, L, swz); break;
      case 8: stage<8>(src, dst, n, Ns, f, L, swz); break;
      default:
        if (kAll) {
          if (R == 2) stage<2>(src, dst, n, Ns, f, L, swz);
          else if (R == 7) stage<7>(src, dst, n, Ns, f, L, swz);
          else stage<11>(src, dst, n, Ns, f, L, swz);
        }
        break;
    }
    __syncthreads();
    float4* t = src; src = dst; dst = t;
    Ns *= R;
  }
  // result element i of this CTA is element S i + h of the line
  if (mode != 1) {
    float4* out = reinterpret_cast<float4*>(data) + base;
    for (int i = threadIdx.x; i < n; i += T) {
      const int o = S * i + h;
      if (o < shalf || o >= nfull - shalf) out[(int64_t)o * elem_stride] = src[swizzle(i, swz)];
    }
  } else {
    double2* out = reinterpret_cast<double2*>(data) + base;
    for (int i = threadIdx.x; i < n; i += T) {
      const int o = S * i + h;
      if (o >= shalf && o < nfull - shalf) continue;   // not needed downstream
      const cdd x = load_cdd(src[swizzle(i, swz)]);
      double2 v; v.x = join_double(x.r); v.y = join_double(x.i);
      out[(int64_t)o * elem_stride] = v;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Pairs of lines (fft_engine.cuh): the kernel of every line that splits into 1, 2, 4 or 8 parts
// of at most kPairMaxPart points with radices up to 12
//
// A CTA (a cluster of S CTAs when the line is split) transforms two lines of a plane at once,
// packed into the two halves of the FP32 x2 instructions.  Bound: the FP32 pipes.  Layout:
//  * one shared-memory buffer of n packed points, two 16-byte arrays (real pairs, imaginary
//    pairs); a stage reads its butterflies into registers, synchronises and writes them back in
//    place (registers hold about 8 - 12 points per thread, so a second buffer would only cost
//    CTAs per SM);
//  * the first stage reads its points straight from global memory and the last one writes its
//    results there, so a three-stage line crosses shared memory twice;
//  * a split line's radix-S decimation-in-frequency step is done where the points are loaded:
//    CTA h takes the j-range [h n / S, (h + 1) n / S), forms all S outputs of each butterfly and
//    writes output r into CTA r's buffer through distributed shared memory;
//  * where one pair leaves lanes of its warps idle, several share a CTA (kPack, see pair_pack);
//  * radices up to 12 (10, 6 and 12 by coprime factors, no inner twiddles): 1728 = 12 12 12 in
//    three stages instead of 8 8 3 3 3 in five;
//  * twiddles are stored per stage in the order the threads read them, each float twice.
// ---------------------------------------------------------------------------------------
constexpr int kPairMaxPart = 2048, kPairStages = 12;

struct PairLine {
  int n, S, T, cls, nst;         // points per CTA, CTAs per line, threads, register class, stages
  int P, TL;                     // pairs of lines per CTA, threads of a pair
  int radix[kPairStages];
  unsigned magic[kPairStages];   // j / Ns = umulhi(j, magic) for Ns > 1
  int twofs[kPairStages];        // first entry of the stage's twiddles, entry (kk - 1) Ns + jm
  const float4* tw;              // two float4 per entry: (rh, rh, rl, rl), (ih, ih, il, il)
  const float4* tw2;             // split lines: e^{-2 pi i j r / (S n)} at entry (r - 1) n + j
};

// butterflies of radix R a thread holds at once: class 9 about 8 points, class 12 about 12
__host__ __device__ constexpr int pair_nb(int cls, int R) {
  return cls == 9 ? (R >= 5 ? 1 : R == 4 ? 2 : R == 3 ? 3 : 4)
                  : (R >= 7 ? 1 : R >= 5 ? 2 : R == 4 ? 3 : R == 3 ? 4 : 5);
}

struct PairIo {
  float4* data;
  int64_t base0, base1, es;      // the two lines' first elements, element stride
  int nfull, lhalf, shalf;
  bool inv, two;                 // inverse: real and imaginary parts exchanged; second line exists
  __device__ __forceinline__ Cx<d2> load(int o) const {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (o < lhalf || o >= nfull - lhalf) {
      a = data[base0 + (int64_t)o * es];
      if (two) b = data[base1 + (int64_t)o * es];
    }
    Cx<d2> x;
    x.r.h = f2_make(inv ? a.z : a.x, inv ? b.z : b.x);
    x.r.l = f2_make(inv ? a.w : a.y, inv ? b.w : b.y);
    x.i.h = f2_make(inv ? a.x : a.z, inv ? b.x : b.z);
    x.i.l = f2_make(inv ? a.y : a.w, inv ? b.y : b.w);
    return x;
  }
  __device__ __forceinline__ void store(int o, const Cx<d2>& x) const {
    if (o >= shalf && o < nfull - shalf) return;   // not needed downstream
    const float2 rh = f2_split(x.r.h), rl = f2_split(x.r.l), ih = f2_split(x.i.h), il = f2_split(x.i.l);
    data[base0 + (int64_t)o * es] = inv ? make_float4(ih.x, il.x, rh.x, rl.x)
                                        : make_float4(rh.x, rl.x, ih.x, il.x);
    if (two)
      data[base1 + (int64_t)o * es] = inv ? make_float4(ih.y, il.y, rh.y, rl.y)
                                          : make_float4(rh.y, rl.y, ih.y, il.y);
  }
};

// shared-memory slot of point e: the low three bits XORed with the next three (a permutation
// inside aligned groups of 8; the buffers are allocated in whole groups)
__device__ __forceinline__ int pair_slot(int e) { return e ^ ((e >> 3) & 7); }

__device__ __forceinline__ Cx<d2> pair_get(const ulonglong2* sr, const ulonglong2* si, int e) {
  const int s = pair_slot(e);
  const ulonglong2 a = sr[s], b = si[s];
  return Cx<d2>{{{a.x}, {a.y}}, {{b.x}, {b.y}}};
}
__device__ __forceinline__ void pair_put(ulonglong2* sr, ulonglong2* si, int e, const Cx<d2>& x) {
  const int s = pair_slot(e);
  sr[s] = make_ulonglong2(x.r.h.v, x.r.l.v);
  si[s] = make_ulonglong2(x.i.h.v, x.i.l.v);
}
__device__ __forceinline__ Tw<d2> pair_tw(const float4* __restrict__ tw, int t) {
  const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(tw) + 2 * t);
  const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2*>(tw) + 2 * t + 1);
  return Tw<d2>{{a.x}, {a.y}, {b.x}, {b.y}};
}

struct PairStageArgs {
  ulonglong2 *sr, *si;
  const float4* tw;              // the stage's twiddles
  int n, Ns;
  unsigned magic;
  int S, h;                      // the line's element S o + h is result o of this CTA
  int j, TL;                     // thread within the pair's, and how many these are
};
// One stage: read the butterflies and transform them, synchronise, write them back in place.
// kIn: 0 the first stage of a whole line, from global memory; 1 the first stage of a split line,
// from the buffer that the decimation step has filled (both without twiddles); 2 a later stage.
// kLast: results to global memory.  (Separate instances: with both destinations in one body the
// compiler keeps the results in registers for both and spills.)
// Idle lanes of a warp repeat the last butterfly and store nothing, and the barrier between
// reading and writing stands inside the branch that skips idle warps: points that live across
// the end of a branch are spilled, all of them.
template <int R, int kIn, bool kLast>
__device__ __forceinline__ int pair_compute(const PairIo& io, const PairStageArgs& a, int j, int M,
                                            int Ns, Cx<d2>* x) {
#pragma unroll
  for (int k = 0; k < R; ++k)
    x[k] = kIn == 0 ? io.load(j + k * M) : pair_get(a.sr, a.si, j + k * M);
  int o = j * R;
  if constexpr (kIn == 2) {
    const int jq = kLast ? 0 : (int)__umulhi((unsigned)j, a.magic), jm = j - jq * Ns;
    o = jq * Ns * R + jm;
#pragma unroll
    for (int k = 1; k < R; ++k) x[k] = cx_mul(x[k], pair_tw(a.tw, jm + (k - 1) * Ns));
  }
  dft<R>(x);
  return o;
}
template <int R, bool kLast>
__device__ __forceinline__ void pair_result(const PairIo& io, const PairStageArgs& a, int o, int Ns,
                                            const Cx<d2>* x) {
#pragma unroll
  for (int q = 0; q < R; ++q) {
    if (kLast) io.store(a.S * (o + q * Ns) + a.h, x[q]);
    else pair_put(a.sr, a.si, o + q * Ns, x[q]);
  }
}
// all warps of the CTA arrive, from either side of a warp-uniform branch
__device__ __forceinline__ void pair_barrier() { asm volatile("barrier.sync 0;" ::: "memory"); }

// NB: butterflies per thread, exactly as many as the CTA's threads need (idle rounds cost as much
// as full ones)
template <int R, int NB, int kIn, bool kLast, bool kPack>
__device__ __forceinline__ void pair_stage_nb(const PairIo& io, const PairStageArgs& a) {
  constexpr bool kWait = kIn != 0 && !kLast;   // every point of the buffer is read before it is written
  const int M = a.n / R, T = kPack ? a.TL : blockDim.x, Ns = kIn == 2 ? a.Ns : 1;
  const int j = kPack ? a.j : threadIdx.x;
  if constexpr (NB == 1) {
    if (kPack ? __any_sync(0xffffffffu, j < M) : (j & ~31) < M) {
      Cx<d2> x[R];
      const int o = pair_compute<R, kIn, kLast>(io, a, min(j, M - 1), M, Ns, x);
      if (kWait) pair_barrier();
      if (j < M) pair_result<R, kLast>(io, a, o, Ns, x);
    } else if (kWait) {
      pair_barrier();
    }
  } else {
    Cx<d2> x[NB][R];
    int o[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b)
      o[b] = pair_compute<R, kIn, kLast>(io, a, min(j + b * T, M - 1), M, Ns, x[b]);
    if (kWait) pair_barrier();
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if ((!kPack || j < T) && j + b * T < M) pair_result<R, kLast>(io, a, o[b], Ns, x[b]);
  }
  if (!kLast) pair_barrier();
}
template <int R, int CLS, int kIn, bool kLast, bool kPack>
__device__ __forceinline__ void pair_stage(const PairIo& io, const PairStageArgs& a) {
  constexpr int kMost = pair_nb(CLS, R);
  const int M = a.n / R, T = kPack ? a.TL : blockDim.x;
  if (kMost == 1 || M <= T) pair_stage_nb<R, 1, kIn, kLast, kPack>(io, a);
  else if (kMost == 2 || M <= 2 * T) pair_stage_nb<R, kMost < 2 ? 1 : 2, kIn, kLast, kPack>(io, a);
  else if (kMost == 3 || M <= 3 * T) pair_stage_nb<R, kMost < 3 ? 1 : 3, kIn, kLast, kPack>(io, a);
  else pair_stage_nb<R, kMost < 4 ? 1 : kMost, kIn, kLast, kPack>(io, a);
}
template <int CLS, int kIn, bool kLast, bool kPack>
__device__ __forceinline__ void pair_dispatch(int R, const PairIo& io, const PairStageArgs& a) {
  if constexpr (kIn != 2) {   // first radix: 8 or 9 (class 9), 8 to 12 (class 12), see pair_plan
    if constexpr (CLS == 9) {
      if (R == 8) pair_stage<8, CLS, kIn, kLast, kPack>(io, a);
      else pair_stage<9, CLS, kIn, kLast, kPack>(io, a);
    } else {
      switch (R) {
        case 8: pair_stage<8, CLS, kIn, kLast, kPack>(io, a); break;
        case 9: pair_stage<9, CLS, kIn, kLast, kPack>(io, a); break;
        case 10: pair_stage<10, CLS, kIn, kLast, kPack>(io, a); break;
        case 11: pair_stage<11, CLS, kIn, kLast, kPack>(io, a); break;
        default: pair_stage<12, CLS, kIn, kLast, kPack>(io, a); break;
      }
    }
  } else {
    switch (R) {
      case 2: pair_stage<2, CLS, kIn, kLast, kPack>(io, a); break;
      case 3: pair_stage<3, CLS, kIn, kLast, kPack>(io, a); break;
      case 4: pair_stage<4, CLS, kIn, kLast, kPack>(io, a); break;
      case 5: pair_stage<5, CLS, kIn, kLast, kPack>(io, a); break;
      case 6: pair_stage<6, CLS, kIn, kLast, kPack>(io, a); break;
      case 7: pair_stage<7, CLS, kIn, kLast, kPack>(io, a); break;
      case 8: pair_stage<8, CLS, kIn, kLast, kPack>(io, a); break;
      case 9: pair_stage<9, CLS, kIn, kLast, kPack>(io, a); break;
      default:
        if constexpr (CLS == 12) {
          if (R == 10) pair_stage<10, CLS, kIn, kLast, kPack>(io, a);
          else if (R == 11) pair_stage<11, CLS, kIn, kLast, kPack>(io, a);
          else pair_stage<12, CLS, kIn, kLast, kPack>(io, a);
        }
        break;
    }
  }
}

// the radix-S decimation step of a split line (see above); the cluster barriers are the caller's
template <int S>
__device__ __forceinline__ void pair_split(const PairLine& L, const PairIo& io, ulonglong2* sr,
                                           ulonglong2* si, int h) {
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int n = L.n, per = (n + S - 1) / S;
  const int j1 = min(n, (h + 1) * per);
  for (int j = h * per + threadIdx.x; j < j1; j += blockDim.x) {
    Cx<d2> x[S];
#pragma unroll
    for (int r = 0; r < S; ++r) x[r] = io.load(j + r * n);
    dft<S>(x);
#pragma unroll
    for (int r = 0; r < S; ++r) {
      if (r > 0) x[r] = cx_mul(x[r], pair_tw(L.tw2, (r - 1) * n + j));
      pair_put(cl.map_shared_rank(sr, r), cl.map_shared_rank(si, r), j, x[r]);
    }
  }
}

// Lines q = 2 p, 2 p + 1 (p = pair index in the plane) of `lines` per plane; line q >= split is
// shifted by skip.  lhalf, shalf as in k_fft_lines; float pairs in and out.
template <int CLS, int TMAX, bool kPack>
__global__ void __launch_bounds__(TMAX, 2)
k_fft_pairs(const __grid_constant__ PairLine L, float4* __restrict__ data, int64_t plane_elems,
            int lines, int64_t line_stride, int64_t elem_stride, int inv, int split, int skip,
            int lhalf, int shalf) {
  extern __shared__ __align__(16) float4 fsm[];
  const int S = L.S;
  const unsigned cid = S > 1 ? blockIdx.x / (unsigned)S : blockIdx.x;
  const int h = (int)(blockIdx.x - cid * S);   // rank in the cluster (S, 1, 1)
  const unsigned pairs = (unsigned)(lines + 1) / 2, groups = kPack ? (pairs + L.P - 1) / L.P : pairs;
  const unsigned plane = cid / groups;
  // threads past the last pair's are idle; pairs past the plane's last repeat it (they read and
  // write what it does, on the same sides of the barriers)
  const int sub = kPack ? min((int)threadIdx.x / L.TL, L.P - 1) : 0;
  const int at = (int)(cid - plane * groups);
  const int q0 = 2 * (kPack ? min(at * L.P + sub, (int)pairs - 1) : at), q1 = q0 + 1;
  PairIo io;
  io.data = data;
  const int64_t pb = (int64_t)plane * plane_elems;
  io.base0 = pb + (int64_t)(q0 < split ? q0 : q0 + skip) * line_stride;
  io.base1 = pb + (int64_t)(q1 < split ? q1 : q1 + skip) * line_stride;
  io.es = elem_stride;
  io.nfull = S * L.n;
  io.lhalf = lhalf; io.shalf = shalf;
  io.inv = inv != 0; io.two = q1 < lines;
  PairStageArgs a;
  const int room = (L.n + 7) & ~7;
  a.sr = reinterpret_cast<ulonglong2*>(fsm) + (kPack ? 2 * room * sub : 0);
  a.si = a.sr + room;
  if (kPack) { a.j = (int)threadIdx.x - sub * L.TL; a.TL = L.TL; }
  a.n = L.n; a.S = S; a.h = h;
  if (S > 1) {
    // every CTA of the cluster must have started before its buffer is written
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    if (S == 2) pair_split<2>(L, io, a.sr, a.si, h);
    else if (S == 4) pair_split<4>(L, io, a.sr, a.si, h);
    else pair_split<8>(L, io, a.sr, a.si, h);
    cl.sync();
    pair_dispatch<CLS, 1, false, kPack>(L.radix[0], io, a);
  } else {
    pair_dispatch<CLS, 0, false, kPack>(L.radix[0], io, a);
  }
  a.Ns = L.radix[0];
  int st = 1;
  for (; st < L.nst - 1; ++st) {
    a.tw = L.tw + 2 * L.twofs[st];
    a.magic = L.magic[st];
    pair_dispatch<CLS, 2, false, kPack>(L.radix[st], io, a);
    a.Ns *= L.radix[st];
  }
  a.tw = L.tw + 2 * L.twofs[st];
  pair_dispatch<CLS, 2, true, kPack>(L.radix[st], io, a);
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
static dd host_dd(long double v) {
  float h = (float)v;
  float l = (float)(v - (long double)h);
  dd x; x.h = h; x.l = l;
  return x;
}

// One side's transform: pairs of lines where the side allows it, else one line per CTA / cluster.
constexpr int kFewLines = 1024;   // lines of a pass, points of a line: see on_pairs
struct SideFft {
  bool pairs = false, lines = false;   // which kernels have tables
  bool fwd_lines = false;              // one line per CTA for the forward transform
  PairLine pl{};
  FftLine fl{};
  // twiddles of pl, then those of fl: each the line's, then (split lines) the decimation step's
  float4* tw = nullptr;
};
struct Df64Fft {
  int nu = 0, nv = 0;
  SideFft u, v;
};

// FP32 operations per point of a radix-R butterfly in double-float arithmetic (5, 10 and 12 as
// they measure, 10 % above their count)
static double pair_radix_ops(int R) {
  switch (R) {
    case 2: return 22; case 3: return 50; case 4: return 44; case 5: return 95; case 6: return 72;
    case 7: return 130; case 8: return 75; case 9: return 117; case 10: return 118;
    case 11: return 190; default: return 108;
  }
}
constexpr int pair_threads(int cls) { return cls == 9 ? 256 : 192; }   // CTA limit of a class
// Cheapest radices of n points for a register class, largest first: butterflies, 38 per twiddle
// product and about 75 per trip through shared memory (with its two barriers) from the second
// stage on; at least two stages, the first of radix 8 or more, all within the class's CTA size.
// Class 12 (168 registers) counts 1.18 times: it pays where it saves a stage (1200 points as 12 10
// 10 measured 1.2 times as fast as 8 6 5 5), else not (1344 as 12 7 4 4: 0.85 of 8 7 6 4).
static void pair_search(int m, int maxr, int depth, double cost, PairLine* cur, double* best,
                        PairLine* out) {
  if (m == 1) {
    if (cur->cls == 12) cost *= 1.18;
    if (cost >= *best || depth < 2 || cur->radix[0] < 8) return;
    int T = 32;
    for (int i = 0; i < depth; ++i) {
      const int per = cur->n / cur->radix[i], nb = pair_nb(cur->cls, cur->radix[i]);
      T = std::max(T, ((per + nb - 1) / nb + 31) / 32 * 32);
    }
    if (T > pair_threads(cur->cls)) return;
    *best = cost;
    *out = *cur;
    out->nst = depth;
    out->T = T;
    out->P = 1;
    out->TL = T;
    return;
  }
  if (depth == kPairStages) return;
  for (int R = std::min(maxr, cur->cls); R >= 2; --R) {
    if (m % R != 0) continue;
    cur->radix[depth] = R;
    pair_search(m / R, R, depth + 1,
                cost + pair_radix_ops(R) + (depth > 0 ? 38.0 * (R - 1) / R + 75.0 : 0.0), cur, best, out);
  }
}
static bool pair_part(int N, int S, PairLine* L) {
  if (N % S != 0 || N / S > kPairMaxPart) return false;
  double best = 1e30;
  for (int cls : {9, 12}) {
    PairLine cur;
    std::memset(&cur, 0, sizeof(cur));
    cur.n = N / S; cur.S = S; cur.cls = cls;
    pair_search(cur.n, cls, 0, 0.0, &cur, &best, L);
  }
  return best < 1e30;
}
// Radices, class and threads for a line of N points; false: the line kernels above.  Measured
// against those on the pruned transforms of square sides (forward / inverse, per plane): one CTA
// up to 2048 points (512: 7.1 -> 5.9 and 14.0 -> 6.2 us; 2048: 139 -> 108 and 150 -> 107 us).  From
// 3072 points on a cluster of four beats two where the parts are of class 9 and at most 160
// threads (3584: 1.23 / 1.11 times the line kernels' speed against 1.12 / 1.04; 3840 in parts of 192
// threads 1.04 / 0.97 against 1.11 / 1.07).  Left to one line per CTA, which is as fast or faster: up
// to 2048 points what one CTA cannot take (2016: 0.89 / 0.93), and between 3072 and 4096 points
// sides with a factor 11, or with 7 and 5 (3168: 1.08 / 0.95, 3520: 0.98 / 0.91, 3360: 1.02 / 0.86).
// Several pairs per CTA where their threads fill its warps better: as many as give the most pairs
// per SM, from 33 threads a pair up (576 points, 72 threads a pair: one to a CTA of 96 measured
// 0.95 / 1.66 times the line kernels' speed forward / inverse, two to a CTA of 160 1.04 / 1.77;
// 672, 112 threads: 1.19 / 1.86 alone and 1.09 / 1.74 with two, no more pairs per SM; 128, 16
// threads: 0.97 / 1.86 alone and 0.78 / 1.40 with four, too few CTAs).
static void pair_pack(PairLine* L) {
  int tl = 1;
  for (int i = 0; i < L->nst; ++i) {
    const int per = L->n / L->radix[i], nb = pair_nb(L->cls, L->radix[i]);
    tl = std::max(tl, (per + nb - 1) / nb);
  }
  if (tl <= 32) return;
  const int room = L->cls == 9 ? 512 : 384;   // threads an SM holds
  int best = room / L->T;
  for (int P = 2; P * tl <= pair_threads(L->cls) && P * ((L->n + 7) & ~7) <= kPairMaxPart; ++P) {
    const int T = (P * tl + 31) / 32 * 32;
    if (P * (room / T) > best) { best = P * (room / T); L->P = P; L->TL = tl; L->T = T; }
  }
}
static bool pair_plan(int N, PairLine* L) {
  if (N <= kPairMaxPart) {
    if (!pair_part(N, 1, L)) return false;
    pair_pack(L);
    return true;
  }
  if (N > 3072 && N < 4096 && (N % 11 == 0 || N % 35 == 0)) return false;
  if (N >= 3072 && pair_part(N, 4, L) && L->n <= 1024 && L->cls == 9 && L->T <= 160) return true;
  for (int S : {2, 4, 8})
    if (pair_part(N, S, L)) return true;
  return false;
}

// a root of unity as a twiddle entry (each float twice)
static void pair_entry(const UnitRoots& roots, int64_t t, float4* e) {
  float w[4];
  roots.pair(t, w);
  e[0] = make_float4(w[0], w[0], w[1], w[1]);
  e[1] = make_float4(w[2], w[2], w[3], w[3]);
}

// appends the line's twiddles; returns where those of the decimation step start
static size_t pair_table(PairLine* L, std::vector<float4>* table) {
  int entries = 0, Ns = 1;
  for (int s = 0; s < L->nst; ++s) {
    L->twofs[s] = entries;
    L->magic[s] = Ns > 1 ? (unsigned)(0x100000000ull / (unsigned)Ns) + 1u : 0u;
    if (Ns > 1) entries += (L->radix[s] - 1) * Ns;
    Ns *= L->radix[s];
  }
  const int own = entries;
  entries += (L->S - 1) * L->n;
  const size_t at = table->size();
  table->resize(at + 2 * (size_t)std::max(1, entries));
  float4* h = table->data() + at;
  const int64_t N = (int64_t)L->S * L->n;
  const UnitRoots roots(N);
  Ns = 1;
  for (int s = 0; s < L->nst; ++s) {
    const int R = L->radix[s];
    if (Ns > 1)
      for (int k = 1; k < R; ++k)
        for (int jm = 0; jm < Ns; ++jm)
          pair_entry(roots, (int64_t)jm * k * (N / ((int64_t)Ns * R)),
                     &h[2 * (size_t)(L->twofs[s] + (k - 1) * Ns + jm)]);
    Ns *= R;
  }
  for (int r = 1; r < L->S; ++r)
    for (int j = 0; j < L->n; ++j)
      pair_entry(roots, (int64_t)j * r, &h[2 * (size_t)(own + (r - 1) * L->n + j)]);
  return at + 2 * (size_t)own;
}

// Launch configuration of `blocks` CTAs (a multiple of L.S) of the pair kernel
struct PairLaunch {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  PairLaunch(const PairLine& L, unsigned blocks, cudaStream_t s) {
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3((unsigned)L.T);
    cfg.dynamicSmemBytes = 2 * sizeof(float4) * (size_t)((L.n + 7) & ~7) * L.P;
    cfg.stream = s;
    std::memset(attr, 0, sizeof(attr));
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)L.S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = L.S > 1 ? 1 : 0;
  }
  PairLaunch(const PairLaunch&) = delete;   // cfg points into the object
};

static cudaError_t pair_smem_attributes() {
  const int bytes = (int)(2 * sizeof(float4) * kPairMaxPart);
  cudaError_t e = cudaSuccess;
#define WG_SMEM_ATTR(...)                                                                        \
  if (e == cudaSuccess)                                                                          \
    e = cudaFuncSetAttribute(k_fft_pairs<__VA_ARGS__>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)
  WG_SMEM_ATTR(9, 256, false);  WG_SMEM_ATTR(9, 256, true);
  WG_SMEM_ATTR(12, 192, false); WG_SMEM_ATTR(12, 192, true);
#undef WG_SMEM_ATTR
  return e;
}

// whether the GPU, as the process sees it, can place a cluster of the line's CTAs at all (a share of
// it with few SMs to a cluster's domain may not): where it cannot, the line goes to the kernels of
// one line per CTA, which do without clusters when they must
static bool pair_cluster_fits(const PairLine& L) {
  if (L.S == 1) return true;
  const PairLaunch l(L, (unsigned)L.S, 0);
  int clusters = 0;
  const cudaError_t e = L.cls == 9
      ? cudaOccupancyMaxActiveClusters(&clusters, k_fft_pairs<9, 256, false>, &l.cfg)
      : cudaOccupancyMaxActiveClusters(&clusters, k_fft_pairs<12, 192, false>, &l.cfg);
  if (e == cudaSuccess) return clusters > 0;
  cudaGetLastError();
  return false;
}

static cudaError_t launch_pairs(const PairLine& L, double2* data, int64_t batch, int64_t plane,
                                int lines, int64_t line_stride, int64_t elem_stride, int fwd,
                                int split, int skip, int lhalf, int shalf, cudaStream_t s) {
  if (lines == 0 || batch == 0) return cudaSuccess;
  const int64_t blocks = batch * (((lines + 1) / 2 + L.P - 1) / L.P) * L.S;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  const PairLaunch l(L, (unsigned)blocks, s);
  float4* d = reinterpret_cast<float4*>(data);
  const int inv = fwd ? 0 : 1;
#define WG_PAIRS(C, TM, P)                                                                       \
  cudaLaunchKernelEx(&l.cfg, k_fft_pairs<C, TM, P>, L, d, plane, lines, line_stride, elem_stride, inv, \
                     split, skip, lhalf, shalf)
  if (L.P > 1) return L.cls == 9 ? WG_PAIRS(9, 256, true) : WG_PAIRS(12, 192, true);
  return L.cls == 9 ? WG_PAIRS(9, 256, false) : WG_PAIRS(12, 192, false);
#undef WG_PAIRS
}

// Two buffers of n df64 complex values in shared memory per CTA (two CTAs per SM up to n =
// 3584); split lines (df64_line_split) run on clusters of two or four CTAs.
static constexpr int64_t kMaxSide = kDf64MaxSide;

bool df64_fft_supported(int64_t nu, int64_t nv) { return df64_side_ok(nu) && df64_side_ok(nv); }

// e^{-2 pi i t / len}, t = 0 .. len - 1, as df64 (float4: re hi, re lo, im hi, im lo)
static void twiddles(int len, float4* h) {
  const UnitRoots roots(len);
  for (int t = 0; t < len; ++t) roots.pair(t, &h[t].x);
}

static DftConst dft_constants() {
  DftConst k;
  const long double pi = 3.141592653589793238462643383279L;
  k.c31 = host_dd(sinl(2 * pi / 3));
  k.c51 = host_dd(cosl(2 * pi / 5));
  k.c52 = host_dd(cosl(4 * pi / 5));
  k.s51 = host_dd(sinl(2 * pi / 5));
  k.s52 = host_dd(sinl(4 * pi / 5));
  k.r2 = host_dd(sqrtl(2.0L) / 2);
  for (int q = 1; q <= 3; ++q) {
    k.c7[q - 1] = host_dd(cosl(2 * pi * q / 7));
    k.s7[q - 1] = host_dd(sinl(2 * pi * q / 7));
  }
  for (int q = 1; q <= 5; ++q) {
    k.c11[q - 1] = host_dd(cosl(2 * pi * q / 11));
    k.s11[q - 1] = host_dd(sinl(2 * pi * q / 11));
  }
  return k;
}

// appends the line's twiddles
static cudaError_t line_table(int nline, FftLine* L, std::vector<float4>* table) {
  std::memset(L, 0, sizeof(*L));
  const int S = df64_line_split(nline);
  if (S == 0) return cudaErrorInvalidValue;
  const int n = nline / S;
  L->n = n;
  L->split = S;
  Df64LinePlan lp;
  if (!df64_line_plan(n, &lp) || lp.nst > kMaxStages) return cudaErrorInvalidValue;
  L->nst = lp.nst;
  L->threads = lp.threads;
  for (int i = 0; i < lp.nst; ++i) L->radix[i] = lp.radix[i];
  const size_t at = table->size();
  table->resize(at + n + (S > 1 ? nline : 0));
  twiddles(n, table->data() + at);
  if (S > 1) twiddles(nline, table->data() + at + n);
  static const DftConst k = dft_constants();
  L->k = k;
  return cudaSuccess;
}

// sides of the radices 2 and 5 only, which pairs take in four stages with idle lanes: forward
// and inverse at the pairs' speed against the lines', on square sides with pruning: 640 0.92 /
// 1.65, 800 0.98 / 1.44, 1280 1.02 / 1.28, 1600 0.92 / 1.10 (other sides from 0.97 up: 128; 1152
// 1.03 / 1.40, 960 and up)
static bool forward_by_lines(const PairLine& pl) {
  const int n = pl.n;
  return pl.S == 1 && n >= 640 && n % 5 == 0 && n % 3 && n % 7 && n % 11;
}

static cudaError_t make_side(int n, int64_t most_lines, SideFft* f) {
  f->pairs = pair_plan(n, &f->pl) && pair_cluster_fits(f->pl);
  std::vector<float4> table;
  size_t pair_split = 0, line = 0;
  cudaError_t e = cudaSuccess;
  f->fwd_lines = f->pairs && forward_by_lines(f->pl);
  f->lines = !f->pairs || f->fwd_lines || (n <= kFewLines && most_lines <= 2 * kFewLines);   // see on_pairs
  if (f->pairs) pair_split = pair_table(&f->pl, &table);
  if (f->lines) {
    line = table.size();
    e = line_table(n, &f->fl, &table);
  }
  if (e == cudaSuccess) e = cudaMalloc((void**)&f->tw, sizeof(float4) * table.size());
  if (e == cudaSuccess) e = cudaMemcpy(f->tw, table.data(), sizeof(float4) * table.size(), cudaMemcpyHostToDevice);
  f->pl.tw = f->tw;
  f->pl.tw2 = f->tw + pair_split;
  f->fl.tw = f->tw + line;
  f->fl.tw2 = f->fl.split > 1 ? f->fl.tw + f->fl.n : nullptr;
  return e;
}

int df64_fft_line(int64_t n, bool forward, bool* pairs, int* parts, int* radix) {
  if (!df64_side_ok(n)) return 0;
  PairLine pl;
  *pairs = pair_plan((int)n, &pl) && !(forward && forward_by_lines(pl));
  if (*pairs) {
    *parts = pl.S;
    std::copy(pl.radix, pl.radix + pl.nst, radix);
    return pl.nst;
  }
  Df64LinePlan lp;
  *parts = df64_line_split(n);
  df64_line_plan(n / *parts, &lp);
  std::copy(lp.radix, lp.radix + lp.nst, radix);
  return lp.nst;
}

cudaError_t df64_fft_create(int64_t nu, int64_t nv, int64_t batch, Df64Fft** out) {
  *out = nullptr;
  if (!df64_fft_supported(nu, nv)) return cudaErrorInvalidValue;
  Df64Fft* f = new Df64Fft();
  f->nu = (int)nu; f->nv = (int)nv;
  cudaError_t e = pair_smem_attributes();
  if (e == cudaSuccess) e = make_side((int)nu, batch * nv, &f->u);
  if (e == cudaSuccess) e = make_side((int)nv, batch * nu, &f->v);
  const int smax = (int)(2 * kMaxSide * sizeof(float4));
#define WG_SMEM_ATTR(K, BYTES)                                                                   \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, BYTES)
  if (f->u.lines || f->v.lines) {
    WG_SMEM_ATTR((k_fft_lines<448, 2, false, false, false>), smax); WG_SMEM_ATTR((k_fft_lines<448, 2, false, true, false>), smax);
    WG_SMEM_ATTR((k_fft_lines<448, 2, true, false, false>), smax);  WG_SMEM_ATTR((k_fft_lines<448, 2, true, true, false>), smax);
    WG_SMEM_ATTR((k_fft_lines<832, 1, false, false, false>), smax); WG_SMEM_ATTR((k_fft_lines<832, 1, false, true, false>), smax);
    WG_SMEM_ATTR((k_fft_lines<832, 1, true, false, false>), smax);  WG_SMEM_ATTR((k_fft_lines<832, 1, true, true, false>), smax);
    WG_SMEM_ATTR((k_fft_lines<448, 2, false, false, true>), smax);  WG_SMEM_ATTR((k_fft_lines<448, 2, true, false, true>), smax);
    WG_SMEM_ATTR((k_fft_lines<832, 1, false, false, true>), smax);  WG_SMEM_ATTR((k_fft_lines<832, 1, true, false, true>), smax);
    WG_SMEM_ATTR((k_fft_lines_cluster<448, 2, false>), smax); WG_SMEM_ATTR((k_fft_lines_cluster<448, 2, true>), smax);
    WG_SMEM_ATTR((k_fft_lines_cluster<832, 1, false>), smax); WG_SMEM_ATTR((k_fft_lines_cluster<832, 1, true>), smax);
  }
#undef WG_SMEM_ATTR
  if (e != cudaSuccess) {
    df64_fft_destroy(f);
    return e;
  }
  *out = f;
  return cudaSuccess;
}

void df64_fft_destroy(Df64Fft* f) {
  if (f == nullptr) return;
  for (SideFft* side : {&f->u, &f->v})
    if (side->tw) cudaFree(side->tw);
  delete f;
}

static cudaError_t launch_lines(const FftLine& L, double2* data, int64_t batch, int64_t plane,
                                int lines_per_plane, int64_t line_stride, int64_t elem_stride,
                                int mode, int fwd, int split, int skip, int lhalf, int shalf,
                                cudaStream_t s) {
  if (lines_per_plane == 0 || batch == 0) return cudaSuccess;
  const size_t smem = 2 * sizeof(float4) * (size_t)L.n;
  // split lines: L.split CTAs per line
  const int64_t nlines = batch * lines_per_plane * L.split;
  // persistent CTAs: as many as fit the GPU at once (two per SM up to 448 threads, else one)
  int dev = 0, sms = 0;
  cudaError_t ea = cudaGetDevice(&dev);
  if (ea == cudaSuccess) ea = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (ea != cudaSuccess) return ea;
  // pairs in, every element loaded: persistent CTAs with asynchronous loads (inverse row pass
  // 40.8 -> 38.5 ms per bench grid call); doubles in (converted on load) or pruned loads: one
  // line per CTA (the persistent form measured 1.2 ms slower on the forward row pass)
  const bool async = mode != 0 && 2 * (int64_t)lhalf >= L.n && L.split == 1;
  const int64_t blocks =
      async ? std::min<int64_t>(nlines, (int64_t)sms * (L.threads <= 448 ? 2 : 1)) : nlines;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  bool common = true;   // radices 8, 4, 5, 3 only
  for (int i = 0; i < L.nst; ++i)
    if (L.radix[i] == 2 || L.radix[i] == 7 || L.radix[i] == 11) common = false;
  if (L.split > 1) {
    // a cluster of L.split CTAs per line (k_fft_lines_cluster); the register-path split below if
    // the cluster cannot be launched
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)nlines);
    cfg.blockDim = dim3((unsigned)L.threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    std::memset(attr, 0, sizeof(attr));
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)L.split;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (nlines > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaError_t ec;
#define WG_CLUSTER(TM, MB, A)                                                                   \
    ec = cudaLaunchKernelEx(&cfg, k_fft_lines_cluster<TM, MB, A>, L, data, plane,               \
                            lines_per_plane, line_stride, elem_stride, mode, fwd, split, skip,  \
                            lhalf, shalf)
    if (L.threads <= 448) { if (common) WG_CLUSTER(448, 2, false); else WG_CLUSTER(448, 2, true); }
    else { if (common) WG_CLUSTER(832, 1, false); else WG_CLUSTER(832, 1, true); }
#undef WG_CLUSTER
    if (ec == cudaSuccess) return cudaSuccess;
    cudaGetLastError();   // the launch was refused (no kernel ran): the register-path split
  }
#define WG_LINES1(TM, MB, A, Y, P)                                                              \
  k_fft_lines<TM, MB, A, Y, P><<<(unsigned)blocks, L.threads, smem, s>>>(                       \
      L, data, plane, lines_per_plane, line_stride, elem_stride, mode, fwd, split, skip, lhalf, \
      shalf, nlines)
#define WG_LINES(TM, MB, A)                                                                     \
  if (L.split > 1) WG_LINES1(TM, MB, A, false, true);                                           \
  else if (async) WG_LINES1(TM, MB, A, true, false);                                            \
  else WG_LINES1(TM, MB, A, false, false)
  if (L.threads <= 448) {
    if (common) { WG_LINES(448, 2, false); } else { WG_LINES(448, 2, true); }
  } else {
    if (common) { WG_LINES(832, 1, false); } else { WG_LINES(832, 1, true); }
  }
#undef WG_LINES1
#undef WG_LINES
  return cudaGetLastError();
}

// Whether a pass over `lines` lines of a side runs on pairs of lines.  Forward passes of few short lines
// do not: half as many CTAs then leave SMs idle, each takes longer, and the code of the pair
// kernels, a stage of its own for every radix and place, comes from L2 or beyond.  Forward transforms of a
// plan, line by line against in pairs, right after the last one / after 640 MB of other traffic: one plane of
// 128^2 15.6 / 14.3 against 21.5 / 30.7 us, 512^2 23.6 / 26.6 against 31.8 / 45.1, 896^2 40.3 / 43.0 against
// 42.0 / 57.3; 1024^2 48.3 / 49.2 against 44.1 / 59.4; planes of 128^2: 11 of them 20.9 / 20.5 against 21.6 /
// 28.7, 15 of them 23.9 / 22.5 against 21.5 / 30.7; of 256^2, 11: 38.2 / 36.9 against 33.8 / 47.1.
static bool on_pairs(const SideFft& f, int fwd, int64_t lines) {
  return f.pairs && !(fwd && f.lines && (f.fwd_lines || lines <= kFewLines));
}

static cudaError_t launch_side(const SideFft& f, double2* data, int64_t batch, int64_t plane,
                               int lines, int64_t line_stride, int64_t elem_stride, int mode,
                               int fwd, int split, int skip, int lhalf, int shalf, cudaStream_t s) {
  return on_pairs(f, fwd, batch * lines)
             ? launch_pairs(f.pl, data, batch, plane, lines, line_stride, elem_stride, fwd, split,
                            skip, lhalf, shalf, s)
             : launch_lines(f.fl, data, batch, plane, lines, line_stride, elem_stride, mode, fwd,
                            split, skip, lhalf, shalf, s);
}

// complex128 planes to float pairs and back, in place (the FFT utilities; the plans keep pairs)
__global__ void k_to_pairs(double2* __restrict__ data, int64_t count, int back) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (back) {
      const float4 v = reinterpret_cast<const float4*>(data)[i];
      data[i] = make_double2(join_double(dd_make(v.x, v.y)), join_double(dd_make(v.z, v.w)));
    } else {
      const double2 d = data[i];
      const dd r = split_double(d.x), m = split_double(d.y);
      reinterpret_cast<float4*>(data)[i] = make_float4(r.h, r.l, m.h, m.l);
    }
  }
}

// In-place transform of `batch` nu x nv complex128 planes; sign -1 forward, +1 inverse.
// df64_planes: the planes on the grid side are double-float pairs (float4 per complex value:
// re hi, re lo, im hi, im lo) instead of doubles -- the forward transform's output and the
// inverse transform's input; image_pairs: the image side (forward input, inverse output) is
// pairs as well.
// keep_rows = keep_cols = 0: the full 2-D transform.  Otherwise only the image block -- the first
// and last keep_rows/2 rows and keep_cols/2 columns of a plane -- matters, and the column pass
// (strided, the slower pass per line) runs over the image columns only:
//  forward: the image block holds the only nonzero input: the column pass over the image
//    columns loads only their image rows, then the row pass over all rows loads only the image
//    columns (the rest is zero and never read, so the caller need not write it);
//  inverse: only the image block is read afterwards: the row pass over all rows stores only the
//    image columns, then the column pass over those columns stores only the image rows (other
//    cells are left undefined).
cudaError_t df64_fft_exec(Df64Fft* f, double2* data, int64_t batch, int sign, cudaStream_t s,
                          int64_t keep_rows, int64_t keep_cols, bool df64_planes, bool image_pairs) {
  const int64_t plane = (int64_t)f->nu * f->nv;
  const int fwd = sign < 0 ? 1 : 0;
  const bool prune = keep_rows > 0 && keep_cols > 0;
  if (prune && ((keep_rows & 1) || (keep_cols & 1) || keep_rows > f->nu || keep_cols > f->nv))
    return cudaErrorInvalidValue;
  // pass modes of the line kernels: 0 loads doubles and stores pairs, 1 loads pairs and stores
  // doubles, 2 pairs in and out; between the passes pairs.  The line-pair kernels take and give pairs
  // only: complex128 data are converted before a first pass and after a second pass that they run
  const SideFft &first = prune && fwd ? f->u : f->v, &second = prune && fwd ? f->v : f->u;
  const bool in_pairs = fwd ? image_pairs : df64_planes, out_pairs = fwd ? df64_planes : image_pairs;
  const int64_t of_u = batch * (prune ? 2 * (keep_cols / 2) : f->nv), of_v = batch * f->nu;   // lines of a pass
  const bool conv_in = !in_pairs && on_pairs(first, fwd, &first == &f->u ? of_u : of_v);
  const bool conv_out = !out_pairs && on_pairs(second, fwd, &second == &f->u ? of_u : of_v);
  const int mode_in = in_pairs || conv_in ? 2 : 0, mode_out = out_pairs || conv_out ? 2 : 1;
  cudaError_t e;
  auto convert = [&](int back) {
    k_to_pairs<<<152 * 8, 256, 0, s>>>(data, batch * plane, back);
    return cudaGetLastError();
  };
  if (conv_in && (e = convert(0)) != cudaSuccess) return e;
  auto done = [&](cudaError_t r) { return r == cudaSuccess && conv_out ? convert(1) : r; };
  if (!prune) {
    // rows (length nv, contiguous), then columns (length nu, stride nv)
    e = launch_side(f->v, data, batch, plane, f->nu, f->nv, 1, mode_in, fwd,
                     f->nu, 0, f->nv, f->nv, s);
    if (e != cudaSuccess) return e;
    return done(launch_side(f->u, data, batch, plane, f->nv, 1, f->nv, mode_out, fwd,
                            f->nv, 0, f->nu, f->nu, s));
  }
  const int rh = (int)(keep_rows / 2);   // image half-extent along u (rows)
  const int ch = (int)(keep_cols / 2);   // along v (columns)
  const int ncols = 2 * ch, cskip = f->nv - ncols;   // image columns: [0, ch) and [nv - ch, nv)
  if (fwd) {
    // image columns (length nu, stride nv), image rows loaded; then all rows (length nv),
    // image columns loaded
    e = launch_side(f->u, data, batch, plane, ncols, 1, f->nv, mode_in, fwd, ch, cskip, rh,
                     f->nu, s);
    if (e != cudaSuccess) return e;
    return done(launch_side(f->v, data, batch, plane, f->nu, f->nv, 1, mode_out, fwd, f->nu, 0, ch,
                            f->nv, s));
  }
  // inverse: all rows, image columns stored; then the image columns, image rows stored
  e = launch_side(f->v, data, batch, plane, f->nu, f->nv, 1, mode_in, fwd, f->nu, 0, f->nv, ch, s);
  if (e != cudaSuccess) return e;
  return done(launch_side(f->u, data, batch, plane, ncols, 1, f->nv, mode_out, fwd, ch, cskip, f->nu,
                          rh, s));
}

}  // namespace wg
