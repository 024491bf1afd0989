// Register-level DFT building blocks of the double-float plane FFT, on values that carry TWO lines
// at once: every scalar is a packed pair of floats (one per line) and every operation a packed
// FP32 instruction (add / sub / mul / fma .f32x2).
//
// Why pairs of lines: GB300's packed FP32 instructions run at the same lane rate as the scalar
// ones (measured 39.7 T against 38.4 T operations/s) but take one issue slot for two operations,
// and the line kernels were bound by issue (785 instructions per element and pass for 460 FP32
// operations).  With two lines side by side the arithmetic needs half the slots, and one address
// computation, one shared-memory access pattern and one twiddle load serve both lines; inside a
// line (real and imaginary part packed together) every rotation by i and every complex product
// would need moves.
//
// All transforms are forward (e^{-2 pi i}); the inverse is the forward transform with real and
// imaginary parts exchanged on load and on store.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace wg {

typedef unsigned long long pk64;

// ---- f2: two floats, one per line --------------------------------------------------------
struct f2 { pk64 v; };

__device__ __forceinline__ f2 f2_make(float a, float b) {
  f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b)); return r;
}
__device__ __forceinline__ float2 f2_split(f2 x) {
  float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x.v)); return r;
}
// a constant in both lines.  volatile: the constants of a radix stay with its code; hoisted out of
// the stage loop, those of all radices together would be spilled
__device__ __forceinline__ f2 f2_dup(float a) {
  f2 r; asm volatile("mov.b64 %0, {%1, %1};" : "=l"(r.v) : "f"(a)); return r;
}
__device__ __forceinline__ f2 s_add(f2 a, f2 b) {
  f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f2 s_sub(f2 a, f2 b) {
  f2 r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f2 s_mul(f2 a, f2 b) {
  f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f2 s_fma(f2 a, f2 b, f2 c) {
  f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v)); return r;
}

// ---- d2: two double-float values, one per line -------------------------------------------
struct d2 { f2 h, l; };

__device__ __forceinline__ d2 d2_two_sum(f2 a, f2 b) {   // h + l = a + b exactly (Knuth)
  d2 r;
  r.h = s_add(a, b);
  const f2 bb = s_sub(r.h, a);
  r.l = s_add(s_sub(a, s_sub(r.h, bb)), s_sub(b, bb));
  return r;
}
__device__ __forceinline__ d2 d2_fast_two_sum(f2 a, f2 b) {   // the same for |a| >= |b| (Dekker)
  d2 r;
  r.h = s_add(a, b);
  r.l = s_sub(b, s_sub(r.h, a));
  return r;
}
__device__ __forceinline__ d2 s_add(d2 a, d2 b) {
  const d2 s = d2_two_sum(a.h, b.h);
  return d2_fast_two_sum(s.h, s_add(s.l, s_add(a.l, b.l)));
}
__device__ __forceinline__ d2 s_sub(d2 a, d2 b) {   // a - b, the two-sum written for -b
  const f2 s = s_sub(a.h, b.h);
  const f2 bb = s_sub(s, a.h);                       // rounded -b
  const f2 e = s_sub(s_sub(a.h, s_sub(s, bb)), s_add(b.h, bb));
  return d2_fast_two_sum(s, s_add(e, s_sub(a.l, b.l)));
}

// ---- compile-time constants --------------------------------------------------------------
// cos(2 pi k / N), sin(2 pi k / N) from the Taylor series of the reduced angle, in double-double
// arithmetic: a pair of floats resolves 2^-50 of a value, and of a double's last bit (2^-53) it would
// keep the error (in double, 13 of the 74 constants of the radices 3 to 11 were not the nearest
// pair, among them those of the radices 7 and 9)
namespace trig {
struct wide { double h, l; };   // h + l
__host__ __device__ constexpr wide sum(double a, double b) {   // exact (Knuth)
  const double s = a + b, bb = s - a;
  return wide{s, (a - (s - bb)) + (b - bb)};
}
__host__ __device__ constexpr wide prod(double a, double b) {   // exact (Dekker)
  const double ca = 134217729.0 * a, cb = 134217729.0 * b;
  const double ah = ca - (ca - a), al = a - ah, bh = cb - (cb - b), bl = b - bh;
  const double p = a * b;
  return wide{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
__host__ __device__ constexpr wide neg(wide a) { return wide{-a.h, -a.l}; }
__host__ __device__ constexpr wide add(wide a, wide b) {
  const wide s = sum(a.h, b.h);
  return sum(s.h, s.l + (a.l + b.l));
}
__host__ __device__ constexpr wide mul(wide a, wide b) {
  const wide p = prod(a.h, b.h);
  return sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
__host__ __device__ constexpr wide div(wide a, double n) {
  const double q = a.h / n;
  const wide p = prod(q, n);
  return sum(q, (((a.h - p.h) - p.l) + a.l) / n);
}
__host__ __device__ constexpr wide angle(int k, int N) {   // 2 pi k / N
  return div(mul(wide{2.0 * k, 0.0}, wide{3.14159265358979311600e+00, 1.22464679914735317636e-16}), N);
}
// |x| <= pi / 4
__host__ __device__ constexpr wide sin_small(wide x) {
  const wide x2 = mul(x, x);
  wide t = x, s = x;
  for (int i = 1; i <= 14; ++i) { t = neg(div(mul(t, x2), (2.0 * i) * (2.0 * i + 1.0))); s = add(s, t); }
  return s;
}
__host__ __device__ constexpr wide cos_small(wide x) {
  const wide x2 = mul(x, x);
  wide t{1.0, 0.0}, s = t;
  for (int i = 1; i <= 14; ++i) { t = neg(div(mul(t, x2), (2.0 * i - 1.0) * (2.0 * i))); s = add(s, t); }
  return s;
}
// octant reduction in exact integer arithmetic: angle k / N of a turn
__host__ __device__ constexpr wide cos2pi(int k, int N);
__host__ __device__ constexpr wide sin2pi(int k, int N) {
  k %= N; if (k < 0) k += N;
  if (2 * k > N) return neg(sin2pi(N - k, N));
  if (4 * k > N) return sin2pi(N - 2 * k, 2 * N);     // sin(pi - x)
  if (8 * k > N) return cos2pi(N - 4 * k, 4 * N);     // sin(x) = cos(pi/2 - x)
  return sin_small(angle(k, N));
}
__host__ __device__ constexpr wide cos2pi(int k, int N) {
  k %= N; if (k < 0) k += N;
  if (2 * k > N) return cos2pi(N - k, N);
  if (4 * k > N) return neg(cos2pi(N - 2 * k, 2 * N));
  if (8 * k > N) return sin2pi(N - 4 * k, 4 * N);
  return cos_small(angle(k, N));
}
}  // namespace trig

struct Konst {   // a real constant, the nearest pair of floats
  float h, l;
  __host__ __device__ constexpr explicit Konst(trig::wide v)
      : h((float)v.h), l((float)((v.h - (double)(float)v.h) + v.l)) {}
};

// a * k: p - n with p the rounded product of the high parts and n minus everything below it
__device__ __forceinline__ d2 s_mulk(d2 a, const Konst k) {
  const f2 H = f2_dup(k.h), nH = f2_dup(-k.h), nL = f2_dup(-k.l);
  const f2 p = s_mul(a.h, H);
  f2 n = s_fma(a.h, nH, p);
  n = s_fma(a.h, nL, n);
  n = s_fma(a.l, nH, n);
  d2 r;
  r.h = s_sub(p, n);
  r.l = s_sub(s_sub(p, r.h), n);
  return r;
}
// a * k + c
__device__ __forceinline__ d2 s_fmak(d2 a, const Konst k, d2 c) {
  const f2 H = f2_dup(k.h), nH = f2_dup(-k.h), nL = f2_dup(-k.l);
  const f2 p = s_mul(a.h, H);
  f2 n = s_fma(a.h, nH, p);
  n = s_fma(a.h, nL, n);
  n = s_fma(a.l, nH, n);
  const d2 s = d2_two_sum(c.h, p);
  return d2_fast_two_sum(s.h, s_add(s.l, s_sub(c.l, n)));
}
// c - a / 2 (the half is exact)
__device__ __forceinline__ d2 s_submhalf(d2 c, d2 a) {
  d2 m;
  m.h = s_mul(a.h, f2_dup(0.5f));
  m.l = s_mul(a.l, f2_dup(0.5f));
  return s_sub(c, m);
}

// ---- complex values ----------------------------------------------------------------------
template <class S> struct Cx { S r, i; };

template <class S> __device__ __forceinline__ Cx<S> cx_add(const Cx<S>& a, const Cx<S>& b) {
  return Cx<S>{s_add(a.r, b.r), s_add(a.i, b.i)};
}
template <class S> __device__ __forceinline__ Cx<S> cx_sub(const Cx<S>& a, const Cx<S>& b) {
  return Cx<S>{s_sub(a.r, b.r), s_sub(a.i, b.i)};
}
template <class S> __device__ __forceinline__ Cx<S> cx_add_mi(const Cx<S>& a, const Cx<S>& b) {   // a - i b
  return Cx<S>{s_add(a.r, b.i), s_sub(a.i, b.r)};
}
template <class S> __device__ __forceinline__ Cx<S> cx_add_pi(const Cx<S>& a, const Cx<S>& b) {   // a + i b
  return Cx<S>{s_sub(a.r, b.i), s_add(a.i, b.r)};
}
template <class S> __device__ __forceinline__ Cx<S> cx_mulk(const Cx<S>& a, const Konst k) {
  return Cx<S>{s_mulk(a.r, k), s_mulk(a.i, k)};
}

// Twiddle factors as loaded from the tables: every float twice (one per line).
template <class S> struct Tw;
template <> struct Tw<d2> { f2 rh, rl, ih, il; };

// x u + y v with the cross terms, one normalised pair: both leading products are split exactly
// (n1, n2 are minus their errors), summed exactly, the small terms accumulated in float.
// nuh, nvh: -u.h, -v.h.
__device__ __forceinline__ d2 d2_dot(const d2& x, f2 uh, f2 nuh, f2 ul, const d2& y, f2 vh, f2 nvh, f2 vl) {
  const f2 p1 = s_mul(x.h, uh), n1 = s_fma(x.h, nuh, p1);
  const f2 p2 = s_mul(y.h, vh), n2 = s_fma(y.h, nvh, p2);
  const d2 s = d2_two_sum(p1, p2);
  f2 t = s_sub(s.l, s_add(n1, n2));
  t = s_fma(x.h, ul, t);
  t = s_fma(x.l, uh, t);
  t = s_fma(y.h, vl, t);
  t = s_fma(y.l, vh, t);
  return d2_fast_two_sum(s.h, t);
}
__device__ __forceinline__ Cx<d2> cx_mul(const Cx<d2>& a, const Tw<d2>& w) {
  const f2 m1 = f2_dup(-1.0f);
  const f2 nrh = s_mul(w.rh, m1), nih = s_mul(w.ih, m1), nil = s_mul(w.il, m1);
  return Cx<d2>{d2_dot(a.r, w.rh, nrh, w.rl, a.i, nih, w.ih, nil),
                d2_dot(a.r, w.ih, nih, w.il, a.i, w.rh, nrh, w.rl)};
}
// a e^{-2 pi i k / N} for compile-time k, N
template <int N, int K>
__device__ __forceinline__ Cx<d2> cx_root(const Cx<d2>& a) {
  constexpr Konst c{trig::cos2pi(K, N)}, s{trig::neg(trig::sin2pi(K, N))};
  return Cx<d2>{d2_dot(a.r, f2_dup(c.h), f2_dup(-c.h), f2_dup(c.l), a.i, f2_dup(-s.h), f2_dup(s.h), f2_dup(-s.l)),
                d2_dot(a.r, f2_dup(s.h), f2_dup(-s.h), f2_dup(s.l), a.i, f2_dup(c.h), f2_dup(-c.h), f2_dup(c.l))};
}

// ---- DFTs of R values in registers (in place, natural order in and out) -------------------
template <class S> __device__ __forceinline__ void dft_2(Cx<S>* x) {
  const Cx<S> a = cx_add(x[0], x[1]), b = cx_sub(x[0], x[1]);
  x[0] = a; x[1] = b;
}
template <class S> __device__ __forceinline__ void dft_3(Cx<S>* x) {
  const Cx<S> t = cx_add(x[1], x[2]), d = cx_sub(x[1], x[2]);
  const Cx<S> m{s_submhalf(x[0].r, t.r), s_submhalf(x[0].i, t.i)};
  constexpr Konst k{trig::sin2pi(1, 3)};
  const Cx<S> s = cx_mulk(d, k);
  x[0] = cx_add(x[0], t);
  x[1] = cx_add_mi(m, s);
  x[2] = cx_add_pi(m, s);
}
template <class S> __device__ __forceinline__ void dft_4(Cx<S>* x) {
  const Cx<S> t0 = cx_add(x[0], x[2]), t1 = cx_sub(x[0], x[2]);
  const Cx<S> t2 = cx_add(x[1], x[3]), d = cx_sub(x[1], x[3]);
  x[0] = cx_add(t0, t2);
  x[2] = cx_sub(t0, t2);
  x[1] = cx_add_mi(t1, d);
  x[3] = cx_add_pi(t1, d);
}
template <class S> __device__ __forceinline__ void dft_8(Cx<S>* x) {
  Cx<S> e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
  dft_4(e);
  dft_4(o);
  constexpr Konst c{trig::cos2pi(1, 8)};
  const Cx<S> o1{s_mulk(s_add(o[1].r, o[1].i), c), s_mulk(s_sub(o[1].i, o[1].r), c)};  // (1 - i) / sqrt 2
  // o3 (-1 - i) / sqrt 2 = (a, -q)
  const S a = s_mulk(s_sub(o[3].i, o[3].r), c), q = s_mulk(s_add(o[3].r, o[3].i), c);
  x[0] = cx_add(e[0], o[0]);
  x[4] = cx_sub(e[0], o[0]);
  x[1] = cx_add(e[1], o1);
  x[5] = cx_sub(e[1], o1);
  x[2] = cx_add_mi(e[2], o[2]);
  x[6] = cx_add_pi(e[2], o[2]);
  x[3] = Cx<S>{s_add(e[3].r, a), s_sub(e[3].i, q)};
  x[7] = Cx<S>{s_sub(e[3].r, a), s_add(e[3].i, q)};
}
// odd prime R: with a_k = x_k + x_{R-k}, b_k = x_k - x_{R-k} (k = 1 .. P = (R - 1) / 2),
//   y_q = x_0 + sum_k a_k cos(2 pi k q / R) - i sum_k b_k sin(2 pi k q / R), y_{R-q} with + i
template <int R, int Q, int K, class S>
__device__ __forceinline__ void odd_terms(const Cx<S>* a, const Cx<S>* b, Cx<S>& re, Cx<S>& im) {
  if constexpr (K <= (R - 1) / 2) {
    constexpr Konst c{trig::cos2pi(K * Q, R)}, s{trig::sin2pi(K * Q, R)};
    re.r = s_fmak(a[K - 1].r, c, re.r);
    re.i = s_fmak(a[K - 1].i, c, re.i);
    if constexpr (K == 1) im = cx_mulk(b[0], s);
    else im = Cx<S>{s_fmak(b[K - 1].r, s, im.r), s_fmak(b[K - 1].i, s, im.i)};
    odd_terms<R, Q, K + 1>(a, b, re, im);
  }
}
template <int R, int Q, class S>
__device__ __forceinline__ void odd_outputs(const Cx<S>* a, const Cx<S>* b, const Cx<S>& x0, Cx<S>* x) {
  if constexpr (Q <= (R - 1) / 2) {
    Cx<S> re = x0, im;
    odd_terms<R, Q, 1>(a, b, re, im);
    x[Q] = cx_add_mi(re, im);
    x[R - Q] = cx_add_pi(re, im);
    odd_outputs<R, Q + 1>(a, b, x0, x);
  }
}
template <int R, class S> __device__ __forceinline__ void dft_odd_prime(Cx<S>* x) {
  constexpr int P = (R - 1) / 2;
  Cx<S> a[P], b[P];
#pragma unroll
  for (int k = 1; k <= P; ++k) {
    a[k - 1] = cx_add(x[k], x[R - k]);
    b[k - 1] = cx_sub(x[k], x[R - k]);
  }
  const Cx<S> x0 = x[0];
#pragma unroll
  for (int k = 0; k < P; ++k) x[0] = cx_add(x[0], a[k]);
  odd_outputs<R, 1>(a, b, x0, x);
}
template <int R, class S> __device__ __forceinline__ void dft(Cx<S>* x);

// R = A B with A, B coprime (Good-Thomas): no twiddles between the two
__host__ __device__ constexpr int inv_mod(int a, int m) {
  for (int i = 1; i < m; ++i)
    if (a * i % m == 1) return i;
  return 0;
}
template <int A, int B, class S> __device__ __forceinline__ void dft_coprime(Cx<S>* x) {
  constexpr int N = A * B, kInvB = inv_mod(B % A, A), kInvA = inv_mod(A % B, B);
  Cx<S> y[N];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    Cx<S> t[A];
#pragma unroll
    for (int a = 0; a < A; ++a) t[a] = x[(B * a + A * b) % N];
    dft<A>(t);
#pragma unroll
    for (int a = 0; a < A; ++a) y[a * B + b] = t[a];
  }
#pragma unroll
  for (int a = 0; a < A; ++a) {
    dft<B>(y + a * B);
#pragma unroll
    for (int b = 0; b < B; ++b)
      x[(B * kInvB * a + A * kInvA * b) % N] = y[a * B + b];
  }
}
// R = A A: columns, constant twiddles, rows
template <int N, int K, class S> __device__ __forceinline__ Cx<S> cx_tw(const Cx<S>& a) {
  if constexpr (K % N == 0) return a;
  else return cx_root<N, K>(a);
}
template <int A, int B, int b, int a, class S> __device__ __forceinline__ void tw_col(Cx<S>* t) {
  if constexpr (a < A) {
    t[a] = cx_tw<A * B, a * b>(t[a]);
    tw_col<A, B, b, a + 1>(t);
  }
}
template <int A, int B, int b, class S> __device__ __forceinline__ void cols(const Cx<S>* x, Cx<S>* y) {
  if constexpr (b < B) {
    Cx<S> t[A];
#pragma unroll
    for (int a = 0; a < A; ++a) t[a] = x[b + B * a];
    dft<A>(t);
    tw_col<A, B, b, 1>(t);
#pragma unroll
    for (int a = 0; a < A; ++a) y[a * B + b] = t[a];
    cols<A, B, b + 1>(x, y);
  }
}
template <int A, int B, class S> __device__ __forceinline__ void dft_product(Cx<S>* x) {
  Cx<S> y[A * B];
  cols<A, B, 0>(x, y);
#pragma unroll
  for (int a = 0; a < A; ++a) {
    dft<B>(y + a * B);
#pragma unroll
    for (int b = 0; b < B; ++b) x[a + A * b] = y[a * B + b];
  }
}
template <int R, class S> __device__ __forceinline__ void dft(Cx<S>* x) {
  if constexpr (R == 2) dft_2(x);
  else if constexpr (R == 3) dft_3(x);
  else if constexpr (R == 4) dft_4(x);
  else if constexpr (R == 5 || R == 7 || R == 11) dft_odd_prime<R>(x);
  else if constexpr (R == 6) dft_coprime<3, 2>(x);
  else if constexpr (R == 8) dft_8(x);
  else if constexpr (R == 9) dft_product<3, 3>(x);
  else if constexpr (R == 10) dft_coprime<5, 2>(x);
  else dft_coprime<3, 4>(x);   // 12
}

}  // namespace wg
