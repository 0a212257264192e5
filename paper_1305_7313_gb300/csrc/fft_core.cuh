// fft_core.cuh — the transforms of the Fock apply: in-register DFTs of radix 2,
// 3, 4, 5, 7 and 8 and of their composites up to 24, and the stages that
// put them together on lines and planes held in shared memory, specialised at
// compile time for one line length N.
//
// The 3D FFTs of the Fock apply (orbitals to real space, pair densities to G
// space and back, V_x psi back to G space; §4 of the paper computes all of
// them "via Fast Fourier Transform") are done as one pass over planes and one
// pass over columns.  A line of N = A B points takes two stages, A-point DFTs
// and B-point DFTs with twiddles on their inputs, each in place; the twiddle
// products are not rounded on their own in float and double but folded into the
// first butterfly sums as fused multiply-adds (Dft::run_tw).
//
// Thread mapping: consecutive threads take consecutive lines, which keeps
// shared-memory accesses conflict-free when lines are contiguous (columns) or
// when the line stride is odd (rows with a padded stride).
//
// Twiddles come from a table w[t] = exp(-2 pi i t / N), t < N, computed on the
// host in FP64; a kernel stages the N products a stage reads in shared memory.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "df64.cuh"

// The butterflies and their complex helpers compile for the host too, so that
// they can be checked on a CPU; the kernels use them on the device only.
#define FFT_HD __host__ __device__ __forceinline__

namespace fockx {

constexpr int kMaxStages = 8;
constexpr int kTwiddleTable = 2;  // forward and inverse twiddles
constexpr int kMaxThreads = 1024;
constexpr int kEmax = 24;  // elements a thread may hold across a stage

// Radix plans: factorisations of a line into stages with whole lines shared by
// tl threads.  No kernel is laid out by them (the passes' factors are two_factor's
// and their geometry PairGeo's); the host checks of the radices and of Geo are.
struct RadixPlan {
  int nst;                 // number of stages
  int r[kMaxStages];       // radices, in stage order
  int tl_plane;            // sub-threads per line, plane passes (N lines)
  int tl_colh;             // sub-threads per line, half-spectrum column pass (2(N/2+1) lines)
};

// sin and cos of 2 pi m / R for integers, evaluated at compile time from their
// Taylor series after reducing the angle to [0, pi/4] with the octant
// symmetries (exact for the multiples of pi/4).
__host__ __device__ constexpr double ct_taylor_sin(double x) {
  double term = x, sum = x;
  for (int k = 1; k < 14; ++k) {
    term *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr double ct_taylor_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 14; ++k) {
    term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
    sum += term;
  }
  return sum;
}
// cos(2 pi m / R) (want_sin = false) or sin(2 pi m / R) (want_sin = true)
__host__ __device__ constexpr double ct_trig(int m, int R, bool want_sin) {
  m = ((m % R) + R) % R;
  // angle = 2 pi m / R = (pi / 4) * (8 m / R): octant o and remainder in [0, 1)
  const int num = 8 * m;
  const int o = num / R;
  const double f = (double)(num - o * R) / (double)R;  // fraction of an octant
  const double quarter_pi = 0.78539816339744830961566084581987572;
  double c = 0.0, s = 0.0;
  // angle within the octant, measured from its start (even octant) or its end (odd)
  const double y = ((o & 1) ? (1.0 - f) : f) * quarter_pi;
  const double cy = ct_taylor_cos(y), sy = ct_taylor_sin(y);
  switch (o) {  // angle = o * pi/4 + f * pi/4
    case 0: c = cy; s = sy; break;      // [0, 45)
    case 1: c = sy; s = cy; break;      // [45, 90): 90 - y
    case 2: c = -sy; s = cy; break;     // [90, 135): 90 + y
    case 3: c = -cy; s = sy; break;     // [135, 180): 180 - y
    case 4: c = -cy; s = -sy; break;    // [180, 225): 180 + y
    case 5: c = -sy; s = -cy; break;    // [225, 270): 270 - y
    case 6: c = sy; s = -cy; break;     // [270, 315): 270 + y
    default: c = cy; s = -sy; break;    // [315, 360): 360 - y
  }
  return want_sin ? s : c;
}

__host__ __device__ constexpr int cgcd(int a, int b) {
  while (b != 0) {
    const int t = a % b;
    a = b;
    b = t;
  }
  return a;
}

__host__ __device__ constexpr int best_tl(int n, const int* r, int nst, int nlines, int maxt, int emax) {
  int g = 0;
  for (int s = 0; s < nst; ++s) g = cgcd(g, n / r[s]);
  for (int t = g; t >= 1; --t)
    if (g % t == 0 && n / t <= emax && (nlines * t + 31) / 32 * 32 <= maxt) return t;
  return 0;
}

constexpr int kRadices[8] = {16, 12, 9, 8, 6, 4, 3, 2};

// Depth-first search over radix multisets (in descending order) whose product
// is n; keeps the plan with the fewest stages, then the most threads per line.
__host__ __device__ constexpr void radix_search(int n, int rem, int first, RadixPlan& cur, RadixPlan& best,
                                                int& best_score, int maxt, int emax) {
  if (rem == 1) {
    RadixPlan p = cur;
    p.tl_plane = best_tl(n, p.r, p.nst, n, maxt, emax);
    p.tl_colh = best_tl(n, p.r, p.nst, 2 * (n / 2 + 1), maxt, emax);
    if (p.tl_plane == 0 || p.tl_colh == 0) return;
    const int score = p.nst * 4096 - p.tl_plane;
    if (score < best_score) {
      best_score = score;
      best = p;
    }
    return;
  }
  if (cur.nst >= 4) return;
  for (int k = first; k < 8; ++k) {
    const int r = kRadices[k];
    if (rem % r != 0) continue;
    cur.r[cur.nst++] = r;
    radix_search(n, rem / r, k, cur, best, best_score, maxt, emax);
    --cur.nst;
  }
}

// Fewest stages first, then the most threads per line, with CTAs of at most
// maxt threads.
__host__ __device__ constexpr RadixPlan make_radix_plan(int n, int maxt = kMaxThreads, int emax = kEmax) {
  RadixPlan best{};
  best.nst = 0;
  RadixPlan cur{};
  cur.nst = 0;
  int best_score = 1 << 30;
  radix_search(n, n, 0, cur, best, best_score, maxt, emax);
  return best;
}

// Per working type.  fused: the type has a hardware fused multiply-add, so twiddle
// products are folded into the butterfly sums (Dft::run_tw) instead of being
// rounded on their own.  emax: elements a thread may hold across a stage of a radix
// plan (RadixPlan).
template <class T> struct FftTraits {
  static constexpr int emax = kEmax;
  static constexpr bool fused = true;
};

template <class T> struct CplxOf;
template <> struct CplxOf<float> { using type = float2; };
template <> struct CplxOf<double> { using type = double2; };
template <> struct CplxOf<df64> { using type = cdf64; };
template <> struct FftTraits<double> {
  static constexpr int emax = 12;
  static constexpr bool fused = true;
};
template <> struct FftTraits<df64> {
  static constexpr int emax = 12;
  static constexpr bool fused = false;
};
template <class T> using cplx = typename CplxOf<T>::type;

// Elements a thread may hold across a stage of radix plan (N, MAXT, EMAX) (0:
// FftTraits<T>::emax).
template <class T, int EMAX> __host__ __device__ constexpr int plan_emax() {
  return EMAX > 0 ? EMAX : FftTraits<T>::emax;
}

// S * x for S = +1 or -1 (a sign flip, never a multiplication)
template <int S, class T> FFT_HD T sgn(T x) {
  if constexpr (S > 0) return x;
  else return -x;
}
// x / 2, exact
FFT_HD float half_of(float x) { return 0.5f * x; }
FFT_HD double half_of(double x) { return 0.5 * x; }
__device__ __forceinline__ df64 half_of(df64 x) { return ldexp_pow2(x, 0.5f); }

// a * b + c with one rounding
FFT_HD float fmadd(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}
FFT_HD double fmadd(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return __fma_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}

template <class T>
FFT_HD cplx<T> cmake(T x, T y) {
  cplx<T> r;
  r.x = x;
  r.y = y;
  return r;
}
template <class C> FFT_HD C cadd(C a, C b);
// x y and x + S y rounded once, in any type.
template <class T> FFT_HD T rmul(T x, T y) { return x * y; }
// a compile-time factor as the multiplications take it
template <class T> FFT_HD T factor(T c) { return c; }
template <int S, class T> FFT_HD T radd(T x, T y) { return S > 0 ? x + y : x - y; }
#ifdef __CUDA_ARCH__
// FP64: as fused multiply-adds, x y + (-0) and x + y 1, which round the same, with
// every operand in a register.  A DADD, a DMUL or a DFMA with an immediate or
// constant operand occupies the FP64 unit of an SM for 20 clocks a warp, a DFMA of
// registers for 16.8 (measured with independent operations: 504 against 598 G a
// second over the chip).  The factors come from a register the compiler cannot see
// through (%smid < 2^24), or it would turn them back.  FP64 pair passes at 96^3:
// 165 -> 151 us a chain, the FP64 unit 92-97% busy.
__device__ __forceinline__ double opaque_one() {
  double o;
  asm("{.reg .u32 t; mov.u32 t, %%smid; shr.u32 t, t, 24; add.u32 t, t, 1; cvt.rn.f64.u32 %0, t;}" : "=d"(o));
  return o;
}
__device__ __forceinline__ double opaque_minus_zero() {
  double o;
  asm("{.reg .u32 t; mov.u32 t, %%smid; shr.u32 t, t, 24; cvt.rn.f64.u32 %0, t; neg.f64 %0, %0;}" : "=d"(o));
  return o;
}
template <> __device__ __forceinline__ double rmul<double>(double x, double y) {
  return __fma_rn(x, y, opaque_minus_zero());
}
template <> __device__ __forceinline__ double factor<double>(double c) { return __dmul_rn(c, opaque_one()); }
template <> __device__ __forceinline__ double radd<1, double>(double x, double y) { return __fma_rn(y, opaque_one(), x); }
template <> __device__ __forceinline__ double radd<-1, double>(double x, double y) {
  return __fma_rn(-y, opaque_one(), x);
}
#endif

template <class C> FFT_HD C cadd(C a, C b) {
  a.x = radd<1>(a.x, b.x);
  a.y = radd<1>(a.y, b.y);
  return a;
}
template <class C> FFT_HD C csub(C a, C b) {
  a.x = radd<-1>(a.x, b.x);
  a.y = radd<-1>(a.y, b.y);
  return a;
}
// c b and a + c b for a real c (one rounding per component where T has a fused
// multiply-add).
template <class T, class C> FFT_HD C cscale(T c, C b) {
  const T f = factor(c);
  b.x = rmul(f, b.x);
  b.y = rmul(f, b.y);
  return b;
}
template <class T, class C> FFT_HD C caxpy(T c, C b, C a) {
  if constexpr (FftTraits<T>::fused) {
    const T f = factor(c);
    a.x = fmadd(f, b.x, a.x);
    a.y = fmadd(f, b.y, a.y);
  } else {
    a = cadd(a, cscale(c, b));
  }
  return a;
}
#ifdef __CUDA_ARCH__
// FP32: both components in one instruction, with the same roundings.  The FP32
// pipe runs the two-wide forms at the rate of two scalar ones, but an instruction
// takes one issue slot: the forward plane pass at 96^3 went from 3.01 to 2.83 us a
// chain, the apply (256 bands) from 136.8 to 134.4 ms.
template <> __device__ __forceinline__ float2 cadd<float2>(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; add.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
template <> __device__ __forceinline__ float2 csub<float2>(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; sub.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
template <> __device__ __forceinline__ float2 cscale<float, float2>(float c, float2 b) {
  float2 r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %2}; mov.b64 b, {%3, %4}; mul.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(c), "f"(b.x), "f"(b.y));
  return r;
}
template <> __device__ __forceinline__ float2 caxpy<float, float2>(float c, float2 b, float2 a) {
  float2 r;
  asm("{.reg .b64 a, b, c, d; mov.b64 a, {%2, %2}; mov.b64 b, {%3, %4}; mov.b64 c, {%5, %6}; fma.rn.f32x2 d, a, b, c; "
      "mov.b64 {%0, %1}, d;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(c), "f"(b.x), "f"(b.y), "f"(a.x), "f"(a.y));
  return r;
}
#endif
#ifdef __CUDA_ARCH__
// Double-float: the sums, products and scalings of df64.cuh on both components at
// once (pairs (x.hi, y.hi) and (x.lo, y.lo)), operation for operation with the
// same roundings, in half the issue slots (96^3 column pass 12.5 -> 11.1 us a
// chain, 64^3 forward pass 4.38 -> 3.95).
struct DfPair {
  float2 hi, lo;
};
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; mul.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{.reg .b64 a, b, c, d; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; mov.b64 c, {%6, %7}; fma.rn.f32x2 d, a, b, c; "
      "mov.b64 {%0, %1}, d;}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ DfPair df_pair(cdf64 a) {
  return DfPair{make_float2(a.x.hi, a.y.hi), make_float2(a.x.lo, a.y.lo)};
}
__device__ __forceinline__ DfPair df_swapped(cdf64 a) {
  return DfPair{make_float2(a.y.hi, a.x.hi), make_float2(a.y.lo, a.x.lo)};
}
__device__ __forceinline__ cdf64 df_join(float2 hi, float2 lo) {
  cdf64 r;
  r.x = df64(hi.x, lo.x);
  r.y = df64(hi.y, lo.y);
  return r;
}
// a + b
__device__ __forceinline__ cdf64 df_add2(DfPair a, DfPair b) {
  const float2 s = cadd(a.hi, b.hi), bb = csub(s, a.hi);
  float2 e = cadd(csub(a.hi, csub(s, bb)), csub(b.hi, bb));
  e = cadd(e, cadd(a.lo, b.lo));
  const float2 h = cadd(s, e);
  return df_join(h, csub(e, csub(h, s)));
}
// a - b
__device__ __forceinline__ cdf64 df_sub2(DfPair a, DfPair b) {
  const float2 s = csub(a.hi, b.hi), bb = csub(s, a.hi);
  float2 e = csub(csub(a.hi, csub(s, bb)), cadd(b.hi, bb));
  e = cadd(e, csub(a.lo, b.lo));
  const float2 h = cadd(s, e);
  return df_join(h, csub(e, csub(h, s)));
}
// a + (g.x b.x, g.y b.y), g = +-1
__device__ __forceinline__ cdf64 df_addsub2(DfPair a, DfPair b, float2 g) {
  const float2 s = f2fma(b.hi, g, a.hi), nbb = csub(a.hi, s);
  float2 e = cadd(csub(a.hi, cadd(s, nbb)), f2fma(b.hi, g, nbb));
  e = cadd(e, f2fma(b.lo, g, a.lo));
  const float2 h = cadd(s, e);
  return df_join(h, csub(e, csub(h, s)));
}
// c b for a real c (the errors kept negated: n = -(error so far))
__device__ __forceinline__ DfPair df_scale2(df64 c, DfPair b) {
  const float2 ch = make_float2(c.hi, c.hi), nh = make_float2(-c.hi, -c.hi), nl = make_float2(-c.lo, -c.lo);
  const float2 p = f2mul(ch, b.hi);
  float2 n = f2fma(nh, b.hi, p);
  n = f2fma(nh, b.lo, n);
  n = f2fma(nl, b.hi, n);
  const float2 h = csub(p, n);
  return DfPair{h, csub(csub(p, h), n)};
}
template <> __device__ __forceinline__ cdf64 cadd<cdf64>(cdf64 a, cdf64 b) { return df_add2(df_pair(a), df_pair(b)); }
template <> __device__ __forceinline__ cdf64 csub<cdf64>(cdf64 a, cdf64 b) { return df_sub2(df_pair(a), df_pair(b)); }
template <> __device__ __forceinline__ cdf64 cscale<df64, cdf64>(df64 c, cdf64 b) {
  const DfPair r = df_scale2(c, df_pair(b));
  return df_join(r.hi, r.lo);
}
#endif
// a + S i b and a - S i b for S = +1 or -1
template <int S, class C> FFT_HD C cadd_si(C a, C b) {
  C r;
  r.x = radd<-S>(a.x, b.y);
  r.y = radd<S>(a.y, b.x);
  return r;
}
#ifdef __CUDA_ARCH__
template <int S> __device__ __forceinline__ cdf64 df_add_si(cdf64 a, cdf64 b) {
  return df_addsub2(df_pair(a), df_swapped(b), make_float2(S > 0 ? -1.f : 1.f, S > 0 ? 1.f : -1.f));
}
template <> __device__ __forceinline__ cdf64 cadd_si<1, cdf64>(cdf64 a, cdf64 b) { return df_add_si<1>(a, b); }
template <> __device__ __forceinline__ cdf64 cadd_si<-1, cdf64>(cdf64 a, cdf64 b) { return df_add_si<-1>(a, b); }
#endif
template <int S, class C> FFT_HD C csub_si(C a, C b) { return cadd_si<-S>(a, b); }
template <class C> FFT_HD C cmul(C a, C b) {
  C r;
  if constexpr (std::is_same<decltype(a.x), double>::value) {
    r.x = fmadd(-a.y, b.y, rmul(a.x, b.x));
    r.y = fmadd(a.y, b.x, rmul(a.x, b.y));
  } else {
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
  }
  return r;
}
#ifdef __CUDA_ARCH__
template <> __device__ __forceinline__ cdf64 cmul<cdf64>(cdf64 a, cdf64 b) {
  return df_addsub2(df_scale2(b.x, df_pair(a)), df_scale2(b.y, df_swapped(a)), make_float2(-1.f, 1.f));
}
#endif
// S * i * a for S = +1 or -1
template <int S, class C> FFT_HD C cmul_si(C a) {
  C r;
  r.x = S > 0 ? -a.y : a.y;
  r.y = S > 0 ? a.x : -a.x;
  return r;
}

// In-register DFTs, y_q = sum_r x_r exp(SIGN 2 pi i r q / R).
template <int SIGN, class T> struct Dft {
  using C = cplx<T>;
  static FFT_HD void r2(C* x) {
    C a = x[0];
    x[0] = cadd(a, x[1]);
    x[1] = csub(a, x[1]);
  }
  static FFT_HD void r3(C* x) { r3_sd(x, cadd(x[1], x[2]), csub(x[1], x[2])); }
  // the length-3 DFT from x0, s = x1 + x2 and d = x1 - x2
  static FFT_HD void r3_sd(C* x, C s, C d) {
    constexpr T h0 = T(0.86602540378443864676372317075293618);  // sin(2 pi / 3)
    if constexpr (FftTraits<T>::fused) {
      const T h = factor(SIGN > 0 ? h0 : -h0);
      const C m = caxpy(T(-0.5), s, x[0]);
      x[0] = cadd(x[0], s);
      x[1] = cmake<T>(fmadd(-h, d.y, m.x), fmadd(h, d.x, m.y));
      x[2] = cmake<T>(fmadd(h, d.y, m.x), fmadd(-h, d.x, m.y));
    } else {
      const C m = csub(x[0], cmake<T>(half_of(s.x), half_of(s.y)));
      const C u = cscale(h0, d);
      x[0] = cadd(x[0], s);
      x[1] = cadd_si<SIGN>(m, u);
      x[2] = csub_si<SIGN>(m, u);
    }
  }
  static FFT_HD void r4v(C& x0, C& x1, C& x2, C& x3) {
    C a = cadd(x0, x2), b = csub(x0, x2), c = cadd(x1, x3), d = csub(x1, x3);
    x0 = cadd(a, c);
    x2 = csub(a, c);
    x1 = cadd_si<SIGN>(b, d);
    x3 = csub_si<SIGN>(b, d);
  }
  static FFT_HD void r4(C* x) { r4v(x[0], x[1], x[2], x[3]); }
  static FFT_HD void r8(C* x) {
    constexpr T c = T(0.70710678118654752440084436210484904);  // cos(pi / 4)
    C e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    C o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
    r4v(e0, e1, e2, e3);
    r4v(o0, o1, o2, o3);
    // x_q = e_q +- exp(SIGN 2 pi i q / 8) o_q, the pi/4 rotations as c * p
    const C p = cadd_si<SIGN>(o1, o1), q = csub_si<SIGN>(o3, o3);
    x[0] = cadd(e0, o0);
    x[4] = csub(e0, o0);
    x[1] = caxpy(c, p, e1);
    x[5] = caxpy(-c, p, e1);
    x[2] = cadd_si<SIGN>(e2, o2);
    x[6] = csub_si<SIGN>(e2, o2);
    x[3] = caxpy(-c, q, e3);
    x[7] = caxpy(c, q, e3);
  }
  // x *= exp(SIGN 2 pi i M / R) with compile-time M, R (exact for the quarter turns)
  template <int M, int R> static FFT_HD C twiddle(C x) {
    constexpr int m = ((M % R) + R) % R;
    if constexpr (m == 0) {
      return x;
    } else if constexpr (4 * m == R) {
      return cmul_si<SIGN>(x);
    } else if constexpr (2 * m == R) {
      return cmake<T>(-x.x, -x.y);
    } else if constexpr (4 * m == 3 * R) {
      return cmul_si<-SIGN>(x);
    } else {
      const T c = factor(T(ct_trig(m, R, false))), s = factor(T(SIGN * ct_trig(m, R, true)));
      return cmul(x, cmake<T>(c, s));
    }
  }
  // ---- twiddled inputs, for types with a fused multiply-add (FftTraits::fused).
  // DFT of (x_0, w_1 x_1, ..., w_{R-1} x_{R-1}): each twiddle product is folded
  // into the first sum it feeds (a + w x as two fused multiply-adds per
  // component), and the matching difference is taken as 2 a - (a + w x), which
  // saves the separate rounding of w x and a quarter of the instructions of the
  // twiddled sums.
  // a + w x
  static FFT_HD C cfma(C a, C w, C x) {
    return cmake<T>(fmadd(w.x, x.x, fmadd(-w.y, x.y, a.x)), fmadd(w.x, x.y, fmadd(w.y, x.x, a.y)));
  }
  // 2 a - b
  static FFT_HD C ctwice_sub(C a, C b) {
    const T two = factor(T(2));
    return cmake<T>(fmadd(two, a.x, -b.x), fmadd(two, a.y, -b.y));
  }
  // a - 2 b
  static FFT_HD C csub_twice(C a, C b) {
    return caxpy(T(-2), b, a);
  }
  static FFT_HD void r2_tw(C& x0, C& x1, C w1) {
    const C a = cfma(x0, w1, x1);
    x1 = ctwice_sub(x0, a);
    x0 = a;
  }
  static FFT_HD void r3_tw(C* x, C w1, C w2) {
    const C x1w = cmul(x[1], w1);
    const C s = cfma(x1w, w2, x[2]);  // w1 x1 + w2 x2
    r3_sd(x, s, ctwice_sub(x1w, s));
  }
  static FFT_HD void r4v_tw(C& x0, C& x1, C& x2, C& x3, C w1, C w2, C w3) {
    const C a = cfma(x0, w2, x2);      // x0 + w2 x2
    const C b = ctwice_sub(x0, a);     // x0 - w2 x2
    const C x3w = cmul(x3, w3);
    const C c = cfma(x3w, w1, x1);     // w1 x1 + w3 x3
    const C d = csub_twice(c, x3w);  // w1 x1 - w3 x3
    x0 = cadd(a, c);
    x2 = csub(a, c);
    x1 = cadd_si<SIGN>(b, d);
    x3 = csub_si<SIGN>(b, d);
  }
  static FFT_HD void r8_tw(C* x, const C* w) {
    constexpr T c = T(0.70710678118654752440084436210484904);  // cos(pi / 4)
    C e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    C o0 = cmul(x[1], w[1]), o1 = x[3], o2 = x[5], o3 = x[7];
    r4v_tw(e0, e1, e2, e3, w[2], w[4], w[6]);
    r4v_tw(o0, o1, o2, o3, w[3], w[5], w[7]);
    // x_q = e_q +- exp(SIGN 2 pi i q / 8) o_q, the pi/4 rotations as c * p
    const C p = cadd_si<SIGN>(o1, o1), q = csub_si<SIGN>(o3, o3);
    x[0] = cadd(e0, o0);
    x[4] = csub(e0, o0);
    x[1] = caxpy(c, p, e1);
    x[5] = caxpy(-c, p, e1);
    x[2] = cadd_si<SIGN>(e2, o2);
    x[6] = csub_si<SIGN>(e2, o2);
    x[3] = caxpy(-c, q, e3);
    x[7] = caxpy(c, q, e3);
  }
  // DFT of odd prime length: with s_j = x_j + x_R-j and d_j = x_j - x_R-j (j = 1 ..
  // (R-1)/2), y_q = a_q +- SIGN i u_q, a_q = x_0 + sum_j cos(2 pi j q / R) s_j, u_q =
  // sum_j sin(2 pi j q / R) d_j.
  template <int R, int Q, int J = 1> static FFT_HD void odd_sums(const C* s, const C* d, C& a, C& u) {
    if constexpr (2 * J < R) {
      constexpr T c = T(ct_trig(J * Q, R, false)), h = T(ct_trig(J * Q, R, true));
      a = caxpy(c, s[J], a);
      if constexpr (J == 1) u = cscale(h, d[1]);
      else u = caxpy(h, d[J], u);
      odd_sums<R, Q, J + 1>(s, d, a, u);
    }
  }
  template <int R, int Q = 1> static FFT_HD void odd_outputs(const C* s, const C* d, C x0, C* y) {
    if constexpr (2 * Q < R) {
      C a = x0, u = x0;
      odd_sums<R, Q>(s, d, a, u);
      y[Q] = cadd_si<SIGN>(a, u);
      y[R - Q] = csub_si<SIGN>(a, u);
      odd_outputs<R, Q + 1>(s, d, x0, y);
    }
  }
  template <int R> static FFT_HD void odd_prime(C* x) {
    constexpr int H = (R + 1) / 2;
    C s[H], d[H], sum = x[0];
#pragma unroll
    for (int j = 1; j < H; ++j) {
      s[j] = cadd(x[j], x[R - j]);
      d[j] = csub(x[j], x[R - j]);
      sum = cadd(sum, s[j]);
    }
    odd_outputs<R>(s, d, x[0], x);
    x[0] = sum;
  }
  // W0: x_0 carries a twiddle w_0 too
  template <int R, bool W0> static FFT_HD void run_tw(C* x, const C* w) {
    if constexpr (W0) x[0] = cmul(x[0], w[0]);
    if constexpr (R == 2) r2_tw(x[0], x[1], w[1]);
    else if constexpr (R == 3) r3_tw(x, w[1], w[2]);
    else if constexpr (R == 4) r4v_tw(x[0], x[1], x[2], x[3], w[1], w[2], w[3]);
    else if constexpr (R == 8) r8_tw(x, w);
    else if constexpr (R == 6) prime_factor<2, 3, true>(x, w);
    else if constexpr (R == 9) composite<3, 3, true>(x, w);
    else if constexpr (R == 12) prime_factor<4, 3, true>(x, w);
    else if constexpr (R == 5 || R == 7) {
#pragma unroll
      for (int r = 1; r < R; ++r) x[r] = cmul(x[r], w[r]);
      odd_prime<R>(x);
    }
    else if constexpr (R == 10) prime_factor<2, 5, true>(x, w);
    else if constexpr (R == 14) prime_factor<2, 7, true>(x, w);
    else if constexpr (R == 15) prime_factor<3, 5, true>(x, w);
    else if constexpr (R == 20) prime_factor<4, 5, true>(x, w);
    else if constexpr (R == 18) prime_factor<9, 2, true>(x, w);
    else if constexpr (R == 24) prime_factor<8, 3, true>(x, w);
    else composite<4, 4, true>(x, w);  // R == 16
  }

  // R = R1 R2 with R1, R2 coprime, in registers (the prime-factor algorithm of
  // Good and Thomas): input (R2 n1 + R1 n2) mod R and output (R2 i2 k1 + R1 i1
  // k2) mod R, i2 = R2^-1 mod R1, i1 = R1^-1 mod R2, turn the DFT into R2 DFTs
  // of length R1 and R1 of length R2 with no twiddles between them (12 = 4 x 3
  // by Cooley-Tukey spends 12 more additions or multiply-adds a butterfly on
  // them: 5% of a 96-point line's arithmetic; without them an apply at 96^3
  // went from 116.7 to 111.5 ms in FP64, 48 bands, and from 64.8 to 62.9 ms in
  // double-float, 64 bands; the FP32 passes wait on shared memory and did not
  // change).  TW: stage twiddles w[n] on the inputs, x_0 without one.
  static __host__ __device__ constexpr int inverse_mod(int a, int m) {
    for (int k = 1; k < m; ++k)
      if ((a * k) % m == 1) return k;
    return 0;
  }
  template <int R1, int R2, bool TW, int N2 = 0>
  static FFT_HD void pfa_inner(C* x, const C* w, C* a) {
    if constexpr (N2 < R2) {
      C t[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) t[n1] = x[(R2 * n1 + R1 * N2) % (R1 * R2)];
      if constexpr (TW) {
        C wt[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) wt[n1] = w[(R2 * n1 + R1 * N2) % (R1 * R2)];
        run_tw<R1, (N2 > 0)>(t, wt);
      } else {
        run<R1>(t);
      }
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) a[N2 * R1 + k1] = t[k1];
      pfa_inner<R1, R2, TW, N2 + 1>(x, w, a);
    }
  }
  template <int R1, int R2, bool TW = false>
  static FFT_HD void prime_factor(C* x, const C* w = nullptr) {
    constexpr int R = R1 * R2, c1 = R2 * inverse_mod(R2, R1), c2 = R1 * inverse_mod(R1, R2);
    C a[R];
    pfa_inner<R1, R2, TW>(x, w, a);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      C t[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) t[n2] = a[n2 * R1 + k1];
      run<R2>(t);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) x[(c1 * k1 + c2 * k2) % R] = t[k2];
    }
  }

  // w_R^m is a quarter turn (a sign change or a swap, no arithmetic)
  static __host__ __device__ constexpr bool quarter_turn(int m, int R) { return (4 * (((m % R) + R) % R)) % R == 0; }
  // every twiddle w_R^(n2 k1), 0 < n2 < R2, needs arithmetic
  template <int R2, int R> static __host__ __device__ constexpr bool all_general(int k1) {
    for (int n2 = 1; n2 < R2; ++n2)
      if (quarter_turn(n2 * k1, R)) return false;
    return true;
  }

  // R = R1 R2 in registers: R2 DFTs of length R1 over x[R2 n1 + n2] (TW: with
  // the stage twiddles w[R2 n1 + n2] on their inputs), twiddle w_R^(n2 k1),
  // R1 DFTs of length R2; output k = k1 + R1 k2.
  template <int R1, int R2, bool TW, int N2 = 0>
  static FFT_HD void inner(C* x, const C* w, C* a) {
    if constexpr (N2 < R2) {
      C t[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) t[n1] = x[R2 * n1 + N2];
      if constexpr (TW) {
        C wt[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) wt[n1] = w[R2 * n1 + N2];
        run_tw<R1, (N2 > 0)>(t, wt);
      } else {
        run<R1>(t);
      }
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) a[N2 * R1 + k1] = t[k1];
      inner<R1, R2, TW, N2 + 1>(x, w, a);
    }
  }
  template <int R1, int R2, int K1 = 0>
  static FFT_HD void outer(const C* a, C* x) {
    if constexpr (K1 < R1) {
      C t[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) t[n2] = a[n2 * R1 + K1];
      if constexpr (FftTraits<T>::fused && K1 > 0 && all_general<R2, R1 * R2>(K1)) {
        C wc[R2];
#pragma unroll
        for (int n2 = 0; n2 < R2; ++n2)
          wc[n2] = cmake<T>(factor(T(ct_trig(n2 * K1, R1 * R2, false))), factor(T(SIGN * ct_trig(n2 * K1, R1 * R2, true))));
        run_tw<R2, false>(t, wc);
      } else {
        twiddle_col<R1, R2, K1, 1>(t);
        run<R2>(t);
      }
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) x[K1 + R1 * k2] = t[k2];
      outer<R1, R2, K1 + 1>(a, x);
    }
  }
  template <int R1, int R2, int K1, int N2>
  static FFT_HD void twiddle_col(C* t) {
    if constexpr (N2 < R2) {
      t[N2] = twiddle<N2 * K1, R1 * R2>(t[N2]);
      twiddle_col<R1, R2, K1, N2 + 1>(t);
    }
  }
  template <int R1, int R2, bool TW = false>
  static FFT_HD void composite(C* x, const C* w = nullptr) {
    C a[R1 * R2];
    inner<R1, R2, TW>(x, w, a);
    outer<R1, R2>(a, x);
  }
  template <int R> static FFT_HD void run(C* x) {
    if constexpr (R == 2) r2(x);
    else if constexpr (R == 3) r3(x);
    else if constexpr (R == 4) r4(x);
    else if constexpr (R == 8) r8(x);
    else if constexpr (R == 6) prime_factor<2, 3>(x);
    else if constexpr (R == 9) composite<3, 3>(x);
    else if constexpr (R == 12) prime_factor<4, 3>(x);
    else if constexpr (R == 5 || R == 7) odd_prime<R>(x);
    else if constexpr (R == 10) prime_factor<2, 5>(x);
    else if constexpr (R == 14) prime_factor<2, 7>(x);
    else if constexpr (R == 15) prime_factor<3, 5>(x);
    else if constexpr (R == 20) prime_factor<4, 5>(x);
    else if constexpr (R == 18) prime_factor<9, 2>(x);
    else if constexpr (R == 24) prime_factor<8, 3>(x);
    else composite<4, 4>(x);  // R == 16
  }
};

// ------------------------------------------------ two-factor transforms in place
//
// The pair passes transform lines of N = A B points as
//
//   n = b + B r  (r < A, b < B),   k = q + A s  (q < A, s < B):
//   X[k] = sum_b w_B^(b s) w_N^(b q) sum_r x[b + B r] w_A^(r q)
//
// A-stage (item (line, b)): the A-point DFT over r, output q left at position
// b + B q, where the inputs came from.  B-stage (item (line, q)): the B values
// at positions B q .. B q + B - 1, twiddles w_N^(b q) on the inputs, B-point
// DFT, output s left at B q + s.  Every item reads and writes the same B or A
// positions, so a stage needs one barrier after it and none between its reads
// and writes, an item's registers are free before the next item's loads, and a
// thread holds one item (max(A, B) values) instead of all its elements of the
// line.  The frequency k ends at position spec_pos(k) = k / A + B (k mod A).
// The inverse of a spectrum in that order runs the stages backwards (B-point
// DFT over s, twiddles on the A-stage's inputs, A-point DFT over q) and leaves
// natural order.
//
// Factors: the larger one first, its DFTs without twiddles; N / 4 and 4 need the
// fewest operations (96: 24 x 4 takes 1,584 additions and multiply-adds, 8 x 12
// 1,648; FP64 forward pass at 96^3 58.9 -> 57.4 us a chain, at 60^3 15 x 4 against
// 12 x 5 15.9 -> 15.5) except at 72 and 36, and in double-float at 96, whose
// 24-point DFT is too long for the instruction cache (17.7 us against 17.2 with
// 12 x 8).
struct TwoFactor {
  int a, b;
};
template <class T, int N, int TILE = 0> constexpr TwoFactor two_factor() {
  static_assert(N == 8 || N == 12 || N == 16 || N == 20 || N == 24 || N == 28 || N == 32 || N == 36 || N == 40 ||
                    N == 48 || N == 56 || N == 60 || N == 64 || N == 72 || N == 80 || N == 96,
                "no factors chosen for this line length");
  if (TILE == 1) return N == 16 ? TwoFactor{8, 2} : TwoFactor{12, 8};
  if (N == 96 && !FftTraits<T>::fused) return TwoFactor{12, 8};
  if (N == 72) return TwoFactor{12, 6};
  if (N == 36) return TwoFactor{12, 3};
  if (N == 8 || N == 12) return TwoFactor{4, N / 4};
  return TwoFactor{N / 4, 4};
}
template <int A, int B> FFT_HD constexpr int spec_pos(int k) { return k / A + B * (k % A); }

// R consecutive twiddles in shared memory, two to a 16-byte load in FP32 (w_0 is
// not used: x_0 carries no twiddle).
template <class T, int R> __device__ __forceinline__ void load_twiddle_row(cplx<T>* w, const cplx<T>* wp) {
  if constexpr (sizeof(cplx<T>) == 8 && R % 2 == 0) {
    const float4* w4 = reinterpret_cast<const float4*>(wp);
#pragma unroll
    for (int r = 0; r < R; r += 2) {
      const float4 t = w4[r / 2];
      w[r] = cmake<T>(t.x, t.y);
      w[r + 1] = cmake<T>(t.z, t.w);
    }
  } else {
#pragma unroll
    for (int r = 1; r < R; ++r) w[r] = wp[r];
    w[0] = w[1];
  }
}

// DFT of x_0, w[1] x_1, ..., w[R-1] x_{R-1} (wp: the R twiddles in shared memory).
template <class T, int R, int SIGN>
__device__ __forceinline__ void dft_twiddled(cplx<T>* x, const cplx<T>* wp) {
  cplx<T> w[R];
  load_twiddle_row<T, R>(w, wp);
  if constexpr (FftTraits<T>::fused) {
    Dft<SIGN, T>::template run_tw<R, false>(x, w);
  } else {
#pragma unroll
    for (int r = 1; r < R; ++r) x[r] = cmul(x[r], w[r]);
    Dft<SIGN, T>::template run<R>(x);
  }
}

// item / n and item % n for a run-time 1 <= n <= 1024 and item < 65536 (one
// multiplication by a reciprocal computed once per kernel).
struct RtDiv {
  unsigned n, mag;
  __device__ __forceinline__ explicit RtDiv(int n_) : n((unsigned)n_), mag(n_ > 1 ? 0xffffffffu / (unsigned)n_ + 1u : 0u) {}
  __device__ __forceinline__ int div(int item) const { return mag ? (int)__umulhi((unsigned)item, mag) : item; }
};

// A-stage (or, with the roles of A and B exchanged by the caller, any stage) on
// lines in shared memory: item (line l, j), j < NJ, takes the R elements at
// buf + off(l) + j JS + r STEP in place.  TW: twiddles tw[j R + r].  Threads
// take items line-fast, so a warp's items are consecutive lines.
template <class T, int R, int SIGN, int NJ, int JS, int STEP, bool TW, int THR, class Off>
__device__ __forceinline__ void stage_rt(cplx<T>* buf, const cplx<T>* tw, int nlines, const RtDiv& by, const Off& off) {
  for (int item = threadIdx.x; item < nlines * NJ; item += THR) {
    const int j = by.div(item), l = item - j * nlines;
    cplx<T>* p = buf + off(l) + j * JS;
    cplx<T> x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = p[r * STEP];
    if constexpr (TW) dft_twiddled<T, R, SIGN>(x, tw + j * R);
    else Dft<SIGN, T>::template run<R>(x);
#pragma unroll
    for (int r = 0; r < R; ++r) p[r * STEP] = x[r];
  }
  __syncthreads();
}
// Items of a stage unrolled together: all of a thread's in FP32 and FP64; one
// in double-float, whose items are over a thousand instructions each.
template <class T> constexpr int kItemUnroll = FftTraits<T>::fused ? 16 : 1;

// The same with a compile-time line count and line stride LS.
template <class T, int R, int SIGN, int NJ, int JS, int STEP, bool TW, int THR, int NLINES, int LS>
__device__ __forceinline__ void stage_ct(cplx<T>* buf, const cplx<T>* tw) {
#pragma unroll(kItemUnroll<T>)
  for (int item0 = 0; item0 < NLINES * NJ; item0 += THR) {
    const int item = item0 + threadIdx.x;
    if ((NLINES * NJ) % THR == 0 || item < NLINES * NJ) {
      const int j = item / NLINES, l = item - j * NLINES;
      cplx<T>* p = buf + l * LS + j * JS;
      cplx<T> x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = p[r * STEP];
      if constexpr (TW) dft_twiddled<T, R, SIGN>(x, tw + j * R);
      else Dft<SIGN, T>::template run<R>(x);
#pragma unroll
      for (int r = 0; r < R; ++r) p[r * STEP] = x[r];
    }
  }
  __syncthreads();
}

// ------------------------------------------------ a plane in three passes
//
// With N = 4 M a plane takes three trips through registers instead of four: two
// M-point stages and one pass of 4 x 4 blocks, which does the 4-point stages of
// both axes.
//
// Inverse: the columns' M-point stage (its input read from global memory), the
// blocks, the rows' M-point stage.  For lines n = b + 4 r, k = q + M s along the
// columns (place b + 4 q after the first stage, 4 q + s after the second) and
// n = b + M r, k = q + 4 s along the rows (place b + M q, then M q + s).
template <int M> FFT_HD constexpr int plane_row_place(int k) { return 4 * (k % M) + k / M; }
template <int M> FFT_HD constexpr int plane_col_place(int k) { return M * (k % 4) + k / 4; }

// The middle pass: block item (x, y), x, y < M, rows 4x .. 4x + 3, columns y + M j.
// 4-point DFTs with twiddles tw[4 x + b] down the columns, then 4-point DFTs
// along the rows, in place.  A half warp takes 4 y of 4 consecutive x: 4 RP = 4
// modulo 16 values, so its accesses fall on distinct banks.  M is padded to a
// multiple of 4 for it; items in plain order of y collide in pairs where M is not
// one (six mixed systems on grids of 48 to 96 in one batch: 10.6 ms, 10.4 so).
template <class T, int M, int SIGN, int THR, int RP>
__device__ __forceinline__ void plane_block_pass(cplx<T>* P, const cplx<T>* tw) {
  constexpr int MG = (M + 3) / 4;  // groups of four
#pragma unroll(kItemUnroll<T>)
  for (int item0 = 0; item0 < 16 * MG * MG; item0 += THR) {
    const int item = item0 + threadIdx.x;
    const int h = item >> 4, g = h / MG;
    const int x = 4 * g + ((item >> 2) & 3), y = 4 * (h - g * MG) + (item & 3);
    if ((M % 4 != 0 || M * M % THR != 0) && (x >= M || y >= M)) continue;
    cplx<T>* p = P + 4 * x * RP + y;
    cplx<T> v[4][4];  // [row along r][column j]
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      cplx<T> c[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) c[b] = p[b * RP + j * M];
      dft_twiddled<T, 4, SIGN>(c, tw + 4 * x);
#pragma unroll
      for (int b = 0; b < 4; ++b) v[b][j] = c[b];
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      Dft<SIGN, T>::r4(v[b]);
#pragma unroll
      for (int j = 0; j < 4; ++j) p[b * RP + j * M] = v[b][j];
    }
  }
  __syncthreads();
}

// Forward: the columns' M-point stage from global memory, the rows' M-point stage,
// the blocks straight to global memory, so that shared memory holds the plane
// between the passes only: two writes and two reads, where the rows' M-point stage
// last would leave its lines across the warp's threads and need a third of each to
// store whole runs (forward pass of a chain, 96^3 2.89 -> 2.37 us, 72^3 0.87 -> 0.67,
// 48^3 0.32 -> 0.29).  The inverse ends on the rows, whose four consecutive points a
// thread the 16-byte updates want: with the blocks last and scalar updates it takes
// 3.79 us against 3.26.  Along both axes n = b + 4 r, k = q + M s; place 4 q + b of
// a row and M b + q of a column after the M-point stages.
//
// The rows' M-point stage, item (row, b): columns b + 4 r to columns M b + q.  The
// items of a row exchange columns, so they write after all have read.
template <class T, int M, int SIGN, int THR, int RP>
__device__ __forceinline__ void plane_row_stage(cplx<T>* P) {
  constexpr int N = 4 * M;
  static_assert(THR >= 4 * N, "an item a thread");
  const bool on = THR == 4 * N || threadIdx.x < 4 * N;
  const int b = threadIdx.x / N;
  cplx<T>* p = P + (threadIdx.x - b * N) * RP;
  cplx<T> x[M];
  if (on) {
#pragma unroll
    for (int r = 0; r < M; ++r) x[r] = p[b + 4 * r];
    Dft<SIGN, T>::template run<M>(x);
  }
  __syncthreads();
  if (on) {
#pragma unroll
    for (int q = 0; q < M; ++q) p[M * b + q] = x[q];
  }
  __syncthreads();
}
// The blocks, item (x, y), x, y < M: rows 4 x + b, columns y + M b; put(v, x, y)
// takes elements (x + M s, y + M t) in v[s][t].  tw[4 x + b]: e^{SIGN 2 pi i x b / N}.  Items go in
// order of y: a warp's elements are runs of M.
template <class T, int M, int SIGN, int THR, int RP, class Put>
__device__ __forceinline__ void plane_block_out(const cplx<T>* P, const cplx<T>* tw, const Put& put) {
#pragma unroll 1
  for (int item = threadIdx.x; item < M * M; item += THR) {
    const int x = item / M, y = item - x * M;
    const cplx<T>* p = P + 4 * x * RP + y;
    cplx<T> v[4][4];  // [row][column]
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      cplx<T> t[4] = {p[c * M], p[RP + c * M], p[2 * RP + c * M], p[3 * RP + c * M]};
      dft_twiddled<T, 4, SIGN>(t, tw + 4 * x);
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r][c] = t[r];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) dft_twiddled<T, 4, SIGN>(v[r], tw + 4 * y);
    put(v, x, y);
  }
}

}  // namespace fockx
