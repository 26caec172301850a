// Block fixed point for the FP64 line transforms (sm_103a).
//
// The GPU issues two FP64 instructions per clock and SM, against 64 to 128
// integer ones: an FP64 transform spends its time in the FP64 pipe (ncu: 82 to
// 86 % busy, DRAM at 3 to 7 %).  A transform needs little of what a floating
// format gives: every intermediate of a line is a sum of the line's elements
// times unit factors, so |intermediate| <= L1 = sum |x_n| of the line, known
// before the first stage.  Each line is therefore scaled by a power of two to
// L1 < 2^62, transformed in 64-bit integers, and scaled back: an add is two
// integer adds, a multiplication by a twiddle (62 fraction bits) three 32 x 32
// -> 64 multiply-adds, and nothing is rounded but the products, at 2^-62 L1.
//
// Accuracy: one unit q = 2^-62 L1 (2^-61 L1 at worst: the scale is a power of
// two).  L1 <= N rms, so q <= 2^-52 rms at 512 points, and the input rounding
// (0.29 q per component) and the product rounding (about 0.45 q per stage)
// stay at or below the rounding of an FP64 transform (2^-53 of every
// intermediate at every operation); twiddles carry 62 bits instead of 53.
// Measured against 80-bit transforms (right-hand side without diffusion, 64^3,
// 96x48x64, 256x16x128, 512x16x16): relative L2 error 2.6e-16 to 2.7e-16, with
// FP64 transforms 5.4e-16 to 6.2e-16.  256^3 RK4 step: 35.4 -> 14.0 ms (10.7 with
// the x pass one line at a time, ps_passes.cuh).
//
// Range: a line with an Inf or a NaN (or whose L1 overflows) becomes NaN as a
// whole; a line whose L1 is below 2^-937 loses bits (the scale is capped at
// 2^1021, so that results need no gradual underflow), zero lines stay zero.
// Scaling such lines by 2^512 and back, with a branch per line, restored them at
// 2 to 9 % of every FP64 right-hand side (128^3: 338 -> 356 us).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ps {

// A complex number in units of 2^-s of its line.
struct __align__(16) fx2 {
  long long x, y;
};
// A unit-circle factor: (h 2^32 + l) / 2^62 per component, |h| <= 2^30, l a
// signed word above -2^31 (both can be negated).
struct __align__(16) fxw {
  int xh, xl, yh, yl;
};

template <typename V> struct fft_of { using val = V; using tw = V; };
template <> struct fft_of<double2> { using val = fx2; using tw = fxw; };

__host__ __device__ __forceinline__ fxw cconj(fxw w) {
  fxw r;
  r.xh = w.xh;
  r.xl = w.xl;
  r.yh = -w.yh;
  r.yl = -w.yl;
  return r;
}

// v = h 2^32 + l with the low word as a signed remainder
__host__ __device__ __forceinline__ void fx_split(long long v, int& h, int& l) {
  l = (int)(unsigned)(unsigned long long)v;
  h = (int)(v >> 32) + (int)((unsigned)l >> 31);
}
// 4 P + round(Q / 2^30): P the products of high words, Q (started at 2^29)
// those of a high and a low word; the low-low products are below one unit and
// of either sign (both low words are signed).
__host__ __device__ __forceinline__ long long fx_join(long long p, long long q) {
  return (long long)((unsigned long long)p << 2) + (q >> 30);
}
constexpr long long FX_HALF = 1LL << 29;

// a w
__host__ __device__ __forceinline__ fx2 cmul(fx2 a, fxw w) {
  int xh, xl, yh, yl;
  fx_split(a.x, xh, xl);
  fx_split(a.y, yh, yl);
  const int nh = -w.yh, nl = -w.yl;
  const long long pr = (long long)xh * w.xh + (long long)yh * nh;
  const long long qr = FX_HALF + (long long)xh * w.xl + (long long)xl * w.xh + (long long)yh * nl + (long long)yl * nh;
  const long long pi = (long long)xh * w.yh + (long long)yh * w.xh;
  const long long qi = FX_HALF + (long long)xh * w.yl + (long long)xl * w.yh + (long long)yh * w.xl + (long long)yl * w.xh;
  fx2 r;
  r.x = fx_join(pr, qr);
  r.y = fx_join(pi, qi);
  return r;
}
// a times the real factor (h 2^32 + l) / 2^62
__host__ __device__ __forceinline__ long long fx_mul(long long a, int h, int l) {
  int ah, al;
  fx_split(a, ah, al);
  return fx_join((long long)ah * h, FX_HALF + (long long)ah * l + (long long)al * h);
}
// cos(pi/8), sin(pi/8), sqrt(1/2) and sqrt(3)/2 as (h, l)
constexpr int FX_C1H = 992008094, FX_C1L = 1696238673;
constexpr int FX_S1H = 410903207, FX_S1L = -1364630830;
constexpr int FX_HH = 759250125, FX_HL = -25716447;
constexpr int FX_S3H = 929887697, FX_S3L = -1332128537;
constexpr int FX_5H = 1 << 29;  // 1/2

// exp(-2 pi i m / n) for 0 <= m < n <= 2^20: the first octant by the Taylor
// series of sin and cos in unsigned 64-bit fractions (truncation below 2^-62),
// the others by symmetry.
__host__ __device__ __forceinline__ unsigned long long fx_umulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ inline fxw fx_twiddle(int m, int n) {
  const int k8 = (int)((8LL * m) % n), oct = (int)((8LL * m) / n);
  const unsigned k = (unsigned)((oct & 1) ? n - k8 : k8);  // angle k/n pi/4 from the nearer axis
  const unsigned long long pi4 = 0xC90FDAA22168C235ull;    // pi/4 2^64
  const unsigned long long x = (pi4 / n) * k + ((pi4 % n) * k) / n;
  const unsigned long long x2 = fx_umulhi(x, x);
  // sin x = x (1 - x2/6 (1 - x2/20 (...))), 1 - cos x = x2/2 (1 - x2/12 (...))
  unsigned long long ts = 0, tc = 0;
  for (int i = 10; i >= 1; --i) {
    ts = fx_umulhi(x2, 0ull - 1 - ts) / (unsigned)(2 * i * (2 * i + 1));
    if (i > 1) tc = fx_umulhi(x2, 0ull - 1 - tc) / (unsigned)((2 * i - 1) * (2 * i));
  }
  const unsigned long long sn = x - fx_umulhi(x, ts);
  const unsigned long long oc = fx_umulhi(x2, 0ull - 1 - tc) / 2;  // 1 - cos x
  const long long s = (long long)((sn + 2) >> 2), c = (1LL << 62) - (long long)((oc + 2) >> 2);
  const bool swap = ((oct + 1) >> 1) & 1;  // octants 1, 2, 5, 6
  const bool cneg = oct >= 2 && oct <= 5, sneg = oct >= 4;
  long long cv = swap ? s : c, sv = swap ? c : s;
  if (cneg) cv = -cv;
  if (!sneg) sv = -sv;  // exp(-i theta)
  fxw w;
  fx_split(cv, w.xh, w.xl);
  fx_split(sv, w.yh, w.yl);
  if (w.xl == (int)0x80000000) w.xl += 1;
  if (w.yl == (int)0x80000000) w.yl += 1;
  return w;
}

// The scale of a line from the high word u of (an upper bound of) its L1 norm
// as an FP64 number.
struct FxScale {
  int s;        // fixed = value 2^s
  int poison;   // or-ed into the high words of the results (a quiet NaN for a line with Inf or NaN)
};
__host__ __device__ __forceinline__ FxScale fx_scale(int u) {
  FxScale f;
  const int e = u >> 20;
  f.poison = e >= 0x7ff ? 0x7ff80000 : 0;
  f.s = 1084 - e < 1021 ? 1084 - e : 1021;  // L1 < 2^(e - 1022)
  return f;
}

// d 2^s to the nearest integer; |d| 2^s < 2^62.
__host__ __device__ __forceinline__ long long fx_from(int hi, int lo, int s) {
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = ((unsigned long long)((mh << 10) | ((unsigned)lo >> 22)) << 32) | ((unsigned)lo << 10);
  // value = m 2^-(1085 - s - e); one bit is left for the rounding
  unsigned r = (unsigned)(1084 - s - e);
  r = r < 63u ? r : 63u;
  const unsigned long long t = ((m >> r) + 1) >> 1;
  const long long sg = (long long)(hi >> 31);
  return ((long long)t ^ sg) - sg;
}
// v 2^-s, rounded to nearest, as the high and low word of an FP64 number.
__host__ __device__ __forceinline__ void fx_to(long long v, FxScale f, int& hi, int& lo) {
  const int vh = (int)(v >> 32);
  const long long sg = (long long)(vh >> 31);
  const unsigned long long a = (unsigned long long)((v ^ sg) - sg);
#ifdef __CUDA_ARCH__
  const int n = __clzll((long long)a);
#else
  const int n = a ? __builtin_clzll(a) : 64;
#endif
  const unsigned long long t = ((a << (n - 1)) + 0x200) >> 10;  // 53 bits: a = t 2^(11 - n)
  const int eb = a ? (1085 - f.s - n) << 20 : 0;
  hi = ((int)(t >> 32) + eb) | (vh & (int)0x80000000) | f.poison;
  lo = (int)(unsigned)t;
}

#ifdef __CUDACC__
// v over the lanes lane ^ FROM, ^ 2 FROM, ... below WIDTH: every lane of the
// aligned group of WIDTH lanes gets the same largest value or sum.
template <int FROM, int WIDTH, class V, class OP>
__device__ __forceinline__ V fx_lanes(V v, OP op) {
  unsigned mask = 0xffffffffu;
  if constexpr (WIDTH < 32) mask = ((1u << WIDTH) - 1u) << (threadIdx.x & 31 & ~(WIDTH - 1));
#pragma unroll
  for (int o = FROM; o < WIDTH; o *= 2) v = op(v, __shfl_xor_sync(mask, v, o));
  return v;
}
// High word of an upper bound of sum |re| + |im| over the E elements of each
// lane of such a group (0 when all are zero or subnormal, that of Inf for an Inf
// or NaN).  The terms are added as FP32 numbers relative to the largest exponent
// of the group: FP64 additions would take the pipe this format avoids.
template <int FROM, int WIDTH, int E>
__device__ __forceinline__ int fx_bound(const double2 (&a)[E]) {
  int hm = 0;
#pragma unroll
  for (int m = 0; m < E; ++m) {
    hm = max(hm, __double2hiint(a[m].x) & 0x7fffffff);
    hm = max(hm, __double2hiint(a[m].y) & 0x7fffffff);
  }
  if constexpr (FROM == 1 && WIDTH == 32) hm = __reduce_max_sync(0xffffffffu, hm);
  else hm = fx_lanes<FROM, WIDTH>(hm, [](int x, int y) { return max(x, y); });
  const int base = (hm & 0x7ff00000) - (127 << 20);
  float f = 0.f;
#pragma unroll
  for (int m = 0; m < E; ++m) {
    f += __int_as_float(max((__double2hiint(a[m].x) & 0x7fffffff) - base, 0) << 3);
    f += __int_as_float(max((__double2hiint(a[m].y) & 0x7fffffff) - base, 0) << 3);
  }
  f = fx_lanes<FROM, WIDTH>(f, [](float x, float y) { return x + y; });
  // truncated terms (2^-20 of each) and the FP32 sums: raised by 2^-9
  const unsigned u = (unsigned)((__float_as_int(f) >> 3) + base + (1 << 11));
  return hm < 0x00100000 ? 0 : (int)min(u, 0x7ff00000u);
}
// u + v of two such words
__device__ __forceinline__ int fx_add_bound(int u, int v) {
  const unsigned w = (unsigned)__double2hiint(__hiloint2double(u, 0) + __hiloint2double(v, 0)) + 1u;
  return (int)min(w, 0x7ff00000u);
}
template <int E>
__device__ __forceinline__ void fx_load(fx2 (&b)[E], const double2 (&a)[E], FxScale f) {
#pragma unroll
  for (int m = 0; m < E; ++m) {
    b[m].x = fx_from(__double2hiint(a[m].x), __double2loint(a[m].x), f.s);
    b[m].y = fx_from(__double2hiint(a[m].y), __double2loint(a[m].y), f.s);
  }
}
__device__ __forceinline__ double2 fx_value(fx2 v, FxScale f) {
  int xh, xl, yh, yl;
  fx_to(v.x, f, xh, xl);
  fx_to(v.y, f, yh, yl);
  return make_double2(__hiloint2double(xh, xl), __hiloint2double(yh, yl));
}
#endif

}  // namespace ps
