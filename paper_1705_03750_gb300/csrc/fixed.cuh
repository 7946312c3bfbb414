// 64-bit fixed-point arithmetic for the FP64 paths.
//
// FP64 executes at two lanes per SM per clock here, 1/64 of the 32-bit rate,
// so a value that feeds no integer decision of the method is evaluated on the
// integer pipes instead, with more fraction bits than a double's 53: offsets
// in cells with FX_Q = 52 bits after the point (their FP64 evaluation, an
// index position of up to 2^13 cells, keeps 39 to 52), and sums of node
// values in units of 2^-59 of the largest one.
#pragma once

#include <stdint.h>

namespace vm {

constexpr int FX_Q = 52;        // fraction bits of offsets in cells
constexpr int FX_LIM = 32;      // largest site offset from an element's start site
constexpr double FX_MAX = 1900.0;  // bound on |offset| in cells (2^11 is the format's range)
// A node decision is taken from the fixed-point offset when it clears the
// half-integer by 2^-26 cells; the FP64 evaluation in the fixed order is
// within 1e-10 cells of it (terms up to FX_MAX, positions up to 2^14 cells,
// some forty roundings).
constexpr long long FX_MARGIN = 1ll << (FX_Q - 26);

// Record of one element's inverse map, 128 bytes: the index position of
// Q(P) along each axis at site (i0 + j, l0 + l), relative to the integer
// anchor B, is c0 + j (c1 + j c3 + l c4) + l (c2 + l c5) cells, exactly the
// second-order map of Sec. 2.1 expanded about the element's start site; the
// coefficients of the x axis, then of the v axis, then the integers.
struct __align__(16) FxRec {
  long long c[12];
  int i0, l0, Bu, Bw;
  int lim;  // the record serves sites with |j|, |l| < lim (0: none, not the start site either)
  int pad[3];
};
static_assert(sizeof(FxRec) == 128, "one cache line per element");

// c0 + j (c1 + j c3 + l c4) + l (c2 + l c5), integers throughout.
__device__ __forceinline__ long long fx_poly(const longlong2 a, const longlong2 b, const longlong2 c, int j, int l) {
  return a.x + (long long)j * (a.y + (long long)j * b.y + (long long)l * c.x) +
         (long long)l * (b.x + (long long)l * c.y);
}

// Distance in cells from P to site i of the axis lo + i d: |i d + (lo - P)|
// is at most half a cell, so the fused operation is exact but for the
// rounding of lo - P, which is carried (TwoSum).
__device__ __forceinline__ double cells_from(double P, double lo, double d, double inv_d, double i) {
  const double a = lo - P, b = a - lo, e = (lo - (a - b)) - (P + b);
  return (fma(i, d, a) + e) * inv_d;
}

// c in units of 2^-q, rounded to nearest, |c| 2^q < 2^63 (from the bits of c).
__device__ __forceinline__ long long fx_of(double c, int q) {
  const int hi = __double2hiint(c);
  const unsigned long long mant =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(c);
  const int sh = 1075 - q - ((hi >> 20) & 0x7ff);  // bits to drop
  unsigned long long v;
  if (sh <= 0)
    v = mant << -sh;
  else
    v = sh > 62 ? 0ull : (mant + (1ull << (sh - 1))) >> sh;
  const long long sg = (long long)(hi >> 31);
  return ((long long)v ^ sg) - sg;
}

// a * E / 2^62 (|E| <= 2^62: a factor of at most 1).
__device__ __forceinline__ long long fx_mul62(long long a, long long E) {
  return (long long)(((unsigned long long)__mul64hi(a, E) << 2) | ((unsigned long long)(a * E) >> 62));
}

// a * X / 2^64, X a non-negative Q64 fraction below 1/2.
__device__ __forceinline__ long long fx_mul(long long a, long long X) { return __mul64hi(a, X); }

__device__ __forceinline__ int fx_exp(double F) { return (__double2hiint(F) >> 20) & 0x7ff; }

// F in units of 2^(emax - 1075 - UP): |result| <= 2^(53 + UP) (truncated
// towards zero), emax the largest biased exponent of the values used together.
template <int UP = 7>
__device__ __forceinline__ long long fx_int(double F, int emax) {
  const int hi = __double2hiint(F);
  const unsigned long long mant =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(F);
  const int sh = emax - ((hi >> 20) & 0x7ff);
  const long long v = (long long)((mant << UP) >> (sh < 63 ? sh : 63));
  const long long sg = (long long)(hi >> 31);
  return (v ^ sg) - sg;
}

// S * 2^(emax - 1082) for 128 <= emax <= 2040 and |S| < 2^63.
__device__ __forceinline__ double fx_double(long long S, int emax) {
  const double d = __ll2double_rn(S);
  return S ? __hiloint2double(__double2hiint(d) + ((emax - 1082) << 20), __double2loint(d)) : 0.0;
}

// Sum of at most four products of values (|v| <= 2^60) with non-negative
// weights w (2^-60 units, their sum at most 1): four 32-bit products a term
// accumulated in 64 bits each, to about two units.
struct FxDot {
  long long hh = 0, hl = 0;
  unsigned long long lh = 0, ll = 0;
  __device__ __forceinline__ void add(long long v, int wh, int wl) {
    const int vh = (int)(v >> 32);
    const unsigned vl = (unsigned)v;
    hh += (long long)vh * wh;
    hl += (long long)vh * wl;
    lh += (unsigned long long)vl * (unsigned)wh;
    ll += (unsigned long long)(vl >> 2) * (unsigned)wl;
  }
  __device__ __forceinline__ long long sum() const {
    return (hh << 3) + (hl >> 28) + (long long)(lh >> 29) + (long long)(ll >> 58);
  }
};
// A weight in 2^-62 units as the two halves FxDot takes.
__device__ __forceinline__ void fx_split(long long w, int& wh, int& wl) {
  wh = (int)(w >> 33);
  wl = (int)((unsigned)(w >> 2) & 0x7fffffffu);
}

// Is site (i, j) within the record's reach?  Then its offset from the anchor
// o.z, o.w along each axis.
__device__ __forceinline__ bool fx_offset(const FxRec* __restrict__ X, int i, int j, long long& ru, long long& rw,
                                          int4& o) {
  o = __ldg(reinterpret_cast<const int4*>(&X->i0));
  const int lim = __ldg(&X->lim);
  const longlong2* c = reinterpret_cast<const longlong2*>(X->c);
  const longlong2 x0 = __ldg(c), x1 = __ldg(c + 1), x2 = __ldg(c + 2);
  const longlong2 v0 = __ldg(c + 3), v1 = __ldg(c + 4), v2 = __ldg(c + 5);
  const int dj = i - o.x, dl = j - o.y;
  ru = fx_poly(x0, x1, x2, dj, dl);
  rw = fx_poly(v0, v1, v2, dj, dl);
  return max(abs(dj), abs(dl)) < lim;
}

// Square root of d2 (2^-60 units, 0 <= d2 < 2^60) in 2^-62 units: an FP32
// root and two corrections from the exact remainder, each of some 23 bits.
__device__ __forceinline__ long long fx_sqrt(long long d2) {
  if (d2 < 16) return 0;
  const float f = (float)d2, r = rsqrtf(f);
  long long D = (long long)(f * r * 4294967296.f);  // sqrt(d2) 2^30 -> 2^62 units
#pragma unroll
  for (int it = 0; it < 2; it++) {
    const long long rem = d2 - __mul64hi(D, D);      // 2^-60 units
    D += (long long)((float)rem * r * 2147483648.f);  // rem / (2 d)
  }
  return D;
}

// The Monaghan kernel W(2d) (Sec. 2.3.2) from d^2 (2^-60 units, below 1), in
// 2^-62 units: 1 - 6 d^2 (1 - d) up to d = 1/2, 2 (1 - d)^3 beyond.
__device__ __forceinline__ long long fx_kernel(long long d2) {
  constexpr long long one = 1ll << 62;
  const long long e = one - fx_sqrt(d2);
  if (e >= (one >> 1)) return one - 6 * (__mul64hi(d2, e) << 4);
  return __mul64hi(__mul64hi(e << 1, e << 1) << 2, e << 1);
}

// num / den, den in 2^-59 units and positive, to about 2^-46 |num / den|
// after the third term.
__device__ __forceinline__ long long fx_div(long long num, long long den) {
  const float r = 1.f / (float)den * 5.764607523034235e17f;  // 2^59 / den
  long long q = (long long)((float)num * r);
#pragma unroll
  for (int it = 0; it < 2; it++) {
    const long long rem = num - ((__mul64hi(q, den) << 5) | (long long)((unsigned long long)(q * den) >> 59));
    q += (long long)((float)rem * r);
  }
  return q;
}

// Cubic B-spline weights of the four nodes around fraction t (2^-62 units).
__device__ __forceinline__ void fx_bspline(long long t, long long (&b)[4]) {
  constexpr long long one = 1ll << 62, two3 = 0x2AAAAAAAAAAAAAABll, sixth = 0x2AAAAAAAAAAAAAABll;  // 2/3 2^62; 2^64/6
  const long long z = one - t;
  const long long t2 = __mul64hi(t, t), t3 = __mul64hi(t2, t), z2 = __mul64hi(z, z), z3 = __mul64hi(z2, z);
  b[0] = __mul64hi(z3 << 4, sixth);
  b[1] = two3 - (t2 << 2) + (t3 << 3);
  b[2] = two3 - (z2 << 2) + (z3 << 3);
  b[3] = __mul64hi(t3 << 4, sixth);
}

}  // namespace vm
