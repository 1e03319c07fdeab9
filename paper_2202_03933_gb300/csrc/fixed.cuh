// Fixed-point arithmetic of the quadrature loops on the integer pipe.
//
// GB300 issues 2 FP64 operations per SM and clock but 32 lanes of the
// 32 x 32 + 64 bit multiply-add (mad.wide; 24.9 measured against 1.68 DFMA at
// the same clock), so a 64-bit fixed-point product made of three mad.wide runs
// about five times as fast as a DFMA, and additions, shifts and comparisons of
// 64-bit integers cost next to nothing.  The quantities of a quadrature point
// are bounded -- in-plane coordinates by the pair's extent, element parameters
// and shape functions by 1, weights by the polygon's area -- which is all that
// fixed point needs.  Resolution: in-plane coordinates of a pair are held to
// 2^-62 of the pair's extent in their direction (FP64 has 2^-53 of the
// coordinate), parameters to about 2^-57 (2^-54 at worst, kMaxMapBits); factors
// that stay small over a whole pair are scaled up first, so that small entries
// keep their relative accuracy.
//
// A value is an int64 with a fixed number of fraction bits ("Q60" = 60).  For
// a product it is written with balanced digits v = h 2^32 + l, l in
// [-2^31, 2^31), and
//     a b / 2^64 = a.h b.h + (a.h b.l + a.l b.h) / 2^32 + a.l b.l / 2^64;
// the last term (at most 1/4 unit of 2^64) is dropped.  Sums of products keep
// the two remaining parts apart and are normalised once.  Overflow: with
// |h| <= 2^29 a cross product is at most 2^60, so the cross sum of up to three
// products stays below 2^63; where a longer sum is formed its bound is given.
#pragma once

#include "clip.cuh"

namespace mortar {

struct Dg {
  int h, l;
};

__device__ __forceinline__ Dg fx_split(long long v) {
  const int l = (int)v;
  return {(int)(v >> 32) + (int)((unsigned)l >> 31), l};
}

// Written as the instruction: from C expressions the compiler forms the
// product and a separate 64-bit addition (7 instead of 3 multiply-pipe
// instructions for a product of the sums below).
#ifdef __CUDA_ARCH__
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ long long mul_wide(int a, int b) {
  long long d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ int mul_hi(int a, int b) { return __mulhi(a, b); }
__device__ __forceinline__ unsigned shift_in(unsigned lo, unsigned hi, int k) { return __funnelshift_l(lo, hi, k); }
__device__ __forceinline__ float rcp_f32(float x) {   // about 1 ulp; seeds only
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
#else
inline long long mad_wide(int a, int b, long long c) { return (long long)a * b + c; }
inline long long mul_wide(int a, int b) { return (long long)a * b; }
inline int mul_hi(int a, int b) { return (int)(((long long)a * b) >> 32); }
inline unsigned shift_in(unsigned lo, unsigned hi, int k) {
  return (unsigned)((((unsigned long long)hi << 32 | lo) << k) >> 32);
}
inline float rcp_f32(float x) { return 1.0f / x; }
#endif

// Sum of products in units of 2^64: hh + cr / 2^32.
struct FxAcc {
  long long hh, cr;
  __device__ __forceinline__ void zero() { hh = 0; cr = 0; }
  __device__ __forceinline__ void mul(Dg a, Dg b) {   // first product
    hh = mul_wide(a.h, b.h);
    cr = mad_wide(a.l, b.h, mul_wide(a.h, b.l));
  }
  __device__ __forceinline__ void mac(Dg a, Dg b) {
    hh = mad_wide(a.h, b.h, hh);
    cr = mad_wide(a.l, b.h, mad_wide(a.h, b.l, cr));
  }
  // the sum times 2^k, 0 <= k < 32: the cross sum's whole units are added by a
  // multiply-add (one instruction), then both words shifted
  __device__ __forceinline__ long long get(int k) const {
    const long long t = mad_wide((int)(cr >> 32), 1, hh);
    return (long long)((unsigned long long)shift_in((unsigned)t, (unsigned)((unsigned long long)t >> 32), k) << 32 |
                       shift_in((unsigned)cr, (unsigned)t, k));
  }
  template <int K>
  __device__ __forceinline__ long long get() const { return get(K); }
  // the low digits' product of the last mul or mac, where 2^-2 unit matters
  __device__ __forceinline__ void low(Dg a, Dg b) { cr += mul_hi(a.l, b.l); }
  // moves the whole units of the cross sum into hh (keeps the fraction): bounds cr between runs of products
  __device__ __forceinline__ void carry() {
    hh += cr >> 32;
    cr = (long long)(unsigned)cr;
  }
};

// d 2^k as an integer (truncated); |d| 2^k < 2^63.
__device__ __forceinline__ long long fx_of_double(double d, int k) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7ffu);
  const int sh = 1085 - e - k;   // (mantissa << 10) >> sh
  unsigned long long m = ((b << 10) & 0x3ffffffffffffc00ull) | 0x4000000000000000ull;
  m = (e == 0 || sh > 62) ? 0ull : m >> (sh < 0 ? 0 : sh);
  return (long long)b < 0 ? -(long long)m : (long long)m;
}

// Exponent E with |d| < 2^E (normal numbers; very small for zero).
__device__ __forceinline__ int fx_exponent(unsigned hi_abs) { return (int)(hi_abs >> 20) - 1022; }
__device__ __forceinline__ unsigned fx_hi_abs(double d) {
  return (unsigned)((unsigned long long)__double_as_longlong(d) >> 32) & 0x7fffffffu;
}

// (hh + cr / 2^32) 2^k rounded to FP64; the result is zero or a normal number.
__device__ __forceinline__ double fx_to_double(long long hh, long long cr, int k) {
  long long hi = hh + (cr >> 32);
  unsigned lo = (unsigned)cr;
  const bool neg = hi < 0;
  if (neg) {
    lo = 0u - lo;
    hi = ~hi + (lo == 0u ? 1 : 0);
  }
  if (hi == 0) {
    if (lo == 0u) return 0.0;
    hi = (long long)lo;
    lo = 0u;
    k -= 32;
  }
  const int n = __clzll(hi);
  unsigned long long top = (unsigned long long)hi << n;
  if (n > 0) top |= n <= 32 ? (unsigned long long)lo >> (32 - n) : (unsigned long long)lo << (n - 32);
  const unsigned long long m = (top >> 11) + ((top >> 10) & 1ull);   // 2^52 <= m <= 2^53
  const long long e = 1023 + 63 - n + k;
  const unsigned long long bits = ((unsigned long long)(e - 1) << 52) + m;
  return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
}

__device__ __forceinline__ float fx_f32(long long v) { return (float)(int)(v >> 32); }   // in units of 2^32

constexpr Dg fx_const(double v) {   // digits of v 2^62
  const long long q = (long long)(v * 4611686018427387904.0);
  const int l = (int)(unsigned)(unsigned long long)q;
  return {(int)(q >> 32) + (l < 0 ? 1 : 0), l};
}

// The 7-point rule (Tri7) in Q62: weights by point, and of its orbits (0: the
// centroid, 1: points 1-3, 2: points 4-6, barycentric (a, b), (b, a), (a, a)
// as in tri7_point) the coordinate a and the difference b - a.
struct Tri7Fx {
  Dg w[7];
};
struct OrbitFx {
  Dg a[3], d[3];
};
constexpr Tri7Fx tri7_fx() {
  return {{fx_const(Tri7::w0), fx_const(Tri7::w1), fx_const(Tri7::w1), fx_const(Tri7::w1), fx_const(Tri7::w2),
           fx_const(Tri7::w2), fx_const(Tri7::w2)}};
}
constexpr OrbitFx orbit_fx() {
  return {{fx_const(1.0 / 3.0), fx_const(Tri7::a1), fx_const(Tri7::a2)},
          {fx_const(0.0), fx_const(Tri7::b1 - Tri7::a1), fx_const(Tri7::b2 - Tri7::a2)}};
}
static __constant__ Tri7Fx kTri7Fx = tri7_fx();
static __constant__ OrbitFx kOrbitFx = orbit_fx();

// 1 / n in Q62 (the vertex-mean centroid)
struct InvCountFx {
  Dg d[17];
};
constexpr InvCountFx inv_count_fx() {
  InvCountFx t{};
  for (int n = 1; n < 17; ++n) t.d[n] = fx_const(n == 1 ? 0.9999999999999999 : 1.0 / n);
  return t;
}
static __constant__ InvCountFx kInvCountFx = inv_count_fx();

// Most bits that an element's inverse map may amplify the frame's 2^-62 by: xi
// is then resolved to 2^-54 (FP64: 2^-53 of the element).  Elements 2^6 or so
// smaller than the frame, and needles that lie across its axes, exceed it, and
// the pair takes the FP64 path.  Stretched elements along the axes do not: the
// frame has an exponent for each direction.  Parallelogram pairs (random
// overlaps, 1.1 times as large masters, geometric mean of the block's largest
// error over its largest entry): with one exponent for both directions and kb up
// to 20 1.7e-16, 7.5e-16, 7e-15, 7e-14 at aspects 1, 1e3, 1e4, 1e5; FP64 2e-16
// throughout, and this form 1.7e-16 throughout.
constexpr int kMaxMapBits = 8;

// One element's map in the pair's frame (in-plane coordinates u 2^-Eu, v 2^-Ev,
// Q62, below 1/2) and its inverse; parameters are Q61.  Affine maps: xi = B (x - c0)
// with B = 2^kb B', |B'| < 1 in Q61.  Bilinear maps: FP32 Newton in units of
// 2^-30, then two steps with the residual in fixed point and the FP32
// iteration's last Jacobian inverse G.  The last FP32 step is at most 1e-4, so
// G is J^-1 to a relative d ~ 1e-5 (1e-4 |c3| / |J|) and the FP32 iterate is
// within a few 1e-7: the steps leave d 1e-7 and d^2 1e-7 ~ 1e-17, so what
// remains is the residual's rounding, 2^-60 over the Jacobian (about 2^-57 in
// xi).  A second step above 2^-36 means that G was no good approximation, and
// the point goes to the FP64 Newton.
struct FxMap {
  bool affine;
  long long c0u, c0v, c1u, c1v;
  Dg k1u, k1v, k2u, k2v, k3u, k3v;   // bilinear: c1, c2, c3 (Q62); affine: the rows k1u k1v, k2u k2v of B'
  int kb;                            // 2^kb above the inverse map's entries (bilinear: at the centre)
  float f1u, f1v, f2u, f2v, f3u, f3v, b00, b01, b10, b11;
  float g00, g01, g10, g11;          // last solve's FP32 Jacobian inverse (xi per 2^-30 of the frame)

  // false if the inverse amplifies too much
  __device__ __forceinline__ bool setup_bilinear(const PlaneMap& m, int Eu, int Ev) {
    affine = false;
    const int ku = 62 - Eu, kv = 62 - Ev;
    c0u = fx_of_double(m.c0u, ku);
    c0v = fx_of_double(m.c0v, kv);
    k1u = fx_split(fx_of_double(m.c1u, ku));
    k1v = fx_split(fx_of_double(m.c1v, kv));
    k2u = fx_split(fx_of_double(m.c2u, ku));
    k2v = fx_split(fx_of_double(m.c2v, kv));
    k3u = fx_split(fx_of_double(m.c3u, ku));
    k3v = fx_split(fx_of_double(m.c3v, kv));
    bilinear_floats();
    const float b = fmaxf(fmaxf(fabsf(b00), fabsf(b01)), fmaxf(fabsf(b10), fabsf(b11)));   // xi per 2^-30
    kb = min(max(0, (int)(__float_as_uint(b) >> 23) - 126 + 30), 31);
    return kb <= kMaxMapBits;
  }
  // what follows from the digits
  __device__ __forceinline__ void bilinear_floats() {
    c1u = ((long long)k1u.h << 32) + k1u.l;
    c1v = ((long long)k1v.h << 32) + k1v.l;
    f1u = (float)k1u.h; f1v = (float)k1v.h;
    f2u = (float)k2u.h; f2v = (float)k2v.h;
    f3u = (float)k3u.h; f3v = (float)k3v.h;
    const float fd = rcp_f32(f1u * f2v - f2u * f1v);
    b00 = f2v * fd; b01 = -f2u * fd; b10 = -f1v * fd; b11 = f1u * fd;
  }
  // i: inverse of [c1 c2] (rows); false if it amplifies too much
  __device__ __forceinline__ bool setup_affine(const PlaneMap& m, double i00, double i01, double i10, double i11,
                                               int Eu, int Ev) {
    affine = true;
    c0u = fx_of_double(m.c0u, 62 - Eu);
    c0v = fx_of_double(m.c0v, 62 - Ev);
    const int eu = fx_exponent(max(fx_hi_abs(i00), fx_hi_abs(i10))), ev = fx_exponent(max(fx_hi_abs(i01), fx_hi_abs(i11)));
    kb = max(0, max(eu + Eu, ev + Ev));   // |B|, a column times 2^Eu, the other 2^Ev, < 2^kb
    if (kb > kMaxMapBits) return false;
    const int ku = 61 + Eu - kb, kv = 61 + Ev - kb;
    k1u = fx_split(fx_of_double(i00, ku));
    k1v = fx_split(fx_of_double(i01, kv));
    k2u = fx_split(fx_of_double(i10, ku));
    k2v = fx_split(fx_of_double(i11, kv));
    const float f = __uint_as_float((unsigned)(127 - 59 + kb) << 23);   // high words: B' 2^29, x 2^30
    b00 = (float)k1u.h * f; b01 = (float)k1v.h * f; b10 = (float)k2u.h * f; b11 = (float)k2v.h * f;
    return true;
  }

  // FP32 xi of a bilinear map's point (error a few 2^(kb - 24)); false if the
  // iteration did not settle.  Three Newton updates without a test settle
  // ordinary elements, and their straight code lets several points of a thread
  // overlap.
  __device__ __forceinline__ void newton_f32(float tu, float tv, float& x, float& y, float& step) {
    const float ru = fmaf(f3u * x, y, fmaf(f1u, x, fmaf(f2u, y, -tu)));
    const float rv = fmaf(f3v * x, y, fmaf(f1v, x, fmaf(f2v, y, -tv)));
    const float j00 = fmaf(f3u, y, f1u), j01 = fmaf(f3u, x, f2u);
    const float j10 = fmaf(f3v, y, f1v), j11 = fmaf(f3v, x, f2v);
    const float id = rcp_f32(j00 * j11 - j01 * j10);
    g00 = j11 * id; g01 = -j01 * id; g10 = -j10 * id; g11 = j00 * id;
    const float d0 = fmaf(g00, ru, g01 * rv), d1 = fmaf(g10, ru, g11 * rv);
    x -= d0;
    y -= d1;
    step = fabsf(d0) + fabsf(d1);
  }
  __device__ __forceinline__ bool settle(float tu, float tv, float& x, float& y) {
    float step;
    x = b00 * tu + b01 * tv;
    y = b10 * tu + b11 * tv;
#pragma unroll
    for (int it = 0; it < 3; ++it) newton_f32(tu, tv, x, y, step);
    if (!(step <= 1e-4f)) {
#pragma unroll 1
      for (int it = 0; it < 13 && !(step <= 1e-4f); ++it) newton_f32(tu, tv, x, y, step);
    }
    return step <= 1e-4f;
  }
  __device__ __forceinline__ bool coarse(float tu, float tv, float& x, float& y) {
    return settle(tu, tv, x, y) && fabsf(x) < 1.01f && fabsf(y) < 1.01f;
  }

  // FP32 xi of the point x (Q62), for bounds only; false if it did not settle
  template <int NEN>
  __device__ __forceinline__ bool solve_f32(long long xu, long long xv, float& x, float& y) {
    const float tu = fx_f32(xu - c0u), tv = fx_f32(xv - c0v);
    if (NEN == 3 || affine) {
      x = b00 * tu + b01 * tv;
      y = b10 * tu + b11 * tv;
      return true;
    }
    return coarse(tu, tv, x, y);
  }

  // |c| < 1/2 and |xi| < 1.01: the cross sums stay below 2^62.4
  __device__ __forceinline__ void residual(long long du, long long dv, long long xi, long long eta, long long& ru,
                                           long long& rv) const {
    const Dg x = fx_split(xi), y = fx_split(eta);
    FxAcc a;
    a.mul(k3u, y);
    const Dg ju = fx_split(c1u + a.get<3>());
    a.mul(k3v, y);
    const Dg jv = fx_split(c1v + a.get<3>());
    a.mul(ju, x);
    a.mac(k2u, y);
    ru = a.get<3>() - du;
    a.mul(jv, x);
    a.mac(k2v, y);
    rv = a.get<3>() - dv;
  }

  // affine: xi (Q61) at d = x - c0
  __device__ __forceinline__ void solve_affine(long long du, long long dv, long long& xi, long long& eta) const {
    const Dg a = fx_split(du), b = fx_split(dv);
    FxAcc s;
    s.mul(k1u, a);
    s.mac(k1v, b);
    xi = s.get(2 + kb);
    s.mul(k2u, a);
    s.mac(k2v, b);
    eta = s.get(2 + kb);
  }
  // bilinear: the two fixed-point steps from the FP32 iterate (x, y)
  __device__ __forceinline__ bool refine(long long du, long long dv, float x, float y, long long& xi,
                                         long long& eta) const {
    xi = (long long)__float2int_rn(x * 0x1p30f) << 31;
    eta = (long long)__float2int_rn(y * 0x1p30f) << 31;
    long long ru, rv;
    residual(du, dv, xi, eta, ru, rv);
    {
      const float fu = (float)(int)(ru >> 18), fv = (float)(int)(rv >> 18);   // units of 2^-44
      xi -= (long long)__float2int_rn(fmaf(g00, fu, g01 * fv) * 0x1p27f) << 20;
      eta -= (long long)__float2int_rn(fmaf(g10, fu, g11 * fv) * 0x1p27f) << 20;
    }
    residual(du, dv, xi, eta, ru, rv);
    if (ru != (int)ru || rv != (int)rv) return false;
    const float fu = (float)(int)ru, fv = (float)(int)rv;   // units of 2^-62
    const float d0 = fmaf(g00, fu, g01 * fv) * 0x1p29f, d1 = fmaf(g10, fu, g11 * fv) * 0x1p29f;
    xi -= (long long)__float2int_rn(d0);
    eta -= (long long)__float2int_rn(d1);
    return fmaxf(fabsf(d0), fabsf(d1)) < 0x1p25f;
  }
  // xi (Q61) of the point x (Q62); false if the FP32 or the fixed-point steps did not settle
  template <int NEN>
  __device__ __forceinline__ bool solve(long long xu, long long xv, long long& xi, long long& eta) {
    const long long du = xu - c0u, dv = xv - c0v;
    if (NEN == 3 || affine) {
      solve_affine(du, dv, xi, eta);
      return true;
    }
    float x, y;
    return coarse(fx_f32(du), fx_f32(dv), x, y) && refine(du, dv, x, y, xi, eta);
  }
};

// Left shift that brings values up to `m` + err to 1 at most.
__device__ __forceinline__ int fx_room(float m, float err) {
  const int e = (int)(__float_as_uint(fmaxf(m, 0.0f) + err) >> 23) - 126;   // m + err < 2^e
  return min(max(-e, 0), 16);
}

// Scales of the shape-function factors of one element over a pair's polygon:
// a factor (1 -+ xi) / 2, (1 -+ eta) / 2 (quad4) or a shape function itself
// (tri3) that is below 2^-k at every vertex is held with k more bits.  The
// level sets of xi and eta are straight lines, so the polygon's vertices bound
// them.
struct FxScales {
  int k[4];   // quad4: 1 - xi, 1 + xi, 1 - eta, 1 + eta; tri3: N0, N1, N2
  template <int NEN>
  __device__ __forceinline__ int shape(int a) const {   // of shape function a
    if (NEN == 3) return k[a];
    return (a == 1 || a == 2 ? k[1] : k[0]) + (a < 2 ? k[2] : k[3]);
  }
};
template <int NEN>
__device__ __forceinline__ bool fx_scales(FxMap& m, const long long* X, const long long* Y, int nr, FxScales& s) {
  float lo1 = 1.0f, hi1 = -1.0f, lo2 = 1.0f, hi2 = -1.0f, lo3 = 1.0f;
  bool ok = true;
#pragma unroll 1
  for (int k = 0; k < nr; ++k) {
    float x, y;
    ok &= m.template solve_f32<NEN>(X[k], Y[k], x, y);
    lo1 = fminf(lo1, x); hi1 = fmaxf(hi1, x);
    lo2 = fminf(lo2, y); hi2 = fmaxf(hi2, y);
    lo3 = fminf(lo3, x + y);
  }
  if (!ok) {   // no bound: unscaled
    s.k[0] = s.k[1] = s.k[2] = s.k[3] = 0;
    return true;
  }
  // FP32 rounding of the parameters, whose sums' terms are up to 2^kb
  const float err = 1e-5f + __uint_as_float((unsigned)(127 - 21 + m.kb) << 23);
  if (NEN == 4) {
    s.k[0] = fx_room(0.5f * (1.0f - lo1), err); s.k[1] = fx_room(0.5f * (1.0f + hi1), err);
    s.k[2] = fx_room(0.5f * (1.0f - lo2), err); s.k[3] = fx_room(0.5f * (1.0f + hi2), err);
  } else {
    s.k[0] = fx_room(1.0f - lo3, err); s.k[1] = fx_room(hi1, err); s.k[2] = fx_room(hi2, err); s.k[3] = 0;
  }
  return fmaxf(fmaxf(-lo1, hi1), fmaxf(-lo2, hi2)) < 1.01f;
}

// Common frame of a pair, an exponent for each in-plane direction: 2^Eu at
// least twice the largest u of the slave window and the largest u coefficient
// of the master map, 2^Ev as much for v.  (The slave's first edge is along u, so
// that stretched elements are, as a rule, along the axes.)  Not ok out of range.
struct FxFrame {
  int Eu, Ev;
  bool ok;
};
template <int NS, int NM>
__device__ __forceinline__ FxFrame fx_frame(const double* __restrict__ r, const PlaneMap& m) {
  unsigned hu = max(max(fx_hi_abs(m.c0u), fx_hi_abs(m.c1u)), fx_hi_abs(m.c2u));
  unsigned hv = max(max(fx_hi_abs(m.c0v), fx_hi_abs(m.c1v)), fx_hi_abs(m.c2v));
  if (NM == 4) {
    hu = max(hu, fx_hi_abs(m.c3u));
    hv = max(hv, fx_hi_abs(m.c3v));
  }
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    hu = max(hu, fx_hi_abs(r[SR_PS + 2 * k]));
    hv = max(hv, fx_hi_abs(r[SR_PS + 2 * k + 1]));
  }
  const int Eu = fx_exponent(hu) + 1, Ev = fx_exponent(hv) + 1;
  return {Eu, Ev, Eu > -300 && Eu < 300 && Ev > -300 && Ev < 300};
}

// FP64 Newton from xi = 0 for a point whose fixed-point steps did not settle
// (strongly distorted elements); false if it fails or leaves the element.
static __device__ __noinline__ bool fx_slow_solve(PlaneMap m, int Eu, int Ev, long long xu, long long xv,
                                                  long long& xi, long long& eta) {
  MapInverse mi;
  mi.m = m;
  double a = 0.0, b = 0.0;
  if (!mi.newton64(fx_to_double(xu, 0, Eu - 62), fx_to_double(xv, 0, Ev - 62), a, b)) return false;
  if (!(fabs(a) < 1.01 && fabs(b) < 1.01)) return false;
  xi = fx_of_double(a, 61);
  eta = fx_of_double(b, 61);
  return true;
}

__device__ __forceinline__ PlaneMap slave_plane_map(const double* __restrict__ r) {
  return {r[SR_C], r[SR_C + 1], r[SR_C + 2], r[SR_C + 3], r[SR_C + 4], r[SR_C + 5], r[SR_C + 6], r[SR_C + 7]};
}

// The projected map of master element m in the plane of slave record r (as clip_polygon forms it).
template <int NM>
__device__ __noinline__ PlaneMap master_plane_map(const double* __restrict__ r, const double* __restrict__ xm,
                                                  const int32_t* __restrict__ conn_m, int32_t m) {
  double mu[4], mv[4];
  project_master<NM>(r, xm, conn_m + (int64_t)NM * m, mu, mv);
  return plane_map<NM>(mu, mv);
}

}  // namespace mortar
