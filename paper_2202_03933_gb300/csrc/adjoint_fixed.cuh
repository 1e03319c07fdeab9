// Reverse sweep of the quadrature points of one cell in fixed point.
//
// With the monomial form of the pair's functional (k_adjoint.cu),
//   f = -m_s^T CY m_m [+ m_s^T SX m_s / 2],
// a point needs u = CY^T m_s, v = CY m_m [and SX m_s], the parameter adjoints
//   b_s = df/dxi_s, b_m = df/dxi_m,   y = J^-T b on both sides,
// and adds W y (x) (1, xi, eta, xi eta) to the map-coefficient adjoints, the
// l1, l2 moments of W y to the cell's vertices, and w f to its area.
//
// Scales.  The pair's forms mix quantities of different size: CY's first
// column holds the multipliers times the mean position (as large as the
// coordinates), the others the multipliers times the element's extent, and its
// first row the mean multiplier.  Each part has its own power of two, set from
// sums of absolute entries so that the sums it enters stay below 1/2:
//   s11: CY[i][j], i, j >= 1;  sv: CY[i][0], i >= 1, v and b_s;
//   s1: CY[0][j], u and b_m;   s0: CY[0][0] and f.
// y is held as y 2^-ky in the pair's frame, with 2^ky a bound of the inverse
// Jacobian over the element; on stretched elements, where one component is
// smaller than the other by the aspect and W y (the fewest bits of the sweep) would
// lose as many of it, times 2^l with a shift of its own for each component, from a
// bound of that component over the pair (bound_y).
#pragma once

#include "quadrature.cuh"

namespace mortar {

// Words of the adjoint's record beyond FxRecord's (which keep their places):
// 45 + i: CY[i][0], 49 + 3 i + j: CY[i][j + 1] (digits, j < 3); 61, 103: scales;
// 62..: the clip record (pool vertices u, v, t; 12 each, then meta, polygon,
// counts); 104..: SX (digits, segment D).  The cell kernel leaves its results
// in the places of what it has read: G 0..15, slave map adjoint 16..23, master
// map adjoint 24..31, vertices 45 + 2 k (nr of them), H 104..119.
struct AdjRecord {
  static constexpr int kC0 = 45, kC1 = 49, kScales = 61, kPool = 62, kScales2 = 103, kSX = 104;
  static constexpr int kWords = 104, kWordsSeg = 120;
  static constexpr int kG = 0, kMapS = 16, kMapM = 24, kVertex = 45, kH = 104;
};

// Lower bound of a bilinear map's |determinant| over the element (xi to 1.01),
// in units of 2^-60 of the frame: it is linear in xi and eta.
__device__ __forceinline__ float fx_smallest_det(const FxMap& m) {
  const float d = fabsf(m.f1u * m.f2v - m.f2u * m.f1v), d1 = fabsf(m.f1u * m.f3v - m.f3u * m.f1v),
              d2 = fabsf(m.f3u * m.f2v - m.f2u * m.f3v);
  const float dmin = d - 1.01f * (d1 + d2);
  return dmin > 1e-3f * d ? dmin : 0.0f;   // 0: nearly singular somewhere
}

// 2^ky above |J^-T b| for |b| <= 1/2, in the frame (99: nearly singular somewhere in the element).
__device__ __forceinline__ int fx_inverse_exponent(const FxMap& m) {
  if (m.affine) return m.kb;
  const float a = fmaxf(fmaxf(fabsf(m.f1u), fabsf(m.f1v)), fmaxf(fabsf(m.f2u), fabsf(m.f2v))) +
                  fmaxf(fabsf(m.f3u), fabsf(m.f3v));
  const float dmin = fx_smallest_det(m);
  if (!(dmin > 0.0f)) return 99;
  return max(0, (int)(__float_as_uint(a / dmin) >> 23) - 126 + 30);   // f in units of 2^-30
}

// Pairs whose frame is stretched by more than 2^kMaxStretch = 2^|Eu - Ev| take
// the FP64 path: the smaller component of the master's y is smaller by about as
// much, either because its b is (the forms' resolution is 2^-62 of their scale)
// or, on sheared elements, by cancellation.  From a stretch of 2^2 on, its bound
// is used to hold it at full width.  Errors of the master's map adjoints relative
// to their largest (400 random pairs, geometric mean; here, FP64), aspects 1, 16,
// 100: parallelograms along the axes 1.8e-16, 1.4e-16, 2.3e-16 (2.5e-16, 2.3e-16,
// 2.1e-16), sheared ones 2.3e-16, 5.7e-16, 2.5e-15 (3.1e-16, 6.3e-16, 2.1e-15),
// distorted quads 6e-17, 1.3e-16, 7e-16 (1.4e-14).
constexpr int kMaxStretch = 7;

// Exponents: of the pair's forms (a Q62 value c stands for c 2^s), of y, and
// the shifts su, sv that bring the fan's edges to full width; and of a cell's
// sums (an integer stands for integer 2^x).
struct AdjScale {
  int s0, sv, s1, s11, kys, kym, eu, ev;
  unsigned l;                   // shifts of y of slave u, v, master u, v, in 8 bits each
  int xsu, xsv, xmu, xmv;       // W y of slave, master
  int xau, xav;   // half the area adjoint times an edge's u (v) component: (Q61 x Q62) / 2^64
  int xvu, xvv;   // common scale of the vertex adjoints' u and v components
  __device__ __forceinline__ long long word1() const {
    return (long long)((unsigned long long)(unsigned short)s0 | (unsigned long long)(unsigned short)sv << 16 |
                       (unsigned long long)(unsigned short)s1 << 32 | (unsigned long long)(unsigned short)s11 << 48);
  }
  __device__ __forceinline__ long long word2() const {
    return (long long)((unsigned long long)(unsigned)(kys | kym << 8 | eu << 16 | ev << 24) |
                       (unsigned long long)l << 32);
  }
  __device__ __forceinline__ int shift(int k) const { return (int)(l >> (8 * k) & 0xffu); }
  __device__ __forceinline__ void load(long long w1, long long w2, int ke, int Eu, int Ev) {
    s0 = (int)(short)w1;
    sv = (int)(short)(w1 >> 16);
    s1 = (int)(short)(w1 >> 32);
    s11 = (int)(short)(w1 >> 48);
    kys = (int)w2 & 0xff;
    kym = (int)(w2 >> 8) & 0xff;
    eu = (int)(w2 >> 16) & 0xff;
    ev = (int)(w2 >> 24) & 0xff;
    l = (unsigned)((unsigned long long)w2 >> 32);
    const int ku = ke - 5 - Eu, kv = ke - 5 - Ev;   // weights are 4 omega w
    xsu = ku + kys + sv - shift(0);
    xsv = kv + kys + sv - shift(1);
    xmu = ku + kym + s1 - shift(2);
    xmv = kv + kym + s1 - shift(3);
    xau = s0 + Eu - 60 - eu;
    xav = s0 + Ev - 60 - ev;
    xvu = max(xsu, max(xmu, xav)) + 2;   // the u adjoint takes the area times v components
    xvv = max(xsv, max(xmv, xau)) + 2;
  }
  __device__ __forceinline__ int xs(int c) const { return c == 0 ? xsu : xsv; }
  __device__ __forceinline__ int xm(int c) const { return c == 0 ? xmu : xmv; }
  // From the forms C (and, SEG, S) and the element maps, in a frame of
  // 2^stretch = 2^(Eu - Ev).  False if the forms leave the FP32 range that the
  // bounds are formed in, or a map is nearly singular or stretched too far.
  template <int NS, int NM, bool SEG>
  __device__ __forceinline__ bool set(const double C[4][4], const double S[4][4], const FxMap& sm, const FxMap& mm,
                                      int stretch) {
    float all = 0.0f, col = 0.0f, row = 0.0f, in_row = 0.0f, in_col[4] = {0.0f, 0.0f, 0.0f, 0.0f}, cols[4], rows[4];
    rows[3] = cols[3] = 0.0f;
    unsigned long long any = 0;   // of the forms' bits but the sign
#pragma unroll
    for (int j = 0; j < NM; ++j) cols[j] = 0.0f;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      float r = 0.0f, rin = 0.0f;
#pragma unroll
      for (int j = 0; j < NM; ++j) {
        const float c = fabsf(f32_trunc(C[i][j]));
        any |= (unsigned long long)__double_as_longlong(C[i][j]) << 1;
        r += c;
        cols[j] += c;
        if (i > 0 && j > 0) { rin += c; in_col[j] += c; }
      }
      if (SEG)
#pragma unroll
        for (int j = 0; j < NS; ++j) {
          r += fabsf(f32_trunc(S[i][j]));
          any |= (unsigned long long)__double_as_longlong(S[i][j]) << 1;
        }
      all += r;
      rows[i] = r;
      if (i > 0) { row = fmaxf(row, r); in_row = fmaxf(in_row, rin); }
    }
#pragma unroll
    for (int j = 1; j < NM; ++j) { col = fmaxf(col, cols[j]); in_row = fmaxf(in_row, in_col[j]); }
    auto ex = [](float v) { return (int)(__float_as_uint(v) >> 23) - 126; };   // v < 2^ex
    s11 = ex(in_row) + 1;
    sv = max(ex(row) + 2, s11);
    s1 = max(ex(col) + 2, s11);
    s0 = max(ex(all) + 1, max(sv, s1));
    if (!(all < 1e37f && (all > 1e-30f || any == 0))) return false;   // no multipliers at all: zero forms
    kys = fx_inverse_exponent(sm);
    kym = fx_inverse_exponent(mm);
    if (kys >= 20 || kym >= 20 || abs(stretch) > kMaxStretch) return false;
    l = 0;
    if (abs(stretch) >= 2) {   // |b| is at most the row's (column's) sum, that of xi eta added to both
      l = bound_y(sm, kys, rows[1] + rows[3], rows[2] + rows[3], sv);
      l |= bound_y(mm, kym, cols[1] + cols[3], cols[2] + cols[3], s1) << 16;
    }
    return true;
  }
  // Shifts (8 bits each) that bring y = J^-T b up to 2^59 (of 2^61: the high digits
  // of W y then add at most 2^59 to a cross sum of seven products in
  // fx_cell_moments, whose low digits take 7 2^60), from bounds of |b|.
  static __device__ __forceinline__ unsigned bound_y(const FxMap& m, int ky, float b0, float b1, int s) {
    float p[2], q[2];   // |y_c| <= p[c] |b_0| + q[c] |b_1|, in units of 2^ky
    if (m.affine) {
      p[0] = fabsf((float)m.k1u.h) * 0x1p-29f; q[0] = fabsf((float)m.k2u.h) * 0x1p-29f;
      p[1] = fabsf((float)m.k1v.h) * 0x1p-29f; q[1] = fabsf((float)m.k2v.h) * 0x1p-29f;
    } else {
      const float a3u = fabsf(m.f3u), a3v = fabsf(m.f3v);
      const float i = __uint_as_float((unsigned)(127 + 30 - ky) << 23) / fx_smallest_det(m);
      p[0] = (fabsf(m.f2v) + a3v) * i; q[0] = (fabsf(m.f1v) + a3v) * i;
      p[1] = (fabsf(m.f2u) + a3u) * i; q[1] = (fabsf(m.f1u) + a3u) * i;
    }
    unsigned l = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float y = 1.02f * (p[c] * b0 + q[c] * b1);                 // 1.02: parameters up to 1.01, FP32 sums
      const int e = (int)(__float_as_uint(y) >> 23) - 126 - s;         // y < 2^(e + s)
      l |= (unsigned)min(max(-e - 2, 0), 20) << (8 * c);
    }
    return l;
  }
};

// v 2^-k, rounded
__device__ __forceinline__ long long fx_down(long long v, int k) {
  k = min(max(k, 1), 62);
  return ((v >> (k - 1)) + 1) >> 1;
}

// y = J^-T b 2^-ky (Q61) at xi, eta (digits of Q61), b in Q62.  Affine: B'^T b.  Bilinear: FP32 inverse Jacobian at xi, then two
// refinements with the residual b - J^T y in fixed point (each gains the FP32
// inverse's 20 bits).  False if |y| leaves the range or a
// refinement did not settle.
template <int NEN>
__device__ __forceinline__ bool fx_pull_back(const FxMap& m, int ky, Dg x, Dg y, long long b0, long long b1,
                                             long long& y0, long long& y1) {
  FxAcc a;
  if (NEN == 3 || m.affine) {
    const Dg p = fx_split(b0), q = fx_split(b1);
    a.mul(m.k1u, p);
    a.mac(m.k2u, q);
    y0 = a.get<2>();
    a.mul(m.k1v, p);
    a.mac(m.k2v, q);
    y1 = a.get<2>();
    return true;
  }
  a.mul(m.k3u, y);
  const Dg j00 = fx_split(m.c1u + a.get<3>());
  a.mul(m.k3v, y);
  const Dg j10 = fx_split(m.c1v + a.get<3>());
  a.mul(m.k3u, x);
  const long long c2u = ((long long)m.k2u.h << 32) + m.k2u.l, c2v = ((long long)m.k2v.h << 32) + m.k2v.l;
  const Dg j01 = fx_split(c2u + a.get<3>());
  a.mul(m.k3v, x);
  const Dg j11 = fx_split(c2v + a.get<3>());
  const float f00 = (float)j00.h, f01 = (float)j01.h, f10 = (float)j10.h, f11 = (float)j11.h;   // units of 2^-30
  const float id = rcp_f32(f00 * f11 - f01 * f10);
  const float sc = __uint_as_float((unsigned)(127 - ky) << 23);
  const float g00 = f11 * id * sc, g01 = -f01 * id * sc, g10 = -f10 * id * sc, g11 = f00 * id * sc;
  float r0 = (float)(int)(b0 >> 32), r1 = (float)(int)(b1 >> 32);   // b 2^30
  float d0 = fmaf(g00, r0, g10 * r1), d1 = fmaf(g01, r0, g11 * r1);   // y 2^-ky
  if (!(fmaxf(fabsf(d0), fabsf(d1)) < 1.9f)) return false;
  const int h0 = __float2int_rn(d0 * 0x1p29f), h1 = __float2int_rn(d1 * 0x1p29f);
  // first residual: y has no low digit yet
  a.hh = mad_wide(j00.h, h0, mul_wide(j10.h, h1));
  a.cr = mad_wide(j00.l, h0, mul_wide(j10.l, h1));
  const long long q0 = b0 - a.get(3 + ky);
  a.hh = mad_wide(j01.h, h0, mul_wide(j11.h, h1));
  a.cr = mad_wide(j01.l, h0, mul_wide(j11.l, h1));
  const long long q1 = b1 - a.get(3 + ky);
  r0 = (float)(int)(q0 >> 16);   // 2^46
  r1 = (float)(int)(q1 >> 16);
  d0 = fmaf(g00, r0, g10 * r1);   // y 2^-ky 2^16
  d1 = fmaf(g01, r0, g11 * r1);
  y0 = ((long long)h0 << 32) + ((long long)__float2int_rn(d0 * 0x1p33f) << 12);
  y1 = ((long long)h1 << 32) + ((long long)__float2int_rn(d1 * 0x1p33f) << 12);
  const Dg p = fx_split(y0), q = fx_split(y1);
  a.mul(j00, p);
  a.mac(j10, q);
  a.low(j00, p);
  a.low(j10, q);
  const long long t0 = b0 - a.get(3 + ky);   // 2^62
  a.mul(j01, p);
  a.mac(j11, q);
  a.low(j01, p);
  a.low(j11, q);
  const long long t1 = b1 - a.get(3 + ky);
  if (t0 != (int)t0 || t1 != (int)t1) return false;
  r0 = (float)(int)t0;
  r1 = (float)(int)t1;
  y0 += __float2int_rn(fmaf(g00, r0, g10 * r1) * 0x1p29f);   // y 2^-ky 2^32
  y1 += __float2int_rn(fmaf(g01, r0, g11 * r1) * 0x1p29f);
  return true;
}

// One cell's sums.  W y of each side: the plain sum, and with xi, eta, xi eta;
// and the l1, l2 moments.
struct AdjSums {
  long long s1[2], m1[2];
  FxAcc sx[3][2], mx[3][2];
  long long es1[2], es2[2], em1[2], em2[2];
};

// The reverse sweep over the points of one cell: W y of slave u, v, master u, v
// into pts[(28 + 4 q + 0..3) * stride], and area = sum w f (Q61 at 2^s0).
// o: the record (word w at o[32 w]); pts: back-projections.  False if an
// inverse Jacobian leaves its range.
template <int NS, int NM, bool SEG, int stride>
__device__ __forceinline__ bool fx_cell_sweep(const FxMap& sm, const FxMap& mm, const AdjScale& sc,
                                              const long long* __restrict__ o, long long weight,
                                              long long* __restrict__ pts, long long& area) {
  constexpr int KS = NS, KM = NM;
  auto dg = [&](int w) { const long long v = o[32 * w]; return Dg{(int)(v >> 32), (int)v}; };
  auto val = [](Dg d) { return ((long long)d.h << 32) + d.l; };
  auto c1 = [&](int i, int j) { return dg(AdjRecord::kC1 + 3 * i + j - 1); };   // j >= 1
  area = 0;
  const Dg om = fx_split(weight);
  const int d0v = min(sc.s0 - sc.sv, 63), d01 = min(sc.s0 - sc.s1, 63);
  const int dv = min(sc.sv - sc.s11, 63), d1 = min(sc.s1 - sc.s11, 63);
  bool ok = true;
#pragma unroll 1
  for (int q = 0; q < 7; ++q) {
    FxAcc a;
    const Dg x1 = fx_split(pts[(4 * q) * stride]), x2 = fx_split(pts[(4 * q + 1) * stride]);
    const Dg z1 = fx_split(pts[(4 * q + 2) * stride]), z2 = fx_split(pts[(4 * q + 3) * stride]);
    a.mul(x1, x2);
    const Dg x12 = fx_split(a.get<3>());
    a.mul(z1, z2);
    const Dg z12 = fx_split(a.get<3>());
    // u_j = (CY^T m_s)_j, j >= 1; f = -(u_0 + sum_j u_j m_m[j])
    long long u[4];
#pragma unroll
    for (int j = 1; j < KM; ++j) {
      a.mul(c1(1, j), x1);
      a.mac(c1(2, j), x2);
      if (KS == 4) a.mac(c1(3, j), x12);
      u[j] = val(c1(0, j)) + (a.get<3>() >> d1);
    }
    a.mul(dg(AdjRecord::kC0 + 1), x1);
    a.mac(dg(AdjRecord::kC0 + 2), x2);
    if (KS == 4) a.mac(dg(AdjRecord::kC0 + 3), x12);
    long long f = -(val(dg(AdjRecord::kC0)) + (a.get<3>() >> d0v));
    a.mul(fx_split(u[1]), z1);
    a.mac(fx_split(u[2]), z2);
    if (KM == 4) a.mac(fx_split(u[3]), z12);
    f -= a.get<3>() >> d01;
    // g_i = -(CY m_m)_i [+ (SX m_s)_i], i >= 1
    long long g[4];
#pragma unroll
    for (int i = 1; i < KS; ++i) {
      a.mul(c1(i, 1), z1);
      a.mac(c1(i, 2), z2);
      if (KM == 4) a.mac(c1(i, 3), z12);
      g[i] = -(val(dg(AdjRecord::kC0 + i)) + (a.get<3>() >> dv));
    }
    if (SEG) {
      FxAcc h;   // m_s^T SX m_s
      long long w0 = 0;
#pragma unroll
      for (int i = 0; i < KS; ++i) {
        const int k = AdjRecord::kSX + 4 * i;
        a.mul(dg(k + 1), x1);
        a.mac(dg(k + 2), x2);
        if (KS == 4) a.mac(dg(k + 3), x12);
        const long long t = val(dg(k)) + a.get<3>();
        if (i == 0) w0 = t;
        else {
          g[i] += t;
          if (i == 1) h.mul(fx_split(t), x1);
          else h.mac(fx_split(t), i == 2 ? x2 : x12);
        }
      }
      f += (w0 + (h.get<3>() >> d0v)) >> 1;
    }
    a.mul(kTri7Fx.w[q], fx_split(f));
    area += a.get<1>();
    long long bs0, bs1, bm0, bm1;
    if (KS == 4) {
      const Dg g3 = fx_split(g[3]);
      a.mul(g3, x2);
      bs0 = g[1] + a.get<3>();
      a.mul(g3, x1);
      bs1 = g[2] + a.get<3>();
    } else {
      bs0 = g[1];
      bs1 = g[2];
    }
    if (KM == 4) {
      const Dg u3 = fx_split(u[3]);
      a.mul(u3, z2);
      bm0 = -(u[1] + a.get<3>());
      a.mul(u3, z1);
      bm1 = -(u[2] + a.get<3>());
    } else {
      bm0 = -u[1];
      bm1 = -u[2];
    }
    long long y[4];   // J^-T b: slave u, v, master u, v
    ok &= fx_pull_back<NS>(sm, sc.kys, x1, x2, bs0, bs1, y[0], y[1]);
    ok &= fx_pull_back<NM>(mm, sc.kym, z1, z2, bm0, bm1, y[2], y[3]);
    if (sc.l != 0u)   // stretched frames
#pragma unroll
      for (int k = 0; k < 4; ++k) y[k] <<= sc.shift(k);
    a.mul(om, kTri7Fx.w[q]);
    const Dg W = fx_split(a.get<4>());   // 4 omega w < 2^60
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const Dg yd = fx_split(y[k]);
      a.mul(W, yd);
      a.low(W, yd);
      a.cr += 1ll << 28;   // rounded: these are the smallest integers of the sweep
      pts[(28 + 4 * q + k) * stride] = a.get<3>();
    }
  }
  return ok;
}

// The cell's sums over the points' W y.  A loop of its own: the sweep holds the
// element maps, this one the accumulators.
template <int NS, int NM, int stride>
__device__ __forceinline__ void fx_cell_moments(const long long* __restrict__ pts, AdjSums& r) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    r.s1[k] = r.m1[k] = r.es1[k] = r.es2[k] = r.em1[k] = r.em2[k] = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) { r.sx[i][k].zero(); r.mx[i][k].zero(); }
  }
  // per orbit: sums over its points, and the points where l2, l1 are b
  long long os[4], o1[4], o2[4];
#pragma unroll 1
  for (int q = 0; q < 7; ++q) {
    FxAcc a;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const Dg x1 = fx_split(pts[(4 * q + 2 * side) * stride]), x2 = fx_split(pts[(4 * q + 2 * side + 1) * stride]);
      a.mul(x1, x2);
      const Dg x12 = fx_split(a.get<3>());
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int k = 2 * side + c;
        const long long y = pts[(28 + 4 * q + k) * stride];
        const Dg d = fx_split(y);
        FxAcc(&m)[3][2] = side == 0 ? r.sx : r.mx;
        (side == 0 ? r.s1 : r.m1)[c] += y;
        m[0][c].mac(d, x1);
        m[1][c].mac(d, x2);
        if ((side == 0 ? NS : NM) == 4) m[2][c].mac(d, x12);
        // moments with l1, l2: (1/3, 1/3), and per orbit (a, b), (b, a), (a, a)
        os[k] = q == 0 || q == 1 || q == 4 ? y : os[k] + y;
        if (q == 1 || q == 4) o2[k] = y;
        if (q == 2 || q == 5) o1[k] = y;
      }
    }
    if (q == 0 || q == 3 || q == 6) {
      const int n = (q + 2) / 3;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        a.mul(kOrbitFx.a[n], fx_split(os[k]));
        const long long t = a.get<2>();
        long long t1 = t, t2 = t;
        if (n > 0) {
          a.mul(kOrbitFx.d[n], fx_split(o1[k]));
          t1 += a.get<2>();
          a.mul(kOrbitFx.d[n], fx_split(o2[k]));
          t2 += a.get<2>();
        }
        const int c = k & 1;
        if (k < 2) { r.es1[c] += t1; r.es2[c] += t2; } else { r.em1[c] += t1; r.em2[c] += t2; }
      }
    }
  }
}

}  // namespace mortar
