// Pieces of the pair geometry shared by the pair kernels (forward, adjoint of
// the weighted gap, linearisation of D and M): the Sutherland-Hodgman clip
// with its stages recorded (Sec. 2.3, Algorithm 1: master polygon clipped by
// the slave window in the slave element's auxiliary plane), the reverse sweep
// through the clip and merge, and the reverse of the projection onto the
// auxiliary plane (x0, n0, t1, t2 as functions of the slave nodes).  The
// forward decisions are the ones clip_polygon takes, so every kernel agrees on
// which pairs contribute.
#pragma once

#include "clip.cuh"

namespace mortar {

constexpr int kPolyA = 10;   // vertex cap per recorded clipping stage (convex polygons need <= 8)

struct V3 {
  double x, y, z;
};
__device__ __forceinline__ V3 v3(double x, double y, double z) { return {x, y, z}; }
__device__ __forceinline__ V3 operator+(V3 a, V3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 operator-(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 operator*(double s, V3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ V3 cross(V3 a, V3 b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

template <int NEN>
__device__ __forceinline__ void shape_grad(double xi, double eta, double dN[4][2]) {
  if constexpr (NEN == 4) {
    dN[0][0] = -0.25 * (1.0 - eta); dN[0][1] = -0.25 * (1.0 - xi);
    dN[1][0] = 0.25 * (1.0 - eta);  dN[1][1] = -0.25 * (1.0 + xi);
    dN[2][0] = 0.25 * (1.0 + eta);  dN[2][1] = 0.25 * (1.0 + xi);
    dN[3][0] = -0.25 * (1.0 + eta); dN[3][1] = 0.25 * (1.0 - xi);
  } else {
    dN[0][0] = -1.0; dN[0][1] = -1.0;
    dN[1][0] = 1.0;  dN[1][1] = 0.0;
    dN[2][0] = 0.0;  dN[2][1] = 1.0;
    dN[3][0] = 0.0;  dN[3][1] = 0.0;
  }
}

// Element quadrature point k (same rule as the precomputation).
template <int NEN>
__device__ __forceinline__ void elem_point_a(int k, double& xi, double& eta, double& w) {
  if constexpr (NEN == 4) {
    const double g = 0.7745966692414834;
    const double pp[3] = {-g, 0.0, g};
    const double ww[3] = {5.0 / 9.0, 8.0 / 9.0, 5.0 / 9.0};
    xi = pp[k / 3];
    eta = pp[k % 3];
    w = ww[k / 3] * ww[k % 3];
  } else {
    tri7_point(k, xi, eta, w);
    w *= 0.5;
  }
}

// Map-coefficient adjoint (c0u c0v c1u c1v c2u c2v c3u c3v) -> in-plane node adjoints.
template <int NEN>
__device__ __forceinline__ void map_coeff_reverse(const double* cb, double* pbu, double* pbv) {
  if constexpr (NEN == 4) {
    for (int c = 0; c < 2; ++c) {   // corners (-1,-1), (1,-1), (1,1), (-1,1): sums and differences shared
      double* pb = c == 0 ? pbu : pbv;
      const double s0 = 0.25 * cb[c], s1 = 0.25 * cb[2 + c], s2 = 0.25 * cb[4 + c], s3 = 0.25 * cb[6 + c];
      const double a = s0 - s2, b = s1 - s3, d = s0 + s2, e = s1 + s3;
      pb[0] += a - b;
      pb[1] += a + b;
      pb[2] += d + e;
      pb[3] += d - e;
    }
  } else {
    pbu[0] += cb[0] - cb[2] - cb[4];
    pbv[0] += cb[1] - cb[3] - cb[5];
    pbu[1] += cb[2]; pbv[1] += cb[3];
    pbu[2] += cb[4]; pbv[2] += cb[5];
  }
}

// Clip of one pair with every stage recorded, and its reverse.
template <int NS>
struct ClipRec {
  double Vu[NS + 1][kPolyA], Vv[NS + 1][kPolyA], tt[NS][kPolyA];
  int8_t src[NS][kPolyA];   // output vertex o of stage i: input edge k; +64 if an intersection
  int nv[NS + 1];
  int last = 0, nl = 0, nr = 0;
  int sel[kPolyA];          // merged polygon: vertices of the last stage

  // Master polygon (in-plane coordinates, reversed to CCW if mrev) clipped by
  // the slave window of record r, then merged.  Returns true for a non-empty
  // polygon (same decisions as clip_polygon).
  template <int NM>
  __device__ __forceinline__ bool run(const double* __restrict__ r, const double* mu, const double* mv, bool mrev,
                                      unsigned long long& clip_over) {
    const double eps_in = r[SR_EPSIN];
    const long long eps_bits = __double_as_longlong(eps_in >= 0.0 ? eps_in : 0.0);
    for (int k = 0; k < NM; ++k) {
      const int l = mrev ? NM - 1 - k : k;
      Vu[0][k] = mu[l];
      Vv[0][k] = mv[l];
    }
    nv[0] = NM;
    last = 0;
    for (int i = 0; i < NS; ++i) {
      const int n = nv[i];
      if (n == 0) break;
      const int i1 = i + 1 == NS ? 0 : i + 1;
      const double au = r[SR_PS + 2 * i], av = r[SR_PS + 2 * i + 1];
      const double eu = r[SR_PS + 2 * i1] - au, ev = r[SR_PS + 2 * i1 + 1] - av;
      double d[kPolyA];
      int side[kPolyA];
      for (int k = 0; k < n; ++k) {
        d[k] = cross2(eu, ev, Vu[i][k] - au, Vv[i][k] - av);
        side[k] = band_side(d[k], eps_bits);
      }
      int o = 0;
      for (int k = 0; k < n; ++k) {
        const int k1 = k + 1 == n ? 0 : k + 1;
        const double dp = d[k], dq = d[k1];
        const int sp = side[k], sq = side[k1];
        if ((sp == 1 && sq == -1) || (sp == -1 && sq == 1)) {   // dp, dq beyond the band on both sides
          const double t = dp / (dp - dq);
          if (o < kPolyA) {
            Vu[i + 1][o] = Vu[i][k] + t * (Vu[i][k1] - Vu[i][k]);
            Vv[i + 1][o] = Vv[i][k] + t * (Vv[i][k1] - Vv[i][k]);
            tt[i][o] = t;
            src[i][o] = (int8_t)(k + 64);
          }
          ++o;
        }
        if (sq == 0 || sq == 1) {   // dq >= -eps_in
          if (o < kPolyA) {
            Vu[i + 1][o] = Vu[i][k1];
            Vv[i + 1][o] = Vv[i][k1];
            src[i][o] = (int8_t)k;
          }
          ++o;
        }
      }
      if (o > kPolyA) { clip_over++; o = kPolyA; }
      nv[i + 1] = o;
      last = i + 1;
    }
    // merge consecutive (cyclic) vertices closer than eps_merge: a selection
    const double em2 = r[SR_EPSM2];
    nr = 0;
    nl = nv[last];
    const bool clipped = last == NS;
    for (int k = 0; clipped && k < nl; ++k) {
      if (nr > 0) {
        const double du = Vu[last][k] - Vu[last][sel[nr - 1]], dv = Vv[last][k] - Vv[last][sel[nr - 1]];
        if (du * du + dv * dv < em2) continue;
      }
      sel[nr++] = k;
    }
    while (nr > 1) {
      const double du = Vu[last][sel[nr - 1]] - Vu[last][sel[0]], dv = Vv[last][sel[nr - 1]] - Vv[last][sel[0]];
      if (du * du + dv * dv < em2) --nr; else break;
    }
    double pa2 = 0.0;
    for (int k = 0; k < nr; ++k) {
      const int k1 = k + 1 == nr ? 0 : k + 1;
      pa2 += cross2(Vu[last][sel[k]], Vv[last][sel[k]], Vu[last][sel[k1]], Vv[last][sel[k1]]);
    }
    return eps_in >= 0.0 && clipped && nr >= 3 && !(0.5 * fabs(pa2) < r[SR_EPSA]);
  }

  __device__ __forceinline__ double pu(int k) const { return Vu[last][sel[k]]; }
  __device__ __forceinline__ double pv(int k) const { return Vv[last][sel[k]]; }

  // Reverse of merge and clip: adjoints (Rbu, Rbv) of the nr merged vertices
  // are ADDED to the in-plane adjoints of the slave nodes (sbu, sbv; element
  // node order) and of the master nodes (mbu, mbv).
  template <int NM>
  __device__ __forceinline__ void reverse(const double* __restrict__ r, const double* Rbu, const double* Rbv,
                                          bool srev, bool mrev, double* sbu, double* sbv, double* mbu,
                                          double* mbv) const {
    double Bu[NS + 1][kPolyA], Bv[NS + 1][kPolyA];
    for (int k = 0; k < nl; ++k) { Bu[last][k] = 0.0; Bv[last][k] = 0.0; }
    for (int k = 0; k < nr; ++k) { Bu[last][sel[k]] += Rbu[k]; Bv[last][sel[k]] += Rbv[k]; }
    double Wbu[4] = {0, 0, 0, 0}, Wbv[4] = {0, 0, 0, 0};
    for (int i = NS - 1; i >= 0; --i) {
      const int n = nv[i];
      const int i1 = i + 1 == NS ? 0 : i + 1;
      const double au = r[SR_PS + 2 * i], av = r[SR_PS + 2 * i + 1];
      const double eu = r[SR_PS + 2 * i1] - au, ev = r[SR_PS + 2 * i1 + 1] - av;
      for (int k = 0; k < n; ++k) { Bu[i][k] = 0.0; Bv[i][k] = 0.0; }
      double abu2 = 0.0, abv2 = 0.0, ebu = 0.0, ebv = 0.0;
      for (int o = 0; o < nv[i + 1]; ++o) {
        const double gbu = Bu[i + 1][o], gbv = Bv[i + 1][o];
        const int code = src[i][o];
        const int k = code & 63;
        const int k1 = k + 1 == n ? 0 : k + 1;
        if (code < 64) {   // copied vertex
          Bu[i][k1] += gbu;
          Bv[i][k1] += gbv;
          continue;
        }
        // intersection x = p + t (q - p), t = d_p / (d_p - d_q),
        // d = eu (y_v - a_v) - ev (y_u - a_u) for y = p, q
        const double tk = tt[i][o];
        const double pu_ = Vu[i][k], pv_ = Vv[i][k], qu = Vu[i][k1], qv = Vv[i][k1];
        Bu[i][k] += (1.0 - tk) * gbu; Bv[i][k] += (1.0 - tk) * gbv;
        Bu[i][k1] += tk * gbu;        Bv[i][k1] += tk * gbv;
        const double tb = gbu * (qu - pu_) + gbv * (qv - pv_);
        const double dp = cross2(eu, ev, pu_ - au, pv_ - av);
        const double dq = cross2(eu, ev, qu - au, qv - av);
        const double den = dp - dq;
        const double i2 = 1.0 / (den * den);
        const double dpb = -tb * dq * i2, dqb = tb * dp * i2;
        Bu[i][k] += -ev * dpb;  Bv[i][k] += eu * dpb;
        Bu[i][k1] += -ev * dqb; Bv[i][k1] += eu * dqb;
        abu2 += ev * (dpb + dqb);
        abv2 += -eu * (dpb + dqb);
        ebu += (pv_ - av) * dpb + (qv - av) * dqb;
        ebv += -(pu_ - au) * dpb - (qu - au) * dqb;
      }
      Wbu[i] += abu2 - ebu; Wbv[i] += abv2 - ebv;
      Wbu[i1] += ebu;       Wbv[i1] += ebv;
    }
    for (int k = 0; k < NS; ++k) {
      const int a = srev ? NS - 1 - k : k;
      sbu[a] += Wbu[k];
      sbv[a] += Wbv[k];
    }
    for (int k = 0; k < NM; ++k) {
      const int l = mrev ? NM - 1 - k : k;
      mbu[l] += Bu[0][k];
      mbv[l] += Bv[0][k];
    }
  }
};

// Orientation of the projected master polygon: true if clockwise.  In FP32
// where the area is above 1e-4 of its terms.
template <int NM>
__device__ __forceinline__ bool polygon_reversed(const double* mu, const double* mv) {
  float u[4], v[4], a = 0.0f, s = 0.0f;
#pragma unroll
  for (int l = 0; l < NM; ++l) { u[l] = f32_trunc(mu[l]); v[l] = f32_trunc(mv[l]); }
#pragma unroll
  for (int l = 0; l < NM; ++l) {
    const float x = u[l] * v[(l + 1) % NM], y = v[l] * u[(l + 1) % NM];
    a += x - y;
    s += fabsf(x) + fabsf(y);
  }
  if (fabsf(a) > 1e-4f * s && s < 1e37f && fabsf(a) > 1e-30f) return a < 0.0f;
  double ma2 = 0.0;
#pragma unroll
  for (int l = 0; l < NM; ++l) ma2 += cross2(mu[l], mv[l], mu[(l + 1) % NM], mv[(l + 1) % NM]);
  return ma2 < 0.0;
}

// Compact clip record: the same Sutherland-Hodgman clip and merge as
// ClipRec (identical decisions, quotients to an ulp), recorded as a pool of
// vertices instead of whole stages.  Pool slots [0, NM) are the master
// polygon's vertices (counter-clockwise), every later slot is an edge
// intersection x = p + t (q - p) made at stage i from pool slots p and q; a
// copied vertex keeps its slot.  The working polygon of a stage is a list of
// 4-bit slot ids packed into 64 bits.  Reverse: slots are visited from the
// last intersection down, so that each slot's adjoint is complete before it
// is passed on to its two parents and to the clip edge.
template <int NS, int NM>
struct ClipPool {
  static constexpr int kSlots = 12;   // master vertices + intersections (convex quads: <= 4 + 8)
  double pu[kSlots], pv[kSlots], tt[kSlots];
  uint16_t meta[kSlots];              // intersection: p | q << 4 | stage << 8
  int nv = 0, nr = 0;
  uint64_t poly = 0;                  // merged polygon: slot ids, 4 bits each

  bool over = false;                  // more vertices than fit: the pair is not decided

  __device__ __forceinline__ int id(int k) const { return (int)((poly >> (4 * k)) & 15); }
  __device__ __forceinline__ double u(int k) const { return pu[id(k)]; }
  __device__ __forceinline__ double v(int k) const { return pv[id(k)]; }

  // Vertices a and b closer than eps_merge?  In FP32 where that settles it (the
  // distance is above 1e-5 of the coordinates and well above eps_merge).
  __device__ __forceinline__ bool close(int a, int b, double em2) const {
    const float ua = f32_trunc(pu[a]), va = f32_trunc(pv[a]), ub = f32_trunc(pu[b]), vb = f32_trunc(pv[b]);
    const float d = fabsf(ua - ub) + fabsf(va - vb);
    const float e = f32_trunc(em2);   // 0: none, or below FP32's range
    if (e > 0.0f && d > 1e-5f * (fabsf(ua) + fabsf(va) + fabsf(ub) + fabsf(vb)) && 0.25f * d * d > e) return false;
    const double du = pu[a] - pu[b], dv = pv[a] - pv[b];
    return du * du + dv * dv < em2;
  }

  // FP64 work: the distances to the window's edges, and per edge two rounds of
  // intersections (a lane's crossings are found first and computed together, so
  // that a warp runs as many rounds as its lane with the most crossings has).
  __device__ __forceinline__ bool run(const double* __restrict__ r, const double* mu, const double* mv, bool mrev,
                                      unsigned long long& clip_over) {
    const double eps_in = r[SR_EPSIN];
    const long long eps_bits = __double_as_longlong(eps_in >= 0.0 ? eps_in : 0.0);
    uint64_t cur = 0;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      const int l = mrev ? NM - 1 - k : k;
      pu[k] = mu[l];
      pv[k] = mv[l];
      cur |= (uint64_t)k << (4 * k);
    }
    nv = NM;
    int n = NM;
    over = false;
    for (int i = 0; i < NS && n > 0; ++i) {
      const int i1 = i + 1 == NS ? 0 : i + 1;
      const double au = r[SR_PS + 2 * i], av = r[SR_PS + 2 * i + 1];
      const double eu = r[SR_PS + 2 * i1] - au, ev = r[SR_PS + 2 * i1 + 1] - av;
      double d[16];                            // of the vertices of cur
      unsigned in = 0, pos = 0, neg = 0;       // dq >= -eps_in; beyond the band on either side
      for (int k = 0; k < n; ++k) {
        const int id = (int)((cur >> (4 * k)) & 15);
        d[k] = cross2(eu, ev, pu[id] - au, pv[id] - av);
        const int s = band_side(d[k], eps_bits);
        pos |= (s == 1 ? 1u : 0u) << k;
        neg |= (s == -1 ? 1u : 0u) << k;
        in |= (s == 0 || s == 1 ? 1u : 0u) << k;
      }
      // bit k: of the edge's end k + 1
      const unsigned in1 = in >> 1 | (in & 1u) << (n - 1), pos1 = pos >> 1 | (pos & 1u) << (n - 1);
      const unsigned neg1 = neg >> 1 | (neg & 1u) << (n - 1);
      const unsigned cross = (pos & neg1) | (neg & pos1);
      if (nv + __popc(cross) > kSlots || __popc(cross) + __popc(in) > 16) {
        over = true;
        break;
      }
      int w = nv;
      for (unsigned c = cross; c != 0u; c &= c - 1u) {
        const int k = __ffs(c) - 1, k1 = k + 1 == n ? 0 : k + 1;
        const int idp = (int)((cur >> (4 * k)) & 15), idq = (int)((cur >> (4 * k1)) & 15);
        const double dp = d[k], t = quotient(dp, dp - d[k1]);
        pu[w] = pu[idp] + t * (pu[idq] - pu[idp]);
        pv[w] = pv[idp] + t * (pv[idq] - pv[idp]);
        tt[w] = t;
        meta[w] = (uint16_t)(idp | (idq << 4) | (i << 8));
        ++w;
      }
      uint64_t nxt = 0;
      int o = 0;
      for (int k = 0; k < n; ++k) {
        if (cross >> k & 1u) {
          nxt |= (uint64_t)nv << (4 * o);
          ++nv;
          ++o;
        }
        if (in1 >> k & 1u) {
          nxt |= ((cur >> (k + 1 == n ? 0 : 4 * (k + 1))) & 15) << (4 * o);
          ++o;
        }
      }
      cur = nxt;
      n = o;
    }
    if (over) {   // cannot happen for convex elements; reported, pair dropped
      clip_over++;
      nr = 0;
      return false;
    }
    // merge consecutive (cyclic) vertices closer than eps_merge: a selection
    const double em2 = r[SR_EPSM2];
    nr = 0;
    poly = 0;
    int last_id = -1, first_id = -1;
    for (int k = 0; k < n; ++k) {
      const int q = (int)((cur >> (4 * k)) & 15);
      if (nr > 0) {
        if (close(q, last_id, em2)) continue;
      } else {
        first_id = q;
      }
      poly |= (uint64_t)q << (4 * nr);
      last_id = q;
      ++nr;
    }
    while (nr > 1 && close(id(nr - 1), first_id, em2)) {
      --nr;
      poly &= ~((uint64_t)15 << (4 * nr));
    }
    if (!(eps_in >= 0.0 && nr >= 3)) return false;
    // area above the threshold?  In FP32 where that settles it
    float fa = 0.0f, fs = 0.0f;
    for (int k = 0; k < nr; ++k) {
      const int a = id(k), b = id(k + 1 == nr ? 0 : k + 1);
      const float x = f32_trunc(pu[a]) * f32_trunc(pv[b]), y = f32_trunc(pv[a]) * f32_trunc(pu[b]);
      fa += x - y;
      fs += fabsf(x) + fabsf(y);
    }
    const float ea = f32_trunc(r[SR_EPSA]);   // 0: none, or below FP32's range
    if (ea > 0.0f && fabsf(fa) > 1e-4f * fs && 0.25f * fabsf(fa) > ea) return true;
    double pa2 = 0.0;
    for (int k = 0; k < nr; ++k) {
      const int a = id(k), b = id(k + 1 == nr ? 0 : k + 1);
      pa2 += cross2(pu[a], pv[a], pu[b], pv[b]);
    }
    return !(0.5 * fabs(pa2) < r[SR_EPSA]);
  }

  // Reverse of merge and clip.  Bu, Bv (kSlots, caller-owned) hold on entry
  // the adjoints of the merged polygon's vertices ADDED at their slots (all
  // other slots zero); the in-plane adjoints of the slave window vertices
  // (element node order) and of the master nodes are ADDED to sbu, sbv, mbu, mbv.
  __device__ __forceinline__ void reverse(const double* __restrict__ r, double* Bu, double* Bv, bool srev,
                                          bool mrev, double* sbu, double* sbv, double* mbu, double* mbv) const {
    double Wbu[NS], Wbv[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) { Wbu[k] = 0.0; Wbv[k] = 0.0; }
    for (int w = nv - 1; w >= NM; --w) {
      const double gbu = Bu[w], gbv = Bv[w];
      const int p = meta[w] & 15, q = (meta[w] >> 4) & 15, i = meta[w] >> 8;
      const int i1 = i + 1 == NS ? 0 : i + 1;
      const double au = r[SR_PS + 2 * i], av = r[SR_PS + 2 * i + 1];
      const double eu = r[SR_PS + 2 * i1] - au, ev = r[SR_PS + 2 * i1 + 1] - av;
      // intersection x = p + t (q - p), t = d_p / (d_p - d_q),
      // d = eu (y_v - a_v) - ev (y_u - a_u) for y = p, q; with
      // s = tb / (d_p - d_q): adjoints of d_p and d_q are (1 - t) s and t s, and
      // those of the edge combine to s (x - a)
      const double tk = tt[w], omt = 1.0 - tk;
      const double qpu = pu[q] - pu[p], qpv = pv[q] - pv[p];
      const double tb = gbu * qpu + gbv * qpv;
      const double sb = tb * rcp_newton(ev * qpu - eu * qpv);
      const double gu = gbu - ev * sb, gv = gbv + eu * sb;
      Bu[p] += omt * gu;
      Bv[p] += omt * gv;
      Bu[q] += tk * gu;
      Bv[q] += tk * gv;
      const double abu2 = ev * sb, abv2 = -eu * sb;
      const double ebu = (pv[w] - av) * sb;
      const double ebv = -(pu[w] - au) * sb;
#pragma unroll
      for (int s = 0; s < NS; ++s) {   // window vertices i and i + 1 (registers, no indexed array)
        const int s1 = s + 1 == NS ? 0 : s + 1;
        if (s == i) {
          Wbu[s] += abu2 - ebu;
          Wbv[s] += abv2 - ebv;
          Wbu[s1] += ebu;
          Wbv[s1] += ebv;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const int a = srev ? NS - 1 - k : k;
      sbu[a] += Wbu[k];
      sbv[a] += Wbv[k];
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      const int l = mrev ? NM - 1 - k : k;
      mbu[l] += Bu[k];
      mbv[l] += Bv[k];
    }
  }
};

// clip_polygon's stages as they stand (clip.cuh), for polygons beyond the pool.
template <int NS, int NM, int CAP>
__device__ __noinline__ int clip_polygon_large(const double* __restrict__ r, const double* __restrict__ xm,
                                               const int32_t* __restrict__ conn_m, int32_t m, PlaneMap& mmap,
                                               double* Pu, double* Pv, unsigned long long& clip_over) {
  return clip_polygon<NS, NM, CAP>(r, xm, conn_m, m, mmap, Pu, Pv, clip_over);
}

// clip_polygon by way of the pool: the same projection, stages and decisions.
// Bound by the FP64 pipe; the pool's moves are packed slot ids instead of
// coordinates, a warp computes two intersections per window edge instead of one
// at every vertex, and merge distances, areas and orientation go to FP64 only
// where FP32 leaves them open.  k_pair_clip at 1000x866 (3.5 M pairs) 3.29 ->
// 2.78 ms, the adjoint's finish kernel on 128 batched interfaces (1.9 M pairs),
// with the shorter reverse of an intersection, 1.30 -> 1.10 ms.
template <int NS, int NM, int CAP>
__device__ __forceinline__ int clip_polygon_pool(const double* __restrict__ r, const double* __restrict__ xm,
                                                 const int32_t* __restrict__ conn_m, int32_t m, PlaneMap& mmap,
                                                 double* Pu, double* Pv, unsigned long long& clip_over) {
  if (!(r[SR_EPSIN] >= 0.0)) return 0;
  double mu[4], mv[4];
  project_master<NM>(r, xm, conn_m + (int64_t)NM * m, mu, mv);
  mmap = plane_map<NM>(mu, mv);
  ClipPool<NS, NM> cp;
  unsigned long long over = 0;
  if (!cp.run(r, mu, mv, polygon_reversed<NM>(mu, mv), over))
    return over == 0 ? 0 : clip_polygon_large<NS, NM, CAP>(r, xm, conn_m, m, mmap, Pu, Pv, clip_over);
  if (cp.nr > CAP) {   // cannot happen for convex elements; reported, pair dropped
    clip_over++;
    return 0;
  }
  for (int k = 0; k < cp.nr; ++k) { Pu[k] = cp.u(k); Pv[k] = cp.v(k); }
  return cp.nr;
}

// Adjoints of the auxiliary plane: point x0 and in-plane basis t1, t2.
struct PlaneBar {
  V3 x0, t1, t2;
};

// Reverse of the projection u = (P - x0).t1, v = (P - x0).t2 of N nodes P:
// in-plane adjoints (bu, bv) in; 3D coordinate adjoints ADDED to g, the plane's
// to pb.
template <int N>
__device__ __forceinline__ void project_reverse(const V3* P, V3 x0, V3 t1, V3 t2, const double* bu, const double* bv,
                                                double g[4][3], PlaneBar& pb) {
  for (int l = 0; l < N; ++l) {
    const V3 dd = P[l] - x0;
    const V3 db = bu[l] * t1 + bv[l] * t2;
    g[l][0] += db.x; g[l][1] += db.y; g[l][2] += db.z;
    pb.x0 = pb.x0 - db;
    pb.t1 = pb.t1 + bu[l] * dd;
    pb.t2 = pb.t2 + bv[l] * dd;
  }
}

// Reverse of the auxiliary plane (x0 = element centre, n0 = unit normal there,
// t1 = normalised projected first edge, t2 = n0 x t1) as a function of the slave
// nodes X: what several reverse sweeps of one element share (the square roots
// and divisions), and one sweep, ADDED to gX.
template <int NS>
struct PlaneBasis {
  V3 t1, t2, n0, g1, g2, ed;
  double iln, ile, en;
  __device__ __forceinline__ PlaneBasis(const V3* X, V3 t1_, V3 t2_, V3 n0_) : t1(t1_), t2(t2_), n0(n0_) {
    if constexpr (NS == 4) {
      g1 = 0.25 * ((X[1] - X[0]) + (X[2] - X[3]));
      g2 = 0.25 * ((X[2] - X[1]) + (X[3] - X[0]));
    } else {
      g1 = X[1] - X[0];
      g2 = X[2] - X[0];
    }
    const V3 nn = cross(g1, g2);
    iln = 1.0 / sqrt(dot(nn, nn));
    ed = X[1] - X[0];
    en = dot(ed, n0);
    const V3 ep = ed - en * n0;
    ile = 1.0 / sqrt(dot(ep, ep));
  }
  __device__ __forceinline__ void reverse(const PlaneBar& pb, double gX[4][3]) const {
    const V3 x0b = pb.x0, t2b = pb.t2;
    V3 t1b = pb.t1;
    V3 n0b = cross(t1, t2b);   // t2 = n0 x t1
    t1b = t1b + cross(t2b, n0);
    const V3 epb = ile * (t1b - dot(t1, t1b) * t1);
    V3 edb = epb;
    const double enb = -dot(epb, n0);
    n0b = n0b - en * epb;
    edb = edb + enb * n0;
    n0b = n0b + enb * ed;
    const V3 nb = iln * (n0b - dot(n0, n0b) * n0);
    const V3 g1b = cross(g2, nb), g2b = cross(nb, g1);
    V3 Xb[4];
    for (int a = 0; a < 4; ++a) Xb[a] = v3(0, 0, 0);
    Xb[1] = Xb[1] + edb;
    Xb[0] = Xb[0] - edb;
    if constexpr (NS == 4) {
      const V3 a1 = 0.25 * g1b, a2 = 0.25 * g2b, ax = 0.25 * x0b;
      Xb[0] = Xb[0] - a1 - a2 + ax;
      Xb[1] = Xb[1] + a1 - a2 + ax;
      Xb[2] = Xb[2] + a1 + a2 + ax;
      Xb[3] = Xb[3] - a1 + a2 + ax;
    } else {
      const V3 ax = (1.0 / 3.0) * x0b;
      Xb[0] = Xb[0] - g1b - g2b + ax;
      Xb[1] = Xb[1] + g1b + ax;
      Xb[2] = Xb[2] + g2b + ax;
    }
    for (int a = 0; a < NS; ++a) {
      gX[a][0] += Xb[a].x; gX[a][1] += Xb[a].y; gX[a][2] += Xb[a].z;
    }
  }
};

template <int NS>
__device__ __forceinline__ void plane_basis_reverse(const V3* X, V3 t1, V3 t2, V3 n0, const PlaneBar& pb,
                                                    double gX[4][3]) {
  PlaneBasis<NS>(X, t1, t2, n0).reverse(pb, gX);
}

// Monomial form of the element shape functions, N(xi) = T m(xi): quad4
// m = (1, xi, eta, xi eta) and row a of T is (1, xi_a, eta_a, xi_a eta_a) / 4
// with the corners (xi_a, eta_a) = (-1,-1), (1,-1), (1,1), (-1,1); tri3
// m = (1, xi, eta) and N = (1 - xi - eta, xi, eta).  A bilinear form
// N_s^T P N_m of nodal quantities equals m_s^T (T_s^T P T_m) m_m, which a
// quadrature point evaluates without forming N.

// out_i = sum_a T[a][i] in_a: monomial coefficients of the nodal field `in`.
template <int NEN, class T>
__device__ __forceinline__ void nodal_to_mono(const T* in, T* out) {
  if constexpr (NEN == 4) {
    const T s02 = in[0] + in[2], s13 = in[1] + in[3], d20 = in[2] - in[0], d13 = in[1] - in[3];
    out[0] = 0.25 * (s02 + s13);
    out[1] = 0.25 * (d20 + d13);
    out[2] = 0.25 * (d20 - d13);
    out[3] = 0.25 * (s02 - s13);
  } else {
    out[0] = in[0];
    out[1] = in[1] - in[0];
    out[2] = in[2] - in[0];
  }
}

}  // namespace mortar
