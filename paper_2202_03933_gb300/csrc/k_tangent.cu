// Linearisation of the mortar coupling terms (Sec. 1: the consistent
// linearisation of D and M enters every nonlinear iteration):
//     K = d/dX [ (D (x) I3) ys - (M (x) I3) ym ],   ys, ym held fixed,
// a block-sparse matrix of 3x3 blocks: block rows = slave nodes, block
// columns = slave nodes, then master nodes.
//
// Per pair (s, m), in the standard basis N_e of the slave element,
//     O_e,c = sum over quadrature points of W N_e(xi_s) Z_c,
//     Z_c   = [segment D] sum_b N_b(xi_s) ys_b,c - sum_l N_l(xi_m) ym_l,c,
// and the pair's rows are sum_e A[a][e] O_e,c (A = I for standard LMs).
// Three lanes own one pair, one component c each, and run the reverse sweep
// of the four outputs together: each lane computes every third quadrature
// point's back-projections and shares them with the other two through shared
// memory, the per-point adjoints of the four seeds are accumulated side by
// side (their map-coefficient adjoints in shared memory), and only the reverse
// of the clip and of the projection runs once per seed.  The seeds are the
// monomials 1, x, y, x y (triangles: 1, x, y) in coordinates of the slave element
// that are zero at its corner nearest to the pair's polygon and one at that
// corner's neighbours (Corner), of which the N_e are combinations: a seed's
// point adjoint is then a product or two, and the slave map's adjoints of all
// four follow from 12 moments.  Seen from that corner, N_e that are small all
// over the pair are small seeds themselves or differences in which nothing
// cancels, so that a row that is small keeps its digits: with a pair of 1 % of
// the element's size at a corner, the far node's row has errors up to 3.2e-13 of
// itself, as with the N_e as seeds, and 2.9e-12 with monomials about the centre.
// Bound by the FP64 pipe (about 75 % busy); 300x260 quads, dual (0.31 M pairs):
// 21.8 ms with the N_e as seeds, 18.9 ms this way (18.7 about the centre), square
// roots and divisions of the plane once per pair.
//
// The derivatives through A (dual LMs) and of the element-domain D depend on
// the slave element alone: a per-element kernel pushes the pair sums of O and
// the D term through A = Dh Me^-1 and the element integrals in forward mode
// over the 12 slave coordinates.  Rows are gathered per slave node in a fixed
// order into BSR with no floating-point atomics: bitwise reproducible.
#include <algorithm>

#include "clip.cuh"
#include "context.h"
#include "reverse.cuh"

namespace mortar {

namespace {

constexpr int kTanWarps = 4;
constexpr int kTanThreads = 32 * kTanWarps;
constexpr int kThreads = 128;

struct TanArgs {
  const int32_t* ps;
  const int32_t* pm;
  const double* srec;
  const double* xs;
  const double* xm;
  const int32_t* conn_s;
  const int32_t* conn_m;
  const double* ys;
  const double* ym;
  double* Kp;          // per pair 288: [a][c][k][d], k < 4 slave node, k >= 4 master node k - 4
  double* Op;          // per pair 12: O_e,c (dual LMs)
  const uint8_t* flag; // per pair: non-empty in the forward run (FP64 clip)
  int64_t pair_cap;
  DevStatus* st;
  int32_t watchdog_us;
};

// Corner of a slave element, and the coordinates (x, y) about it: quad4
// x = (1 -+ xi) / 2, y = (1 -+ eta) / 2; tri3 the barycentric coordinates of the
// two other corners.
template <int NS>
struct Corner {
  bool rx = false, ry = false;   // quad4: at xi = 1, at eta = 1
  int k = 0;                     // tri3: corner

  __device__ __forceinline__ Corner(double xi, double eta) {
    if constexpr (NS == 4) {
      rx = xi > 0.0;
      ry = eta > 0.0;
    } else {
      const double n0 = 1.0 - xi - eta;
      k = xi > n0 ? (eta > xi ? 2 : 1) : (eta > n0 ? 2 : 0);
    }
  }
  __device__ __forceinline__ void coordinates(double xi, double eta, double& x, double& y) const {
    if constexpr (NS == 4) {
      x = 0.5 * (rx ? 1.0 - xi : 1.0 + xi);
      y = 0.5 * (ry ? 1.0 - eta : 1.0 + eta);
    } else {
      const double n0 = 1.0 - xi - eta;
      x = k == 0 ? xi : (k == 1 ? eta : n0);
      y = k == 0 ? eta : (k == 1 ? n0 : xi);
    }
  }
  // rows of the inverse Jacobian of (xi, eta) to those of (x, y)
  __device__ __forceinline__ void rows(double* a) const {
    if constexpr (NS == 4) {
      const double f = rx ? -0.5 : 0.5, g = ry ? -0.5 : 0.5;
      a[0] *= f; a[1] *= f; a[2] *= g; a[3] *= g;
    } else {
      const double b0 = -a[0] - a[2], b1 = -a[1] - a[3];
      const double x0 = k == 0 ? a[0] : (k == 1 ? a[2] : b0), x1 = k == 0 ? a[1] : (k == 1 ? a[3] : b1);
      const double y0 = k == 0 ? a[2] : (k == 1 ? b0 : a[0]), y1 = k == 0 ? a[3] : (k == 1 ? b1 : a[1]);
      a[0] = x0; a[1] = x1; a[2] = y0; a[3] = y1;
    }
  }
  // values at the corner, its neighbours in x and y and (quad4) the opposite corner <-> in node order
  __device__ __forceinline__ void to_nodes(double c, double x, double y, double o, double* n) const {
    if constexpr (NS == 4) {
      const double p = rx ? x : c, q = rx ? c : x, r = rx ? o : y, t = rx ? y : o;   // xi = -1, 1; then the far eta's
      n[0] = ry ? r : p; n[1] = ry ? t : q; n[2] = ry ? q : t; n[3] = ry ? p : r;
    } else {
      n[0] = k == 0 ? c : (k == 1 ? y : x);
      n[1] = k == 0 ? x : (k == 1 ? c : y);
      n[2] = k == 0 ? y : (k == 1 ? x : c);
      n[3] = 0.0;
    }
  }
  // N_e of the seeds' values f: rows, and (transposed coefficients) the nodes' adjoints of a map's coefficients
  __device__ __forceinline__ void nodal(const double* f, double* n) const {
    if constexpr (NS == 4) {
      const double x = f[1] - f[3], y = f[2] - f[3];
      to_nodes((f[0] - f[1]) - y, x, y, f[3], n);
    } else {
      to_nodes(f[0] - f[1] - f[2], f[1], f[2], 0.0, n);
    }
  }
  // coefficients in the seeds of the field with nodal values n
  __device__ __forceinline__ void coefficients(const double* n, double* f) const {
    if constexpr (NS == 4) {
      const double p = ry ? n[3] : n[0], q = ry ? n[2] : n[1], r = ry ? n[0] : n[3], t = ry ? n[1] : n[2];
      const double c = rx ? q : p, x = rx ? p : q, y = rx ? t : r, o = rx ? r : t;
      f[0] = c;
      f[1] = x - c;
      f[2] = y - c;
      f[3] = (c - x) + (o - y);
    } else {
      const double c = k == 0 ? n[0] : (k == 1 ? n[1] : n[2]);
      f[0] = c;
      f[1] = (k == 0 ? n[1] : (k == 1 ? n[2] : n[0])) - c;
      f[2] = (k == 0 ? n[2] : (k == 1 ? n[0] : n[1])) - c;
      f[3] = 0.0;
    }
  }
};

// Quadrature-point data one lane computes and the other two lanes of its
// pair group read (shared memory), what does not depend on the component:
// the seeds, the master's back-projection and its product, and W J_s^-1 (rows of
// the corner's coordinates), -W J_m^-1.
struct GPX {
  double s1, s2, s12, m1, m2, m12;
  double a[4], b[4];
  double s11, s22, s122, s112;
};

// One value in the basis (1, xi, eta, xi eta) of an element
template <int NEN>
__device__ __forceinline__ double mono_value(const double* y, double x1, double x2, double x12) {
  const double v = fma(y[2], x2, fma(y[1], x1, y[0]));
  return NEN == 4 ? fma(y[3], x12, v) : v;
}
template <int NEN>
__device__ __forceinline__ void mono_grad(const double* y, double x1, double x2, double& g0, double& g1) {
  g0 = NEN == 4 ? fma(y[3], x2, y[1]) : y[1];
  g1 = NEN == 4 ? fma(y[3], x1, y[2]) : y[2];
}

// Accumulators of a thread (shared memory).  Slave side, element D: moments of
// su_1, su_2 = W J_s^-T e_1, e_2 times Z, with (1, x, y, x y) and, on quad4,
// (y^2, x y^2) for su_1, (x^2, x^2 y) for su_2, from which the map adjoints of
// all seeds follow (grad x y = y e_1 + x e_2); segment D: the map adjoints
// themselves.  Then the master map adjoints.
template <int NS, bool SEG>
constexpr int kSlaveSums = SEG ? 8 * NS : (NS == 4 ? 24 : 12);
template <int NS, int NM, bool SEG>
constexpr int kTanSums = kSlaveSums<NS, SEG> + (NM == 4 ? 8 : 6) * NS;
// the sums of every thread, then 32 exchange slots per warp
template <int NS, int NM, bool SEG>
constexpr size_t kTanSmem = sizeof(double) * kTanSums<NS, NM, SEG> * kTanThreads + sizeof(GPX) * kTanThreads;

// Pair p, component cp, for the lanes of one pair group (lanes 3g, 3g + 1,
// 3g + 2 hold components 0, 1, 2 of the same pair).  Every lane of the warp
// calls this with the same control flow around the exchanges: lanes with
// live = false (no pair) take part in the loops and exchanges without work.
// acc: this thread's shared-memory accumulators, entry i at acc[i * kTanThreads];
// gx: the warp's 32 exchange slots.
template <int NS, int NM, bool SEG, bool DUAL>
__device__ void tangent_pair(const TanArgs& g, int64_t p, int cp, bool live, double* __restrict__ acc,
                             GPX* __restrict__ gx, unsigned long long& clip_over, unsigned long long& newton_fail) {
  const int lane = threadIdx.x & 31;
  const int32_t s = g.ps[p], m = g.pm[p];
  const double* r = g.srec + (int64_t)SR_STRIDE * s;
  const int32_t* cs = g.conn_s + (int64_t)NS * s;
  const int32_t* cm = g.conn_m + (int64_t)NM * m;
  double yS[4] = {0, 0, 0, 0}, yM[4] = {0, 0, 0, 0};
  {   // monomial coefficients of the held field
    double y[4] = {0, 0, 0, 0};
    for (int l = 0; l < NM; ++l) y[l] = g.ym[3 * (int64_t)cm[l] + cp];
    nodal_to_mono<NM>(y, yM);
  }
  const V3 x0 = v3(r[SR_X0], r[SR_X0 + 1], r[SR_X0 + 2]);
  const V3 t1 = v3(r[SR_T1], r[SR_T1 + 1], r[SR_T1 + 2]);
  const V3 t2 = v3(r[SR_T2], r[SR_T2 + 1], r[SR_T2 + 2]);
  double mu[4], mv[4];
  for (int l = 0; l < NM; ++l) {
    const int64_t n = cm[l];
    const double dx = g.xm[3 * n] - x0.x, dy = g.xm[3 * n + 1] - x0.y, dz = g.xm[3 * n + 2] - x0.z;
    mu[l] = dx * t1.x + dy * t1.y + dz * t1.z;
    mv[l] = dx * t2.x + dy * t2.y + dz * t2.z;
  }
  const PlaneMap mmap = plane_map<NM>(mu, mv);
  PlaneMap smap;
  smap.c0u = r[SR_C + 0]; smap.c0v = r[SR_C + 1]; smap.c1u = r[SR_C + 2]; smap.c1v = r[SR_C + 3];
  smap.c2u = r[SR_C + 4]; smap.c2v = r[SR_C + 5]; smap.c3u = r[SR_C + 6]; smap.c3v = r[SR_C + 7];
  const bool mrev = polygon_reversed<NM>(mu, mv);
  const bool srev = r[SR_REV] != 0.0;
  ClipPool<NS, NM> clip;   // compact record: master corners + intersections
  unsigned long long clip_dummy = 0;
  const bool nonempty = clip.run(r, mu, mv, mrev, live ? clip_over : clip_dummy);
  // row a at + 72 a; written with streaming (evict-first) stores, so that L2
  // keeps the threads' stack lines rather than these write-once blocks
  double* kout = g.Kp + 288 * p + 24 * cp;
  const int nr = nonempty ? clip.nr : 0;
  MapInverse mi;
  mi.setup(mmap, NM == 3 || map_is_affine(mmap));
  MapInverse si;
  if (r[SR_AFF] != 0.0) {
    si.m = smap;
    si.affine = true;
    si.i00 = r[SR_BINV]; si.i01 = r[SR_BINV + 1]; si.i10 = r[SR_BINV + 2]; si.i11 = r[SR_BINV + 3];
  } else {
    si.setup(smap, false);
  }
  // per-seed adjoints of the polygon vertices, kept at the vertices' pool slots
  constexpr int kSlots = ClipPool<NS, NM>::kSlots;
  double Rbu[4][kSlots], Rbv[4][kSlots];
  for (int k = 0; k < clip.nv; ++k)
    for (int e = 0; e < NS; ++e) { Rbu[e][k] = 0.0; Rbv[e][k] = 0.0; }
  double cu = 0.0, cv = 0.0;
  int ncell = nr >= 3 ? 1 : 0;
  if (nr > 3) {
    double su = 0.0, sv = 0.0;
    for (int k = 0; k < nr; ++k) { su += clip.u(k); sv += clip.v(k); }
    cu = su * kInvCount[nr];
    cv = sv * kInvCount[nr];
    ncell = nr;
  }
  const Corner<NS> corner = [&] {   // nearest to the polygon's vertex mean (distorted elements: by the map's linear part)
    double u = cu - smap.c0u, v = cv - smap.c0v;
    if (nr == 3) {
      u = (1.0 / 3.0) * (clip.u(0) + clip.u(1) + clip.u(2)) - smap.c0u;
      v = (1.0 / 3.0) * (clip.v(0) + clip.v(1) + clip.v(2)) - smap.c0v;
    }
    const float fu = f32_trunc(u) * si.scf, fv = f32_trunc(v) * si.scf;
    return si.affine ? Corner<NS>(si.i00 * u + si.i01 * v, si.i10 * u + si.i11 * v)
                     : Corner<NS>(f64_of_f32(si.b00 * fu + si.b01 * fv), f64_of_f32(si.b10 * fu + si.b11 * fv));
  }();
  if (SEG) {
    double y[4] = {0, 0, 0, 0};
    for (int a = 0; a < NS; ++a) y[a] = g.ys[3 * (int64_t)cs[a] + cp];
    corner.coefficients(y, yS);
  }
  if (!live) ncell = 0;
  constexpr int KS = kSlaveSums<NS, SEG>, KM = NM == 4 ? 8 : 6;   // master sums per seed
  for (int i = 0; i < KS + KM * NS; ++i) acc[i * kTanThreads] = 0.0;
  double O[4] = {0, 0, 0, 0}, cbu[4] = {0, 0, 0, 0}, cbv[4] = {0, 0, 0, 0};
  const int ncell_w = __reduce_max_sync(0xffffffffu, ncell);
  const int gbase = 3 * (lane / 3);
  for (int cI = 0; cI < ncell_w; ++cI) {
    const bool cell_ok = cI < ncell;
    int ib = 0, iw = 0;   // pool slots of the cell's two polygon vertices
    double au = 0.0, av = 0.0;
    if (cell_ok) {
      if (nr == 3) {
        au = clip.u(0); av = clip.v(0); ib = clip.id(1); iw = clip.id(2);
      } else {
        au = cu; av = cv; ib = clip.id(cI); iw = clip.id(cI + 1 == nr ? 0 : cI + 1);
      }
    }
    const double e1u = cell_ok ? clip.pu[ib] - au : 0.0, e1v = cell_ok ? clip.pv[ib] - av : 0.0;
    const double e2u = cell_ok ? clip.pu[iw] - au : 0.0, e2v = cell_ok ? clip.pv[iw] - av : 0.0;
    const double crs = cross2(e1u, e1v, e2u, e2v);
    const double area = 0.5 * fabs(crs);
    double arb[4], e1bu[4], e1bv[4], e2bu[4], e2bv[4], xbu_c[4], xbv_c[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      arb[e] = 0.0; e1bu[e] = 0.0; e1bv[e] = 0.0; e2bu[e] = 0.0; e2bv[e] = 0.0; xbu_c[e] = 0.0; xbv_c[e] = 0.0;
    }
#pragma unroll 1
    for (int rr = 0; rr < 3; ++rr) {
      // this lane's quadrature point of the round (component cp computes point 3 rr + cp)
      const int qo = 3 * rr + cp;
      if (cell_ok && qo < 7) {
        double l1, l2, w;
        tri7_point(qo, l1, l2, w);
        const double W = w * area;
        const double xu = au + l1 * e1u + l2 * e2u;
        const double xv = av + l1 * e1v + l2 * e2v;
        GPX& o = gx[lane];
        double xs1, xs2, xm1, xm2, a00, a01, a10, a11;
        if (!si.solve(xu, xv, xs1, xs2)) newton_fail++;
        if (!mi.solve(xu, xv, xm1, xm2)) newton_fail++;
        double x, y;
        corner.coordinates(xs1, xs2, x, y);
        o.s1 = x; o.s2 = y; o.s12 = x * y;
        o.m1 = xm1; o.m2 = xm2; o.m12 = xm1 * xm2;
        si.jinv(xs1, xs2, a00, a01, a10, a11);
        o.a[0] = W * a00; o.a[1] = W * a01; o.a[2] = W * a10; o.a[3] = W * a11;
        corner.rows(o.a);
        mi.jinv(xm1, xm2, a00, a01, a10, a11);
        o.b[0] = -W * a00; o.b[1] = -W * a01; o.b[2] = -W * a10; o.b[3] = -W * a11;
        if (NS == 4 && !SEG) {
          o.s11 = x * x; o.s22 = y * y;
          o.s122 = o.s12 * y; o.s112 = o.s12 * x;
        }
      }
      __syncwarp();
#pragma unroll 1
      for (int jj = 0; jj < 3; ++jj) {
        const int q = 3 * rr + jj;
        if (!(cell_ok && q < 7)) continue;
        const GPX& x = gx[gbase + jj];
        double l1, l2, w;
        tri7_point(q, l1, l2, w);
        const double s1 = x.s1, s2 = x.s2, s12 = x.s12, m1 = x.m1, m2 = x.m2, m12 = x.m12;
        double Z = -mono_value<NM>(yM, m1, m2, m12);
        if (SEG) Z += mono_value<NS>(yS, s1, s2, s12);
        const double wZ = w * Z;
        arb[0] += wZ;
        arb[1] = fma(wZ, s1, arb[1]);
        arb[2] = fma(wZ, s2, arb[2]);
        if (NS == 4) arb[3] = fma(wZ, s12, arb[3]);
        // J_m^-T (adjoint of xi_m) of the seed 1
        double g0, g1;
        mono_grad<NM>(yM, m1, m2, g0, g1);
        double tu[4], tv[4], su[4], sv[4];   // master and slave point adjoints of the seeds 1, x, y, x y
        tu[0] = fma(x.b[0], g0, x.b[2] * g1);
        tv[0] = fma(x.b[1], g0, x.b[3] * g1);
        tu[1] = s1 * tu[0]; tv[1] = s1 * tv[0];
        tu[2] = s2 * tu[0]; tv[2] = s2 * tv[0];
        if (NS == 4) { tu[3] = s12 * tu[0]; tv[3] = s12 * tv[0]; }
        su[0] = 0.0; sv[0] = 0.0;
        su[1] = x.a[0] * Z; sv[1] = x.a[1] * Z;
        su[2] = x.a[2] * Z; sv[2] = x.a[3] * Z;
        if (NS == 4) {
          su[3] = fma(s2, su[1], s1 * su[2]);
          sv[3] = fma(s2, sv[1], s1 * sv[2]);
        }
        auto add = [&](int i, double f, double v) { acc[i * kTanThreads] = fma(f, v, acc[i * kTanThreads]); };
        if constexpr (SEG) {
          mono_grad<NS>(yS, s1, s2, g0, g1);
          const double gu = fma(x.a[0], g0, x.a[2] * g1), gv = fma(x.a[1], g0, x.a[3] * g1);
          su[0] = gu; sv[0] = gv;
          su[1] = fma(s1, gu, su[1]); sv[1] = fma(s1, gv, sv[1]);
          su[2] = fma(s2, gu, su[2]); sv[2] = fma(s2, gv, sv[2]);
          if (NS == 4) { su[3] = fma(s12, gu, su[3]); sv[3] = fma(s12, gv, sv[3]); }
#pragma unroll
          for (int e = 0; e < NS; ++e) {
            add(8 * e + 0, 1.0, su[e]); add(8 * e + 1, 1.0, sv[e]);
            add(8 * e + 2, s1, su[e]); add(8 * e + 3, s1, sv[e]);
            add(8 * e + 4, s2, su[e]); add(8 * e + 5, s2, sv[e]);
            if (NS == 4) { add(8 * e + 6, s12, su[e]); add(8 * e + 7, s12, sv[e]); }
          }
        } else {
#pragma unroll
          for (int e = 1; e < 3; ++e) {
            constexpr int N = NS == 4 ? 12 : 6;
            const int o = N * (e - 1);
            add(o + 0, 1.0, su[e]); add(o + 1, 1.0, sv[e]);
            add(o + 2, s1, su[e]); add(o + 3, s1, sv[e]);
            add(o + 4, s2, su[e]); add(o + 5, s2, sv[e]);
            if (NS == 4) {
              add(o + 6, s12, su[e]); add(o + 7, s12, sv[e]);
              add(o + 8, e == 1 ? x.s22 : x.s11, su[e]); add(o + 9, e == 1 ? x.s22 : x.s11, sv[e]);
              add(o + 10, e == 1 ? x.s122 : x.s112, su[e]); add(o + 11, e == 1 ? x.s122 : x.s112, sv[e]);
            }
          }
        }
#pragma unroll
        for (int e = 0; e < NS; ++e) {
          const int o = KS + KM * e;
          add(o + 0, 1.0, tu[e]); add(o + 1, 1.0, tv[e]);
          add(o + 2, m1, tu[e]); add(o + 3, m1, tv[e]);
          add(o + 4, m2, tu[e]); add(o + 5, m2, tv[e]);
          if (NM == 4) { add(o + 6, m12, tu[e]); add(o + 7, m12, tv[e]); }
          const double xbu = e == 0 && !SEG ? tu[e] : su[e] + tu[e], xbv = e == 0 && !SEG ? tv[e] : sv[e] + tv[e];
          xbu_c[e] += xbu; xbv_c[e] += xbv;
          e1bu[e] = fma(l1, xbu, e1bu[e]); e1bv[e] = fma(l1, xbv, e1bv[e]);
          e2bu[e] = fma(l2, xbu, e2bu[e]); e2bv[e] = fma(l2, xbv, e2bv[e]);
        }
      }
      __syncwarp();   // the slots are rewritten by the next three points
    }
    if (cell_ok) {
#pragma unroll
      for (int e = 0; e < NS; ++e) {   // area = |cross| / 2, cell vertices, centroid
        O[e] = fma(area, arb[e], O[e]);
        const double crb = 0.5 * (crs < 0.0 ? -arb[e] : arb[e]);
        e1bu[e] += crb * e2v; e1bv[e] -= crb * e2u;
        e2bu[e] -= crb * e1v; e2bv[e] += crb * e1u;
        Rbu[e][ib] += e1bu[e]; Rbv[e][ib] += e1bv[e];
        Rbu[e][iw] += e2bu[e]; Rbv[e][iw] += e2bv[e];
        const double abu = xbu_c[e] - (e1bu[e] + e2bu[e]), abv = xbv_c[e] - (e1bv[e] + e2bv[e]);
        if (nr == 3) {
          const int s0 = clip.id(0);
          Rbu[e][s0] += abu; Rbv[e][s0] += abv;
        } else {
          cbu[e] += abu; cbv[e] += abv;
        }
      }
    }
  }
  if (!live) return;
  if (!nonempty) {   // not reached for pairs the count pass found non-empty; blocks stay defined
    for (int a = 0; a < 4; ++a)
      for (int k = 0; k < 24; ++k) __stcs(kout + 72 * a + k, 0.0);
    if (DUAL)
      for (int e = 0; e < 4; ++e) __stcs(g.Op + 12 * p + 3 * e + cp, 0.0);
    return;
  }
  if (nr > 3) {
    const double inv = kInvCount[nr];
    for (int e = 0; e < NS; ++e)
      for (int k = 0; k < nr; ++k) {
        const int sk = clip.id(k);
        Rbu[e][sk] += cbu[e] * inv; Rbv[e][sk] += cbv[e] * inv;
      }
  }
  // ---- per seed: clip and merge, map coefficients, projection and plane;
  //      node coordinates read again here (L1/L2) rather than held through
  //      the quadrature loop
  const V3 n0 = v3(r[SR_N0], r[SR_N0 + 1], r[SR_N0 + 2]);
  V3 X[4], Y[4];
  for (int a = 0; a < NS; ++a) {
    const int64_t n = cs[a];
    X[a] = v3(g.xs[3 * n], g.xs[3 * n + 1], g.xs[3 * n + 2]);
  }
  for (int l = 0; l < NM; ++l) {
    const int64_t n = cm[l];
    Y[l] = v3(g.xm[3 * n], g.xm[3 * n + 1], g.xm[3 * n + 2]);
  }
  const PlaneBasis<NS> basis(X, t1, t2, n0);
  double Ks[NS][24];   // rows of the seeds
#pragma unroll 1
  for (int e = 0; e < NS; ++e) {
    double sbu[4] = {0, 0, 0, 0}, sbv[4] = {0, 0, 0, 0}, mbu[4] = {0, 0, 0, 0}, mbv[4] = {0, 0, 0, 0};
    clip.reverse(r, Rbu[e], Rbv[e], srev, mrev, sbu, sbv, mbu, mbv);
    double smb[8], mmb[8];   // map adjoints: minus the sums
    auto sum = [&](int i) { return acc[i * kTanThreads]; };
    for (int k = 0; k < 8; ++k) {
      const int c = k & 1;
      if constexpr (SEG) {
        smb[k] = NS == 4 || k < 6 ? -sum(8 * e + k) : 0.0;
      } else if constexpr (NS == 3) {
        smb[k] = e > 0 && k < 6 ? -sum(6 * (e - 1) + k) : 0.0;
      } else {
        if (e == 0) smb[k] = 0.0;
        else if (e < 3) smb[k] = -sum(12 * (e - 1) + k);
        else   // y su_1 + x su_2 with 1, x, y, x y
          smb[k] = -(sum((k < 2 ? 4 : (k < 4 ? 6 : (k < 6 ? 8 : 10))) + c) +
                     sum(12 + (k < 2 ? 2 : (k < 4 ? 8 : (k < 6 ? 6 : 10))) + c));
      }
      mmb[k] = k < KM ? -sum(KS + KM * e + k) : 0.0;
    }
    {
      const double cbu_e[4] = {smb[0], smb[2], smb[4], smb[6]}, cbv_e[4] = {smb[1], smb[3], smb[5], smb[7]};
      double n[4];
      corner.nodal(cbu_e, n);
      for (int a = 0; a < NS; ++a) sbu[a] += n[a];
      corner.nodal(cbv_e, n);
      for (int a = 0; a < NS; ++a) sbv[a] += n[a];
    }
    map_coeff_reverse<NM>(mmb, mbu, mbv);
    double gX[4][3], gY[4][3];
    for (int a = 0; a < 4; ++a)
      for (int d = 0; d < 3; ++d) { gX[a][d] = 0.0; gY[a][d] = 0.0; }
    PlaneBar pb{v3(0, 0, 0), v3(0, 0, 0), v3(0, 0, 0)};
    project_reverse<NS>(X, x0, t1, t2, sbu, sbv, gX, pb);
    project_reverse<NM>(Y, x0, t1, t2, mbu, mbv, gY, pb);
    basis.reverse(pb, gX);
    for (int a = 0; a < 4; ++a)
      for (int d = 0; d < 3; ++d) {
        Ks[e][3 * a + d] = gX[a][d];
        Ks[e][12 + 3 * a + d] = gY[a][d];
      }
  }
  double AT[4][4];   // dual: rows of A in the seeds
  if (DUAL)
    for (int a = 0; a < NS; ++a) {
      double v[4];
      for (int e = 0; e < NS; ++e) v[e] = r[SR_A + 4 * a + e];
      corner.coefficients(v, AT[a]);
    }
  for (int k = 0; k < 24; ++k) {
    double f[4], row[4];
    for (int e = 0; e < NS; ++e) f[e] = Ks[e][k];
    if (DUAL) {
      for (int a = 0; a < NS; ++a) {
        double v = 0.0;
        for (int e = 0; e < NS; ++e) v = fma(AT[a][e], f[e], v);
        row[a] = v;
      }
    } else {
      corner.nodal(f, row);
    }
    for (int a = 0; a < 4; ++a) __stcs(kout + 72 * a + k, a < NS ? row[a] : 0.0);
  }
  if (DUAL) {
    double On[4];
    corner.nodal(O, On);
    for (int e = 0; e < 4; ++e) __stcs(g.Op + 12 * p + 3 * e + cp, e < NS ? On[e] : 0.0);
  }
}

// Persistent kernel over warp batches of 32 R pairs, each sorted by the cell
// count and edge intersections of an FP32 clip (ballot counting sort) and
// swept in rounds of 10 pairs x 3 components.
template <int NS, int NM, bool SEG, bool DUAL, int R>
__global__ void __launch_bounds__(kTanThreads) k_tangent_pairs(TanArgs g) {
  extern __shared__ double tan_acc[];
  constexpr int B = 32 * R;
  __shared__ uint8_t perm_s[kTanWarps][B];
  __shared__ unsigned pres_s[kTanWarps][8];   // key values present in the batch (256 bits)
  uint8_t* perm = perm_s[threadIdx.x >> 5];
  unsigned* pres = pres_s[threadIdx.x >> 5];
  double* acc = tan_acc + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  unsigned long long clip_over = 0, newton_fail = 0;
  DevStatus* st = g.st;
  const bool ok = st->over_pairs == 0 && st->over_bins == 0;
  const int64_t n = ok ? (int64_t)min((unsigned long long)g.pair_cap, st->n_pairs) : 0;
  const int64_t items = (n + B - 1) / B;
  GPX* gx = reinterpret_cast<GPX*>(tan_acc + kTanSums<NS, NM, SEG> * kTanThreads) + 32 * (threadIdx.x >> 5);
  const Watchdog wd(g.watchdog_us);
  for (;;) {   // bounded: the shared counter only grows
    if (wd.expired(&st->timeout)) break;
    int64_t item = 0;
    if (lane == 0) item = (int64_t)atomicAdd(&st->work_ctr3, 1ull);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= items) break;
    const int64_t base = item * B;
    // sort key: 0 for pairs the forward run found empty (their blocks are
    // never read), else 1 + 16 x the cell count + the edge intersections of
    // an FP32 clip (a cost estimate only; the FP64 clip of the pair kernel
    // decides)
    if (lane < 8) pres[lane] = 0u;
    __syncwarp();
    int key[R];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int64_t p = base + rr * 32 + lane;
      int k = 0;
      if (p < n && g.flag[p]) {
        int n_int = 0;
        const int nr = clip_count_f32<NS, NM>(g.srec + (int64_t)SR_STRIDE * g.ps[p], g.xm, g.conn_m, g.pm[p],
                                              n_int);
        k = 1 + 16 * (nr == 0 ? 0 : (nr == 3 ? 1 : min(nr, kPolyS))) + min(n_int, 15);
        atomicOr(&pres[k >> 5], 1u << (k & 31));
      }
      key[rr] = k;
    }
    __syncwarp();
    int pos[R];
    int basecnt = 0;
#pragma unroll 1
    for (int w = 7; w >= 0; --w) {
      unsigned bits = pres[w];
      while (bits != 0u) {   // uniform across the warp
        const int b = 31 - __clz(bits);
        bits &= ~(1u << b);
        const int v = 32 * w + b;
        int before = 0;
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
          const unsigned mk = __ballot_sync(0xffffffffu, key[rr] == v);
          if (key[rr] == v) pos[rr] = basecnt + before + __popc(mk & lt_mask);
          before += __popc(mk);
        }
        basecnt += before;
      }
    }
    const int n_live = basecnt;
#pragma unroll
    for (int rr = 0; rr < R; ++rr)
      if (key[rr] > 0) perm[pos[rr]] = (uint8_t)(rr * 32 + lane);
    __syncwarp();
    // rounds of 10 pairs: lanes 3 g .. 3 g + 2 take components 0..2 of pair g
    const int grp = lane / 3, cp = lane - 3 * (lane / 3);
    for (int i0 = 0; i0 < n_live; i0 += 10) {
      const int i = i0 + grp;
      const bool live = lane < 30 && i < n_live;
      const int64_t p = base + perm[live ? i : i0];
      tangent_pair<NS, NM, SEG, DUAL>(g, p, cp, live, acc, gx, clip_over, newton_fail);
      __syncwarp();
    }
    __syncwarp();
  }
  (void)clip_over;     // both counted once already by the forward pass
  (void)newton_fail;
}

// Per slave element (forward mode over its 12 coordinates X_b,d):
//   Ke[a][c][b][d] = sum_e dA[a][e]/dX_bd S[e][c]                     (dual LMs)
//                  + sum_b' dDe[a][b']/dX_bd ys_b',c                  (element D)
// with S = sum of O over the element's non-empty pairs, A = Dh Me^-1 (so
// dA S = dDh T - A dMe T, T = Me^-1 S = Dh^-1 A S) and De = A Me (dual:
// De = Dh, dDe = dDh; standard: dDe = dMe).  Every element integral is
// sum_q w f(q) J(q), and dJ(q)/dX_bd = dN_b/dxi (g2 x n)_d + dN_b/deta (n x g1)_d,
// so Ke[a][c][b][d] = sum_q rho[a][c](q) dJ(q)/dX_bd with
//   rho[a][c] = w (N_a T[a][c] - Phi_a tau_c) + [element D] w N_a yD_a,c,
//   tau_c = sum_j N_j T[j][c], Phi_a = sum_i A[a][i] N_i,
//   yD_a,c = ys_a,c (dual) or sum_b N_b ys_b,c (standard).
template <int NS, bool DUAL, bool ELEMD>
__global__ void __launch_bounds__(kThreads) k_tangent_elems(
    const double* __restrict__ xs, const int32_t* __restrict__ conn_s, const double* __restrict__ ys,
    const double* __restrict__ srec, const int64_t* __restrict__ pair_off, const uint8_t* __restrict__ flag,
    const double* __restrict__ Op, int64_t Es, double* __restrict__ Ke, const DevStatus* st) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Es) return;
  double* out = Ke + 144 * e;
  for (int k = 0; k < 144; ++k) out[k] = 0.0;
  const double* r = srec + (int64_t)SR_STRIDE * e;
  if (r[SR_EPSIN] < 0.0 || st->over_pairs) return;
  V3 X[4];
  double yS[4][3];
  for (int a = 0; a < 4; ++a) {
    X[a] = v3(0, 0, 0);
    yS[a][0] = yS[a][1] = yS[a][2] = 0.0;
  }
  for (int a = 0; a < NS; ++a) {
    const int64_t n = conn_s[(int64_t)NS * e + a];
    X[a] = v3(xs[3 * n], xs[3 * n + 1], xs[3 * n + 2]);
    for (int c = 0; c < 3; ++c) yS[a][c] = ys[3 * n + c];
  }
  double A[4][4];
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b) A[a][b] = r[SR_A + 4 * a + b];
  constexpr int nq = NS == 4 ? 9 : 7;
  double T[4][3];
  for (int a = 0; a < 4; ++a) T[a][0] = T[a][1] = T[a][2] = 0.0;
  if (DUAL) {
    double S[4][3];
    for (int a = 0; a < 4; ++a) S[a][0] = S[a][1] = S[a][2] = 0.0;
    for (int64_t p = pair_off[e]; p < pair_off[e + 1]; ++p) {
      if (!flag[p]) continue;
      for (int a = 0; a < NS; ++a)
        for (int c = 0; c < 3; ++c) S[a][c] += Op[12 * p + 3 * a + c];
    }
    double Dh[4] = {0, 0, 0, 0};
    for (int q = 0; q < nq; ++q) {
      double xi, eta, w;
      elem_point_a<NS>(q, xi, eta, w);
      double N[4], dN[4][2];
      shape_fn<NS>(xi, eta, N);
      shape_grad<NS>(xi, eta, dN);
      V3 g1 = v3(0, 0, 0), g2 = v3(0, 0, 0);
      for (int a = 0; a < NS; ++a) { g1 = g1 + dN[a][0] * X[a]; g2 = g2 + dN[a][1] * X[a]; }
      const V3 nq3 = cross(g1, g2);
      const double wj = w * sqrt(dot(nq3, nq3));
      for (int a = 0; a < NS; ++a) Dh[a] += wj * N[a];
    }
    for (int j = 0; j < NS; ++j)
      for (int c = 0; c < 3; ++c) {
        double v = 0.0;
        for (int k = 0; k < NS; ++k) v = fma(A[j][k], S[k][c], v);
        T[j][c] = v / Dh[j];
      }
  }
  // flat element (parallelogram, every tri3): constant tangents g1, g2, so
  // dJ/dX_bd = dN_b/dxi c1_d + dN_b/deta c2_d with constant c1, c2, and the
  // point sums of rho dN_b are taken first (96 sums instead of 144 per point)
  bool flat;
  V3 g1c, g2c;
  if constexpr (NS == 4) {
    g1c = 0.25 * ((X[1] - X[0]) + (X[2] - X[3]));
    g2c = 0.25 * ((X[2] - X[1]) + (X[3] - X[0]));
    const V3 d3 = 0.25 * ((X[0] - X[1]) + (X[2] - X[3]));
    const double s3 = fabs(d3.x) + fabs(d3.y) + fabs(d3.z);
    const double s12 = fabs(g1c.x) + fabs(g1c.y) + fabs(g1c.z) + fabs(g2c.x) + fabs(g2c.y) + fabs(g2c.z);
    flat = s3 <= 1e-15 * s12;
  } else {
    g1c = X[1] - X[0];
    g2c = X[2] - X[0];
    flat = true;
  }
  if (flat) {
    const V3 ncv = cross(g1c, g2c);
    const V3 nu = (1.0 / sqrt(dot(ncv, ncv))) * ncv;
    const V3 c1 = cross(g2c, nu), c2 = cross(nu, g1c);
    const double c1d[3] = {c1.x, c1.y, c1.z}, c2d[3] = {c2.x, c2.y, c2.z};
    double P1[4][3][4], P2[4][3][4];
    for (int a = 0; a < 4; ++a)
      for (int c = 0; c < 3; ++c)
        for (int b = 0; b < 4; ++b) { P1[a][c][b] = 0.0; P2[a][c][b] = 0.0; }
    for (int q = 0; q < nq; ++q) {
      double xi, eta, w;
      elem_point_a<NS>(q, xi, eta, w);
      double N[4], dN[4][2];
      shape_fn<NS>(xi, eta, N);
      shape_grad<NS>(xi, eta, dN);
      double tau[3] = {0, 0, 0}, yq[3] = {0, 0, 0};
      for (int j = 0; j < NS; ++j)
        for (int c = 0; c < 3; ++c) {
          tau[c] = fma(N[j], T[j][c], tau[c]);
          yq[c] = fma(N[j], yS[j][c], yq[c]);
        }
      for (int a = 0; a < NS; ++a) {
        double phi = 0.0;
        for (int i = 0; i < NS; ++i) phi = fma(A[a][i], N[i], phi);
        for (int c = 0; c < 3; ++c) {
          double rho = 0.0;
          if (DUAL) rho = w * (N[a] * T[a][c] - phi * tau[c]);
          if (ELEMD) rho = fma(w * N[a], DUAL ? yS[a][c] : yq[c], rho);
          for (int b = 0; b < NS; ++b) {
            P1[a][c][b] = fma(rho, dN[b][0], P1[a][c][b]);
            P2[a][c][b] = fma(rho, dN[b][1], P2[a][c][b]);
          }
        }
      }
    }
    for (int a = 0; a < NS; ++a)
      for (int c = 0; c < 3; ++c)
        for (int b = 0; b < NS; ++b)
          for (int d = 0; d < 3; ++d)
            out[36 * a + 12 * c + 3 * b + d] = fma(P1[a][c][b], c1d[d], P2[a][c][b] * c2d[d]);
    return;
  }
  for (int q = 0; q < nq; ++q) {
    double xi, eta, w;
    elem_point_a<NS>(q, xi, eta, w);
    double N[4], dN[4][2];
    shape_fn<NS>(xi, eta, N);
    shape_grad<NS>(xi, eta, dN);
    V3 g1 = v3(0, 0, 0), g2 = v3(0, 0, 0);
    for (int a = 0; a < NS; ++a) { g1 = g1 + dN[a][0] * X[a]; g2 = g2 + dN[a][1] * X[a]; }
    const V3 nq3 = cross(g1, g2);
    const V3 nu = (1.0 / sqrt(dot(nq3, nq3))) * nq3;
    const V3 c1 = cross(g2, nu), c2 = cross(nu, g1);
    const double c1d[3] = {c1.x, c1.y, c1.z}, c2d[3] = {c2.x, c2.y, c2.z};
    double tau[3] = {0, 0, 0}, yq[3] = {0, 0, 0};
    for (int j = 0; j < NS; ++j)
      for (int c = 0; c < 3; ++c) {
        tau[c] = fma(N[j], T[j][c], tau[c]);
        yq[c] = fma(N[j], yS[j][c], yq[c]);
      }
    for (int a = 0; a < NS; ++a) {
      double phi = 0.0;
      for (int i = 0; i < NS; ++i) phi = fma(A[a][i], N[i], phi);
      for (int c = 0; c < 3; ++c) {
        double rho = 0.0;
        if (DUAL) rho = w * (N[a] * T[a][c] - phi * tau[c]);
        if (ELEMD) rho = fma(w * N[a], DUAL ? yS[a][c] : yq[c], rho);
        if (rho == 0.0) continue;
        double* o = out + 36 * a + 12 * c;
        for (int b = 0; b < NS; ++b) {
          const double u = rho * dN[b][0], v = rho * dN[b][1];
          for (int d = 0; d < 3; ++d) o[3 * b + d] = fma(u, c1d[d], fma(v, c2d[d], o[3 * b + d]));
        }
      }
    }
  }
}

// Sources of one block row j, visited in a fixed order: the slave elements
// around j (sorted), for each its non-empty pairs in (s, m) order, then the
// element block.  f(col, block pointer, row stride of the block, diagonal add).
template <int NS, int NM, bool SEG, bool DUAL, bool ELEMD>
struct TanRowSource {
  const int64_t* n2e_ptr;
  const int64_t* n2e_ent;
  const int64_t* pair_off;
  const int32_t* pm;
  const uint8_t* flag;
  const int32_t* conn_s;
  const int32_t* conn_m;
  const double* Kp;
  const double* Ke;
  const double* Mblk;
  const double* Dblk;
  const double* De;
  int64_t Ns;
  int direct;

  template <class F>
  __device__ __forceinline__ void visit(int64_t j, F&& f) const {
    for (int64_t q = n2e_ptr[j]; q < n2e_ptr[j + 1]; ++q) {
      const int64_t ee = n2e_ent[q];
      const int64_t e = ee >> 2;
      const int a = (int)(ee & 3);
      bool any = false;
      for (int64_t p = pair_off[e]; p < pair_off[e + 1]; ++p) {
        if (!flag[p]) continue;
        any = true;
        const double* kb = Kp + 288 * p + 72 * a;
        for (int k = 0; k < NS; ++k)
          f(conn_s[(int64_t)NS * e + k], kb + 3 * k, 24, (SEG && direct) ? Dblk[16 * p + 4 * a + k] : 0.0);
        const int64_t m = pm[p];
        for (int l = 0; l < NM; ++l)
          f((int32_t)(Ns + conn_m[(int64_t)NM * m + l]), kb + 12 + 3 * l, 24,
            direct ? -Mblk[16 * p + 4 * a + l] : 0.0);
      }
      if (ELEMD || (DUAL && any)) {
        const double* kb = Ke + 144 * e + 36 * a;
        for (int k = 0; k < NS; ++k)
          f(conn_s[(int64_t)NS * e + k], kb + 3 * k, 12, (ELEMD && direct) ? De[16 * e + 4 * a + k] : 0.0);
      }
    }
  }
};

// Sorted unique column ids of a row (block columns).
template <int CAP>
struct RowKeys {
  int32_t col[CAP];
  int u = 0;
  bool over = false;
  __device__ __forceinline__ void add(int32_t c) {
    int lo = 0, hi = u;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (col[mid] < c) lo = mid + 1; else hi = mid;
    }
    if (lo < u && col[lo] == c) return;
    if (u == CAP) { over = true; return; }
    for (int k = u; k > lo; --k) col[k] = col[k - 1];
    col[lo] = c;
    ++u;
  }
};

constexpr int kRowCap = 64;

// One thread per block row.  MODE 0: count the unique block columns.
// MODE 1: write them, sorted (the values follow in k_tangent_rows_warp).
template <int MODE, class Src>
__global__ void __launch_bounds__(kThreads) k_tangent_rows(Src src, int64_t N, int32_t* __restrict__ cnt,
                                                           const int64_t* __restrict__ rp, int64_t cap,
                                                           int32_t* __restrict__ col, double* __restrict__ val,
                                                           DevStatus* st) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= N) return;
  if (st->over_pairs) {
    if (MODE == 0) cnt[j] = 0;
    return;
  }
  if (MODE == 1 && rp[N] > cap) {
    if (j == 0) atomicMax(&st->over_K, 1ull);
    return;
  }
  RowKeys<kRowCap> keys;
  src.visit(j, [&](int32_t c, const double*, int, double) { keys.add(c); });
  int u = keys.u;
  const int64_t o = MODE == 1 ? rp[j] : 0;
  if (keys.over) {   // long row: repeated selection of the next column
    u = 0;
    int32_t last = -1;
    for (;;) {
      int32_t next = 0x7fffffff;
      src.visit(j, [&](int32_t c, const double*, int, double) { if (c > last && c < next) next = c; });
      if (next == 0x7fffffff) break;
      if (MODE == 1) col[o + u] = next;
      ++u;
      last = next;
    }
  } else if (MODE == 1) {
    for (int k = 0; k < u; ++k) col[o + k] = keys.col[k];
  }
  if (MODE == 0) cnt[j] = u;
  (void)val;
}

// Value pass, one warp per block row: the row's sorted columns (written by
// k_tangent_rows<1>) go to shared memory, then the row's sources are visited
// in the fixed order and each source's
// entries (72 of a pair row, 36 of an element row, contiguous in memory) are
// read by the 32 lanes together and added to the row's blocks held in shared
// memory.  Within one source no two entries share a block entry, and sources
// follow each other after a warp barrier, so every block entry is summed in
// the same order (sources in visit order).  Rows with more than kRowCap
// columns are summed by lane 0 alone in global memory, in the same order.
constexpr int kRowWarps = 4;

template <int NS, int NM, bool SEG, bool DUAL, bool ELEMD>
__global__ void __launch_bounds__(32 * kRowWarps) k_tangent_rows_warp(TanRowSource<NS, NM, SEG, DUAL, ELEMD> src,
                                                                      int64_t N, const int64_t* __restrict__ rp,
                                                                      int64_t cap, int32_t* __restrict__ col,
                                                                      double* __restrict__ val, DevStatus* st) {
  __shared__ int32_t keys_s[kRowWarps][kRowCap];
  __shared__ double acc_s[kRowWarps][kRowCap * 9];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int32_t* keys = keys_s[w];
  double* acc = acc_s[w];
  if (st->over_pairs) return;
  if (rp[N] > cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(&st->over_K, 1ull);
    return;
  }
  const int64_t nw = (int64_t)gridDim.x * kRowWarps;
  for (int64_t j = (int64_t)blockIdx.x * kRowWarps + w; j < N; j += nw) {
    const int64_t o = rp[j];
    const int u = (int)(rp[j + 1] - o);
    if (u > kRowCap) {   // long row: lane 0 accumulates in global memory, in the same order
      if (lane == 0) {
        double* vrow = val + 9 * o;
        for (int k = 0; k < 9 * u; ++k) vrow[k] = 0.0;
        const int32_t* crow = col + o;
        src.visit(j, [&](int32_t c, const double* blk, int stride, double diag) {
          int lo = 0, hi = u;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (crow[mid] < c) lo = mid + 1; else hi = mid;
          }
          double* vb = vrow + 9 * lo;
          for (int cc = 0; cc < 3; ++cc)
            for (int d = 0; d < 3; ++d) vb[3 * cc + d] += blk[stride * cc + d] + (cc == d ? diag : 0.0);
        });
      }
      __syncwarp();
      continue;
    }
    for (int k = lane; k < u; k += 32) keys[k] = col[o + k];
    for (int k = lane; k < 9 * u; k += 32) acc[k] = 0.0;
    __syncwarp();
    auto find = [&](int32_t c) {
      int lo = 0, hi = u;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (keys[mid] < c) lo = mid + 1; else hi = mid;
      }
      return lo;
    };
    for (int64_t q = src.n2e_ptr[j]; q < src.n2e_ptr[j + 1]; ++q) {
      const int64_t ee = src.n2e_ent[q];
      const int64_t e = ee >> 2;
      const int a = (int)(ee & 3);
      bool any = false;
      for (int64_t p = src.pair_off[e]; p < src.pair_off[e + 1]; ++p) {
        if (!src.flag[p]) continue;
        any = true;
        const int64_t m = src.pm[p];
        int mypos = 0;   // lanes 0..7: block position of the pair's node k = lane
        if (lane < NS) mypos = find(src.conn_s[(int64_t)NS * e + lane]);
        else if (lane >= 4 && lane < 4 + NM) mypos = find((int32_t)(src.Ns + src.conn_m[(int64_t)NM * m + lane - 4]));
        const double* kb = src.Kp + 288 * p + 72 * a;
        for (int it = 0; it < 3; ++it) {   // entries lane, lane + 32, lane + 64 (< 72)
          const int idx = lane + 32 * it;
          const int ic = idx < 72 ? idx : 0;
          const int c = ic / 24, rem = ic - 24 * c, k = rem / 3, d = rem - 3 * k;
          const int pos = __shfl_sync(0xffffffffu, mypos, k);   // every lane takes part
          const bool valid = idx < 72 && (k < NS || (k >= 4 && k - 4 < NM));
          if (!valid) continue;
          double v = kb[idx];
          if (src.direct && c == d)
            v += k < 4 ? (SEG ? src.Dblk[16 * p + 4 * a + k] : 0.0) : -src.Mblk[16 * p + 4 * a + (k - 4)];
          acc[9 * pos + 3 * c + d] += v;
        }
        __syncwarp();
      }
      if (ELEMD || (DUAL && any)) {
        int mypos = 0;
        if (lane < NS) mypos = find(src.conn_s[(int64_t)NS * e + lane]);
        const double* kb = src.Ke + 144 * e + 36 * a;
        for (int it = 0; it < 2; ++it) {   // entries lane, lane + 32 (< 36)
          const int idx = lane + 32 * it;
          const int ic = idx < 36 ? idx : 0;
          const int c = ic / 12, rem = ic - 12 * c, k = rem / 3, d = rem - 3 * k;
          const int pos = __shfl_sync(0xffffffffu, mypos, k);   // every lane takes part
          if (idx >= 36 || k >= NS) continue;
          double v = kb[idx];
          if (ELEMD && src.direct && c == d) v += src.De[16 * e + 4 * a + k];
          acc[9 * pos + 3 * c + d] += v;
        }
        __syncwarp();
      }
    }
    double* vrow = val + 9 * o;
    for (int k = lane; k < 9 * u; k += 32) vrow[k] = acc[k];
    __syncwarp();
  }
}

#ifdef MORTAR_PAIR_NS
__global__ void k_tangent_nnzb(const int64_t* __restrict__ rp, int64_t N, DevStatus* st) {
  if (threadIdx.x == 0 && blockIdx.x == 0) st->nnzb_K = (unsigned long long)rp[N];
}

template <int NS, int NM, bool SEG, bool DUAL>
void launch_pairs_t(mortar_ctx* c) {
  TanArgs g{c->pairs_s.as<int32_t>(), c->pairs_m.as<int32_t>(), c->srec.as<double>(), c->xs.as<double>(),
            c->xm.as<double>(), c->conn_s.as<int32_t>(), c->conn_m.as<int32_t>(), c->tan_ys.as<double>(),
            c->tan_ym.as<double>(), c->tan_Kp.as<double>(), c->tan_Op.as<double>(), c->flag.as<uint8_t>(),
            c->tan_pair_cap, c->dstat.as<DevStatus>(), c->watchdog_us};
  // batches of 160 pairs: 16 full rounds of 10 pair groups (lanes 30, 31 idle)
  auto kern = k_tangent_pairs<NS, NM, SEG, DUAL, 5>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTanSmem<NS, NM, SEG>);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kTanThreads, kTanSmem<NS, NM, SEG>);
  if (per_sm < 1) per_sm = 1;
  kern<<<(unsigned)(c->n_sm * per_sm), kTanThreads, kTanSmem<NS, NM, SEG>, c->stream>>>(g);
}

template <int NS, int NM, bool SEG, bool DUAL, bool ELEMD>
void rows_t(mortar_ctx* c, int mode) {
  TanRowSource<NS, NM, SEG, DUAL, ELEMD> src{
      c->n2e_s_ptr.as<int64_t>(), c->n2e_s_ent.as<int64_t>(), c->pair_off.as<int64_t>(), c->pairs_m.as<int32_t>(),
      c->flag.as<uint8_t>(), c->conn_s.as<int32_t>(), c->conn_m.as<int32_t>(), c->tan_Kp.as<double>(),
      c->tan_Ke.as<double>(), c->Mblk.as<double>(), c->Dblk.as<double>(), c->De.as<double>(), c->Ns,
      c->tan_direct};
  const int64_t N = c->Ns;
  const unsigned g = (unsigned)((N + kThreads - 1) / kThreads);
  DevStatus* st = c->dstat.as<DevStatus>();
  if (mode == 0) {
    if (N > 0)
      k_tangent_rows<0><<<g, kThreads, 0, c->stream>>>(src, N, c->row_cnt.as<int32_t>(), nullptr, 0, nullptr,
                                                       nullptr, st);
    launch_exclusive_scan_i32(c->row_cnt.as<int32_t>(), c->tan_rowptr.as<int64_t>(), nullptr, N,
                              c->scan_tmp.as<int64_t>(), c->stream);
    k_tangent_nnzb<<<1, 32, 0, c->stream>>>(c->tan_rowptr.as<int64_t>(), N, st);
  } else if (N > 0) {
    k_tangent_rows<1><<<g, kThreads, 0, c->stream>>>(src, N, nullptr, c->tan_rowptr.as<int64_t>(), c->tan_nnzb_cap,
                                                     c->tan_col.as<int32_t>(), nullptr, st);
    const int64_t blocks = std::min<int64_t>((N + kRowWarps - 1) / kRowWarps, (int64_t)c->n_sm * 64);
    k_tangent_rows_warp<NS, NM, SEG, DUAL, ELEMD><<<(unsigned)blocks, 32 * kRowWarps, 0, c->stream>>>(
        src, N, c->tan_rowptr.as<int64_t>(), c->tan_nnzb_cap, c->tan_col.as<int32_t>(), c->tan_val.as<double>(), st);
  }
}

}  // namespace

template <int NS, int NM>
void tangent_pairs_nsnm(mortar_ctx* c, const RunParams& rp) {
  const bool seg = rp.d_domain == 1, dual = rp.lm == 1;
  if (seg && dual) launch_pairs_t<NS, NM, true, true>(c);
  else if (seg) launch_pairs_t<NS, NM, true, false>(c);
  else if (dual) launch_pairs_t<NS, NM, false, true>(c);
  else launch_pairs_t<NS, NM, false, false>(c);
}

template <int NS, int NM>
void tangent_rows_nsnm(mortar_ctx* c, const RunParams& rp, int mode) {
  const bool seg = rp.d_domain == 1, dual = rp.lm == 1;
  if (seg && dual) rows_t<NS, NM, true, true, false>(c, mode);
  else if (seg) rows_t<NS, NM, true, false, false>(c, mode);
  else if (dual) rows_t<NS, NM, false, true, true>(c, mode);
  else rows_t<NS, NM, false, false, true>(c, mode);
}

template void tangent_pairs_nsnm<MORTAR_PAIR_NS, MORTAR_PAIR_NM>(mortar_ctx*, const RunParams&);
template void tangent_rows_nsnm<MORTAR_PAIR_NS, MORTAR_PAIR_NM>(mortar_ctx*, const RunParams&, int);
#else   // the main part: element blocks, dispatch

template <int NS, bool DUAL, bool ELEMD>
void launch_elems_t(mortar_ctx* c) {
  if (c->Es == 0) return;
  k_tangent_elems<NS, DUAL, ELEMD><<<(unsigned)((c->Es + kThreads - 1) / kThreads), kThreads, 0, c->stream>>>(
      c->xs.as<double>(), c->conn_s.as<int32_t>(), c->tan_ys.as<double>(), c->srec.as<double>(),
      c->pair_off.as<int64_t>(), c->flag.as<uint8_t>(), c->tan_Op.as<double>(), c->Es, c->tan_Ke.as<double>(),
      c->dstat.as<DevStatus>());
}

}  // namespace

bool tangent_needs_elems(const mortar_ctx* c) {
  return c->opt.lm == MORTAR_LM_DUAL || c->opt.d_domain == MORTAR_D_ELEMENT;
}

void launch_tangent_blocks(mortar_ctx* c, const RunParams& rp) {
  if (c->nen_s == 4 && c->nen_m == 4) tangent_pairs_nsnm<4, 4>(c, rp);
  else if (c->nen_s == 4 && c->nen_m == 3) tangent_pairs_nsnm<4, 3>(c, rp);
  else if (c->nen_s == 3 && c->nen_m == 4) tangent_pairs_nsnm<3, 4>(c, rp);
  else tangent_pairs_nsnm<3, 3>(c, rp);
  if (!tangent_needs_elems(c)) return;
  const bool elemd = rp.d_domain == 0, dual = rp.lm == 1;
  if (c->nen_s == 4) {
    if (dual && elemd) launch_elems_t<4, true, true>(c);
    else if (dual) launch_elems_t<4, true, false>(c);
    else launch_elems_t<4, false, true>(c);
  } else {
    if (dual && elemd) launch_elems_t<3, true, true>(c);
    else if (dual) launch_elems_t<3, true, false>(c);
    else launch_elems_t<3, false, true>(c);
  }
}

void launch_tangent_rows(mortar_ctx* c, const RunParams& rp, int mode) {
  if (c->nen_s == 4 && c->nen_m == 4) tangent_rows_nsnm<4, 4>(c, rp, mode);
  else if (c->nen_s == 4 && c->nen_m == 3) tangent_rows_nsnm<4, 3>(c, rp, mode);
  else if (c->nen_s == 3 && c->nen_m == 4) tangent_rows_nsnm<3, 4>(c, rp, mode);
  else tangent_rows_nsnm<3, 3>(c, rp, mode);
}
#endif  // MORTAR_PAIR_NS

}  // namespace mortar
