// Adjoint (reverse-mode gradient) of the weighted gap functional
//     J = sum_j lambda_j . ( (D X_s)_j - (M X_m)_j )
// with respect to every slave and master nodal coordinate -- the consistent
// linearisation of the mortar terms (Sec. 1 of arXiv 2202.03933).
//
// Per pair, J_pair = sum over quadrature points of W * Lh . q with
//   Lh = sum_c Lambda_c N_c(xi_s),  Lambda_c = sum_a A[a][c] lambda_a,
//   q  = [segment D] x_s(xi_s) - x_m(xi_m)   (x_s, x_m: isoparametric
//        interpolation of the ORIGINAL 3D nodes).
// The kernel recomputes the pair's geometry (nothing is stored between the
// forward and the adjoint) while recording the clip (every intersection vertex
// with its two parent vertices and its clip edge), then runs the reverse sweep:
//   quadrature point -> back-projection (implicit function theorem at the
//   converged xi: dxi = J^-1 (dx - d map)) -> cell vertices and cell area ->
//   centroid fan -> merge (selection) -> clipping stages (vertex copies and
//   edge intersections x = p + t (q - p), t = d_p / (d_p - d_q)) -> in-plane
//   coordinates u = (X - x0).t1, v = (X - x0).t2 -> auxiliary plane (x0, n0,
//   t1, t2 as functions of the slave nodes).
// The LM coefficients A (dual basis, A = Dh Me^-1) depend on the slave
// element only: each pair emits dJ/dA, a per-element kernel sums it over the
// element's pairs, adds the element-domain D term and propagates both through
// A and the element integrals to the slave nodes.  Per-pair and per-element
// gradient blocks are then gathered per node in a fixed order (no floating
// point atomics), and J is reduced with a fixed tree: results are bitwise
// reproducible.
#include <algorithm>
#include <type_traits>

#include "adjoint_fixed.cuh"
#include "clip.cuh"
#include "context.h"
#include "pair_sort.cuh"
#include "reverse.cuh"

namespace mortar {

namespace {

constexpr int kThreads = 128;


// Reverse of the back-projection at a converged xi: accumulates the adjoint of
// the query point (xb) and of the map coefficients (cb[8] = c0u c0v c1u c1v ...).
__device__ __forceinline__ void invert_map_reverse(const PlaneMap& m, double xi, double eta, double xib0,
                                                   double xib1, double& xbu, double& xbv, double* cb) {
  const double j00 = m.c1u + m.c3u * eta, j01 = m.c2u + m.c3u * xi;
  const double j10 = m.c1v + m.c3v * eta, j11 = m.c2v + m.c3v * xi;
  const double inv = 1.0 / (j00 * j11 - j01 * j10);
  const double mu = (j11 * xib0 - j10 * xib1) * inv;   // mu = J^-T xib
  const double mv = (-j01 * xib0 + j00 * xib1) * inv;
  xbu += mu;
  xbv += mv;
  const double xe = xi * eta;
  cb[0] -= mu;      cb[1] -= mv;
  cb[2] -= xi * mu; cb[3] -= xi * mv;
  cb[4] -= eta * mu; cb[5] -= eta * mv;
  cb[6] -= xe * mu; cb[7] -= xe * mv;
}

struct AdjCounters {
  unsigned long long clip_over = 0, newton_fail = 0, nonempty = 0, cells = 0, gp = 0;
};

// Forward outputs written by the fused kernel (M, D blocks and flags).
struct FwdOut {
  double* Mblk;
  double* Dblk;
  uint8_t* flag;
};

// What a pair contributes to its slave element, summed per element by
// k_adjoint_elems before the steps that depend on the element alone (dual
// basis, J, auxiliary plane): Lb_c = dJ/dLambda_c (12), in-plane adjoints of the
// slave nodes (4 + 4), adjoints of the plane from the master nodes (x0, t1, t2),
// one word of padding, and (segment D) the direct slave node gradients (12).
template <bool SEG>
constexpr int kSlavePair = SEG ? 42 : 30;

template <bool SEG>
__device__ __forceinline__ void store_slave_pair(double* __restrict__ sl, int64_t p, const V3* Lb, const double* sbu,
                                                 const double* sbv, const PlaneBar& pb, const double gX[4][3]) {
  double2* o = reinterpret_cast<double2*>(sl + kSlavePair<SEG> * p);
  auto put = [&](int k, double a, double b) { __stcs(o + k, make_double2(a, b)); };
  for (int c = 0; c < 4; c += 2) {
    put(3 * c / 2, Lb[c].x, Lb[c].y);
    put(3 * c / 2 + 1, Lb[c].z, Lb[c + 1].x);
    put(3 * c / 2 + 2, Lb[c + 1].y, Lb[c + 1].z);
  }
  put(6, sbu[0], sbu[1]); put(7, sbu[2], sbu[3]);
  put(8, sbv[0], sbv[1]); put(9, sbv[2], sbv[3]);
  put(10, pb.x0.x, pb.x0.y); put(11, pb.x0.z, pb.t1.x); put(12, pb.t1.y, pb.t1.z);
  put(13, pb.t2.x, pb.t2.y); put(14, pb.t2.z, 0.0);
  if (SEG)
    for (int k = 0; k < 6; ++k) put(15 + k, gX[2 * k / 3][2 * k % 3], gX[(2 * k + 1) / 3][(2 * k + 1) % 3]);
}

template <int NS, int NM, bool SEG, bool DUAL>
__device__ void adjoint_one(int64_t p, const int32_t* __restrict__ ps, const int32_t* __restrict__ pm,
                            const double* __restrict__ srec, const double* __restrict__ xs,
                            const double* __restrict__ xm, const int32_t* __restrict__ conn_s,
                            const int32_t* __restrict__ conn_m, const double* __restrict__ lambda,
                            const RunParams& rp, double* __restrict__ sl_out, double* __restrict__ gm_out,
                            AdjCounters& ctr) {
  const int32_t s = ps[p], m = pm[p];
  const double* r = srec + (int64_t)SR_STRIDE * s;
  double gX[4][3], gY[4][3], Lb[4][3];
  for (int a = 0; a < 4; ++a)
    for (int k = 0; k < 3; ++k) { gX[a][k] = 0.0; gY[a][k] = 0.0; Lb[a][k] = 0.0; }
  const double eps_in = r[SR_EPSIN];
  bool nonempty = false;
  V3 X[4], Y[4], lam[4], Lam[4];
  if (eps_in >= 0.0) {
    for (int a = 0; a < NS; ++a) {
      const int64_t n = conn_s[(int64_t)NS * s + a];
      X[a] = v3(xs[3 * n], xs[3 * n + 1], xs[3 * n + 2]);
      lam[a] = v3(lambda[3 * n], lambda[3 * n + 1], lambda[3 * n + 2]);
    }
    for (int l = 0; l < NM; ++l) {
      const int64_t n = conn_m[(int64_t)NM * m + l];
      Y[l] = v3(xm[3 * n], xm[3 * n + 1], xm[3 * n + 2]);
    }
    const V3 x0 = v3(r[SR_X0], r[SR_X0 + 1], r[SR_X0 + 2]);
    const V3 t1 = v3(r[SR_T1], r[SR_T1 + 1], r[SR_T1 + 2]);
    const V3 t2 = v3(r[SR_T2], r[SR_T2 + 1], r[SR_T2 + 2]);
    // ---- forward: projection, maps, orientation (as in the integration kernel)
    double mu[4], mv[4];
    for (int l = 0; l < NM; ++l) {
      const double dx = Y[l].x - x0.x, dy = Y[l].y - x0.y, dz = Y[l].z - x0.z;
      mu[l] = dx * t1.x + dy * t1.y + dz * t1.z;
      mv[l] = dx * t2.x + dy * t2.y + dz * t2.z;
    }
    const PlaneMap mmap = plane_map<NM>(mu, mv);
    PlaneMap smap;
    smap.c0u = r[SR_C + 0]; smap.c0v = r[SR_C + 1]; smap.c1u = r[SR_C + 2]; smap.c1v = r[SR_C + 3];
    smap.c2u = r[SR_C + 4]; smap.c2v = r[SR_C + 5]; smap.c3u = r[SR_C + 6]; smap.c3v = r[SR_C + 7];
    const bool mrev = polygon_reversed<NM>(mu, mv);
    const bool srev = r[SR_REV] != 0.0;
    // ---- forward clip with recorded stages and merge
    ClipRec<NS> cr;
    nonempty = cr.template run<NM>(r, mu, mv, mrev, ctr.clip_over);
    const int nr = cr.nr;
    if (nonempty) {
      // LM-weighted multipliers Lambda_c
      double A[4][4];
      for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b) A[a][b] = r[SR_A + 4 * a + b];
      for (int c = 0; c < NS; ++c) {
        if (DUAL) {
          V3 acc = v3(0, 0, 0);
          for (int a = 0; a < NS; ++a) acc = acc + A[a][c] * lam[a];
          Lam[c] = acc;
        } else {
          Lam[c] = lam[c];
        }
      }
      double Ru[kPolyA], Rv[kPolyA], Rbu[kPolyA], Rbv[kPolyA];
      for (int k = 0; k < nr; ++k) {
        Ru[k] = cr.pu(k);
        Rv[k] = cr.pv(k);
        Rbu[k] = 0.0;
        Rbv[k] = 0.0;
      }
      double cu = 0.0, cv = 0.0, cbu = 0.0, cbv = 0.0;
      int ncell = 1;
      if (nr > 3) {
        double su = 0.0, sv = 0.0;
        for (int k = 0; k < nr; ++k) { su += Ru[k]; sv += Rv[k]; }
        cu = su / (double)nr;
        cv = sv / (double)nr;
        ncell = nr;
      }
      double smb[8] = {0, 0, 0, 0, 0, 0, 0, 0}, mmb[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      for (int cI = 0; cI < ncell; ++cI) {
        int ib, iw;
        double au, av;
        if (nr == 3) {
          au = Ru[0]; av = Rv[0]; ib = 1; iw = 2;
        } else {
          au = cu; av = cv; ib = cI; iw = cI + 1 == nr ? 0 : cI + 1;
        }
        const double e1u = Ru[ib] - au, e1v = Rv[ib] - av, e2u = Ru[iw] - au, e2v = Rv[iw] - av;
        const double cr = cross2(e1u, e1v, e2u, e2v);
        const double area = 0.5 * fabs(cr);
        double area_b = 0.0, e1bu = 0.0, e1bv = 0.0, e2bu = 0.0, e2bv = 0.0, abu = 0.0, abv = 0.0;
#pragma unroll 1
        for (int q = 0; q < 7; ++q) {
          double l1, l2, w;
          tri7_point(q, l1, l2, w);
          const double xu = au + l1 * e1u + l2 * e2u;
          const double xv = av + l1 * e1v + l2 * e2v;
          const double W = w * area;
          double xs1, xs2, xm1, xm2;
          if (!invert_plane_map<NS>(smap, xu, xv, rp.newton_tol, rp.newton_max_iter, xs1, xs2)) ctr.newton_fail++;
          if (!invert_plane_map<NM>(mmap, xu, xv, rp.newton_tol, rp.newton_max_iter, xm1, xm2)) ctr.newton_fail++;
          double Ns[4], Nm[4];
          shape_fn<NS>(xs1, xs2, Ns);
          shape_fn<NM>(xm1, xm2, Nm);
          V3 Lh = v3(0, 0, 0), xsI = v3(0, 0, 0), xmI = v3(0, 0, 0);
          for (int c = 0; c < NS; ++c) Lh = Lh + Ns[c] * Lam[c];
          if (SEG)
            for (int b = 0; b < NS; ++b) xsI = xsI + Ns[b] * X[b];
          for (int l = 0; l < NM; ++l) xmI = xmI + Nm[l] * Y[l];
          const V3 qv = xsI - xmI;
          const double f = dot(Lh, qv);
          // ---- reverse of this quadrature point
          area_b += w * f;
          const V3 Lhb = W * qv, qb = W * Lh;
          double Nsb[4] = {0, 0, 0, 0}, Nmb[4] = {0, 0, 0, 0};
          for (int c = 0; c < NS; ++c) {
            Lb[c][0] += Ns[c] * Lhb.x; Lb[c][1] += Ns[c] * Lhb.y; Lb[c][2] += Ns[c] * Lhb.z;
            Nsb[c] += dot(Lam[c], Lhb);
          }
          if (SEG)
            for (int b = 0; b < NS; ++b) {
              gX[b][0] += Ns[b] * qb.x; gX[b][1] += Ns[b] * qb.y; gX[b][2] += Ns[b] * qb.z;
              Nsb[b] += dot(X[b], qb);
            }
          for (int l = 0; l < NM; ++l) {
            gY[l][0] -= Nm[l] * qb.x; gY[l][1] -= Nm[l] * qb.y; gY[l][2] -= Nm[l] * qb.z;
            Nmb[l] -= dot(Y[l], qb);
          }
          double dNs[4][2], dNm[4][2];
          shape_grad<NS>(xs1, xs2, dNs);
          shape_grad<NM>(xm1, xm2, dNm);
          double xsb0 = 0.0, xsb1 = 0.0, xmb0 = 0.0, xmb1 = 0.0;
          for (int c = 0; c < NS; ++c) { xsb0 += Nsb[c] * dNs[c][0]; xsb1 += Nsb[c] * dNs[c][1]; }
          for (int l = 0; l < NM; ++l) { xmb0 += Nmb[l] * dNm[l][0]; xmb1 += Nmb[l] * dNm[l][1]; }
          double xbu = 0.0, xbv = 0.0;
          invert_map_reverse(smap, xs1, xs2, xsb0, xsb1, xbu, xbv, smb);
          invert_map_reverse(mmap, xm1, xm2, xmb0, xmb1, xbu, xbv, mmb);
          abu += xbu; abv += xbv;
          e1bu += l1 * xbu; e1bv += l1 * xbv;
          e2bu += l2 * xbu; e2bv += l2 * xbv;
        }
        // area = |cr| / 2
        const double crb = 0.5 * (cr < 0.0 ? -area_b : area_b);
        e1bu += crb * e2v; e1bv -= crb * e2u;
        e2bu -= crb * e1v; e2bv += crb * e1u;
        Rbu[ib] += e1bu; Rbv[ib] += e1bv;
        Rbu[iw] += e2bu; Rbv[iw] += e2bv;
        abu -= e1bu + e2bu;
        abv -= e1bv + e2bv;
        if (nr == 3) { Rbu[0] += abu; Rbv[0] += abv; } else { cbu += abu; cbv += abv; }
      }
      if (nr > 3) {
        const double inv = 1.0 / (double)nr;
        for (int k = 0; k < nr; ++k) { Rbu[k] += cbu * inv; Rbv[k] += cbv * inv; }
      }
      // ---- reverse merge and clipping stages, projection, auxiliary plane
      double sbu[4] = {0, 0, 0, 0}, sbv[4] = {0, 0, 0, 0}, mbu[4] = {0, 0, 0, 0}, mbv[4] = {0, 0, 0, 0};
      cr.template reverse<NM>(r, Rbu, Rbv, srev, mrev, sbu, sbv, mbu, mbv);
      map_coeff_reverse<NS>(smb, sbu, sbv);
      map_coeff_reverse<NM>(mmb, mbu, mbv);
      PlaneBar pb{v3(0, 0, 0), v3(0, 0, 0), v3(0, 0, 0)};
      project_reverse<NM>(Y, x0, t1, t2, mbu, mbv, gY, pb);
      V3 L[4];
      for (int c = 0; c < 4; ++c) L[c] = v3(Lb[c][0], Lb[c][1], Lb[c][2]);
      store_slave_pair<SEG>(sl_out, p, L, sbu, sbv, pb, gX);
      double* gmo = gm_out + 12 * p;
      for (int a = 0; a < 4; ++a)
        for (int k = 0; k < 3; ++k) gmo[3 * a + k] = gY[a][k];
    }
  }
}

template <int NS, int NM, bool SEG, bool DUAL>
__global__ void __launch_bounds__(kMaxPairBlock) k_adjoint_pairs(
    const int32_t* __restrict__ ps, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xs, const double* __restrict__ xm, const int32_t* __restrict__ conn_s,
    const int32_t* __restrict__ conn_m, const double* __restrict__ lambda, RunParams rp, int64_t pair_cap,
    int32_t chunk, double* __restrict__ sl_out, double* __restrict__ gm_out, DevStatus* st) {
  AdjCounters ctr;
  const int lane = threadIdx.x & 31;
  const bool ok = st->over_pairs == 0 && st->over_bins == 0;
  const int64_t n = ok ? (int64_t)min((unsigned long long)pair_cap, st->n_pairs) : 0;
  const Watchdog wd(rp.watchdog_us);
  for (;;) {   // bounded: the shared counter only grows
    if (wd.expired(&st->timeout)) break;
    int64_t base = 0;
    if (lane == 0) base = (int64_t)atomicAdd(&st->work_ctr2, (unsigned long long)chunk);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= n) break;
    const int64_t end = min(base + (int64_t)chunk, n);
    for (int64_t p = base + lane; p < end; p += 32)
      adjoint_one<NS, NM, SEG, DUAL>(p, ps, pm, srec, xs, xm, conn_s, conn_m, lambda, rp, sl_out, gm_out, ctr);
  }
  block_count_add(&st->clip_overflow, ctr.clip_over);
  block_count_add(&st->newton_fail, ctr.newton_fail);
}

// Node coordinates and multipliers of a pair.  Read for the set-up and again
// (from L1/L2) after the quadrature: keeping them in registers would spill.
template <int NS, int NM>
__device__ __forceinline__ void load_pair_nodes(const int32_t* __restrict__ cs, const int32_t* __restrict__ cm,
                                                const double* __restrict__ xs, const double* __restrict__ xm,
                                                const double* __restrict__ lambda, V3* X, V3* Y, V3* lam) {
  for (int a = 0; a < NS; ++a) {
    const int64_t n = cs[a];
    X[a] = v3(xs[3 * n], xs[3 * n + 1], xs[3 * n + 2]);
    lam[a] = v3(lambda[3 * n], lambda[3 * n + 1], lambda[3 * n + 2]);
  }
  for (int l = 0; l < NM; ++l) {
    const int64_t n = cm[l];
    Y[l] = v3(xm[3 * n], xm[3 * n + 1], xm[3 * n + 2]);
  }
}

// Lambda_c = sum_a A[a][c] lambda_a (dual LMs), lambda_c (standard)
template <int NS, bool DUAL>
__device__ __forceinline__ void lm_weights(const double* __restrict__ r, const V3* lam, V3* Lam) {
  for (int c = 0; c < NS; ++c) {
    if (DUAL) {
      V3 acc = v3(0, 0, 0);
      for (int a = 0; a < NS; ++a) acc = acc + r[SR_A + 4 * a + c] * lam[a];
      Lam[c] = acc;
    } else {
      Lam[c] = lam[c];
    }
  }
}

// Lambda_c (12 words) and its monomial coefficients LM_i (12) of every slave
// element: the pairs of an element share them.
template <int NS, bool DUAL>
__global__ void __launch_bounds__(kThreads) k_multipliers(const int32_t* __restrict__ conn_s,
                                                          const double* __restrict__ lambda,
                                                          const double* __restrict__ srec, int64_t Es,
                                                          double* __restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Es) return;
  V3 lam[4], Lam[4], LM[4];
  for (int a = 0; a < 4; ++a) Lam[a] = LM[a] = v3(0, 0, 0);
  for (int a = 0; a < NS; ++a) {
    const int64_t n = conn_s[(int64_t)NS * e + a];
    lam[a] = v3(lambda[3 * n], lambda[3 * n + 1], lambda[3 * n + 2]);
  }
  lm_weights<NS, DUAL>(srec + (int64_t)SR_STRIDE * e, lam, Lam);
  nodal_to_mono<NS>(Lam, LM);
  double* o = out + 24 * e;
  for (int a = 0; a < 4; ++a) {
    o[3 * a] = Lam[a].x; o[3 * a + 1] = Lam[a].y; o[3 * a + 2] = Lam[a].z;
    o[12 + 3 * a] = LM[a].x; o[12 + 3 * a + 1] = LM[a].y; o[12 + 3 * a + 2] = LM[a].z;
  }
}

template <int N>
__device__ __forceinline__ void load_v3(const double* __restrict__ o, V3* v) {
  for (int a = 0; a < N; ++a) v[a] = v3(o[3 * a], o[3 * a + 1], o[3 * a + 2]);
}

// M = A G and D = A H of a pair from FP64 sums.
template <int NS, int NM, bool SEG, bool DUAL>
__device__ __forceinline__ void adjoint_blocks(int64_t p, const double* __restrict__ r, const double G[4][4],
                                               const double H[4][4], const FwdOut& fo) {
  double* mo = fo.Mblk + 16 * p;
  for (int a = 0; a < 4; ++a)
    for (int l = 0; l < 4; ++l) {
      double v = 0.0;
      if (a < NS && l < NM) {
        if (DUAL)
          for (int c = 0; c < NS; ++c) v += r[SR_A + 4 * a + c] * G[c][l];
        else
          v = G[a][l];
      }
      __stcs(mo + 4 * a + l, v);
    }
  if (SEG) {
    double* dout = fo.Dblk + 16 * p;
    for (int a = 0; a < 4; ++a)
      for (int b = 0; b < 4; ++b) {
        double v = 0.0;
        if (a < NS && b < NS) {
          if (DUAL)
            for (int c = 0; c < NS; ++c) v += r[SR_A + 4 * a + c] * H[c][b];
          else
            v = H[a][b];
        }
        __stcs(dout + 4 * a + b, v);
      }
  }
  __stcs(fo.flag + p, (uint8_t)1);
}

// From a pair's sums (G, H, map-coefficient adjoints smb and mmb, adjoints Bu,
// Bv of the polygon's vertices at their pool slots): the reverse of the clip,
// the master's part of the projection, and the direct terms.  Outputs go out
// with streaming (evict-first) stores: each is written once and read by a later
// kernel, and L2 keeps the threads' stack lines instead.
template <int NS, int NM, bool SEG>
__device__ __forceinline__ void adjoint_finish(int64_t p, const int32_t* __restrict__ cs,
                                               const int32_t* __restrict__ cm, const double* __restrict__ r,
                                               const double* __restrict__ xs, const double* __restrict__ xm,
                                               const V3* Lam, const ClipPool<NS, NM>& cp, double* Bu, double* Bv,
                                               bool mrev, const double* smb, const double* mmb,
                                               const double G[4][4], const double H[4][4],
                                               double* __restrict__ sl_out, double* __restrict__ gm_out) {
  double sbu[4] = {0, 0, 0, 0}, sbv[4] = {0, 0, 0, 0}, mbu[4] = {0, 0, 0, 0}, mbv[4] = {0, 0, 0, 0};
  cp.reverse(r, Bu, Bv, r[SR_REV] != 0.0, mrev, sbu, sbv, mbu, mbv);
  map_coeff_reverse<NS>(smb, sbu, sbv);
  map_coeff_reverse<NM>(mmb, mbu, mbv);
  V3 X[4], Y[4], Lb[4];
  for (int l = 0; l < NM; ++l) {
    const int64_t n = cm[l];
    Y[l] = v3(xm[3 * n], xm[3 * n + 1], xm[3 * n + 2]);
  }
  if (SEG)
    for (int a = 0; a < NS; ++a) {
      const int64_t n = cs[a];
      X[a] = v3(xs[3 * n], xs[3 * n + 1], xs[3 * n + 2]);
    }
  double gX[4][3], gY[4][3];
  for (int c = 0; c < 4; ++c) {
    V3 acc = v3(0, 0, 0);
    if (c < NS) {
      if (SEG)
        for (int b = 0; b < NS; ++b) acc = acc + H[c][b] * X[b];
      for (int l = 0; l < NM; ++l) acc = acc - G[c][l] * Y[l];
    }
    Lb[c] = acc;
  }
  for (int l = 0; l < 4; ++l) {
    V3 acc = v3(0, 0, 0), acx = v3(0, 0, 0);
    for (int c = 0; c < NS; ++c) {
      if (l < NM) acc = acc - G[c][l] * Lam[c];
      if (SEG && l < NS) acx = acx + H[c][l] * Lam[c];
    }
    gY[l][0] = acc.x; gY[l][1] = acc.y; gY[l][2] = acc.z;
    if (SEG) { gX[l][0] = acx.x; gX[l][1] = acx.y; gX[l][2] = acx.z; }
  }
  PlaneBar pb{v3(0, 0, 0), v3(0, 0, 0), v3(0, 0, 0)};
  project_reverse<NM>(Y, v3(r[SR_X0], r[SR_X0 + 1], r[SR_X0 + 2]), v3(r[SR_T1], r[SR_T1 + 1], r[SR_T1 + 2]),
                      v3(r[SR_T2], r[SR_T2 + 1], r[SR_T2 + 2]), mbu, mbv, gY, pb);
  store_slave_pair<SEG>(sl_out, p, Lb, sbu, sbv, pb, gX);
  double2* gmo = reinterpret_cast<double2*>(gm_out + 12 * p);
  for (int k = 0; k < 6; ++k)
    __stcs(gmo + k, make_double2(gY[2 * k / 3][2 * k % 3], gY[(2 * k + 1) / 3][(2 * k + 1) % 3]));
}

// Forward outputs of a pair without a polygon.
template <bool SEG>
__device__ __forceinline__ void adjoint_empty(int64_t p, const FwdOut& fo) {
  double2* mo = reinterpret_cast<double2*>(fo.Mblk + 16 * p);
  for (int k = 0; k < 8; ++k) __stcs(mo + k, make_double2(0.0, 0.0));
  if (SEG) {
    double2* dd = reinterpret_cast<double2*>(fo.Dblk + 16 * p);
    for (int k = 0; k < 8; ++k) __stcs(dd + k, make_double2(0.0, 0.0));
  }
  __stcs(fo.flag + p, (uint8_t)0);
}

// ------------------------------------------------- variant 0, FP64 fallback
// Pairs that do not fit the fixed-point frame.  Same functional, reorganised
// for the FP64 pipe:
//  * the per-point work is written in the monomial basis of the shape
//    functions, N = T m with m = (1, xi, eta, xi eta) (quad4) or (1, xi, eta)
//    (tri3).  With the monomial coefficients LM_i = sum_c T_s[c][i] Lambda_c,
//    YM_j = sum_l T_m[l][j] Y_l and XM_j = sum_b T_s[b][j] X_b (per pair),
//      f = Lh . q = [seg] m_s^T CX m_s - m_s^T CY m_m,
//      CY[i][j] = LM_i . YM_j,  CX[i][j] = LM_i . XM_j,
//    so a point needs v = CY m_m, u = CY^T m_s (and [seg] w = (CX + CX^T) m_s):
//      f = [seg] m_s^T w / 2 - m_s^T v,
//      W df/dxi_s = W (dm_s/dxi_s)^T (w - v),  W df/dxi_m = -W (dm_m/dxi_m)^T u;
//  * the terms that hold the shape functions fixed come from the forward
//    accumulators G = sum W N Nm^T and H = sum W N N^T (summed in the nodal
//    basis: non-negative terms keep small entries accurate) at the end:
//      dJ/dY_l |direct = -sum_c G[c][l] Lambda_c,  dJ/dX_b |direct = sum_c H[c][b] Lambda_c,
//      dJ/dLambda_c = sum_b H[c][b] X_b - sum_l G[c][l] Y_l,  J = sum_c Lambda_c . dJ/dLambda_c;
//  * element maps are inverted with MapInverse (affine 2x2 inverse, or FP32
//    Newton + one Newton step on the FP64 residual), and the
//    implicit-function step applies the FP64 inverse Jacobian at the
//    converged xi (MapInverse::jinvT);
//  * the clip is the record's vertex pool (ClipPool).
template <int NS, int NM, bool SEG, bool DUAL>
__device__ __noinline__ void adjoint_pair_fast(int64_t p, const ClipPool<NS, NM>& cp, bool mrev,
                                  const int32_t* __restrict__ ps, const int32_t* __restrict__ pm,
                                  const double* __restrict__ srec, const double* __restrict__ xs,
                                  const double* __restrict__ xm, const int32_t* __restrict__ conn_s,
                                  const int32_t* __restrict__ conn_m, const double* __restrict__ lambda,
                                  double* __restrict__ sl_out, double* __restrict__ gm_out, const FwdOut& fo,
                                  AdjCounters& ctr) {
  constexpr int KS = NS, KM = NM;   // monomials per side (quad4: 4, tri3: 3)
  double CYv[16], SXv[SEG ? 16 : 1];
  auto CYs = [&](int i, int j) -> double& { return CYv[4 * i + j]; };
  auto SXs = [&](int i, int j) -> double& { return SXv[4 * i + j]; };
  const int32_t s = ps[p], m = pm[p];
  const double* r = srec + (int64_t)SR_STRIDE * s;
  const int32_t* cs = conn_s + (int64_t)NS * s;
  const int32_t* cm = conn_m + (int64_t)NM * m;
  double mu[4], mv[4];
  project_master<NM>(r, xm, cm, mu, mv);
  const PlaneMap mmap = plane_map<NM>(mu, mv);
  PlaneMap smap;
  smap.c0u = r[SR_C + 0]; smap.c0v = r[SR_C + 1]; smap.c1u = r[SR_C + 2]; smap.c1v = r[SR_C + 3];
  smap.c2u = r[SR_C + 4]; smap.c2v = r[SR_C + 5]; smap.c3u = r[SR_C + 6]; smap.c3v = r[SR_C + 7];
  const int nr = cp.nr;
  {
    // monomial coefficients and the pair's bilinear forms
    {
      V3 X[4], Y[4], lam[4], Lam[4], LM[4], YM[4];
      load_pair_nodes<NS, NM>(cs, cm, xs, xm, lambda, X, Y, lam);
      lm_weights<NS, DUAL>(r, lam, Lam);
      nodal_to_mono<NS>(Lam, LM);
      nodal_to_mono<NM>(Y, YM);
#pragma unroll
      for (int i = 0; i < KS; ++i)
#pragma unroll
        for (int j = 0; j < KM; ++j) CYs(i, j) = dot(LM[i], YM[j]);
      if (SEG) {
        V3 XM[4];
        nodal_to_mono<NS>(X, XM);
        double CX[4][4];
#pragma unroll
        for (int i = 0; i < KS; ++i)
#pragma unroll
          for (int j = 0; j < KS; ++j) CX[i][j] = dot(LM[i], XM[j]);
#pragma unroll
        for (int i = 0; i < KS; ++i)
#pragma unroll
          for (int j = 0; j < KS; ++j) SXs(i, j) = CX[i][j] + CX[j][i];
      }
    }
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
    // polygon vertex adjoints, kept at the vertices' pool slots
    double Bu[ClipPool<NS, NM>::kSlots], Bv[ClipPool<NS, NM>::kSlots];
    for (int k = 0; k < cp.nv; ++k) { Bu[k] = 0.0; Bv[k] = 0.0; }
    double cu = 0.0, cv = 0.0, cbu = 0.0, cbv = 0.0;
    int ncell = 1;
    if (nr > 3) {
      double su = 0.0, sv = 0.0;
      for (int k = 0; k < nr; ++k) { su += cp.u(k); sv += cp.v(k); }
      cu = su * kInvCount[nr];
      cv = sv * kInvCount[nr];
      ncell = nr;
    }
    // forward accumulators G = sum W N_s N_m^T, H = sum W N_s N_s^T, summed
    // from the nodal shape functions: all terms are non-negative, so small
    // entries keep their relative accuracy (monomial moments would cancel)
    double G[4][4], H[4][4];
    for (int a = 0; a < 4; ++a)
      for (int b = 0; b < 4; ++b) { G[a][b] = 0.0; H[a][b] = 0.0; }
    double smb[8] = {0, 0, 0, 0, 0, 0, 0, 0}, mmb[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int cI = 0; cI < ncell; ++cI) {
      int ib, iw;
      double au, av;
      if (nr == 3) {
        au = cp.u(0); av = cp.v(0); ib = 1; iw = 2;
      } else {
        au = cu; av = cv; ib = cI; iw = cI + 1 == nr ? 0 : cI + 1;
      }
      const int sb = cp.id(ib), sw = cp.id(iw);
      const double e1u = cp.pu[sb] - au, e1v = cp.pv[sb] - av, e2u = cp.pu[sw] - au, e2v = cp.pv[sw] - av;
      const double cr = cross2(e1u, e1v, e2u, e2v);
      const double area = 0.5 * fabs(cr);
      double area_b = 0.0, e1bu = 0.0, e1bv = 0.0, e2bu = 0.0, e2bv = 0.0, abu = 0.0, abv = 0.0;
      ctr.cells++;
      ctr.gp += 7;
#pragma unroll 1
      for (int q = 0; q < 7; ++q) {
        double l1, l2, w;
        tri7_point(q, l1, l2, w);
        const double xu = au + l1 * e1u + l2 * e2u;
        const double xv = av + l1 * e1v + l2 * e2v;
        const double W = w * area;
        double xs1, xs2, xm1, xm2;
        if (!si.solve(xu, xv, xs1, xs2)) ctr.newton_fail++;
        if (!mi.solve(xu, xv, xm1, xm2)) ctr.newton_fail++;
        const double xs12 = xs1 * xs2, xm12 = xm1 * xm2;
        // v = CY m_m (rows 1.. only: the derivative in xi_s needs no v_0),
        // u = CY^T m_s, and m_s^T CY m_m = u . m_m
        double v[4], u[4];
#pragma unroll
        for (int i = 1; i < KS; ++i) {
          double t = fma(CYs(i, 2), xm2, fma(CYs(i, 1), xm1, CYs(i, 0)));
          if (KM == 4) t = fma(CYs(i, 3), xm12, t);
          v[i] = t;
        }
#pragma unroll
        for (int j = 0; j < KM; ++j) {
          double t = fma(CYs(2, j), xs2, fma(CYs(1, j), xs1, CYs(0, j)));
          if (KS == 4) t = fma(CYs(3, j), xs12, t);
          u[j] = t;
        }
        // g = [seg] (CX + CX^T) m_s - v;  f = [seg] m_s^T w / 2 - m_s^T v
        double g[4], f;
        {
          double fv = fma(u[2], xm2, fma(u[1], xm1, u[0]));
          if (KM == 4) fv = fma(u[3], xm12, fv);
          if (SEG) {
            double fw = 0.0;
#pragma unroll
            for (int i = 0; i < KS; ++i) {
              double t = fma(SXs(i, 2), xs2, fma(SXs(i, 1), xs1, SXs(i, 0)));
              if (KS == 4) t = fma(SXs(i, 3), xs12, t);
              if (i > 0) g[i] = t - v[i];
              fw = i == 0 ? t : fma(i == 1 ? xs1 : (i == 2 ? xs2 : xs12), t, fw);
            }
            f = fma(0.5, fw, -fv);
          } else {
#pragma unroll
            for (int i = 1; i < KS; ++i) g[i] = -v[i];
            f = -fv;
          }
        }
        area_b = fma(w, f, area_b);
        // W df/dxi on both sides
        double xsb0, xsb1, xmb0, xmb1;
        if (KS == 4) {
          xsb0 = W * fma(xs2, g[3], g[1]);
          xsb1 = W * fma(xs1, g[3], g[2]);
        } else {
          xsb0 = W * g[1];
          xsb1 = W * g[2];
        }
        if (KM == 4) {
          xmb0 = -W * fma(xm2, u[3], u[1]);
          xmb1 = -W * fma(xm1, u[3], u[2]);
        } else {
          xmb0 = -W * u[1];
          xmb1 = -W * u[2];
        }
        // forward accumulators (nodal shape functions).  The factors 1/4 of
        // quad4 shape functions are folded into W: with ks, km = 1/4 for a
        // quad4 side (1 for tri3), WNs = (ks km W) N_s / ks and Nm = N_m / km,
        // so that WNs Nm = W N_s N_m
        {
          constexpr double km = NM == 4 ? 0.25 : 1.0;
          constexpr double kw = km * (NS == 4 ? 0.25 : 1.0);
          double WNs[4], Nm[4];
          const double wk = kw * W;
          if constexpr (NS == 4) {
            // products of (1 -+ xi)(1 -+ eta) as FMAs: q (1 -+ eta) = q -+ q eta
            const double qa = fma(-wk, xs1, wk), qb = fma(wk, xs1, wk);
            WNs[0] = fma(-qa, xs2, qa); WNs[1] = fma(-qb, xs2, qb); WNs[2] = fma(qb, xs2, qb);
            WNs[3] = fma(qa, xs2, qa);
          } else {
            WNs[1] = wk * xs1; WNs[2] = wk * xs2; WNs[0] = wk - WNs[1] - WNs[2]; WNs[3] = 0.0;
          }
          if constexpr (NM == 4) {
            const double a = 1.0 - xm1, b = 1.0 + xm1;
            Nm[0] = fma(-a, xm2, a); Nm[1] = fma(-b, xm2, b); Nm[2] = fma(b, xm2, b); Nm[3] = fma(a, xm2, a);
          } else {
            shape_fn<NM>(xm1, xm2, Nm);
          }
#pragma unroll
          for (int a = 0; a < NS; ++a)
#pragma unroll
            for (int l = 0; l < NM; ++l) G[a][l] = fma(WNs[a], Nm[l], G[a][l]);
          if (SEG) {   // H = sum W N_s N_s^T = sum WNs (N_s / km)
            double Ns[4];
            if constexpr (NS == 4 && NM == 4) {
              const double a = 1.0 - xs1, b = 1.0 + xs1;
              Ns[0] = fma(-a, xs2, a); Ns[1] = fma(-b, xs2, b); Ns[2] = fma(b, xs2, b); Ns[3] = fma(a, xs2, a);
            } else {
              shape_fn<NS>(xs1, xs2, Ns);
              if (NM == 4)
                for (int b = 0; b < NS; ++b) Ns[b] *= 4.0;
            }
#pragma unroll
            for (int a = 0; a < NS; ++a)
#pragma unroll
              for (int b = 0; b < NS; ++b) H[a][b] = fma(WNs[a], Ns[b], H[a][b]);
          }
        }
        double msu, msv, mmu, mmv;   // J^-T xib on both sides
        si.jinvT(xs1, xs2, xsb0, xsb1, msu, msv);
        mi.jinvT(xm1, xm2, xmb0, xmb1, mmu, mmv);
        smb[0] -= msu; smb[1] -= msv;
        smb[2] = fma(-xs1, msu, smb[2]); smb[3] = fma(-xs1, msv, smb[3]);
        smb[4] = fma(-xs2, msu, smb[4]); smb[5] = fma(-xs2, msv, smb[5]);
        smb[6] = fma(-xs12, msu, smb[6]); smb[7] = fma(-xs12, msv, smb[7]);
        mmb[0] -= mmu; mmb[1] -= mmv;
        mmb[2] = fma(-xm1, mmu, mmb[2]); mmb[3] = fma(-xm1, mmv, mmb[3]);
        mmb[4] = fma(-xm2, mmu, mmb[4]); mmb[5] = fma(-xm2, mmv, mmb[5]);
        mmb[6] = fma(-xm12, mmu, mmb[6]); mmb[7] = fma(-xm12, mmv, mmb[7]);
        const double xbu = msu + mmu, xbv = msv + mmv;
        abu += xbu; abv += xbv;
        e1bu = fma(l1, xbu, e1bu); e1bv = fma(l1, xbv, e1bv);
        e2bu = fma(l2, xbu, e2bu); e2bv = fma(l2, xbv, e2bv);
      }
      const double crb = 0.5 * (cr < 0.0 ? -area_b : area_b);
      e1bu += crb * e2v; e1bv -= crb * e2u;
      e2bu -= crb * e1v; e2bv += crb * e1u;
      Bu[sb] += e1bu; Bv[sb] += e1bv;
      Bu[sw] += e2bu; Bv[sw] += e2bv;
      abu -= e1bu + e2bu;
      abv -= e1bv + e2bv;
      if (nr == 3) { const int s0 = cp.id(0); Bu[s0] += abu; Bv[s0] += abv; } else { cbu += abu; cbv += abv; }
    }
    if (nr > 3) {
      const double inv = kInvCount[nr];
      for (int k = 0; k < nr; ++k) { const int sk = cp.id(k); Bu[sk] += cbu * inv; Bv[sk] += cbv * inv; }
    }
    V3 X[4], Y[4], lam[4], Lam[4];
    load_pair_nodes<NS, NM>(cs, cm, xs, xm, lambda, X, Y, lam);
    lm_weights<NS, DUAL>(r, lam, Lam);
    adjoint_blocks<NS, NM, SEG, DUAL>(p, r, G, H, fo);
    adjoint_finish<NS, NM, SEG>(p, cs, cm, r, xs, xm, Lam, cp, Bu, Bv, mrev, smb, mmb, G, H, sl_out, gm_out);
    ctr.nonempty++;
  }
}

// Words of the clip record in a pair's adjoint record.
template <int NS, int NM>
__device__ __forceinline__ void store_pool(long long* o, const ClipPool<NS, NM>& cp, bool mrev) {
  constexpr int K = ClipPool<NS, NM>::kSlots;
  static_assert(K == 12, "record layout");
  o += 32 * AdjRecord::kPool;
  for (int k = 0; k < cp.nv; ++k) {
    o[32 * k] = __double_as_longlong(cp.pu[k]);
    o[32 * (K + k)] = __double_as_longlong(cp.pv[k]);
    if (k >= NM) o[32 * (2 * K + k)] = __double_as_longlong(cp.tt[k]);
  }
#pragma unroll
  for (int w = 0; w < 3; ++w) {
    unsigned long long v = 0;
    for (int k = 0; k < 4; ++k)
      if (4 * w + k >= NM && 4 * w + k < cp.nv) v |= (unsigned long long)cp.meta[4 * w + k] << (16 * k);
    o[32 * (3 * K + w)] = (long long)v;
  }
  o[32 * (3 * K + 3)] = (long long)cp.poly;
  o[32 * (3 * K + 4)] = cp.nv | cp.nr << 8 | (mrev ? 1 : 0) << 16;
}
template <int NS, int NM>
__device__ __forceinline__ bool load_pool(const long long* o, ClipPool<NS, NM>& cp) {
  constexpr int K = ClipPool<NS, NM>::kSlots;
  o += 32 * AdjRecord::kPool;
  const int n = (int)o[32 * (3 * K + 4)];
  cp.nv = n & 0xff;
  cp.nr = n >> 8 & 0xff;
  cp.poly = (uint64_t)o[32 * (3 * K + 3)];
  for (int k = 0; k < cp.nv; ++k) {
    cp.pu[k] = __longlong_as_double(o[32 * k]);
    cp.pv[k] = __longlong_as_double(o[32 * (K + k)]);
    if (k >= NM) {
      cp.tt[k] = __longlong_as_double(o[32 * (2 * K + k)]);
      cp.meta[k] = (uint16_t)(o[32 * (3 * K + (k >> 2))] >> (16 * (k & 3)));
    }
  }
  return (n >> 16 & 1) != 0;
}

// nr of a record whose pair the finish kernel runs in FP64: set by the clip
// kernel, or by the cell kernel (the clip kernel has counted the pair then)
constexpr int kSlowPair = 0xff, kSlowCounted = 0xfe;

struct AdjArgs {
  const int32_t* ps;
  const int32_t* pm;
  const double* srec;
  const double* xs;
  const double* xm;
  const int32_t* conn_s;
  const int32_t* conn_m;
  const double* lambda;
  int64_t pair_cap;
  int64_t first;   // first pair of the chunk
  const int32_t* order;
  long long* rec;
  const double* mult;   // k_multipliers
  double* sl;
  double* gm;
  FwdOut fo;
  DevStatus* st;
  int32_t watchdog_us;
};

// Group of 32 pairs for a warp; false when none are left.
__device__ __forceinline__ bool next_group(unsigned long long* ctr, int64_t n, int64_t& g) {
  unsigned long long v = 0;
  if ((threadIdx.x & 31) == 0) v = atomicAdd(ctr, 1ull);
  g = (int64_t)__shfl_sync(0xffffffffu, v, 0);
  return 32 * g < n;
}

// Variant 0 (default; the forward blocks come with it) is split like the
// forward integration, where the work's character changes: k_pair_sort,
// k_adjoint_clip, k_adjoint_cells, k_adjoint_finish, with a record per pair in
// between (832 B, 960 B with segment D).  planar 600x520, dual (1.35 M pairs):
// 0.20 + 1.35 + 4.3 + 1.36 ms against 14.5 to 16.8 ms (by batch size) of one FP64
// kernel with the same sweep.
//
// First kernel: FP64 clip with its record, the pair's bilinear forms CY [and
// SX], and the conversion to fixed point.  Bound by the FP64 pipe and the
// latency of its chains.  One record per pair, in sorted order.
template <int NS, int NM, bool SEG>
__global__ void __launch_bounds__(kMaxPairBlock, 2) k_adjoint_clip(AdjArgs g, unsigned long long* cta_t) {
  cta_mark(cta_t, 0);
  constexpr int W = SEG ? AdjRecord::kWordsSeg : AdjRecord::kWords;
  AdjCounters ctr;
  DevStatus* st = g.st;
  const int64_t n = chunk_pairs(st, g.pair_cap, g.first, kPairChunk);
  const Watchdog wd(g.watchdog_us);
  int64_t grp;
  while (!wd.expired(&st->timeout) && next_group(&st->pair_ctr[1], n, grp)) {   // bounded: the counter only grows
    const int64_t i = 32 * grp + (threadIdx.x & 31);
    long long* o = g.rec + grp * (32 * W) + (threadIdx.x & 31);
    int mark = 0;   // nr of a record with nothing for the cell kernel
    if (i < n) {
      const int64_t p = g.first + g.order[i];
      const int32_t s = g.ps[p], m = g.pm[p];
      const double* r = g.srec + (int64_t)SR_STRIDE * s;
      const int32_t* cm = g.conn_m + (int64_t)NM * m;
      o[32 * FxRecord::kPair] = p;
      double mu[4], mv[4];
      project_master<NM>(r, g.xm, cm, mu, mv);
      const PlaneMap mmap = plane_map<NM>(mu, mv);
      const bool mrev = polygon_reversed<NM>(mu, mv);
      ClipPool<NS, NM> cp;
      if (!cp.run(r, mu, mv, mrev, ctr.clip_over)) {
        adjoint_empty<SEG>(p, g.fo);
      } else {
        store_pool(o, cp, mrev);
        double pu[FxPolygon::kCap], pv[FxPolygon::kCap];
        for (int k = 0; k < min(cp.nr, FxPolygon::kCap); ++k) {
          pu[k] = cp.u(k);
          pv[k] = cp.v(k);
        }
        FxPolygon f;
        mark = kSlowPair;
        if (f.setup<NS, NM>(r, mmap, pu, pv, cp.nr)) {
          // bilinear forms of the pair, and their scales
          // (segment D: x_s - x_m does not change with the origin, and about the
          // element's centre the forms are as large as the element, not as the
          // coordinates: what cancels in fixed point is small)
          const V3 org = SEG ? v3(r[SR_X0], r[SR_X0 + 1], r[SR_X0 + 2]) : v3(0.0, 0.0, 0.0);
          V3 Y[4], LM[4], YM[4];
          for (int l = 0; l < NM; ++l) {
            const int64_t nd = cm[l];
            Y[l] = v3(g.xm[3 * nd], g.xm[3 * nd + 1], g.xm[3 * nd + 2]) - org;
          }
          load_v3<NS>(g.mult + 24 * (int64_t)s + 12, LM);
          nodal_to_mono<NM>(Y, YM);
          double C[4][4], S[4][4];
#pragma unroll
          for (int a = 0; a < NS; ++a)
#pragma unroll
            for (int b = 0; b < NM; ++b) C[a][b] = dot(LM[a], YM[b]);
          if (SEG) {
            V3 X[4], XM[4];
            for (int a = 0; a < NS; ++a) {
              const int64_t nd = g.conn_s[(int64_t)NS * s + a];
              X[a] = v3(g.xs[3 * nd], g.xs[3 * nd + 1], g.xs[3 * nd + 2]) - org;
            }
            nodal_to_mono<NS>(X, XM);
#pragma unroll
            for (int a = 0; a < NS; ++a)
#pragma unroll
              for (int b = 0; b < NS; ++b) S[a][b] = dot(LM[a], XM[b]);
#pragma unroll
            for (int a = 0; a < NS; ++a)
#pragma unroll
              for (int b = 0; b <= a; ++b) {
                S[a][b] += S[b][a];   // a == b: doubled
                S[b][a] = S[a][b];
              }
          }
          AdjScale sc;
          sc.eu = f.su;
          sc.ev = f.sv;
          if (sc.set<NS, NM, SEG>(C, S, f.s, f.m, f.Eu - f.Ev)) {
            FxRecord::store<NS, NM>(o, f, p);
            auto put = [&](int w, double v, int sc) {
              const Dg d = fx_split(fx_of_double(v, 62 - sc));
              o[32 * w] = (long long)(((unsigned long long)(unsigned)d.h << 32) | (unsigned)d.l);
            };
#pragma unroll
            for (int a = 0; a < NS; ++a) {
              put(AdjRecord::kC0 + a, C[a][0], a == 0 ? sc.s0 : sc.sv);
#pragma unroll
              for (int b = 1; b < NM; ++b) put(AdjRecord::kC1 + 3 * a + b - 1, C[a][b], a == 0 ? sc.s1 : sc.s11);
              if (SEG)
#pragma unroll
                for (int b = 0; b < NS; ++b) put(AdjRecord::kSX + 4 * a + b, S[a][b], a == 0 ? sc.s0 : sc.sv);
            }
            o[32 * AdjRecord::kScales] = sc.word1();
            o[32 * AdjRecord::kScales2] = sc.word2();
            mark = -1;
            ctr.cells += f.ncell;
            ctr.gp += 7 * f.ncell;
            ctr.nonempty++;
          }
        }
      }
    }
    if (mark >= 0) o[32 * FxRecord::kInfo] = mark;
    __syncwarp();
  }
  block_count_add(&st->clip_overflow, ctr.clip_over);
  block_count_add(&st->nonempty, ctr.nonempty);
  block_count_add(&st->cells, ctr.cells);
  block_count_add(&st->gauss_points, ctr.gp);
  __syncthreads();
  cta_mark(cta_t, 1);
}

constexpr int kAdjSlots = 56;      // shared 64-bit words per thread of the cell kernel: points, W y or sums
constexpr int kCellThreads = 384;  // the registers of an SM at 168 a thread

// Second kernel: one cell of a pair per lane, as k_pair_quadrature.  Leaves G
// [and H], the map-coefficient adjoints and the polygon vertices' adjoints in
// the record.  Bound by issue (0.4 per scheduler and clock) over the
// multiply-add pipe (43 %) and the integer pipe (38 %), with 3 warps per
// scheduler.  Its loop is beyond the instruction cache's full-rate size (about
// 2,300 instructions), so the warps of a block stay in the same part
// (__syncthreads): 5.2 ms at 600x520, 5.8 ms with every warp on its own.  4.3 ms
// with what later parts need read again from the record instead of held.
// Other shapes (all adjoint kernels together 7.9 ms): 512 threads of 128
// registers 8.6, two blocks of 256 threads of 128 registers 8.3.
template <int NS, int NM, bool SEG>
__global__ void __maxnreg__(168) k_adjoint_cells(AdjArgs ar) {
  constexpr int W = SEG ? AdjRecord::kWordsSeg : AdjRecord::kWords;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pts = reinterpret_cast<long long*>(smem_raw) + threadIdx.x;
  constexpr int stride = kCellThreads;
  long long* sums = pts + 28 * stride;
  const int lane = threadIdx.x & 31;
  DevStatus* st = ar.st;
  const int64_t n = chunk_pairs(st, ar.pair_cap, ar.first, kPairChunk);
  const int turn = cell_turn(n);
  const Watchdog wd(ar.watchdog_us);
  // The warps of a block run their rounds in step: every round costs the same
  // (one cell per lane), and the round's code, about 3,000 instructions, does not
  // fit the instruction cache that all warps of an SM share unless they are in
  // the same part of it.  A warp takes a new turn when its last is used up.
  int64_t r0 = 0;
  int records = 0, w = 0;
  bool more = true;
  for (;;) {
    int ncell = 0;
    for (;;) {   // to the next records with cells; bounded: the shared counter only grows
      if (w >= records) {
        if (!more) break;
        unsigned long long g0 = ~0ull >> 1;
        if (!wd.expired(&st->timeout)) {
          if (lane == 0) g0 = atomicAdd(&st->pair_ctr[2], (unsigned long long)turn);
          g0 = __shfl_sync(0xffffffffu, g0, 0);
        }
        more = (int64_t)g0 < n;
        r0 = (int64_t)g0;
        records = more ? (int)min((int64_t)turn, n - r0) : 0;
        w = 0;
        continue;
      }
      if (w + lane < records) {
        const int64_t i = r0 + w + lane;
        ncell = record_cells(ar.rec[((i >> 5) * W + FxRecord::kInfo) * 32 + (i & 31)]);
      }
      if (__any_sync(0xffffffffu, ncell > 0)) break;
      w += 32;
    }
    if (!__syncthreads_or(w < records)) break;
    const CellSlot cs = assign_cells(ncell);
    const int64_t i = w < records ? r0 + w + cs.rec : 0;
    w += cs.taken;
    long long* o = ar.rec + (i >> 5) * (32 * W) + (i & 31);
    bool ok = cs.cell >= 0;
    // what later parts need they load again: registers are what bounds the warps
    long long weight = 0, area = 0;
    FxView f;
    if (ok) {
      const int64_t p = o[32 * FxRecord::kPair];
      const double* sr = ar.srec + (int64_t)SR_STRIDE * ar.ps[p];
      f.load<NS, NM>(o);
      weight = f.weight(cs.cell);
      ok = fx_back_project<NS, NM, stride>(f, cs.cell, sr, ar.xm, ar.conn_m, ar.pm[p], pts);
    }
    __syncthreads();
    if (ok) {
      AdjScale sc;
      sc.load(o[32 * AdjRecord::kScales], o[32 * AdjRecord::kScales2], f.ke, f.Eu, f.Ev);
      ok = fx_cell_sweep<NS, NM, SEG, stride>(f.s, f.m, sc, o, weight, pts, area);
    }
    const unsigned bad = __ballot_sync(0xffffffffu, cs.cell >= 0 && !ok);
    const bool slow = cs.cell >= 0 && (bad >> cs.first & (cs.cells < 32 ? (1u << cs.cells) - 1u : ~0u)) != 0;
    ok &= !slow;
    // every lane of the pair has read the record by now: results take its words' places
    __syncthreads();
    {
      AdjSums r;
      fx_cell_moments<NS, NM, stride>(pts, r);
      const long long info = o[32 * FxRecord::kInfo];
      const int nr = (int)(info & 0xff);
      AdjScale sc;
      sc.load(o[32 * AdjRecord::kScales], o[32 * AdjRecord::kScales2], FxRecord::info_ke(info), FxRecord::info_eu(info),
              FxRecord::info_ev(info));
      // map-coefficient adjoints: minus the sums of W y (x) (1, xi, eta, xi eta), units of 2^64 of Q61 x Q61
      __syncwarp();
      if (ok) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {   // the plain sums are whole; the others have a fraction, words 16..21
          const int c = e & 1, k = (e & 7) >> 1;
          if (k == 0) {
            sums[e * stride] = e < 8 ? r.s1[c] : r.m1[c];
          } else {
            const FxAcc& a = e < 8 ? r.sx[k - 1][c] : r.mx[k - 1][c];
            const int i = e - (e < 8 ? 2 : 4);
            sums[e * stride] = a.hh + (a.cr >> 32);
            reinterpret_cast<unsigned*>(sums + (16 + (i >> 1)) * stride)[i & 1] = (unsigned)a.cr;
          }
        }
        // vertex adjoints of the cell: moments of both sides and the area's part,
        // d area = +-(1/2)(e2v de1u - e2u de1v + e1u de2v - e1v de2u)
        const int ib = nr > 3 ? cs.cell : 1, iw = nr > 3 ? (cs.cell + 1 == nr ? 0 : cs.cell + 1) : 2;
        const long long cu = o[32 * 24], cv = o[32 * 25];
        const long long e1u = o[64 * ib] - cu, e1v = o[64 * ib + 32] - cv;
        const long long e2u = o[64 * iw] - cu, e2v = o[64 * iw + 32] - cv;
        FxAcc a;
        a.mul(fx_split(e1u), fx_split(e2v));
        FxAcc b;
        b.mul(fx_split(e1v), fx_split(e2u));
        const bool neg = (a.hh - b.hh) + ((a.cr - b.cr) >> 32) < 0;
        const Dg ar2 = fx_split(neg ? -area : area);
        // one component of a vertex: the moments, and the area with the other component of an edge
        auto part = [&](int c, long long s, long long mv, long long e, int es, int xa) {
          const int xv = c == 0 ? sc.xvu : sc.xvv;
          a.mul(ar2, fx_split(e << es));
          return fx_down(s, xv - sc.xs(c)) + fx_down(mv, xv - sc.xm(c)) + fx_down(a.hh + (a.cr >> 32), xv - xa);
        };
        const long long v1u = part(0, r.es1[0], r.em1[0], e2v, sc.ev, sc.xav);
        const long long v1v = part(1, r.es1[1], r.em1[1], -e2u, sc.eu, sc.xau);
        const long long v2u = part(0, r.es2[0], r.em2[0], -e1v, sc.ev, sc.xav);
        const long long v2v = part(1, r.es2[1], r.em2[1], e1u, sc.eu, sc.xau);
        sums[22 * stride] = v1u; sums[23 * stride] = v1v;
        sums[24 * stride] = v2u; sums[25 * stride] = v2v;
        sums[26 * stride] = fx_down(r.s1[0], sc.xvu - sc.xsu) + fx_down(r.m1[0], sc.xvu - sc.xmu) - v1u - v2u;
        sums[27 * stride] = fx_down(r.s1[1], sc.xvv - sc.xsv) + fx_down(r.m1[1], sc.xvv - sc.xmv) - v1v - v2v;
      }
      __syncwarp();
      if (ok) {
        const long long* pair = sums - lane + cs.first;
#pragma unroll 1
        for (int e = cs.cell; e < 16; e += cs.cells) {
          const bool plain = (e & 6) == 0;
          const int i = e - (e < 8 ? 2 : 4);
          long long hh = 0, cr = 0;
          for (int k = 0; k < cs.cells; ++k) {
            hh += pair[e * stride + k];
            if (!plain) cr += reinterpret_cast<const unsigned*>(pair + (16 + (i >> 1)) * stride + k)[i & 1];
          }
          const double v = -fx_to_double(hh, cr, (plain ? 0 : 3) + (e < 8 ? sc.xs(e & 1) : sc.xm(e & 1)));
          o[32 * (AdjRecord::kMapS + e)] = __double_as_longlong(v);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          long long* ov = o + 32 * (AdjRecord::kVertex + c);
          const int xv = c == 0 ? sc.xvu : sc.xvv;
          if (nr == 3) {   // one cell: its corner, then the two vertices
            ov[0] = __double_as_longlong(fx_to_double(pair[(26 + c) * stride], 0, xv));
            ov[64] = __double_as_longlong(fx_to_double(pair[(22 + c) * stride], 0, xv));
            ov[128] = __double_as_longlong(fx_to_double(pair[(24 + c) * stride], 0, xv));
          } else {   // vertex k: cell k's first, cell k - 1's second, 1 / nr of the centre's
            long long centre = 0;
            for (int k = 0; k < cs.cells; ++k) centre += pair[(26 + c) * stride + k];
            FxAcc a;
            a.mul(fx_split(centre), kInvCountFx.d[nr]);
            const int prev = cs.cell == 0 ? cs.cells - 1 : cs.cell - 1;
            const long long v = a.get<2>() + pair[(22 + c) * stride + cs.cell] + pair[(24 + c) * stride + prev];
            ov[64 * cs.cell] = __double_as_longlong(fx_to_double(v, 0, xv));
          }
        }
      }
    }
    __syncthreads();
    {
      FxScales ss, sm;
      FxRecord::load_scales(o, ss, sm);
      const int ke = FxRecord::info_ke(o[32 * FxRecord::kInfo]);
      FxAcc g[4][4];
      if (SEG) {
        fx_cell_products<NS, NS, true, stride>(ss, ss, weight, pts, g);
        fx_sum_cells<NS, NS, stride>(g, cs, ok, sums, [&](int a, int b, long long hh, long long cr) {
          o[32 * (AdjRecord::kH + 4 * a + b)] =
              __double_as_longlong(fx_to_double(hh, cr, ke - ss.shape<NS>(a) - ss.shape<NS>(b)));
        });
      }
      fx_cell_products<NS, NM, false, stride>(ss, sm, weight, pts, g);
      fx_sum_cells<NS, NM, stride>(g, cs, ok, sums, [&](int a, int l, long long hh, long long cr) {
        o[32 * (AdjRecord::kG + 4 * a + l)] =
            __double_as_longlong(fx_to_double(hh, cr, ke - ss.shape<NS>(a) - sm.shape<NM>(l)));
      });
    }
    if (slow && cs.cell == 0) o[32 * FxRecord::kInfo] = kSlowCounted;
  }
}

// Third kernel: per pair, the forward blocks, the reverse of the clip and of
// the master's projection, and the direct terms; bound by the FP64 pipe.  The
// blocks M = A G belong here: inside the cell kernel they cost 0.8 ms more at
// 600x520 (4.5 -> 5.3) than they save.  What depends on the slave element alone
// (the plane's reverse) is done once per element (k_adjoint_elems): pairs
// leave 30 words, 42 with segment D.
template <int NS, int NM, bool SEG, bool DUAL>
__global__ void __launch_bounds__(kMaxPairBlock, 2) k_adjoint_finish(AdjArgs g) {
  constexpr int W = SEG ? AdjRecord::kWordsSeg : AdjRecord::kWords;
  AdjCounters ctr, counted;
  DevStatus* st = g.st;
  const int64_t n = chunk_pairs(st, g.pair_cap, g.first, kPairChunk);
  const Watchdog wd(g.watchdog_us);
  int64_t grp;
  while (!wd.expired(&st->timeout) && next_group(&st->pair_ctr[3], n, grp)) {   // bounded: the counter only grows
    const long long* o = g.rec + grp * (32 * W) + (threadIdx.x & 31);
    const int nr = (int)(o[32 * FxRecord::kInfo] & 0xff);
    if (nr == kSlowPair || nr == kSlowCounted) {
      ClipPool<NS, NM> cp;
      const bool mrev = load_pool(o, cp);
      adjoint_pair_fast<NS, NM, SEG, DUAL>(o[32 * FxRecord::kPair], cp, mrev, g.ps, g.pm, g.srec, g.xs, g.xm, g.conn_s, g.conn_m,
                                           g.lambda, g.sl, g.gm, g.fo, nr == kSlowPair ? ctr : counted);
    } else if (nr != 0) {
      const int64_t p = o[32 * FxRecord::kPair];
      const int32_t s = g.ps[p], m = g.pm[p];
      ClipPool<NS, NM> cp;
      const bool mrev = load_pool(o, cp);
      auto word = [&](int w) { return __longlong_as_double(o[32 * w]); };
      double G[4][4], H[4][4], smb[8], mmb[8];
#pragma unroll
      for (int a = 0; a < NS; ++a) {
#pragma unroll
        for (int l = 0; l < NM; ++l) G[a][l] = word(AdjRecord::kG + 4 * a + l);
        if (SEG)
#pragma unroll
          for (int b = 0; b < NS; ++b) H[a][b] = word(AdjRecord::kH + 4 * a + b);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        smb[k] = word(AdjRecord::kMapS + k);
        mmb[k] = word(AdjRecord::kMapM + k);
      }
      double Bu[ClipPool<NS, NM>::kSlots], Bv[ClipPool<NS, NM>::kSlots];
      for (int k = 0; k < cp.nv; ++k) { Bu[k] = 0.0; Bv[k] = 0.0; }
      for (int k = 0; k < cp.nr; ++k) {
        const int id = cp.id(k);
        Bu[id] += word(AdjRecord::kVertex + 2 * k);
        Bv[id] += word(AdjRecord::kVertex + 2 * k + 1);
      }
      adjoint_blocks<NS, NM, SEG, DUAL>(p, g.srec + (int64_t)SR_STRIDE * s, G, H, g.fo);
      V3 Lam[4];
      load_v3<NS>(g.mult + 24 * (int64_t)s, Lam);
      adjoint_finish<NS, NM, SEG>(p, g.conn_s + (int64_t)NS * s, g.conn_m + (int64_t)NM * m,
                                  g.srec + (int64_t)SR_STRIDE * s, g.xs, g.xm, Lam, cp, Bu, Bv, mrev, smb, mmb, G, H,
                                  g.sl, g.gm);
    }
    __syncwarp();
  }
  // pairs that the clip kernel did not count
  block_count_add(&st->clip_overflow, ctr.clip_over);
  block_count_add(&st->newton_fail, ctr.newton_fail + counted.newton_fail);
  block_count_add(&st->nonempty, ctr.nonempty);
  block_count_add(&st->cells, ctr.cells);
  block_count_add(&st->gauss_points, ctr.gp);
}

// Constant tables of a flat element with dual LMs.  There Dh_a = d for every
// a, Me = d Mref and A is the constant matrix ac (quad4: 4 on the diagonal,
// -2 for edge neighbours, 1 across; tri3: 3 and -1), so the adjoint of the
// element integrals through A = Dh Me^-1 is Meb = -(1/d) ac Ab ac.  The flat
// reverse below needs Meb only through weighted sums sum_ab w_ab Meb_ab, which
// equal -(1/d) sum_cd Ab_cd (ac w ac)_cd: w[k] holds ac w_k ac for the weights
// of the closed-form reference integrals (quad4: the three of S1 / S2; tri3:
// int N_a N_b).
struct FlatDualTables {
  double ac[4][4];
  double w[3][4][4];
};

template <int NS>
constexpr FlatDualTables flat_dual_tables() {
  FlatDualTables t{};
  const double cx[4] = {-1.0, 1.0, 1.0, -1.0}, cy[4] = {-1.0, -1.0, 1.0, 1.0};
  double wk[3][4][4] = {};
  for (int a = 0; a < NS; ++a)
    for (int b = 0; b < NS; ++b) {
      if (NS == 4) {
        const int dd = (a - b + 4) % 4;
        t.ac[a][b] = dd == 0 ? 4.0 : (dd == 2 ? 1.0 : -2.0);
        const double px = 2.0 + (2.0 / 3.0) * cx[a] * cx[b], py = 2.0 + (2.0 / 3.0) * cy[a] * cy[b];
        wk[0][a][b] = px * py;
        wk[1][a][b] = px * (cy[a] + cy[b]);
        wk[2][a][b] = py * (cx[a] + cx[b]);
      } else {
        t.ac[a][b] = a == b ? 3.0 : -1.0;
        wk[0][a][b] = a == b ? 1.0 / 12.0 : 1.0 / 24.0;
      }
    }
  for (int k = 0; k < 3; ++k)
    for (int c = 0; c < NS; ++c)
      for (int d = 0; d < NS; ++d) {
        double v = 0.0;
        for (int a = 0; a < NS; ++a)
          for (int b = 0; b < NS; ++b) v += t.ac[a][c] * wk[k][a][b] * t.ac[d][b];
        t.w[k][c][d] = v;
      }
  return t;
}

// The tables' ac is the dual matrix of the reference element: ac Mref = dref I
// (quad4: Mref = (4, 2, 1) / 9 by node distance, dref = 1; tri3: Mref = 1/12 on
// the diagonal, 1/24 off it, dref = 1/6).
template <int NS>
constexpr bool flat_dual_biorthogonal() {
  const FlatDualTables t = flat_dual_tables<NS>();
  for (int a = 0; a < NS; ++a)
    for (int c = 0; c < NS; ++c) {
      double v = 0.0;
      for (int b = 0; b < NS; ++b) {
        const int dd = (b - c + NS) % NS;
        const double mref = NS == 4 ? (dd == 0 ? 4.0 / 9.0 : (dd == 2 ? 1.0 / 9.0 : 2.0 / 9.0))
                                    : (dd == 0 ? 1.0 / 12.0 : 1.0 / 24.0);
        v += t.ac[a][b] * mref;
      }
      const double want = a == c ? (NS == 4 ? 1.0 : 1.0 / 6.0) : 0.0;
      const double err = v - want;
      if (err > 1e-14 || err < -1e-14) return false;
    }
  return true;
}
static_assert(flat_dual_biorthogonal<4>() && flat_dual_biorthogonal<3>(),
              "flat-element dual coefficients are not the reference element's dual matrix");

// Per slave element: sum dJ/dA over its pairs, add the element-domain D term,
// propagate through A = Dh Me^-1 and the element integrals to the nodes.
template <int NS, bool DUAL, bool ELEMD>
__global__ void __launch_bounds__(kThreads) k_adjoint_elems(
    const double* __restrict__ xs, const int32_t* __restrict__ conn_s, const double* __restrict__ lambda,
    const double* __restrict__ srec, const double* __restrict__ De, const int64_t* __restrict__ pair_off,
    const uint8_t* __restrict__ flag, const double* __restrict__ sl, int64_t Es, double* __restrict__ ge,
    const DevStatus* st) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Es) return;
  double* out = ge + 16 * e;
  for (int k = 0; k < 16; ++k) out[k] = 0.0;
  const double* r = srec + (int64_t)SR_STRIDE * e;
  if (r[SR_EPSIN] < 0.0 || st->over_pairs) return;
  V3 X[4], lam[4];
  for (int a = 0; a < NS; ++a) {
    const int64_t n = conn_s[(int64_t)NS * e + a];
    X[a] = v3(xs[3 * n], xs[3 * n + 1], xs[3 * n + 2]);
    lam[a] = v3(lambda[3 * n], lambda[3 * n + 1], lambda[3 * n + 2]);
  }
  double A[4][4], Ab[4][4], Meb[4][4], Dhb[4];
  for (int a = 0; a < 4; ++a) {
    Dhb[a] = 0.0;
    for (int b = 0; b < 4; ++b) { A[a][b] = r[SR_A + 4 * a + b]; Ab[a][b] = 0.0; Meb[a][b] = 0.0; }
  }
  // what the element's pairs contribute (store_slave_pair)
  constexpr int W = kSlavePair<!ELEMD>;
  double sum[W];
  for (int k = 0; k < W; ++k) sum[k] = 0.0;
  for (int64_t p = pair_off[e]; p < pair_off[e + 1]; ++p) {
    if (!flag[p]) continue;
    const double2* o = reinterpret_cast<const double2*>(sl + W * p);
#pragma unroll
    for (int k = 0; k < W / 2; ++k) {
      const double2 v = __ldcs(o + k);
      sum[2 * k] += v.x;
      sum[2 * k + 1] += v.y;
    }
  }
  V3 Xb[4];
  for (int a = 0; a < 4; ++a) Xb[a] = v3(0, 0, 0);
  double Je = 0.0;
  {   // pairs' part of J, dJ/dA (dual LMs), and the slave's side of projection and plane
    V3 Lb[4], Lam[4];
    load_v3<4>(sum, Lb);
    lm_weights<NS, DUAL>(r, lam, Lam);
    for (int c = 0; c < NS; ++c) {
      Je += dot(Lam[c], Lb[c]);
      if (DUAL)
        for (int a = 0; a < NS; ++a) Ab[a][c] = dot(lam[a], Lb[c]);
    }
    double g[4][3];
    for (int a = 0; a < 4; ++a)
      for (int k = 0; k < 3; ++k) g[a][k] = ELEMD ? 0.0 : sum[(ELEMD ? 0 : 30) + 3 * a + k];
    const V3 x0 = v3(r[SR_X0], r[SR_X0 + 1], r[SR_X0 + 2]), t1 = v3(r[SR_T1], r[SR_T1 + 1], r[SR_T1 + 2]),
             t2 = v3(r[SR_T2], r[SR_T2 + 1], r[SR_T2 + 2]);
    PlaneBar pb{v3(sum[20], sum[21], sum[22]), v3(sum[23], sum[24], sum[25]), v3(sum[26], sum[27], sum[28])};
    project_reverse<NS>(X, x0, t1, t2, sum + 12, sum + 16, g, pb);
    plane_basis_reverse<NS>(X, t1, t2, v3(r[SR_N0], r[SR_N0 + 1], r[SR_N0 + 2]), pb, g);
    load_v3<NS>(&g[0][0], Xb);
  }
  constexpr int nq = NS == 4 ? 9 : 7;
  // element integrals Me, Dh (recomputed).  A flat element (negligible
  // bilinear term: parallelograms, every tri3) has constant tangents g1, g2
  // and Jacobian J0, so Me = J0 Mref and Dh = J0 dref, and in the reverse
  // sweep below the Jacobian's gradient directions are the same at every
  // quadrature point.
  double Me[4][4], Dh[4];
  for (int a = 0; a < 4; ++a) {
    Dh[a] = 0.0;
    for (int b = 0; b < 4; ++b) Me[a][b] = 0.0;
  }
  V3 g1c, g2c;
  bool flat;
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
  const V3 nc = cross(g1c, g2c);
  const double J0 = sqrt(dot(nc, nc));
  if (flat) {
    if constexpr (NS == 4) {
      const double m4 = J0 * (4.0 / 9.0), m2 = J0 * (2.0 / 9.0), m1 = J0 * (1.0 / 9.0);
      for (int a = 0; a < 4; ++a) {
        Dh[a] = J0;
        for (int b = 0; b < 4; ++b) {
          const int dd = (a - b + 4) % 4;
          Me[a][b] = dd == 0 ? m4 : (dd == 2 ? m1 : m2);
        }
      }
    } else {
      for (int a = 0; a < 3; ++a) {
        Dh[a] = J0 * (1.0 / 6.0);
        for (int b = 0; b < 3; ++b) Me[a][b] = J0 * (a == b ? 1.0 / 12.0 : 1.0 / 24.0);
      }
    }
  }
  for (int q = 0; q < nq && !flat; ++q) {
    double xi, eta, w;
    elem_point_a<NS>(q, xi, eta, w);
    double N[4], dN[4][2];
    shape_fn<NS>(xi, eta, N);
    shape_grad<NS>(xi, eta, dN);
    V3 g1 = v3(0, 0, 0), g2 = v3(0, 0, 0);
    for (int a = 0; a < NS; ++a) { g1 = g1 + dN[a][0] * X[a]; g2 = g2 + dN[a][1] * X[a]; }
    const V3 nq3 = cross(g1, g2);
    const double wj = w * sqrt(dot(nq3, nq3));
    for (int a = 0; a < NS; ++a) {
      Dh[a] += wj * N[a];
      for (int b = 0; b < NS; ++b) Me[a][b] += wj * N[a] * N[b];
    }
  }
  if (ELEMD && DUAL) {
    // dual LMs: De = A Me = diag(Dh) exactly, J_e = sum_a Dh_a (lam_a . X_a)
    for (int a = 0; a < NS; ++a) {
      const double dla = dot(lam[a], X[a]);
      const double dab = De[16 * e + 5 * a];
      Je += dab * dla;
      Xb[a] = Xb[a] + dab * lam[a];
      Dhb[a] += dla;
    }
  } else if (ELEMD) {
    // J_e = sum_ab (lam_a . X_b) De_ab with De = A Me
    for (int a = 0; a < NS; ++a)
      for (int b = 0; b < NS; ++b) {
        const double dab = De[16 * e + 4 * a + b];
        Je += dab * dot(lam[a], X[b]);
        Xb[b] = Xb[b] + dab * lam[a];
        const double deb = dot(lam[a], X[b]);
        for (int c = 0; c < NS; ++c) {
          Ab[a][c] += deb * Me[c][b];
          Meb[c][b] += A[a][c] * deb;
        }
      }
  }
  constexpr FlatDualTables kFD = flat_dual_tables<NS>();
  const bool flat_dual = DUAL && flat;
  const double inv_d = flat_dual ? 1.0 / Dh[0] : 0.0;
  if (flat_dual) {
    // Dhb_a += sum_b Ab_ab K_ab with K = ac / d; Meb enters below as weighted sums
#pragma unroll
    for (int a = 0; a < NS; ++a) {
      double t = 0.0;
#pragma unroll
      for (int b = 0; b < NS; ++b) t = fma(kFD.ac[a][b], Ab[a][b], t);
      Dhb[a] = fma(t, inv_d, Dhb[a]);
    }
  } else if (DUAL) {
    // A = Dh K, K = Me^-1 = Dh^-1 A
    double K[4][4], Kb[4][4];
    for (int a = 0; a < NS; ++a) {
      const double inv = 1.0 / Dh[a];   // one division per row
      for (int b = 0; b < NS; ++b) {
        K[a][b] = A[a][b] * inv;
        Kb[a][b] = Dh[a] * Ab[a][b];
      }
    }
    for (int a = 0; a < NS; ++a) {
      double s = 0.0;
      for (int b = 0; b < NS; ++b) s += Ab[a][b] * K[a][b];
      Dhb[a] += s;
    }
    // Meb -= K Kb K
    double T[4][4];
    for (int a = 0; a < NS; ++a)
      for (int b = 0; b < NS; ++b) {
        double s = 0.0;
        for (int c = 0; c < NS; ++c) s += K[a][c] * Kb[c][b];
        T[a][b] = s;
      }
    for (int a = 0; a < NS; ++a)
      for (int b = 0; b < NS; ++b) {
        double s = 0.0;
        for (int c = 0; c < NS; ++c) s += T[a][c] * K[c][b];
        Meb[a][b] -= s;
      }
  }
  // element integrals -> nodes.  The adjoint of the surface Jacobian at a
  // point is jb = sum_ab (Dhb_a + Meb_ab N_b) N_a; a flat element only needs
  // S1_c = int jb dN_c/dxi and S2_c = int jb dN_c/deta over the reference
  // element, which are exact polynomial integrals:
  //   quad4 (corners (xi_a, eta_a) = (-1,-1), (1,-1), (1,1), (-1,1)):
  //     int N_a dN_c/dxi         = xi_c / 4 (1 + eta_a eta_c / 3)
  //     int N_a N_b dN_c/dxi     = xi_c / 64 (2 + 2/3 xi_a xi_b)(2 + 2/3 (eta_a eta_b + eta_c (eta_a + eta_b)))
  //   (and the same with xi and eta exchanged for dN_c/deta);
  //   tri3: dN_c constant, int N_a = 1/6, int N_a N_b = 1/12 (a = b) or 1/24.
  double S1[4] = {0, 0, 0, 0}, S2[4] = {0, 0, 0, 0};
  if (flat) {
    if constexpr (NS == 4) {
      constexpr double cx[4] = {-1.0, 1.0, 1.0, -1.0}, cy[4] = {-1.0, -1.0, 1.0, 1.0};
      double A0 = 0.0, A1 = 0.0, C1 = 0.0, B0 = 0.0, Bx = 0.0, By = 0.0;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        B0 += Dhb[a];
        Bx = fma(cx[a], Dhb[a], Bx);
        By = fma(cy[a], Dhb[a], By);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (flat_dual) {
            A0 = fma(kFD.w[0][a][b], Ab[a][b], A0);
            A1 = fma(kFD.w[1][a][b], Ab[a][b], A1);
            C1 = fma(kFD.w[2][a][b], Ab[a][b], C1);
          } else {
            const double px = 2.0 + (2.0 / 3.0) * cx[a] * cx[b], py = 2.0 + (2.0 / 3.0) * cy[a] * cy[b];
            A0 = fma(px * py, Meb[a][b], A0);
            A1 = fma(px * (cy[a] + cy[b]), Meb[a][b], A1);
            C1 = fma(py * (cx[a] + cx[b]), Meb[a][b], C1);
          }
        }
      }
      if (flat_dual) { A0 *= -inv_d; A1 *= -inv_d; C1 *= -inv_d; }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        S1[c] = cx[c] * fma(1.0 / 64.0, fma((2.0 / 3.0) * cy[c], A1, A0), 0.25 * fma(cy[c] / 3.0, By, B0));
        S2[c] = cy[c] * fma(1.0 / 64.0, fma((2.0 / 3.0) * cx[c], C1, A0), 0.25 * fma(cx[c] / 3.0, Bx, B0));
      }
    } else {
      double T = 0.0, Tm = 0.0;
      for (int a = 0; a < 3; ++a) {
        T = fma(1.0 / 6.0, Dhb[a], T);
        for (int b = 0; b < 3; ++b)
          Tm = flat_dual ? fma(kFD.w[0][a][b], Ab[a][b], Tm) : fma(a == b ? 1.0 / 12.0 : 1.0 / 24.0, Meb[a][b], Tm);
      }
      T = flat_dual ? fma(-inv_d, Tm, T) : T + Tm;
      S1[0] = -T; S1[1] = T; S1[2] = 0.0;
      S2[0] = -T; S2[1] = 0.0; S2[2] = T;
    }
  }
  for (int q = 0; q < nq && !flat; ++q) {
    double xi, eta, w;
    elem_point_a<NS>(q, xi, eta, w);
    double N[4], dN[4][2];
    shape_fn<NS>(xi, eta, N);
    shape_grad<NS>(xi, eta, dN);
    double jb = 0.0;
    for (int a = 0; a < NS; ++a) {
      double v = Dhb[a];
      for (int b = 0; b < NS; ++b) v = fma(Meb[a][b], N[b], v);
      jb = fma(v, N[a], jb);
    }
    jb *= w;
    if (jb == 0.0) continue;
    V3 g1 = v3(0, 0, 0), g2 = v3(0, 0, 0);
    for (int a = 0; a < NS; ++a) { g1 = g1 + dN[a][0] * X[a]; g2 = g2 + dN[a][1] * X[a]; }
    const V3 nq3 = cross(g1, g2);
    const double J = sqrt(dot(nq3, nq3));
    const V3 nb = (jb / J) * nq3;
    const V3 g1b = cross(g2, nb), g2b = cross(nb, g1);
    for (int a = 0; a < NS; ++a) Xb[a] = Xb[a] + dN[a][0] * g1b + dN[a][1] * g2b;
  }
  if (flat && J0 > 0.0) {   // d J / d g1 = g2 x n / J, d J / d g2 = n / J x g1 (same at every point)
    const V3 nu = (1.0 / J0) * nc;
    const V3 d1 = cross(g2c, nu), d2 = cross(nu, g1c);
    for (int a = 0; a < NS; ++a) Xb[a] = Xb[a] + S1[a] * d1 + S2[a] * d2;
  }
  for (int a = 0; a < NS; ++a) {
    out[3 * a] = Xb[a].x;
    out[3 * a + 1] = Xb[a].y;
    out[3 * a + 2] = Xb[a].z;
  }
  out[12] = Je;
}

#ifndef MORTAR_PAIR_NS
// master element -> pairs (non-empty ones), counting sort + per-element sort
__global__ void k_mp_count(const int32_t* __restrict__ pm, const uint8_t* __restrict__ flag, int64_t pair_cap,
                           int32_t* __restrict__ cnt, const DevStatus* st) {
  const int64_t n = st->over_pairs ? 0 : (int64_t)min((unsigned long long)pair_cap, st->n_pairs);
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    if (flag[p]) atomicAdd(&cnt[pm[p]], 1);
}

__global__ void k_mp_fill(const int32_t* __restrict__ pm, const uint8_t* __restrict__ flag, int64_t pair_cap,
                          const int64_t* __restrict__ off, int32_t* __restrict__ cnt, int32_t* __restrict__ list,
                          const DevStatus* st) {
  const int64_t n = st->over_pairs ? 0 : (int64_t)min((unsigned long long)pair_cap, st->n_pairs);
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    if (flag[p]) {
      const int32_t m = pm[p];
      const int32_t slot = atomicSub(&cnt[m], 1) - 1;
      list[off[m] + slot] = (int32_t)p;
    }
}

__global__ void k_mp_sort(const int64_t* __restrict__ off, int64_t Em, int32_t* __restrict__ list) {
  const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= Em) return;
  const int64_t b0 = off[f], b1 = off[f + 1];
  for (int64_t a = b0 + 1; a < b1; ++a) {
    const int32_t v = list[a];
    int64_t b = a - 1;
    while (b >= b0 && list[b] > v) { list[b + 1] = list[b]; --b; }
    list[b + 1] = v;
  }
}

__global__ void k_grad_slave(const int64_t* __restrict__ n2e_ptr, const int64_t* __restrict__ n2e_ent,
                             const double* __restrict__ ge, int64_t Ns, double* __restrict__ grad,
                             const DevStatus* st) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= Ns) return;
  double g0 = 0.0, g1 = 0.0, g2 = 0.0;
  if (!st->over_pairs)
    for (int64_t q = n2e_ptr[j]; q < n2e_ptr[j + 1]; ++q) {
      const int64_t e = n2e_ent[q] >> 2;
      const int a = (int)(n2e_ent[q] & 3);
      g0 += ge[16 * e + 3 * a]; g1 += ge[16 * e + 3 * a + 1]; g2 += ge[16 * e + 3 * a + 2];
    }
  grad[3 * j] = g0;
  grad[3 * j + 1] = g1;
  grad[3 * j + 2] = g2;
}

__global__ void k_grad_master(const int64_t* __restrict__ n2e_ptr, const int64_t* __restrict__ n2e_ent,
                              const int64_t* __restrict__ mp_off, const int32_t* __restrict__ mp_list,
                              const double* __restrict__ gm_pair, int64_t Nm, double* __restrict__ grad,
                              const DevStatus* st) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= Nm) return;
  double g0 = 0.0, g1 = 0.0, g2 = 0.0;
  if (!st->over_pairs)
    for (int64_t q = n2e_ptr[j]; q < n2e_ptr[j + 1]; ++q) {
      const int64_t f = n2e_ent[q] >> 2;
      const int l = (int)(n2e_ent[q] & 3);
      for (int64_t k = mp_off[f]; k < mp_off[f + 1]; ++k) {
        const int64_t p = mp_list[k];
        g0 += gm_pair[12 * p + 3 * l]; g1 += gm_pair[12 * p + 3 * l + 1]; g2 += gm_pair[12 * p + 3 * l + 2];
      }
    }
  grad[3 * j] = g0;
  grad[3 * j + 1] = g1;
  grad[3 * j + 2] = g2;
}

constexpr int kJBlocks = 256;

// Fixed-shape reduction of J over the elements (deterministic).
__global__ void __launch_bounds__(256) k_J_partial(const double* __restrict__ ge, int64_t Es, double* __restrict__ part) {
  const int64_t per = (Es + gridDim.x - 1) / gridDim.x;
  const int64_t b0 = per * blockIdx.x, b1 = min(Es, b0 + per);
  double s = 0.0;
  for (int64_t i = b0 + threadIdx.x; i < b1; i += blockDim.x) s += ge[16 * i + 12];
  __shared__ double sh[256];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void __launch_bounds__(256) k_J_final(const double* __restrict__ part, DevStatus* st) {
  __shared__ double sh[256];
  sh[threadIdx.x] = part[threadIdx.x];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) st->J = sh[0];
}
#endif  // !MORTAR_PAIR_NS

#ifdef MORTAR_PAIR_NS
template <int NS, int NM, bool SEG, bool DUAL>
void launch_pairs_t(mortar_ctx* c, const RunParams& rp, unsigned grid, unsigned block, int32_t chunk) {
  if (grid == 0) {   // persistent grid: every SM filled to the kernel's occupancy
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_adjoint_pairs<NS, NM, SEG, DUAL>, (int)block, 0);
    grid = (unsigned)(c->n_sm * (per_sm < 1 ? 1 : per_sm));
  }
  k_adjoint_pairs<NS, NM, SEG, DUAL><<<grid, block, 0, c->stream>>>(
      c->pairs_s.as<int32_t>(), c->pairs_m.as<int32_t>(), c->srec.as<double>(), c->xs.as<double>(),
      c->xm.as<double>(), c->conn_s.as<int32_t>(), c->conn_m.as<int32_t>(), c->lambda.as<double>(), rp, c->pair_cap,
      chunk, c->sl_pair.as<double>(), c->gm_pair.as<double>(), c->dstat.as<DevStatus>());
}

// The default adjoint always produces the forward blocks as well (the run
// pipeline fuses the two); a non-fused call only rewrites the same blocks.
template <int NS, int NM, bool SEG, bool DUAL>
void launch_fixed(mortar_ctx* c, const RunParams& rp, int block, int rounds) {
  IntegrateArgs ia{c->pairs_s.as<int32_t>(), c->pairs_m.as<int32_t>(), c->srec.as<double>(), c->xm.as<double>(),
                   c->conn_m.as<int32_t>(), nullptr, nullptr, nullptr, c->pair_cap, c->dstat.as<DevStatus>(),
                   c->stream};
  ia.order = c->order.as<int32_t>();
  AdjArgs a{ia.ps, ia.pm, ia.srec, c->xs.as<double>(), ia.xm, c->conn_s.as<int32_t>(), ia.conn_m,
            c->lambda.as<double>(), c->pair_cap, 0, ia.order, c->rec.as<long long>(), c->mult.as<double>(),
            c->sl_pair.as<double>(), c->gm_pair.as<double>(),
            FwdOut{c->Mblk.as<double>(), c->Dblk.as<double>(), c->flag.as<uint8_t>()}, ia.st, c->watchdog_us};
  auto grid = [&](auto kern, int threads, size_t shm) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, shm);
    return (unsigned)(c->n_sm * (per_sm < 1 ? 1 : per_sm));
  };
  unsigned long long* cta_t = (c->timing && c->cta_t.p) ? c->cta_t.as<unsigned long long>() : nullptr;
  auto clip = k_adjoint_clip<NS, NM, SEG>;
  auto cells = k_adjoint_cells<NS, NM, SEG>;
  auto fin = k_adjoint_finish<NS, NM, SEG, DUAL>;
  const size_t shm = (size_t)kCellThreads * kAdjSlots * 8;
  cudaFuncSetAttribute(cells, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
  const unsigned gc = grid(clip, block, 0), gq = grid(cells, kCellThreads, shm), gf = grid(fin, block, 0);
  if (cta_t) c->pair_grid = (int)gc;
  if (c->Es > 0)
    k_multipliers<NS, DUAL><<<(unsigned)((c->Es + kThreads - 1) / kThreads), kThreads, 0, c->stream>>>(
        a.conn_s, a.lambda, a.srec, c->Es, c->mult.as<double>());
  for (; a.first < c->pair_cap; a.first += kPairChunk) {
    launch_pair_sort<NS, NM>(ia, rp, c->n_sm, 32 * rounds, a.first);
    clip<<<gc, block, 0, c->stream>>>(a, a.first == 0 ? cta_t : nullptr);   // a full chunk's balance
    cells<<<gq, kCellThreads, shm, c->stream>>>(a);
    fin<<<gf, block, 0, c->stream>>>(a);
  }
}

}  // namespace

template <int NS, int NM>
void adjoint_pairs_nsnm(mortar_ctx* c, const RunParams& rp, unsigned grid, unsigned block, int32_t chunk) {
  const bool seg = rp.d_domain == 1, dual = rp.lm == 1;
  if (c->variant == 1) {
    if (seg && dual) launch_pairs_t<NS, NM, true, true>(c, rp, grid, block, chunk);
    else if (seg) launch_pairs_t<NS, NM, true, false>(c, rp, grid, block, chunk);
    else if (dual) launch_pairs_t<NS, NM, false, true>(c, rp, grid, block, chunk);
    else launch_pairs_t<NS, NM, false, false>(c, rp, grid, block, chunk);
    return;
  }
  const int rounds = c->rounds > 0 ? c->rounds : kSortBatch / 32;
  if (seg && dual) launch_fixed<NS, NM, true, true>(c, rp, (int)block, rounds);
  else if (seg) launch_fixed<NS, NM, true, false>(c, rp, (int)block, rounds);
  else if (dual) launch_fixed<NS, NM, false, true>(c, rp, (int)block, rounds);
  else launch_fixed<NS, NM, false, false>(c, rp, (int)block, rounds);
}
template void adjoint_pairs_nsnm<MORTAR_PAIR_NS, MORTAR_PAIR_NM>(mortar_ctx*, const RunParams&, unsigned, unsigned,
                                                                  int32_t);
#else   // the main part: element adjoint, gathers, J, dispatch

template <int NS>
void launch_elems_ns(mortar_ctx* c, const RunParams& rp) {
  const unsigned g = (unsigned)((c->Es + kThreads - 1) / kThreads);
  if (c->Es == 0) return;
  const bool elemd = rp.d_domain == 0, dual = rp.lm == 1;
  auto args = [&](auto kern) {
    kern<<<g, kThreads, 0, c->stream>>>(c->xs.as<double>(), c->conn_s.as<int32_t>(), c->lambda.as<double>(),
                                        c->srec.as<double>(), c->De.as<double>(), c->pair_off.as<int64_t>(),
                                        c->flag.as<uint8_t>(), c->sl_pair.as<double>(), c->Es, c->ge_elem.as<double>(),
                                        c->dstat.as<DevStatus>());
  };
  if (dual && elemd) args(k_adjoint_elems<NS, true, true>);
  else if (dual) args(k_adjoint_elems<NS, true, false>);
  else if (elemd) args(k_adjoint_elems<NS, false, true>);
  else args(k_adjoint_elems<NS, false, false>);
}

}  // namespace

int prepare_adjoint_buffers(mortar_ctx* c) {
  const size_t P = (size_t)std::max<int64_t>(c->pair_cap, 1);
  int r;
  if (c->variant == 0) {
    const size_t words = c->opt.d_domain == MORTAR_D_SEGMENT ? AdjRecord::kWordsSeg : AdjRecord::kWords;
    const size_t need = (std::min<size_t>(P, kPairChunk) + 31) / 32 * 32 * words * 8;
    if (c->rec.bytes < need && c->graph_exec) {   // a captured forward run holds the records' address
      cudaGraphExecDestroy(c->graph_exec);
      c->graph_exec = nullptr;
    }
    if ((r = buf_reserve(c->rec, need)) != MORTAR_OK) return r;
  }
  const size_t sl = c->opt.d_domain == MORTAR_D_SEGMENT ? kSlavePair<true> : kSlavePair<false>;
  if ((r = buf_reserve(c->sl_pair, P * sl * 8)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->gm_pair, P * 12 * 8)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->mp_list, P * 4)) != MORTAR_OK) return r;
  const size_t Es = (size_t)std::max<int64_t>(c->Es, 1), Em = (size_t)std::max<int64_t>(c->Em, 1);
  if ((r = buf_reserve(c->ge_elem, Es * 16 * 8)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->mult, Es * 24 * 8)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->mp_cnt, Em * 4)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->mp_off, (Em + 1) * 8)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->grad_s, (size_t)std::max<int64_t>(c->Ns, 1) * 24)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->grad_m, (size_t)std::max<int64_t>(c->Nm, 1) * 24)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->J_part, kJBlocks * 8)) != MORTAR_OK) return r;
  if ((r = buf_reserve(c->lambda, (size_t)std::max<int64_t>(c->Ns, 1) * 24)) != MORTAR_OK) return r;
  return MORTAR_OK;
}

bool adjoint_fuses_forward(const mortar_ctx* c) { return c->variant == 0; }

void launch_adjoint_pairs(mortar_ctx* c, const RunParams& rp) {
  const unsigned block = c->block_size > 0 ? (unsigned)c->block_size : 128u;
  const int32_t chunk = c->chunk_pairs > 0 ? c->chunk_pairs : 32;
  const unsigned grid = 0;   // the one-pair-per-thread kernels size their own grid
  if (c->nen_s == 4 && c->nen_m == 4) adjoint_pairs_nsnm<4, 4>(c, rp, grid, block, chunk);
  else if (c->nen_s == 4 && c->nen_m == 3) adjoint_pairs_nsnm<4, 3>(c, rp, grid, block, chunk);
  else if (c->nen_s == 3 && c->nen_m == 4) adjoint_pairs_nsnm<3, 4>(c, rp, grid, block, chunk);
  else adjoint_pairs_nsnm<3, 3>(c, rp, grid, block, chunk);
}

void launch_adjoint_rest(mortar_ctx* c, const RunParams& rp) {
  DevStatus* st = c->dstat.as<DevStatus>();
  if (c->nen_s == 4) launch_elems_ns<4>(c, rp); else launch_elems_ns<3>(c, rp);
  // master element -> pair lists
  cudaMemsetAsync(c->mp_cnt.p, 0, (size_t)std::max<int64_t>(c->Em, 1) * 4, c->stream);
  const unsigned pg = (unsigned)(c->n_sm * 8);
  k_mp_count<<<pg, 256, 0, c->stream>>>(c->pairs_m.as<int32_t>(), c->flag.as<uint8_t>(), c->pair_cap,
                                        c->mp_cnt.as<int32_t>(), st);
  launch_exclusive_scan_i32(c->mp_cnt.as<int32_t>(), c->mp_off.as<int64_t>(), nullptr, c->Em,
                            c->scan_tmp.as<int64_t>(), c->stream);
  k_mp_fill<<<pg, 256, 0, c->stream>>>(c->pairs_m.as<int32_t>(), c->flag.as<uint8_t>(), c->pair_cap,
                                       c->mp_off.as<int64_t>(), c->mp_cnt.as<int32_t>(), c->mp_list.as<int32_t>(), st);
  if (c->Em > 0)
    k_mp_sort<<<(unsigned)((c->Em + kThreads - 1) / kThreads), kThreads, 0, c->stream>>>(
        c->mp_off.as<int64_t>(), c->Em, c->mp_list.as<int32_t>());
  if (c->Ns > 0)
    k_grad_slave<<<(unsigned)((c->Ns + kThreads - 1) / kThreads), kThreads, 0, c->stream>>>(
        c->n2e_s_ptr.as<int64_t>(), c->n2e_s_ent.as<int64_t>(), c->ge_elem.as<double>(), c->Ns, c->grad_s.as<double>(),
        st);
  if (c->Nm > 0)
    k_grad_master<<<(unsigned)((c->Nm + kThreads - 1) / kThreads), kThreads, 0, c->stream>>>(
        c->n2e_m_ptr.as<int64_t>(), c->n2e_m_ent.as<int64_t>(), c->mp_off.as<int64_t>(), c->mp_list.as<int32_t>(),
        c->gm_pair.as<double>(), c->Nm, c->grad_m.as<double>(), st);
  k_J_partial<<<kJBlocks, 256, 0, c->stream>>>(c->ge_elem.as<double>(), c->Es, c->J_part.as<double>());
  k_J_final<<<1, 256, 0, c->stream>>>(c->J_part.as<double>(), st);
}
#endif  // MORTAR_PAIR_NS

}  // namespace mortar
