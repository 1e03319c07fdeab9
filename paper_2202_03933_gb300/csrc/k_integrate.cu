// Per-pair segment-based mortar integration (Algorithm 1 body, Sec. 2.3).
//
// For one slave/master pair: project the master nodes onto the slave
// element's auxiliary plane (Fig. 1: x0, n0), clip the master polygon by the
// slave polygon (Sutherland-Hodgman with an absolute inside band eps_in),
// merge near-duplicate vertices, discard slivers, split the clip polygon
// into a centroid fan of triangular cells, and integrate with the 7-point
// degree-5 rule.  At every quadrature point both elements are inverted
// (chi_h: the element map in the plane solved for xi) and
//     G[c][l] += W N_c(xi_s) N_l(xi_m),   H[c][b] += W N_c(xi_s) N_b(xi_s)
// so that M_pair = A G and D_pair = A H with the slave element's LM
// coefficients A (Phi_a = sum_c A[a][c] N_c, Eq. AnsatzDiscretizationLagrangeMult).
//
// GB300 has two FP64 lanes per SM and clock, and a warp-wide FP64 instruction
// costs the same with 1 or 32 active lanes, so the FP64 work is kept small and
// in full warps:
//
//  * variant 0 (default): three kernels.  k_pair_sort orders batches of pairs
//    by the cell count and edge intersections of an FP32 clip; k_pair_clip clips
//    in FP64 (which decides what a pair contributes) and turns the polygon, the
//    element maps and the cell weights into a fixed-point record;
//    k_pair_quadrature integrates the records on the integer pipe, one cell of
//    a pair per lane (fixed.cuh, quadrature.cuh).
//    planar_600x520 (1.35 M pairs, dual LMs): 0.20 + 0.95 + 1.63 ms, against
//    6.2 ms (batches of 64 pairs, the former default) and 5.6 ms (1024) of the
//    one-kernel FP64 form.  The clip kernel is bound by the FP64 pipe (50 %
//    busy, 400 instructions a pair) and instruction fetch, the quadrature
//    kernel by issue (0.52 per scheduler and clock) over the multiply-add and
//    integer pipes.
//  * one kernel (k_integrate_fused): for callers without workspace.  Clip
//    records in shared memory, then the same quadrature.
//  * pairs that do not fit the fixed-point frame are integrated in FP64 in
//    either form (integrate_polygon_fp64): affine maps are inverted with one
//    precomputed 2x2 inverse, bilinear ones by Newton in FP32, then one step
//    with an FP64 residual (MapInverse in clip.cuh).
//  * variant 1: one pair per thread, FP64 Newton from xi = 0 at every point
//    (the oracle's iteration), kept as the reference schedule.
//
// All are persistent grids taking work from a global counter; the loops are
// bounded by the pair count.
#include "clip.cuh"
#include "context.h"
#include "pair_sort.cuh"
#include "quadrature.cuh"
#include "reverse.cuh"

namespace mortar {

static_assert(kRecordGroupBytes == 32 * FxRecord::kWords * 8, "record size");

namespace {

struct PairCounters {
  unsigned long long nonempty = 0, gp = 0, cells = 0, newton_fail = 0, xi_oor = 0, clip_over = 0;
  __device__ __forceinline__ void add(DevStatus* st) const {
    block_count_add(&st->nonempty, nonempty);
    block_count_add(&st->gauss_points, gp);
    block_count_add(&st->cells, cells);
    block_count_add(&st->newton_fail, newton_fail);
    block_count_add(&st->xi_oor, xi_oor);
    block_count_add(&st->clip_overflow, clip_over);
  }
};

// Writes M = A G (and D = A H) for pair p.
template <int NS, int NM, bool SEG>
__device__ __forceinline__ void write_blocks(int64_t p, const double* __restrict__ r, const double G[4][4],
                                             const double H[4][4], bool dual, double* __restrict__ Mblk,
                                             double* __restrict__ Dblk) {
  double* mo = Mblk + 16 * p;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      double v = 0.0;
      if (a < NS && l < NM) {
        if (dual) {
#pragma unroll
          for (int c = 0; c < NS; ++c) v += r[SR_A + 4 * a + c] * G[c][l];
        } else {
          v = G[a][l];
        }
      }
      mo[4 * a + l] = v;
    }
  if (SEG) {
    double* dout = Dblk + 16 * p;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        double v = 0.0;
        if (a < NS && b < NS) {
          if (dual) {
#pragma unroll
            for (int c = 0; c < NS; ++c) v += r[SR_A + 4 * a + c] * H[c][b];
          } else {
            v = H[a][b];
          }
        }
        dout[4 * a + b] = v;
      }
  }
}

__device__ __forceinline__ void write_zero_blocks(int64_t p, bool seg, double* __restrict__ Mblk,
                                                  double* __restrict__ Dblk) {
  double2* mo = reinterpret_cast<double2*>(Mblk + 16 * p);
#pragma unroll
  for (int k = 0; k < 8; ++k) mo[k] = make_double2(0.0, 0.0);
  if (seg) {
    double2* dout = reinterpret_cast<double2*>(Dblk + 16 * p);
#pragma unroll
    for (int k = 0; k < 8; ++k) dout[k] = make_double2(0.0, 0.0);
  }
}

// ---------------------------------------------------------------- variant 1
template <int NS, int NM, bool SEG>
__device__ __forceinline__ void integrate_one(int64_t p, const int32_t* __restrict__ ps,
                                              const int32_t* __restrict__ pm, const double* __restrict__ srec,
                                              const double* __restrict__ xm, const int32_t* __restrict__ conn_m,
                                              const RunParams& rp, double* __restrict__ Mblk,
                                              double* __restrict__ Dblk, uint8_t* __restrict__ flag,
                                              PairCounters& ctr) {
  const int32_t s = ps[p], m = pm[p];
  const double* r = srec + (int64_t)SR_STRIDE * s;
  double G[4][4], H[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) { G[a][b] = 0.0; H[a][b] = 0.0; }
  PlaneMap mmap;
  double Pu[kMaxPoly], Pv[kMaxPoly];
  const int nr = clip_polygon<NS, NM, kMaxPoly>(r, xm, conn_m, m, mmap, Pu, Pv, ctr.clip_over);
  if (nr == 0) {
    write_zero_blocks(p, SEG, Mblk, Dblk);
    flag[p] = 0;
    return;
  }
  PlaneMap smap;
  smap.c0u = r[SR_C + 0]; smap.c0v = r[SR_C + 1]; smap.c1u = r[SR_C + 2]; smap.c1v = r[SR_C + 3];
  smap.c2u = r[SR_C + 4]; smap.c2v = r[SR_C + 5]; smap.c3u = r[SR_C + 6]; smap.c3v = r[SR_C + 7];
  double cu, cv;
  int ncell;
  if (nr == 3) {
    ncell = 1;
    cu = Pu[0]; cv = Pv[0];
  } else {
    ncell = nr;
    double su = 0.0, sv = 0.0;
    for (int k = 0; k < nr; ++k) { su += Pu[k]; sv += Pv[k]; }
    cu = su / (double)nr;
    cv = sv / (double)nr;
  }
  ctr.cells += ncell;
  ctr.nonempty++;
  for (int cI = 0; cI < ncell; ++cI) {
    double au, av, bu, bv, wu, wv;
    if (nr == 3) {
      au = Pu[0]; av = Pv[0]; bu = Pu[1]; bv = Pv[1]; wu = Pu[2]; wv = Pv[2];
    } else {
      const int k1 = cI + 1 == nr ? 0 : cI + 1;
      au = cu; av = cv; bu = Pu[cI]; bv = Pv[cI]; wu = Pu[k1]; wv = Pv[k1];
    }
    const double e1u = bu - au, e1v = bv - av, e2u = wu - au, e2v = wv - av;
    const double area = 0.5 * fabs(cross2(e1u, e1v, e2u, e2v));
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
      if (xi_out_of_range<NS>(xs1, xs2)) ctr.xi_oor++;
      if (xi_out_of_range<NM>(xm1, xm2)) ctr.xi_oor++;
      double Ns[4], Nm[4];
      shape_fn<NS>(xs1, xs2, Ns);
      shape_fn<NM>(xm1, xm2, Nm);
#pragma unroll
      for (int a = 0; a < NS; ++a) {
        const double wn = W * Ns[a];
#pragma unroll
        for (int l = 0; l < NM; ++l) G[a][l] += wn * Nm[l];
        if (SEG) {
#pragma unroll
          for (int b = 0; b < NS; ++b) H[a][b] += wn * Ns[b];
        }
      }
      ctr.gp++;
    }
  }
  write_blocks<NS, NM, SEG>(p, r, G, H, rp.lm == 1, Mblk, Dblk);
  flag[p] = 1;
}

template <int NS, int NM, bool SEG>
__global__ void __launch_bounds__(kMaxPairBlock) k_integrate(const int32_t* __restrict__ ps, const int32_t* __restrict__ pm,
                                                   const double* __restrict__ srec, const double* __restrict__ xm,
                                                   const int32_t* __restrict__ conn_m, RunParams rp,
                                                   double* __restrict__ Mblk, double* __restrict__ Dblk,
                                                   uint8_t* __restrict__ flag, int64_t pair_cap, int32_t chunk,
                                                   DevStatus* st) {
  PairCounters ctr;
  const int lane = threadIdx.x & 31;
  const bool ok = st->over_pairs == 0 && st->over_bins == 0;
  const int64_t n = ok ? (int64_t)min((unsigned long long)pair_cap, st->n_pairs) : 0;
  const Watchdog wd(rp.watchdog_us);
  // bounded work loop: the counter only grows, so at most n / chunk fetches succeed
  for (;;) {
    if (wd.expired(&st->timeout)) break;
    int64_t base = 0;
    if (lane == 0) base = (int64_t)atomicAdd(&st->work_ctr, (unsigned long long)chunk);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= n) break;
    const int64_t end = min(base + (int64_t)chunk, n);
    for (int64_t p = base + lane; p < end; p += 32)
      integrate_one<NS, NM, SEG>(p, ps, pm, srec, xm, conn_m, rp, Mblk, Dblk, flag, ctr);
  }
  ctr.add(st);
}

// ---------------------------------------------------------------- variant 0
constexpr int kQuadThreads = 128;   // of the quadrature kernel's blocks
// shared memory per thread: a cell's seven back-projections [and, SEG, its sums apart from them]
template <bool SEG>
constexpr int kPtsBytes = (SEG ? 52 : 28) * 8;

// The clip polygon (pu, pv, nr vertices) of pair p in FP64, for pairs whose
// geometry does not fit the fixed-point frame: the 7-point rule on the centroid
// fan with the map inversions of MapInverse.
template <int NS, int NM, bool SEG>
__device__ __forceinline__ void polygon_fp64(int64_t p, const double* __restrict__ r, const PlaneMap& mmap,
                                             const double* pu, const double* pv, int nr, const RunParams& rp,
                                             double* __restrict__ Mblk, double* __restrict__ Dblk,
                                             uint8_t* __restrict__ flag, PairCounters& ctr) {
  MapInverse mi;
  mi.setup(mmap, NM == 3 || map_is_affine(mmap));
  MapInverse si;
  {
    PlaneMap smap;
    smap.c0u = r[SR_C + 0]; smap.c0v = r[SR_C + 1]; smap.c1u = r[SR_C + 2]; smap.c1v = r[SR_C + 3];
    smap.c2u = r[SR_C + 4]; smap.c2v = r[SR_C + 5]; smap.c3u = r[SR_C + 6]; smap.c3v = r[SR_C + 7];
    if (r[SR_AFF] != 0.0) {
      si.m = smap;
      si.affine = true;
      si.i00 = r[SR_BINV]; si.i01 = r[SR_BINV + 1]; si.i10 = r[SR_BINV + 2]; si.i11 = r[SR_BINV + 3];
    } else {
      si.setup(smap, false);
    }
  }
  double G[4][4], H[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) { G[a][b] = 0.0; H[a][b] = 0.0; }
  const int ncell = nr == 3 ? 1 : nr;
  double cu = pu[0], cv = pv[0];
  if (nr > 3) {
    double su = 0.0, sv = 0.0;
    for (int k = 0; k < nr; ++k) { su += pu[k]; sv += pv[k]; }
    cu = su * kInvCount[nr];
    cv = sv * kInvCount[nr];
  }
  ctr.cells += ncell;
  ctr.nonempty++;
  // the quad4 factors 1/4 of both sides are folded into the weight
  constexpr double km = NM == 4 ? 0.25 : 1.0;
  constexpr double kw = km * (NS == 4 ? 0.25 : 1.0);
  for (int cI = 0; cI < ncell; ++cI) {
    const int ib = nr == 3 ? 1 : cI;
    const int iw = nr == 3 ? 2 : (cI + 1 == nr ? 0 : cI + 1);
    const double e1u = pu[ib] - cu, e1v = pv[ib] - cv, e2u = pu[iw] - cu, e2v = pv[iw] - cv;
    const double area = 0.5 * fabs(cross2(e1u, e1v, e2u, e2v));
#pragma unroll 1
    for (int q = 0; q < 7; ++q) {
      double l1, l2, w;
      tri7_point(q, l1, l2, w);
      const double xu = cu + l1 * e1u + l2 * e2u;
      const double xv = cv + l1 * e1v + l2 * e2v;
      double xs1, xs2, xm1, xm2;
      if (!si.solve(xu, xv, xs1, xs2)) ctr.newton_fail++;
      if (!mi.solve(xu, xv, xm1, xm2)) ctr.newton_fail++;
      const double wk = kw * (w * area);
      double Ns[4], Nm[4];   // Ns = (kw W) N_s / ks, Nm = N_m / km
      if constexpr (NS == 4) {   // (1 -+ xi)(1 -+ eta) products as FMAs
        const double qa = fma(-wk, xs1, wk), qb = fma(wk, xs1, wk);
        Ns[0] = fma(-qa, xs2, qa); Ns[1] = fma(-qb, xs2, qb); Ns[2] = fma(qb, xs2, qb); Ns[3] = fma(qa, xs2, qa);
      } else {
        Ns[1] = wk * xs1; Ns[2] = wk * xs2; Ns[0] = wk - Ns[1] - Ns[2]; Ns[3] = 0.0;
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
        for (int l = 0; l < NM; ++l) G[a][l] = fma(Ns[a], Nm[l], G[a][l]);
      if (SEG) {   // H = sum W N_s N_s^T = sum Ns (N_s / km)
        double Nu[4];
        if constexpr (NS == 4 && NM == 4) {
          const double a = 1.0 - xs1, b = 1.0 + xs1;
          Nu[0] = fma(-a, xs2, a); Nu[1] = fma(-b, xs2, b); Nu[2] = fma(b, xs2, b); Nu[3] = fma(a, xs2, a);
        } else {
          shape_fn<NS>(xs1, xs2, Nu);
          if (NM == 4)
            for (int b = 0; b < NS; ++b) Nu[b] *= 4.0;
        }
#pragma unroll
        for (int a = 0; a < NS; ++a)
#pragma unroll
          for (int b = 0; b < NS; ++b) H[a][b] = fma(Ns[a], Nu[b], H[a][b]);
      }
      ctr.gp++;
    }
  }
  write_blocks<NS, NM, SEG>(p, r, G, H, rp.lm == 1, Mblk, Dblk);
  flag[p] = 1;
}

template <int NS, int NM, bool SEG>
__device__ __noinline__ void integrate_polygon_fp64(int64_t p, const double* __restrict__ r, const PlaneMap& mmap,
                                                    const double* __restrict__ pu, const double* __restrict__ pv, int nr,
                                                    const RunParams& rp, double* __restrict__ Mblk,
                                                    double* __restrict__ Dblk, uint8_t* __restrict__ flag,
                                                    PairCounters& ctr) {
  polygon_fp64<NS, NM, SEG>(p, r, mmap, pu, pv, nr, rp, Mblk, Dblk, flag, ctr);
}

// One pair in FP64 from its clip on (pairs that the cell kernel hands back; in
// the one-kernel form, whose code is short of room, all of them).
template <int NS, int NM, bool SEG>
__device__ __noinline__ void integrate_pair_fp64(int64_t p, const int32_t* __restrict__ ps,
                                                 const int32_t* __restrict__ pm, const double* __restrict__ srec,
                                                 const double* __restrict__ xm, const int32_t* __restrict__ conn_m,
                                                 const RunParams& rp, double* __restrict__ Mblk,
                                                 double* __restrict__ Dblk, uint8_t* __restrict__ flag,
                                                 PairCounters& ctr) {
  const double* r = srec + (int64_t)SR_STRIDE * ps[p];
  PlaneMap mmap;
  double pu[kPolyS], pv[kPolyS];
  const int nr = clip_polygon_pool<NS, NM, kPolyS>(r, xm, conn_m, pm[p], mmap, pu, pv, ctr.clip_over);
  if (nr > 0) {
    polygon_fp64<NS, NM, SEG>(p, r, mmap, pu, pv, nr, rp, Mblk, Dblk, flag, ctr);
  } else {
    write_zero_blocks(p, SEG, Mblk, Dblk);
    flag[p] = 0;
  }
}

// FP64 clip of pair p, and its record at o (word w at o[32 w]).  Empty pairs
// get zero blocks; pairs that do not fit the fixed-point frame are integrated
// in FP64 here.  Either way the record says that no cells are left.
// AGAIN: such pairs are clipped again rather than their polygon passed on.
template <int NS, int NM, bool SEG, bool AGAIN>
__device__ __forceinline__ void clip_record(bool has, int64_t p, const int32_t* __restrict__ ps,
                                            const int32_t* __restrict__ pm, const double* __restrict__ srec,
                                            const double* __restrict__ xm, const int32_t* __restrict__ conn_m,
                                            const RunParams& rp, double* __restrict__ Mblk,
                                            double* __restrict__ Dblk, uint8_t* __restrict__ flag,
                                            long long* __restrict__ o, PairCounters& ctr) {
  bool stored = false;
  if (has) {
    const double* r = srec + (int64_t)SR_STRIDE * ps[p];
    PlaneMap mmap;
    double pu[kPolyS], pv[kPolyS];
    const int nr = clip_polygon_pool<NS, NM, kPolyS>(r, xm, conn_m, pm[p], mmap, pu, pv, ctr.clip_over);
    if (nr == 0) {
      write_zero_blocks(p, SEG, Mblk, Dblk);
      flag[p] = 0;
    } else {
      FxPolygon f;
      stored = f.setup<NS, NM>(r, mmap, pu, pv, nr);
      if (stored) {
        FxRecord::store<NS, NM>(o, f, p);
        ctr.cells += f.ncell;
        ctr.gp += 7 * f.ncell;
        ctr.nonempty++;
      } else if (AGAIN) {
        integrate_pair_fp64<NS, NM, SEG>(p, ps, pm, srec, xm, conn_m, rp, Mblk, Dblk, flag, ctr);
      } else {
        integrate_polygon_fp64<NS, NM, SEG>(p, r, mmap, pu, pv, nr, rp, Mblk, Dblk, flag, ctr);
      }
    }
  }
  if (!stored) o[32 * FxRecord::kInfo] = 0;   // nr = 0
}

// One cell of a record (at o, where this lane has one) per lane of the warp:
// the cell's back-projections, then its products, then the pair's sums through
// shared memory, and the pair's blocks.  STRIDE: the block's threads; pts:
// this thread's slice of kPtsBytes.
template <int NS, int NM, bool SEG, int STRIDE>
__device__ __forceinline__ void integrate_cells(const CellSlot& cs, const long long* o,
                                                const int32_t* __restrict__ ps, const int32_t* __restrict__ pm,
                                                const double* __restrict__ srec, const double* __restrict__ xm,
                                                const int32_t* __restrict__ conn_m, const RunParams& rp,
                                                double* __restrict__ Mblk, double* __restrict__ Dblk,
                                                uint8_t* __restrict__ flag, long long* __restrict__ pts,
                                                PairCounters& slow) {
  bool ok = cs.cell >= 0;
  int64_t p = 0;
  int32_t m = 0;
  const double* r = srec;
  FxScales ss, sm;
  int ke = 0;
  long long weight = 0;
  if (ok) {
    FxView f;
    f.load<NS, NM>(o);
    p = o[32 * FxRecord::kPair];
    r = srec + (int64_t)SR_STRIDE * ps[p];
    m = pm[p];
    weight = f.weight(cs.cell);
    ss = f.ss;
    sm = f.sm;
    ke = f.ke;
    ok = fx_back_project<NS, NM, STRIDE>(f, cs.cell, r, xm, conn_m, m, pts);
  }
  const unsigned bad = __ballot_sync(0xffffffffu, cs.cell >= 0 && !ok);
  const bool slow_pair = cs.cell >= 0 && (bad >> cs.first & ((1u << cs.cells) - 1u)) != 0;
  ok &= !slow_pair;
  FxAcc g[4][4];
  if (SEG) {   // the sums' memory is apart from the points', which M's products read again
    fx_cell_products<NS, NS, true, STRIDE>(ss, ss, weight, pts, g);
    write_block<NS, NS, STRIDE>(g, cs, ok, ke, ss, ss, rp.lm == 1, r, Dblk + 16 * p, pts + 28 * STRIDE);
  }
  fx_cell_products<NS, NM, false, STRIDE>(ss, sm, weight, pts, g);
  write_block<NS, NM, STRIDE>(g, cs, ok, ke, ss, sm, rp.lm == 1, r, Mblk + 16 * p, SEG ? pts + 28 * STRIDE : pts);
  if (cs.cell == 0) {
    if (ok) flag[p] = 1;
    else integrate_pair_fp64<NS, NM, SEG>(p, ps, pm, srec, xm, conn_m, rp, Mblk, Dblk, flag, slow);
  }
  __syncwarp();
}

// -------------------------------------------------------- one-kernel form
// For callers without workspace: records live in shared memory, one group of
// pairs per warp and turn.  Small pair lists are latency-bound (14,400 pairs
// fill 3 of 16 warps of a scheduler at 8 pairs a warp), so a group is as small
// as spreads the list over all warps, 8 pairs (about a warp full of cells) to 32.
// 14,400 pairs of quad4 elements through the no-allocation entry point: 251 us a
// call with the former FP64 kernel (one pair per lane, all of it in one round
// of 450 warps), 158 us with this one.
constexpr int kFusedThreads = 128;
template <bool SEG>
constexpr size_t kFusedSmem = (size_t)kFusedThreads * (kPtsBytes<SEG> + FxRecord::kWords * 8);
template <int NS, int NM, bool SEG>
__global__ void __launch_bounds__(kFusedThreads, 3) k_integrate_fused(
    const int32_t* __restrict__ ps, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, RunParams rp, double* __restrict__ Mblk,
    double* __restrict__ Dblk, uint8_t* __restrict__ flag, int64_t pair_cap, DevStatus* st,
    unsigned long long* cta_t) {
  cta_mark(cta_t, 0);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  long long* pts = reinterpret_cast<long long*>(smem_raw) + threadIdx.x;
  long long* rec = reinterpret_cast<long long*>(smem_raw) + kFusedThreads * (kPtsBytes<SEG> / 8) +
                   warp * (32 * FxRecord::kWords);
  PairCounters ctr, slow;
  const int64_t n = chunk_pairs(st, pair_cap, 0, pair_cap);
  const int64_t warps = (int64_t)gridDim.x * (kFusedThreads / 32);
  const int turn = (int)max((int64_t)8, min((int64_t)32, (n + warps - 1) / warps));
  const Watchdog wd(rp.watchdog_us);
  for (;;) {   // bounded: the shared counter only grows
    if (wd.expired(&st->timeout)) break;
    unsigned long long g0 = 0;
    if (lane == 0) g0 = atomicAdd(&st->work_ctr, (unsigned long long)turn);
    const int64_t p0 = (int64_t)__shfl_sync(0xffffffffu, g0, 0);
    if (p0 >= n) break;
    const int pairs = (int)min((int64_t)turn, n - p0);
    clip_record<NS, NM, SEG, true>(lane < pairs, p0 + lane, ps, pm, srec, xm, conn_m, rp, Mblk, Dblk, flag, rec + lane, ctr);
    __syncwarp();
    for (int w = 0; w < pairs;) {
      int ncell = 0;
      if (w + lane < pairs) ncell = record_cells(rec[32 * FxRecord::kInfo + w + lane]);
      const CellSlot cs = assign_cells(ncell);
      const long long* o = rec + w + cs.rec;
      w += cs.taken;
      integrate_cells<NS, NM, SEG, kFusedThreads>(cs, o, ps, pm, srec, xm, conn_m, rp, Mblk, Dblk, flag, pts, slow);
    }
    __syncwarp();
  }
  ctr.newton_fail += slow.newton_fail;   // slow pairs' cells and points were counted with their records
  ctr.xi_oor += slow.xi_oor;
  ctr.add(st);
  __syncthreads();
  cta_mark(cta_t, 1);
}

// ------------------------------------------- three-kernel form (default)
// Split where the work's character changes: a sort kernel
// (FP32 keys, k_pair_sort), a clip kernel (FP64 clip, and the polygon's
// conversion to fixed point) that leaves one record per pair in sorted order,
// and a quadrature kernel on the integer pipe.  One kernel with all of it does
// not fit the instruction cache (about 2,300 instructions run at full rate,
// measured with straight-line loops; IPC 0.75 -> 0.35 beyond that): its warps,
// each in another phase, issued 0.24 instructions per scheduler and clock at 8
// and at 16 warps per SM alike.
template <int NS, int NM, bool SEG>
__global__ void __launch_bounds__(kMaxPairBlock, 2) k_pair_clip(
    const int32_t* __restrict__ ps, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, RunParams rp, double* __restrict__ Mblk,
    double* __restrict__ Dblk, uint8_t* __restrict__ flag, int64_t pair_cap, int64_t first, const int32_t* __restrict__ order,
    long long* __restrict__ rec, DevStatus* st, unsigned long long* cta_t) {
  cta_mark(cta_t, 0);
  const int lane = threadIdx.x & 31;
  PairCounters ctr;
  const int64_t n = chunk_pairs(st, pair_cap, first, kPairChunk);
  const Watchdog wd(rp.watchdog_us);
  for (;;) {   // bounded: the shared counter only grows; one group of 32 pairs per turn
    if (wd.expired(&st->timeout)) break;
    unsigned long long g = 0;
    if (lane == 0) g = atomicAdd(&st->pair_ctr[1], 1ull);
    g = __shfl_sync(0xffffffffu, g, 0);
    const int64_t i = 32 * (int64_t)g + lane;
    if (32 * (int64_t)g >= n) break;
    clip_record<NS, NM, SEG, false>(i < n, i < n ? first + order[i] : 0, ps, pm, srec, xm, conn_m, rp, Mblk, Dblk, flag,
                             rec + (int64_t)g * (32 * FxRecord::kWords) + lane, ctr);
    __syncwarp();
  }
  ctr.add(st);
  __syncthreads();
  cta_mark(cta_t, 1);
}

// Quadrature of the clip kernel's records, one cell of a pair per lane (all
// cells cost the same, so lanes idle only at the ends of warps).
template <int NS, int NM, bool SEG>
__global__ void __launch_bounds__(kQuadThreads, 4) k_pair_quadrature(
    const int32_t* __restrict__ ps, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, RunParams rp, double* __restrict__ Mblk,
    double* __restrict__ Dblk, uint8_t* __restrict__ flag, int64_t pair_cap, int64_t first,
    const long long* __restrict__ rec, DevStatus* st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pts = reinterpret_cast<long long*>(smem_raw) + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const int64_t n = chunk_pairs(st, pair_cap, first, kPairChunk);
  const int turn = cell_turn(n);
  const Watchdog wd(rp.watchdog_us);
  PairCounters slow;
  for (;;) {   // bounded: the shared counter only grows
    if (wd.expired(&st->timeout)) break;
    unsigned long long g0 = 0;
    if (lane == 0) g0 = atomicAdd(&st->pair_ctr[2], (unsigned long long)turn);
    const int64_t r0 = (int64_t)__shfl_sync(0xffffffffu, g0, 0);
    if (r0 >= n) break;
    const int records = (int)min((int64_t)turn, n - r0);
    for (int w = 0; w < records;) {
      int ncell = 0;
      if (w + lane < records) {
        const int64_t i = r0 + w + lane;
        ncell = record_cells(rec[((i >> 5) * FxRecord::kWords + FxRecord::kInfo) * 32 + (i & 31)]);
      }
      if (!__any_sync(0xffffffffu, ncell > 0)) {   // empty pairs, or pairs done in FP64
        w += 32;
        continue;
      }
      const CellSlot cs = assign_cells(ncell);
      const int64_t i = r0 + w + cs.rec;
      w += cs.taken;
      integrate_cells<NS, NM, SEG, kQuadThreads>(cs, rec + (i >> 5) * (32 * FxRecord::kWords) + (i & 31), ps, pm, srec,
                                                 xm, conn_m, rp, Mblk, Dblk, flag, pts, slow);
    }
  }
  // pairs, cells and points were counted by the clip kernel
  block_count_add(&st->newton_fail, slow.newton_fail);
  block_count_add(&st->xi_oor, slow.xi_oor);
}

#ifdef MORTAR_PAIR_NS
template <int NS, int NM, bool SEG>
void launch_split(const IntegrateArgs& a, const RunParams& rp, int n_sm, int rounds, int warps) {
  auto clip = k_pair_clip<NS, NM, SEG>;
  auto quad = k_pair_quadrature<NS, NM, SEG>;
  const size_t shq = (size_t)kQuadThreads * kPtsBytes<SEG>;
  cudaFuncSetAttribute(quad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shq);
  int clip_sm = 0, quad_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&clip_sm, clip, warps * 32, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&quad_sm, quad, kQuadThreads, shq);
  const unsigned gc = (unsigned)(n_sm * (clip_sm < 1 ? 1 : clip_sm)), gq = (unsigned)(n_sm * (quad_sm < 1 ? 1 : quad_sm));
  if (a.grid_out) *a.grid_out = (int)gc;
  for (int64_t first = 0; first < a.pair_cap; first += kPairChunk) {
    launch_pair_sort<NS, NM>(a, rp, n_sm, 32 * rounds, first);
    clip<<<gc, warps * 32, 0, a.stream>>>(a.ps, a.pm, a.srec, a.xm, a.conn_m, rp, a.Mblk, a.Dblk, a.flag, a.pair_cap,
                                          first, a.order, a.rec, a.st,
                                          first == 0 ? a.cta_t : nullptr);   // a full chunk's balance
    quad<<<gq, kQuadThreads, shq, a.stream>>>(a.ps, a.pm, a.srec, a.xm, a.conn_m, rp, a.Mblk, a.Dblk, a.flag,
                                            a.pair_cap, first, a.rec, a.st);
  }
}

template <int NS, int NM, bool SEG>
void launch_fused(const IntegrateArgs& a, const RunParams& rp, int n_sm) {
  auto kern = k_integrate_fused<NS, NM, SEG>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmem<SEG>);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kFusedThreads, kFusedSmem<SEG>);
  const unsigned grid = (unsigned)(n_sm * (per_sm < 1 ? 1 : per_sm));
  if (a.grid_out) *a.grid_out = (int)grid;
  kern<<<grid, kFusedThreads, kFusedSmem<SEG>, a.stream>>>(a.ps, a.pm, a.srec, a.xm, a.conn_m, rp, a.Mblk, a.Dblk,
                                                           a.flag, a.pair_cap, a.st, a.cta_t);
}

template <int NS, int NM, bool SEG>
void launch_one_pair_per_thread(const IntegrateArgs& a, const RunParams& rp, int n_sm, int block, int chunk) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_integrate<NS, NM, SEG>, block, 0);
  if (per_sm < 1) per_sm = 1;
  const unsigned grid = (unsigned)(n_sm * per_sm);
  k_integrate<NS, NM, SEG><<<grid, block, 0, a.stream>>>(a.ps, a.pm, a.srec, a.xm, a.conn_m, rp, a.Mblk, a.Dblk,
                                                         a.flag, a.pair_cap, chunk, a.st);
}

}  // namespace

template <int NS, int NM>
void integrate_nsnm(const IntegrateArgs& a, const RunParams& rp, int n_sm, int variant, int block, int chunk,
                    int rounds) {
  const bool seg = rp.d_domain == 1;
  if (variant == 1) {
    if (seg) launch_one_pair_per_thread<NS, NM, true>(a, rp, n_sm, block, chunk);
    else launch_one_pair_per_thread<NS, NM, false>(a, rp, n_sm, block, chunk);
    return;
  }
  if (a.rec) {
    if (seg) launch_split<NS, NM, true>(a, rp, n_sm, rounds, block / 32);
    else launch_split<NS, NM, false>(a, rp, n_sm, rounds, block / 32);
    return;
  }
  if (seg) launch_fused<NS, NM, true>(a, rp, n_sm);
  else launch_fused<NS, NM, false>(a, rp, n_sm);
}
template void integrate_nsnm<MORTAR_PAIR_NS, MORTAR_PAIR_NM>(const IntegrateArgs&, const RunParams&, int, int, int,
                                                              int, int);
#else   // the main part: dispatch

void launch_dispatch(const IntegrateArgs& a, const RunParams& rp, int nen_s, int nen_m, int n_sm, int variant,
                     int block, int chunk, int rounds) {
  if (nen_s == 4 && nen_m == 4) integrate_nsnm<4, 4>(a, rp, n_sm, variant, block, chunk, rounds);
  else if (nen_s == 4 && nen_m == 3) integrate_nsnm<4, 3>(a, rp, n_sm, variant, block, chunk, rounds);
  else if (nen_s == 3 && nen_m == 4) integrate_nsnm<3, 4>(a, rp, n_sm, variant, block, chunk, rounds);
  else integrate_nsnm<3, 3>(a, rp, n_sm, variant, block, chunk, rounds);
}

}  // namespace

bool integrate_batched_fits(int rounds, int block) {
  return block >= 32 && block <= kMaxPairBlock &&
         (size_t)(kSortThreads / 32) * batch_smem_bytes(32 * rounds) <= kMaxDynSmem;
}

void launch_integrate_raw(const IntegrateArgs& a, const RunParams& rp, int nen_s, int nen_m, int n_sm) {
  launch_dispatch(a, rp, nen_s, nen_m, n_sm, 0, 128, 32, 2);
}

void launch_integrate(mortar_ctx* c, const RunParams& rp) {
  if (quadratic_slave(c)) {
    launch_integrate_quadratic(c, rp);
    return;
  }
  if (rp.integration == 1) {
    c->pair_grid = 0;
    launch_integrate_element_based(c, rp);
    return;
  }
  IntegrateArgs a{c->pairs_s.as<int32_t>(), c->pairs_m.as<int32_t>(), c->srec.as<double>(), c->xm.as<double>(),
                  c->conn_m.as<int32_t>(), c->Mblk.as<double>(), c->Dblk.as<double>(), c->flag.as<uint8_t>(),
                  c->pair_cap, c->dstat.as<DevStatus>(), c->stream};
  a.rec = c->rec.as<long long>();
  a.order = c->order.as<int32_t>();
  c->pair_grid = 0;
  if (c->timing && c->cta_t.p) {
    a.cta_t = c->cta_t.as<unsigned long long>();
    a.grid_out = &c->pair_grid;
  }
  const int block = c->block_size > 0 ? c->block_size : 128;
  const int chunk = c->chunk_pairs > 0 ? c->chunk_pairs : 32;
  const int rounds = c->rounds > 0 ? c->rounds : kSortBatch / 32;
  launch_dispatch(a, rp, c->nen_s, c->nen_m, c->n_sm, c->variant, block, chunk, rounds);
}
#endif  // MORTAR_PAIR_NS

}  // namespace mortar
