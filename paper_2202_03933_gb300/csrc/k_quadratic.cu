// Segment-based integration of quadratic slave elements (tri6, quad8; the
// paper's isoparametric discretisation, Eq. AnsatzDiscretization, with
// quadratic shape functions and standard Lagrange multipliers).
//
// The slave surface is integrated on its piecewise flat approximation
// (Sec. 2.3): every quadratic element is split into four linear sub-elements
// (precomputed records 4 s + k: auxiliary plane, window, map), and for a pair
// (s, m) each sub-element runs the body of Algorithm 1 against the master
// element -- project, clip, centroid fan, 7-point rule, back-projection.  A
// quadrature point's sub-element parameters map affinely to the parent's,
// where the quadratic shape functions are evaluated:
//     M_pair[a][l] += W N_a(xi_parent) N_l(xi_m)      (8 x 4 block per pair).
// D is the element-domain integral of the precomputation.
//
// Work unit = (pair, sub-element), u = 4 p + k: the four sub-elements of a
// pair overlap the master element in different cell counts (often none), so
// one pair per lane would leave most lanes idle.  As for linear elements
// (k_integrate.cu), three kernels: the units are sorted by an FP32 clip
// (k_pair_sort), clipped in FP64 and turned into fixed-point records
// (k_quadratic_clip), and integrated on the integer pipe with one cell of a unit
// per lane (k_quadratic_cells).  A last kernel sums the non-empty unit blocks
// of every pair in the fixed order k = 0..3 (bitwise reproducible) into the pair
// block and its flag.  quad8 450x390 (0.71 M pairs, 2.8 M units): 0.43 + 2.06 +
// 4.55 + 0.19 ms against 14.7 ms of one FP64 kernel; the clip is bound by the FP64 pipe
// (most units are empty), the cells by issue over the integer pipes.
#include "clip.cuh"
#include "context.h"
#include "pair_sort.cuh"
#include "quadrature.cuh"
#include "reverse.cuh"
#include "quadratic.cuh"

namespace mortar {

namespace {

constexpr int kQThreads = 128;
constexpr int kQPtsBytes = 52 * 8;   // shared memory per thread: a cell's seven back-projections, and its sums

struct QCounters {
  unsigned long long gp = 0, cells = 0, newton_fail = 0, clip_over = 0;
};

// The clip polygon (Pu, Pv, nr vertices) of unit u in FP64, for units that do
// not fit the fixed-point frame.  Writes the unit's 8 x 4 block and flag.
template <int NP, int NM>
__device__ __noinline__ void integrate_unit_polygon(int64_t u, const double* __restrict__ r, const PlaneMap& mmap,
                                                    const double* __restrict__ Pu, const double* __restrict__ Pv, int nr,
                                                    double* __restrict__ U, uint8_t* __restrict__ uflag,
                                                    QCounters& ctr) {
  const int k = (int)(u & 3);
  double2* out = reinterpret_cast<double2*>(U + 32 * u);
  double Mq[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int l = 0; l < 4; ++l) Mq[a][l] = 0.0;
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
  double cu = Pu[0], cv = Pv[0];
  int ncell = 1;
  if (nr > 3) {
    double su = 0.0, sv = 0.0;
    for (int j = 0; j < nr; ++j) { su += Pu[j]; sv += Pv[j]; }
    cu = su * kInvCount[nr];
    cv = sv * kInvCount[nr];
    ncell = nr;
  }
  ctr.cells += ncell;
  for (int cI = 0; cI < ncell; ++cI) {
    const int ib = nr == 3 ? 1 : cI;
    const int iw = nr == 3 ? 2 : (cI + 1 == nr ? 0 : cI + 1);
    const double e1u = Pu[ib] - cu, e1v = Pv[ib] - cv, e2u = Pu[iw] - cu, e2v = Pv[iw] - cv;
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
      double xp, ep;
      sub_to_parent<NP>(k, xs1, xs2, xp, ep);
      double Np[8], WNm[4];   // W folded into the master side (4 products instead of NP)
      shape_quadratic<NP>(xp, ep, Np);
      if constexpr (NM == 4) {   // 1/4 of the quad4 shape functions folded into W
        const double wq = 0.25 * (w * area);
        const double qa = fma(-wq, xm1, wq), qb = fma(wq, xm1, wq);
        WNm[0] = fma(-qa, xm2, qa); WNm[1] = fma(-qb, xm2, qb); WNm[2] = fma(qb, xm2, qb); WNm[3] = fma(qa, xm2, qa);
      } else {
        const double W = w * area;
        WNm[1] = W * xm1; WNm[2] = W * xm2; WNm[0] = W - WNm[1] - WNm[2]; WNm[3] = 0.0;
      }
#pragma unroll
      for (int a = 0; a < NP; ++a)
#pragma unroll
        for (int l = 0; l < NM; ++l) Mq[a][l] = fma(Np[a], WNm[l], Mq[a][l]);
      ctr.gp++;
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    __stcs(out + 2 * a, make_double2(Mq[a][0], Mq[a][1]));
    __stcs(out + 2 * a + 1, make_double2(Mq[a][2], NM == 4 ? Mq[a][3] : 0.0));
  }
  uflag[u] = 1;
}

// One unit in FP64 from its clip on (units that the cell kernel hands back).
template <int NP, int NM>
__device__ __noinline__ void integrate_unit(int64_t u, const int32_t* __restrict__ ps, const int32_t* __restrict__ pm,
                                            const double* __restrict__ srec, const double* __restrict__ xm,
                                            const int32_t* __restrict__ conn_m, double* __restrict__ U,
                                            uint8_t* __restrict__ uflag, QCounters& ctr) {
  const int64_t p = u >> 2;
  const double* r = srec + (int64_t)SR_STRIDE * (4 * (int64_t)ps[p] + (u & 3));
  PlaneMap mmap;
  double Pu[kPolyS], Pv[kPolyS];
  const int nr = clip_polygon_pool<NP == 8 ? 4 : 3, NM, kPolyS>(r, xm, conn_m, pm[p], mmap, Pu, Pv, ctr.clip_over);
  if (nr > 0) integrate_unit_polygon<NP, NM>(u, r, mmap, Pu, Pv, nr, U, uflag, ctr);
  else uflag[u] = 0;
}

// Half of a quadratic element's shape functions in Q61 (HALF 0: corners, 1:
// mid-sides) at the parent point of sub-element k's (xi, eta) (Q61).  quad8
// with A, B = 1 -+ xi_p, C, D = 1 -+ eta_p:
//   corners (AC (A + C - 3), BC (B + C - 3), BD (B + D - 3), AD (A + D - 3)) / 4,
//   mid-sides (AB C, CD B, AB D, CD A) / 2.
template <int NP, int HALF>
__device__ __forceinline__ void fx_shape_quadratic(int k, long long xi, long long eta, Dg* N) {
  FxAcc p;
  const long long one = 1ll << 61;
  if constexpr (NP == 8) {
    const long long xp = (xi + (k == 1 || k == 2 ? one : -one)) >> 1, ep = (eta + (k >= 2 ? one : -one)) >> 1;
    const long long A = one - xp, B = one + xp, C = one - ep, D = one + ep;
    const Dg a = fx_split(A), b = fx_split(B), c = fx_split(C), d = fx_split(D);
    if (HALF == 0) {
      auto corner = [&](Dg u, Dg v, long long s) {
        p.mul(u, v);
        const Dg uv = fx_split(p.get<2>());   // Q60, at most 4
        p.mul(uv, fx_split(s - 3 * one));
        return fx_split(p.get<2>());
      };
      N[0] = corner(a, c, A + C);
      N[1] = corner(b, c, B + C);
      N[2] = corner(b, d, B + D);
      N[3] = corner(a, d, A + D);
    } else {
      p.mul(a, b);
      const Dg ab = fx_split(p.get<3>());   // at most 1
      p.mul(c, d);
      const Dg cd = fx_split(p.get<3>());
      p.mul(ab, c);
      N[0] = fx_split(p.get<2>());
      p.mul(cd, b);
      N[1] = fx_split(p.get<2>());
      p.mul(ab, d);
      N[2] = fx_split(p.get<2>());
      p.mul(cd, a);
      N[3] = fx_split(p.get<2>());
    }
  } else {
    const long long hx = xi >> 1, he = eta >> 1, half = one >> 1;
    const long long xp = k == 1 ? half + hx : (k == 3 ? half - he : hx);
    const long long ep = k == 2 ? half + he : (k == 3 ? hx + he : he);
    const long long L[3] = {one - xp - ep, xp, ep};
    const Dg l0 = fx_split(L[0]), l1 = fx_split(L[1]), l2 = fx_split(L[2]);
    if (HALF == 0) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        p.mul(i == 0 ? l0 : (i == 1 ? l1 : l2), fx_split(2 * L[i] - one));
        N[i] = fx_split(p.get<3>());
      }
    } else {
      p.mul(l0, l1);
      N[0] = fx_split(p.get<5>());
      p.mul(l1, l2);
      N[1] = fx_split(p.get<5>());
      p.mul(l2, l0);
      N[2] = fx_split(p.get<5>());
    }
  }
}

// Sums over one cell's points of N_p (W N_m)^T for half of the parent's shape
// functions (bounds as in fx_cell_products, with the roles exchanged).
template <int NP, int NM, int HALF, int stride>
__device__ __forceinline__ void fx_cell_quadratic(int k, const FxScales& sm, long long weight,
                                                  const long long* __restrict__ pts, FxAcc g[4][4]) {
  constexpr int NR = NP / 2;
#pragma unroll
  for (int a = 0; a < NR; ++a)
#pragma unroll
    for (int l = 0; l < NM; ++l) g[a][l].zero();
  const Dg om = fx_split(weight);
#pragma unroll 1
  for (int q = 0; q < 7; ++q) {
    Dg Nm[4], Np[4];
    FxAcc a;
    a.mul(om, kTri7Fx.w[q]);
    const Dg W = fx_split(a.get<2>());
    fx_shape<NM>(sm, pts[(4 * q + 2) * stride], pts[(4 * q + 3) * stride], Nm);
#pragma unroll
    for (int l = 0; l < NM; ++l) {
      a.mul(W, Nm[l]);
      Nm[l] = fx_split(a.get<3>());
    }
    fx_shape_quadratic<NP, HALF>(k, pts[(4 * q) * stride], pts[(4 * q + 1) * stride], Np);
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
      for (int l = 0; l < NM; ++l) g[i][l].mac(Nm[l], Np[i]);
  }
}

// Clip of the chunk's units in sorted order, one record each (see k_pair_clip).
template <int NP, int NM>
__global__ void __launch_bounds__(kQThreads, 4) k_quadratic_clip(
    const int32_t* __restrict__ ps, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, RunParams rp, double* __restrict__ U,
    uint8_t* __restrict__ uflag, int64_t pair_cap, int64_t first, const int32_t* __restrict__ order,
    long long* __restrict__ rec, DevStatus* st) {
  constexpr int NSUB = NP == 8 ? 4 : 3;
  const int lane = threadIdx.x & 31;
  QCounters ctr;
  const int64_t n = 4 * chunk_pairs(st, pair_cap, first, kPairChunk / 4);   // units
  const Watchdog wd(rp.watchdog_us);
  for (;;) {   // bounded: the shared counter only grows; one group of 32 units per turn
    if (wd.expired(&st->timeout)) break;
    unsigned long long g = 0;
    if (lane == 0) g = atomicAdd(&st->pair_ctr[1], 1ull);
    g = __shfl_sync(0xffffffffu, g, 0);
    const int64_t i = 32 * (int64_t)g + lane;
    if (32 * (int64_t)g >= n) break;
    long long* o = rec + (int64_t)g * (32 * FxRecord::kWords) + lane;
    bool stored = false;
    int nr = 0;
    int64_t u = 0;
    const double* r = srec;
    PlaneMap mmap;
    double pu[kPolyS], pv[kPolyS];
    if (i < n) {
      u = 4 * first + order[i];
      const int64_t p = u >> 2;
      r = srec + (int64_t)SR_STRIDE * (4 * (int64_t)ps[p] + (u & 3));
      nr = clip_polygon_pool<NSUB, NM, kPolyS>(r, xm, conn_m, pm[p], mmap, pu, pv, ctr.clip_over);
      if (nr == 0) {
        uflag[u] = 0;
      } else {
        FxPolygon f;
        stored = f.setup<NSUB, NM>(r, mmap, pu, pv, nr);
        if (stored) {
          FxRecord::store<NSUB, NM>(o, f, u);
          ctr.cells += f.ncell;
          ctr.gp += 7 * f.ncell;
        }
      }
    }
    __syncwarp();   // lanes leave setup in several places; those for FP64 run together
    if (nr > 0 && !stored) integrate_unit_polygon<NP, NM>(u, r, mmap, pu, pv, nr, U, uflag, ctr);
    if (!stored) o[32 * FxRecord::kInfo] = 0;   // nr = 0: nothing left for the cell kernel
    __syncwarp();
  }
  block_count_add(&st->gauss_points, ctr.gp);
  block_count_add(&st->cells, ctr.cells);
  block_count_add(&st->newton_fail, ctr.newton_fail);
  block_count_add(&st->clip_overflow, ctr.clip_over);
}

// Quadrature of the units' records, one cell per lane (see k_pair_quadrature);
// the corner and the mid-side rows one after the other, so that each pass has
// 16 sums.  Bound by issue over the integer pipes, as for linear elements.
template <int NP, int NM>
__global__ void __launch_bounds__(kQThreads, 4) k_quadratic_cells(
    const int32_t* __restrict__ ps, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, RunParams rp, double* __restrict__ U,
    uint8_t* __restrict__ uflag, int64_t pair_cap, int64_t first, const long long* __restrict__ rec, DevStatus* st) {
  constexpr int NSUB = NP == 8 ? 4 : 3, NR = NP / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* pts = reinterpret_cast<long long*>(smem_raw) + threadIdx.x;
  constexpr int stride = kQThreads;
  const int lane = threadIdx.x & 31;
  const int64_t n = 4 * chunk_pairs(st, pair_cap, first, kPairChunk / 4);
  const int turn = cell_turn(n);
  const Watchdog wd(rp.watchdog_us);
  QCounters slow;
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
      if (!__any_sync(0xffffffffu, ncell > 0)) {   // empty units, or units done in FP64
        w += 32;
        continue;
      }
      const CellSlot cs = assign_cells(ncell);
      const int64_t i = r0 + w + cs.rec;
      w += cs.taken;
      bool ok = cs.cell >= 0;
      int64_t u = 0;
      FxScales sm;
      int ke = 0;
      long long weight = 0;
      if (ok) {
        const long long* o = rec + (i >> 5) * (32 * FxRecord::kWords) + (i & 31);
        FxView f;
        f.load<NSUB, NM>(o);
        u = o[32 * FxRecord::kPair];
        weight = f.weight(cs.cell);
        sm = f.sm;
        ke = f.ke;
        ok = fx_back_project<NSUB, NM, stride>(f, cs.cell, srec + (int64_t)SR_STRIDE * (4 * (int64_t)ps[u >> 2] + (u & 3)), xm,
                                       conn_m, pm[u >> 2], pts);
      }
      const unsigned bad = __ballot_sync(0xffffffffu, cs.cell >= 0 && !ok);
      ok &= !(cs.cell >= 0 && (bad >> cs.first & ((1u << cs.cells) - 1u)) != 0);
      double* out = U + 32 * u;
      auto emit = [&](int a, int l, long long hh, long long cr) {
        __stcs(out + 4 * a + l, fx_to_double(hh, cr, ke - sm.shape<NM>(l)));
      };
      long long* sums = pts + 28 * stride;
      FxAcc g[4][4];
      fx_cell_quadratic<NP, NM, 0, stride>((int)(u & 3), sm, weight, pts, g);
      fx_sum_cells<NR, NM, stride>(g, cs, ok, sums, emit);
      out += 4 * NR;
      fx_cell_quadratic<NP, NM, 1, stride>((int)(u & 3), sm, weight, pts, g);
      fx_sum_cells<NR, NM, stride>(g, cs, ok, sums, emit);
      if (ok && (NP < 8 || NM < 4))   // the block is padded with zeros
        for (int e = cs.cell; e < 32; e += cs.cells)
          if ((e >> 2) >= NP || (e & 3) >= NM) __stcs(U + 32 * u + e, 0.0);
      if (cs.cell == 0) {
        if (ok) uflag[u] = 1;
        else integrate_unit<NP, NM>(u, ps, pm, srec, xm, conn_m, U, uflag, slow);
      }
      __syncwarp();
    }
  }
  // cells and points were counted by the clip kernel
  block_count_add(&st->newton_fail, slow.newton_fail);
}

// Pair block = sum of its non-empty unit blocks in the order k = 0..3; flag = any.
// Sixteen threads per pair, thread j summing the j-th 16-byte pair of entries
// of the four blocks: every load and store of a half-warp is one contiguous
// 256-byte segment.
__global__ void __launch_bounds__(256) k_quadratic_reduce(const double* __restrict__ U,
                                                          const uint8_t* __restrict__ uflag, int64_t pair_cap,
                                                          double* __restrict__ Mblk, uint8_t* __restrict__ flag,
                                                          DevStatus* st) {
  const bool ok = st->over_pairs == 0 && st->over_bins == 0;
  const int64_t n = ok ? (int64_t)min((unsigned long long)pair_cap, st->n_pairs) : 0;
  const int j = threadIdx.x & 15;
  unsigned long long ne = 0;
  for (int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4; p < n;
       p += ((int64_t)gridDim.x * blockDim.x) >> 4) {
    const double2* u0 = reinterpret_cast<const double2*>(U + 128 * p) + j;
    const uint32_t f = *reinterpret_cast<const uint32_t*>(uflag + 4 * p);
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if ((f >> (8 * k) & 0xffu) == 0u) continue;   // an empty unit's block is not written
      const double2 t = __ldcs(u0 + 16 * k);
      acc.x += t.x;
      acc.y += t.y;
    }
    __stcs(reinterpret_cast<double2*>(Mblk + 32 * p) + j, acc);
    if (j == 0) {
      flag[p] = f != 0u ? 1 : 0;
      ne += f != 0u ? 1ull : 0ull;
    }
  }
  block_count_add(&st->nonempty, ne);
}

template <int NP, int NM>
void launch_q(mortar_ctx* c, const RunParams& rp) {
  constexpr int NSUB = NP == 8 ? 4 : 3;
  IntegrateArgs a{c->pairs_s.as<int32_t>(), c->pairs_m.as<int32_t>(), c->srec.as<double>(), c->xm.as<double>(),
                  c->conn_m.as<int32_t>(), nullptr, nullptr, nullptr, c->pair_cap, c->dstat.as<DevStatus>(), c->stream};
  a.order = c->order.as<int32_t>();
  auto clip = k_quadratic_clip<NP, NM>;
  auto cells = k_quadratic_cells<NP, NM>;
  const size_t shm = (size_t)kQThreads * kQPtsBytes;
  cudaFuncSetAttribute(cells, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
  int clip_sm = 0, cell_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&clip_sm, clip, kQThreads, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&cell_sm, cells, kQThreads, shm);
  const unsigned gc = (unsigned)(c->n_sm * (clip_sm < 1 ? 1 : clip_sm)), gq = (unsigned)(c->n_sm * (cell_sm < 1 ? 1 : cell_sm));
  for (int64_t first = 0; first < c->pair_cap; first += kPairChunk / 4) {
    launch_pair_sort<NSUB, NM, 4>(a, rp, c->n_sm, kSortBatch, first);
    clip<<<gc, kQThreads, 0, c->stream>>>(a.ps, a.pm, a.srec, a.xm, a.conn_m, rp, c->Qunit.as<double>(),
                                          c->Qflag.as<uint8_t>(), c->pair_cap, first, a.order, c->rec.as<long long>(),
                                          a.st);
    cells<<<gq, kQThreads, shm, c->stream>>>(a.ps, a.pm, a.srec, a.xm, a.conn_m, rp, c->Qunit.as<double>(),
                                             c->Qflag.as<uint8_t>(), c->pair_cap, first, c->rec.as<long long>(), a.st);
  }
  k_quadratic_reduce<<<(unsigned)(c->n_sm * 8), 256, 0, c->stream>>>(c->Qunit.as<double>(), c->Qflag.as<uint8_t>(),
                                                                     c->pair_cap, c->Mblk.as<double>(),
                                                                     c->flag.as<uint8_t>(), c->dstat.as<DevStatus>());
}

}  // namespace

void launch_integrate_quadratic(mortar_ctx* c, const RunParams& rp) {
  c->pair_grid = 0;
  if (c->nen_s == 8 && c->nen_m == 4) launch_q<8, 4>(c, rp);
  else if (c->nen_s == 8) launch_q<8, 3>(c, rp);
  else if (c->nen_m == 4) launch_q<6, 4>(c, rp);
  else launch_q<6, 3>(c, rp);
}

}  // namespace mortar
