// Element-based integration of the mortar matrices (Sec. 1 and Sec. 2.3 set
// it against the segment-based Algorithm 1: no clipping or triangulation; a
// higher-order rule on the slave element copes with the kinks of the
// integrand at master element edges, at lower accuracy).
//
// One thread per slave element (points outermost, see the kernels).  Rule: n x n
// Gauss-Legendre points on quad4 (collapsed n x n points on tri3), mapped into the element's auxiliary plane
// by the projected slave map, weights w |det J_s|.  The element's candidate
// pairs are visited in pair order; each takes the points not taken yet whose
// back-projection onto its projected master element converges inside it
// (|xi|, |eta| <= 1 + 1e-10 on quad4, barycentric >= -1e-10 on tri3) and adds
//     M_p[a][l] += W Phi_a(xi_s) N_l(xi_m),   D_p[a][b] += W Phi_a N_b(xi_s) (segment D).
// Points no master covers contribute nothing.  Ownership is a bit mask per
// thread.  The blocks keep the layout of the segment-based ones, so the
// assembly is shared.
#include <cmath>
#include <vector>

#include "clip.cuh"
#include "context.h"
#include "quadrature.cuh"

namespace mortar {

namespace {

constexpr int kThreads = 128;
constexpr int kMaxRule = 16;
constexpr double kInsideTol = 1e-10;

constexpr int kChunk = 8;   // candidate pairs held per pass over the points
constexpr int kFixedPairs = 12;   // ... in the fixed-point form
constexpr int kMaxFixedRule = 12;   // n of the largest fixed-point rule (rule_boost)

// One element in FP64, points outermost: for each rule point the
// element's candidate pairs (a chunk of up to kChunk, with their projected
// master maps kept in thread-local memory) are tried in pair order with a box
// reject and the FP32 Newton iterate, and only the owner's FP64 step and the
// point's contribution are computed.  The FP64 work then runs once per point
// on every lane (interior elements own all points), instead of once per
// (pair, point) behind lane-divergent tests.  Contributions are added into
// the owner's block in global memory (this thread's own blocks, L1-resident)
// in point order.  Elements with more than kChunk pairs take further passes
// over the points not yet owned, so "first covering pair in pair order" holds.
// Dual LMs: G = sum W N_s N_m^T in the nodal basis, and A applied once per pair.
template <int NS, int NM, bool SEG, bool DUAL>
__device__ __noinline__ void element_fp64(int64_t e, const int64_t* __restrict__ pair_off,
                                          const int32_t* __restrict__ pm, const double* __restrict__ srec,
                                          const double* __restrict__ xm, const int32_t* __restrict__ conn_m,
                                          const double* __restrict__ rule, int n, double* __restrict__ Mblk,
                                          double* __restrict__ Dblk, uint8_t* __restrict__ flag,
                                          unsigned long long& n_live, unsigned long long& n_gp) {
  const int nq = n * n;
  const int64_t p0 = pair_off[e], p1 = pair_off[e + 1];
  if (p0 == p1) return;
  const double* r = srec + (int64_t)SR_STRIDE * e;
  const bool live = r[SR_EPSIN] >= 0.0;
  PlaneMap smap;
  smap.c0u = r[SR_C + 0]; smap.c0v = r[SR_C + 1]; smap.c1u = r[SR_C + 2]; smap.c1v = r[SR_C + 3];
  smap.c2u = r[SR_C + 4]; smap.c2v = r[SR_C + 5]; smap.c3u = r[SR_C + 6]; smap.c3v = r[SR_C + 7];
  const double x0x = r[SR_X0], x0y = r[SR_X0 + 1], x0z = r[SR_X0 + 2];
  const double t1x = r[SR_T1], t1y = r[SR_T1 + 1], t1z = r[SR_T1 + 2];
  const double t2x = r[SR_T2], t2y = r[SR_T2 + 1], t2z = r[SR_T2 + 2];
  double Phi_c[4][4];   // dual: Phi_a = sum_c A[a][c] N_c
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) Phi_c[a][c] = r[SR_A + 4 * a + c];
  uint32_t taken[kMaxRule * kMaxRule / 32];
#pragma unroll
  for (int k = 0; k < kMaxRule * kMaxRule / 32; ++k) taken[k] = 0u;
  for (int64_t c0 = p0; c0 < p1; c0 += kChunk) {
    const int kc = (int)min((int64_t)kChunk, p1 - c0);
    MapInverse mic[kChunk];
    float box[kChunk][4];
    int got[kChunk];
    for (int k = 0; k < kc; ++k) {
      got[k] = 0;
      const int64_t p = c0 + k;
      double* mo = Mblk + 16 * p;
      for (int t = 0; t < 16; ++t) mo[t] = 0.0;
      if (SEG) {
        double* dout = Dblk + 16 * p;
        for (int t = 0; t < 16; ++t) dout[t] = 0.0;
      }
      const int32_t m = pm[p];
      double mu[4], mv[4];
      double lo_u = 1e300, hi_u = -1e300, lo_v = 1e300, hi_v = -1e300;
#pragma unroll
      for (int l = 0; l < NM; ++l) {
        const int64_t nd = conn_m[(int64_t)NM * m + l];
        const double dx = xm[3 * nd] - x0x, dy = xm[3 * nd + 1] - x0y, dz = xm[3 * nd + 2] - x0z;
        mu[l] = dx * t1x + dy * t1y + dz * t1z;
        mv[l] = dx * t2x + dy * t2y + dz * t2z;
        lo_u = fmin(lo_u, mu[l]); hi_u = fmax(hi_u, mu[l]);
        lo_v = fmin(lo_v, mv[l]); hi_v = fmax(hi_v, mv[l]);
      }
      // box of the projected master element in FP32, widened far beyond the
      // inside tolerance and the FP32 rounding of the test point: a quick reject only
      const double band = 1e-4 * fmax(hi_u - lo_u, hi_v - lo_v);
      box[k][0] = f32_trunc(lo_u - band); box[k][1] = f32_trunc(hi_u + band);
      box[k][2] = f32_trunc(lo_v - band); box[k][3] = f32_trunc(hi_v + band);
      const PlaneMap mmap = plane_map<NM>(mu, mv);
      mic[k].setup(mmap, NM == 3 || map_is_affine(mmap));
    }
    if (live) {
      for (int q = 0; q < nq; ++q) {
        if ((taken[q >> 5] >> (q & 31)) & 1u) continue;
        const int i = q / n, j = q - (q / n) * n;
        double xi, eta, wq;
        if constexpr (NS == 4) {
          xi = rule[i]; eta = rule[j];
          wq = rule[n + i] * rule[n + j];
        } else {
          const double s = 0.5 * (rule[i] + 1.0), tt = 0.5 * (rule[j] + 1.0);
          xi = s; eta = tt * (1.0 - s);
          wq = 0.25 * rule[n + i] * rule[n + j] * (1.0 - s);
        }
        const double xe = xi * eta;
        const double xu = smap.c0u + smap.c1u * xi + smap.c2u * eta + smap.c3u * xe;
        const double xv = smap.c0v + smap.c1v * xi + smap.c2v * eta + smap.c3v * xe;
        const float fu = f32_trunc(xu), fv = f32_trunc(xv);
        // Owner search in two parts: an FP32 scan (box reject, FP32 Newton
        // iterate within 1e-5 of the element) finds the next candidate, then
        // its FP64 step and inside test run for all lanes together; a
        // candidate that fails the FP64 test (a point within 1e-5 of a
        // master edge) resumes the scan after it.  Same owner as testing
        // the candidates one by one in pair order.
        int owner = -1;
        double m1 = 0.0, m2 = 0.0;
        int k = 0;
        while (owner < 0 && k < kc) {
          int kn = -1, mode = 0;   // 1: affine (solved), 2: FP32 iterate near, 3: FP32 did not settle
          double a1 = 0.0, a2 = 0.0;
          CoarseInv ci;
          for (; k < kc; ++k) {
            if (fu < box[k][0] || fu > box[k][1] || fv < box[k][2] || fv > box[k][3]) continue;
            const MapInverse& mk = mic[k];
            if (mk.affine) { mode = 1; kn = k; break; }
            if (mk.coarse(xu, xv, a1, a2, ci)) {   // points clearly outside skip the FP64 step
              const bool near = NM == 4
                  ? (fabs(a1) <= 1.0 + 1e-5 && fabs(a2) <= 1.0 + 1e-5)
                  : (a1 >= -1e-5 && a2 >= -1e-5 && a1 + a2 <= 1.0 + 1e-5);
              if (!near) continue;
              mode = 2;
            } else {
              mode = 3;
            }
            kn = k;
            break;
          }
          if (kn < 0) break;
          k = kn + 1;
          MapInverse& mi = mic[kn];
          if (mode == 1) {
            mi.solve(xu, xv, a1, a2);
          } else if (mode == 2) {
            mi.polish(xu, xv, a1, a2, ci);
          } else if (!mi.newton64(xu, xv, a1, a2)) {   // FP32 did not settle: FP64 Newton from its iterate
            continue;
          }
          const bool inside = NM == 4
              ? (fabs(a1) <= 1.0 + kInsideTol && fabs(a2) <= 1.0 + kInsideTol)
              : (a1 >= -kInsideTol && a2 >= -kInsideTol && a1 + a2 <= 1.0 + kInsideTol);
          if (!inside) continue;
          owner = kn;
          m1 = a1;
          m2 = a2;
        }
        if (owner < 0) continue;
        taken[q >> 5] |= 1u << (q & 31);
        got[owner] += 1;
        const double j00 = smap.c1u + smap.c3u * eta, j01 = smap.c2u + smap.c3u * xi;
        const double j10 = smap.c1v + smap.c3v * eta, j11 = smap.c2v + smap.c3v * xi;
        const double W = wq * fabs(j00 * j11 - j01 * j10);
        double Ns[4], Nm[4], Phi[4];
        shape_fn<NS>(xi, eta, Ns);
        shape_fn<NM>(m1, m2, Nm);
#pragma unroll
        for (int a = 0; a < NS; ++a) Phi[a] = W * Ns[a];
        double* mo = Mblk + 16 * (c0 + owner);
#pragma unroll
        for (int a = 0; a < NS; ++a)
#pragma unroll
          for (int l = 0; l < NM; ++l) mo[4 * a + l] = fma(Phi[a], Nm[l], mo[4 * a + l]);
        if (SEG) {
          double* dout = Dblk + 16 * (c0 + owner);
#pragma unroll
          for (int a = 0; a < NS; ++a)
#pragma unroll
            for (int b = 0; b < NS; ++b) dout[4 * a + b] = fma(Phi[a], Ns[b], dout[4 * a + b]);
        }
      }
      if (DUAL)   // every point of this chunk's pairs is in: M = A G, D = A H
        for (int k = 0; k < kc; ++k) {
          if (got[k] == 0) continue;
          double* mo = Mblk + 16 * (c0 + k);
          double G[4][4];
#pragma unroll
          for (int c = 0; c < NS; ++c)
#pragma unroll
            for (int l = 0; l < NM; ++l) G[c][l] = mo[4 * c + l];
#pragma unroll
          for (int a = 0; a < NS; ++a)
#pragma unroll
            for (int l = 0; l < NM; ++l) {
              double v = 0.0;
#pragma unroll
              for (int c = 0; c < NS; ++c) v = fma(Phi_c[a][c], G[c][l], v);
              mo[4 * a + l] = v;
            }
          if (SEG) {
            double* dout = Dblk + 16 * (c0 + k);
#pragma unroll
            for (int c = 0; c < NS; ++c)
#pragma unroll
              for (int b = 0; b < NS; ++b) G[c][b] = dout[4 * c + b];
#pragma unroll
            for (int a = 0; a < NS; ++a)
#pragma unroll
              for (int b = 0; b < NS; ++b) {
                double v = 0.0;
#pragma unroll
                for (int c = 0; c < NS; ++c) v = fma(Phi_c[a][c], G[c][b], v);
                dout[4 * a + b] = v;
              }
          }
        }
    }
    for (int k = 0; k < kc; ++k) {
      flag[c0 + k] = got[k] > 0 ? 1 : 0;
      n_live += got[k] > 0 ? 1 : 0;
      n_gp += (unsigned long long)got[k];
    }
  }
}

template <int NS, int NM, bool SEG, bool DUAL>
__global__ void __launch_bounds__(kThreads) k_integrate_elembased(
    const int64_t* __restrict__ pair_off, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, const double* __restrict__ rule, int n,
    int64_t Es, double* __restrict__ Mblk, double* __restrict__ Dblk, uint8_t* __restrict__ flag,
    DevStatus* st) {
  unsigned long long n_live = 0, n_gp = 0;
  const bool ok = st->over_pairs == 0 && st->over_bins == 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; ok && e < Es;
       e += (int64_t)gridDim.x * blockDim.x)
    element_fp64<NS, NM, SEG, DUAL>(e, pair_off, pm, srec, xm, conn_m, rule, n, Mblk, Dblk, flag, n_live, n_gp);
  block_count_add(&st->nonempty, n_live);
  block_count_add(&st->gauss_points, n_gp);
}

// ------------------------------------------------------------- fixed point
// The same loop on the integer pipe (fixed.cuh).  Slave side: the rule's
// points xi, eta (Q61) and the products w N_a / sum w (Q62 times 2^boost) are
// a table in shared memory; a point's weight is the table times |det J_s|.
// Master side: the FP32 scan decides for points farther than 1e-5 from an
// element's edge, the fixed-point back-projection (2^-57 in xi) for the others
// with the same 1e-10 tolerance.  The owner's sums stay in registers while
// consecutive points have the same owner, and are exchanged with thread-local
// memory when it changes.  Digits: a product's size goes down to 2^-22 of the
// largest at a rule's corners, so the table, and its products with |det J_s|,
// have a third digit (32 more bits), the products' low terms are kept and a sum
// holds 96 bits: an entry that only such points contribute to has all the bits
// that FP64 gives it.  (Blocks of at most four points, n = 12, parallelograms:
// geometric mean of the largest relative error of an entry 7e-14 with two
// digits, 4e-15 with three, FP64 3e-15.)
// 600x520 quad4, n = 8, dual: 5.95 ms in FP64 (FP64 pipe), 3.2 ms here, of which
// the instructions would take half: the candidates' maps and the exchanged sums
// (about 2 KB a thread) miss L1 in 58 % of their sectors.  Sums added in memory
// point by point: 4.07 ms; without the warp in step: 9.0 ms; 2 or 4 blocks per SM
// instead of 3: 3.6, 3.8 ms.  An element that falls back to FP64 holds up its
// warp: with 8 pairs the most, 275x332 quads (nine pairs here and there) took
// 1.2 times the FP64 form's call, with chunks of 12 0.84 times.
struct ElemCandidate {
  FxMap map;
  int lo_u, hi_u, lo_v, hi_v;   // box in 2^-29 of the frame, widened by 2^-13 of its size
};

__host__ __device__ inline void rule_point(int nen, const double* rule, int n, int q, double& xi, double& eta,
                                           double& w) {
  const int i = q / n, j = q - i * n;
  if (nen == 4) {
    xi = rule[i]; eta = rule[j];
    w = rule[n + i] * rule[n + j];
  } else {
    const double s = 0.5 * (rule[i] + 1.0), t = 0.5 * (rule[j] + 1.0);
    xi = s; eta = t * (1.0 - s);
    w = 0.25 * rule[n + i] * rule[n + j] * (1.0 - s);
  }
}
__host__ __device__ inline double rule_shape(int nen, int a, double xi, double eta) {
  if (nen == 3) return a == 0 ? 1.0 - xi - eta : (a == 1 ? xi : eta);
  return 0.25 * (a == 1 || a == 2 ? 1.0 + xi : 1.0 - xi) * (a < 2 ? 1.0 - eta : 1.0 + eta);
}

// corners of a projected map in 2^-29 of the frame: min and max of one coordinate
template <int NEN>
__device__ __forceinline__ void corner_range(long long c0, Dg c1, Dg c2, Dg c3, int& lo, int& hi) {
  const int a = (int)(c0 >> 33), b = c1.h >> 1, c = c2.h >> 1, d = NEN == 4 ? c3.h >> 1 : 0;
  const int x0 = NEN == 4 ? a - b - c + d : a, x1 = NEN == 4 ? a + b - c - d : a + b;
  const int x2 = NEN == 4 ? a + b + c + d : a + c, x3 = NEN == 4 ? a - b + c - d : a;
  lo = min(min(x0, x1), min(x2, x3));
  hi = max(max(x0, x1), max(x2, x3));
  const int band = ((hi - lo) >> 13) + 4;   // 4: the truncated digits
  lo -= band;
  hi += band;
}

// Exchanges the sums of pair `from` (null: none) for those of pair `to`.
template <int NR, int NC>
__device__ __forceinline__ void exchange(FxAcc g[4][4], FxAcc* __restrict__ from, const FxAcc* __restrict__ to) {
#pragma unroll
  for (int a = 0; a < NR; ++a)
#pragma unroll
    for (int l = 0; l < NC; ++l) {
      if (from) {
        g[a][l].carry();
        from[NC * a + l] = g[a][l];
      }
      g[a][l] = to[NC * a + l];
    }
}
// Three digits: d + x 2^-32 in units of the last place of d, |x| <= 2^31.
struct Dg3 {
  Dg d;
  int x;
};
template <int NR, int NC>
__device__ __forceinline__ void add_products(FxAcc g[4][4], const Dg3* Ns, const Dg* Nc) {
#pragma unroll
  for (int a = 0; a < NR; ++a)
#pragma unroll
    for (int l = 0; l < NC; ++l) {
      g[a][l].mac(Ns[a].d, Nc[l]);
      g[a][l].cr += mul_hi(Ns[a].d.l, Nc[l].l) + mul_hi(Ns[a].x, Nc[l].h);   // below 2^30 + 2^29
    }
}
// t W / 2^61 with t of three digits, W Q61 and at most 1
__device__ __forceinline__ Dg3 weigh(Dg t, int x, Dg W) {
  FxAcc a;
  a.mul(t, W);
  const long long low = mad_wide(x, W.h, mul_wide(t.l, W.l));   // below 2^62 + 2^60
  a.cr += low >> 32;
  const unsigned digit = shift_in((unsigned)low, (unsigned)a.cr, 3);
  return {fx_split(a.get<3>() + (digit >> 31)), (int)digit};
}
// Table entry of the product v = w N_a / sum w (at least 0, below 2^-2): digits of v 2^k, balanced.
__device__ __forceinline__ void put_product(double v, int k, long long& t, int& x) {
  t = fx_of_double(v, k);
  const double up = __longlong_as_double((long long)(1023 + k) << 52);
  const double rest = v * up - (double)t;   // exact: not zero only where t has fewer bits than v
  const unsigned d = (unsigned)(long long)(rest * 0x1p32);
  t += d >> 31;
  x = (int)d;
}
template <int NR, int NC>
__device__ __forceinline__ void carry_all(FxAcc g[4][4]) {
#pragma unroll
  for (int a = 0; a < NR; ++a)
#pragma unroll
    for (int l = 0; l < NC; ++l) g[a][l].carry();
}

// The block of one pair from its sums: G, or A G with dual LMs.
template <int NR, int NC, bool DUAL>
__device__ __forceinline__ void put_block(const FxAcc* __restrict__ acc, int ke, const double* __restrict__ A,
                                          double* __restrict__ out) {
  double G[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int l = 0; l < 4; ++l) G[a][l] = a < NR && l < NC ? fx_to_double(acc[NC * a + l].hh, acc[NC * a + l].cr, ke) : 0.0;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      double v = G[a][l];
      if (DUAL && a < NR && l < NC) {
        v = 0.0;
#pragma unroll
        for (int c = 0; c < NR; ++c) v = fma(A[4 * a + c], G[c][l], v);
      }
      out[4 * a + l] = v;
    }
}

// The table: per point xi, eta, the NS products, and their third digits (two a word).
template <int NS>
constexpr int kTableWords = 2 + NS + (NS + 1) / 2;
template <int NS>
__device__ __forceinline__ void put_point(long long* t, double xi, double eta, double w, int boost) {
  t[0] = fx_of_double(xi, 61);
  t[1] = fx_of_double(eta, 61);
  int* third = reinterpret_cast<int*>(t + 2 + NS);
  for (int a = 0; a < NS; ++a)
    put_product(w * (NS == 4 ? 0.25 : 2.0) * rule_shape(NS, a, xi, eta), 62 + boost, t[2 + a], third[a]);
}

// One element per lane, the warp in step (__syncwarp between the parts, which
// lanes with another owner or candidate would otherwise run one by one).
// Candidate pairs in chunks of kFixedPairs: 12 holds what meshes of about the
// same size have (three by three, four by three), further chunks take the
// points without an owner yet.  False (blocks not final) for a lane whose
// element does not fit: degenerate, or a master whose map is out of range (kMaxMapBits).
// tab: the table (kTableWords).
template <int NS, int NM, bool SEG, bool DUAL>
__device__ __forceinline__ bool element_fixed(bool valid, int64_t e, const int64_t* __restrict__ pair_off,
                                              const int32_t* __restrict__ pm, const double* __restrict__ srec,
                                              const double* __restrict__ xm, const int32_t* __restrict__ conn_m,
                                              const long long* __restrict__ tab, int nq, int boost,
                                              double* __restrict__ Mblk, double* __restrict__ Dblk,
                                              uint8_t* __restrict__ flag, unsigned long long& n_live,
                                              unsigned long long& n_gp) {
  int64_t p0 = 0, p1 = 0;
  const double* r = srec;
  if (valid) {
    p0 = pair_off[e];
    p1 = pair_off[e + 1];
    r = srec + (int64_t)SR_STRIDE * e;
  }
  bool ok = p0 == p1 || r[SR_EPSIN] >= 0.0;
  unsigned taken[(kMaxFixedRule * kMaxFixedRule + 31) / 32];
#pragma unroll
  for (int k = 0; k < (int)(sizeof(taken) / sizeof(taken[0])); ++k) taken[k] = 0u;
  unsigned live = 0, owned = 0;
  const bool more = __any_sync(0xffffffffu, p1 - p0 > kFixedPairs);
  for (; __any_sync(0xffffffffu, ok && p0 < p1); p0 += kFixedPairs) {   // p0 of a finished lane moves on, unused
    int kc = ok ? (int)max((int64_t)0, min(p1 - p0, (int64_t)kFixedPairs)) : 0;
    const PlaneMap smap = kc > 0 ? slave_plane_map(r) : PlaneMap{0.0, 0.0, 1.0, 0.0, 0.0, 1.0, 0.0, 0.0};
    PlaneMap maps[kFixedPairs];
    int Eu = -1000, Ev = -1000;
    for (int k = 0; k < kc; ++k) {
      maps[k] = master_plane_map<NM>(r, xm, conn_m, pm[p0 + k]);
      const FxFrame f = fx_frame<NS, NM>(r, maps[k]);
      Eu = max(Eu, f.Eu);
      Ev = max(Ev, f.Ev);
    }
    __syncwarp();
    // det J_s = d0 + d1 xi + d2 eta, in units of 2^ED (Q61)
    const double f0 = cross2(smap.c1u, smap.c1v, smap.c2u, smap.c2v), f1 = cross2(smap.c1u, smap.c1v, smap.c3u, smap.c3v);
    const double f2 = cross2(smap.c3u, smap.c3v, smap.c2u, smap.c2v);
    const int ED = fx_exponent(fx_hi_abs(fabs(f0) + fabs(f1) + fabs(f2)));
    if (kc > 0 && !(Eu > -200 && Eu < 200 && Ev > -200 && Ev < 200 && ED > -500 && ED < 500)) {
      ok = false;
      kc = 0;
    }
    if (kc == 0) Eu = Ev = 4;   // lanes without work run along on the unit map
    const long long d0 = fx_of_double(f0, 61 - ED);
    const Dg d1 = fx_split(fx_of_double(f1, 61 - ED)), d2 = fx_split(fx_of_double(f2, 61 - ED));
    const bool varies = NS == 4 && !(f1 == 0.0 && f2 == 0.0);
    FxMap sm;
    sm.setup_bilinear(smap, Eu, Ev);   // not inverted
    ElemCandidate cand[kFixedPairs];
    FxAcc acc[kFixedPairs][NS * NM], accD[SEG ? kFixedPairs : 1][SEG ? NS * NS : 1];
    for (int k = 0; k < kc; ++k) {
      FxMap& m = cand[k].map;
      const bool fits = m.setup_bilinear(maps[k], Eu, Ev);   // and for the box
      corner_range<NM>(m.c0u, m.k1u, m.k2u, m.k3u, cand[k].lo_u, cand[k].hi_u);
      corner_range<NM>(m.c0v, m.k1v, m.k2v, m.k3v, cand[k].lo_v, cand[k].hi_v);
      if (NM == 3 || map_is_affine(maps[k])) {
        const double id = 1.0 / (maps[k].c1u * maps[k].c2v - maps[k].c2u * maps[k].c1v);
        ok &= m.setup_affine(maps[k], maps[k].c2v * id, -maps[k].c2u * id, -maps[k].c1v * id, maps[k].c1u * id, Eu, Ev);
      } else {
        ok &= fits;
      }
      for (int t = 0; t < NS * NM; ++t) acc[k][t].zero();
      if (SEG)
        for (int t = 0; t < NS * NS; ++t) accD[SEG ? k : 0][SEG ? t : 0].zero();
    }
    if (!ok) kc = 0;
    __syncwarp();
    const FxScales none = {{0, 0, 0, 0}};
    FxAcc g[4][4], h[4][4];   // sums of pair cur
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int l = 0; l < 4; ++l) { g[i][l].zero(); h[i][l].zero(); }
    int cur = -1;
    unsigned got[3] = {0u, 0u, 0u};   // points of pair k in byte k (at most 144)
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
      const long long* t = tab + kTableWords<NS> * q;
      const long long xs = t[0], es = t[1];
      long long xu, xv;
      sm.residual(-sm.c0u, -sm.c0v, xs, es, xu, xv);
      const int iu = (int)(xu >> 33), iv = (int)(xv >> 33);
      unsigned near_box = 0;   // candidates left to try, in pair order
      const bool open = !more || !(taken[q >> 5] >> (q & 31) & 1u);
      for (int k = 0; k < (open ? kc : 0); ++k)
        near_box |= (iu >= cand[k].lo_u && iu <= cand[k].hi_u && iv >= cand[k].lo_v && iv <= cand[k].hi_v ? 1u : 0u) << k;
      int owner = -1;
      long long x1 = 0, x2 = 0;
      while (__any_sync(0xffffffffu, near_box != 0u)) {   // at most kFixedPairs rounds: each takes a bit of every lane
        bool near = false, settled = true;
        float x = 0.0f, y = 0.0f;
        const int k = near_box != 0u ? __ffs(near_box) - 1 : 0;
        FxMap m;
        if (near_box != 0u) {
          m = cand[k].map;
          near_box &= near_box - 1u;
          const float tu = fx_f32(xu - m.c0u), tv = fx_f32(xv - m.c0v);
          float band = 1e-5f;
          if (NM == 3 || m.affine) {
            const float xa = m.b00 * tu, xb = m.b01 * tv, ya = m.b10 * tu, yb = m.b11 * tv;
            x = xa + xb;
            y = ya + yb;
            band = fmaf(1e-6f, fabsf(xa) + fabsf(xb) + fabsf(ya) + fabsf(yb), band);   // FP32 rounding of a needle's sums
            if (!(band < 0.25f)) ok = false;   // nothing is written before the end
          } else {
            settled = m.settle(tu, tv, x, y);
          }
          // points clearly outside skip the fixed-point step
          near = !settled || (NM == 4 ? (fabsf(x) <= 1.0f + band && fabsf(y) <= 1.0f + band)
                                      : (x >= -band && y >= -band && x + y <= 1.0f + band));
        }
        __syncwarp();
        if (near) {
          bool solved = settled;
          if (NM == 3 || m.affine) m.solve_affine(xu - m.c0u, xv - m.c0v, x1, x2);
          else if (settled) solved = m.refine(xu - m.c0u, xv - m.c0v, x, y, x1, x2);
          if (!solved) solved = fx_slow_solve(maps[k], Eu, Ev, xu, xv, x1, x2);
          constexpr long long one = 1ll << 61, tol = (long long)(kInsideTol * (double)(1ll << 61));
          const bool inside = NM == 4
              ? (x1 <= one + tol && x1 >= -(one + tol) && x2 <= one + tol && x2 >= -(one + tol))
              : (x1 >= -tol && x2 >= -tol && x1 + x2 <= one + tol);
          if (solved && inside) {
            owner = k;
            near_box = 0u;
          }
        }
        __syncwarp();
      }
      if (owner >= 0 && owner != cur) {
        exchange<NS, NM>(g, cur >= 0 ? acc[cur] : nullptr, acc[owner]);
        if (SEG) exchange<NS, NS>(h, cur >= 0 ? accD[SEG ? cur : 0] : nullptr, accD[SEG ? owner : 0]);
        cur = owner;
      }
      __syncwarp();
      long long det = d0;
      FxAcc a;
      if (varies) {
        a.mul(d1, fx_split(xs));
        a.mac(d2, fx_split(es));
        det += a.get<3>();
      }
      const Dg W = fx_split(det < 0 ? -det : det);
      if (owner >= 0) {
        const unsigned one = 1u << (8 * (owner & 3));
        got[0] += owner < 4 ? one : 0u;
        got[1] += owner >= 4 && owner < 8 ? one : 0u;
        got[2] += owner >= 8 ? one : 0u;
        if (more) taken[q >> 5] |= 1u << (q & 31);
        Dg3 Ns[4];
        Dg Nc[4];
        const int* third = reinterpret_cast<const int*>(t + 2 + NS);
#pragma unroll
        for (int i = 0; i < NS; ++i) Ns[i] = weigh(fx_split(t[2 + i]), third[i], W);
        fx_shape<NM>(none, x1, x2, Nc);
        add_products<NS, NM>(g, Ns, Nc);
        if (SEG) {
          fx_shape<NS>(none, xs, es, Nc);
          add_products<NS, NS>(h, Ns, Nc);
        }
      }
      if ((q & 3) == 3) {   // four products: cross sums below 2^63
        carry_all<NS, NM>(g);
        if (SEG) carry_all<NS, NS>(h);
      }
      __syncwarp();
    }
    if (ok && cur >= 0) {
      exchange<NS, NM>(g, acc[cur], acc[cur]);
      if (SEG) exchange<NS, NS>(h, accD[SEG ? cur : 0], accD[SEG ? cur : 0]);
    }
    const int ke = ED - 59 - boost + (NS == 4 ? 2 : -1);   // sum w = 4 or 1/2
    for (int k = 0; k < (ok ? kc : 0); ++k) {
      const unsigned points = (k < 4 ? got[0] : (k < 8 ? got[1] : got[2])) >> (8 * (k & 3)) & 0xffu;
      put_block<NS, NM, DUAL>(acc[k], ke, r + SR_A, Mblk + 16 * (p0 + k));
      if (SEG) put_block<NS, NS, DUAL>(accD[SEG ? k : 0], ke, r + SR_A, Dblk + 16 * (p0 + k));
      flag[p0 + k] = points > 0 ? 1 : 0;
      live += points > 0 ? 1u : 0u;
      owned += points;
    }
    __syncwarp();
  }
  if (!ok) return false;
  n_live += live;
  n_gp += owned;
  return true;
}

template <int NS, int NM, bool SEG, bool DUAL>
__global__ void __launch_bounds__(kThreads, SEG ? 2 : 3) k_integrate_elembased_fixed(
    const int64_t* __restrict__ pair_off, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, const double* __restrict__ rule, int n,
    int boost, int64_t Es, double* __restrict__ Mblk, double* __restrict__ Dblk, uint8_t* __restrict__ flag,
    DevStatus* st) {
  extern __shared__ long long tab[];
  const int nq = n * n;
  for (int q = threadIdx.x; q < nq; q += blockDim.x) {   // rows to and fro: fewer changes of owner
    const int i = q / n, j = q - i * n;
    double xi, eta, w;
    rule_point(NS, rule, n, n * i + (i & 1 ? n - 1 - j : j), xi, eta, w);
    put_point<NS>(tab + kTableWords<NS> * q, xi, eta, w, boost);
  }
  __syncthreads();
  unsigned long long n_live = 0, n_gp = 0;
  const bool ok = st->over_pairs == 0 && st->over_bins == 0;
  for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); ok && e0 < Es;
       e0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = e0 + (threadIdx.x & 31);
    if (!element_fixed<NS, NM, SEG, DUAL>(e < Es, e, pair_off, pm, srec, xm, conn_m, tab, nq, boost, Mblk, Dblk, flag,
                                          n_live, n_gp))
      element_fp64<NS, NM, SEG, DUAL>(e, pair_off, pm, srec, xm, conn_m, rule, n, Mblk, Dblk, flag, n_live, n_gp);
    __syncwarp();
  }
  block_count_add(&st->nonempty, n_live);
  block_count_add(&st->gauss_points, n_gp);
}

template <int NS, int NM>
void launch_nsnm(mortar_ctx* c, const RunParams& rp) {
  const bool seg = rp.d_domain == 1, dual = rp.lm == 1;
  const int n = c->rule_1d_n, boost = c->rule_boost[NS == 4 ? 0 : 1];
  auto grid = [&](auto kern, size_t shm) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, shm);
    if (per_sm < 1) per_sm = 1;
    return (unsigned)std::min<int64_t>((c->Es + kThreads - 1) / kThreads, (int64_t)c->n_sm * per_sm * 8);
  };
  auto go = [&](auto fixed, auto fp64) {
    if (boost >= 0) {
      const size_t shm = sizeof(long long) * kTableWords<NS> * n * n;
      fixed<<<grid(fixed, shm), kThreads, shm, c->stream>>>(
          c->pair_off.as<int64_t>(), c->pairs_m.as<int32_t>(), c->srec.as<double>(), c->xm.as<double>(),
          c->conn_m.as<int32_t>(), c->rule_1d.as<double>(), n, boost, c->Es, c->Mblk.as<double>(),
          c->Dblk.as<double>(), c->flag.as<uint8_t>(), c->dstat.as<DevStatus>());
    } else {
      fp64<<<grid(fp64, 0), kThreads, 0, c->stream>>>(
          c->pair_off.as<int64_t>(), c->pairs_m.as<int32_t>(), c->srec.as<double>(), c->xm.as<double>(),
          c->conn_m.as<int32_t>(), c->rule_1d.as<double>(), n, c->Es, c->Mblk.as<double>(), c->Dblk.as<double>(),
          c->flag.as<uint8_t>(), c->dstat.as<DevStatus>());
    }
  };
  if (seg && dual) go(k_integrate_elembased_fixed<NS, NM, true, true>, k_integrate_elembased<NS, NM, true, true>);
  else if (seg) go(k_integrate_elembased_fixed<NS, NM, true, false>, k_integrate_elembased<NS, NM, true, false>);
  else if (dual) go(k_integrate_elembased_fixed<NS, NM, false, true>, k_integrate_elembased<NS, NM, false, true>);
  else go(k_integrate_elembased_fixed<NS, NM, false, false>, k_integrate_elembased<NS, NM, false, false>);
}

// Boost of the fixed-point table of an n x n rule: up to three bits, as far as
// every product stays below 1/4.  -1: the smallest product (rules beyond 12 x
// 12 on quad4, 8 x 8 on tri3) would keep less than 40 bits, and the rule
// stays in FP64.
int rule_boost(int nen, const double* rule, int n) {
  double lo = 1.0, hi = 0.0;
  for (int q = 0; q < n * n; ++q) {
    double xi, eta, w;
    rule_point(nen, rule, n, q, xi, eta, w);
    for (int a = 0; a < nen; ++a) {
      const double v = w * (nen == 4 ? 0.25 : 2.0) * rule_shape(nen, a, xi, eta);
      lo = std::min(lo, v);
      hi = std::max(hi, v);
    }
  }
  int b = 0;
  while (b < 3 && std::ldexp(hi, b + 1) < 0.25) ++b;
  return n <= kMaxFixedRule && std::ldexp(lo, b) >= std::ldexp(1.0, -22) ? b : -1;
}

}  // namespace

// n-point Gauss-Legendre rule on [-1, 1] (points ascending, then weights):
// roots of P_n by Newton from cos(pi (i + 3/4) / (n + 1/2)), P_n and P_n' by
// the three-term recurrence, weights 2 / ((1 - x^2) P_n'(x)^2).
int upload_gauss_legendre(mortar_ctx* c, int n) {
  std::vector<double> h(2 * (size_t)n);
  const double pi = std::acos(-1.0);
  for (int i = 0; i < n; ++i) {
    double x = std::cos(pi * (n - i - 0.25) / (n + 0.5));   // ascending order
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double pk = 1.0, pk1 = 0.0;   // P_k, P_{k-1}
      for (int k = 1; k <= n; ++k) {
        const double pn = ((2.0 * k - 1.0) * x * pk - (k - 1.0) * pk1) / k;
        pk1 = pk;
        pk = pn;
      }
      dp = n * (x * pk - pk1) / (x * x - 1.0);
      const double dx = pk / dp;
      x -= dx;
      if (std::fabs(dx) < 1e-16) break;
    }
    double pk = 1.0, pk1 = 0.0;
    for (int k = 1; k <= n; ++k) {
      const double pn = ((2.0 * k - 1.0) * x * pk - (k - 1.0) * pk1) / k;
      pk1 = pk;
      pk = pn;
    }
    dp = n * (x * pk - pk1) / (x * x - 1.0);
    h[i] = x;
    h[n + i] = 2.0 / ((1.0 - x * x) * dp * dp);
  }
  int r = buf_reserve(c->rule_1d, h.size() * sizeof(double));
  if (r != MORTAR_OK) return r;
  if (cudaMemcpy(c->rule_1d.p, h.data(), h.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    return MORTAR_ERR_CUDA;
  }
  c->rule_1d_n = n;
  c->rule_boost[0] = rule_boost(4, h.data(), n);
  c->rule_boost[1] = rule_boost(3, h.data(), n);
  return MORTAR_OK;
}

void launch_integrate_element_based(mortar_ctx* c, const RunParams& rp) {
  if (c->Es == 0) return;
  if (c->nen_s == 4 && c->nen_m == 4) launch_nsnm<4, 4>(c, rp);
  else if (c->nen_s == 4 && c->nen_m == 3) launch_nsnm<4, 3>(c, rp);
  else if (c->nen_s == 3 && c->nen_m == 4) launch_nsnm<3, 4>(c, rp);
  else launch_nsnm<3, 3>(c, rp);
}

}  // namespace mortar
