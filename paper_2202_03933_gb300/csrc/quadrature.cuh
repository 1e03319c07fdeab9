// Quadrature of one pair's clip polygon in fixed point.
#pragma once

#include "fixed.cuh"

namespace mortar {

// A pair's clip polygon in the pair's frame with its element maps and weights.
struct FxPolygon {
  static constexpr int kCap = 8;
  long long X[kCap], Y[kCap], A[kCap];   // vertices (Q62), cell weights omega
  long long cu, cv;                      // fan centre
  int su, sv;                            // shifts that bring the fan's edges to 2^61 .. 2^62
  int nr, ncell, Eu, Ev, ke;             // 2^ke: unit of sums of omega w N_s N_m / 2^64 with N Q61
  FxScales ss, sm;
  FxMap s, m;

  __device__ __forceinline__ long long x(int k) const { return X[k]; }
  __device__ __forceinline__ long long y(int k) const { return Y[k]; }
  __device__ __forceinline__ long long weight(int c) const { return A[c]; }
  // vertices of cell c besides the centre
  __device__ __forceinline__ int ib(int c) const { return nr > 3 ? c : 1; }
  __device__ __forceinline__ int iw(int c) const { return nr > 3 ? (c + 1 == nr ? 0 : c + 1) : 2; }

  // From the FP64 polygon (pu, pv, n vertices).  False if the pair does not fit:
  // more than 8 vertices, an element map out of range (elements about 2^6 apart
  // in size, kMaxMapBits) or a vertex outside its element; the caller then takes
  // the FP64 path.  Cell areas are formed from differences scaled up to full
  // width per direction (a sliver's area keeps its digits); the weights are
  // omega = area 2^t with 2^60 <= sum omega < 2^61.
  template <int NS, int NM>
  __device__ __forceinline__ bool setup(const double* __restrict__ r, const PlaneMap& mmap, const double* pu,
                                        const double* pv, int n) {
    nr = n;
    PlaneMap smap;
    smap.c0u = r[SR_C + 0]; smap.c0v = r[SR_C + 1]; smap.c1u = r[SR_C + 2]; smap.c1v = r[SR_C + 3];
    smap.c2u = r[SR_C + 4]; smap.c2v = r[SR_C + 5]; smap.c3u = r[SR_C + 6]; smap.c3v = r[SR_C + 7];
    const FxFrame fr = fx_frame<NS, NM>(r, mmap);
    bool ok = fr.ok && n <= kCap;   // one exit, so that the lanes that take the FP64 path run it together
    Eu = fr.Eu;
    Ev = fr.Ev;
    if (NM == 3 || map_is_affine(mmap)) {
      const double id = 1.0 / (mmap.c1u * mmap.c2v - mmap.c2u * mmap.c1v);
      ok &= m.setup_affine(mmap, mmap.c2v * id, -mmap.c2u * id, -mmap.c1v * id, mmap.c1u * id, Eu, Ev);
    } else {
      ok &= m.setup_bilinear(mmap, Eu, Ev);
    }
    if (NS == 3 || r[SR_AFF] != 0.0) {
      ok &= s.setup_affine(smap, r[SR_BINV], r[SR_BINV + 1], r[SR_BINV + 2], r[SR_BINV + 3], Eu, Ev);
    } else {
      ok &= s.setup_bilinear(smap, Eu, Ev);
    }
    if (!ok) return false;
    cu = 0;
    cv = 0;
    for (int k = 0; k < nr; ++k) {
      X[k] = fx_of_double(pu[k], 62 - Eu);
      Y[k] = fx_of_double(pv[k], 62 - Ev);
      cu += X[k] >> 2;   // eight values below 2^61
      cv += Y[k] >> 2;
    }
    if (nr > 3) {   // vertex mean
      FxAcc a;
      a.mul(fx_split(cu), kInvCountFx.d[nr]);
      cu = a.get<4>();
      a.mul(fx_split(cv), kInvCountFx.d[nr]);
      cv = a.get<4>();
      ncell = nr;
    } else {
      cu = X[0];
      cv = Y[0];
      ncell = 1;
    }
    unsigned long long mu = 0, mv = 0;
    for (int k = 0; k < nr; ++k) {
      const long long a = X[k] - cu, b = Y[k] - cv;
      mu |= (unsigned long long)(a < 0 ? ~a : a);
      mv |= (unsigned long long)(b < 0 ? ~b : b);
    }
    su = min(max(__clzll((long long)mu) - 2, 0), 60);
    sv = min(max(__clzll((long long)mv) - 2, 0), 60);
    unsigned long long sum = 0;
    for (int c = 0; c < ncell; ++c) {
      const int b = ib(c), w = iw(c);
      FxAcc p, q;
      p.mul(fx_split((X[b] - cu) << su), fx_split((Y[w] - cv) << sv));
      q.mul(fx_split((Y[b] - cv) << sv), fx_split((X[w] - cu) << su));
      const long long a2 = (p.hh - q.hh) + (p.cr >> 32) - (q.cr >> 32);   // twice the area, below 2^61
      A[c] = a2 < 0 ? -a2 : a2;
      sum += (unsigned long long)A[c] >> 3;
    }
    // sum = (total / 8) rounded down by less than 8: one more bit of room covers it
    const int t = __clzll((long long)sum) - 3 - 3 - 1;
    for (int c = 0; c < ncell; ++c) A[c] = t >= 0 ? A[c] << min(t, 62) : A[c] >> -t;
    ke = Eu + Ev - 58 - t - su - sv;
    return sum > 0 && fx_scales<NS>(s, X, Y, nr, ss) && fx_scales<NM>(m, X, Y, nr, sm);
  }
};

// Shape functions of one element in Q61, scaled by 2^shape(a), from xi (Q61).
template <int NEN>
__device__ __forceinline__ void fx_shape(const FxScales& s, long long xi, long long eta, Dg* N) {
  if constexpr (NEN == 4) {
    const long long one = 1ll << 61;
    const Dg a = fx_split((one - xi) << s.k[0]), b = fx_split((one + xi) << s.k[1]);
    const Dg c = fx_split((one - eta) << s.k[2]), d = fx_split((one + eta) << s.k[3]);
    FxAcc p;
    p.mul(a, c);
    N[0] = fx_split(p.get<1>());
    p.mul(b, c);
    N[1] = fx_split(p.get<1>());
    p.mul(b, d);
    N[2] = fx_split(p.get<1>());
    p.mul(a, d);
    N[3] = fx_split(p.get<1>());
  } else {
    N[0] = fx_split(((1ll << 61) - xi - eta) << s.k[0]);
    N[1] = fx_split(xi << s.k[1]);
    N[2] = fx_split(eta << s.k[2]);
  }
}

// A pair's polygon, maps and weights as a record of 64-bit words in global
// memory.  Records are stored in groups of 32, word w of lane i of group g at
// rec[(g kWords + w) 32 + i]: a warp reads or writes 256 contiguous bytes.
struct FxRecord {
  static constexpr int kMapS = 26, kMapM = 34, kScale = 42, kPair = 43, kInfo = 44, kWords = 45;
  // words: 2k, 2k + 1: vertex k; 16 + c: weight of cell c; 24, 25: centre;
  // 26.., 34..: maps (c0, then the digits k1 k2 k3); 42: the eight factor scales; 43: pair id;
  // 44: nr | kb_s << 8 | kb_m << 13 | affine_s << 18 | affine_m << 19 | Ev << 20 (12 bits) | ke << 32 | Eu << 48
  static __device__ __forceinline__ int info_ke(long long info) { return (int)(short)(info >> 32); }
  static __device__ __forceinline__ int info_eu(long long info) { return (int)(short)(info >> 48); }
  static __device__ __forceinline__ int info_ev(long long info) { return (int)info >> 20; }
  static __device__ __forceinline__ void store_map(long long* o, const FxMap& m, bool bilinear_possible) {
    auto put = [&](int w, Dg d) { o[32 * w] = (long long)(((unsigned long long)(unsigned)d.h << 32) | (unsigned)d.l); };
    o[0] = m.c0u;
    o[32] = m.c0v;
    put(2, m.k1u); put(3, m.k1v); put(4, m.k2u); put(5, m.k2v);
    if (bilinear_possible && !m.affine) { put(6, m.k3u); put(7, m.k3v); }
  }
  static __device__ __forceinline__ void load_map(const long long* o, FxMap& m, bool bilinear_possible) {
    auto get = [&](int w) { const long long v = o[32 * w]; return Dg{(int)(v >> 32), (int)v}; };
    m.c0u = o[0];
    m.c0v = o[32];
    m.k1u = get(2); m.k1v = get(3); m.k2u = get(4); m.k2v = get(5);
    if (bilinear_possible && !m.affine) {
      m.k3u = get(6); m.k3v = get(7);
      m.bilinear_floats();
    }
  }
  static __device__ __forceinline__ void load_scales(const long long* o, FxScales& ss, FxScales& sm) {
    const unsigned long long sc = (unsigned long long)o[32 * kScale];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ss.k[k] = (int)(sc >> (8 * k)) & 0xff;
      sm.k[k] = (int)(sc >> (32 + 8 * k)) & 0xff;
    }
  }
  template <int NS, int NM>
  static __device__ __forceinline__ void store(long long* o, const FxPolygon& f, int64_t pair) {
    for (int k = 0; k < f.nr; ++k) {
      o[64 * k] = f.X[k];
      o[64 * k + 32] = f.Y[k];
    }
    for (int c = 0; c < f.ncell; ++c) o[32 * (16 + c)] = f.A[c];
    o[32 * 24] = f.cu;
    o[32 * 25] = f.cv;
    o[32 * kPair] = pair;
    o[32 * kInfo] = (long long)((unsigned long long)((unsigned)(f.nr | f.s.kb << 8 | f.m.kb << 13 |
                                                                (f.s.affine ? 1 : 0) << 18 | (f.m.affine ? 1 : 0) << 19) |
                                                     (unsigned)f.Ev << 20) |
                                (unsigned long long)(unsigned short)f.ke << 32 |
                                (unsigned long long)(unsigned short)f.Eu << 48);
    unsigned long long sc = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      sc |= (unsigned long long)f.ss.k[k] << (8 * k) | (unsigned long long)f.sm.k[k] << (32 + 8 * k);
    o[32 * kScale] = (long long)sc;
    store_map(o + 32 * kMapS, f.s, NS == 4);
    store_map(o + 32 * kMapM, f.m, NM == 4);
  }
};

// The view of a record that the quadrature reads: maps and scales in
// registers, vertices and weights where they are.
struct FxView {
  const long long* o;
  long long cu, cv;
  int nr, ncell, Eu, Ev, ke;
  FxScales ss, sm;
  FxMap s, m;
  __device__ __forceinline__ long long x(int k) const { return o[64 * k]; }
  __device__ __forceinline__ long long y(int k) const { return o[64 * k + 32]; }
  __device__ __forceinline__ long long weight(int c) const { return o[32 * (16 + c)]; }
  __device__ __forceinline__ int ib(int c) const { return nr > 3 ? c : 1; }
  __device__ __forceinline__ int iw(int c) const { return nr > 3 ? (c + 1 == nr ? 0 : c + 1) : 2; }
  template <int NS, int NM>
  __device__ __forceinline__ void load(const long long* rec) {
    o = rec;
    const long long info = o[32 * FxRecord::kInfo];
    nr = (int)(info & 0xff);
    ncell = nr > 3 ? nr : 1;
    s.kb = (int)(info >> 8) & 31;
    m.kb = (int)(info >> 13) & 31;
    s.affine = (info >> 18) & 1;
    m.affine = (info >> 19) & 1;
    ke = FxRecord::info_ke(info);
    Eu = FxRecord::info_eu(info);
    Ev = FxRecord::info_ev(info);
    FxRecord::load_scales(o, ss, sm);
    cu = o[32 * 24];
    cv = o[32 * 25];
    FxRecord::load_map(o + 32 * FxRecord::kMapS, s, NS == 4);
    FxRecord::load_map(o + 32 * FxRecord::kMapM, m, NM == 4);
  }
};

// Back-projections of the seven points of cell c, in fixed point: xi, eta of the
// slave and the master element into pts[(4 q + 0..3) * stride] (pts: this
// thread's slice of shared memory, stride: the block's threads).  False if one
// fails.  The rule's points are c + (e1 + e2) / 3 and, per orbit (a, b),
// c + a (e1 + e2) plus (b - a) e2, (b - a) e1 or nothing: three products a
// coordinate for three points.
template <int NS, int NM, int stride, class F>
__device__ __forceinline__ bool fx_back_project(F& f, int c, const double* __restrict__ r,
                                                const double* __restrict__ xm, const int32_t* __restrict__ conn_m,
                                                int32_t m, long long* __restrict__ pts) {
  const int ib = f.ib(c), iw = f.iw(c);
  const Dg e1u = fx_split(f.x(ib) - f.cu), e1v = fx_split(f.y(ib) - f.cv);
  const Dg e2u = fx_split(f.x(iw) - f.cu), e2v = fx_split(f.y(iw) - f.cv);
  long long d1u = 0, d1v = 0, d2u = 0, d2v = 0, ou = 0, ov = 0;
  bool ok = true;
#pragma unroll 1
  for (int q = 0; q < 7; ++q) {
    if (q == 0 || q == 1 || q == 4) {
      const int k = (q + 2) / 3;
      FxAcc a;   // l1 + l2 < 1 bounds the cross sum by 2^62.6
      a.mul(kOrbitFx.a[k], e1u);
      a.mac(kOrbitFx.a[k], e2u);
      ou = f.cu + a.get<2>();
      a.mul(kOrbitFx.a[k], e1v);
      a.mac(kOrbitFx.a[k], e2v);
      ov = f.cv + a.get<2>();
      if (q > 0) {
        a.mul(kOrbitFx.d[k], e2u);
        d2u = a.get<2>();
        a.mul(kOrbitFx.d[k], e2v);
        d2v = a.get<2>();
        a.mul(kOrbitFx.d[k], e1u);
        d1u = a.get<2>();
        a.mul(kOrbitFx.d[k], e1v);
        d1v = a.get<2>();
      }
    }
    const bool p1 = q == 1 || q == 4, p2 = q == 2 || q == 5;
    const long long xu = ou + (p1 ? d2u : (p2 ? d1u : 0)), xv = ov + (p1 ? d2v : (p2 ? d1v : 0));
    long long xi, eta;
    long long* o = pts + (4 * q) * stride;
    if (!f.s.template solve<NS>(xu, xv, xi, eta))
      ok &= fx_slow_solve(slave_plane_map(r), f.Eu, f.Ev, xu, xv, xi, eta);
    o[0] = xi;
    o[stride] = eta;
    if (!f.m.template solve<NM>(xu, xv, xi, eta))
      ok &= fx_slow_solve(master_plane_map<NM>(r, xm, conn_m, m), f.Eu, f.Ev, xu, xv, xi, eta);
    o[2 * stride] = xi;
    o[3 * stride] = eta;
  }
  return ok;
}

// Sums over one cell's points of W N_s N_m^T (NC = NM columns) or, with
// SLAVE2, of W N_s N_s^T, from the back-projections in pts.  om: the cell's
// weight omega.  Every entry is summed from its own products, so small entries
// keep their digits.  Bounds: a product's cross terms are l h of at most
// 2^31 2^29, seven of them, and h l ones that sum to at most 2^29 2^31 (both
// cannot be met at once: N = 1 at all seven points).
template <int NS, int NC, bool SLAVE2, int stride>
__device__ __forceinline__ void fx_cell_products(const FxScales& ss, const FxScales& sc, long long weight,
                                                 const long long* __restrict__ pts, FxAcc g[4][4]) {
#pragma unroll
  for (int a = 0; a < NS; ++a)
#pragma unroll
    for (int l = 0; l < NC; ++l) g[a][l].zero();
  const Dg om = fx_split(weight);
#pragma unroll 1
  for (int q = 0; q < 7; ++q) {
    Dg Ns[4], Nc[4];   // W N_s, N_m (or N_s)
    FxAcc a;
    a.mul(om, kTri7Fx.w[q]);
    const Dg W = fx_split(a.get<2>());
    const long long xi = pts[(4 * q) * stride], eta = pts[(4 * q + 1) * stride];
    if constexpr (NS == 4) {
      const long long one = 1ll << 61;
      const Dg c2 = fx_split((one - eta) << ss.k[2]), d2 = fx_split((one + eta) << ss.k[3]);
      a.mul(W, fx_split((one - xi) << ss.k[0]));
      const Dg qa = fx_split(a.get<2>());
      a.mul(W, fx_split((one + xi) << ss.k[1]));
      const Dg qb = fx_split(a.get<2>());
      a.mul(qa, c2);
      Ns[0] = fx_split(a.get<2>());
      a.mul(qb, c2);
      Ns[1] = fx_split(a.get<2>());
      a.mul(qb, d2);
      Ns[2] = fx_split(a.get<2>());
      a.mul(qa, d2);
      Ns[3] = fx_split(a.get<2>());
    } else {
      fx_shape<NS>(ss, xi, eta, Nc);
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        a.mul(W, Nc[k]);
        Ns[k] = fx_split(a.get<3>());
      }
    }
    if (SLAVE2) fx_shape<NS>(ss, xi, eta, Nc);
    else fx_shape<NC>(sc, pts[(4 * q + 2) * stride], pts[(4 * q + 3) * stride], Nc);
#pragma unroll
    for (int i = 0; i < NS; ++i)
#pragma unroll
      for (int l = 0; l < NC; ++l) g[i][l].mac(Ns[i], Nc[l]);
  }
}

// Pairs [first, first + count) that the run has; 0 after an overflow, and when
// an earlier kernel of the run stopped early (Watchdog): the kernels of a chunk
// hand each other an order and records, of which such a kernel has left a part
// unwritten.  Lane 0 decides for its warp, since a block of the same kernel may
// set the flag meanwhile.  Every lane of the warp calls it.
__device__ __forceinline__ int64_t chunk_pairs(const DevStatus* st, int64_t pair_cap, int64_t first, int64_t count) {
  int64_t n = 0;
  if ((threadIdx.x & 31) == 0 && st->over_pairs == 0 && st->over_bins == 0 &&
      *reinterpret_cast<const volatile unsigned long long*>(&st->timeout) == 0)
    n = max((int64_t)0, min((int64_t)min((unsigned long long)pair_cap, st->n_pairs) - first, count));
  return __shfl_sync(0xffffffffu, n, 0);
}

// Cells of a record with nr vertices: none for an empty pair's, or one that is
// not the cell kernels' to run (nr beyond the polygon's capacity).
__device__ __forceinline__ int record_cells(long long info) {
  const int nr = (int)(info & 0xff);
  return nr < 3 || nr > FxPolygon::kCap ? 0 : (nr > 3 ? nr : 1);
}

// Records per turn of a cell kernel's warp: about 16 turns a warp, 8 (a warp's
// lanes) to 256 records.
__device__ __forceinline__ int cell_turn(int64_t n) {
  const int64_t t = n / (16 * (int64_t)gridDim.x * (blockDim.x >> 5));
  return (int)max((int64_t)8, min((int64_t)256, t & ~(int64_t)7));
}

// Cells of consecutive records on consecutive lanes: each lane gets one cell
// of one pair, whole pairs only, as many as fit in a warp.
struct CellSlot {
  int rec;      // record relative to the window's first
  int cell;     // cell of this lane within its pair, -1: none
  int first;    // lane of the pair's cell 0
  int cells;    // cells of the pair
  int taken;    // records used up by this round, at least 1
};
// ncell: this lane's record's cells (lane i: record i of the window; at most 8)
__device__ __forceinline__ CellSlot assign_cells(int ncell) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int cum = ncell;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(kAll, cum, d);
    if (lane >= d) cum += v;
  }
  const unsigned fit = __ballot_sync(kAll, cum <= 32);   // a prefix of the lanes
  CellSlot s;
  s.taken = max(__popc(fit), 1);   // a lane's cells fit a warp (record_cells), so that 0 does not happen
  const bool has = cum <= 32 && ncell > 0;
  const int start = cum - ncell;
  const unsigned starts = __reduce_or_sync(kAll, has ? 1u << start : 0u);
  const unsigned owners = __ballot_sync(kAll, has);   // records with cells, in the order of their starts
  const int total = __reduce_max_sync(kAll, has ? cum : 0);
  const unsigned upto = starts & (0xffffffffu >> (31 - lane));
  s.cell = -1;
  s.rec = 0;
  s.first = 0;
  if (lane < total) {
    const int rank = __popc(upto) - 1;
    s.first = 31 - __clz(upto);
    s.cell = lane - s.first;
    s.rec = __fns(owners, 0, rank + 1);
  }
  s.cells = __shfl_sync(kAll, ncell, s.rec);
  return s;
}

// Adds up the cells' sums g of every pair of the warp: the lanes of a pair take
// its entries (a, l) in turn and pass each sum, hh + cr / 2^32, to emit.  buf:
// this thread's slice of shared memory (24 words; entry i at buf[i * stride],
// lane L's at buf - lane + L), free to use by the whole warp.
template <int NR, int NC, int stride, class Emit>
__device__ __forceinline__ void fx_sum_cells(const FxAcc g[4][4], const CellSlot& cs, bool ok,
                                             long long* __restrict__ buf, Emit emit) {
  __syncwarp();
#pragma unroll
  for (int a = 0; a < NR; ++a)
#pragma unroll
    for (int l = 0; l < NC; ++l) {
      const int e = NC * a + l;
      buf[e * stride] = g[a][l].hh + (g[a][l].cr >> 32);
      reinterpret_cast<unsigned*>(buf + (16 + (e >> 1)) * stride)[e & 1] = (unsigned)g[a][l].cr;
    }
  __syncwarp();
  const long long* pair = buf - (threadIdx.x & 31) + cs.first;
  if (ok)
#pragma unroll 1
    for (int e = cs.cell; e < NR * NC; e += cs.cells) {
      long long hh = 0, cr = 0;
      for (int k = 0; k < cs.cells; ++k) {
        hh += pair[e * stride + k];
        cr += reinterpret_cast<const unsigned*>(pair + (16 + (e >> 1)) * stride + k)[e & 1];
      }
      emit(e / NC, e % NC, hh, cr);
    }
}

// Writes the 4x4 block M = A G (standard LMs: G) of every pair of the warp from
// its cells' sums g (fx_sum_cells).
template <int NS, int NC, int stride>
__device__ __forceinline__ void write_block(const FxAcc g[4][4], const CellSlot& cs, bool ok, int ke,
                                            const FxScales& ss, const FxScales& sc, bool dual,
                                            const double* __restrict__ r, double* __restrict__ out,
                                            long long* __restrict__ buf) {
  double G[16];   // dual: this lane's entries, until every lane has read the sums
  int n = 0;
  fx_sum_cells<NS, NC, stride>(g, cs, ok, buf, [&](int a, int l, long long hh, long long cr) {
    const double v = fx_to_double(hh, cr, ke - ss.shape<NS>(a) - sc.shape<NC>(l));
    if (dual) G[n++] = v;
    else __stcs(out + 4 * a + l, v);
  });
  if (ok && NS * NC < 16)   // the block is padded with zeros
    for (int e = cs.cell; e < 16; e += cs.cells)
      if ((e >> 2) >= NS || (e & 3) >= NC) __stcs(out + e, 0.0);
  if (dual) {
    __syncwarp();
    double* Gs = reinterpret_cast<double*>(buf - (threadIdx.x & 31) + cs.first);
    if (ok) {
      n = 0;
      for (int e = cs.cell; e < NS * NC; e += cs.cells) Gs[e * stride] = G[n++];
    }
    __syncwarp();
    if (ok)
#pragma unroll 1
      for (int e = cs.cell; e < NS * NC; e += cs.cells) {
        const int a = e / NC, l = e - NC * a;
        double v = 0.0;
#pragma unroll
        for (int c = 0; c < NS; ++c) v = fma(r[SR_A + 4 * a + c], Gs[(NC * c + l) * stride], v);
        __stcs(out + 4 * a + l, v);
      }
  }
}

}  // namespace mortar
