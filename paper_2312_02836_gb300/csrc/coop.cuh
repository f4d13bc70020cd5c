// coop.cuh -- one zone per team of threads: 4, 8 or 16 lanes of a warp, a
// warp, or a block of two to eight warps.  The network evaluation, the linear
// algebra and the per-step scalars of the integrator (integrator.cuh) are
// spread over the team.
//
// What it is for.  On this GPU a warp's FP64 instruction takes its scheduler
// 64 cycles, dependent or not, whatever its active lanes, and four warps
// (one per scheduler) keep the SM's FP64 unit busy.  So a zone's time is its
// count of FP64 warp instructions times 64 cycles, and an SM's throughput is
// that count over all its zones.  One zone per lane (device.cuh) does the
// fewest instructions per zone, but needs thousands of zones per SM and
// 3 to 120 KB of work arrays each; a team cuts the longest zone's time by
// what it spreads and needs a few zones per SM, their arrays in shared
// memory.
//
// Two orders of arithmetic:
//  * S = 0, the lane order: every sum in the order of the lane kernels, so a
//    team gives a lane kernel's bits;
//  * S = 32, 64, 128, the team order: sums are S strided partial sums added
//    by a butterfly in each 32 and then in order, triangular solves go
//    column by column.  The result depends on S only, not on the threads P
//    that share the work: every warp forms the whole sum itself, so no
//    barrier is spent on it.
// The LU is the same in both: each slot sees its updates in pivot order.
// Every thread holds the zone's scalars (time, step, order, counters) and
// computes them identically, so branches are uniform across the team.
#pragma once
#include "device.cuh"
#include "integrator.cuh"

namespace nb {

// The compiled network as a team reads it.  The header is a kernel parameter,
// so its sizes and offsets are operands from the constant bank: read from
// the blob, they were loads in front of every loop.
struct BlobDims {
  const unsigned char* b;
  const BlobHeader& h;
  const int &n, &N, &R, &sh, &hasE;
  double inv_n;
  __device__ __forceinline__ BlobDims(const unsigned char* blob, const BlobHeader& H)
      : b(blob), h(H), n(H.n), N(H.N), R(H.R), sh(H.self_heating), hasE(H.has_E),
        inv_n(1.0 / H.n) {}
  template <class T>
  __device__ __forceinline__ const T* arr(int off) const {
    return reinterpret_cast<const T*>(b + off);
  }
};

// coefficients of the series of delta_phi_series, one row per power of T9:
// 1/T9, T9^(-1/3), T9^(1/3), T9^(5/3), ln T9, T9^(-3/2)
__device__ const double g_series[6][4] = {
    {-1.0, 1.0, -1.0, 1.0},
    {-1.0 / 3.0, 2.0 / 9.0, -14.0 / 81.0, 35.0 / 243.0},
    {1.0 / 3.0, -1.0 / 9.0, 5.0 / 81.0, -10.0 / 243.0},
    {5.0 / 3.0, 5.0 / 9.0, -5.0 / 81.0, 5.0 / 243.0},
    {1.0, -0.5, 1.0 / 3.0, -0.25},
    {-1.5, 15.0 / 8.0, -35.0 / 16.0, 315.0 / 128.0}};

template <int P_, int S_, class D_ = BlobDims>
struct TNet : D_ {
  static constexpr int P = P_, S = S_, width = P_;
  static constexpr int SW = P_ < 32 ? P_ : 32;   // threads of the team in one warp
  int lane;        // 0 .. P-1
  unsigned mask;   // the team's lanes in this warp
  unsigned long long* slot;   // P > 32: broadcast slot in shared memory
  // Per-point values (history times, weights, powers of T9) sit one per lane,
  // or two where the team has fewer than 8 lanes: point j in slot j / SW of
  // lane j % SW
  static constexpr int NP = P_ < 8 ? 8 / P_ : 1;
  double ser[NP][4];   // this lane's rows of g_series

  __device__ __forceinline__ TNet(const D_& d, unsigned long long* bslot) : D_(d), slot(bslot) {
    lane = threadIdx.x % P;
    mask = P >= 32 ? 0xffffffffu : ((1u << (P & 31)) - 1u) << (threadIdx.x & 31 & ~(P - 1));
#pragma unroll
    for (int r = 0; r < NP; ++r) {
      const int row = point(r) < 6 ? point(r) : 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) ser[r][c] = g_series[row][c];
    }
  }
  __device__ __forceinline__ int wl() const { return lane & (SW - 1); }
  __device__ __forceinline__ double shfl(double x, int src) const {
    return __shfl_sync(mask, x, src, SW);
  }
  // the point in this lane's slot r, and point m's value in every lane
  __device__ __forceinline__ int point(int r) const { return wl() + SW * r; }
  __device__ __forceinline__ double pick(const double (&v)[NP], int m) const {
    if constexpr (NP == 1) return shfl(v[0], m);
    else return shfl(m < SW ? v[0] : v[1], m & (SW - 1));
  }
  // sum of f over i < cnt: acc <- f(i, acc).  sum1: the lane kernel's single
  // chain, sum2: its two interleaved partial sums; the same in team order.
  template <class F>
  __device__ __forceinline__ double sum_team(int cnt, F f) const {
    static_assert(P >= 32, "one partial sum of each 32 per lane");
    double tot = 0.0;
#pragma unroll
    for (int q = 0; q < S / 32; ++q) {
      double x = 0.0;
      for (int i = (lane & 31) + 32 * q; i < cnt; i += S) x = f(i, x);
#pragma unroll
      for (int m = 16; m >= 1; m >>= 1) x += __shfl_xor_sync(mask, x, m);
      tot = q == 0 ? x : tot + x;
    }
    return tot;
  }
  template <class F>
  __device__ __forceinline__ double sum1(int cnt, F f) const {
    if constexpr (S > 0) {
      return sum_team(cnt, f);
    } else {
      double acc = 0.0;
      for (int i = 0; i < cnt; ++i) acc = f(i, acc);
      return acc;
    }
  }
  template <class F>
  __device__ __forceinline__ double sum2(int cnt, F f) const {
    if constexpr (S > 0) {
      return sum_team(cnt, f);
    } else {
      // even lanes take the first partial sum, odd lanes the second
      double acc = 0.0;
      for (int i = lane & 1; i < cnt; i += 2) acc = f(i, acc);
      return acc + __shfl_xor_sync(mask, acc, 1);
    }
  }
  __device__ __forceinline__ bool all(bool b) const {
    if constexpr (P > 32) return __syncthreads_and(b) != 0;
    else return __all_sync(mask, b);
  }
  __device__ __forceinline__ void sync() const {
    if constexpr (P > 32) __syncthreads();
    else __syncwarp(mask);
  }
  // thread 0's value in every thread of the team
  __device__ __forceinline__ unsigned long long bcast(unsigned long long v) const {
    if constexpr (P > 32) {
      __syncthreads();
      if (lane == 0) *slot = v;
      __syncthreads();
      return *slot;
    } else {
      return __shfl_sync(mask, v, 0, SW);
    }
  }
};

// shared-memory bytes a block needs for its team's broadcasts
__host__ __device__ constexpr int team_scratch_bytes(int P) { return P > 32 ? 16 : 0; }

template <int P, int S, class D>
struct is_coop<TNet<P, S, D>> {
  static constexpr bool value = true;
};

// contiguous view of one of the team's arrays
struct CV {
  double* p;
  __device__ __forceinline__ double& operator[](int i) const { return p[i]; }
};

// the team's arrays: y holds a solve's partial sums ([2 n]) and its solution
// ([n]), both in position order
struct CWS {
  CV x, xp, psi, f, iw, tmp, pv, f0, xh, eh, th, k, g, rr, kp, dt, lu, y;
};

// The Newton-loop part of the arrays at hot, f0 and the history at cold
__device__ __forceinline__ CWS make_cws(const BlobHeader& h, double* hot, double* cold) {
  CWS w;
  w.x.p = hot + h.th_x; w.xp.p = hot + h.th_xp; w.psi.p = hot + h.th_psi;
  w.iw.p = hot + h.th_iw; w.tmp.p = hot + h.th_tmp;
  w.pv.p = hot + h.th_pv;
  w.k.p = hot + h.th_k; w.rr.p = hot + h.th_rr;
  w.lu.p = hot + h.th_lu; w.y.p = hot + h.th_y; w.f.p = hot + h.th_f;
  w.dt.p = hot + h.th_dt; w.eh.p = hot + h.th_eh; w.th.p = hot + h.th_th;
  // the T9 slopes and reference rates sit with the cold part at fixed T9
  w.g.p = h.th_g >= 0 ? hot + h.th_g : cold + h.tc_g;
  w.kp.p = h.th_kp >= 0 ? hot + h.th_kp : cold + h.tc_kp;
  w.f0.p = cold + h.tc_f0;
  w.xh.p = cold + h.tc_xh;
  return w;
}

// ---------------------------------------------------------------- rates

// what rate_full reads of the network
struct RateNet {
  const double *coef, *scale, *apc, *scr, *tab_lnl;
  const int32_t *ap, *nrho, *tab_of;
  int tab_nd, tab_nt;
};

template <class D>
__device__ __forceinline__ RateNet rate_net(const D& t) {
  RateNet r;
  const BlobHeader& h = t.h;
  r.coef = t.template arr<double>(h.o_coef); r.scale = t.template arr<double>(h.o_scale);
  r.apc = t.template arr<double>(h.o_apc); r.ap = t.template arr<int32_t>(h.o_ap);
  r.nrho = t.template arr<int32_t>(h.o_nrho);
  r.scr = h.has_scr ? t.template arr<double>(h.o_scr) : nullptr;
  r.tab_of = h.n_tab > 0 ? t.template arr<int32_t>(h.o_tab_of) : nullptr;
  r.tab_lnl = t.template arr<double>(h.o_tab_lnl);
  r.tab_nd = h.tab_nd; r.tab_nt = h.tab_nt;
  return r;
}

template <class D>
__device__ __forceinline__ TCell team_cell(const D& t, const RateNet& r, double T9) {
  return r.tab_of ? t_cell(t.template arr<double>(t.h.o_tab_t9), r.tab_nt, T9)
                  : TCell{0, 0.0, 1.0, false};
}

template <int P, int S, class D>
__device__ __forceinline__ void eval_rates(const TNet<P, S, D>& t, const Zone& s, const CWS& w,
                                           const TPow& p, double T9, bool with_g) {
  t.sync();
  const RateNet rn = rate_net(t);
  const TCell tc = team_cell(t, rn, T9);
  for (int r = t.lane; r < t.R; r += P) {
    double gr;
    w.k[r] = rate_full(rn, s, r, p, T9, tc, with_g ? &gr : nullptr);
    if (with_g) w.g[r] = gr;
  }
  t.sync();
}

template <int P, int S, class D>
__device__ __forceinline__ void save_ref_rates(const TNet<P, S, D>& t, const CWS& w) {
  for (int r = t.lane; r < t.R; r += P) w.kp[r] = w.k[r];
  t.sync();
}

// delta_phi_series with one power per lane: 7 FP64 instructions for the
// team, where one lane alone takes 31
template <int P, int S, class D>
__device__ __forceinline__ bool delta_phi_team(const TNet<P, S, D>& t, const TPow& r, double T9,
                                               double T9r, DPhi& d) {
  const double dT = T9 - T9r;
  const double x = dT * r.iT;
  if ((dbits(x) & 0x7fffffffffffffffLL) > 0x3f10000000000000LL) return false;
  double v[TNet<P, S, D>::NP];
#pragma unroll
  for (int q = 0; q < TNet<P, S, D>::NP; ++q) {
    const int l = t.point(q);
    const double pre = l == 0 ? r.iT : l == 1 ? r.it13 : l == 2 ? r.t13 : l == 3 ? r.T53
                     : l == 4 ? 1.0 : r.hz;
    v[q] = pre * binom4(x, t.ser[q][0], t.ser[q][1], t.ser[q][2], t.ser[q][3]);
  }
  d.d1 = t.pick(v, 0);
  d.d2 = t.pick(v, 1);
  d.d3 = t.pick(v, 2);
  d.d4 = dT;
  d.d5 = t.pick(v, 3);
  d.d6 = t.pick(v, 4);
  d.d7 = t.pick(v, 5);
  return true;
}

template <int P, int S, class D>
__device__ __forceinline__ void eval_rates_near(const TNet<P, S, D>& t, const Zone& s,
                                                const CWS& w, double T9, const TPow& ref,
                                                double T9ref) {
  t.sync();
  const RateNet rn = rate_net(t);
  DPhi d;
  TPow p;
  bool have_p = !delta_phi_team(t, ref, T9, T9ref, d);
  if (have_p) {
    p = t_powers(T9, false, s.scr);
    d = delta_phi(p, ref, T9, T9ref);
  }
  const TCell tc = team_cell(t, rn, T9);
  for (int r = t.lane; r < t.R; r += P) {
    const double* a = rn.coef + 7 * r;
    double de = rate_delta(a[1], a[2], a[3], a[4], a[5], a[6], d);
    if (rn.scr) de = fma(rn.scr[r], d.d7, de);
    if (rn.ap[r] < 0 && !(rn.tab_of && rn.tab_of[r] >= 0) && small_delta(de)) {
      w.k[r] = rate_near(w.kp[r], de);
    } else {
      if (!have_p) {
        p = t_powers(T9, false, s.scr);
        have_p = true;
      }
      w.k[r] = rate_full(rn, s, r, p, T9, tc, nullptr);
    }
  }
  t.sync();
}

// the zone's density cell of the rate tables (every thread, the same sum)
template <int P, int S, class D, class V>
__device__ __forceinline__ void tab_zone(const TNet<P, S, D>& t, Zone& s, const V& x0) {
  t.sync();
  s.tab_i = 0;
  s.tab_u = 0.0;
  if (t.h.n_tab <= 0) return;
  const double* charge = t.template arr<double>(t.h.o_charge);
  double ye = 0.0;
  for (int i = 0; i < t.N; ++i) ye = fma(charge[i], x0[i], ye);
  density_cell(t.template arr<double>(t.h.o_tab_dens), t.h.tab_nd, s.rho, ye, s);
}

// ---------------------------------------------------------------- terms, f, M

template <int P, int S, class D>
__device__ __forceinline__ void eval_terms(const TNet<P, S, D>& t, const CWS& w, const CV& v) {
  t.sync();
  const int16_t* reac = t.template arr<int16_t>(t.h.o_reac);
  const int32_t* nreac = t.template arr<int32_t>(t.h.o_nreac);
  for (int r = t.lane; r < t.R; r += P) {
    const int16_t* ra = reac + 3 * r;
    const int m = nreac[r];
    double q = w.k[r];
    q *= v[ra[0]];
    if (m > 1) q *= v[ra[1]];
    if (m > 2) q *= v[ra[2]];
    w.rr[r] = q;
  }
  t.sync();
}

// sum_r Q_r rr_r, the same value in every thread
template <int P, int S, class D>
__device__ __forceinline__ double eval_edot(const TNet<P, S, D>& t, const CWS& w) {
  const double* Q = t.template arr<double>(t.h.o_Q);
  return t.sum2(t.R, [&](int r, double e) { return fma(Q[r], w.rr[r], e); });
}

// sum_e c[e] v[idx[e]] over [beg, end), two interleaved partial sums
template <class TI, class V>
__device__ __forceinline__ double gather(const double* c, const TI* idx, int beg, int end,
                                         const V& v) {
  double a0 = 0.0, a1 = 0.0;
  int e = beg;
  for (; e + 1 < end; e += 2) {
    a0 = fma(c[e], v[idx[e]], a0);
    a1 = fma(c[e + 1], v[idx[e + 1]], a1);
  }
  if (e < end) a0 = fma(c[e], v[idx[e]], a0);
  return a0 + a1;
}

// The gathers of `cnt` rows in order of decreasing length: the first `split`
// (more than 4 entries) by two threads each, one partial sum a thread, the
// rest one per thread.  store(row, sum) is called by one thread per row.
// Sorted, the rows that share an instruction are of like length; unsorted
// (rows by index), the 48-species Jacobian's 1,333 slots took three times
// the instructions.
template <int P, int S, class D, class V, class ST>
__device__ __forceinline__ void gather_rows(const TNet<P, S, D>& t, const int16_t* ord, int split,
                                            int cnt, const int32_t* ptr, const int16_t* idx,
                                            const double* c, const V& v, ST store) {
  const int par = t.lane & 1;
  for (int b = 0; b < split; b += P / 2) {
    const int q = b + (t.lane >> 1);
    const int row = ord[q < split ? q : 0];
    double a = 0.0;
    if (q < split)
      for (int e = ptr[row] + par; e < ptr[row + 1]; e += 2) a = fma(c[e], v[idx[e]], a);
    const double o = __shfl_xor_sync(t.mask, a, 1);
    if (q < split && par == 0) store(row, a + o);
  }
  for (int q = split + t.lane; q < cnt; q += P) {
    const int row = ord[q];
    store(row, gather(c, idx, ptr[row], ptr[row + 1], v));
  }
}

template <int P, int S, class D>
__device__ __forceinline__ void eval_f(const TNet<P, S, D>& t, const CWS& w,
                                       const HeatRate& hr, const CV& out) {
  t.sync();
  const BlobHeader& h = t.h;
  gather_rows(t, t.template arr<int16_t>(h.o_rhs_ord), h.rhs_split, t.N,
              t.template arr<int32_t>(h.o_rhs_ptr), t.template arr<int16_t>(h.o_rhs_r),
              t.template arr<double>(h.o_rhs_c), w.rr,
              [&](int i, double a) { out[i] = a; });
  if (t.sh) {
    const double fT = hr.ed / hr.cv;
    if (t.lane == 0) out[t.N] = fT;
  }
  t.sync();
}

// M = alpha0 I - h J(v) into w.lu (needs w.k, w.g (self-heating), w.rr at v)
template <int P, int S, class D>
__device__ __forceinline__ void assemble_M(const TNet<P, S, D>& t, const CWS& w, const CV& v,
                                           const HeatRate& hr, double alpha0, double h) {
  t.sync();
  const BlobHeader& hd = t.h;
  const int nd = hd.nd;
  {
    const int16_t *dt_o = t.template arr<int16_t>(hd.o_dt_o),
                  *dt_r = t.template arr<int16_t>(hd.o_dt_r);
    const double* dt_m = t.template arr<double>(hd.o_dt_m);
    for (int d = t.lane; d < nd; d += P) {
      const int16_t o0 = dt_o[2 * d], o1 = dt_o[2 * d + 1];
      double q = w.k[dt_r[d]] * dt_m[d];
      if (o0 >= 0) q *= v[o0];
      if (o1 >= 0) q *= v[o1];
      w.dt[d] = q;
    }
  }
  TRow tr{0.0, 0.0, 0.0};
  if (t.sh) {
    for (int r = t.lane; r < t.R; r += P) w.dt[nd + r] = w.rr[r] * w.g[r];
    tr = t_row(hr.ed, hr.cv, v[t.N]);
  }
  t.sync();
  const double mh = -h;
  const uint8_t* flag = t.template arr<uint8_t>(hd.o_js_flag);
  const int16_t* ord = t.template arr<int16_t>(hd.o_js_ord);
  gather_rows(t, ord, hd.js_split, hd.js_fill, t.template arr<int32_t>(hd.o_js_ptr),
              t.template arr<int16_t>(hd.o_js_src), t.template arr<double>(hd.o_js_c), w.dt,
              [&](int sl, double acc) {
                const uint8_t fl = flag[sl];
                if (fl & SLOT_TROW) acc = fma(acc, tr.a1, tr.b1);
                else if (fl & SLOT_TT) acc = fma(acc, tr.a1, tr.b2);
                double m = mh * acc;
                if (fl & SLOT_DIAG) m += alpha0;
                w.lu[sl] = m;
              });
  // slots of the fill: -h times an empty sum
  const double m0 = mh * 0.0, md = m0 + alpha0;
  for (int q = hd.js_fill + t.lane; q < hd.nnz; q += P) {
    const int sl = ord[q];
    w.lu[sl] = flag[sl] & SLOT_DIAG ? md : m0;
  }
  t.sync();
}

// ---------------------------------------------------------------- LU

// quotient of small numbers (a < 2^15, b < 2^8 or so) in single precision:
// (a + 1/2) / b is at least 1/(2 b) away from an integer
__device__ __forceinline__ int small_div(int a, int b) {
  return (int)__fdividef((float)a + 0.5f, (float)b);
}

// a[D(i,j)] -= a[L_i] a[U_j] over the |L| x |U| pairs of one pivot, a pair
// per thread and round (93 % and 99 % of the lanes busy on the 48- and
// 128-species networks).  at(e, li, u, ds, ls, us) names pair e's slots.  The
// pairs are independent, so the operands of NBATCH rounds are loaded before
// the first result is stored: one round's shared-memory latency would
// otherwise show between its FMAs.
template <int P, int NBATCH, class AT>
__device__ __forceinline__ void update_pairs(int lane, double* lu, int nl, int nu, AT at) {
  const int np = nl * nu;
  const int qW = small_div(P, nu), rW = P - qW * nu;
  int li = small_div(lane, nu), u = lane - li * nu;
  for (int e = lane; e < np; e += P * NBATCH) {
    int ds[NBATCH];
    double d[NBATCH], l[NBATCH], v[NBATCH];
#pragma unroll
    for (int b = 0; b < NBATCH; ++b) {
      ds[b] = -1;
      if (e + b * P < np) {
        int ls, us;
        at(e + b * P, li, u, ds[b], ls, us);
        d[b] = lu[ds[b]];
        l[b] = lu[ls];
        v[b] = lu[us];
      }
      li += qW;
      u += rW;
      if (u >= nu) { u -= nu; ++li; }
    }
#pragma unroll
    for (int b = 0; b < NBATCH; ++b)
      if (ds[b] >= 0) lu[ds[b]] = fma(-l[b], v[b], d[b]);
  }
}

// Static-pivot LU in place, the diagonal keeping 1/pivot; the lane
// kernel's operations slot by slot.  false if a pivot is zero, not finite
// or eaten by cancellation (pivot_kept, all pivots at the end, in parallel).
// Pivots before the trailing dense block read their pairs' slots from the
// compiled lists; the block itself is stored dense, so its slots are
// computed, which spares the 20 to 450 KB of lists that every factorisation
// would read through the L1.
template <int P, int S, class D>
__device__ __forceinline__ bool factor_M(const TNet<P, S, D>& t, const CWS& w) {
  t.sync();
  const BlobHeader& h = t.h;
  const Pivot* piv = t.template arr<Pivot>(h.o_piv);
  const int16_t *lslot = t.template arr<int16_t>(h.o_lslot),
                *uslot = t.template arr<int16_t>(h.o_uslot),
                *dslot = t.template arr<int16_t>(h.o_dslot),
                *dpos = t.template arr<int16_t>(h.o_dpos);
  constexpr int NB = P > 32 ? 4 : P == 32 ? 2 : 1;
  const int c = h.tail, n = t.n, m = n - c, wbase = t.lane & ~31;
  double* lu = w.lu.p;
  double* pvs = w.pv.p;   // the pivots before they are inverted
  for (int k = t.lane; k < n; k += P) w.tmp[k] = lu[dpos[k]];
  t.sync();
  for (int k = 0; k < c; ++k) {
    const Pivot p = piv[k];
    const int nl = p.lend - p.lbeg, nu = p.uend - p.ubeg;
    double inv = 0.0;
    if (wbase == 0 || wbase < nl) {   // warps without a row spare the pipe
      const double pv = lu[p.dslot];
      inv = recip2(pv);
      if (t.lane == 0) pvs[k] = pv;
      for (int li = t.lane; li < nl; li += P) {
        const int ls = lslot[p.lbeg + li];
        lu[ls] = lu[ls] * inv;
      }
    }
    t.sync();
    if (t.lane == 0) lu[p.dslot] = inv;
    if (nl > 0 && nu > 0)
      update_pairs<P, NB>(t.lane, lu, nl, nu, [&](int e, int li, int u, int& ds, int& ls, int& us) {
        ds = dslot[p.dbeg + e];
        ls = lslot[p.lbeg + li];
        us = uslot[p.ubeg + u];
      });
    t.sync();
  }
  // (i, j) of the block at a[i m + j]
  double* a = lu + h.tail_slot;
  for (int k = 0; k < m; ++k) {
    double* ak = a + k * (m + 1);
    const int r = m - 1 - k;
    double inv = 0.0;
    if (wbase == 0 || wbase < r) {
      const double pv = *ak;
      inv = recip2(pv);
      if (t.lane == 0) pvs[c + k] = pv;
      for (int i = t.lane; i < r; i += P) ak[(i + 1) * m] = ak[(i + 1) * m] * inv;
    }
    t.sync();
    if (t.lane == 0) *ak = inv;
    if (r > 0)
      update_pairs<P, NB>(t.lane, ak, r, r, [&](int, int li, int u, int& ds, int& ls, int& us) {
        ls = (li + 1) * m;
        us = u + 1;
        ds = ls + us;
      });
    t.sync();
  }
  bool ok = true;
  for (int k = t.lane; k < n; k += P) ok = ok && pivot_kept(pvs[k], w.tmp[k]);
  return t.all(ok);
}

// ---------------------------------------------------------------- solves

// Column substitution on y (position order) over columns [k0, k1): column k's
// solved value goes to the rows of its entries.  DIAG: y_k is multiplied by the stored reciprocal
// pivot first.  UP: columns last to first.  In lane order a row keeps its
// two partial sums (y[2 row + parity], seeded with the right-hand side and
// 0) and the solved values go to z; in team order y[row] alone, solved in
// place.  The next column's entry and factor are fetched before the barrier:
// they don't depend on y.
template <int P, int S, bool DIAG, bool UP, class D>
__device__ __forceinline__ void solve_columns(const TNet<P, S, D>& t, const double* lu,
                                              const uint32_t* ent, const int32_t* ptr,
                                              const int16_t* dpos, double* y, double* z,
                                              int k0, int k1) {
  const int n = k1 - k0;
  if (n <= 0) return;
  int k = UP ? k1 - 1 : k0;
  int e0 = ptr[k], e1 = ptr[k + 1];
  uint32_t pk = 0;
  double l = 0.0, dv = 1.0;
  if (e0 + t.lane < e1) { pk = ent[e0 + t.lane]; l = lu[pk & 0xffff]; }
  if (DIAG) dv = lu[dpos[k]];
  for (int it = 0; it < n; ++it) {
    double xk = S > 0 ? y[k] : y[2 * k] + y[2 * k + 1];
    if (DIAG) xk = xk * dv;
    if (e0 + t.lane < e1) {
      double* tgt = y + (S > 0 ? pk >> 17 : pk >> 16);
      *tgt = fma(-l, xk, *tgt);
    }
    for (int e = e0 + t.lane + P; e < e1; e += P) {
      const uint32_t q = ent[e];
      double* tgt = y + (S > 0 ? q >> 17 : q >> 16);
      *tgt = fma(-lu[q & 0xffff], xk, *tgt);
    }
    const int kd = k;
    k += UP ? -1 : 1;
    if (it + 1 < n) {
      e0 = ptr[k];
      e1 = ptr[k + 1];
      if (e0 + t.lane < e1) { pk = ent[e0 + t.lane]; l = lu[pk & 0xffff]; }
      if (DIAG) dv = lu[dpos[k]];
    }
    if (S == 0) {
      if (t.lane == 0) z[kd] = xk;
      t.sync();
    } else {
      t.sync();
      // every thread has read y[kd], and no later column does
      if (DIAG && t.lane == 0) y[kd] = xk;
    }
  }
  if (S > 0 && DIAG) t.sync();
}

// Back substitution in lane order: a row's entries in increasing column, one
// partial sum per thread of a pair; rows of one dependency level together.
template <int P, int S, bool DIAG, class D>
__device__ __forceinline__ void solve_rows(const TNet<P, S, D>& t, const double* lu,
                                           const uint32_t* ent, const int32_t* ptr,
                                           const int16_t* rows, const int16_t* lev, int n_lev,
                                           const int16_t* dpos, double* z) {
  const int par = t.lane & 1;
  for (int v = 0; v < n_lev; ++v) {
    const int r0 = lev[v], r1 = lev[v + 1];
    for (int b = r0; b < r1; b += P / 2) {
      const int q = b + (t.lane >> 1);
      const bool act = q < r1;
      const int row = rows[act ? q : r0];
      double a = 0.0;
      if (act) {
        if (par == 0) a = z[row];
        for (int e = ptr[row] + par; e < ptr[row + 1]; e += 2) {
          const uint32_t pk = ent[e];
          a = fma(-lu[pk & 0xffff], z[pk >> 16], a);
        }
      }
      double acc = a + __shfl_xor_sync(t.mask, a, 1);
      if (DIAG) acc = acc * lu[dpos[row]];
      if (act && par == 0) z[row] = acc;
    }
    t.sync();
  }
}

// The trailing dense block (at most 32 rows, row i's entries from a + i m) of
// both substitutions in team order, by one warp with a row per lane in a
// register: a column costs a shuffle, a load and an FMA, without the
// barrier and the shared-memory round trip between columns.
template <int P, int S, class D>
__device__ __forceinline__ void solve_tail(const TNet<P, S, D>& t, const double* a, double* y,
                                           int m) {
  if (t.lane < 32) {
    const bool row = t.lane < m;
    const double* ai = a + (row ? t.lane : 0) * m;
    double v = row ? y[t.lane] : 0.0;
#pragma unroll 4
    for (int k = 0; k + 1 < m; ++k) {
      const double yk = t.shfl(v, k);
      const double l = ai[k];
      if (t.lane > k) v = fma(-l, yk, v);
    }
#pragma unroll 4
    for (int k = m - 1; k > 0; --k) {
      const double xk = t.shfl(v, k) * a[k * m + k];
      const double u = ai[k];
      if (t.lane < k) v = fma(-u, xk, v);
    }
    if (row) y[t.lane] = v * ai[t.lane];
  }
}

// w.y (right-hand side in position order, as newton_correct lays it out) ->
// M^-1 times it; the array that holds the solution, in position order
template <int P, int S, class D>
__device__ __forceinline__ const double* solve_M(const TNet<P, S, D>& t, const CWS& w) {
  const BlobHeader& h = t.h;
  const int16_t* dpos = t.template arr<int16_t>(h.o_dpos);
  const uint32_t* cl = t.template arr<uint32_t>(h.o_cl);
  const int32_t* cl_ptr = t.template arr<int32_t>(h.o_cl_ptr);
  const int n = t.n, c = h.tail, m = n - c;
  double *y = w.y.p, *z = w.y.p + 2 * n;
  t.sync();
  if constexpr (S > 0) {
    const uint32_t* cu = t.template arr<uint32_t>(h.o_cu);
    const int32_t* cu_ptr = t.template arr<int32_t>(h.o_cu_ptr);
    if (m <= 32) {
      solve_columns<P, S, false, false>(t, w.lu.p, cl, cl_ptr, dpos, y, z, 0, c);
      solve_tail(t, w.lu.p + h.tail_slot, y + c, m);
      t.sync();
      // the rows above the block take its columns, last first
      const uint32_t* ru = t.template arr<uint32_t>(h.o_ru);
      const int32_t* ru_ptr = t.template arr<int32_t>(h.o_ru_ptr);
      const int32_t* ru_tail = t.template arr<int32_t>(h.o_ru_tail);
      for (int i = t.lane; i < c; i += P) {
        double v = y[i];
        const int e0 = ru_tail[i];
#pragma unroll 4
        for (int e = ru_ptr[i + 1] - 1; e >= e0; --e) {
          const uint32_t pk = ru[e];
          v = fma(-w.lu[pk & 0xffff], y[pk >> 16], v);
        }
        y[i] = v;
      }
      t.sync();
      solve_columns<P, S, true, true>(t, w.lu.p, cu, cu_ptr, dpos, y, z, 0, c);
    } else {
      solve_columns<P, S, false, false>(t, w.lu.p, cl, cl_ptr, dpos, y, z, 0, n);
      solve_columns<P, S, true, true>(t, w.lu.p, cu, cu_ptr, dpos, y, z, 0, n);
    }
    return y;
  } else {
    solve_columns<P, S, false, false>(t, w.lu.p, cl, cl_ptr, dpos, y, z, 0, n);
    solve_rows<P, S, true>(t, w.lu.p, t.template arr<uint32_t>(h.o_ru),
                           t.template arr<int32_t>(h.o_ru_ptr),
                           t.template arr<int16_t>(h.o_ru_row),
                           t.template arr<int16_t>(h.o_ru_lev), h.n_ru_lev, dpos, z);
    return z;
  }
}

// ---------------------------------------------------------------- step pieces

// alpha_0 in every thread, alpha_j at point j
template <int P, int S, class D>
struct step_alpha<TNet<P, S, D>> {
  using T = TNet<P, S, D>;
  double a0, aj[T::NP];
  unsigned mask;
  __device__ __forceinline__ double operator[](int j) const {
    if (j == 0) return a0;
    if constexpr (T::NP == 1) return __shfl_sync(mask, aj[0], j, T::SW);
    else return __shfl_sync(mask, j < T::SW ? aj[0] : aj[1], j & (T::SW - 1), T::SW);
  }
};

// out_i = sum_{j<cnt} c_j xh[history j0 + j], c_j held by point j + c0
template <int P, int S, class D, class OUT>
__device__ __forceinline__ void team_combine(const TNet<P, S, D>& t, const Zone& s, const CWS& w,
                                             int cnt, int j0,
                                             const double (&c)[TNet<P, S, D>::NP], int c0,
                                             OUT out) {
  double cj[KMAX + 1];
  int base[KMAX + 1];
#pragma unroll
  for (int j = 0; j <= KMAX; ++j) {
    cj[j] = t.pick(c, j + c0);
    base[j] = hslot(s, j0 + j < HMAX ? j0 + j : 0) * t.n;
  }
  for (int i = t.lane; i < t.n; i += P) {
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j <= KMAX; ++j)
      if (j < cnt) acc = fma(cj[j], w.xh[base[j] + i], acc);
    out(i, acc);
  }
}

// bdf_alpha, point j's lane forming alpha_j from its time tj (t_new at point
// 0 and at idle ones): the team spends one coefficient's instructions instead
// of k
template <int P, int S, class D>
__device__ __forceinline__ void team_alpha(const TNet<P, S, D>& t, int kk, double t_new,
                                           const double (&tj)[TNet<P, S, D>::NP], double h,
                                           step_alpha<TNet<P, S, D>>& alpha) {
  constexpr int NP = TNet<P, S, D>::NP;
  double ej[NP], rj[NP], num[NP], den[NP];
#pragma unroll
  for (int r = 0; r < NP; ++r) {
    const bool mine = t.point(r) >= 1 && t.point(r) <= kk;
    ej[r] = t_new - tj[r];
    rj[r] = 1.0 / (mine ? ej[r] : 1.0);
    num[r] = den[r] = 1.0;
  }
  double acc = 0.0;
  for (int m = 1; m <= kk; ++m) acc += t.pick(rj, m);
  for (int m = 0; m <= kk; ++m) {
    const double em = t.pick(ej, m), tm = t.pick(tj, m);
#pragma unroll
    for (int r = 0; r < NP; ++r)
      if (m != t.point(r)) {
        if (m != 0) num[r] *= em;
        den[r] *= tj[r] - tm;
      }
  }
  alpha.mask = t.mask;
  alpha.a0 = h * acc;
#pragma unroll
  for (int r = 0; r < NP; ++r) {
    const bool mine = t.point(r) >= 1 && t.point(r) <= kk;
    alpha.aj[r] = h * num[r] / (mine ? den[r] : 1.0);
  }
}

template <int P, int S, class D>
__device__ __forceinline__ void step_coeffs(const TNet<P, S, D>& t, const Zone& s, CWS& w,
                                            double atol, double rtol, double h, double t_new,
                                            int kk, step_alpha<TNet<P, S, D>>& alpha) {
  double tj[TNet<P, S, D>::NP];
#pragma unroll
  for (int r = 0; r < TNet<P, S, D>::NP; ++r) {
    const int l = t.point(r);
    tj[r] = l >= 1 && l <= kk ? w.th[hslot(s, l - 1)] : t_new;
  }
  team_alpha(t, kk, t_new, tj, h, alpha);
  team_combine(t, s, w, kk, 0, alpha.aj, 1, [&](int i, double a) { w.psi[i] = a; });
  const int b0 = hslot(s, 0) * t.n;
  for (int i = t.lane; i < t.n; i += P) w.iw[i] = recip1(atol + rtol * fabs(w.xh[b0 + i]));
}

// the Lagrange weights at tt over history j0..j0+q (lagrange_weights), one
// per point
template <int P, int S, class D>
__device__ __forceinline__ void team_lagrange(const TNet<P, S, D>& t, const Zone& s, const CWS& w,
                                              int j0, int q, double tt,
                                              double (&lw)[TNet<P, S, D>::NP]) {
  constexpr int NP = TNet<P, S, D>::NP;
  double tj[NP], ej[NP], num[NP], den[NP];
#pragma unroll
  for (int r = 0; r < NP; ++r) {
    tj[r] = w.th[hslot(s, t.point(r) <= q ? j0 + t.point(r) : j0)];
    ej[r] = tt - tj[r];
    num[r] = den[r] = 1.0;
  }
  for (int m = 0; m <= q; ++m) {
    const double em = t.pick(ej, m), tm = t.pick(tj, m);
#pragma unroll
    for (int r = 0; r < NP; ++r)
      if (m != t.point(r)) {
        num[r] *= em;
        den[r] *= tj[r] - tm;
      }
  }
#pragma unroll
  for (int r = 0; r < NP; ++r) lw[r] = num[r] / (t.point(r) <= q ? den[r] : 1.0);
}

template <int P, int S, class D>
__device__ __forceinline__ void predict(const TNet<P, S, D>& t, const Zone& s, CWS& w, int q,
                                        double t_new) {
  double lw[TNet<P, S, D>::NP];
  team_lagrange(t, s, w, 0, q, t_new, lw);
  team_combine(t, s, w, q + 1, 0, lw, 0, [&](int i, double a) { w.xp[i] = a; });
}

template <int P, int S, class D>
__device__ __forceinline__ double newton_correct(const TNet<P, S, D>& t, CWS& w, double alpha0,
                                                 double h) {
  const int16_t* pos = t.template arr<int16_t>(t.h.o_pos);
  double* y = w.y.p;
  for (int i = t.lane; i < t.n; i += P) {
    const double d = -(fma(alpha0, w.x[i], w.psi[i]) - h * w.f[i]);
    if constexpr (S > 0) {
      y[pos[i]] = d;
    } else {
      y[2 * pos[i]] = d;
      y[2 * pos[i] + 1] = 0.0;
    }
  }
  const double* z = solve_M(t, w);
  double nrm;
  if constexpr (S > 0) {
    nrm = t.sum_team(t.n, [&](int i, double a) {
      const double q = z[pos[i]] * w.iw[i];
      return fma(q, q, a);
    });
    for (int i = t.lane; i < t.n; i += P) w.x[i] += z[pos[i]];
    t.sync();
  } else {
    for (int i = t.lane; i < t.n; i += P) {
      const double d = z[pos[i]];
      w.x[i] += d;
      w.tmp[i] = d * w.iw[i];
    }
    t.sync();
    nrm = t.sum2(t.n, [&](int i, double a) { return fma(w.tmp[i], w.tmp[i], a); });
  }
  return nrm * t.inv_n;
}

// sum of the squares of v(i) over the state
template <int P, int S, class D, class F>
__device__ __forceinline__ double team_square(const TNet<P, S, D>& t, CWS& w, F v) {
  if constexpr (S > 0) {
    return t.sum_team(t.n, [&](int i, double a) {
      const double q = v(i);
      return fma(q, q, a);
    });
  } else {
    t.sync();
    for (int i = t.lane; i < t.n; i += P) w.tmp[i] = v(i);
    t.sync();
    return t.sum1(t.n, [&](int i, double a) { return fma(w.tmp[i], w.tmp[i], a); });
  }
}

template <int P, int S, class D>
__device__ __forceinline__ double error_norm2(const TNet<P, S, D>& t, CWS& w, double c) {
  return team_square(t, w, [&](int i) { return c * (w.x[i] - w.xp[i]) * w.iw[i]; }) * t.inv_n;
}

template <int P, int S, class D>
__device__ __forceinline__ double order_estimate(const TNet<P, S, D>& t, const Zone& s, CWS& w,
                                                 int q, double h) {
  const double t0 = w.th[hslot(s, 0)];
  double lw[TNet<P, S, D>::NP];
  team_lagrange(t, s, w, 1, q, t0, lw);
  const double c = h / (t0 - w.th[hslot(s, q + 1)]);
  const int b0 = hslot(s, 0) * t.n;
  double cj[KMAX + 1];
  int base[KMAX + 1];
#pragma unroll
  for (int j = 0; j <= KMAX; ++j) {
    cj[j] = t.pick(lw, j);
    base[j] = hslot(s, j + 1) * t.n;
  }
  return team_square(t, w, [&](int i) {
    double a = 0.0;
#pragma unroll
    for (int j = 0; j <= KMAX; ++j)
      if (j <= q) a = fma(cj[j], w.xh[base[j] + i], a);
    return c * (w.xh[b0 + i] - a) * w.iw[i];
  }) * t.inv_n;
}

// the step factors of the three orders, one per lane: one exp and log for
// the team instead of three
template <int P, int S, class D>
__device__ __forceinline__ double order_factor(const TNet<P, S, D>& t, const Zone& s, CWS& w,
                                               double err2, double h, int& best_q) {
  const int k = s.k;
  const bool lower = k > 1, higher = k < KMAX && s.nh >= k + 3;
  const double e1 = lower ? order_estimate(t, s, w, k - 1, h) : err2;
  const double e2 = higher ? order_estimate(t, s, w, k + 1, h) : err2;
  const int l = t.wl();
  const double f = step_factor(l == 1 ? e1 : l == 2 ? e2 : err2, l == 1 ? k - 1 : l == 2 ? k + 1 : k);
  best_q = k;
  double best = t.shfl(f, 0);
  const double f1 = t.shfl(f, 1), f2 = t.shfl(f, 2);
  if (lower && f1 > best) { best = f1; best_q = k - 1; }
  if (higher && f2 > best) { best = f2; best_q = k + 1; }
  return best;
}

// ---------------------------------------------------------------- claim loop

// Thread 0 of a team claims zones from the device queue and the team
// integrates them, one step attempt per turn of the loop, so that the teams
// of one warp stay in step.  The watchdog reads thread 0's clock, so the
// team decides as one.
template <int P, int S, class D>
__device__ __forceinline__ void coop_claim_loop(const TNet<P, S, D>& t, CWS& w,
                                                const BurnParams& B) {
  unsigned long long t_start = 0ull;
  if (B.budget_ns) t_start = t.bcast(t.lane == 0 ? gpu_ns() : 0ull);
  Zone s;
  bool active = false;
  for (;;) {
    if (!active) {
      unsigned long long c = 0;
      if (t.lane == 0) c = atomicAdd(B.queue, 1ull);
      c = t.bcast(c);
      if (c >= (unsigned long long)B.Z) break;
      s.z = B.order ? (long long)B.order[c] : (long long)c;
    }
    bool expired = false;
    if (B.budget_ns) expired = t.bcast(t.lane == 0 ? gpu_ns() : 0ull) - t_start > B.budget_ns;
    bool done;
    if (expired) {
      if (!active) {
        zone_timeout_unstarted(t, s.z, B);
        continue;
      }
      s.status = NB_Z_TIMEOUT;
      done = true;
    } else {
      done = active ? zone_attempt(t, s, w, B) : zone_init(t, s, w, B);
    }
    active = !done;
    if (done) {
      zone_finish(t, s, w, B);
      t.sync();
    }
  }
}

}  // namespace nb
