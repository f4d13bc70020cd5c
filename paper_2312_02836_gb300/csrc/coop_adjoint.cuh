// coop_adjoint.cuh -- the reverse sweep's steps (adjoint.cuh) by a team of
// threads (coop.cuh): the K cotangent sets of a step are solved together.
#pragma once
#include "adjoint.cuh"
#include "coop.cuh"

namespace nb {

// a team's adjoint arrays, offsets in doubles from its first one (64 bits: a
// tape's stride may be any number, and the recomputed block has that many
// states)
struct TeamAdj {
  long long lam, ee, gr, gt, mu, de, seg, ce, vs, total;
};

// mu: K solve vectors; ce: e_q h / alpha_0; vs: [K, R] rate terms (lane order
// at fixed temperature: each set's T9 sum is one chain over its rates)
struct TAWS {
  CV lam, ee, gr, gt, mu, de, seg, ce, vs;
};

__device__ __forceinline__ TAWS make_taws(const TeamAdj& A, double* base) {
  TAWS a;
  a.lam.p = base + A.lam; a.ee.p = base + A.ee; a.gr.p = base + A.gr; a.gt.p = base + A.gt;
  a.mu.p = base + A.mu; a.de.p = base + A.de; a.seg.p = base + A.seg; a.ce.p = base + A.ce;
  a.vs.p = base + A.vs;
  return a;
}

// doubles of one solve vector
__host__ __device__ constexpr int team_mu(int n, int S) { return S > 0 ? n : 3 * n; }

// offsets of a team's adjoint arrays for K cotangent sets
inline void team_layout(const BlobHeader& h, int K, int stride, int S, TeamAdj* a) {
  long long off = 0;
  auto take = [&](long long cnt) { const long long o = off; off += cnt; return o; };
  a->lam = take((long long)HMAX * K * h.n);
  a->ee = take(HMAX * K);
  a->gr = take((long long)K * h.R);
  a->gt = take(K);
  a->mu = take((long long)K * team_mu(h.n, S));
  a->de = take(h.n);
  a->seg = take((long long)stride * h.n);
  a->ce = take(K);
  a->vs = take(h.self_heating ? 0 : (long long)(S > 0 ? 1 : K) * h.R);
  a->total = (off + 1) & ~1LL;
}

// v_q <- M^-T v_q of K vectors at once, each n (team order) or 3 n (lane
// order: partial sums, then the solution) doubles from v + q * stride in
// position order.  All vectors share a column's barrier, and their updates
// fill the lanes that one column of one vector leaves idle.
template <int P, int S, bool DIAG, bool UP, class D>
__device__ __forceinline__ void solve_columns_k(const TNet<P, S, D>& t, const double* lu,
                                                const uint32_t* ent, const int32_t* ptr,
                                                const int16_t* dpos, double* v, int stride,
                                                int K) {
  const int n = t.n;
  for (int it = 0; it < n; ++it) {
    const int k = UP ? n - 1 - it : it;
    const int e0 = ptr[k], len = ptr[k + 1] - e0;
    if (S == 0 || DIAG) {
      const double dv = DIAG ? lu[dpos[k]] : 1.0;
      for (int q = t.lane; q < K; q += P) {
        double* y = v + q * stride;
        double xk = S > 0 ? y[k] : y[2 * k] + y[2 * k + 1];
        if (DIAG) xk = xk * dv;
        y[S > 0 ? k : 2 * n + k] = xk;
      }
      t.sync();
    }
    if (len > 0) {
      const int qW = P / len, rW = P - qW * len;
      int q = t.lane / len, r = t.lane - q * len;
      for (int e = t.lane; e < K * len; e += P) {
        const uint32_t pk = ent[e0 + r];
        double* y = v + q * stride;
        double* tgt = y + (S > 0 ? pk >> 17 : pk >> 16);
        *tgt = fma(-lu[pk & 0xffff], y[S > 0 ? k : 2 * n + k], *tgt);
        q += qW;
        r += rW;
        if (r >= len) { r -= len; ++q; }
      }
    }
    t.sync();
  }
}

template <int P, int S, class D>
__device__ __forceinline__ void solve_MT_k(const TNet<P, S, D>& t, const double* lu, double* v,
                                           int stride, int K) {
  const BlobHeader& h = t.h;
  const int16_t* dpos = t.template arr<int16_t>(h.o_dpos);
  t.sync();
  solve_columns_k<P, S, true, false>(t, lu, t.template arr<uint32_t>(h.o_cut),
                                     t.template arr<int32_t>(h.o_cut_ptr), dpos, v, stride, K);
  if constexpr (S > 0) {
    solve_columns_k<P, S, false, true>(t, lu, t.template arr<uint32_t>(h.o_clt),
                                       t.template arr<int32_t>(h.o_clt_ptr), dpos, v, stride, K);
  } else {
    const uint32_t* ent = t.template arr<uint32_t>(h.o_rlt);
    const int32_t* ptr = t.template arr<int32_t>(h.o_rlt_ptr);
    const int16_t *rows = t.template arr<int16_t>(h.o_rlt_row),
                  *lev = t.template arr<int16_t>(h.o_rlt_lev);
    const int par = t.lane & 1;
    for (int g = 0; g < h.n_rlt_lev; ++g) {
      const int r0 = lev[g], cnt = lev[g + 1] - r0;
      for (int b = 0; b < K * cnt; b += P / 2) {
        const int e = b + (t.lane >> 1);
        const bool act = e < K * cnt;
        const int q = act ? e / cnt : 0;
        const int row = rows[r0 + (act ? e - q * cnt : 0)];
        double* z = v + q * stride + 2 * t.n;
        double a = 0.0;
        if (act) {
          if (par == 0) a = z[row];
          for (int i = ptr[row] + par; i < ptr[row + 1]; i += 2) {
            const uint32_t pk = ent[i];
            a = fma(-lu[pk & 0xffff], z[pk >> 16], a);
          }
        }
        const double acc = a + __shfl_xor_sync(t.mask, a, 1);
        if (act && par == 0) z[row] = acc;
      }
      t.sync();
    }
  }
}

template <int P, int S, class D>
__device__ __forceinline__ void adj_alpha(const TNet<P, S, D>& t, const AdjParams& A, long long z,
                                          int s, int kk, double h,
                                          step_alpha<TNet<P, S, D>>& alpha) {
  const double t_new = sched_ptr(A, z, s)[0];
  double tj[TNet<P, S, D>::NP];
#pragma unroll
  for (int r = 0; r < TNet<P, S, D>::NP; ++r) {
    const int l = t.point(r);
    tj[r] = l >= 1 && l <= kk ? sched_ptr(A, z, s - l)[0] : t_new;
  }
  team_alpha(t, kk, t_new, tj, h, alpha);
}

template <int P, int S, class D>
__device__ __forceinline__ void edot_gradient(const TNet<P, S, D>& t, const CWS& w, const TAWS& a) {
  const BlobHeader& h = t.h;
  const double* Q = t.template arr<double>(h.o_Q);
  const int32_t* ptr = t.template arr<int32_t>(h.o_dej_ptr);
  const int16_t *dej = t.template arr<int16_t>(h.o_dej_d),
                *dt_r = t.template arr<int16_t>(h.o_dt_r);
  t.sync();
  for (int j = t.lane; j < t.N; j += P) {
    double acc = 0.0;
    for (int e = ptr[j]; e < ptr[j + 1]; ++e) {
      const int d = dej[e];
      acc += Q[dt_r[d]] * w.dt[d];
    }
    a.de[j] = acc;
  }
  if (t.sh) {
    const double acc = t.sum1(t.R, [&](int r, double e) { return fma(Q[r], w.dt[h.nd + r], e); });
    if (t.lane == 0) a.de[t.N] = acc;
  }
  t.sync();
}

template <int P, int S, class D>
__device__ __forceinline__ void adj_sets(const TNet<P, S, D>& t, const CWS& w, const TAWS& a, int K,
                                         int kk, int sl, const int* sj,
                                         const step_alpha<TNet<P, S, D>>& alpha, double h,
                                         double ia0, double icv) {
  const BlobHeader& hd = t.h;
  const int n = t.n, R = t.R, st = team_mu(n, S), so = S > 0 ? 0 : 2 * n;
  const int16_t* pos = t.template arr<int16_t>(hd.o_pos);
  for (int q = t.lane; q < K; q += P) a.ce[q] = a.ee[sl * K + q] * h * ia0;
  t.sync();
  for (int q = 0; q < K; ++q) {
    const int lo = (sl * K + q) * n;
    double* y = a.mu.p + q * st;
    for (int i = t.lane; i < n; i += P) {
      double v = a.lam[lo + i];
      if (t.hasE) v = fma(a.ce[q], a.de[i], v);
      if constexpr (S > 0) {
        y[pos[i]] = v;
      } else {
        y[2 * pos[i]] = v;
        y[2 * pos[i] + 1] = 0.0;
      }
      a.lam[lo + i] = 0.0;
    }
  }
  solve_MT_k(t, w.lu.p, a.mu.p, st, K);
#pragma unroll
  for (int j = 1; j <= KMAX; ++j) {
    if (j > kk) continue;
    const double aj = alpha[j], ma = -aj;
    for (int q = 0; q < K; ++q) {
      const int lj = (sj[j] * K + q) * n;
      const double* z = a.mu.p + q * st + so;
      for (int i = t.lane; i < n; i += P) a.lam[lj + i] = fma(ma, z[pos[i]], a.lam[lj + i]);
    }
    if (t.hasE)
      for (int q = t.lane; q < K; q += P)
        a.ee[sj[j] * K + q] = fma(-a.ee[sl * K + q] * ia0, aj, a.ee[sj[j] * K + q]);
  }
  for (int q = t.lane; q < K; q += P) a.ee[sl * K + q] = 0.0;
  const double *Q = t.template arr<double>(hd.o_Q), *rg_c = t.template arr<double>(hd.o_rg_c);
  const int32_t* rg_ptr = t.template arr<int32_t>(hd.o_rg_ptr);
  const int16_t* rg_i = t.template arr<int16_t>(hd.o_rg_i);
  for (int q = 0; q < K; ++q) {
    const double* z = a.mu.p + q * st + so;
    const double ce = a.ce[q];
    const double muT = t.sh ? z[pos[t.N]] * icv : 0.0;
    auto term = [&](int r) {
      double acc = 0.0;
      for (int e = rg_ptr[r]; e < rg_ptr[r + 1]; ++e) acc = fma(rg_c[e], z[pos[rg_i[e]]], acc);
      const double Qr = Q[r];
      acc = fma(muT, Qr, acc);
      return w.rr[r] * fma(h, acc, ce * Qr);
    };
    if (t.sh) {
      for (int r = t.lane; r < R; r += P) a.gr[q * R + r] += term(r);
    } else {
      double* vs = a.vs.p + (S > 0 ? 0 : q * R);
      if (S > 0) t.sync();   // the set before has read vs
      for (int r = t.lane; r < R; r += P) {
        const double v = term(r);
        a.gr[q * R + r] += v;
        vs[r] = v;
      }
      if constexpr (S > 0) {
        t.sync();
        const double gt = t.sum_team(R, [&](int r, double e) { return fma(vs[r], w.g[r], e); });
        if (t.lane == 0) a.gt[q] += gt;
      }
    }
  }
  if constexpr (S == 0) {
    if (!t.sh) {
      t.sync();
      for (int q = t.lane; q < K; q += P) {
        double gt = 0.0;
        for (int r = 0; r < R; ++r) gt = fma(a.vs[q * R + r], w.g[r], gt);
        a.gt[q] += gt;
      }
    }
  }
  t.sync();
}

}  // namespace nb
