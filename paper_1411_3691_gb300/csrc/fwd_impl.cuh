// fwd_impl.cuh -- forward correlator kernel, block factors, batched kernel and per-pair probe
// (templates; instantiated once per n class and kernel by fwd_*.cu, batch_nc*.cu and pair_nc*.cu).
//
// One thread block per work item (work family W, tile of `tile` sinks); one thread per
// sink.  Per flavour a thread factorises the family's shared rows against its sink's
// columns (shared_rows) and caches y = det(G) G^{-1} e_r in shared memory; then every
// member of the family costs one O(n) dot product per flavour, Sec. 2.1: in fixed point on the
// integer pipe (fx_dots, fx_det2), or in FP64 (member_det) in calls without tables, on propagators that
// do not suit them, and where a fixed-point value is out of its range, small, or near the lemma guard.
// Two-sided blocks (a family against a sink family) take y from factors stored once per
// block (kapply*).  Members whose lemma factor or whose family pivots fail the guards go
// to a per-warp queue and are refactored from scratch 32 at a time -- pairs that share the
// member and the sink family's columns as one group (group_fresh), so the FP64 pipe stays
// occupied.  Thread sums are reduced in a fixed order into one partial per work item (and
// by reduce_kernel into C): bitwise reproducible.
#pragma once

#include "kernels.cuh"

namespace mhc {

namespace fwd {

struct QEntry {
  int32_t member;  // member slot
  int32_t lane;    // lane (sink) of the warp that produced it
  int32_t fail;    // flavours to refactor (bit f)
  int32_t pguard;  // of those, the flavours whose shared rows failed the pivot guard
  double2 prod;    // product of the flavours that did not fail
  double2 w;       // signed w_i w_j of the pair
};

// Algorithmic flops of the refactor path, counted with the planner's rule (real add/mul 1,
// FMA 2, complex multiply 6, complex FMA 8, complex reciprocal 6, pivot measure 1):
// a fresh partial-pivot LU determinant of one n x n block, ...
__device__ __forceinline__ unsigned long long fresh_flops(int n) {
  const long long m = n;
  return (unsigned long long)(m * (m + 1) / 2 + 6 * (m - 1) + 3 * m * (m - 1) +
                              8 * (m - 1) * m * (2 * m - 1) / 6 + 6 * (m - 1));
}
// ... and a grouped refactor (group_fresh) of pairs whose matrices share their first
// n - rc columns: the group's elimination of those columns and the rows of L^{-1} P of the
// rc remaining rows (one complex multiply-add per unused row and step) ...
__device__ __forceinline__ unsigned long long group_shared_flops(int n, int rc) {
  long long f = 0;
  const int M = n - rc;
  for (int k = 0; k < M; k++)
    f += (n - k) + 6 + 6 * (n - k - 1) + 8 * (n - k - 1) * (M - 1 - k) + 8 * rc * (n - k - 1);
  return (unsigned long long)(f + 6 * (M > 1 ? M - 1 : 0));
}
// ... and each pair's share: rc x rc dot products of length n, the last rc x rc step (for
// rc = 2: two pivot measures, a reciprocal, a multiplier, one update, two products) and
// the product with the shared pivots.
__device__ __forceinline__ unsigned long long group_pair_flops(int n, int rc) {
  return (unsigned long long)(rc * rc * (8LL * n - 2) + (rc == 2 ? 2 + 6 + 6 + 8 + 12 : 6));
}

// Pivot search of one step of group_fresh: the largest |re| + |im| in column k (rk: this
// lane's entry) among the unused rows, by one warp-wide maximum of a key made of the
// measure's sign, exponent and leading 15 mantissa bits with (31 - lane) below them: a pivot
// within 2^-15 of the largest, the lowest row of those -- partial pivoting up to that tie
// tolerance; a zero measure keeps key bits 5..31 zero, which is how an exactly zero pivot
// column shows.  Updates the used rows, the permutation's parity, the determinant and the
// pivot's reciprocal.  Called by the whole warp.
struct PivotState {
  unsigned piv;  // rows already used as pivots
  int mystep;    // the step at which this lane's row became the pivot (NC: never)
  int parity;
  bool zero;
  dev::cd det;
  int p;         // this step's pivot row
  dev::cd rc;    // its reciprocal
};
__device__ __forceinline__ void select_pivot(PivotState& s, dev::cd rk, int k, int n, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  const bool cand = lane < n && !((s.piv >> lane) & 1);
  const unsigned mkey = cand ? (((unsigned)__double2hiint(dev::abs1(rk)) & ~31u) | (unsigned)(31 - lane)) : 0u;
  const unsigned top = __reduce_max_sync(FULL, mkey);
  const int p = 31 - (int)(top & 31u);
  // the permutation's parity: p moves ahead of the unused rows that precede it
  s.parity ^= __popc(~s.piv & ((1u << p) - 1u) & ((1u << n) - 1u)) & 1;
  s.piv |= 1u << p;
  s.mystep = lane == p ? k : s.mystep;
  s.zero |= (top >> 5) == 0u;
  const dev::cd pk = make_double2(__shfl_sync(FULL, rk.x, p), __shfl_sync(FULL, rk.y, p));
  s.det = (k == 0) ? pk : dev::cmul(s.det, pk);
  s.rc = dev::crcp(pk);
  s.p = p;
}

// Fresh determinants of a group of queued pairs that share member m and a two-sided sink
// family Q whose members change RC columns of flavour f (RC = 1 or 2; family of rank rho):
// their matrices G = [R | A_j] agree in the first n - RC columns R (the family's n - rho
// shared rows and the member's rho rows, in member_rows order, against the sink family's
// shared columns) and differ in the last RC columns A_j.  Partial-pivot LU eliminates
// column by column, so the first n - RC steps are those of R for every pair: P R = L [U; 0],
// and the last RC rows of L^{-1} P A_j form the RC x RC block that the last steps factorise,
// det G = sign(P) det(U) det(V A_j) with V the rows of L^{-1} P that belong to the RC rows
// left after the shared steps.  The warp factorises R once (lane i holds row i and keeps
// its multiplier of every step), forms V by walking the steps backwards (the coefficient of
// a step's pivot row is minus the warp sum, over the rows still unused at that step, of
// multiplier times coefficient), and each lane of the group then needs RC x RC dot products
// of length n with its own sink's columns and the last RC x RC step with the same pivot
// rule.  Called by the whole warp; returns the determinant on the lanes in grp.
template <int NC, int RC>
__device__ __forceinline__ dev::cd group_fresh(const FwdArgs& a, int W, int f, int rho, int m, int Q,
                                               int64_t j, unsigned grp, dev::cd* wk) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NR = NC - RC > 0 ? NC - RC : 1;
  const int lane = threadIdx.x & 31;
  const int n = a.n_f[f];
  const int M = n - RC;  // shared columns: the common elimination steps
  const int L = a.L_f[f];
  const dev::cd* S = a.S[f];
  const int32_t* arow = a.fam_arow + (int64_t)W * a.Tn + a.off_f[f];
  const int32_t* mlab = a.mem_lab + ((int64_t)m * a.F + f) * MHC_MAX_RANK;
  const int32_t* scol = a.snk_pos + (int64_t)a.q_off[Q] * a.Tn + a.off_f[f];
  // label of row i: the family's shared rows, then the member's changed rows
  auto row_label = [&](int i) { return i < n - rho ? arow[i] : mlab[min(i - (n - rho), rho - 1)]; };
  const int rlab = row_label(min(lane, n - 1));
  dev::cd R[NR];
#pragma unroll
  for (int u = 0; u < NR; u++)
    R[u] = (lane < n && u < M) ? dev::ldS(S + (size_t)rlab * L + scol[u]) : make_double2(0.0, 0.0);
  PivotState ps;
  ps.piv = 0;
  ps.mystep = NC;
  ps.parity = 0;
  ps.zero = false;
  ps.det = make_double2(1.0, 0.0);
  if (M > 0) select_pivot(ps, R[0], 0, n, lane);
  // Step k: the multipliers of column k, then column k + 1 updated first and the pivot of
  // step k + 1 chosen (with its reciprocal) before the other columns of step k, so that the
  // chain of the next pivot (maximum, broadcast, reciprocal) overlaps independent updates.
  // The values are those of the plain order: each entry sees the same operations.
#pragma unroll
  for (int k = 0; k < NR; k++) {
    if (k >= M) break;
    const int p = ps.p;
    const bool act = lane < n && !((ps.piv >> lane) & 1);
    const dev::cd l = dev::cmul(R[k], ps.rc);
    if (k + 1 < NR && k + 1 < M) {
      const dev::cd pu = make_double2(__shfl_sync(FULL, R[k + 1].x, p), __shfl_sync(FULL, R[k + 1].y, p));
      if (act) R[k + 1] = dev::cfms(l, pu, R[k + 1]);
      select_pivot(ps, R[k + 1], k + 1, n, lane);
    }
#pragma unroll
    for (int u = k + 2; u < NR; u++) {
      if (u >= M) break;
      const dev::cd pu = make_double2(__shfl_sync(FULL, R[u].x, p), __shfl_sync(FULL, R[u].y, p));
      if (act) R[u] = dev::cfms(l, pu, R[u]);
    }
    if (act) R[k] = l;  // this row's multiplier of step k
  }
  const unsigned piv = ps.piv;
  const int mystep = ps.mystep;
  int parity = ps.parity;
  bool zero = ps.zero;
  dev::cd det = ps.det;
  // the RC rows left after the shared steps, ascending
  const unsigned rest = ~piv & ((1u << n) - 1u);
  int left[RC];
  left[0] = __ffs(rest) - 1;
  if (RC == 2) left[RC - 1] = __ffs(rest & ~(1u << left[0])) - 1;
  // V: lane i holds the coefficient of row i in each remaining row's functional.  In the
  // order of the steps (position s < M: the pivot row of step s; M + t: the t-th remaining
  // row), the functional's coefficient at position s is minus the sum, over the later
  // positions s', of the multiplier of row s' at step s times the coefficient at s' -- a
  // back substitution with the unit lower factor.  The multipliers are staged by step in
  // the warp's shared scratch wk (column s: positions s + 1 .. n - 1, packed), and the
  // substitution runs as pushes: once position s' is final it is broadcast and every
  // earlier position adds its term, so the dependency chain per position is one shuffle and
  // one complex multiply-add.
  const int pos = mystep < NC ? mystep : (lane == left[0] ? M : M + RC - 1);
  auto woff = [&](int c) { return c * (n - 1) - c * (c - 1) / 2; };  // column c of the packed store
  __syncwarp();
#pragma unroll
  for (int k = 0; k < NR; k++) {
    if (k >= M) break;
    if (lane < n && k < pos) wk[woff(k) + pos - k - 1] = R[k];  // this row's multiplier at step k
  }
  __syncwarp();
  dev::cd acc[RC];
#pragma unroll
  for (int t = 0; t < RC; t++)  // the remaining rows: coefficient 1 in their own functional
    acc[t] = lane < M ? wk[woff(lane) + M + t - lane - 1] : make_double2(0.0, 0.0);
#pragma unroll
  for (int sp = NR - 1; sp >= 1; sp--) {
    if (sp >= M) continue;
    dev::cd v[RC];
#pragma unroll
    for (int t = 0; t < RC; t++)
      v[t] = dev::cneg(make_double2(__shfl_sync(FULL, acc[t].x, sp), __shfl_sync(FULL, acc[t].y, sp)));
    if (lane < sp) {
      const dev::cd w = wk[woff(lane) + sp - lane - 1];
#pragma unroll
      for (int t = 0; t < RC; t++) acc[t] = dev::cfma(w, v[t], acc[t]);
    }
  }
  // back to row order: row i takes the coefficient of its position
  const int src = pos < M ? pos : 0;
  dev::cd V[RC];
#pragma unroll
  for (int t = 0; t < RC; t++) {
    const dev::cd x = make_double2(-__shfl_sync(FULL, acc[t].x, src), -__shfl_sync(FULL, acc[t].y, src));
    V[t] = lane >= n ? make_double2(0.0, 0.0) : pos < M ? x : make_double2(pos == M + t ? 1.0 : 0.0, 0.0);
  }
  // each lane: its sink's last RC columns against the RC functionals
  const bool mine = (grp >> lane) & 1;
  const int32_t* cj = dev::sink_cols(a, j) + a.off_f[f];
  dev::cd D[RC][RC];
#pragma unroll
  for (int t = 0; t < RC; t++)
#pragma unroll
    for (int u = 0; u < RC; u++) D[t][u] = make_double2(0.0, 0.0);
  int lc[RC];
#pragma unroll
  for (int u = 0; u < RC; u++) lc[u] = mine ? cj[n - RC + u] : 0;
#pragma unroll
  for (int i = 0; i < NC; i++) {
    if (i >= n) break;
    const int li = row_label(i);
    dev::cd vi[RC];
#pragma unroll
    for (int t = 0; t < RC; t++) vi[t] = make_double2(__shfl_sync(FULL, V[t].x, i), __shfl_sync(FULL, V[t].y, i));
#pragma unroll
    for (int u = 0; u < RC; u++) {
      const dev::cd x = mine ? dev::ldS(S + (size_t)li * L + lc[u]) : make_double2(0.0, 0.0);
#pragma unroll
      for (int t = 0; t < RC; t++) D[t][u] = dev::cfma(vi[t], x, D[t][u]);
    }
  }
  if (RC == 1) {
    zero |= __double_as_longlong(dev::abs1(D[0][0])) == 0;
    det = M == 0 ? D[0][0] : dev::cmul(det, D[0][0]);
  } else {
    // last 2 x 2 step: pivot the larger |re| + |im| of the first column, ties to the lower row
    const double b0 = dev::abs1(D[0][0]), b1 = dev::abs1(D[RC - 1][0]);
    const bool swp = dev::gt_nonneg(b1, b0);
    parity ^= (int)swp;
    const dev::cd pv = swp ? D[RC - 1][0] : D[0][0], ov = swp ? D[0][0] : D[RC - 1][0];
    const dev::cd pw = swp ? D[RC - 1][RC - 1] : D[0][RC - 1], ow = swp ? D[0][RC - 1] : D[RC - 1][RC - 1];
    zero |= __double_as_longlong(swp ? b1 : b0) == 0;
    const dev::cd l = dev::cmul(ov, dev::crcp(pv));
    const dev::cd last = dev::cfms(l, pw, ow);
    zero |= __double_as_longlong(dev::abs1(last)) == 0;
    det = M == 0 ? dev::cmul(pv, last) : dev::cmul(dev::cmul(det, pv), last);
  }
  if (zero) return make_double2(0.0, 0.0);
  return parity ? dev::cneg(det) : det;
}

// does the sink family's block hold fixed-point factors of the one-column kind
__device__ __forceinline__ bool fx_block(const FwdArgs& a, int W, int Q, int f, bool qtwo) {
  return a.fx.nf > 0 && qtwo && a.q_rank[(int64_t)Q * a.F + f] == 1 && a.fam_rank[(int64_t)W * a.F + f] <= 2 &&
         !a.kguard[((int64_t)W * a.n_q + Q) * a.F + f];
}

// where the solves' exponents of flavour f start (WarpScratch)
__device__ __forceinline__ int fx_at(const FwdArgs& a, int f) { return f == a.fx.f0 ? 0 : 32; }

// complex factor of a flavour's fixed-point solve: det B of a block solved in fixed point, sd of
// a two-row family, else 1
__device__ __forceinline__ dev::cd fx_factor(const FwdArgs& a, int W, int Q, int f, bool blk, const double2* Yf, int T) {
  const int n = a.n_f[f];
  if (a.fam_rank[(int64_t)W * a.F + f] == 2) return Yf[2 * n * T];
  if (!blk) return make_double2(1.0, 0.0);
  return a.kbuf[((int64_t)W * a.n_q + Q) * a.kstride + a.koff[f] + (n - 1) * (n - 1) + n];
}

// Refactor one pair per lane (the lanes with have; e: the pair, j: its sink position):
// the product of the flavours that passed, times fresh determinants of the flavours that
// failed, accumulated into acc.  With a.rowdiff the row-difference update is tried first
// for members of one- and two-row families.  Pairs that share a member and a two-sided sink
// family with one or two changed columns (n <= 18) are factorised together (group_fresh);
// the others one per lane.  Yw: the warp's cached solves (lane l at Yw + l, stride
// blockDim.x), in fixed point with exponents eyw when fxm; wk: the warp's scratch for group_fresh.
// Called by the whole warp.
template <int NCMAX, bool FX, bool CW>
__device__ __forceinline__ void refactor_pairs(const FwdArgs& a, int W, bool have, const QEntry& e, int64_t j,
                                               const double2* Yw, bool fxm, const short* eyw, double2* wk,
                                               double2& acc, unsigned long long& rflops, unsigned long long& nrd) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int T = blockDim.x;
  const int32_t* cols = dev::sink_cols(a, j);
  double2 prod = have ? e.prod : make_double2(1.0, 0.0);
  int32_t fail = have ? e.fail : 0;
  const int Q = a.snk_orig ? a.snk_q[j] : -1;
  if (a.rowdiff && have) {
    // members of one- and two-row families that failed the lemma guard (not the pivot
    // guard): the row-difference update with the cached solve of the pair's sink (lane
    // e.lane of this warp) and its scale exponent as the solve's producer defines it
    const unsigned cand = (unsigned)(e.fail & ~e.pguard);
    for (int f = 0; f < a.F; f++) {
      const int n = a.n_f[f];
      const int rho = a.fam_rank[(int64_t)W * a.F + f];
      if (!((cand >> f) & 1) || rho > 2 || n < rho + 1) continue;
      const double2* Yf = Yw + (size_t)a.yoff[f] * T + e.lane;
      double2 yl[FX ? 2 * NCMAX + 1 : 1];  // the solve of the pair's sink, when it is not FP64
      const double2* y = Yf;
      int ys = T;
      if constexpr (FX) {
        if (fxm) {
          const int e2 = eyw[fx_at(a, f) + e.lane], eq = e2 >> 1;
          const double2 fac = fx_factor(a, W, Q, f, e2 & 1, Yf, T);
          for (int q = 0; q < rho * n; q++) {
            yl[q] = fx::value(reinterpret_cast<const int4*>(Yf)[q * T], eq);
            if (rho == 1) yl[q] = dev::cmul(yl[q], fac);
          }
          if (rho == 2) yl[2 * n] = fac;
          y = yl;
          ys = 1;
        }
      }
      const int ey = dev::cached_scale(y, ys, n, rho);
      bool f2 = true;
      const int32_t* mlab = a.mem_lab + ((int64_t)e.member * a.F + f) * MHC_MAX_RANK;
      const int32_t* arow = a.fam_arow + (int64_t)W * a.Tn + a.off_f[f];
      double2 d;
      if constexpr (NCMAX >= 10)  // two-row families need n_f >= 10
        d = rho == 1 ? dev::rowdiff_det(a.S[f], a.L_f[f], n, mlab[0], arow, cols + a.off_f[f], y, ys, ey, a.kc, &f2)
                     : dev::rowdiff2_det(a.S[f], a.L_f[f], n, mlab, arow, cols + a.off_f[f], y, ys, ey, a.kc, &f2);
      else
        d = dev::rowdiff_det(a.S[f], a.L_f[f], n, mlab[0], arow, cols + a.off_f[f], y, ys, ey, a.kc, &f2);
      rflops += rho == 1 ? dev::rowdiff_flops(n) : dev::rowdiff2_flops(n);
      if (!f2) {
        prod = dev::cmul(prod, d);
        fail &= ~(1 << f);
        nrd++;
      }
    }
  }
  int32_t rows[NCMAX];
  for (int f = 0; f < a.F; f++) {
    const bool need = have && ((fail >> f) & 1);
    const int n = a.n_f[f];
    const int rho = a.fam_rank[(int64_t)W * a.F + f];
    const int sig = (Q >= 0 && a.q_two[Q]) ? a.q_rank[(int64_t)Q * a.F + f] : 0;
    const bool grouped = need && NCMAX <= 18 && n >= 2 && sig == 1;
    const bool grouped2 = need && NCMAX <= 18 && n >= 3 && sig == 2;
    unsigned todo = __ballot_sync(FULL, grouped || grouped2);
    while (todo) {
      const int leader = __ffs(todo) - 1;
      const int lm = __shfl_sync(FULL, have ? e.member : 0, leader);
      const int lq = __shfl_sync(FULL, Q, leader);
      const int lsig = __shfl_sync(FULL, sig, leader);
      const unsigned grp = __ballot_sync(FULL, ((todo >> lane) & 1) && e.member == lm && Q == lq);
      const double2 d = lsig == 1 ? group_fresh<NCMAX <= 18 ? NCMAX : 18, 1>(a, W, f, rho, lm, lq, j, grp, wk)
                                  : group_fresh<NCMAX <= 18 ? NCMAX : 18, 2>(a, W, f, rho, lm, lq, j, grp, wk);
      if ((grp >> lane) & 1) {
        prod = dev::cmul(prod, d);
        rflops += group_pair_flops(n, lsig) + (lane == leader ? group_shared_flops(n, lsig) : 0ull);
      }
      todo &= ~grp;
    }
    if (need && !grouped && !grouped2) {
      dev::member_rows(a, W, e.member, f, rho, rows);
      const double2 d = dev::dispatch_fresh<NCMAX>(n, a.S[f], a.L_f[f], rows, cols + a.off_f[f]);
      prod = dev::cmul(prod, d);
      rflops += fresh_flops(n);
    }
  }
  if (have) acc = dev::add_weighted<CW>(a, e.w, prod, acc);
}

// With the fixed-point member loop a call, not inlined: that loop keeps its registers and the
// instruction cache its lines.
template <int NCMAX, bool CW>
__device__ __noinline__ void refactor_call(const FwdArgs& a, int W, bool have, const QEntry& e, int64_t j,
                                           const double2* Yw, bool fxm, const short* eyw, double2* wk, double2& acc,
                                           unsigned long long& rflops, unsigned long long& nrd) {
  refactor_pairs<NCMAX, true, CW>(a, W, have, e, j, Yw, fxm, eyw, wk, acc, rflops, nrd);
}

template <int NCMAX, bool FX, bool CW>
__device__ void process_pairs(const FwdArgs& a, int W, bool have, const QEntry& e, int64_t j, const double2* Yw,
                              bool fxm, const short* eyw, double2* wk, double2& acc, unsigned long long& rflops,
                              unsigned long long& nrd) {
  if constexpr (FX)
    refactor_call<NCMAX, CW>(a, W, have, e, j, Yw, fxm, eyw, wk, acc, rflops, nrd);
  else
    refactor_pairs<NCMAX, false, CW>(a, W, have, e, j, Yw, fxm, eyw, wk, acc, rflops, nrd);
}

// Refactor the first count queued pairs (one per lane).  Called by the whole warp.
template <int NCMAX, bool FX, bool CW>
__device__ void process_queue(const FwdArgs& a, int W, QEntry* q, int count, int64_t jbase,
                              const double2* Yw, bool fxm, const short* eyw, double2* wk, double2& acc,
                              unsigned long long& rflops, unsigned long long& nrd) {
  const int lane = threadIdx.x & 31;
  const bool have = lane < count;
  QEntry e = {};
  if (have) e = q[lane];
  process_pairs<NCMAX, FX, CW>(a, W, have, e, jbase + (have ? e.lane : 0), Yw, fxm, eyw, wk, acc, rflops, nrd);
}

// ---- solves and member dots in fixed point (fx.cuh) -------------------------------------
// The warp's cached solves are fixed-point vectors in the y cache (rank 1: the n entries of y up
// to a complex factor; rank 2: the 2 n entries of z1 and z2, sd stays FP64).  In its scratch
// (WarpScratch): the column labels, [slot][lane], from the start of the member loop; the solves'
// exponents (fx_at), [flavour][lane]: 2 e_y (an entry of 2^56 stands for 2^e_y), + 1 when the block's
// det B is a factor.

// Solve of one flavour in fixed point; false: the lane takes the FP64 factorisation.  Ks: the
// block's factors staged in shared memory, or null.
__device__ __forceinline__ bool fx_solve(const FwdArgs& a, int W, int Q, int f, const int32_t* col, const int4* Ks,
                                         double2* Yf, int T, short* ey) {
  const int n = a.n_f[f], rho = a.fam_rank[(int64_t)W * a.F + f];
  const double2* K = a.kbuf + ((int64_t)W * a.n_q + Q) * a.kstride + a.koff[f];
  const int c = col[n - 1], ea = a.fx.cexp[f][c];
  int4* Yx = reinterpret_cast<int4*>(Yf);
  int e2 = 0;
  double2 sd;
  const bool ok = Ks ? fx::solve_sink<true>(n, rho, a.fx.sc[f] + c, ea, Ks, K, Yx, T, &e2, &sd)
                     : fx::solve_sink<false>(n, rho, a.fx.sc[f] + c, ea, reinterpret_cast<const int4*>(K), K, Yx, T, &e2, &sd);
  if (!ok) return false;
  if (rho == 2) Yf[2 * n * T] = sd;
  *ey = (short)e2;
  return true;
}

// The block factors of flavour f of the warp's sinks, copied to its scratch: a solve walks them
// row by row, every row waiting for a few loads, which from global memory cost hundreds of clocks
// each.  Sinks stand in family order, so the warp's blocks are those of families Q0 .. Q1.  Returns
// the lane's block, or null (kept in global memory) when they do not fit.  Called by the whole
// warp; the caller's solves end before the next call.
template <int NCMAX>
__device__ __forceinline__ const int4* fx_stage(const FwdArgs& a, int W, int Q, int f, int lane, void* scratch) {
  constexpr unsigned FULL = 0xffffffffu;
  const int M = a.n_f[f] - a.fam_rank[(int64_t)W * a.F + f], blk = M * (M + 1);
  const int Q0 = __shfl_sync(FULL, Q, 0), cnt = __shfl_sync(FULL, Q, 31) - Q0 + 1;
  if (Q0 < 0 || cnt * blk > WarpScratch<NCMAX>::kBytes / 16) return nullptr;
  const int4* src = reinterpret_cast<const int4*>(a.kbuf + ((int64_t)W * a.n_q + Q0) * a.kstride + a.koff[f]);
  int4* dst = reinterpret_cast<int4*>(scratch);
  __syncwarp();
  for (int q = 0; q < cnt; q++)
    for (int e = lane; e < blk; e += 32) dst[q * blk + e] = __ldg(src + (size_t)q * a.kstride + e);
  __syncwarp();
  return dst + (Q - Q0) * blk;
}

// A flavour's FP64 solve to fixed point, in place; ey: the member guard's scale exponent as the
// FP64 producers define it.  false (and nothing changed): not finite, or without a normal exponent.
__device__ __forceinline__ bool fx_from_fp64(int n, int rho, double2* Yf, int T, int ey, short* out_e) {
  if (rho == 2) {
    const double2 sd = Yf[2 * n * T];
    if (!dev::finite2(sd) || dev::expo(sd) < -900) return false;
    ey = (ey - dev::expo(sd)) >> 1;
  }
  if (ey >= 900 || ey <= -900) return false;
  for (int q = 0; q < rho * n; q++) reinterpret_cast<int4*>(Yf)[q * T] = fx::quant(Yf[q * T], ey + 1, fx::kFracBits);
  *out_e = (short)(2 * (ey + 1));
  return true;
}

// back to FP64 in place (the lanes of a warp that leaves the fixed-point path)
static __device__ __noinline__ void fx_to_fp64(int n, int rho, double2* Yf, int T, int ey, dev::cd factor) {
  for (int q = 0; q < rho * n; q++) {
    const dev::cd v = fx::value(reinterpret_cast<const int4*>(Yf)[q * T], ey);
    Yf[q * T] = rho == 1 ? dev::cmul(v, factor) : v;
  }
}

// g . y of kN members' rows (rank 1).  The members share each load of y and give the integer pipe
// independent sums; the rows' entries are one address for the lanes of a sink family but in its
// changed column.
template <int kN>
__device__ __forceinline__ void fx_dots(int n, const int4* const (&r)[kN], const unsigned short* lab, const int4* Y,
                                        int T, fx::Val (&v)[kN]) {
  fx::Acc s[kN];
#pragma unroll 1
  for (int q = 0; q < n; q++) {
    const int o = lab[q * 32];
    const int4 y = Y[q * T];
#pragma unroll
    for (int k = 0; k < kN; k++) fx::mac(s[k], __ldg(r[k] + o), y);
  }
#pragma unroll
  for (int k = 0; k < kN; k++) v[k] = fx::finish(s[k]);
}

// det(B Z) of one member's two rows against z1, z2 (rank 2); a dot too large for the product's
// limbs gives 0, which no threshold lets pass.
__device__ __forceinline__ fx::Val fx_det2(int n, const int4* __restrict__ r1, const int4* __restrict__ r2,
                                           const unsigned short* lab, const int4* Y, int T) {
  fx::Acc s11, s12, s21, s22;
#pragma unroll 1
  for (int q = 0; q < n; q++) {
    const int o = lab[q * 32];
    const int4 z1 = Y[q * T], z2 = Y[(n + q) * T];
    const int4 a = __ldg(r1 + o), b = __ldg(r2 + o);
    fx::mac(s11, a, z1);
    fx::mac(s12, a, z2);
    fx::mac(s21, b, z1);
    fx::mac(s22, b, z2);
  }
  const fx::Val d11 = fx::finish(s11), d12 = fx::finish(s12), d21 = fx::finish(s21), d22 = fx::finish(s22);
  const bool ok = max(max(fx::magnitude(d11), fx::magnitude(d12)), max(fx::magnitude(d21), fx::magnitude(d22))) < fx::kMulHi;
  const fx::Val p = fx::mul(fx::split(d11), fx::split(d22)), m = fx::mul(fx::split(d12), fx::split(d21));
  return ok ? fx::Val{p.re - m.re, p.im - m.im} : fx::Val{0, 0};  // half the determinant
}

// One member's determinant in FP64 from a fixed-point solve, with the FP64 lemma guard: the pairs
// whose fixed-point value is out of range, too small to be sure of, or near the guard.  The solve's
// entries carry at least the accuracy of FP64 ones at their largest entry's scale, which is the guard's
// scale; where every product is far below it and the determinant too, that is not enough, and the pair
// is refactored (kFloorBits and kCarryBits, with floor exponents).
static __device__ __noinline__ dev::cd fx_member64(const dev::cd* __restrict__ S, int L, int n, int rho,
                                            const int32_t* __restrict__ lab, const int32_t* __restrict__ col,
                                            const int4* Y, int T, int e, dev::cd factor, int kc, bool* fail) {
  const dev::cd* r1 = S + (size_t)lab[0] * L;
  dev::cd d = make_double2(0.0, 0.0);
  int eb = -4096, ez = -4096;
  if (rho == 1) {
    int ep = -8192;
    for (int q = 0; q < n; q++) {
      const dev::cd y = dev::cmul(fx::value(Y[q * T], e), factor), b = dev::ldS(r1 + col[q]);
      ez = max(ez, dev::expo(y));
      eb = max(eb, dev::expo(b));
      ep = max(ep, dev::expo(y) + dev::expo(b));
      d = dev::cfma(b, y, d);
    }
    const int ed = dev::expo(d), es = eb + ez;
    *fail = ed < es - kc || (ed < es - fx::kFloorBits && ep < es - fx::kCarryBits);
    return d;
  }
  const dev::cd* r2 = S + (size_t)lab[1] * L;
  dev::cd d11 = d, d12 = d, d21 = d, d22 = d;
  int e2 = -4096, p11 = -8192, p12 = -8192, p21 = -8192, p22 = -8192;
  for (int q = 0; q < n; q++) {
    const dev::cd z1 = fx::value(Y[q * T], e), z2 = fx::value(Y[(n + q) * T], e);
    const dev::cd b1 = dev::ldS(r1 + col[q]), b2 = dev::ldS(r2 + col[q]);
    const int ez1 = dev::expo(z1), ez2 = dev::expo(z2), eb1 = dev::expo(b1), eb2 = dev::expo(b2);
    ez = max(ez, max(ez1, ez2));
    eb = max(eb, eb1);
    e2 = max(e2, eb2);
    p11 = max(p11, eb1 + ez1);
    p12 = max(p12, eb1 + ez2);
    p21 = max(p21, eb2 + ez1);
    p22 = max(p22, eb2 + ez2);
    d11 = dev::cfma(b1, z1, d11);
    d12 = dev::cfma(b1, z2, d12);
    d21 = dev::cfma(b2, z1, d21);
    d22 = dev::cfma(b2, z2, d22);
  }
  ez = max(ez, 0);
  d = dev::cmul(factor, dev::cfms(d12, d21, dev::cmul(d11, d22)));
  const int ed = dev::expo(d), es = eb + e2 + dev::expo(factor) + 2 * ez;
  const bool carried = min(p11, p12) >= eb + ez - fx::kCarryBits && min(p21, p22) >= e2 + ez - fx::kCarryBits;
  *fail = ed < es - kc || (ed < es - fx::kFloorBits2 && !carried);
  return d;
}

// A sum of products of two dots (of one dot with nf = 1) in FP64; e: the exponent of their scale, lf: the
// lane's factors.
__device__ __forceinline__ double2 fx_sum(const fx::Acc2& s, int nf, int e, double2 lf) {
  double re, im;
  if (nf == 1) {
    re = (double)s.rp;
    im = (double)s.ih;
    e -= fx::kDotBits;
  } else {
    constexpr double k30 = 1073741824.0;
    re = fma((double)s.hi_re(), k30, (double)s.lo_re());
    im = fma((double)s.hi_im(), k30, (double)s.lo_im());
    e += 30 - 2 * fx::kSplitBits;
  }
  return dev::cmul(make_double2(fx::scale2(re, e), fx::scale2(im, e)), lf);
}
// One member's product: a call, as the member loop needs it now and then only.
static __device__ __noinline__ double2 fx_far(fx::Val u, fx::Val t, int nf, int e, double2 lf) {
  fx::Acc2 s;
  if (nf == 1) {
    s.rp = u.re;
    s.ih = u.im;
  } else {
    fx::mac(s, fx::split(u), fx::split(t));
  }
  return fx_sum(s, nf, e, lf);
}

// One work item (family W x sink tile) by the whole thread block; the block's sum goes
// to *partial.  Shared by the per-plan launch and the persistent batched launch.  FX: the call takes the
// fixed-point path (dev::fx_on); else the FP64 path alone.  CW: the weights may be complex.
template <int NCMAX, bool FX, bool CW>
__device__ __forceinline__ void fwd_item(const FwdArgs& a, int W, int tile, double2* smem,
                                         double2* partial) {
  const int T = blockDim.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t jraw = (int64_t)tile * T + tid;
  const bool valid = jraw < a.n_snk;
  const int64_t j = valid ? jraw : a.n_snk - 1;  // sink position
  const int32_t* cols = dev::sink_cols(a, j);
  const int Q = a.snk_orig ? a.snk_q[j] : -1;
  const bool qtwo = Q >= 0 && a.q_two[Q];
  const int mem0 = a.fam_info[4 * W], kW = a.fam_info[4 * W + 1];
  using WS = WarpScratch<NCMAX>;
  char* scratch = reinterpret_cast<char*>(smem + (size_t)a.slots * T) + (size_t)warp * WS::bytes(a.slots, a.fx.nf > 0);
  QEntry* queue = reinterpret_cast<QEntry*>(scratch);
  double2* Y = smem + tid;
  const double2* Yw = smem + (tid & ~31);  // the warp's cached solves (lane l: Yw + l)

  // ---- per flavour: solve, or factorise the shared rows, for this sink ----------------
  constexpr bool kFx = FX;
  unsigned short* lab = reinterpret_cast<unsigned short*>(scratch + WS::kQueue + WS::kWalk) + lane;
  short* eyw = reinterpret_cast<short*>(scratch + WS::exponents(a.slots));
  bool fxm = kFx && a.fx.nf > 0 && kW <= fx::kMaxMembers, bad = false;
  for (int f = 0; f < a.F; f++) fxm &= a.fam_rank[(int64_t)W * a.F + f] <= 2;
  // flavours solved in fixed point; left to the FP64 factorisation; FP64 solves converted
  unsigned infx = 0, solo = 0, made = 0;
  unsigned pguard = 0;
  dev::ScalesFor<NCMAX> eys;
  for (int f = 0; f < a.F; f++) {
    const int n = a.n_f[f];
    int ey = 0;
    if (n == 0) continue;
    const int rho = a.fam_rank[(int64_t)W * a.F + f];
    const int32_t* arow = a.fam_arow + (int64_t)W * a.Tn + a.off_f[f];
    const int sig = qtwo ? a.q_rank[(int64_t)Q * a.F + f] : 0;
    double2* Yf = Y + (size_t)a.yoff[f] * T;
    bool done = false;
    if constexpr (kFx) {
      const bool blk = fx_block(a, W, Q, f, qtwo);
      const int4* Ks = __any_sync(0xffffffffu, blk) ? fx_stage<NCMAX>(a, W, Q, f, lane, scratch) : nullptr;
      if (blk) {
        done = fx_solve(a, W, Q, f, cols + a.off_f[f], Ks, Yf, T, eyw + fx_at(a, f) + lane);
        if (done) infx |= 1u << f; else solo |= 1u << f;
      }
    }
    if (!done) {
      if (!((solo >> f) & 1) && qtwo && (rho == 1 || sig == 1 || (rho == 2 && sig == 2)) &&
          !a.kguard[((int64_t)W * a.n_q + Q) * a.F + f]) {
        const double2* K = a.kbuf + ((int64_t)W * a.n_q + Q) * a.kstride + a.koff[f];
        if (rho == 2 && sig == 2)
          dev::dispatch_kapply22<NCMAX>(n, a.S[f], a.L_f[f], arow, cols + a.off_f[f], K, Yf, T, &ey);
        else if (sig == 2)
          dev::dispatch_kapply12<NCMAX>(n, a.S[f], a.L_f[f], arow, cols + a.off_f[f], K, Yf, T, &ey);
        else if (rho == 2)
          dev::dispatch_kapply2<NCMAX>(n, a.S[f], a.L_f[f], arow, cols + a.off_f[f], K, Yf, T, &ey);
        else
          dev::dispatch_kapply<NCMAX>(n, a.S[f], a.L_f[f], arow, cols + a.off_f[f], K, Yf, T, &ey);
      } else {
        const bool g = dev::dispatch_shared<NCMAX>(n, rho, a.S[f], a.L_f[f], arow, cols + a.off_f[f], Yf, T, &ey, a.kp);
        pguard |= (unsigned)g << f;
      }
      if constexpr (kFx) {
        if (fxm && fx_from_fp64(n, rho, Yf, T, ey, eyw + fx_at(a, f) + lane)) made |= 1u << f;
        bad |= fxm && !((made >> f) & 1);
      }
    }
    eys.set(f, ey);
  }

  // ---- the member dots in fixed point, unless a sink of the warp has no usable solve (not
  // finite, or its pivot guard fired) ------------------------------------------------------
  int le = 0;                           // exponent of the lane's solves, all flavours
  double2 lf = make_double2(1.0, 0.0);  // their factors
  if constexpr (kFx) {
    const bool keep = fxm && !__any_sync(0xffffffffu, bad || pguard != 0);
    __syncwarp();  // the labels lie where the solves read the staged block factors
    for (int f = 0; f < a.F; f++) {
      const int n = a.n_f[f];
      if (n == 0) continue;
      const int rho = a.fam_rank[(int64_t)W * a.F + f];
      double2* Yf = Y + (size_t)a.yoff[f] * T;
      const bool blk = (infx >> f) & 1;
      if (keep) {
        lf = dev::cmul(lf, fx_factor(a, W, Q, f, blk, Yf, T));
        le += rho * (eyw[fx_at(a, f) + lane] >> 1) + (rho == 2);  // fx::mul halves
        for (int q = 0; q < n; q++) lab[(a.yoff[f] + q) * 32] = (unsigned short)cols[a.off_f[f] + q];
      } else if (blk || ((made >> f) & 1)) {
        fx_to_fp64(n, rho, Yf, T, eyw[fx_at(a, f) + lane] >> 1, fx_factor(a, W, Q, f, blk, Yf, T));
        eys.set(f, dev::cached_scale(Yf, T, n, rho));
      }
    }
    fxm = keep;
    __syncwarp();
  }

  // ---- rank-2 flavours against a one-column sink family shared by the warp's sinks: the
  // members' dots with the block's first null vector, once per warp (lane t: member t) -----
  // (two-row families need n_f >= 10: the classes below compile none of this)
  constexpr bool kZ1 = NCMAX >= 10;
  int zf0 = -1, zf1 = -1;
  double2* z1d = reinterpret_cast<double2*>(scratch + WS::kQueue + WS::kWalk);
  // the warp's scratch for the grouped refactors' multipliers (group_fresh)
  double2* wk = reinterpret_cast<double2*>(scratch + WS::kQueue);
  // (the shuffle and the vote run on every lane: qtwo differs between lanes whose sinks
  // belong to a two-sided family and lanes whose sinks stand alone)
  const int Q0 = kZ1 ? __shfl_sync(0xffffffffu, Q, 0) : 0;
  const bool z1_warp = kZ1 && __all_sync(0xffffffffu, qtwo && Q == Q0);
  if (kZ1 && z1_warp && kW <= 32 && !fxm) {
    // the flavours are chosen from warp-uniform data only (W, Q), so every lane assigns the
    // same slots; such a flavour took kapply2 on every lane
    for (int f = 0; f < a.F && zf1 < 0; f++) {
      const int n = a.n_f[f];
      if (n == 0 || a.fam_rank[(int64_t)W * a.F + f] != 2 || a.q_rank[(int64_t)Q * a.F + f] != 1 ||
          a.kguard[((int64_t)W * a.n_q + Q) * a.F + f])
        continue;
      const int slot = zf0 < 0 ? 0 : 1;
      if (lane < kW) {
        double2 d11, d21;
        dev::dispatch_dots_z1<NCMAX>(n, a.S[f], a.L_f[f],
                                     a.mem_lab + ((int64_t)(mem0 + lane) * a.F + f) * MHC_MAX_RANK,
                                     cols + a.off_f[f], Y + (size_t)a.yoff[f] * T, T, &d11, &d21);
        z1d[(slot * 32 + lane) * 2] = d11;
        z1d[(slot * 32 + lane) * 2 + 1] = d21;
      }
      if (slot == 0) zf0 = f; else zf1 = f;
    }
    __syncwarp();
  }

  // ---- per member: one dot product per flavour --------------------------------------
  const double2 wj = valid ? dev::sink_weight<CW>(a, j) : make_double2(0.0, 0.0);
  // acc: sum over the members of w_i prod_f det (this lane's sink; times w_j once, at the
  // end); accq: the refactored pairs, w_i w_j included (a queue lane holds other sinks' pairs)
  double2 acc = make_double2(0.0, 0.0), accq = make_double2(0.0, 0.0);
  int qn = 0;
  unsigned long long n_parent = 0, n_child = 0, n_rowdiff = 0, rflops = 0;
  // one member in FP64: the lanes with part (the others' pairs are already summed)
  auto member64 = [&](int c, bool part) {
    const int m = mem0 + c;
    unsigned fail = pguard;
    double2 prod = make_double2(1.0, 0.0);
    bool first = true;
    for (int f = 0; f < a.F; f++) {
      const int n = a.n_f[f];
      if (n == 0 || ((pguard >> f) & 1)) continue;
      const int rho = a.fam_rank[(int64_t)W * a.F + f];
      bool cf = false;
      const int32_t* mlab = a.mem_lab + ((int64_t)m * a.F + f) * MHC_MAX_RANK;
      const double2* Yf = Y + (size_t)a.yoff[f] * T;
      double2 d;
      bool fixed = false;
      if constexpr (kFx) {
        if (fxm) {
          d = fx_member64(a.S[f], a.L_f[f], n, rho, mlab, cols + a.off_f[f], reinterpret_cast<const int4*>(Yf), T,
                          eyw[fx_at(a, f) + lane] >> 1, fx_factor(a, W, Q, f, (infx >> f) & 1, Yf, T), a.kc, &cf);
          fixed = true;
        }
      }
      if (fixed) {
      } else if (kZ1 && (f == zf0 || f == zf1)) {
        const double2* zd = z1d + ((f == zf0 ? 0 : 32) + c) * 2;
        d = dev::dispatch_member_z1<NCMAX>(n, a.S[f], a.L_f[f], mlab, cols + a.off_f[f], Yf, T, eys.get(f),
                                           a.kc, &cf, zd[0], zd[1]);
      } else {
        d = dev::dispatch_member<NCMAX>(n, rho, a.S[f], a.L_f[f], mlab, cols + a.off_f[f], Yf, T, eys.get(f),
                                        a.kc, &cf);
      }
      if (cf) {
        fail |= 1u << f;
      } else {
        prod = first ? d : dev::cmul(prod, d);
        first = false;
      }
    }
    const bool need = valid && part && fail != 0;
    const double2 wi = dev::source_weight<CW>(a, m);
    if (part && !fail) acc = dev::add_weighted<CW>(a, wi, prod, acc);
    const unsigned ball = __ballot_sync(0xffffffffu, need);
    if (ball == 0xffffffffu) {
      // every lane refactors this member (a member near-singular against its family): the
      // pairs go straight to the refactor as one group, past the queue, so that a queue
      // flush never splits the group that group_fresh factorises once
      QEntry e;
      e.member = m;
      e.lane = lane;
      e.fail = (int32_t)fail;
      e.pguard = (int32_t)pguard;
      e.prod = prod;
      e.w = dev::add_weighted<CW>(a, wi, wj, make_double2(0.0, 0.0));
      process_pairs<NCMAX, FX, CW>(a, W, true, e, j, Yw, fxm, eyw, wk, accq, rflops, n_rowdiff);
      n_parent += __popc(fail & pguard);
      n_child += __popc(fail & ~pguard);
    } else if (ball) {
      if (need) {
        const int pos = qn + __popc(ball & ((1u << lane) - 1u));
        QEntry e;
        e.member = m;
        e.lane = lane;
        e.fail = (int32_t)fail;
        e.pguard = (int32_t)pguard;
        e.prod = prod;
        e.w = dev::add_weighted<CW>(a, wi, wj, make_double2(0.0, 0.0));
        queue[pos] = e;
        n_parent += __popc(fail & pguard);
        n_child += __popc(fail & ~pguard);
      }
      qn += __popc(ball);
      __syncwarp();
      if (qn >= 32) {
        process_queue<NCMAX, FX, CW>(a, W, queue, 32, (int64_t)tile * T + warp * 32, Yw, fxm, eyw, wk, accq, rflops, n_rowdiff);
        __syncwarp();
        if (lane < qn - 32) queue[lane] = queue[32 + lane];
        __syncwarp();
        qn -= 32;
      }
    }
  };
  if constexpr (!kFx) {
    for (int c = 0; c < kW; c++) member64(c, true);
  } else {
    // Sum of the members' products at the family's exponent, in integers: to FP64 every kFlush members.
    fx::Acc2 tot;
    auto add = [&]() {
      const double2 v = fx_sum(tot, a.fx.nf, a.fx.fexp[W] + le, lf);
      acc.x += v.x;
      acc.y += v.y;
      tot = fx::Acc2();
    };
    constexpr int kFloorN = NCMAX <= 8 ? 8 : 18;
    const int thr1 = fx::accepted(kFloorN, a.kc, 1), thr2 = fx::accepted(kFloorN, a.kc, 2);
    // members four at a time (a step that they do not fill repeats the last one)
    constexpr int kN = 4;
    const int step = fxm ? kN : 1;
    for (int c = 0; c < kW; c += step) {
      unsigned slow = 15;  // bit k: this lane's pair with member c + k goes through FP64
      if (fxm) {
        const unsigned ds = __ldg(a.fx.align + mem0 + c);
        fx::Val u[kN], t[kN];
        int at = 0;
        slow = 0;
        for (int f = 0; f < a.F; f++) {
          const int n = a.n_f[f], L = a.L_f[f];
          if (n == 0) continue;
          const int rho = a.fam_rank[(int64_t)W * a.F + f];
          const unsigned short* lb = lab + a.yoff[f] * 32;
          const int4* Yf = reinterpret_cast<const int4*>(Y + (size_t)a.yoff[f] * T);
          fx::Val v[kN];
          const int4* r[kN];
  #pragma unroll
          for (int k = 0; k < kN; k++) {
            const int m = mem0 + min(c + k, kW - 1);
            r[k] = at == 0 ? a.fx.ws + (size_t)m * L
                           : a.fx.s[f] + (size_t)a.mem_lab[((int64_t)m * a.F + f) * MHC_MAX_RANK] * L;
          }
          if (NCMAX >= 10 && rho == 2) {
  #pragma unroll
            for (int k = 0; k < kN; k++) {
              const int m = mem0 + min(c + k, kW - 1);
              v[k] = fx_det2(n, r[k], a.fx.s[f] + (size_t)a.mem_lab[((int64_t)m * a.F + f) * MHC_MAX_RANK + 1] * L, lb, Yf, T);
            }
          } else {
            fx_dots<kN>(n, r, lb, Yf, T, v);
          }
          const int thr = rho == 2 ? thr2 : thr1;
  #pragma unroll
          for (int k = 0; k < kN; k++) {
            u[k] = at == 0 ? v[k] : u[k];
            t[k] = v[k];
            slow |= (unsigned)!fx::usable(fx::magnitude(v[k]), thr) << k;
          }
          at++;
        }
        unsigned far = 0;
        if (ds & 0x80808080u) {
  #pragma unroll
          for (int k = 0; k < kN; k++) {
            const unsigned d = (ds >> (8 * k)) & 255u;
            far |= (unsigned)(d == fx::kFar) << k;
            slow |= (unsigned)(d == fx::kOnlyFp64) << k;
          }
        }
  #pragma unroll
        for (int k = 0; k < kN; k++) {
          const unsigned d = (ds >> (8 * k)) & 255u;
          const bool use = d < fx::kFar && !((slow >> k) & 1);
          if (a.fx.nf == 1) {  // kFlush values below 2^60
            const fx::Val x = fx::rounded(u[k], d & 31u);
            tot.rp += use ? x.re : 0;
            tot.ih += use ? x.im : 0;
          } else {
            const fx::Val x = d & 127u ? fx::aligned(u[k], d & 31u) : u[k];
            fx::mac(tot, fx::split(use ? x : fx::Val{0, 0}), fx::split(t[k]));
          }
        }
        if (((c + kN) & (fx::kFlush - 1)) == 0 || c + kN >= kW) add();
        while (far) {
          const int k = __ffs(far) - 1;
          far &= far - 1;
          const fx::Val x = k == 0 ? u[0] : k == 1 ? u[1] : k == 2 ? u[2] : u[3];
          const fx::Val y = k == 0 ? t[0] : k == 1 ? t[1] : k == 2 ? t[2] : t[3];
          const double2 v = fx_far(x, y, a.fx.nf, a.fx.fexp[W] + le - __ldg(a.fx.below + mem0 + c + k), lf);
          if (!((slow >> k) & 1)) acc = dev::cadd(acc, v);
        }
      }
      // pairs out of the fixed-point range or below its floor (every pair of a family or warp that the format
      // does not take)
      slow &= (1u << min(step, kW - c)) - 1u;
      for (unsigned todo = __reduce_or_sync(0xffffffffu, slow); todo; todo &= todo - 1) {
        const int k = __ffs(todo) - 1;
        member64(c + k, (slow >> k) & 1);
      }
    }
  }
  __syncwarp();
  if (qn > 0) process_queue<NCMAX, FX, CW>(a, W, queue, qn, (int64_t)tile * T + warp * 32, Yw, fxm, eyw, wk, accq, rflops, n_rowdiff);
  acc = dev::add_weighted<CW>(a, wj, acc, accq);

  // ---- fixed-order reduction: lanes, then warps --------------------------------------
  acc = dev::warp_sum(acc);
  for (int o = 16; o > 0; o >>= 1) {
    n_parent += __shfl_xor_sync(0xffffffffu, n_parent, o);
    n_child += __shfl_xor_sync(0xffffffffu, n_child, o);
    n_rowdiff += __shfl_xor_sync(0xffffffffu, n_rowdiff, o);
    rflops += __shfl_xor_sync(0xffffffffu, rflops, o);
  }
  __syncthreads();
  double2* red = smem;  // reuse: the factor cache is no longer needed
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (tid == 0) {
    double2 s = red[0];
    for (int w = 1; w < (T >> 5); w++) {
      s.x += red[w].x;
      s.y += red[w].y;
    }
    *partial = s;
    if (!dev::finite2(s)) atomicOr(&a.counters[0], kStatusNonFinite);
  }
  if (lane == 0 && (n_parent | n_child | n_rowdiff)) {
    atomicAdd(&a.counters[1], n_parent);
    atomicAdd(&a.counters[2], n_child - n_rowdiff);  // queued for the lemma guard, less those the
    atomicAdd(&a.counters[3], rflops);               // row-difference update resolved
    atomicAdd(&a.counters[4], n_rowdiff);
  }
}

// The last block of a call to finish sums the items' partials in a fixed order (smem: past the
// entries that fwd_item's own sum uses).
__device__ __forceinline__ void fold_partials(const FwdArgs& a, double2* smem) {
  const int T = blockDim.x, tid = threadIdx.x;
  double2* red = smem + 8;
  int* last = reinterpret_cast<int*>(smem + 16);
  if (tid == 0) {
    __threadfence();
    const unsigned n1 = (unsigned)a.fold_items - 1;
    *last = atomicInc(a.reduce_done, n1) == n1;  // the last one wraps it to 0
  }
  __syncthreads();
  if (!*last) return;
  __threadfence();
  double2 s = make_double2(0.0, 0.0);
#pragma unroll 8
  for (int64_t i = tid; i < a.fold_items; i += T) s = dev::cadd(s, __ldcg(a.partials + i));
  s = dev::warp_sum(s);
  if ((tid & 31) == 0) red[tid >> 5] = s;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < (T >> 5); w++) s = dev::cadd(s, red[w]);
    a.out[0] = s.x;
    a.out[1] = s.y;
  }
}

// Registers: the n <= 8 class keeps 168 (12 one-warp blocks per SM, or 3 blocks of its
// 128-thread tile); the larger classes may use all 255, measured fastest for n = 18 (8 blocks
// per SM against 9 at 216 and 10 at 200, whose spills cost more than the warps gain).
// FX: the plan has fixed-point tables, or the weights are complex; else the kernel holds the FP64 path for
// real weights alone (n <= 32: for both).  512 x 512 terms of n = 3: 55 us per call, and 64 us when it
// also carried the complex weights, converted solves for the refactors and a launch for the partials'
// sum.  The FX kernels (CW: for complex weights, else real ones) keep the FP64 path apart, for plans without
// tables and for propagators that are not flat: a copy of its own, for n <= 8 called, so that its registers
// stay out of the other's (4096 x 4096 terms of n = 6: 1177 us, 1200 us inlined; n = 9, 7 with families of
// three 1983 us, 1895 us inlined).  The arguments stay in constant memory (__grid_constant__): calls take
// their address, for which every thread had copied all 1.4 KB of them (n = 9, 7: 2185 us; n = 18, 4096 x 4096
// terms 9.8 ms, 9.3 ms without the copy).
template <int NCMAX, bool CW>
__device__ __noinline__ void fwd_item_fp64(const FwdArgs& a, int W, int tile, double2* partial) {
  extern __shared__ double2 smem[];
  fwd_item<NCMAX, false, CW>(a, W, tile, smem, partial);
}
template <int NCMAX, bool FX, bool CW>
__global__ void __maxnreg__(NCMAX <= 8 ? 168 : 255) fwd_kernel(const __grid_constant__ FwdArgs a) {
  extern __shared__ double2 smem[];
  const int64_t item = a.item0 + blockIdx.x;
  const int64_t pos = item / a.n_tiles;
  const int W = a.fam_order ? a.fam_order[pos] : (int)pos;
  const int tile = (int)(item % a.n_tiles);
  if constexpr (FX) {
    if (dev::fx_on(a))
      fwd_item<NCMAX, true, CW>(a, W, tile, smem, &a.partials[item]);
    else if (NCMAX <= 8)
      fwd_item_fp64<NCMAX, CW>(a, W, tile, &a.partials[item]);
    else
      fwd_item<NCMAX, false, CW>(a, W, tile, smem, &a.partials[item]);
  } else {
    fwd_item<NCMAX, false, CW>(a, W, tile, smem, &a.partials[item]);
  }
  if (a.fold_items > 0) fold_partials(a, smem);
}

// Flavours of a pair that pair_group_kernel takes: blocks that do not fit in a thread's registers.
__device__ __forceinline__ bool pair_grouped(int n, int rho) { return n > 6 && rho <= 2; }

// Per-pair determinants by the update scheme in FP64 (one thread per pair): the flavours with
// n <= 6 or more than two changed rows.
template <int NCMAX>
__global__ void __launch_bounds__(64) pair_kernel(const FwdArgs a, int64_t n_pairs, int64_t n_src,
                                                  const int64_t* __restrict__ ii,
                                                  const int64_t* __restrict__ jj,
                                                  const int32_t* __restrict__ src_member,
                                                  const int32_t* __restrict__ mem_family,
                                                  double2* __restrict__ dets, int32_t* path) {
  extern __shared__ double2 smem[];
  const int T = blockDim.x;
  const int64_t p = (int64_t)blockIdx.x * T + threadIdx.x;
  if (p >= n_pairs) return;
  const int64_t i = ii[p], j = jj[p];
  if (i < 0 || i >= n_src || j < 0 || j >= a.n_snk) {
    atomicOr(&a.counters[0], kStatusBadIndex);
    return;
  }
  const int m = src_member[i];
  const int W = mem_family[m];
  double2* Y = smem + threadIdx.x;
  int32_t rows[NCMAX];
  int32_t bits = 0;
  for (int f = 0; f < a.F; f++) {
    const int n = a.n_f[f];
    if (pair_grouped(n, a.fam_rank[(int64_t)W * a.F + f])) continue;
    double2 d = make_double2(1.0, 0.0);
    if (n > 0) {
      const int rho = a.fam_rank[(int64_t)W * a.F + f];
      const int32_t* col = a.snk_lab + j * a.Tn + a.off_f[f];
      int ey = 0;
      bool fail = dev::dispatch_shared<NCMAX>(n, rho, a.S[f], a.L_f[f],
                                              a.fam_arow + (int64_t)W * a.Tn + a.off_f[f], col,
                                              Y, T, &ey, a.kp);
      if (!fail) {
        const int32_t* mlab = a.mem_lab + ((int64_t)m * a.F + f) * MHC_MAX_RANK;
        d = dev::dispatch_member<NCMAX>(n, rho, a.S[f], a.L_f[f], mlab, col, Y, T, ey, a.kc, &fail);
        if (fail && rho <= 2 && n >= rho + 1 && a.rowdiff) {
          bool f2 = true;
          const int32_t* arow = a.fam_arow + (int64_t)W * a.Tn + a.off_f[f];
          double2 d2;
          if constexpr (NCMAX >= 10)  // two-row families need n_f >= 10
            d2 = rho == 1 ? dev::rowdiff_det(a.S[f], a.L_f[f], n, mlab[0], arow, col, Y, T, ey, a.kc, &f2)
                          : dev::rowdiff2_det(a.S[f], a.L_f[f], n, mlab, arow, col, Y, T, ey, a.kc, &f2);
          else
            d2 = dev::rowdiff_det(a.S[f], a.L_f[f], n, mlab[0], arow, col, Y, T, ey, a.kc, &f2);
          if (!f2) {
            d = d2;
            fail = false;
            bits |= 1 << (8 + f);
          }
        }
      }
      if (fail) {
        dev::member_rows(a, W, m, f, rho, rows);
        d = dev::dispatch_fresh<NCMAX>(n, a.S[f], a.L_f[f], rows, col);
        bits |= 1 << f;
      }
      if ((a.mem_par[m] >> f) & 1) d = dev::cneg(d);
    }
    dets[p * a.F + f] = d;
  }
  if (path) path[p] = bits;
}

// One two-sided block (family W, sink family Q, flavour f) of plan a: factorise B
// (rank-1 family) or the two-row family's shared rows (see kapply2), or nothing.
template <int NCMAX>
__device__ __forceinline__ void kfac_one(const FwdArgs& a, int64_t t, int64_t n_fam) {
  const int f = (int)(t % a.F);
  const int64_t wq = t / a.F;
  const int Q = (int)(wq % a.n_q);
  const int W = (int)(wq / a.n_q);
  const int n = a.n_f[f];
  if (n == 0 || n > 6 || !a.q_two[Q]) return;  // n > 6: kfac_group_kernel
  const int rho = a.fam_rank[(int64_t)W * a.F + f];
  const int sig = a.q_rank[(int64_t)Q * a.F + f];
  const dev::cd* S = a.S[f];
  const int L = a.L_f[f];
  const int32_t* arow = a.fam_arow + (int64_t)W * a.Tn + a.off_f[f];
  const int32_t* scol = a.snk_pos + (int64_t)a.q_off[Q] * a.Tn + a.off_f[f];
  dev::cd* K = const_cast<dev::cd*>(a.kbuf) + wq * a.kstride + a.koff[f];
  if ((rho == 2 && sig == 2) || rho >= 3) {  // one-sided update for these blocks
    a.kguard[t] = 1;
    return;
  }
  bool g;
  if (sig == 2) {
#define MHC_K12(N) \
  case N:          \
    g = dev::kfac_block12<N, N>(S, L, N, arow, scol, K, a.kp); \
    break;
    switch (n) {
      MHC_K12(2)
      MHC_K12(3)
      MHC_K12(4)
      MHC_K12(5)
      MHC_K12(6)
      default:
        return;
    }
#undef MHC_K12
    a.kguard[t] = g ? 1 : 0;
    return;
  }
#define MHC_KF(N)                                                                         \
  case N:                                                                                 \
    g = rho == 1 ? dev::kfac_block<N, N, 1>(S, L, N, arow, scol, K, a.kp, dev::fx_on(a))    \
                 : dev::kfac_block<N, N, (N >= 2 ? 2 : 1)>(S, L, N, arow, scol, K, a.kp, false); \
    break;
  switch (n) {
    MHC_KF(1)
    MHC_KF(2)
    MHC_KF(3)
    MHC_KF(4)
    MHC_KF(5)
    MHC_KF(6)
    default:
      return;
  }
#undef MHC_KF
  a.kguard[t] = g ? 1 : 0;
}

// Thread u of a plan's block grid takes flavour u / (n_fam n_q) and block u mod (n_fam n_q):
// the flavour varies slowest, so a warp's threads share n_f (flavours of different sizes
// would otherwise alternate across the lanes and run both code paths).  Returns the index
// of the block in the [W][Q][f] layout of the factor buffer.
__device__ __forceinline__ int64_t kfac_index(const FwdArgs& a, int64_t u, int64_t n_fam) {
  const int64_t nwq = n_fam * a.n_q;
  return (u % nwq) * a.F + u / nwq;
}

// two-sided blocks of one plan: one thread per (W, Q, f)
template <int NCMAX>
__global__ void __launch_bounds__(128) kfac_kernel(const FwdArgs a, int64_t n_fam) {
  const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= n_fam * a.n_q * a.F) return;
  kfac_one<NCMAX>(a, kfac_index(a, u, n_fam), n_fam);
}

// two-sided blocks of every plan of a batch in one launch: kpref[k] is the first thread of
// correlator k (prefix sums of n_fam * n_q * F; kpref[count] = total)
template <int NCMAX>
__global__ void __launch_bounds__(128) kfac_batch_kernel(const FwdArgs* __restrict__ desc,
                                                         const int64_t* __restrict__ kpref,
                                                         const int64_t* __restrict__ nfam, int count) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= kpref[count]) return;
  int lo = 0, hi = count - 1;
  while (lo < hi) {  // last k with kpref[k] <= t
    const int mid = (lo + hi + 1) >> 1;
    if (kpref[mid] <= t) lo = mid; else hi = mid - 1;
  }
  const FwdArgs& a = desc[lo];
  if (!a.snk_orig) return;
  kfac_one<NCMAX>(a, kfac_index(a, t - kpref[lo], nfam[lo]), nfam[lo]);
}

// Two-sided blocks with n > 6: G lanes per block, the block in shared memory (see
// dev::group_lu).  One warp per thread block; GPW blocks per warp.
template <int NCMAX>
struct KGroup {
  static constexpr int G = NCMAX <= 8 ? 4 : (NCMAX <= 18 ? 8 : 16);  // lanes per block
  static constexpr int GPW = 32 / G;                           // blocks per warp
  // complex per block (matrix + back-substitution vector), padded to 4 mod 8 16-byte units
  // so that two groups sharing an 8-lane shared-memory phase use disjoint bank groups
  static constexpr int RAW = (NCMAX - 1) * (NCMAX - 1) + (NCMAX - 1);
  static constexpr int BS = RAW + ((4 - RAW % 8) + 8) % 8;
  static constexpr int PS = 3 * NCMAX;                         // ints per block: row order, two exponents
  static constexpr size_t smem() { return (size_t)GPW * (BS * sizeof(double2) + PS * sizeof(int)); }
};

// Per-pair determinants of the other flavours: G lanes per (pair, flavour), the shared rows in shared
// memory (group_lu), the null vectors by a back substitution over the lanes, the member's dots and a
// guarded pair's fresh factorisation likewise.  A thread's own (n - 1) x n matrix lived in local
// memory: 100 000 pairs of n = 18 took 26.4 ms; here 5.4 ms, of which the factorisations' FP64 work is
// 2.5 ms.
template <int NCMAX>
struct PairGroup {
  static constexpr int G = KGroup<NCMAX>::G, GPW = KGroup<NCMAX>::GPW;
  static constexpr int RAW = NCMAX * (NCMAX | 1) + 2 * NCMAX + 1;
  static constexpr int BS = RAW + ((4 - RAW % 8) + 8) % 8;  // as KGroup
  static constexpr size_t smem() { return (size_t)GPW * (BS * sizeof(double2) + NCMAX * sizeof(int)); }
};
template <int NCMAX>
__global__ void __launch_bounds__(32) pair_group_kernel(const FwdArgs a, int64_t n_pairs, int64_t n_src,
                                                        const int64_t* __restrict__ ii,
                                                        const int64_t* __restrict__ jj,
                                                        const int32_t* __restrict__ src_member,
                                                        const int32_t* __restrict__ mem_family,
                                                        double2* __restrict__ dets, int32_t* path) {
  using PG = PairGroup<NCMAX>;
  constexpr int G = PG::G;
  extern __shared__ double2 smem[];
  const int lane = threadIdx.x, grp = lane / G, g = lane % G;
  const unsigned gm = ((1u << G) - 1u) << (grp * G);
  const int64_t u = (int64_t)blockIdx.x * PG::GPW + grp;
  const int f = (int)(u / n_pairs);  // the flavour varies slowest
  if (f >= a.F) return;
  const int64_t p = u % n_pairs, i = ii[p], j = jj[p];
  if (i < 0 || i >= n_src || j < 0 || j >= a.n_snk) return;  // reported by pair_kernel
  const int m = src_member[i], W = mem_family[m];
  const int n = a.n_f[f], rho = a.fam_rank[(int64_t)W * a.F + f], M = n - rho;
  if (!pair_grouped(n, rho)) return;
  dev::cd* B = smem + (size_t)grp * PG::BS;
  dev::cd* Y = B + NCMAX * (NCMAX | 1);
  int* perm = reinterpret_cast<int*>(smem + (size_t)PG::GPW * PG::BS) + grp * NCMAX;
  const int L = a.L_f[f], P = n | 1;
  const dev::cd* S = a.S[f];
  const int32_t* arow = a.fam_arow + (int64_t)W * a.Tn + a.off_f[f];
  const int32_t* col = a.snk_lab + j * a.Tn + a.off_f[f];
  const int32_t* mlab = a.mem_lab + ((int64_t)m * a.F + f) * MHC_MAX_RANK;
  auto load = [&](int rows) {  // the shared rows, then the member's
    for (int e = g; e < rows * n; e += G) {
      const int r = e / n, q = e - r * n;
      B[r * P + q] = dev::ldS(S + (size_t)(r < M ? arow[r] : mlab[r - M]) * L + col[q]);
    }
    __syncwarp(gm);
  };
  auto sum = [&](dev::cd v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
      v.x += __shfl_xor_sync(gm, v.x, o);
      v.y += __shfl_xor_sync(gm, v.y, o);
    }
    return v;
  };
  auto most = [&](int v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v = max(v, __shfl_xor_sync(gm, v, o));
    return v;
  };
  load(M);
  dev::cd det, d = make_double2(0.0, 0.0);
  int parity, bits = 0;
  bool fail = dev::group_lu<G>(B, P, perm, M, n, M, g, gm, a.kp, &det, &parity);
  if (!fail) {
    const dev::cd sd = parity ? dev::cneg(det) : det;
    // null vectors z_t = [-U1^{-1} u_t ; e_t] (Y + t n); rank 1: y = sd z; rank 2: sd at Y + 2 n
    for (int t = 0; t < rho; t++) {
      dev::cd* z = Y + t * n;
      for (int k = M - 1; k >= 0; k--) {
        dev::cd s = make_double2(0.0, 0.0);
        for (int q = k + 1 + g; q < M; q += G) s = dev::cfma(B[k * P + q], z[q], s);
        s = sum(s);
        if (g == 0) z[k] = dev::cmul(dev::cadd(s, B[k * P + M + t]), dev::cneg(B[k * P + k]));
        __syncwarp(gm);
      }
      for (int v = g; v < rho; v += G) z[M + v] = make_double2(v == t ? 1.0 : 0.0, 0.0);
      __syncwarp(gm);
      if (rho == 1)
        for (int q = g; q < n; q += G) z[q] = dev::cmul(sd, z[q]);
    }
    if (rho == 2 && g == 0) Y[2 * n] = sd;
    __syncwarp(gm);
    int ez = rho == 1 ? -4096 : 0, e1 = -4096, e2 = -4096;
    for (int q = g; q < rho * n; q += G) ez = max(ez, dev::expo(Y[q]));
    ez = most(ez);
    const int ey = rho == 1 ? ez : dev::expo(sd) + 2 * ez;
    if (rho == 1) {
      for (int q = g; q < n; q += G) {
        const dev::cd b = dev::ldS(S + (size_t)mlab[0] * L + col[q]);
        e1 = max(e1, dev::expo(b));
        d = dev::cfma(b, Y[q], d);
      }
      d = sum(d);
      e2 = 0;
    } else {
      dev::cd d11 = d, d12 = d, d21 = d, d22 = d;
      for (int q = g; q < n; q += G) {
        const dev::cd b1 = dev::ldS(S + (size_t)mlab[0] * L + col[q]), b2 = dev::ldS(S + (size_t)mlab[1] * L + col[q]);
        e1 = max(e1, dev::expo(b1));
        e2 = max(e2, dev::expo(b2));
        d11 = dev::cfma(b1, Y[q], d11);
        d12 = dev::cfma(b1, Y[n + q], d12);
        d21 = dev::cfma(b2, Y[q], d21);
        d22 = dev::cfma(b2, Y[n + q], d22);
      }
      d11 = sum(d11);
      d12 = sum(d12);
      d21 = sum(d21);
      d22 = sum(d22);
      d = dev::cmul(sd, dev::cfms(d12, d21, dev::cmul(d11, d22)));
      e2 = most(e2);
    }
    fail = dev::expo(d) < most(e1) + e2 + ey - a.kc;
    if (fail && a.rowdiff) {  // one lane; the others take its result
      bool f2 = true;
      dev::cd d2 = d;
      if (g == 0)
        d2 = rho == 1 ? dev::rowdiff_det(S, L, n, mlab[0], arow, col, Y, 1, ey, a.kc, &f2)
                      : dev::rowdiff2_det(S, L, n, mlab, arow, col, Y, 1, ey, a.kc, &f2);
      f2 = __shfl_sync(gm, (int)f2, grp * G);
      if (!f2) {
        d = make_double2(__shfl_sync(gm, d2.x, grp * G), __shfl_sync(gm, d2.y, grp * G));
        fail = false;
        bits = 1 << (8 + f);
      }
    }
  }
  if (fail) {
    __syncwarp(gm);
    load(n);
    const bool zero = dev::group_lu<G>(B, P, perm, n, n, n, g, gm, 1 << 20, &det, &parity);
    d = zero ? make_double2(0.0, 0.0) : parity ? dev::cneg(det) : det;
    bits = 1 << f;
  }
  if (g == 0) {
    dets[p * a.F + f] = (a.mem_par[m] >> f) & 1 ? dev::cneg(d) : d;
    if (path && bits) atomicOr(&path[p], bits);
  }
}

template <int NCMAX>
__device__ __forceinline__ void kfac_group_one(const FwdArgs& a, int64_t t) {
  using KG = KGroup<NCMAX>;
  extern __shared__ double2 ksm[];
  const int lane = threadIdx.x & 31;
  const int j = lane / KG::G, g = lane % KG::G;
  const unsigned gm = KG::G == 32 ? 0xffffffffu : (((1u << KG::G) - 1u) << (j * KG::G));
  dev::cd* Bs = ksm + (size_t)j * KG::BS;
  dev::cd* Ws = Bs + (NCMAX - 1) * (NCMAX - 1);
  int* Ps = reinterpret_cast<int*>(ksm + (size_t)KG::GPW * KG::BS) + j * KG::PS;
  const int f = (int)(t % a.F);
  const int64_t wq = t / a.F;
  const int Q = (int)(wq % a.n_q);
  const int W = (int)(wq / a.n_q);
  const int n = a.n_f[f];
  if (n <= 6 || !a.q_two[Q]) return;
  const int rho = a.fam_rank[(int64_t)W * a.F + f];
  const int sig = a.q_rank[(int64_t)Q * a.F + f];
  const dev::cd* S = a.S[f];
  const int L = a.L_f[f];
  const int32_t* arow = a.fam_arow + (int64_t)W * a.Tn + a.off_f[f];
  const int32_t* scol = a.snk_pos + (int64_t)a.q_off[Q] * a.Tn + a.off_f[f];
  dev::cd* K = const_cast<dev::cd*>(a.kbuf) + wq * a.kstride + a.koff[f];
  bool gd;
  if (rho >= 3)  // one-sided update for these blocks
    gd = true;
  else if (rho == 2 && sig == 2)  // the (n-2) x (n-2) shared block, kapply's layout (kapply22)
    gd = dev::group_kfac_block<KG::G>(S, L, n - 1, 1, arow, scol, K, a.kp, g, gm, Bs, Ws, Ps, NCMAX, false);
  else if (sig == 2)
    gd = dev::group_kfac_block12<KG::G>(S, L, n, arow, scol, K, a.kp, g, gm, Bs, Ps);
  else
    gd = dev::group_kfac_block<KG::G>(S, L, n, rho, arow, scol, K, a.kp, g, gm, Bs, Ws, Ps, NCMAX, dev::fx_on(a));
  if (g == 0) a.kguard[t] = gd ? 1 : 0;
}

template <int NCMAX>
__global__ void __launch_bounds__(32) kfac_group_kernel(const FwdArgs a, int64_t n_fam) {
  const int64_t u = (int64_t)blockIdx.x * KGroup<NCMAX>::GPW + (threadIdx.x / KGroup<NCMAX>::G);
  if (u >= n_fam * a.n_q * a.F) return;
  kfac_group_one<NCMAX>(a, kfac_index(a, u, n_fam));
}

template <int NCMAX>
__global__ void __launch_bounds__(32) kfac_group_batch_kernel(const FwdArgs* __restrict__ desc,
                                                              const int64_t* __restrict__ kpref,
                                                              const int64_t* __restrict__ nfam, int count) {
  const int64_t t = (int64_t)blockIdx.x * KGroup<NCMAX>::GPW + (threadIdx.x / KGroup<NCMAX>::G);
  if (t >= kpref[count]) return;
  int lo = 0, hi = count - 1;
  while (lo < hi) {  // last k with kpref[k] <= t
    const int mid = (lo + hi + 1) >> 1;
    if (kpref[mid] <= t) lo = mid; else hi = mid - 1;
  }
  const FwdArgs& a = desc[lo];
  if (!a.snk_orig) return;
  kfac_group_one<NCMAX>(a, kfac_index(a, t - kpref[lo], nfam[lo]));
}

}  // namespace fwd

// Block factors of every plan of a batch: blocks with n <= 6 one per thread, blocks with
// n > 6 (present when big != 0) by lane groups.
template <int NCMAX>
cudaError_t launch_kfac_batch_nc(const FwdArgs* desc, const int64_t* kpref, const int64_t* nfam,
                                 int count, int64_t total, int big, cudaStream_t s) {
  if (total == 0) return cudaSuccess;
  fwd::kfac_batch_kernel<NCMAX><<<(unsigned)((total + 127) / 128), 128, 0, s>>>(desc, kpref, nfam, count);
  if (big) {
    using KG = fwd::KGroup<NCMAX>;
    fwd::kfac_group_batch_kernel<NCMAX><<<(unsigned)((total + KG::GPW - 1) / KG::GPW), 32, KG::smem(), s>>>(
        desc, kpref, nfam, count);
  }
  return cudaGetLastError();
}

template <int NCMAX>
cudaError_t launch_kfac_nc(const FwdArgs& a, int64_t n_fam, cudaStream_t s) {
  const int64_t threads = n_fam * a.n_q * a.F;
  if (threads == 0) return cudaSuccess;
  fwd::kfac_kernel<NCMAX><<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(a, n_fam);
  bool big = false;
  for (int f = 0; f < a.F; f++) big |= a.n_f[f] > 6;
  if (big) {
    using KG = fwd::KGroup<NCMAX>;
    fwd::kfac_group_kernel<NCMAX><<<(unsigned)((threads + KG::GPW - 1) / KG::GPW), 32, KG::smem(), s>>>(a, n_fam);
  }
  return cudaGetLastError();
}

// Persistent batched launch: blocks pull (correlator, family, tile) items from a list
// ordered by decreasing cost through one atomic counter; each item's partial goes to its
// own slot (see batch.cu).  Registers as fwd_kernel's (at most 128 threads per block).  The paths with
// and without tables are copies of their own (FP64 items ran 4 % slower through the one that has both).
template <int NCMAX>
__global__ void __maxnreg__(NCMAX <= 8 ? 168 : 255) batch_kernel(const FwdArgs* __restrict__ desc,
                                                    const BatchItem* __restrict__ items,
                                                    int64_t n_items, unsigned long long* head,
                                                    const int64_t* __restrict__ part_off,
                                                    double2* __restrict__ partials) {
  extern __shared__ double2 smem[];
  __shared__ int64_t s_item;
  for (;;) {
    if (threadIdx.x == 0) s_item = (int64_t)atomicAdd(head, 1ull);
    __syncthreads();
    const int64_t it = s_item;
    if (it >= n_items) break;
    const BatchItem bi = items[it];
    const FwdArgs& a = desc[bi.corr];
    double2* partial = &partials[part_off[bi.corr] + (int64_t)bi.W * a.n_tiles + bi.tile];
    if (NCMAX <= 18 && dev::fx_on(a))
      fwd::fwd_item<NCMAX, (NCMAX <= 18), false>(a, bi.W, bi.tile, smem, partial);
    else
      fwd::fwd_item<NCMAX, false, false>(a, bi.W, bi.tile, smem, partial);
    __syncthreads();
  }
}

template <int NCMAX>
cudaError_t launch_batch_nc(int grid, int T, size_t smem, cudaStream_t s, const FwdArgs* desc,
                            const BatchItem* items, int64_t n_items, unsigned long long* head,
                            const int64_t* part_off, double2* partials) {
  // the shared-memory limit was raised by batch_occupancy_nc, outside any stream capture
  batch_kernel<NCMAX><<<grid, T, smem, s>>>(desc, items, n_items, head, part_off, partials);
  return cudaGetLastError();
}

template <int NCMAX>
int batch_occupancy_nc(int T, size_t smem) {
  int nb = 0, dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, batch_kernel<NCMAX>) == cudaSuccess) optin -= (int)fa.sharedSizeBytes;
  cudaFuncSetAttribute(batch_kernel<NCMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_kernel<NCMAX>, T, smem) != cudaSuccess)
    return 1;
  return nb > 0 ? nb : 1;
}

template <int NCMAX, bool FX, bool CW>
cudaError_t launch_fwd_nc(const FwdArgs& a, int tile, int64_t items, size_t smem, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(fwd::fwd_kernel<NCMAX, FX, CW>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  fwd::fwd_kernel<NCMAX, FX, CW><<<(unsigned)items, tile, smem, s>>>(a);
  return cudaGetLastError();
}

template <int NCMAX>
cudaError_t launch_pairs_nc(const FwdArgs& a, int64_t n_pairs, int64_t n_src, const int64_t* ii,
                            const int64_t* jj, const int32_t* src_member, const int32_t* mem_family,
                            double* dets, int32_t* path, cudaStream_t s) {
  const int T = 64;
  const size_t smem = (size_t)a.slots * T * sizeof(double2);
  if (n_pairs == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fwd::pair_kernel<NCMAX>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)((n_pairs + T - 1) / T);
  fwd::pair_kernel<NCMAX><<<grid, T, smem, s>>>(a, n_pairs, n_src, ii, jj, src_member, mem_family,
                                                reinterpret_cast<double2*>(dets), path);
  bool big = false;
  for (int f = 0; f < a.F; f++) big |= a.n_f[f] > 6;
  if (big) {  // after pair_kernel, which writes every pair's path word
    using PG = fwd::PairGroup<NCMAX>;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(fwd::pair_group_kernel<NCMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)PG::smem())) != cudaSuccess)
      return e;
    const int64_t units = n_pairs * a.F;
    fwd::pair_group_kernel<NCMAX><<<(unsigned)((units + PG::GPW - 1) / PG::GPW), 32, PG::smem(), s>>>(
        a, n_pairs, n_src, ii, jj, src_member, mem_family, reinterpret_cast<double2*>(dets), path);
  }
  return cudaGetLastError();
}

}  // namespace mhc
