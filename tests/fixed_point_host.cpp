// Host test of csrc/fx.cuh: the solves and the determinants that the fixed-point path accepts, against
// long double, beside the FP64 path's (csrc/device.cuh: kfac_block, kapply, member_det).  Prints: blocks,
// those refused, sinks, those refused, and the accepted solves' largest error by their largest entry,
// median and maximum, then the same for FP64; determinants accepted, left to the FP64 path, and the
// accepted ones' relative error, median and maximum, then the same for FP64; whether the propagator is
// flat (a call on others takes the FP64 path throughout).
// usage: fixed_point_host n pattern spread kp kc [seed]
//   pattern: rows | cols | both: scaled by random powers of two over 2^spread; decay: by
//   2^-spread per step between 12-label sites; onerow, onecol: one label in eight scaled by 2^-spread;
//   flip: rows and columns alternately by 2^spread; unused: columns that no sink has scaled by 2^spread
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>
#include <vector>

#include "../paper_1411_3691_gb300/csrc/fx.cuh"

using namespace mhc;
typedef std::complex<long double> CL;
typedef dev::cd cd;

static CL wide(cd z) { return CL(z.x, z.y); }

static CL exact_det(std::vector<std::vector<CL>> A) {
  const int n = (int)A.size();
  CL det = 1;
  for (int k = 0; k < n; k++) {
    int p = k;
    for (int i = k; i < n; i++)
      if (std::abs(A[i][k]) > std::abs(A[p][k])) p = i;
    if (p != k) {
      std::swap(A[p], A[k]);
      det = -det;
    }
    det *= A[k][k];
    for (int i = k + 1; i < n; i++) {
      const CL l = A[i][k] / A[k][k];
      for (int q = k; q < n; q++) A[i][q] -= l * A[k][q];
    }
  }
  return det;
}

// z = -B^{-1} a in long double
static std::vector<CL> exact_solve(std::vector<std::vector<CL>> A, std::vector<CL> x) {
  const int n = (int)A.size();
  for (int k = 0; k < n; k++) {
    int p = k;
    for (int i = k; i < n; i++)
      if (std::abs(A[i][k]) > std::abs(A[p][k])) p = i;
    std::swap(A[p], A[k]);
    std::swap(x[p], x[k]);
    for (int i = k + 1; i < n; i++) {
      const CL l = A[i][k] / A[k][k];
      for (int q = k; q < n; q++) A[i][q] -= l * A[k][q];
      x[i] -= l * x[k];
    }
  }
  for (int i = n - 1; i >= 0; i--) {
    for (int q = i + 1; q < n; q++) x[i] -= A[i][q] * x[q];
    x[i] /= A[i][i];
  }
  for (CL& z : x) z = -z;
  return x;
}

int main(int argc, char** argv) {
  const int n = atoi(argv[1]), spread = atoi(argv[3]), kp = atoi(argv[4]), kc = atoi(argv[5]);
  const std::string pattern = argv[2];
  std::mt19937_64 g(argc > 6 ? atoi(argv[6]) : 1);
  std::normal_distribution<double> N(0, std::sqrt(.5));
  const int L = n == 18 ? 96 : 12 * ((n + 2) / 3) + 12, M = n - 1;
  std::vector<cd> S((size_t)L * L);
  std::vector<int> used(L, 1);
  for (int l = 0; l < L; l++)
    if (pattern == "unused" && l % 4 == 3) used[l] = 0;
  std::vector<int> re(L), ce(L);
  for (int l = 0; l < L; l++) re[l] = (int)(g() % (spread + 1)), ce[l] = (int)(g() % (spread + 1));
  for (int a = 0; a < L; a++)
    for (int b = 0; b < L; b++) {
      int e = 0;
      if (pattern == "rows" || pattern == "both") e += re[a];
      if (pattern == "cols" || pattern == "both") e += ce[b];
      if (pattern == "decay") e = -spread * std::abs(a / 12 - b / 12);
      if (pattern == "onerow") e = a % 8 ? 0 : -spread;
      if (pattern == "onecol") e = b % 8 ? 0 : -spread;
      if (pattern == "unused" && !used[b]) e = spread;
      if (pattern == "flip") e = (a ^ b) & 1 ? spread : 0;
      const double f = std::ldexp(1.0, e);
      S[(size_t)a * L + b] = {(N(g) + (a == b ? (n == 18 ? 3 : 2) : 0)) * f, N(g) * f};
    }
  std::vector<int> rexp(L), cexp(L);
  fx::Scan scan;
  for (int l = 0; l < L; l++) {
    int er = -4096, ec = -4096, small = 0, total = 0;
    for (int k = 0; k < L; k++) {
      if (used[k]) er = max(er, dev::expo(S[(size_t)l * L + k]));
      ec = max(ec, dev::expo(S[(size_t)k * L + l]));
    }
    rexp[l] = er + 1;
    cexp[l] = ec + 1;
    for (int k = 0; k < L; k++) {
      total += used[k];
      small += used[k] && fx::small_entry(S[(size_t)l * L + k], rexp[l]);
    }
    scan.row(rexp[l], small, total);
    if (used[l]) scan.column(cexp[l]);
  }
  std::vector<double> efx, e64, dfx, d64;
  long blocks = 0, brefused = 0, sinks = 0, srefused = 0, accepted = 0, left = 0;
  for (int t = 0; t < (n > 9 ? 500 : 1500); t++) {
    std::vector<int> p(L);
    for (int i = 0; i < L; i++) p[i] = i;
    std::shuffle(p.begin(), p.end(), g);
    std::vector<int32_t> rows(p.begin(), p.begin() + M), members(p.begin() + M, p.begin() + M + 4);
    std::shuffle(p.begin(), p.end(), g);
    std::vector<int32_t> cols;
    for (int l : p)
      if (used[l] && (int)cols.size() < n + 3) cols.push_back(l);
    std::vector<cd> K(M * M + M + 2), KX(M * M + M + 2), Y(n);
    const bool guard = dev::kfac_block<18, 0, 1>(S.data(), L, n, rows.data(), cols.data(), K.data(), kp, false);
    if (guard) continue;
    blocks++;
    if (dev::kfac_block<18, 0, 1>(S.data(), L, n, rows.data(), cols.data(), KX.data(), kp, true)) {
      brefused++;
      continue;
    }
    for (int k = 0; k < 4; k++) {  // the sinks of the family: the last column changes
      std::vector<int32_t> c(cols.begin(), cols.begin() + M);
      c.push_back(cols[M + k]);
      int ey = 0;
      dev::kapply<18, 0>(S.data(), L, n, rows.data(), c.data(), K.data(), Y.data(), 1, &ey);
      std::vector<int4> a((size_t)L * L), y(n);
      for (int r : rows) a[(size_t)r * L] = fx::quant(S[(size_t)r * L + c[M]], cexp[c[M]], fx::kABits);
      sinks++;
      int e2 = 0;
      cd sd;
      const int4* F = reinterpret_cast<const int4*>(KX.data());
      if (!fx::solve_sink<true>(n, 1, a.data(), cexp[c[M]], F, KX.data(), y.data(), 1, &e2, &sd)) {
        srefused++;
        continue;
      }
      std::vector<std::vector<CL>> B(M, std::vector<CL>(M));
      std::vector<CL> x(M);
      for (int i = 0; i < M; i++) {
        for (int q = 0; q < M; q++) B[i][q] = wide(S[(size_t)rows[i] * L + c[q]]);
        x[i] = wide(S[(size_t)rows[i] * L + c[M]]);
      }
      const std::vector<CL> z = exact_solve(B, x);
      long double top = 1, dx = 0, dy = 0;  // the unit entry
      for (int i = 0; i < M; i++) {
        const fx::Val v = fx::joined(y[i]);
        top = max(top, std::abs(z[i]));
        const int u = (e2 >> 1) - fx::kFracBits;
        dx = max(dx, std::abs(CL(std::ldexp((long double)v.re, u), std::ldexp((long double)v.im, u)) - z[i]));
        dy = max(dy, std::abs(wide(Y[i]) / wide(Y[M]) - z[i]));  // y = det B z
      }
      efx.push_back((double)(dx / top));
      e64.push_back((double)(dy / top));
      for (int m : members) {
        bool fail = false;
        const cd det64 = dev::member_det<18, 0, 1>(S.data(), L, n, &m, c.data(), Y.data(), 1, ey, kc, &fail);
        if (fail) continue;  // refactored
        fx::Acc s;
        std::vector<int4> row(n);
        for (int q = 0; q < n; q++) {
          row[q] = fx::quant(S[(size_t)m * L + c[q]], rexp[m], fx::kRowBits);
          fx::mac(s, row[q], y[q]);
        }
        const fx::Val v = fx::finish(s);
        const int mag = fx::magnitude(v);
        if (!fx::usable(mag, fx::accepted(n, kc, 1))) {
          left++;
          continue;
        }
        accepted++;
        std::vector<std::vector<CL>> A(n, std::vector<CL>(n));
        for (int i = 0; i < n; i++)
          for (int q = 0; q < n; q++) A[i][q] = wide(S[(size_t)(i < M ? rows[i] : m) * L + c[q]]);
        const CL ref = exact_det(A);
        const int u = (e2 >> 1) + rexp[m] - fx::kDotBits;
        const CL got = CL(std::ldexp((long double)v.re, u), std::ldexp((long double)v.im, u)) * wide(KX[M * M + M + 1]);
        dfx.push_back((double)(std::abs(got - ref) / std::abs(ref)));
        d64.push_back((double)(std::abs(wide(det64) - ref) / std::abs(ref)));
      }
    }
  }
  auto stat = [](std::vector<double> v, double* med, double* mx) {
    *med = *mx = 0;
    if (v.empty()) return;
    std::sort(v.begin(), v.end());
    *med = v[v.size() / 2];
    *mx = v.back();
  };
  double a, b, c, d;
  stat(efx, &a, &b);
  stat(e64, &c, &d);
  printf("%ld %ld %ld %ld %.3e %.3e %.3e %.3e ", blocks, brefused, sinks, srefused, a, b, c, d);
  stat(dfx, &a, &b);
  stat(d64, &c, &d);
  printf("%ld %ld %.3e %.3e %.3e %.3e %d\n", accepted, left, a, b, c, d, (int)scan.flat());
  return 0;
}
