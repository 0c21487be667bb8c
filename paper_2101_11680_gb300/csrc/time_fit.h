// Host side of the time-compressed operator (time_basis.cu): the windows of
// bins and the orthonormal basis of each, fitted on sampled rows of W_hat.
// Plain C++, no device code.  Internal header: not part of the C ABI.
#pragma once

#include <math.h>
#include <stddef.h>

#include <algorithm>
#include <utility>
#include <vector>

namespace time_fit {

constexpr int TZ_R = 16;             // columns of one window's basis at most (row pitch of the device table)
constexpr int TZ_FIRST = 16;         // bins of the first window
constexpr double TZ_FALL = 1e-3;     // a window ends where the response has fallen by this factor
constexpr double TZ_EPS = 1e-10;     // scaled residual at which a window's rank is reached
constexpr double TZ_FLOOR = 1e-6;    // depths below this share of a bin's response are scaled by it instead

inline double dot(const double* a, const double* b, size_t n) {
  double s[4] = {0, 0, 0, 0};
  size_t i = 0;
  for (; i + 4 <= n; i += 4)
    for (int u = 0; u < 4; ++u) s[u] += a[i + u] * b[i + u];
  for (; i < n; ++i) s[0] += a[i] * b[i];
  return (s[0] + s[1]) + (s[2] + s[3]);
}

inline void axpy(double f, const double* x, double* y, size_t n) {
  for (size_t i = 0; i < n; ++i) y[i] += f * x[i];
}

// Basis of the rows [a, b) of w [nt][cols] (column z of sample s at s nz + z):
// q[t - a][j], j < rank; the rank, or -1 when it is above TZ_R.
inline int window_basis(const double* w, int nz, int ns, const double* d, int a, int b, double* q) {
  const int len = b - a;
  const size_t cols = (size_t)nz * ns;
  // scaled rows, columns of no weight dropped
  std::vector<double> cz(nz, TZ_FLOOR);
  for (int t = a; t < b; ++t)
    for (int z = 0; z < nz; ++z) cz[z] = std::max(cz[z], w[t * cols + z] / d[t]);  // sample 0 is DC
  std::vector<char> keep(cols, 0);
  for (int t = a; t < b; ++t)
    for (size_t i = 0; i < cols; ++i)
      if (fabs(w[t * cols + i]) > 0.1 * TZ_EPS * d[t] * cz[i % nz]) keep[i] = 1;
  std::vector<size_t> idx;
  for (size_t i = 0; i < cols; ++i)
    if (keep[i]) idx.push_back(i);
  if (idx.empty()) idx.push_back(0);
  const size_t n = idx.size();
  std::vector<double> e(len * n), res;
  for (int t = 0; t < len; ++t)
    for (size_t i = 0; i < n; ++i) e[t * n + i] = w[(a + t) * cols + idx[i]] / (d[a + t] * cz[idx[i] % nz]);
  res = e;
  // rows pivoted by norm, orthonormalised twice, until the residual is below TZ_EPS everywhere
  std::vector<double> v;
  int r = 0;
  for (; r < len; ++r) {
    double top = 0.0, best = -1.0;
    int piv = 0;
    for (int t = 0; t < len; ++t) {
      const double* x = res.data() + t * n;
      for (size_t i = 0; i < n; ++i) top = std::max(top, fabs(x[i]));
      const double nn = dot(x, x, n);
      if (nn > best) {
        best = nn;
        piv = t;
      }
    }
    if (!(top >= TZ_EPS)) break;
    if (r == TZ_R) return -1;
    std::vector<double> x(res.begin() + piv * n, res.begin() + (piv + 1) * n);
    for (int pass = 0; pass < 2; ++pass)
      for (int j = 0; j < r; ++j) axpy(-dot(x.data(), &v[j * n], n), &v[j * n], x.data(), n);
    const double nrm = sqrt(dot(x.data(), x.data(), n));
    if (!(nrm > 0.0)) break;
    for (double& u : x) u /= nrm;
    v.insert(v.end(), x.begin(), x.end());
    for (int t = 0; t < len; ++t) axpy(-dot(&res[t * n], x.data(), n), x.data(), &res[t * n], n);
  }
  if (r >= len - 1 && len <= TZ_R) {  // nothing to gain: the bins themselves
    for (int t = 0; t < len; ++t)
      for (int j = 0; j < len; ++j) q[t * TZ_R + j] = t == j ? 1.0 : 0.0;
    return len;
  }
  // the same space in unscaled bins, orthonormal (the pivot order keeps it graded)
  std::vector<double> g((size_t)r * len);
  for (int j = 0; j < r; ++j)
    for (int t = 0; t < len; ++t) g[j * len + t] = dot(&e[t * n], &v[j * n], n) * d[a + t];
  for (int j = 0; j < r; ++j) {
    for (int pass = 0; pass < 3; ++pass) {
      for (int l = 0; l < j; ++l) axpy(-dot(&g[j * len], &g[l * len], len), &g[l * len], &g[j * len], len);
      const double nrm = sqrt(dot(&g[j * len], &g[j * len], len));
      if (!(nrm > 0.0) || !isfinite(nrm)) return -1;
      for (int t = 0; t < len; ++t) g[j * len + t] /= nrm;
    }
    for (int t = 0; t < len; ++t) q[t * TZ_R + j] = g[j * len + t];
  }
  return r;
}

struct Window {
  int begin, end;     // bins
  int plane, planes;  // first column, columns
};

struct Basis {
  std::vector<double> q;      // [nt][TZ_R]
  std::vector<Window> win;
  std::vector<double> dinv;   // [nt] 1 / DC response of each bin
  int rank = 0;
};

inline bool fit(const std::vector<double>& w, int nt, int nz, int ns, Basis* out) {
  const size_t cols = (size_t)nz * ns;
  std::vector<double> d(nt);
  for (int t = 0; t < nt; ++t) {
    double mx = 0.0;
    for (size_t i = 0; i < cols; ++i) {
      if (!isfinite(w[t * cols + i])) return false;
      if (i < (size_t)nz) mx = std::max(mx, fabs(w[t * cols + i]));
    }
    d[t] = mx > 1e-280 ? mx : 1.0;
  }
  std::vector<std::pair<int, int>> todo;
  for (int a = 0; a < nt;) {
    int b = std::min(nt, a == 0 ? TZ_FIRST : 2 * a);
    double mx = d[a];
    for (int t = a + 1; t < b; ++t) {
      mx = std::max(mx, d[t]);
      if (d[t] < TZ_FALL * mx) b = t;
    }
    todo.push_back({a, b});
    a = b;
  }
  std::reverse(todo.begin(), todo.end());
  out->q.assign((size_t)nt * TZ_R, 0.0);
  out->dinv.resize(nt);
  for (int t = 0; t < nt; ++t) out->dinv[t] = 1.0 / d[t];
  while (!todo.empty()) {
    const auto [a, b] = todo.back();
    todo.pop_back();
    const int r = window_basis(w.data(), nz, ns, d.data(), a, b, out->q.data() + (size_t)a * TZ_R);
    if (r < 0) {
      if (b - a <= 1) return false;
      std::fill(out->q.begin() + (size_t)a * TZ_R, out->q.begin() + (size_t)b * TZ_R, 0.0);
      const int mid = (a + b) / 2;
      todo.push_back({mid, b});
      todo.push_back({a, mid});
      continue;
    }
    out->win.push_back({a, b, out->rank, r});
    out->rank += r;
  }
  return true;
}

}  // namespace time_fit
