// Host side of the time-compressed operator (time_basis.cu): the windows of
// bins and the orthonormal basis of each, fitted on sampled rows of W_hat.
// Plain C++, no device code.  Internal header: not part of the C ABI.
#pragma once

#include <math.h>
#include <stddef.h>
#include <string.h>

#include <algorithm>
#include <utility>
#include <vector>

namespace time_fit {

constexpr int TZ_R = 16;             // columns of one window's basis at most (row pitch of the device table)
constexpr int TZ_FIRST = 16;         // bins of the first window
constexpr double TZ_FALL = 1e-3;     // a window ends where the response has fallen by this factor
constexpr double TZ_EPS = 1e-10;     // scaled residual at which a window's rank is reached
constexpr double TZ_FLOOR = 1e-30;   // share of a bin's response below which a depth is not looked at
constexpr double TZ_OWN = 2e-8;      // residual of a bin and depth relative to its own DC response
constexpr double TZ_CHECK = 2e-8;    // residual over all classes, relative to a bin's DC response
constexpr double TZ_CHECK_OWN = 1e-7;  // the same relative to that of the depth in the bin
constexpr double TZ_CANCEL = 20.0;   // largest sum_j |Q V| / |sum_j Q V| over the bins and depths of a window

// Pairs of doubles (the 128-bit vectors of either host), four sums: the fit is
// bound by these loops.
typedef double pair_t __attribute__((vector_size(16)));
inline pair_t pair_at(const double* p) {
  pair_t v;
  memcpy(&v, p, sizeof(v));
  return v;
}

inline double dot(const double* a, const double* b, size_t n) {
  pair_t s = {0.0, 0.0}, t = {0.0, 0.0};
  size_t i = 0;
  for (; i + 4 <= n; i += 4) {
    s += pair_at(a + i) * pair_at(b + i);
    t += pair_at(a + i + 2) * pair_at(b + i + 2);
  }
  for (; i < n; ++i) s[0] += a[i] * b[i];
  return (s[0] + s[1]) + (t[0] + t[1]);
}

// y += f x; the squared norm of the new y (as dot forms it).
inline double axpy(double f, const double* x, double* y, size_t n) {
  const pair_t ff = {f, f};
  pair_t s = {0.0, 0.0}, t = {0.0, 0.0};
  size_t i = 0;
  for (; i + 4 <= n; i += 4) {
    const pair_t u = pair_at(y + i) + ff * pair_at(x + i), v = pair_at(y + i + 2) + ff * pair_at(x + i + 2);
    memcpy(y + i, &u, sizeof(u));
    memcpy(y + i + 2, &v, sizeof(v));
    s += u * u;
    t += v * v;
  }
  for (; i < n; ++i) {
    y[i] += f * x[i];
    s[0] += y[i] * y[i];
  }
  return (s[0] + s[1]) + (t[0] + t[1]);
}

// Largest cancellation in the products of an orthonormal basis g [r][len]: over
// bins and depths of the DC class (sample 0), sum_j |g_j v_j| / |w| with v = g w.
// FP32 rounding of Q and V grows by it.  Infinite where the basis, in FP64, does
// not give the response back.
inline double cancellation(const double* w, int nz, size_t cols, const double* d, int a, int len,
                           const std::vector<double>& g, int r) {
  double worst = 1.0;
  std::vector<double> v(r);
  for (int z = 0; z < nz; ++z) {
    for (int j = 0; j < r; ++j) {
      v[j] = 0.0;
      for (int t = 0; t < len; ++t) v[j] += g[(size_t)j * len + t] * w[(a + t) * cols + z];
    }
    for (int t = 0; t < len; ++t) {
      const double own = w[(a + t) * cols + z];
      if (!(fabs(own) > TZ_FLOOR * d[a + t])) continue;
      double sum = 0.0, mag = 0.0;
      for (int j = 0; j < r; ++j) {
        const double f = g[(size_t)j * len + t] * v[j];
        sum += f;
        mag += fabs(f);
      }
      if (!(fabs(sum - own) <= 2.0 * TZ_OWN * fabs(own))) return INFINITY;
      worst = std::max(worst, mag / fabs(own));
    }
  }
  return worst;
}

// The same space in an order of bins: basis vector i is zero at the bins that the
// vectors before it were taken for.  A deep layer's response rises by many decades
// over the early windows; in the order of size its early bins are the small
// difference of large products, in the order of time each is its own product.  A bin is
// taken in turn when what the vectors so far leave of it is above `theta` (smooth
// neighbours are not), then the largest remainders complete the basis.
inline std::vector<double> in_time_order(const std::vector<double>& g, int r, int len, double theta) {
  std::vector<double> u((size_t)r * r), c(r), h((size_t)r * len, 0.0);
  std::vector<char> used(len, 0);
  int m = 0;
  auto remainder = [&](int t) {
    for (int j = 0; j < r; ++j) c[j] = g[(size_t)j * len + t];
    for (int pass = 0; pass < 2; ++pass)
      for (int l = 0; l < m; ++l) axpy(-dot(c.data(), &u[(size_t)l * r], r), &u[(size_t)l * r], c.data(), r);
    return sqrt(dot(c.data(), c.data(), r));
  };
  auto take = [&](int t) {
    const double nrm = remainder(t);
    for (int j = 0; j < r; ++j) u[(size_t)m * r + j] = c[j] / nrm;
    used[t] = 1;
    ++m;
  };
  for (int t = 0; t < len && m < r; ++t)
    if (remainder(t) >= theta) take(t);
  while (m < r) {
    int best = -1;
    double most = 0.0;
    for (int t = 0; t < len; ++t) {
      const double nrm = used[t] ? 0.0 : remainder(t);
      if (nrm > most) {
        most = nrm;
        best = t;
      }
    }
    if (best < 0) return g;
    take(best);
  }
  for (int i = 0; i < r; ++i)
    for (int j = 0; j < r; ++j) axpy(u[(size_t)i * r + j], &g[(size_t)j * len], &h[(size_t)i * len], len);
  return h;
}

// Basis of the rows [a, b) of w [nt][cols] (column z of sample s at s nz + z):
// q[t - a][j], j < rank; the rank, or -1 when it is above TZ_R or the products
// cancel more than TZ_CANCEL.
inline int window_basis(const double* w, int nz, int ns, const double* d, int a, int b, double* q) {
  const int len = b - a;
  const size_t cols = (size_t)nz * ns;
  // scaled rows, columns of no weight dropped
  std::vector<double> cz(nz, TZ_FLOOR);
  for (int t = a; t < b; ++t)
    for (int z = 0; z < nz; ++z) cz[z] = std::max(cz[z], w[t * cols + z] / d[t]);  // sample 0 is DC
  std::vector<char> keep(cols, 0);
  std::vector<double> thr(nz);
  for (int t = a; t < b; ++t) {
    for (int z = 0; z < nz; ++z) thr[z] = 0.1 * TZ_EPS * d[t] * cz[z];
    for (int s = 0; s < ns; ++s)
      for (int z = 0; z < nz; ++z) keep[(size_t)s * nz + z] |= fabs(w[t * cols + (size_t)s * nz + z]) > thr[z];
  }
  std::vector<size_t> idx;
  for (size_t i = 0; i < cols; ++i)
    if (keep[i]) idx.push_back(i);
  if (idx.empty()) idx.push_back(0);
  const size_t n = idx.size();
  std::vector<int> zi(n);
  std::vector<double> den(nz), nn(len);  // a bin's scale per depth, squared norms of the residual rows
  for (size_t i = 0; i < n; ++i) zi[i] = (int)(idx[i] % nz);
  std::vector<double> e(len * n), res;
  for (int t = 0; t < len; ++t) {
    for (int z = 0; z < nz; ++z) den[z] = d[a + t] * cz[z];
    for (size_t i = 0; i < n; ++i) e[t * n + i] = w[(a + t) * cols + idx[i]] / den[zi[i]];
    nn[t] = dot(&e[t * n], &e[t * n], n);
  }
  res = e;
  std::vector<double> lim((size_t)len * nz);  // a residual's factor to its bin's and depth's own response
  for (int t = 0; t < len; ++t)
    for (int z = 0; z < nz; ++z)
      lim[t * nz + z] = cz[z] / std::max(fabs(w[(a + t) * cols + z]) / d[a + t], TZ_FLOOR);
  // rows pivoted by norm, orthonormalised twice, until the residual is below TZ_EPS everywhere
  std::vector<double> v;
  int r = 0;
  for (; r < len; ++r) {
    int piv = (int)(std::max_element(nn.begin(), nn.end()) - nn.begin());
    double top = sqrt(nn[piv] / n);  // bounds the largest entry from below; the entries themselves where that is too low
    if (!(top >= TZ_EPS))
      for (double u : res) top = std::max(top, fabs(u));
    if (!(top >= TZ_EPS)) {  // in the window's scale; then every bin and depth in its own
      double over = TZ_OWN;
      piv = -1;
      for (int t = 0; t < len; ++t)
        for (size_t i = 0; i < n; ++i) {
          const double rel = fabs(res[t * n + i]) * lim[t * nz + zi[i]];
          if (rel > over) {
            over = rel;
            piv = t;
          }
        }
      if (piv < 0) break;
    }
    if (r == TZ_R) return -1;
    std::vector<double> x(res.begin() + piv * n, res.begin() + (piv + 1) * n);
    for (int pass = 0; pass < 2; ++pass)
      for (int j = 0; j < r; ++j) axpy(-dot(x.data(), &v[j * n], n), &v[j * n], x.data(), n);
    const double nrm = sqrt(dot(x.data(), x.data(), n));
    if (!(nrm > 0.0)) break;
    for (double& u : x) u /= nrm;
    v.insert(v.end(), x.begin(), x.end());
    for (int t = 0; t < len; ++t) nn[t] = axpy(-dot(&res[t * n], x.data(), n), x.data(), &res[t * n], n);
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
  }
  double least = cancellation(w, nz, cols, d, a, len, g, r);
  std::vector<double> pick = g;
  if (!(least <= TZ_CANCEL))
    for (double theta : {0.7, 0.5, 0.25, 0.1}) {
      std::vector<double> h = in_time_order(g, r, len, theta);
      const double c = cancellation(w, nz, cols, d, a, len, h, r);
      if (c < least) {
        least = c;
        pick.swap(h);
      }
    }
  if (!(least <= TZ_CANCEL)) return -1;
  for (int j = 0; j < r; ++j)
    for (int t = 0; t < len; ++t) q[t * TZ_R + j] = pick[(size_t)j * len + t];
  return r;
}

struct Window {
  int begin, end;     // bins
  int plane, planes;  // first column, columns
};

struct Basis {
  std::vector<double> q;      // [nt][TZ_R]
  std::vector<Window> win;
  std::vector<double> tol;    // [nt][nz] largest residual that any class may leave
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
  out->tol.resize((size_t)nt * nz);
  for (int t = 0; t < nt; ++t)
    for (int z = 0; z < nz; ++z)
      out->tol[(size_t)t * nz + z] =
          std::min(TZ_CHECK * d[t], TZ_CHECK_OWN * std::max(fabs(w[t * cols + z]), TZ_FLOOR * d[t]));
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
