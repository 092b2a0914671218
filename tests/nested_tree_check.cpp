// Host check of the nested elimination's tables (csrc/sca_nested_tree.h), compiled and run by
// tests/test_nested_cpu.py.  For every lattice and both forms of the leaves: each site is
// eliminated once and every index lies in its table.  For the smaller lattices the elimination
// is carried out on those tables in complex double, with bounds-checked accesses, exactly as the
// kernels index them, and compared with a pivoted dense inverse.
// Output per lattice and form: L form entries m_max panel_max ld_error g_error (errors -1 where
// not computed).
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <stdexcept>

#include "sca_nested_tree.h"

using namespace sca::nested;
typedef std::complex<double> Z;

static void need(bool ok, const char* what) {
  if (!ok) throw std::runtime_error(what);
}

static void structure(const Tree& t, int* mmax, int* wmax) {
  const int N = t.L * t.L;
  std::vector<int> seen(N, 0);
  *mmax = *wmax = 0;
  long long entries = 0;
  for (const Node& n : t.nodes) {
    const int m = n.p + n.q;
    need(n.front == entries, "fronts overlap");
    entries += (long long)m * m;
    *mmax = std::max(*mmax, m);
    *wmax = std::max(*wmax, n.pw);
    for (int i = 0; i < m; ++i) {
      const int s = t.table.at(n.sites + i);
      need(s >= 0 && s < N, "site");
      if (i < n.p) ++seen[s];
    }
    for (int b = 0; b < n.blacks; ++b) ++seen.at(t.table.at(n.bsite + b));
    for (int k = 0; k < 4 * n.blacks; ++k)
      need(t.table.at(n.bnbr + k) >= 0 && t.table[n.bnbr + k] < m, "black's neighbour");
    for (int k = 0; n.blacks && k < m; ++k)
      need((t.table.at(n.adj + k) >> n.blacks) == 0, "adjacent black");
    need(n.blacks <= 15 && n.pw <= 32, "a warp's width");
    need(n.p > 0 && n.npan * n.pw >= n.p && (n.npan - 1) * n.pw < n.p, "panels");
    need((n.child[0] < 0) == (n.child[1] < 0), "one child");
    if (n.parent >= 0) {
      const Node& par = t.nodes.at(n.parent);
      int prev = -1;
      for (int i = 0; i < n.q; ++i) {
        const int v = t.table.at(n.pmap + i);
        need(v > prev && v < par.p + par.q, "map to the parent");
        need(t.table[par.sites + v] == t.table[n.sites + n.p + i], "site in the parent");
        prev = v;
      }
    }
  }
  need(entries == t.entries && t.levels.size() <= kMaxLevels, "entries");
  for (int s : seen) need(s == 1, "site not eliminated once");
}

static void eliminate(const Tree& t, double* ld_err, double* g_err) {
  const int L = t.L, N = L * L;
  std::mt19937 rng(L);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  std::vector<Z> a(N);
  for (Z& x : a) x = Z(u(rng), 0.3);
  const double tt = 1.3;
  auto adjacent = [&](int i, int j) {
    const int dx = std::abs(i / L - j / L), dy = std::abs(i % L - j % L);
    return (dx == 0 && (dy == 1 || dy == L - 1)) || (dy == 0 && (dx == 1 || dx == L - 1));
  };
  // dense, partial pivoting
  std::vector<Z> W(N * N), I(N * N);
  for (int i = 0; i < N; ++i) {
    I[i * N + i] = 1.0;
    for (int j = 0; j < N; ++j) W[i * N + j] = i == j ? a[i] : adjacent(i, j) ? Z(tt) : Z(0.0);
  }
  double ld = 0.0, ldn = 0.0;
  for (int c = 0; c < N; ++c) {
    int p = c;
    for (int r = c; r < N; ++r)
      if (std::abs(W[r * N + c]) > std::abs(W[p * N + c])) p = r;
    for (int j = 0; j < N; ++j) {
      std::swap(W[c * N + j], W[p * N + j]);
      std::swap(I[c * N + j], I[p * N + j]);
    }
    const Z d = W[c * N + c];
    ld += std::log(std::abs(d));
    for (int j = 0; j < N; ++j) {
      W[c * N + j] /= d;
      I[c * N + j] /= d;
    }
    for (int r = 0; r < N; ++r) {
      const Z f = W[r * N + c];
      if (r == c || f == 0.0) continue;
      for (int j = 0; j < N; ++j) {
        W[r * N + j] -= f * W[c * N + j];
        I[r * N + j] -= f * I[c * N + j];
      }
    }
  }
  // nested
  std::vector<Z> F(t.entries), G(N);
  auto tab = [&](int o) { return (int)t.table.at(o); };
  auto front = [&](const Node& n, int i, int j) -> Z& {
    const int m = n.p + n.q;
    need(i >= 0 && j >= 0 && i < m && j < m, "front index");
    return F.at(n.front + (long long)i * m + j);
  };
  for (int lv = (int)t.levels.size() - 1; lv >= 0; --lv)
    for (int k = t.levels[lv].first; k < t.levels[lv].first + t.levels[lv].count; ++k) {
      const Node& n = t.nodes[k];
      const int m = n.p + n.q;
      std::vector<Z> bt(n.blacks);
      for (int b = 0; b < n.blacks; ++b) {
        bt[b] = tt * tt / a[tab(n.bsite + b)];
        ldn += std::log(std::abs(a[tab(n.bsite + b)]));
      }
      auto at = [&](int hi, int lo) {
        Z v = 0.0;
        for (int c = 0; c < 2; ++c)
          if (n.child[c] >= 0) {
            const Node& ch = t.nodes[n.child[c]];
            const int x = tab(n.cmap[c] + hi), y = tab(n.cmap[c] + lo);
            if (x >= 0 && y >= 0) {
              need(y <= x, "monotonic map");
              v += front(ch, ch.p + x, ch.p + y);
            }
          }
        if (lo < n.p) {
          if (hi == lo) v += a[tab(n.sites + hi)];
          else if (adjacent(tab(n.sites + hi), tab(n.sites + lo))) v += tt;
        }
        for (int b = 0; b < n.blacks; ++b)
          if (tab(n.adj + hi) >> b & tab(n.adj + lo) >> b & 1) v -= bt[b];
        return v;
      };
      for (int pa = 0; pa < n.npan; ++pa) {
        const int o = pa * n.pw, w = std::min(n.pw, n.p - o), l = m - o, r = l - w;
        std::vector<Z> A(w * l), X(w * r);
        for (int i = 0; i < w; ++i)
          for (int j = 0; j < l; ++j) {
            const int hi = std::max(i, j) + o, lo = std::min(i, j) + o;
            A[i * l + j] = pa == 0 ? at(hi, lo) : front(n, hi, lo);
          }
        for (int c = 0; c < w; ++c) {
          const Z d = A[c * l + c];
          ldn += std::log(std::abs(d));
          std::vector<Z> row(w), col(w);
          for (int j = 0; j < w; ++j) {
            row[j] = A[c * l + j] / d;
            col[j] = A[j * l + c];
          }
          for (int i = 0; i < w; ++i)
            for (int j = 0; j < w; ++j)
              A[i * l + j] = i == c ? (j == c ? 1.0 / d : row[j])
                                    : (j == c ? -col[i] / d : A[i * l + j] - col[i] * row[j]);
        }
        for (int i = 0; i < w; ++i)
          for (int j = 0; j < r; ++j)
            for (int c = 0; c < w; ++c) X[i * r + j] += A[i * l + c] * A[c * l + w + j];
        for (int i = 0; i < r; ++i)
          for (int j = 0; j <= i; ++j) {
            Z v = pa == 0 ? at(o + w + i, o + w + j) : front(n, o + w + i, o + w + j);
            for (int c = 0; c < w; ++c) v -= A[c * l + w + i] * X[c * r + j];
            front(n, o + w + i, o + w + j) = v;
          }
        for (int i = 0; i < w; ++i) {
          for (int j = 0; j < w; ++j) front(n, o + i, o + j) = A[i * l + j];
          for (int j = 0; j < r; ++j) front(n, o + i, o + w + j) = X[i * r + j];
        }
      }
    }
  for (const Node& n : t.nodes) {
    const int m = n.p + n.q;
    if (n.parent >= 0)
      for (int i = 0; i < n.q; ++i)
        for (int j = 0; j < n.q; ++j)
          front(n, n.p + i, n.p + j) = front(t.nodes[n.parent], tab(n.pmap + i), tab(n.pmap + j));
    for (int pa = n.npan - 1; pa >= 0; --pa) {
      const int o = pa * n.pw, w = std::min(n.pw, n.p - o), r = m - o - w;
      std::vector<Z> X(w * r), Y(w * r);
      for (int i = 0; i < w; ++i)
        for (int j = 0; j < r; ++j) X[i * r + j] = front(n, o + i, o + w + j);
      for (int i = 0; i < w; ++i)
        for (int j = 0; j < r; ++j)
          for (int c = 0; c < r; ++c) Y[i * r + j] += X[i * r + c] * front(n, o + w + c, o + w + j);
      for (int i = 0; i < w; ++i)
        for (int j = 0; j <= i; ++j) {
          Z s = front(n, o + i, o + j);
          for (int c = 0; c < r; ++c) s += Y[i * r + c] * X[j * r + c];
          front(n, o + i, o + j) = front(n, o + j, o + i) = s;
          if (i == j) G[tab(n.sites + o + i)] = s;
        }
      for (int i = 0; i < w; ++i)
        for (int j = 0; j < r; ++j)
          front(n, o + i, o + w + j) = front(n, o + w + j, o + i) = -Y[i * r + j];
    }
    for (int b = 0; b < n.blacks; ++b) {
      Z s = 0.0;
      for (int x = 0; x < 4; ++x)
        for (int y = 0; y < 4; ++y) s += front(n, tab(n.bnbr + 4 * b + x), tab(n.bnbr + 4 * b + y));
      const Z ai = 1.0 / a[tab(n.bsite + b)];
      G[tab(n.bsite + b)] = ai + ai * ai * tt * tt * s;
    }
  }
  *ld_err = std::abs(ldn - ld);
  *g_err = 0.0;
  for (int i = 0; i < N; ++i) *g_err = std::max(*g_err, std::abs(G[i] - I[i * N + i]));
}

int main(int argc, char** argv) {
  const int dense_up_to = argc > 1 ? std::atoi(argv[1]) : 20;
  for (int L = kMinL; L <= 64; L += 2)
    for (int form = 0; form < 2; ++form) {
      const Tree t = Builder(L).build(form != 0);
      int mmax, wmax;
      structure(t, &mmax, &wmax);
      double le = -1.0, ge = -1.0;
      if (L <= dense_up_to) eliminate(t, &le, &ge);
      std::printf("%d %d %lld %d %d %.3e %.3e\n", L, form, t.entries, mmax, wmax, le, ge);
    }
  return 0;
}
