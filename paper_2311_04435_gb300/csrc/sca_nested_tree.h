// Elimination tree of the L x L periodic square lattice for the nested elimination
// (sca_nested.cu): host-side index tables only, no arithmetic.
//
// A_{n,sigma} couples a site to its four neighbours, so a separator (a set of sites whose removal
// splits the lattice) decouples the rest.  The tree is the nested dissection of George (SIAM J.
// Numer. Anal. 10, 345 (1973)) on the torus: the root removes the columns x = 0 and x = L/2; each
// of the two cylinders left removes its rows y = 0 and y = L/2; each of the four rectangles left
// is halved by its middle line, again and again, until a region holds at most kLeafSites sites.  A
// node eliminates its own separator ("pivots"); what it leaves couples only the sites around its
// region ("boundary"), all of which are pivots of its ancestors.  In a leaf the sites of one
// checkerboard colour couple only to the other colour and to the boundary: those ("blacks") can be
// eliminated in closed form, which leaves the other colour as the node's pivots.
//
// A black is a pivot of modulus |A_bb|, which can be as small as w_n, while on disordered fields the
// leaf's block as a whole is far better conditioned (on weak ones it has levels near zero too: see
// the arithmetics in sca_internal.h).  The tree therefore has two forms with the same nodes, which
// differ in the leaves only: `dense_leaves` (every site of a leaf is a pivot of its front), for
// blocks without column dominance (w_n <= 4|t|), and the closed form for the others.  In float64
// on random site energies in [-1, 1] (t = 1, L = 14 and 18) the largest error of G_ii is, dense
// leaves against blacks, 2.4e-15 against 7e-14 at w_n = 0.157 and 9e-16 against 1.2e-14 at 0.314
// (a pivoted dense elimination: 1.4e-15); a dense leaf of 16 sites costs four times the
// multiply-adds of the closed form, a fifth more over the whole tree.
//
// Node `k` works on a front of m = p + q variables: its p pivots, then its q boundary sites in
// the order in which the parent's front lists them (so that maps between fronts are monotonic).
// Fronts are eliminated in panels of at most `panel_width(m)` pivots.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace sca {
namespace nested {

constexpr int kMinL = 6;        // smallest lattice the tree is built for
// A leaf's region: a 4 x 4 leaf has 8 blacks and 8 pivots (or 16 pivots) under 16 boundary sites.
constexpr int kLeafSites = 20;
// Widest panel of a front of m variables: F12 and X of a panel, 2 w (m - w) entries of 16 bytes,
// and two w x w blocks take at most 50 KB of shared memory.
inline int panel_width(int m) {
  int w = 20;
  while (16 * (w * (2 * (m - w) + 2) + 2 * w * w) > 50 * 1024) --w;
  return w;
}
constexpr int kRows = 2;        // rows of a thread's output tile at most
constexpr int kSlots = 2;       // entries of a pivots' block that a thread can hold
constexpr int kMaxLevels = 10;

struct Node {
  int p, q;            // pivots, boundary sites
  int parent;          // node index, -1 for the root
  int child[2];        // node indices, -1 where there is none
  int sites;           // table offset: site of each of the m local variables
  int cmap[2];         // table offset: local variable -> boundary index in child c, -1 if absent
  int pmap;            // table offset: boundary index -> local variable of the parent
  int blacks;          // number of blacks (leaves only)
  int bsite;           // table offset: site of each black
  int bnbr;            // table offset: 4 local variables per black
  int adj;             // table offset: bit mask of the blacks next to each local variable
  int npan, pw;        // panels and the width of the first ones (the last may be narrower)
  long long front;     // offset of the m x m front in a block's storage (entries)
};

struct Level {
  int first, count;    // nodes [first, first + count), all at one depth
};

struct Tree {
  int L = 0;
  std::vector<Node> nodes;      // root first, level by level
  std::vector<Level> levels;    // root level first
  std::vector<int16_t> table;
  long long entries = 0;        // front entries per block
};

class Builder {
 public:
  explicit Builder(int L) : L_(L), pos_(L * L, -1), stamp_(L * L, 0) {}

  Tree build(bool dense_leaves) {
    dense_leaves_ = dense_leaves;
    Tree t;
    t.L = L_;
    const int H = L_ / 2;
    std::vector<Region> cur, next;
    Region root;
    root.kind = 0;
    root.parent = -1;
    cur.push_back(root);
    while (!cur.empty()) {
      const Level lv{(int)t.nodes.size(), (int)cur.size()};
      next.clear();
      for (const Region& r : cur) {
        const int id = (int)t.nodes.size();
        Node n{};
        n.parent = r.parent;
        n.child[0] = n.child[1] = -1;
        std::vector<int> piv, black;
        Region ch[2];
        int nch = 0;
        split(r, H, piv, black, ch, nch);
        std::vector<int> bnd = boundary(r);
        if (r.parent >= 0) {  // order of the parent's front
          const Node& par = t.nodes[r.parent];
          for (int i = 0; i < par.p + par.q; ++i) pos_[t.table[par.sites + i]] = i;
          std::sort(bnd.begin(), bnd.end(), [&](int a, int b) { return pos_[a] < pos_[b]; });
          n.pmap = (int)t.table.size();
          for (int s : bnd) t.table.push_back((int16_t)pos_[s]);
        }
        n.p = (int)piv.size();
        n.q = (int)bnd.size();
        const int m = n.p + n.q;
        n.sites = (int)t.table.size();
        for (int s : piv) t.table.push_back((int16_t)s);
        for (int s : bnd) t.table.push_back((int16_t)s);
        n.blacks = (int)black.size();
        if (n.blacks) {
          for (int i = 0; i < m; ++i) pos_[t.table[n.sites + i]] = i;
          n.bsite = (int)t.table.size();
          for (int s : black) t.table.push_back((int16_t)s);
          n.bnbr = (int)t.table.size();
          std::vector<int> adj(m, 0);
          for (int b = 0; b < n.blacks; ++b) {
            int nb[4];
            neighbours(black[b], nb);
            for (int k = 0; k < 4; ++k) {
              t.table.push_back((int16_t)pos_[nb[k]]);
              adj[pos_[nb[k]]] |= 1 << b;
            }
          }
          n.adj = (int)t.table.size();
          for (int i = 0; i < m; ++i) t.table.push_back((int16_t)adj[i]);
        }
        // (a leaf is one panel)
        const int pw = panel_width(m);
        n.npan = (n.p + pw - 1) / pw;
        n.pw = n.npan ? (n.p + n.npan - 1) / n.npan : 0;
        n.front = t.entries;
        t.entries += (long long)m * m;
        if (r.parent >= 0) {
          Node& par = t.nodes[r.parent];
          const int c = par.child[0] < 0 ? 0 : 1;
          par.child[c] = id;
        }
        t.nodes.push_back(n);
        for (int k = 0; k < nch; ++k) {
          ch[k].parent = id;
          next.push_back(ch[k]);
        }
      }
      t.levels.push_back(lv);
      cur.swap(next);
    }
    // local variable -> boundary index in each child
    for (Node& n : t.nodes)
      for (int c = 0; c < 2; ++c) {
        if (n.child[c] < 0) continue;
        const int m = n.p + n.q;
        n.cmap[c] = (int)t.table.size();
        t.table.resize(t.table.size() + m, -1);
        const Node& k = t.nodes[n.child[c]];
        for (int i = 0; i < k.q; ++i) t.table[n.cmap[c] + t.table[k.pmap + i]] = (int16_t)i;
      }
    return t;
  }

 private:
  // kind 0: the torus, 1: a cylinder (columns [x0, x0 + w), all rows), 2: a rectangle
  struct Region {
    int kind = 0, x0 = 0, w = 0, y0 = 0, h = 0, parent = -1;
  };

  int site(int x, int y) const { return ((x + L_) % L_) * L_ + (y + L_) % L_; }

  void neighbours(int s, int* nb) const {
    const int x = s / L_, y = s % L_;
    nb[0] = site(x + 1, y);
    nb[1] = site(x - 1, y);
    nb[2] = site(x, y + 1);
    nb[3] = site(x, y - 1);
  }

  bool inside(const Region& r, int s) const {
    if (r.kind == 0) return true;
    const int dx = (s / L_ - r.x0 + L_) % L_, dy = (s % L_ - r.y0 + L_) % L_;
    return dx < r.w && (r.kind == 1 || dy < r.h);
  }

  // Sites outside r with a neighbour in r, each once (stamp_ marks what this call has listed).
  std::vector<int> boundary(const Region& r) {
    std::vector<int> out;
    if (r.kind == 0) return out;
    ++stamp_now_;
    const int h = r.kind == 1 ? L_ : r.h;
    for (int a = 0; a < r.w; ++a)
      for (int b = 0; b < h; ++b) {
        if (a > 0 && a < r.w - 1 && (r.kind == 1 || (b > 0 && b < h - 1))) continue;
        int nb[4];
        neighbours(site(r.x0 + a, r.y0 + b), nb);
        for (int k = 0; k < 4; ++k)
          if (!inside(r, nb[k]) && stamp_[nb[k]] != stamp_now_) {
            stamp_[nb[k]] = stamp_now_;
            out.push_back(nb[k]);
          }
      }
    return out;
  }

  static void add(Region* ch, int& n, int kind, int x0, int w, int y0, int h) {
    if (w <= 0 || h <= 0) return;
    ch[n].kind = kind;
    ch[n].x0 = x0;
    ch[n].w = w;
    ch[n].y0 = y0;
    ch[n].h = h;
    ++n;
  }

  void split(const Region& r, int H, std::vector<int>& piv, std::vector<int>& black, Region* ch,
             int& nch) const {
    if (r.kind == 0) {
      for (int x : {0, H})
        for (int y = 0; y < L_; ++y) piv.push_back(site(x, y));
      add(ch, nch, 1, 1, H - 1, 0, L_);
      add(ch, nch, 1, H + 1, L_ - H - 1, 0, L_);
      return;
    }
    if (r.kind == 1) {
      for (int y : {0, H})
        for (int a = 0; a < r.w; ++a) piv.push_back(site(r.x0 + a, y));
      add(ch, nch, 2, r.x0, r.w, 1, H - 1);
      add(ch, nch, 2, r.x0, r.w, H + 1, L_ - H - 1);
      return;
    }
    if (r.w * r.h <= kLeafSites) {
      std::vector<int> col[2];
      for (int a = 0; a < r.w; ++a)
        for (int b = 0; b < r.h; ++b) {
          const int s = site(r.x0 + a, r.y0 + b);
          col[(s / L_ + s % L_) & 1].push_back(s);
        }
      const int k = col[0].size() >= col[1].size() ? 0 : 1;
      if (!dense_leaves_) black = col[k];
      piv = col[1 - k];
      if (dense_leaves_) piv.insert(piv.end(), col[k].begin(), col[k].end());
      return;
    }
    if (r.w >= r.h) {
      const int c = r.w / 2;
      for (int b = 0; b < r.h; ++b) piv.push_back(site(r.x0 + c, r.y0 + b));
      add(ch, nch, 2, r.x0, c, r.y0, r.h);
      add(ch, nch, 2, r.x0 + c + 1, r.w - c - 1, r.y0, r.h);
    } else {
      const int c = r.h / 2;
      for (int a = 0; a < r.w; ++a) piv.push_back(site(r.x0 + a, r.y0 + c));
      add(ch, nch, 2, r.x0, r.w, r.y0, c);
      add(ch, nch, 2, r.x0, r.w, r.y0 + c + 1, r.h - c - 1);
    }
  }

  int L_;
  bool dense_leaves_ = false;
  std::vector<int> pos_;    // local variable of a site in the front at hand
  std::vector<int> stamp_;
  int stamp_now_ = 0;
};

}  // namespace nested
}  // namespace sca
