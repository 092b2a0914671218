// Nested elimination of the blocks A_{n,sigma} (Eq. 2): ln|det A| and diag(A^{-1}) from the
// lattice's own sparsity instead of a dense sweep.
//
// A = (i w_n + mu) I - H_sigma couples a site to its four neighbours only.  The tree of
// sca_nested_tree.h eliminates it front by front, children before parents ("up"): a node
// assembles its m x m front (its own entries of A plus its children's Schur complements), inverts
// its pivots' block P = F11^{-1}, keeps P and X = P F12, and leaves F22 - F12^T X to its parent.
// The pivots' product is det A.  Then parents before children ("down"), with G the front's part of
// A^{-1} (Takahashi's recurrence; symmetric like A): from G on the boundary, which is part of the
// parent's front,
//   G_pb = -X G_bb,   G_pp = P + (X G_bb) X^T,
// so the diagonal of A^{-1} comes out of entries inside the fronts, exactly, with no full inverse.
// A block of N = 1600 sites takes 3.4 M complex multiply-adds this way, against N^3 = 4.1 G in the
// dense Gauss-Jordan sweep.
//
// No pivot is searched for: -i A has the Hermitian part (Im z) I with Im z = w_n > 0 (eta for a
// density of states), and so has every Schur complement and every leading block of one; each
// pivot is at least Im z in modulus.  Rounding errors grow by powers of |t| / Im z, which is why
// callers with Im z below kMinImag |t| take the pivoted dense elimination (nested_rule).
//
// Arithmetic: float64, or on the reduced-precision paths double-float (an unevaluated sum of two
// float32, 48 bits): products exact by FMA, sums by two-sums, 12 float32 instructions per real
// multiply-add.  This GPU does 64 float32 FMAs in the time of one float64 FMA, so double-float is
// 5 times as fast as float64 and keeps 24 bits more than the float32 blocks of the dense paths.
//
// Work split: one CTA per (node, block), one launch per tree level and direction, fronts in
// global memory (a block's fronts take 3.2 MB at N = 1600), the current panel of at most 20 pivot
// rows and its X in shared memory.  Both number types are bound by their arithmetic: a panel of w
// rows does w / 2 multiply-adds per front entry that it reads and writes.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "sca_device.cuh"
#include "sca_internal.h"
#include "sca_nested_tree.h"

namespace sca {
namespace {

using nested::Node;

// ------------------------------------------------------------------ numbers
struct alignas(16) Zd {
  double re, im;
};
struct alignas(16) Zf {  // re = rh + rl, im = ih + il
  float rh, rl, ih, il;
};

// Running sums: float64, or a float32 sum with the sum of its rounding errors.
struct Ad {
  double re, im;
};
struct Af {
  float rs, rc, is, ic;
};
template <typename Z>
struct AccOf;
template <>
struct AccOf<Zd> {
  using type = Ad;
};
template <>
struct AccOf<Zf> {
  using type = Af;
};

__device__ __forceinline__ void zset(Zd& z, double re, double im) { z = {re, im}; }
__device__ __forceinline__ void zset(Zf& z, double re, double im) {
  const dsf a = ds_of(re), b = ds_of(im);
  z = {a.h, a.l, b.h, b.l};
}
__device__ __forceinline__ double zre(Zd z) { return z.re; }
__device__ __forceinline__ double zim(Zd z) { return z.im; }
__device__ __forceinline__ double zre(Zf z) { return (double)z.rh + (double)z.rl; }
__device__ __forceinline__ double zim(Zf z) { return (double)z.ih + (double)z.il; }
__device__ __forceinline__ Zd zneg(Zd z) { return {-z.re, -z.im}; }
__device__ __forceinline__ Zf zneg(Zf z) { return {-z.rh, -z.rl, -z.ih, -z.il}; }
__device__ __forceinline__ Zd zadd(Zd a, Zd b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Zf zadd(Zf a, Zf b) {
  const dsf r = ds_add({a.rh, a.rl}, {b.rh, b.rl}), i = ds_add({a.ih, a.il}, {b.ih, b.il});
  return {r.h, r.l, i.h, i.l};
}

__device__ __forceinline__ void acc_of(Ad& a, Zd z) { a = {z.re, z.im}; }
__device__ __forceinline__ void acc_of(Af& a, Zf z) { a = {z.rh, z.rl, z.ih, z.il}; }
__device__ __forceinline__ Zd acc_get(Ad a) { return {a.re, a.im}; }
__device__ __forceinline__ Zf acc_get(Af a) {
  const dsf r = two_sum(a.rs, a.rc), i = two_sum(a.is, a.ic);
  return {r.h, r.l, i.h, i.l};
}

__device__ __forceinline__ void mac(Ad& s, Zd a, Zd b) {
  s.re = fma(a.re, b.re, s.re);
  s.im = fma(a.re, b.im, s.im);
  s.re = fma(-a.im, b.im, s.re);
  s.im = fma(a.im, b.re, s.im);
}
// (s + c) += (ah + al)(bh + bl): the product's leading part exactly (p + e), its cross terms to
// float32 relative accuracy, the sum's rounding error kept in c.  The intrinsics keep the
// compiler from contracting p into the additions.
__device__ __forceinline__ void mac1(float& s, float& c, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = fmaf(ah, bh, -p);
  e = fmaf(ah, bl, e);
  e = fmaf(al, bh, e);
  const float t = __fadd_rn(s, p), z = __fadd_rn(t, -s);
  const float r = __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -z)), __fadd_rn(p, -z));
  s = t;
  c = __fadd_rn(c, __fadd_rn(r, e));
}
__device__ __forceinline__ void mac(Af& s, Zf a, Zf b) {
  mac1(s.rs, s.rc, a.rh, a.rl, b.rh, b.rl);
  mac1(s.is, s.ic, a.rh, a.rl, b.ih, b.il);
  mac1(s.rs, s.rc, -a.ih, -a.il, b.ih, b.il);
  mac1(s.is, s.ic, a.ih, a.il, b.rh, b.rl);
}
template <typename Z>
__device__ __forceinline__ Z zmul(Z a, Z b) {
  typename AccOf<Z>::type s{};
  mac(s, a, b);
  return acc_get(s);
}
__device__ __forceinline__ Zd zinv(Zd z) {
  const double d = 1.0 / (z.re * z.re + z.im * z.im);
  return {z.re * d, -z.im * d};
}
__device__ __forceinline__ Zf zinv(Zf z) {
  float s = 0.f, c = 0.f;
  mac1(s, c, z.rh, z.rl, z.rh, z.rl);
  mac1(s, c, z.ih, z.il, z.ih, z.il);
  const dsf d = two_sum(s, c);
  const float q = 1.0f / d.h;  // then one Newton step: q + q (1 - d q)
  float e = fmaf(-q, d.h, 1.0f);
  e = fmaf(-q, d.l, e);
  const float ql = __fmul_rn(q, e);
  float rs = 0.f, rc = 0.f, is = 0.f, ic = 0.f;
  mac1(rs, rc, z.rh, z.rl, q, ql);
  mac1(is, ic, -z.ih, -z.il, q, ql);
  const dsf r = two_sum(rs, rc), i = two_sum(is, ic);
  return {r.h, r.l, i.h, i.l};
}

// ------------------------------------------------------------------ kernels
template <typename Z>
struct NestArgs {
  const Node* nodes;     // the two forms of the tree, nnodes each: closed-form, dense leaves
  const int16_t* tab;
  Z* fronts;             // fronts of the pass's blocks, `stride` entries apart
  long long stride;
  double* ldp;           // [block of the pass][node]: the node's share of ln|det A|
  int nnodes;
  int b0;                // block of the pass's first slot
  Lattice la;
  double* ld;            // ln|det A_b|
  double* gd;            // [b][site]: sigma Re G_ii (or Im G_ii where zshift is set)
  int* flags;
};

// The nodes of the form that a block with shift imaginary part zi takes: dense leaves unless its
// columns are diagonally dominant (the line of the dense elimination's pivoted group).
template <typename Z>
__device__ __forceinline__ const Node* tree_of(const NestArgs<Z>& a, double t, double zi) {
  return a.nodes + (zi > 4.0 * fabs(t) * (1.0 + 1e-3) ? 0 : a.nnodes);
}

__device__ __forceinline__ bool adjacent(int L, int a, int b) {
  const int dx = abs(a / L - b / L), dy = abs(a % L - b % L);
  return (dx == 0 && (dy == 1 || dy == L - 1)) || (dy == 0 && (dx == 1 || dx == L - 1));
}

// Entry (hi, lo) of a front before its own elimination, hi >= lo: A's entry where lo is a pivot
// (entries between boundary sites belong to an ancestor), the children's Schur complements, and
// in a leaf the closed-form elimination of the blacks next to both sites (bt = t^2 / a_b).
template <typename Z>
struct Front {
  int L;
  double t;
  const Z* c[2];        // children's Schur complements (their boundary parts), row stride cm
  int cm[2];
  int p, leaf;
  const int16_t *site, *cmap0, *cmap1, *adj;
  const Z* bt;
  const Z* diag;        // A_ii of the pivots
  __device__ __forceinline__ Z at(int hi, int lo) const {
    Z v;
    zset(v, 0.0, 0.0);
    if (leaf) {
      for (int x = 0; x < 4; ++x) {
        const int b = adj[4 * hi + x];
        if (b < 0) break;
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (adj[4 * lo + y] == b) v = zadd(v, zneg(bt[b]));
      }
    } else {
      if (c[0]) {
        const int i = cmap0[hi], j = cmap0[lo];
        if (i >= 0 && j >= 0) v = c[0][(size_t)i * cm[0] + j];
      }
      if (c[1]) {
        const int i = cmap1[hi], j = cmap1[lo];
        if (i >= 0 && j >= 0) v = zadd(v, c[1][(size_t)i * cm[1] + j]);
      }
    }
    if (lo < p) {
      if (hi == lo) {
        v = zadd(v, diag[lo]);
      } else if (adjacent(L, site[hi], site[lo])) {
        Z b;
        zset(b, t, 0.0);
        v = zadd(v, b);
      }
    }
    return v;
  }
};

// One node of one block, up: see the file comment.  Shared memory: the panel's rows A (w x the
// rest of the front), X, the leaf's blacks, the pivots' diagonal and the index maps.
template <typename Z, int NT>
__global__ void __launch_bounds__(NT) k_nest_up(NestArgs<Z> a, int first) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Acc = typename AccOf<Z>::type;
  constexpr int kEntries = (nested::kPanel * nested::kPanel + NT - 1) / NT;
  const int mat = blockIdx.y, tid = threadIdx.x;
  int n, sg;
  const Lattice la = block_lattice(a.la, a.b0 + mat, n, sg);
  double zr = la.mu, zi = (2.0 * n + 1.0) * kPi * la.T;
  if (la.zshift) {
    zr = la.zshift[2 * n];
    zi = la.zshift[2 * n + 1];
  }
  const Node* nodes = tree_of(a, la.t, zi);
  const Node nd = nodes[first + blockIdx.x];
  const int p = nd.p, m = nd.p + nd.q;
  Z* base = a.fronts + (size_t)mat * a.stride;
  Z* F = base + nd.front;
  Z* A = reinterpret_cast<Z*>(smem);
  Z* X = A + nd.pw * m;
  Z* bt = X + nd.pw * (m - nd.pw);
  Z* diag = bt + nd.blacks;
  double* mag = reinterpret_cast<double*>(diag + p);
  int16_t* site = reinterpret_cast<int16_t*>(mag + 32);
  int16_t* cm0 = site + m;
  int16_t* cm1 = cm0 + m;
  int16_t* adj = cm1 + m;
  double ld = 0.0;  // warp 0
  for (int i = tid; i < m; i += NT) {
    site[i] = a.tab[nd.sites + i];
    cm0[i] = nd.child[0] >= 0 ? a.tab[nd.cmap[0] + i] : (int16_t)-1;
    cm1[i] = nd.child[1] >= 0 ? a.tab[nd.cmap[1] + i] : (int16_t)-1;
    if (i < p) zset(diag[i], zr - site_energy(la, a.tab[nd.sites + i], sg), zi);
  }
  if (nd.blacks) {
    for (int i = tid; i < 4 * m; i += NT) adj[i] = a.tab[nd.adj + i];
    for (int b0 = 0; b0 < nd.blacks; b0 += 32)
      if (tid < 32) {
        double l = 0.0;
        if (b0 + tid < nd.blacks) {
          const double ar = zr - site_energy(la, a.tab[nd.bsite + b0 + tid], sg);
          Z z, t2;
          zset(z, ar, zi);
          zset(t2, la.t * la.t, 0.0);
          bt[b0 + tid] = zmul(t2, zinv(z));
          const double m2 = ar * ar + zi * zi;
          const bool ok = m2 > 0.0 && isfinite(m2);
          if (!ok) atomicOr(a.flags, 1);
          l = 0.5 * log(ok ? m2 : 1.0);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        ld += l;
      }
  }
  Front<Z> f;
  f.L = la.L;
  f.t = la.t;
  for (int c = 0; c < 2; ++c) {
    f.c[c] = nullptr;
    f.cm[c] = 0;
    if (nd.child[c] >= 0) {
      const Node k = nodes[nd.child[c]];
      const int mc = k.p + k.q;
      f.c[c] = base + k.front + (size_t)k.p * mc + k.p;
      f.cm[c] = mc;
    }
  }
  f.p = p;
  f.leaf = nd.blacks > 0;
  f.site = site;
  f.cmap0 = cm0;
  f.cmap1 = cm1;
  f.adj = adj;
  f.bt = bt;
  f.diag = diag;
  __syncthreads();
  for (int pa = 0; pa < nd.npan; ++pa) {
    const int o = pa * nd.pw, w = min(nd.pw, p - o), l = m - o, r = l - w;
    // ---- the panel's rows
    for (int e = tid; e < w * l; e += NT) {
      const int i = e / l, j = e - i * l;
      const int hi = max(i, j) + o, lo = min(i, j) + o;
      A[i * l + j] = pa == 0 ? f.at(hi, lo) : F[(size_t)hi * m + lo];
    }
    __syncthreads();
    // ---- P = F11^{-1} in place (Gauss-Jordan, diagonal pivots in order)
    for (int c = 0; c < w; ++c) {
      const Z d = A[c * l + c];
      const Z dinv = zinv(d);
      if (tid == 0) mag[c] = zre(d) * zre(d) + zim(d) * zim(d);
      Z val[kEntries];
#pragma unroll
      for (int u = 0; u < kEntries; ++u) {
        const int e = tid + u * NT;
        if (e >= w * w) break;
        const int i = e / w, j = e - i * w;
        const Z row = A[c * l + j], col = A[i * l + c];
        if (i == c) {
          val[u] = j == c ? dinv : zmul(row, dinv);
        } else if (j == c) {
          val[u] = zneg(zmul(col, dinv));
        } else {
          Acc s;
          acc_of(s, A[i * l + j]);
          mac(s, zneg(col), zmul(row, dinv));
          val[u] = acc_get(s);
        }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kEntries; ++u) {
        const int e = tid + u * NT;
        if (e >= w * w) break;
        const int i = e / w, j = e - i * w;
        A[i * l + j] = val[u];
      }
      __syncthreads();
    }
    if (tid < 32) {
      const double m2 = tid < w ? mag[tid] : 1.0;
      const bool ok = m2 > 0.0 && isfinite(m2);
      if (!ok) atomicOr(a.flags, 1);
      double v = 0.5 * log(ok ? m2 : 1.0);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      ld += v;
    }
    // ---- X = P F12, two rows per thread
    const int hw = (w + 1) / 2;
    for (int e = tid; e < hw * r; e += NT) {
      const int i = e / r, j = e - i * r;
      const int i1 = min(i + hw, w - 1);
      Acc s0{}, s1{};
#pragma unroll 2
      for (int k = 0; k < w; ++k) {
        const Z v = A[k * l + w + j];
        mac(s0, A[i * l + k], v);
        mac(s1, A[i1 * l + k], v);
      }
      X[i * r + j] = acc_get(s0);
      if (i + hw < w) X[i1 * r + j] = acc_get(s1);
    }
    __syncthreads();
    // ---- P and X to the front's panel rows
    for (int e = tid; e < w * l; e += NT) {
      const int i = e / l, j = e - i * l;
      F[(size_t)(o + i) * m + o + j] = j < w ? A[i * l + j] : X[i * r + j - w];
    }
    // ---- F22 - F12^T X, lower triangle: each thread four entries, rows and columns h apart so
    // that neighbouring lanes read neighbouring entries
    const int h = (r + 1) / 2, tiles = h * (h + 1) / 2;
    Z* R = F + (size_t)(o + w) * (m + 1);
    for (int e = tid; e < tiles; e += NT) {
      int ti = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
      while ((ti + 1) * (ti + 2) / 2 <= e) ++ti;
      while (ti * (ti + 1) / 2 > e) --ti;
      const int tj = e - ti * (ti + 1) / 2;
      const bool in_i = ti + h < r, in_j = tj + h < r;
      const int i1 = in_i ? ti + h : ti, j1 = in_j ? tj + h : tj;
      Acc s00{}, s10{}, s01{}, s11{};
#pragma unroll 2
      for (int k = 0; k < w; ++k) {
        const Z* Ak = A + k * l + w;
        const Z a0 = zneg(Ak[ti]), a1 = zneg(Ak[i1]);
        const Z x0 = X[k * r + tj], x1 = X[k * r + j1];
        mac(s00, a0, x0);
        mac(s10, a1, x0);
        mac(s01, a0, x1);
        mac(s11, a1, x1);
      }
      auto put = [&](int i, int j, const Acc& s) {
        const Z v = pa == 0 ? f.at(o + w + i, o + w + j) : R[(size_t)i * m + j];
        R[(size_t)i * m + j] = zadd(v, acc_get(s));
      };
      put(ti, tj, s00);
      if (in_i) put(i1, tj, s10);
      if (in_i && in_j) put(i1, j1, s11);
      if (in_j && ti != tj) put(j1, ti, s01);
    }
    __syncthreads();
  }
  double* ldp = a.ldp + (size_t)mat * a.nnodes;
  if (tid == 0) ldp[first + blockIdx.x] = ld;
  if (nd.parent < 0) {  // the root: ln|det A| over all nodes in a fixed order
    __syncthreads();
    __shared__ double part[NT];
    double v = 0.0;
    for (int k = tid; k < a.nnodes; k += NT) v += ldp[k];
    part[tid] = v;
    __syncthreads();
    for (int s = NT / 2; s > 0; s >>= 1) {
      if (tid < s) part[tid] += part[tid + s];
      __syncthreads();
    }
    if (tid == 0) a.ld[a.b0 + mat] = part[0];
  }
}

// One node of one block, down.  Panels in reverse; R is the part of the front after the panel,
// already G.  Four rows of Y = X R per thread: R is read from global memory (L1 and L2 hold it),
// X broadcast from shared memory.
template <typename Z, int NT>
__global__ void __launch_bounds__(NT) k_nest_down(NestArgs<Z> a, int first) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Acc = typename AccOf<Z>::type;
  const int mat = blockIdx.y, tid = threadIdx.x;
  int n, sg;
  const Lattice la = block_lattice(a.la, a.b0 + mat, n, sg);
  double zr = la.mu, zi = (2.0 * n + 1.0) * kPi * la.T;
  if (la.zshift) {
    zr = la.zshift[2 * n];
    zi = la.zshift[2 * n + 1];
  }
  const Node* nodes = tree_of(a, la.t, zi);
  const Node nd = nodes[first + blockIdx.x];
  const int p = nd.p, q = nd.q, m = nd.p + nd.q;
  Z* base = a.fronts + (size_t)mat * a.stride;
  Z* F = base + nd.front;
  const int ldx = (m - nd.pw) | 1;  // odd: rows of 16-byte entries start in different banks
  Z* X = reinterpret_cast<Z*>(smem);
  Z* Y = X + nd.pw * ldx;
  int16_t* map = reinterpret_cast<int16_t*>(Y + nd.pw * ldx);
  double* gd = a.gd + (size_t)(a.b0 + mat) * la.N;
  if (nd.parent >= 0) {
    const Node pr = nodes[nd.parent];
    const int mp = pr.p + pr.q;
    const Z* G = base + pr.front;
    for (int i = tid; i < q; i += NT) map[i] = a.tab[nd.pmap + i];
    __syncthreads();
    for (int e = tid; e < q * q; e += NT) {
      const int i = e / q, j = e - i * q;
      F[(size_t)(p + i) * m + p + j] = G[(size_t)map[i] * mp + map[j]];
    }
    __syncthreads();
  }
  for (int pa = nd.npan - 1; pa >= 0; --pa) {
    const int o = pa * nd.pw, w = min(nd.pw, p - o), r = m - o - w;
    Z* R = F + (size_t)(o + w) * (m + 1);
    for (int e = tid; e < w * r; e += NT) {
      const int i = e / r, j = e - i * r;
      X[i * ldx + j] = F[(size_t)(o + i) * m + o + w + j];
    }
    __syncthreads();
    const int hw = (w + 3) / 4;
    for (int e = tid; e < hw * r; e += NT) {
      const int i = e / r, j = e - i * r;
      const int i1 = min(i + hw, w - 1), i2 = min(i + 2 * hw, w - 1), i3 = min(i + 3 * hw, w - 1);
      Acc s0{}, s1{}, s2{}, s3{};
#pragma unroll 2
      for (int k = 0; k < r; ++k) {
        const Z g = R[(size_t)k * m + j];
        mac(s0, X[i * ldx + k], g);
        mac(s1, X[i1 * ldx + k], g);
        mac(s2, X[i2 * ldx + k], g);
        mac(s3, X[i3 * ldx + k], g);
      }
      Y[i * ldx + j] = acc_get(s0);
      if (i + hw < w) Y[i1 * ldx + j] = acc_get(s1);
      if (i + 2 * hw < w) Y[i2 * ldx + j] = acc_get(s2);
      if (i + 3 * hw < w) Y[i3 * ldx + j] = acc_get(s3);
    }
    __syncthreads();
    for (int e = tid; e < w * (w + 1) / 2; e += NT) {
      int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
      while ((i + 1) * (i + 2) / 2 <= e) ++i;
      while (i * (i + 1) / 2 > e) --i;
      const int j = e - i * (i + 1) / 2;
      Acc s;
      acc_of(s, F[(size_t)(o + i) * m + o + j]);
#pragma unroll 2
      for (int k = 0; k < r; ++k) mac(s, Y[i * ldx + k], X[j * ldx + k]);
      const Z g = acc_get(s);
      F[(size_t)(o + i) * m + o + j] = g;
      if (i != j) F[(size_t)(o + j) * m + o + i] = g;
      if (i == j)
        gd[a.tab[nd.sites + o + i]] = la.zshift ? zim(g) : sg * zre(g);
    }
    for (int e = tid; e < w * r; e += NT) {
      const int i = e / r, j = e - i * r;
      F[(size_t)(o + i) * m + o + w + j] = zneg(Y[i * ldx + j]);
    }
    for (int e = tid; e < w * r; e += NT) {
      const int j = e / w, i = e - j * w;
      F[(size_t)(o + w + j) * m + o + i] = zneg(Y[i * ldx + j]);
    }
    __syncthreads();
  }
  // blacks: G_bb = 1/a + (t/a)^2 sum_{u,v} G_uv over the black's neighbours
  if (nd.blacks) {
    for (int b = tid; b < nd.blacks; b += NT) {
      const int s = a.tab[nd.bsite + b];
      Z z, t2, sum;
      zset(z, zr - site_energy(la, s, sg), zi);
      zset(t2, la.t * la.t, 0.0);
      zset(sum, 0.0, 0.0);
      for (int u = 0; u < 4; ++u) {
        const int iu = a.tab[nd.bnbr + 4 * b + u];
        for (int v = 0; v < 4; ++v) sum = zadd(sum, F[(size_t)iu * m + a.tab[nd.bnbr + 4 * b + v]]);
      }
      const Z ai = zinv(z);
      const Z g = zadd(ai, zmul(zmul(zmul(ai, t2), ai), sum));
      gd[s] = la.zshift ? zim(g) : sg * zre(g);
    }
  }
}

// Im Tr G per block for a density of states: fixed-order sum of the row that k_nest_down wrote.
__global__ void __launch_bounds__(256) k_nest_trace(int N, int b0, const double* gd, double* tr) {
  __shared__ double part[256];
  const int b = b0 + blockIdx.x;
  double v = 0.0;
  for (int i = threadIdx.x; i < N; i += 256) v += gd[(size_t)b * N + i];
  part[threadIdx.x] = v;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) part[threadIdx.x] += part[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) tr[b] = part[0];
}

#define SCA_LAUNCH_CHECK(where)                                   \
  do {                                                            \
    g_launches.fetch_add(1, std::memory_order_relaxed);           \
    cudaError_t err__ = cudaGetLastError();                       \
    if (err__ != cudaSuccess) return cuda_fail(err__, where);     \
  } while (0)

size_t up_smem(const nested::Node& n) {
  const size_t m = n.p + n.q;
  return 16 * ((size_t)n.pw * (2 * m - n.pw) + n.blacks + n.p) + 32 * sizeof(double) +
         sizeof(int16_t) * m * (n.blacks ? 7 : 3);
}
size_t down_smem(const nested::Node& n) {
  const size_t m = n.p + n.q;
  return 32 * (size_t)n.pw * ((m - n.pw) | 1) + sizeof(int16_t) * n.q;
}

struct LevelPlan {
  int first, count, nt;
  size_t smem_up, smem_down;
};

}  // namespace

// Per-context state: the tree's tables on the device and the launch plan.
struct Nested {
  Node* d_nodes = nullptr;
  int16_t* d_tab = nullptr;
  std::vector<LevelPlan> levels;
  int nnodes = 0;
  long long stride = 0;   // entries per block
  int cap = 0;            // blocks per pass
};

namespace {

template <typename Z, int NT>
sca_status allow_smem() {
  static ContextOnce once;
  if (once.done()) return SCA_OK;
  int dev = 0, optin = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa;
  if (err == cudaSuccess) err = cudaFuncGetAttributes(&fa, k_nest_up<Z, NT>);
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_nest_up<Z, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               optin - (int)fa.sharedSizeBytes);
  if (err == cudaSuccess) err = cudaFuncGetAttributes(&fa, k_nest_down<Z, NT>);
  if (err == cudaSuccess)
    err = cudaFuncSetAttribute(k_nest_down<Z, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               optin - (int)fa.sharedSizeBytes);
  if (err != cudaSuccess) return cuda_fail(err, "nested elimination set-up");
  once.mark();
  return SCA_OK;
}

template <typename Z, int NT>
sca_status launch_level(Engine& e, const NestArgs<Z>& a, const LevelPlan& lv, int cnt, bool up,
                        cudaStream_t s) {
  sca_status st = allow_smem<Z, NT>();
  if (st != SCA_OK) return st;
  const int kind = up ? kNestUp : kNestDown;
  prof_begin(e, kind, s);
  if (up)
    k_nest_up<Z, NT><<<dim3(lv.count, cnt), NT, lv.smem_up, s>>>(a, lv.first);
  else
    k_nest_down<Z, NT><<<dim3(lv.count, cnt), NT, lv.smem_down, s>>>(a, lv.first);
  prof_end(e, kind, s);
  SCA_LAUNCH_CHECK(up ? "nested elimination" : "nested inverse diagonal");
  return SCA_OK;
}

template <typename Z>
sca_status run_nested_t(Engine& e, const Lattice& la, bool up, bool down, cudaStream_t s) {
  const Nested& ne = *e.nest;
  NestArgs<Z> a;
  a.nodes = ne.d_nodes;
  a.tab = ne.d_tab;
  a.fronts = static_cast<Z*>(e.M);
  a.stride = ne.stride;
  a.nnodes = ne.nnodes;
  a.la = la;
  a.ld = e.ld;
  a.gd = e.gd;
  a.flags = e.flags;
  const int cap = std::min(ne.cap, 65535);
  for (int b0 = 0; b0 < e.B; b0 += cap) {
    const int cnt = std::min(cap, e.B - b0);
    a.b0 = b0;
    a.ldp = reinterpret_cast<double*>(a.fronts + (size_t)cnt * ne.stride);
    const int nl = (int)ne.levels.size();
    for (int pass = 0; pass < 2; ++pass) {
      if (!(pass == 0 ? up : down)) continue;
      for (int k = 0; k < nl; ++k) {
        const LevelPlan& lv = ne.levels[pass == 0 ? nl - 1 - k : k];
        const sca_status st = lv.nt == 64    ? launch_level<Z, 64>(e, a, lv, cnt, pass == 0, s)
                              : lv.nt == 128 ? launch_level<Z, 128>(e, a, lv, cnt, pass == 0, s)
                                             : launch_level<Z, 256>(e, a, lv, cnt, pass == 0, s);
        if (st != SCA_OK) return st;
      }
    }
    if (down && la.zshift) {
      prof_begin(e, kRefine, s);
      k_nest_trace<<<cnt, 256, 0, s>>>(e.N, b0, e.gd, e.tr);
      prof_end(e, kRefine, s);
      SCA_LAUNCH_CHECK("nested trace");
    }
  }
  return SCA_OK;
}

}  // namespace

bool nested_rule(double t, double imag_min, double imag_max) {
  return imag_min >= kNestedMinImag * std::fabs(t) && imag_min >= 1e-9 && imag_max <= 1e9 &&
         std::fabs(t) <= 1e9;
}

sca_status nested_prepare(Engine& e) {
  e.nest = nullptr;
  if (e.L < nested::kMinL) return SCA_OK;
  nested::Tree t = nested::Builder(e.L).build(false);
  const nested::Tree td = nested::Builder(e.L).build(true);
  const size_t S = e.fp64 ? 8 : 4;
  const long long stride = std::max(t.entries, td.entries);
  const size_t per_block = 16 * (size_t)stride + sizeof(double) * t.nodes.size();
  const size_t room = e.block_room;
  const long long cap = (long long)(room / per_block);
  if (cap < e.chunk) return SCA_OK;
  Nested* ne = new (std::nothrow) Nested();
  if (!ne) { set_error("host allocation failed"); return SCA_ENOMEM; }
  e.nest = ne;
  ne->nnodes = (int)td.nodes.size();
  ne->stride = stride;
  ne->cap = (int)std::min<long long>(cap, e.B);
  for (const nested::Level& lv : t.levels) {
    LevelPlan p{lv.first, lv.count, lv.mmax >= 80 ? 256 : lv.mmax >= 40 ? 128 : 64, 0, 0};
    for (int k = lv.first; k < lv.first + lv.count; ++k)
      for (const nested::Tree* f : {(const nested::Tree*)&t, &td}) {
        p.smem_up = std::max(p.smem_up, up_smem(f->nodes[k]));
        p.smem_down = std::max(p.smem_down, down_smem(f->nodes[k]));
      }
    ne->levels.push_back(p);
  }
  // both forms in one table: the second's offsets follow the first's entries
  const int toff = (int)t.table.size();
  t.table.insert(t.table.end(), td.table.begin(), td.table.end());
  for (nested::Node n : td.nodes) {
    for (int* o : {&n.sites, &n.cmap[0], &n.cmap[1], &n.pmap, &n.bsite, &n.bnbr, &n.adj}) *o += toff;
    t.nodes.push_back(n);
  }
  cudaError_t err = cudaMalloc((void**)&ne->d_nodes, sizeof(Node) * t.nodes.size());
  if (err == cudaSuccess) err = cudaMalloc((void**)&ne->d_tab, sizeof(int16_t) * t.table.size());
  if (err != cudaSuccess) {
    nested_release(e);
    (void)cudaGetLastError();
    set_error("cudaMalloc failed for the elimination tree");
    return SCA_ENOMEM;
  }
  err = cudaMemcpy(ne->d_nodes, t.nodes.data(), sizeof(Node) * t.nodes.size(), cudaMemcpyHostToDevice);
  if (err == cudaSuccess)
    err = cudaMemcpy(ne->d_tab, t.table.data(), sizeof(int16_t) * t.table.size(), cudaMemcpyHostToDevice);
  if (err != cudaSuccess) { nested_release(e); return cuda_fail(err, "elimination tree upload"); }
  return SCA_OK;
}

void nested_release(Engine& e) {
  if (!e.nest) return;
  if (e.nest->d_nodes) cudaFree(e.nest->d_nodes);
  if (e.nest->d_tab) cudaFree(e.nest->d_tab);
  delete e.nest;
  e.nest = nullptr;
}

sca_status run_nested(Engine& e, const Lattice& la, bool up, bool down, cudaStream_t s) {
  if (up) {
    const cudaError_t err = cudaMemsetAsync(e.flags, 0, sizeof(int), s);
    if (err != cudaSuccess) return cuda_fail(err, "flags reset");
  }
  return e.fp64 ? run_nested_t<Zd>(e, la, up, down, s) : run_nested_t<Zf>(e, la, up, down, s);
}

}  // namespace sca
