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
// pivot is at least Im z in modulus.  Rounding errors grow by powers of |t| / Im z on weak fields,
// which is why blocks of small Im z take wider arithmetic (nested_wide) and callers with Im z below
// kNestedMinImag |t| the pivoted dense elimination (nested_rule).
//
// Arithmetic: float64, or on the reduced-precision paths double-float (an unevaluated sum of two
// float32, 48 bits): products exact by FMA, sums by two-sums, 12 float32 operations per real
// multiply-add, two of them per instruction (real and imaginary part side by side: 20x20 with 512
// blocks 1150 to 1080 us per gradient, 40x40 with 256 3794 to 3490, 64x64 with 128 8281 to 7360).
// This GPU does 64 float32 FMAs in the time of one float64 FMA, so double-float is 5 times as
// fast as float64 and keeps 24 bits more than the float32 blocks of the dense paths.  The few
// blocks of small Im z: sums of three float32 (72 bits, 46 operations per real multiply-add, which
// takes no longer than one of float64 does here: a 20x20 float64 density of states 1013 us in
// float64, 1004 in these, 11324 in double-double).  They go beside the others, on a stream of their
// own, in clusters of up to eight CTAs per block: a 20x20 gradient, T = 0.05, 124 blocks in float64
// and 4 in these, 1009 us, 1004 with all 128 in float64; 512 blocks, T = 0.1, 2 of them in these, 2273 / 2264
// (2296 with clusters of eight where the others take longer than one block's time per SM).
// On small lattices their dependent chain shows: 8x8 densities of states 287 us, 151 in float64.
//
// Work split: a group of threads per front (a warp for the smallest, 256 or 512 threads for the
// largest), fronts in global memory (a block's take 3.2 MB at N = 1600), the current panel of at
// most 20 pivot rows and its X in shared memory.  Up to one block per SM the whole elimination is
// one launch, a CTA of 512 threads per block or a cluster of them, with a barrier per tree level;
// more blocks take one launch per level and direction, spread over the chip, in parts side by side:
// the blocks with dense leaves, and two halves of the others.  Microseconds per gradient, one launch
// against one per level: 16x16 with 64 blocks 176 / 254, 24x24 with 128 578 / 687, 32x32 with 128
// 1100 / 1217, 64x64 with 128 7850 / 8281; 20x20 with 512 blocks 1313 / 1150, float64 2892 / 2429,
// 40x40 with 256 5766 / 3570 (all before the packed instructions, which took 4 to 11 % off, and
// the halves; with both, dealing 128 blocks out by level still loses: 64x64 7333 / 7595, 32x32
// 1086 / 1108, 20x20 density of states 461 / 521).  An entry's arithmetic is the same in every
// split: results do not depend on it.
//
// What bounds it: float64, the float64 pipe (80 % active at 20x20: 2.1 times the instructions that
// the products alone need, for lanes that idle at the edges of small fronts); double-float, the
// float32 pipe, busy half of the time (1.9 instructions issued per cycle, most of them packed, which
// hold the pipe for two), the latency of reads of the parents' fronts (30 % of the downward
// products at 64x64), and the dependent chain of a panel's pivots, some 1800 cycles per pivot,
// which other fronts' products overlap only in part.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <type_traits>
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
struct alignas(16) Zf {  // re = rh + rl, im = ih + il: two pairs for the packed instructions
  float rh, ih, rl, il;
};
struct Zt {  // sums of three float32 each, 72 bits, as pairs (re, im)
  unsigned long long h, m, l;
};
struct alignas(16) Zw {  // as Zf, of two float64 each: 106 bits
  double rh, ih, rl, il;
};

// Running sums of products a b: float64, or float32 sums s with the sums c of their rounding
// errors, two to a register pair.  Af holds (re, im); Aw holds (a.re, a.im) b.re in (s1, c1) and
// (a.re, a.im) b.im in (s2, c2), so that a is used as it is loaded and only b, which the rows of a
// thread share, is spread over pairs: for the long sums, as its result takes more to put together.
struct Ad {
  double re, im;
};
using f2 = unsigned long long;  // two float32 in a register pair
struct Af {
  f2 s, c;
};
struct Aw {
  f2 s1, c1, s2, c2;
};
struct At {  // sums, their rounding errors', and those sums' own
  f2 s, c, d;
};
struct Aq {  // sums and the sums of their rounding errors, float64
  double rs, rc, is, ic;
};
__device__ __forceinline__ f2 f2_of(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_get(f2 a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
template <typename Z>
struct AccOf;
template <>
struct AccOf<Zd> {
  using type = Ad;
  using wide = Ad;
};
template <>
struct AccOf<Zf> {
  using type = Af;
  using wide = Aw;
};
template <>
struct AccOf<Zt> {
  using type = At;
  using wide = At;
};
template <>
struct AccOf<Zw> {
  using type = Aq;
  using wide = Aq;
};

__device__ __forceinline__ void zset(Zd& z, double re, double im) { z = {re, im}; }
__device__ __forceinline__ void zset(Zf& z, double re, double im) {
  const dsf a = ds_of(re), b = ds_of(im);
  z = {a.h, b.h, a.l, b.l};
}
__device__ __forceinline__ void zset(Zt& z, double re, double im) {
  const dsf a = ds_of(re), b = ds_of(im);
  z.h = f2_of(a.h, b.h);
  z.m = f2_of(a.l, b.l);
  z.l = f2_of((float)((re - a.h) - a.l), (float)((im - b.h) - b.l));
}
__device__ __forceinline__ void zset0(Zt& z) { z = {0, 0, 0}; }
__device__ __forceinline__ double zre(Zt z) {
  float h, m, l, u;
  f2_get(z.h, h, u);
  f2_get(z.m, m, u);
  f2_get(z.l, l, u);
  return ((double)h + (double)m) + (double)l;
}
__device__ __forceinline__ double zim(Zt z) {
  float h, m, l, u;
  f2_get(z.h, u, h);
  f2_get(z.m, u, m);
  f2_get(z.l, u, l);
  return ((double)h + (double)m) + (double)l;
}
__device__ __forceinline__ Zt zneg(Zt z) {
  constexpr unsigned long long sign = 0x8000000080000000ull;
  return {z.h ^ sign, z.m ^ sign, z.l ^ sign};
}
__device__ __forceinline__ void zset(Zw& z, double re, double im) { z = {re, im, 0.0, 0.0}; }
__device__ __forceinline__ void zset0(Zw& z) { z = {0.0, 0.0, 0.0, 0.0}; }
__device__ __forceinline__ void zset0(Zd& z) { z = {0.0, 0.0}; }
__device__ __forceinline__ void zset0(Zf& z) { z = {0.f, 0.f, 0.f, 0.f}; }
__device__ __forceinline__ double zre(Zd z) { return z.re; }
__device__ __forceinline__ double zim(Zd z) { return z.im; }
__device__ __forceinline__ double zre(Zf z) { return (double)z.rh + (double)z.rl; }
__device__ __forceinline__ double zim(Zf z) { return (double)z.ih + (double)z.il; }
__device__ __forceinline__ double zre(Zw z) { return z.rh + z.rl; }
__device__ __forceinline__ double zim(Zw z) { return z.ih + z.il; }
__device__ __forceinline__ Zw zneg(Zw z) { return {-z.rh, -z.ih, -z.rl, -z.il}; }
__device__ __forceinline__ Zd zneg(Zd z) { return {-z.re, -z.im}; }
__device__ __forceinline__ Zf zneg(Zf z) { return {-z.rh, -z.ih, -z.rl, -z.il}; }
__device__ __forceinline__ Zd zadd(Zd a, Zd b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Zf zadd(Zf a, Zf b) {
  const dsf r = ds_add({a.rh, a.rl}, {b.rh, b.rl}), i = ds_add({a.ih, a.il}, {b.ih, b.il});
  return {r.h, i.h, r.l, i.l};
}
// Sum s and rounding error r of a + b, of a - b.
__device__ __forceinline__ void two_sum_f2(f2 a, f2 b, f2& s, f2& r) {
  const f2 t = f2_add(a, b), z = f2_sub(t, a);
  r = f2_add(f2_sub(a, f2_sub(t, z)), f2_sub(b, z));
  s = t;
}
__device__ __forceinline__ void two_diff_f2(f2 a, f2 b, f2& s, f2& r) {
  const f2 t = f2_sub(a, b), z = f2_sub(t, a);
  r = f2_sub(f2_sub(a, f2_sub(t, z)), f2_add(b, z));
  s = t;
}
// A number of three parts from sums of falling size.
__device__ __forceinline__ Zt three(f2 s, f2 c, f2 d) {
  two_sum_f2(c, d, c, d);
  two_sum_f2(s, c, s, c);
  two_sum_f2(c, d, c, d);
  return {s, c, d};
}
__device__ __forceinline__ Zt zadd(Zt a, Zt b) {
  f2 s, c, e, u;
  two_sum_f2(a.h, b.h, s, e);
  two_sum_f2(a.m, b.m, c, u);
  f2 d = f2_add(f2_add(a.l, b.l), u);
  two_sum_f2(c, e, c, u);
  return three(s, c, f2_add(d, u));
}
// The same in float64 (the intrinsics keep the compiler from contracting).
__device__ __forceinline__ void two_sum_d(double a, double b, double& s, double& r) {
  s = __dadd_rn(a, b);
  const double z = __dadd_rn(s, -a);
  r = __dadd_rn(__dadd_rn(a, -__dadd_rn(s, -z)), __dadd_rn(b, -z));
}
__device__ __forceinline__ Zw zadd(Zw a, Zw b) {
  double rs, rr, is, ir;
  two_sum_d(a.rh, b.rh, rs, rr);
  two_sum_d(a.ih, b.ih, is, ir);
  Zw z;
  two_sum_d(rs, rr + (a.rl + b.rl), z.rh, z.rl);
  two_sum_d(is, ir + (a.il + b.il), z.ih, z.il);
  return z;
}

__device__ __forceinline__ Zd zsel(bool c, Zd a, Zd b) {
  return {c ? a.re : b.re, c ? a.im : b.im};
}
__device__ __forceinline__ Zf zsel(bool c, Zf a, Zf b) {
  return {c ? a.rh : b.rh, c ? a.ih : b.ih, c ? a.rl : b.rl, c ? a.il : b.il};
}
__device__ __forceinline__ Zt zsel(bool c, Zt a, Zt b) {
  return {c ? a.h : b.h, c ? a.m : b.m, c ? a.l : b.l};
}
__device__ __forceinline__ Zt zshfl_xor(Zt z, int off) {
  return {__shfl_xor_sync(0xffffffffu, z.h, off), __shfl_xor_sync(0xffffffffu, z.m, off),
          __shfl_xor_sync(0xffffffffu, z.l, off)};
}
__device__ __forceinline__ Zw zsel(bool c, Zw a, Zw b) {
  return {c ? a.rh : b.rh, c ? a.ih : b.ih, c ? a.rl : b.rl, c ? a.il : b.il};
}
__device__ __forceinline__ Zw zshfl_xor(Zw z, int off) {
  return {__shfl_xor_sync(0xffffffffu, z.rh, off), __shfl_xor_sync(0xffffffffu, z.ih, off),
          __shfl_xor_sync(0xffffffffu, z.rl, off), __shfl_xor_sync(0xffffffffu, z.il, off)};
}
__device__ __forceinline__ Zd zshfl_xor(Zd z, int off) {
  return {__shfl_xor_sync(0xffffffffu, z.re, off), __shfl_xor_sync(0xffffffffu, z.im, off)};
}
__device__ __forceinline__ Zf zshfl_xor(Zf z, int off) {
  return {__shfl_xor_sync(0xffffffffu, z.rh, off), __shfl_xor_sync(0xffffffffu, z.ih, off),
          __shfl_xor_sync(0xffffffffu, z.rl, off), __shfl_xor_sync(0xffffffffu, z.il, off)};
}

__device__ __forceinline__ void acc_of(Ad& a, Zd z) { a = {z.re, z.im}; }
__device__ __forceinline__ void acc_of(Af& a, Zf z) {
  a = {f2_of(z.rh, z.ih), f2_of(z.rl, z.il)};
}
__device__ __forceinline__ void acc_of(At& a, Zt z) { a = {z.h, z.m, z.l}; }
__device__ __forceinline__ Zt acc_get(At a) { return three(a.s, a.c, a.d); }
__device__ __forceinline__ void acc_of(Aq& a, Zw z) { a = {z.rh, z.rl, z.ih, z.il}; }
__device__ __forceinline__ Zw acc_get(Aq a) {
  Zw z;
  two_sum_d(a.rs, a.rc, z.rh, z.rl);
  two_sum_d(a.is, a.ic, z.ih, z.il);
  return z;
}
__device__ __forceinline__ Zd acc_get(Ad a) { return {a.re, a.im}; }
__device__ __forceinline__ Zf acc_get(Af a) {
  float rs, rc, is, ic;
  f2_get(a.s, rs, is);
  f2_get(a.c, rc, ic);
  const dsf r = two_sum(rs, rc), i = two_sum(is, ic);
  return {r.h, i.h, r.l, i.l};
}

__device__ __forceinline__ Zf acc_get(Aw a) {
  float p, q, pc, qc, u, v, uc, vc;
  f2_get(a.s1, p, q);
  f2_get(a.c1, pc, qc);
  f2_get(a.s2, u, v);
  f2_get(a.c2, uc, vc);
  dsf r = two_sum(p, -v), i = two_sum(q, u);
  r = two_sum(r.h, r.l + (pc - vc));
  i = two_sum(i.h, i.l + (qc + uc));
  return {r.h, i.h, r.l, i.l};
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
__device__ __forceinline__ void mac1(double& s, double& c, double ah, double al, double bh,
                                     double bl) {
  const double p = __dmul_rn(ah, bh);
  double e = fma(ah, bh, -p);
  e = fma(ah, bl, e);
  e = fma(al, bh, e);
  double t, r;
  two_sum_d(s, p, t, r);
  s = t;
  c = __dadd_rn(c, __dadd_rn(r, e));
}
__device__ __forceinline__ void mac(Aq& s, Zw a, Zw b) {
  mac1(s.rs, s.rc, a.rh, a.rl, b.rh, b.rl);
  mac1(s.is, s.ic, a.rh, a.rl, b.ih, b.il);
  mac1(s.rs, s.rc, -a.ih, -a.il, b.ih, b.il);
  mac1(s.is, s.ic, a.ih, a.il, b.rh, b.rl);
}
// The same for both halves of a pair, in half the instructions.  A pair cannot be negated in
// place: -p is taken apart and put together again, or, in the second form, minus b comes in.
__device__ __forceinline__ void mac2(f2& s, f2& c, f2 ah, f2 al, f2 bh, f2 bl) {
  const f2 p = f2_mul(ah, bh);
  float p0, p1;
  f2_get(p, p0, p1);
  f2 e = f2_fma(ah, bh, f2_of(-p0, -p1));
  e = f2_fma(ah, bl, e);
  e = f2_fma(al, bh, e);
  const f2 t = f2_add(s, p), z = f2_sub(t, s);
  const f2 r = f2_add(f2_sub(s, f2_sub(t, z)), f2_sub(p, z));
  s = t;
  c = f2_add(c, f2_add(r, e));
}
__device__ __forceinline__ void mac(Af& s, Zf a, Zf b) {
  mac2(s.s, s.c, f2_of(a.rh, a.rh), f2_of(a.rl, a.rl), f2_of(b.rh, b.ih), f2_of(b.rl, b.il));
  mac2(s.s, s.c, f2_of(a.ih, a.ih), f2_of(a.il, a.il), f2_of(-b.ih, b.rh), f2_of(-b.il, b.rl));
}
__device__ __forceinline__ void mac2(f2& s, f2& c, f2 ah, f2 al, f2 bh, f2 nbh, f2 nbl) {
  const f2 p = f2_mul(ah, bh);
  f2 e = f2_fma(ah, nbh, p);  // minus the rest of the product
  e = f2_fma(ah, nbl, e);
  e = f2_fma(al, nbh, e);
  const f2 t = f2_add(s, p), z = f2_sub(t, s);
  const f2 r = f2_add(f2_sub(s, f2_sub(t, z)), f2_sub(p, z));
  s = t;
  c = f2_add(c, f2_sub(r, e));
}
__device__ __forceinline__ void mac(Aw& s, Zf a, Zf b) {
  const f2 ah = f2_of(a.rh, a.ih), al = f2_of(a.rl, a.il);
  mac2(s.s1, s.c1, ah, al, f2_of(b.rh, b.rh), f2_of(-b.rh, -b.rh), f2_of(-b.rl, -b.rl));
  mac2(s.s2, s.c2, ah, al, f2_of(b.ih, b.ih), f2_of(-b.ih, -b.ih), f2_of(-b.il, -b.il));
}
// (s, c, d) += (a0 + a1 + a2)(b0 + b1 + b2), n = -b: the leading product with its error exactly, the
// two of the next order likewise, the three of the order after (and the errors of the second) to
// float32 accuracy; what is added to c keeps its errors in d.
__device__ __forceinline__ void mac3(At& s, f2 a0, f2 a1, f2 a2, f2 b0, f2 b1, f2 b2, f2 n0, f2 n1) {
  const f2 p = f2_mul(a0, b0), p1 = f2_mul(a0, b1), p2 = f2_mul(a1, b0);
  const f2 e = f2_fma(a0, n0, p), e1 = f2_fma(a0, n1, p1), e2 = f2_fma(a1, n0, p2);  // minus them
  const f2 q = f2_fma(a0, b2, f2_fma(a1, b1, f2_mul(a2, b0)));
  f2 r, u, ue, v, ve, we, r1;
  two_sum_f2(s.s, p, s.s, r);
  two_sum_f2(p1, p2, u, ue);
  two_diff_f2(r, e, v, ve);
  two_sum_f2(u, v, u, we);
  two_sum_f2(s.c, u, s.c, r1);
  s.d = f2_add(s.d, f2_add(f2_add(f2_add(ue, ve), f2_add(we, r1)), f2_sub(q, f2_add(e1, e2))));
}
__device__ __forceinline__ void mac(At& s, Zt a, Zt b) {
  float ar, ai, mr, mi, lr, li, br[3], bi[3];
  f2_get(a.h, ar, ai);
  f2_get(a.m, mr, mi);
  f2_get(a.l, lr, li);
  f2_get(b.h, br[0], bi[0]);
  f2_get(b.m, br[1], bi[1]);
  f2_get(b.l, br[2], bi[2]);
  mac3(s, f2_of(ar, ar), f2_of(mr, mr), f2_of(lr, lr), b.h, b.m, b.l, f2_of(-br[0], -bi[0]),
       f2_of(-br[1], -bi[1]));
  mac3(s, f2_of(ai, ai), f2_of(mi, mi), f2_of(li, li), f2_of(-bi[0], br[0]), f2_of(-bi[1], br[1]),
       f2_of(-bi[2], br[2]), f2_of(bi[0], -br[0]), f2_of(bi[1], -br[1]));
}
template <typename Z>
__device__ __forceinline__ Z zmul(Z a, Z b) {
  typename AccOf<Z>::type s{};
  mac(s, a, b);
  return acc_get(s);
}
// 1 / z, and |z|^2 in float64.  (Which of the two products goes into the FMA is written out: left
// to the compiler it differed between the kernels, and a result's last bit with the split.)
__device__ __forceinline__ Zd zinv(Zd z, double* mag2 = nullptr) {
  const double m = fma(z.im, z.im, __dmul_rn(z.re, z.re));
  const double d = recip(m);
  if (mag2) *mag2 = m;
  return {z.re * d, -z.im * d};
}
__device__ __forceinline__ Zf zinv(Zf z, double* mag2 = nullptr) {
  float s = 0.f, c = 0.f;
  mac1(s, c, z.rh, z.rl, z.rh, z.rl);
  mac1(s, c, z.ih, z.il, z.ih, z.il);
  const dsf d = two_sum(s, c);
  if (mag2) *mag2 = (double)d.h + (double)d.l;
  const float q = __frcp_rn(d.h);  // then one Newton step: q + q (1 - d q)
  float e = fmaf(-q, d.h, 1.0f);
  e = fmaf(-q, d.l, e);
  const float ql = __fmul_rn(q, e);
  float rs = 0.f, rc = 0.f, is = 0.f, ic = 0.f;
  mac1(rs, rc, z.rh, z.rl, q, ql);
  mac1(is, ic, -z.ih, -z.il, q, ql);
  const dsf r = two_sum(rs, rc), i = two_sum(is, ic);
  return {r.h, i.h, r.l, i.l};
}
__device__ __forceinline__ Zt zinv(Zt z, double* mag2 = nullptr) {
  At s{};
  const Zt n = zneg(z);
  mac3(s, z.h, z.m, z.l, z.h, z.m, z.l, n.h, n.m);  // re^2, im^2
  const Zt sq = acc_get(s);
  float h0, h1, m0, m1, l0, l1;
  f2_get(sq.h, h0, h1);
  f2_get(sq.m, m0, m1);
  f2_get(sq.l, l0, l1);
  dsf h = two_sum(h0, h1), m = two_sum(m0, m1);
  float l = __fadd_rn(__fadd_rn(l0, l1), m.l);
  m = two_sum(m.h, h.l);  // |z|^2 = h.h + m.h + l
  l = __fadd_rn(l, m.l);
  const dsf d = two_sum(h.h, m.h);
  const dsf d2 = two_sum(d.l, l);
  if (mag2) *mag2 = ((double)d.h + (double)d2.h) + (double)d2.l;
  // 1 / |z|^2 = q (1 + e + e^2) to e^3 < 2^-69, e = 1 - q |z|^2 to 48 bits
  const float q = __frcp_rn(d.h);
  const float e0 = fmaf(-q, d.h, 1.0f), p = __fmul_rn(q, d2.h), pe = fmaf(q, d2.h, -p);
  dsf e = two_sum(e0, -p);
  e.l = __fadd_rn(e.l, -fmaf(q, d2.l, pe));
  e = two_sum(e.h, fmaf(e.h, e.h, e.l));
  const float f = __fmul_rn(q, e.h), fe = fmaf(q, e.l, fmaf(q, e.h, -f));
  const dsf i0 = two_sum(q, f);
  const dsf i1 = two_sum(i0.l, fe);
  const f2 qh = f2_of(i0.h, i0.h), qm = f2_of(i1.h, i1.h), ql = f2_of(i1.l, i1.l);
  float zr[3], zi[3];
  f2_get(z.h, zr[0], zi[0]);
  f2_get(z.m, zr[1], zi[1]);
  f2_get(z.l, zr[2], zi[2]);
  At r{};
  mac3(r, qh, qm, ql, f2_of(zr[0], -zi[0]), f2_of(zr[1], -zi[1]), f2_of(zr[2], -zi[2]),
       f2_of(-zr[0], zi[0]), f2_of(-zr[1], zi[1]));
  return acc_get(r);
}
__device__ __forceinline__ Zw zinv(Zw z, double* mag2 = nullptr) {
  double s = 0.0, c = 0.0;
  mac1(s, c, z.rh, z.rl, z.rh, z.rl);
  mac1(s, c, z.ih, z.il, z.ih, z.il);
  double d, dl;
  two_sum_d(s, c, d, dl);
  if (mag2) *mag2 = d;
  const double q = recip(d);  // then one Newton step: q + q (1 - d q)
  double e = fma(-q, d, 1.0);
  e = fma(-q, dl, e);
  const double ql = __dmul_rn(q, e);
  double rs = 0.0, rc = 0.0, is = 0.0, ic = 0.0;
  mac1(rs, rc, z.rh, z.rl, q, ql);
  mac1(is, ic, -z.ih, -z.il, q, ql);
  Zw r;
  two_sum_d(rs, rc, r.rh, r.rl);
  two_sum_d(is, ic, r.ih, r.il);
  return r;
}

// The float32 forms square numbers within float32's range, so site terms of 2^60 and more come in as
// 2^60: what such a site couples with changes by 2^-60 t^2 or less, and its own G_ii, 1 / a, is as
// far below rounding either way.  Its share of |det A|^2 is put right where it is read: `far`.
// (No pivot is too small: each is at least Im z >= 1e-9 in modulus.)
template <typename Z>
constexpr bool kNarrow = std::is_same<Z, Zf>::value || std::is_same<Z, Zt>::value;
__device__ __forceinline__ bool beyond(double x) {  // |x| >= 2^60 or not finite, off the slow pipe
  return (__double2hiint(x) & 0x7fffffff) >= 0x43b00000;
}
__device__ __forceinline__ bool beyond(Zf z) { return fabsf(z.rh) >= 0x1p60f; }
__device__ __forceinline__ bool beyond(Zt z) {
  float r, i;
  f2_get(z.h, r, i);
  return fabsf(r) >= 0x1p60f;
}
__device__ __forceinline__ bool beyond(Zd) { return false; }
__device__ __forceinline__ bool beyond(Zw) { return false; }
template <typename Z>
__device__ __forceinline__ double near_term(double re) {
  return kNarrow<Z> && beyond(re) ? copysign(0x1p60, re) : re;
}
// (|a| / 2^60)^2 of a site term beyond 2^60, not finite where it is not.
__device__ __forceinline__ double far(double re) { return (re * 0x1p-60) * (re * 0x1p-60); }

// A product of moduli squared as mantissa in [1, 2) and exponent: a node's share of |det A|^2.
// One logarithm per node at the root instead of one per pivot (a float64 logarithm costs about
// 40 instructions of the slowest pipe of this GPU).
struct alignas(16) Det {
  double mant;
  int exp, pad;
};
// Product over the warp's lanes of m2 (1.0 where a lane has none), in a fixed order, times
// (mant, exp); flags non-positive or non-finite moduli.
__device__ __forceinline__ void det_mul(double m2, double& mant, int& exp, int* flags) {
  if (!(m2 > 0.0 && isfinite(m2))) {
    atomicOr(flags, 1);
    m2 = 1.0;
  }
  int e = 0;
  det_norm(m2, e);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    m2 *= __shfl_xor_sync(0xffffffffu, m2, off);
    e += __shfl_xor_sync(0xffffffffu, e, off);
  }
  mant *= m2;
  exp += e;
  det_norm(mant, exp);
}

// ------------------------------------------------------------------ kernels
constexpr int kRows = nested::kRows;    // rows of a thread's output tile at most
constexpr int kSlots = nested::kSlots;  // entries of a pivots' block that a thread holds at most

// Blocks from which a launch per level takes them in two halves on two streams (20x20 with 500
// such blocks 1072 / 1000 us per gradient in one part / in halves, float64 2413 / 2249, 40x40 with
// 244 3478 / 3185, its potential 1628 / 1555).  A pass with a launch per level has more blocks
// than SMs, so the line only keeps a small rest beside blocks with dense leaves in one piece.
constexpr int kHalves = 64;

// How one level's fronts are worked on: `group` threads per front, each group with `smem` bytes.
struct LevelPlan {
  int first, count, group, smem;
};

template <typename Z>
struct NestArgs {
  const Node* nodes;     // the two forms of the tree, nnodes each: closed-form, dense leaves
  const int16_t* tab;
  Z* fronts;             // fronts of the pass's blocks, `stride` entries apart
  long long stride;
  Det* det;              // [block of the pass][node]: the node's share of |det A|^2
  int nnodes, nlevels;
  int b0;                // block of the pass's first slot
  int csize;             // CTAs per block
  int ndense;            // leading slots of the pass that take the dense leaves
  int range;             // 1: not blocks whose entries leave float32's range; 2: those alone
  int k0, k1;            // phases: [0, nlevels) up from the leaves, [nlevels, 2 nlevels) down
  Lattice la;
  double* ld;            // ln|det A_b|
  double* gd;            // [b][site]: sigma Re G_ii (or Im G_ii where zshift is set)
  int* flags;
  LevelPlan lv[2][nested::kMaxLevels];  // by form; root first
};

// Whether two sites, packed as 256 x + y, are neighbours.
__device__ __forceinline__ bool adjacent(int L, int a, int b) {
  const int dx = abs((a >> 8) - (b >> 8)), dy = abs((a & 255) - (b & 255));
  return (dx == 0 && (dy == 1 || dy == L - 1)) || (dy == 0 && (dx == 1 || dx == L - 1));
}

// Entry (hi, lo) of a front before its own elimination, hi >= lo: A's entry where lo is a pivot
// (entries between boundary sites belong to an ancestor), the children's Schur complements, and
// in a leaf the closed-form elimination of the blacks next to both sites (bt = -t^2 / a_b).
template <typename Z>
struct Front {
  int L;
  const Z* c[2];        // children's Schur complements (their boundary parts), row stride cm
  int cm[2];
  int p, leaf;
  int site, cmap0, cmap1, adj;  // shared-memory offsets of the index maps,
  int bt, diag;                 // of the blacks' terms, of A_ii of the pivots followed by t
  __device__ __forceinline__ Z at(int hi, int lo) const {
    extern __shared__ __align__(16) unsigned char smem[];
    auto tab = [&](int o, int i) { return (int)reinterpret_cast<const int16_t*>(smem + o)[i]; };
    Z v;
    zset0(v);
    if (leaf) {
      for (int both = tab(adj, hi) & tab(adj, lo); both; both &= both - 1)
        v = zadd(v, reinterpret_cast<const Z*>(smem + bt)[__ffs(both) - 1]);
    } else if (c[0]) {  // (a node with children has two)
      const int i = tab(cmap0, hi), j = tab(cmap0, lo), k = tab(cmap1, hi), l = tab(cmap1, lo);
      Z x;
      zset0(x);
      const Z *c0 = c[0], *c1 = c[1];
      __builtin_assume(__isGlobal(c0));
      __builtin_assume(__isGlobal(c1));
      if (i >= 0 && j >= 0) v = c0[i * cm[0] + j];
      if (k >= 0 && l >= 0) x = c1[k * cm[1] + l];
      v = zadd(v, x);
    }
    if (lo < p) {
      if (hi == lo)
        v = zadd(v, reinterpret_cast<const Z*>(smem + diag)[lo]);
      else if (adjacent(L, tab(site, hi), tab(site, lo)))
        v = zadd(v, reinterpret_cast<const Z*>(smem + diag)[p]);
    }
    return v;
  }
};

// Row and column of entry e of a lower triangle stored row after row.
__device__ __forceinline__ void triangle(int e, int& i, int& j) {
  i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  if ((i + 1) * (i + 2) / 2 <= e) ++i;
  if (i * (i + 1) / 2 > e) --i;
  j = e - i * (i + 1) / 2;
}

// Block of KR rows and column of task e where row block b has KR (b + 1) columns.
template <int KR>
__device__ __forceinline__ void row_block(int e, int& b, int& j) {
  b = (int)((sqrtf((8.0f / KR) * (float)e + 1.0f) - 1.0f) * 0.5f);
  if (KR * (b + 1) * (b + 2) / 2 <= e) ++b;
  if (KR * b * (b + 1) / 2 > e) --b;
  j = e - KR * b * (b + 1) / 2;
}

// The threads that work on one front: `size` of them (a power of two, a whole warp at least) with
// a barrier of their own.
struct Group {
  int size, tid, bar;
  __device__ __forceinline__ void sync() const {
    if (size == 32)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(size) : "memory");
  }
};

// Offset of a pointer into the CTA's dynamic shared memory.
__device__ __forceinline__ int off(const void* p) {
  extern __shared__ __align__(16) unsigned char smem[];
  return (int)(static_cast<const unsigned char*>(p) - smem);
}

// What the fronts of one block share.
template <typename Z>
struct Block {
  const Node* nodes;
  const int16_t* tab;
  Z* fronts;
  Det* det;
  double* gd;
  int* flags;
  Lattice la;
  double zr, zi;
  int sg;
};

// The functions below are calls of their own, with offsets into shared memory instead of pointers:
// inlined into one kernel their registers add up (as calls, the forms of 128 registers spill 72
// bytes or less in float64 and double-float, those of 64 registers up to 296), and through a call a
// pointer would lose its address space.
// Their inner loops have no branch per row, which would split them into blocks of two dependent
// chains each; rows past the end repeat the last one and are dropped.

// -F11^{-1} by w Gauss-Jordan steps, diagonal pivots in order: thread (g, j) holds the entries
// (g, j), (g + G, j), ... of the w x w block, S of them, G = size / w.  A step needs the pivot's
// row, its column and its reciprocal; their owners write them to shared memory as soon as they
// have them (two buffers, one barrier per step).  The result replaces F11, negated, and goes to
// the front.
template <typename Z, int S>
__device__ __noinline__ void invert(const Group gr, int w, int F11o, int rowo, int colo,
                                    int mago, Z* Fo, int m) {
  using Acc = typename AccOf<Z>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  Z* F11 = reinterpret_cast<Z*>(smem + F11o);
  Z* rowb = reinterpret_cast<Z*>(smem + rowo);
  Z* colb = reinterpret_cast<Z*>(smem + colo);
  double* mag = reinterpret_cast<double*>(smem + mago);
  __builtin_assume(__isGlobal(Fo));
  const int G = min(w, gr.size / w), g = gr.tid / w, j = gr.tid - g * w;
  const bool on = g < G;
  Z reg[S];
  int row[S];
#pragma unroll
  for (int s = 0; s < S; ++s) row[s] = min(g + s * G, w - 1);
  if (on) {
#pragma unroll
    for (int s = 0; s < S; ++s) reg[s] = F11[row[s] * w + j];
    if (g == 0) rowb[j] = reg[0];
    if (j == 0) {
#pragma unroll
      for (int s = 0; s < S; ++s) colb[row[s]] = zneg(reg[s]);
    }
    if (gr.tid == 0) colb[w] = zinv(reg[0], mag);
  }
#pragma unroll 1
  for (int c = 0; c < w; ++c) {
    gr.sync();
    const Z* rb = rowb + (c & 1) * w;
    const Z* cb = colb + (c & 1) * (w + 1);
    Z* rn = rowb + ((c + 1) & 1) * w;
    Z* cn = colb + ((c + 1) & 1) * (w + 1);
    if (on) {
      const bool own = j == c;
      const Z dinv = cb[w];
      const Z u = zsel(own, dinv, zmul(rb[j], dinv));
      Z zero;
      zset0(zero);
#pragma unroll
      for (int s = 0; s < S; ++s) {
        Acc x;
        acc_of(x, zsel(own, zero, reg[s]));
        mac(x, cb[row[s]], u);
        reg[s] = zsel(row[s] == c, u, acc_get(x));
      }
      if (c + 1 < w && g == (c + 1) % G) {  // the next pivot's row
        Z nr = reg[0];
#pragma unroll
        for (int s = 1; s < S; ++s) nr = zsel(row[s] == c + 1, reg[s], nr);
        rn[j] = nr;
        if (j == c + 1) cn[w] = zinv(nr, mag + j);
      }
      if (j == c + 1) {
#pragma unroll
        for (int s = 0; s < S; ++s) cn[row[s]] = zneg(reg[s]);
      }
    }
  }
  if (on) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      F11[row[s] * w + j] = zneg(reg[s]);
      Fo[(size_t)row[s] * m + j] = reg[s];
    }
  }
}

// Lower triangle of the rest, F22 - F12^T X: each thread one column and KR rows.  Neighbouring lanes
// take neighbouring columns, so the front's rows, X and the children's rows are read and written
// along them, and F12 is broadcast.
template <typename Z, int KR>
__device__ __noinline__ void update_rest(const Group gr, const Front<Z>& f, bool first, int at0,
                                            int w, int r, int m, int Ao, int lda, int Xo, Z* R) {
  using Acc = typename AccOf<Z>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  const Z* A = reinterpret_cast<const Z*>(smem + Ao);
  const Z* X = reinterpret_cast<const Z*>(smem + Xo);
  __builtin_assume(__isGlobal(R));
  const int nb = (r + KR - 1) / KR, tasks = KR * nb * (nb + 1) / 2;
  for (int e = gr.tid; e < tasks; e += gr.size) {
    int b, j;
    row_block<KR>(e, b, j);
    if (j >= r) continue;
    const int i0 = b * KR;
    Acc s[KR];
#pragma unroll
    for (int u = 0; u < KR; ++u) s[u] = Acc{};
    const Z *Ai = A + i0, *Xj = X + j;
#pragma unroll 2
    for (int k = 0; k < w; ++k) {
      const Z x = *Xj;
#pragma unroll
      for (int u = 0; u < KR; ++u) mac(s[u], Ai[u], x);
      Ai += lda;
      Xj += r;
    }
    Z v[KR];
    if (!first) {
#pragma unroll
      for (int u = 0; u < KR; ++u) v[u] = R[max(j, min(i0 + u, r - 1)) * m + j];
    } else {
#pragma unroll
      for (int u = 0; u < KR; ++u) v[u] = f.at(at0 + max(j, min(i0 + u, r - 1)), at0 + j);
    }
#pragma unroll
    for (int u = 0; u < KR; ++u) {
      const int i = i0 + u;
      if (i < r && j <= i) R[i * m + j] = zadd(v[u], acc_get(s[u]));
    }
  }
}

// Y = X R (w x r, inner length n): one column and KR rows per thread, the rows nrb apart, X (row
// stride ldx) broadcast from shared memory, R (row stride step) from shared or global memory (L1
// and L2 hold it).  kAhead > 0: R is Rg, in global memory, read kAhead rows ahead; else at Ro, and
// the rows of Y go to Yg (row stride m) too.  Four rows ahead where a CTA of 512 threads has the SM
// to itself (64x64: 7.6 ms with two, 7.3 with four, 7.2 with six, which costs 12x12 and densities
// of states 1.5 %), two where four CTAs of 256 share it (64 registers; three cost 2 %).  kMap: R's
// rows and columns go through map (R in the parent's front).
template <typename Z, int KR, bool kMap, int kAhead>
__device__ __noinline__ void times(const Group gr, int w, int n, int r, int Xo, int ldx, int Yo,
                                   int ldy, const Z* Rg, int Ro, int step, int mapo, Z* Yg, int m) {
  constexpr bool kGlobal = kAhead > 0;
  using Acc = std::conditional_t<(kAhead > 0), typename AccOf<Z>::wide, typename AccOf<Z>::type>;
  extern __shared__ __align__(16) unsigned char smem[];
  const Z* X = reinterpret_cast<const Z*>(smem + Xo);
  Z* Y = reinterpret_cast<Z*>(smem + Yo);
  const Z* Rs = reinterpret_cast<const Z*>(smem + Ro);
  const int16_t* map = reinterpret_cast<const int16_t*>(smem + mapo);
  __builtin_assume(__isGlobal(Rg));
  const int nrb = (w + KR - 1) / KR;
  for (int e = gr.tid; e < nrb * r; e += gr.size) {
    const int b = e / r, j = e - b * r;
    Acc s[KR];
    int Xi[KR];
#pragma unroll
    for (int u = 0; u < KR; ++u) {
      s[u] = Acc{};
      Xi[u] = min(b + u * nrb, w - 1) * ldx;
    }
    const int jj = kMap ? map[j] : j;
    if constexpr (kGlobal) {
      auto load = [&](int k) {
        k = min(k, n - 1);
        return Rg[(kMap ? map[k] : k) * step + jj];
      };
      Z g[kAhead];
#pragma unroll
      for (int d = 0; d < kAhead; ++d) g[d] = load(d);
      int k = 0;
#pragma unroll 1
      for (; k + kAhead <= n; k += kAhead) {
#pragma unroll
        for (int d = 0; d < kAhead; ++d) {
          const Z x = g[d];
          g[d] = load(k + kAhead + d);
#pragma unroll
          for (int u = 0; u < KR; ++u) mac(s[u], X[Xi[u] + k + d], x);
        }
      }
#pragma unroll
      for (int d = 0; d + 1 < kAhead; ++d)
        if (k + d < n) {
#pragma unroll
          for (int u = 0; u < KR; ++u) mac(s[u], X[Xi[u] + k + d], g[d]);
        }
    } else {
#pragma unroll 2
      for (int k = 0; k < n; ++k) {
        const Z g = Rs[k * step + jj];
#pragma unroll
        for (int u = 0; u < KR; ++u) mac(s[u], X[Xi[u] + k], g);
      }
    }
#pragma unroll
    for (int u = 0; u < KR; ++u) {
      const int i = b + u * nrb;
      if (i < w) {
        const Z v = acc_get(s[u]);
        Y[i * ldy + j] = v;
        if (!kGlobal) Yg[i * m + j] = v;
      }
    }
  }
}

// The row count that fits the outputs per thread: passes over the threads, each of KR products and
// about a third of a product's overhead.
template <typename Z, bool kMap, int kAhead>
__device__ __forceinline__ void times_fit(const Group& gr, int w, int n, int r, int Xo, int ldx,
                                          int Yo, int ldy, const Z* Rg, int Ro, int step, int mapo,
                                          Z* Yg, int m) {
  auto cost = [&](int kr) {
    return ((w + kr - 1) / kr * r + gr.size - 1) / gr.size * (3 * kr + 1);
  };
  if (cost(2) <= cost(1) || kMap)
    times<Z, 2, kMap, kAhead>(gr, w, n, r, Xo, ldx, Yo, ldy, Rg, Ro, step, mapo, Yg, m);
  else
    times<Z, 1, kMap, kAhead>(gr, w, n, r, Xo, ldx, Yo, ldy, Rg, Ro, step, mapo, Yg, m);
}

// One front, up: see the file comment.  -X is kept (in the front and here), as both later products
// want it with that sign.  Shared memory: F12 and -X (w x r each), F11 (then -P), the inversion's
// buffers, the leaf's blacks, the pivots' diagonal, index maps.
template <typename Z>
__device__ __forceinline__ void front_up(const Block<Z>& B, int node, const Group& gr, int at) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Acc = typename AccOf<Z>::type;
  const int tid = gr.tid, size = gr.size;
  const Node nd = B.nodes[node];
  const int p = nd.p, m = nd.p + nd.q, pw = nd.pw;
  Z* F = B.fronts + nd.front;
  Z* A = reinterpret_cast<Z*>(smem + at);
  Z* X = A + pw * (m - pw + kRows);
  Z* F11 = X + pw * (m - pw);
  Z* rowb = F11 + pw * pw;        // [2][pw]: the pivot's row
  Z* colb = rowb + 2 * pw;        // [2][pw + 1]: minus its column, then the reciprocal
  Z* bt = colb + 2 * (pw + 1);
  Z* diag = bt + nd.blacks;
  double* mag = reinterpret_cast<double*>(diag + p + 1);
  int16_t* site = reinterpret_cast<int16_t*>(mag + 32);
  int16_t* cm0 = site + m;
  int16_t* cm1 = cm0 + m;
  int16_t* adj = cm1 + m;
  double mant = 1.0;  // first warp: the node's share of |det A|^2
  int expo = 0;
  for (int i = tid; i < m; i += size) {
    const int s = B.tab[nd.sites + i], x = s / B.la.L;
    site[i] = (int16_t)((x << 8) | (s - x * B.la.L));
    cm0[i] = nd.child[0] >= 0 ? B.tab[nd.cmap[0] + i] : (int16_t)-1;
    cm1[i] = nd.child[1] >= 0 ? B.tab[nd.cmap[1] + i] : (int16_t)-1;
  }
  for (int i = tid; i <= p; i += size)
    zset(diag[i],
         i < p ? near_term<Z>(B.zr - site_energy(B.la, B.tab[nd.sites + i], B.sg)) : B.la.t,
         i < p ? B.zi : 0.0);
  if (nd.blacks) {
    for (int i = tid; i < m; i += size) adj[i] = B.tab[nd.adj + i];
    if (tid < 32) {
      double m2 = 1.0;
      if (tid < nd.blacks) {
        Z z, t2;
        const double re = B.zr - site_energy(B.la, B.tab[nd.bsite + tid], B.sg);
        zset(z, near_term<Z>(re), B.zi);
        zset(t2, B.la.t * B.la.t, 0.0);
        bt[tid] = zneg(zmul(t2, zinv(z, &m2)));
        if (kNarrow<Z> && beyond(re)) m2 *= far(re);
      }
      det_mul(m2, mant, expo, B.flags);
    }
  }
  Front<Z> f;
  f.L = B.la.L;
  for (int c = 0; c < 2; ++c) {
    f.c[c] = nullptr;
    f.cm[c] = 0;
    if (nd.child[c] >= 0) {
      const Node k = B.nodes[nd.child[c]];
      const int mc = k.p + k.q;
      f.c[c] = B.fronts + k.front + (size_t)k.p * mc + k.p;
      f.cm[c] = mc;
    }
  }
  f.p = p;
  f.leaf = nd.blacks > 0;
  f.site = off(site);
  f.cmap0 = off(cm0);
  f.cmap1 = off(cm1);
  f.adj = off(adj);
  f.bt = off(bt);
  f.diag = off(diag);
  gr.sync();
  for (int pa = 0; pa < nd.npan; ++pa) {
    const int o = pa * pw, w = min(pw, p - o), l = m - o, r = l - w;
    const int lda = r + kRows;  // row blocks read up to kRows - 1 entries past r
    // ---- the panel to shared memory (F12 stays there), then to the registers
    for (int i = tid >> 5; i < w; i += size >> 5)
#pragma unroll 2
      for (int j = tid & 31; j < l; j += 32) {
        const int hi = max(i, j) + o, lo = min(i, j) + o;
        const Z v = pa == 0 ? f.at(hi, lo) : F[hi * m + lo];
        if (j < w)
          F11[i * w + j] = v;
        else
          A[i * lda + j - w] = v;
      }
    gr.sync();
    Z* Fo = F + (size_t)o * (m + 1);
    if (w <= size / w)
      invert<Z, 1>(gr, w, off(F11), off(rowb), off(colb), off(mag), Fo, m);
    else
      invert<Z, kSlots>(gr, w, off(F11), off(rowb), off(colb), off(mag), Fo, m);
    gr.sync();
    if (r > 0)
      times_fit<Z, false, 0>(gr, w, w, r, off(F11), w, off(X), r, (const Z*)F, off(A), lda, 0,
                                 Fo + w, m);
    gr.sync();
    if (tid < 32) {
      double m2 = tid < w ? mag[tid] : 1.0;
      if (kNarrow<Z> && tid < w && beyond(diag[o + tid]))
        m2 *= far(B.zr - site_energy(B.la, B.tab[nd.sites + o + tid], B.sg));
      det_mul(m2, mant, expo, B.flags);
    }
    // ---- the rest; fewer rows per thread where more would leave threads idle
    Z* R = F + (size_t)(o + w) * (m + 1);
    auto cost = [&](int kr) {
      const int nb = (r + kr - 1) / kr;
      return (kr * nb * (nb + 1) / 2 + size - 1) / size * (3 * kr + 1);
    };
    if (cost(2) <= cost(1))
      update_rest<Z, 2>(gr, f, pa == 0, o + w, w, r, m, off(A), lda, off(X), R);
    else
      update_rest<Z, 1>(gr, f, pa == 0, o + w, w, r, m, off(A), lda, off(X), R);
    gr.sync();
  }
  if (tid == 0) B.det[node] = {mant, expo, 0};
}

// One front, down.  Panels in reverse; R is the part of the front after the panel, already G.  A
// node without children keeps nothing but its own rows: R is then read from the parent's front.
template <typename Z, int NT>
__device__ __forceinline__ void front_down(const Block<Z>& B, int node, const Group& gr, int at) {
  extern __shared__ __align__(16) unsigned char smem[];
  using Acc = typename AccOf<Z>::type;
  const int tid = gr.tid, size = gr.size;
  const Node nd = B.nodes[node];
  const int p = nd.p, q = nd.q, m = nd.p + nd.q;
  Z* F = B.fronts + nd.front;
  const int ldx = (m - nd.pw) | 1;  // odd: rows of 16-byte entries start in different banks
  Z* X = reinterpret_cast<Z*>(smem + at);
  Z* Y = X + nd.pw * ldx;
  Z* P = Y + nd.pw * ldx;
  int16_t* map = reinterpret_cast<int16_t*>(P + nd.pw * nd.pw);
  const bool direct = nd.child[0] < 0 && nd.npan <= 1 && nd.parent >= 0;
  const Z* G = nullptr;  // the parent's front
  int mp = 0;
  if (nd.parent >= 0) {
    const Node pr = B.nodes[nd.parent];
    mp = pr.p + pr.q;
    G = B.fronts + pr.front;
    for (int i = tid; i < q; i += size) map[i] = B.tab[nd.pmap + i];
    gr.sync();
    if (!direct) {
      // G_bb into the front, several entries in flight per thread
      for (int i = tid >> 5; i < q; i += size >> 5) {
        const Z* Gi = G + map[i] * mp;
        Z* Fi = F + (p + i) * m + p;
        for (int j0 = tid & 31; j0 < q; j0 += 128) {
          Z v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = Gi[map[min(j0 + 32 * u, q - 1)]];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (j0 + 32 * u < q) Fi[j0 + 32 * u] = v[u];
        }
      }
      gr.sync();
    }
  }
  for (int pa = nd.npan - 1; pa >= 0; --pa) {
    const int o = pa * nd.pw, w = min(nd.pw, p - o), r = m - o - w;
    const Z* R = F + (size_t)(o + w) * (m + 1);
    for (int i = tid >> 5; i < w; i += size >> 5)
      for (int j = tid & 31; j < r; j += 32) X[i * ldx + j] = F[(o + i) * m + o + w + j];
    gr.sync();
    if (direct)
      times_fit<Z, true, NT == 512 ? 4 : 2>(gr, w, r, r, off(X), ldx, off(Y), ldx, G, 0, mp,
                                            off(map), (Z*)nullptr, 0);
    else if (r > 0)
      times_fit<Z, false, NT == 512 ? 4 : 2>(gr, w, r, r, off(X), ldx, off(Y), ldx, R, 0, m, 0,
                                             (Z*)nullptr, 0);
    gr.sync();
    // ---- G_pp = P + Y (-X)^T, lower triangle; ks threads share an entry's sum (by the front's
    // shape alone: the order of a sum must not depend on how many threads there are)
    const int outs = w * (w + 1) / 2, ks = r >= 48 ? 4 : 2;
    for (int e0 = 0; e0 < outs; e0 += size / ks) {
      const int e = min(e0 + tid / ks, outs - 1), k0 = tid % ks;
      int i, j;
      triangle(e, i, j);
      Acc s{};
      if (k0 == 0) acc_of(s, F[(size_t)(o + i) * m + o + j]);
#pragma unroll 2
      for (int k = k0; k < r; k += ks) mac(s, Y[i * ldx + k], X[j * ldx + k]);
      Z g = acc_get(s);
      for (int off = 1; off < ks; off <<= 1) g = zadd(g, zshfl_xor(g, off));
      if (k0 == 0 && e0 + tid / ks < outs) {
        if (direct) {
          P[i * w + j] = g;
          P[j * w + i] = g;
        } else {
          F[(size_t)(o + i) * m + o + j] = g;
          F[(size_t)(o + j) * m + o + i] = g;
        }
        if (i == j) B.gd[B.tab[nd.sites + o + i]] = B.la.zshift ? zim(g) : B.sg * zre(g);
      }
    }
    if (!direct) {
      for (int i = tid >> 5; i < w; i += size >> 5)
        for (int j = tid & 31; j < r; j += 32) F[(o + i) * m + o + w + j] = Y[i * ldx + j];
      for (int j = tid >> 4; j < r; j += size >> 4)
        for (int i = tid & 15; i < w; i += 16) F[(o + w + j) * m + o + i] = Y[i * ldx + j];
    }
    gr.sync();
  }
  // blacks: G_bb = 1/a + (t/a)^2 sum_{u,v} G_uv over the black's neighbours, four threads each
  // (one neighbour u per thread); such leaves have one panel
  if (nd.blacks) {
    for (int b0 = 0; b0 < nd.blacks; b0 += size / 4) {
      const int b = min(b0 + tid / 4, nd.blacks - 1), u = tid & 3;
      const int s = B.tab[nd.bsite + b];
      const int iu = B.tab[nd.bnbr + 4 * b + u];
      Z sum;
      zset(sum, 0.0, 0.0);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int iv = B.tab[nd.bnbr + 4 * b + v], hi = max(iu, iv), lo = min(iu, iv);
        sum = zadd(sum, hi < p    ? P[hi * p + lo]
                        : lo < p  ? Y[lo * ldx + hi - p]
                                  : G[(size_t)map[hi - p] * mp + map[lo - p]]);
      }
      sum = zadd(sum, zshfl_xor(sum, 1));
      sum = zadd(sum, zshfl_xor(sum, 2));
      if (u == 0 && b0 + tid / 4 < nd.blacks) {
        Z z, t2;
        zset(z, near_term<Z>(B.zr - site_energy(B.la, s, B.sg)), B.zi);
        zset(t2, B.la.t * B.la.t, 0.0);
        const Z ai = zinv(z);
        const Z g = zadd(ai, zmul(zmul(zmul(ai, t2), ai), sum));
        B.gd[s] = B.la.zshift ? zim(g) : B.sg * zre(g);
      }
    }
    gr.sync();
  }
}

// Barrier of the CTAs that share a block (global memory written before it is visible after it).
template <bool kCluster>
__device__ __forceinline__ void block_sync() {
  if (kCluster)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                     : "memory");
  else
    __syncthreads();
}

// The elimination of one block by one CTA, or by a cluster of them: level after level, up and then
// down, each level's fronts dealt out to the CTAs' thread groups.  A launch of a single level
// (k1 = k0 + 1) needs no barrier and may spread a block over any number of CTAs.
template <typename Z, int NT, bool kCluster>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : 1) k_nested(NestArgs<Z> a) {
  const int tid = threadIdx.x;
  const int csize = a.csize, rank = blockIdx.x % csize;
  const int mat = blockIdx.x / csize;
  __shared__ Block<Z> B;  // read where needed: in registers it would be live everywhere
  __shared__ int form;
  if (tid == 0) {
    int n;
    B.la = block_lattice(a.la, a.b0 + mat, n, B.sg);
    B.zr = B.la.mu;
    B.zi = (2.0 * n + 1.0) * kPi * B.la.T;
    if (B.la.zshift) {
      B.zr = B.la.zshift[2 * n];
      B.zi = B.la.zshift[2 * n + 1];
    }
    form = mat < a.ndense ? 1 : 0;
    B.nodes = a.nodes + form * a.nnodes;
    B.tab = a.tab;
    B.fronts = a.fronts + (size_t)mat * a.stride;
    B.det = a.det + (size_t)mat * a.nnodes;
    B.gd = a.gd + (size_t)(a.b0 + mat) * B.la.N;
    B.flags = a.flags;
  }
  __syncthreads();
  if (a.range) {
    int big = 0;
    for (int i = tid; i < B.la.N; i += NT)
      if (beyond(B.zr - site_energy(B.la, i, B.sg))) big = 1;
    if (__syncthreads_or(big) != (a.range == 2)) return;  // (alike in all CTAs of a block)
  }
  for (int k = a.k0; k < a.k1; ++k) {
    const bool up = k < a.nlevels;
    const LevelPlan& lv = a.lv[form][up ? a.nlevels - 1 - k : k - a.nlevels];
    const int group = tid / lv.group, groups = NT / lv.group;
    const Group gr{lv.group, tid - group * lv.group, 1 + group};
    const int at = group * lv.smem;
    for (int f = rank + csize * group; f < lv.count; f += csize * groups) {
      if (up)
        front_up(B, lv.first + f, gr, at);
      else
        front_down<Z, NT>(B, lv.first + f, gr, at);
    }
    if (k + 1 == a.k1 && k != a.nlevels - 1) break;
    block_sync<kCluster>();
    if (k == a.nlevels - 1 && rank == 0 && tid < 32) {  // ln|det A| over all nodes, fixed order
      double v = 0.0;
      int e = 0;
      for (int i = tid; i < a.nnodes; i += 32) {
        v += log(B.det[i].mant);
        e += B.det[i].exp;
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, off);
        e += __shfl_xor_sync(0xffffffffu, e, off);
      }
      if (tid == 0) a.ld[a.b0 + mat] = 0.5 * (v + (double)e * 0.69314718055994530942);
    }
  }
}

// Im Tr G per block for a density of states: fixed-order sum of the row that k_nested wrote.
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

// z: bytes of an entry
size_t up_smem(const nested::Node& n, size_t z) {
  const size_t m = n.p + n.q, pw = n.pw;
  return z * (pw * (2 * (m - pw) + kRows) + pw * pw + 2 * pw + 2 * (pw + 1) + n.blacks + n.p + 1) +
         32 * sizeof(double) + sizeof(int16_t) * m * (n.blacks ? 4 : 3);
}
size_t down_smem(const nested::Node& n, size_t z) {
  const size_t m = n.p + n.q;
  return z * (2 * (size_t)n.pw * ((m - n.pw) | 1) + (size_t)n.pw * n.pw) + sizeof(int16_t) * n.q;
}

}  // namespace

// The two forms of one lattice size's tree, as every context of that size takes them: the tables in
// one piece (nodes, then indices) and the shapes that the launch plans follow.
struct NestedForms {
  struct Shape {
    int first, count, group;  // group: the fewest threads for a front
    int bytes[3];             // shared memory of a front with entries of 16, 24 and 32 bytes
    template <typename Z>
    int smem() const { return bytes[sizeof(Z) / 8 - 2]; }
  };
  std::vector<Shape> levels[2];
  std::vector<char> tables;
  size_t index_at = 0;    // offset of the indices
  int nnodes = 0;
  long long stride = 0;   // entries per block

  // A block's fronts, and with its shares of |det A|^2.  (A float64 context's wider blocks have
  // room for double-double, at the same place for both arithmetics that they may take.)
  size_t front_bytes(NestedArith a) const {
    return (a == NestedArith::kWide64 ? 32 : a == NestedArith::kWide32 ? 24 : 16) * (size_t)stride;
  }
  size_t block_bytes(NestedArith a) const { return front_bytes(a) + sizeof(Det) * nnodes; }
  // Room for all blocks in their arithmetic where all are to be resident, and for one block of the
  // wider one in any case.  From 10 x 10 sites up the dense blocks take more than either.
  size_t room_for(const Engine& e) const {
    const size_t base = block_bytes(e.fp64 ? NestedArith::kFloat64 : NestedArith::kFloat2);
    const size_t wide = block_bytes(e.fp64 ? NestedArith::kWide64 : NestedArith::kWide32);
    if (e.chunk < e.B) return wide;
    return std::max(wide, e.nest_wide * wide + (e.B - e.nest_wide) * base + 256);
  }
};

// Per-context state: the tables on the device, memory, streams.
struct Nested {
  const NestedForms& f;
  explicit Nested(const NestedForms& forms) : f(forms) {}
  char* d_tables = nullptr;
  char* fronts = nullptr; // where they are kept: the context's blocks, or `own`
  size_t room = 0;
  void* own = nullptr;    // their own memory where the blocks' is too small
  int sms = 1;
  // more blocks than SMs: the second half of a pass that takes a launch per level (a stream of its
  // own only where there is no second stream of the dense elimination), and the blocks in wider
  // arithmetic (which otherwise take the side stream)
  cudaStream_t half = nullptr, wide = nullptr;
  bool half_own = false;
  cudaEvent_t ev_half = nullptr, ev_wide = nullptr;
};

namespace {

// Plan of a whole elimination by CTAs of 512 threads, a.csize of them per block: a level's fronts
// are dealt out over the CTAs' groups, whose size is the fewest threads for a front where there
// are fronts enough and grows to the whole CTA where there are not, or where shared memory needs
// fewer groups.  Returns the shared memory that a CTA needs.
template <typename Z>
size_t plan_levels(const Nested& ne, NestArgs<Z>& a) {
  constexpr int nt = 512, room = 220 << 10;
  static_assert(nt / 64 < 16, "a group above a warp needs one of the 15 barriers left");
  size_t need = 0;
  for (int form = 0; form < 2; ++form)
    for (size_t k = 0; k < ne.f.levels[form].size(); ++k) {
      const NestedForms::Shape& s = ne.f.levels[form][k];
      const int smem = s.smem<Z>();
      int g = s.group;
      while (2 * g <= nt && ((nt / (2 * g)) * a.csize >= s.count || nt / g * smem > room)) g *= 2;
      a.lv[form][k] = {s.first, s.count, g, smem};
      need = std::max(need, (size_t)(nt / g) * smem);
    }
  return need;
}

template <typename Z, int NT, bool kCluster>
sca_status launch(Engine& e, const NestArgs<Z>& a, int cnt, size_t smem, cudaStream_t s) {
  static ContextOnce once;
  cudaError_t err;
  if (!once.done()) {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    if ((err = cudaGetDevice(&dev)) != cudaSuccess ||
        (err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess ||
        (err = cudaFuncGetAttributes(&fa, k_nested<Z, NT, kCluster>)) != cudaSuccess ||
        (err = cudaFuncSetAttribute(k_nested<Z, NT, kCluster>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    optin - (int)fa.sharedSizeBytes)) != cudaSuccess)
      return cuda_fail(err, "nested elimination set-up");
    once.mark();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(cnt * a.csize));
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.csize;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = kCluster ? 1 : 0;
  const int kind = a.k0 < a.nlevels ? kNestUp : kNestDown;
  prof_begin(e, kind, s);
  err = cudaLaunchKernelEx(&cfg, k_nested<Z, NT, kCluster>, a);
  prof_end(e, kind, s);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (err != cudaSuccess) return cuda_fail(err, "nested elimination");
  return SCA_OK;
}

// Blocks [b0, b0 + cnt) in arithmetic Z, their fronts at `mem`, `bytes` for each, on `s`; `free_sms`
// SMs are for them.
template <typename Z>
sca_status run_blocks_of(Engine& e, const Lattice& la, int b0, int cnt, char* mem, size_t bytes,
                         int free_sms, bool up, bool down, cudaStream_t s, int max_cluster,
                         int range = 0) {
  const Nested& ne = *e.nest;
  NestArgs<Z> a;
  a.nodes = reinterpret_cast<const Node*>(ne.d_tables);
  a.tab = reinterpret_cast<const int16_t*>(ne.d_tables + ne.f.index_at);
  a.fronts = reinterpret_cast<Z*>(mem);
  a.stride = (long long)(bytes / sizeof(Z));
  a.nnodes = ne.f.nnodes;
  a.nlevels = (int)ne.f.levels[0].size();
  a.la = la;
  a.ld = e.ld;
  a.gd = e.gd;
  a.flags = e.flags;
  a.b0 = b0;
  a.det = reinterpret_cast<Det*>(mem + (size_t)cnt * bytes);
  const int nl = a.nlevels, p0 = up ? 0 : nl, p1 = down ? 2 * nl : nl;
  sca_status st = SCA_OK;
  const int dense = std::min(cnt, std::max(0, e.nest_dense - b0));
  a.ndense = dense;
  a.range = range;
  if (cnt > ne.sms && sizeof(Z) == 16) {
    // side by side: the few blocks with dense leaves on the high-priority stream, and the others
    // in two halves, so that one half's fronts fill the SMs that the last wave of the other's
    // level leaves idle
    struct Part {
      int form, first, n, all;  // all: blocks of the form, which the group sizes follow
      cudaStream_t s;
      cudaEvent_t join;
    } parts[4];
    int nparts = 0;
    const bool two = dense > 0 && dense < cnt && e.side != nullptr;
    for (int form = 1; form >= 0; --form) {
      const int n = form ? dense : cnt - dense, first = form ? 0 : dense;
      const int h = ne.half && n >= kHalves && !(form && two) ? n / 2 : 0;
      if (n == 0) continue;
      if (form && two)
        parts[nparts++] = {form, first, n, n, e.side, e.ev_join};
      else
        parts[nparts++] = {form, first, n - h, n, s, nullptr};
      if (h) parts[nparts++] = {form, first + n - h, h, n, ne.half, ne.ev_half};
    }
    cudaError_t err = cudaSuccess;
    if (nparts > 1) err = cudaEventRecord(e.ev_fork, s);
    for (int i = 0; i < nparts && err == cudaSuccess; ++i)
      if (parts[i].join) err = cudaStreamWaitEvent(parts[i].s, e.ev_fork, 0);
    if (err != cudaSuccess) return cuda_fail(err, "fork");
    for (int k = p0; k < p1; ++k)
      for (int i = 0; i < nparts; ++i) {
        const Part& pt = parts[i];
        NestArgs<Z> f = a;  // the part's blocks alone
        f.b0 = b0 + pt.first;
        f.fronts = a.fronts + (size_t)pt.first * a.stride;
        f.det = a.det + (size_t)pt.first * a.nnodes;
        f.ndense = pt.form ? pt.n : 0;
        const int level = k < nl ? nl - 1 - k : k - nl;
        f.k0 = k;
        f.k1 = k + 1;
        const NestedForms::Shape& sh = ne.f.levels[pt.form][level];
        const int smem = sh.smem<Z>();
        int g = sh.group;  // the fewest threads while they fill the SMs; four CTAs per SM
        while (2 * g <= 256 && ((long long)sh.count * pt.all * g < 1024ll * ne.sms ||
                                256 / g * smem > 55 << 10))
          g *= 2;
        f.lv[pt.form][level] = {sh.first, sh.count, g, smem};
        f.csize = (sh.count + 256 / g - 1) / (256 / g);
        if constexpr (sizeof(Z) == 16)
          st = launch<Z, 256, false>(e, f, pt.n, (size_t)(256 / g) * smem, pt.s);
        if (st != SCA_OK) return st;
      }
    for (int i = 0; i < nparts && err == cudaSuccess; ++i)
      if (parts[i].join) {
        err = cudaEventRecord(parts[i].join, parts[i].s);
        if (err == cudaSuccess) err = cudaStreamWaitEvent(s, parts[i].join, 0);
      }
    if (err != cudaSuccess) return cuda_fail(err, "join");
  } else {
    // CTAs per block: as many as there are SMs for, up to the portable cluster size
    a.k0 = p0;
    a.k1 = p1;
    a.csize = 1;
    while (2 * a.csize <= max_cluster && 2 * a.csize * cnt <= free_sms) a.csize *= 2;
    const size_t smem = plan_levels(ne, a);
    st = a.csize > 1 ? launch<Z, 512, true>(e, a, cnt, smem, s)
                     : launch<Z, 512, false>(e, a, cnt, smem, s);
  }
  if (st != SCA_OK) return st;
  if (down && la.zshift && range != 1) {
    prof_begin(e, kRefine, s);
    k_nest_trace<<<cnt, 256, 0, s>>>(e.N, b0, e.gd, e.tr);
    prof_end(e, kRefine, s);
    SCA_LAUNCH_CHECK("nested trace");
  }
  return SCA_OK;
}

sca_status run_blocks_in(NestedArith ar, Engine& e, const Lattice& la, int b0, int cnt, char* mem,
                         int free_sms, bool up, bool down, cudaStream_t s, int max_cluster = 8) {
  const size_t by = e.nest->f.front_bytes(ar);
  const int mc = max_cluster;
  if (ar == NestedArith::kFloat2)
    return run_blocks_of<Zf>(e, la, b0, cnt, mem, by, free_sms, up, down, s, mc);
  if (ar == NestedArith::kFloat64)
    return run_blocks_of<Zd>(e, la, b0, cnt, mem, by, free_sms, up, down, s, mc);
  if (ar == NestedArith::kWide32)
    return run_blocks_of<Zt>(e, la, b0, cnt, mem, by, free_sms, up, down, s, mc);
  // a float64 context: entries beyond float32's range take double-double (a launch that ends at
  // once where there are none)
  sca_status st = run_blocks_of<Zt>(e, la, b0, cnt, mem, by, free_sms, up, down, s, mc, 1);
  if (st == SCA_OK) st = run_blocks_of<Zw>(e, la, b0, cnt, mem, by, free_sms, up, down, s, mc, 2);
  return st;
}

}  // namespace

bool nested_rule(double t, double imag_min, double imag_max) {
  return imag_min >= kNestedMinImag * std::fabs(t) && imag_min >= 1e-9 && imag_max <= 1e9 &&
         std::fabs(t) <= 1e9;
}

bool nested_wide(bool fp64, int L, double t, double imag) {
  const double enough = fp64 ? kFloat64Enough : L <= 10 ? kFloat2EnoughSmall : kFloat2Enough;
  return imag < enough * std::fabs(t);
}

int nested_wide_blocks(bool fp64, int L, double t, double T, int n_omega) {
  int n = 0;
  while (n < n_omega && nested_wide(fp64, L, t, (2.0 * n + 1.0) * M_PI * T)) ++n;
  return 2 * n;
}

// The forms of lattice size L: constant data, built by the first context of that size (64x64: 0.6 ms)
// and kept, 0.3 MB at most each.  Null where host memory is short.
static const NestedForms* nested_forms(int L) {
  static std::mutex mu;
  static std::unique_ptr<const NestedForms> built[33];
  if (L < nested::kMinL || L > 64) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  std::unique_ptr<const NestedForms>& slot = built[L / 2];
  if (slot) return slot.get();
  try {
    std::unique_ptr<NestedForms> f(new NestedForms());
    nested::Tree t[2] = {nested::Builder(L).build(false), nested::Builder(L).build(true)};
    f->nnodes = (int)t[0].nodes.size();
    // whole entries of 16, 24 and 32 bytes
    f->stride = (std::max(t[0].entries, t[1].entries) + 5) / 6 * 6;
    std::vector<Node> nodes;
    std::vector<int16_t> table;
    for (int form = 0; form < 2; ++form) {
      for (const nested::Level& lv : t[form].levels) {
        NestedForms::Shape sh{lv.first, lv.count, 32, {0, 0, 0}};
        for (int k = lv.first; k < lv.first + lv.count; ++k) {
          const nested::Node& n = t[form].nodes[k];
          while (10 * sh.group < 9 * (n.p + n.q) || n.pw > kSlots * (sh.group / n.pw)) sh.group *= 2;
          for (int z = 16; z <= 32; z += 8) {
            int& by = sh.bytes[z / 8 - 2];
            by = std::max(by, ((int)std::max(up_smem(n, z), down_smem(n, z)) + 15) / 16 * 16);
          }
        }
        f->levels[form].push_back(sh);
      }
      // one table: a form's offsets follow the entries before it
      const int at = (int)table.size();
      table.insert(table.end(), t[form].table.begin(), t[form].table.end());
      for (nested::Node n : t[form].nodes) {
        for (int* o : {&n.sites, &n.cmap[0], &n.cmap[1], &n.pmap, &n.bsite, &n.bnbr, &n.adj}) *o += at;
        nodes.push_back(n);
      }
    }
    f->index_at = (sizeof(Node) * nodes.size() + 15) / 16 * 16;
    f->tables.resize(f->index_at + sizeof(int16_t) * table.size());
    std::memcpy(f->tables.data(), nodes.data(), sizeof(Node) * nodes.size());
    std::memcpy(f->tables.data() + f->index_at, table.data(), sizeof(int16_t) * table.size());
    slot = std::move(f);
  } catch (const std::bad_alloc&) {
    return nullptr;
  }
  return slot.get();
}

size_t nested_bytes(const Engine& e) {
  const NestedForms* f = e.dense_switch ? nullptr : nested_forms(e.L);
  if (!f) return 0;
  const size_t need = f->room_for(e);
  return f->tables.size() + (need > e.block_room ? need : 0);
}

sca_status nested_wide_stream(Engine& e) {
  Nested* ne = e.nest;
  if (!ne || ne->wide || e.B <= ne->sms) return SCA_OK;
  int least = 0, greatest = 0;
  cudaError_t err = cudaDeviceGetStreamPriorityRange(&least, &greatest);
  if (err == cudaSuccess)
    err = cudaStreamCreateWithPriority(&ne->wide, cudaStreamNonBlocking, greatest);
  return err == cudaSuccess ? SCA_OK : cuda_fail(err, "nested elimination set-up");
}

sca_status nested_prepare(Engine& e) {
  if (e.nest || e.L < nested::kMinL) return SCA_OK;
  const NestedForms* forms = nested_forms(e.L);
  Nested* ne = forms ? new (std::nothrow) Nested(*forms) : nullptr;
  if (!ne) { set_error("host allocation failed"); return SCA_ENOMEM; }
  e.nest = ne;
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess)
    err = cudaDeviceGetAttribute(&ne->sms, cudaDevAttrMultiProcessorCount, dev);
  if (err == cudaSuccess) err = cudaEventCreateWithFlags(&ne->ev_wide, cudaEventDisableTiming);
  if (err == cudaSuccess && e.B > ne->sms) {
    ne->half = e.aux;
    if (!ne->half) {
      err = cudaStreamCreateWithFlags(&ne->half, cudaStreamNonBlocking);
      ne->half_own = err == cudaSuccess;
    }
    if (err == cudaSuccess) err = cudaEventCreateWithFlags(&ne->ev_half, cudaEventDisableTiming);
  }
  if (err != cudaSuccess) { nested_release(e); return cuda_fail(err, "nested elimination set-up"); }
  if (e.nest_wide > 0) {
    const sca_status st = nested_wide_stream(e);
    if (st != SCA_OK) { nested_release(e); return st; }
  }
  const size_t need = forms->room_for(e);
  ne->fronts = static_cast<char*>(e.M);
  ne->room = e.block_room;
  if (need > ne->room) {
    err = device_malloc(&ne->own, need);
    ne->fronts = static_cast<char*>(ne->own);
    ne->room = need;
  }
  if (err == cudaSuccess) err = device_malloc((void**)&ne->d_tables, forms->tables.size());
  if (err != cudaSuccess) {
    nested_release(e);
    (void)cudaGetLastError();
    set_error("cudaMalloc failed for the elimination tree or its fronts");
    return SCA_ENOMEM;
  }
  err = cudaMemcpy(ne->d_tables, forms->tables.data(), forms->tables.size(), cudaMemcpyHostToDevice);
  // (a copy from pageable memory may still be under way, and the context's streams do not wait for
  // the default one)
  if (err == cudaSuccess) err = cudaStreamSynchronize(cudaStreamLegacy);
  if (err != cudaSuccess) { nested_release(e); return cuda_fail(err, "elimination tree upload"); }
  return SCA_OK;
}

void nested_release(Engine& e) {
  if (!e.nest) return;
  if (e.nest->half_own) {
    cudaStreamSynchronize(e.nest->half);
    cudaStreamDestroy(e.nest->half);
  }
  if (e.nest->wide) {
    cudaStreamSynchronize(e.nest->wide);
    cudaStreamDestroy(e.nest->wide);
  }
  if (e.nest->ev_half) cudaEventDestroy(e.nest->ev_half);
  if (e.nest->ev_wide) cudaEventDestroy(e.nest->ev_wide);
  if (e.nest->own) cudaFree(e.nest->own);
  if (e.nest->d_tables) cudaFree(e.nest->d_tables);
  delete e.nest;
  e.nest = nullptr;
}

sca_status run_nested(Engine& e, const Lattice& la, bool up, bool down, cudaStream_t s) {
  const Nested& ne = *e.nest;
  cudaError_t err = cudaSuccess;
  if (up) {
    err = cudaMemsetAsync(e.flags, 0, sizeof(int), s);
    if (err != cudaSuccess) return cuda_fail(err, "flags reset");
  }
  // the blocks in wider arithmetic first, then the others
  struct Group {
    NestedArith ar;
    int first, n;
    size_t bytes;
  } groups[2];
  int ng = 0;
  const int nw = std::min(e.B, e.nest_wide);
  const int ends[3] = {0, nw, e.B};
  const NestedArith kinds[2] = {e.fp64 ? NestedArith::kWide64 : NestedArith::kWide32,
                                e.fp64 ? NestedArith::kFloat64 : NestedArith::kFloat2};
  size_t total = 0;
  for (int k = 0; k < 2; ++k)
    if (const int n = ends[k + 1] - ends[k]) {
      groups[ng] = {kinds[k], ends[k], n, (n * ne.f.block_bytes(kinds[k]) + 255) / 256 * 256};
      total += k == 0 && nw < e.B ? groups[ng].bytes : n * ne.f.block_bytes(kinds[k]);
      ++ng;
    }
  if (total > ne.room) {  // one after another, in passes that fit
    if (!up) {
      set_error("the eliminated fronts are not all resident");
      return SCA_ENOSTATE;
    }
    for (int g = 0; g < ng; ++g) {
      const int cap = (int)std::min<size_t>(ne.room / ne.f.block_bytes(groups[g].ar), groups[g].n);
      for (int b = 0; b < groups[g].n; b += cap) {
        const sca_status st = run_blocks_in(groups[g].ar, e, la, groups[g].first + b,
                                            std::min(cap, groups[g].n - b), ne.fronts, ne.sms, up,
                                            down, s);
        if (st != SCA_OK) return st;
      }
    }
    return SCA_OK;
  }
  if (ng < 2)
    return run_blocks_in(groups[0].ar, e, la, groups[0].first, groups[0].n, ne.fronts, ne.sms, up,
                         down, s);
  // Side by side: the few in wider arithmetic on a stream of their own, with the SMs that the
  // others leave at one block per SM.  Where those take a launch per level, over several blocks' time
  // per SM, clusters are smaller by as much.
  const cudaStream_t ws = ne.wide ? ne.wide : e.side;
  err = cudaEventRecord(ne.ev_wide, s);
  if (err == cudaSuccess) err = cudaStreamWaitEvent(ws, ne.ev_wide, 0);
  if (err != cudaSuccess) return cuda_fail(err, "fork");
  const int others = e.B - nw, free_sms = ne.sms - (others <= ne.sms ? others : 0);
  const int max_cluster = others <= ne.sms ? 8 : std::max(1, 8 * ne.sms / others);
  int c = 1;
  while (2 * c <= max_cluster && 2 * c * nw <= free_sms) c *= 2;
  sca_status st =
      run_blocks_in(groups[0].ar, e, la, 0, nw, ne.fronts, free_sms, up, down, ws, max_cluster);
  if (st == SCA_OK)
    st = run_blocks_in(groups[1].ar, e, la, nw, others, ne.fronts + groups[0].bytes,
                       std::max(1, ne.sms - c * nw), up, down, s);
  if (st != SCA_OK) return st;
  err = cudaEventRecord(ne.ev_wide, ws);
  if (err == cudaSuccess) err = cudaStreamWaitEvent(s, ne.ev_wide, 0);
  if (err != cudaSuccess) return cuda_fail(err, "join");
  return SCA_OK;
}

}  // namespace sca
