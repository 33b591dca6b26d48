// Loop hafnian by elimination of index pairs with polynomial entries.
//
// Write the loop hafnian's Gaussian generating function with one variable x_p per index pair
// p = (j, j+n): lhaf(A) is the coefficient of x_1 x_2 ... x_n. Integrating the pairs out one
// after the other and keeping each x_p to first order only (a higher power of x_p can never
// end in that coefficient) turns the matrix of the remaining vertices into polynomials:
//     A'_jk = A_jk + x_p (A_ja A_kb + A_jb A_ka)
//     v'_j  = v_j  + x_p (A_ja v_b  + A_jb v_a)
//     g'    = g (1 + x_p (A_ab + v_a v_b)),                 p = (a, b).
// Setting x_p = d_p x with signs d_p = +-1 leaves polynomials in one x, and the signed mean
// over the sign patterns keeps exactly the monomials in which every x_p occurs to an odd
// power; in degree n that is x_1 ... x_n alone. This is the inclusion-exclusion idea of
// Bjorklund ("Counting perfect matchings as fast as Ryser", SODA 2012) with signs in place
// of subsets, extended by the loop weights v. Flipping all signs and x changes nothing, so
// the first sign is +. After d pairs only degrees <= d matter, so everything is truncated
// there. The last two pairs are not signed: with four vertices left,
//     lhaf = [x^{n-2}] g (w01 w23 + w02 w13 + w03 w12 - 2 v0 v1 v2 v3),  w_jk = A_jk + v_j v_k.
// The sign patterns form a binary tree; all nodes of one depth have the same shapes, so a
// level is a set of equal truncated polynomial products.
//
// Work: 2^{n-3} leaves with about 62 products of truncated polynomials each, ~8 n^2 2^n / 15
// complex multiply-adds in all, against ~n^3 2^n for building every subset term from scratch
// (N = 40: 1.1e9 against 1.1e10), and the signed mean cancels by 10^2..10^4 where the signed
// subset sum cancels by 10^7..10^12.
//
// Arithmetic. Products of polynomials are sums of products with no division, so they run in
// fixed point: a real number is an 84-bit integer times 2^-81, held as three 28-bit limbs
// with signs (h 2^56 + m 2^28 + l). GB300 issues 64 32x32+64-bit integer multiply-adds per SM
// and clock (measured 18.7e12/s), a limb product is at most 2^54, and up to 2^9 of them add
// up in 64 bits without a carry, so a whole convolution accumulates exactly and is normalised
// once. Six limb products per real product (the three below 2^-81 are dropped) make 24
// multiply-adds per complex one: 0.78e12 complex multiply-adds/s, against 0.17e12/s for
// triple-float (216 FP32 instructions) and 0.15e12/s for FP64. Fixed point needs a scale: the
// matrix is scaled by one factor such that its root-mean-fourth singular value is about one,
// which keeps the coefficients of every matrix tried between 2^-10 and 1.5 (the format holds
// |x| < 4). Overflow anywhere, or a result so small that the 2^-81 resolution could show, sets
// a flag and the caller evaluates the problem by the subset sum instead.
//
// The code of one level is a function of (level, task number) that reads the level's nodes
// and writes the next level's, so it compiles for the host as well and is checked there
// against the definition, with every index bounds-checked.
#pragma once

#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define GBSH_HD __host__ __device__ __forceinline__
#else
#define GBSH_HD inline
#endif

namespace gbsh {

constexpr int kTreeFrac = 81;        // value = integer * 2^-81
constexpr int kLimbBits = 28;

// A complex fixed-point number: limbs of the real and the imaginary part (32 bytes, so that
// an element is two 16-byte loads).
struct alignas(16) Fxc {
  int rh, rm, rl, ih;
  int im, il, pad0, pad1;
};

// 64-bit limb-product sums of one complex accumulator, by weight: s2 2^112, s1 2^84, s0 2^56
// (in units of 2^-162).
struct FxAcc {
  long long s2r, s1r, s0r, s2i, s1i, s0i;
};

GBSH_HD FxAcc fx_acc_zero() { return FxAcc{0, 0, 0, 0, 0, 0}; }

GBSH_HD Fxc fx_load(const Fxc* p) {
#ifdef __CUDA_ARCH__
  const int4 a = reinterpret_cast<const int4*>(p)[0];
  const int2 b = reinterpret_cast<const int2*>(p)[2];
  return Fxc{a.x, a.y, a.z, a.w, b.x, b.y, 0, 0};
#else
  return *p;
#endif
}
GBSH_HD void fx_store(Fxc* p, const Fxc& v) {
#ifdef __CUDA_ARCH__
  reinterpret_cast<int4*>(p)[0] = make_int4(v.rh, v.rm, v.rl, v.ih);
  reinterpret_cast<int2*>(p)[2] = make_int2(v.im, v.il);
#else
  *p = v;
#endif
}

// acc += a * b. The limb products of weight 2^28 and 1 are below the result's resolution.
GBSH_HD void fx_mac(FxAcc& s, const Fxc& a, const Fxc& b) {
  const int nh = -a.ih, nm = -a.im, nl = -a.il;
  s.s2r += (long long)a.rh * b.rh;
  s.s2r += (long long)nh * b.ih;
  s.s1r += (long long)a.rh * b.rm;
  s.s1r += (long long)a.rm * b.rh;
  s.s1r += (long long)nh * b.im;
  s.s1r += (long long)nm * b.ih;
  s.s0r += (long long)a.rh * b.rl;
  s.s0r += (long long)a.rl * b.rh;
  s.s0r += (long long)a.rm * b.rm;
  s.s0r += (long long)nh * b.il;
  s.s0r += (long long)nl * b.ih;
  s.s0r += (long long)nm * b.im;
  s.s2i += (long long)a.rh * b.ih;
  s.s2i += (long long)a.ih * b.rh;
  s.s1i += (long long)a.rh * b.im;
  s.s1i += (long long)a.rm * b.ih;
  s.s1i += (long long)a.ih * b.rm;
  s.s1i += (long long)a.im * b.rh;
  s.s0i += (long long)a.rh * b.il;
  s.s0i += (long long)a.rl * b.ih;
  s.s0i += (long long)a.rm * b.im;
  s.s0i += (long long)a.ih * b.rl;
  s.s0i += (long long)a.il * b.rh;
  s.s0i += (long long)a.im * b.rm;
}

GBSH_HD int sext28(long long x) { return (int)((unsigned)x << 4) >> 4; }

// The accumulated real number rounded to the format; bad |= it does not fit (|x| < 2).
GBSH_HD void fx_norm(long long s2, long long s1, long long s0, int& h, int& m, int& l, unsigned& bad) {
  bad |= (unsigned)((unsigned long long)(s2 + (1ll << 51)) >> 52);
  // in units of 2^-81: s2 2^31 + s1 2^3 + s0 2^-25
  const long long lo = ((s1 & ((1ll << 25) - 1)) << 3) + ((s0 + (1ll << 24)) >> 25);
  l = sext28(lo);
  const long long v = (long long)((unsigned long long)s2 << 3) + (s1 >> 25) + ((lo - l) >> 28);
  m = sext28(v);
  h = (int)((v - m) >> 28);
}
GBSH_HD Fxc fx_norm(const FxAcc& s, unsigned& bad) {
  Fxc r{};
  fx_norm(s.s2r, s.s1r, s.s0r, r.rh, r.rm, r.rl, bad);
  fx_norm(s.s2i, s.s1i, s.s0i, r.ih, r.im, r.il, bad);
  return r;
}

// (h, m, l) = a + sg b, carries propagated; bad |= |result| >= 4.
GBSH_HD void fx_add1(int ah, int am, int al, int bh, int bm, int bl, int sg, int& h, int& m, int& l,
                     unsigned& bad) {
  const int x = al + sg * bl;
  l = sext28(x);
  const int y = am + sg * bm + ((x - l) >> 28);
  m = sext28(y);
  h = ah + sg * bh + ((y - m) >> 28);
  bad |= (unsigned)(h + (1 << 27)) >> 28;
}
GBSH_HD Fxc fx_add(const Fxc& a, const Fxc& b, int sg, unsigned& bad) {
  Fxc r{};
  fx_add1(a.rh, a.rm, a.rl, b.rh, b.rm, b.rl, sg, r.rh, r.rm, r.rl, bad);
  fx_add1(a.ih, a.im, a.il, b.ih, b.im, b.il, sg, r.ih, r.im, r.il, bad);
  return r;
}

// acc0, acc1 += coefficients t0, t0 + 1 of the polynomial product a * b, a[u] at a + u sa, b[u]
// at b + u sb; t0 = -1 leaves acc0 alone. t0 + 1 must not exceed the last coefficient of either
// factor. Two coefficients a task: each step loads one new element of each factor for two
// multiply-adds (b in a sliding window of two). Four would halve the loads, but with the
// accumulators of four (48 registers) the code spilled and outgrew the instruction cache.
GBSH_HD void fx_conv2(FxAcc& acc0, FxAcc& acc1, const Fxc* a, int sa, const Fxc* b, int sb, int t0) {
  b += (ptrdiff_t)(t0 + 1) * sb;
  Fxc w1 = fx_load(b), w0{};
  int u = t0 + 1;  // steps before the last one
  if (u > 0) {
    b -= sb;
    w0 = fx_load(b);
    if (u & 1) {
      const Fxc x = fx_load(a);
      a += sa;
      fx_mac(acc0, x, w0);
      fx_mac(acc1, x, w1);
      w1 = w0;
      if (u > 1) {
        b -= sb;
        w0 = fx_load(b);
      }
    }
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
    for (u >>= 1; u > 0; --u) {
      Fxc x = fx_load(a);
      a += sa;
      fx_mac(acc0, x, w0);
      fx_mac(acc1, x, w1);
      b -= sb;
      w1 = fx_load(b);
      x = fx_load(a);
      a += sa;
      fx_mac(acc0, x, w1);
      fx_mac(acc1, x, w0);
      if (u > 1) {
        b -= sb;
        w0 = fx_load(b);
      }
    }
  }
  fx_mac(acc1, fx_load(a), w1);
}

// ------------------------------------------------------------------ levels of the tree
// Level M holds nodes with M pairs left: r = 2M vertices, L = n - M + 1 coefficients per
// polynomial. A node's polynomials are the A_jk, j < k < r, at k (k - 1) / 2 + j (so that
// eliminating the last pair leaves the others in place) and the loop weights v_j at
// r (r - 1) / 2 + j. Coefficient u of polynomial p of node x is A[(u ld + x) P + p]; g and
// h = A_ab + v_a v_b (of the pair that is eliminated next) are at [u ld + x].
GBSH_HD constexpr int tree_polys(int M) { return M * (2 * M + 1); }

struct TreeLevel {
  Fxc* A;
  Fxc* g;
  Fxc* h;
  int q;   // nodes, from the pointers on
  int ld;  // nodes stored side by side
};

// Elements of a level of q nodes (level 2 holds the eight w and v v polynomials in place of h).
GBSH_HD size_t tree_level_elems(int M, int n, int q) {
  return (size_t)q * (n - M + 1) * (tree_polys(M) + 1 + (M == 2 ? 8 : 1));
}
GBSH_HD TreeLevel tree_level(Fxc* base, int M, int n, int q) {
  const size_t L = n - M + 1;
  TreeLevel v;
  v.A = base;
  v.g = base + (size_t)q * L * tree_polys(M);
  v.h = v.g + (size_t)q * L;
  v.q = v.ld = q;
  return v;
}
// Node x of a level as a level of one node.
GBSH_HD TreeLevel tree_node(const TreeLevel& v, int M, int x) {
  return TreeLevel{v.A + (size_t)x * tree_polys(M), v.g + x, v.h + (M == 2 ? 8 * x : x), 1, v.ld};
}
// Nodes of level M of the whole tree, and the element offset of that level when the levels
// n, n - 1, ... follow each other.
GBSH_HD int tree_width(int M, int n) { return n - M < 2 ? 1 : 1 << (n - M - 1); }
GBSH_HD size_t tree_offset(int M, int n) {
  size_t off = 0;
  for (int m = n; m > M; --m) off += tree_level_elems(m, n, tree_width(m, n));
  return off;
}

// (j, k), j < k, of polynomial p = k (k - 1) / 2 + j.
GBSH_HD void tree_pair(int p, int& j, int& k) {
#ifdef __CUDA_ARCH__
  k = (int)((1.0f + sqrtf((float)(8 * p + 1))) * 0.5f);
#else
  k = (int)((1.0f + __builtin_sqrtf((float)(8 * p + 1))) * 0.5f);
#endif
  if (k * (k - 1) / 2 > p) --k;
  if (k * (k + 1) / 2 <= p) ++k;
  j = p - k * (k - 1) / 2;
}

// One phase of a node set's way down the tree; its tasks are independent of each other.
//   step    one elimination, level M (src) to level M - 1 (dst): both children of every node
//           x, 2 x with + and 2 x + 1 with -, or (`single`, at the root) the + child alone. The
//           g of src's nodes are made here too, from their parents' (par, one level up), and h
//           of src's nodes: both lag a level so that a level has no chain of products. `psign` =
//           0: src holds both children of each node of par, and `gsel` tells by how many nodes
//           its pointers are past the first; +-1: src is that child of par's one node. At the
//           root (M = n) g is one and has no parent.
//   last1   level 2 (src): w_jk = A_jk + v_j v_k at 8 x + p (p the pair's number), -2 v0 v1 at
//           8 x + 6 and v2 v3 at 8 x + 7, in place of h; and g of the level's nodes.
//   last2   level 2 (src): the products w01 w23, w02 w13, w03 w12, -2 v0 v1 v2 v3 of a node,
//           each multiplied with g: the node's [x^{n-2}] g (...), in parts.
enum TreeKind { kTreeStep, kTreeLast1, kTreeLast2 };
struct TreePhase {
  TreeLevel src, dst, par;
  int kind, n, M, psign, gsel;
  bool single;
};

GBSH_HD int tree_items(const TreePhase& s) {
  if (s.kind == kTreeLast2) return 4 * s.src.q;
  const int g = s.M < s.n ? s.par.q : 0;
  return s.kind == kTreeStep ? s.src.q * (tree_polys(s.M - 1) + 1) + g : 6 * s.src.q + g;
}
GBSH_HD unsigned tree_tasks(const TreePhase& s) {
  return (unsigned)((s.n - s.M + 2) / 2 * tree_items(s));
}

// Runs one task. In phase last2 returns true with a part of node `node`'s term in z.
GBSH_HD bool tree_task(const TreePhase& s, unsigned task, int& node, Fxc& z, unsigned& bad) {
  const int M = s.M, L = s.n - M + 1, q = s.src.q, ld = s.src.ld, r = 2 * M;
  const int items = tree_items(s);
  const int tile = (int)(task / (unsigned)items), it = (int)(task - (unsigned)tile * (unsigned)items);
  int t0 = L - 2 - 2 * tile;  // the costliest coefficients first
  // The task: coefficients t0, t0 + 1 of f0 * f1 (+ f2 * f3), then one of three ends.
  const Fxc *f0, *f1, *f2 = nullptr, *f3 = nullptr;
  int stride;
  enum { kChild, kStore, kDot } end;
  const Fxc* old;      // kChild: the polynomial to which +- x (product) is added; kStore: (product)
  int ostride = 0;
  Fxc* dst = nullptr;
  int dstride = 0, twin = 0;  // kChild: the - child's distance (0: one child, sign `sg`)
  int sg = 1, Lold = L, extra = 0;
  const int nmain = s.kind == kTreeStep ? q * (tree_polys(M - 1) + 1) : 6 * q;
  if (s.kind == kTreeLast2) {
    // pairs (01,23) = (0,5), (02,13) = (1,4), (03,12) = (3,2), then (6,7)
    const int x = it >> 2, c = it & 3;
    stride = ld * 8;
    const Fxc* w = s.src.h + (ptrdiff_t)x * 8;
    f0 = w + (c == 0 ? 0 : (c == 1 ? 1 : (c == 2 ? 3 : 6)));
    f1 = w + (c == 3 ? 7 : (c == 2 ? 2 : 5 - c));
    end = kDot;
    old = s.src.g + x;
    ostride = ld;
    node = x;
  } else if (it >= nmain) {  // g' = g +- x g h of node(s) of src
    const int x = it - nmain;
    --t0;
    if (t0 < -1) return false;
    stride = s.par.ld;
    f0 = s.par.g + x;
    f1 = s.par.h + x;
    end = kChild;
    old = f0;
    ostride = stride;
    Lold = L - 1;
    sg = s.psign;
    twin = s.psign == 0 ? 1 : 0;
    dst = s.psign == 0 ? s.src.g - s.gsel + 2 * x : s.src.g;
    dstride = ld;
  } else {
    const int P = tree_polys(M);
    const int col_a = (r - 2) * (r - 3) / 2, col_b = (r - 1) * (r - 2) / 2, col_v = r * (r - 1) / 2;
    stride = ld * P;
    const int nA = nmain - q;  // phase step
    if (s.kind == kTreeLast1) {
      const int x = it / 6, p = it - 6 * x;
      int j, k;
      tree_pair(p, j, k);
      const Fxc* A = s.src.A + (ptrdiff_t)x * P;
      f0 = A + 6 + j;
      f1 = A + 6 + k;
      end = kStore;
      old = A + p;
      dst = s.src.h + (ptrdiff_t)x * 8 + p;
      dstride = ld * 8;
      extra = p == 0 ? 6 : (p == 5 ? 2 : 0);
    } else if (it < nA) {
      const int Pc = tree_polys(M - 1), rc = r - 2, loop0 = rc * (rc - 1) / 2;
      const int x = it / Pc, p = it - x * Pc;
      const Fxc* A = s.src.A + (ptrdiff_t)x * P;
      int j, k;
      if (p >= loop0) {  // v'_j
        j = p - loop0;
        f1 = A + col_v + r - 1;
        f3 = A + col_v + r - 2;
        old = A + col_v + j;
      } else {
        tree_pair(p, j, k);
        f1 = A + col_b + k;
        f3 = A + col_a + k;
        old = A + p;
      }
      f0 = A + col_a + j;
      f2 = A + col_b + j;
      end = kChild;
      twin = s.single ? 0 : Pc;
      dst = s.dst.A + (ptrdiff_t)(s.single ? x : 2 * x) * Pc + p;
      dstride = s.dst.ld * Pc;
    } else {  // h = A_ab + v_a v_b
      const int x = it - nA;
      const Fxc* A = s.src.A + (ptrdiff_t)x * P;
      f0 = A + col_v + r - 2;
      f1 = A + col_v + r - 1;
      end = kStore;
      old = A + col_b + r - 2;
      dst = s.src.h + x;
      dstride = ld;
    }
    ostride = stride;
  }
  FxAcc acc0 = fx_acc_zero(), acc1 = fx_acc_zero();
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
  for (;;) {
    fx_conv2(acc0, acc1, f0, stride, f1, stride, t0);
    if (!f2) break;
    f0 = f2;
    f1 = f3;
    f2 = nullptr;
  }
  FxAcc dot = fx_acc_zero();
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
  for (int t = t0; t < t0 + 2; ++t) {
    const Fxc v = fx_norm(acc0, bad);
    acc0 = acc1;
    if (t < 0) continue;
    if (end == kChild) {
      Fxc o{};
      if (t + 1 < Lold) o = fx_load(old + (ptrdiff_t)(t + 1) * ostride);
      Fxc* d = dst + (ptrdiff_t)(t + 1) * dstride;
      fx_store(d, fx_add(o, v, twin ? 1 : sg, bad));
      if (twin) fx_store(d + twin, fx_add(o, v, -1, bad));
      if (t == 0) {
        const Fxc c = fx_load(old);
        fx_store(dst, c);
        if (twin) fx_store(dst + twin, c);
      }
    } else if (end == kStore) {
      Fxc* d = dst + (ptrdiff_t)t * dstride;
      fx_store(d, fx_add(fx_load(old + (ptrdiff_t)t * ostride), v, 1, bad));
      if (extra == 2) fx_store(d + extra, v);
      if (extra == 6) {
        const Fxc zero{};
        fx_store(d + extra, fx_add(fx_add(zero, v, -1, bad), v, -1, bad));
      }
    } else {
      fx_mac(dot, v, fx_load(old + (ptrdiff_t)(L - 1 - t) * ostride));
    }
  }
  if (end != kDot) return false;
  z = fx_norm(dot, bad);
  return true;
}

// ------------------------------------------------------------------ cutting the tree
// Step `step` of the breadth-first part (level n - step to n - step - 1) of a tree whose levels
// n, n - 1, ... follow each other from `base`.
GBSH_HD TreePhase tree_step_phase(Fxc* base, int n, int step) {
  TreePhase s;
  const int M = n - step;
  s.kind = kTreeStep;
  s.n = n;
  s.M = M;
  s.src = tree_level(base + tree_offset(M, n), M, n, tree_width(M, n));
  s.dst = tree_level(base + tree_offset(M - 1, n), M - 1, n, tree_width(M - 1, n));
  s.par = s.src;
  if (step > 0) s.par = tree_level(base + tree_offset(M + 1, n), M + 1, n, tree_width(M + 1, n));
  s.single = step == 0;
  s.psign = step == 1 ? 1 : 0;
  s.gsel = 0;
  return s;
}

// A unit: node `unit` of level m1 and all below it, in scratch of tree_scratch elements. Levels
// m1 - 1 .. top are walked depth first and hold the two children of one node each; from level
// `top` on the subtree is worked off breadth first.
GBSH_HD size_t tree_scratch(int n, int m1, int top) {
  size_t e = 0;
  for (int M = m1 - 1; M >= 2; --M) e += tree_level_elems(M, n, M >= top ? 2 : 1 << (top - M));
  return e;
}
GBSH_HD void tree_unit_levels(TreeLevel* lv, Fxc* base, Fxc* scratch, int n, int m1, int top, int unit) {
  lv[m1] = tree_node(tree_level(base + tree_offset(m1, n), m1, n, tree_width(m1, n)), m1, unit);
  if (m1 < n)
    lv[m1 + 1] = tree_node(tree_level(base + tree_offset(m1 + 1, n), m1 + 1, n, tree_width(m1 + 1, n)),
                           m1 + 1, unit >> 1);
  for (int M = m1 - 1; M >= 2; --M) {
    const int q = M >= top ? 2 : 1 << (top - M);
    lv[M] = tree_level(scratch, M, n, q);
    scratch += tree_level_elems(M, n, q);
  }
}
// Phase i (of m1) of walk b (of 2^(m1 - top)). Bit M - top of b tells which child of level M
// the walk is in. Walk b > 0 shares with walk b - 1 the levels above the one whose child
// changes, so it starts at phase tree_first_phase.
GBSH_HD int tree_first_phase(int m1, int top, unsigned b) {
  if (b == 0) return 0;
  int low = 0;
  while (!((b >> low) & 1)) ++low;
  return m1 - top - low;
}
GBSH_HD TreePhase tree_unit_phase(const TreeLevel* lv, int n, int m1, int top, int unit, unsigned b, int i) {
  TreePhase s;
  const int M = m1 - i > 2 ? m1 - i : 2;
  s.n = n;
  s.M = M;
  s.kind = i < m1 - 2 ? kTreeStep : (i < m1 - 1 ? kTreeLast1 : kTreeLast2);
  s.single = M == n;
  s.src = lv[M];
  s.dst = lv[M > 2 ? M - 1 : 2];
  s.par = lv[M < n ? M + 1 : M];
  s.psign = 0;
  s.gsel = 0;
  if (M < m1 && M >= top) {
    s.gsel = (b >> (M - top)) & 1;
    s.src = tree_node(s.src, M, s.gsel);
  }
  if (M + 1 < m1 && M + 1 >= top) s.par = tree_node(s.par, M + 1, (b >> (M + 1 - top)) & 1);
  if (M == m1) s.psign = m1 < n - 1 && (unit & 1) ? -1 : 1;
  return s;
}

}  // namespace gbsh
