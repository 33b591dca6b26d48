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
// (N = 40: 1.0e9 against 1.1e10, 4.7 ms against 184), and the signed mean cancels by 10^2..10^4 where the signed
// subset sum cancels by 10^7..10^12.
//
// Arithmetic. Products of polynomials are sums of products with no division, so they run in
// fixed point: a real number is an integer times 2^-81, held as three limbs with signs,
// h 2^54 + m 2^27 + l, |m|, |l| <= 2^26, |h| < 2^29. The limb products of a whole convolution
// add up in 64 bits, so it accumulates exactly and is normalised once. Six limb products per real
// product (the three below 2^-81 are dropped) and three real products per complex one (Gauss) make
// 18 32x32+64-bit integer multiply-adds per complex one: 0.45e12 complex multiply-adds/s with
// operands from L1, against 0.17e12/s at best for triple-float (216 FP32 instructions) and
// 0.15e12/s for FP64. (The integer multiply-add issues every 2 cycles when it repeats its
// operands, 18.7e12/s, and every 4.4 in this code: its operand fetch is the limit.) Fixed point
// needs a scale: each vertex gets one, such that the root-mean-fourth singular value of the matrix is
// about one and no loop weight stands out (tree_root, lhaf_tree.cu). The coefficients of configuration
// matrices then stay below 2.4 up to N = 32 and below 3.4 up to N = 50; the format holds |x| < 4,
// long levels a little less (fx_limit). Overflow anywhere, or a result so small that the resolution could
// show, sets a flag and the caller evaluates the problem by the subset sum instead: strongly graded
// matrices, and from N = 26 on loop weights well above the entries (up to a seventh of them at N = 28, half at
// N = 32, where weights of one phase and those above 1 come out too small).
//
// The code of one level is a function of (level, task number) that reads the level's nodes
// and writes the next level's, so it compiles for the host as well and is checked there
// against the definition.
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

constexpr int kTreeFrac = 81;  // value = integer * 2^-81
constexpr int kLimbBits = 27;
constexpr int kLimbHalf = 1 << (kLimbBits - 1);
constexpr int kLimbMask = (1 << kLimbBits) - 1;

// A complex fixed-point number: limbs of the real and the imaginary part.
struct Fxc {
  int rh, rm, rl, ih, im, il;
};

// In memory a row of numbers lies in blocks of 32: 32 (rh, rm), 32 (rl, ih), 32 (im, il) pairs.
// A warp that reads 32 neighbours then takes three 256-byte runs, where 24- or 32-byte
// structures cost it five times the L1 wavefronts. Numbers are addressed by bytes.
GBSH_HD constexpr int fx_at(int i) { return (i >> 5) * 768 + (i & 31) * 8; }
GBSH_HD constexpr int fx_row(int count) { return ((count + 31) >> 5) * 768; }

GBSH_HD Fxc fx_load(const char* p) {
#ifdef __CUDA_ARCH__
  const int2 a = *reinterpret_cast<const int2*>(p), b = *reinterpret_cast<const int2*>(p + 256),
             c = *reinterpret_cast<const int2*>(p + 512);
  return Fxc{a.x, a.y, b.x, b.y, c.x, c.y};
#else
  const int *a = reinterpret_cast<const int*>(p), *b = a + 64, *c = a + 128;
  return Fxc{a[0], a[1], b[0], b[1], c[0], c[1]};
#endif
}
GBSH_HD void fx_store(char* p, const Fxc& v) {
#ifdef __CUDA_ARCH__
  *reinterpret_cast<int2*>(p) = make_int2(v.rh, v.rm);
  *reinterpret_cast<int2*>(p + 256) = make_int2(v.rl, v.ih);
  *reinterpret_cast<int2*>(p + 512) = make_int2(v.im, v.il);
#else
  int *a = reinterpret_cast<int*>(p), *b = a + 64, *c = a + 128;
  a[0] = v.rh, a[1] = v.rm, b[0] = v.rl, b[1] = v.ih, c[0] = v.im, c[1] = v.il;
#endif
}

// 64-bit limb-product sums of one complex number, by weight: s2 2^108, s1 2^81, s0 2^54 (in units
// of 2^-162).
struct FxSum {
  long long s2r, s1r, s0r, s2i, s1i, s0i;
};
// Such sums while they grow: p = sum of re re, q = sum of im im, t = sum of (re + im) (re + im),
// from which re = p - q and im = t - p - q (Gauss): 18 multiply-adds a complex product instead of
// 24. The products alone run at 450 against 350 G complex multiply-adds/s; with it N = 40 took
// 4.72 ms instead of 5.00. t may wrap in 64 bits; the differences fit. The sums start at
// half a unit of the next limb, which turns the cuts in fx_norm into roundings to the nearest.
struct FxAcc {
  long long p2, p1, p0, q2, q1, q0, t2, t1, t0;
};
GBSH_HD FxAcc fx_acc_empty() { return FxAcc{0, 0, 0, 0, 0, 0, 0, 0, 0}; }
GBSH_HD FxAcc fx_acc_zero() {
  return FxAcc{kLimbHalf, kLimbHalf, kLimbHalf, 0, 0, 0, 2 * kLimbHalf, 2 * kLimbHalf, 2 * kLimbHalf};
}
GBSH_HD long long fx_wrap(unsigned long long x) { return (long long)x; }
GBSH_HD FxSum fx_sum(const FxAcc& s) {
  typedef unsigned long long u;
  return FxSum{s.p2 - s.q2, s.p1 - s.q1, s.p0 - s.q0, fx_wrap((u)s.t2 - (u)s.p2 - (u)s.q2),
               fx_wrap((u)s.t1 - (u)s.p1 - (u)s.q1), fx_wrap((u)s.t0 - (u)s.p0 - (u)s.q0)};
}
GBSH_HD void fx_wide(long long& s, int a, int b) {
  s = (long long)((unsigned long long)s + (unsigned long long)((long long)a * b));
}
// (s2, s1, s0) += a b of two real numbers. The limb products of weight 2^27 and 1 are below the
// result's resolution.
GBSH_HD void fx_mac1(long long& s2, long long& s1, long long& s0, int ah, int am, int al, int bh, int bm, int bl) {
  fx_wide(s2, ah, bh);
  fx_wide(s1, ah, bm);
  fx_wide(s0, ah, bl);
  fx_wide(s1, am, bh);
  fx_wide(s0, am, bm);
  fx_wide(s0, al, bh);
}
GBSH_HD void fx_mac(FxAcc& s, const Fxc& a, const Fxc& b) {
  fx_mac1(s.p2, s.p1, s.p0, a.rh, a.rm, a.rl, b.rh, b.rm, b.rl);
  fx_mac1(s.q2, s.q1, s.q0, a.ih, a.im, a.il, b.ih, b.im, b.il);
  fx_mac1(s.t2, s.t1, s.t0, a.rh + a.ih, a.rm + a.im, a.rl + a.il, b.rh + b.ih, b.rm + b.im, b.rl + b.il);
}

// Range checks set the sign bit of `over`: three instructions each, and they run on every number
// (with the limit in a register N = 32 takes 1 % longer than with a constant 4, N = 44 4 % less).
GBSH_HD void fx_check(int h, int lim, unsigned& over) {
  over |= ((unsigned)lim - (unsigned)h) | ((unsigned)lim + (unsigned)h);  // |h| > lim
}

// The accumulated real number rounded to the format: s2 2^27 + s1 + s0 2^-27; `over` if |x| >= 4. s2
// wraps at |x| = 512, so a sum is told from one below 4 as long as it is below 1020: see fx_limit.
GBSH_HD void fx_norm1(long long s2, long long s1, long long s0, int& h, int& m, int& l, unsigned& over) {
  const long long t = s1 + (s0 >> kLimbBits);
  l = ((int)t & kLimbMask) - kLimbHalf;
  const long long v = s2 + (t >> kLimbBits);
  m = ((int)v & kLimbMask) - kLimbHalf;
  h = (int)(v >> kLimbBits);
  fx_check((int)(v >> 32), (1 << 24) - 1, over);
}
GBSH_HD Fxc fx_norm(const FxSum& s, unsigned& over) {
  Fxc r;
  fx_norm1(s.s2r, s.s1r, s.s0r, r.rh, r.rm, r.rl, over);
  fx_norm1(s.s2i, s.s1i, s.s0i, r.ih, r.im, r.il, over);
  return r;
}

// Largest |h| of a number that a level of L coefficients may hold. A coefficient of its products
// is a sum of up to 2 L complex products (two factors' pairs), 4 L real ones in each part, which
// stays below the 1020 that fx_norm1 needs if the numbers are below sqrt(255 / L): 4 up to 15
// coefficients (N = 34), then less, 3.57 at N = 44 (where a configuration matrix was seen to reach
// 3.31), 3.02 at N = 60. Level 2's numbers enter single products and may be as large as 4 at any length.
constexpr int kFxLimitFree = 15;  // coefficients up to which it is 4
constexpr int kFxLimit = (4 << (kTreeFrac - 2 * kLimbBits)) - 1;
GBSH_HD int fx_limit(int L) {
  constexpr int kOne = 1 << (kTreeFrac - 2 * kLimbBits);
  if (L <= kFxLimitFree) return kFxLimit;
#ifdef __CUDA_ARCH__
  return (int)(sqrtf(255.0f / (float)L) * (float)kOne) - 64;  // 64: roundings of the root
#else
  return (int)(__builtin_sqrtf(255.0f / (float)L) * (float)kOne) - 64;
#endif
}

// (h, m, l) from limbs with carries to propagate; `over` if |h| > lim.
GBSH_HD void fx_carry(int xh, int xm, int xl, int& h, int& m, int& l, int lim, unsigned& over) {
  const int a = xl + kLimbHalf;
  l = (a & kLimbMask) - kLimbHalf;
  const int b = xm + kLimbHalf + (a >> kLimbBits);
  m = (b & kLimbMask) - kLimbHalf;
  h = xh + (b >> kLimbBits);
  fx_check(h, lim, over);
}
GBSH_HD Fxc fx_add(const Fxc& a, const Fxc& b, int lim, unsigned& over) {
  Fxc r;
  fx_carry(a.rh + b.rh, a.rm + b.rm, a.rl + b.rl, r.rh, r.rm, r.rl, lim, over);
  fx_carry(a.ih + b.ih, a.im + b.im, a.il + b.il, r.ih, r.im, r.il, lim, over);
  return r;
}
GBSH_HD Fxc fx_sub(const Fxc& a, const Fxc& b, int lim, unsigned& over) {
  Fxc r;
  fx_carry(a.rh - b.rh, a.rm - b.rm, a.rl - b.rl, r.rh, r.rm, r.rl, lim, over);
  fx_carry(a.ih - b.ih, a.im - b.im, a.il - b.il, r.ih, r.im, r.il, lim, over);
  return r;
}

// acc0, acc1 += coefficients t0, t0 + 1 of the polynomial product a * b, coefficient u at a + u sa
// and b + u sb; t0 = -1 leaves acc0 alone. t0 + 1 must not exceed the last coefficient of either
// factor. Two coefficients a task: each step loads one new element of each factor for two
// multiply-adds (b in a sliding window of two, a one step ahead of its use). Four would halve the
// loads, but with the accumulators of four the code spilled and outgrew the instruction cache
// (N = 40: 9.0 ms against 5.7 ms). Bound by how fast the register file feeds the 64-bit
// multiply-adds: one a warp and 4.4 cycles, not the 2 of a chain on fixed registers, whatever the
// order of operands or the pairing of registers.
GBSH_HD void fx_conv2(FxAcc& acc0, FxAcc& acc1, const char* a, int sa, const char* b, int sb, int t0) {
  b += (ptrdiff_t)(t0 + 1) * sb;
  Fxc w1 = fx_load(b), x = fx_load(a), w0{};
  int u = t0 + 1;  // steps before the last one
  if (u > 0) {
    b -= sb;
    w0 = fx_load(b);
    if (u & 1) {
      a += sa;
      const Fxc y = fx_load(a);
      fx_mac(acc0, x, w0);
      fx_mac(acc1, x, w1);
      x = y;
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
      a += sa;
      const Fxc y = fx_load(a);
      fx_mac(acc1, x, w1);
      b -= sb;
      w1 = fx_load(b);
      fx_mac(acc0, x, w0);
      a += sa;
      x = fx_load(a);
      fx_mac(acc1, y, w0);
      if (u > 1) {
        b -= sb;
        w0 = fx_load(b);
      }
      fx_mac(acc0, y, w1);
    }
  }
  fx_mac(acc1, x, w1);
}

// ------------------------------------------------------------------ levels of the tree
// Level M holds nodes with M pairs left: r = 2M vertices, L = n - M + 1 coefficients per
// polynomial. A node's polynomials are the A_jk, j < k < r, at k (k - 1) / 2 + j (so that
// eliminating the last pair leaves the others in place) and the loop weights v_j at
// r (r - 1) / 2 + j: P(M) in all. Coefficient u of the polynomials of all nodes is a row, number
// x P + p of it belongs to node x; the rows of g and of h = A_ab + v_a v_b (of the pair that is
// eliminated next) have one number per node.
GBSH_HD constexpr int tree_polys(int M) { return M * (2 * M + 1); }

struct TreeLevel {
  char* A;           // row 0 of the A_jk and v_j
  int g, h;          // bytes from there to the rows of g and h
  int sA, sg, sh;    // bytes from row to row
  int q, x0;         // nodes x0 .. x0 + q - 1
};

// Level 2 holds the eight w and v v polynomials per node in place of h.
GBSH_HD size_t tree_level_bytes(int M, int n, int q) {
  return (size_t)(n - M + 1) * (fx_row(q * tree_polys(M)) + fx_row(q) + fx_row(M == 2 ? 8 * q : q));
}
GBSH_HD TreeLevel tree_level(char* base, int M, int n, int q) {
  const int L = n - M + 1;
  TreeLevel v;
  v.sA = fx_row(q * tree_polys(M));
  v.sg = fx_row(q);
  v.sh = fx_row(M == 2 ? 8 * q : q);
  v.A = base;
  v.g = L * v.sA;
  v.h = v.g + L * v.sg;
  v.q = q;
  v.x0 = 0;
  return v;
}
// Node x of a level as a level of one node.
GBSH_HD TreeLevel tree_node(TreeLevel v, int x) {
  v.x0 += x;
  v.q = 1;
  return v;
}
// Nodes of level M of the whole tree, and the byte offset of that level when the levels
// n, n - 1, ... follow each other.
GBSH_HD int tree_width(int M, int n) { return n - M < 2 ? 1 : 1 << (n - M - 1); }
GBSH_HD size_t tree_offset(int M, int n) {
  size_t off = 0;
  for (int m = n; m > M; --m) off += tree_level_bytes(m, n, tree_width(m, n));
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

// a / b for 0 <= a < 2^23, b > 0, inv = 1 / b in single precision.
GBSH_HD int tree_div(int a, int b, float inv) {
  int x = (int)((float)a * inv);
  if (x * b > a) --x;
  if ((x + 1) * b <= a) ++x;
  return x;
}

// One phase of a node set's way down the tree; its tasks are independent of each other.
//   step    one elimination, level M (src) to level M - 1 (dst): both children of every node
//           x, 2 x with + and 2 x + 1 with -, or (`single`, at the root) the + child alone. The
//           g of src's nodes are made here too, from their parents' (par, one level up), and h
//           of src's nodes: both lag a level so that a level has no chain of products. `psign` =
//           0: src's storage holds both children of each node of par; +-1: src is that child of
//           par's one node. At the root (M = n) g is one and has no parent.
//   last1   level 2 (src): w_jk = A_jk + v_j v_k at 8 x + p (p the pair's number), -2 v0 v1 at
//           8 x + 6 and v2 v3 at 8 x + 7, in place of h; and g of the level's nodes.
//   last2   level 2 (src): the products w01 w23, w02 w13, w03 w12, -2 v0 v1 v2 v3 of a node,
//           each multiplied with g: the node's [x^{n-2}] g (...), in parts.
enum TreeKind { kTreeStep, kTreeLast1, kTreeLast2 };
struct TreePhase {
  TreeLevel src, dst, par;
  int kind, n, M, psign;
  bool single;
  int src_bit, par_bit;  // a level walked depth first: its node is this bit of the walk's number;
                         // -1: its nodes are those of src and par
  // set by tree_ready
  int nmain, items, tasks, lim;
  float inv_items, inv_node;
};

// A task makes coefficients in twos: a tile near the top and its mirror tile near the bottom of
// an item's triangle of products, so that all tasks of a phase cost the same.
// kShort: n is at most kFxLimitFree, and the limit is known without the root's code.
template <bool kShort = false>
GBSH_HD void tree_ready(TreePhase& s) {
  const int L = s.n - s.M + 1, g = s.M < s.n ? s.par.q : 0;
  const int per = s.kind == kTreeStep ? tree_polys(s.M - 1) : (s.kind == kTreeLast1 ? 6 : 4);
  s.nmain = s.src.q * (s.kind == kTreeStep ? per + 1 : per);
  s.items = s.nmain + (s.kind == kTreeLast2 ? 0 : g);
  s.tasks = ((L + 1) / 2 + 1) / 2 * s.items;
  s.lim = kShort ? kFxLimit : fx_limit(s.kind == kTreeStep && s.M > 3 ? L + 1 : 0);
  s.inv_items = 1.0f / (float)s.items;
  s.inv_node = 1.0f / (float)per;
}

// An item of a phase: the products f0 * f1 (+ g0 * g1) and what becomes of them. Byte offsets
// from fb and db instead of pointers: the accumulators leave few registers.
enum TreeEnd { kChild, kStore, kDot };
struct TreeJob {
  const char* fb;
  char* db;
  int f0, f1, g0, g1;  // factors; g0 < 0: one product
  int sa, sb;          // row strides of the factors
  TreeEnd end;
  int old, so;         // kChild: the polynomial to which +- x (product) is added; kStore: (product)
  int dst, twin, sd;   // kChild: the + and the - child (or one, the - child if `neg`)
  int top, last;       // two below the number of coefficients; last coefficient of `old`
  int lim;             // fx_limit of what is stored
  int node;
  bool neg;
};
GBSH_HD TreeJob tree_job(const TreePhase& s, unsigned walk, int it) {
  const int xs = s.src_bit < 0 ? s.src.x0 : (int)(walk >> s.src_bit) & 1;
  const int L = s.n - s.M + 1;
  TreeJob J;
  J.fb = s.src.A;
  J.db = s.src.A;
  J.g0 = J.g1 = -1;
  J.dst = 0;
  J.twin = -1;
  J.sd = 0;
  J.top = L - 2;
  J.last = L - 1;
  J.lim = s.lim;
  J.neg = false;
  J.node = 0;
  if (s.kind == kTreeLast2) {
    // pairs (01,23) = (0,5), (02,13) = (1,4), (03,12) = (3,2), then (6,7)
    const int x = it >> 2, c = it & 3, at = 8 * (xs + x);
    J.sa = J.sb = s.src.sh;
    J.f0 = s.src.h + fx_at(at + (c == 0 ? 0 : (c == 1 ? 1 : (c == 2 ? 3 : 6))));
    J.f1 = s.src.h + fx_at(at + (c == 3 ? 7 : (c == 2 ? 2 : 5 - c)));
    J.end = kDot;
    J.old = s.src.g + fx_at(xs + x);
    J.so = s.src.sg;
    J.node = x;
  } else if (it >= s.nmain) {  // g' = g +- x g h of node(s) of src
    const int x = it - s.nmain;
    const int xp = (s.par_bit < 0 ? s.par.x0 : (int)(walk >> s.par_bit) & 1) + x;
    J.fb = s.par.A;
    --J.top;
    --J.last;
    J.sa = J.so = s.par.sg;
    J.sb = s.par.sh;
    J.f0 = J.old = s.par.g + fx_at(xp);
    J.f1 = s.par.h + fx_at(xp);
    J.end = kChild;
    J.neg = s.psign < 0;
    J.dst = s.src.g + fx_at(s.psign == 0 ? 2 * x : xs + x);
    if (s.psign == 0) J.twin = s.src.g + fx_at(2 * x + 1);
    J.sd = s.src.sg;
  } else {
    const int M = s.M, r = 2 * M, P = tree_polys(M);
    const int col_a = (r - 2) * (r - 3) / 2, col_b = (r - 1) * (r - 2) / 2, col_v = r * (r - 1) / 2;
    J.sa = J.sb = J.so = s.src.sA;
    const int nA = s.nmain - s.src.q;  // phase step
    if (s.kind == kTreeLast1) {
      const int x = tree_div(it, 6, s.inv_node), p = it - 6 * x, at = (xs + x) * P;
      int j, k;
      tree_pair(p, j, k);
      J.f0 = fx_at(at + 6 + j);
      J.f1 = fx_at(at + 6 + k);
      J.end = kStore;
      J.old = fx_at(at + p);
      const int w = 8 * (xs + x);
      J.dst = s.src.h + fx_at(w + p);
      J.sd = s.src.sh;
      if (p == 0) J.twin = s.src.h + fx_at(w + 6);
      if (p == 5) J.twin = s.src.h + fx_at(w + 7);
      J.neg = p == 0;
    } else if (it < nA) {
      const int Pc = tree_polys(M - 1), rc = r - 2, loop0 = rc * (rc - 1) / 2;
      const int x = tree_div(it, Pc, s.inv_node), p = it - x * Pc, at = (xs + x) * P;
      int j, ka, kb, o = p;
      if (p >= loop0) {  // v'_j
        j = p - loop0;
        ka = col_v + r - 2;
        kb = col_v + r - 1;
        o = col_v + j;
      } else {
        int k;
        tree_pair(p, j, k);
        ka = col_a + k;
        kb = col_b + k;
      }
      J.f0 = fx_at(at + col_a + j);
      J.f1 = fx_at(at + kb);
      J.g0 = fx_at(at + col_b + j);
      J.g1 = fx_at(at + ka);
      J.old = fx_at(at + o);
      J.end = kChild;
      J.db = s.dst.A;
      const int c = (s.single ? x : 2 * x) * Pc + p;  // the children's storage starts at node 0
      J.dst = fx_at(c);
      if (!s.single) J.twin = fx_at(c + Pc);
      J.sd = s.dst.sA;
    } else {  // h = A_ab + v_a v_b
      const int x = it - nA, at = (xs + x) * P;
      J.f0 = fx_at(at + col_v + r - 2);
      J.f1 = fx_at(at + col_v + r - 1);
      J.end = kStore;
      J.old = fx_at(at + col_b + r - 2);
      J.dst = s.src.h + fx_at(xs + x);
      J.sd = s.src.sh;
    }
  }
  return J;
}

// What becomes of coefficient t of the product.
GBSH_HD void tree_end(const TreeJob& J, int t, const Fxc& v, unsigned& over) {
  if (J.end == kChild) {
    Fxc o{};
    if (t < J.last) o = fx_load(J.fb + J.old + (ptrdiff_t)(t + 1) * J.so);
    char* d = J.db + (ptrdiff_t)(t + 1) * J.sd;
    if (!J.neg) fx_store(d + J.dst, fx_add(o, v, J.lim, over));
    if (J.twin >= 0 || J.neg) fx_store(d + (J.neg ? J.dst : J.twin), fx_sub(o, v, J.lim, over));
    if (t == 0) {
      const Fxc c = fx_load(J.fb + J.old);
      fx_store(J.db + J.dst, c);
      if (J.twin >= 0) fx_store(J.db + J.twin, c);
    }
  } else {
    char* d = J.db + (ptrdiff_t)t * J.sd;
    fx_store(d + J.dst, fx_add(fx_load(J.fb + J.old + (ptrdiff_t)t * J.so), v, J.lim, over));
    if (J.twin >= 0) {
      const Fxc zero{};
      fx_store(d + J.twin, J.neg ? fx_sub(fx_sub(zero, v, J.lim, over), v, J.lim, over) : v);
    }
  }
}

// The same in four independent parts, and the number that a part starts from.
GBSH_HD Fxc tree_end_old(const TreeJob& J, int t, int role) {
  if (J.end == kDot) return role == 0 ? fx_load(J.fb + J.old + (ptrdiff_t)(J.last - t) * J.so) : Fxc{};
  if (J.end == kStore) return role == 0 ? fx_load(J.fb + J.old + (ptrdiff_t)t * J.so) : Fxc{};
  if (role < 2) return t < J.last ? fx_load(J.fb + J.old + (ptrdiff_t)(t + 1) * J.so) : Fxc{};
  return t == 0 ? fx_load(J.fb + J.old) : Fxc{};
}
GBSH_HD void tree_end_part(const TreeJob& J, int t, int role, const Fxc& o, const Fxc& v, unsigned& over) {
  if (J.end == kStore) {
    char* d = J.db + (ptrdiff_t)t * J.sd;
    if (role == 0) {
      fx_store(d + J.dst, fx_add(o, v, J.lim, over));
    } else if (role == 1 && J.twin >= 0) {
      const Fxc zero{};
      fx_store(d + J.twin, J.neg ? fx_sub(fx_sub(zero, v, J.lim, over), v, J.lim, over) : v);
    }
    return;
  }
  char* d = J.db + (ptrdiff_t)(t + 1) * J.sd;
  if (role < 2) {
    if (role == 1 && J.twin < 0) return;
    if (role == 0 && !J.neg) fx_store(d + J.dst, fx_add(o, v, J.lim, over));
    else fx_store(d + (role == 0 ? J.dst : J.twin), fx_sub(o, v, J.lim, over));
  } else if (t == 0 && (role == 2 || J.twin >= 0)) {
    fx_store(J.db + (role == 2 ? J.dst : J.twin), o);
  }
}

// A task's work in pieces for phases with few items: piece `sub` (of four) of coefficient t of
// item `it`, a quarter of its products. The four sums are added (by the caller: exactly, they are
// integers) before tree_end_part.
GBSH_HD FxSum tree_piece(const TreeJob& J, int t, int sub) {
  FxAcc acc = fx_acc_empty();
  if (sub == 0) acc = fx_acc_zero();
  if (t > J.top + 1) return fx_sum(acc);
  const bool two = J.g0 >= 0;
  const int u0 = two ? sub >> 1 : sub, du = two ? 2 : 4;
  const char* a = J.fb + (two && (sub & 1) ? J.g0 : J.f0) + (ptrdiff_t)u0 * J.sa;
  const char* b = J.fb + (two && (sub & 1) ? J.g1 : J.f1) + (ptrdiff_t)(t - u0) * J.sb;
#ifdef __CUDA_ARCH__
#pragma unroll 4
#endif
  for (int u = u0; u <= t; u += du) {
    fx_mac(acc, fx_load(a), fx_load(b));
    a += (ptrdiff_t)du * J.sa;
    b -= (ptrdiff_t)du * J.sb;
  }
  return fx_sum(acc);
}
GBSH_HD int tree_pieces(const TreePhase& s) { return (s.n - s.M + 1) * s.items * 4; }

// The parts of a job that a task does not need during its products, kept outside the registers
// (on the GPU in shared memory, a column per thread): two FxAcc and three operands with their
// sums take 63 of the 96 registers that 640 threads an SM leave.
constexpr int kSlotInts = 11;
template <class Slot>
GBSH_HD void tree_put(const Slot& m, const TreeJob& J) {
  const long long db = (long long)(size_t)J.db;
  m.put(0, (int)db);
  m.put(1, (int)(db >> 32));
  m.put(2, J.g0);
  m.put(3, J.g1);
  m.put(4, J.old);
  m.put(5, J.so);
  m.put(6, J.dst);
  m.put(7, J.twin);
  m.put(8, J.sd);
  m.put(9, J.last);
  m.put(10, (int)J.end + (J.neg ? 4 : 0));
}
template <class Slot>
GBSH_HD TreeJob tree_get(const Slot& m, const char* fb, int lim) {
  TreeJob J;
  J.fb = fb;
  J.lim = lim;
  J.db = (char*)(size_t)((unsigned long long)(unsigned)m.get(0) | (unsigned long long)(unsigned)m.get(1) << 32);
  J.old = m.get(4);
  J.so = m.get(5);
  J.dst = m.get(6);
  J.twin = m.get(7);
  J.sd = m.get(8);
  J.last = m.get(9);
  const int e = m.get(10);
  J.end = (TreeEnd)(e & 3);
  J.neg = (e & 4) != 0;
  J.f0 = J.f1 = J.g0 = J.g1 = J.sa = J.sb = J.top = J.node = 0;
  return J;
}

// Runs one task of walk `walk`. In phase last2 returns true with a part of node `node`'s term in
// z (sums of limbs, carries not propagated). bad: 0, or 1 once a number left the range. kShort: n is
// at most kFxLimitFree, and the limit is known without the phase.
template <bool kShort = false, class Slot>
GBSH_HD bool tree_task(const TreePhase& s, unsigned walk, int task, const Slot& slot, int& node, Fxc& z,
                       unsigned& bad) {
  int tile = tree_div(task, s.items, s.inv_items);
  const char* fb;
  int f0, f1, sa, sb, top;
  {
    const TreeJob J = tree_job(s, walk, task - tile * s.items);
    tree_put(slot, J);
    node = J.node;
    fb = J.fb;
    f0 = J.f0;
    f1 = J.f1;
    sa = J.sa;
    sb = J.sb;
    top = J.top;
  }
  z = Fxc{};
  unsigned& over = bad;  // one register: the sign bit until the end of the task
  bad <<= 31;
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
  for (int side = 0;; ++side) {
    const int t0 = top - 2 * tile;
    if (t0 >= -1) {
      FxAcc acc0 = fx_acc_zero(), acc1 = fx_acc_zero();
      int a = f0, b = f1;
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
      for (int c = 0;; ++c) {
        fx_conv2(acc0, acc1, fb + a, sa, fb + b, sb, t0);
        if (c) break;
        a = slot.get(2);
        b = slot.get(3);
        if (a < 0) break;
      }
      FxSum sum = fx_sum(acc0);
      const FxSum sum1 = fx_sum(acc1);
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
      for (int t = t0; t < t0 + 2; ++t) {
        const Fxc v = fx_norm(sum, over);
        sum = sum1;
        if (t < 0) continue;
        const TreeJob J = tree_get(slot, fb, kShort ? kFxLimit : s.lim);
        if (J.end == kDot) {
          FxAcc dot = fx_acc_zero();
          fx_mac(dot, v, fx_load(fb + J.old + (ptrdiff_t)(J.last - t) * J.so));
          const Fxc part = fx_norm(fx_sum(dot), over);
          z = Fxc{z.rh + part.rh, z.rm + part.rm, z.rl + part.rl, z.ih + part.ih, z.im + part.im, z.il + part.il};
        } else {
          tree_end(J, t, v, over);
        }
      }
    }
    const int tiles = (s.n - s.M + 2) / 2, mirror = tiles - 1 - tile;
    if (side == 1 || mirror == tile) break;
    tile = mirror;
  }
  bad >>= 31;
  return s.kind == kTreeLast2;
}

// ------------------------------------------------------------------ cutting the tree
// Phase i of n of the whole tree breadth first; its levels n, n - 1, ... follow each other from
// `base`.
template <bool kShort = false>
GBSH_HD TreePhase tree_whole_phase(char* base, int n, int i) {
  TreePhase s;
  const int M = n - i > 2 ? n - i : 2;
  const int up = M < n ? M + 1 : M, down = M > 2 ? M - 1 : 2;
  s.src = tree_level(base + tree_offset(M, n), M, n, tree_width(M, n));
  s.dst = tree_level(base + tree_offset(down, n), down, n, tree_width(down, n));
  s.par = tree_level(base + tree_offset(up, n), up, n, tree_width(up, n));
  s.kind = i < n - 2 ? kTreeStep : (i == n - 2 ? kTreeLast1 : kTreeLast2);
  s.n = n;
  s.M = M;
  s.single = i == 0 && n > 2;
  s.psign = M == n - 1 ? 1 : 0;
  s.src_bit = s.par_bit = -1;
  tree_ready<kShort>(s);
  return s;
}

// CTAs of a cluster that works off whole trees of n pairs, of `count` problems: as many as the widest
// levels can use, at most `most` (what the device can hold), and so few that `count` clusters
// need no more than `slots` CTAs.
GBSH_HD int tree_cluster(int n, int count, int slots, int most) {
  int c = n <= 3 ? 1 : (n <= 4 ? 4 : (n <= 6 ? 8 : 16));
  while (c > 1 && (c > most || (long long)count * c > slots)) c >>= 1;
  return c;
}

// A unit: node `unit` of level m1 and all below it, in scratch of tree_scratch bytes. Levels
// m1 - 1 .. top are walked depth first and hold the two children of one node each; from level
// `top` on the subtree is worked off breadth first.
GBSH_HD size_t tree_scratch(int n, int m1, int top) {
  size_t e = 0;
  for (int M = m1 - 1; M >= 2; --M) e += tree_level_bytes(M, n, M >= top ? 2 : 1 << (top - M));
  return e;
}
GBSH_HD void tree_unit_levels(TreeLevel* lv, char* base, char* scratch, int n, int m1, int top, int unit) {
  lv[m1] = tree_node(tree_level(base + tree_offset(m1, n), m1, n, tree_width(m1, n)), unit);
  if (m1 < n)
    lv[m1 + 1] = tree_node(tree_level(base + tree_offset(m1 + 1, n), m1 + 1, n, tree_width(m1 + 1, n)), unit >> 1);
  for (int M = m1 - 1; M >= 2; --M) {
    const int q = M >= top ? 2 : 1 << (top - M);
    lv[M] = tree_level(scratch, M, n, q);
    scratch += tree_level_bytes(M, n, q);
  }
}
// The unit is worked off in walks b = 0 .. 2^(m1 - top) - 1 of m1 phases each. Bit M - top of b
// tells which child of level M the walk is in. Walk b > 0 shares with walk b - 1 the levels above
// the one whose child changes, so it starts at phase tree_first_phase.
GBSH_HD int tree_first_phase(int m1, int top, unsigned b) {
  if (b == 0) return 0;
  int low = 0;
  while (!((b >> low) & 1)) ++low;
  return m1 - top - low;
}
GBSH_HD TreePhase tree_unit_phase(const TreeLevel* lv, int n, int m1, int top, int unit, int i) {
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
  s.src_bit = s.par_bit = -1;
  if (M < m1 && M >= top) {
    s.src_bit = M - top;
    s.src.q = 1;
  }
  if (M + 1 < m1 && M + 1 >= top) {
    s.par_bit = M + 1 - top;
    s.par.q = 1;
  }
  if (M == m1) s.psign = m1 < n - 1 && (unit & 1) ? -1 : 1;
  tree_ready(s);
  return s;
}

}  // namespace gbsh
