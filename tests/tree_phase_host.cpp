// Host build of one elimination step (csrc/lhaf_tree.cuh) on a level that the caller fills, and of
// the rule for cluster sizes. C entries for ctypes.
#include <cmath>
#include <vector>

#include "lhaf_tree.cuh"

using namespace gbsh;

namespace {
Fxc to_fixed(const double* z) {
  Fxc v{};
  for (int c = 0; c < 2; ++c) {
    const __int128 x = (__int128)std::llrint(std::ldexp(z[c], 54)) << (kTreeFrac - 54);
    const __int128 a = x + kLimbHalf, b = (a >> kLimbBits) + kLimbHalf;
    (c ? v.il : v.rl) = ((int)(long long)a & kLimbMask) - kLimbHalf;
    (c ? v.im : v.rm) = ((int)(long long)b & kLimbMask) - kLimbHalf;
    (c ? v.ih : v.rh) = (int)(long long)(b >> kLimbBits);
  }
  return v;
}
double value(int h, int m, int l) {
  return std::ldexp(h, -27) + std::ldexp(m, -54) + std::ldexp(l, -81);
}
struct HostSlot {
  int* m;
  void put(int k, int v) const { m[k] = v; }
  int get(int k) const { return m[k]; }
};
}  // namespace

// src: n - M + 1 coefficients of each of the M (2 M + 1) polynomials of one node of level M of n
// (polynomial p's coefficient t at t polys + p; re, im), whose g and h are zero. dst: the same of
// its + child. Returns whether the step flagged the problem.
extern "C" int tree_host_step(int n, int M, const double* src, double* dst) {
  std::vector<char> a(tree_level_bytes(M, n, 1)), b(tree_level_bytes(M - 1, n, 2)), c(tree_level_bytes(M + 1, n, 1));
  TreePhase s{};
  s.kind = kTreeStep;
  s.n = n;
  s.M = M;
  s.psign = 1;
  s.src_bit = s.par_bit = -1;
  s.src = tree_level(a.data(), M, n, 1);
  s.dst = tree_level(b.data(), M - 1, n, 2);
  s.par = tree_level(c.data(), M + 1, n, 1);
  tree_ready(s);
  const int L = n - M + 1, P = tree_polys(M), Pc = tree_polys(M - 1);
  for (int t = 0; t < L; ++t)
    for (int p = 0; p < P; ++p) fx_store(s.src.A + t * s.src.sA + fx_at(p), to_fixed(src + 2 * (t * P + p)));
  unsigned bad = 0;
  int node, ints[kSlotInts];
  Fxc z;
  for (int t = 0; t < s.tasks; ++t) tree_task(s, 0, t, HostSlot{ints}, node, z, bad);
  for (int t = 0; t <= L; ++t)
    for (int p = 0; p < Pc; ++p) {
      const Fxc v = fx_load(s.dst.A + t * s.dst.sA + fx_at(p));
      dst[2 * (t * Pc + p)] = value(v.rh, v.rm, v.rl);
      dst[2 * (t * Pc + p) + 1] = value(v.ih, v.im, v.il);
    }
  return bad ? 1 : 0;
}

extern "C" int tree_host_cluster(int n, int count, int slots, int most) { return tree_cluster(n, count, slots, most); }
