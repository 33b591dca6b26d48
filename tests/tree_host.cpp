// Host build of the elimination tree (csrc/lhaf_tree.cuh): the same level code as the GPU
// kernels, driven serially, with the limb sums in 128-bit integers. C entry for ctypes.
#include <cmath>
#include <cstdlib>
#include <vector>

#include "lhaf_tree.cuh"

using namespace gbsh;

namespace {
void to_fixed(double x, int m, int e, int& h, int& mm, int& l) {  // x m 2^e
  int ex;
  const double f = std::frexp(x, &ex);
  __int128 v = (__int128)((long long)std::ldexp(f, 53)) * m;
  const int sh = ex - 53 + e + kTreeFrac;
  if (sh >= 0) v <<= sh;
  else if (sh < -100) v = 0;
  else v = (v + ((__int128)1 << (-sh - 1))) >> (-sh);
  l = sext28((long long)v);
  v = (v - l) >> kLimbBits;
  mm = sext28((long long)v);
  v = (v - mm) >> kLimbBits;
  h = (int)v;
}

// Guarded storage: a level's elements and a canary on each side.
struct Guarded {
  std::vector<Fxc> mem;
  explicit Guarded(size_t n) : mem(n + 64, Fxc{7, 7, 7, 7, 7, 7, 7, 7}) {}
  Fxc* data() { return mem.data() + 32; }
  bool intact() const {
    for (int i = 0; i < 32; ++i)
      if (mem[i].rh != 7 || mem[mem.size() - 1 - i].rh != 7 || mem[i].il != 7 || mem[mem.size() - 1 - i].il != 7)
        return false;
    return true;
  }
};
}  // namespace

// lhaf of the N x N row-major complex matrix a (re, im pairs) whose vertices are scaled by
// m / 16 2^e; units are the nodes of level m1, breadth first from level top. Returns 0, or 1 on
// overflow, 2 on a write outside a buffer.
extern "C" int tree_host_lhaf(const double* a, int N, int m, int e, int m1, int top, double* out) {
  const int Ne = std::max(4, N + (N & 1)), n = Ne / 2;
  Guarded levels(tree_offset(m1 - 1, n)), scratch(tree_scratch(n, m1, top));
  Fxc* root = levels.data();
  const int edges = Ne * (Ne - 1) / 2;
  for (int p = 0; p < tree_polys(n); ++p) {
    int j, k;
    if (p < edges) tree_pair(p, j, k); else j = k = p - edges;
    const int r = (j & 1) ? j / 2 + n : j / 2, c = (k & 1) ? k / 2 + n : k / 2;
    Fxc v{};
    if (r < N && c < N) {
      const double* z = a + 2 * ((size_t)r * N + c);
      to_fixed(z[0], j == k ? m : m * m, j == k ? e - 4 : 2 * e - 8, v.rh, v.rm, v.rl);
      to_fixed(z[1], j == k ? m : m * m, j == k ? e - 4 : 2 * e - 8, v.ih, v.im, v.il);
    } else if (j == k) {
      v.rh = 1 << (kTreeFrac - 1 - 2 * kLimbBits);
    }
    fx_store(root + p, v);
  }
  Fxc one{};
  one.rh = 1 << (kTreeFrac - 2 * kLimbBits);
  fx_store(root + tree_polys(n), one);
  unsigned bad = 0;
  int node;
  Fxc z;
  for (int step = 0; n - step > m1; ++step) {
    const TreePhase s = tree_step_phase(root, n, step);
    for (unsigned t = 0; t < tree_tasks(s); ++t) tree_task(s, t, node, z, bad);
  }
  __int128 re = 0, im = 0;
  for (int unit = 0; unit < tree_width(m1, n); ++unit) {
    TreeLevel lv[34];
    tree_unit_levels(lv, root, scratch.data(), n, m1, top, unit);
    for (unsigned b = 0; b < 1u << (m1 - top); ++b)
      for (int i = tree_first_phase(m1, top, b); i < m1; ++i) {
        const TreePhase s = tree_unit_phase(lv, n, m1, top, unit, b, i);
        for (unsigned t = 0; t < tree_tasks(s); ++t)
          if (tree_task(s, t, node, z, bad)) {
            const bool neg = (__builtin_popcount(node) + __builtin_popcount(unit) + __builtin_popcount(b)) & 1;
            const __int128 x = (((__int128)z.rh << 28) + z.rm) * (1 << 28) + z.rl;
            const __int128 y = (((__int128)z.ih << 28) + z.im) * (1 << 28) + z.il;
            re += neg ? -x : x;
            im += neg ? -y : y;
          }
      }
  }
  const int exp2 = -kTreeFrac - (n >= 3 ? n - 3 : 0) - e * N + (Ne - N);
  const long double fac = std::pow(16.0L / m, (long double)N);
  out[0] = (double)std::ldexp((long double)re * fac, exp2);
  out[1] = (double)std::ldexp((long double)im * fac, exp2);
  return bad ? 1 : (levels.intact() && scratch.intact() ? 0 : 2);
}
