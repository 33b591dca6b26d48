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
  v += kLimbHalf;
  l = ((int)(long long)v & kLimbMask) - kLimbHalf;
  v = (v >> kLimbBits) + kLimbHalf;
  mm = ((int)(long long)v & kLimbMask) - kLimbHalf;
  h = (int)(long long)(v >> kLimbBits);
}

struct HostSlot {
  int* m;
  void put(int k, int v) const { m[k] = v; }
  int get(int k) const { return m[k]; }
};

// Guarded storage: a buffer with a canary on each side.
struct Guarded {
  std::vector<char> mem;
  explicit Guarded(size_t n) : mem(n + 2048, 7) {}
  char* data() { return mem.data() + 1024; }
  bool intact() const {
    for (int i = 0; i < 1024; ++i)
      if (mem[i] != 7 || mem[mem.size() - 1 - i] != 7) return false;
    return true;
  }
};
}  // namespace

// (level m1 = 0: the whole tree breadth first.)
// lhaf of the N x N row-major complex matrix a (re, im pairs) whose vertices are scaled by
// m / 16 2^e; units are the nodes of level m1, breadth first from level top. Returns 0, or 1 on
// overflow, 2 on a write outside a buffer.
extern "C" int tree_host_lhaf(const double* a, int N, int m, int e, int m1, int top, double* out) {
  const int Ne = std::max(4, N + (N & 1)), n = Ne / 2;
  const bool whole = m1 == 0;
  Guarded levels(tree_offset(whole ? 1 : m1 - 1, n)), scratch(whole ? 0 : tree_scratch(n, m1, top));
  const TreeLevel root = tree_level(levels.data(), n, n, 1);
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
    fx_store(root.A + fx_at(p), v);
  }
  Fxc one{};
  one.rh = 1 << (kTreeFrac - 2 * kLimbBits);
  fx_store(root.A + root.g, one);
  unsigned bad = 0;
  int node, ints[kSlotInts];
  const HostSlot slot{ints};
  Fxc z;
  __int128 re = 0, im = 0;
  auto add = [&](bool neg) {
    const __int128 x = (((__int128)z.rh << kLimbBits) + z.rm) * (1 << kLimbBits) + z.rl;
    const __int128 y = (((__int128)z.ih << kLimbBits) + z.im) * (1 << kLimbBits) + z.il;
    re += neg ? -x : x;
    im += neg ? -y : y;
  };
  for (int i = 0; whole && i < n; ++i) {
    const TreePhase s = tree_whole_phase(levels.data(), n, i);
    for (int t = 0; t < s.tasks; ++t)
      if (tree_task(s, 0, t, slot, node, z, bad)) add(__builtin_popcount(node) & 1);
  }
  for (int step = 0; !whole && n - step > m1; ++step) {
    const TreePhase s = tree_whole_phase(levels.data(), n, step);
    for (int t = 0; t < s.tasks; ++t) tree_task(s, 0, t, slot, node, z, bad);
  }
  for (int unit = 0; !whole && unit < tree_width(m1, n); ++unit) {
    TreeLevel lv[34];
    tree_unit_levels(lv, levels.data(), scratch.data(), n, m1, top, unit);
    for (unsigned b = 0; b < 1u << (m1 - top); ++b)
      for (int i = tree_first_phase(m1, top, b); i < m1; ++i) {
        const TreePhase s = tree_unit_phase(lv, n, m1, top, unit, i);
        for (int t = 0; t < s.tasks; ++t)
          if (tree_task(s, b, t, slot, node, z, bad))
            add((__builtin_popcount(node) + __builtin_popcount(unit) + __builtin_popcount(b)) & 1);
      }
  }
  const int exp2 = -kTreeFrac - (n >= 3 ? n - 3 : 0) - e * N + (Ne - N);
  const long double fac = std::pow(16.0L / m, (long double)N);
  out[0] = (double)std::ldexp((long double)re * fac, exp2);
  out[1] = (double)std::ldexp((long double)im * fac, exp2);
  return bad ? 1 : (levels.intact() && scratch.intact() ? 0 : 2);
}
