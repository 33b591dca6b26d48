// Kernels and launches of the elimination-tree evaluation (lhaf_tree.cuh).
//
//   tree_root_kernel   one CTA per problem: gathers the matrix (pattern, fill vector, padding),
//                      picks the scale and writes the fixed-point root level.
//   tree_step_kernel   one breadth-first elimination of every problem, one task per thread; the
//                      first levels, until there are nodes enough for all CTAs.
//   tree_kernel        persistent CTAs claim units (nodes of that level) and work off the subtree
//                      below in their own scratch, which stays small (in L1 and L2) because all
//                      but the last levels are walked depth first, two nodes a level. The
//                      leaves go to the problem's limb sums; integer sums are exact, so a result
//                      does not depend on how the tree is cut or on which CTA took which unit.
//                      The CTA that finishes a problem's last unit converts the sums to double.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <numeric>

#include <cooperative_groups.h>

#include "lhaf_kernels.cuh"
#include "lhaf_tree.cuh"
#include "lhaf_tree.h"

namespace cg = cooperative_groups;

namespace gbsh {

namespace {

// CTAs of tree_step_kernel and tree_kernel. 5 of 128 threads leave 96 registers a thread, which
// hold fx_conv2's operands a step ahead: N = 32 318 us and 512 patterns of up to 30 photons
// 6.38 ms, against 338 us and 6.71 ms with 6 (80 registers, nothing loaded ahead), 324 us and
// 6.77 ms with 4 (N = 44: 22.1, 22.0, 23.0 ms). Other widths (64 to 256 threads) were 4 to 28 %
// slower at N = 40.
constexpr int kTreeThreads = 128;
constexpr int kTreeCtasPerSm = 5;
// Largest n of a small problem (tree_small_kernel). Alone, n = 8 takes 53 us that way against 72
// by launches; n = 9 and 10 the same either way, n = 11 takes 104 against 91 and n = 12 162
// against 108: their levels are wider than 16 CTAs. 128 unrelated matrices of up to 16 indices
// take 195 us with this line at 8 or 9, 255 at 7.
constexpr int kTreeSmallMax = 8;
static_assert(kTreeSmallMax <= kFxLimitFree, "the limit of small problems is a constant");
// Units (tasks of one CTA) that a launch aims at, per CTA that runs at a time, shared out by work:
// a tree's work grows 2.26-fold with an index pair (n = 16 to 22). 512 patterns of up to 30
// photons take 7.6 ms with 2, 7.06 with 4, 6.75 with 8, 6.63 with 16, and 10.0 with 2 shared
// out evenly; the storage for the levels above the units grows with it.
constexpr double kTreeUnits = 8;
constexpr double kTreeGrowth = 2.26;
// Levels above the units at most, which bounds their storage: 2048 units, fewer than kTreeUnits asks
// for from one problem of N = 27 on. N = 50 takes 212 ms and 1.8 GB with 12, 218 and 1.8 with 11, 211 and 2.0 with
// 13; N = 56 2.10 s, 2.21 and 2.12. 13 suits N = 40 (4.21 ms, 4.70 with 12) and 48 (94 ms, 100), but takes
// 375 us instead of 319 at N = 32 and 1.05 ms instead of 1.02 at N = 36.
constexpr int kTreeDepth = 12;
// Level from which a unit is worked off breadth first: 5 takes 5.31 ms at N = 40 (levels too narrow
// for a CTA), 7 takes 23.6 ms at N = 44 (its storage leaves the L2), 6 takes 4.7 and 22.0.
constexpr int kTreeTop = 6;
// Smallest scaled result that is kept: where the tree's absolute error is 2^-53 of it. The error is
// a mean over the leaves: against a 113-bit evaluation, over matrices with loop weights of 0.2 to 2,
// at most 2^-81.4 at N = 20, 2^-82.2 at 24, 2^-83.5 at 28 and 2^-84.0 at 32. (Configuration matrices
// come out at 2^-20 for N = 40, 2^-27 for N = 50.)
__device__ __forceinline__ int tree_min_exp(int n) { return n > 10 ? -28 - (n - 10) / 2 : -28; }

// The scale of a vertex: d_j with lhaf(D A D) = det D lhaf(A). The edges alone ask for d^-2 = rho
// (below) and for entries below 0.8; where the loop weights are large their vertices get a smaller
// one, d_j |v_j| = sqrt(tau), such that sum d^2 |v|^2 <= kWeightSum: the weights enter g as exp of half
// that sum spread over n pairs. Large weights and a full matrix together grow faster than each alone, so
// d^-2 is raised by up to kWeightEdge as the sum approaches its limit. One scale for all vertices, as
// the largest weight needs it, loses the smaller ones: of 152 matrices with weights of 0.3 to 2 a size (in and out
// of phase, and random real ones) 35 were handed back to the subset sum at N = 20, 70 at 24, 105 at
// 28; this way 0, 2 and 21. kWeightSum = 6.25 or 6.75: 1 or 4 at N = 24, 45 or 20 at N = 28.
constexpr float kWeightSum = 6.5f, kWeightMax = 0.8f;
constexpr float kWeightEdge = 0.75f, kWeightFree = 0.2f;
// Weights beyond 2^32 times what the edges scale to one stay with the subset sum, whose value
// test_handed_back_to_the_subset_sum (tests/test_gpu_tree.py) asks for there.
constexpr float kWeightRange = 18446744073709551616.f;

__device__ __forceinline__ void dd_two_prod(double a, double b, double& p, double& e) {
  p = __dmul_rn(a, b);
  e = __fma_rn(a, b, -p);
}
__device__ __forceinline__ void dd_mul(double ah, double al, double bh, double bl, double& h, double& l) {
  double p, e;
  dd_two_prod(ah, bh, p, e);
  e = __fma_rn(ah, bl, __fma_rn(al, bh, e));
  h = __dadd_rn(p, e);
  l = __dsub_rn(e, __dsub_rn(h, p));
}

// x m 2^e in units of 2^-81 as limbs; bad |= it does not fit (or x is not finite). Integer
// instructions only: FP64 ones are slow.
__device__ void to_fixed(double x, int m, int e, int& h, int& mm, int& l, unsigned& bad) {
  const long long bits = __double_as_longlong(x);
  const int ex = (int)(bits >> 52) & 0x7ff;
  if (ex == 0x7ff) bad = 1;
  const long long mant = (bits & ((1ll << 52) - 1)) | (ex ? 1ll << 52 : 0);
  __int128 v = (bits < 0 ? -mant : mant) * m;  // < 2^63: 53 bits times at most 31^2
  const int sh = (ex ? ex : 1) - 1075 + e + kTreeFrac;
  if (v == 0 || sh < -100) {
    v = 0;
  } else if (sh >= 0) {
    if (sh > 62) bad = 1;
    v <<= (sh > 62 ? 62 : sh);
  } else {
    v = (v + ((__int128)1 << (-sh - 1))) >> (-sh);
  }
  const __int128 lim = (__int128)1 << kTreeFrac;  // |x| < 1: room for the first products
  if (v >= lim || v <= -lim) bad = 1;
  v += kLimbHalf;
  l = ((int)(long long)v & kLimbMask) - kLimbHalf;
  v = (v >> kLimbBits) + kLimbHalf;
  mm = ((int)(long long)v & kLimbMask) - kLimbHalf;
  h = (int)(long long)(v >> kLimbBits);
}

__device__ __forceinline__ double2 tree_entry(const BatchInput& in, int r, int c) {
  const int ir = in.idx ? in.idx[r] : r, ic = in.idx ? in.idx[c] : c;
  if (r == c && in.diag) return in.diag[ir];
  return in.base[(size_t)ir * in.ld + ic];
}
// Biased exponent of a double, and x 2^(1023 - ex) in single precision (0 where that underflows).
__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ float scaled_float(double x, int ex) {
  const int hi = __double2hiint(x), e = ((hi >> 20) & 0x7ff) - ex + 127;
  if (e <= 0) return 0.f;
  return __int_as_float((hi & 0x80000000) | (e << 23) | ((hi & 0xfffff) << 3) |
                        (int)((unsigned)__double2loint(x) >> 29));
}

constexpr int kRootThreads = 256;  // of the root kernel and of a cluster's CTAs
constexpr int kRootWarps = kRootThreads / 32;

struct RootShared {
  float2 a[kMaxN * kMaxN];
  float v2[kMaxN];          // |v_j|^2
  short m[kMaxN], e[kMaxN];  // scale of index j: m / 16 2^e
  unsigned ea[kRootWarps], ev[kRootWarps];
  float f[3][kRootWarps];
};

__device__ __forceinline__ float warp_sum(float x) {
  for (int d = 16; d; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
  return x;
}
__device__ __forceinline__ float warp_max(float x) {
  for (int d = 16; d; d >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, d));
  return x;
}

// Root level and state of a problem, by one CTA of kThreads threads: gathers the matrix, picks
// the scale, writes the fixed-point numbers. Latency matters here (small problems take 20 us in
// all), so the scale is worked out in single precision from exponent-shifted entries.
template <int kThreads>
__device__ void tree_root(const TreeProblem& P, const TreeLevel& root, TreeState* S, RootShared& sh) {
  constexpr int kWarps = kThreads / 32;
  const int tid = threadIdx.x, N = P.in.N, lane = tid & 31, warp = tid >> 5;
  unsigned bad = 0, ea = 0, ev = 0;
  for (int e = tid; e < N * N; e += kThreads) {
    const int r = e / N, c = e - r * N;
    const double2 z = tree_entry(P.in, r, c);
    const unsigned x = (unsigned)max(exponent_of(z.x), exponent_of(z.y));
    if (x == 0x7ff) bad = 1;
    if (r == c) ev = max(ev, x); else ea = max(ea, x);
  }
  ea = __reduce_max_sync(0xffffffffu, ea);
  ev = __reduce_max_sync(0xffffffffu, ev);
  if (lane == 0) {
    sh.ea[warp] = ea;
    sh.ev[warp] = ev;
  }
  __syncthreads();
  for (int w = 0; w < kWarps; ++w) {
    ea = max(ea, sh.ea[w]);
    ev = max(ev, sh.ev[w]);
  }
  // entries and weights as floats below 2
  float f2 = 0.f, am = 0.f;
  for (int e = tid; e < N * N; e += kThreads) {
    const int r = e / N, c = e - r * N;
    const double2 z = tree_entry(P.in, r, c);
    const int ex = r == c ? (int)ev : (int)ea;
    float2 w = make_float2(scaled_float(z.x, ex), scaled_float(z.y, ex));
    const float m2 = w.x * w.x + w.y * w.y;
    if (r == c) {
      sh.v2[r] = m2;
      w = make_float2(0.f, 0.f);
    } else {
      f2 += m2;
      am = fmaxf(am, m2);
    }
    sh.a[e] = w;
  }
  __syncthreads();
  // rho = |A^H A|_F / |A|_F, the root of the mean of sigma^2 weighted by sigma^2: equal to the
  // spectral norm for flat and for rank-one spectra
  float g2 = 0.f;
  for (int e = tid; e < N * (N + 1) / 2; e += kThreads) {
    int i, j;
    tree_pair(e, i, j);  // i < j: (i, j - 1) runs over the upper triangle
    --j;
    float re = 0.f, im = 0.f;
    for (int k = 0; k < N; ++k) {
      const float2 x = sh.a[k * N + i], y = sh.a[k * N + j];  // conj(x) y
      re += x.x * y.x + x.y * y.y;
      im += x.x * y.y - x.y * y.x;
    }
    g2 += (i == j ? 1.f : 2.f) * (re * re + im * im);
  }
  f2 = warp_sum(f2);
  g2 = warp_sum(g2);
  am = warp_max(am);
  if (lane == 0) {
    sh.f[0][warp] = f2;
    sh.f[1][warp] = g2;
    sh.f[2][warp] = am;
  }
  __syncthreads();
  if (warp == 0) {  // short code: a CTA runs it once and waits for its instructions
    f2 = warp_sum(lane < kWarps ? sh.f[0][lane] : 0.f);
    g2 = warp_sum(lane < kWarps ? sh.f[1][lane] : 0.f);
    am = warp_max(lane < kWarps ? sh.f[2][lane] : 0.f);
    // d^-2 of the edges alone, in units of 2^xa; |v|^2 is in units of 2^xv. Without edges the
    // weights alone set the scales.
    const int xv = 2 * ((int)ev - 1023);
    int xa = (int)ea - 1023;
    float da = fmaxf(f2 > 0.f ? sqrtf(__fdividef(g2, f2)) : 0.f, 1.25f * sqrtf(am));
    if (ea == 0 || !(da > 0.f)) {
      da = 1.f;
      xa = ev ? xv - 60 : 0;
    }
    // d^2 |v|^2 of indices lane and lane + 32
    const float m0 = lane < N ? sh.v2[lane] : 0.f, m1 = lane + 32 < N ? sh.v2[lane + 32] : 0.f;
    const float unit = __fdividef(__int_as_float((min(max(xv - xa, -126), 126) + 127) << 23), da);
    float w0 = m0 * unit, w1 = m1 * unit;
    if (fmaxf(w0, w1) > kWeightRange) bad = 1;
    const float full = warp_sum(fminf(w0, kWeightMax) + fminf(w1, kWeightMax)) * (1.f / kWeightSum);
    const float edge = 1.f + kWeightEdge / (1.f - kWeightFree) * fmaxf(0.f, fminf(full, 1.f) - kWeightFree);
    da *= edge;
    w0 = __fdividef(w0, edge);
    w1 = __fdividef(w1, edge);
    float tau = kWeightMax;
    if (full > 1.f && warp_sum(fminf(w0, tau) + fminf(w1, tau)) > kWeightSum) {
      // the tau at which the sum of min(w, tau) is kWeightSum, from below
      tau = __fdividef(kWeightSum, (float)N);
#pragma unroll 1
      for (int it = 0; it < 6; ++it) {
        const float small = warp_sum((w0 <= tau ? w0 : 0.f) + (w1 <= tau ? w1 : 0.f));
        const int big = __popc(__ballot_sync(0xffffffffu, w0 > tau)) + __popc(__ballot_sync(0xffffffffu, w1 > tau));
        if (big) tau = fminf(__fdividef(kWeightSum - small, (float)big), kWeightMax);
      }
    }
#pragma unroll 1
    for (int j = lane; j < N; j += 32) {
      const bool heavy = (j < 32 ? w0 : w1) > tau;
      const float den = heavy ? __fdividef(j < 32 ? m0 : m1, tau) : da;
      const int top = heavy ? xv : xa;
      // 1 / sqrt(den 2^top), a little below, as m / 16 2^e with m of 5 bits: exact products
      const int f = __float_as_int(rsqrtf((top & 1) ? 2.f * den : den) * 0.999999f);
      const int e = (f >> 23) - 127 - (top >> 1);
      if (e > 900 || e < -900) bad = 1;
      sh.m[j] = (short)(16 + ((f >> 19) & 15));
      sh.e[j] = (short)min(max(e, -900), 900);
    }
  }
  __syncthreads();
  if (warp == kWarps - 1) {  // 1 / det D: the product of the m / 16, and the exponents apart
    double h = 1.0, l = 0.0;
    int e = 0;
    for (int j = lane; j < N; j += 32) {
      h *= sh.m[j];
      e += sh.e[j];
    }
    for (int d = 1; d < 4; d <<= 1) h *= __shfl_xor_sync(0xffffffffu, h, d);  // exact: 8 factors of 5 bits
#pragma unroll 1
    for (int d = 4; d < 32; d <<= 1)
      dd_mul(h, l, __shfl_xor_sync(0xffffffffu, h, d), __shfl_xor_sync(0xffffffffu, l, d), h, l);
    e = __reduce_add_sync(0xffffffffu, e);
    if (lane == 0) {
      const double r = __drcp_rn(h);
      S->fac_hi = r;
      S->fac_lo = __fma_rn(-r, l, __fma_rn(-r, h, 1.0)) * r;
      S->exp2 = -kTreeFrac - (P.n >= 3 ? P.n - 3 : 0) - e + 4 * N + (P.Ne - N);
    }
  }
  // root level: vertex 2 p is index p, vertex 2 p + 1 is index p + n; padding vertices have no
  // edges, loop weight one and scale one half
  const int polys = tree_polys(P.n), edges = P.Ne * (P.Ne - 1) / 2;
  for (int p = tid; p < polys; p += kThreads) {
    int j, k;
    if (p < edges) tree_pair(p, j, k); else j = k = p - edges;
    const int r = (j & 1) ? (j >> 1) + P.n : (j >> 1), c = (k & 1) ? (k >> 1) + P.n : (k >> 1);
    Fxc v{};
    if (r < N && c < N) {
      const double2 z = tree_entry(P.in, r, c);
      const int mm = j == k ? sh.m[r] : sh.m[r] * sh.m[c], ee = j == k ? sh.e[r] - 4 : sh.e[r] + sh.e[c] - 8;
      to_fixed(z.x, mm, ee, v.rh, v.rm, v.rl, bad);
      to_fixed(z.y, mm, ee, v.ih, v.im, v.il, bad);
    } else if (j == k) {
      v.rh = 1 << (kTreeFrac - 1 - 2 * kLimbBits);
    }
    fx_store(root.A + fx_at(p), v);
  }
  if (tid == 0) {
    Fxc v{};
    v.rh = 1 << (kTreeFrac - 2 * kLimbBits);
    fx_store(root.A + root.g, v);  // g = 1
    for (int i = 0; i < 6; ++i) S->sum[i] = 0;
    S->done = 0;
  }
  const int any = __syncthreads_or((int)bad);
  if (tid == 0) S->bad = any ? 1 : 0;
}

// Scales a problem and makes its level n. One CTA a problem: 8 to 13 us of dependent steps (norms,
// scale, conversion), hidden in a batch. kOne: one problem, passed as a kernel argument;
// otherwise a table in device memory.
template <bool kOne>
__global__ void __launch_bounds__(kRootThreads)
tree_root_kernel(const TreeProblem* __restrict__ table, TreeProblem one, TreeState* __restrict__ state,
                 unsigned* __restrict__ counter, char* __restrict__ levels) {
  __shared__ RootShared sh;
  cudaTriggerProgrammaticLaunchCompletion();  // launched the plain way: nothing to wait for
  const TreeProblem P = kOne ? one : table[blockIdx.x];
  if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0;
  tree_root<kRootThreads>(P, tree_level(levels + P.root, P.n, P.n, 1), state + blockIdx.x, sh);
}

// The problem's signed mean from its limb sums, to double.
__device__ void tree_result(const TreeProblem& P, TreeState* S, double* out, bool flags) {
  double v[2];
  double top = 0.0;
  for (int c = 0; c < 2; ++c) {
    const long long h = (long long)__ldcg(&S->sum[3 * c]), m = (long long)__ldcg(&S->sum[3 * c + 1]),
                    l = (long long)__ldcg(&S->sum[3 * c + 2]);
    __int128 r = ((__int128)h << kLimbBits) + m;
    r = (r << kLimbBits) + l;
    const bool neg = r < 0;
    if (neg) r = -r;
    const unsigned long long hi = (unsigned long long)(r >> 64), lo = (unsigned long long)r;
    // exact pieces: hi < 2^53, the halves of lo
    const double x = (double)hi * 18446744073709551616.0, y = (double)(lo >> 32) * 4294967296.0,
                 z = (double)(lo & 0xffffffffull);
    double s = x + y, e = y - (s - x);
    const double s2 = s + z, e2 = z - (s2 - s) + e;
    const double ah = s2 + e2, al = e2 - (ah - s2);
    double ph, pl;
    dd_mul(ah, al, S->fac_hi, S->fac_lo, ph, pl);
    v[c] = ldexp(neg ? -ph : ph, S->exp2);
    top = fmax(top, ah);
  }
  const int shift = kTreeFrac + (P.n >= 3 ? P.n - 3 : 0);
  const bool fail = __ldcg(&S->bad) != 0 || !(ldexp(top, -shift) >= ldexp(1.0, tree_min_exp(P.n)));
  if (fail) S->bad = 1;
  out[0] = v[0];
  out[1] = v[1];
  if (flags) out[2] = fail ? 1.0 : 0.0;
}

// One piece (tree_piece) per lane, four neighbouring lanes per coefficient; all lanes of a warp
// call it together. A phase with few items is a chain of loads and products in each thread:
// in pieces the chain is a quarter as long. `J`: tree_piece_job of `id`. Returns true in the lane
// that holds a term in z.
__device__ __forceinline__ TreeJob tree_piece_job(const TreePhase& s, int id, int& t) {
  const int L = s.n - s.M + 1, q = id >> 2;
  const bool active = q < L * s.items;
  const int row = active ? tree_div(q, s.items, s.inv_items) : 0;
  t = active ? L - 1 - row : 1 << 20;
  return tree_job(s, 0, active ? q - row * s.items : 0);
}
__device__ __forceinline__ bool tree_piece_task(const TreeJob& J, int t, int sub, Fxc& z, unsigned& bad) {
  const bool active = t <= J.top + 1;
  FxSum acc{0, 0, 0, 0, 0, 0};
  Fxc old{};
  if (active) {
    old = tree_end_old(J, t, sub);
    acc = tree_piece(J, t, sub);
  }
#pragma unroll
  for (int d = 1; d <= 2; d <<= 1) {
    acc.s2r += __shfl_xor_sync(0xffffffffu, acc.s2r, d);
    acc.s1r += __shfl_xor_sync(0xffffffffu, acc.s1r, d);
    acc.s0r += __shfl_xor_sync(0xffffffffu, acc.s0r, d);
    acc.s2i += __shfl_xor_sync(0xffffffffu, acc.s2i, d);
    acc.s1i += __shfl_xor_sync(0xffffffffu, acc.s1i, d);
    acc.s0i += __shfl_xor_sync(0xffffffffu, acc.s0i, d);
  }
  if (!active) return false;
  unsigned& over = bad;  // as in tree_task
  bad <<= 31;
  const Fxc v = fx_norm(acc, over);
  if (J.end != kDot) {
    tree_end_part(J, t, sub, old, v, over);
  } else if (sub == 0) {
    FxAcc dot = fx_acc_zero();
    fx_mac(dot, v, old);
    z = fx_norm(fx_sum(dot), over);
  }
  bad >>= 31;
  return J.end == kDot && sub == 0;
}

// Column of a thread in its CTA's job storage (tree_put). Volatile: the compiler would keep the
// values in registers, and spill those of the products instead.
template <int kThreads>
struct JobSlot {
  volatile int (*m)[kThreads];
  __device__ __forceinline__ void put(int k, int v) const { m[k][threadIdx.x] = v; }
  __device__ __forceinline__ int get(int k) const { return m[k][threadIdx.x]; }
};

// One breadth-first level of the large problems, the whole GPU on it: 3 to 17 us, the latency of a
// launch and of its loads for the narrow levels, the products for the wide ones. kOne: the phase
// of the one problem is set up on the host. Phases of at most `fine` pieces, a quarter of a
// coefficient a thread, run that way: a narrow level is as long as one thread's work (N = 20
// 59 us an evaluation, 80 without; N = 25 116 and 130; N = 40 the same).
template <bool kOne>
__global__ void __launch_bounds__(kTreeThreads, kTreeCtasPerSm)
tree_step_kernel(const TreeProblem* __restrict__ table, const __grid_constant__ TreePhase one, int step, int fine,
                 TreeState* __restrict__ state, char* __restrict__ levels) {
  __shared__ TreePhase many;
  __shared__ int slots[kSlotInts][kTreeThreads];
  chain_wait();
  if (!kOne) {
    if (table[blockIdx.y].n - step <= table[blockIdx.y].m1) return;  // fewer steps than another's
    if (threadIdx.x == 0)
      many = tree_whole_phase(levels + table[blockIdx.y].root, table[blockIdx.y].n, step);
    __syncthreads();
  }
  const TreePhase& s = kOne ? one : many;
  const int t = (int)(blockIdx.x * kTreeThreads + threadIdx.x);
  unsigned bad = 0;
  int x;
  Fxc z;
  if (tree_pieces(s) <= fine) {
    if ((t & ~31) < tree_pieces(s)) {
      const TreeJob J = tree_piece_job(s, t, x);
      tree_piece_task(J, x, t & 3, z, bad);
    }
  } else if (t < s.tasks) {
    tree_task(s, 0, t, JobSlot<kTreeThreads>{slots}, x, z, bad);
  }
  if (bad) atomicOr(&state[blockIdx.y].bad, 1u);
}

// Limb sums of the terms a thread met, one column per thread (64-bit atomics on one shared sum
// were a third of a small problem's time).
template <int kThreads>
struct LimbSums {
  long long v[6][kThreads];
  __device__ void clear() {
    for (int i = 0; i < 6; ++i) v[i][threadIdx.x] = 0;
  }
  __device__ void add(const Fxc& z, bool neg) {
    const int sg = neg ? -1 : 1, t = threadIdx.x;
    v[0][t] += sg * z.rh;
    v[1][t] += sg * z.rm;
    v[2][t] += sg * z.rl;
    v[3][t] += sg * z.ih;
    v[4][t] += sg * z.im;
    v[5][t] += sg * z.il;
  }
  // After a barrier: warp w adds up the sums w, w + warps, ... into v[.][0].
  __device__ void reduce() {
    for (int i = threadIdx.x >> 5; i < 6; i += kThreads / 32) {
      long long x = 0;
      for (int t = threadIdx.x & 31; t < kThreads; t += 32) x += v[i][t];
      for (int d = 16; d; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
      if ((threadIdx.x & 31) == 0) v[i][0] = x;
    }
  }
};

// The units of all large problems, claimed from a counter by one resident wave of CTAs: nearly all
// of a large evaluation. A unit's levels live in the CTA's own scratch (walked depth first, two
// nodes a level, so that the scratch of all CTAs stays in the L2) and its tasks are independent
// within a phase. Bound by the convolutions' multiply-adds (their pipe is busy 69 % of the time, see
// fx_conv2), and the latency of their loads (4.4 warps a scheduler; 50 % hit L1, and a
// warp waits for one during 15 % of its time). N = 40: 4.70 ms, 0.21e12 complex
// multiply-adds/s (184 ms for the subset sum); N = 44: 20.8 ms (919).
template <bool kOne>
__global__ void __launch_bounds__(kTreeThreads, kTreeCtasPerSm)
tree_kernel(const TreeProblem* __restrict__ table, TreeProblem one, int count, unsigned total_units,
            TreeState* __restrict__ state, unsigned* __restrict__ counter, char* __restrict__ levels,
            char* __restrict__ scratch, size_t cta_bytes, double* __restrict__ out, bool flags) {
  __shared__ TreeLevel lv[kMaxN / 2 + 2];  // levels m1 + 1 and m1: the unit and its parent
  __shared__ TreePhase phase[kMaxN / 2];
  __shared__ LimbSums<kTreeThreads> sum;
  __shared__ int slots[kSlotInts][kTreeThreads];
  __shared__ unsigned s_unit;
  __shared__ int s_prob;
  const int tid = threadIdx.x;
  char* ws = scratch + (size_t)blockIdx.x * cta_bytes;
  chain_wait();
  for (;;) {
    if (tid == 0) {
      const unsigned u = atomicAdd(counter, 1u);
      s_unit = u;
      int lo = 0, hi = count - 1;  // last problem with unit_base <= u
      while (!kOne && lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (table[mid].unit_base <= u) lo = mid; else hi = mid - 1;
      }
      s_prob = lo;
    }
    sum.clear();
    __syncthreads();
    if (s_unit >= total_units) return;
    const int prob = s_prob;
    const TreeProblem P = kOne ? one : table[prob];
    const int n = P.n, m1 = P.m1, top = P.top, unit = (int)(s_unit - P.unit_base);
    if (tid == 0) tree_unit_levels(lv, levels + P.root, ws, n, m1, top, unit);
    __syncthreads();
    // in shared memory because the accumulators leave no registers for them
    if (tid < m1) phase[tid] = tree_unit_phase(lv, n, m1, top, unit, tid);
    __syncthreads();
    unsigned bad = 0;
    for (unsigned b = 0; b < 1u << (m1 - top); ++b)
      for (int i = tree_first_phase(m1, top, b); i < m1; ++i) {
        const TreePhase& s = phase[i];
        for (int t = tid; t < s.tasks; t += kTreeThreads) {
          int x;
          Fxc z;
          if (tree_task(s, b, t, JobSlot<kTreeThreads>{slots}, x, z, bad))
            sum.add(z, (__popc((unsigned)x) + __popc((unsigned)unit) + __popc(b)) & 1);
        }
        __syncthreads();
      }
    const int any = __syncthreads_or((int)bad);
    TreeState* S = state + prob;
    sum.reduce();
    __syncthreads();
    if (tid < 6) atomicAdd(&S->sum[tid], (unsigned long long)sum.v[tid][0]);
    if (tid == 0 && any) atomicOr(&S->bad, 1u);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      if (atomicAdd(&S->done, 1u) == P.units - 1) {
        __threadfence();
        tree_result(P, S, out + 3 * (size_t)prob, flags);
      }
    }
    __syncthreads();
  }
}

// Small problems in one launch: a cluster of CTAs works a whole tree off breadth first, one
// cluster barrier a level (a grid-wide step is a launch, 3 us; the levels of a small tree take
// less). Its scratch holds every level. Bound by the barriers and the latency of a level's loads:
// N = 16 takes 31 us (42 with the gated launches behind it; 135 by the subset sum).
template <bool kOne>
__global__ void __launch_bounds__(kRootThreads, 2)
tree_small_kernel(const TreeProblem* __restrict__ table, TreeProblem one, int first, int count,
                  TreeState* __restrict__ state, char* __restrict__ scratch, size_t bytes,
                  double* __restrict__ out, bool flags) {
  __shared__ union {
    RootShared root;
    LimbSums<kRootThreads> sum;
  } sh;
  __shared__ TreePhase phase[kTreeSmallMax];
  __shared__ int slots[kSlotInts][kRootThreads];
  __shared__ unsigned s_bad;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank(), tid = threadIdx.x;
  const int id = (int)blockIdx.x / C, clusters = (int)gridDim.x / C, stride = C * kRootThreads;
  char* base = scratch + (size_t)id * bytes;
  for (int p = first + id; p < first + count; p += clusters) {
    const TreeProblem P = kOne ? one : table[p];
    TreeState* S = state + p;
    if (tid < P.n) phase[tid] = tree_whole_phase<true>(base, P.n, tid);
    if (tid == P.n) s_bad = 0;
    if (rank == 0) tree_root<kRootThreads>(P, tree_level(base, P.n, P.n, 1), S, sh.root);
    __syncthreads();
    sh.sum.clear();
    const int t0 = rank * kRootThreads + tid;
    unsigned bad = 0;
    int t;
    TreeJob J = tree_piece_job(phase[0], t0, t);
    cl.sync();
    for (int i = 0; i < P.n; ++i) {
      const TreePhase& s = phase[i];
      const int pieces = tree_pieces(s);
      int x;
      Fxc z;
      if (pieces <= 3 * stride) {
        for (int q = t0; (q & ~31) < pieces; q += stride) {
          if (q != t0) J = tree_piece_job(s, q, t);
          J.lim = kFxLimit;
          if (tree_piece_task(J, t, q & 3, z, bad)) sh.sum.add(z, __popc((unsigned)J.node) & 1);
        }
      } else {
        for (int q = t0; q < s.tasks; q += stride)
          if (tree_task<true>(s, 0, q, JobSlot<kRootThreads>{slots}, x, z, bad)) sh.sum.add(z, __popc((unsigned)x) & 1);
      }
      if (i == P.n - 1) {
        if (bad) atomicOr(&s_bad, 1u);
        __syncthreads();
        sh.sum.reduce();
      }
      // the next phase's first job is worked out while the others arrive
      auto token = cl.barrier_arrive();
      if (i + 1 < P.n) J = tree_piece_job(phase[i + 1], t0, t);
      cl.barrier_wait(std::move(token));
    }
    if (rank == 0) {
      if (tid < 6) {
        long long total = sh.sum.v[tid][0];
        for (int r = 1; r < C; ++r) total += *cl.map_shared_rank(&sh.sum.v[tid][0], r);
        S->sum[tid] = (unsigned long long)total;
      }
      if (tid == 6) {
        unsigned b = s_bad;
        for (int r = 1; r < C; ++r) b |= *cl.map_shared_rank(&s_bad, r);
        if (b) S->bad = 1;
      }
      __syncthreads();
      if (tid == 0) tree_result(P, S, out + 3 * (size_t)p, flags);
    }
    cl.sync();  // the other CTAs' sums were read
  }
}

constexpr int kMaxGridY = 65535;

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

using SmallKernel = void (*)(const TreeProblem*, TreeProblem, int, int, TreeState*, char*, size_t, double*, bool);

static cudaLaunchConfig_t small_config(int cluster, int clusters, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(clusters * cluster));
  cfg.blockDim = dim3(kRootThreads);
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)cluster;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// CTAs of tree_small_kernel's largest cluster on the current device: 16 is not a portable size, and
// a partition of the device may hold fewer. Asked once a device.
static cudaError_t max_cluster(int* out) {
  static std::mutex mu;
  static int most[64] = {};
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (!most[dev]) {
    int c = 16;
    for (; c > 1; c >>= 1) {
      bool fits = true;
      for (const SmallKernel k : {tree_small_kernel<true>, tree_small_kernel<false>}) {
        cudaLaunchAttribute attr{};
        const cudaLaunchConfig_t cfg = small_config(c, 1, &attr);
        int n = 0;
        fits = fits && (c <= 8 || cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
               cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0;
      }
      if (fits) break;
      cudaGetLastError();
    }
    most[dev] = c;
  }
  *out = most[dev];
  return cudaSuccess;
}

}  // namespace

// Callers sit behind C entry points: no exception leaves.
cudaError_t tree_plan(const int* Ns, int count, size_t base_off, TreePlan* plan) try {
  DeviceInfo dev;
  cudaError_t e = device_info(&dev);
  if (e != cudaSuccess) return e;
  TreePlan& T = *plan;
  T.order.resize(count);
  std::iota(T.order.begin(), T.order.end(), 0);
  std::stable_sort(T.order.begin(), T.order.end(), [&](int a, int b) { return Ns[a] > Ns[b]; });
  T.prob.resize(count);
  T.steps.clear();
  auto pairs = [&](int q) { return std::max(4, Ns[T.order[q]] + (Ns[T.order[q]] & 1)) / 2; };
  // in launch order: large, small
  const int cluster_slots = 2 * dev.sm_count;
  T.nbig = 0;
  double work = 0;
  while (T.nbig < count && pairs(T.nbig) > kTreeSmallMax) work += std::pow(kTreeGrowth, pairs(T.nbig++));
  const int nsmall = count - T.nbig;
  T.cluster = T.clusters = 0;
  T.small_bytes = 0;
  if (nsmall > 0) {
    const int n = pairs(T.nbig);  // of the largest
    int most = 1;
    e = max_cluster(&most);
    if (e != cudaSuccess) return e;
    T.cluster = tree_cluster(n, nsmall, cluster_slots, most);
    T.clusters = std::min(nsmall, cluster_slots / T.cluster);
    T.small_bytes = align256(tree_offset(1, n));
  }
  const unsigned slots = (unsigned)(kTreeCtasPerSm * dev.sm_count);
  unsigned base = 0;
  size_t root = 0;
  T.cta_bytes = 0;
  T.fine = (int)slots * kTreeThreads / std::max(T.nbig, 1);  // pieces that still run all at once
  for (int q = 0; q < count; ++q) {
    TreeProblem& P = T.prob[q];
    const int n = pairs(q);
    P.Ne = 2 * n;
    P.n = n;
    P.m1 = P.top = n;
    P.units = 0;
    P.unit_base = base;
    P.root = root;
    if (q >= T.nbig) continue;
    P.m1 = n - 1;
    const double want = kTreeUnits * slots * std::pow(kTreeGrowth, n) / work;
    while (P.m1 > 2 && tree_width(P.m1, n) < want && n - P.m1 < kTreeDepth) --P.m1;
    P.top = std::min(kTreeTop, P.m1);
    P.units = (unsigned)tree_width(P.m1, n);
    base += P.units;
    root += align256(tree_offset(P.m1 - 1, n));
    T.cta_bytes = std::max(T.cta_bytes, tree_scratch(n, P.m1, P.top));
    for (int i = 0; i < n - P.m1; ++i) {
      if ((int)T.steps.size() <= i) T.steps.push_back(TreePlan::Step{0, 0});
      T.steps[i].problems = q + 1;
      const TreePhase s = tree_whole_phase(nullptr, n, i);
      T.steps[i].tasks = std::max(T.steps[i].tasks, tree_pieces(s) <= T.fine ? tree_pieces(s) : s.tasks);
    }
  }
  T.total_units = base;
  T.blocks = (int)std::min<unsigned>(slots, base);
  size_t off = align256(base_off);
  T.off_prob = off; off = align256(off + sizeof(TreeProblem) * (size_t)count);
  T.off_state = off; off = align256(off + sizeof(TreeState) * (size_t)count);
  T.off_counter = off; off = align256(off + sizeof(unsigned));
  T.off_out = off; off = align256(off + 3 * sizeof(double) * (size_t)count);
  T.off_root = off; off = align256(off + root);
  T.off_cta = off; off = align256(off + T.cta_bytes * (size_t)T.blocks);
  T.off_small = off; off = align256(off + T.small_bytes * (size_t)T.clusters);
  T.bytes = off;
  return cudaSuccess;
} catch (const std::bad_alloc&) {
  return cudaErrorMemoryAllocation;
}

cudaError_t tree_stage(TreePlan* plan, const BatchInput* in, void* ws, cudaStream_t st) {
  for (size_t q = 0; q < plan->prob.size(); ++q) plan->prob[q].in = in[plan->order[q]];
  if (plan->prob.size() < 2) return cudaSuccess;
  return cudaMemcpyAsync(static_cast<char*>(ws) + plan->off_prob, plan->prob.data(),
                         sizeof(TreeProblem) * plan->prob.size(), cudaMemcpyHostToDevice, st);
}

static cudaError_t launch_small(const TreePlan& plan, char* b, cudaStream_t st, double* out, bool flags) {
  const int count = (int)plan.prob.size();
  const bool one = count == 1;
  const SmallKernel k = one ? tree_small_kernel<true> : tree_small_kernel<false>;
  cudaLaunchAttribute attr{};
  cudaLaunchConfig_t cfg = small_config(plan.cluster, plan.clusters, &attr);
  cfg.stream = st;
  const TreeProblem* table = one ? nullptr : reinterpret_cast<const TreeProblem*>(b + plan.off_prob);
  return cudaLaunchKernelEx(&cfg, k, table, plan.prob[0], plan.nbig, count - plan.nbig,
                            reinterpret_cast<TreeState*>(b + plan.off_state), b + plan.off_small,
                            plan.small_bytes, out, flags);
}

static cudaError_t launch_large(const TreePlan& plan, char* b, cudaStream_t st, double* out, bool flags) {
  const bool one = plan.prob.size() == 1;
  const TreeProblem* table = one ? nullptr : reinterpret_cast<const TreeProblem*>(b + plan.off_prob);
  TreeState* state = reinterpret_cast<TreeState*>(b + plan.off_state);
  unsigned* counter = reinterpret_cast<unsigned*>(b + plan.off_counter);
  char* levels = b + plan.off_root;
  const TreeProblem& p0 = plan.prob[0];
  if (one)
    tree_root_kernel<true><<<1, kRootThreads, 0, st>>>(table, p0, state, counter, levels);
  else
    tree_root_kernel<false><<<plan.nbig, kRootThreads, 0, st>>>(table, p0, state, counter, levels);
  cudaError_t e = cudaGetLastError();
  for (int i = 0; i < (int)plan.steps.size() && e == cudaSuccess; ++i) {
    const TreePhase s = tree_whole_phase(levels + p0.root, p0.n, i);
    const unsigned x = (unsigned)(plan.steps[i].tasks + kTreeThreads - 1) / kTreeThreads;
    for (int f = 0; f < plan.steps[i].problems && e == cudaSuccess; f += kMaxGridY) {
      const dim3 grid(x, (unsigned)std::min(plan.steps[i].problems - f, kMaxGridY));
      e = launch_chained(one ? tree_step_kernel<true> : tree_step_kernel<false>, grid, kTreeThreads, st, true,
                         one ? table : table + f, s, i, plan.fine, state + f, levels);
    }
  }
  if (e != cudaSuccess) return e;
  return launch_chained(one ? tree_kernel<true> : tree_kernel<false>, dim3(plan.blocks), kTreeThreads, st, true,
                        table, p0, plan.nbig, plan.total_units, state, counter, levels, b + plan.off_cta,
                        plan.cta_bytes, out, flags);
}

cudaError_t tree_launch(const TreePlan& plan, void* ws, cudaStream_t st, cudaStream_t side, double* out, bool flags) {
  const int count = (int)plan.prob.size();
  char* b = static_cast<char*>(ws);
  if (count == 0) return cudaSuccess;
  if (plan.nbig == 0) return launch_small(plan, b, st, out, flags);
  if (plan.nbig == count) return launch_large(plan, b, st, out, flags);
  // Both kinds: chains of dependent steps that leave most of the GPU idle, so side by side (a
  // sampler run of 16 samples, 40 modes, 3.18 ms; 3.70 one after the other).
  if (!side) {
    const cudaError_t e = launch_small(plan, b, st, out, flags);
    return e == cudaSuccess ? launch_large(plan, b, st, out, flags) : e;
  }
  cudaEvent_t fork = nullptr, join = nullptr;
  cudaError_t e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(fork, st);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(side, fork, 0);
  if (e == cudaSuccess) {
    e = launch_small(plan, b, side, out, flags);
    cudaError_t j = cudaEventRecord(join, side);  // whatever was launched is waited for
    if (e == cudaSuccess && j == cudaSuccess) e = launch_large(plan, b, st, out, flags);
    if (j == cudaSuccess) j = cudaStreamWaitEvent(st, join, 0);
    if (e == cudaSuccess) e = j;
  }
  if (fork) cudaEventDestroy(fork);
  if (join) cudaEventDestroy(join);
  return e;
}

cudaError_t tree_run(TreePlan* plan, const BatchInput* in, void* ws, void* host, cudaStream_t st,
                     cudaStream_t side, double* out3, std::vector<int>* again) try {
  const size_t count = plan->prob.size();
  // The kernels write the results straight to page-locked memory: with a copy to pageable memory
  // instead (and the matrix of gbsh_lhaf copied from there), a call takes 75 us at N = 16, not 61.
  std::vector<double> pageable(host ? 0 : 3 * count);
  double* res = host ? static_cast<double*>(host) : pageable.data();
  double* out = host ? res : reinterpret_cast<double*>(static_cast<char*>(ws) + plan->off_out);
  cudaError_t e = tree_stage(plan, in, ws, st);
  if (e == cudaSuccess) e = tree_launch(*plan, ws, st, side, out, true);
  if (e == cudaSuccess && !host && count > 0)
    e = cudaMemcpyAsync(res, out, sizeof(double) * 3 * count, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  for (size_t q = 0; q < count; ++q) {
    const int p = plan->order[q];
    if (res[3 * q + 2] != 0.0) again->push_back(p);
    out3[3 * (size_t)p] = res[3 * q];
    out3[3 * (size_t)p + 1] = res[3 * q + 1];
    out3[3 * (size_t)p + 2] = 0.0;
  }
  std::sort(again->begin(), again->end());
  return cudaSuccess;
} catch (const std::bad_alloc&) {  // before anything is launched or after it has ended
  return cudaErrorMemoryAllocation;
}

const unsigned* tree_flag(const TreePlan& plan, void* ws) {
  return &reinterpret_cast<const TreeState*>(static_cast<const char*>(ws) + plan.off_state)->bad;
}

}  // namespace gbsh
