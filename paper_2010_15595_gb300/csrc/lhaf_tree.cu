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
#include <numeric>

#include "lhaf_kernels.cuh"
#include "lhaf_tree.cuh"
#include "lhaf_tree.h"

namespace gbsh {

namespace {

constexpr int kTreeThreads = 128;
constexpr int kTreeCtasPerSm = 6;
constexpr int kTreeTop = 6;  // level from which a unit is worked off breadth first
// Smallest scaled result that is kept. The tree's absolute error is about 2^-80 (against a
// 113-bit evaluation), so 2^-28 leaves it at 2^-52 of the result. The subset sum it would be
// handed back to is itself 2^-47 off at N = 32, 2^-42 at N = 40 and 2^-31 at N = 56, so the line
// follows it down from N = 28 on: 2^-44 relative at N = 40, 2^-34 at N = 56.
__device__ __forceinline__ int tree_min_exp(int n) { return n > 14 ? -28 - (4 * (n - 14)) / 3 : -28; }

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

// x m 2^e in units of 2^-81 as limbs; bad |= it does not fit (or x is not finite).
__device__ void to_fixed(double x, int m, int e, int& h, int& mm, int& l, unsigned& bad) {
  if (!(fabs(x) <= 1.7976931348623157e308)) bad = 1;
  int ex;
  const double f = frexp(x, &ex);
  const long long i = (long long)ldexp(f, 53) * m;  // < 2^63: 53 bits times at most 31^2
  const int sh = ex - 53 + e + kTreeFrac;
  __int128 v = i;
  if (i == 0) {
    v = 0;
  } else if (sh >= 0) {
    if (sh > 62) bad = 1;
    v <<= (sh > 62 ? 62 : sh);
  } else if (sh < -100) {
    v = 0;
  } else {
    v = (v + ((__int128)1 << (-sh - 1))) >> (-sh);
  }
  const __int128 lim = (__int128)1 << 82;
  if (v >= lim || v <= -lim) bad = 1;
  l = sext28((long long)v);
  v = (v - l) >> kLimbBits;
  mm = sext28((long long)v);
  v = (v - mm) >> kLimbBits;
  h = (int)(long long)v;
}

template <class T, class F>
__device__ T block_reduce(T x, T* sh, F f) {
  __syncthreads();
  sh[threadIdx.x] = x;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] = f(sh[threadIdx.x], sh[threadIdx.x + w]);
    __syncthreads();
  }
  return sh[0];
}

__device__ __forceinline__ double2 tree_entry(const BatchInput& in, int r, int c) {
  const int ir = in.idx ? in.idx[r] : r, ic = in.idx ? in.idx[c] : c;
  if (r == c && in.diag) return in.diag[ir];
  return in.base[(size_t)ir * in.ld + ic];
}

constexpr int kRootThreads = 256;

// kOne: one problem, passed as a kernel argument; otherwise a table in device memory.
template <bool kOne>
__global__ void __launch_bounds__(kRootThreads)
tree_root_kernel(const TreeProblem* __restrict__ table, TreeProblem one,
                 TreeState* __restrict__ state, unsigned* __restrict__ counter, Fxc* __restrict__ roots) {
  __shared__ float2 a[kMaxN * kMaxN];
  __shared__ double sh[kRootThreads];
  __shared__ int s_m, s_e;
  const TreeProblem P = kOne ? one : table[blockIdx.x];
  const int tid = threadIdx.x, N = P.in.N;
  auto dmax = [](double x, double y) { return x > y ? x : (y > x ? y : (x == x ? x : (y == y ? y : x))); };
  auto dsum = [](double x, double y) { return x + y; };
  unsigned bad = 0;
  // largest entry off the diagonal, loop weights
  double am = 0.0, vm = 0.0, v2 = 0.0;
  for (int e = tid; e < N * N; e += kRootThreads) {
    const int r = e / N, c = e - r * N;
    const double2 z = tree_entry(P.in, r, c);
    const double m = hypot(z.x, z.y);
    if (!(m <= 1.7976931348623157e308)) bad = 1;
    if (r == c) {
      vm = dmax(vm, m);
      v2 += m * m;
    } else {
      am = dmax(am, m);
    }
  }
  am = block_reduce(am, sh, dmax);
  vm = block_reduce(vm, sh, dmax);
  v2 = block_reduce(v2, sh, dsum);
  // rho = |A^H A|_F / |A|_F, the root of the mean of sigma^2 weighted by sigma^2: equal to the
  // spectral norm for flat and for rank-one spectra. Single precision is plenty for a scale.
  const double inv = am > 0.0 ? 1.0 / am : 0.0;
  float f2 = 0.f, g2 = 0.f;
  for (int e = tid; e < N * N; e += kRootThreads) {
    const int r = e / N, c = e - r * N;
    float2 w = make_float2(0.f, 0.f);
    if (r != c) {
      const double2 z = tree_entry(P.in, r, c);
      w = make_float2((float)(z.x * inv), (float)(z.y * inv));
    }
    a[e] = w;
    f2 += w.x * w.x + w.y * w.y;
  }
  __syncthreads();
  for (int e = tid; e < N * (N + 1) / 2; e += kRootThreads) {
    int i, j;
    tree_pair(e, i, j);  // i < j + 1: (i, j - 1) runs over the upper triangle
    --j;
    float re = 0.f, im = 0.f;
    for (int k = 0; k < N; ++k) {
      const float2 x = a[k * N + i], y = a[k * N + j];  // conj(x) y
      re += x.x * y.x + x.y * y.y;
      im += x.x * y.y - x.y * y.x;
    }
    g2 += (i == j ? 1.f : 2.f) * (re * re + im * im);
  }
  const double F2 = block_reduce((double)f2, sh, dsum);
  const double G2 = block_reduce((double)g2, sh, dsum);
  if (tid == 0) {
    // The loop weights enter g as exp of about |v|^2 / 2 spread over n pairs, hence |v|^2 / 8;
    // no single entry may come near the format's limit.
    double den = F2 > 0.0 ? am * sqrt(G2 / F2) : 0.0;
    den = dmax(dmax(den, am), dmax(v2 * 0.125, vm * vm));
    if (!(den > 0.0)) den = 1.0;
    const double s = rsqrt(den);  // vertex scale, its mantissa cut to 5 bits: exact products
    if (!(s > 1e-300 && s < 1e300)) bad = 1;
    int ex;
    const double f = frexp(s, &ex);
    s_m = (int)(f * 32.0);
    s_e = ex - 1;  // scale = m / 16 * 2^e
    if (s_m < 16 || s_m > 31) { s_m = 16; s_e = 0; bad = 1; }
    // 1 / scale^N: (16 / m)^N in double-double by squaring, exponents apart
    double bh = 16.0 / s_m, bl = __fma_rn(-bh, (double)s_m, 16.0) / s_m, h = 1.0, l = 0.0;
    for (int k = N; k > 0; k >>= 1) {
      if (k & 1) dd_mul(h, l, bh, bl, h, l);
      dd_mul(bh, bl, bh, bl, bh, bl);
    }
    TreeState& S = state[blockIdx.x];
    for (int i = 0; i < 6; ++i) S.sum[i] = 0;
    S.fac_hi = h;
    S.fac_lo = l;
    S.exp2 = -kTreeFrac - (P.n >= 3 ? P.n - 3 : 0) - s_e * N + (P.Ne - N);
    S.done = 0;
    S.bad = 0;
    if (blockIdx.x == 0) *counter = 0;
  }
  __syncthreads();
  const int m = s_m, e2 = s_e;
  // root level: vertex 2 p is index p, vertex 2 p + 1 is index p + n; padding vertices have no
  // edges, loop weight one and scale one half
  Fxc* A = roots + P.root;
  const int polys = tree_polys(P.n), edges = P.Ne * (P.Ne - 1) / 2;
  for (int p = tid; p < polys; p += kRootThreads) {
    int j, k;
    if (p < edges) tree_pair(p, j, k); else j = k = p - edges;
    const int r = (j & 1) ? (j >> 1) + P.n : (j >> 1), c = (k & 1) ? (k >> 1) + P.n : (k >> 1);
    Fxc v{};
    if (r < N && c < N) {
      const double2 z = tree_entry(P.in, r, c);
      const int mm = j == k ? m : m * m, ee = j == k ? e2 - 4 : 2 * e2 - 8;
      to_fixed(z.x, mm, ee, v.rh, v.rm, v.rl, bad);
      to_fixed(z.y, mm, ee, v.ih, v.im, v.il, bad);
    } else if (j == k) {
      v.rh = 1 << (kTreeFrac - 1 - 2 * kLimbBits);
    }
    fx_store(A + p, v);
  }
  if (tid == 0) {
    Fxc v{};
    v.rh = 1 << (kTreeFrac - 2 * kLimbBits);
    fx_store(A + polys, v);  // g = 1
  }
  if (__syncthreads_or((int)bad) && tid == 0) state[blockIdx.x].bad = 1;
}

// The problem's signed mean from its limb sums, to double.
__device__ void tree_result(const TreeProblem& P, TreeState* S, double* out, bool flags) {
  double v[2];
  double top = 0.0;
  for (int c = 0; c < 2; ++c) {
    const long long h = (long long)__ldcg(&S->sum[3 * c]), m = (long long)__ldcg(&S->sum[3 * c + 1]),
                    l = (long long)__ldcg(&S->sum[3 * c + 2]);
    __int128 r = (((__int128)h << kLimbBits) + m);
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

template <bool kOne>
__global__ void __launch_bounds__(kTreeThreads, kTreeCtasPerSm)
tree_step_kernel(const TreeProblem* __restrict__ table, TreeProblem one, int step,
                 TreeState* __restrict__ state, Fxc* __restrict__ levels) {
  const TreeProblem P = kOne ? one : table[blockIdx.y];
  if (P.n - step <= P.m1) return;  // fewer steps than another problem's
  const TreePhase s = tree_step_phase(levels + P.root, P.n, step);
  const unsigned t = blockIdx.x * kTreeThreads + threadIdx.x;
  unsigned bad = 0;
  if (t < tree_tasks(s)) {
    int x;
    Fxc z;
    tree_task(s, t, x, z, bad);
  }
  if (bad) atomicOr(&state[blockIdx.y].bad, 1u);
}

template <bool kOne>
__global__ void __launch_bounds__(kTreeThreads, kTreeCtasPerSm)
tree_kernel(const TreeProblem* __restrict__ table, TreeProblem one, int count, unsigned total_units,
            TreeState* __restrict__ state, unsigned* __restrict__ counter, Fxc* __restrict__ levels,
            Fxc* __restrict__ scratch, size_t cta_elems, double* __restrict__ out, bool flags) {
  __shared__ TreeLevel lv[kMaxN / 2 + 2];  // levels m1 + 1 and m1: the unit and its parent
  __shared__ unsigned long long sum[6];
  __shared__ unsigned s_unit;
  __shared__ int s_prob;
  const int tid = threadIdx.x;
  Fxc* ws = scratch + (size_t)blockIdx.x * cta_elems;
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
    if (tid < 6) sum[tid] = 0;
    __syncthreads();
    if (s_unit >= total_units) return;
    const int prob = s_prob;
    const TreeProblem P = kOne ? one : table[prob];
    const int n = P.n, m1 = P.m1, top = P.top, unit = (int)(s_unit - P.unit_base);
    if (tid == 0) tree_unit_levels(lv, levels + P.root, ws, n, m1, top, unit);
    __syncthreads();
    unsigned bad = 0;
    for (unsigned b = 0; b < 1u << (m1 - top); ++b) {
      const int parity = __popc((unsigned)unit) + __popc(b);
      for (int i = tree_first_phase(m1, top, b); i < m1; ++i) {
        const TreePhase s = tree_unit_phase(lv, n, m1, top, unit, b, i);
        const unsigned nt = tree_tasks(s);
        for (unsigned t = tid; t < nt; t += kTreeThreads) {
          int x;
          Fxc z;
          if (tree_task(s, t, x, z, bad)) {
            const int sg = ((__popc((unsigned)x) + parity) & 1) ? -1 : 1;
            atomicAdd(&sum[0], (unsigned long long)(long long)(sg * z.rh));
            atomicAdd(&sum[1], (unsigned long long)(long long)(sg * z.rm));
            atomicAdd(&sum[2], (unsigned long long)(long long)(sg * z.rl));
            atomicAdd(&sum[3], (unsigned long long)(long long)(sg * z.ih));
            atomicAdd(&sum[4], (unsigned long long)(long long)(sg * z.im));
            atomicAdd(&sum[5], (unsigned long long)(long long)(sg * z.il));
          }
        }
        __syncthreads();
      }
    }
    const int any = __syncthreads_or((int)bad);
    TreeState* S = state + prob;
    if (tid < 6) atomicAdd(&S->sum[tid], sum[tid]);
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

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

cudaError_t tree_plan(const int* Ns, int count, size_t base_off, TreePlan* plan) {
  DeviceInfo dev;
  cudaError_t e = device_info(&dev);
  if (e != cudaSuccess) return e;
  TreePlan& T = *plan;
  T.order.resize(count);
  std::iota(T.order.begin(), T.order.end(), 0);
  std::stable_sort(T.order.begin(), T.order.end(), [&](int a, int b) { return Ns[a] > Ns[b]; });
  T.prob.resize(count);
  T.steps.clear();
  const unsigned slots = (unsigned)(kTreeCtasPerSm * dev.sm_count);
  unsigned base = 0;
  size_t root = 0;
  T.cta_elems = 1;
  for (int q = 0; q < count; ++q) {
    TreeProblem& P = T.prob[q];
    const int N = Ns[T.order[q]];
    P.Ne = std::max(4, N + (N & 1));
    P.n = P.Ne / 2;
    const int n = P.n;
    P.m1 = n;
    P.top = std::min(n, kTreeTop);
    if (n > 2) {
      --P.m1;
      const unsigned want = count == 1 ? 4 * slots : 2 * slots / (unsigned)count;
      while (P.m1 > 2 && (unsigned)tree_width(P.m1, n) < want && n - P.m1 < (n > 24 ? 11 : 12)) --P.m1;
    }
    P.top = std::min(P.top, P.m1);
    P.units = (unsigned)tree_width(P.m1, n);
    P.unit_base = base;
    base += P.units;
    P.root = root;
    root += tree_offset(P.m1 - 1, n);
    T.cta_elems = std::max(T.cta_elems, tree_scratch(n, P.m1, P.top));
    for (int i = 0; i < n - P.m1; ++i) {
      if ((int)T.steps.size() <= i) T.steps.push_back(TreePlan::Step{0, 0});
      TreePhase s{};
      s.kind = kTreeStep;
      s.n = n;
      s.M = n - i;
      s.src.q = tree_width(n - i, n);
      s.par.q = i > 0 ? tree_width(n - i + 1, n) : 0;
      T.steps[i].problems = q + 1;
      T.steps[i].tasks = std::max(T.steps[i].tasks, tree_tasks(s));
    }
  }
  T.total_units = base;
  T.blocks = (int)std::min<unsigned>(slots, base);
  size_t off = align256(base_off);
  T.off_prob = off; off = align256(off + sizeof(TreeProblem) * (size_t)count);
  T.off_state = off; off = align256(off + sizeof(TreeState) * (size_t)count);
  T.off_counter = off; off = align256(off + sizeof(unsigned));
  T.off_out = off; off = align256(off + 3 * sizeof(double) * (size_t)count);
  T.off_root = off; off = align256(off + sizeof(Fxc) * root);
  T.off_cta = off; off = align256(off + sizeof(Fxc) * T.cta_elems * (size_t)T.blocks);
  T.bytes = off;
  return cudaSuccess;
}

cudaError_t tree_stage(TreePlan* plan, const BatchInput* in, void* ws, cudaStream_t st) {
  for (size_t q = 0; q < plan->prob.size(); ++q) plan->prob[q].in = in[plan->order[q]];
  if (plan->prob.size() < 2) return cudaSuccess;
  return cudaMemcpyAsync(static_cast<char*>(ws) + plan->off_prob, plan->prob.data(),
                         sizeof(TreeProblem) * plan->prob.size(), cudaMemcpyHostToDevice, st);
}

cudaError_t tree_launch(const TreePlan& plan, void* ws, cudaStream_t st, double* value) {
  const int count = (int)plan.prob.size();
  if (count == 0) return cudaSuccess;
  char* b = static_cast<char*>(ws);
  const TreeProblem* table = count > 1 ? reinterpret_cast<const TreeProblem*>(b + plan.off_prob) : nullptr;
  TreeState* state = reinterpret_cast<TreeState*>(b + plan.off_state);
  unsigned* counter = reinterpret_cast<unsigned*>(b + plan.off_counter);
  Fxc* roots = reinterpret_cast<Fxc*>(b + plan.off_root);
  Fxc* scratch = reinterpret_cast<Fxc*>(b + plan.off_cta);
  double* out = value ? value : reinterpret_cast<double*>(b + plan.off_out);
  const bool one = count == 1;
  const TreeProblem& p0 = plan.prob[0];
  if (one)
    tree_root_kernel<true><<<1, kRootThreads, 0, st>>>(table, p0, state, counter, roots);
  else
    tree_root_kernel<false><<<count, kRootThreads, 0, st>>>(table, p0, state, counter, roots);
  for (size_t i = 0; i < plan.steps.size(); ++i) {
    const dim3 grid((plan.steps[i].tasks + kTreeThreads - 1) / kTreeThreads, plan.steps[i].problems);
    if (one)
      tree_step_kernel<true><<<grid, kTreeThreads, 0, st>>>(table, p0, (int)i, state, roots);
    else
      tree_step_kernel<false><<<grid, kTreeThreads, 0, st>>>(table, p0, (int)i, state, roots);
  }
  if (one)
    tree_kernel<true><<<plan.blocks, kTreeThreads, 0, st>>>(table, p0, count, plan.total_units, state,
                                                            counter, roots, scratch, plan.cta_elems,
                                                            out, value == nullptr);
  else
    tree_kernel<false><<<plan.blocks, kTreeThreads, 0, st>>>(table, p0, count, plan.total_units, state,
                                                             counter, roots, scratch, plan.cta_elems,
                                                             out, value == nullptr);
  return cudaGetLastError();
}

const unsigned* tree_flag(const TreePlan& plan, void* ws) {
  return &reinterpret_cast<const TreeState*>(static_cast<const char*>(ws) + plan.off_state)->bad;
}

}  // namespace gbsh
