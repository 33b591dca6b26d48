// Host interface of the elimination-tree evaluation (lhaf_tree.cu; the method is described in
// lhaf_tree.cuh).
#pragma once

#include <cstddef>
#include <vector>

#include <cuda_runtime.h>

#include "lhaf_types.cuh"

namespace gbsh {

// One problem of a launch. A small one is worked off whole by a cluster of CTAs. Of the others the
// levels n .. m1 are computed breadth first by the whole GPU; each node of level m1 is a unit that
// one CTA works off: depth first, two nodes a level, down to level `top`, then breadth first.
struct TreeProblem {
  BatchInput in;
  int Ne, n;       // padded size, Ne = 2 n >= 4
  int m1, top;
  unsigned unit_base, units;
  size_t root;     // byte offset of its levels n .. m1
};

// Running state of a problem: exact limb sums of the signed mean, and how to undo the scale.
struct TreeState {
  unsigned long long sum[6];
  double fac_hi, fac_lo;
  int exp2;
  unsigned done;
  unsigned bad;    // overflow, or a result too small for the fixed-point resolution
  unsigned pad;
};

// Layout of the evaluation of `count` problems in one workspace (byte offsets).
struct TreePlan {
  std::vector<TreeProblem> prob;   // in launch order
  std::vector<int> order;          // prob[q] is the caller's problem order[q]
  int nbig;                        // prob[0 .. nbig) are large, the others small
  int cluster, clusters;           // CTAs per cluster and clusters of the small ones' launch
  size_t small_bytes;              // scratch per cluster
  unsigned total_units;
  int fine;                        // breadth-first steps of at most so many pieces run in pieces
  int blocks;
  struct Step { int problems; int tasks; };
  std::vector<Step> steps;         // breadth-first eliminations: problems that take part (the
                                   // first ones), most tasks of one of them
  size_t cta_bytes;                // scratch per CTA
  size_t off_prob, off_state, off_counter, off_out, off_root, off_cta, off_small, bytes;
};

// Sizes 0 are left out (their loop hafnian is 1): `Ns` entries must be 1..kMaxN.
cudaError_t tree_plan(const int* Ns, int count, size_t base_off, TreePlan* plan);

// Evaluates the problems of `plan` (in[i]: input of the caller's problem i) in `ws` on `st`. `side`: a
// stream that nothing else uses until `st` has been waited for, to which part of the work may be
// forked from `st` and joined back, or null.
// Result of launch-order problem q, if `flags`: three doubles at out + 3 q: re, im, and 1 where
// the problem has to be evaluated by the subset sum instead (0 otherwise). Without (one-problem
// launches): re, im, and the flag at tree_flag().
cudaError_t tree_launch(const TreePlan& plan, void* ws, cudaStream_t st, cudaStream_t side, double* out, bool flags);

// Fills in the inputs and, for more than one problem, uploads the table.
cudaError_t tree_stage(TreePlan* plan, const BatchInput* in, void* ws, cudaStream_t st);

// Stages and launches `plan`, waits, and copies the results to out3[3 i ..] of the caller's
// problem i (re, im, 0); problems to be evaluated by the subset sum are added to `again`.
// `host`: page-locked memory of at least 24 bytes a problem that the call may use, or null.
cudaError_t tree_run(TreePlan* plan, const BatchInput* in, void* ws, void* host, cudaStream_t st,
                     cudaStream_t side, double* out3, std::vector<int>* again);

// Device address of a one-problem launch's fallback flag (nonzero: evaluate by the subset sum).
const unsigned* tree_flag(const TreePlan& plan, void* ws);

}  // namespace gbsh
