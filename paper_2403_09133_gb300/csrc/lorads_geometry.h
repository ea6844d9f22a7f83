// The library's choice of CTAs for a single-problem solve (lorads_params::grid = 0).
#pragma once
#include <stdint.h>

namespace lorads {

constexpr int SOLVER_THREADS = 256;       // one-CTA solver: default CTA size ...
constexpr int BLOCK_THREADS_MAX = 384;    // ... and the largest (batches autotune 128..384)
constexpr int GRID_THREADS_MAX = 320;     // grid solver: CTA size chosen per problem
constexpr int SOLVER_THREADS_MIN = 128;   // every solver CTA: four warps, one per Lanczos chain

struct SolveSize {
  int64_t n;          // rows
  bool fp64;          // the plain FP64 form (else the mixed form)
  bool diag_only;     // every constraint one diagonal entry, at most one per row
  int threads;        // the caller's CTA size; 0: library choice
  int sms;
};

// One CTA for small problems, the whole GPU from a few hundred rows up (n >= 512).  The FP64 form
// goes over earlier, since one SM's FP64 unit (a warp instruction every 16 clocks) bounds it: from
// n = 256 with diagonal constraints (60 iterations on ER graphs of degree 6, one CTA / 152: n = 200
// 9.5 / 10.3 ms, 256 10.4 / 10.5, 320 22.7 / 11.5, 500 31.9 / 11.5), and from n = 40 in the general form,
// whose rows carry many entries (matrix completion n = 60 42.5 / 12.7 ms, 400 338 / 15; theta n = 20
// 31.5 / 34.4, 40 28.5 / 23.9).  The mixed form stays on one CTA below 512: another geometry sums in
// another order, and its FP32 iterates then differ by far more than rounding.  A CTA size that only
// the one-CTA kernel takes keeps a solve of fewer than 512 rows there.
inline int default_ctas(const SolveSize& p) {
  if (p.n >= 512) return p.sms;
  if (!p.fp64 || p.n < (p.diag_only ? 256 : 40) || p.threads > GRID_THREADS_MAX) return 1;
  return p.sms;
}

}  // namespace lorads
