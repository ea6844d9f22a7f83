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
  int lanes;          // lanes of a factor row at the largest rank
  int threads;        // the caller's CTA size; 0: library choice
  int sms;
};

// One CTA for small problems, the whole GPU from a few hundred rows up (n >= 512).  The FP64 form
// leaves one CTA earlier, since one SM's FP64 unit (a warp instruction every 16 clocks) bounds it: from
// n = 256 with diagonal constraints and from n = 40 in the general form, whose rows carry many
// entries.  It takes the CTAs that its rows fill and no more, a team of lanes per row with diagonal
// constraints and a warp per row in the general form: further CTAs only wait at the barriers, and they
// keep other callers' solves off the GPU.  Measured (ms, grids of 1 / 8 / 16 / 32 / 76 / 152):
//   ER degree 6, 60 iterations      n = 256   10.4  10.2  10.3  10.3  10.4  10.4
//                                   n = 300   21.2  10.4  10.3  10.3  10.5  10.7
//                                   n = 511   32.1  11.3  11.3  11.2  11.4  11.6
//   the same, row-block direct      n = 511   21.2   8.7   8.7   8.6   8.7   8.9
//   completion, 15 iterations       n = 60    42.5  15.7  12.4  12.4  12.6  13.0
//                                   n = 200    157  36.4  24.4  16.5  12.7  13.2
//                                   n = 500    329  79.3  47.6  32.4  25.3  22.1
//   theta, 15 iterations            n = 20    31.5  33.6  33.6  33.8  34.0  34.6
//                                   n = 40    24.6  21.0  19.8  19.7  19.8  19.7
// Eight callers side by side, a thread, stream and problem each (solves a second, grids of 1 / 8 /
// 16 / 152): ER n = 256 705 / 714 / 712 / 169, n = 500 238 / 651 / 646 / 158; completion n = 60
// 108 / 270 / 328 / 148, n = 400 19 / 99 / 163 / 121 (on one CTA each, completions of n = 400 overtake
// a grid of 100 at about 50 callers).  The mixed form stays on one CTA below 512: another geometry
// sums in another order, and its FP32 iterates then differ by far more than rounding.  A CTA size
// that only the one-CTA kernel takes keeps a solve of fewer than 512 rows there.
inline int default_ctas(const SolveSize& p) {
  if (p.n >= 512) return p.sms;
  if (!p.fp64 || p.n < (p.diag_only ? 256 : 40) || p.threads > GRID_THREADS_MAX) return 1;
  const int64_t lanes = p.n * (p.diag_only ? p.lanes : 32);
  const int64_t threads = p.threads > 0 ? p.threads : SOLVER_THREADS_MIN;
  const int64_t ctas = (lanes + threads - 1) / threads;
  return (int)(ctas < 2 ? 2 : ctas > p.sms ? p.sms : ctas);
}

// Operators with a warp per row, whose 32 / G sub-teams of G lanes take an entry of the row each: whether
// the rows of A hold at most one entry per sub-team on average (an entry off the diagonal lies in two
// rows).  The Hessian then takes one entry a round, for longer rows two: with short ones the second
// is mostly past the row's end, and without it two CTAs of the FP64 kernel fit an SM where one does
// (r = 9, one / two entries a round: n = 20,000 with 6 entries a row FP64 96 / 119 us, FP32 16.5 / 18.6;
// n = 3,000 with 133 entries FP64 84 / 69).
// The FP32 product's sub-teams then form their own entries' weights, for longer rows the warp
// forms 32 at once (r = 9: 6 entries a row 13.3 / 22.1 us; 200 entries a row 41.6 / 31).
inline bool short_rows(int64_t n, int64_t entries, int lanes) {
  return entries <= n * (32 / (lanes < 32 ? lanes : 32));
}

constexpr int OP_CTAS_PER_SM = 8;   // CTAs of an operator call's launch, per SM

// FP64 operators: a row of ld doubles (ld <= 256) is ld / 2 units of 16 bytes, dealt to G lanes, at most
// 8 units each.
enum UnitWork { UNIT_SDDMM_DIAG, UNIT_SDDMM, UNIT_HESSIAN, UNIT_SPMM };
inline int unit_count(int ld, int G) { return (ld / 2 + G - 1) / G; }

// G: the fewest lanes, which issue the fewest FP64 instructions, widened up to 8 while the rows leave
// SMs idle and latency counts instead.  How many lanes per SM are too few grows with the units that a
// lane handles, one after the other; the product with C handles them once per entry of the row.
// Measured at 1,000 to 80,000 rows, r = 9, 20, 32, 48, 2 / 4 / 8 lanes (us):
//   sampled, on the diagonal   r = 9, n = 30,000  3.26 4.36 6.52     r = 32, n = 10,000  4.10 3.52 3.86
//   sampled, off the diagonal  r = 9, n = 30,000  4.07 5.41 8.62     r = 32, n = 10,000  6.04 4.60 4.65
//   Hessian                    r = 9, n = 30,000  5.24 7.16 9.73     r = 32, n = 20,000  10.6 8.47 8.92
//   product, 7 entries a row   r = 9, n = 10,000  11.5 10.1 9.19     r = 20, n = 30,000  25.0 26.0 27.8
// The Hessian and the product with 6 to 8 units per lane, whose rows take most registers, are widened
// further (Hessian r = 48, n = 10,000, 6 units 8.2, 3 units 7.3; product of degree 7,
// wider / not: r = 48, 6 units, n = 40,000 50.7 / 60.1, n = 400,000 473 / 470; r = 32, 8 units, 41.6 / 53.6 and
// 318 / 367).
inline int unit_lanes(UnitWork work, int ld, long long rows, int sms) {
  int G = 2;
  while (unit_count(ld, G) > 8 || (work == UNIT_SPMM && G < 8 && unit_count(ld, G) == 8)) G <<= 1;
  while (G < 8 && 2 * G <= ld / 2) {
    const int N = unit_count(ld, G);
    const int few = work == UNIT_SPMM         ? (N > 5 ? 3072 : 512)
                    : work == UNIT_SDDMM_DIAG ? 26 * N
                    : work == UNIT_SDDMM      ? 52 * N
                    : N > 5                   ? 512
                                              : 36 * N;
    if (rows * G >= (long long)sms * few) break;
    G <<= 1;
  }
  return G;
}

}  // namespace lorads
