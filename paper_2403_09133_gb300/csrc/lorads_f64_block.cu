// Plain FP64 form of the one-CTA solver kernel (small problems and batches), a unit of its own
// so that the units compile in parallel.  Earlier builds of this kernel diverged on matrix
// completion after code changes elsewhere in the solver; not seen since the lanes of a warp converge at
// team_sum (see there).  By default FP64 solves leave one CTA from n = 40 or 256 (default_ctas); batches
// and grid = 1 come here, and the GPU tests ask for it by grid = 1: bit-identical repeats, agreement with
// the whole-GPU kernel and, step by step, with the oracle.
#include "lorads_kernels.cuh"
namespace lorads {
LORADS_DEFINE_SOLVE_LAUNCH_BLOCK(double, 0)
}
