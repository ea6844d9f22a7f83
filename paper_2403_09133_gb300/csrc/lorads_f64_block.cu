// Plain FP64 form of the one-CTA solver kernel (small problems and batches), a unit of its own
// so that the units compile in parallel.  Earlier builds of this kernel diverged on matrix
// completion after code changes elsewhere in the solver; the cause was the missing convergence of
// a team's lanes described at team_sum.
#include "lorads_kernels.cuh"
namespace lorads {
LORADS_DEFINE_SOLVE_LAUNCH_BLOCK(double, 0)
}
