// solve_hyb.cu - the per-sweep-point solve with the factored routes of hybrid columns.
#include "solve_body.cuh"
#include "solve_launch.h"

namespace ssm {

SolveKernel solve_kernel_hyb() { return solve_kernel<true>; }

}  // namespace ssm
