// solve_launch.h - the pieces of the per-sweep-point solve that live in files of their own.
#pragma once

#include "internal.h"

namespace ssm {

using SolveKernel = void (*)(const double* Kfull, const double* KZ, int64_t n_t, int nv, int nvh, double tau,
                             double xlo, double xhi, const double* mu, int ldmu, int K, double floor_scale,
                             double* work, double* dos, int32_t* rank, int* flag, const double* floor_pt,
                             const int32_t* perm, int64_t n_slot, bool pinv, const int32_t* n_dev);

// The kernel whose hybrid columns take the factored routes (solve_hyb.cu).
SolveKernel solve_kernel_hyb();

// Points of n_v <= SOLVE_SMALL_N without hybrid columns, a warp each (solve_small.cu); what
// it leaves goes into pend (pend[0]: the number).
constexpr int SOLVE_SMALL_N = 32;
cudaError_t launch_solve_small(const double* Kfull, const double* KZ, int64_t n_t, int n_v, double tau, double xlo,
                               double xhi, const double* mu, int ldmu, int K, double floor_scale, double* dos,
                               int32_t* rank, const double* floor_pt, int32_t* pend, cudaStream_t s);

}  // namespace ssm
