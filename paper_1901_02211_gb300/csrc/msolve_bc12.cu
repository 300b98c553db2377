// The multi-shift solver for RHS tiles of 12 columns.
#include "msolve.cuh"

template int solve_bc<12>(const std::vector<LatIn> &, double, int, double *, int, int);
template float time_kind_bc<12>(smpq_ctx *, int, int, int, int, int, void *, double *, double *, int *);
