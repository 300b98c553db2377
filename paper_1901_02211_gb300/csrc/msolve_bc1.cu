// The multi-shift solver for RHS tiles of 1 column.
#include "msolve.cuh"

template int solve_bc<1>(const std::vector<LatIn> &, double, int, double *, int, int);
template float time_kind_bc<1>(smpq_ctx *, int, int, int, int, int, void *, double *, double *, int *);
