// The multi-shift solver for RHS tiles of 24 columns.
#include "msolve.cuh"

template int solve_bc<24>(const std::vector<LatIn> &, double, int, double *, int, int);
template float time_kind_bc<24>(smpq_ctx *, int, int, int, int, int, void *, double *, double *, int *);
