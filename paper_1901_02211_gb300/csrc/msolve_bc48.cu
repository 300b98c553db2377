// The multi-shift solver for RHS tiles of 48 columns.
#include "msolve.cuh"

template int solve_bc<48>(const std::vector<LatIn> &, double, int, double *, int, int);
template float time_kind_bc<48>(smpq_ctx *, int, int, int, int, int, void *, double *, double *, int *);
