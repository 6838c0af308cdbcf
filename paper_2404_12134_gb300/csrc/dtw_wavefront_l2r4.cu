// DTW wavefront instances: rows per lane R = 4, no band, l2-norm local cost
// (paths and the pairwise matrix).
#include "dtw_lean_impl.cuh"

WTS_LEAN_ENTRY(l2r4, 4, kCostL2)
