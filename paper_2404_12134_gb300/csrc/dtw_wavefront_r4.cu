// DTW wavefront instances: rows per lane R = 4, no band, squared l2 local cost.
#include "dtw_lean_impl.cuh"

WTS_LEAN_ENTRY(r4, 4, kCostSqEuclid)
