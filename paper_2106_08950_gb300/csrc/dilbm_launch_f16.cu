// The launchers for __half storage: every launch shape (2, 4 or 8 warps per
// block; with and without edge handling).  One translation unit per storage
// type so that the library compiles in parallel.
#include "dilbm_launch_impl.cuh"

template struct dilbm::Launch<__half>;
