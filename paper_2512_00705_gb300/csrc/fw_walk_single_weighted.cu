// fw_walk_single_weighted.cu -- the walk kernel's variants for one weighted job.
#include "fw_walk.cuh"

WALK_LAUNCHES(single_weighted, 1, ALGO_WEIGHTED)
