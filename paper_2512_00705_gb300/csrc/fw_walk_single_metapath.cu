// fw_walk_single_metapath.cu -- the walk kernel's variants for one metapath job.
#include "fw_walk.cuh"

WALK_LAUNCHES(single_metapath, 1, ALGO_METAPATH)
