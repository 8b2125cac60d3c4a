// fw_walk_table_weighted.cu -- the walk kernel's variants for tables of weighted jobs.
#include "fw_walk.cuh"

WALK_LAUNCHES(table_weighted, kMaxJobs, ALGO_WEIGHTED)
