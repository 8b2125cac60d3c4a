// fw_walk_table_metapath.cu -- the walk kernel's variants for tables of metapath jobs.
#include "fw_walk.cuh"

WALK_LAUNCHES(table_metapath, kMaxJobs, ALGO_METAPATH)
