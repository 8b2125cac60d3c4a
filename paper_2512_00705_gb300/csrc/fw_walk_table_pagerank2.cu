// fw_walk_table_pagerank2.cu -- the walk kernel's variants for tables of pagerank2 jobs.
#include "fw_walk.cuh"

WALK_LAUNCHES(table_pagerank2, kMaxJobs, ALGO_PAGERANK2)
