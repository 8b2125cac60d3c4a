// fw_walk_single_pagerank2.cu -- the walk kernel's variants for one pagerank2 job.
#include "fw_walk.cuh"

WALK_LAUNCHES(single_pagerank2, 1, ALGO_PAGERANK2)
