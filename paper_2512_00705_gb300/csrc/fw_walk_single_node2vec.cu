// fw_walk_single_node2vec.cu -- the walk kernel's variants for one node2vec job.
#include "fw_walk.cuh"

WALK_LAUNCHES(single_node2vec, 1, ALGO_NODE2VEC)
