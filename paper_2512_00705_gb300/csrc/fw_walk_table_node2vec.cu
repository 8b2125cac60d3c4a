// fw_walk_table_node2vec.cu -- the walk kernel's variants for tables of node2vec jobs.
#include "fw_walk.cuh"

WALK_LAUNCHES(table_node2vec, kMaxJobs, ALGO_NODE2VEC)
