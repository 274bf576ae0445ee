// Row kernel, FP32: the fused solve, an instance over a cluster.
#include "ucn_launch.cuh"

UCN_DEFINE_ROWS_SCP(Quat13, false, true, ROWS_THREADS, false)
