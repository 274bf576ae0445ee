// Row kernel, FP32 scenario groups: the fused solve, 168 registers per thread.
#include "ucn_launch.cuh"

UCN_DEFINE_ROWS_SCP(Quad12, true, false, ROWS_WIDE_THREADS, false)
