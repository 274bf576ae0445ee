// Row kernel, FP32: the fused solve, 255 registers per thread.
#include "ucn_launch.cuh"

UCN_DEFINE_ROWS_SCP(Mars14, false, false, ROWS_THREADS, false)
