// Row kernel, FP32: the stand-alone ADMM call.
#include "ucn_launch.cuh"

UCN_DEFINE_ROWS_ADMM(Mars14, false, ROWS_THREADS, false)
UCN_DEFINE_ROWS_ADMM(Mars14, true, ROWS_THREADS, false)
