// Row kernel, FP32: the stand-alone ADMM call.
#include "ucn_launch.cuh"

UCN_DEFINE_ROWS_ADMM(Quad12, false, ROWS_THREADS, true)
UCN_DEFINE_ROWS_ADMM(Quad12, false, ROWS_WIDE_THREADS, false)
UCN_DEFINE_ROWS_ADMM(Quad12, true, ROWS_THREADS, true)
