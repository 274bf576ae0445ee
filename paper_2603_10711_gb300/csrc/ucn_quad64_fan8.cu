// Fan kernel, FP64 12-state quadrotor: 8 lanes per node.
#include "ucn_launch.cuh"

UCN_DEFINE_FAN(8, false)
