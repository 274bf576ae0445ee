// Fan kernel, FP64 12-state quadrotor: 16 lanes per node.
#include "ucn_launch.cuh"

UCN_DEFINE_FAN(16, false)
