// Fan kernel, FP64 12-state quadrotor: 16 lanes per node, an instance over a cluster.
#include "ucn_launch.cuh"

UCN_DEFINE_FAN(16, true)
