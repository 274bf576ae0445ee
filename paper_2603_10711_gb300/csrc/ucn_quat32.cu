// Kernel instantiations: 13-state quaternion quadrotor, FP32 path with refinement:
// the linearisation; solves and ADMM calls run on the row kernel, in its own units
// (ucn_quat32_rows*.cu).
#include "ucn_launch.cuh"
UCN_DEFINE_LAUNCHERS(quat32, Quat13, float, true)
