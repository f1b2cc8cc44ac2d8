// Pair kernel, d = 32, f32 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(32, float, d32_f32)
