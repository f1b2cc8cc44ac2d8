// Pair kernel, d = 16, f32 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(16, float, d16_f32)
