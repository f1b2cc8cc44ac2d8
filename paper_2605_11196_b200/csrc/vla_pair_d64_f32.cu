// Pair kernel, d = 64, f32 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(64, float, d64_f32)
