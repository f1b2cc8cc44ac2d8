// Pair kernel, d = 128, f32 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(128, float, d128_f32)
