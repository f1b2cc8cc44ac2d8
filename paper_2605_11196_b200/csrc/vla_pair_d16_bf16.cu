// Pair kernel, d = 16, bf16 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(16, uint16_t, d16_bf16)
