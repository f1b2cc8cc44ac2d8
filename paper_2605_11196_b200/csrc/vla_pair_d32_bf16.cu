// Pair kernel, d = 32, bf16 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(32, uint16_t, d32_bf16)
