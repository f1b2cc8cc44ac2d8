// Pair kernel, d = 64, bf16 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(64, uint16_t, d64_bf16)
