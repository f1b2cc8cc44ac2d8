// Pair kernel, d = 128, bf16 inputs.
#include "vla_pair_launch.cuh"

VLA_DEFINE_PAIR_TU(128, uint16_t, d128_bf16)
