// Chunked backward pass, d = 32, bf16 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(32, uint16_t, d32_bf16)
