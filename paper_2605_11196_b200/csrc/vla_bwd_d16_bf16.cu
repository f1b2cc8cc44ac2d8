// Chunked backward pass, d = 16, bf16 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(16, uint16_t, d16_bf16)
