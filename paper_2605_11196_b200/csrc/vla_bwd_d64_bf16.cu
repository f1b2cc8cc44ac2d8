// Chunked backward pass, d = 64, bf16 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(64, uint16_t, d64_bf16)
