// Chunked backward pass, d = 128, bf16 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(128, uint16_t, d128_bf16)
