// Chunked backward pass, d = 32, f32 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(32, float, d32_f32)
