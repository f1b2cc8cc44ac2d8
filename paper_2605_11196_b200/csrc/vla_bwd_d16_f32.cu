// Chunked backward pass, d = 16, f32 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(16, float, d16_f32)
