// Chunked backward pass, d = 64, f32 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(64, float, d64_f32)
