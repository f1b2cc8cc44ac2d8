// Chunked backward pass, d = 128, f32 inputs.
#include "vla_bwd_launch.cuh"

VLA_DEFINE_BWD_TU(128, float, d128_f32)
