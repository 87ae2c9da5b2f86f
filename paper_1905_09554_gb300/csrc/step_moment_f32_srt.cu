// Moment kernels for CodecF32 storage with the COLL_SRT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(f32_srt, CodecF32, COLL_SRT)
