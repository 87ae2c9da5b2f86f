// Moment kernels for CodecF16Dev storage with the COLL_SRT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(f16_srt, CodecF16Dev, COLL_SRT)
