// Moment kernels for CodecBF16Dev storage with the COLL_SRT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(bf16_srt, CodecBF16Dev, COLL_SRT)
