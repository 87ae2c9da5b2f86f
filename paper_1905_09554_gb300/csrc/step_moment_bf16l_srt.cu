// Moment kernels for CodecBF16Local storage with the COLL_SRT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(bf16l_srt, CodecBF16Local, COLL_SRT)
