// Moment kernels for CodecF16Local storage with the COLL_SRT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(f16l_srt, CodecF16Local, COLL_SRT)
