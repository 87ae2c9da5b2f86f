// Moment kernels for CodecBF16Local storage with the COLL_MRT_UNIT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(bf16l_mrtu, CodecBF16Local, COLL_MRT_UNIT)
