// Moment kernels for CodecF16Local storage with the COLL_MRT_UNIT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(f16l_mrtu, CodecF16Local, COLL_MRT_UNIT)
