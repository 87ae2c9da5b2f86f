// Moment kernels for CodecF16Dev storage with the COLL_MRT_UNIT collision.
#include "step_moment.cuh"

LBM_MOMENT_INSTANCE(f16_mrtu, CodecF16Dev, COLL_MRT_UNIT)
