// The two-kernel FP64 step of every collision.
#include "step_split.cuh"

namespace lbm {

cudaError_t split_step_f64(const SplitLaunch& l, int coll, void* src, void* dst, void* psi) {
    switch (coll) {
        case COLL_SRT: return split_step<COLL_SRT>(l, src, dst, psi);
        case COLL_MRT: return split_step<COLL_MRT>(l, src, dst, psi);
        case COLL_MRT_SPARSE: return split_step<COLL_MRT_SPARSE>(l, src, dst, psi);
        case COLL_MRT_UNIT: return split_step<COLL_MRT_UNIT>(l, src, dst, psi);
        default: return split_step<COLL_MRT_SHEAR>(l, src, dst, psi);
    }
}

}  // namespace lbm
