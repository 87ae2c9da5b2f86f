// The two-kernel step of every collision for CodecF32 storage.
#include "step_split.cuh"

namespace lbm {

cudaError_t split_step_f32(const SplitLaunch& l, int coll, void* src, void* dst, void* psi) {
    return split_collisions<CodecF32>(l, coll, src, dst, psi);
}

}  // namespace lbm
