// The two-kernel step of every collision for CodecF16Local storage.
#include "step_split.cuh"

namespace lbm {

cudaError_t split_step_f16l(const SplitLaunch& l, int coll, void* src, void* dst, void* psi) {
    return split_collisions<CodecF16Local>(l, coll, src, dst, psi);
}

}  // namespace lbm
