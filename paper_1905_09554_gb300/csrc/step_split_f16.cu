// The two-kernel step of every collision for CodecF16Dev storage.
#include "step_split.cuh"

namespace lbm {

cudaError_t split_step_f16(const SplitLaunch& l, int coll, void* src, void* dst, void* psi) {
    return split_collisions<CodecF16Dev>(l, coll, src, dst, psi);
}

}  // namespace lbm
