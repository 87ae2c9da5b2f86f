// The two-kernel step of every collision for CodecBF16Dev storage.
#include "step_split.cuh"

namespace lbm {

cudaError_t split_step_bf16(const SplitLaunch& l, int coll, void* src, void* dst, void* psi) {
    return split_collisions<CodecBF16Dev>(l, coll, src, dst, psi);
}

}  // namespace lbm
