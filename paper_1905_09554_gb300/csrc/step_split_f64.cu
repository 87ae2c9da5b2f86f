// The two-kernel step of every collision for CodecF64 storage.
#include "step_split.cuh"

namespace lbm {

cudaError_t split_step_f64(const SplitLaunch& l, int coll, void* src, void* dst, void* psi) {
    return split_collisions<CodecF64>(l, coll, src, dst, psi);
}

}  // namespace lbm
