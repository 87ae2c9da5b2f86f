// Launches of kernels that follow one another on a stream without waiting for
// the previous one's end to be set up (programmatic dependent launch): a
// kernel's blocks are placed while the last blocks of the one before finish, and
// wait in chain_begin() until that one is complete.  Between
// kernels of a few microseconds this hides the launch: 65,536 cells, FP32, two
// kernels a step: 8.2 -> 5.0 us a step.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace lbm {

// First statement of a kernel launched with launch_chained: nothing that an
// earlier kernel wrote is read, and nothing that it reads is written, before.
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's blocks be placed once every block got here: late in
// the kernel, so that they find the SMs evenly free (placed from the start
// they piled up on some: FP64 32x32x64 1.41 -> 2.38 ms per 50 steps).
__device__ __forceinline__ void chain_end() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Cells up to which kernels are chained: of the moment and adjoint kernels,
// whose launches take some 30 us there, and of the two-kernel step's pair.
// Beyond, grids are many rounds of blocks long and want plain stream order: their
// successor's blocks would take places among their last ones (FP32 steps of 19.6 M
// cells in two kernels 583 us plain, 712 chained).
constexpr long long kChainCells = 1500000, kChainSplitCells = 400000;

// chain: false launches in plain stream order.
template <class... P, class... A>
cudaError_t launch_chained(bool chain, void (*kernel)(P...), dim3 grid, dim3 block, size_t shared, cudaStream_t stream,
                           A&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = shared;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
}

}  // namespace lbm
