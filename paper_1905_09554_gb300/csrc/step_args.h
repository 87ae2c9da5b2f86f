// Arguments of the step kernels and the launch description shared between
// the host API (lbm_sc.cu) and the per-storage kernel translation units
// (step_f64.cu, step_f32.cu, step_f16.cu, step_bf16.cu).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "codec.cuh"
#include "lattice.cuh"

namespace lbm {

// Collision kernels: SRT; MRT with general rates; MRT whose rates outside
// {e, 3pxx, pww, pxy, pyz, pxz} are 1; MRT with every rate 1; MRT whose
// rates outside {3pxx, pww, pxy, pyz, pxz} are 1 (the shear rule).
enum { COLL_SRT = 0, COLL_MRT = 1, COLL_MRT_SPARSE = 2, COLL_MRT_UNIT = 3, COLL_MRT_SHEAR = 4, COLL_COUNT = 5 };

// Moments that an operator reads before the collision: rho, jx, jy, jz, then
// the second moments whose rates differ from 1.
//   SRT at tau = 1, MRT with every rate 1:      4
//   MRT, shear rule: 2 xx - yy - zz, yy - zz, xy, yz, xz:  9
//   MRT, paper's rule: xx, yy, zz, xy, yz, xz:  10
// (SRT at another tau and MRT with general rates need all 19 populations.)
__host__ __device__ constexpr int moments_of_operator(int coll) {
    return coll == COLL_MRT_SHEAR ? 9 : (coll == COLL_MRT_SPARSE ? 10 : 4);
}

struct StepArgs {
    int nx, ny, nz;
    int zchunk;           // planes per block (work item) along z
    int tiles_x, n_tiles; // xy tiles of the persistent kernel
    int n_items;          // n_tiles * number of z chunks
    long long n;          // cells = nx*ny*nz (population stride)
    double G;             // interaction strength G0 (first belt)
    double G2;            // second-belt strength of the two-belt force (kernel 6)
    double tau, omega;    // SRT relaxation time and 1/tau
    double rho0, inv_rho0;
    double s[Q];          // MRT rates, moment order
    double gw;            // the force's strength as force_of takes it: -G (gwf: -G/36)
    // (1 - s_k)/norm_k of the rows e (times 19), 3pxx, pww, pxy, pyz, pxz
    double kk[6];
    // The same parameters rounded to float once on the host, for the float
    // arithmetic of the 32- and 16-bit formats: a double-to-float conversion
    // inside the cell loop would occupy the FP64 pipe (2 lanes per SM clock).
    float Gf, tauf, omegaf, rho0f, inv_rho0f;
    float sf[Q];
    float gwf, kkf[6];
    DevParams dev;
    int* err;             // device error word (bit 0: a bounded wait timed out)
    const float* ref_src; // local-reference storage: density field of the source copy
    float* ref_dst;       // ... and of the destination copy
    int test_stall;       // failure test of the bounded waits (bulk kernel)
    // Optional (kernels 1 and 3): psi of the input state, one value per cell
    // in the arithmetic type (the adjoint's recomputation keeps it for the
    // reverse step); nullptr normally.
    void* psi_out;
    void* psi_ws;         // kernel 6: field of psi in the arithmetic type, or nullptr
};

// MRT rates in the arithmetic type R (see par() in lattice.cuh).
template <class R>
__host__ __device__ __forceinline__ const R (&rates(const StepArgs& a))[Q] {
    if constexpr (sizeof(R) == sizeof(double)) return a.s;
    else return a.sf;
}
template <class R>
__host__ __device__ __forceinline__ const R (&row_rates(const StepArgs& a))[6] {
    if constexpr (sizeof(R) == sizeof(double)) return a.kk;
    else return a.kkf;
}
// Fill the derived parameters and the float copies from the double fields.
inline void round_params(StepArgs& a) {
    constexpr int rows[6] = {1, 9, 11, 13, 14, 15};
    a.gw = -a.G;
    a.gwf = float(-a.G / 36.0);
    for (int i = 0; i < 6; ++i) {
        a.kk[i] = (1.0 - a.s[rows[i]]) / mrt_norm(rows[i]) * (i == 0 ? 19.0 : 1.0);
        a.kkf[i] = float(a.kk[i]);
    }
    a.Gf = float(a.G);
    a.tauf = float(a.tau);
    a.omegaf = float(a.omega);
    a.rho0f = float(a.rho0);
    a.inv_rho0f = float(a.inv_rho0);
    for (int k = 0; k < Q; ++k) a.sf[k] = float(a.s[k]);
}

// One box of a batch: geometry, work items and where its populations start
// (element offset) in the batch's population copies.
struct BatchBox {
    int nx, ny, nz;
    int tiles_x, n_tiles, zchunk;
    int item_begin;       // first work item of the box (items are box-major)
    long long base;       // element offset of the box's 19 population fields
    long long n;          // cells of the box (population stride)
};

struct BatchArgs {
    int nbox;
    int n_items;
    const BatchBox* boxes;  // device array of nbox entries
};

// Launch description of one step.
struct StepLaunch {
    StepArgs args;
    int kernel;           // 1 register-staged, 2 cp.async-staged, 3 pipelined,
                          // 4 bulk-copy, 5 tensor-copy, 6 two-belt force
    const CUtensorMap* tmap;  // kernel 5: tensor map of the source copy
    int tile_y;           // 4, 8 or 16 (tile width is 32)
    int grid;             // persistent grid (kernels 2 and 3)
    int coll;             // COLL_SRT .. COLL_MRT_SHEAR
    cudaStream_t stream;
};

// Kernel entry points of one (storage, collision) pair, defined in
// step_<storage>_<collision>.cu.  launch enqueues one step src -> dst;
// prepare opts kernels 2/3 in to their shared memory and returns their
// resident blocks per SM (0 = cannot run); batch / batch_prepare do the same
// for the batched step (FP64/FP32 only).
struct StepKernels {
    cudaError_t (*launch)(const StepLaunch& l, const void* src, void* dst);
    int (*prepare)(const StepLaunch& l);
    cudaError_t (*batch)(const StepLaunch& l, const BatchArgs& b, const void* src, void* dst);
    int (*batch_prepare)(const StepLaunch& l);
};

// storage: LBM_F64 .. LBM_BF16_LOCAL (0..5); coll: COLL_SRT .. COLL_MRT_SHEAR.
const StepKernels& step_kernels(int storage, int coll);

// Row length of the moment fields, and the floats of one field.
__host__ __device__ inline int moment_pitch(int nx) { return ((nx + 3) & ~3) + 4; }
inline long long moment_cells(int nx, int ny, int nz) { return (long long)moment_pitch(nx) * ny * nz; }

// Planes zs .. ze - 1 of a tile of a box: what a block of the moment kernel goes through at a time.
struct alignas(16) MomentPiece {
    int box, tile, zs, ze;
};

// Launch description of the moment kernels (step_moment.cuh).  args.tiles_x is
// that of the moment kernel's tiles; boxes: the batch's box table (nbox > 0).
struct MomentLaunch {
    StepArgs args;
    BatchArgs batch;
    const MomentPiece* pieces;  // device: block b takes pieces first[b] .. first[b + 1] - 1
    const int* first;
    int grid;             // blocks of the step
    int gather_grid;      // blocks (per box) of the populations -> moments pass
    int src_hi, dst_hi;   // which of a copy's two sets of moment fields
    cudaStream_t stream;
};

struct MomentKernels {
    // opts the step kernels in to their shared memory and returns their
    // resident blocks per SM (0 or less: cannot run)
    int (*prepare)(bool batch);
    cudaError_t (*gather)(const MomentLaunch& l, const void* pops, void* moments);
    cudaError_t (*step)(const MomentLaunch& l, const void* moments, void* out);
    cudaError_t (*emit)(const MomentLaunch& l, const void* moments, void* pops);
    int fields;           // moment fields of the collision
    int tile_x, tile_y;   // an output tile
};

// nullptr where the collision (or the storage) has no moment form.
const MomentKernels* moment_kernels(int storage, int coll);

// The step in two kernels (step_split.cuh), of one lattice or of a batch's
// boxes (batch.nbox > 0).  Its first kernel leaves, for the second, either
//  * moments != nullptr (FP64 and FP32; not for general MRT rates, and SRT only
//    at tau = 1): the moments and psi there, fields of n cells each; this may be
//    `src`, whose populations are then overwritten; or
//  * psi of `src` in the field `psi` (not for batches).
struct SplitLaunch {
    StepArgs args;
    BatchArgs batch;
    unsigned max_cells;   // of the largest box
    cudaStream_t stream;
    void* moments = nullptr;
};
cudaError_t split_step(const SplitLaunch& l, int storage, int coll, void* src, void* dst, void* psi);

}  // namespace lbm
