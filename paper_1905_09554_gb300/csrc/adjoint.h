// Launchers of the discrete-adjoint kernels (adjoint_kernels.cu), used by the
// host API in lbm_sc.cu.
#pragma once
#include <cuda_runtime.h>

namespace lbm {

struct AdjointArgs {
    int nx, ny, nz;
    long long n;
    double G, tau, omega, rho0;
    double gw;                      // -G (gwf: -G/36), as force_of takes it
    float Gf, tauf, omegaf, rho0f, gwf;  // rounded on the host for the FP32 kernels
    int grid;  // blocks of adjoint_threads() threads (grid-stride loops)
    bool tau1; // tau = 1: lam holds four values a cell {A, B}, lam_a = A + c_a.B, and gr is not used
};

int adjoint_threads();
int adjoint_rows_per_block();  // the step kernels walk x rows, this many per block
// The adjoint field is kept as lam_a(x) + gr(x): the force's contribution to
// dJ/drho is the same for every population, so it is stored once per cell
// (gr, n values) instead of being added to the 19 populations.
//
// One reverse step: (lam_out, gr_out) = (dS/df)^T (lam_next + gr_next) at the
// forward state f; this step's dJ/dG and dJ/dtau are added to the per-block
// running sums in `partials` (2 * grid doubles, zeroed before the first
// step), which adjoint_reduce adds into acc[0..1] once after the last step.
// psi (n) and gF (4n: {psi gF, S.gF} per cell, see adj_collide_kernel) are
// scratch; lam and gF are 16-byte aligned;
// acc is not touched here.  Needs nx*ny*nz < 2^32 (32-bit cell indices).
// psi_ready: psi already holds psi of f (the step kernel wrote it during the
// recomputation); otherwise it is computed first.
cudaError_t adjoint_step(const AdjointArgs& a, bool f64, const void* f, void* psi, bool psi_ready,
                         const void* lam_next, const void* gr_next, void* lam_out, void* gr_out, void* gF,
                         double* partials, double* acc, cudaStream_t st);
// The same at tau = 1 in FP32 from a state's moment fields (step_moment.cuh,
// 4 fields).  lam_next2: lam of two steps on, nullptr in the last step; first:
// step 0, from a state at rest.
cudaError_t adjoint_step_moments(const AdjointArgs& a, const float* moments, float* psi, bool psi_ready,
                                 const void* lam_next, const void* lam_next2, void* lam_out, void* gF,
                                 double* partials, bool first, cudaStream_t st);
cudaError_t adjoint_reduce(const AdjointArgs& a, const double* partials, double* acc, cudaStream_t st);
// lam_a = dJ/drho (every a), gr = 0.
cudaError_t adjoint_seed(const AdjointArgs& a, bool f64, const double* dJdrho, void* lam, void* gr, cudaStream_t st);
// dJ/drho0 = sum_a w_a lam_a + gr.
cudaError_t adjoint_rho0(const AdjointArgs& a, bool f64, const void* lam, const void* gr, double* out,
                         cudaStream_t st);

}  // namespace lbm
