// The FP64 step in two kernels without any redundant arithmetic.
//
// GB300 issues FP64 at 2 lanes an SM and clock, so an FP64 step is bound by
// its ~150 FP64 operations a cell (150 / (152 x 2 x 2.07 GHz) = 0.24 ns) while
// HBM would deliver 1600 bytes in that time.  The one-kernel steps compute psi
// of their tiles' rims again (19 additions, an exponential and a division's
// worth of work per rim cell; 0.6 rim cells per cell on the 32 x 4 tiles that
// FP64 needs) and the density twice.  Here
//   sc_fields_kernel  forms psi of every cell once, from its populations; where
//       the collision needs no more than the moments (collide.cuh), it leaves
//       those and psi in the first slots of the cell's own populations,
//   sc_push_kernel    reads psi of the 18 neighbours (through L1) and the
//       moments or populations, collides and pushes.
// The extra traffic (72 to 88 B a cell) hides behind the FP64 pipe.  Cells are dealt
// linearly to 64-thread blocks, so that small boxes fill the chip too.
#pragma once
#include "collide.cuh"
#include "step_kernel.cuh"

namespace lbm {

constexpr int kSplitThreads = 64;

// psi in slot kMoments<COLL> behind the moments (IN_PLACE), or in its own field.
template <int COLL, bool IN_PLACE>
__global__ void __launch_bounds__(kSplitThreads)
sc_fields_kernel(double* f_all, double* psi_all, const StepArgs a, const BatchArgs b) {
    constexpr int NF = kMoments<COLL>;
    unsigned n = unsigned(a.n);
    long long base = 0;
    if (b.nbox) {
        const BatchBox& bx = b.boxes[blockIdx.y];
        n = unsigned(bx.n);
        base = bx.base;
    }
    const unsigned i = blockIdx.x * kSplitThreads + threadIdx.x;
    if (i >= n) return;
    double* const f = f_all + base;
    double v[Q];
    static_for<0, Q>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        v[q] = f[q * (long long)n + i];
    });
    if constexpr (IN_PLACE) {
        double m[NF];
        moments_of<COLL, double>(v, m);
        static_for<0, NF>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            f[k * (long long)n + i] = m[k];
        });
        f[NF * (long long)n + i] = psi_of<double>(m[0], a.rho0, a.inv_rho0);
    } else {
        double m[NF];
        moments_of<COLL, double>(v, m);  // (the sums that the density does not need fall away)
        psi_all[i] = psi_of<double>(m[0], a.rho0, a.inv_rho0);
    }
}

// psi of a cell's neighbours in one plane; yo, xo: offsets of its rows and columns -1, 0, +1.
struct NeighbourPsi {
    const double* plane;
    const unsigned (&yo)[3];
    const unsigned (&xo)[3];
    template <class DX, class DY>
    __device__ __forceinline__ double operator()(DX, DY) const {
        return __ldg(plane + (yo[DY::value + 1] + xo[DX::value + 1]));
    }
};

template <int COLL, bool IN_PLACE>
__global__ void __launch_bounds__(kSplitThreads)
sc_push_kernel(const double* __restrict__ src_all, const double* __restrict__ psi_all, double* __restrict__ dst_all,
               const StepArgs a, const BatchArgs b) {
    constexpr int NF = kMoments<COLL>;
    int nx = a.nx, ny = a.ny, nz = a.nz;
    long long base = 0;
    if (b.nbox) {
        const BatchBox& bx = b.boxes[blockIdx.y];
        nx = bx.nx;
        ny = bx.ny;
        nz = bx.nz;
        base = bx.base;
    }
    const unsigned plane = unsigned(nx) * unsigned(ny), n = plane * unsigned(nz);
    const unsigned i = blockIdx.x * kSplitThreads + threadIdx.x;
    if (i >= n) return;
    const double* __restrict__ src = src_all + base;
    double* __restrict__ dst = dst_all + base;
    const double* __restrict__ psi = IN_PLACE ? src + NF * (long long)n : psi_all;
    const int z = int(i / plane), y = int((i - unsigned(z) * plane) / unsigned(nx)),
              x = int(i - unsigned(z) * plane - unsigned(y) * unsigned(nx));
    const unsigned zo[3] = {unsigned(z == 0 ? nz - 1 : z - 1) * plane, unsigned(z) * plane,
                            unsigned(z + 1 == nz ? 0 : z + 1) * plane};
    const unsigned yo[3] = {unsigned(y == 0 ? ny - 1 : y - 1) * nx, unsigned(y) * nx,
                            unsigned(y + 1 == ny ? 0 : y + 1) * nx};
    const unsigned xo[3] = {unsigned(x == 0 ? nx - 1 : x - 1), unsigned(x), unsigned(x + 1 == nx ? 0 : x + 1)};

    PsiView<double> w[3];
    static_for<0, 3>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const NeighbourPsi at{psi + zo[k], yo, xo};
        w[k].c = __ldg(psi + (zo[k] + yo[1] + xo[1]));
        psi_axis(w[k], at);
        if constexpr (k == 1) psi_diag(w[k], at);
    });
    const Force<double> F = force_of(w[0], w[1], w[2], a.gw);
    double f[Q];
    if constexpr (IN_PLACE) {
        double m[NF];
        static_for<0, NF>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            m[k] = __ldg(src + (k * (long long)n + i));
        });
        collide_moments<COLL, double, true>(m, F, a, [&](auto qc, double v) {
            constexpr int q = decltype(qc)::value;
            f[q] = v;
        });
    } else {
        static_for<0, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            f[q] = __ldg(src + (q * (long long)n + i));
        });
        collide<COLL, double>(f, F, a);
    }
    // Eq. LBE streaming: f_a(x + c_a, t + 1) = f*_a(x, t).
    static_for<0, Q>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        dst[q * (long long)n + (zo[cz(q) + 1] + yo[cy(q) + 1] + xo[cx(q) + 1])] = f[q];
    });
}

template <int COLL>
cudaError_t split_step(const SplitLaunch& l, void* src, void* dst, void* psi) {
    const dim3 grid((l.max_cells + kSplitThreads - 1) / kSplitThreads, l.batch.nbox ? l.batch.nbox : 1);
    double* const s = static_cast<double*>(src);
    double* const d = static_cast<double*>(dst);
    double* const p = static_cast<double*>(psi);
    if constexpr (COLL != COLL_MRT) {
        if (!psi) {
            sc_fields_kernel<COLL, true><<<grid, kSplitThreads, 0, l.stream>>>(s, nullptr, l.args, l.batch);
            sc_push_kernel<COLL, true><<<grid, kSplitThreads, 0, l.stream>>>(s, nullptr, d, l.args, l.batch);
            return cudaGetLastError();
        }
    }
    if (!psi || l.batch.nbox) return cudaErrorInvalidValue;
    sc_fields_kernel<COLL, false><<<grid, kSplitThreads, 0, l.stream>>>(s, p, l.args, l.batch);
    sc_push_kernel<COLL, false><<<grid, kSplitThreads, 0, l.stream>>>(s, p, d, l.args, l.batch);
    return cudaGetLastError();
}

}  // namespace lbm
