// The step in two kernels without any redundant arithmetic.
//
//   sc_fields_kernel  forms psi of every cell once, from its populations; where
//       the collision needs no more than the moments (collide.cuh), it leaves
//       those and psi in the first slots of the cell's own populations, or in
//       fields of their own where the populations have to stay,
//   sc_push_kernel    reads psi of the 18 neighbours (through L1) and the
//       moments or populations, collides and pushes.
// Cells are dealt linearly to small blocks: no tile, rim, chunk or barrier.
//
// FP64: GB300 issues FP64 at 2 lanes an SM and clock, so a step is bound by its
// ~150 FP64 operations a cell (150 / (152 x 2 x 2.07 GHz) = 0.24 ns) while HBM
// would deliver 1600 bytes in that time.  The one-kernel steps compute psi of
// their tiles' rims again (19 additions and an exponential per rim cell, 0.6
// rim cells per cell on the 32 x 4 tiles that FP64 needs) and the density
// twice; the 72 to 88 B a cell that the second kernel adds hide behind the
// FP64 pipe.
//
// Measured: 32 x 32 x 64, SRT, 50 steps 8.10 -> 1.12 ms (of that the marching
// kernel's 32 blocks on 152 SMs cost most); 128 x 128 x 288, MRT, 10 steps
// 30.7 -> 14.8 ms, 3.18 GLUPS.
//
// 32- and 16-bit storage: the extra passes cost bytes, so large boxes keep the
// marching kernels.  Boxes that live in L2 are bound by the marching kernels'
// latency instead (a few planes per block, one barrier each), and 16-bit
// storage with odd rows has no pipelined kernel at all (bound by latency and the
// partly filled sectors of its unaligned rows; BF16 97 x 85 x 131, 20 steps:
// 1.14 -> 0.78 ms).
#pragma once
#include "collide.cuh"
#include "launch.cuh"
#include "step_kernel.cuh"

namespace lbm {

// Threads a block.  FP64: 64, so that the few blocks of a small box spread over all SMs (32 x 32 x 64, 50 steps: 1.10 ms
// with 64, 1.18 with 128, 1.24 with 256).  32- and 16-bit storage: 256, because placing blocks of 64 takes longer than
// their work (BF16 97 x 85 x 131, 20 steps: 983 us with 64, 824 with 128, 775 with 256; FP32 48 x 48 x 96: 10.4 / 8.6 /
// 8.4 us a step).
template <class R>
constexpr int kSplitThreads = sizeof(R) == 8 ? 64 : 256;

// Element k of cell i of a field array with n cells each.
template <class S>
__device__ __forceinline__ S* cell_at(S* p, int k, unsigned n, unsigned i) {
    return p + (k * (long long)n + i);
}

// MOMENTS: `fields` receives the moments and, behind them, psi (it may be f_all);
// otherwise psi alone.  Local-reference storage: the density goes to ref_dst as
// well.
template <class Codec, int COLL, bool MOMENTS>
__global__ void __launch_bounds__(kSplitThreads<typename Codec::R>)
sc_fields_kernel(const typename Codec::S* f_all, typename Codec::R* fields, const StepArgs a, const BatchArgs b) {
    using R = typename Codec::R;
    constexpr int NF = kMoments<COLL>;
    chain_begin();
    unsigned n = unsigned(a.n);
    long long base = 0;
    if (b.nbox) {
        const BatchBox& bx = b.boxes[blockIdx.y];
        n = unsigned(bx.n);
        base = bx.base;
    }
    const unsigned i = blockIdx.x * kSplitThreads<R> + threadIdx.x;
    if (i >= n) return;
    const typename Codec::S* const f = f_all + base;
    float ref = 0.0f;
    if constexpr (Codec::kLocal) ref = __ldg(a.ref_src + i);
    R v[Q], m[NF];
    static_for<0, Q>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const typename Codec::S s = *cell_at(f, q, n, i);
        if constexpr (Codec::kLocal) v[q] = Codec::template decode_ref<q>(s, ref, a.dev);
        else v[q] = Codec::template decode<q>(s, a.dev);
    });
    moments_of<COLL, R>(v, m);  // (the sums that are not needed fall away)
    const R p = psi_of<R>(m[0], par<R>(a.rho0, a.rho0f), par<R>(a.inv_rho0, a.inv_rho0f));
    chain_end();
    if constexpr (MOMENTS) {
        static_for<0, NF>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            *cell_at(fields + base, k, n, i) = m[k];
        });
        *cell_at(fields + base, NF, n, i) = p;
    } else {
        fields[i] = p;
        if constexpr (Codec::kLocal) a.ref_dst[i] = m[0];
    }
}

// psi of a cell's neighbours in one plane; yo, xo: offsets of its rows and columns -1, 0, +1.
template <class R>
struct NeighbourPsi {
    const R* plane;
    const unsigned (&yo)[3];
    const unsigned (&xo)[3];
    template <class DX, class DY>
    __device__ __forceinline__ R operator()(DX, DY) const {
        return __ldg(plane + (yo[DY::value + 1] + xo[DX::value + 1]));
    }
};

template <class Codec, int COLL, bool MOMENTS>
__global__ void __launch_bounds__(kSplitThreads<typename Codec::R>)
sc_push_kernel(const typename Codec::S* __restrict__ src_all, const typename Codec::R* __restrict__ fields,
               typename Codec::S* __restrict__ dst_all, const StepArgs a, const BatchArgs b) {
    using R = typename Codec::R;
    using S = typename Codec::S;
    constexpr int NF = kMoments<COLL>;
    chain_begin();
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
    const unsigned i = blockIdx.x * kSplitThreads<R> + threadIdx.x;
    if (i >= n) return;
    const S* __restrict__ src = src_all + base;
    S* __restrict__ dst = dst_all + base;
    const R* __restrict__ psi = fields;
    if constexpr (MOMENTS) psi += base + NF * (long long)n;
    const int z = int(i / plane), y = int((i - unsigned(z) * plane) / unsigned(nx)),
              x = int(i - unsigned(z) * plane - unsigned(y) * unsigned(nx));
    const unsigned zo[3] = {unsigned(z == 0 ? nz - 1 : z - 1) * plane, unsigned(z) * plane,
                            unsigned(z + 1 == nz ? 0 : z + 1) * plane};
    const unsigned yo[3] = {unsigned(y == 0 ? ny - 1 : y - 1) * nx, unsigned(y) * nx,
                            unsigned(y + 1 == ny ? 0 : y + 1) * nx};
    const unsigned xo[3] = {unsigned(x == 0 ? nx - 1 : x - 1), unsigned(x), unsigned(x + 1 == nx ? 0 : x + 1)};

    R f[Q], m[NF];
    if constexpr (MOMENTS) {
        static_for<0, NF>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            m[k] = __ldg(cell_at(fields + base, k, n, i));
        });
    } else {
        float ref = 0.0f;
        if constexpr (Codec::kLocal) ref = __ldg(a.ref_src + i);
        static_for<0, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            if constexpr (Codec::kLocal) f[q] = Codec::template load_ref<q>(cell_at(src, q, n, i), ref, a.dev);
            else f[q] = Codec::template load<q>(cell_at(src, q, n, i), a.dev);
        });
    }
    PsiView<R> w[3];
    static_for<0, 3>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const NeighbourPsi<R> at{psi + zo[k], yo, xo};
        w[k].c = __ldg(psi + (zo[k] + yo[1] + xo[1]));
        psi_axis(w[k], at);
        if constexpr (k == 1) psi_diag(w[k], at);
    });
    const Force<R> F = force_of(w[0], w[1], w[2], par<R>(a.gw, a.gwf));
    if constexpr (MOMENTS) {
        collide_moments<COLL, R, true>(m, F, a, [&](auto qc, R v) {
            constexpr int q = decltype(qc)::value;
            f[q] = v;
        });
    } else {
        collide<COLL, R>(f, F, a);
    }
    chain_end();
    // Eq. LBE streaming: f_a(x + c_a, t + 1) = f*_a(x, t).
    static_for<0, Q>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const unsigned to = zo[cz(q) + 1] + yo[cy(q) + 1] + xo[cx(q) + 1];
        S* const d = cell_at(dst, q, n, to);
        if constexpr (Codec::kLocal) {
            // deviation from the rest equilibrium at the destination's density (written by the first kernel)
            Codec::template store_ref<q>(d, f[q], __ldg(a.ref_dst + to), a.dev);
        } else {
            Codec::template store<q>(d, f[q], a.dev);
        }
    });
}

template <class Codec, int COLL>
cudaError_t split_step(const SplitLaunch& l, void* src, void* dst, void* psi) {
    using S = typename Codec::S;
    using R = typename Codec::R;
    const dim3 grid((l.max_cells + kSplitThreads<R> - 1) / kSplitThreads<R>, l.batch.nbox ? l.batch.nbox : 1);
    S* const s = static_cast<S*>(src);
    S* const d = static_cast<S*>(dst);
    const bool chain = (long long)grid.x * grid.y * kSplitThreads<R> <= kChainSplitCells;
    auto both = [&](auto with_moments, void* fields) {
        constexpr bool M = decltype(with_moments)::value;
        R* const p = static_cast<R*>(fields);
        cudaError_t e = launch_chained(chain, sc_fields_kernel<Codec, COLL, M>, grid, kSplitThreads<R>, 0, l.stream, s, p, l.args,
                                       l.batch);
        if (e == cudaSuccess)
            e = launch_chained(chain, sc_push_kernel<Codec, COLL, M>, grid, kSplitThreads<R>, 0, l.stream, s, p, d, l.args,
                               l.batch);
        return e;
    };
    if constexpr (COLL != COLL_MRT && sizeof(S) == sizeof(R)) {
        if (l.moments) return both(std::true_type{}, l.moments);
    }
    if (!psi || l.batch.nbox) return cudaErrorInvalidValue;
    return both(std::false_type{}, psi);
}

template <class Codec>
cudaError_t split_collisions(const SplitLaunch& l, int coll, void* src, void* dst, void* psi) {
    switch (coll) {
        case COLL_SRT: return split_step<Codec, COLL_SRT>(l, src, dst, psi);
        case COLL_MRT: return split_step<Codec, COLL_MRT>(l, src, dst, psi);
        case COLL_MRT_SPARSE: return split_step<Codec, COLL_MRT_SPARSE>(l, src, dst, psi);
        case COLL_MRT_UNIT: return split_step<Codec, COLL_MRT_UNIT>(l, src, dst, psi);
        default: return split_step<Codec, COLL_MRT_SHEAR>(l, src, dst, psi);
    }
}

}  // namespace lbm
