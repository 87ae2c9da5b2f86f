// The sums of the ligament diagnostics, shared by lbm_diag and
// lbm_diag_noalloc so that both give the same numbers, to the last bit.
//
// Each cell's rho and j come from its 19 populations in the codec's
// arithmetic type (float for 32- and 16-bit storage, double for FP64).  The
// thread sums its cells in that type over runs of kRun cells (the run is
// unrolled, so its loads are in flight together) and adds each run's
// partial sums to float64 accumulators.  With float storage this does one
// float64 add per quantity and run instead of per cell: the FP64 pipe of the
// GPU issues at a small fraction of the FP32 rate and bounded the per-cell
// form.  The order of all sums is fixed, so results are deterministic.
#pragma once
#include <algorithm>

#include "codec.cuh"
#include "lattice.cuh"

namespace lbm {

template <class Codec>
__device__ __forceinline__ void diag_cell(const typename Codec::S* __restrict__ p, long long n,
                                          const DevParams& dev, float ref, typename Codec::R& rho,
                                          typename Codec::R& jx, typename Codec::R& jy,
                                          typename Codec::R& jz) {
    using R = typename Codec::R;
    R r = R(0), ax = R(0), ay = R(0), az = R(0);
    static_for<0, Q>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        R fq;
        if constexpr (Codec::kLocal) fq = Codec::template load_ref<q>(p + q * n, ref, dev);
        else fq = Codec::template load<q>(p + q * n, dev);
        r += fq;
        if constexpr (cx(q) != 0) ax += R(cx(q)) * fq;
        if constexpr (cy(q) != 0) ay += R(cy(q)) * fq;
        if constexpr (cz(q) != 0) az += R(cz(q)) * fq;
    });
    rho = r;
    jx = ax;
    jy = ay;
    jz = az;
}

constexpr int kDiagThreads = 256;
constexpr int kDiagRun = 8;
constexpr int kDiagRunCells = kDiagRun * kDiagThreads;  // cells of one run of every thread

// Parts that a slice is summed in, one block each: as many as leave 3.5 blocks an
// SM over all slices, so that one round of blocks takes them all, at least one run
// of cells a part, and, for more than one part, at most kDiagMaxParts in all.
// us a call of lbm_diag with one part / 8 blocks an SM rounded up / this rule:
//   FP32 64x64x144 48.9 / 41.0 / 42.2, 128x128x288 109.5 / 136.7 / 100.8, 256x256x575 563 / 580 / 544,
//   300x200x100 230 / 156 / 133, 384x384x300 634 / 652 / 616; FP64 128x128x288 614 / 629 / 603
// (the one part by a tree in shared memory).
constexpr int kDiagMaxParts = 4096;
inline int diag_parts(long long plane, int nz, int num_sms) {
    const long long runs = (plane + kDiagRunCells - 1) / kDiagRunCells, want = 7LL * num_sms / (2LL * nz);
    const long long most = nz < kDiagMaxParts ? kDiagMaxParts / nz : 1;
    return int(std::max(1LL, std::min(std::min(want, runs), most)));
}

// Cells first, first + stride, ... < count (in runs of kRun of them; with
// parts > 1 only every parts-th run from the part-th on, so that several
// blocks share a slice without changing what a run sums) of the slice whose
// populations start at fz (population stride n; refz: the slice's reference densities for
// the local-reference codecs).  acc: mass, jx, jy, jz, liquid area, max rho,
// cells with rho <= 0 / NaN / Inf.
template <class Codec>
__device__ __forceinline__ void diag_accumulate(const typename Codec::S* __restrict__ fz, long long n,
                                                long long count, long long first, int stride, const DevParams& dev,
                                                double rho_v, double inv, const float* __restrict__ refz,
                                                double (&acc)[7], int part = 0, int parts = 1) {
    using R = typename Codec::R;
    constexpr int kRun = kDiagRun;
    for (int k = 0; k < 7; ++k) acc[k] = 0.0;
    const R rv = R(rho_v), iv = R(inv);
    for (long long i = first + (long long)part * kRun * stride; i < count; i += (long long)parts * kRun * stride) {
        R m = R(0), jx = R(0), jy = R(0), jz = R(0), area = R(0), mx = R(0);
        int bad = 0;
#pragma unroll
        for (int k = 0; k < kRun; ++k) {
            const long long c = i + (long long)k * stride;
            if (c < count) {
                R r, ax, ay, az;
                float rf = 0.0f;
                if constexpr (Codec::kLocal) rf = refz[c];
                diag_cell<Codec>(fz + c, n, dev, rf, r, ax, ay, az);
                m += r;
                jx += ax;
                jy += ay;
                jz += az;
                area += fmin(fmax((r - rv) * iv, R(0)), R(1));
                mx = fmax(mx, r);
                if (!(r > R(0)) || !isfinite(r)) ++bad;
            }
        }
        acc[0] += double(m);
        acc[1] += double(jx);
        acc[2] += double(jy);
        acc[3] += double(jz);
        acc[4] += double(area);
        acc[5] = fmax(acc[5], double(mx));
        acc[6] += double(bad);
    }
}

__device__ __forceinline__ double diag_join(int k, double a, double b) { return k == 5 ? fmax(a, b) : a + b; }

// One block's sum of a part of a slice, by a fixed tree: threads 0 .. 6 return
// quantity threadIdx.x of `acc`'s order.
template <class Codec>
__device__ __forceinline__ double diag_part(const typename Codec::S* __restrict__ fz, long long n, long long plane,
                                            const DevParams& dev, double rho_l, double rho_v,
                                            const float* __restrict__ refz, int part, int parts) {
    __shared__ double red[7][kDiagThreads / 32];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    double acc[7];
    diag_accumulate<Codec>(fz, n, plane, threadIdx.x, kDiagThreads, dev, rho_v, 1.0 / (rho_l - rho_v), refz, acc, part,
                           parts);
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        for (int s = 16; s > 0; s >>= 1) acc[k] = diag_join(k, acc[k], __shfl_down_sync(0xffffffffu, acc[k], s));
        if (lane == 0) red[k][warp] = acc[k];
    }
    __syncthreads();
    double v = 0.0;
    if (threadIdx.x < 7) {
        v = red[threadIdx.x][0];
        for (int w = 1; w < kDiagThreads / 32; ++w) v = diag_join(threadIdx.x, v, red[threadIdx.x][w]);
    }
    return v;
}

}  // namespace lbm
