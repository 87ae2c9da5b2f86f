// Step kernel with the two-belt (multirange) pseudo-potential force, the
// extension of Eq. SC_force that Sec. 2 of the paper names as the way to set
// the surface tension independently of the equation of state:
//
//   F(x) = -psi(x) [ G1 sum_{a in D3Q19} w_a psi(x + c_a) c_a
//                  + G2 sum_{b in E8} (p_b / 3) psi(x + e_b) e_b ]
//
// E8: the 92 vectors with components in {-2..2} and |e|^2 in
// {1, 2, 3, 4, 5, 6, 8}; p: per shell 4/45, 1/21, 2/105, 5/504, 1/315, 1/630,
// 1/5040, the weights with unit second moment whose moment tensors are
// isotropic to eighth order.  The factor 1/3 gives belt 2 the lattice's
// second moment cs2, so the bulk equation of state is
// P = rho cs2 + cs2 (G1 + G2) psi^2 / 2 whatever the split of G1 + G2.
//
// Two kernels per step.  sc_psi_kernel turns the populations into a field of
// psi (80 B a cell); sc_step_mr_kernel then reads one value per cell and
// two-cell halo instead of summing 19 populations 1.7 times a cell.  It
// marches along z with two planes of (TX + 4) x (TY + 4) psi values in shared
// memory.  What plane p contributes to the force at distance 0, 1 and 2 along
// z differs only in the coefficients of the same five in-plane sums (by
// a^2 + b^2 of the offset (a, b)), so each thread reads its 5 x 5 patch of a
// plane once and adds to the forces of planes p - 2 .. p + 2: 25 shared loads
// and ~110 operations per cell where the 92 neighbours one by one took 92 and
// ~260.  Plane p - 2 then has its force, is collided and pushed (the streaming
// itself is the D3Q19 one).
//
// Bound: latency (a plane's 25 shared loads behind one barrier, 16 warps an SM),
// at half the HBM rate.  10 steps of
// 128 x 128 x 288 with FP32 SRT: 3.05 -> 2.46 ms, 221 us a step.
//
// Without the psi field (no memory for it) the halo planes are summed from
// the populations as before.
#pragma once
#include "e8.cuh"
#include "step_kernel.cuh"

namespace lbm {

template <class Codec>
__global__ void __launch_bounds__(256)
sc_psi_kernel(const typename Codec::S* __restrict__ f, typename Codec::R* __restrict__ psi, const StepArgs a) {
    using R = typename Codec::R;
    const R rho0 = par<R>(a.rho0, a.rho0f), inv_rho0 = par<R>(a.inv_rho0, a.inv_rho0f);
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < a.n; i += gridDim.x * 256LL)
        psi[i] = psi_of<R>(cell_density<Codec>(f + i, a.n, a.dev), rho0, inv_rho0);
}

template <class Codec, int COLL, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, sizeof(typename Codec::R) == 4 ? 512 / (TX * TY) : 1)
sc_step_mr_kernel(const typename Codec::S* __restrict__ src, typename Codec::S* __restrict__ dst, const StepArgs a) {
    using R = typename Codec::R;
    static_assert(!Codec::kLocal, "the multirange kernel stores populations directly");
    constexpr int NT = TX * TY, PX = TX + 4, PY = TY + 4, PLANE = PX * PY, NS = (PLANE + NT - 1) / NT;
    __shared__ R psi_s[2][PLANE];

    const int tid = threadIdx.x;
    const int lx = tid % TX, ly = tid / TX;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const long long n = a.n;
    const long long plane = (long long)nx * ny;
    const int zs = blockIdx.z * a.zchunk;
    if (zs >= nz) return;  // uniform over the block
    const int ze = min(zs + a.zchunk, nz);

    const int gx = wrap_index(x0 + lx, nx), gy = wrap_index(y0 + ly, ny);
    const bool active = (x0 + lx < nx) && (y0 + ly < ny);
    const int my_slot = (ly + 2) * PX + (lx + 2);
    const long long my_xy = (long long)gy * nx + gx;
    const int xp = (gx + 1 == nx) ? 0 : gx + 1, xm = (gx == 0) ? nx - 1 : gx - 1;
    const int yp = (gy + 1 == ny) ? 0 : gy + 1, ym = (gy == 0) ? ny - 1 : gy - 1;
    const long long yoff[3] = {(long long)ym * nx, (long long)gy * nx, (long long)yp * nx};
    const int xidx[3] = {xm, gx, xp};

    const R rho0 = par<R>(a.rho0, a.rho0f), inv_rho0 = par<R>(a.inv_rho0, a.inv_rho0f);
    const DevParams dev = a.dev;
    const R* const psi_ws = static_cast<const R*>(a.psi_ws);
    // G1 w(s) + G2 p(s) / 3 per shell s = |e|^2
    R c[9];
#pragma unroll
    for (int s = 0; s < 9; ++s) c[s] = R(a.G * mr::w_d3q19(s) + a.G2 * mr::p_e8(s) / 3.0);

    // cells of the psi plane that this thread fills
    long long cell[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int s = min(tid + k * NT, PLANE - 1);
        cell[k] = (long long)wrap_index(y0 + s / PX - 2, ny) * nx + wrap_index(x0 + s % PX - 2, nx);
    }
    R v[NS];  // psi of the next plane, on its way
    auto fetch = [&](int z) {
        const long long zo = (long long)wrap_index(z, nz) * plane;
#pragma unroll
        for (int k = 0; k < NS; ++k)
            v[k] = psi_ws ? __ldg(psi_ws + zo + cell[k])
                          : psi_of<R>(cell_density<Codec>(src + zo + cell[k], n, dev), rho0, inv_rho0);
    };

    // Force sums of planes p - 2 .. p + 1 so far (ax[0]: p - 2), and psi of planes p - 1, p - 2.
    R ax[4] = {}, ay[4] = {}, az[4] = {}, c1 = R(0), c2 = R(0);
    fetch(zs - 2);
    // One plane: fc holds the populations of plane p - 2; those of plane p - 1 are loaded into fl meanwhile.
    auto turn = [&](R (&fc)[Q], R (&fl)[Q], int p) {
        R* const buf = psi_s[p & 1];
#pragma unroll
        for (int k = 0; k < NS; ++k)
            if (tid + k * NT < PLANE) buf[tid + k * NT] = v[k];
        __syncthreads();
        if (p <= ze) fetch(p + 1);
        const int z = p - 2;
        const bool go = z >= zs && active;
        const long long zo = (long long)z * plane;
        if (z + 1 >= zs && z + 1 < ze) {
            const typename Codec::S* const s1 = src + (zo + plane + my_xy);
            static_for<0, Q>([&](auto qc) {
                constexpr int q = decltype(qc)::value;
                fl[q] = Codec::template load<q>(s1 + q * n, dev);
            });
        }
        const R* const b = buf + my_slot;
        auto at = [&](int dx, int dy) { return b[dx + dy * PX]; };
        const R v00 = at(0, 0);
        // opposite neighbours along x (u) and y (w), by shell: differences and sums
        const R d1x = at(1, 0) - at(-1, 0), d1y = at(0, 1) - at(0, -1);
        const R S1 = (at(1, 0) + at(-1, 0)) + (at(0, 1) + at(0, -1));
        const R e1 = at(1, 1) - at(-1, -1), e2 = at(1, -1) - at(-1, 1);
        const R g2x = e1 + e2, g2y = e1 - e2;
        const R S2 = (at(1, 1) + at(-1, -1)) + (at(1, -1) + at(-1, 1));
        const R d4x = R(2) * (at(2, 0) - at(-2, 0)), d4y = R(2) * (at(0, 2) - at(0, -2));
        const R S4 = (at(2, 0) + at(-2, 0)) + (at(0, 2) + at(0, -2));
        const R h1 = at(2, 1) - at(-2, -1), h2 = at(2, -1) - at(-2, 1);
        const R i1 = at(1, 2) - at(-1, -2), i2 = at(1, -2) - at(-1, 2);
        const R g5x = R(2) * (h1 + h2) + (i1 + i2), g5y = (h1 - h2) + R(2) * (i1 - i2);
        const R S5 = ((at(2, 1) + at(-2, -1)) + (at(2, -1) + at(-2, 1))) +
                     ((at(1, 2) + at(-1, -2)) + (at(1, -2) + at(-1, 2)));
        const R k1 = at(2, 2) - at(-2, -2), k2 = at(2, -2) - at(-2, 2);
        const R g8x = R(2) * (k1 + k2), g8y = R(2) * (k1 - k2);

        const R X2 = c[5] * d1x + c[6] * g2x + c[8] * d4x, Y2 = c[5] * d1y + c[6] * g2y + c[8] * d4y;
        const R X1 = c[2] * d1x + c[3] * g2x + c[5] * d4x + c[6] * g5x;
        const R Y1 = c[2] * d1y + c[3] * g2y + c[5] * d4y + c[6] * g5y;
        const R X0 = c[1] * d1x + c[2] * g2x + c[4] * d4x + c[5] * g5x + c[8] * g8x;
        const R Y0 = c[1] * d1y + c[2] * g2y + c[4] * d4y + c[5] * g5y + c[8] * g8y;
        const R Z1 = c[1] * v00 + c[2] * S1 + c[3] * S2 + c[5] * S4 + c[6] * S5;
        const R Z2 = R(2) * (c[4] * v00 + c[5] * S1 + c[6] * S2 + c[8] * S4);

        const Force<R> F{-c2, ax[0] + X2, ay[0] + Y2, az[0] + Z2};
        ax[0] = ax[1] + X1; ay[0] = ay[1] + Y1; az[0] = az[1] + Z1;
        ax[1] = ax[2] + X0; ay[1] = ay[2] + Y0; az[1] = az[2];
        ax[2] = ax[3] + X1; ay[2] = ay[3] + Y1; az[2] = az[3] - Z1;
        ax[3] = X2;         ay[3] = Y2;         az[3] = -Z2;
        c2 = c1;
        c1 = v00;

        if (go) {
            collide<COLL, R>(fc, F, a);
            // Eq. LBE streaming: f_a(x + c_a, t + 1) = f*_a(x, t).
            const int zm = (z == 0) ? nz - 1 : z - 1, zn = (z + 1 == nz) ? 0 : z + 1;
            const long long zoff[3] = {(long long)zm * plane, zo, (long long)zn * plane};
            static_for<0, Q>([&](auto qc) {
                constexpr int q = decltype(qc)::value;
                const long long idx = zoff[cz(q) + 1] + yoff[cy(q) + 1] + xidx[cx(q) + 1];
                Codec::template store<q>(dst + (q * n + idx), fc[q], a.dev);
            });
        }
    };
    R fa[Q], fb[Q];
    for (int p = zs - 2; p <= ze + 1; p += 2) {
        turn(fa, fb, p);
        if (p + 1 <= ze + 1) turn(fb, fa, p + 1);
    }
}

}  // namespace lbm
