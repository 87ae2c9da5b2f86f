// Discrete adjoint of the SRT Shan-Chen step (Sec. 2: Eqs. LBE, local_eq,
// momentum, SC_force, vel_shift), for FP32 or FP64 populations.
//
// Forward step at time t (state f = post-streaming populations):
//   rho = sum f, j = sum c f, psi = psi(rho), S(x) = sum_a w_a psi(x + c_a) c_a,
//   F = -G psi S, u' = (j + tau F)/rho, f* = f + omega (f_eq(rho, u') - f),
//   f_a(x + c_a, t + 1) = f*_a(x).
// Reverse step, given lam(t+1) = dJ/df(t+1):
//   1. streaming adjoint (pull): lam*_a(x) = lam_a(x + c_a, t+1);
//   2. collision adjoint (local, adj_collide_kernel): lam_loc = (df*/df)^T lam*,
//      gF = (df*/dF)^T lam*, and the tau and G terms of the parameter
//      gradients;
//   3. force adjoint (a gather over neighbours, adj_force_kernel):
//      g_psi(y) = -G [ S(y).gF(y) + sum_a w_a psi(y - c_a) c_a . gF(y - c_a) ],
//      g_rho = g_psi psi'(rho) with psi' = exp(-rho/rho0) = 1 - psi/rho0,
//      lam_a(y, t) = lam_loc_a(y) + g_rho(y) for every a.  Step 2 already
//      knows S(y) and psi(y), so it stores T = S.gF and V = psi gF per cell
//      and the gather reads only V of the 18 neighbours.
// Parameter gradients are summed in float64 per block and reduced in a fixed
// order (deterministic).
//
// psi and 1/rho are the step's own functions (psi_of, recip), also where FP32
// takes the hardware's approximations: psi of a state that no step recomputed is
// then the same wherever the checkpoints lie, and the equilibrium is the one the
// step took.  With expf and the division the error of the three gradients of
// 64 x 64 x 180, 500 steps, grew from 4.3e-6 to 4.7e-6 (and 38.0 to 39.1 ms).
//
// At tau = 1 the collision forgets the populations, so their adjoint is
// lam_a(y) = A(y) + c_a.B(y): four values a cell instead of 20 (lam and gr).
// adj_collide1_kernel and adj_force_kernel then keep {A, B} as one 16- or
// 32-byte vector per cell: one vector load per neighbour where the general
// form loads two values, and 128 + 40 B a cell and step instead of 250 + 40.
// 64 x 64 x 180 in FP32, 500 steps back with their recomputation: 64.1 ms with
// 20 values, 50.2 with {A, B}, 41.4 with the recomputed states kept as moments
// too, 37.7 with the block shape and block sums below.  Both kernels are bound
// by the latency of their gathers from L2 (about 39 and 17 us a step from a
// cold cache before those two).
#include <cuda_runtime.h>

#include "adjoint.h"
#include "collide.cuh"
#include "launch.cuh"
#include "lattice.cuh"

namespace lbm {
namespace {

// 64 x 64 x 180, 500 steps back: 41.3 ms with blocks of 256 threads, 39.8 with 128, 39.7 with 64, 40.3 with 32.
constexpr int kThreads = 128;
constexpr int kRowThreads = 32, kRows = kThreads / kRowThreads;  // (32, 4) blocks: 4 rows at a time

// The cells of one x row and the periodic neighbour offsets of the row and
// of its cells (32-bit: the adjoint needs nx*ny*nz < 2^32).  Blocks of
// (32, 4) threads walk the ny*nz rows (grid-stride); a warp covers 32
// consecutive x of a row, so the neighbour gathers stay coalesced and no
// cell index is ever divided.
struct Row {
    unsigned row;           // its number, y + ny z
    unsigned zo[3], yo[3];  // offsets of planes z-1, z, z+1 and rows y-1, y, y+1
};

__device__ __forceinline__ Row row_of(unsigned r, int nx, int ny, int nz) {
    const int y = int(r % unsigned(ny)), z = int(r / unsigned(ny));
    const int ym = y == 0 ? ny - 1 : y - 1, yp = y + 1 == ny ? 0 : y + 1;
    const int zm = z == 0 ? nz - 1 : z - 1, zp = z + 1 == nz ? 0 : z + 1;
    const unsigned plane = unsigned(nx) * unsigned(ny);
    Row w;
    w.row = r;
    w.zo[0] = unsigned(zm) * plane;
    w.zo[1] = unsigned(z) * plane;
    w.zo[2] = unsigned(zp) * plane;
    w.yo[0] = unsigned(ym) * unsigned(nx);
    w.yo[1] = unsigned(y) * unsigned(nx);
    w.yo[2] = unsigned(yp) * unsigned(nx);
    return w;
}

// Index of x + (dx, dy, dz), |d| <= 1, with xs = {x-1, x, x+1} wrapped.
__device__ __forceinline__ unsigned nb_of(const Row& w, const unsigned (&xs)[3], int dx, int dy, int dz) {
    return w.zo[dz + 1] + w.yo[dy + 1] + xs[dx + 1];
}

// psi of a cell's neighbours in the plane at offset zo.
template <class R>
struct RowPsi {
    const R* psi;
    unsigned zo;
    const Row& w;
    const unsigned (&xs)[3];
    template <class DX, class DY>
    __device__ __forceinline__ R operator()(DX, DY) const {
        return __ldg(psi + (zo + w.yo[DY::value + 1] + xs[DX::value + 1]));
    }
};
// The step's force of cell xs[1] of row w (collide.cuh).
template <class R>
__device__ __forceinline__ Force<R> row_force(const R* psi, const Row& w, const unsigned (&xs)[3], R gw) {
    PsiView<R> v[3];
    static_for<0, 3>([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const RowPsi<R> at{psi, w.zo[k], w, xs};
        v[k].c = __ldg(psi + (w.zo[k] + w.yo[1] + xs[1]));
        psi_axis(v[k], at);
        if constexpr (k == 1) psi_diag(v[k], at);
    });
    return force_of(v[0], v[1], v[2], gw);
}

// c_q . (x, y, z)
template <int q, class R>
__device__ __forceinline__ R dot_c(R x, R y, R z) {
    R s = R(0);
    if constexpr (cx(q) != 0) s = cx(q) > 0 ? x : -x;
    if constexpr (cy(q) != 0) s = cx(q) != 0 ? (cy(q) > 0 ? s + y : s - y) : (cy(q) > 0 ? y : -y);
    if constexpr (cz(q) != 0)
        s = (cx(q) != 0 || cy(q) != 0) ? (cz(q) > 0 ? s + z : s - z) : (cz(q) > 0 ? z : -z);
    return s;
}

template <class F>
__device__ __forceinline__ void for_each_cell(int nx, int ny, int nz, F&& body) {
    const unsigned rows = unsigned(ny) * unsigned(nz);
    for (unsigned r = blockIdx.x * kRows + threadIdx.y; r < rows; r += gridDim.x * kRows) {
        const Row w = row_of(r, nx, ny, nz);
        for (int x = threadIdx.x; x < nx; x += kRowThreads) {
            const unsigned xs[3] = {unsigned(x == 0 ? nx - 1 : x - 1), unsigned(x), unsigned(x + 1 == nx ? 0 : x + 1)};
            body(w, xs, w.zo[1] + w.yo[1] + unsigned(x));
        }
    }
}

// Four values of one cell, loaded and stored whole.
template <class R>
struct alignas(16) Vec4 {
    R x, y, z, w;
};
__device__ __forceinline__ Vec4<float> load4(const Vec4<float>* p) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Vec4<double> load4(const Vec4<double>* p) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void store4(Vec4<float>* p, const Vec4<float>& v) {
    *reinterpret_cast<float4*>(p) = make_float4(v.x, v.y, v.z, v.w);
}
__device__ __forceinline__ void store4(Vec4<double>* p, const Vec4<double>& v) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v.x, v.y);
    reinterpret_cast<double2*>(p)[1] = make_double2(v.z, v.w);
}

template <class R>
__global__ void __launch_bounds__(kThreads) adj_psi_kernel(const R* __restrict__ f, R* __restrict__ psi, unsigned n,
                                                           R rho0, R inv_rho0) {
    for (unsigned i = blockIdx.x * kThreads + threadIdx.y * kRowThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) {
        const R r = density_of<R>([&](auto qc) { return f[size_t(decltype(qc)::value) * n + i]; });
        psi[i] = psi_of<R>(r, rho0, inv_rho0);
    }
}

// The same from the moment fields of step_moment.cuh.
__global__ void __launch_bounds__(kThreads) adj_psi_moments_kernel(const float* __restrict__ moments,
                                                                   float* __restrict__ psi, AdjointArgs a) {
    const unsigned pitch = unsigned(moment_pitch(a.nx));
    const float rho0 = a.rho0f, inv_rho0 = float(1.0 / a.rho0);
    for_each_cell(a.nx, a.ny, a.nz, [&](const Row& w, const unsigned (&xs)[3], unsigned i) {
        const unsigned o = w.row * pitch + xs[1] + 2;
        psi[i] = psi_of<float>(moments[o], rho0, inv_rho0);
    });
}

// Sum of (a, b) over the block, added to out2[0..1] (the block's running
// sums over the reverse steps); fixed order.  One warp adds up what all have
// written, a in its lower and b in its upper lanes: an FP64 instruction holds
// the pipe of 2 lanes for 16 cycles a warp, and a tree by shuffles in every
// warp takes 10 of them (64 x 64 x 180, 500 steps back: 39.8 -> 38.5 ms).
__device__ __forceinline__ void block_sum2(double a, double b, double* out2) {
    __shared__ double red[2][kThreads];
    const int t = threadIdx.y * kRowThreads + threadIdx.x;
    red[0][t] = a;
    red[1][t] = b;
    __syncthreads();
    if (t < 32) {
        const double* const r = red[t >> 4];
        double s = r[t & 15];
        for (int k = 16; k < kThreads; k += 16) s += r[k + (t & 15)];
        for (int k = 8; k > 0; k >>= 1) s += __shfl_down_sync(0xffffffffu, s, k, 16);
        if ((t & 15) == 0) out2[t >> 4] += s;
    }
}

// Collision adjoint.  Besides lam_out it writes, per cell, the two pieces of
// the force adjoint that the gather of adj_force_kernel needs:
//   V = psi gF (the cell's force sensitivity weighted by its psi)
//   T = S . gF (S = sum_a w_a psi(x + c_a) c_a, known here),
// one vector {V, T} per cell.
template <class R>
__global__ void __launch_bounds__(kThreads)
adj_collide_kernel(const R* __restrict__ f, const R* __restrict__ psi, const R* __restrict__ lam_next,
                   const R* __restrict__ gr_next, R* __restrict__ lam_out, Vec4<R>* __restrict__ fa,
                   double* __restrict__ partials, AdjointArgs a) {
    const unsigned n = unsigned(a.n);
    chain_begin();
    const R tau = par<R>(a.tau, a.tauf), omega = par<R>(a.omega, a.omegaf);
    double accG = 0.0, accT = 0.0;
    for_each_cell(a.nx, a.ny, a.nz, [&](const Row& w, const unsigned (&xs)[3], unsigned i) {
        R fv[Q], ls[Q];
        static_for<0, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            fv[q] = f[size_t(q) * n + i];
            const unsigned nb = nb_of(w, xs, cx(q), cy(q), cz(q));
            ls[q] = lam_next[size_t(q) * n + nb] + gr_next[nb];  // streaming adjoint: pull from x + c_q
        });
        R m[4];
        moments_of<COLL_SRT, R>(fv, m);
        const R rho = m[0];
        const Force<R> F = row_force(psi, w, xs, par<R>(a.gw, a.gwf));
        const R Fx = F.g * F.sx, Fy = F.g * F.sy, Fz = F.g * F.sz;
        const R sx = R(1.0 / 36.0) * F.sx, sy = R(1.0 / 36.0) * F.sy, sz = R(1.0 / 36.0) * F.sz;
        const R ps = psi[i];
        const R inv_rho = recip(rho);
        const R ux = (m[1] + tau * Fx) * inv_rho, uy = (m[2] + tau * Fy) * inv_rho, uz = (m[3] + tau * Fz) * inv_rho;
        const R u2 = ux * ux + uy * uy + uz * uz;
        // adjoint of f* = (1 - omega) f + omega f_eq(rho, u')
        R g_rho = R(0), gux = R(0), guy = R(0), guz = R(0), g_tau = R(0);
        // w_a rho with the rest weight from sum_a w_a = 1, as the step forms it: with the rounded weights
        // (their sum is 1 + 3e-8 in float) the adjoint field grew by 3e-8 a step, 1e-5 over 500 steps.
        const R r2 = R(1.0 / 36.0) * rho, r1 = r2 + r2, r0 = fma(R(-24), r2, rho);
        R s_mw = R(0);
        static_for<0, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            const R cu = dot_c<q>(ux, uy, uz);
            const R wr = q == 0 ? r0 : (q < 7 ? r1 : r2);
            const R feq = wr * (R(1) - R(1.5) * u2 + cu * (R(3) + R(4.5) * cu));
            const R mu = omega * ls[q], mw = mu * wr;
            g_rho += mu * feq;
            // d f_eq / d u' = w rho (3 c + 9 (c.u') c - 3 u')
            const R k = mw * (R(3) + R(9) * cu);
            if constexpr (cx(q) != 0) gux += R(cx(q)) * k;
            if constexpr (cy(q) != 0) guy += R(cy(q)) * k;
            if constexpr (cz(q) != 0) guz += R(cz(q)) * k;
            s_mw += mw;
            g_tau -= ls[q] * (feq - fv[q]);
        });
        gux -= R(3) * s_mw * ux;
        guy -= R(3) * s_mw * uy;
        guz -= R(3) * s_mw * uz;
        g_tau *= omega * omega;  // d omega / d tau = -1/tau^2
        // u' = (j + tau F)/rho
        const R gjx = gux * inv_rho, gjy = guy * inv_rho, gjz = guz * inv_rho;
        g_rho = (g_rho - (gux * ux + guy * uy + guz * uz)) * inv_rho;
        g_tau += (gux * Fx + guy * Fy + guz * Fz) * inv_rho;
        const R gFx = tau * gjx, gFy = tau * gjy, gFz = tau * gjz;
        static_for<0, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            R v = (R(1) - omega) * ls[q] + g_rho;
            if constexpr (q != 0) v += dot_c<q>(gjx, gjy, gjz);
            lam_out[size_t(q) * n + i] = v;
        });
        store4(fa + i, Vec4<R>{ps * gFx, ps * gFy, ps * gFz, sx * gFx + sy * gFy + sz * gFz});
        // dF/dG = -psi S
        accG += double(-(ps * sx) * gFx - (ps * sy) * gFy - (ps * sz) * gFz);
        accT += double(g_tau);
    });
    chain_end();
    block_sum2(accG, accT, partials + 2 * blockIdx.x);
}

// The same at tau = 1, from lam_a(y) = A(y) + c_a.B(y) kept as {A, B}: the
// pulled value of velocity q is A + c_q.B of the neighbour x + c_q.  Opposite
// velocities share the even part e and odd part o of f_eq = e +/- o.  Writes
// {g_rho, B} (adj_force_kernel adds the force's part of A) and {V, T}.
//
// The gradient with respect to tau, sum_x sum_q ls_q (f_eq_q - f_q), needs the
// populations before the collision.  FROM_MOMENTS has only a state's moments
// (as step_moment.cuh stores them: 16 B a cell are kept per state instead of
// 76).  There f_q(x + c_q, t + 1) = f_eq_q(x, t), so the populations of step
// t + 1 are weighted here, in step t, with the adjoint two links on:
//   sum_x sum_q f_eq_q(x, t) [ lam_q(x + c_q, t + 1) - lam_q(x + 2 c_q, t + 2) ],
// a difference along the velocity that is as small as f_eq - f itself.
// lam_next2: lam(t + 2), nullptr in the last step; first: step 0, whose
// populations are at rest, f_q = w_q rho.
template <class R, bool FROM_MOMENTS>
__global__ void __launch_bounds__(kThreads, 4)
adj_collide1_kernel(const R* __restrict__ f, const R* __restrict__ psi, const Vec4<R>* __restrict__ lam_next,
                    const Vec4<R>* __restrict__ lam_next2, Vec4<R>* __restrict__ lam_out, Vec4<R>* __restrict__ fa,
                    double* __restrict__ partials, bool first, AdjointArgs a) {
    chain_begin();
    const unsigned n = unsigned(a.n);
    const int pitch = moment_pitch(a.nx);
    const long long nf = (long long)pitch * a.ny * a.nz;
    double accG = 0.0, accT = 0.0;
    for_each_cell(a.nx, a.ny, a.nz, [&](const Row& w, const unsigned (&xs)[3], unsigned i) {
        R fv[Q], m[4];
        if constexpr (FROM_MOMENTS) {
            // rows of `pitch` floats from column 2 on; rho, then jx and jy by pairs of cells, then jz
            const unsigned col = xs[1] + 2, o = w.row * unsigned(pitch) + col;
            const R* const pj = f + (nf + 2 * (long long)(o - (col & 1)) + (col & 1));
            m[0] = __ldg(f + o);
            m[1] = __ldg(pj);
            m[2] = __ldg(pj + 2);
            m[3] = __ldg(f + (3 * nf + o));
        } else {
            static_for<0, Q>([&](auto qc) {
                constexpr int q = decltype(qc)::value;
                fv[q] = f[size_t(q) * n + i];
            });
            moments_of<COLL_SRT, R>(fv, m);
        }
        const R rho = m[0];
        const Force<R> F = row_force(psi, w, xs, par<R>(a.gw, a.gwf));
        const R Fx = F.g * F.sx, Fy = F.g * F.sy, Fz = F.g * F.sz;
        const R ps = psi[i], inv_rho = recip(rho);
        const R ux = (m[1] + Fx) * inv_rho, uy = (m[2] + Fy) * inv_rho, uz = (m[3] + Fz) * inv_rho;
        const R base = R(1) - R(1.5) * (ux * ux + uy * uy + uz * uz);
        const R r2 = R(1.0 / 36.0) * rho, r1 = r2 + r2, r0 = fma(R(-24), r2, rho);

        const R l0 = load4(lam_next + i).x;
        R s_feq = r0 * base * l0;          // sum_q ls_q f_eq_q
        R s_f;                             // sum_q ls_q (f_eq_q - f_q), or its rearrangement
        if constexpr (FROM_MOMENTS) s_f = r0 * base * (lam_next2 ? l0 - load4(lam_next2 + i).x : l0);
        else s_f = (r0 * base - fv[0]) * l0;
        R s_w1 = R(0), s_w2 = R(0);        // sums of ls over the axis and the edge velocities
        R gx = R(0), gy = R(0), gz = R(0);
        // rows, planes and columns two links away
        unsigned zo2[3], yo2[3], xs2[3];
        if constexpr (FROM_MOMENTS) {
            const unsigned plane = unsigned(a.nx) * unsigned(a.ny), vol = plane * unsigned(a.nz);
            auto two = [](unsigned lo, unsigned hi, unsigned step, unsigned end, unsigned (&o)[3]) {
                o[0] = lo == 0 ? end - step : lo - step;
                o[2] = hi + step == end ? 0 : hi + step;
            };
            two(w.zo[0], w.zo[2], plane, vol, zo2);
            two(w.yo[0], w.yo[2], unsigned(a.nx), plane, yo2);
            two(xs[0], xs[2], 1u, unsigned(a.nx), xs2);
            zo2[1] = w.zo[1];
            yo2[1] = w.yo[1];
            xs2[1] = xs[1];
        }
        static_for<0, 9>([&](auto pc) {
            constexpr int q = 2 * decltype(pc)::value + 1;
            const Vec4<R> p = load4(lam_next + nb_of(w, xs, cx(q), cy(q), cz(q)));
            const Vec4<R> o = load4(lam_next + nb_of(w, xs, -cx(q), -cy(q), -cz(q)));
            // streaming adjoint: pull from x + c_q
            const R lp = p.x + dot_c<q>(p.y, p.z, p.w), lm = o.x - dot_c<q>(o.y, o.z, o.w);
            const R sl = lp + lm, dl = lp - lm;
            const R cu = dot_c<q>(ux, uy, uz);
            const R wr = q < 7 ? r1 : r2;
            const R e = wr * (base + R(4.5) * cu * cu), od = wr * (R(3) * cu);
            s_feq += e * sl + od * dl;
            if constexpr (FROM_MOMENTS) {
                R kp = lp, km = lm;
                if (lam_next2) {
                    const Vec4<R> p2 = load4(lam_next2 + (zo2[cz(q) + 1] + yo2[cy(q) + 1] + xs2[cx(q) + 1]));
                    const Vec4<R> o2 = load4(lam_next2 + (zo2[1 - cz(q)] + yo2[1 - cy(q)] + xs2[1 - cx(q)]));
                    kp -= p2.x + dot_c<q>(p2.y, p2.z, p2.w);
                    km -= o2.x - dot_c<q>(o2.y, o2.z, o2.w);
                }
                s_f += (e + od) * kp + (e - od) * km;
            } else {
                s_f += ((e + od) - fv[q]) * lp + ((e - od) - fv[q + 1]) * lm;
            }
            if constexpr (q < 7) s_w1 += sl;
            else s_w2 += sl;
            // d f_eq / d u' = w rho (3 c + 9 (c.u') c - 3 u')
            const R k = wr * (R(3) * dl + R(9) * cu * sl);
            if constexpr (cx(q) != 0) gx += R(cx(q)) * k;
            if constexpr (cy(q) != 0) gy += R(cy(q)) * k;
            if constexpr (cz(q) != 0) gz += R(cz(q)) * k;
        });
        const R s_wr = r0 * l0 + r1 * s_w1 + r2 * s_w2;  // sum_q w_q rho ls_q
        if constexpr (FROM_MOMENTS) {
            if (first) s_f -= s_wr;
        }
        gx -= R(3) * s_wr * ux;
        gy -= R(3) * s_wr * uy;
        gz -= R(3) * s_wr * uz;
        // u' = (j + F)/rho at tau = 1
        const R gjx = gx * inv_rho, gjy = gy * inv_rho, gjz = gz * inv_rho;
        const R g_rho = (s_feq - (gx * ux + gy * uy + gz * uz)) * inv_rho;
        store4(lam_out + i, Vec4<R>{g_rho, gjx, gjy, gjz});
        const R sg = R(1.0 / 36.0) * (F.sx * gjx + F.sy * gjy + F.sz * gjz);
        store4(fa + i, Vec4<R>{ps * gjx, ps * gjy, ps * gjz, sg});
        accG += double(-ps * sg);                                        // dF/dG = -psi S
        accT += double((gjx * Fx + gjy * Fy + gjz * Fz) - s_f);          // d omega / d tau = -1
    });
    chain_end();
    block_sum2(accG, accT, partials + 2 * blockIdx.x);
}

// Force adjoint: g_psi(y) = -G [ T(y) + sum_a w_a c_a . V(y - c_a) ] and the
// density term g_psi(y) psi'(rho(y)), psi' = 1 - psi/rho0.  It is the same for
// every population: kept in gr and added where it is read, or (TAU1) added to
// the A of {A, B}.
template <class R, bool TAU1>
__global__ void __launch_bounds__(kThreads, 4)
adj_force_kernel(const R* __restrict__ psi, const Vec4<R>* __restrict__ fa, R* __restrict__ gr, AdjointArgs a) {
    chain_begin();
    const R G = par<R>(a.G, a.Gf), inv_rho0 = R(1.0 / a.rho0);
    for_each_cell(a.nx, a.ny, a.nz, [&](const Row& w, const unsigned (&xs)[3], unsigned i) {
        R axis = R(0), edge = R(0);
        static_for<1, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            const Vec4<R> v = load4(fa + nb_of(w, xs, -cx(q), -cy(q), -cz(q)));  // y - c_q
            if constexpr (q < 7) axis += dot_c<q>(v.x, v.y, v.z);
            else edge += dot_c<q>(v.x, v.y, v.z);
        });
        const R term = load4(fa + i).w + (R(1.0 / 18.0) * axis + R(1.0 / 36.0) * edge);
        const R g = -G * term * (R(1) - psi[i] * inv_rho0);
        if constexpr (TAU1) gr[4 * size_t(i)] += g;
        else gr[i] = g;
    });
}

// lam_a(x, T) = dJ/drho(x) for every a (rho = sum_a f_a); no force term yet.
template <class R>
__global__ void adj_seed1_kernel(const double* __restrict__ g, Vec4<R>* __restrict__ lam, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        store4(lam + i, Vec4<R>{R(g[i]), R(0), R(0), R(0)});
}
template <class R>
__global__ void adj_seed_kernel(const double* __restrict__ g, R* __restrict__ lam, R* __restrict__ gr, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const R v = R(g[i]);
        gr[i] = R(0);
        static_for<0, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            lam[q * n + i] = v;
        });
    }
}

// f_a(x, 0) = w_a rho0(x): dJ/drho0(x) = sum_a w_a lam_a(x, 0), with
// lam_a = stored part + force term gr (sum_a w_a = 1).
template <class R>
__global__ void adj_rho0_kernel(const R* __restrict__ lam, const R* __restrict__ gr, double* __restrict__ out,
                                long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double s = double(gr[i]);
        static_for<0, Q>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            s += wq(q) * double(lam[q * n + i]);
        });
        out[i] = s;
    }
}

// At tau = 1 the sum is A: sum_a w_a (A + c_a.B) = A.
template <class R>
__global__ void adj_rho01_kernel(const Vec4<R>* __restrict__ lam, double* __restrict__ out, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = double(load4(lam + i).x);
}

// Fixed-order sum of the per-block partials into acc[0..1]: each of 128
// threads sums a strided subset in block order, then a fixed tree.
__global__ void __launch_bounds__(kThreads) adj_reduce_kernel(const double* __restrict__ partials, int nblocks,
                                                             double* __restrict__ acc) {
    __shared__ double red[2][kThreads];
    double g = 0.0, t = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kThreads) {
        g += partials[2 * b];
        t += partials[2 * b + 1];
    }
    red[0][threadIdx.x] = g;
    red[1][threadIdx.x] = t;
    __syncthreads();
    for (int s = kThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] += red[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        acc[0] += red[0][0];
        acc[1] += red[1][0];
    }
}

template <class R>
cudaError_t run_adjoint_step(const AdjointArgs& a, const void* f, void* psi, bool psi_ready, const void* lam_next,
                             const void* gr_next, void* lam_out, void* gr_out, void* gF, double* partials,
                             double* acc, cudaStream_t st) {
    const int grid = a.grid;
    const dim3 block(kRowThreads, kRows);
    if (!psi_ready)
        adj_psi_kernel<R><<<grid, block, 0, st>>>(static_cast<const R*>(f), static_cast<R*>(psi), unsigned(a.n),
                                                  par<R>(a.rho0, a.rho0f), R(1.0 / a.rho0));
    Vec4<R>* const v = static_cast<Vec4<R>*>(gF);
    if (a.tau1) {
        cudaError_t e = launch_chained(a.n <= kChainCells, adj_collide1_kernel<R, false>, grid, block, 0, st, static_cast<const R*>(f),
                                       static_cast<const R*>(psi), static_cast<const Vec4<R>*>(lam_next), nullptr,
                                       static_cast<Vec4<R>*>(lam_out), v, partials, false, a);
        if (e != cudaSuccess) return e;
        return launch_chained(a.n <= kChainCells, adj_force_kernel<R, true>, grid, block, 0, st, static_cast<const R*>(psi), v,
                              static_cast<R*>(lam_out), a);
    }
    cudaError_t e = launch_chained(a.n <= kChainCells, adj_collide_kernel<R>, grid, block, 0, st, static_cast<const R*>(f),
                                   static_cast<const R*>(psi), static_cast<const R*>(lam_next),
                                   static_cast<const R*>(gr_next), static_cast<R*>(lam_out), v, partials, a);
    if (e != cudaSuccess) return e;
    e = launch_chained(a.n <= kChainCells, adj_force_kernel<R, false>, grid, block, 0, st, static_cast<const R*>(psi), v,
                       static_cast<R*>(gr_out), a);
    (void)acc;  // the per-block sums stay in `partials` until adjoint_reduce
    return e;
}

}  // namespace

cudaError_t adjoint_step(const AdjointArgs& a, bool f64, const void* f, void* psi, bool psi_ready,
                         const void* lam_next, const void* gr_next, void* lam_out, void* gr_out, void* gF,
                         double* partials, double* acc, cudaStream_t st) {
    return f64 ? run_adjoint_step<double>(a, f, psi, psi_ready, lam_next, gr_next, lam_out, gr_out, gF, partials,
                                          acc, st)
               : run_adjoint_step<float>(a, f, psi, psi_ready, lam_next, gr_next, lam_out, gr_out, gF, partials,
                                         acc, st);
}

cudaError_t adjoint_step_moments(const AdjointArgs& a, const float* moments, float* psi, bool psi_ready,
                                 const void* lam_next, const void* lam_next2, void* lam_out, void* gF,
                                 double* partials, bool first, cudaStream_t st) {
    const dim3 block(kRowThreads, kRows);
    if (!psi_ready) adj_psi_moments_kernel<<<a.grid, block, 0, st>>>(moments, psi, a);
    Vec4<float>* const v = static_cast<Vec4<float>*>(gF);
    cudaError_t e = launch_chained(
        a.n <= kChainCells, adj_collide1_kernel<float, true>, a.grid, block, 0, st, moments, psi, static_cast<const Vec4<float>*>(lam_next),
        static_cast<const Vec4<float>*>(lam_next2), static_cast<Vec4<float>*>(lam_out), v, partials, first, a);
    if (e != cudaSuccess) return e;
    return launch_chained(a.n <= kChainCells, adj_force_kernel<float, true>, a.grid, block, 0, st, psi, v, static_cast<float*>(lam_out), a);
}

cudaError_t adjoint_seed(const AdjointArgs& a, bool f64, const double* dJdrho, void* lam, void* gr, cudaStream_t st) {
    if (a.tau1) {
        if (f64) adj_seed1_kernel<double><<<a.grid, kThreads, 0, st>>>(dJdrho, static_cast<Vec4<double>*>(lam), a.n);
        else adj_seed1_kernel<float><<<a.grid, kThreads, 0, st>>>(dJdrho, static_cast<Vec4<float>*>(lam), a.n);
        return cudaGetLastError();
    }
    if (f64)
        adj_seed_kernel<double><<<a.grid, kThreads, 0, st>>>(dJdrho, static_cast<double*>(lam),
                                                             static_cast<double*>(gr), a.n);
    else
        adj_seed_kernel<float><<<a.grid, kThreads, 0, st>>>(dJdrho, static_cast<float*>(lam), static_cast<float*>(gr),
                                                            a.n);
    return cudaGetLastError();
}

cudaError_t adjoint_rho0(const AdjointArgs& a, bool f64, const void* lam, const void* gr, double* out,
                         cudaStream_t st) {
    if (a.tau1) {
        if (f64) adj_rho01_kernel<double><<<a.grid, kThreads, 0, st>>>(static_cast<const Vec4<double>*>(lam), out, a.n);
        else adj_rho01_kernel<float><<<a.grid, kThreads, 0, st>>>(static_cast<const Vec4<float>*>(lam), out, a.n);
        return cudaGetLastError();
    }
    if (f64)
        adj_rho0_kernel<double><<<a.grid, kThreads, 0, st>>>(static_cast<const double*>(lam),
                                                             static_cast<const double*>(gr), out, a.n);
    else
        adj_rho0_kernel<float><<<a.grid, kThreads, 0, st>>>(static_cast<const float*>(lam),
                                                            static_cast<const float*>(gr), out, a.n);
    return cudaGetLastError();
}

int adjoint_threads() { return kThreads; }
int adjoint_rows_per_block() { return kRows; }

cudaError_t adjoint_reduce(const AdjointArgs& a, const double* partials, double* acc, cudaStream_t st) {
    adj_reduce_kernel<<<1, kThreads, 0, st>>>(partials, a.grid, acc);
    return cudaGetLastError();
}

}  // namespace lbm
