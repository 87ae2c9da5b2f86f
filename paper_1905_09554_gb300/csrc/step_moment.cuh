// The step of the operators whose post-collision state follows from a few
// moments (32- and 16-bit storage).
//
// SRT at tau = 1 and MRT with its rates at 1 outside {e, 3pxx, pww, pxy, pyz,
// pxz} forget all but 4, 9 or 10 moments of a cell's 19 populations in the
// collision (collide.cuh), so between two steps of one lbm_step call only
// those moments have to be kept: 32, 72 or 80 bytes are read and written per
// cell and step instead of 152.  A call of n steps runs
//   sc_moments_kernel   populations -> moments,
//   sc_moment_kernel    moments -> moments, n - 1 times,
//   sc_moment_kernel    with EMIT: moments -> populations.
// Every population is formed, streamed and summed in the order and rounding
// of the population kernels (for 16-bit storage through its rounding too), so
// n steps at once and n calls of one step give the same bits.
//
// One block marches along z with the cells of a 68 x 15 region (pairs along x,
// one pair per thread, in packed arithmetic) around an output tile of 64 x 13
// (9 or 10 fields: 68 x 11 around 64 x 9, 384 threads of up to 168 registers,
// where 512 of 128 spill and single cells take twice the instructions: 97 and
// 76 against 67 ms for 20 steps of 384 x 384 x 1024).  Per plane p, after one
// barrier, a thread
//   * takes the populations of plane p - 2 that stream in from its
//     neighbours out of shared memory and adds them to the sums of planes
//     p - 3 (complete: written), p - 2 and p - 1,
//   * reads psi of its in-plane neighbours (8 values; what it saw of the two
//     planes below is kept in registers), and collides its cell of plane
//     p - 1, leaving the 16 populations that move within the plane in shared
//     memory for the next turn,
//   * turns the density of plane p + 1, loaded one turn earlier, into psi.
// The region's rim is computed twice (by the neighbouring tiles as well):
// 416 of 512 threads own output cells.  The rim columns sit in one warp of
// their own, so that all other warps load and store whole rows.
//
// Bound: not HBM (47 B a cell and step at 4 fields, 32 without the rims of cut spans, are 60% of the copy rate) but,
// with 4 fields, issue slots and the chain within a plane (224 instructions a
// cell, 49% of the slots at 16 warps an SM), with 9 and 10 the shared memory
// their planes in flight take (384 threads an SM).  Measured, one call: SRT tau = 1, 256 x 256 x 575, 50
// steps 55.9 -> 23.1 ms; FP16 with local references, unit-rate MRT, 20 steps
// 23.4 -> 12.9 ms; 64 uneven boxes, 50 steps 52.6 -> 26.0 ms; the paper's MRT,
// 384 x 384 x 1024, 20 steps 100.8 -> 66.8 ms.
//
// Layout of the fields: rows of nx (rounded up to a multiple of 4) + 4 cells,
// two periodic copies of cells at either end, so that no load wraps along x
// and pairs stay aligned for any nx.  The density comes first by itself; the
// other moments follow two by two, interleaved by thread (one cell's, or one
// pair's, two values side by side), and a last odd one by itself: 3 loads and
// 3 stores for 4 fields, 5 or 6 for 9 or 10.
#pragma once
#include "collide.cuh"
#include "launch.cuh"
#include "step_kernel.cuh"

namespace lbm {

template <int NF>
struct MomentTile {
    static constexpr int ROWS = NF == 4 ? 15 : 11, OUT = ROWS - 2, NT = 32 * (ROWS + 1);
    static constexpr int TXO = 64;
    static constexpr int XP = 35;               // exchange pitch, in region columns
    static constexpr int SLOTS = ROWS * XP;
    static constexpr int NS = 14;               // scalar exchange arrays
    static constexpr int NP = 6;                // pair exchange arrays
    static constexpr int EXCH = SLOTS * (NS + 2 * NP);  // floats per exchange buffer
    // psi: rows -1 .. ROWS, even and odd cells apart
    static constexpr int PP = 35;
    static constexpr int PSI = (ROWS + 2) * PP + 2;
    static constexpr int NRING = 2 * 34;
    // Two turns' buffers (exchange arrays and psi), then the moments in flight:
    // the density of 8 planes (with the ring cells'), the others of 3 or 4, each
    // thread's in slots of its own.
    static constexpr int BUF = (EXCH + 2 * PSI + 3) / 4 * 4;
    static constexpr int RHO = 2 * (NT + NRING);
    static constexpr int REST = 2 * NT * (NF - 1);
    // slot of plane p >= -1 in the ring of the other moments (4 where they fit: a mask instead of a remainder)
    static constexpr int STAGES = NF == 4 ? 4 : 3;
    static constexpr size_t bytes = sizeof(float) * (size_t)(2 * BUF + 8 * RHO + STAGES * REST);
    __device__ static unsigned stage(int p) { return NF == 4 ? unsigned(p) & 3u : unsigned(p + 3) % 3u; }
    static_assert(bytes <= 227 * 1024, "shared memory of one block");
};

// Exchange arrays of a population that changes column: scalar arrays for those
// moving along x (1, 11, 13 / 2, 14, 12; the value that leaves the pair) and,
// two each, along the diagonals; pair arrays for those moving along y only.
__host__ __device__ constexpr int exch_index(int q) {
    constexpr int t[Q] = {-1, 0, 3, 0, 1, -1, -1, 6, 8, 10, 12, 1, 5, 2, 4, 2, 5, 3, 4};
    return t[q];
}

struct MomentArgs {
    int src_hi, dst_hi;  // the buffer's second set of moment fields (0: its first)
    const MomentPiece* pieces;
    const int* first;
};

// The moments of a thread's pair at float offset od of a field.
template <int NF>
__device__ __forceinline__ void store_moments(float* d, long long nf, unsigned od, const F2 (&o)[NF]) {
    static_for<0, (NF + 2) / 2>([&](auto gc) {
        constexpr int g = decltype(gc)::value, k = g == 0 ? 0 : 2 * g - 1;
        if constexpr (k > 0 && k + 1 < NF)
            *reinterpret_cast<ulonglong2*>(d + k * nf + 2 * (long long)od) = make_ulonglong2(o[k].v, o[k + 1].v);
        else if constexpr (k < NF)
            *reinterpret_cast<unsigned long long*>(d + k * nf + od) = o[k].v;
    });
}
// Field k of the cell in column col (0 .. pitch - 1) of the row that starts at
// `row`: rho by itself, then two by two, interleaved by pairs of cells.
template <int NF>
__device__ __forceinline__ float* moment_at(float* d, long long nf, unsigned row, int col, int k) {
    const bool two = k > 0 && ((k - 1) / 2) * 2 + 2 < NF;
    if (!two) return d + k * nf + (row + unsigned(col));
    const int k0 = ((k - 1) / 2) * 2 + 1, which = k - k0;
    return d + k0 * nf + 2 * (long long)(row + unsigned(col / 2 * 2)) + which * 2 + col % 2;
}
// The pair of a thread near the ends of an odd row: value by value, the
// periodic copy of every cell that has one (and, for the pair that sticks out
// of the row, the cell itself).
template <int NF>
__device__ __forceinline__ void store_ends(float* d, long long nf, unsigned od, const F2 (&o)[NF], int x, int nx,
                                           bool stick) {
    const unsigned row = od - unsigned(x + 2);
#pragma unroll 1
    for (int j = stick ? 0 : 2; j < 4; ++j) {  // first the cells, then their copies
        const int e = j % 2, xe = x + e;
        if (xe >= nx) continue;
        int col = xe + 2;
        if (j >= 2) {
            if (xe >= 2 && xe < nx - 2) continue;
            col += xe < 2 ? nx : -nx;
        }
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            float lo, hi;
            unpack2(o[k], lo, hi);
            *moment_at<NF>(d, nf, row, col, k) = e ? hi : lo;
        }
    }
}

template <class Codec, int COLL, bool EMIT, bool BATCH, bool KEEP_PSI = false>
__global__ void __launch_bounds__(MomentTile<kMoments<COLL>>::NT, 1)
sc_moment_kernel(const void* __restrict__ src_all, void* __restrict__ dst_all, const StepArgs a, const BatchArgs b,
                 const MomentArgs ma) {
    using V = F2;
    using S = typename Codec::S;
    constexpr int NF = kMoments<COLL>;
    using T = MomentTile<NF>;
    constexpr int XP = T::XP, PP = T::PP, ROWS = T::ROWS, SLOTS = T::SLOTS;
    constexpr bool LOCAL = Codec::kLocal, HALF = sizeof(S) == 2;
    static_assert(!BATCH || !HALF, "batches hold 32-bit populations");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* const buf0 = reinterpret_cast<float*>(smem_raw);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // region column rp (0 .. 33) and row ry (0 .. 14): rows in warps 0 .. 14, the two rim columns in the last warp
    const bool rim = warp == ROWS;
    // (its two spare lanes keep to the unused column 34)
    const int rp = !rim ? lane + 1 : (lane < ROWS ? 0 : (lane < 2 * ROWS ? 33 : 34));
    const int ry = !rim ? warp : lane % ROWS;
    const bool inner = !rim && ry >= 1 && ry <= T::OUT;  // owns output cells
    const int xs = ry * XP + rp;
    const int ps = (ry + 1) * PP + rp + 1;
    // ring cells (psi only) around the region
    const bool ring = tid < T::NRING;
    const int hp = tid % 34, hy = tid < 34 ? -1 : ROWS;
    const int hs = (hy + 1) * PP + hp + 1;

    constexpr int REST = T::REST;
    float* const rho_st = buf0 + 2 * T::BUF;       // [8][RHO]
    float* const rest_st = rho_st + 8 * T::RHO;    // [STAGES][REST]

    chain_begin();
    const float rho0 = a.rho0f, inv_rho0 = a.inv_rho0f;
    const DevParams& dev = a.dev;
    auto psi_v = [&](V r) { return vmap(r, [&](float x) { return psi_of<float>(x, rho0, inv_rho0); }); };

    for (int piece = ma.first[blockIdx.x]; piece < ma.first[blockIdx.x + 1]; ++piece) {
        const MomentPiece work = ma.pieces[piece];
        int nx, ny, nz, tiles_x;
        long long base = 0;
        if constexpr (BATCH) {
            const BatchBox& bx = b.boxes[work.box];
            nx = bx.nx; ny = bx.ny; nz = bx.nz;
            tiles_x = bx.tiles_x;
            base = bx.base;
        } else {
            nx = a.nx; ny = a.ny; nz = a.nz;
            tiles_x = a.tiles_x;
        }
        const int pitch = moment_pitch(nx);
        const unsigned plane = unsigned(pitch) * unsigned(ny);
        const long long nf = (long long)plane * nz;
        const float* __restrict__ src = static_cast<const float*>(src_all) + base + (ma.src_hi ? NF * nf : 0);

        const int x0 = (work.tile % tiles_x) * T::TXO, y0 = (work.tile / tiles_x) * T::OUT;
        const int zs = work.zs, ze = work.ze;
        const int x = x0 + (rp - 1) * 2, y = y0 + ry - 1;
        const unsigned off = unsigned(wrap_index(y, ny)) * pitch + min(x + 2, pitch - 2);
        const unsigned hoff =
            unsigned(wrap_index(y0 + hy - 1, ny)) * pitch + min(x0 + (hp - 1) * 2 + 2, pitch - 2);
        const bool own = inner && y < ny && x < nx;
        // any cell of this thread with a periodic copy, or a pair that sticks out of an odd row
        const bool edge = x < 2 || x + 2 > nx - 2;
        float* const dst_m = EMIT ? nullptr : static_cast<float*>(dst_all) + base + (ma.dst_hi ? NF * nf : 0);

        auto put_psi = [&](float* buf, int slot, V p) {
            float e, o;
            unpack2(p, e, o);
            buf[slot] = e;
            buf[T::PSI + slot] = o;
        };

        // What a thread keeps of three consecutive planes, rotated by the caller.
        struct Plane {
            PsiView<V> w;
        };
        V own0, own5, own6;          // populations of the last collided plane that stay in the column
        float kept[6];               // those that move along x within the pair
        SumUp<V> up1, upz;           // what plane q sent up (to q + 1), and plane q - 1 (to q)
        V z_r, z_jx, z_jy, z_xx, z_yy, z_xy;  // sums of plane q's cell without what comes from above

        // The density of plane p (and of the ring cells), and the other moments of plane p: copied
        // asynchronously four and three turns before their use, so that no register waits for them.
        int zr = wrap_index(zs - 2, nz), zm = wrap_index(zs - 1, nz);  // planes fetched next
        unsigned rrow = unsigned(zr) * plane, mrow = unsigned(zm) * plane;
        auto fetch_rho = [&](int p) {
            float* const st = rho_st + (p & 7) * T::RHO + 2 * tid;
            async_copy::copy<8>(st, src + (rrow + off));
            if (ring) async_copy::copy<8>(st + 2 * T::NT, src + (rrow + hoff));
            rrow += plane;
            if (++zr == nz) { zr = 0; rrow = 0; }
        };
        auto fetch_rest = [&](int p) {
            const unsigned o = mrow + off;
            float* const st = rest_st + T::stage(p) * REST;
            static_for<0, (NF - 1) / 2>([&](auto gc) {
                constexpr int k = 2 * decltype(gc)::value + 1;
                async_copy::copy<16>(st + (k - 1) * T::NT * 2 + 4 * tid, src + k * nf + 2 * (long long)o);
            });
            if constexpr (NF % 2 == 0)
                async_copy::copy<8>(st + (NF - 2) * T::NT * 2 + 2 * tid, src + (NF - 1) * nf + o);
            mrow += plane;
            if (++zm == nz) { zm = 0; mrow = 0; }
        };
        auto rho_of = [&](int p) -> V { return *reinterpret_cast<const V*>(rho_st + (p & 7) * T::RHO + 2 * tid); };
        // psi of plane p into its turn's buffer
        auto fill_psi = [&](Plane& q, int p) {
            float* const buf = buf0 + (p & 1) * T::BUF + T::EXCH;
            q.w.c = psi_v(rho_of(p));
            put_psi(buf, ps, q.w.c);
            if constexpr (KEEP_PSI) {  // for the adjoint
                if (own && p >= zs && p < ze) {
                    float* d = static_cast<float*>(a.psi_out) + ((long long)p * ny + y) * nx + x;
                    float lo, hi;
                    unpack2(q.w.c, lo, hi);
                    d[0] = lo;
                    if (x + 1 < nx) d[1] = hi;
                }
            }
            if (ring)
                put_psi(buf, hs,
                        psi_v(*reinterpret_cast<const V*>(rho_st + (p & 7) * T::RHO + 2 * (tid + T::NT))));
        };

        Plane pa, pb, pc;
        for (int p = zs - 2; p <= zs; ++p) {
            fetch_rho(p);
            async_copy::commit();
        }
        fetch_rho(zs + 1);
        fetch_rest(zs - 1);
        async_copy::commit();
        async_copy::wait<3>();
        fill_psi(pc, zs - 2);

        // One turn: plane p has its psi in shared memory; prev, cur: planes p - 2, p - 1.
        auto turn = [&](Plane& prev, Plane& cur, Plane& nxt, int p) {
            float* const ex_r = buf0 + (p & 1) * T::BUF;
            float* const ex_w = buf0 + (~p & 1) * T::BUF;
            const float* const psi_r = ex_r + T::EXCH;
            async_copy::wait<2>();  // the density of plane p + 1 and the rest of plane p - 1 are here
            __syncthreads();

            if (p >= zs + 1 && inner) {
                // local-reference storage: this cell's density in the planes that receive
                V ref_dn = vset<V>(0.0f), ref_fl = ref_dn, ref_up = ref_dn;
                if constexpr (LOCAL) {
                    ref_dn = rho_of(p - 3);
                    ref_fl = rho_of(p - 2);
                    ref_up = rho_of(p - 1);
                }
                // population q of plane p - 2 arriving at this thread's cell(s)
                auto got = [&](auto qc) -> V {
                    constexpr int q = decltype(qc)::value;
                    if constexpr (q == 0) return own0;
                    else if constexpr (q == 5) return own5;
                    else if constexpr (q == 6) return own6;
                    else if constexpr (cx(q) == 0) {
                        F2 r;
                        r.v = reinterpret_cast<const unsigned long long*>(ex_r)[exch_index(q) * SLOTS + xs -
                                                                                 cy(q) * XP];
                        return r;
                    } else {
                        // one cell of the pair receives from the neighbouring pair, the other from this
                        // column: along a diagonal out of shared memory, along x it never left the thread
                        const float* e = ex_r + 2 * T::NP * SLOTS + exch_index(q) * SLOTS + xs - cy(q) * XP;
                        const float far = e[-cx(q)];
                        float near;
                        if constexpr (cy(q) == 0) near = kept[exch_index(q)];
                        else near = e[SLOTS];
                        return cx(q) > 0 ? pack2(far, near) : pack2(near, far);
                    }
                };
                auto in = [&](auto qc, V ref) -> V {
                    constexpr int q = decltype(qc)::value;
                    V v = got(qc);
                    if constexpr (LOCAL && !EMIT) {  // through the 16-bit storage of the destination cell
                        float lo, hi, r0, r1;
                        unpack2(v, lo, hi);
                        unpack2(ref, r0, r1);
                        v = pack2(Codec::template decode_ref<q>(Codec::template encode_ref<q>(lo, r0, dev), r0, dev),
                                  Codec::template decode_ref<q>(Codec::template encode_ref<q>(hi, r1, dev), r1, dev));
                    }
                    return v;
                };
                // opposite populations qp and qm.  Along x a pair takes one value of each from this thread
                // and one from a neighbour, in opposite cells: added cell by cell, no register is moved.
                auto both = [&](auto qpc, auto qmc, V ref) -> Opp<V> {
                    constexpr int qp = decltype(qpc)::value, qm = decltype(qmc)::value;
                    if constexpr (!LOCAL && cx(qp) == 1 && cy(qp) == 0) {
                        const float* e = ex_r + 2 * T::NP * SLOTS + xs;
                        const float pl = e[exch_index(qp) * SLOTS - 1], mh = e[exch_index(qm) * SLOTS + 1];
                        const float ph = kept[exch_index(qp)], ml = kept[exch_index(qm)];
                        return {pack2(vadd(pl, ml), vadd(ph, mh)), pack2(vsub(pl, ml), vsub(ph, mh))};
                    } else {
                        return opp(in(qpc, ref), in(qmc, ref));
                    }
                };
#define LBM_IN(q, ref) in(std::integral_constant<int, q>{}, ref)
#define LBM_BOTH(p, m, ref) both(std::integral_constant<int, p>{}, std::integral_constant<int, m>{}, ref)
                if constexpr (EMIT) {
                    S* const dst = static_cast<S*>(dst_all) + base;
                    const long long cells = (long long)nx * ny * nz;
                    auto put = [&](auto qc, int t, V ref) {
                        constexpr int q = decltype(qc)::value;
                        if (own && t >= zs && t < ze) {
                            S* d = dst + q * cells + ((long long)t * ny + y) * nx + x;
                            const V v = got(qc);
                            float lo, hi, r0, r1;
                            unpack2(v, lo, hi);
                            unpack2(ref, r0, r1);
                            const bool two = x + 1 < nx;
                            if constexpr (LOCAL) {
                                Codec::template store_ref<q>(d, lo, r0, dev);
                                if (two) Codec::template store_ref<q>(d + 1, hi, r1, dev);
                            } else if constexpr (HALF) {
                                Codec::template store<q>(d, lo, dev);
                                if (two) Codec::template store<q>(d + 1, hi, dev);
                            } else if ((nx & 1) == 0) {
                                *reinterpret_cast<unsigned long long*>(d) = v.v;
                            } else {
                                d[0] = lo;
                                if (two) d[1] = hi;
                            }
                        }
                    };
                    const int q = p - 2;
#define LBM_PUT(k, t, ref) put(std::integral_constant<int, k>{}, t, ref)
                    LBM_PUT(6, q - 1, ref_dn); LBM_PUT(12, q - 1, ref_dn); LBM_PUT(13, q - 1, ref_dn);
                    LBM_PUT(16, q - 1, ref_dn); LBM_PUT(17, q - 1, ref_dn);
                    LBM_PUT(0, q, ref_fl); LBM_PUT(1, q, ref_fl); LBM_PUT(2, q, ref_fl);
                    LBM_PUT(3, q, ref_fl); LBM_PUT(4, q, ref_fl); LBM_PUT(7, q, ref_fl);
                    LBM_PUT(8, q, ref_fl); LBM_PUT(9, q, ref_fl); LBM_PUT(10, q, ref_fl);
                    LBM_PUT(5, q + 1, ref_up); LBM_PUT(11, q + 1, ref_up); LBM_PUT(14, q + 1, ref_up);
                    LBM_PUT(15, q + 1, ref_up); LBM_PUT(18, q + 1, ref_up);
#undef LBM_PUT
                    if constexpr (LOCAL) {  // the density before this step: the reference of what the cell holds
                        if (own && q >= zs && q < ze) {
                            float* d = a.ref_dst + ((long long)q * ny + y) * nx + x;
                            float lo, hi;
                            unpack2(ref_fl, lo, hi);
                            d[0] = lo;
                            if (x + 1 < nx) d[1] = hi;
                        }
                    }
                } else {
                    // from above: plane p - 3 is complete
                    const SumUp<V> dn =
                        sum_vertical(LBM_IN(6, ref_dn), LBM_BOTH(13, 12, ref_dn), LBM_BOTH(17, 16, ref_dn));
                    const int t = p - 3;
                    if (own && t >= zs) {
                        V o[NF];
                        moments_from<COLL, V>(upz, z_r, z_jx, z_jy, z_xx, z_yy, z_xy, dn, o);
                        float* const d = dst_m;
                        const unsigned od = unsigned(t) * plane + unsigned(y) * pitch + unsigned(x + 2);
                        const bool stick = x + 1 >= nx;
                        if (!stick) store_moments<NF>(d, nf, od, o);
                        if (edge) {
                            if ((nx & 1) == 0) store_moments<NF>(d, nf, od + (x < 2 ? nx : -nx), o);
                            else store_ends<NF>(d, nf, od, o, x, nx, stick);
                        }
                    }
                    const SumFlat<V> fl = sum_flat(LBM_IN(0, ref_fl), LBM_BOTH(1, 2, ref_fl),
                                                   LBM_BOTH(3, 4, ref_fl), LBM_BOTH(7, 8, ref_fl),
                                                   LBM_BOTH(9, 10, ref_fl));
                    upz = up1;
                    z_r = vadd(upz.r, fl.r);
                    z_jx = vadd(upz.dx, fl.jx);
                    z_jy = vadd(upz.dy, fl.jy);
                    if constexpr (NF > 4) {
                        z_xx = vadd(upz.sx, fl.xx);
                        z_yy = vadd(upz.sy, fl.yy);
                        z_xy = fl.xy;
                    }
                    up1 = sum_vertical(LBM_IN(5, ref_up), LBM_BOTH(11, 14, ref_up), LBM_BOTH(15, 18, ref_up));
                }
#undef LBM_IN
#undef LBM_BOTH
            }

            if (p <= ze + 1) {
                {
                    // rows y - 1, y, y + 1: left neighbour, the pair, right neighbour; differences along x
                    // are formed cell by cell (they mix the halves of neighbouring pairs)
                    float l[3], e[3], o[3], r[3];
                    unpack2(nxt.w.c, e[1], o[1]);
                    static_for<0, 3>([&](auto kc) {
                        constexpr int k = decltype(kc)::value;
                        const float* pe = psi_r + ps + (k - 1) * PP;
                        const float* po = pe + T::PSI;
                        if constexpr (k != 1) { e[k] = pe[0]; o[k] = po[0]; }
                        l[k] = po[-1];
                        r[k] = pe[1];
                    });
                    const F2 ym = pack2(e[0], o[0]), yp = pack2(e[2], o[2]);
                    nxt.w.ex = pack2(vsub(o[1], l[1]), vsub(r[1], e[1]));
                    nxt.w.ey = vsub(yp, ym);
                    nxt.w.s4 = vadd(pack2(vadd(o[1], l[1]), vadd(r[1], e[1])), vadd(yp, ym));
                    const F2 da = pack2(vsub(o[2], l[0]), vsub(r[2], e[0]));
                    const F2 db = pack2(vsub(o[0], l[2]), vsub(r[0], e[2]));
                    nxt.w.dx = vadd(da, db);
                    nxt.w.dy = vsub(da, db);
                }
                if (p >= zs) {  // collide plane p - 1
                    const Force<V> F = force_of(prev.w, cur.w, nxt.w, a.gwf);
                    V m[NF];
                    m[0] = rho_of(p - 1);
                    const float* const st = rest_st + T::stage(p - 1) * REST;
                    static_for<0, (NF - 1) / 2>([&](auto gc) {
                        constexpr int k = 2 * decltype(gc)::value + 1;
                        const float* q = st + (k - 1) * T::NT * 2 + 4 * tid;
                        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(q);
                        m[k].v = v.x;
                        m[k + 1].v = v.y;
                    });
                    if constexpr (NF % 2 == 0)
                        m[NF - 1] = *reinterpret_cast<const V*>(st + (NF - 2) * T::NT * 2 + 2 * tid);
                    collide_moments<COLL, V, true>(m, F, a, [&](auto qc, V f) {
                        constexpr int q = decltype(qc)::value;
                        if constexpr (HALF && !LOCAL && !EMIT) {  // through the 16-bit storage
                            f = vmap(f, [&](float v) {
                                return Codec::template decode<q>(Codec::template encode<q>(v, dev), dev);
                            });
                        }
                        if constexpr (q == 0) own0 = f;
                        else if constexpr (q == 5) own5 = f;
                        else if constexpr (q == 6) own6 = f;
                        else {
                            float lo, hi;
                            unpack2(f, lo, hi);
                            float* e = ex_w + 2 * T::NP * SLOTS + exch_index(q) * SLOTS + xs;
                            if constexpr (cx(q) == 0) {
                                reinterpret_cast<unsigned long long*>(ex_w)[exch_index(q) * SLOTS + xs] = f.v;
                            } else {
                                const float near = cx(q) > 0 ? lo : hi;
                                e[0] = cx(q) > 0 ? hi : lo;
                                if constexpr (cy(q) == 0) kept[exch_index(q)] = near;
                                else e[SLOTS] = near;
                            }
                        }
                    });
                }
                if (p <= ze) fill_psi(prev, p + 1);
                if (p <= ze - 3) fetch_rho(p + 4);
                if (p <= ze - 2) fetch_rest(p + 2);
            }
            async_copy::commit();
        };
        for (int p = zs - 2; p <= ze + 2; p += 3) {
            turn(pa, pb, pc, p);
            if (p + 1 <= ze + 2) turn(pb, pc, pa, p + 1);
            if (p + 2 <= ze + 2) turn(pc, pa, pb, p + 2);
        }
    }
    chain_end();
}

// Populations -> moment fields (all the operators above read of a state).
// One thread per cell along x rows; of a batch, blockIdx.y takes every
// gridDim.y-th box (a grid has at most 65,535 rows of blocks, a batch has no
// such limit).
constexpr int kMomentGatherRows = 65535;

template <class Codec, int COLL, bool BATCH>
__global__ void __launch_bounds__(256)
sc_moments_kernel(const void* __restrict__ src_all, void* __restrict__ dst_all, const StepArgs a, const BatchArgs b) {
    using S = typename Codec::S;
    constexpr int NF = kMoments<COLL>;
    chain_begin();
    const DevParams& dev = a.dev;
    auto gather = [&](int nx, int ny, int nz, long long base) {
        const long long n = (long long)nx * ny * nz;
        const int pitch = moment_pitch(nx);
        const unsigned rows = unsigned(ny) * unsigned(nz);
        const long long nf = (long long)pitch * rows;
        const S* __restrict__ src = static_cast<const S*>(src_all) + base;
        float* dst = static_cast<float*>(dst_all) + base;
        for (unsigned r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8) {
            for (int x = threadIdx.x & 31; x < nx; x += 32) {
                const long long cell = (long long)r * nx + x;
                float f[Q], m[NF];
                float ref = 0.0f;
                if constexpr (Codec::kLocal) ref = __ldg(a.ref_src + cell);
                static_for<0, Q>([&](auto qc) {
                    constexpr int q = decltype(qc)::value;
                    const S* p = src + (q * n + cell);
                    if constexpr (Codec::kLocal) f[q] = Codec::template load_ref<q>(p, ref, dev);
                    else f[q] = Codec::template load<q>(p, dev);
                });
                moments_of<COLL, float>(f, m);
                const unsigned row = r * unsigned(pitch);
                const int g = x < 2 ? nx : (x >= nx - 2 ? -nx : 0);
                static_for<0, NF>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
                    *moment_at<NF>(dst, nf, row, x + 2, k) = m[k];
                    if (g) *moment_at<NF>(dst, nf, row, x + 2 + g, k) = m[k];
                });
            }
        }
    };
    if constexpr (BATCH) {
        for (int i = int(blockIdx.y); i < b.nbox; i += int(gridDim.y)) {
            const BatchBox& bx = b.boxes[i];
            gather(bx.nx, bx.ny, bx.nz, bx.base);
        }
    } else {
        gather(a.nx, a.ny, a.nz, 0);
    }
}

inline bool moment_chain(const MomentLaunch& l) { return !l.batch.nbox && l.args.n <= kChainCells; }

template <class Codec, int COLL, bool EMIT, bool BATCH>
cudaError_t moment_launch(const MomentLaunch& l, const void* src, void* dst) {
    using T = MomentTile<kMoments<COLL>>;
    const int sm = (int)T::bytes;
    if constexpr (COLL == COLL_SRT && !EMIT && !BATCH && std::is_same_v<Codec, CodecF32>) {
        if (l.args.psi_out) {
            auto kern = sc_moment_kernel<Codec, COLL, EMIT, BATCH, true>;
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
            if (e != cudaSuccess) return e;
            return launch_chained(moment_chain(l), kern, l.grid, T::NT, sm, l.stream, src, dst, l.args, l.batch,
                                  MomentArgs{l.src_hi, l.dst_hi, l.pieces, l.first});
        }
    }
    return launch_chained(moment_chain(l), sc_moment_kernel<Codec, COLL, EMIT, BATCH>, l.grid, T::NT,
                          sm, l.stream, src, dst, l.args, l.batch, MomentArgs{l.src_hi, l.dst_hi, l.pieces, l.first});
}

template <class Codec, int COLL, bool EMIT>
cudaError_t moment_dispatch(const MomentLaunch& l, const void* src, void* dst) {
    if constexpr (sizeof(typename Codec::S) == 4) {
        if (l.batch.nbox) return moment_launch<Codec, COLL, EMIT, true>(l, src, dst);
    }
    return moment_launch<Codec, COLL, EMIT, false>(l, src, dst);
}

template <class Codec, int COLL>
cudaError_t moment_gather(const MomentLaunch& l, const void* src, void* dst) {
    if constexpr (sizeof(typename Codec::S) == 4) {
        if (l.batch.nbox)
            return launch_chained(moment_chain(l), sc_moments_kernel<Codec, COLL, true>,
                                  dim3(l.gather_grid, l.batch.nbox < kMomentGatherRows ? l.batch.nbox : kMomentGatherRows),
                                  256, 0, l.stream, src, dst, l.args, l.batch);
    }
    return launch_chained(moment_chain(l), sc_moments_kernel<Codec, COLL, false>, l.gather_grid, 256, 0, l.stream, src, dst, l.args,
                          l.batch);
}

template <class Codec, int COLL, bool EMIT, bool BATCH>
int moment_prepare_one() {
    using T = MomentTile<kMoments<COLL>>;
    auto kern = sc_moment_kernel<Codec, COLL, EMIT, BATCH>;
    const int sm = (int)T::bytes;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    int per_sm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T::NT, sm);
    return e == cudaSuccess ? per_sm : -int(e);
}

template <class Codec, int COLL>
int moment_prepare(bool batch) {
    int k = 0, e = 0;
    if constexpr (sizeof(typename Codec::S) == 4) {
        if (batch) {
            k = moment_prepare_one<Codec, COLL, false, true>();
            e = moment_prepare_one<Codec, COLL, true, true>();
            return k < e ? k : e;
        }
    }
    k = moment_prepare_one<Codec, COLL, false, false>();
    e = moment_prepare_one<Codec, COLL, true, false>();
    return k < e ? k : e;
}

}  // namespace lbm

// Defines the moment kernels of one (storage, collision) pair.
#define LBM_MOMENT_INSTANCE(NAME, CODEC, COLL)                                                       \
    namespace lbm {                                                                                  \
    extern const MomentKernels kMoment_##NAME = {moment_prepare<CODEC, COLL>, moment_gather<CODEC, COLL>, \
                                                 moment_dispatch<CODEC, COLL, false>,                \
                                                 moment_dispatch<CODEC, COLL, true>, kMoments<COLL>, \
                                                 MomentTile<kMoments<COLL>>::TXO,                    \
                                                 MomentTile<kMoments<COLL>>::OUT};     \
    }
