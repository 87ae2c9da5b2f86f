// Moments, force and collision of one cell, shared by every step kernel.
//
// Every operation below is written as a single rounded add, subtract,
// multiply or fused multiply-add, in one fixed order, so that a kernel that
// holds a cell's 19 populations and a kernel that holds only its moments
// (step_moment.cuh) give the same bits, whatever the compiler contracts.
//
// V is float, double, or F2 (two cells of float in one 64-bit register: GB300
// issues a packed add / multiply / fma for both cells at once, each rounded
// as the scalar operation).
#pragma once
#include "lattice.cuh"
#include "step_args.h"

namespace lbm {

struct F2 {
    unsigned long long v;
};

template <class V> struct VecTraits { using R = V; static constexpr int N = 1; };
template <> struct VecTraits<F2> { using R = float; static constexpr int N = 2; };

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float vfnma(float a, float b, float c) { return __fmaf_rn(-a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double vfnma(double a, double b, double c) { return __fma_rn(-a, b, c); }

__device__ __forceinline__ F2 pack2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 vadd(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vsub(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 vfnma(F2 a, F2 b, F2 c) {
    a.v ^= 0x8000000080000000ull;
    return vfma(a, b, c);
}

// The scalar s in every cell of a V.
template <class V, class S>
__device__ __forceinline__ V vset(S s) {
    if constexpr (VecTraits<V>::N == 2) return pack2(float(s), float(s));
    else return V(s);
}
// Element-wise scalar function.
template <class V, class F>
__device__ __forceinline__ V vmap(V a, F&& f) {
    if constexpr (VecTraits<V>::N == 2) {
        float lo, hi;
        unpack2(a, lo, hi);
        return pack2(f(lo), f(hi));
    } else {
        return f(a);
    }
}

// c a and c a + b for a number c, the same for every cell: two scalar
// instructions for a pair, whose c is an immediate or a constant-bank operand
// (a packed one would need c twice in a register pair).
template <class V, class S>
__device__ __forceinline__ V vmulc(S c, V a) {
    using R = typename VecTraits<V>::R;
    return vmap(a, [&](R x) { return vmul(x, R(c)); });
}
// -a, and 2 a + b (doubling is exact: one rounding either way).
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ F2 vneg(F2 a) { return vmulc(-1.0f, a); }
__device__ __forceinline__ float vtwice(float a, float b) { return vfma(2.0f, a, b); }
__device__ __forceinline__ double vtwice(double a, double b) { return vfma(2.0, a, b); }
__device__ __forceinline__ F2 vtwice(F2 a, F2 b) { return vadd(vadd(a, a), b); }
__device__ __forceinline__ float vmul1(float a, float b) { return vmul(a, b); }
__device__ __forceinline__ double vmul1(double a, double b) { return vmul(a, b); }
__device__ __forceinline__ F2 vmul1(F2 a, F2 b) {
    float al, ah, bl, bh;
    unpack2(a, al, ah);
    unpack2(b, bl, bh);
    return pack2(vmul(al, bl), vmul(ah, bh));
}
template <class V, class S>
__device__ __forceinline__ V vfmac(S c, V a, V b) {
    if constexpr (VecTraits<V>::N == 2) {
        float al, ah, bl, bh;
        unpack2(a, al, ah);
        unpack2(b, bl, bh);
        return pack2(vfma(al, float(c), bl), vfma(ah, float(c), bh));
    } else {
        return vfma(a, V(c), b);
    }
}
template <class V, class S, class T>
__device__ __forceinline__ V vfmac(S c, V a, T b) {  // b a number, too
    using R = typename VecTraits<V>::R;
    return vmap(a, [&](R x) { return vfma(x, R(c), R(b)); });
}

// psi = rho0 (1 - exp(-rho/rho0)).  Float arithmetic uses the hardware's base-2
// exponential (2 ulp, and the rounding of its argument: a few ulp for the
// densities of a two-phase state, |rho/rho0| < 4) instead of the correctly
// rounded expf, whose range reduction costs about eight more instructions per
// call.  Subnormal arguments and results are flushed (psi rounds to the same
// value), which saves the scaling around them.
//
// FP64: the table-driven method of Tang (ACM Trans. Math. Softw. 15, 1989) with
// 64 entries, 11 FP64 operations where exp takes 16: with
// a = n ln2/64 + r, |r| <= ln2/128, and n = 64 m + j,
//   e^a = 2^m 2^(j/64) e^r,  e^r - 1 = r + c2 r^2 + ... + c5 r^5.
// An entry is 2^(j/64) as the sum of two doubles, so that only the last sum
// rounds visibly; ln2/64 is split so that n times its upper part is exact.  The
// c are the Taylor series' with its next two terms economised: r^6 and r^7
// replaced by the combinations of r^2, r^4 and r^3, r^5 that stay closest to
// them on the interval (Chebyshev's T_3 in r^2 with its first zero moved to 0),
// which leaves 1.4e-18 of the 3.5e-17 that the plain series leaves off.
// Below the range of normal results, and for NaN and infinities, exp itself is
// called.
// Worst error over 500 k arguments in [-4.6, 0]: 0.52 ulp (exp: 0.86; with entries
// of one double and the plain series 1.25, two operations fewer a step: 14.51
// against 14.77 ms for 10 steps of 128 x 128 x 288, the division below included).
__device__ const double2 kExp2Table[64] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
    {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55}, {0x1.0874518759bc8p+0, 0x1.186be4bb284ffp-57},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.03a1727c57b53p-59},
    {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54}, {0x1.1429aaea92de0p+0, -0x1.32fbf9af1369ep-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1a35beb6fcb75p+0, 0x1.e5b4c7b4968e4p-55},
    {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54}, {0x1.2063b88628cd6p+0, 0x1.dc775814a8495p-55},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.26b4565e27cddp+0, 0x1.2bd339940e9d9p-55},
    {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55}, {0x1.2d285a6e4030bp+0, 0x1.0024754db41d5p-54},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.33c08b26416ffp+0, 0x1.32721843659a6p-54},
    {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54}, {0x1.3a7db34e59ff7p+0, -0x1.5e436d661f5e3p-56},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.4160a21f72e2ap+0, -0x1.ef3691c309278p-58},
    {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59}, {0x1.486a2b5c13cd0p+0, 0x1.3c1a3b69062f0p-56},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.4b309d25957e3p-54},
    {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55}, {0x1.56f4736b527dap+0, 0x1.9bb2c011d93adp-54},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.5e76f15ad2148p+0, 0x1.ba6f93080e65ep-54},
    {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54}, {0x1.6623882552225p+0, -0x1.bb60987591c34p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.6dfb23c651a2fp+0, -0x1.bbe3a683c88abp-57},
    {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55}, {0x1.75feb564267c9p+0, -0x1.0245957316dd3p-54},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.7e2f336cf4e62p+0, 0x1.05d02ba15797ep-56},
    {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54}, {0x1.868d99b4492edp+0, -0x1.fc6f89bd4f6bap-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.8f1ae99157736p+0, 0x1.5cc13a2e3976cp-55},
    {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57}, {0x1.97d829fde4e50p+0, -0x1.d185b7c1b85d1p-54},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a0c667b5de565p+0, -0x1.359495d1cd533p-54},
    {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.0fac90ef7fd31p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b33a2b84f15fbp+0, -0x1.2805e3084d708p-57},
    {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56}, {0x1.bcc1e904bc1d2p+0, 0x1.23dd07a2d9e84p-55},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.c67f12e57d14bp+0, 0x1.2884dff483cadp-54},
    {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56}, {0x1.d072d4a07897cp+0, -0x1.cbc3743797a9cp-54},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.da9e603db3285p+0, 0x1.c2300696db532p-54},
    {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54}, {0x1.e502ee78b3ff6p+0, 0x1.39e8980a9cc8fp-55},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.efa1bee615a27p+0, 0x1.dc7f486a4b6b0p-54},
    {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54}, {0x1.fa7c1819e90d8p+0, 0x1.74853f3a5931ep-55}};

__device__ __forceinline__ double exp_table(double a) {
    if (!(fabs(a) < 700.0)) return exp(a);
    const double shift = 6755399441055744.0;  // 1.5 2^52: adding it rounds to an integer in the low bits
    const double t = __fma_rn(a, 0x1.71547652b82fep+6, shift);
    const int n = __double2loint(t);
    const double k = __dsub_rn(t, shift);
    double r = __fma_rn(k, -0x1.62e4200000000p-7, a);
    r = __fma_rn(k, -0x1.fdf473de6af28p-28, r);
    double p = __fma_rn(r, 0x1.1111227699597p-7, 0x1.555573c703d40p-5);
    p = __fma_rn(r, p, 0x1.5555555554afdp-3);
    p = __fma_rn(r, p, 0x1.fffffffffdbccp-2);
    p = __fma_rn(__dmul_rn(r, r), p, r);
    const double2 s = __ldg(kExp2Table + (n & 63));
    const double e = __dadd_rn(s.x, __fma_rn(s.x, p, s.y));
    return __hiloint2double(__double2hiint(e) + ((n >> 6) << 20), __double2loint(e));
}

template <class R>
__device__ __forceinline__ R psi_of(R rho, R rho0, R inv_rho0);
template <>
__device__ __forceinline__ double psi_of<double>(double rho, double rho0, double inv_rho0) {
    return __dmul_rn(rho0, __dsub_rn(1.0, exp_table(__dmul_rn(-rho, inv_rho0))));
}
template <>
__device__ __forceinline__ float psi_of<float>(float rho, float rho0, float inv_rho0) {
    float e;  // inv_rho0 times -log2(e): the same for every cell, formed once
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(__fmul_rn(rho, __fmul_rn(inv_rho0, -1.4426950408889634f))));
    return __fmul_rn(rho0, __fsub_rn(1.0f, e));
}

// 1/rho.  FP64 divides.  Float arithmetic uses the hardware reciprocal (within 1
// ulp) instead of the IEEE division, whose special-case check adds a branch per
// cell.
template <class R>
__device__ __forceinline__ R recip(R x);
template <>
__device__ __forceinline__ double recip<double>(double x) {
    return 1.0 / x;
}
template <>
__device__ __forceinline__ float recip<float>(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ------------------------------------------------------------------ moments
// The populations that move up (c_z = +1), stay in the plane (c_z = 0) and
// move down (c_z = -1) are summed apart, because a kernel that marches along
// z receives them from three different planes.

template <class V>
struct SumUp {  // one of the two groups with c_z != 0
    V r;        // its density
    V dx, dy;   // x and y momentum
    V sx, sy;   // sums of its two x-moving and its two y-moving populations
};

template <class V>
struct Opp {  // two opposite populations: their sum and difference
    V s, d;
};
template <class V>
__device__ __forceinline__ Opp<V> opp(V p, V m) {
    return {vadd(p, m), vsub(p, m)};
}

// f0: straight along z; x, y: the two with c_x (c_y) = +1, -1.
template <class V>
__device__ __forceinline__ SumUp<V> sum_vertical(V f0, const Opp<V>& x, const Opp<V>& y) {
    SumUp<V> s;
    s.sx = x.s;
    s.sy = y.s;
    s.r = vadd(f0, vadd(x.s, y.s));
    s.dx = x.d;
    s.dy = y.d;
    return s;
}

template <class V>
struct SumFlat {  // the nine populations with c_z = 0
    V r, jx, jy;
    V xx, yy, xy;  // second moments
};

// f0 and the opposite pairs (1, 2), (3, 4), (7, 8), (9, 10) of the library's velocity order.
template <class V>
__device__ __forceinline__ SumFlat<V> sum_flat(V f0, const Opp<V>& a, const Opp<V>& b, const Opp<V>& c,
                                               const Opp<V>& d) {
    SumFlat<V> s;
    const V sdiag = vadd(c.s, d.s);
    s.r = vadd(f0, vadd(vadd(a.s, b.s), sdiag));
    s.jx = vadd(a.d, vadd(c.d, d.d));
    s.jy = vadd(b.d, vsub(c.d, d.d));
    s.xx = vadd(a.s, sdiag);
    s.yy = vadd(b.s, sdiag);
    s.xy = vsub(c.s, d.s);
    return s;
}

template <int COLL>
constexpr int kMoments = moments_of_operator(COLL);

template <int COLL, class V>
__device__ __forceinline__ void moments_from(const SumUp<V>& up, const V& rho_uf, const V& jx_uf, const V& jy_uf,
                                             const V& xx_uf, const V& yy_uf, const V& xy, const SumUp<V>& dn,
                                             V (&m)[kMoments<COLL>]) {
    // rho_uf etc.: the sums of the up and flat groups
    m[0] = vadd(rho_uf, dn.r);
    m[1] = vadd(jx_uf, dn.dx);
    m[2] = vadd(jy_uf, dn.dy);
    m[3] = vsub(up.r, dn.r);
    if constexpr (COLL == COLL_MRT_SHEAR || COLL == COLL_MRT_SPARSE) {
        const V xx = vadd(xx_uf, dn.sx), yy = vadd(yy_uf, dn.sy), zz = vadd(up.r, dn.r);
        const V yz = vsub(up.dy, dn.dy), xz = vsub(up.dx, dn.dx);
        if constexpr (COLL == COLL_MRT_SHEAR) {
            m[4] = vsub(vadd(xx, xx), vadd(yy, zz));
            m[5] = vsub(yy, zz);
            m[6] = xy;
            m[7] = yz;
            m[8] = xz;
        } else {
            m[4] = xx;
            m[5] = yy;
            m[6] = zz;
            m[7] = xy;
            m[8] = yz;
            m[9] = xz;
        }
    }
}

// Moments of 19 populations in registers.
template <int COLL, class V>
__device__ __forceinline__ void moments_of(const V (&f)[Q], V (&m)[kMoments<COLL>]) {
    const SumUp<V> up = sum_vertical(f[5], opp(f[11], f[14]), opp(f[15], f[18]));
    const SumUp<V> dn = sum_vertical(f[6], opp(f[13], f[12]), opp(f[17], f[16]));
    const SumFlat<V> fl = sum_flat(f[0], opp(f[1], f[2]), opp(f[3], f[4]), opp(f[7], f[8]), opp(f[9], f[10]));
    moments_from<COLL, V>(up, vadd(up.r, fl.r), vadd(up.dx, fl.jx), vadd(up.dy, fl.jy), vadd(up.sx, fl.xx),
                          vadd(up.sy, fl.yy), fl.xy, dn, m);
}

// Density of a cell alone, from a getter of population q: the rho of
// moments_of.
template <class V, class Get>
__device__ __forceinline__ V density_of(Get&& f) {
    auto at = [&](auto qc) { return f(qc); };
#define LBM_AT(q) at(std::integral_constant<int, q>{})
    const V up = vadd(LBM_AT(5), vadd(vadd(LBM_AT(11), LBM_AT(14)), vadd(LBM_AT(15), LBM_AT(18))));
    const V fl = vadd(LBM_AT(0), vadd(vadd(vadd(LBM_AT(1), LBM_AT(2)), vadd(LBM_AT(3), LBM_AT(4))),
                                      vadd(vadd(LBM_AT(7), LBM_AT(8)), vadd(LBM_AT(9), LBM_AT(10)))));
    const V dn = vadd(LBM_AT(6), vadd(vadd(LBM_AT(13), LBM_AT(12)), vadd(LBM_AT(17), LBM_AT(16))));
#undef LBM_AT
    return vadd(vadd(up, fl), dn);
}

// -------------------------------------------------------------------- force
// Eq. SC_force, F = -G psi sum_a w_a psi(x + c_a) c_a, from what a cell sees
// of each of three planes.  36 w_a = 2 on the axes and 1 on the edges, so
//   36 S_x = 2 ex(z) + dx(z) + ex(z-1) + ex(z+1),
//   36 S_z = 2 (c(z+1) - c(z-1)) + s4(z+1) - s4(z-1).
template <class V>
struct PsiView {
    V c;       // psi of the cell
    V s4;      // sum over its four axis neighbours in the plane
    V ex, ey;  // differences along x and y
    V dx, dy;  // the same from the four diagonal neighbours
};

// psi at an offset in a plane of row pitch PX.
template <class R, int PX>
struct PsiAt {
    const R* p;
    template <class DX, class DY>
    __device__ __forceinline__ R operator()(DX, DY) const {
        return p[DX::value + DY::value * PX];
    }
};

// p(dx, dy): psi of the neighbour in the plane (compile-time offsets).
template <class V, class P>
__device__ __forceinline__ void psi_axis(PsiView<V>& w, P&& p) {
    const V xp = p(std::integral_constant<int, 1>{}, std::integral_constant<int, 0>{});
    const V xm = p(std::integral_constant<int, -1>{}, std::integral_constant<int, 0>{});
    const V yp = p(std::integral_constant<int, 0>{}, std::integral_constant<int, 1>{});
    const V ym = p(std::integral_constant<int, 0>{}, std::integral_constant<int, -1>{});
    w.ex = vsub(xp, xm);
    w.ey = vsub(yp, ym);
    w.s4 = vadd(vadd(xp, xm), vadd(yp, ym));
}
template <class V, class P>
__device__ __forceinline__ void psi_diag(PsiView<V>& w, P&& p) {
    const V a = vsub(p(std::integral_constant<int, 1>{}, std::integral_constant<int, 1>{}),
                     p(std::integral_constant<int, -1>{}, std::integral_constant<int, -1>{}));
    const V b = vsub(p(std::integral_constant<int, 1>{}, std::integral_constant<int, -1>{}),
                     p(std::integral_constant<int, -1>{}, std::integral_constant<int, 1>{}));
    w.dx = vadd(a, b);
    w.dy = vsub(a, b);
}

// F = g (sx, sy, sz), kept as factors: every use multiplies and adds.
template <class V>
struct Force {
    V g, sx, sy, sz;
};
// gw: float -G/36, double -G: there the weight 1/36 is a factor of its own, with
// the same rounding (5.6e-17 low) as in the equilibrium's w rho, so that the two
// cancel in the balance of pressure and force that sets the densities of the
// phases.  -G/36 rounded once is off by another amount (8.1e-17 high at G =
// -5.5): 20 steps then left the vapour's density 4e-16 to 9e-16 low.
template <class V, class R>
__device__ __forceinline__ Force<V> force_of(const PsiView<V>& lo, const PsiView<V>& mid, const PsiView<V>& hi,
                                             R gw) {
    Force<V> F;
    F.g = vmulc(gw, mid.c);
    if constexpr (sizeof(R) == sizeof(double)) F.g = vmul(F.g, 1.0 / 36.0);
    const V dc = vsub(hi.c, lo.c);
    F.sx = vtwice(mid.ex, vadd(mid.dx, vadd(lo.ex, hi.ex)));
    F.sy = vtwice(mid.ey, vadd(mid.dy, vadd(lo.ey, hi.ey)));
    F.sz = vtwice(dc, vsub(hi.s4, lo.s4));
    return F;
}

// ---------------------------------------------------------------- collision
// With a = 3 u' and h = w rho / 2, the equilibrium is
//   f_eq = h (b + (c.a)^2) +/- 2 h c.a,   b = 2 - a.a/3,
// an even and an odd part for each pair of opposite velocities.
//
// SRT (Eq. vel_shift): u' = (j + tau F)/rho, f* = f + omega (f_eq - f).
//
// MRT with Guo-like forcing (Eq. barycentric) at u_b = (j + F/2)/rho, rates 1
// outside K = {e, 3pxx, pww, pxy, pyz, pxz}: writing
// m* = m_eq + S/2 + (1 - s)(m - m_eq + S/2), the conserved rows vanish (rho:
// m = m_eq, S = 0; j: m - m_eq = -F/2, S = F), rows with s = 1 vanish, and
//   f* = f_eq(rho, u_b) + S_pop/2 + sum_{k in K} M_k^T (1 - s_k)(m_k - m_eq_k + S_k/2)/norm_k.
// With phi = 1.5 F/rho and a = 3 (j + F)/rho the first two terms are
//   h (b + (c.a)^2 - (c.phi)^2) +/- 2 h c.a,   b = 2 - (a.a - phi.phi)/3,
// and with g = a - 2 phi the second moments entering the rows of K are
//   N_ij = Pi_ij - rho delta_ij/3 - (rho/9)(g_i g_j - phi_i phi_j).
// The energy row is left out under the shear rule, where its rate is 1.
//
// w_a rho per speed shell, the rest one from sum_a w_a = 1: the rounded
// weights float(1/3) + 6 float(1/18) + 12 float(1/36) sum to 1 + 3e-8, which
// made FP32 runs gain ~3e-8 of their mass every step.

// put(q, value) receives f*_q (for SRT at tau != 1: omega f_eq_q, to which
// the caller adds (1 - omega) f_q).  TAU1: SRT at tau = 1, known when compiled
// (multiplications by 1 are left out; the values are the same).
template <int COLL, class V, bool TAU1 = false, class Put>
__device__ __forceinline__ void collide_moments(const V (&m)[kMoments<COLL>], const Force<V>& F, const StepArgs& a,
                                                Put&& put) {
    using R = typename VecTraits<V>::R;
    constexpr bool SRT = COLL == COLL_SRT;
    constexpr bool ROWS = COLL == COLL_MRT_SHEAR || COLL == COLL_MRT_SPARSE;
    const V rho = m[0];
    const V inv = vmap(rho, [](R r) { return recip(r); });
    const V inv3 = vmulc(R(3), inv);
    V ax, ay, az, px, py, pz;
    V b;
    V gt = F.g;  // a = 3 (j + tau F)/rho (SRT), 3 (j + F)/rho (MRT)
    if constexpr (SRT && !TAU1) gt = vmulc(par<R>(a.tau, a.tauf), F.g);
    ax = vmul(inv3, vfma(gt, F.sx, m[1]));
    ay = vmul(inv3, vfma(gt, F.sy, m[2]));
    az = vmul(inv3, vfma(gt, F.sz, m[3]));
    const V aa = vfma(az, az, vfma(ay, ay, vmul(ax, ax)));
    if constexpr (SRT) {
        px = py = pz = aa;  // not used
        b = vfmac(R(-1.0 / 3.0), aa, R(2));
    } else {
        const V i15 = vmul(vmulc(R(1.5), inv), F.g);
        px = vmul(i15, F.sx);
        py = vmul(i15, F.sy);
        pz = vmul(i15, F.sz);
        b = vfmac(R(-1.0 / 3.0), vfnma(pz, pz, vfnma(py, py, vfnma(px, px, aa))), R(2));
    }
    // 2 h per speed shell: w rho on the axes (r1) and edges (r2 = rho/36, and r1 = 2 r2)
    V r2 = vmulc(R(1.0 / 36.0), rho);
    V r0 = vfmac(R(-24), r2, rho);

    // corrections of the even part: rest, axis x / y / z, edges xy / xz / yz (+/- for the two pairs of an edge)
    V k0, kx, ky, kz, kxy, kxz, kyz, cxy, cxz, cyz;
    if constexpr (ROWS) {
        const V gx = vfmac(R(-2), px, ax), gy = vfmac(R(-2), py, ay), gz = vfmac(R(-2), pz, az);
        const V r9 = vmulc(R(1.0 / 9.0), rho);
        auto flow = [&](V g1, V g2, V p1, V p2) { return vfnma(p1, p2, vmul(g1, g2)); };
        const V xx = flow(gx, gx, px, px), yy = flow(gy, gy, py, py), zz = flow(gz, gz, pz, pz);
        const R(&kk)[6] = row_rates<R>(a);
        V d1, d2, pxy, pyz, pxz;
        if constexpr (COLL == COLL_MRT_SHEAR) {
            d1 = m[4];
            d2 = m[5];
            pxy = m[6];
            pyz = m[7];
            pxz = m[8];
        } else {
            d1 = vsub(vadd(m[4], m[4]), vadd(m[5], m[6]));
            d2 = vsub(m[5], m[6]);
            pxy = m[7];
            pyz = m[8];
            pxz = m[9];
        }
        const V A = vmulc(kk[1], vfnma(r9, vsub(vadd(xx, xx), vadd(yy, zz)), d1));
        const V B = vmulc(kk[2], vfnma(r9, vsub(yy, zz), d2));
        cxy = vmulc(kk[3], vfnma(r9, flow(gx, gy, px, py), pxy));
        cyz = vmulc(kk[4], vfnma(r9, flow(gy, gz, py, pz), pyz));
        cxz = vmulc(kk[5], vfnma(r9, flow(gx, gz, px, pz), pxz));
        kx = vadd(A, A);
        ky = vsub(B, A);
        kxy = vadd(A, B);
        kxz = vsub(A, B);
        kz = vneg(kxy);
        kyz = vneg(kx);
        if constexpr (COLL == COLL_MRT_SPARSE) {
            // e = 19 tr N; coefficients -30, -11, 8 at rest, axis and edge velocities
            const V tr = vsub(vadd(vadd(m[4], m[5]), m[6]), rho);
            const V E = vmulc(kk[0], vfnma(r9, vadd(vadd(xx, yy), zz), tr));
            k0 = vmulc(R(-30), E);
            kx = vfmac(R(-11), E, kx);
            ky = vfmac(R(-11), E, ky);
            kz = vfmac(R(-11), E, kz);
            kxy = vfmac(R(8), E, kxy);
            kxz = vfmac(R(8), E, kxz);
            kyz = vfmac(R(8), E, kyz);
        }
    }
    if constexpr (SRT && !TAU1) {
        const R om = par<R>(a.omega, a.omegaf);
        r0 = vmulc(om, r0);
        r2 = vmulc(om, r2);
    }
    const V r1 = vadd(r2, r2), h2 = vmulc(R(0.5), r2), n2 = vneg(r2), n1 = vneg(r1);
    const V& h1 = r2;

    {
        // (the product cell by cell: a packed one may be contracted with the sum it enters later)
        const V e0 = vmulc(R(0.5), r0);
        if constexpr (COLL == COLL_MRT_SPARSE) put(std::integral_constant<int, 0>{}, vfma(e0, b, k0));
        else put(std::integral_constant<int, 0>{}, vmul1(e0, b));
    }
    static_for<0, 9>([&](auto pc) {
        constexpr int q = 2 * decltype(pc)::value + 1;
        constexpr bool axis = q < 7;
        // c.a and c.phi (one or two components)
        auto dot = [&](V x, V y, V z) {
            if constexpr (q == 1) return x;
            else if constexpr (q == 3) return y;
            else if constexpr (q == 5) return z;
            else if constexpr (q == 7) return vadd(x, y);
            else if constexpr (q == 9) return vsub(x, y);
            else if constexpr (q == 11) return vadd(x, z);
            else if constexpr (q == 13) return vsub(x, z);
            else if constexpr (q == 15) return vadd(y, z);
            else return vsub(y, z);
        };
        const V ca = dot(ax, ay, az);
        V T = vfma(ca, ca, b);
        if constexpr (!SRT) {
            const V cp = dot(px, py, pz);
            T = vfnma(cp, cp, T);
        }
        const V h = axis ? h1 : h2;
        V e;
        if constexpr (ROWS) {
            V k;
            if constexpr (q == 1) k = kx;
            else if constexpr (q == 3) k = ky;
            else if constexpr (q == 5) k = kz;
            else if constexpr (q == 7) k = vadd(kxy, cxy);
            else if constexpr (q == 9) k = vsub(kxy, cxy);
            else if constexpr (q == 11) k = vadd(kxz, cxz);
            else if constexpr (q == 13) k = vsub(kxz, cxz);
            else if constexpr (q == 15) k = vadd(kyz, cyz);
            else k = vsub(kyz, cyz);
            e = vfma(h, T, k);
        } else {
            e = vmul(h, T);
        }
        put(std::integral_constant<int, q>{}, vfma(axis ? r1 : r2, ca, e));
        put(std::integral_constant<int, q + 1>{}, vfma(axis ? n1 : n2, ca, e));
    });
}

}  // namespace lbm
