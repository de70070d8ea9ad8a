// Moments and collision of a cell (Otomo et al., arXiv:1601.01237, Eqs. 1-11),
// written once over the ways the kernels hold the two components:
//
//   PairF32  both components of a cell in one thread, as a packed pair.  The
//            components go through the same polynomials with their own density,
//            velocity and relaxation rate, so every operation of the pair is
//            one packed instruction (FFMA2 and its kin issue two FP32
//            operations each), and the pairs are the units in which the
//            populations are stored.  The packed form freed the registers that
//            the scalar one spilled (up to 120 bytes a thread in the
//            third-order FP32 instances of the fused step, now 0).
//   LaneF64  one component per lane; lanes l and l ^ 1 hold the two components
//            of a cell and exchange what couples them by shuffles.  FP64 retires
//            one warp instruction per 64 cycles on each of an SM's four
//            schedulers, so its instances are bound by the FP64 instructions of
//            the busiest scheduler, and half a cell per lane spreads a lattice
//            over twice as many of them.
//
// V is what a lane holds of a quantity that both components have, U what it
// holds of a mixture quantity (in PairF32 a pair of equal halves, which costs
// the same issue slots as a scalar and no packing moves).
#pragma once

#include "d3q19.cuh"

namespace lbm {

__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 p, q;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tsub.rn.f32x2 p, p, q;\n\t"
        "mov.b64 {%0, %1}, p;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }

struct PairF32 {
    using R = float;
    using V = float2;
    using U = float2;
    __device__ __forceinline__ static V dup(R a) { return make_float2(a, a); }
    __device__ __forceinline__ V of(R a, R b) const { return make_float2(a, b); }     // (component 1, component 2)
    __device__ __forceinline__ R both(V a) const { return a.x + a.y; }                // sum over the components
};
struct LaneF64 {
    using R = double;
    using V = double;
    using U = double;
    int a;   // component of this lane
    __device__ __forceinline__ static V dup(R x) { return x; }
    __device__ __forceinline__ V of(R x, R y) const { return a ? y : x; }
    __device__ __forceinline__ R both(V x) const { return x + __shfl_xor_sync(0xffffffffu, x, 1); }
};
__device__ __forceinline__ float2 vswap(float2 a) { return make_float2(a.y, a.x); }

// c_i . (x, y, z) for i odd (the opposite direction has the negative)
template <class T>
__device__ __forceinline__ T vdot(int i, T x, T y, T z)
{
    T r = x;
    bool first = true;
    auto term = [&](int c, T t) {
        if (c == 0) return;
        if (first) r = t;              // the first non-zero component of an odd direction is +1
        else r = c > 0 ? vadd(r, t) : vsub(r, t);
        first = false;
    };
    term(cx(i), x);
    term(cy(i), y);
    term(cz(i), z);
    return r;
}
__host__ __device__ constexpr bool odd_dirs_lead_positive()
{
    for (int i = 1; i < Q; i += 2) {
        const int l = cx(i) ? cx(i) : (cy(i) ? cy(i) : cz(i));
        if (l != 1) return false;
    }
    return true;
}
static_assert(odd_dirs_lead_positive(), "vdot takes the leading component of odd directions as +1");

// x / N (N = 3, 36) with 1 / N in two parts: within an ulp of the quotient and
// unbiased.  (A product with the rounded reciprocal alone carries that constant's
// relative error, in FP64 5.55e-17 low, into every collision with the same sign.)
template <int N>
__device__ __forceinline__ float2 vdivc(float2 x)
{
    constexpr float hi = (float)(1.0 / N), lo = (float)(1.0 / N - (double)hi);
    return vfma(x, make_float2(hi, hi), vmul(x, make_float2(lo, lo)));
}
template <int N>
__device__ __forceinline__ double vdivc(double x)
{
    // lo = (1 - N hi) / N; the products of N with the two halves of hi are exact
    constexpr double hi = 1.0 / N, up = (double)(float)hi, lo = ((1.0 - N * up) - N * (hi - up)) / N;
    return fma(x, hi, x * lo);
}

// Collision kinds of the kernels: the three operators, and EQ for tau = 1 in
// both components, where 1 - 1/tau = 0: all three operators then give
// f* = f^eq (with the forcing term) whatever the populations' non-equilibrium
// part, so that a cell's densities and momentum are all that its collision
// needs of them.
enum CollisionKind { COLL_BGK = 0, COLL_REG = 1, COLL_REG3 = 2, COLL_EQ = 3 };

// What the regularized operators keep of a cell's populations: the second
// moments sum_i c c f (xx, yy, zz, xy, xz, yz) and, for the third-order filter,
// the sums of h3s3 f and h3d f (struct Third).
template <class C, int REG>
struct RegMoments {
    using V = typename C::V;
    using R = typename C::R;
    static constexpr int n = REG == COLL_REG ? 6 : (REG == COLL_REG3 ? 12 : 0);
    V m[n > 0 ? n : 1];

    __device__ __forceinline__ void of(const V (&f)[Q])
    {
        if constexpr (n > 0) {
            // opposite directions carry the same products and opposite odd moments
            V e[Q / 2 + 1];
#pragma unroll
            for (int i = 1; i < Q; i += 2) e[i / 2] = vadd(f[i], f[i + 1]);
            // directions (odd members): 1 x, 3 y, 5 z, 7 9 xy, 11 13 xz, 15 17 yz
            const V xy = vadd(e[3], e[4]), xz = vadd(e[5], e[6]), yz = vadd(e[7], e[8]);
            m[0] = vadd(e[0], vadd(xy, xz));
            m[1] = vadd(e[1], vadd(xy, yz));
            m[2] = vadd(e[2], vadd(xz, yz));
            m[3] = vsub(e[3], e[4]);
            m[4] = vsub(e[5], e[6]);
            m[5] = vsub(e[7], e[8]);
        }
        if constexpr (REG == COLL_REG3) {
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                V s = C::dup(R(0));
                bool first = true;
#pragma unroll
                for (int i = 1; i < Q; i += 2) {
                    const int h = k < 3 ? h3s3(i, k) : h3d(i, k - 3);
                    if (h == 0) continue;
                    const V d = vsub(f[i], f[i + 1]);
                    if (first) s = h == 1 ? d : vmul(d, C::dup(R(h)));
                    else s = h == 1 ? vadd(s, d) : (h == -1 ? vsub(s, d) : vfma(d, C::dup(R(h)), s));
                    first = false;
                }
                m[6 + k] = s;
            }
        }
    }
};
static_assert(cx(7) * cy(7) == 1 && cx(9) * cy(9) == -1 && cx(11) * cz(11) == 1 && cx(13) * cz(13) == -1 &&
                  cy(15) * cz(15) == 1 && cy(17) * cz(17) == -1,
              "signs of the off-diagonal second moments");

// Density of a gathered population set, in the grouping of the fused step's
// halo partials, (directions 0-6 + 7-12) + 13-18.
template <class V>
__device__ __forceinline__ V density(const V (&f)[Q])
{
    V g0 = f[0], g1 = f[7], g2 = f[13];
#pragma unroll
    for (int i = 1; i < 7; ++i) g0 = vadd(g0, f[i]);
#pragma unroll
    for (int i = 8; i < 13; ++i) g1 = vadd(g1, f[i]);
#pragma unroll
    for (int i = 14; i < Q; ++i) g2 = vadd(g2, f[i]);
    return vadd(vadd(g0, g1), g2);
}

// Mixture momentum over opposite pairs, sum_{i odd} c_i (t_i - t_opp(i)): each
// difference of two nearly equal populations is taken first (exactly, in FP32,
// when they are within a factor of two), so that the rounding scales with the
// momentum and not with the density.
template <class C>
__device__ __forceinline__ void momentum(const C &c, const typename C::V (&f)[Q], typename C::R &jx, typename C::R &jy,
                                         typename C::R &jz)
{
    using V = typename C::V;
    V a[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) a[d] = vsub(f[1 + 2 * d], f[2 + 2 * d]);
#pragma unroll
    for (int i = 7; i < Q; i += 2) {
        const V t = vsub(f[i], f[i + 1]);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (ca(i, d) == 1) a[d] = vadd(a[d], t);
            else if (ca(i, d) == -1) a[d] = vsub(a[d], t);
        }
    }
    jx = c.both(a[0]);
    jy = c.both(a[1]);
    jz = c.both(a[2]);
}

// Interaction sums S^b = sum_i w_i c_i rho^b(x + c_i) (Eq. 7) from the
// differences rho(x + c_i) - rho(x - c_i) of opposite neighbours (i odd, given
// by diff(i)): the differences of nearby densities come first, so that the
// rounding scales with the gradient and not with the density.
template <class C, class D>
__device__ __forceinline__ void interaction(D diff, typename C::V (&S)[3])
{
    using V = typename C::V;
    using R = typename C::R;
    V g[3];
    bool first[3] = {true, true, true};
#pragma unroll
    for (int i = 7; i < Q; i += 2) {
        const V t = diff(i);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (ca(i, d) == 0) continue;
            if (first[d]) g[d] = t;   // (its sign is +1, checked below)
            else g[d] = ca(i, d) > 0 ? vadd(g[d], t) : vsub(g[d], t);
            first[d] = false;
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
        S[d] = vfma(diff(1 + 2 * d), C::dup(w<R>(1)), vmul(g[d], C::dup(w<R>(7))));
}
static_assert(cx(7) == 1 && cy(7) == 1 && cz(11) == 1, "first diagonal of each axis is positive");

// Collision with forcing (Eq. 1 with Eq. 2, or Eq. 10; the two readings of the
// forcing term, see collide() in d3q19.cuh).
//   r     rho^a;  inv = 1 / (rho^1 + rho^2);  u = mixture velocity j / rho
//   So    interaction sums of the other component
//   mom   raw moments of the populations (REG and REG3)
//   get   get(i): the pre-collision population of direction i (BGK only)
//   put   put(i, o): receives the post-collision population of direction i
// DEV: populations in and out are deviations d = f - w_i rho0 of the deviation
// formats (and rho0 T0 less on the diagonal of the second moments).
//
// f^eq of Eq. 3 is taken in s_i = 3 c_i . v: with B = -3/2 v^2 and A = 1 + B,
//   f^eq_i, f^eq_opp = rho w_i (1 + E +- O),  E = B + s^2 / 2,  O = s (A + s^2 / 6).
// With q = rho / 36 the parts q k E and q k O are small and q k is added last, so
// that roundings of a population's size are made once per opposite pair and once per
// direction (tau = 1 in FP32: once per direction); q, which all directions share, takes
// its rounding out of the mass again by the rest direction, which has rho - 24 q in the
// place of 12 q.  One collision's rms error in units of 2^-24 rho (2^-53 in FP64), BGK
// with tau != 1 / regularized / tau = 1: mass 0.24 / 0.23 / 0.22, momentum 0.08 / 0.08 /
// 0.06, pressure 0.22 / 0.20 / 0.15; with each direction's polynomial formed at scale 1
// and multiplied by rho w_i 0.63 / 0.55 / 0.55, 0.11 / 0.08 / 0.08, 0.24 / 0.25 / 0.21;
// with q A rounded once for all directions 0.90 / 0.83 / 0.68, 0.09 / 0.08 / 0.08, 0.31 /
// 0.33 / 0.23, and in FP64 with q = rho times the rounded 1/36 a mean of -0.50 per step.
// Parameter derivatives of 50 steps at 96^3 (six droplets, largest error over largest
// value): with the last of these 6.5e-8 / 8.2e-8 / 7.6e-8 / 3.3e-8, here 2.0e-8 / 2.2e-8 /
// 2.2e-8 / 3.1e-8.  us per step, that form and this one in the same kernels: runs in
// moment space 512^3 3052 / 3044, 256^3 393 / 402, regularized 617 / 631, FP64 1 x 64 x 64
// 8.8 / 9.1.
template <class C, int REG, int FORCE, bool DEV, class GET, class PUT>
__device__ __forceinline__ void collide_cell(const C &c, const Phys<typename C::R> &p, typename C::V r,
                                             typename C::R inv, typename C::R ux, typename C::R uy, typename C::R uz,
                                             const typename C::V (&So)[3], const RegMoments<C, REG> &mom, GET get,
                                             PUT put)
{
    using R = typename C::R;
    using V = typename C::V;
    using U = typename C::U;
    const V one = C::dup(R(1));
    const V om = c.of(p.omega[0], p.omega[1]);
    const V G = c.of(p.G12, p.G21);
    // accelerations g^a = G^{ab} S^b + g_ext
    const V gx = vfma(G, So[0], C::dup(p.gext[0]));
    const V gy = vfma(G, So[1], C::dup(p.gext[1]));
    const V gz = vfma(G, So[2], C::dup(p.gext[2]));
    V Fx, Fy, Fz;   // Guo: F^a = rho^a g^a, both components relax toward u* = u + (F^1 + F^2) / (2 rho)
    if constexpr (FORCE == FORCE_GUO) {
        Fx = vmul(r, gx); Fy = vmul(r, gy); Fz = vmul(r, gz);
        const R hi = R(0.5) * inv;
        ux += c.both(Fx) * hi;
        uy += c.both(Fy) * hi;
        uz += c.both(Fz) * hi;
    }
    const R usq = ux * ux + uy * uy + uz * uz;
    const U Ux = C::dup(ux), Uy = C::dup(uy), Uz = C::dup(uz);
    const U Bu = C::dup(usq * R(-1.5)), Au = C::dup(fma(usq, R(-1.5), R(1)));
    const U three = C::dup(R(3));
    const U Sx = vmul(three, Ux), Sy = vmul(three, Uy), Sz = vmul(three, Uz);   // 3 u
    const V rq = vdivc<36>(r);   // rho w_i = rq k_i
    V rd = r, dq = rq;           // less rho0 in the deviation formats
    if constexpr (DEV) {
        rd = vsub(r, C::dup(p.rho0));
        dq = vdivc<36>(rd);
    }
    V vx, vy, vz, A, B;   // 3 v^a, A(v^a) and B(v^a)
    if constexpr (FORCE == FORCE_EDM) {
        vx = vadd(gx, Ux); vy = vadd(gy, Uy); vz = vadd(gz, Uz);
        const V sq = vfma(vx, vx, vfma(vy, vy, vmul(vz, vz)));
        B = vmul(sq, C::dup(R(-1.5)));
        A = vfma(sq, C::dup(R(-1.5)), one);
        vx = vmul(vx, three); vy = vmul(vy, three); vz = vmul(vz, three);
    } else {
        vx = Sx; vy = Sy; vz = Sz;
        A = Au;
        B = Bu;
    }
    // Guo's forcing term k_i ((c.u*)(c.Q) 3 - u*.Q +- c.Q), Q = (3 cf / 36) F,
    // cf = 1 - 1/(2 tau) (BGK) or 1/2
    V Qx, Qy, Qz, uQ;
    if constexpr (FORCE == FORCE_GUO) {
        const V cq = REG != COLL_BGK ? C::dup(R(1.0 / 24.0)) : vmul(vfma(om, C::dup(R(-0.5)), one), C::dup(R(1.0 / 12.0)));
        Qx = vmul(Fx, cq); Qy = vmul(Fy, cq); Qz = vmul(Fz, cq);
        uQ = vfma(Qx, Ux, vfma(Qy, Uy, vmul(Qz, Uz)));
    }
    if constexpr (REG == COLL_BGK) {
        // f* = f^eq(v) - keep f^eq(u) + keep f; with Guo's forcing v = u and
        // f^eq(v) - keep f^eq(u) = omega f^eq(u)
        const V keep = vsub(one, om), oc = vsub(one, keep);   // oc: exactly what keep leaves (1 - omega rounds below 1/2)
        const V re = FORCE == FORCE_GUO ? vmul(rq, oc) : rq;
        const V ra = vmul(re, A);
        const V h = vmul(re, C::dup(R(0.5))), t = vmul(re, C::dup(R(1.0 / 6.0)));
        V nh, nt, na;             // -keep rq / 2, -keep rq / 6, -keep rq A(u)
        V even0 = vmul(re, B);    // E at s = 0
        if constexpr (FORCE == FORCE_EDM) {
            const V nk = vmul(vmul(keep, C::dup(R(-1))), rq);
            nh = vmul(nk, C::dup(R(0.5)));
            nt = vmul(nk, C::dup(R(1.0 / 6.0)));
            na = vmul(nk, Au);
            even0 = vfma(nk, Bu, even0);
        } else {
            even0 = vsub(even0, uQ);
        }
        // omega rho - 36 q: 32 q is exact, and what is left after it a ninth of the size
        const V q = vmul(oc, dq), q2 = vadd(q, q);
        const V left = vfma(q, C::dup(R(-4)), vfma(oc, rd, vmul(q, C::dup(R(-32)))));
        put(0, vfma(even0, C::dup(R(12)), vfma(q, C::dup(R(12)), vfma(keep, get(0), left))));
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            const V s = vdot(i, vx, vy, vz), m = vmul(s, s);
            V P = vfma(m, h, even0), M = vmul(s, vfma(m, t, ra));
            if constexpr (FORCE == FORCE_EDM) {
                const U su = vdot(i, Sx, Sy, Sz), mu = vmul(su, su);
                P = vfma(nh, mu, P);
                M = vfma(vfma(nt, mu, na), su, M);
            } else {
                const V cQ = vdot(i, Qx, Qy, Qz);
                P = vfma(cQ, s, P);
                M = vadd(M, cQ);
            }
            // (keep f + k q has the size of a population, so that two roundings of that size are made)
            const V a = vfma(keep, get(i), i < 7 ? q2 : q), b = vfma(keep, get(i + 1), i < 7 ? q2 : q);
            const V x = vadd(P, M), y = vsub(P, M);
            put(i, i < 7 ? vfma(x, C::dup(R(2)), a) : vadd(a, x));
            put(i + 1, i < 7 ? vfma(y, C::dup(R(2)), b) : vadd(b, y));
        }
    } else {
        // Pi = sum c c f - rho (T0 I + u u) [+ (u F + F u) / 2], times keep / 8:
        // f^neq_i = k_i (c c : Pi - tr(Pi) / 3) keep / 8  (none of it at tau = 1)
        constexpr bool kNeq = REG != COLL_EQ;
        const V nr = vmul(r, C::dup(R(-1)));
        const V k8 = vmul(vsub(one, om), C::dup(R(0.125)));
        const V ra = vmul(rq, A);
        const V h = vmul(rq, C::dup(R(0.5))), t6 = vmul(rq, C::dup(R(1.0 / 6.0)));
        V even0 = vmul(rq, B);   // E at s = 0
        if constexpr (FORCE == FORCE_GUO) even0 = vsub(even0, uQ);
        V P[6], axis[3], diag[3];   // even0 + f^neq / k_i of the axes and, but for the P_ab term, of the diagonals
        if constexpr (kNeq) {
            const R T0 = R(1) / R(3);
            auto dia = [&](int k, R u, V F) {
                V m = mom.m[k];
                if constexpr (DEV) m = vadd(m, C::dup(p.rho0 * T0));
                m = vfma(nr, C::dup(T0 + u * u), m);
                if constexpr (FORCE == FORCE_GUO) m = vfma(F, C::dup(u), m);
                return vmul(k8, m);
            };
            auto off = [&](int k, R ua, R ub, V Fa, V Fb) {
                V m = vfma(nr, C::dup(ua * ub), mom.m[k]);
                if constexpr (FORCE == FORCE_GUO)
                    m = vfma(Fb, C::dup(R(0.5) * ua), vfma(Fa, C::dup(R(0.5) * ub), m));
                m = vmul(k8, m);
                return vadd(m, m);
            };
            P[0] = dia(0, ux, Fx);
            P[1] = dia(1, uy, Fy);
            P[2] = dia(2, uz, Fz);
            P[3] = off(3, ux, uy, Fx, Fy);
            P[4] = off(4, ux, uz, Fx, Fz);
            P[5] = off(5, uy, uz, Fy, Fz);
            even0 = vsub(even0, vdivc<3>(vadd(P[0], vadd(P[1], P[2]))));
            axis[0] = vadd(even0, P[0]);
            axis[1] = vadd(even0, P[1]);
            axis[2] = vadd(even0, P[2]);
            diag[0] = vadd(axis[0], P[1]);   // xy
            diag[1] = vadd(axis[0], P[2]);   // xz
            diag[2] = vadd(axis[1], P[2]);   // yz
        }
        V s3[3], d3[3];
        if constexpr (REG == COLL_REG3) {
            const R u[3] = {ux, uy, uz};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const R ub = u[a == 0 ? 1 : 0], uc = u[a == 2 ? 1 : 2];
                const R hs = R(0.5) * u[a] * (ub * ub + uc * uc), hd = R(1.5) * u[a] * (ub * ub - uc * uc);
                s3[a] = vmul(k8, vfma(nr, C::dup(hs), vdivc<3>(mom.m[6 + a])));
                d3[a] = vmul(k8, vfma(nr, C::dup(hd), mom.m[9 + a]));
            }
        }
        constexpr bool kPlain = !kNeq && FORCE == FORCE_EDM;   // f^eq(v) alone
        const V q2 = vadd(dq, dq), rq2 = vadd(rq, rq);
        // rho - 24 q is rounded before E joins it: half of its values are ties, which an E
        // that is never positive at tau = 1 would all turn down
        put(0, vfma(even0, C::dup(R(12)), vfma(dq, C::dup(R(-24)), rd)));
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            V b = even0;
            if constexpr (kNeq) {
                if (i < 7) b = axis[i / 2];
                else b = ((i - 7) % 4) == 0 ? vadd(diag[(i - 7) / 4], P[3 + (i - 7) / 4])
                                            : vsub(diag[(i - 7) / 4], P[3 + (i - 7) / 4]);
            }
            const V s = vdot(i, vx, vy, vz), m = vmul(s, s);
            if constexpr (kPlain && sizeof(R) == 4) {
                // (q outside the polynomials: constants in the place of the pairs h, t6 and ra, for
                // which the moment step's tiles of 16 rows have no registers: 512^3 3044 us per step,
                // with them 3954)
                const V x = vfma(m, C::dup(R(0.5)), B), y = vmul(s, vfma(m, C::dup(R(1.0 / 6.0)), A));
                put(i, vfma(i < 7 ? rq2 : rq, vadd(x, y), i < 7 ? q2 : dq));
                put(i + 1, vfma(i < 7 ? rq2 : rq, vsub(x, y), i < 7 ? q2 : dq));
                continue;
            }
            V e = vfma(m, h, b);
            if constexpr (sizeof(R) == 8 && FORCE == FORCE_EDM && REG != COLL_REG3) {
                // (an operation less; a negated factor costs the packed form one)
                const V O = vfma(m, t6, ra), t = i < 7 ? vadd(s, s) : s;
                e = i < 7 ? vfma(e, C::dup(R(2)), q2) : vadd(e, dq);
                put(i, vfma(t, O, e));
                put(i + 1, vfma(-t, O, e));
                continue;
            }
            V o = vmul(s, vfma(m, t6, ra));
            if constexpr (FORCE == FORCE_GUO) {
                const V cQ = vdot(i, Qx, Qy, Qz);
                e = vfma(cQ, s, e);
                o = vadd(o, cQ);
            }
            if constexpr (REG == COLL_REG3) {
                V t = o;
                auto term = [&](int hh, V v) {
                    if (hh) t = hh == 1 ? vadd(t, v) : (hh == -1 ? vsub(t, v) : vfma(v, C::dup(R(hh)), t));
                };
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    term(h3s3(i, a), s3[a]);
                    term(h3d(i, a), d3[a]);
                }
                o = t;
            }
            if (i < 7) {   // k_i = 2
                e = vfma(e, C::dup(R(2)), q2);
                put(i, vfma(o, C::dup(R(2)), e));
                put(i + 1, vfma(o, C::dup(R(-2)), e));
            } else {
                e = vadd(e, dq);
                put(i, vadd(e, o));
                put(i + 1, vsub(e, o));
            }
        }
    }
}

}  // namespace lbm
