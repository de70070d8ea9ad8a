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

// x / 36 and x / 3.  FP32 splits the constant in two: within an ulp of the
// rounded quotient and unbiased (a product with the rounded 1/36 alone would
// add that constant's relative error to the mass at every collision); FP64
// multiplies (its relative error 5e-17 stays below the rounding of the sums).
__device__ __forceinline__ float2 vdivc(float2 x, double c)
{
    const float hi = (float)c, lo = (float)(c - (double)hi);
    return vfma(x, make_float2(hi, hi), vmul(x, make_float2(lo, lo)));
}
__device__ __forceinline__ double vdivc(double x, double c) { return x * c; }

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
// formats: a constant per unit weight more in each output, -omega rho0 under
// BGK (keep f = keep d + keep w rho0), -rho0 under the regularized filter,
// and rho0 T0 on the diagonal of the second moments.
//
// f^eq of Eq. 3 is taken in s_i = 3 c_i . v: with A = 1 - 3/2 v^2,
//   f^eq_i, f^eq_opp = rho w_i (E +- O),  E = A + s^2 / 2,  O = s (A + s^2 / 6),
// with the density folded into A and the two factors once per weight, seven
// operations per opposite pair (nine in c_i . v with a product by rho w_i).
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
    const U Au = C::dup(fma(usq, R(-1.5), R(1)));
    const U three = C::dup(R(3));
    const U Sx = vmul(three, Ux), Sy = vmul(three, Uy), Sz = vmul(three, Uz);   // 3 u
    const V rq = vdivc(r, 1.0 / 36.0);                                          // rho w_i = rq k_i
    V vx, vy, vz, A;   // 3 v^a and A(v^a)
    if constexpr (FORCE == FORCE_EDM) {
        vx = vadd(gx, Ux); vy = vadd(gy, Uy); vz = vadd(gz, Uz);
        A = vfma(vfma(vx, vx, vfma(vy, vy, vmul(vz, vz))), C::dup(R(-1.5)), one);
        vx = vmul(vx, three); vy = vmul(vy, three); vz = vmul(vz, three);
    } else {
        vx = Sx; vy = Sy; vz = Sz;
        A = Au;
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
        const V keep = vsub(one, om);
        const V re = FORCE == FORCE_GUO ? vmul(rq, om) : rq;
        const V ra = vmul(re, A);
        const V h = vmul(re, C::dup(R(0.5))), t = vmul(re, C::dup(R(1.0 / 6.0)));
        V nh, nt, na;    // -keep rq / 2, -keep rq / 6, -keep rq A(u)
        V even0 = ra;    // k_i of it is what f* has at s = 0
        if constexpr (FORCE == FORCE_EDM) {
            const V nk = vmul(vsub(om, one), rq);
            nh = vmul(nk, C::dup(R(0.5)));
            nt = vmul(nk, C::dup(R(1.0 / 6.0)));
            na = vmul(nk, Au);
            even0 = vadd(ra, na);
        } else {
            even0 = vsub(ra, uQ);
        }
        if constexpr (DEV) even0 = vfma(om, C::dup(p.rho0 * R(-1.0 / 36.0)), even0);
        put(0, vfma(even0, C::dup(R(12)), vmul(keep, get(0))));
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
            if (i < 7) { P = vadd(P, P); M = vadd(M, M); }
            put(i, vfma(keep, get(i), vadd(P, M)));
            put(i + 1, vfma(keep, get(i + 1), vsub(P, M)));
        }
    } else {
        // Pi = sum c c f - rho (T0 I + u u) [+ (u F + F u) / 2], times keep / 8:
        // f^neq_i = k_i (c c : Pi - tr(Pi) / 3) keep / 8  (none of it at tau = 1)
        constexpr bool kNeq = REG != COLL_EQ;
        const V nr = vmul(r, C::dup(R(-1)));
        const V k8 = vmul(vsub(one, om), C::dup(R(0.125)));
        const V ra = vmul(rq, A);
        const V h = vmul(rq, C::dup(R(0.5))), t6 = vmul(rq, C::dup(R(1.0 / 6.0)));
        V even0 = ra;   // the part of f* / k_i that all directions share
        if constexpr (FORCE == FORCE_GUO) even0 = vsub(even0, uQ);
        if constexpr (DEV) even0 = vsub(even0, C::dup(p.rho0 * R(1.0 / 36.0)));
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
            even0 = vsub(even0, vdivc(vadd(P[0], vadd(P[1], P[2])), 1.0 / 3.0));
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
                const R eq = R(0.5) * u[a] * (ub * ub + uc * uc), dq = R(1.5) * u[a] * (ub * ub - uc * uc);
                s3[a] = vmul(k8, vfma(nr, C::dup(eq), vdivc(mom.m[6 + a], 1.0 / 3.0)));
                d3[a] = vmul(k8, vfma(nr, C::dup(dq), mom.m[9 + a]));
            }
        }
        put(0, vmul(even0, C::dup(R(12))));
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            V b = even0;
            if constexpr (kNeq) {
                if (i < 7) b = axis[i / 2];
                else b = ((i - 7) % 4) == 0 ? vadd(diag[(i - 7) / 4], P[3 + (i - 7) / 4])
                                            : vsub(diag[(i - 7) / 4], P[3 + (i - 7) / 4]);
            }
            const V s = vdot(i, vx, vy, vz), m = vmul(s, s);
            V e = vfma(m, h, b), o = vmul(s, vfma(m, t6, ra));
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
            if (i < 7) { e = vadd(e, e); o = vadd(o, o); }
            put(i, vadd(e, o));
            put(i + 1, vsub(e, o));
        }
    }
}

}  // namespace lbm
