// Moments and collision of both components of one cell (Otomo et al.,
// arXiv:1601.01237, Eqs. 1-11), written on pairs (component 1, component 2).
//
// The two components go through the same polynomials with their own density,
// velocity and relaxation rate, so in FP32 every operation of the pair is one
// packed instruction (FFMA2 and its kin issue two FP32 operations each), and
// the pairs are the units in which the populations are stored.  In FP64 a pair
// operation is two scalar ones; what depends on the mixture velocity alone is
// shared by the components there (type U: one double; in FP32 a pair of equal
// halves, which costs the same issue slots as a scalar and no packing moves).
// The packed form freed the registers that the scalar one spilled (up to 120
// bytes a thread in the third-order FP32 instances of the fused step, now 0).
#pragma once

#include "d3q19.cuh"

namespace lbm {

template <class R> struct PairOf;
template <> struct PairOf<float> { using V = float2; using U = float2; };
template <> struct PairOf<double> { using V = double2; using U = double; };

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
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
// a pair and a shared factor
__device__ __forceinline__ double2 vmul(double2 a, double b) { return make_double2(a.x * b, a.y * b); }
__device__ __forceinline__ double2 vfma(double2 a, double b, double2 c)
{
    return make_double2(fma(a.x, b, c.x), fma(a.y, b, c.y));
}
__device__ __forceinline__ double2 vadd(double2 a, double b) { return make_double2(a.x + b, a.y + b); }
template <class R> __device__ __forceinline__ typename PairOf<R>::V vpair(R a, R b);
template <> __device__ __forceinline__ float2 vpair<float>(float a, float b) { return make_float2(a, b); }
template <> __device__ __forceinline__ double2 vpair<double>(double a, double b) { return make_double2(a, b); }
template <class R> __device__ __forceinline__ typename PairOf<R>::V vdup(R a) { return vpair<R>(a, a); }
template <class R> __device__ __forceinline__ typename PairOf<R>::U udup(R a);
template <> __device__ __forceinline__ float2 udup<float>(float a) { return make_float2(a, a); }
template <> __device__ __forceinline__ double udup<double>(double a) { return a; }
template <class V> __device__ __forceinline__ V vswap(V a) { V r; r.x = a.y; r.y = a.x; return r; }

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

// x / 36 and x / 3 with the constant split in two: within an ulp of the
// rounded quotient and unbiased (a product with the rounded 1/36 alone would
// add that constant's relative error to the mass at every collision).
template <class V, class R>
__device__ __forceinline__ V vdiv_const(V x, R hi, R lo) { return vfma(x, vdup<R>(hi), vmul(x, vdup<R>(lo))); }
template <class R>
struct Recip {
    static constexpr R hi36 = (R)(1.0 / 36.0), lo36 = (R)(1.0 / 36.0 - (double)(R)(1.0 / 36.0));
    static constexpr R hi3 = (R)(1.0 / 3.0), lo3 = (R)(1.0 / 3.0 - (double)(R)(1.0 / 3.0));
};
template <class R>
__device__ __forceinline__ typename PairOf<R>::V vdiv36(typename PairOf<R>::V x)
{
    if constexpr (sizeof(R) == 8) return vmul(x, vdup<R>(R(1.0 / 36.0)));
    else return vdiv_const(x, Recip<R>::hi36, Recip<R>::lo36);
}
template <class R>
__device__ __forceinline__ typename PairOf<R>::V vdiv3(typename PairOf<R>::V x)
{
    if constexpr (sizeof(R) == 8) return vmul(x, vdup<R>(R(1.0 / 3.0)));
    else return vdiv_const(x, Recip<R>::hi3, Recip<R>::lo3);
}

// Collision kinds of the kernels: the three operators, and EQ for tau = 1 in
// both components, where 1 - 1/tau = 0: all three operators then give
// f* = f^eq (with the forcing term) whatever the populations' non-equilibrium
// part, so that a cell's densities and momentum are all that its collision
// needs of them.
enum CollisionKind { COLL_BGK = 0, COLL_REG = 1, COLL_REG3 = 2, COLL_EQ = 3 };

// What the regularized operators keep of a cell's populations: the second
// moments sum_i c c f (xx, yy, zz, xy, xz, yz) and, for the third-order filter,
// the sums of h3s3 f and h3d f (struct Third), as pairs.
template <class R, int REG>
struct RegMoments {
    using V = typename PairOf<R>::V;
    static constexpr int n = REG == COLL_REG ? 6 : (REG == COLL_REG3 ? 12 : 0);
    V m[n > 0 ? n : 1];

    __device__ __forceinline__ void of(const V (&f)[Q])
    {
        if (n == 0) return;
        // opposite directions carry the same products and opposite odd moments
        V e[Q / 2 + 1];
#pragma unroll
        for (int i = 1; i < Q; i += 2) e[i / 2] = vadd(f[i], f[i + 1]);
        // directions (odd members): 1 x, 3 y, 5 z, 7 9 xy, 11 13 xz, 15 17 yz
        const V xy = vadd(e[3], e[4]), xz = vadd(e[5], e[6]), yz = vadd(e[7], e[8]);
        if constexpr (n > 0) {
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
                V s = vdup<R>(R(0));
                bool first = true;
#pragma unroll
                for (int i = 1; i < Q; i += 2) {
                    const int h = k < 3 ? h3s3(i, k) : h3d(i, k - 3);
                    if (h == 0) continue;
                    const V d = vsub(f[i], f[i + 1]);
                    if (first) s = vmul(d, vdup<R>(R(h)));
                    else s = h == 1 ? vadd(s, d) : (h == -1 ? vsub(s, d) : vfma(d, vdup<R>(R(h)), s));
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

// Densities of a gathered population set, summed in the grouping of the fused
// step's halo partials, (directions 0-6 + 7-12) + 13-18, and the mixture
// momentum over opposite pairs, sum_{i odd} c_i (t_i - t_opp(i)), t = f^1 + f^2:
// each difference of two nearly equal populations is taken first (exactly, in
// FP32, when they are within a factor of two), so that the rounding scales
// with the momentum and not with the density.
template <class R>
__device__ __forceinline__ void sums2(const typename PairOf<R>::V (&f)[Q], typename PairOf<R>::V &rho, R &jx, R &jy, R &jz)
{
    using V = typename PairOf<R>::V;
    V g0 = f[0], g1 = f[7], g2 = f[13];
#pragma unroll
    for (int i = 1; i < 7; ++i) g0 = vadd(g0, f[i]);
#pragma unroll
    for (int i = 8; i < 13; ++i) g1 = vadd(g1, f[i]);
#pragma unroll
    for (int i = 14; i < Q; ++i) g2 = vadd(g2, f[i]);
    rho = vadd(vadd(g0, g1), g2);
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
    jx = a[0].x + a[0].y;
    jy = a[1].x + a[1].y;
    jz = a[2].x + a[2].y;
}

// Interaction sums S^b = sum_i w_i c_i rho^b(x + c_i) (Eq. 7) from the
// differences d_i = rho(x + c_i) - rho(x - c_i) of opposite neighbours (i odd,
// given by diff(i)): the differences of nearby densities come first, so that
// the rounding scales with the gradient and not with the density.
template <class R, class D>
__device__ __forceinline__ void interaction2(D diff, typename PairOf<R>::V (&S)[3])
{
    using V = typename PairOf<R>::V;
    V g[3];
    bool first[3] = {true, true, true};
#pragma unroll
    for (int i = 7; i < Q; i += 2) {
        const V t = diff(i);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (ca(i, d) == 0) continue;
            if (first[d]) g[d] = t;   // (+1: the leading component, checked for z below)
            else g[d] = ca(i, d) > 0 ? vadd(g[d], t) : vsub(g[d], t);
            first[d] = false;
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
        S[d] = vfma(diff(1 + 2 * d), vdup<R>(w<R>(1)), vmul(g[d], vdup<R>(w<R>(7))));
}
static_assert(cx(7) == 1 && cy(7) == 1 && cz(11) == 1, "first diagonal of each axis is positive");

// Collision with forcing of both components (Eq. 1 with Eq. 2, or Eq. 10; the
// two readings of the forcing term, see collide() in d3q19.cuh).
//   r     (rho^1, rho^2);  inv = 1 / (rho^1 + rho^2);  u = mixture velocity j / rho
//   S     interaction sums
//   mom   raw moments of the populations (REG > 0)
//   get   get(i): the pre-collision pair of direction i (BGK only)
//   put   put(i, o): receives the post-collision pair of direction i
// DEV: populations in and out are deviations d = f - w_i rho0 of the deviation
// formats: a constant per unit weight more in each output, -omega rho0 under
// BGK (keep f = keep d + keep w rho0), -rho0 under the regularized filter,
// and rho0 T0 on the diagonal of the second moments.
template <class R, int REG, int FORCE, bool DEV, class GET, class PUT>
__device__ __forceinline__ void collide2(const Phys<R> &p, typename PairOf<R>::V r, R inv, R ux, R uy, R uz,
                                         const typename PairOf<R>::V (&S)[3], const RegMoments<R, REG> &mom, GET get,
                                         PUT put)
{
    using V = typename PairOf<R>::V;
    using U = typename PairOf<R>::U;
    const V one = vdup<R>(R(1));
    const V om = vpair<R>(p.omega[0], p.omega[1]);
    const V keep = vsub(one, om);
    const V G = vpair<R>(p.G12, p.G21);
    // accelerations g^a = G^{ab} S^b + g_ext
    V gx = vfma(G, vswap(S[0]), vdup<R>(p.gext[0]));
    V gy = vfma(G, vswap(S[1]), vdup<R>(p.gext[1]));
    V gz = vfma(G, vswap(S[2]), vdup<R>(p.gext[2]));
    V Fx = gx, Fy = gy, Fz = gz;   // Guo: rho^a g^a
    if constexpr (FORCE == FORCE_GUO) {
        Fx = vmul(r, gx); Fy = vmul(r, gy); Fz = vmul(r, gz);
        const R hi = R(0.5) * inv;
        ux += (Fx.x + Fx.y) * hi;
        uy += (Fy.x + Fy.y) * hi;
        uz += (Fz.x + Fz.y) * hi;
    }
    const R usq = ux * ux + uy * uy + uz * uz;
    const U Ux = udup<R>(ux), Uy = udup<R>(uy), Uz = udup<R>(uz);
    const U Au = udup<R>(R(1) - R(1.5) * usq), Bu = udup<R>(R(3) - R(4.5) * usq);
    const V rq = vdiv36<R>(r), rq2 = vadd(rq, rq);   // rho w_i = (rho / 36) k_i
    const V c45 = vdup<R>(R(4.5));
    const U u45 = udup<R>(R(4.5));
    V vx, vy, vz, A, B;
    if constexpr (FORCE == FORCE_EDM) {
        vx = vadd(gx, Ux); vy = vadd(gy, Uy); vz = vadd(gz, Uz);
        const V vsq = vfma(vx, vx, vfma(vy, vy, vmul(vz, vz)));
        A = vfma(vsq, vdup<R>(R(-1.5)), one);
        B = vfma(vsq, vdup<R>(R(-4.5)), vdup<R>(R(3)));
    }
    // Guo's forcing term, scaled: cq = 3 cf / 36, cf = 1 - 1/(2 tau) (BGK) or 1/2
    V Qx, Qy, Qz, uQ;
    if constexpr (FORCE == FORCE_GUO) {
        const V cq = REG != COLL_BGK ? vdup<R>(R(1) / R(24)) : vmul(vfma(om, vdup<R>(R(-0.5)), one), vdup<R>(R(1) / R(12)));
        Qx = vmul(Fx, cq); Qy = vmul(Fy, cq); Qz = vmul(Fz, cq);
        uQ = vfma(Qx, Ux, vfma(Qy, Uy, vmul(Qz, Uz)));
    }
    if constexpr (REG == COLL_BGK) {
        const V nk = vsub(om, one);
        // constant per unit k of the deviation formats
        const V dc = vmul(om, vdup<R>(DEV ? p.rho0 * R(-1.0 / 36.0) : R(0)));
        {
            V o;
            if constexpr (FORCE == FORCE_EDM) o = vmul(rq, vfma(nk, Au, A));
            else o = vsub(vmul(vmul(rq, om), Au), uQ);
            if constexpr (DEV) o = vadd(o, dc);
            put(0, vfma(o, vdup<R>(R(12)), vmul(keep, get(0))));
        }
        V rwo, rwo2;
        if constexpr (FORCE == FORCE_GUO) { rwo = vmul(rq, om); rwo2 = vadd(rwo, rwo); }
        const V dc2 = vadd(dc, dc);
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            const bool axis = i < 7;
            const U cu = vdot(i, Ux, Uy, Uz), hu = vmul(cu, u45);
            const U Eu = vfma(hu, cu, Au), Ou = vmul(cu, vfma(hu, cu, Bu));
            V P, M;   // even and odd part of f^eq(v) - keep f^eq(u), forcing included
            if constexpr (FORCE == FORCE_EDM) {
                const V c = vdot(i, vx, vy, vz), h = vmul(c, c45);
                const V E = vfma(nk, Eu, vfma(h, c, A)), O = vfma(nk, Ou, vmul(c, vfma(h, c, B)));
                const V rw = axis ? rq2 : rq;
                P = DEV ? vfma(rw, E, axis ? dc2 : dc) : vmul(rw, E);
                M = vmul(rw, O);
            } else {
                const V rw = axis ? rwo2 : rwo;
                V cQ = vdot(i, Qx, Qy, Qz), uq = uQ;
                if (axis) { cQ = vadd(cQ, cQ); uq = vadd(uq, uq); }
                const V e = vsub(vmul(cQ, vmul(cu, udup<R>(R(3)))), uq);
                P = vfma(rw, Eu, e);
                if constexpr (DEV) P = vadd(P, axis ? dc2 : dc);
                M = vfma(rw, Ou, cQ);
            }
            put(i, vfma(keep, get(i), vadd(P, M)));
            put(i + 1, vfma(keep, get(i + 1), vsub(P, M)));
        }
    } else {
        // Pi = sum c c f - rho (T0 I + u u) [+ (u F + F u) / 2], times keep / 8:
        // f^neq_i = k_i (c c : Pi - tr(Pi) / 3) keep / 8  (none of it at tau = 1)
        constexpr bool kNeq = REG != COLL_EQ;
        const V nr = vmul(r, vdup<R>(R(-1)));
        const V k8 = vmul(keep, vdup<R>(R(0.125)));
        V P[6], t = vdup<R>(R(0));
        if constexpr (kNeq) {
            const R T0 = R(1) / R(3);
            auto diag = [&](int k, R u, V F) {
                V m = mom.m[k];
                if constexpr (DEV) m = vadd(m, vdup<R>(p.rho0 * T0));
                m = vfma(nr, vdup<R>(T0 + u * u), m);
                if constexpr (FORCE == FORCE_GUO) m = vfma(F, vdup<R>(u), m);
                return vmul(k8, m);
            };
            auto off = [&](int k, R ua, R ub, V Fa, V Fb) {
                V m = vfma(nr, vdup<R>(ua * ub), mom.m[k]);
                if constexpr (FORCE == FORCE_GUO)
                    m = vfma(Fb, vdup<R>(R(0.5) * ua), vfma(Fa, vdup<R>(R(0.5) * ub), m));
                m = vmul(k8, m);
                return vadd(m, m);
            };
            P[0] = diag(0, ux, Fx);
            P[1] = diag(1, uy, Fy);
            P[2] = diag(2, uz, Fz);
            P[3] = off(3, ux, uy, Fx, Fy);
            P[4] = off(4, ux, uz, Fx, Fz);
            P[5] = off(5, uy, uz, Fy, Fz);
            t = vdiv3<R>(vadd(P[0], vadd(P[1], P[2])));
        }
        // the deviation formats' constant, per unit k
        if constexpr (DEV) t = vadd(t, vdup<R>(p.rho0 * R(1.0 / 36.0)));
        V s3[3], d3[3];
        if constexpr (REG == COLL_REG3) {
            const R u[3] = {ux, uy, uz};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const R ub = u[a == 0 ? 1 : 0], uc = u[a == 2 ? 1 : 2];
                const R eq = R(0.5) * u[a] * (ub * ub + uc * uc), dq = R(1.5) * u[a] * (ub * ub - uc * uc);
                s3[a] = vmul(k8, vfma(nr, vdup<R>(eq), vdiv3<R>(mom.m[6 + a])));
                d3[a] = vmul(k8, vfma(nr, vdup<R>(dq), mom.m[9 + a]));
            }
        }
        {
            V o;
            if constexpr (FORCE == FORCE_EDM) o = vmul(rq, A);
            else o = vsub(vmul(rq, Au), uQ);
            if constexpr (kNeq || DEV) o = vsub(o, t);
            put(0, vmul(o, vdup<R>(R(12))));
        }
        // k_i (c c : Pi - tr / 3): axis pairs 2 (P_aa - t), diagonal pairs
        // (P_aa + P_bb - t) +- 2 P_ab
        V xt, yt, zt, base[3];   // base: xy, xz, yz
        if constexpr (kNeq) {
            xt = vsub(P[0], t); yt = vsub(P[1], t); zt = vsub(P[2], t);
            base[0] = vadd(xt, P[1]); base[1] = vadd(xt, P[2]); base[2] = vadd(yt, P[2]);
        }
        // even part of f*: rw E + n
        auto even = [&](int i, V rw, auto E) {
            if constexpr (kNeq) {
                V n;
                if (i < 7) {
                    const V d = i == 1 ? xt : (i == 3 ? yt : zt);
                    n = vadd(d, d);
                } else {
                    const int k = (i - 7) / 4;
                    n = ((i - 7) % 4) == 0 ? vadd(base[k], P[3 + k]) : vsub(base[k], P[3 + k]);
                }
                return vfma(rw, E, n);
            } else {
                const V e = vmul(rw, E);
                if constexpr (DEV) return vsub(e, i < 7 ? vadd(t, t) : t);
                else return e;
            }
        };
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            const bool axis = i < 7;
            V e, o;
            if constexpr (FORCE == FORCE_EDM) {
                const V c = vdot(i, vx, vy, vz), h = vmul(c, c45);
                const V rw = axis ? rq2 : rq;
                e = even(i, rw, vfma(h, c, A));
                o = vmul(rw, vmul(c, vfma(h, c, B)));
            } else {
                const U cu = vdot(i, Ux, Uy, Uz), hu = vmul(cu, u45);
                const V rw = axis ? rq2 : rq;
                V cQ = vdot(i, Qx, Qy, Qz), uq = uQ;
                if (axis) { cQ = vadd(cQ, cQ); uq = vadd(uq, uq); }
                e = vadd(even(i, rw, vfma(hu, cu, Au)), vsub(vmul(cQ, vmul(cu, udup<R>(R(3)))), uq));
                o = vfma(rw, vmul(cu, vfma(hu, cu, Bu)), cQ);
            }
            if constexpr (REG == COLL_REG3) {
                V m = vdup<R>(R(0));
                bool first = true;
                auto term = [&](int h, V v) {
                    if (h == 0) return;
                    if (first) m = h == 1 ? v : vmul(v, vdup<R>(R(h)));
                    else m = h == 1 ? vadd(m, v) : (h == -1 ? vsub(m, v) : vfma(v, vdup<R>(R(h)), m));
                    first = false;
                };
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    term(h3s3(i, a), s3[a]);
                    term(h3d(i, a), d3[a]);
                }
                o = axis ? vadd(o, vadd(m, m)) : vadd(o, m);
            }
            put(i, vadd(e, o));
            put(i + 1, vsub(e, o));
        }
    }
}

}  // namespace lbm
