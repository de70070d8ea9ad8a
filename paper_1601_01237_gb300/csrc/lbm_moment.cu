// Runs of steps in moment space (FP32 arithmetic).
//
// Under the regularized operator a step reads its 38 populations only to form
// the densities, the mixture momentum and (for tau != 1) the second moments
// of each component, and the post-collision populations are a polynomial in
// them and in the densities' gradient; at tau = 1 that holds for every
// operator.  So between the first and the last step of a call nothing else
// has to travel through memory: a run of n steps is
//   k_moment_in    populations -> moments m(t) of the gathered populations,
//   k_step_moment  m(t) -> m(t + 1), n - 1 times,
//   k_moment_out   m(t + n - 1) -> populations after its collision,
// with 5 values per cell at tau = 1 (rho^1, rho^2, u; 40 bytes per cell and step
// instead of 304) and 17 regularized (with sum c c f of both components; 136
// bytes).  Every value is held and every sum taken in FP32, opposite neighbours and
// opposite populations subtracted first in x and y and in z, where they come planes
// apart, taken relative to the column's densities (rms errors of u_z, u_x in runs of 5 to
// 100 steps over those of population steps: 0.92 to 0.97, 0.89 to 0.94; u_z with plain sums
// 1.04 to 1.13); the state at the end of the call is the population state.
// us per step in calls of 10 (512^3), 20 (256^3) and 100 steps, population steps and
// these with their ends: tau = 1 512^3 6991 / 3251, 256^3 869 / 414, 128^3 122 / 57, 96^3
// 55 / 33, regularized 256^3 873 / 649, 384 x 512 x 512 with walls 5424 / 3728, tau = 1 under
// a mask 256^3 1042 / 455.
#include <cuda_runtime.h>

#include <atomic>

#include "collide.cuh"
#include "d3q19.cuh"
#include "lbm_internal.h"

namespace lbm {

namespace {

// Moment state of N cells: pairs rho, (ux, uy), uz, and NP pairs of second
// moments (xx, yy, zz, xy, xz, yz), one array behind the other.
template <int KIND>
struct MomentState {
    static constexpr int NP = RegMoments<PairF32, KIND>::n;
    static_assert(KIND == COLL_EQ || KIND == COLL_REG, "operators that act on moments alone");
    float2 *rho, *uxy, *P;
    float *uz;
    __host__ __device__ MomentState(void *base, long long N)
    {
        rho = (float2 *)base;
        uxy = rho + N;
        P = uxy + N;                 // P[k N + cell]
        uz = (float *)(P + (long long)NP * N);
    }
    __device__ __forceinline__ void put_solid(unsigned cell, float2 r, unsigned N32) const
    {
        rho[cell] = r;
        uxy[cell] = make_float2(0.f, 0.f);
        uz[cell] = 0.f;
#pragma unroll
        for (int k = 0; k < NP; ++k) P[(size_t)k * N32 + cell] = make_float2(0.f, 0.f);
    }
};
template <int KIND>
constexpr size_t moment_floats() { return 5 + 2 * (size_t)RegMoments<PairF32, KIND>::n; }

struct Nb3 {
    unsigned cell, xo[3], yo[3], zo[3];
    bool zlo, zhi;
};

__device__ __forceinline__ Nb3 nb3(const Phys<float> &p, unsigned cell)
{
    const unsigned nx = (unsigned)p.nx, ny = (unsigned)p.ny, nz = (unsigned)p.nz, plane = nx * ny;
    const unsigned z = cell / plane, rem = cell - z * plane, y = rem / nx, x = rem - y * nx;
    Nb3 n;
    n.cell = cell;
    n.xo[0] = x == 0 ? nx - 1 : x - 1;
    n.xo[1] = x;
    n.xo[2] = x == nx - 1 ? 0 : x + 1;
    n.yo[0] = (y == 0 ? ny - 1 : y - 1) * nx;
    n.yo[1] = y * nx;
    n.yo[2] = (y == ny - 1 ? 0 : y + 1) * nx;
    n.zo[0] = (z == 0 ? nz - 1 : z - 1) * plane;
    n.zo[1] = z * plane;
    n.zo[2] = (z == nz - 1 ? 0 : z + 1) * plane;
    n.zlo = p.wall_z && z == 0;
    n.zhi = p.wall_z && z == nz - 1;
    return n;
}

constexpr int kThreadsM = 256;

// One thread per cell, bound by the bytes it gathers (152 in FP32, 76 in 16 bits).
// links (nullptr without a mask): every cell's link word (bit 0: the cell is
// solid; bit i: x - c_i is solid, so that link bounces back).  A solid site
// holds the density that it presents to Eq. 13 and no motion.
template <int S, int KIND>
__global__ void __launch_bounds__(kThreadsM)
k_moment_in(const typename Store<S>::T *__restrict__ f, MomentState<KIND> m, Phys<float> p, const unsigned *__restrict__ links)
{
    const unsigned cell = blockIdx.x * kThreadsM + threadIdx.x, N32 = (unsigned)p.N;
    if (cell >= N32) return;
    const Nb3 n = nb3(p, cell);
    const unsigned lw = links ? __ldg(links + cell) : 0u;
    if (lw & 1u) {
        m.put_solid(cell, make_float2(p.rho_s[0], p.rho_s[1]), N32);
        return;
    }
    float2 v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const bool wall = (cz(i) == 1 && n.zlo) || (cz(i) == -1 && n.zhi) || ((lw >> i) & 1u);
        const unsigned src = n.zo[1 - cz(i)] + n.yo[1 - cy(i)] + n.xo[1 - cx(i)];
        const typename Store<S>::T *q = f + 2 * (size_t)(wall ? (unsigned)opp(i) * N32 + cell : (unsigned)i * N32 + src);
        if constexpr (Store<S>::kDev) Store<S>::load2_d(q, v[i].x, v[i].y);   // (deviations have the momentum of the populations)
        else v[i] = ld_pair_f32(q);
    }
    float2 r = density(v);
    if constexpr (Store<S>::kDev) r = vadd(r, PairF32::dup(p.rho0));
    float jx, jy, jz;
    momentum(PairF32(), v, jx, jy, jz);
    const float inv = 1.0f / (r.x + r.y);
    m.rho[cell] = r;
    m.uxy[cell] = make_float2(jx * inv, jy * inv);
    m.uz[cell] = jz * inv;
    RegMoments<PairF32, KIND> mo;
    mo.of(v);
#pragma unroll
    for (int k = 0; k < MomentState<KIND>::NP; ++k) {
        if constexpr (Store<S>::kDev) {
            if (k < 3) mo.m[k] = vadd(mo.m[k], PairF32::dup(p.rho0 * (1.0f / 3.0f)));
        }
        m.P[(size_t)k * N32 + cell] = mo.m[k];
    }
}

// One thread per cell, bound by the bytes it stores.
template <int FMT, int KIND, int FORCE>
__global__ void __launch_bounds__(kThreadsM)
k_moment_out(MomentState<KIND> m, typename Store<FMT>::T *__restrict__ f, Phys<float> p, const unsigned *__restrict__ links)
{
    const unsigned cell = blockIdx.x * kThreadsM + threadIdx.x, N32 = (unsigned)p.N;
    if (cell >= N32) return;
    const Nb3 n = nb3(p, cell);
    if (links && (__ldg(links + cell) & 1u)) {   // nothing in a solid site
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const float e = w<float>(i) * p.rho0;
            Store<FMT>::store2(f + 2 * (size_t)((unsigned)i * N32 + cell), 0.f, 0.f, e, e);
        }
        return;
    }
    const float2 rs = make_float2(p.rho_s[0], p.rho_s[1]);
    const float2 *__restrict__ rho = m.rho;
    auto at = [&](int dx, int dy, int dz) {
        if ((dz == -1 && n.zlo) || (dz == 1 && n.zhi))
            return p.wall_mirror ? vadd(__ldg(rho + n.zo[1] + n.yo[1 + dy] + n.xo[1 + dx]), rs) : rs;
        return __ldg(rho + n.zo[1 + dz] + n.yo[1 + dy] + n.xo[1 + dx]);
    };
    float2 S[3];
    interaction<PairF32>([&](int i) { return vsub(at(cx(i), cy(i), cz(i)), at(-cx(i), -cy(i), -cz(i))); }, S);
    const float2 So[3] = {vswap(S[0]), vswap(S[1]), vswap(S[2])};
    const float2 r = m.rho[cell], uxy = m.uxy[cell];
    RegMoments<PairF32, KIND> mo;
#pragma unroll
    for (int k = 0; k < MomentState<KIND>::NP; ++k) mo.m[k] = m.P[(size_t)k * N32 + cell];
    auto get = [](int) { return make_float2(0.f, 0.f); };
    auto put = [&](int i, float2 v) {
        typename Store<FMT>::T *q = f + 2 * (size_t)((unsigned)i * N32 + cell);
        if constexpr (Store<FMT>::kDev) Store<FMT>::store2_d(q, v.x, v.y);
        else Store<FMT>::store2(q, v.x, v.y, 0.f, 0.f);
    };
    if constexpr (Store<FMT>::kDev) {   // collide_cell takes the second moments of the deviations
#pragma unroll
        for (int k = 0; k < 3 && k < MomentState<KIND>::NP; ++k)
            mo.m[k] = vsub(mo.m[k], PairF32::dup(p.rho0 * (1.0f / 3.0f)));
    }
    collide_cell<PairF32, KIND, FORCE, Store<FMT>::kDev>(PairF32(), p, r, 1.0f / (r.x + r.y), uxy.x, uxy.y, m.uz[cell], So, mo, get, put);
}

// Wall densities of the mirror model under a mask, after each new moment state:
// each solid site with a fluid neighbour takes the w_i-weighted mean of its fluid
// neighbours' densities plus rho_s (Eq. 13).  One thread per site: the sites are a
// surface, so launch and one gather's latency bound it (8.5 us beside the 425 of a
// 256^3 step with an inclined slab).
__global__ void __launch_bounds__(kThreadsM)
k_moment_walls(float2 *__restrict__ rho, Phys<float> p, const unsigned *__restrict__ links,
               const unsigned *__restrict__ sites, long long n_sites)
{
    const long long t = (long long)blockIdx.x * kThreadsM + threadIdx.x;
    if (t >= n_sites) return;
    const Nb3 n = nb3(p, sites[t]);
    const unsigned lw = __ldg(links + n.cell);   // bit i: x - c_i is solid
    float2 num = make_float2(0.f, 0.f);
    int den36 = 0;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        if ((lw >> i) & 1u) continue;
        num = vfma(PairF32::dup((float)k36(i)), rho[n.zo[1 - cz(i)] + n.yo[1 - cy(i)] + n.xo[1 - cx(i)]], num);
        den36 += k36(i);
    }
    const float d = (float)den36;
    rho[n.cell] = den36 ? make_float2(num.x / d + p.rho_s[0], num.y / d + p.rho_s[1]) : make_float2(p.rho_s[0], p.rho_s[1]);
}

// ---------------------------------------------------------------------------
// m(t) -> m(t + 1).  A CTA owns 30 x (EY - 2) columns and marches along z over
// lz planes; its 32 x EY threads are those columns and the ring around them, one
// thread per column.  Per plane p:
//   a. each thread completes the interaction sums of its cell from the density
//      planes p - 1, p, p + 1 (each plane is read once from shared memory and
//      adds to the sums of the three planes that see it), collides the cell and
//      leaves the 16 pairs of its post-collision populations that move in x or
//      y in shared memory;
//   -- barrier --
//   b. each thread picks up the 16 pairs that stream into its column, from the
//      plane's own direction group (c_z = 0), into plane p + 1 (c_z = +1) and into
//      plane p - 1 (c_z = -1), as sums and differences of opposite sources, adds
//      them to the moments of those planes and stores the moments of plane
//      p - 1, which are then complete;
//   -- barrier, unless the next plane's pairs go to another copy --
// The next plane's moments and the density plane after it are loaded one
// iteration ahead.  The ring's collisions are computed by every neighbouring
// CTA too (512 collisions for 420 cells in tiles of 16 rows), and a CTA computes one plane more at
// each end of its chunk; densities reach one cell further, loaded by 68 + 2 EY
// of the threads.
// MASK: a solid site lets nothing out, so that what streams from it is zero, and a
// cell with a link into a solid site (a bit of its link word) adds its own
// populations of these links, reversed, to its plane; the solid sites' densities
// stand in the moment state (k_moment_walls), and the gradient needs no case.
constexpr int kEX = 32, kOX = kEX - 2, kRX = kEX + 2;   // along x: threads, tile, densities
constexpr int kPad = 40;                                // a neighbour's offset is at most 33
constexpr int kMove = 16;
static_assert(kPad >= kEX + 1, "");
// Tiles of EY thread rows.  NB = 2 copies of the moving populations leave one
// barrier per plane instead of two, where shared memory holds them.  ns: measured
// time per plane of an SM full of such CTAs, so that the tile with the least work
// (rings, ragged edges and the last wave counted) is taken.  us per step at tau = 1,
// tiles 12 / 16 / 24: 512^3 3323 / 3252 / 3342, 256^3 414 / 422 / 417, 128^3 67 / 67 / 57,
// 96^3 33 / 36 / 34; regularized 12 / 16: 256^3 651 / 649, 131 x 150 x 173 135 / 141,
// 384 x 512 x 512 with walls 3754 / 3724.  Under a mask tiles of 16 rows spill at tau = 1
// (256^3 835 us, the others 454 and 464), and regularized ones of 18 or more rows do.
template <int KIND, int EY_>
struct Tile {
    static constexpr int EY = EY_, ctas = KIND == COLL_EQ && EY <= 16 ? 2 : 1, NB = KIND == COLL_EQ && EY == 16 ? 1 : 2;
    static constexpr int ns = KIND == COLL_EQ ? (EY == 12 ? 1870 : (EY == 16 ? 2580 : 2060)) : (EY == 12 ? 1460 : 2005);
    static constexpr int threads = kEX * EY, OY = EY - 2, RY = EY + 2;
    static constexpr int rim = 2 * kRX + 2 * EY;   // cells of a density plane beyond the threads' own
    // density planes held: 4 leave a column's densities at q - 1, q and q + 1 in place
    // where the 64 registers of two CTAs of 512 threads do not hold them
    static constexpr int NR = KIND == COLL_EQ && EY == 16 ? 4 : 2;
    static_assert(rim <= threads, "");
};

template <class T>
struct MomentSmem {
    float2 lead[kPad];                    // (threads of the ring read past the ends; what they collect is not stored)
    float2 f[T::NB][kMove][T::threads];   // moving populations of a plane
    float2 tail[kPad];
    float2 rho[T::NR][T::RY][kRX];        // density planes p + 1 and p + 2 (T::NR = 4: from p - 1 on)
};

// The direction with given components.
__host__ __device__ constexpr int dir_of(int x, int y, int z)
{
    for (int i = 0; i < Q; ++i)
        if (cx(i) == x && cy(i) == y && cz(i) == z) return i;
    return -1;
}

constexpr int kUp = dir_of(0, 0, 1), kDown = dir_of(0, 0, -1);
static_assert(kUp == 5 && kDown == 6, "");
// Place of a moving direction in MomentSmem::f (put() below has the same rule).
// A template, so that it is a constant: the search is not folded at run time
// (the kernel took 1744 us per step at 256^3 with it, 382 without).
template <int X, int Y, int Z>
struct MoveSlot {
    static constexpr int i = dir_of(X, Y, Z), value = i < kUp ? i - 1 : i - 3;
    static_assert(X != 0 || Y != 0, "moves in x or y");
};

// Moments of a plane's cells as they collect: density and second moments as
// pairs, momentum of the mixture.
template <int KIND>
struct Collect {
    static constexpr int NP = RegMoments<PairF32, KIND>::n;
    static constexpr float kShare = 7.f / 256.f;
    float2 rho, P[NP > 0 ? NP : 1];
    float jx, jy, jz;
    __device__ __forceinline__ void zero()
    {
        rho = make_float2(0.f, 0.f);
        jx = jy = jz = 0.f;
#pragma unroll
        for (int k = 0; k < NP; ++k) P[k] = make_float2(0.f, 0.f);
    }
    // the eight populations of c_z = 0 that move, along +x, -x, +y, -y and the
    // diagonals (+,+), (-,-), (+,-), (-,+)
    __device__ __forceinline__ void add_plane(float2 xp, float2 xm, float2 yp, float2 ym, float2 a, float2 b, float2 c,
                                              float2 d)
    {
        const float2 ab = vadd(a, b), cd = vadd(c, d), da = vsub(a, b), dc = vsub(c, d);
        const float2 ex = vadd(xp, xm), ey = vadd(yp, ym), dg = vadd(ab, cd);
        const float2 mx = vadd(vsub(xp, xm), vadd(da, dc)), my = vadd(vsub(yp, ym), vsub(da, dc));
        rho = vadd(rho, vadd(vadd(ex, ey), dg));
        jx += mx.x + mx.y;
        jy += my.x + my.y;
        if constexpr (NP > 0) {
            P[0] = vadd(P[0], vadd(ex, dg));
            P[1] = vadd(P[1], vadd(ey, dg));
            P[3] = vadd(P[3], vsub(ab, cd));
        }
    }
    // the five populations of a group c_z = Z = +-1: the one that stays in its
    // column, and those from the columns at -x, +x, -y, +y (moving the other way).
    // REF: less a share of the cell's density r one step before, which both groups of the
    // cell know: they come two planes apart, and the z momentum would else be the
    // difference of two sums of the populations' size.  (kShare is near w_7 and has three
    // bits, so that the products are exact; with w_7 rounded what is left is a rounding
    // with a sign of its own, and the density's sum swallows it: mass drifts.)  finish()
    // adds the shares back.
    template <int Z, bool REF>
    __device__ __forceinline__ void add_group(float2 n0, float2 xp, float2 xm, float2 yp, float2 ym, float2 r)
    {
        const float2 dx = vsub(xp, xm), dy = vsub(yp, ym);
        const float2 ex = vadd(xp, xm), ey = vadd(yp, ym);
        float2 s = vadd(ex, ey);
        if (REF) {
            n0 = vfma(r, PairF32::dup(-2.f * kShare), n0);
            s = vfma(r, PairF32::dup(-4.f * kShare), s);
        }
        s = vadd(n0, s);
        rho = vadd(rho, s);
        jx += dx.x + dx.y;
        jy += dy.x + dy.y;
        if (Z > 0) jz += s.x + s.y;
        else jz -= s.x + s.y;
        if constexpr (NP > 0) {
            P[0] = vadd(P[0], ex);
            P[1] = vadd(P[1], ey);
            P[2] = vadd(P[2], s);
            P[4] = Z > 0 ? vadd(P[4], dx) : vsub(P[4], dx);
            P[5] = Z > 0 ? vadd(P[5], dy) : vsub(P[5], dy);
        }
    }
    __device__ __forceinline__ void finish(float2 r)
    {
        rho = vfma(r, PairF32::dup(12.f * kShare), rho);
        if constexpr (NP > 0) P[2] = vfma(r, PairF32::dup(12.f * kShare), P[2]);
    }
};

template <int KIND, int FORCE, int EY, bool WALLZ, bool MASK>
__global__ void __launch_bounds__(Tile<KIND, EY>::threads, Tile<KIND, EY>::ctas)
k_step_moment(const MomentState<KIND> in, MomentState<KIND> out, Phys<float> p, int ntx, int lz,
              const unsigned *__restrict__ links)
{
    static_assert(!(MASK && WALLZ), "a solid mask needs a lattice periodic along z");
    constexpr int NP = MomentState<KIND>::NP;
    using T = Tile<KIND, EY>;
    constexpr int kOY = T::OY, kRY = T::RY, kRim = T::rim, kThreadsS = T::threads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MomentSmem<T> &sm = *reinterpret_cast<MomentSmem<T> *>(smem_raw);
    const int tid = threadIdx.x, ex = tid % kEX, ey = tid / kEX;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const unsigned plane = (unsigned)nx * (unsigned)ny, N32 = (unsigned)p.N;
    const int x0 = (int)(blockIdx.x % (unsigned)ntx) * kOX, y0 = (int)(blockIdx.x / (unsigned)ntx) * kOY;
    const int z0 = (int)blockIdx.y * lz, z1 = min(z0 + lz, nz);
    const bool stores = ex >= 1 && ex <= kOX && ey >= 1 && ey <= kOY && x0 + ex - 1 < nx && y0 + ey - 1 < ny;
    auto column = [&](int x, int y) {   // periodic in x and y
        x %= nx; if (x < 0) x += nx;
        y %= ny; if (y < 0) y += ny;
        return (unsigned)y * (unsigned)nx + (unsigned)x;
    };
    const unsigned col = column(x0 + ex - 1, y0 + ey - 1);
    // the rim cell of the density plane that this thread also loads
    int rx = 0, ry = 0;
    if (tid < kRX) { rx = tid; ry = 0; }
    else if (tid < 2 * kRX) { rx = tid - kRX; ry = kRY - 1; }
    else { const int k = tid - 2 * kRX; rx = (k & 1) ? kRX - 1 : 0; ry = 1 + (k >> 1); }
    const bool rim = tid < kRim;
    const unsigned rcol = rim ? column(x0 + rx - 2, y0 + ry - 2) : 0u;
    // offset of plane q: periodic, or the mirror plane of a wall site
    auto offset = [&](int q) {
        if (WALLZ) q = q < 0 ? 0 : (q >= nz ? nz - 1 : q);
        else { q %= nz; if (q < 0) q += nz; }
        return (unsigned)q * plane;
    };
    const float2 rs = make_float2(p.rho_s[0], p.rho_s[1]);
    auto present = [&](int q, float2 r) {   // what plane q presents to Eq. 13
        if (WALLZ && (q < 0 || q >= nz)) return p.wall_mirror ? vadd(r, rs) : rs;
        return r;
    };
    cudaTriggerProgrammaticLaunchCompletion();   // the next step may be set up
    cudaGridDependencySynchronize();             // the previous step's moments
    // density plane z0 - 2 into its slot, z0 - 1 into registers
    const int first = z0 - 1;   // first plane that collides
    float2 r_next, h_next = make_float2(0.f, 0.f);
    {
        const unsigned o = offset(first - 1);
        sm.rho[(first - 1) & (T::NR - 1)][ey + 1][ex + 1] = present(first - 1, in.rho[o + col]);
        if (rim) sm.rho[(first - 1) & (T::NR - 1)][ry][rx] = present(first - 1, in.rho[o + rcol]);
        const unsigned o1 = offset(first);
        r_next = in.rho[o1 + col];
        if (rim) h_next = in.rho[o1 + rcol];
    }
    float2 uxy = make_float2(0.f, 0.f);
    float uz = 0.f;
    unsigned lw = 0, lw_p = 0;   // link words of the column at plane q + 1, q - 1
    RegMoments<PairF32, KIND> mo;
    // x and y sums of plane q so far, what it adds to q + 1's, its Laplacian's two
    // predecessors, and the column's densities at q and q - 1
    const float2 zero = make_float2(0.f, 0.f);
    constexpr bool keep = T::NR == 2;
    auto own = [&](int k) { return sm.rho[k & (T::NR - 1)][ey + 1][ex + 1]; };
    float2 S[2] = {zero, zero}, lo[2] = {zero, zero}, L0 = zero, L1 = zero, r_own = zero, r_old = zero;
    Collect<KIND> c0, c1;   // planes p - 1 and p
    c0.zero();
    c1.zero();
    const float2 w1 = PairF32::dup(w<float>(1)), w2 = PairF32::dup(w<float>(7));
    __syncthreads();
    // p = first - 2, first - 1: only the density planes first - 1 and first come in
    for (int q = first - 2; q <= z1; ++q) {
        // ---- a. plane q + 1's densities are in place: they complete plane q's
        //      sums and start plane q + 1's and q + 2's
        const bool collides = q >= first && !(WALLZ && (q < 0 || q >= nz));
        // (density plane q + 2 into its slot, where plane q, of four held plane q - 2, was: the
        // neighbours read it before the last iteration's barrier, so that their reads have to
        // stay in section a; a thread's own() reads are of cells that it writes itself)
        sm.rho[(q + 2) & (T::NR - 1)][ey + 1][ex + 1] = present(q + 2, r_next);
        if (rim) sm.rho[(q + 2) & (T::NR - 1)][ry][rx] = present(q + 2, h_next);
        // loads for the next iteration
        const float2 uxy_c = uxy;
        const float uz_c = uz;
        const unsigned lw_c = lw;
        const RegMoments<PairF32, KIND> mo_c = mo;
        if (q < z1) {
            const unsigned o3 = offset(q + 3), o1 = offset(q + 1);
            r_next = in.rho[o3 + col];
            if (rim) h_next = in.rho[o3 + rcol];
            uxy = in.uxy[o1 + col];
            uz = in.uz[o1 + col];
            if (MASK) lw = __ldg(links + o1 + col);
#pragma unroll
            for (int k = 0; k < NP; ++k) mo.m[k] = in.P[(size_t)k * N32 + o1 + col];
        }
        float2 So[3], rc;
        {
            const float2(*R)[kRX] = &sm.rho[(q + 1) & (T::NR - 1)][ey];   // rows ey, ey + 1, ey + 2: y - 1, y, y + 1
            const float2 xp = R[1][ex + 2], xm = R[1][ex], yp = R[2][ex + 1], ym = R[0][ex + 1];
            rc = R[1][ex + 1];
            const float2 dx = vsub(xp, xm), dy = vsub(yp, ym);
            const float2 a = vsub(R[2][ex + 2], R[0][ex]), b = vsub(R[0][ex + 2], R[2][ex]);   // (1,1), (1,-1)
            // S_z = w_7 (6 (rho(q + 1) - rho(q - 1)) + L(q + 1) - L(q - 1)) with L the sum of the four
            // neighbours less 4 rho: differences first, as in x and y (x_- - rho = x_+ - rho - dx)
            const float2 L = vfma(vadd(vsub(xp, rc), vsub(yp, rc)), make_float2(2.f, 2.f), vsub(zero, vadd(dx, dy)));
            const float2 lx = vmul(w2, dx), ly = vmul(w2, dy);
            // plane q: this plane lies above it
            So[0] = vswap(vadd(S[0], lx));
            So[1] = vswap(vadd(S[1], ly));
            So[2] = vswap(vmul(w2, vfma(vsub(rc, keep ? r_old : own(q - 1)), make_float2(6.f, 6.f), vsub(L, L0))));
            // plane q + 1: its own plane
            S[0] = vadd(lo[0], vfma(w1, dx, vmul(w2, vadd(a, b))));
            S[1] = vadd(lo[1], vfma(w1, dy, vmul(w2, vsub(a, b))));
            // plane q + 2: this plane lies below it
            lo[0] = lx;
            lo[1] = ly;
            L0 = L1;
            L1 = L;
        }
        float2 *const F = &sm.f[T::NB == 2 ? (q & 1) : 0][0][tid];
        const float2 r = keep ? r_own : own(q);   // density of plane q at this column
        if (keep) r_own = rc;
        float2 f0, fu, fd;        // populations that stay in the column: c_z = 0, +1, -1
        if (collides) {
            auto get = [](int) { return make_float2(0.f, 0.f); };
            auto put = [&](int i, float2 v) {
                if (i == 0) f0 = v;
                else if (i == kUp) fu = v;
                else if (i == kDown) fd = v;
                else F[(i < kUp ? i - 1 : i - 3) * kThreadsS] = v;
            };
            if (MASK && (lw_c & 1u)) {   // nothing leaves a solid site
#pragma unroll
                for (int i = 0; i < Q; ++i) put(i, make_float2(0.f, 0.f));
            } else {
                collide_cell<PairF32, KIND, FORCE, false>(PairF32(), p, r, 1.0f / (r.x + r.y), uxy_c.x, uxy_c.y, uz_c, So,
                                                          mo_c, get, put);
            }
        }
        __syncthreads();
        // ---- b. what streams into this column
        const float2 r_dn = keep ? r_old : own(q - 1);
        Collect<KIND> c2;         // plane q + 1
        c2.zero();
        if (collides) {
            // the population (X, Y, Z) out of column - (X, Y), and the cell's own
#define LBM_FROM(X, Y, Z) F[MoveSlot<X, Y, Z>::value * kThreadsS - (X) - (Y) * kEX]
#define LBM_OWN(X, Y, Z) F[MoveSlot<X, Y, Z>::value * kThreadsS]
            {   // c_z = 0
                const float2 xp = LBM_FROM(1, 0, 0), xm = LBM_FROM(-1, 0, 0), yp = LBM_FROM(0, 1, 0), ym = LBM_FROM(0, -1, 0);
                const float2 a = LBM_FROM(1, 1, 0), b = LBM_FROM(-1, -1, 0), c = LBM_FROM(1, -1, 0), d = LBM_FROM(-1, 1, 0);
                c1.rho = vadd(c1.rho, f0);
                c1.add_plane(xp, xm, yp, ym, a, b, c, d);
            }
            c2.template add_group<1, true>(fu, LBM_FROM(1, 0, 1), LBM_FROM(-1, 0, 1), LBM_FROM(0, 1, 1), LBM_FROM(0, -1, 1),
                                           keep ? r_own : own(q + 1));
            c0.template add_group<-1, true>(fd, LBM_FROM(1, 0, -1), LBM_FROM(-1, 0, -1), LBM_FROM(0, 1, -1),
                                            LBM_FROM(0, -1, -1), r_dn);
            if (WALLZ) {   // half-way bounce-back: the cell's own populations come back reversed
                if (q == 0)
                    c1.template add_group<1, true>(fd, LBM_OWN(-1, 0, -1), LBM_OWN(1, 0, -1), LBM_OWN(0, -1, -1),
                                                   LBM_OWN(0, 1, -1), r);
                if (q == nz - 1)
                    c1.template add_group<-1, true>(fu, LBM_OWN(-1, 0, 1), LBM_OWN(1, 0, 1), LBM_OWN(0, -1, 1),
                                                    LBM_OWN(0, 1, 1), r);
            }
            if (MASK && lw_c > 1u) {   // links into solid sites
#define LBM_BACK(X, Y, Z) (((lw_c >> dir_of(X, Y, Z)) & 1u) ? LBM_OWN(-(X), -(Y), -(Z)) : make_float2(0.f, 0.f))
                {   // c_z = 0
                    const float2 xp = LBM_BACK(1, 0, 0), xm = LBM_BACK(-1, 0, 0), yp = LBM_BACK(0, 1, 0), ym = LBM_BACK(0, -1, 0);
                    const float2 a = LBM_BACK(1, 1, 0), b = LBM_BACK(-1, -1, 0), c = LBM_BACK(1, -1, 0), d = LBM_BACK(-1, 1, 0);
                    c1.add_plane(xp, xm, yp, ym, a, b, c, d);
                }
                // (what takes the place of the zeros out of the solid sites, whose w_i t is off already)
                c1.template add_group<1, false>(((lw_c >> kUp) & 1u) ? fd : make_float2(0.f, 0.f), LBM_BACK(1, 0, 1),
                                                LBM_BACK(-1, 0, 1), LBM_BACK(0, 1, 1), LBM_BACK(0, -1, 1), zero);
                c1.template add_group<-1, false>(((lw_c >> kDown) & 1u) ? fu : make_float2(0.f, 0.f), LBM_BACK(1, 0, -1),
                                                 LBM_BACK(-1, 0, -1), LBM_BACK(0, 1, -1), LBM_BACK(0, -1, -1), zero);
#undef LBM_BACK
            }
#undef LBM_FROM
#undef LBM_OWN
        }
        if (q > z0 && stores) {   // plane q - 1 is complete
            const unsigned cell = (unsigned)(q - 1) * plane + col;
            if (MASK && (lw_p & 1u)) {
                out.put_solid(cell, rs, N32);
            } else {
                c0.finish(r_dn);
                const float inv = 1.0f / (c0.rho.x + c0.rho.y);
                out.rho[cell] = c0.rho;
                out.uxy[cell] = make_float2(c0.jx * inv, c0.jy * inv);
                out.uz[cell] = c0.jz * inv;
#pragma unroll
                for (int k = 0; k < NP; ++k) out.P[(size_t)k * N32 + cell] = c0.P[k];
            }
        }
        lw_p = lw_c;
        if (keep) r_old = r;
        c0 = c1;
        c1 = c2;
        if (T::NB == 1) __syncthreads();   // (two copies: a copy's readers passed the next plane's barrier)
    }
}

Phys<float> make_phys_m(const HostPhys &h)
{
    Phys<float> p;
    p.nx = h.nx; p.ny = h.ny; p.nz = h.nz; p.N = h.N;
    p.wall_z = h.wall_z;
    p.wall_mirror = h.wall_mirror;
    p.omega[0] = (float)(1.0 / h.tau[0]);
    p.omega[1] = (float)(1.0 / h.tau[1]);
    p.G12 = (float)h.G12; p.G21 = (float)h.G21;
    for (int d = 0; d < 3; ++d) p.gext[d] = (float)h.gext[d];
    p.rho_s[0] = (float)h.rho_s[0]; p.rho_s[1] = (float)h.rho_s[1];
    p.rho0 = (float)h.rho0;
    return p;
}

// Planes per CTA: equal chunks of at most 128, the fewest waves x (planes + 4) (the
// collisions beyond the two ends of a chunk and the density planes before it); waves:
// their number.
int moment_planes(long long cols, int nz, long long slots, long long *waves)
{
    int best = nz;
    long long least = -1;
    for (int most = nz < 128 ? nz : 128; most >= 1; --most) {   // (by length: few of them however tall the lattice)
        const int nch = (nz + most - 1) / most, lz = (nz + nch - 1) / nch;
        if (lz < 4 && nch > 1) break;
        const long long w = (cols * ((nz + lz - 1) / lz) + slots - 1) / slots;
        if (least < 0 || w * (lz + 4) < least) { least = w * (lz + 4); best = lz; *waves = w; }
    }
    return best;
}

// Takes the tile of EY rows into the plan if it is the cheapest so far (cost: that of the others).
template <int KIND, int EY>
void plan_tile(const HostPhys &h, MomentPlan &q, double &cost)
{
    using T = Tile<KIND, EY>;
    const int ntx = (h.nx + kOX - 1) / kOX;
    const long long cols = (long long)ntx * ((h.ny + T::OY - 1) / T::OY);
    long long waves = 1;
    const int lz = moment_planes(cols, h.nz, (long long)T::ctas * current_device_sms(), &waves);
    const double c = (double)waves * (lz + 4) * T::ns;
    if (q.rows && !(c < cost)) return;
    cost = c;
    q.rows = EY;
    q.ntx = ntx;
    q.lz = lz;
    q.cols = cols;
    // (the planes beyond a chunk that do not collide cost less: all four count near four
    // only regularized; at z walls there is no plane beyond)
    const double planes = lz + (KIND == COLL_EQ ? 3.3 : 4.2) - (h.wall_z && lz == h.nz ? 1.0 : 0.0);
    q.step_us = 1e-3 * (double)waves * planes * T::ns;
}

constexpr int kMaxAttrDevices = 64;

template <int KIND, int FORCE, int EY, bool WALLZ, bool MASK>
cudaError_t launch_tile(const HostPhys &h, const MomentPlan &q, const void *in, void *out, cudaStream_t s)
{
    using T = Tile<KIND, EY>;
    static std::atomic<int> attr_set[kMaxAttrDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool cached = dev >= 0 && dev < kMaxAttrDevices;
    if (!cached || !attr_set[dev].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute((const void *)k_step_moment<KIND, FORCE, EY, WALLZ, MASK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(MomentSmem<T>));
        if (e != cudaSuccess) return e;
        if (cached) attr_set[dev].store(1, std::memory_order_release);
    }
    const dim3 grid((unsigned)q.cols, (unsigned)((h.nz + q.lz - 1) / q.lz));
    // Successive steps overlap at their ends (programmatic stream serialization):
    // a step's CTAs are set up while the last wave of the previous one drains, and
    // wait for it before their first access (us per step without and with: tau = 1 61 x
    // 65 x 70 16.4 / 14.0, 100^3 35.0 / 32.9, regularized 20.5 / 17.1, 54.0 / 51.9).
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(T::threads);
    c.dynamicSmemBytes = sizeof(MomentSmem<T>);
    c.stream = s;
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k_step_moment<KIND, FORCE, EY, WALLZ, MASK>, MomentState<KIND>(const_cast<void *>(in), h.N),
                              MomentState<KIND>(out, h.N), make_phys_m(h), q.ntx, q.lz, h.links);
}

template <int KIND, bool WALLZ, bool MASK>
cudaError_t launch_step(const HostPhys &h, const MomentPlan &q, const void *in, void *out, cudaStream_t s)
{
    if (h.forcing == FORCE_GUO) return launch_tile<KIND, FORCE_GUO, 12, WALLZ, MASK>(h, q, in, out, s);
    if (q.rows == 12) return launch_tile<KIND, FORCE_EDM, 12, WALLZ, MASK>(h, q, in, out, s);
    if constexpr (KIND == COLL_EQ) {
        if (q.rows == 24) return launch_tile<KIND, FORCE_EDM, 24, WALLZ, MASK>(h, q, in, out, s);
    }
    if constexpr (KIND != COLL_EQ || !MASK) {
        if (q.rows == 16) return launch_tile<KIND, FORCE_EDM, 16, WALLZ, MASK>(h, q, in, out, s);
    }
    return cudaErrorInvalidValue;
}

template <int KIND>
MomentPlan plan_kind(const HostPhys &h)
{
    MomentPlan q = {};
    double cost = 0;
    plan_tile<KIND, 12>(h, q, cost);
    if (h.forcing == FORCE_GUO) {   // (it needs the registers of that tile: 256^3 467 us, exact difference 414)
        q.step_us *= 1.15;
    } else {
        if (KIND != COLL_EQ || !h.links) plan_tile<KIND, 16>(h, q, cost);
        if constexpr (KIND == COLL_EQ) plan_tile<KIND, 24>(h, q, cost);
    }
    q.bytes = sizeof(float) * moment_floats<KIND>() * (size_t)h.N;
    // the two ends are bound by their bytes: ps per cell (256^3: 410 + 448 us, 528 + 559;
    // 16 bits 263 + 354, 366 + 464)
    const bool f32 = h.storage == ST_F32;
    q.ends_us = 4.0 + 1e-6 * (double)h.N * (KIND == COLL_EQ ? (f32 ? 52 : 38) : (f32 ? 66 : 51));
    q.fused_us = marching_us(h);
    return q;
}

bool tau_one(const HostPhys &h) { return (float)(1.0 / h.tau[0]) == 1.0f && (float)(1.0 / h.tau[1]) == 1.0f; }

inline unsigned grid_m(long long N) { return (unsigned)((N + kThreadsM - 1) / kThreadsM); }

}  // namespace

// A run of n steps takes the two ends and n - 1 steps on moments, where that is estimated
// to be less than n steps on populations: lattices of a few planes, or much narrower than
// a tile, collide too many cells twice.  us per step in runs of 20, populations / moments:
// FP32 regularized 1 x 2100^2 395 / 640, 2 x 2100^2 631 / 829, 6 x 2100^2 1668 / 1437,
// 20000 x 32 x 32 1029 / 1464, 256^3 878 / 653; tau = 1 1 x 2100^2 374 / 361; FP16 deviations tau = 1
// 1 x 2100^2 275 / 358, 6 x 2100^2 1020 / 797, regularized 6 x 2100^2 1267 / 1416, 256^3 696 / 640
// (two steps there 696 / 728).
MomentPlan moment_plan(const HostPhys &h)
{
    const MomentPlan none = {};
    // The relative formats stay step by step: they hand out FP32 reference densities,
    // which carry every step's rounding to 16 bits.
    if (h.storage != ST_F32 && h.storage != ST_F16_DEV && h.storage != ST_BF16_DEV) return none;
    if (!tau_one(h) && h.collision != LBM_REGULARIZED) return none;
    if (!fused_supported(h) || use_box(h)) return none;
    const long long cols = (long long)((h.nx + kOX - 1) / kOX) * ((h.ny + Tile<COLL_REG, 12>::OY - 1) / Tile<COLL_REG, 12>::OY);
    if (cols >= (1LL << 31) || h.nz > 4 * 65535) return none;   // grid limits
    return tau_one(h) ? plan_kind<COLL_EQ>(h) : plan_kind<COLL_REG>(h);
}

namespace {

template <int KIND>
cudaError_t moment_walls(const HostPhys &h, void *m, cudaStream_t s)
{
    if (h.links && h.wall_mirror && h.n_bsolid > 0)
        k_moment_walls<<<grid_m(h.n_bsolid), kThreadsM, 0, s>>>(MomentState<KIND>(m, h.N).rho, make_phys_m(h), h.links,
                                                                h.bsolid, h.n_bsolid);
    return cudaGetLastError();
}

template <int S, int KIND>
cudaError_t moment_in_t(const HostPhys &h, const void *f, void *m, cudaStream_t s)
{
    k_moment_in<S, KIND><<<grid_m(h.N), kThreadsM, 0, s>>>((const typename Store<S>::T *)f, MomentState<KIND>(m, h.N),
                                                           make_phys_m(h), h.links);
    return moment_walls<KIND>(h, m, s);
}

template <int KIND>
cudaError_t moment_step_t(const HostPhys &h, const MomentPlan &q, const void *in, void *out, cudaStream_t s)
{
    const cudaError_t e = h.wall_z ? launch_step<KIND, true, false>(h, q, in, out, s)
                          : h.links ? launch_step<KIND, false, true>(h, q, in, out, s)
                                    : launch_step<KIND, false, false>(h, q, in, out, s);
    return e == cudaSuccess ? moment_walls<KIND>(h, out, s) : e;
}

template <int S, int KIND, int FORCE>
cudaError_t moment_out_t(const HostPhys &h, const void *m, void *f, cudaStream_t s)
{
    k_moment_out<S, KIND, FORCE><<<grid_m(h.N), kThreadsM, 0, s>>>(MomentState<KIND>(const_cast<void *>(m), h.N),
                                                            (typename Store<S>::T *)f, make_phys_m(h), h.links);
    return cudaGetLastError();
}

template <int S>
cudaError_t in_s(const HostPhys &h, const void *f, void *m, cudaStream_t s)
{
    return tau_one(h) ? moment_in_t<S, COLL_EQ>(h, f, m, s) : moment_in_t<S, COLL_REG>(h, f, m, s);
}

template <int S>
cudaError_t out_s(const HostPhys &h, const void *m, void *f, cudaStream_t s)
{
    if (h.forcing == FORCE_GUO)
        return tau_one(h) ? moment_out_t<S, COLL_EQ, FORCE_GUO>(h, m, f, s) : moment_out_t<S, COLL_REG, FORCE_GUO>(h, m, f, s);
    return tau_one(h) ? moment_out_t<S, COLL_EQ, FORCE_EDM>(h, m, f, s) : moment_out_t<S, COLL_REG, FORCE_EDM>(h, m, f, s);
}

}  // namespace

cudaError_t launch_moment_in(const HostPhys &h, const void *f, void *m, cudaStream_t s)
{
    switch (h.storage) {
    case ST_F32: return in_s<ST_F32>(h, f, m, s);
    case ST_F16_DEV: return in_s<ST_F16_DEV>(h, f, m, s);
    case ST_BF16_DEV: return in_s<ST_BF16_DEV>(h, f, m, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_moment_step(const HostPhys &h, const MomentPlan &q, const void *in, void *out, cudaStream_t s)
{
    return tau_one(h) ? moment_step_t<COLL_EQ>(h, q, in, out, s) : moment_step_t<COLL_REG>(h, q, in, out, s);
}

cudaError_t launch_moment_out(const HostPhys &h, const void *m, void *f, cudaStream_t s)
{
    switch (h.storage) {
    case ST_F32: return out_s<ST_F32>(h, m, f, s);
    case ST_F16_DEV: return out_s<ST_F16_DEV>(h, m, f, s);
    case ST_BF16_DEV: return out_s<ST_BF16_DEV>(h, m, f, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
