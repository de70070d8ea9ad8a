// Forward-step kernels of the two-component D3Q19 Shan-Chen LBM
// (Otomo et al., arXiv:1601.01237, Sec. 2 and Sec. 4.1), plus state set-up,
// output fields and FP64 reductions.
//
// Two-kernel design:
//   k_density : f* (pull-gathered) -> rho^a(x)                     (Eq. 4)
//   k_collide : f* (pull-gathered), rho^b stencil -> f* (next)     (Eqs. 3-7, 13, 1/2/10)
// Populations are stored post-collision at their origin cell; a cell's
// pre-collision population f_i(x, t) is gathered from x - c_i (streaming is
// the gather), or is the reversed population of x itself when x - c_i lies
// behind a half-way bounce-back wall.
//
// Staircase walls (the inclined walls of Sec. 4.2) are a mask of solid sites
// (Phys::solid): links into a solid site bounce back, solid sites hold zero
// populations, and the density pass is followed by k_wall_rho_list,
// which gives each solid site next to fluid the density it presents to Eq. 13.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "collide.cuh"
#include "d3q19.cuh"
#include "lbm_internal.h"

namespace lbm {

namespace {

constexpr int kThreads = 256;

// Kernel parameters of the two-kernel step: the lattice's Phys plus the link
// flags of a solid mask (N words, bit i set when x - c_i is a solid site;
// nullptr without a mask).
template <class R>
struct PhysF : Phys<R> {
    const unsigned *links = nullptr;
};

// Neighbourhood of one cell: offsets of x-1, x, x+1 (and likewise y, z) as
// linear cell offsets with periodic wrap.  Index k = d + 1 for neighbour x + d.
struct Nbr {
    long long cell;
    long long xo[3], yo[3], zo[3];
    bool zlo_wall, zhi_wall;   // z - 1 (resp. z + 1) is a wall site
    int z;
};

template <class R>
__device__ __forceinline__ bool decode_cell(const Phys<R> &p, long long cell, Nbr &n)
{
    if (cell >= p.N) return false;
    const long long plane = (long long)p.nx * p.ny;
    int x, y, z;
    if (p.N <= 0x7fffffffLL) {   // (64-bit divisions cost more than the rest of the index arithmetic)
        const unsigned c = (unsigned)cell, pl = (unsigned)plane, nx = (unsigned)p.nx;
        const unsigned zu = c / pl, rem = c - zu * pl, yu = rem / nx;
        x = (int)(rem - yu * nx); y = (int)yu; z = (int)zu;
    } else {
        z = (int)(cell / plane);
        const long long rem = cell - (long long)z * plane;
        y = (int)(rem / p.nx);
        x = (int)(rem - (long long)y * p.nx);
    }
    n.cell = cell;
    n.z = z;
    n.xo[0] = (x == 0 ? p.nx - 1 : x - 1);
    n.xo[1] = x;
    n.xo[2] = (x == p.nx - 1 ? 0 : x + 1);
    n.yo[0] = (long long)(y == 0 ? p.ny - 1 : y - 1) * p.nx;
    n.yo[1] = (long long)y * p.nx;
    n.yo[2] = (long long)(y == p.ny - 1 ? 0 : y + 1) * p.nx;
    n.zo[0] = (long long)(z == 0 ? p.nz - 1 : z - 1) * plane;
    n.zo[1] = (long long)z * plane;
    n.zo[2] = (long long)(z == p.nz - 1 ? 0 : z + 1) * plane;
    n.zlo_wall = p.wall_z && z == 0;
    n.zhi_wall = p.wall_z && z == p.nz - 1;
    return true;
}

// Pre-collision populations of both components at one cell (streaming as a
// gather, with half-way bounce-back at z walls).
template <int S>
__device__ __forceinline__ void gather(const typename Store<S>::T *__restrict__ f,
                                       const PhysF<typename Store<S>::R> &p, const Nbr &n,
                                       typename Store<S>::R (&fa)[2][Q])
{
    using R = typename Store<S>::R;
    const unsigned lf = p.links ? __ldg(p.links + n.cell) : 0u;   // bit i: x - c_i is solid
    // reference densities of the cell (the *_REL formats code every population
    // a cell gathers relative to the cell's own stored pair; rho0 otherwise)
    R ra = p.rho0, rb = p.rho0;
    if constexpr (Store<S>::kRel) {
        const float2 rr = state_ref(f, p.ref_off)[n.cell];
        ra = rr.x; rb = rr.y;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const long long src = n.zo[1 - cz(i)] + n.yo[1 - cy(i)] + n.xo[1 - cx(i)];
        const bool wall = (cz(i) == 1 && n.zlo_wall) || (cz(i) == -1 && n.zhi_wall) || ((lf >> i) & 1u);
        const long long idx = wall ? pair_index(opp(i), n.cell, p.N) : pair_index(i, src, p.N);
        Store<S>::load2(f + idx, w<R>(i) * ra, w<R>(i) * rb, fa[0][i], fa[1][i]);
    }
}

// Interaction sum of Eqs. 7 and 13 for both density fields at one cell:
//   S^b = sum_{i != 0} w_i c_i rho^b(x + c_i),
// where a wall site contributes rho'_b = rho_b(mirror) + rho_s^b (modified
// model) or rho_s^b (point-wise potential).  The mirror of a wall site
// x + c_i across the z wall is x + c_i with its z component replaced by z.
// The sum runs over opposite neighbours, sum_{i odd} w_i c_i (r_i - r_opp(i)),
// so that the differences of nearby densities are taken first.
template <class R>
__device__ __forceinline__ void interaction_sums(const R *__restrict__ rho, const Phys<R> &p,
                                                 const Nbr &n, R (&S)[2][3])
{
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        R sx = 0, sy = 0, sz = 0;
        const R *rb = rho + (long long)b * p.N;
        R r[Q];
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const bool wall = (cz(i) == -1 && n.zlo_wall) || (cz(i) == 1 && n.zhi_wall);
            if (wall) {
                r[i] = p.rho_s[b];
                if (p.wall_mirror) r[i] += __ldg(rb + n.zo[1] + n.yo[1 + cy(i)] + n.xo[1 + cx(i)]);
            } else {
                r[i] = __ldg(rb + n.zo[1 + cz(i)] + n.yo[1 + cy(i)] + n.xo[1 + cx(i)]);
            }
        }
#pragma unroll
        for (int i = 1; i < Q; i += 2) {
            const R wr = w<R>(i) * (r[i] - r[i + 1]);
            if (cx(i) == 1) sx += wr; else if (cx(i) == -1) sx -= wr;
            if (cy(i) == 1) sy += wr; else if (cy(i) == -1) sy -= wr;
            if (cz(i) == 1) sz += wr; else if (cz(i) == -1) sz -= wr;
        }
        S[b][0] = sx; S[b][1] = sy; S[b][2] = sz;
    }
}

// Densities of both components and the mixture velocity (Eqs. 4-6); the
// momentum is summed over opposite pairs, sum_{i odd} c_i (t_i - t_opp(i)),
// t_i = f^1_i + f^2_i (the differences of nearly equal populations first).
template <class R>
__device__ __forceinline__ void local_moments(const R (&fa)[2][Q], R &r1, R &r2, R &ux, R &uy, R &uz)
{
    R rr[2], jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        R s = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) s += fa[a][i];
        rr[a] = s;
    }
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
        const R v = (fa[0][i] + fa[1][i]) - (fa[0][i + 1] + fa[1][i + 1]);
        if (cx(i) == 1) jx += v; else if (cx(i) == -1) jx -= v;
        if (cy(i) == 1) jy += v; else if (cy(i) == -1) jy -= v;
        if (cz(i) == 1) jz += v; else if (cz(i) == -1) jz -= v;
    }
    r1 = rr[0];
    r2 = rr[1];
    const R inv = R(1) / (r1 + r2);
    ux = jx * inv;
    uy = jy * inv;
    uz = jz * inv;
}

// ---------------------------------------------------------------------------
template <int S>
__global__ void __launch_bounds__(kThreads)
k_density(const typename Store<S>::T *__restrict__ f, typename Store<S>::R *__restrict__ rho,
          PhysF<typename Store<S>::R> p)
{
    using R = typename Store<S>::R;
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * kThreads + threadIdx.x, n)) return;
    if (p.solid && p.solid[n.cell]) return;   // k_wall_rho_list writes the solid sites that are read
    R fa[2][Q];
    gather<S>(f, p, n, fa);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        R s = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) s += fa[a][i];
        rho[(long long)a * p.N + n.cell] = s;
    }
}

// Link flags of a mask: bit i of cell x set when x - c_i is a solid site (so
// bit 0, x - c_0 = x, marks a solid site itself), so that the gather tests
// one word per cell instead of one byte per link.
__global__ void __launch_bounds__(kThreads)
k_link_flags(const unsigned char *__restrict__ solid, unsigned *__restrict__ links, PhysF<float> p)
{
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * kThreads + threadIdx.x, n)) return;
    unsigned f = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i)
        if (solid[n.zo[1 - cz(i)] + n.yo[1 - cy(i)] + n.xo[1 - cx(i)]]) f |= 1u << i;
    links[n.cell] = f;
}

// Mask set-up of the fused step: wall_rho = rho_s at solid sites, and the
// boundary cells of the mirror model counted (lists == nullptr) or listed
// (positions from the counters; the order of a list does not matter, every
// entry is processed on its own).
__global__ void __launch_bounds__(kThreads)
k_mask_setup(const unsigned char *__restrict__ solid, const unsigned *__restrict__ links, PhysF<float> p,
             float2 *__restrict__ wall_rho, unsigned *__restrict__ bfluid, unsigned *__restrict__ bsolid,
             unsigned long long *__restrict__ counts)
{
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * kThreads + threadIdx.x, n)) return;
    const unsigned lf = links[n.cell];
    if (!(lf & 1u)) {
        if (lf) {   // a fluid cell with a solid neighbour
            const unsigned long long k = atomicAdd(counts, 1ull);
            if (bfluid) bfluid[k] = (unsigned)n.cell;
        }
        return;
    }
    wall_rho[n.cell] = make_float2(p.rho_s[0], p.rho_s[1]);
    bool fluid_nb = false;
#pragma unroll
    for (int i = 1; i < Q; ++i)
        if (!solid[n.zo[1 + cz(i)] + n.yo[1 + cy(i)] + n.xo[1 + cx(i)]]) fluid_nb = true;
    if (fluid_nb) {
        const unsigned long long k = atomicAdd(counts + 1, 1ull);
        if (bsolid) bsolid[k] = (unsigned)n.cell;
    }
}

template <int S, int REG, int FORCE>
__global__ void __launch_bounds__(kThreads)
k_collide(const typename Store<S>::T *__restrict__ fin, typename Store<S>::T *__restrict__ fout,
          const typename Store<S>::R *__restrict__ rho, PhysF<typename Store<S>::R> p)
{
    using R = typename Store<S>::R;
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * kThreads + threadIdx.x, n)) return;
    if (p.solid && p.solid[n.cell]) {   // solid sites hold no populations
        const R e = Store<S>::kRel ? R(1) : p.rho0;   // (never read: any finite code)
#pragma unroll
        for (int i = 0; i < Q; ++i) Store<S>::store2(fout + pair_index(i, n.cell, p.N), R(0), R(0), w<R>(i) * e, w<R>(i) * e);
        if constexpr (Store<S>::kRel) state_ref(fout, p.ref_off)[n.cell] = make_float2(1.0f, 1.0f);
        return;
    }
    R fa[2][Q];
    gather<S>(fin, p, n, fa);
    R r1, r2, ux, uy, uz;
    local_moments(fa, r1, r2, ux, uy, uz);
    R Sb[2][3];
    interaction_sums(rho, p, n, Sb);
    // g^a = sum_b F^{ab} / rho^a + g_ext with F^{ab} = G^{ab} rho^a S^b (G^{aa} = 0)
    const R g1x = p.G12 * Sb[1][0] + p.gext[0], g1y = p.G12 * Sb[1][1] + p.gext[1],
            g1z = p.G12 * Sb[1][2] + p.gext[2];
    const R g2x = p.G21 * Sb[0][0] + p.gext[0], g2y = p.G21 * Sb[0][1] + p.gext[1],
            g2z = p.G21 * Sb[0][2] + p.gext[2];
    if (FORCE == FORCE_GUO) {   // common equilibrium velocity u* = u + g/2 (Eqs. 8-9)
        const R hi = R(0.5) / (r1 + r2);
        ux += (r1 * g1x + r2 * g2x) * hi;
        uy += (r1 * g1y + r2 * g2y) * hi;
        uz += (r1 * g1z + r2 * g2z) * hi;
    }
    collide<R, REG, FORCE>(fa[0], r1, ux, uy, uz, g1x, g1y, g1z, p.omega[0]);
    collide<R, REG, FORCE>(fa[1], r2, ux, uy, uz, g2x, g2y, g2z, p.omega[1]);
    if constexpr (Store<S>::kRel) {
        // each population coded relative to the density of the cell that reads
        // it next (x + c_i, or x itself across a wall); the cell's own pair is
        // its reference for the next gather
        const unsigned lf = p.links ? __ldg(p.links + n.cell) : 0u;
        const R d1 = rho[n.cell], d2 = rho[p.N + n.cell];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const bool wall = (cz(i) == -1 && n.zlo_wall) || (cz(i) == 1 && n.zhi_wall) ||
                              (i != 0 && ((lf >> opp(i)) & 1u));
            const long long dst = n.zo[1 + cz(i)] + n.yo[1 + cy(i)] + n.xo[1 + cx(i)];
            const R e1 = wall || i == 0 ? d1 : rho[dst], e2 = wall || i == 0 ? d2 : rho[p.N + dst];
            Store<S>::store2(fout + pair_index(i, n.cell, p.N), fa[0][i], fa[1][i], Store<S>::enc(w<R>(i) * e1),
                             Store<S>::enc(w<R>(i) * e2));
        }
        state_ref(fout, p.ref_off)[n.cell] = make_float2(d1, d2);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i)
            Store<S>::store2(fout + pair_index(i, n.cell, p.N), fa[0][i], fa[1][i], w<R>(i) * p.rho0, w<R>(i) * p.rho0);
    }
}

// ---------------------------------------------------------------------------
// The two-kernel step in FP64, one component of a cell per lane (LaneF64 of
// collide.cuh) and 32-bit indices (19 N < 2^32).  FP64 arithmetic is scarce on
// this GPU: a scheduler retires one FP64 warp instruction per 64 cycles, so
// the step is bound by the FP64 instructions of the busiest scheduler at every
// size (34^3: 37 us of them against 3.5 us of memory traffic).  Hence
//   - small CTAs of half-cell lanes: 256-thread CTAs of whole cells put all of a
//     34^3 lattice on 2 CTAs per busy SM, and a 64^2 one on 16 SMs;
//   - the densities are formed once, in the density pass, and the collision
//     reads its own back instead of summing them again;
//   - the collision in 3 c.v, six or seven operations per pair;
//   - warps inside a wall do no arithmetic.
// Of CTAs of 32, 64 and 128 threads the smallest leaves the least imbalance
// (34^3 39.5 / 42.7 / 42.7 us per step).  us per step before and now: 1 x 64 x 64
// 39.8 / 9.1, 1 x 300 x 300 115 / 60, 34^3 periodic 94.7 / 39.5, 128^3 2046 / 1225.
constexpr int kThreads64 = 32;

struct Nbr32 {
    unsigned cell;
    unsigned xo[3], yo[3], zo[3];
    bool zlo, zhi;   // z - 1 (z + 1) is a wall site
};

template <class P>
__device__ __forceinline__ Nbr32 neighbours32(const P &p, unsigned cell)
{
    const unsigned nx = (unsigned)p.nx, ny = (unsigned)p.ny, nz = (unsigned)p.nz, plane = nx * ny;
    const unsigned z = cell / plane, rem = cell - z * plane, y = rem / nx, x = rem - y * nx;
    Nbr32 n;
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

__device__ __forceinline__ void gather64(const double *__restrict__ f, const PhysF<double> &p, const Nbr32 &n,
                                         unsigned lf, int a, double (&v)[Q])
{
    const unsigned N32 = (unsigned)p.N;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const unsigned src = n.zo[1 - cz(i)] + n.yo[1 - cy(i)] + n.xo[1 - cx(i)];
        const bool wall = (cz(i) == 1 && n.zlo) || (cz(i) == -1 && n.zhi) || (i != 0 && ((lf >> i) & 1u));
        v[i] = __ldg(f + 2 * (size_t)(wall ? (unsigned)opp(i) * N32 + n.cell : (unsigned)i * N32 + src) + a);
    }
}

__global__ void __launch_bounds__(kThreads64)
k_density64(const double *__restrict__ f, double *__restrict__ rho, PhysF<double> p)
{
    const unsigned t = blockIdx.x * kThreads64 + threadIdx.x, cell = t >> 1;
    if (cell >= (unsigned)p.N) return;
    const unsigned lf = p.links ? __ldg(p.links + cell) : 0u;
    const int a = (int)(t & 1u);
    const Nbr32 n = neighbours32(p, cell);
    if (lf & 1u) return;   // k_wall_rho_list writes the solid sites that are read
    double v[Q];
    gather64(f, p, n, lf, a, v);
    rho[(size_t)a * (unsigned)p.N + cell] = density(v);
}

// Density that a solid site of the mask presents to the interaction sum of
// Eq. 13, written into rho after the density pass: the modified model takes
// the mean of rho^b over the site's fluid neighbours weighted by w_i (zero
// normal derivative for fields that vary along the wall normal) plus rho_s^b;
// the original model takes rho_s^b.  Over the sites next to fluid, the only ones
// that are read, one component per lane.
// PAIRS: rho holds (rho^1, rho^2) per cell instead of one array per component.
template <class R, bool PAIRS>
__global__ void __launch_bounds__(kThreads64)
k_wall_rho_list(R *__restrict__ rho, PhysF<R> p, const unsigned *__restrict__ sites, unsigned n_sites)
{
    const unsigned t = blockIdx.x * kThreads64 + threadIdx.x;
    if ((t >> 1) >= n_sites) return;
    const int a = (int)(t & 1u);
    const Nbr32 n = neighbours32(p, sites[t >> 1]);
    const unsigned lf = __ldg(p.links + n.cell);   // bit opp(i): x + c_i is solid
    auto r = [&](unsigned c) -> R & { return PAIRS ? rho[2 * (size_t)c + a] : rho[(size_t)a * (unsigned)p.N + c]; };
    R num = 0;
    int den36 = 0;
    if (p.wall_mirror) {
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            // (every neighbour is read, so that the loads are in flight together)
            const R v = r(n.zo[1 + cz(i)] + n.yo[1 + cy(i)] + n.xo[1 + cx(i)]);
            const bool fluid = !((lf >> opp(i)) & 1u);
            num += fluid ? R(k36(i)) * v : R(0);
            den36 += fluid ? k36(i) : 0;
        }
    }
    r(n.cell) = (den36 ? num / R(den36) : R(0)) + p.rho_s[a];
}

template <int KIND, int FORCE>
__global__ void __launch_bounds__(kThreads64)
k_collide64(const double *__restrict__ fin, double *__restrict__ fout, const double *__restrict__ rho, PhysF<double> p)
{
    const unsigned t = blockIdx.x * kThreads64 + threadIdx.x, N32 = (unsigned)p.N;
    // both lanes of every cell stay for the shuffles; lanes past the end repeat the last cell
    const unsigned cell = min(t >> 1, N32 - 1u);
    const bool store = (t >> 1) < N32;
    const LaneF64 c{(int)(t & 1u)};
    const Nbr32 n = neighbours32(p, cell);
    const unsigned lf = p.links ? __ldg(p.links + cell) : 0u;
    const bool solid = lf & 1u;
    double *o = fout + 2 * (size_t)cell + c.a;
    if (__all_sync(0xffffffffu, solid)) {   // inside a wall: no arithmetic
#pragma unroll
        for (int i = 0; i < Q && store; ++i) o[2 * (size_t)((unsigned)i * N32)] = 0.0;
        return;
    }
    double f[Q];
    gather64(fin, p, n, lf, c.a, f);
    double r = __ldg(rho + (size_t)c.a * N32 + cell);
    if (solid) r = 1.0;   // (nothing of a solid site's arithmetic is kept)
    const double *ro = rho + (size_t)(1 - c.a) * N32;
    const double rs = c.of(p.rho_s[1], p.rho_s[0]);   // of the other component
    double So[3];
    auto at = [&](int dx, int dy, int dz) {
        const bool wall = (dz == -1 && n.zlo) || (dz == 1 && n.zhi);
        if (wall) return p.wall_mirror ? rs + __ldg(ro + n.zo[1] + n.yo[1 + dy] + n.xo[1 + dx]) : rs;
        return __ldg(ro + n.zo[1 + dz] + n.yo[1 + dy] + n.xo[1 + dx]);
    };
    interaction<LaneF64>([&](int i) { return at(cx(i), cy(i), cz(i)) - at(-cx(i), -cy(i), -cz(i)); }, So);
    double jx, jy, jz;
    momentum(c, f, jx, jy, jz);
    RegMoments<LaneF64, KIND> mom;
    mom.of(f);
    const double inv = 1.0 / c.both(r);
    auto get = [&](int i) { return f[i]; };
    auto put = [&](int i, double v) {
        if (store) o[2 * (size_t)((unsigned)i * N32)] = solid ? 0.0 : v;
    };
    collide_cell<LaneF64, KIND, FORCE, false>(c, p, r, inv, jx * inv, jy * inv, jz * inv, So, mom, get, put);
}

// Initial populations f_i(x) = f^eq_i(rho(x), u(x)) of Eq. 3, each written where
// the first gather of cell x reads it: population i at x - c_i, or in the place
// of opp(i) at x itself where x - c_i is a wall site.  A cell's polynomials are
// formed once, opposite directions sharing them, and its densities are read
// once (a gather form had every cell's polynomials repeated by its 19 readers:
// 128^3 FP32 with u 1576 us, this one 590 us, at rest 128 / 64 us; bound by its 150 FP64 operations
// per cell).  At rest the values are the roundings of the FP64 products rho w_i.
template <int S>
__global__ void __launch_bounds__(kThreads)
k_init_feq(const double *__restrict__ rho1, const double *__restrict__ rho2, const double *__restrict__ u,
           typename Store<S>::T *__restrict__ f, PhysF<typename Store<S>::R> p)
{
    using R = typename Store<S>::R;
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * blockDim.x + threadIdx.x, n)) return;
    const unsigned lf = p.links ? __ldg(p.links + n.cell) : 0u;   // bit i: x - c_i is solid
    if (lf & 1u) {   // solid sites hold no populations
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            const R e = Store<S>::kRel ? Store<S>::enc(w<R>(j)) : w<R>(j) * p.rho0;
            Store<S>::store2(f + pair_index(j, n.cell, p.N), R(0), R(0), e, e);
        }
        if constexpr (Store<S>::kRel) state_ref(f, p.ref_off)[n.cell] = make_float2(1.0f, 1.0f);
        return;
    }
    const double r1 = rho1[n.cell], r2 = rho2[n.cell];
    // coded relative to the reader's initial density, which is this cell's
    const R e1 = Store<S>::kRel ? (R)r1 : p.rho0, e2 = Store<S>::kRel ? (R)r2 : p.rho0;
    auto put = [&](int i, R v1, R v2) {
        const bool wall = (cz(i) == 1 && n.zlo_wall) || (cz(i) == -1 && n.zhi_wall) || (i != 0 && ((lf >> i) & 1u));
        const long long at = wall ? pair_index(opp(i), n.cell, p.N)
                                  : pair_index(i, n.zo[1 - cz(i)] + n.yo[1 - cy(i)] + n.xo[1 - cx(i)], p.N);
        Store<S>::store2(f + at, v1, v2, Store<S>::enc(w<R>(i) * e1), Store<S>::enc(w<R>(i) * e2));
    };
    if constexpr (Store<S>::kRel) state_ref(f, p.ref_off)[n.cell] = make_float2((float)r1, (float)r2);
    const double a0 = r1 * wd(0), a1 = r1 * wd(1), a2 = r1 * wd(7), b0 = r2 * wd(0), b1 = r2 * wd(1), b2 = r2 * wd(7);
    if (!u) {
        const R v0 = (R)a0, v1 = (R)a1, v2 = (R)a2, w0 = (R)b0, w1 = (R)b1, w2 = (R)b2;
#pragma unroll
        for (int i = 0; i < Q; ++i) put(i, i == 0 ? v0 : (i < 7 ? v1 : v2), i == 0 ? w0 : (i < 7 ? w1 : w2));
        return;
    }
    const double ux = u[3 * n.cell], uy = u[3 * n.cell + 1], uz = u[3 * n.cell + 2];
    const double A = 1.0 - 1.5 * (ux * ux + uy * uy + uz * uz);
    put(0, (R)(a0 * A), (R)(b0 * A));
    const double sx = 3.0 * ux, sy = 3.0 * uy, sz = 3.0 * uz;
#pragma unroll
    for (int i = 1; i < Q; i += 2) {   // f^eq_+- / (rho w) = A + s^2/2 +- s (A + s^2/6), s = 3 c.u
        const double s = vdot(i, sx, sy, sz), m = s * s;
        const double E = fma(m, 0.5, A), O = s * fma(m, 1.0 / 6.0, A);
        const double a = i < 7 ? a1 : a2, b = i < 7 ? b1 : b2;
        put(i, (R)(a * (E + O)), (R)(b * (E + O)));
        put(i + 1, (R)(a * (E - O)), (R)(b * (E - O)));
    }
}

// Reference densities of a state set from explicit populations (the *_REL
// formats): each cell's densities sum_i f_i^a of the given populations
// (solid sites: 1, never read).
template <int S>
__global__ void __launch_bounds__(kThreads)
k_set_ref(const double *__restrict__ src, typename Store<S>::T *__restrict__ f, PhysF<typename Store<S>::R> p)
{
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * kThreads + threadIdx.x, n)) return;
    float2 r = make_float2(1.0f, 1.0f);
    if (!(p.solid && p.solid[n.cell])) {
        double a = 0, b = 0;
        for (int k = 0; k < Q; ++k) {
            a += src[(long long)k * p.N + n.cell];
            b += src[(long long)(Q + k) * p.N + n.cell];
        }
        r = make_float2((float)a, (float)b);
    }
    state_ref(f, p.ref_off)[n.cell] = r;
}

template <int S>
__global__ void __launch_bounds__(kThreads)
k_set_pop(const double *__restrict__ src, typename Store<S>::T *__restrict__ f,
          PhysF<typename Store<S>::R> p)
{
    using R = typename Store<S>::R;
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * kThreads + threadIdx.x, n)) return;
    const bool here_solid = p.solid && p.solid[n.cell];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            const long long dst = n.zo[1 + cz(j)] + n.yo[1 + cy(j)] + n.xo[1 + cx(j)];
            const bool wall = (cz(j) == -1 && n.zlo_wall) || (cz(j) == 1 && n.zhi_wall) ||
                              (j != 0 && p.solid && p.solid[dst]);
            const long long sc = wall ? n.cell : dst;
            const int k = wall ? opp(j) : j;
            R e = p.rho0;   // *_REL: the reader's reference (written by k_set_ref)
            if constexpr (Store<S>::kRel) {
                const float2 rr = state_ref(f, p.ref_off)[sc];
                e = here_solid ? R(1) : (a == 0 ? rr.x : rr.y);
            }
            Store<S>::store(f + pair_index(j, n.cell, p.N) + a,
                            here_solid ? R(0) : (R)src[(long long)(a * Q + k) * p.N + sc], Store<S>::enc(w<R>(j) * e));
        }
}

template <int S>
__global__ void __launch_bounds__(kThreads)
k_get_pop(const typename Store<S>::T *__restrict__ f, double *__restrict__ dst,
          PhysF<typename Store<S>::R> p)
{
    using R = typename Store<S>::R;
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * kThreads + threadIdx.x, n)) return;
    const bool here_solid = p.solid && p.solid[n.cell];
    R fa[2][Q];
    gather<S>(f, p, n, fa);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int i = 0; i < Q; ++i) dst[(long long)(a * Q + i) * p.N + n.cell] = here_solid ? 0.0 : (double)fa[a][i];
}

// Velocity of Eq. 8: u_F = u + g/2 with g = sum_a g^a rho^a / rho (Eq. 9).
template <class R>
__device__ __forceinline__ void velocity_uF(const Phys<R> &p, R r1, R r2, R ux, R uy, R uz,
                                            const R (&Sb)[2][3], R &fx, R &fy, R &fz)
{
    const R g1[3] = {p.G12 * Sb[1][0] + p.gext[0], p.G12 * Sb[1][1] + p.gext[1], p.G12 * Sb[1][2] + p.gext[2]};
    const R g2[3] = {p.G21 * Sb[0][0] + p.gext[0], p.G21 * Sb[0][1] + p.gext[1], p.G21 * Sb[0][2] + p.gext[2]};
    const R half_inv = R(0.5) / (r1 + r2);
    fx = ux + (g1[0] * r1 + g2[0] * r2) * half_inv;
    fy = uy + (g1[1] * r1 + g2[1] * r2) * half_inv;
    fz = uz + (g1[2] * r1 + g2[2] * r2) * half_inv;
}

// Output fields and reductions run in two passes: this one gathers every cell
// once and leaves its densities (as pairs, where the second pass needs them,
// and the output fields o1, o2) and its velocity u = j / rho (three planes
// behind each other); the second one adds the force from the densities'
// stencil.  u lies in the state copy that is free between steps.  (One pass that
// gathered again beside a density pass took 1.54 ms for the fields at 256^3
// FP32, these two 0.68 ms against a floor of 0.43; pairs instead of one array
// per component halve the second pass's 36 stencil loads.)
template <class R> struct VecOf;
template <> struct VecOf<float> { using T = float2; };
template <> struct VecOf<double> { using T = double2; };

template <int S, class O>
__global__ void __launch_bounds__(kThreads)
k_sums(const typename Store<S>::T *__restrict__ f, typename VecOf<typename Store<S>::R>::T *__restrict__ rho,
       typename Store<S>::R *__restrict__ u, O *__restrict__ o1, O *__restrict__ o2, PhysF<typename Store<S>::R> p)
{
    using R = typename Store<S>::R;
    Nbr n;
    if (!decode_cell(p, (long long)blockIdx.x * blockDim.x + threadIdx.x, n)) return;
    if (p.solid && p.solid[n.cell]) {   // no fluid at a solid site
        if (o1) o1[n.cell] = (O)0;
        if (o2) o2[n.cell] = (O)0;
        return;
    }
    R fa[2][Q];
    gather<S>(f, p, n, fa);
    R r1, r2, ux, uy, uz;
    local_moments(fa, r1, r2, ux, uy, uz);
    if (o1) o1[n.cell] = (O)r1;
    if (o2) o2[n.cell] = (O)r2;
    if (rho) {
        typename VecOf<R>::T v;
        v.x = r1;
        v.y = r2;
        rho[n.cell] = v;
        u[n.cell] = ux;
        u[p.N + n.cell] = uy;
        u[2 * p.N + n.cell] = uz;
    }
}

// The same in FP64 with one component per lane.
template <class O>
__global__ void __launch_bounds__(kThreads64)
k_sums64(const double *__restrict__ f, double *__restrict__ rho, double *__restrict__ u, O *__restrict__ o1,
         O *__restrict__ o2, PhysF<double> p)
{
    const unsigned t = blockIdx.x * kThreads64 + threadIdx.x, N32 = (unsigned)p.N;
    const unsigned cell = min(t >> 1, N32 - 1u);
    const bool store = (t >> 1) < N32;
    const LaneF64 c{(int)(t & 1u)};
    O *o = c.a ? o2 : o1;
    const unsigned lf = p.links ? __ldg(p.links + cell) : 0u;
    double v[Q];
    gather64(f, p, neighbours32(p, cell), lf, c.a, v);
    const double r = density(v);
    if (o && store) o[cell] = (lf & 1u) ? (O)0 : (O)r;
    if (!rho) return;
    double jx, jy, jz;
    momentum(c, v, jx, jy, jz);
    const double inv = 1.0 / c.both(r);
    if (!store || (lf & 1u)) return;
    rho[2 * (size_t)cell + c.a] = r;
    if (c.a == 0) {
        u[cell] = jx * inv;
        u[(size_t)N32 + cell] = jy * inv;
    } else {
        u[2 * (size_t)N32 + cell] = jz * inv;
    }
}

// u_F = u + g / 2 of one cell from the first pass (Eqs. 8-9), with the
// interaction sums of Eqs. 7 and 13 over opposite neighbours as interaction_sums.
template <class R>
__device__ __forceinline__ void velocity_of(const typename VecOf<R>::T *__restrict__ rho, const R *__restrict__ u,
                                            const PhysF<R> &p, const Nbr32 &n, R &r1, R &r2, R &fx, R &fy, R &fz)
{
    using V = typename VecOf<R>::T;
    auto at = [&](int dx, int dy, int dz) {
        V v;
        if ((dz == -1 && n.zlo) || (dz == 1 && n.zhi)) {   // a wall site: its mirror cell's and rho_s, or rho_s
            v.x = p.rho_s[0];
            v.y = p.rho_s[1];
            if (p.wall_mirror) {
                const V m = __ldg(rho + n.zo[1] + n.yo[1 + dy] + n.xo[1 + dx]);
                v.x += m.x;
                v.y += m.y;
            }
        } else {
            v = __ldg(rho + n.zo[1 + dz] + n.yo[1 + dy] + n.xo[1 + dx]);
        }
        return v;
    };
    R Sb[2][3] = {{0, 0, 0}, {0, 0, 0}};
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
        const V a = at(cx(i), cy(i), cz(i)), b = at(-cx(i), -cy(i), -cz(i));
        const R d1 = w<R>(i) * (a.x - b.x), d2 = w<R>(i) * (a.y - b.y);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (ca(i, d) == 1) { Sb[0][d] += d1; Sb[1][d] += d2; }
            else if (ca(i, d) == -1) { Sb[0][d] -= d1; Sb[1][d] -= d2; }
        }
    }
    const V own = rho[n.cell];
    const size_t N = (size_t)p.N;
    r1 = own.x;
    r2 = own.y;
    velocity_uF(p, r1, r2, u[n.cell], u[N + n.cell], u[2 * N + n.cell], Sb, fx, fy, fz);
}

// The three components of a cell's u_F lie side by side in the output; a CTA's
// are put in order in shared memory and stored in whole rows.
template <class R, class O>
__global__ void __launch_bounds__(kThreads)
k_uF(const typename VecOf<R>::T *__restrict__ rho, const R *__restrict__ u, O *__restrict__ ouF, PhysF<R> p)
{
    __shared__ O sh[3 * kThreads];
    const unsigned c0 = blockIdx.x * blockDim.x, N32 = (unsigned)p.N, cell = c0 + threadIdx.x;
    R fx = 0, fy = 0, fz = 0;
    if (cell < N32 && !(p.solid && p.solid[cell])) {
        R r1, r2;
        velocity_of<R>(rho, u, p, neighbours32(p, cell), r1, r2, fx, fy, fz);
    }
    sh[3 * threadIdx.x] = (O)fx;
    sh[3 * threadIdx.x + 1] = (O)fy;
    sh[3 * threadIdx.x + 2] = (O)fz;
    __syncthreads();
    const unsigned m = 3 * min(blockDim.x, N32 - c0);
    O *out = ouF + 3 * (size_t)c0;
    for (unsigned k = threadIdx.x; k < m; k += blockDim.x) out[k] = sh[k];
}

constexpr int kReduceBlocks = 1216;   // 152 SMs x 8

template <class R>
__global__ void __launch_bounds__(kThreads, 4)
k_reduce(const typename VecOf<R>::T *__restrict__ rho, const R *__restrict__ u, double *__restrict__ partials,
         PhysF<R> p)
{
    double acc[6] = {0, 0, 0, 0, 0, 0};
    unsigned bad = 0;
    R top = 0;   // acc[5] in the arithmetic type
    const unsigned N32 = (unsigned)p.N;
    for (unsigned c = blockIdx.x * kThreads + threadIdx.x; c < N32; c += gridDim.x * kThreads) {
        if (p.solid && p.solid[c]) continue;   // solid sites hold no fluid
        R r1, r2, fx, fy, fz;
        velocity_of<R>(rho, u, p, neighbours32(p, c), r1, r2, fx, fy, fz);
        const double rho_t = (double)r1 + (double)r2;
        if (!(r1 > R(0)) || !(r2 > R(0)) || !isfinite(r1) || !isfinite(r2)) ++bad;
        acc[0] += (double)r1;
        acc[1] += (double)r2;
        acc[2] += rho_t * (double)fx;
        acc[3] += rho_t * (double)fy;
        acc[4] += rho_t * (double)fz;
        // max |u_F|^2; the host takes the square root of the maximum, which
        // equals the maximum of the (correctly rounded, monotonic) roots.  The
        // FP64 square is formed only where the rounded one can exceed the
        // maximum so far.
        const R q = fx * fx + fy * fy + fz * fz;
        if (!(q * R(1.00001) < top) || top < R(1e-30)) {
            acc[5] = fmax(acc[5], (double)fx * fx + (double)fy * fy + (double)fz * fz);
            top = (R)acc[5];
        }
    }
    // fixed-order block reduction (deterministic)
    __shared__ double sh[7][kThreads];
    for (int k = 0; k < 6; ++k) sh[k][threadIdx.x] = acc[k];
    sh[6][threadIdx.x] = (double)bad;
    __syncthreads();
    for (int stride = kThreads / 2; stride > 0; stride >>= 1) {
        if (threadIdx.x < stride) {
            for (int k = 0; k < 7; ++k) {
                if (k == 5)
                    sh[k][threadIdx.x] = fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + stride]);
                else
                    sh[k][threadIdx.x] += sh[k][threadIdx.x + stride];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x < 7) partials[(long long)blockIdx.x * 8 + threadIdx.x] = sh[threadIdx.x][0];
    if (threadIdx.x == 7) partials[(long long)blockIdx.x * 8 + 7] = 0.0;
}

template <class R>
PhysF<R> make_phys(const HostPhys &h)
{
    PhysF<R> p;
    p.nx = h.nx; p.ny = h.ny; p.nz = h.nz; p.N = h.N;
    p.wall_z = h.wall_z;
    p.wall_mirror = h.wall_mirror;
    p.omega[0] = (R)(1.0 / h.tau[0]);
    p.omega[1] = (R)(1.0 / h.tau[1]);
    p.G12 = (R)h.G12; p.G21 = (R)h.G21;
    for (int d = 0; d < 3; ++d) p.gext[d] = (R)h.gext[d];
    p.rho_s[0] = (R)h.rho_s[0]; p.rho_s[1] = (R)h.rho_s[1];
    p.rho0 = (R)h.rho0;
    p.solid = h.solid;
    p.links = h.links;
    p.ref_off = h.ref_off;
    return p;
}

inline unsigned grid_for(long long N) { return (unsigned)((N + kThreads - 1) / kThreads); }

// FP64 lattices that the half-cell kernels take: 32-bit element indices (and,
// with a mask, the lists of its boundary, which lbm_set_solid makes).
inline bool lanes64(const HostPhys &h) { return (long long)Q * h.N < (1LL << 32) && (!h.links || h.bsolid); }
inline unsigned grid64(long long cells) { return (unsigned)((2 * cells + kThreads64 - 1) / kThreads64); }

// Densities that the solid sites of a mask present to Eq. 13, into rho.
template <class R, bool PAIRS>
void wall_pass(const HostPhys &h, R *rho, const PhysF<R> &p, cudaStream_t s)
{
    if (h.n_bsolid > 0)
        k_wall_rho_list<R, PAIRS><<<grid64(h.n_bsolid), kThreads64, 0, s>>>(rho, p, h.bsolid, (unsigned)h.n_bsolid);
}

// Threads per CTA of the one-thread-per-cell kernels that run once per call:
// CTAs of 64 spread a small lattice over more SMs (FP64 above all).
inline int threads_for(long long N) { return N < 152LL * 4 * kThreads ? 64 : kThreads; }
inline unsigned grid_by(long long N, int threads) { return (unsigned)((N + threads - 1) / threads); }

// Density pass: rho^a of every fluid cell, then (with a mask) the densities
// the solid sites present to Eq. 13.
template <int S>
void density_pass(const HostPhys &h, const typename Store<S>::T *f, typename Store<S>::R *rho, cudaStream_t s)
{
    using R = typename Store<S>::R;
    const PhysF<R> p = make_phys<R>(h);
    bool lanes = false;
    if constexpr (S == ST_F64) {
        lanes = lanes64(h);
        if (lanes) k_density64<<<grid64(h.N), kThreads64, 0, s>>>(f, rho, p);
    }
    if (!lanes) k_density<S><<<grid_for(h.N), kThreads, 0, s>>>(f, rho, p);
    if (h.solid) wall_pass<R, false>(h, rho, p, s);
}

template <int S>
cudaError_t step_split_t(const HostPhys &h, const void *fin, void *fout, void *rho, cudaStream_t s,
                         cudaEvent_t *ev)
{
    using T = typename Store<S>::T;
    using R = typename Store<S>::R;
    const PhysF<R> p = make_phys<R>(h);
    const unsigned g = grid_for(h.N);
    if (ev) cudaEventRecord(ev[0], s);
    density_pass<S>(h, (const T *)fin, (R *)rho, s);
    if (ev) cudaEventRecord(ev[1], s);
    if constexpr (S == ST_F64) {
        if (lanes64(h)) {
            const unsigned g64 = grid64(h.N);
            const bool guo = h.forcing == FORCE_GUO;
#define LBM_COLLIDE64(K_)                                                                                            \
    do {                                                                                                             \
        if (guo) k_collide64<K_, FORCE_GUO><<<g64, kThreads64, 0, s>>>((const T *)fin, (T *)fout, (const R *)rho, p); \
        else k_collide64<K_, FORCE_EDM><<<g64, kThreads64, 0, s>>>((const T *)fin, (T *)fout, (const R *)rho, p);     \
    } while (0)
            if (h.tau[0] == 1.0 && h.tau[1] == 1.0) LBM_COLLIDE64(COLL_EQ);
            else if (h.collision == LBM_REGULARIZED) LBM_COLLIDE64(COLL_REG);
            else if (h.collision == LBM_REGULARIZED3) LBM_COLLIDE64(COLL_REG3);
            else LBM_COLLIDE64(COLL_BGK);
#undef LBM_COLLIDE64
            if (ev) cudaEventRecord(ev[2], s);
            return cudaGetLastError();
        }
    }
#define LBM_COLLIDE(REG_, F_) k_collide<S, REG_, F_><<<g, kThreads, 0, s>>>((const T *)fin, (T *)fout, (const R *)rho, p)
    const int reg = h.collision == LBM_REGULARIZED ? 1 : (h.collision == LBM_REGULARIZED3 ? 2 : 0);
    if (h.forcing == FORCE_GUO) {
        if (reg == 1) LBM_COLLIDE(1, FORCE_GUO); else if (reg == 2) LBM_COLLIDE(2, FORCE_GUO); else LBM_COLLIDE(0, FORCE_GUO);
    } else {
        if (reg == 1) LBM_COLLIDE(1, FORCE_EDM); else if (reg == 2) LBM_COLLIDE(2, FORCE_EDM); else LBM_COLLIDE(0, FORCE_EDM);
    }
#undef LBM_COLLIDE
    if (ev) cudaEventRecord(ev[2], s);
    return cudaGetLastError();
}

template <int S>
cudaError_t init_t(const HostPhys &h, const double *r1, const double *r2, const double *u, void *f, cudaStream_t s)
{
    const int t = threads_for(h.N);
    k_init_feq<S><<<grid_by(h.N, t), t, 0, s>>>(r1, r2, u, (typename Store<S>::T *)f, make_phys<typename Store<S>::R>(h));
    return cudaGetLastError();
}

template <int S>
cudaError_t setpop_t(const HostPhys &h, const double *src, void *f, cudaStream_t s)
{
    using T = typename Store<S>::T;
    using R = typename Store<S>::R;
    if constexpr (Store<S>::kRel) k_set_ref<S><<<grid_for(h.N), kThreads, 0, s>>>(src, (T *)f, make_phys<R>(h));
    k_set_pop<S><<<grid_for(h.N), kThreads, 0, s>>>(src, (T *)f, make_phys<R>(h));
    return cudaGetLastError();
}

template <int S>
cudaError_t getpop_t(const HostPhys &h, const void *f, double *dst, cudaStream_t s)
{
    using T = typename Store<S>::T;
    using R = typename Store<S>::R;
    k_get_pop<S><<<grid_for(h.N), kThreads, 0, s>>>((const T *)f, dst, make_phys<R>(h));
    return cudaGetLastError();
}

// First pass of the output fields and reductions; with rho also the densities of
// the solid sites.
template <int S, class O>
void sums_pass(const HostPhys &h, const void *f, typename Store<S>::R *rho, typename Store<S>::R *u, O *o1, O *o2,
               cudaStream_t s)
{
    using R = typename Store<S>::R;
    const PhysF<R> p = make_phys<R>(h);
    bool lanes = false;
    if constexpr (S == ST_F64) {
        lanes = lanes64(h);
        if (lanes) k_sums64<O><<<grid64(h.N), kThreads64, 0, s>>>((const double *)f, rho, u, o1, o2, p);
    }
    if (!lanes) {
        const int t = threads_for(h.N);
        k_sums<S, O><<<grid_by(h.N, t), t, 0, s>>>((const typename Store<S>::T *)f, (typename VecOf<R>::T *)rho, u, o1, o2, p);
    }
    if (rho && h.solid) wall_pass<R, true>(h, rho, p, s);
}

template <int S, class O>
void fields_t(const HostPhys &h, const void *f, void *rho, void *u, O *o1, O *o2, O *ouF, cudaStream_t s)
{
    using R = typename Store<S>::R;
    sums_pass<S, O>(h, f, ouF ? (R *)rho : nullptr, (R *)u, o1, o2, s);
    if (!ouF) return;
    const int t = threads_for(h.N);
    k_uF<R, O><<<grid_by(h.N, t), t, 0, s>>>((const typename VecOf<R>::T *)rho, (const R *)u, ouF, make_phys<R>(h));
}

template <int S>
cudaError_t moments_t(const HostPhys &h, const void *f, void *rho, void *u, int out_f64, void *o1, void *o2,
                      void *ouF, cudaStream_t s)
{
    if (out_f64) fields_t<S, double>(h, f, rho, u, (double *)o1, (double *)o2, (double *)ouF, s);
    else fields_t<S, float>(h, f, rho, u, (float *)o1, (float *)o2, (float *)ouF, s);
    return cudaGetLastError();
}

template <int S>
cudaError_t reduce_t(const HostPhys &h, const void *f, void *rho, void *u, double *partials, cudaStream_t s)
{
    using R = typename Store<S>::R;
    sums_pass<S, R>(h, f, (R *)rho, (R *)u, nullptr, nullptr, s);
    k_reduce<R><<<reduce_grid(h.N), kThreads, 0, s>>>((const typename VecOf<R>::T *)rho, (const R *)u, partials, make_phys<R>(h));
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_step_split(const HostPhys &p, const void *f_in, void *f_out, void *rho, cudaStream_t s,
                              cudaEvent_t *ev)
{
    switch (p.storage) {
    case ST_F64: return step_split_t<ST_F64>(p, f_in, f_out, rho, s, ev);
    case ST_F32: return step_split_t<ST_F32>(p, f_in, f_out, rho, s, ev);
    case ST_F16_DEV: return step_split_t<ST_F16_DEV>(p, f_in, f_out, rho, s, ev);
    case ST_BF16_DEV: return step_split_t<ST_BF16_DEV>(p, f_in, f_out, rho, s, ev);
    case ST_F16_REL: return step_split_t<ST_F16_REL>(p, f_in, f_out, rho, s, ev);
    case ST_BF16_REL: return step_split_t<ST_BF16_REL>(p, f_in, f_out, rho, s, ev);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_init_feq(const HostPhys &p, const double *r1, const double *r2, const double *u,
                            void *f, cudaStream_t s)
{
    switch (p.storage) {
    case ST_F64: return init_t<ST_F64>(p, r1, r2, u, f, s);
    case ST_F32: return init_t<ST_F32>(p, r1, r2, u, f, s);
    case ST_F16_DEV: return init_t<ST_F16_DEV>(p, r1, r2, u, f, s);
    case ST_BF16_DEV: return init_t<ST_BF16_DEV>(p, r1, r2, u, f, s);
    case ST_F16_REL: return init_t<ST_F16_REL>(p, r1, r2, u, f, s);
    case ST_BF16_REL: return init_t<ST_BF16_REL>(p, r1, r2, u, f, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_set_populations(const HostPhys &p, const double *src, void *f, cudaStream_t s)
{
    switch (p.storage) {
    case ST_F64: return setpop_t<ST_F64>(p, src, f, s);
    case ST_F32: return setpop_t<ST_F32>(p, src, f, s);
    case ST_F16_DEV: return setpop_t<ST_F16_DEV>(p, src, f, s);
    case ST_BF16_DEV: return setpop_t<ST_BF16_DEV>(p, src, f, s);
    case ST_F16_REL: return setpop_t<ST_F16_REL>(p, src, f, s);
    case ST_BF16_REL: return setpop_t<ST_BF16_REL>(p, src, f, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_get_populations(const HostPhys &p, const void *f, double *dst, cudaStream_t s)
{
    switch (p.storage) {
    case ST_F64: return getpop_t<ST_F64>(p, f, dst, s);
    case ST_F32: return getpop_t<ST_F32>(p, f, dst, s);
    case ST_F16_DEV: return getpop_t<ST_F16_DEV>(p, f, dst, s);
    case ST_BF16_DEV: return getpop_t<ST_BF16_DEV>(p, f, dst, s);
    case ST_F16_REL: return getpop_t<ST_F16_REL>(p, f, dst, s);
    case ST_BF16_REL: return getpop_t<ST_BF16_REL>(p, f, dst, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_moments(const HostPhys &p, const void *f, void *rho, void *u, int out_f64, void *o1, void *o2,
                           void *ouF, cudaStream_t s)
{
    switch (p.storage) {
    case ST_F64: return moments_t<ST_F64>(p, f, rho, u, out_f64, o1, o2, ouF, s);
    case ST_F32: return moments_t<ST_F32>(p, f, rho, u, out_f64, o1, o2, ouF, s);
    case ST_F16_DEV: return moments_t<ST_F16_DEV>(p, f, rho, u, out_f64, o1, o2, ouF, s);
    case ST_BF16_DEV: return moments_t<ST_BF16_DEV>(p, f, rho, u, out_f64, o1, o2, ouF, s);
    case ST_F16_REL: return moments_t<ST_F16_REL>(p, f, rho, u, out_f64, o1, o2, ouF, s);
    case ST_BF16_REL: return moments_t<ST_BF16_REL>(p, f, rho, u, out_f64, o1, o2, ouF, s);
    default: return cudaErrorInvalidValue;
    }
}

int reduce_blocks() { return kReduceBlocks; }
int reduce_grid(long long N) { return (int)(N < (long long)kReduceBlocks * kThreads ? (N + kThreads - 1) / kThreads : kReduceBlocks); }

cudaError_t launch_mask_setup(const HostPhys &h, const unsigned char *solid, float *wall_rho, unsigned *bfluid,
                              unsigned *bsolid, unsigned long long *counts, cudaStream_t s)
{
    k_mask_setup<<<grid_for(h.N), kThreads, 0, s>>>(solid, h.links, make_phys<float>(h), (float2 *)wall_rho, bfluid,
                                                     bsolid, counts);
    return cudaGetLastError();
}

cudaError_t launch_link_flags(const HostPhys &h, const unsigned char *solid, unsigned *links, cudaStream_t s)
{
    k_link_flags<<<grid_for(h.N), kThreads, 0, s>>>(solid, links, make_phys<float>(h));
    return cudaGetLastError();
}

cudaError_t launch_density(const HostPhys &h, const void *f, void *rho, cudaStream_t s)
{
    switch (h.storage) {
    case ST_F64: density_pass<ST_F64>(h, (const double *)f, (double *)rho, s); break;
    case ST_F32: density_pass<ST_F32>(h, (const float *)f, (float *)rho, s); break;
    case ST_F16_DEV: density_pass<ST_F16_DEV>(h, (const __half *)f, (float *)rho, s); break;
    case ST_BF16_DEV: density_pass<ST_BF16_DEV>(h, (const __nv_bfloat16 *)f, (float *)rho, s); break;
    case ST_F16_REL: density_pass<ST_F16_REL>(h, (const __half *)f, (float *)rho, s); break;
    case ST_BF16_REL: density_pass<ST_BF16_REL>(h, (const __nv_bfloat16 *)f, (float *)rho, s); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_reduce(const HostPhys &p, const void *f, void *rho, void *u, double *partials, cudaStream_t s)
{
    switch (p.storage) {
    case ST_F64: return reduce_t<ST_F64>(p, f, rho, u, partials, s);
    case ST_F32: return reduce_t<ST_F32>(p, f, rho, u, partials, s);
    case ST_F16_DEV: return reduce_t<ST_F16_DEV>(p, f, rho, u, partials, s);
    case ST_BF16_DEV: return reduce_t<ST_BF16_DEV>(p, f, rho, u, partials, s);
    case ST_F16_REL: return reduce_t<ST_F16_REL>(p, f, rho, u, partials, s);
    case ST_BF16_REL: return reduce_t<ST_BF16_REL>(p, f, rho, u, partials, s);
    default: return cudaErrorInvalidValue;
    }
}

size_t storage_bytes(int storage)
{
    switch (storage) {
    case ST_F64: return 8;
    case ST_F32: return 4;
    default: return 2;
    }
}

bool storage_is_rel(int storage) { return storage == ST_F16_REL || storage == ST_BF16_REL; }

size_t ref_offset(int storage, long long N)
{
    if (!storage_is_rel(storage)) return 0;
    const size_t pop = (size_t)2 * Q * (size_t)N * storage_bytes(storage);
    return (pop + 255) / 256 * 256;
}

size_t state_bytes(int storage, long long N)
{
    const size_t pop = (size_t)2 * Q * (size_t)N * storage_bytes(storage);
    return storage_is_rel(storage) ? ref_offset(storage, N) + sizeof(float) * 2 * (size_t)N : pop;
}

size_t real_bytes(int storage) { return storage == ST_F64 ? 8 : 4; }

namespace {
constexpr int kMaxSmDevices = 64;
std::atomic<int> g_device_sms[kMaxSmDevices];   // 0 = not looked up yet
}  // namespace

int current_device_sms()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 152;
    if (dev < 0 || dev >= kMaxSmDevices) {   // beyond the table: look it up every time
        int n = 0;
        return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0 ? n : 152;
    }
    int n = g_device_sms[dev].load(std::memory_order_acquire);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 152;
    g_device_sms[dev].store(n, std::memory_order_release);
    return n;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the two-kernel step.  Its density scratch is a
// file-scope device array (2 components x kNoallocMaxCells x 8 bytes = 32 MiB),
// present on every device that loads the library.  Host code cannot use the
// array's name as a device address, so the address is looked up once per
// device with cudaGetSymbolAddress while that device is current.
static __device__ __align__(256) unsigned char g_noalloc_rho[2 * kNoallocMaxCells * sizeof(double)];

namespace {

constexpr int kMaxDevices = 64;
void *g_noalloc_ptr[kMaxDevices] = {};

cudaError_t noalloc_scratch(void **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    void *ptr = __atomic_load_n(&g_noalloc_ptr[dev], __ATOMIC_ACQUIRE);
    if (!ptr) {
        e = cudaGetSymbolAddress(&ptr, g_noalloc_rho);
        if (e != cudaSuccess) return e;
        __atomic_store_n(&g_noalloc_ptr[dev], ptr, __ATOMIC_RELEASE);
    }
    *out = ptr;
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_step_split_noalloc(const HostPhys &p, const void *f_in, void *f_out, cudaStream_t s)
{
    if (p.N > kNoallocMaxCells) return cudaErrorInvalidValue;
    void *rho = nullptr;
    cudaError_t e = noalloc_scratch(&rho);
    if (e != cudaSuccess) return e;
    return launch_step_split(p, f_in, f_out, rho, s);
}

}  // namespace lbm
