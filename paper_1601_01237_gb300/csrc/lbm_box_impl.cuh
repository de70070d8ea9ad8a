// Single-pass time step of small and thin lattices (kernel template;
// instantiated per storage format in lbm_box_<format>.cu).
//
// The marching kernel (lbm_fused_impl.cuh) pays for its low traffic with a
// serial chain of planes and 32 x 8 tiles: a quasi-2D lattice of 160 x 64 cells
// (ny = 1) gives it 40 CTAs whose rows are all images of one row, each marching
// 10 planes, and a 64^2 one 16 CTAs.  Such lattices live in L2 and are bound by
// the length of that chain, so here every cell has its own thread and nothing
// marches: a CTA takes a box of cells, each thread gathers its cell's
// populations (19 paired loads in flight at once), the CTA gathers the
// one-cell halo of the box for its densities alone, and after one barrier every
// thread forms the interaction sums from the densities in shared memory and
// collides its cell from registers.  The halo is gathered again by each
// neighbouring box (8 x 8: 1.6 gathers per cell, 8 x 8 x 4: 2.3), from L2.
//
// FP32, us per step in a long run, the marching step and this one: 64 x 1 x 160
// with z walls 14.7 / 2.7, 1 x 80 x 80 5.9 / 2.2, 1 x 700 x 700 56 / 29,
// 300 x 1 x 600 41 / 10, 24^3 18.5 / 4.9, 48^3 19.5 / 10.5, 64^3 19.8 / 22.6.
// What is left of the small ones is two dependent L2 round trips (gathers and
// stores) and the launch; the larger ones are bound by the L2 reads of the halo.
//
// Successive steps are launched with programmatic stream serialization: a
// step's CTAs are set up while the previous step drains and wait for it with
// griddepcontrol.wait before their first access (without it: 64 x 1 x 160 3.0 us,
// 80 x 80 2.7, 48^3 11.1).
#pragma once

#include <cuda_runtime.h>

#include "collide.cuh"
#include "d3q19.cuh"
#include "lbm_internal.h"

namespace lbm {
namespace box {

// Tile shapes.  FY / FZ: the y (z) direction is one periodic layer, which is its
// own neighbour, so the box has no halo along it.
struct TileXY { static constexpr int TX = 8, TY = 8, TZ = 1; static constexpr bool FY = false, FZ = true; };
struct TileXZ { static constexpr int TX = 8, TY = 1, TZ = 8; static constexpr bool FY = true, FZ = false; };
struct Tile3D { static constexpr int TX = 8, TY = 8, TZ = 4; static constexpr bool FY = false, FZ = false; };

// Where a box cell lies: offsets of its neighbours, and what its density is.
struct Site {
    int xo[3], yo[3], zo[3];   // x-1, x, x+1; (y-1, y, y+1) nx; (z-1, z, z+1) nx ny
    bool zlo, zhi;             // half-way wall below / above the (mirror) cell
    bool ghost;                // a wall site: its density is the mirror cell's + rho_s, or rho_s
};

template <class T>
__device__ __forceinline__ Site site_at(const Phys<float> &p, int gx, int gy, int gz)
{
    Site s;
    const int nx = p.nx, ny = p.ny, nz = p.nz, plane = nx * ny;
    gx = gx < 0 ? gx + nx : (gx >= nx ? gx % nx : gx);
    s.xo[0] = gx == 0 ? nx - 1 : gx - 1;
    s.xo[1] = gx;
    s.xo[2] = gx == nx - 1 ? 0 : gx + 1;
    if (T::FY) {
        s.yo[0] = s.yo[1] = s.yo[2] = 0;
    } else {
        gy = gy < 0 ? gy + ny : (gy >= ny ? gy % ny : gy);
        s.yo[0] = (gy == 0 ? ny - 1 : gy - 1) * nx;
        s.yo[1] = gy * nx;
        s.yo[2] = (gy == ny - 1 ? 0 : gy + 1) * nx;
    }
    s.ghost = false;
    s.zlo = s.zhi = false;
    if (T::FZ) {
        s.zo[0] = s.zo[1] = s.zo[2] = 0;
    } else {
        if (p.wall_z) {
            s.ghost = gz < 0 || gz >= nz;
            gz = gz < 0 ? 0 : (gz >= nz ? nz - 1 : gz);
            s.zlo = gz == 0;
            s.zhi = gz == nz - 1;
        } else {
            gz = gz < 0 ? gz + nz : (gz >= nz ? gz % nz : gz);
        }
        s.zo[0] = (gz == 0 ? nz - 1 : gz - 1) * plane;
        s.zo[1] = gz * plane;
        s.zo[2] = (gz == nz - 1 ? 0 : gz + 1) * plane;
    }
    return s;
}

// Populations of the previous step's output, as the kernel holds them.  The
// loads follow griddepcontrol.wait, so they are coherent (the data was written
// while this grid was resident) and volatile (nothing moves them above the
// wait, or out of the order that puts the halo's loads in flight with the
// cell's own).
__device__ __forceinline__ float2 ld_coherent(const float2 *p)
{
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}

template <int S>
__device__ __forceinline__ float2 ld_pair(const typename Store<S>::T *f, unsigned e)
{
    if constexpr (Store<S>::kDev) {
        unsigned u;
        float2 v;
        asm volatile("ld.global.b32 %0, [%1];" : "=r"(u) : "l"(f + 2 * (size_t)e) : "memory");
        Store<S>::decode2_d(u, v.x, v.y);
        return v;
    } else {
        return ld_coherent(reinterpret_cast<const float2 *>(f + 2 * (size_t)e));
    }
}

// Pull gather of a cell's populations (lw: its link word under a solid mask).
template <int S>
__device__ __forceinline__ void gather(const typename Store<S>::T *__restrict__ f, unsigned N32, const Site &s,
                                       unsigned lw, float2 (&v)[Q])
{
    const unsigned own = (unsigned)(s.zo[1] + s.yo[1] + s.xo[1]);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const bool wall = (cz(i) == 1 && s.zlo) || (cz(i) == -1 && s.zhi) || (i != 0 && ((lw >> i) & 1u));
        const unsigned src = (unsigned)(s.zo[1 - cz(i)] + s.yo[1 - cy(i)] + s.xo[1 - cx(i)]);
        v[i] = ld_pair<S>(f, wall ? (unsigned)opp(i) * N32 + own : (unsigned)i * N32 + src);
    }
}

template <int S, int REG, int FORCE, class T>
__global__ void __launch_bounds__(T::TX *T::TY *T::TZ)
k_step_box(const typename Store<S>::T *__restrict__ fin, typename Store<S>::T *__restrict__ fout, Phys<float> p,
           float *__restrict__ s_out, const unsigned *__restrict__ links, const float2 *__restrict__ wrho)
{
    constexpr int TX = T::TX, TY = T::TY, TZ = T::TZ, NT = TX * TY * TZ;
    constexpr int HY = T::FY ? 0 : 1, HZ = T::FZ ? 0 : 1;   // halo depth along y, z
    constexpr int BX = TX + 2, BY = TY + 2 * HY, BZ = TZ + 2 * HZ;
    static_assert(!Store<S>::kRel, "the relative formats step with the marching kernel");
    __shared__ float2 rho[BZ][BY][BX];
    const int tid = threadIdx.x;
    const int lx = tid % TX, ly = (tid / TX) % TY, lz = tid / (TX * TY);
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * TZ;
    const unsigned N32 = (unsigned)p.N;
    const bool active = x0 + lx < p.nx && y0 + ly < p.ny && z0 + lz < p.nz;
    const Site me = site_at<T>(p, x0 + lx, y0 + ly, z0 + lz);
    const unsigned own = (unsigned)(me.zo[1] + me.yo[1] + me.xo[1]);
    // halo: the z faces (whole planes of the box), then the y faces, then the x faces
    constexpr int NZ = HZ * 2 * BX * BY, NY = HY * 2 * BX * TZ, NX = 2 * TY * TZ, NH = NZ + NY + NX;
    auto halo_pos = [](int h, int &hx, int &hy, int &hz) {
        if (HZ && h < NZ) {
            hx = h % BX; hy = (h / BX) % BY; hz = h < BX * BY ? 0 : BZ - 1;
        } else if (HY && h < NZ + NY) {
            const int k = h - NZ;
            hx = k % BX; hz = HZ + (k / BX) % TZ; hy = k < BX * TZ ? 0 : BY - 1;
        } else {
            const int k = h - NZ - NY;
            hy = HY + k % TY; hz = HZ + (k / TY) % TZ; hx = k < TY * TZ ? 0 : BX - 1;
        }
    };
    cudaTriggerProgrammaticLaunchCompletion();   // the next step may be set up
    const float2 rs = make_float2(p.rho_s[0], p.rho_s[1]);
    // density of a box cell from its gathered populations, or what a wall site presents
    auto density_of = [&](const float2 (&g)[Q], bool ghost) {
        float2 q = density(g);
        if constexpr (Store<S>::kDev) q = vadd(q, PairF32::dup(p.rho0));
        if (ghost) q = p.wall_mirror ? vadd(q, rs) : rs;
        return q;
    };
    auto wall_rho = [&](unsigned cell) { return p.wall_mirror ? ld_coherent(wrho + cell) : rs; };
    int h = tid, hx = 0, hy = 0, hz = 0;
    halo_pos(h, hx, hy, hz);
    Site hs = site_at<T>(p, x0 + hx - 1, y0 + hy - HY, z0 + hz - HZ);
    unsigned hcell = (unsigned)(hs.zo[1] + hs.yo[1] + hs.xo[1]);
    unsigned lw = 0, hl = 0;
    if (links) {   // (the mask is set with the stream idle)
        lw = __ldg(links + own);
        hl = __ldg(links + hcell);
    }
    cudaGridDependencySynchronize();             // the previous step's populations
    float2 f[Q], g[Q];
    gather<S>(fin, N32, me, lw, f);              // (a solid site's own are read and not used)
    if (h < NH) gather<S>(fin, N32, hs, hl, g);
    const bool solid = lw & 1u;
    const float2 r = solid ? wall_rho(own) : density_of(f, me.ghost);
    float jx, jy, jz;
    momentum(PairF32(), f, jx, jy, jz);
    RegMoments<PairF32, REG> mom;
    mom.of(f);
    rho[lz + HZ][ly + HY][lx + 1] = r;
    if (h < NH) rho[hz][hy][hx] = (hl & 1u) ? wall_rho(hcell) : density_of(g, hs.ghost);
    if constexpr (NH > NT) {
#pragma unroll 1
        for (h += NT; h < NH; h += NT) {
            halo_pos(h, hx, hy, hz);
            hs = site_at<T>(p, x0 + hx - 1, y0 + hy - HY, z0 + hz - HZ);
            hcell = (unsigned)(hs.zo[1] + hs.yo[1] + hs.xo[1]);
            hl = links ? __ldg(links + hcell) : 0u;
            gather<S>(fin, N32, hs, hl, g);
            rho[hz][hy][hx] = (hl & 1u) ? wall_rho(hcell) : density_of(g, hs.ghost);
        }
    }
    __syncthreads();
    if (!active) return;
    if (solid) {   // a solid site holds no populations
        if (fout) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float ref = w<float>(i) * p.rho0;
                Store<S>::store2(fout + 2 * (size_t)((unsigned)i * N32 + own), 0.f, 0.f, ref, ref);
            }
        }
        if (s_out) {
#pragma unroll
            for (int k = 0; k < 6; ++k) s_out[(size_t)k * N32 + own] = 0.f;
        }
        return;
    }
    float2 Sb[3];
    interaction<PairF32>([&](int i) {
        const int dx = cx(i), dy = HY * cy(i), dz = HZ * cz(i);
        return vsub(rho[lz + HZ + dz][ly + HY + dy][lx + 1 + dx], rho[lz + HZ - dz][ly + HY - dy][lx + 1 - dx]);
    }, Sb);
    if (s_out) {   // interaction sums of this step (reverse-mode replay)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            s_out[(size_t)d * N32 + own] = Sb[d].x;
            s_out[(size_t)(3 + d) * N32 + own] = Sb[d].y;
        }
    }
    if (!fout) return;
    const float inv = 1.0f / (r.x + r.y);
    const float2 So[3] = {vswap(Sb[0]), vswap(Sb[1]), vswap(Sb[2])};
    auto get = [&](int i) { return f[i]; };
    auto put = [&](int i, float2 v) {
        typename Store<S>::T *q = fout + 2 * (size_t)((unsigned)i * N32 + own);
        if constexpr (Store<S>::kDev) Store<S>::store2_d(q, v.x, v.y);
        else Store<S>::store2(q, v.x, v.y, 0.f, 0.f);
    };
    collide_cell<PairF32, REG, FORCE, Store<S>::kDev>(PairF32(), p, r, inv, jx * inv, jy * inv, jz * inv, So, mom, get,
                                                      put);
}

inline Phys<float> make_phys_b(const HostPhys &h)
{
    using R = float;
    Phys<R> p;
    p.nx = h.nx; p.ny = h.ny; p.nz = h.nz; p.N = h.N;
    p.wall_z = h.wall_z;
    p.wall_mirror = h.wall_mirror;
    p.omega[0] = (R)(1.0 / h.tau[0]);
    p.omega[1] = (R)(1.0 / h.tau[1]);
    p.G12 = (R)h.G12; p.G21 = (R)h.G21;
    for (int d = 0; d < 3; ++d) p.gext[d] = (R)h.gext[d];
    p.rho_s[0] = (R)h.rho_s[0]; p.rho_s[1] = (R)h.rho_s[1];
    p.rho0 = (R)h.rho0;
    return p;
}

template <int S, int REG, int FORCE, class T>
cudaError_t launch(const HostPhys &h, const void *fin, void *fout, cudaStream_t s, void *s_out)
{
    using E = typename Store<S>::T;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)((h.nx + T::TX - 1) / T::TX), (unsigned)((h.ny + T::TY - 1) / T::TY),
                     (unsigned)((h.nz + T::TZ - 1) / T::TZ));
    c.blockDim = dim3(T::TX * T::TY * T::TZ);
    c.stream = s;
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k_step_box<S, REG, FORCE, T>, (const E *)fin, (E *)fout, make_phys_b(h),
                              (float *)s_out, h.links, (const float2 *)h.wall_rho);
}

template <int S, class T>
cudaError_t launch_kind(const HostPhys &h, const void *fin, void *fout, cudaStream_t s, void *s_out)
{
    const bool guo = h.forcing == FORCE_GUO;
#define LBM_BOX(REG_) \
    (guo ? launch<S, REG_, FORCE_GUO, T>(h, fin, fout, s, s_out) : launch<S, REG_, FORCE_EDM, T>(h, fin, fout, s, s_out))
    if ((float)(1.0 / h.tau[0]) == 1.0f && (float)(1.0 / h.tau[1]) == 1.0f) return LBM_BOX(COLL_EQ);
    if (h.collision == LBM_REGULARIZED) return LBM_BOX(COLL_REG);
    if (h.collision == LBM_REGULARIZED3) return LBM_BOX(COLL_REG3);
    return LBM_BOX(COLL_BGK);
#undef LBM_BOX
}

template <int S>
cudaError_t box_t(const HostPhys &h, const void *fin, void *fout, cudaStream_t s, void *s_out)
{
    if (h.nz == 1 && !h.wall_z) return launch_kind<S, TileXY>(h, fin, fout, s, s_out);
    if (h.ny == 1) return launch_kind<S, TileXZ>(h, fin, fout, s, s_out);
    return launch_kind<S, Tile3D>(h, fin, fout, s, s_out);
}

}  // namespace box
}  // namespace lbm
