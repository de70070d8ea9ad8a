// FP64 diagnostics reductions over the density fields (Sec. 3 and Sec. 4.2 of
// Otomo et al., arXiv:1601.01237): the pressure jump across a droplet
// interface for Young-Laplace (Eq. 12), and droplet volume, centre of mass and
// thin-film density for the wall cases.  The densities come from the density
// pass (k_density) into the lattice's scratch; each block writes fixed-order
// FP64 partials that the host sums in order (deterministic).
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "d3q19.cuh"
#include "lbm_internal.h"

namespace lbm {

namespace {

constexpr int kThreadsD = 256;
constexpr int kDiagBlocks = 1216;
constexpr int kSlots = 8;

template <class R>
struct Geo {
    int nx, ny, nz;
    long long N;
    int per[3];
    const unsigned char *solid;   // mask of solid sites or nullptr
};

// Does fluid cell (x, y, z) of a masked (fully periodic) lattice have a solid
// site among its 18 neighbours?
template <class R>
__device__ __forceinline__ bool next_to_solid(const Geo<R> &g, int x, int y, int z)
{
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const int m = dx * dx + dy * dy + dz * dz;
                if (m == 0 || m > 2) continue;
                const int X = (x + dx + g.nx) % g.nx, Y = (y + dy + g.ny) % g.ny, Z = (z + dz + g.nz) % g.nz;
                if (g.solid[((long long)Z * g.ny + Y) * g.nx + X]) return true;
            }
    return false;
}

__device__ __forceinline__ double min_image(double d, int n, int periodic)
{
    if (!periodic) return d;
    const double L = (double)n;
    if (d > 0.5 * L) d -= L;
    else if (d < -0.5 * L) d += L;
    return d;
}

// Coordinates of a cell (32-bit divisions where the lattice allows).
template <class R>
__device__ __forceinline__ void cell_xyz(const Geo<R> &g, long long c, int &x, int &y, int &z)
{
    if (g.N <= 0x7fffffffLL) {
        const unsigned cu = (unsigned)c, nx = (unsigned)g.nx, plane = nx * (unsigned)g.ny;
        const unsigned zu = cu / plane, rem = cu - zu * plane, yu = rem / nx;
        x = (int)(rem - yu * nx); y = (int)yu; z = (int)zu;
    } else {
        const long long plane = (long long)g.nx * g.ny;
        z = (int)(c / plane);
        const long long rem = c - (long long)z * plane;
        y = (int)(rem / g.nx);
        x = (int)(rem - (long long)y * g.nx);
    }
}

__device__ __forceinline__ float min_image_f(float d, int n, int periodic)
{
    if (!periodic) return d;
    const float L = (float)n;
    if (d > 0.5f * L) d -= L;
    else if (d < -0.5f * L) d += L;
    return d;
}

template <int K>
__device__ __forceinline__ void block_reduce_store(double (&acc)[K], double *__restrict__ partials)
{
    __shared__ double sh[K][kThreadsD];
    for (int k = 0; k < K; ++k) sh[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int s = kThreadsD / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int k = 0; k < K; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < K) partials[(long long)blockIdx.x * kSlots + threadIdx.x] = sh[threadIdx.x][0];
}

// Pressure p = T0 rho - G12 T0 rho^1 rho^2 (bulk pressure of the Eq. 7 force
// with G12 = G21) averaged inside r < r_in and outside r > r_out of `center`
// (minimum image along periodic axes).  Partials: sum_in, n_in, sum_out, n_out.
template <class R>
__global__ void __launch_bounds__(kThreadsD)
k_pressure(const R *__restrict__ rho, Geo<R> g, double G12, double cx, double cy, double cz, double r_in,
           double r_out, double *__restrict__ partials)
{
    double acc[4] = {0, 0, 0, 0};
    long long n_in = 0, n_out = 0;
    const double T0 = 1.0 / 3.0;
    const float fcx = (float)cx, fcy = (float)cy, fcz = (float)cz;
    const float fin = (float)(r_in * r_in), fout = (float)(r_out * r_out);
    const float ext = 4e-6f * (float)(g.nx + g.ny + g.nz) +
                      4e-6f * (fabsf(fcx) + fabsf(fcy) + fabsf(fcz) + (float)r_in + (float)r_out);
    for (long long c = (long long)blockIdx.x * kThreadsD + threadIdx.x; c < g.N; c += (long long)gridDim.x * kThreadsD) {
        int x, y, z;
        cell_xyz(g, c, x, y, z);
        if (g.solid && g.solid[c]) continue;   // no fluid at a solid site
        // The distance in FP32 decides all cells but those within its rounding of
        // one of the two spheres (the FP64 distance of every cell took 177 us at
        // 128^3, this 51): |d| is wrong by less than 1e-6 of the lattice's
        // extents, d^2 by less than err.
        const float fx = min_image_f(x - fcx, g.nx, g.per[0]), fy = min_image_f(y - fcy, g.ny, g.per[1]),
                    fz = min_image_f(z - fcz, g.nz, g.per[2]);
        const float q = fx * fx + fy * fy + fz * fz;
        const float err = ext * (sqrtf(q) + ext);
        bool in = q + err < fin, out = q - err > fout;
        if (!in && !out && !(q - err > fin && q + err < fout)) {
            const double dx = min_image(x - cx, g.nx, g.per[0]);
            const double dy = min_image(y - cy, g.ny, g.per[1]);
            const double dz = min_image(z - cz, g.nz, g.per[2]);
            const double r = sqrt(dx * dx + dy * dy + dz * dz);
            in = r < r_in;
            out = r > r_out;
        }
        if (!in && !out) continue;
        const double r1 = (double)rho[c], r2 = (double)rho[g.N + c];
        const double p = T0 * (r1 + r2) - G12 * T0 * r1 * r2;
        if (in) { acc[0] += p; ++n_in; }
        if (out) { acc[2] += p; ++n_out; }
    }
    acc[1] = (double)n_in;
    acc[3] = (double)n_out;
    block_reduce_store<4>(acc, partials);
}

// Origin of the droplet's coordinates, and the bounds beyond which a coordinate
// belongs to another periodic image (x - o > n / 2 above hi, < -n / 2 below lo).
struct Origin {
    double o[3];
    int lo[3], hi[3];
};

// Droplet of component 1: cells with rho^1 > threshold.  Partials: volume,
// sum x, sum y, sum z (coordinates relative to `origin`, minimum image along
// periodic axes), sum rho^1 over the droplet, and over the wall layer outside
// the droplet: sum rho^1 and cell count (thin film).  The wall layer is z = 0,
// or with a mask the fluid cells next to a solid site; solid sites count for
// nothing.
template <class R>
__global__ void __launch_bounds__(kThreadsD)
k_droplet(const R *__restrict__ rho, Geo<R> g, double threshold, Origin og, double *__restrict__ partials)
{
    // The coordinates are summed as whole numbers (exact), moved by a period
    // where the minimum image is another one, and the origin is taken off the
    // sums once: FP64 arithmetic is scarce here.
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    long long count = 0, sum[3] = {0, 0, 0}, film = 0;
    const int n[3] = {g.nx, g.ny, g.nz};
    for (long long c = (long long)blockIdx.x * kThreadsD + threadIdx.x; c < g.N; c += (long long)gridDim.x * kThreadsD) {
        int x, y, z;
        cell_xyz(g, c, x, y, z);
        if (g.solid && g.solid[c]) continue;
        const double r1 = (double)rho[c];
        if (r1 > threshold) {
            const int q[3] = {x, y, z};
#pragma unroll
            for (int k = 0; k < 3; ++k) sum[k] += q[k] > og.hi[k] ? q[k] - n[k] : (q[k] < og.lo[k] ? q[k] + n[k] : q[k]);
            ++count;
            acc[4] += r1;
        } else if (g.solid ? next_to_solid(g, x, y, z) : z == 0) {
            acc[5] += r1;
            ++film;
        }
    }
    acc[0] = (double)count;
    // (no cell, no share of the origin: it may be infinite)
    for (int k = 0; k < 3; ++k) acc[1 + k] = count ? fma(-(double)count, og.o[k], (double)sum[k]) : 0.0;
    acc[6] = (double)film;
    block_reduce_store<7>(acc, partials);
}

template <class R>
Geo<R> geo_of(const HostPhys &h)
{
    Geo<R> g;
    g.nx = h.nx; g.ny = h.ny; g.nz = h.nz; g.N = h.N;
    g.per[0] = 1; g.per[1] = 1; g.per[2] = h.wall_z ? 0 : 1;
    g.solid = h.solid;
    return g;
}

}  // namespace

int diag_grid(long long N) { return (int)std::min<long long>(kDiagBlocks, (N + kThreadsD - 1) / kThreadsD); }
int diag_slots() { return kSlots; }

cudaError_t launch_pressure(const HostPhys &h, const void *rho, const double center[3], double r_in, double r_out,
                            double *partials, cudaStream_t s)
{
    if (h.storage == ST_F64)
        k_pressure<double><<<diag_grid(h.N), kThreadsD, 0, s>>>((const double *)rho, geo_of<double>(h), h.G12, center[0],
                                                             center[1], center[2], r_in, r_out, partials);
    else
        k_pressure<float><<<diag_grid(h.N), kThreadsD, 0, s>>>((const float *)rho, geo_of<float>(h), h.G12, center[0],
                                                            center[1], center[2], r_in, r_out, partials);
    return cudaGetLastError();
}

cudaError_t launch_droplet(const HostPhys &h, const void *rho, double threshold, const double origin[3],
                           double *partials, cudaStream_t s)
{
    Origin og;
    const int n[3] = {h.nx, h.ny, h.nz};
    for (int d = 0; d < 3; ++d) {
        const bool per = d < 2 || !h.wall_z;
        const double half = 0.5 * (double)n[d];
        og.o[d] = origin[d];
        og.lo[d] = per ? (int)fmax(fmin(ceil(origin[d] - half), 2e9), -2e9) : INT_MIN;
        og.hi[d] = per ? (int)fmax(fmin(floor(origin[d] + half), 2e9), -2e9) : INT_MAX;
    }
    if (h.storage == ST_F64)
        k_droplet<double><<<diag_grid(h.N), kThreadsD, 0, s>>>((const double *)rho, geo_of<double>(h), threshold, og,
                                                               partials);
    else
        k_droplet<float><<<diag_grid(h.N), kThreadsD, 0, s>>>((const float *)rho, geo_of<float>(h), threshold, og,
                                                              partials);
    return cudaGetLastError();
}

}  // namespace lbm
