// Fused single-pass time step: dispatch over the storage formats.  The kernel
// templates live in lbm_fused_impl.cuh; each storage format is instantiated
// in a translation unit of its own (lbm_fused_<format>.cu), so that they
// compile in parallel.
#include <cuda_runtime.h>

#include <algorithm>

#include "d3q19.cuh"
#include "lbm_internal.h"

namespace lbm {
namespace fused {
template <int S>
cudaError_t fused_t(const HostPhys &h, const void *fin, void *fout, cudaStream_t s, cudaEvent_t *ev, void *s_out);
}  // namespace fused

bool fused_supported(const HostPhys &p)
{
    // 32-bit offsets of the cell pairs inside the 19 direction arrays; tiles of
    // 32 x 8 columns, chunks of at least 8 planes
    return p.storage != ST_F64 && (long long)Q * p.N < (1LL << 32) &&
           (long long)((p.nx + 31) / 32) * ((p.ny + 7) / 8) < (1LL << 31) &&
           (p.nz + 7) / 8 < 65536;
}

int fused_planes(long long cols, int nz, int sms)
{
    // A CTA that marches over lz planes reads lz + 2 planes of populations
    // (the planes below and above its chunk feed its first and last
    // collisions), and the CTAs of one launch run in waves of two per SM.
    // Among equal-length chunkings with lz in [8, 64] (fewer when nz < 8),
    // take the one with the fewest waves x (lz + 2); lz = 64 stays unless
    // another length is at least 5 % cheaper (large lattices, where the last
    // wave is a small part of the launch).
    const long long slots = 2LL * (sms > 0 ? sms : 1);
    auto cost = [&](int lz) {
        const long long ctas = cols * ((nz + lz - 1) / lz);
        return ((ctas + slots - 1) / slots) * (long long)(lz + 2);
    };
    int best = nz < kPlanesMax ? nz : kPlanesMax;
    const long long c64 = cost(best);
    if (c64 > 16LL * (best + 2)) return best;   // more than 16 waves: the last one costs < 6 %
    long long cbest = c64;
    for (int most = best; most >= kPlanesMin; --most) {   // (by length: few of them however tall the lattice)
        const int nch = (nz + most - 1) / most, lz = (nz + nch - 1) / nch;
        if (lz < kPlanesMin && nch > 1) break;
        const long long c = cost(lz);
        if (c < cbest) { cbest = c; best = lz; }
    }
    return cbest * 20 <= c64 * 19 ? best : (nz < kPlanesMax ? nz : kPlanesMax);
}

namespace box {
template <int S>
cudaError_t box_t(const HostPhys &h, const void *fin, void *fout, cudaStream_t s, void *s_out);
}  // namespace box

bool use_box(const HostPhys &p)
{
    if (p.storage != ST_F32 && p.storage != ST_F16_DEV && p.storage != ST_BF16_DEV) return false;
    if (!fused_supported(p) || (p.ny + 7) / 8 > 65535 || (p.nz + 3) / 4 > 65535) return false;
    // One layer along y: the marching tiles would repeat it eight times.
    if (p.ny == 1) return true;
    // One periodic layer along z: the box step is the faster one while its halo
    // comes from L2 (us per step, marching / box: 700^2 47 / 29, 2048^2 363 / 356,
    // 4096^2 1479 / 2328).
    if (p.nz == 1 && !p.wall_z) return p.N <= 2048LL * 2048;
    // Elsewhere by cost: a marching CTA takes about 1.85 us per plane while its
    // SM holds no other (and in proportion beyond), the box step 0.092 ns per cell
    // of its padded boxes, 1/20000 of that (marching / box: 56^3 19.3 / 16.1, 60^3
    // 18.5 / 21.1, 8 x 128 x 128 19.3 / 12.8, 300 x 24 x 24 18.6 / 15.9, 2 x 200 x 200
    // 10.4 / 11.8).
    const int sms = current_device_sms();
    const long long cols = (long long)((p.nx + 31) / 32) * ((p.ny + 7) / 8);
    const int lz = fused_planes(cols, p.nz, sms);
    const long long ctas = cols * ((p.nz + lz - 1) / lz);
    const long long padded = (long long)((p.nx + 7) / 8) * ((p.ny + 7) / 8) * ((p.nz + 3) / 4) * 256;
    return padded * sms < 20000LL * (lz + 2) * (ctas > sms ? ctas : sms);
}

// A CTA takes about 1.9 us per plane, two or more of an SM in proportion, and marches
// lz + 2 planes; a lattice of few periodic planes in one chunk finds the two beyond in
// its caches.  The 16-bit formats take the share of it that their instances' occupancy
// gives them once the SMs are full.  Against measured steps of 2 x 300 x 300 to 256^3, 1 x 2100^2 to
// 6 x 2100^2 and 20000 x 32 x 32 within 15 %.
double marching_us(const HostPhys &p)
{
    const int sms = current_device_sms();
    const long long cols = (long long)((p.nx + 31) / 32) * ((p.ny + 7) / 8);
    const int lz = fused_planes(cols, p.nz, sms);
    const long long ctas = cols * ((p.nz + lz - 1) / lz);
    const double beyond = lz < p.nz ? 2.0 : std::min(2.0, 0.55 + 0.25 * p.nz);
    const double per_sm = ctas <= sms ? 1.0 : (ctas <= 2 * sms ? 2.0 : (double)ctas / sms);
    const bool eq = (float)(1.0 / p.tau[0]) == 1.0f && (float)(1.0 / p.tau[1]) == 1.0f;
    const double share = p.storage == ST_F32 || ctas <= 2 * sms ? 1.0 : (eq ? (p.wall_z ? 0.81 : 0.66) : (p.wall_z ? 0.88 : 0.81));
    return 3.0 + 1.88 * (lz + beyond) * per_sm * share;
}

cudaError_t launch_step_box(const HostPhys &p, const void *f_in, void *f_out, cudaStream_t s, void *s_out)
{
    switch (p.storage) {
    case ST_F32: return box::box_t<ST_F32>(p, f_in, f_out, s, s_out);
    case ST_F16_DEV: return box::box_t<ST_F16_DEV>(p, f_in, f_out, s, s_out);
    case ST_BF16_DEV: return box::box_t<ST_BF16_DEV>(p, f_in, f_out, s, s_out);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step_fused(const HostPhys &p, const void *f_in, void *f_out, cudaStream_t s, cudaEvent_t *ev,
                              void *s_out)
{
    switch (p.storage) {
    case ST_F32: return fused::fused_t<ST_F32>(p, f_in, f_out, s, ev, s_out);
    case ST_F16_DEV: return fused::fused_t<ST_F16_DEV>(p, f_in, f_out, s, ev, s_out);
    case ST_BF16_DEV: return fused::fused_t<ST_BF16_DEV>(p, f_in, f_out, s, ev, s_out);
    case ST_F16_REL: return fused::fused_t<ST_F16_REL>(p, f_in, f_out, s, ev, s_out);
    case ST_BF16_REL: return fused::fused_t<ST_BF16_REL>(p, f_in, f_out, s, ev, s_out);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
