// fhp_resident.cu -- host side of the shared-memory resident kernels
// (fhp_resident.cuh): how many strips a lattice is cut into, and how many steps
// go between exchanges.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "fhp_resident.cuh"

namespace fhp {
namespace {

std::mutex g_res_mutex;
int g_res_sms[64] = {};

int resident_sms() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(g_res_mutex);
    if (!g_res_sms[dev] && cudaDeviceGetAttribute(&g_res_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return g_res_sms[dev];
}

// Bytes one CTA exchanges: 2 slots x 2 sides x units of 32 bytes per quad.
size_t exchange_bytes(const Geometry& g, int gh) {
    const int units = gh == 1 ? kResUnits<1> : gh == 2 ? kResUnits<2> : kResUnits<4>;
    return (size_t)4 * units * g.nq * 32;
}

// Shared memory of one CTA: two staged copies of its strip (nmax owned rows
// and gh ghost rows per side, 7 planes) and the solid rows of all but the
// outermost staged rows.
size_t resident_smem(const Geometry& g, bool has_solid, int grid, int gh) {
    const int staged = (g.H + grid - 1) / grid + 2 * gh;
    return (size_t)(2 * 7 * staged + (has_solid ? staged - 2 : 0)) * g.Pq * 4;
}

// CTAs (strips): at most one per SM, strips of at least 2 gh rows, and no more
// than the exchange buffer (the lattice's byte-staging area) has room for.  A
// single CTA for gh = 1 and lattices of at most kLoneQuads quads (128 x 128,
// 128 quads: 0.75 us a step, 0.98 us in strips with gh = 4; 256 x 128, 256
// quads: 1.1 us).
int resident_grid(const Geometry& g, bool has_solid, size_t staging_bytes, int gh) {
    const int sms = resident_sms();
    if (sms <= 0) return 0;
    if (gh == 1 && (long long)g.nq * g.H <= kLoneQuads && resident_smem(g, has_solid, 1, 1) <= (size_t)kResSmemLimit)
        return 1;
    const size_t room = staging_bytes / exchange_bytes(g, gh);
    const int grid = std::min(std::min(sms, g.H / (2 * gh)), (int)std::min<size_t>(room, 1u << 20));
    return gh > 1 && grid < 2 ? 0 : grid;
}

}  // namespace

bool resident_supported(const Geometry& g, bool has_solid, size_t staging_bytes, int gh) {
    if (gh != 1 && gh != 2 && gh != 4) return false;
    const int grid = resident_grid(g, has_solid, staging_bytes, gh);
    return grid > 0 && resident_smem(g, has_solid, grid, gh) <= (size_t)kResSmemLimit;
}

// More steps between exchanges save hand-offs (about 0.55 us each where nothing
// hides them) and add ghost rows, whose share grows with the row length; a
// larger exchange also leaves room for fewer strips, and forced nodes make
// every extra row dearer.  Measured, us a step with 1 / 2 / 4 steps between
// exchanges: 512 x 512 1.43 / - / 1.01 (p = 1e-3 1.67 / - / 1.50), 512 x 2048
// 1.46 / 1.20 / 1.04, 1024 x 1024 1.34 / 1.12 (1.70 / 1.61), 2048 x 2048 1.51 /
// 1.42 (1.82 / 1.88), 4096 x 1024 1.49 / 1.47 (1.86 / 2.00), 4096 x 2048 1.89 /
// 1.77 (2.44 / 2.48), 8192 x 1024 2.03 / 2.34.
int resident_interval_for(const Geometry& g, bool has_solid, size_t staging_bytes, bool force) {
    if (g.rules != 3 && (long long)g.nq * g.H > kLoneQuads) {
        if (g.nq <= 4 && resident_supported(g, has_solid, staging_bytes, 4)) return 4;
        if (g.nq <= (force ? 8 : 32) && resident_supported(g, has_solid, staging_bytes, 2)) return 2;
    }
    return resident_supported(g, has_solid, staging_bytes, 1) ? 1 : 0;
}

// Moving a lattice in and out costs 8 to 10 us, a direct step 4.15 us while its
// launch bounds it: calls of up to three steps are direct.  Flat lattices of long
// rows have fewer strips than SMs, each of two rows, and a step takes longer the
// longer the rows: 2.0 us for 128 quads, 2.7 for 192, 3.2 for 250 (us a call,
// resident / direct: 32384 x 4, 4 steps 22.8 / 16.8, 8 steps 35.5 / 33.1, 12 steps
// 48.5 / 49.5; 24576 x 32, 6 steps 26.7 / 24.9, 8 steps 31.8 / 33.1; 16384 x 32, 4
// steps 17.3 / 16.7, 5 steps 18.9 / 20.8).  One strip alone has no rows to hand
// over (32768 x 2, 4 steps 12.8 / 16.7), and a forced direct step of more than 2
// million nodes takes longer than its launch (32768 x 152, 5 steps 28.9 / 30.5).
int resident_least_steps(const Geometry& g, bool force) {
    const bool flat = g.H >= 4 && g.H < 2 * resident_sms() && !(force && (long long)g.W * g.H > 2000000);
    return std::max(4, flat ? g.nq / 28 + 1 : 0);
}

cudaError_t launch_resident(const Geometry& g, uint32_t* buf0, uint32_t* buf1, const uint32_t* solid, bool has_solid,
                            bool force, const ForcingTable& ft, Key2 key, uint64_t t0, int nsteps, int gh,
                            uint32_t* halo, size_t halo_bytes, cudaStream_t stream, unsigned int* err) {
    if (nsteps <= 0 || !resident_supported(g, has_solid, halo_bytes, gh)) return cudaErrorInvalidValue;
    const int grid = resident_grid(g, has_solid, halo_bytes, gh);
    const size_t smem = resident_smem(g, has_solid, grid, gh);
    StepArgs a;
    a.src = buf0;
    a.dst = buf1;
    a.solid = solid;
    a.plane_words = g.plane_words;
    a.H = g.H;
    a.Wq = g.Wq;
    a.nq = g.nq;
    a.Pq = g.Pq;
    a.rows_per_warp = a.groups_per_parity = a.warps_per_row = 1;
    a.key = key;
    a.y_base = g.row_base;
    a.rest_rules = rest_rules_mask(g);
    a.t_lo = (uint32_t)t0;
    a.t_hi = (uint32_t)(t0 >> 32);
    a.err = err;
    a.ft = ft;
    ResArgs ra;
    ra.buf0 = buf0;
    ra.buf1 = buf1;
    ra.flip = resident_flips(nsteps, gh);
    ra.halo = halo;
    ra.nsteps = nsteps;
    ra.t0 = t0;
    ra.nmax = (g.H + grid - 1) / grid;
    ra.nq_magic = ((1ull << 32) + g.nq - 1) / g.nq;
    if (grid > 1 && nsteps > gh) {   // no unit carries a step of this call
        const cudaError_t e = cudaMemsetAsync(halo, 0, exchange_bytes(g, gh) * grid, stream);
        if (e != cudaSuccess) return e;
    }
    const bool ragged = g.Wq % 4 != 0, sat = g.rules == 3;
    if (gh == 1) return launch_resident_g<1>(a, ra, grid, smem, has_solid, force, ragged, sat, stream);
    if (gh == 2) return launch_resident_g<2>(a, ra, grid, smem, has_solid, force, ragged, sat, stream);
    return launch_resident_g<4>(a, ra, grid, smem, has_solid, force, ragged, sat, stream);
}

}  // namespace fhp
