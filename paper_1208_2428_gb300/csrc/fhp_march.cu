// fhp_march.cu -- host side of the register-marching kernels: how a lattice
// is cut into bands and the bands' quad columns are dealt to lanes.
#include <cuda_runtime.h>

#include <mutex>

#include "fhp_march.cuh"

namespace fhp {

int sm_count() {
    static std::mutex m;
    static int sms[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(m);
    if (!sms[dev] && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms[dev];
}

namespace {

cudaError_t march_any(int k, const StepArgs& a, const MarchArgs& b, const MarchVariant& v, bool launch, int* n,
                      cudaStream_t s) {
    return k == 2 ? march_k<2>(a, b, v, launch, n, s) : march_k<3>(a, b, v, launch, n, s);
}

MarchVariant march_variant_of(const Geometry& g, bool has_solid, bool force) {
    return MarchVariant{has_solid, force, g.Wq % 4 != 0, g.rules == 3};
}

// Warps of the variant's kernel that are resident at once.
cudaError_t march_resident(int k, const MarchVariant& v, int* warps) {
    int per_sm = 0;
    const cudaError_t e = march_any(k, StepArgs{}, MarchArgs{}, v, false, &per_sm, nullptr);
    if (e != cudaSuccess) return e;
    *warps = sm_count() * per_sm * kMarchWarps;
    return *warps > 0 ? cudaSuccess : cudaErrorInvalidDevice;
}

}  // namespace

// How the quad columns of a lattice's bands go to lanes.  Rows of few quads:
// whole rows side by side in a warp (periodic in x by the shuffles' source
// lanes) where that fills the warp at least as well as the chain.  Else one
// chain of all bands' columns, each band with its halo columns, cut every 30
// lanes: about 92 % of the lanes for rows of 128 quads.
//
// A level spoils one more word inwards from each end of what a warp holds of
// a band, so a halo quad must hold k words.  All do but a partial last quad of
// m < k words.  Then a band has two halo columns to its left, and no warp may
// begin at the second of them or end at the last column: warps begin at the
// multiples of g = gcd(30, pitch) modulo the pitch, so g > 1 must not divide the
// number of quads.  The pitch is raised to the next one with that property, or
// the warps get two halo lanes per side (28 columns) where that is cheaper.
MarchLayout march_layout(const Geometry& g, int k) {
    MarchLayout l{};
    const int m = g.Wq - 4 * (g.nq - 1);
    const int whole = g.nq <= 32 ? 32 / g.nq : 0;
    if (whole && whole * (g.nq + 2) >= 30) {
        l.per_warp = whole;
        return l;
    }
    l.hl = 1;
    l.left = 1;
    l.pitch = g.nq + 2;
    if (m >= k) return l;
    l.left = 2;
    auto gcd30 = [](int v) { return (v % 2 ? 1 : 2) * (v % 3 ? 1 : 3) * (v % 5 ? 1 : 5); };
    for (l.pitch = g.nq + 3; l.pitch * 28 <= (g.nq + 4) * 30; ++l.pitch) {
        const int d = gcd30(l.pitch);
        if (d > 1 && g.nq % d != 0) return l;
    }
    l.hl = 2;
    l.pitch = g.nq + 4;
    return l;
}

long long march_warps(const Geometry& g, const MarchLayout& l, int R) {
    const long long bands = (g.H + R - 1) / R;
    if (!l.pitch) return (bands + l.per_warp - 1) / l.per_warp;
    const int step = 32 - 2 * l.hl;
    return (bands * l.pitch + step - 1) / step;
}

// (Every band, the last one too, has at least k rows, so that a pass reads no
// further than the next band.)
int march_rows(const Geometry& g, int k, int R) {
    if (R < k) R = (k + 1) & ~1;
    while (R < g.H && g.H % R != 0 && g.H % R < k) R += 2;
    return R < g.H ? R : g.H;
}

bool march_supported(const Geometry& g, int k) {
    return (k == 2 || k == 3) && g.H >= 2 * k + 2 && g.plane_words * 4 < ((size_t)1 << 32) - 64;
}

bool march_fits(const Geometry& g, int k, bool has_solid, bool force) {
    int resident = 0;
    return march_supported(g, k) &&
           march_resident(k, march_variant_of(g, has_solid, force), &resident) == cudaSuccess &&
           march_warps(g, march_layout(g, k), g.H) <= resident;
}

// Where register marching is the automatic choice (GB300, GSUPS, marching
// against the kernel it replaces; the lattices hold a cylinder):
//   without forcing   8192 x 2560: 3.8 thousand with k = 2 (3.7 with k = 3)
//     against 3.3; 8192 x 4096 4.8 (4.4) against 3.8; 16384 x 4096 6.1 with k = 3
//     (5.3 with k = 2) against 4.0; 29,984 x 27,990 7.6 (5.5) against 3.3: from 12
//     million nodes on (smaller ones are resident in shared memory anyway),
//     k = 3 from 48 million, where the bands are high enough for a third level;
//   with forcing (p = 5e-4)   12288 x 4096 3.8 against 3.4, 16384 x 4096 4.1
//     against 3.6, 29,984 x 27,990 4.8 against 3.0, but 8192 x 4096 3.5 against
//     3.7: from 40 million nodes, k = 2 (k = 3 has 12 warps an SM to hide the
//     walks behind instead of 16: 3.2 on 16384 x 4096).  The walk's cost grows
//     with p: 3.7 against 3.6 at p = 2e-3, 3.6 against 3.6 at 4e-3;
//   FHP-III   from 200 million nodes on: its network is as long as the memory
//     traffic it hides on smaller lattices;
//   rows of one quad (at most 128 nodes)   every lane marches a band of its own and
//     a warp's loads are 16-byte pieces far apart, each of which costs a whole
//     sector, so beyond L2 the ring and its contiguous tiles win (time marching
//     over the faster single-step kernel, by nodes with padding): with k = 3 53
//     million 0.77 to 0.91, 80 million 0.94, 90 million 1.03 to 1.08, 130 million
//     1.05 to 1.15, 270 million 1.25 to 1.5; with k = 2 53 million 0.90 to 0.95, 66
//     million 1.2 to 1.4, 130 million 1.5 to 2 -- so k = 3 below 85 million without
//     forcing, k = 2 below 60 million with it.
int march_choice(const Geometry& g, const ForcingTable& ft, bool has_solid, bool force) {
    if (!march_supported(g, 3)) return 0;
    const long long nodes = (long long)g.W * g.H;
    int k = 0;
    if (g.nq == 1 && g.plane_words * 32 >= (force ? 60000000u : 85000000u)) return 0;
    if (force) {
        const bool rare = ft.p_plus_1 <= (1ull << 32) / 400;   // p < 2.5e-3
        if (rare && nodes >= (g.rules == 3 ? 200000000LL : 40000000LL)) k = 2;
    } else if (nodes >= 12000000) {
        k = nodes < 48000000 && g.nq > 1 ? 2 : 3;
    }
    return k && march_fits(g, k, has_solid, force) ? k : 0;
}

cudaError_t launch_march(const Geometry& g, uint32_t* src, uint32_t* dst, const uint32_t* solid, bool has_solid,
                         bool force, const ForcingTable& ft, Key2 key, uint64_t t0, int k, int passes,
                         unsigned int* flags, size_t flag_bytes, cudaStream_t stream, unsigned int* err) {
    if (!march_supported(g, k) || passes < 1) return cudaErrorInvalidValue;
    StepArgs a;
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
    a.err = err;
    a.ft = ft;
    MarchArgs b{};
    const MarchVariant v = march_variant_of(g, has_solid, force);
    int resident = 0;
    cudaError_t e = march_resident(k, v, &resident);
    if (e != cudaSuccess) return e;

    const MarchLayout lay = march_layout(g, k);
    b.pitch = lay.pitch;
    b.left = lay.left;
    b.hl = lay.hl;
    b.per_warp = lay.per_warp;
    // The lowest bands that one resident wave of warps covers.
    int R = march_rows(g, k, 2);
    while (R < g.H && march_warps(g, lay, R) > resident) R = march_rows(g, k, R + 2);
    if (march_warps(g, lay, R) > resident) return cudaErrorInvalidConfiguration;
    b.R = R;
    b.nbands = (g.H + R - 1) / R;
    b.nwarps = (int)march_warps(g, lay, R);
    b.flags = flags;
    const size_t need = (size_t)b.nwarps * sizeof(unsigned int);
    const int per_launch = need <= flag_bytes ? passes : 1;
    for (int done = 0; done < passes; done += per_launch) {
        b.passes = per_launch;
        a.src = done & 1 ? dst : src;
        a.dst = done & 1 ? src : dst;
        const uint64_t t = t0 + (uint64_t)done * (uint64_t)k;
        a.t_lo = (uint32_t)t;
        a.t_hi = (uint32_t)(t >> 32);
        if (b.passes > 1) {
            e = cudaMemsetAsync(flags, 0, need, stream);
            if (e != cudaSuccess) return e;
        }
        e = march_any(k, a, b, v, true, nullptr, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace fhp
