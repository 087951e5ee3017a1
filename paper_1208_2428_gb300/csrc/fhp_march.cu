// fhp_march.cu -- host side of the register-marching kernels: how a lattice
// is cut into bands and the bands' quad columns are dealt to lanes.
#include <cuda_runtime.h>

#include <mutex>

#include "fhp_march.cuh"

namespace fhp {
namespace {

int march_sms() {
    static std::mutex m;
    static int sms[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(m);
    if (!sms[dev] && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms[dev];
}

// True if every useful lane of the chain keeps k valid words on both sides:
// a level spoils one more word inwards from each end of a warp, and a partial
// last quad has only m words to spare.
bool chain_valid(int nq, int m, int k, int pitch, int left, int hl) {
    if (m >= k) return true;
    const int step = 32 - 2 * hl;
    // Warps start at chain positions 0, step, 2 step, ...; the positions
    // modulo the pitch repeat after at most `pitch` warps.
    for (int w = 0, start = 0; w < pitch; ++w, start = (start + step) % pitch) {
        for (int lane = hl; lane < 32 - hl; ++lane) {
            const int e = (start + lane) % pitch, q = e - left;
            if (q < 0 || q >= nq) continue;
            int words = 0;
            for (int l = lane - 1; l >= 0 && words < k; --l) {
                const int qq = ((q - (lane - l)) % nq + nq) % nq;
                words += qq == nq - 1 ? m : 4;
            }
            if (words < k) return false;
            words = 0;
            for (int l = lane + 1; l <= 31 && words < k; ++l) {
                const int qq = (q + (l - lane)) % nq;
                words += qq == nq - 1 ? m : 4;
            }
            if (words < k) return false;
        }
    }
    return true;
}

}  // namespace

namespace {

cudaError_t march_any(int k, const StepArgs& a, const MarchArgs& b, const MarchVariant& v, bool launch, int* n,
                      cudaStream_t s) {
    return k == 2 ? march_k<2>(a, b, v, launch, n, s) : march_k<3>(a, b, v, launch, n, s);
}

}  // namespace

bool march_supported(const Geometry& g, int k) {
    return (k == 2 || k == 3) && g.H >= 2 * k + 2 && g.plane_words * 4 < ((size_t)1 << 32) - 64;
}

// Where register marching is the automatic choice (GB300, GSUPS, marching
// against the kernel it replaces; the lattices hold a cylinder):
//   without forcing   12288 x 1024: 2.9 against 2.5 thousand; 4096 x 4096 4.1
//     against 3.2; 8192 x 4096 4.8 (k = 2; 4.2 with k = 3) against 3.8;
//     16384 x 4096 6.6 (k = 3; 6.0 with k = 2) against 4.0; 29,984 x 27,990
//     7.8 against 3.3; but 4096 x 2048 2.9 against 3.1 (resident in shared
//     memory): from 12 million nodes on, and k = 2 between 24 and 48 million,
//     where the rows of a band are too few for a third level;
//   with forcing (p = 5e-4)   12288 x 4096 3.8 against 3.4, 16384 x 4096 4.1
//     against 3.6, 29,984 x 27,990 4.8 against 3.0, but 8192 x 4096 3.5 against
//     3.7: from 40 million nodes, k = 2 (k = 3 has 12 warps an SM to hide the
//     walks behind instead of 16: 3.2 on 16384 x 4096).  The walk's cost grows
//     with p: 3.7 against 3.6 at p = 2e-3, 3.6 against 3.6 at 4e-3;
//   FHP-III   from 200 million nodes on: its network is as long as the memory
//     traffic it hides on smaller lattices.
int march_choice(const Geometry& g, const ForcingTable& ft, bool force) {
    if (!march_supported(g, 3)) return 0;
    const long long nodes = (long long)g.W * g.H;
    if (force) {
        const bool rare = ft.p_plus_1 <= (1ull << 32) / 400;   // p < 2.5e-3
        return rare && nodes >= (g.rules == 3 ? 200000000LL : 40000000LL) ? 2 : 0;
    }
    if (nodes < 12000000) return 0;
    return nodes >= 24000000 && nodes < 48000000 ? 2 : 3;
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
    const MarchVariant v{has_solid, force, g.Wq % 4 != 0, g.rules == 3};
    int per_sm = 0;
    cudaError_t e = march_any(k, a, b, v, false, &per_sm, stream);
    if (e != cudaSuccess) return e;
    const int resident = march_sms() * per_sm * kMarchWarps;
    if (resident <= 0) return cudaErrorInvalidDevice;

    // How a band's columns go to lanes: whole rows side by side in a warp
    // (periodic in x by the shuffles' source lanes) where that fills the warp
    // at least as well, else one chain of all bands' columns, each band with
    // its halo columns, cut every 30 lanes (28 where a partial last quad is
    // too narrow to be a halo): about 92 % of the lanes for rows of 128 quads.
    const int m = g.Wq - 4 * (g.nq - 1);
    const int whole = g.nq <= 32 ? 32 / g.nq : 0;
    if (whole && whole * g.nq * (g.nq + 2) >= 30 * g.nq) {
        b.per_warp = whole;
    } else {
        b.hl = 1;
        b.left = 1;
        b.pitch = g.nq + 2;
        if (!chain_valid(g.nq, m, k, b.pitch, 1, 1)) {
            int best = 0;
            for (int left = 1; left <= 2; ++left)
                for (int pad = left + 1; pad < 32 && (!best || g.nq + pad < best); ++pad)
                    if (chain_valid(g.nq, m, k, g.nq + pad, left, 1)) {
                        best = g.nq + pad;
                        b.left = left;
                    }
            b.pitch = best;
            if (!best || best * 28 > (g.nq + 4) * 30) {   // two halo lanes always hold k words
                b.hl = 2;
                b.left = 2;
                b.pitch = g.nq + 4;
            }
        }
    }
    const int step = 32 - 2 * b.hl;
    auto warps_for = [&](int r) -> long long {
        const long long nb = (g.H + r - 1) / r;
        return b.pitch ? (nb * b.pitch + step - 1) / step : (nb + b.per_warp - 1) / b.per_warp;
    };
    // The lowest bands that one resident wave of warps covers.  Every band,
    // the last one too, has at least k rows, so that a pass reads no further
    // than the next band.
    int R = k <= 2 ? 2 : 4;
    while (R < g.H && (warps_for(R) > resident || (g.H % R != 0 && g.H % R < k))) R += 2;
    if (R > g.H) R = g.H;
    if (warps_for(R) > resident) return cudaErrorInvalidConfiguration;
    b.R = R;
    b.nbands = (g.H + R - 1) / R;
    b.nwarps = (int)warps_for(R);
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
