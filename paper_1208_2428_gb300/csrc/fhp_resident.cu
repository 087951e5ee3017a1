// fhp_resident.cu -- lattices that fit in the SMs' shared memory: the whole
// lattice stays on chip for all steps of a call.
//
// One cooperative launch, one CTA per SM.  CTA b owns rows [y0, y1) of the
// lattice (a contiguous strip of at least two) and keeps them, with one extra
// row below and above, in two shared-memory buffers (steps alternate between
// them).  A step pulls the movers from the rows y-1 (north-going planes 3, 4),
// y (planes 2, 5, 6) and y+1 (south-going planes 0, 1) of the staged strip,
// scatters with the same per-quad code as every other step kernel (random
// words keyed on the lattice's row, so results are identical), and writes the
// new state of the owned rows into the other buffer.  HBM sees the lattice
// once at the start and once at the end of the call.
//
// Between steps only the strips' edge rows travel: planes 0, 1 of the lowest
// row to the CTA below, planes 3, 4 of the highest to the CTA above.  A step
// of a few rows takes less than a hand-off between SMs, so the hand-off is
// what bounds small lattices, and it is one store and one load long: every
// 32-bit word travels in a 64-bit store together with the number of the step
// it belongs to, and the reader polls the word itself until it carries that
// number.  (Rows, fence, release of a counter, acquire, load of the rows -- the
// former protocol -- are five trips to L2 in a row: 3.2 us a step on 4096 x 1024
// (p = 1e-3) with an exchange every second step, 1.9 us with this one every
// step; 6.2 us a direct step.)  Rows
// alternate between two slots: a CTA overwrites a slot two steps later, when
// its neighbours' words of the step between have told it that they had read
// it.  Edge rows are computed first, the draws of a thread's first quad are
// made before the wait, and warps without a quad do the polling, so on larger
// strips the hand-off hides behind the interior rows.
//
// A lattice of at most kLoneQuads quads stays in one SM (its extra rows are
// its own edge rows): 16 warps step it faster than a hand-off takes.
//
// A second kernel (fhp_resident_ghost.cu) keeps two ghost rows per side and
// exchanges every second step (an explicit setting).  This file also holds the
// host side of both.
#include <cuda_runtime.h>

#include <mutex>

#include "fhp_resident.cuh"

namespace fhp {
namespace {

constexpr int kLoneQuads = 256;

// A word and the step it belongs to, as one 64-bit value.
__device__ __forceinline__ unsigned long long tagged(uint32_t word, uint32_t step) {
    return (unsigned long long)step << 32 | word;
}

__device__ __forceinline__ void put_unit(unsigned long long* unit, uint4 v, uint32_t step) {
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(unit), "l"(tagged(v.x, step)),
                 "l"(tagged(v.y, step))
                 : "memory");
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(unit + 2), "l"(tagged(v.z, step)),
                 "l"(tagged(v.w, step))
                 : "memory");
}

// Polls a unit until all of its words belong to `step`; gives up (false)
// after kWaitLimitNs.
__device__ __forceinline__ bool get_unit(const unsigned long long* unit, uint32_t step, uint4& v) {
    unsigned long long start = 0;
    for (unsigned int spin = 0;; ++spin) {
        unsigned long long a, b, c, d;
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(unit) : "memory");
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(c), "=l"(d) : "l"(unit + 2) : "memory");
        if ((uint32_t)(a >> 32) == step && (uint32_t)(b >> 32) == step && (uint32_t)(c >> 32) == step &&
            (uint32_t)(d >> 32) == step) {
            v = make_uint4((uint32_t)a, (uint32_t)b, (uint32_t)c, (uint32_t)d);
            return true;
        }
        if ((spin & 255u) == 255u) {
            const unsigned long long now = global_ns();
            if (start == 0) start = now;
            else if (now - start > kWaitLimitNs) return false;
        }
    }
}

// SAT: the FHP-III rule set.
template <bool SOLID, bool FORCE, bool RAGGED, bool SAT>
__global__ void __launch_bounds__(kRes1Threads, 1) fhp_resident_kernel(const StepArgs a, const ResArgs ra) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int T = kRes1Threads;
    const int G = (int)gridDim.x, b = (int)blockIdx.x;
    const int y0 = (int)(((long long)b * a.H) / G), y1 = (int)(((long long)(b + 1) * a.H) / G);
    const int n = y1 - y0;
    const int Pq = a.Pq, q4 = Pq / 4, nq = a.nq;
    const int rows = ra.nmax + 2;
    const size_t pstride = (size_t)rows * Pq;          // words per staged plane
    uint32_t* X[2];
    X[0] = reinterpret_cast<uint32_t*>(smem_raw);
    X[1] = X[0] + 7 * pstride;
    uint32_t* S = X[1] + 7 * pstride;                  // solid rows of the strip (SOLID only)
    const int below = b == 0 ? G - 1 : b - 1, above = b == G - 1 ? 0 : b + 1;
    const int tid = (int)threadIdx.x;
    unsigned long long* halo = reinterpret_cast<unsigned long long*>(ra.halo);
    // Unit of (parity, CTA, side, plane, quad); side 0: bottom row (planes 0,
    // 1), side 1: top row (planes 3, 4).
    auto unit = [&](int par, int cta, int side, int p, int q) {
        return halo + ((((size_t)(par * G + cta) * 2 + side) * 2 + p) * nq + q) * 4;
    };

    // Stage the owned rows, the two extra rows for step 0 and the solid rows.
    for (int i = tid; i < 7 * n * q4; i += T) {
        const int p = i / (n * q4), rem = i - p * n * q4, lr = rem / q4 + 1, w = 4 * (rem % q4);
        st4(X[0] + p * pstride + (size_t)lr * Pq + w,
            ld4(ra.buf0 + (size_t)p * a.plane_words + (size_t)(y0 + lr - 1) * Pq + w));
    }
    {
        const int yb = y0 == 0 ? a.H - 1 : y0 - 1, ya = y1 == a.H ? 0 : y1;
        for (int i = tid; i < 4 * q4; i += T) {
            const int k = i / q4, w = 4 * (i % q4);
            const int p = k < 2 ? 3 + k : k - 2;         // planes 3, 4 from below; 0, 1 from above
            const int y = k < 2 ? yb : ya, lr = k < 2 ? 0 : n + 1;
            st4(X[0] + p * pstride + (size_t)lr * Pq + w, ld4(ra.buf0 + (size_t)p * a.plane_words + (size_t)y * Pq + w));
        }
    }
    if (SOLID)
        for (int i = tid; i < n * q4; i += T) {
            const int rr = i / q4, w = 4 * (i % q4);
            st4(S + (size_t)rr * Pq + w, ld4(a.solid + (size_t)(y0 + rr) * Pq + w));
        }

    // Quads of a step: the strip's edge rows (row 0, then row n - 1) first,
    // then rows 1 .. n - 2.
    const int edge = 2 * nq, items = n * nq;
    auto place = [&](int e, int& rr, int& q) {
        const uint32_t j = (uint32_t)(e < edge ? e : e - edge);
        const int k = (int)(((unsigned long long)j * ra.nq_magic) >> 32);   // j / nq
        q = (int)j - k * nq;
        rr = e < edge ? (k == 0 ? 0 : n - 1) : 1 + k;
    };
    auto step_of = [&](int s) {
        const unsigned long long t = ra.t0 + (unsigned long long)s;
        return StepVar{nullptr, (uint32_t)t, (uint32_t)(t >> 32)};
    };
    int rr0 = 0, q0 = 0;
    uint4 chi = make_uint4(0u, 0u, 0u, 0u), gate = chi;
    if (tid < items) {
        place(tid, rr0, q0);
        resident_draws<FORCE>(a, step_of(0), q0, y0 + rr0, chi, gate);
    }
    __syncthreads();

    for (int s = 0; s < ra.nsteps; ++s) {
        const uint32_t* src = X[s & 1];
        uint32_t* dst = X[(s & 1) ^ 1];
        const StepVar v = step_of(s);
        const bool more = s + 1 < ra.nsteps;
        const int par = (s + 1) & 1;
        bool ok = true;
        // Edge rows go to the neighbours (or, alone, to the strip's own extra rows).
        auto hand_over = [&](int rr, int q, const uint4 (&o)[7]) {
            if (G == 1) {
                if (rr == 0) {
                    st4(dst + (size_t)(n + 1) * Pq + 4 * q, o[0]);
                    st4(dst + pstride + (size_t)(n + 1) * Pq + 4 * q, o[1]);
                } else {
                    st4(dst + 3 * pstride + 4 * q, o[3]);
                    st4(dst + 4 * pstride + 4 * q, o[4]);
                }
            } else if (more) {
                const int side = rr == 0 ? 0 : 1;
                put_unit(unit(par, b, side, 0, q), side ? o[3] : o[0], (uint32_t)(s + 1));
                put_unit(unit(par, b, side, 1, q), side ? o[4] : o[1], (uint32_t)(s + 1));
            }
        };
        uint4 o[7];
        if (tid < items) {
            resident_quad_drawn<SOLID, FORCE, RAGGED, SAT>(a, v, src, dst, S + (size_t)rr0 * Pq, pstride, rr0 + 1, y0 + rr0,
                                                      q0, chi, gate, o);
            if (tid < edge) hand_over(rr0, q0, o);
            if (more) resident_draws<FORCE>(a, step_of(s + 1), q0, y0 + rr0, chi, gate);
        }
        for (int e = tid + T; e < items; e += T) {
            int rr, q;
            place(e, rr, q);
            resident_quad_at<SOLID, FORCE, RAGGED, SAT>(a, v, src, dst, S + (size_t)rr * Pq, pstride, rr + 1, y0 + rr, q, o);
            if (e < edge) hand_over(rr, q, o);
        }
        if (G > 1 && more) {
            // The neighbours' edge rows of the new state, into the extra rows:
            // units in the order below (planes 3, 4), above (planes 0, 1), the
            // last warps first.
            for (int i = T - 1 - tid; i < 4 * nq; i += T) {
                const int k = (int)(((unsigned long long)(uint32_t)i * ra.nq_magic) >> 32), q = i - k * nq;
                uint4 w;
                if (!get_unit(k < 2 ? unit(par, below, 1, k, q) : unit(par, above, 0, k - 2, q), (uint32_t)(s + 1), w)) {
                    ok = false;
                    break;
                }
                if (k < 2) st4(dst + (3 + k) * pstride + 4 * q, w);
                else st4(dst + (k - 2) * pstride + (size_t)(n + 1) * Pq + 4 * q, w);
            }
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0 && a.err) atomicOr(a.err, 1u);
            return;
        }
    }
    // The owned rows of the final state.
    const uint32_t* fin = X[ra.nsteps & 1];
    uint32_t* out = (ra.nsteps & 1) ? ra.buf1 : ra.buf0;
    for (int i = tid; i < 7 * n * q4; i += T) {
        const int p = i / (n * q4), rem = i - p * n * q4, lr = rem / q4 + 1, w = 4 * (rem % q4);
        st4(out + (size_t)p * a.plane_words + (size_t)(y0 + lr - 1) * Pq + w, ld4(fin + p * pstride + (size_t)lr * Pq + w));
    }
}

std::mutex g_res_mutex;
int g_res_sms[64] = {};
bool g_res_configured[64][2][2][2][2] = {};

template <bool SOLID, bool FORCE, bool RAGGED, bool SAT>
cudaError_t launch_resident_variant(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, cudaStream_t s) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    return launch_resident_coop((const void*)fhp_resident_kernel<SOLID, FORCE, RAGGED, SAT>,
                                &g_res_configured[dev][SOLID][FORCE][RAGGED][SAT], a, ra, grid, kRes1Threads, smem, s);
}

template <bool SOLID, bool FORCE>
cudaError_t launch_resident_sf(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, bool ragged, bool sat,
                               cudaStream_t s) {
    if (sat)
        return ragged ? launch_resident_variant<SOLID, FORCE, true, true>(a, ra, grid, smem, s)
                      : launch_resident_variant<SOLID, FORCE, false, true>(a, ra, grid, smem, s);
    return ragged ? launch_resident_variant<SOLID, FORCE, true, false>(a, ra, grid, smem, s)
                  : launch_resident_variant<SOLID, FORCE, false, false>(a, ra, grid, smem, s);
}

cudaError_t launch_resident_one(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, bool has_solid,
                                bool force, bool ragged, bool sat, cudaStream_t s) {
    if (has_solid)
        return force ? launch_resident_sf<true, true>(a, ra, grid, smem, ragged, sat, s)
                     : launch_resident_sf<true, false>(a, ra, grid, smem, ragged, sat, s);
    return force ? launch_resident_sf<false, true>(a, ra, grid, smem, ragged, sat, s)
                 : launch_resident_sf<false, false>(a, ra, grid, smem, ragged, sat, s);
}

}  // namespace

cudaError_t launch_resident_coop(const void* fn, bool* configured, const StepArgs& a, const ResArgs& ra, int grid,
                                 int threads, size_t smem, cudaStream_t s) {
    {
        std::lock_guard<std::mutex> lock(g_res_mutex);
        if (!*configured) {
            const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmemLimit);
            if (e != cudaSuccess) return e;
            *configured = true;
        }
    }
    StepArgs a_ = a;
    ResArgs ra_ = ra;
    void* args[] = {(void*)&a_, (void*)&ra_};
    const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, smem, s);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Shared memory of one CTA: two staged copies of its strip (nmax owned rows,
// 1 extra row per side for gh = 1, gh ghost rows per side otherwise; 7 planes)
// and its solid rows.
size_t resident_smem(const Geometry& g, bool has_solid, int grid, int gh) {
    if (grid <= 0) return 0;
    const int nmax = (g.H + grid - 1) / grid;
    const int staged = nmax + 2 * gh;
    const int solid_rows = has_solid ? (gh == 1 ? nmax : staged) : 0;
    return (size_t)(2 * 7 * staged + solid_rows) * g.Pq * 4;
}

// CTAs of the resident kernels: at most one per SM; one-row exchange: strips
// of at least two rows, and a single CTA for lattices of at most kLoneQuads
// quads (128 x 128: 0.83 us a step; 256 x 128, 256 quads: 1.1 us; 256 x 256, 512
// quads: 1.66 us in one SM, 1.37 us in 128 strips).
int resident_grid(const Geometry& g, bool has_solid, int gh) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int sms;
    {
        std::lock_guard<std::mutex> lock(g_res_mutex);
        if (!g_res_sms[dev] &&
            cudaDeviceGetAttribute(&g_res_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return 0;
        sms = g_res_sms[dev];
    }
    if (gh > 1) return g.H < sms ? g.H : sms;
    if ((long long)g.nq * g.H <= kLoneQuads && resident_smem(g, has_solid, 1, 1) <= (size_t)kResSmemLimit) return 1;
    return g.H / 2 < sms ? g.H / 2 : sms;
}

// Exchange buffer words: 2 parities x G CTAs x 2 sides x (2 planes of one row
// as nq units of 8 words for gh = 1, 7 (gh - 1) + 2 row planes of Pq words
// otherwise).
size_t resident_halo_words(const Geometry& g, bool has_solid, int gh) {
    const size_t per_side = gh == 1 ? (size_t)2 * g.nq * 8 : (size_t)(7 * (gh - 1) + 2) * g.Pq;
    return (size_t)2 * resident_grid(g, has_solid, gh) * 2 * per_side;
}

bool resident_supported(const Geometry& g, bool has_solid, size_t staging_bytes, int gh) {
    if ((gh != 1 && gh != 2) || (gh > 1 && g.rules == 3)) return false;   // (two ghost rows: not FHP-III)
    const int grid = resident_grid(g, has_solid, gh);
    if (grid <= 0) return false;
    if (gh > 1 && g.H / grid < 2 * gh) return false;   // every strip holds its 2 gh edge rows
    return resident_smem(g, has_solid, grid, gh) <= (size_t)kResSmemLimit &&
           resident_halo_words(g, has_solid, gh) * sizeof(uint32_t) <= staging_bytes;
}

cudaError_t launch_resident(const Geometry& g, uint32_t* buf0, uint32_t* buf1, const uint32_t* solid, bool has_solid,
                            bool force, const ForcingTable& ft, Key2 key, uint64_t t0, int nsteps, int gh,
                            uint32_t* halo, unsigned int* flags, cudaStream_t stream, unsigned int* err) {
    const int grid = resident_grid(g, has_solid, gh);
    if (grid <= 0 || nsteps <= 0 || (gh != 1 && gh != 2) || (gh > 1 && g.H / grid < 2 * gh))
        return cudaErrorInvalidValue;
    const size_t smem = resident_smem(g, has_solid, grid, gh);
    if (smem > (size_t)kResSmemLimit) return cudaErrorInvalidValue;
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
    ra.halo = halo;
    ra.flags = flags;
    ra.nsteps = nsteps;
    ra.t0 = t0;
    ra.nmax = (g.H + grid - 1) / grid;
    ra.nq_magic = ((1ull << 32) + g.nq - 1) / g.nq;
    cudaError_t e = cudaSuccess;
    if (gh > 1) e = cudaMemsetAsync(flags, 0, (size_t)grid * sizeof(unsigned int), stream);
    else if (grid > 1 && nsteps > 1)   // no unit carries a step of this call
        e = cudaMemsetAsync(halo, 0, resident_halo_words(g, has_solid, 1) * sizeof(uint32_t), stream);
    if (e != cudaSuccess) return e;
    const bool ragged = g.Wq % 4 != 0;
    return gh == 1 ? launch_resident_one(a, ra, grid, smem, has_solid, force, ragged, g.rules == 3, stream)
                   : launch_resident_ghost2(a, ra, grid, smem, has_solid, force, ragged, stream);
}

}  // namespace fhp
