// fhp_resident.cuh -- lattices that fit in the SMs' shared memory: the whole
// lattice stays on chip for all steps of a call.
//
// One cooperative launch, one CTA per SM at most.  CTA b owns rows [y0, y1) of
// the lattice (a contiguous strip of at least 2 GH) and keeps them, with GH
// ghost rows below and above, in two shared-memory buffers (steps alternate
// between them).  A step pulls the movers from the rows y-1 (north-going planes
// 3, 4), y (planes 2, 5, 6) and y+1 (south-going planes 0, 1) of the staged
// strip, scatters with the same per-quad code as every other step kernel
// (random words keyed on the lattice's row, so results are identical), and
// writes the new state into the other buffer.  HBM sees the lattice once at
// the start and once at the end of the call.
//
// Every GH steps the strips exchange edge rows.  In step j of such a round the
// rows that can still be computed exactly lose one at each end; after the
// round exactly the owned rows are exact.  From below a strip needs planes 3, 4
// of the outermost ghost row, planes 2 .. 6 of the next and all planes of the
// others (mirrored from above: planes 0, 1, then 0, 1, 2, 5, 6).
//
// The hand-off between SMs is what bounds small lattices, and it is one store
// and one load long: every 32-bit word travels in a 64-bit store together with
// the number of the step it belongs to, and the reader polls the word itself
// until it carries that number.  (Rows, fence, release of a counter, acquire,
// load of the rows -- the former protocol -- are five trips to L2 in a row: 3.2
// us a step on 4096 x 1024, p = 1e-3, with GH = 2; 1.86 us with this one and GH
// = 1.)  Rows alternate between two slots: a CTA
// overwrites a slot two rounds later, when its neighbours' words of the round
// between have told it that they had read it.  Edge rows are computed first,
// the draws of a thread's first quad are made before the wait, and warps
// without a quad do the polling, so on larger strips the hand-off hides behind
// the interior rows.
//
// A lattice of at most kLoneQuads quads stays in one SM (GH = 1; its ghost rows
// are its own edge rows): 16 warps step it faster than a hand-off takes.
#pragma once

#include <cuda_runtime.h>

#include <mutex>

#include "fhp_device.cuh"
#include "fhp_internal.h"
#include "fhp_quad.cuh"

namespace fhp {

constexpr int kRes1Threads = 512;  // 16 warps at <= 128 registers
constexpr int kResSmemLimit = 224 * 1024;
constexpr int kLoneQuads = 160;

struct ResArgs {
    uint32_t* buf0;        // state at t0
    uint32_t* buf1;
    uint32_t* halo;        // exchanged units of 32 bytes: [2 slots][G][2 sides][units][nq], zero at launch
    int nsteps;
    int flip;              // the result goes to buf1 (resident_flips), else to buf0
    unsigned long long t0;
    int nmax;              // most rows any CTA owns
    unsigned long long nq_magic;   // ceil(2^32 / nq): j / nq == (j * nq_magic) >> 32 for small j
};

// Launches the kernel of GH ghost rows per side (1, 2 or 4; fhp_resident_g<GH>.cu).
template <int GH>
cudaError_t launch_resident_g(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, bool has_solid, bool force,
                              bool ragged, bool sat, cudaStream_t s);

namespace {

// One quad (quad q of strip row rr, lattice row y0 + rr) of a step: pulls the
// movers from the staged rows of `src`, scatters, and writes the seven planes
// of the new state into `dst` (padding words of a ragged row stay zero).
// (Local row lr of the staged buffers, lattice row y, `Srow` its solid row.)
// (resident_quad_drawn takes the quad's random blocks from the caller.)
template <bool SOLID, bool FORCE, bool RAGGED, bool SAT = false>
__device__ __forceinline__ void resident_quad_drawn(const StepArgs& a, const StepVar& v, const uint32_t* src,
                                                    uint32_t* dst, const uint32_t* Srow, int pstride, int lr, int y,
                                                    int q, uint4 chi, uint4 gate, uint4 (&o)[7]) {
    const int Pq = a.Pq;
    const int w = 4 * q;
    const int m = RAGGED ? (q == a.nq - 1 ? a.Wq - w : 4) : 4;
    const int wl = q == 0 ? a.Wq - 1 : w - 1;
    const int wr = q == a.nq - 1 ? 0 : w + 4;
    const uint32_t* rm = src + (lr - 1) * Pq;   // row y - 1
    const uint32_t* r0 = src + lr * Pq;         // row y
    const uint32_t* rp = src + (lr + 1) * Pq;   // row y + 1
    const uint4 i3 = ld4(rm + 3 * pstride + w), i4 = ld4(rm + 4 * pstride + w);
    const uint4 i2 = ld4(r0 + 2 * pstride + w), i5 = ld4(r0 + 5 * pstride + w);
    const uint4 i6 = ld4(r0 + 6 * pstride + w);
    const uint4 i0 = ld4(rp + 0 * pstride + w), i1 = ld4(rp + 1 * pstride + w);
    uint4 sd = make_uint4(0u, 0u, 0u, 0u);
    if (SOLID) sd = ld4(Srow + w);
    uint4 n0, n1, n2, n3, n4, n5;
    if ((y & 1) == 0) {
        n2 = pull_left(i2, r0[2 * pstride + wl]);
        n3 = pull_left(i3, rm[3 * pstride + wl]);
        n1 = pull_left(i1, rp[1 * pstride + wl]);
        n5 = pull_right<RAGGED>(i5, r0[5 * pstride + wr], m);
        n4 = i4;
        n0 = i0;
    } else {
        n2 = pull_left(i2, r0[2 * pstride + wl]);
        n5 = pull_right<RAGGED>(i5, r0[5 * pstride + wr], m);
        n4 = pull_right<RAGGED>(i4, rm[4 * pstride + wr], m);
        n0 = pull_right<RAGGED>(i0, rp[0 * pstride + wr], m);
        n3 = i3;
        n1 = i1;
    }
    collide_drawn<SOLID, FORCE, SAT>(a, v, q, y, chi, gate, n0, n1, n2, n3, n4, n5, i6, sd, o);
    if (RAGGED && m < 4) {
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            if (m < 2) o[k].y = 0u;
            if (m < 3) o[k].z = 0u;
            o[k].w = 0u;
        }
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) st4(dst + k * pstride + lr * Pq + w, o[k]);
}

template <bool FORCE>
__device__ __forceinline__ void resident_draws(const StepArgs& a, const StepVar& v, int q, int y, uint4& chi,
                                               uint4& gate) {
    const uint32_t y_key = (uint32_t)(y + a.y_base);
    chi = rng_block((uint32_t)q, y_key, v.t_lo, v.t_hi, 0u, a.key);
    gate = FORCE ? rng_block((uint32_t)q, y_key, v.t_lo, v.t_hi, 1u, a.key) : make_uint4(0u, 0u, 0u, 0u);
}

template <bool SOLID, bool FORCE, bool RAGGED, bool SAT = false>
__device__ __forceinline__ void resident_quad_at(const StepArgs& a, const StepVar& v, const uint32_t* src,
                                                 uint32_t* dst, const uint32_t* Srow, int pstride, int lr, int y,
                                                 int q, uint4 (&o)[7]) {
    uint4 chi, gate;
    resident_draws<FORCE>(a, v, q, y, chi, gate);
    resident_quad_drawn<SOLID, FORCE, RAGGED, SAT>(a, v, src, dst, Srow, pstride, lr, y, q, chi, gate, o);
}

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

// Exchanged planes ("units" of a quad) of one side: the outermost ghost row
// has 2, the next 5, the others 7.
template <int GH>
constexpr int kResUnits = GH == 1 ? 2 : 7 + 7 * (GH - 2);

// Whether a ghost row at distance d from the outermost one is given plane p,
// and as which unit; UP: rows handed upwards (ghost rows below a strip).
template <bool UP>
__device__ __forceinline__ bool res_unit(int d, int p, int& u) {
    if (d == 0) {
        u = UP ? p - 3 : p;
        return UP ? p == 3 || p == 4 : p < 2;
    }
    if (d == 1) {
        u = UP ? p : p < 3 ? 2 + p : p;         // planes 2..6, or 0, 1, 2, 5, 6, as units 2..6
        return UP ? p >= 2 : p < 3 || p >= 5;
    }
    u = 7 + 7 * (d - 2) + p;
    return true;
}

// SAT: the FHP-III rule set.
template <bool SOLID, bool FORCE, bool RAGGED, bool SAT, int GH>
__global__ void __launch_bounds__(kRes1Threads, 1) fhp_resident_kernel(const StepArgs a, const ResArgs ra) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int T = kRes1Threads, NU = kResUnits<GH>;
    const int G = (int)gridDim.x, b = (int)blockIdx.x;
    const int y0 = (int)(((long long)b * a.H) / G), y1 = (int)(((long long)(b + 1) * a.H) / G);
    const int n = y1 - y0, L = n + 2 * GH;             // owned rows; staged rows
    const int Pq = a.Pq, q4 = Pq / 4, nq = a.nq;
    const int pstride = (ra.nmax + 2 * GH) * Pq;       // words per staged plane
    // The two buffers are offsets from one shared-memory pointer: taken from an
    // array of two pointers their loads became generic ones behind a local load.
    uint32_t* const X = reinterpret_cast<uint32_t*>(smem_raw);
    const int half = 7 * pstride;
    uint32_t* const S = X + 2 * half;                  // solid rows of staged rows 1 .. L - 2 (SOLID only)
    const int below = b == 0 ? G - 1 : b - 1, above = b == G - 1 ? 0 : b + 1;
    const int tid = (int)threadIdx.x;
    unsigned long long* halo = reinterpret_cast<unsigned long long*>(ra.halo);
    // Unit u of quad q handed over by `cta` in a round; side 0: downwards
    // (its lowest rows), side 1: upwards.
    auto unit = [&](int par, int cta, int side, int u, int q) {
        return halo + ((((size_t)(par * G + cta) * 2 + side) * NU + u) * nq + q) * 4;
    };
    auto lattice_row = [&](int lr) {                   // lattice row of staged row lr (periodic)
        int y = y0 - GH + lr;
        if (y < 0) y += a.H;
        return y >= a.H ? y - a.H : y;
    };

    for (int i = tid; i < 7 * L * q4; i += T) {
        const int p = i / (L * q4), rem = i - p * L * q4, lr = rem / q4, w = 4 * (rem % q4);
        st4(X + p * pstride + lr * Pq + w,
            ld4(ra.buf0 + (size_t)p * a.plane_words + (size_t)lattice_row(lr) * Pq + w));
    }
    if (SOLID)
        for (int i = tid; i < (L - 2) * q4; i += T) {
            const int lr = 1 + i / q4, w = 4 * (i % q4);
            st4(S + (lr - 1) * Pq + w, ld4(a.solid + (size_t)lattice_row(lr) * Pq + w));
        }

    // Quads of step j of a round: staged rows 1 + j .. L - 2 - j; in the last
    // step (the owned rows) the 2 GH rows that are handed over come first.
    auto items_of = [&](int j) { return (n + 2 * (GH - 1 - j)) * nq; };
    auto place = [&](int j, int e, int& lr, int& q) {
        const int k = (int)(((unsigned long long)(uint32_t)e * ra.nq_magic) >> 32);   // e / nq
        q = e - k * nq;
        if (j < GH - 1) lr = 1 + j + k;
        else lr = GH + (k < GH ? k : k < 2 * GH ? n - 2 * GH + k : k - GH);
    };
    auto step_of = [&](int s) {
        const unsigned long long t = ra.t0 + (unsigned long long)s;
        return StepVar{nullptr, (uint32_t)t, (uint32_t)(t >> 32)};
    };
    int lr0 = 0, q0 = 0;
    uint4 chi = make_uint4(0u, 0u, 0u, 0u), gate = chi;
    if (tid < items_of(0)) {
        place(0, tid, lr0, q0);
        resident_draws<FORCE>(a, step_of(0), q0, lattice_row(lr0), chi, gate);
    }
    __syncthreads();

    int j = 0;          // step of the round
    int round = 1;      // rounds handed over, counting the one under way
    for (int s = 0; s < ra.nsteps; ++s) {
        const uint32_t* src = X + (s & 1 ? half : 0);
        uint32_t* dst = X + (s & 1 ? 0 : half);
        const StepVar v = step_of(s);
        const bool more = s + 1 < ra.nsteps;
        const bool exchange = j == GH - 1 && more;
        const int par = round & 1, items = items_of(j);
        bool ok = true;
        // Edge rows go to the neighbours (or, alone, to the strip's own ghost rows).
        auto hand_over = [&](int lr, int q, const uint4 (&o)[7]) {
            const int rr = lr - GH;
            if (G == 1) {
                if (rr == 0) {
                    st4(dst + (n + 1) * Pq + 4 * q, o[0]);
                    st4(dst + pstride + (n + 1) * Pq + 4 * q, o[1]);
                } else if (rr == n - 1) {
                    st4(dst + 3 * pstride + 4 * q, o[3]);
                    st4(dst + 4 * pstride + 4 * q, o[4]);
                }
                return;
            }
            int u;
            if (rr < GH) {
#pragma unroll
                for (int p = 0; p < 7; ++p)
                    if (res_unit<false>(GH - 1 - rr, p, u)) put_unit(unit(par, b, 0, u, q), o[p], (uint32_t)(s + 1));
            }
            if (rr >= n - GH) {
#pragma unroll
                for (int p = 0; p < 7; ++p)
                    if (res_unit<true>(rr - (n - GH), p, u)) put_unit(unit(par, b, 1, u, q), o[p], (uint32_t)(s + 1));
            }
        };
        uint4 o[7];
        if (tid < items) {
            resident_quad_drawn<SOLID, FORCE, RAGGED, SAT>(a, v, src, dst, S + (lr0 - 1) * Pq, pstride, lr0,
                                                           lattice_row(lr0), q0, chi, gate, o);
            if (exchange) hand_over(lr0, q0, o);
        }
        const int jn = j == GH - 1 ? 0 : j + 1;
        if (more && tid < items_of(jn)) {
            if (GH > 1) place(jn, tid, lr0, q0);
            resident_draws<FORCE>(a, step_of(s + 1), q0, lattice_row(lr0), chi, gate);
        }
        for (int e = tid + T; e < items; e += T) {
            int lr, q;
            place(j, e, lr, q);
            resident_quad_at<SOLID, FORCE, RAGGED, SAT>(a, v, src, dst, S + (lr - 1) * Pq, pstride, lr,
                                                        lattice_row(lr), q, o);
            if (exchange) hand_over(lr, q, o);
        }
        if (exchange && G > 1) {
            // The neighbours' rows of the new state, into the ghost rows (last
            // warps first).
            for (int i = T - 1 - tid; i < 2 * NU * nq; i += T) {
                const int k = (int)(((unsigned long long)(uint32_t)i * ra.nq_magic) >> 32), q = i - k * nq;
                const bool up = k < NU;       // handed upwards by the strip below
                const int u = up ? k : k - NU;
                uint4 w;
                if (!get_unit(unit(par, up ? below : above, up ? 1 : 0, u, q), (uint32_t)(s + 1), w)) {
                    ok = false;
                    break;
                }
                int d, p;
                if (u < 2) {
                    d = 0;
                    p = up ? 3 + u : u;
                } else if (u < 7) {
                    d = 1;
                    p = up || u >= 5 ? u : u - 2;
                } else {
                    d = 2 + (u - 7) / 7;
                    p = (u - 7) % 7;
                }
                st4(dst + p * pstride + (up ? d : L - 1 - d) * Pq + 4 * q, w);
            }
        }
        if (exchange) ++round;
        j = jn;
        if (__syncthreads_or(!ok)) {
            if (tid == 0 && a.err) atomicOr(a.err, 1u);
            return;
        }
    }
    // The owned rows of the final state.
    const uint32_t* fin = X + (ra.nsteps & 1 ? half : 0);
    uint32_t* out = ra.flip ? ra.buf1 : ra.buf0;
    for (int i = tid; i < 7 * n * q4; i += T) {
        const int p = i / (n * q4), rem = i - p * n * q4, rr = rem / q4, w = 4 * (rem % q4);
        st4(out + (size_t)p * a.plane_words + (size_t)(y0 + rr) * Pq + w,
            ld4(fin + p * pstride + (rr + GH) * Pq + w));
    }
}

template <bool SOLID, bool FORCE, bool RAGGED, bool SAT, int GH>
cudaError_t launch_resident_variant(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, cudaStream_t s) {
    static std::mutex m;
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    auto kernel = fhp_resident_kernel<SOLID, FORCE, RAGGED, SAT, GH>;
    {
        std::lock_guard<std::mutex> lock(m);
        if (!configured[dev]) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmemLimit);
            if (e != cudaSuccess) return e;
            configured[dev] = true;
        }
    }
    StepArgs a_ = a;
    ResArgs ra_ = ra;
    void* args[] = {(void*)&a_, (void*)&ra_};
    e = cudaLaunchCooperativeKernel((const void*)kernel, dim3(grid), dim3(kRes1Threads), args, smem, s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <bool SOLID, bool FORCE, int GH>
cudaError_t launch_resident_sf(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, bool ragged, bool sat,
                               cudaStream_t s) {
    if constexpr (GH == 1) {   // (FHP-III: one ghost row only)
        if (sat)
            return ragged ? launch_resident_variant<SOLID, FORCE, true, true, GH>(a, ra, grid, smem, s)
                          : launch_resident_variant<SOLID, FORCE, false, true, GH>(a, ra, grid, smem, s);
    }
    if (sat) return cudaErrorInvalidValue;
    return ragged ? launch_resident_variant<SOLID, FORCE, true, false, GH>(a, ra, grid, smem, s)
                  : launch_resident_variant<SOLID, FORCE, false, false, GH>(a, ra, grid, smem, s);
}

template <int GH>
cudaError_t launch_resident_all(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, bool has_solid, bool force,
                                bool ragged, bool sat, cudaStream_t s) {
    if (has_solid)
        return force ? launch_resident_sf<true, true, GH>(a, ra, grid, smem, ragged, sat, s)
                     : launch_resident_sf<true, false, GH>(a, ra, grid, smem, ragged, sat, s);
    return force ? launch_resident_sf<false, true, GH>(a, ra, grid, smem, ragged, sat, s)
                 : launch_resident_sf<false, false, GH>(a, ra, grid, smem, ragged, sat, s);
}

}  // namespace
}  // namespace fhp
