// fhp_march.cuh -- k steps per pass with the intermediate time levels in
// registers.
//
// A lane owns one quad column (128 nodes of a row) of a band of R rows and
// marches up the band.  At tick t it computes, for every level j = 1..k, the
// quad of row y0 - k + 2 + t - j of S_{t0+j}: level 1 from the lattice in
// global memory, level j from level j - 1.  A row of level j needs planes 0, 1
// of the row above (just computed at this tick), planes 2, 5, 6 of its own row
// (one tick old) and planes 3, 4 of the row below (two ticks old), so a level
// keeps 7 plane quads (28 registers) per lane and nothing passes through
// shared memory or a barrier; the one-node shifts take the neighbour words
// from the neighbouring lanes by shuffles.  Level k goes to the other state
// buffer.  A pass reads and writes the lattice once.
#pragma once

#include <cuda_runtime.h>

#include <mutex>

#include "fhp_debug.cuh"
#include "fhp_device.cuh"
#include "fhp_internal.h"
#include "fhp_quad.cuh"

namespace fhp {

struct MarchArgs {
    int R;          // rows per band (even)
    int nbands;     // ceil(H / R)
    int pitch;      // chain positions per band (0: whole rows in a warp)
    int left;       // chain positions left of a band's quad 0
    int hl;         // halo lanes per side of a warp (chain)
    int per_warp;   // whole rows: bands per warp
    int nwarps;
    int passes;     // passes of k steps in the launch
    unsigned int* flags;   // passes > 1: per warp, passes finished, counted from `epoch`
    unsigned int epoch;    // no flag is above this at launch
};

constexpr int kMarchWarps = 4;   // warps per CTA (independent of one another)

// Shared-memory ring of a warp: STAGES stages of the seven plane quads a tick
// needs, and a ring of solid quads that outlives them by k - 1 ticks.
template <int K, bool SOLID>
struct MarchRing {
    static constexpr int stages = 3;
    static constexpr int solid_slots = SOLID ? (K <= 2 ? 4 : 8) : 0;   // a power of two >= stages + K - 1
    static constexpr int warp_bytes = (stages * 7 + solid_slots) * 512;
};

// The kernel of the lattice's variant (fhp_march_k<k>.cu): launches it, or
// with launch = false only reports how many of its CTAs an SM holds.
struct MarchVariant {
    bool solid, force, ragged, sat;
};
template <int K>
cudaError_t march_k(const StepArgs& a, const MarchArgs& b, const MarchVariant& v, bool launch, int* blocks_per_sm,
                    cudaStream_t s);

namespace {

template <int V>
struct IntC {
    static constexpr int value = V;
};

__device__ __forceinline__ void march_copy16(uint32_t smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(gmem) : "memory");
}

__device__ __forceinline__ uint4 lds4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr)
                 : "memory");
    return v;
}

struct MarchLane {
    int q, y0;
    int src_left, src_right;
    bool useful;
};

__device__ __forceinline__ MarchLane march_lane(const StepArgs& a, const MarchArgs& b, int gw, int lane) {
    MarchLane L;
    int band;
    if (b.pitch) {
        const int step = 32 - 2 * b.hl;
        const int pos = gw * step + lane;
        band = pos / b.pitch;
        const int e = pos - band * b.pitch;
        int q = e - b.left;
        L.useful = lane >= b.hl && lane < 32 - b.hl && q >= 0 && q < a.nq && band < b.nbands;
        if (q < 0) q += a.nq;
        if (q >= a.nq) q -= a.nq;
        L.q = q;
        L.src_left = lane == 0 ? 0 : lane - 1;
        L.src_right = lane == 31 ? 31 : lane + 1;
    } else {
        const int r = lane / a.nq;
        L.q = lane - r * a.nq;
        band = gw * b.per_warp + r;
        L.useful = r < b.per_warp && band < b.nbands;
        L.src_left = L.q == 0 ? lane + a.nq - 1 : lane - 1;
        L.src_right = L.q == a.nq - 1 ? lane - (a.nq - 1) : lane + 1;
        if (L.src_left > 31) L.src_left = 31;   // (lanes beyond the last whole row: never useful)
    }
    if (band >= b.nbands) band = b.nbands - 1;
    L.y0 = band * b.R;
    return L;
}

// The movers of one quad after motion: n0..n5 from the source planes of the
// rows they stream from (odd: parity of the destination row).
template <bool RAGGED, bool ODD>
__device__ __forceinline__ void march_pull(const MarchLane& L, int m, uint4& i0, uint4& i1, uint4& i2, uint4& i3,
                                           uint4& i4, uint4& i5) {
    auto left = [&](const uint4& v) {
        uint32_t offer = v.w;   // the quad's last valid word
        if (RAGGED) offer = m == 4 ? v.w : m == 3 ? v.z : m == 2 ? v.y : v.x;
        return __shfl_sync(0xFFFFFFFFu, offer, L.src_left);
    };
    auto right = [&](const uint4& v) { return __shfl_sync(0xFFFFFFFFu, v.x, L.src_right); };
    if (!ODD) {
        i2 = pull_left(i2, left(i2));
        i3 = pull_left(i3, left(i3));
        i1 = pull_left(i1, left(i1));
        i5 = pull_right<RAGGED>(i5, right(i5), m);
    } else {
        i2 = pull_left(i2, left(i2));
        i5 = pull_right<RAGGED>(i5, right(i5), m);
        i4 = pull_right<RAGGED>(i4, right(i4), m);
        i0 = pull_right<RAGGED>(i0, right(i0), m);
    }
}

// The forcing walk of a whole warp (all lanes take part) over the quads of
// one tick, one per level.  Bit 4 (j - 1) + c of a lane's `todo` says that word
// c of its level-j quad passed the pre-check; `u_last` is the first draw of the
// lane's last such word (most lanes have one at most; the others draw theirs
// again).  Every lane follows the definition (forced_mask) for one word at a
// time; the thresholds Q_1 .. Q_32 sit in the lanes (lane g - 1 holds Q_g - 1,
// so that u < Q_g is u <= its value) and are looked up by shuffles, and a
// forced node is flipped in the quad's planes 2 and 5.
//
// Levels are walked together, after all of them have scattered: a level needs
// planes 2 and 5 of the level below only at the next tick.  That, one copy of
// this code per tick instead of one per level, and branches around what a
// round does not need took the 16384 x 4096 cylinder (p = 5e-4, k = 2) from
// 3100 to 4000 GSUPS against a walk inside every level.
template <int K, class Planes, class Solid>
__device__ __forceinline__ void force_tick(const StepArgs& a, uint32_t todo, uint32_t u_last, uint32_t q_lane,
                                           uint32_t q, int yr, unsigned long long t0, Planes&& planes, Solid&& solid) {
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    const bool single = (todo & (todo - 1u)) == 0u;
    uint32_t u = u_last, rest = 0, bit = 0, draw = 1, y_key = 0, lev = 0;
    bool need = false;
    // (Every round uses up a word or a candidate of each lane that has any: the
    // bound is never reached.)
#pragma unroll 1
    for (int round = 0; round < 4 * K * 33; ++round) {
        const bool fetch = rest == 0u && todo != 0u;
        if (__any_sync(kAll, fetch)) {   // the lane's next word
            if (fetch) {
                bit = todo & (0u - todo);
                todo ^= bit;
                lev = 0;
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const uint4 sd = solid(j), p2 = *planes(j, 2), p5 = *planes(j, 5);
                    if (bit == (1u << (4 * j))) rest = p5.x & ~(p2.x | sd.x);
                    if (bit == (2u << (4 * j))) rest = p5.y & ~(p2.y | sd.y);
                    if (bit == (4u << (4 * j))) rest = p5.z & ~(p2.z | sd.z);
                    if (bit == (8u << (4 * j))) rest = p5.w & ~(p2.w | sd.w);
                    if (j > 0 && bit >= (1u << (4 * j))) lev = j;
                }
                int y = yr - (int)lev;
                if (y < 0) y += a.H;
                if (y >= a.H) y -= a.H;
                y_key = (uint32_t)(y + a.y_base);
                draw = single ? 2u : 1u;
                need = !single;
            }
            __syncwarp(kAll);
        }
        if (__any_sync(kAll, need)) {
            const unsigned long long t = t0 + lev;
            const uint4 r = rng_block(q, y_key, (uint32_t)t, (uint32_t)(t >> 32), draw, a.key);
            if (need) u = bit & 0x11111111u ? r.x : bit & 0x22222222u ? r.y : bit & 0x44444444u ? r.z : r.w;
            draw += need ? 1u : 0u;
        }
        // Is one of the remaining candidates forced?  (Every lane takes part
        // in the shuffles.)
        const int n = __popc(rest);
        const uint32_t last = __shfl_sync(kAll, q_lane, n > 0 ? n - 1 : 0);
        const bool hit = n > 0 && u <= last;
        if (__any_sync(kAll, hit)) {
            // The least g with u < Q_g, from a lower bound up.
            int g = hit ? (int)min(__umulhi(u, a.ft.inv), 31u) : 0;   // g - 1
#pragma unroll 1
            for (int i = 0; i < 32; ++i) {
                const uint32_t qg = __shfl_sync(kAll, q_lane, g);
                const bool more = hit && u > qg && g < 31;
                if (!__any_sync(kAll, more)) break;
                g += more ? 1 : 0;
            }
            uint32_t c = rest;
#pragma unroll 1
            for (; g > 0; --g) c &= c - 1u;
            __syncwarp(kAll);
            const uint32_t here = hit ? c & (0u - c) : 0u;   // the g-th candidate
            rest = hit ? rest & ~(here | (here - 1u)) : 0u;
            const uint4 m = make_uint4(bit & 0x11111111u ? here : 0u, bit & 0x22222222u ? here : 0u,
                                       bit & 0x44444444u ? here : 0u, bit & 0x88888888u ? here : 0u);
#pragma unroll
            for (int j = 0; j < K; ++j) {
                const uint32_t on = K == 1 || lev == (uint32_t)j ? 0xFFFFFFFFu : 0u;
                uint4 *p2 = planes(j, 2), *p5 = planes(j, 5);
                *p2 = make_uint4(p2->x ^ (m.x & on), p2->y ^ (m.y & on), p2->z ^ (m.z & on), p2->w ^ (m.w & on));
                *p5 = make_uint4(p5->x ^ (m.x & on), p5->y ^ (m.y & on), p5->z ^ (m.z & on), p5->w ^ (m.w & on));
            }
        } else {
            rest = 0;
        }
        need = rest != 0u;
        if (!__any_sync(kAll, (rest | todo) != 0u)) break;
    }
}

// The warps whose rows or columns this warp's bands touch, one per lane (-1:
// none): the writers of every lane's column and of the columns two to either
// side, in the lane's band and the bands below and above.  They read what this
// warp writes and write what it reads.
__device__ __noinline__ int march_neighbours(int nq, int nbands, int pitch, int left, int hl, int per_warp, int band,
                                             int q, int lane) {
    int w[9];
    const int step = 32 - 2 * hl;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        int bb = band + i / 3 - 1, qq = q + 2 * (i % 3 - 1);
        bb = bb < 0 ? bb + nbands : bb >= nbands ? bb - nbands : bb;
        if (qq < 0) qq += nq;
        if (qq < 0) qq += nq;   // (rows of one quad)
        if (qq >= nq) qq -= nq;
        if (qq >= nq) qq -= nq;
        w[i] = pitch ? (bb * pitch + left + qq - hl) / step : bb / per_warp;
    }
    int mine = -1, last = -1;
#pragma unroll 1
    for (int k = 0; k < 32; ++k) {
        int m = 0x7FFFFFFF;
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (w[i] > last) m = min(m, w[i]);
        m = __reduce_min_sync(0xFFFFFFFFu, m);
        if (m == 0x7FFFFFFF) break;
        if (lane == k) mine = m;
        last = m;
    }
    return mine;
}

__device__ __forceinline__ unsigned int march_flag(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Wait until every neighbour has finished `target` passes (bounded).
__device__ __noinline__ bool march_wait(const unsigned int* flags, int neighbour, unsigned int target) {
    unsigned long long start = 0;
    for (;;) {
        const bool ok = neighbour < 0 || march_flag(flags + neighbour) >= target;
        if (__all_sync(0xFFFFFFFFu, ok)) {
            __syncwarp();
            return true;
        }
        const unsigned long long now = __shfl_sync(0xFFFFFFFFu, global_ns(), 0);
        if (start == 0) start = now;
        else if (now - start > kWaitLimitNs) return false;
        __nanosleep(40);
    }
}

template <int K, bool SOLID, bool FORCE, bool RAGGED, bool SAT>
__device__ __forceinline__ void march_warp(const StepArgs& a, const MarchArgs& b, int gw, uint32_t ring,
                                           uint32_t q_lane) {
    using Ring = MarchRing<K, SOLID>;
    constexpr int D = Ring::stages;
    const int lane = (int)threadIdx.x & 31;
    const MarchLane L = march_lane(a, b, gw, lane);
    const int H = a.H;
    const int m = RAGGED ? (L.q == a.nq - 1 ? a.Wq - 4 * L.q : 4) : 4;
    const uint32_t row_bytes = (uint32_t)a.Pq * 4u;
    const uint32_t lane_base = ring + 16u * (uint32_t)lane;
    const uint32_t solid_base = lane_base + (uint32_t)(D * 7 * 512);
    const size_t pb = (size_t)a.plane_words * 4;
    const int ticks = b.R + 2 * (K - 1);
    int neighbour = -1;
    if (b.passes > 1) 
        neighbour = march_neighbours(a.nq, b.nbands, b.pitch, b.left, b.hl, b.per_warp, L.y0 / b.R, L.q, lane);

#pragma unroll 1
    for (int pass = 0; pass < b.passes; ++pass) {
    const char* src = reinterpret_cast<const char*>((pass & 1) ? a.dst : a.src);
    char* dst = reinterpret_cast<char*>((pass & 1) ? const_cast<uint32_t*>(a.src) : a.dst);
    if (pass > 0 && !march_wait(b.flags, neighbour, b.epoch + (unsigned int)pass)) {
        if (lane == 0 && a.err) atomicOr(a.err, 1u);
        return;
    }

    // Rows y0 - K + i of the lattice (periodic), as byte offsets in a plane.
    int yc = L.y0 - K;
    if (yc < 0) yc += H;
    uint32_t off_a = (uint32_t)yc * row_bytes + 16u * (uint32_t)L.q;   // row i = t
    auto next_row = [&](uint32_t off) {
        if (++yc == H) {
            yc = 0;
            return 16u * (uint32_t)L.q;
        }
        return off + row_bytes;
    };
    uint32_t off_b = next_row(off_a);   // row t + 1
    uint32_t off_c = next_row(off_b);   // row t + 2
    int st_in = 0, sol_in = 0, bundle = 0;
    auto issue = [&]() {
        if (bundle++ >= ticks) {
            asm volatile("cp.async.commit_group;" ::: "memory");   // (an empty group keeps the count)
            return;
        }
        const uint32_t s = lane_base + (uint32_t)(st_in * 7 * 512);
        if (!dbg_ok(off_a + 16u <= pb && off_b + 16u <= pb && off_c + 16u <= pb, a.err, kSiteMarchLoad)) {
            off_a = off_b = off_c = 0;
            yc = 0;
        }
        march_copy16(s, src + off_c);
        march_copy16(s + 512, src + pb + off_c);
        march_copy16(s + 1024, src + 2 * pb + off_b);
        march_copy16(s + 1536, src + 3 * pb + off_a);
        march_copy16(s + 2048, src + 4 * pb + off_a);
        march_copy16(s + 2560, src + 5 * pb + off_b);
        march_copy16(s + 3072, src + 6 * pb + off_b);
        if (SOLID) {
            march_copy16(solid_base + (uint32_t)sol_in * 512u, reinterpret_cast<const char*>(a.solid) + off_b);
            sol_in = (sol_in + 1) & (Ring::solid_slots - 1);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (++st_in == D) st_in = 0;
        off_a = off_b;
        off_b = off_c;
        off_c = next_row(off_c);
    };
#pragma unroll
    for (int s = 0; s < D - 1; ++s) issue();

    uint4 c256[K > 1 ? K - 1 : 1][3], c34[K > 1 ? K - 1 : 1][2][2];
#pragma unroll
    for (int j = 0; j < K - 1; ++j) {
#pragma unroll
        for (int i = 0; i < 3; ++i) c256[j][i] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int i = 0; i < 4; ++i) c34[j][i >> 1][i & 1] = make_uint4(0u, 0u, 0u, 0u);
    }
    int st_out = 0, sol_out = 0;
    int yr = L.y0 - K + 1;   // row of level 1 (unwrapped)
    uint32_t off_dst = (uint32_t)L.y0 * row_bytes + 16u * (uint32_t)L.q;
    int rows_left = L.useful ? min(b.R, H - L.y0) : 0;
    const unsigned long long t0 =
        (((unsigned long long)a.t_hi << 32) | a.t_lo) + (unsigned long long)pass * (unsigned long long)K;

    // Tick t of parity P (t & 1) with the first J levels running: level j has
    // its first valid row at tick 2 (j - 1).  Without forcing the first ticks are
    // written out, so that the loop holds no conditions and moves fewer
    // registers about (2 to 14 % faster).  With forcing their copies of the walk
    // crowd the instruction cache where bands are low (16384 x 4096, p = 5e-4:
    // 3590 GSUPS against 3930), so the loop skips levels by the tick instead.
    constexpr bool PEEL = !FORCE;
    auto tick = [&](int t, auto par, auto levels) {
        constexpr int P = decltype(par)::value, J = decltype(levels)::value;
        asm volatile("cp.async.wait_group %0;" ::"n"(D - 2) : "memory");
        const uint32_t s = lane_base + (uint32_t)(st_out * 7 * 512);
        uint4 i0 = lds4(s), i1 = lds4(s + 512), i2 = lds4(s + 1024), i3 = lds4(s + 1536), i4 = lds4(s + 2048),
              i5 = lds4(s + 2560), i6 = lds4(s + 3072);
        if (++st_out == D) st_out = 0;
        issue();
        uint4 o[7];
        uint32_t todo = 0, u_last = 0;
#pragma unroll
        for (int j = 1; j <= J; ++j) {
            if (!PEEL && j > 1 && t < 2 * (j - 1)) break;
            uint4 sd = make_uint4(0u, 0u, 0u, 0u);
            if (SOLID) sd = lds4(solid_base + (uint32_t)((sol_out - (j - 1)) & (Ring::solid_slots - 1)) * 512u);
            if (j > 1) {
                uint4 p34[2] = {c34[j - 2][P][0], c34[j - 2][P][1]};
                i0 = o[0];
                i1 = o[1];
                i2 = c256[j - 2][0];
                i5 = c256[j - 2][1];
                i6 = c256[j - 2][2];
                i3 = p34[0];
                i4 = p34[1];
                c34[j - 2][P][0] = o[3];
                c34[j - 2][P][1] = o[4];
                c256[j - 2][0] = o[2];
                c256[j - 2][1] = o[5];
                c256[j - 2][2] = o[6];
            }
            // Row parity: y0 is even, level 1 is at row y0 - K + 1 + t.
            constexpr int kOdd0 = (K + 1 + P) & 1;
            int y = yr - (j - 1);
            if (y < 0) y += H;
            if (y >= H) y -= H;
            const unsigned long long tt = t0 + (unsigned long long)(j - 1);
            const StepVar v{nullptr, (uint32_t)tt, (uint32_t)(tt >> 32)};
            if (((kOdd0 + j - 1) & 1) != 0) march_pull<RAGGED, true>(L, m, i0, i1, i2, i3, i4, i5);
            else march_pull<RAGGED, false>(L, m, i0, i1, i2, i3, i4, i5);
            collide_quad<SOLID, false, SAT>(a, v, L.q, y, i0, i1, i2, i3, i4, i5, i6, sd, o);
            if (FORCE) {
                const uint32_t y_key = (uint32_t)(y + a.y_base);
                const uint4 gate = rng_block((uint32_t)L.q, y_key, v.t_lo, v.t_hi, 1u, a.key);
                const bool dense = a.ft.dense != 0u;
                auto check = [&](uint32_t u, uint32_t cand, uint32_t bit) {
                    if (dense || u < (uint32_t)__popc(cand) * a.ft.pre) {
                        todo |= bit << (4 * j - 4);
                        u_last = u;
                    }
                };
                check(gate.x, o[5].x & ~(o[2].x | sd.x), 1u);
                check(gate.y, o[5].y & ~(o[2].y | sd.y), 2u);
                check(gate.z, o[5].z & ~(o[2].z | sd.z), 4u);
                check(gate.w, o[5].w & ~(o[2].w | sd.w), 8u);
            }
        }
        if constexpr (J < K) {   // the topmost level that runs keeps its newest row
            c34[J - 1][P][0] = o[3];
            c34[J - 1][P][1] = o[4];
            c256[J - 1][0] = o[2];
            c256[J - 1][1] = o[5];
            c256[J - 1][2] = o[6];
        }
        if (!PEEL && K > 1 && t < 2 * (K - 1)) {
#pragma unroll
            for (int j = 1; j < K; ++j)
                if (t >= 2 * (j - 1) && t < 2 * j) {
                    c34[j - 1][P][0] = o[3];
                    c34[j - 1][P][1] = o[4];
                    c256[j - 1][0] = o[2];
                    c256[j - 1][1] = o[5];
                    c256[j - 1][2] = o[6];
                }
        }
        if (FORCE && __any_sync(0xFFFFFFFFu, todo != 0u))
            force_tick<J>(
                a, todo, u_last, q_lane, (uint32_t)L.q, yr, t0,
                [&](int j, int plane) -> uint4* {
                    return j == K - 1 ? &o[plane] : &c256[j][plane == 2 ? 0 : 1];
                },
                [&](int j) {
                    return SOLID ? lds4(solid_base + (uint32_t)((sol_out - j) & (Ring::solid_slots - 1)) * 512u)
                                 : make_uint4(0u, 0u, 0u, 0u);
                });
        if (PEEL ? J == K : t >= 2 * (K - 1)) {
            if (rows_left > 0) {
                if (RAGGED && m < 4) {
#pragma unroll
                    for (int k = 0; k < 7; ++k) {
                        if (m < 2) o[k].y = 0u;
                        if (m < 3) o[k].z = 0u;
                        o[k].w = 0u;
                    }
                }
                char* d = dst + off_dst;
                if (dbg_ok(off_dst + 16u <= pb, a.err, kSiteMarchStore)) {
#pragma unroll
                    for (int k = 0; k < 7; ++k) *reinterpret_cast<uint4*>(d + k * pb) = o[k];
                }
            }
            --rows_left;
            off_dst += row_bytes;
        }
        ++yr;
        ++sol_out;
    };
    if constexpr (PEEL && K >= 2) {
        tick(0, IntC<0>{}, IntC<1>{});
        tick(1, IntC<1>{}, IntC<1>{});
    }
    if constexpr (PEEL && K >= 3) {
        tick(2, IntC<0>{}, IntC<2>{});
        tick(3, IntC<1>{}, IntC<2>{});
    }
#pragma unroll 1
    for (int t = PEEL ? 2 * (K - 1) : 0; t < ticks; t += 2) {
        tick(t, IntC<0>{}, IntC<K>{});
        tick(t + 1, IntC<1>{}, IntC<K>{});
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (pass + 1 < b.passes) {
        __syncwarp();
        if (lane == 0) {
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(b.flags + gw), "r"(b.epoch + (unsigned int)pass + 1u)
                         : "memory");
        }
    }
    }
}

template <int K, bool SOLID, bool FORCE, bool RAGGED, bool SAT>
__global__ void __launch_bounds__(32 * kMarchWarps, K <= 2 ? 4 : (K == 3 ? 3 : 2))
    fhp_march_kernel(const StepArgs a, const MarchArgs b) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int warp = (int)threadIdx.x >> 5;
    const int gw = (int)blockIdx.x * kMarchWarps + warp;
    if (gw >= b.nwarps) return;
    march_warp<K, SOLID, FORCE, RAGGED, SAT>(
        a, b, gw, smem_addr(smem_raw) + (uint32_t)(warp * MarchRing<K, SOLID>::warp_bytes),
        FORCE ? (uint32_t)(a.ft.q[(threadIdx.x & 31) + 1] - 1ull) : 0u);
}

template <int K, bool SOLID, bool FORCE, bool RAGGED, bool SAT>
cudaError_t march_variant(const StepArgs& a, const MarchArgs& b, bool launch, int* blocks_per_sm, cudaStream_t s) {
    constexpr int smem = kMarchWarps * MarchRing<K, SOLID>::warp_bytes;
    auto kernel = fhp_march_kernel<K, SOLID, FORCE, RAGGED, SAT>;
    if (!launch) {
        static std::mutex m;
        static int blocks[64] = {};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(m);
        if (!blocks[dev]) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            int n = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, 32 * kMarchWarps, smem);
            if (e != cudaSuccess) return e;
            if (n < 1) return cudaErrorInvalidConfiguration;
            blocks[dev] = n;
        }
        *blocks_per_sm = blocks[dev];
        return cudaSuccess;
    }
    const dim3 grid((unsigned)((b.nwarps + kMarchWarps - 1) / kMarchWarps)), block(32 * kMarchWarps);
    if (b.passes > 1) {
        // The warps wait for one another between passes: all must be resident.
        StepArgs a_ = a;
        MarchArgs b_ = b;
        void* args[] = {&a_, &b_};
        const cudaError_t e = cudaLaunchCooperativeKernel((const void*)kernel, grid, block, args, smem, s);
        if (e != cudaSuccess) return e;
    } else {
        kernel<<<grid, block, smem, s>>>(a, b);
    }
    return cudaGetLastError();
}

template <int K, bool SOLID, bool FORCE>
cudaError_t march_sf(const StepArgs& a, const MarchArgs& b, const MarchVariant& v, bool launch, int* n,
                     cudaStream_t s) {
    if (v.sat)
        return v.ragged ? march_variant<K, SOLID, FORCE, true, true>(a, b, launch, n, s)
                        : march_variant<K, SOLID, FORCE, false, true>(a, b, launch, n, s);
    return v.ragged ? march_variant<K, SOLID, FORCE, true, false>(a, b, launch, n, s)
                    : march_variant<K, SOLID, FORCE, false, false>(a, b, launch, n, s);
}

template <int K>
cudaError_t march_all(const StepArgs& a, const MarchArgs& b, const MarchVariant& v, bool launch, int* n,
                      cudaStream_t s) {
    if (v.solid)
        return v.force ? march_sf<K, true, true>(a, b, v, launch, n, s) : march_sf<K, true, false>(a, b, v, launch, n, s);
    return v.force ? march_sf<K, false, true>(a, b, v, launch, n, s) : march_sf<K, false, false>(a, b, v, launch, n, s);
}

}  // namespace
}  // namespace fhp
