// fhp_device.cuh -- device building blocks of the FHP step on bit-planes.
//
// A lattice row is stored as words of 32 nodes: bit (x mod 32) of word x/32
// of plane i holds occupation bit i of node x (i = 0..5 movers along c_i at
// (i-2)*60 degrees, 6 rest particle; a separate plane holds the solid flag).
// Every function here works on whole words, so one instruction updates 32
// nodes (multi-spin coding of the node byte of arXiv:1208.2428, Section 2).
#pragma once

#include <cstdint>

#include "fhp_internal.h"
#include "fhp_rules.cuh"

namespace fhp {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of two 32x32
// -> 64-bit products whose halves are swapped and xored with the other two
// counter words and the round key; the key advances by two Weyl constants.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, Key2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned long long a = (unsigned long long)0xD2511F53u * c.x;
        const unsigned long long b = (unsigned long long)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(b >> 32) ^ c.y ^ k.lo, (uint32_t)b, (uint32_t)(a >> 32) ^ c.w ^ k.hi, (uint32_t)a);
        k.lo += 0x9E3779B9u;
        k.hi += 0xBB67AE85u;
    }
    return c;
}

// Random block of the four words 4q..4q+3 of row y at step t for `stream`
// (stream 0: chirality, 1 + d: forcing draw d).  Counter layout:
// (q, y, t mod 2^32, stream + (t div 2^32) * 2^16).
__device__ __forceinline__ uint4 rng_block(uint32_t q, uint32_t y, uint32_t t_lo, uint32_t t_hi,
                                           uint32_t stream, Key2 key) {
    return philox4x32_10(make_uint4(q, y, t_lo, stream | (t_hi << 16)), key);
}

__device__ __forceinline__ uint32_t word_of(const uint4& v, int j) {
    return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w;
}

// ---------------------------------------------------------------------------
// Scattering of 32 nodes at once, as boolean networks (fhp_rules.cuh).
//
// FHP-II: every collision exchanges the particles of a node for another set
// with the same mass and momentum:
//   head-on pair {i, i+3} (others empty)  -> turned by +60 deg (chi 0) or -60 deg (chi 1)
//   triple {0,2,4} <-> {1,3,5}            -> all six movers flip
//   rest + {i}  <->  {i-1, i+1}            -> rest bit and movers i-1, i, i+1 flip
// (each with the rest particle as a spectator where it is not involved).
// FHP-I leaves the last rule out.
//
// FHP-III (collision-saturated): every fluid state that shares its mass and
// momentum with another state changes (k = 0..5, indices of movers mod 6;
// "pair p" = movers p and p+3):
//   zero momentum (every pair full or empty, or a triple): the movers turn
//     by +60 deg (chi 0) or -60 deg (chi 1), the rest particle stays;
//   rest + k <-> {k-1, k+1}                    flip rest, k-1, k, k+1
//   all movers but k+3 <-> rest + {k-1,k,k+1,k+3}   flip rest, k+2, k+3, k+4
//   momentum c_k, mass 3, chi 0: A = k + pair k+1 -> B = k + pair k+2
//     -> C = rest + {k-1, k+1} -> A  (chi 1 backwards)
//   momentum c_k, mass 4, chi 0: D = rest + k + pair k+2 -> E = rest + k +
//     pair k+1 -> F = {k-1, k+1} + pair k -> D  (chi 1 backwards)
//
// Solid nodes reverse every mover (i <-> i+3) and keep the rest particle.
// ---------------------------------------------------------------------------
// RULES 1, 2 or 3; SOLID: the word may hold solid nodes.
template <int RULES, bool SOLID>
__host__ __device__ __forceinline__ Planes7 scatter_rules(const Planes7& in, uint32_t solid, uint32_t chi) {
    if (RULES == 3) return SOLID ? scatter_fhp3_solid(in, chi, solid) : scatter_fhp3(in, chi);
    if (RULES == 1) return SOLID ? scatter_fhp1_solid(in, chi, solid) : scatter_fhp1(in, chi);
    return SOLID ? scatter_fhp2_solid(in, chi, solid) : scatter_fhp2(in, chi);
}

// rest_rules: all ones applies the rest-particle rules (FHP-II), zero skips
// them (FHP-I: head-on and three-body collisions only).
__host__ __device__ __forceinline__ Planes7 scatter(const Planes7& in, uint32_t solid, uint32_t chi,
                                                    uint32_t rest_rules = 0xFFFFFFFFu) {
    return rest_rules ? scatter_rules<2, true>(in, solid, chi) : scatter_rules<1, true>(in, solid, chi);
}

__host__ __device__ __forceinline__ Planes7 scatter_saturated(const Planes7& in, uint32_t solid, uint32_t chi) {
    return scatter_rules<3, true>(in, solid, chi);
}

// ---------------------------------------------------------------------------
// Forcing (ForcingTable: Q_g, g = 0..32, in units of 2^-32 -- a uniform
// u < Q_g means "one of the next g candidates is forced").
// ---------------------------------------------------------------------------
// Forced-node mask of one word: `cand` holds the candidates (fluid, bit 5
// set, bit 2 clear), `u0` is the word's first forcing draw, `more(d)` returns
// draw d >= 1.  Walk: while candidates remain, the least g with u < Q_g picks
// the g-th remaining candidate; candidates before it are not forced; a fresh
// draw decides the ones after it.
template <class MoreDraws>
__device__ __forceinline__ uint32_t forced_mask(uint32_t cand, uint32_t u0, const ForcingTable& ft,
                                                MoreDraws more) {
    uint32_t forced = 0;
    uint32_t u = u0;
    uint32_t draw = 0;
    while (cand) {
        const int remaining = __popc(cand);
        if ((unsigned long long)u >= ft.q[remaining]) break;
        int lo = 1, hi = remaining;  // least g in [1, remaining] with u < Q_g
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((unsigned long long)u < ft.q[mid]) hi = mid; else lo = mid + 1;
        }
        uint32_t c = cand;
        for (int i = 1; i < lo; ++i) c &= c - 1;   // drop the lo-1 lowest candidates
        const int pos = __ffs(c) - 1;              // the lo-th candidate
        forced |= 1u << pos;
        cand = pos == 31 ? 0u : (cand & (0xFFFFFFFFu << (pos + 1)));
        if (!cand) break;   // no candidate left: the next draw would decide nothing
        ++draw;
        u = more(draw);
    }
    return forced;
}

}  // namespace fhp
