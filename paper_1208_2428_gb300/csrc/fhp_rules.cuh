// fhp_rules.cuh -- the collision rules as networks of three-input boolean
// operations (LOP3) on words of 32 nodes.
//
// A GPU thread evaluates any function of three bits for 32 nodes in one
// instruction, so the cost of a collision is the number of three-input
// operations of its network.  The hand-derived sums of products these
// networks replace took about 65 (FHP-II) and 300 (FHP-III) operations per
// word.  The networks below were found by a randomised search written for
// this purpose: starting from such a sum of products, one operation at a time
// is replaced by another three-input function of other values of the network
// that gives the same outputs wherever a difference could be observed, and
// whatever is no longer used is dropped.  They take 25 (FHP-II), 15 (FHP-I)
// and 43 (FHP-III) operations, and 30, 18 and 47 with the bounce-back of solid nodes.
// Every network is equal to its rule table for all node states and both
// chiralities (compared on the host, tests/test_scatter_logic.py).
#pragma once

#include <cstdint>

namespace fhp {

// Any boolean function of three words: bit 4a + 2b + c of IMM is its value
// for bits a, b, c of x, y, z.
template <uint32_t IMM>
__host__ __device__ __forceinline__ uint32_t lop3(uint32_t x, uint32_t y, uint32_t z) {
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(x), "r"(y), "r"(z), "n"(IMM));
    return r;
#else
    uint32_t r = 0;
    for (uint32_t m = 0; m < 8; ++m)
        if ((IMM >> m) & 1u) r |= ((m & 4u) ? x : ~x) & ((m & 2u) ? y : ~y) & ((m & 1u) ? z : ~z);
    return r;
#endif
}

struct Planes7 {
    uint32_t m0, m1, m2, m3, m4, m5, rest;
};

// FHP-I on fluid nodes: 15 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp1(const Planes7& in, uint32_t chi) {
    const uint32_t g0 = lop3<0x4E>(in.m2, in.m5, chi);
    const uint32_t g1 = lop3<0x27>(in.m0, in.m1, in.m2);
    const uint32_t g2 = lop3<0xDC>(in.m0, in.m1, in.m3);
    const uint32_t g3 = lop3<0x35>(in.m3, in.m4, in.m5);
    const uint32_t g4 = lop3<0xA2>(g1, g2, g3);
    const uint32_t g5 = lop3<0x75>(g0, g1, g4);
    const uint32_t g6 = lop3<0xCE>(in.m2, in.m4, in.m5);
    const uint32_t g7 = lop3<0x24>(g2, g5, g6);
    const uint32_t g8 = lop3<0xA9>(g1, g5, g7);
    const uint32_t g9 = lop3<0x58>(in.m0, g0, g8);
    const uint32_t g10 = lop3<0x52>(in.m1, g0, g8);
    const uint32_t g11 = lop3<0x96>(in.m0, in.m3, g9);
    const uint32_t g12 = lop3<0x34>(in.m2, g7, g11);
    const uint32_t g13 = lop3<0x96>(in.m1, in.m4, g10);
    const uint32_t g14 = lop3<0x34>(in.m5, g7, g9);
    return Planes7{g9, g10, g12, g11, g13, g14, in.rest};
}

// FHP-I, bounce-back on solid nodes: 18 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp1_solid(const Planes7& in, uint32_t chi, uint32_t solid) {
    const uint32_t g0 = lop3<0x4E>(in.m2, in.m5, chi);
    const uint32_t g1 = lop3<0x27>(in.m0, in.m1, in.m2);
    const uint32_t g2 = lop3<0xDC>(in.m0, in.m1, in.m3);
    const uint32_t g3 = lop3<0x35>(in.m3, in.m4, in.m5);
    const uint32_t g4 = lop3<0xA2>(g1, g2, g3);
    const uint32_t g5 = lop3<0x75>(g0, g1, g4);
    const uint32_t g6 = lop3<0xCE>(in.m2, in.m4, in.m5);
    const uint32_t g7 = lop3<0x24>(g2, g5, g6);
    const uint32_t g8 = lop3<0xA9>(g1, g5, g7);
    const uint32_t g9 = lop3<0x58>(in.m0, g0, g8);
    const uint32_t g10 = lop3<0xE2>(in.m3, solid, g9);
    const uint32_t g11 = lop3<0x52>(in.m1, g0, g8);
    const uint32_t g12 = lop3<0xE2>(in.m4, solid, g11);
    const uint32_t g13 = lop3<0x96>(in.m0, in.m3, g10);
    const uint32_t g14 = lop3<0x34>(in.m2, g7, g13);
    const uint32_t g15 = lop3<0xE2>(in.m5, solid, g14);
    const uint32_t g16 = lop3<0x96>(in.m1, in.m4, g12);
    const uint32_t g17 = lop3<0x96>(in.m2, in.m5, g15);
    return Planes7{g10, g12, g15, g13, g16, g17, in.rest};
}

// FHP-II on fluid nodes: 25 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp2(const Planes7& in, uint32_t chi) {
    const uint32_t g0 = lop3<0x36>(in.m0, in.m1, in.m2);
    const uint32_t g1 = lop3<0x36>(in.m3, in.m4, in.m5);
    const uint32_t g2 = lop3<0x0A>(in.m1, g1, g1);
    const uint32_t g3 = lop3<0xA6>(in.m4, g0, g2);
    const uint32_t g4 = lop3<0x91>(in.m1, in.m2, in.m5);
    const uint32_t g5 = lop3<0xE9>(in.m1, in.m4, g4);
    const uint32_t g6 = lop3<0x56>(in.m0, in.m3, g5);
    const uint32_t g7 = lop3<0x84>(in.rest, g3, g6);
    const uint32_t g8 = lop3<0x80>(g0, g1, g6);
    const uint32_t g9 = lop3<0xD9>(in.m0, in.m2, chi);
    const uint32_t g10 = lop3<0xC4>(g3, g8, g9);
    const uint32_t g11 = lop3<0xE8>(in.m0, g8, g10);
    const uint32_t g12 = lop3<0xBC>(in.rest, g7, g8);
    const uint32_t g13 = lop3<0x96>(in.m2, in.m5, g12);
    const uint32_t g14 = lop3<0xB7>(g2, g7, g13);
    const uint32_t g15 = lop3<0x58>(g7, g11, g14);
    const uint32_t g16 = lop3<0x16>(in.m0, g7, g15);
    const uint32_t g17 = lop3<0xC8>(in.m1, g8, g9);
    const uint32_t g18 = lop3<0xA6>(g2, g7, g17);
    const uint32_t g19 = lop3<0x1A>(in.m1, g10, g18);
    const uint32_t g20 = lop3<0xA1>(g5, g14, g18);
    const uint32_t g21 = lop3<0x96>(in.m2, g10, g20);
    const uint32_t g22 = lop3<0x1C>(in.m3, g15, g17);
    const uint32_t g23 = lop3<0x16>(in.m4, g7, g18);
    const uint32_t g24 = lop3<0x96>(in.rest, g13, g21);
    return Planes7{g16, g19, g21, g22, g23, g24, g12};
}

// FHP-II, bounce-back on solid nodes: 30 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp2_solid(const Planes7& in, uint32_t chi, uint32_t solid) {
    const uint32_t g0 = lop3<0x03>(in.m2, in.m5, in.m2);
    const uint32_t g1 = lop3<0xE9>(in.m1, in.m4, g0);
    const uint32_t g2 = lop3<0x56>(in.m0, in.m3, g1);
    const uint32_t g3 = lop3<0x36>(in.m3, in.m4, in.m5);
    const uint32_t g4 = lop3<0x36>(in.m0, in.m1, in.m2);
    const uint32_t g5 = lop3<0x80>(g2, g3, g4);
    const uint32_t g6 = lop3<0x0A>(in.m1, g3, g3);
    const uint32_t g7 = lop3<0xD3>(in.m5, chi, g6);
    const uint32_t g8 = lop3<0x4C>(g1, g5, g7);
    const uint32_t g9 = lop3<0xA6>(in.m4, g4, g6);
    const uint32_t g10 = lop3<0x82>(in.rest, g2, g9);
    const uint32_t g11 = lop3<0xCE>(solid, g8, g10);
    const uint32_t g12 = lop3<0xD6>(in.rest, g8, g11);
    const uint32_t g13 = lop3<0x96>(in.m2, in.m5, g12);
    const uint32_t g14 = lop3<0x48>(g6, g10, g13);
    const uint32_t g15 = lop3<0x36>(in.m0, g11, g14);
    const uint32_t g16 = lop3<0xE2>(in.m3, solid, g15);
    const uint32_t g17 = lop3<0xC8>(in.m4, g5, g7);
    const uint32_t g18 = lop3<0xA6>(g6, g10, g17);
    const uint32_t g19 = lop3<0x1A>(in.m1, g8, g18);
    const uint32_t g20 = lop3<0xE2>(in.m4, solid, g19);
    const uint32_t g21 = lop3<0x8C>(g7, g8, g9);
    const uint32_t g22 = lop3<0xA4>(g1, g14, g18);
    const uint32_t g23 = lop3<0x96>(in.m2, g21, g22);
    const uint32_t g24 = lop3<0xE2>(in.m5, solid, g23);
    const uint32_t g25 = lop3<0x9E>(in.m3, g8, g14);
    const uint32_t g26 = lop3<0xE2>(in.m0, solid, g25);
    const uint32_t g27 = lop3<0x16>(in.m4, g10, g18);
    const uint32_t g28 = lop3<0xE2>(in.m1, solid, g27);
    const uint32_t g29 = lop3<0x96>(in.rest, g13, g24);
    return Planes7{g16, g20, g24, g26, g28, g29, g12};
}

// FHP-III on fluid nodes: 43 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp3(const Planes7& in, uint32_t chi) {
    const uint32_t g0 = lop3<0xC3>(in.m1, in.m4, in.m1);
    const uint32_t g1 = lop3<0x82>(in.m0, in.m3, g0);
    const uint32_t g2 = lop3<0x1B>(in.m2, in.m5, g1);
    const uint32_t g3 = lop3<0x81>(in.m0, in.m4, g2);
    const uint32_t g4 = lop3<0x24>(in.m1, in.m2, in.m3);
    const uint32_t g5 = lop3<0x96>(in.m2, in.m5, g0);
    const uint32_t g6 = lop3<0x81>(in.m1, in.m3, in.m5);
    const uint32_t g7 = lop3<0x3A>(g1, g5, g6);
    const uint32_t g8 = lop3<0xD8>(in.m1, in.m3, chi);
    const uint32_t g9 = lop3<0x48>(in.rest, g7, g8);
    const uint32_t g10 = lop3<0xBE>(g3, g4, g9);
    const uint32_t g11 = lop3<0x82>(in.m4, in.rest, g10);
    const uint32_t g12 = lop3<0x81>(in.m0, in.m2, in.m4);
    const uint32_t g13 = lop3<0x96>(g6, g10, g12);
    const uint32_t g14 = lop3<0x82>(in.rest, g2, g13);
    const uint32_t g15 = lop3<0x69>(in.m1, chi, g11);
    const uint32_t g16 = lop3<0x69>(in.m5, g6, g15);
    const uint32_t g17 = lop3<0x09>(g1, g6, g12);
    const uint32_t g18 = lop3<0xA4>(g13, g16, g17);
    const uint32_t g19 = lop3<0x82>(g2, g8, g18);
    const uint32_t g20 = lop3<0x70>(g4, g9, g18);
    const uint32_t g21 = lop3<0x9E>(g14, g19, g20);
    const uint32_t g22 = lop3<0x78>(g10, g12, g14);
    const uint32_t g23 = lop3<0x70>(g22, g16, g17);
    const uint32_t g24 = lop3<0xC6>(g11, g21, g23);
    const uint32_t g25 = lop3<0x5A>(g0, g23, g23);
    const uint32_t g26 = lop3<0x96>(g2, g8, g16);
    const uint32_t g27 = lop3<0xC9>(g24, g25, g26);
    const uint32_t g28 = lop3<0x98>(g11, g21, g27);
    const uint32_t g29 = lop3<0x92>(g1, g13, g24);
    const uint32_t g30 = lop3<0xBA>(g4, g25, g29);
    const uint32_t g31 = lop3<0xE4>(in.m2, in.m4, g19);
    const uint32_t g32 = lop3<0x5A>(in.m0, g31, g31);
    const uint32_t g33 = lop3<0x86>(g17, g30, g32);
    const uint32_t g34 = lop3<0xD4>(g28, g30, g33);
    const uint32_t g35 = lop3<0x78>(g24, g25, g34);
    const uint32_t g36 = lop3<0x5A>(in.m0, g35, g35);
    const uint32_t g37 = lop3<0x5A>(in.m1, g34, g34);
    const uint32_t g38 = lop3<0x5A>(in.m2, g21, g21);
    const uint32_t g39 = lop3<0x96>(in.m3, g23, g35);
    const uint32_t g40 = lop3<0x99>(g25, g25, g37);
    const uint32_t g41 = lop3<0x96>(g5, g25, g38);
    const uint32_t g42 = lop3<0x5A>(in.rest, g23, g23);
    return Planes7{g36, g37, g38, g39, g40, g41, g42};
}

// FHP-III, bounce-back on solid nodes: 47 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp3_solid(const Planes7& in, uint32_t chi, uint32_t solid) {
    const uint32_t g0 = lop3<0x24>(in.m1, in.m2, in.m3);
    const uint32_t g1 = lop3<0xC3>(in.m1, in.m4, in.m1);
    const uint32_t g2 = lop3<0x82>(in.m0, in.m3, g1);
    const uint32_t g3 = lop3<0x1B>(in.m2, in.m5, g2);
    const uint32_t g4 = lop3<0x81>(in.m0, in.m4, g3);
    const uint32_t g5 = lop3<0x96>(in.m2, in.m5, g1);
    const uint32_t g6 = lop3<0x81>(in.m1, in.m3, in.m5);
    const uint32_t g7 = lop3<0x3A>(g2, g5, g6);
    const uint32_t g8 = lop3<0xD8>(in.m1, in.m3, chi);
    const uint32_t g9 = lop3<0x48>(in.rest, g7, g8);
    const uint32_t g10 = lop3<0xBE>(g0, g4, g9);
    const uint32_t g11 = lop3<0x82>(in.m4, in.rest, g10);
    const uint32_t g12 = lop3<0x81>(in.m0, in.m2, in.m4);
    const uint32_t g13 = lop3<0x96>(g6, g10, g12);
    const uint32_t g14 = lop3<0x82>(in.rest, g3, g13);
    const uint32_t g15 = lop3<0x69>(in.m1, chi, g11);
    const uint32_t g16 = lop3<0x96>(g3, g7, g15);
    const uint32_t g17 = lop3<0x09>(g2, g6, g12);
    const uint32_t g18 = lop3<0xA4>(g13, g16, g17);
    const uint32_t g19 = lop3<0x82>(g3, g8, g18);
    const uint32_t g20 = lop3<0x70>(g0, g9, g18);
    const uint32_t g21 = lop3<0x9E>(g14, g19, g20);
    const uint32_t g22 = lop3<0x78>(g10, g12, g14);
    const uint32_t g23 = lop3<0x2A>(g16, g17, g22);
    const uint32_t g24 = lop3<0xC6>(g11, g21, g23);
    const uint32_t g25 = lop3<0xC6>(solid, g1, g23);
    const uint32_t g26 = lop3<0x96>(g7, g8, g15);
    const uint32_t g27 = lop3<0xC9>(g24, g25, g26);
    const uint32_t g28 = lop3<0x98>(g11, g21, g27);
    const uint32_t g29 = lop3<0x98>(g2, g9, g24);
    const uint32_t g30 = lop3<0xBA>(g0, g25, g29);
    const uint32_t g31 = lop3<0x3C>(in.m2, g21, in.m2);
    const uint32_t g32 = lop3<0x74>(in.m4, g19, g31);
    const uint32_t g33 = lop3<0x3C>(in.m0, g32, in.m0);
    const uint32_t g34 = lop3<0x29>(g17, g28, g33);
    const uint32_t g35 = lop3<0xD4>(g28, g30, g34);
    const uint32_t g36 = lop3<0x78>(g24, g25, g35);
    const uint32_t g37 = lop3<0x5A>(in.m0, g36, g36);
    const uint32_t g38 = lop3<0xE2>(in.m3, solid, g37);
    const uint32_t g39 = lop3<0x3C>(in.m1, g35, in.m1);
    const uint32_t g40 = lop3<0xE2>(in.m4, solid, g39);
    const uint32_t g41 = lop3<0xE2>(in.m5, solid, g31);
    const uint32_t g42 = lop3<0x96>(in.m3, g23, g36);
    const uint32_t g43 = lop3<0xE2>(in.m0, solid, g42);
    const uint32_t g44 = lop3<0xC3>(g25, g40, g25);
    const uint32_t g45 = lop3<0x96>(g5, g25, g41);
    const uint32_t g46 = lop3<0x96>(in.rest, g1, g25);
    return Planes7{g38, g40, g41, g43, g44, g45, g46};
}

}  // namespace fhp
