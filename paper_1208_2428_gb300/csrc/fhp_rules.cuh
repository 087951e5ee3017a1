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
// and 46 (FHP-III) operations, and 30, 18 and 52 with the bounce-back of solid nodes.
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

// FHP-III on fluid nodes: 46 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp3(const Planes7& in, uint32_t chi) {
    const uint32_t g0 = lop3<0xC3>(in.m0, in.m3, in.m0);
    const uint32_t g1 = lop3<0xC3>(in.m2, in.m5, in.m2);
    const uint32_t g2 = lop3<0xC3>(in.m1, in.m4, in.m1);
    const uint32_t g3 = lop3<0x81>(g0, g1, g2);
    const uint32_t g4 = lop3<0x4D>(in.m1, in.m4, in.m5);
    const uint32_t g5 = lop3<0x1B>(in.m2, in.rest, g3);
    const uint32_t g6 = lop3<0xA5>(in.m1, g5, g5);
    const uint32_t g7 = lop3<0x59>(chi, g2, g6);
    const uint32_t g8 = lop3<0x82>(in.m1, g4, g7);
    const uint32_t g9 = lop3<0x24>(in.m5, g4, g5);
    const uint32_t g10 = lop3<0xDB>(in.m1, in.m2, in.m3);
    const uint32_t g11 = lop3<0xC3>(in.m0, in.m5, in.m0);
    const uint32_t g12 = lop3<0x24>(in.m0, in.m1, in.m2);
    const uint32_t g13 = lop3<0x3D>(g10, g11, g12);
    const uint32_t g14 = lop3<0x93>(chi, g9, g13);
    const uint32_t g15 = lop3<0x1A>(g2, g9, g14);
    const uint32_t g16 = lop3<0xDC>(g0, g11, g15);
    const uint32_t g17 = lop3<0x41>(in.m0, in.m4, g16);
    const uint32_t g18 = lop3<0xEA>(g7, g12, g17);
    const uint32_t g19 = lop3<0xA0>(g1, g13, g13);
    const uint32_t g20 = lop3<0x36>(g0, g18, g19);
    const uint32_t g21 = lop3<0x2A>(g9, g13, g20);
    const uint32_t g22 = lop3<0x48>(g1, g8, g21);
    const uint32_t g23 = lop3<0xB5>(g9, g15, g17);
    const uint32_t g24 = lop3<0x10>(g6, g10, g18);
    const uint32_t g25 = lop3<0x14>(in.m3, in.m4, g24);
    const uint32_t g26 = lop3<0x92>(g1, g23, g25);
    const uint32_t g27 = lop3<0x27>(g10, g14, g26);
    const uint32_t g28 = lop3<0x88>(g2, g2, g20);
    const uint32_t g29 = lop3<0x60>(g25, g27, g28);
    const uint32_t g30 = lop3<0x5B>(g12, g16, g29);
    const uint32_t g31 = lop3<0x8E>(g21, g27, g30);
    const uint32_t g32 = lop3<0x06>(g3, g22, g31);
    const uint32_t g33 = lop3<0x80>(g0, g19, g20);
    const uint32_t g34 = lop3<0x7E>(g24, g29, g33);
    const uint32_t g35 = lop3<0x5A>(in.m3, g34, g34);
    const uint32_t g36 = lop3<0x69>(g0, g32, g35);
    const uint32_t g37 = lop3<0xF9>(g22, g23, g29);
    const uint32_t g38 = lop3<0x3C>(in.m4, g37, in.m4);
    const uint32_t g39 = lop3<0x69>(g2, g32, g38);
    const uint32_t g40 = lop3<0x28>(g6, g29, g32);
    const uint32_t g41 = lop3<0xB6>(g37, g34, g40);
    const uint32_t g42 = lop3<0xA6>(g2, g29, g41);
    const uint32_t g43 = lop3<0x96>(in.m2, g32, g42);
    const uint32_t g44 = lop3<0x5A>(in.m5, g42, g42);
    const uint32_t g45 = lop3<0x3C>(in.rest, g32, in.rest);
    return Planes7{g36, g39, g43, g35, g38, g44, g45};
}

// FHP-III, bounce-back on solid nodes: 52 operations.
__host__ __device__ __forceinline__ Planes7 scatter_fhp3_solid(const Planes7& in, uint32_t chi, uint32_t solid) {
    const uint32_t g0 = lop3<0xC3>(in.m0, in.m3, in.m0);
    const uint32_t g1 = lop3<0xC3>(in.m2, in.m5, in.m2);
    const uint32_t g2 = lop3<0xC3>(in.m1, in.m4, in.m1);
    const uint32_t g3 = lop3<0x81>(g0, g1, g2);
    const uint32_t g4 = lop3<0x1B>(in.m2, in.rest, g3);
    const uint32_t g5 = lop3<0xA5>(in.m1, g4, g4);
    const uint32_t g6 = lop3<0x59>(chi, g2, g5);
    const uint32_t g7 = lop3<0x27>(in.m1, in.m5, g2);
    const uint32_t g8 = lop3<0x42>(in.m5, g4, g7);
    const uint32_t g9 = lop3<0x48>(g5, g6, g8);
    const uint32_t g10 = lop3<0xDB>(in.m1, in.m2, in.m3);
    const uint32_t g11 = lop3<0xC3>(in.m0, in.m5, in.m0);
    const uint32_t g12 = lop3<0x77>(g10, g10, g11);
    const uint32_t g13 = lop3<0x24>(in.m0, in.m1, in.m2);
    const uint32_t g14 = lop3<0x93>(chi, g8, g12);
    const uint32_t g15 = lop3<0x1A>(g2, g8, g14);
    const uint32_t g16 = lop3<0xDC>(g0, g11, g15);
    const uint32_t g17 = lop3<0x41>(in.m0, in.m4, g16);
    const uint32_t g18 = lop3<0xEA>(g6, g13, g17);
    const uint32_t g19 = lop3<0x88>(g1, g1, g12);
    const uint32_t g20 = lop3<0x36>(g0, g18, g19);
    const uint32_t g21 = lop3<0x2A>(g8, g12, g20);
    const uint32_t g22 = lop3<0x48>(g1, g9, g21);
    const uint32_t g23 = lop3<0xB5>(g8, g15, g17);
    const uint32_t g24 = lop3<0x10>(g5, g10, g18);
    const uint32_t g25 = lop3<0x14>(in.m3, in.m4, g24);
    const uint32_t g26 = lop3<0x82>(g1, g23, g25);
    const uint32_t g27 = lop3<0x27>(g10, g14, g26);
    const uint32_t g28 = lop3<0xA0>(g2, g20, g20);
    const uint32_t g29 = lop3<0x60>(g25, g27, g28);
    const uint32_t g30 = lop3<0x5B>(g13, g16, g29);
    const uint32_t g31 = lop3<0x8E>(g21, g27, g30);
    const uint32_t g32 = lop3<0x46>(g3, g22, g31);
    const uint32_t g33 = lop3<0x20>(g0, g18, g19);
    const uint32_t g34 = lop3<0x3E>(g24, g29, g33);
    const uint32_t g35 = lop3<0x96>(in.m0, g32, g34);
    const uint32_t g36 = lop3<0xE2>(in.m3, solid, g35);
    const uint32_t g37 = lop3<0xFB>(g22, g23, g29);
    const uint32_t g38 = lop3<0x96>(in.m1, g32, g37);
    const uint32_t g39 = lop3<0xE2>(in.m4, solid, g38);
    const uint32_t g40 = lop3<0x28>(g5, g29, g32);
    const uint32_t g41 = lop3<0x9E>(g34, g37, g40);
    const uint32_t g42 = lop3<0xA6>(g2, g29, g41);
    const uint32_t g43 = lop3<0x96>(in.m2, g32, g42);
    const uint32_t g44 = lop3<0xE2>(in.m5, solid, g43);
    const uint32_t g45 = lop3<0x5A>(in.m3, g34, g34);
    const uint32_t g46 = lop3<0xE2>(in.m0, solid, g45);
    const uint32_t g47 = lop3<0x5A>(in.m4, g37, g37);
    const uint32_t g48 = lop3<0xE2>(in.m1, solid, g47);
    const uint32_t g49 = lop3<0x3C>(in.m5, g42, in.m5);
    const uint32_t g50 = lop3<0xE2>(in.m2, solid, g49);
    const uint32_t g51 = lop3<0xD2>(in.rest, solid, g32);
    return Planes7{g36, g39, g44, g46, g48, g50, g51};
}

}  // namespace fhp
