// Test-only: the collision networks without bounce-back (words without solid
// nodes), compiled for the host.  Not part of the product library.
#include <cstdint>

#include "../../paper_1208_2428_gb300/csrc/fhp_device.cuh"

extern "C" __attribute__((visibility("default"))) void host_fluid_scatter_words(int rules, const uint32_t* planes7,
                                                                                uint32_t chi, uint32_t* out7) {
    const fhp::Planes7 in{planes7[0], planes7[1], planes7[2], planes7[3], planes7[4], planes7[5], planes7[6]};
    const fhp::Planes7 o = rules == 1   ? fhp::scatter_rules<1, false>(in, 0u, chi)
                           : rules == 2 ? fhp::scatter_rules<2, false>(in, 0u, chi)
                                        : fhp::scatter_rules<3, false>(in, 0u, chi);
    out7[0] = o.m0; out7[1] = o.m1; out7[2] = o.m2; out7[3] = o.m3;
    out7[4] = o.m4; out7[5] = o.m5; out7[6] = o.rest;
}
