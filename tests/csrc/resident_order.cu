// Test-only: where the resident kernel leaves a call's result, compiled for the
// host.  Not part of the product library.
#include "../../paper_1208_2428_gb300/csrc/fhp_internal.h"

extern "C" __attribute__((visibility("default"))) int resident_flips(int nsteps, int gh) {
    return fhp::resident_flips(nsteps, gh) ? 1 : 0;
}
