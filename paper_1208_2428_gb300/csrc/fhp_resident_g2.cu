// fhp_resident_g2.cu -- the shared-memory resident kernel with 2 ghost rows per
// strip side (its own translation unit so that the library's kernels compile
// in parallel).
#include "fhp_resident.cuh"

namespace fhp {

template <>
cudaError_t launch_resident_g<2>(const StepArgs& a, const ResArgs& ra, int grid, size_t smem, bool has_solid, bool force,
                                 bool ragged, bool sat, cudaStream_t s) {
    return launch_resident_all<2>(a, ra, grid, smem, has_solid, force, ragged, sat, s);
}

}  // namespace fhp
