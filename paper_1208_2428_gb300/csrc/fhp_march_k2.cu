// fhp_march_k2.cu -- register marching with 2 steps per pass (its own
// translation unit so that the library's kernels compile in parallel).
#include "fhp_march.cuh"

namespace fhp {

template <>
cudaError_t march_k<2>(const StepArgs& a, const MarchArgs& b, const MarchVariant& v, bool launch, int* blocks_per_sm,
                       cudaStream_t s) {
    return march_all<2>(a, b, v, launch, blocks_per_sm, s);
}

}  // namespace fhp
