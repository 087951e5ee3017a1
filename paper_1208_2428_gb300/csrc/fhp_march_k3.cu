// fhp_march_k3.cu -- register marching with 3 steps per pass (its own
// translation unit so that the library's kernels compile in parallel).
#include "fhp_march.cuh"

namespace fhp {

template <>
cudaError_t march_k<3>(const StepArgs& a, const MarchArgs& b, const MarchVariant& v, bool launch, int* blocks_per_sm,
                       cudaStream_t s) {
    return march_all<3>(a, b, v, launch, blocks_per_sm, s);
}

}  // namespace fhp
