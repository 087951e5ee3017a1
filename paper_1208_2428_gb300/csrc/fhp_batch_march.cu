// fhp_batch_march.cu -- register marching (fhp_march.cuh) of many lattices in
// one cooperative launch: every warp works on one member's bands for all
// passes of the call and waits only for the warps around it, so the members
// need no launches and no common pace.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "fhp_march.cuh"

namespace fhp {
namespace {

static_assert(kMarchCtaWarps == kMarchWarps, "the member table counts CTAs of the marching kernel");

// FORCE: some member has forcing (the others take the branch without it).
template <int K, bool FORCE, bool RAGGED>
__global__ void __launch_bounds__(32 * kMarchWarps, K <= 2 ? 4 : 3)
    fhp_batch_march_kernel(const __grid_constant__ MarchBatch t) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const MarchJob& J = t.job[t.member[blockIdx.x]];
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const int gw = ((int)blockIdx.x - J.first_cta) * kMarchWarps + warp;
    if (gw >= J.nwarps) return;
    StepArgs a;
    a.src = J.src;
    a.dst = J.dst;
    a.solid = J.solid;
    a.plane_words = J.plane_words;
    a.H = J.H;
    a.Wq = J.Wq;
    a.nq = (J.Wq + 3) >> 2;
    a.Pq = 4 * a.nq;
    a.key = J.key;
    a.t_lo = (uint32_t)J.t0;
    a.t_hi = (uint32_t)(J.t0 >> 32);
    a.err = t.err;
    a.rest_rules = J.rest_rules;
    a.ft.pre = J.pre;
    a.ft.dense = J.dense;
    a.ft.inv = J.inv;
    MarchArgs b;
    b.R = J.R;
    b.nbands = J.nbands;
    b.pitch = J.lay.pitch;
    b.left = J.lay.left;
    b.hl = J.lay.hl;
    b.per_warp = J.lay.per_warp;
    b.nwarps = J.nwarps;
    b.passes = J.passes;
    b.flags = t.flags + J.first_cta * kMarchWarps;
    b.epoch = t.epoch;
    const uint32_t ring = smem_addr(smem_raw) + (uint32_t)(warp * MarchRing<K, true>::warp_bytes);
    if (FORCE && J.P != 0ull) {
        // Threshold Q_(lane + 1): S_0 = 2^32, S_g = floor(S_(g-1) (2^32 - P) / 2^32).
        const unsigned long long one = 1ull << 32, keep = one - J.P;
        unsigned long long S = keep;
        for (int g = 0; g < lane; ++g) S = S * keep >> 32;
        march_warp<K, true, true, RAGGED, false>(a, b, gw, ring, (uint32_t)(one - S - 1ull));
    } else {
        march_warp<K, true, false, RAGGED, false>(a, b, gw, ring, 0u);
    }
}

template <int K, bool FORCE, bool RAGGED>
cudaError_t batch_march_variant(const MarchBatch* t, int* ctas, cudaStream_t s) {
    constexpr int smem = kMarchWarps * MarchRing<K, true>::warp_bytes;
    auto kernel = fhp_batch_march_kernel<K, FORCE, RAGGED>;
    if (!t) {
        static std::mutex m;
        static int count[64] = {};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(m);
        if (!count[dev]) {
            int n = 0, sms = 0;
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, 32 * kMarchWarps, smem);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            if (n < 1) return cudaErrorInvalidConfiguration;
            count[dev] = std::min(n * sms, kMarchMaxCtas);
        }
        *ctas = count[dev];
        return cudaSuccess;
    }
    void* args[] = {const_cast<MarchBatch*>(t)};
    const cudaError_t e = cudaLaunchCooperativeKernel((const void*)kernel, dim3((unsigned)*ctas), dim3(32 * kMarchWarps),
                                                      args, smem, s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t batch_march_any(const MarchBatch* t, int* ctas, int k, bool force, bool ragged, cudaStream_t s) {
    if (k == 3)   // (only without forcing)
        return ragged ? batch_march_variant<3, false, true>(t, ctas, s) : batch_march_variant<3, false, false>(t, ctas, s);
    if (force)
        return ragged ? batch_march_variant<2, true, true>(t, ctas, s) : batch_march_variant<2, true, false>(t, ctas, s);
    return ragged ? batch_march_variant<2, false, true>(t, ctas, s) : batch_march_variant<2, false, false>(t, ctas, s);
}

}  // namespace

cudaError_t batch_march_ctas(int k, bool force, bool ragged, int* ctas) {
    if (k != 2 && (k != 3 || force)) return cudaErrorInvalidValue;
    return batch_march_any(nullptr, ctas, k, force, ragged, nullptr);
}

cudaError_t launch_batch_march(const MarchBatch& t, int ctas, int k, bool force, bool ragged, cudaStream_t stream) {
    int most = 0;
    const cudaError_t e = batch_march_ctas(k, force, ragged, &most);
    if (e != cudaSuccess) return e;
    if (ctas < 1 || ctas > most) return cudaErrorInvalidValue;
    return batch_march_any(&t, &ctas, k, force, ragged, stream);
}

}  // namespace fhp
