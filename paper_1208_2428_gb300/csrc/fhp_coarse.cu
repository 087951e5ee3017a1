// fhp_coarse.cu -- block coarse-graining of the bit-plane lattice.
//
// For each B x B block (B a multiple of 32, so a block row is B/32 whole
// words) the kernel counts, over the fluid nodes of the block, how many carry
// each of the seven particles (population counts of plane & ~solid), the
// number of fluid nodes, and the mass; it then derives density and mean
// particle velocity in double precision:
//   rho = mass / fluid, ux = jx2 / (2 mass), uy = (sqrt(3)/2) jy / mass,
// with the integer momenta jx2 = sum_i n_i 2cos(theta_i) and
// jy = sum_i n_i sgn(sin(theta_i)), theta_i = (i-2)*60 degrees.
//
// The planes are read once, at the speed of memory: a CTA takes the row of
// blocks that 32 neighbouring words hold (one block where a block is wider),
// its eight warps take the blocks' rows in turn, and a lane counts down its
// word column, so every load is one row segment of a plane.  16384 x 4096,
// B = 64: 23.6 us; 49 us when one warp gathered the words of one block.
#include "fhp_internal.h"

namespace fhp {
namespace {

constexpr int kBlock = 256;
constexpr int kWarps = kBlock / 32;

// Bw words per block row, nb blocks per CTA (nb * Bw <= 32, or nb = 1).
template <bool SOLID>
__global__ void __launch_bounds__(kBlock) coarse_kernel(Geometry g, const uint32_t* __restrict__ state,
                                                        const uint32_t* __restrict__ solid, int B, int Bw, int nb,
                                                        int groups, int32_t* __restrict__ counts,
                                                        float* __restrict__ rho,
                                                        float* __restrict__ ux,
                                                        float* __restrict__ uy) {
    __shared__ unsigned part[kWarps][8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nbx = g.W / B;
    const int by = (int)(blockIdx.x / (unsigned)groups), group = (int)(blockIdx.x - (unsigned)by * (unsigned)groups);
    const int bx0 = group * nb;
    const int cols = min(nb, nbx - bx0) * Bw;   // word columns of the CTA
    unsigned n[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // seven particles, fluid nodes
    for (int c = lane; c < cols; c += 32) {
        const size_t base = (size_t)by * B * g.Pq + (size_t)bx0 * Bw + c;
#pragma unroll 4
        for (int r = warp; r < B; r += kWarps) {
            const size_t off = base + (size_t)r * g.Pq;
            const uint32_t f = SOLID ? ~solid[off] : 0xFFFFFFFFu;
            n[7] += __popc(f);
#pragma unroll
            for (int k = 0; k < 7; ++k) n[k] += __popc(state[(size_t)k * g.plane_words + off] & f);
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) part[warp][k][lane] = n[k];
    __syncthreads();
    // Warp k adds counter k over the warps, then thread j adds block j's columns.
    unsigned sum = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) sum += part[w][warp][lane];
    __syncthreads();
    part[0][warp][lane] = sum;
    __syncthreads();
    const int j = (int)threadIdx.x;
    if (j >= nb || bx0 + j >= nbx) return;
    unsigned fluid = 0;
    const int width = min(Bw, 32);
#pragma unroll
    for (int k = 0; k < 8; ++k) n[k] = 0;
    for (int c = 0; c < width; ++c) {
#pragma unroll
        for (int k = 0; k < 8; ++k) n[k] += part[0][k][j * Bw + c];
    }
    fluid = n[7];
    const long long cell = (long long)by * nbx + bx0 + j;
    long long mass = 0;
    for (int k = 0; k < 7; ++k) mass += n[k];
    const long long jx2 = -(long long)n[0] + n[1] + 2LL * n[2] + n[3] - (long long)n[4] - 2LL * n[5];
    const long long jy = -(long long)n[0] - (long long)n[1] + n[3] + n[4];
    int32_t* c = counts + (size_t)cell * 9;
    for (int k = 0; k < 7; ++k) c[k] = (int32_t)n[k];
    c[7] = (int32_t)fluid;
    c[8] = (int32_t)mass;
    const double half_sqrt3 = sqrt(3.0) * 0.5;
    const double r = fluid ? (double)mass / (double)fluid : 0.0;
    const double vx = mass ? (double)jx2 / (2.0 * (double)mass) : 0.0;
    const double vy = mass ? half_sqrt3 * (double)jy / (double)mass : 0.0;
    rho[cell] = __double2float_rn(r);
    ux[cell] = __double2float_rn(vx);
    uy[cell] = __double2float_rn(vy);
}

}  // namespace

cudaError_t launch_coarse_grain(const Geometry& g, const uint32_t* state, const uint32_t* solid,
                                bool has_solid, int B, int32_t* counts, float* rho, float* ux,
                                float* uy, cudaStream_t stream) {
    const int Bw = B / 32, nbx = g.W / B;
    const int nb = Bw >= 32 ? 1 : 32 / Bw;
    const int groups = (nbx + nb - 1) / nb;
    const unsigned grid = (unsigned)((long long)groups * (g.H / B));
    if (has_solid)
        coarse_kernel<true><<<grid, kBlock, 0, stream>>>(g, state, solid, B, Bw, nb, groups, counts, rho, ux, uy);
    else
        coarse_kernel<false><<<grid, kBlock, 0, stream>>>(g, state, solid, B, Bw, nb, groups, counts, rho, ux, uy);
    return cudaGetLastError();
}

}  // namespace fhp
