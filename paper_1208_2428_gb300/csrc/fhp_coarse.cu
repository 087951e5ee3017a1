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
// The planes are read once: a CTA takes the row of blocks that a stretch of a
// row holds, its warps take the blocks' rows in turn, and a lane counts down its
// column, so every load is one row segment of a plane.  Where blocks and quads
// of four words fit each other (1, 2 or a multiple of 4 words per block) a
// lane's column is a quad and a load of a warp 512 bytes; else it is a word.
// The latency of the loads bounds it, so 16 warps take two rows at a time, and
// clusters share the rows of large blocks.  16384 x 4096, B = 64, from HBM:
// 15.3 us; 23.5 us with 8 warps and one row at a time (and with words); 49 us
// when one warp gathered the words of one block (which is left to narrow
// lattices).  Repeated, in L2: B = 32 12.5
// us, 64 8.4, 128 and more 10.4 (256 14.4 and 512 20.6 without clusters); 4096 x
// 4096, B = 128 and more: 8.3 (10.3, 14.2, 20.6).
#include <cooperative_groups.h>

#include "fhp_internal.h"

namespace fhp {
namespace {

constexpr int kBlock = 256;
constexpr int kWarps = kBlock / 32;
constexpr int kQuadBlock = 512;
constexpr int kQuadWarps = kQuadBlock / 32;

// Counts and derived fields of one block from its seven particle counts and its
// fluid nodes.
__device__ __forceinline__ void write_cell(long long cell, const unsigned (&n)[8], int32_t* __restrict__ counts,
                                           float* __restrict__ rho, float* __restrict__ ux, float* __restrict__ uy) {
    long long mass = 0;
    for (int k = 0; k < 7; ++k) mass += n[k];
    const long long jx2 = -(long long)n[0] + n[1] + 2LL * n[2] + n[3] - (long long)n[4] - 2LL * n[5];
    const long long jy = -(long long)n[0] - (long long)n[1] + n[3] + n[4];
    int32_t* c = counts + (size_t)cell * 9;
    for (int k = 0; k < 7; ++k) c[k] = (int32_t)n[k];
    c[7] = (int32_t)n[7];
    c[8] = (int32_t)mass;
    const double half_sqrt3 = sqrt(3.0) * 0.5;
    const double vy = mass ? half_sqrt3 * (double)jy / (double)mass : 0.0;
    uy[cell] = __double2float_rn(vy);
    if (mass < (1 << 23) && n[7] <= (1u << 24)) {
        // Quotients of integers that a float holds exactly: the float division
        // gives what the double one rounded to float gives (53 >= 2 * 24 + 2
        // bits), without two of the three divisions on the few double units.
        rho[cell] = n[7] ? __fdiv_rn((float)mass, (float)n[7]) : 0.0f;
        ux[cell] = mass ? __fdiv_rn((float)jx2, (float)(2 * mass)) : 0.0f;
        return;
    }
    rho[cell] = __double2float_rn(n[7] ? (double)mass / (double)n[7] : 0.0);
    ux[cell] = __double2float_rn(mass ? (double)jx2 / (2.0 * (double)mass) : 0.0);
}

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
    const int width = min(Bw, 32);
#pragma unroll
    for (int k = 0; k < 8; ++k) n[k] = 0;
    for (int c = 0; c < width; ++c) {
#pragma unroll
        for (int k = 0; k < 8; ++k) n[k] += part[0][k][j * Bw + c];
    }
    const long long cell = (long long)by * nbx + bx0 + j;
    write_cell(cell, n, counts, rho, ux, uy);
}

// Quads: a lane counts PER blocks of its four words (4, 2 or 1); `lanes` lanes
// hold one block where PER is 1.  CLUSTER: the `ctas` CTAs of a cluster share the
// rows of their blocks, B a multiple of 32 * ctas, and add their counts up in the
// first one's shared memory.
template <bool SOLID, int PER, bool CLUSTER = false>
__global__ void __launch_bounds__(kQuadBlock, 2) coarse_quads_kernel(Geometry g, const uint32_t* __restrict__ state,
                                                              const uint32_t* __restrict__ solid, int B, int lanes,
                                                              int groups, int ctas, int32_t* __restrict__ counts,
                                                              float* __restrict__ rho, float* __restrict__ ux,
                                                              float* __restrict__ uy) {
    __shared__ unsigned part[8 * PER][32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nbx = g.W / B;
    if (!CLUSTER) ctas = 1;
    const unsigned tile = blockIdx.x / (unsigned)ctas;
    const int rank = CLUSTER ? (int)(blockIdx.x - tile * (unsigned)ctas) : 0;
    const int by = (int)(tile / (unsigned)groups), group = (int)(tile - (unsigned)by * (unsigned)groups);
    const int width = PER == 1 ? lanes * max(1, 32 / lanes) : 32;   // quads of the CTA
    const int q0 = group * width, quads = min(width, g.nq - q0);
    unsigned n[PER][8];
#pragma unroll
    for (int b = 0; b < PER; ++b)
#pragma unroll
        for (int k = 0; k < 8; ++k) n[b][k] = 0u;
    auto add = [&](const uint4& v, int k) {
        if (PER == 4) {
            n[0][k] += __popc(v.x);
            n[1 % PER][k] += __popc(v.y);
            n[2 % PER][k] += __popc(v.z);
            n[3 % PER][k] += __popc(v.w);
        } else if (PER == 2) {
            n[0][k] += __popc(v.x) + __popc(v.y);
            n[1 % PER][k] += __popc(v.z) + __popc(v.w);
        } else {
            n[0][k] += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
        }
    };
    for (int c = lane; c < quads; c += 32) {
        const size_t base = (size_t)by * B * g.Pq + 4 * (size_t)(q0 + c);
        // (B is a multiple of 32 and a warp takes every 16th row: pairs of rows
        // where the counters leave the registers for it.)
        constexpr int ROWS = PER == 4 ? 1 : 2;
        const int stride = ctas * kQuadWarps;
        for (int r = rank * kQuadWarps + warp; r < B; r += ROWS * stride) {
            uint4 p[ROWS][7], f[ROWS];
#pragma unroll
            for (int h = 0; h < ROWS; ++h) {
                const size_t off = base + (size_t)(r + h * stride) * g.Pq;
                f[h] = SOLID ? *reinterpret_cast<const uint4*>(solid + off) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int k = 0; k < 7; ++k)
                    p[h][k] = *reinterpret_cast<const uint4*>(state + (size_t)k * g.plane_words + off);
            }
#pragma unroll
            for (int h = 0; h < ROWS; ++h) {
                add(make_uint4(~f[h].x, ~f[h].y, ~f[h].z, ~f[h].w), 7);
#pragma unroll
                for (int k = 0; k < 7; ++k)
                    add(make_uint4(p[h][k].x & ~f[h].x, p[h][k].y & ~f[h].y, p[h][k].z & ~f[h].z,
                                   p[h][k].w & ~f[h].w), k);
            }
        }
    }
    for (int i = threadIdx.x; i < 8 * PER * 33; i += kQuadBlock) part[i / 33][i % 33] = 0u;
    __syncthreads();
#pragma unroll
    for (int b = 0; b < PER; ++b)
#pragma unroll
        for (int k = 0; k < 8; ++k) atomicAdd(&part[8 * b + k][lane], n[b][k]);
    if (CLUSTER) {
        auto cluster = cooperative_groups::this_cluster();
        cluster.sync();
        if (rank) {
            unsigned* first = cluster.map_shared_rank(&part[0][0], 0);
            for (int i = threadIdx.x; i < 8 * PER * 33; i += kQuadBlock) atomicAdd(first + i, part[i / 33][i % 33]);
        }
        cluster.sync();
        if (rank) return;
    } else {
        __syncthreads();
    }
    // Thread j writes block j of the CTA.
    const int j = (int)threadIdx.x;
    const int blocks = PER == 1 ? max(1, 32 / lanes) : 32 * PER;
    const int bx = (PER == 1 ? q0 / lanes : q0 * PER) + j;
    if (j >= blocks || bx >= nbx) return;
    unsigned sum[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        sum[k] = 0u;
        if (PER == 1) {
            for (int c = 0; c < min(lanes, 32); ++c) sum[k] += part[k][j * lanes + c];
        } else {
            sum[k] = part[8 * (j % PER) + k][j / PER];
        }
    }
    write_cell((long long)by * nbx + bx, sum, counts, rho, ux, uy);
}

// A warp per block: for narrow lattices, whose rows leave the lanes of a CTA's
// warps empty.
template <bool SOLID>
__global__ void __launch_bounds__(kBlock) coarse_warp_kernel(Geometry g, const uint32_t* __restrict__ state,
                                                             const uint32_t* __restrict__ solid, int B, int Bw,
                                                             long long cells, int32_t* __restrict__ counts,
                                                             float* __restrict__ rho, float* __restrict__ ux,
                                                             float* __restrict__ uy) {
    const int lane = threadIdx.x & 31;
    const int nbx = g.W / B;
    const long long cell = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (cell >= cells) return;   // (a whole warp)
    const int by = (int)(cell / nbx), bx = (int)(cell - (long long)by * nbx);
    const size_t base = (size_t)by * B * g.Pq + (size_t)bx * Bw;
    unsigned n[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = lane; i < B * Bw; i += 32) {
        const size_t off = base + (size_t)(i / Bw) * g.Pq + i % Bw;
        const uint32_t f = SOLID ? ~solid[off] : 0xFFFFFFFFu;
        n[7] += __popc(f);
#pragma unroll
        for (int k = 0; k < 7; ++k) n[k] += __popc(state[(size_t)k * g.plane_words + off] & f);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) n[k] = __reduce_add_sync(0xFFFFFFFFu, n[k]);
    if (lane == 0) write_cell(cell, n, counts, rho, ux, uy);
}

// Where a warp per block is the faster (us, a warp per block / the kernels
// above).  These give every row of blocks a CTA, whatever the row's length, so
// what counts is how many rows of blocks there are for the SMs, and how few words
// a row has: 120 rows of blocks of 64 8.3 / 6.5 at every width; 240 rows 8.3 / 10.2
// with 8 words, 10.5 / 10.3 with 16; 1920 rows 10.4 / 37.1 with 2 words, 30.6 / 37.1
// with 12, 39.3 / 37.1 with 16.  B = 32: 3840 rows of 1 word 14.5 / 49.4, of 5 words
// 43.4 / 49.6, of 6 52.7 / 50.3, 120 rows 6.5 / 6.5.  B = 128: 120 rows 12.4 / 10.8,
// 180 rows of 24 words 12.4 / 14.5, of 28 words 14.6 / 14.5, 960 rows of 28 words
// 35.0 / 43.2, of 32 words 51.5 / 45.2.  B = 256: 240 rows 26.9 / 22.7, 480 rows of 16 words 26.9 / 39.2, of 24
// words 39.2 / 41.2.  B = 96: 640 rows of 3 words 9.4 / 10.6, of 6 words 12.0 / 10.5,
// 1280 rows of 6 words 14.6 / 16.5.  Not for larger blocks, whose words one warp
// would take too long to walk (B = 512: 88 / 23).
bool warp_per_block(const Geometry& g, int Bw) {
    const int rows = g.H / (32 * Bw), sms = sm_count();
    switch (Bw) {
        case 1: return rows > sms && g.Wq <= 5;
        case 2: return rows > sms && g.Wq <= 12;
        case 3: return rows > sms && rows > 200 * g.Wq;
        case 4: return rows > sms && g.Wq <= 28;
        case 8: return 2 * rows > 5 * sms && g.Wq <= 24;
        default: return false;
    }
}

}  // namespace

cudaError_t launch_coarse_grain(const Geometry& g, const uint32_t* state, const uint32_t* solid,
                                bool has_solid, int B, int32_t* counts, float* rho, float* ux,
                                float* uy, cudaStream_t stream) {
    const int Bw = B / 32, nbx = g.W / B;
    if (warp_per_block(g, Bw)) {
        const long long cells = (long long)nbx * (g.H / B);
        const unsigned grid = (unsigned)((cells + kWarps - 1) / kWarps);
        auto launch = [&](auto kernel) {
            kernel<<<grid, kBlock, 0, stream>>>(g, state, solid, B, Bw, cells, counts, rho, ux, uy);
        };
        has_solid ? launch(coarse_warp_kernel<true>) : launch(coarse_warp_kernel<false>);
        return cudaGetLastError();
    }
    if (Bw <= 2 || Bw % 4 == 0) {
        const int per = Bw <= 2 ? 4 / Bw : 1, lanes = Bw <= 2 ? 1 : Bw / 4;   // blocks per quad, quads per block
        const int width = per > 1 ? 32 : lanes * (lanes >= 32 ? 1 : 32 / lanes);
        const int groups = (g.Wq + 4 * width - 1) / (4 * width);
        const unsigned grid = (unsigned)((long long)groups * (g.H / B));
        // Blocks of 128 nodes and more leave few CTAs with many rows each: while no
        // more than two per SM come of it, the CTAs of a cluster share the rows.  Not
        // for 32 and 64 nodes, whose few rows gain less than a cluster costs (4096 x
        // 4096: 8.2 us with, 6.3 without).
        int ctas = 1;
        const unsigned most = 2u * (unsigned)sm_count();
        while (per == 1 && ctas < 8 && grid * ctas * 2 <= most && B % (64 * ctas) == 0) ctas *= 2;
        if (ctas > 1) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(grid * ctas);
            cfg.blockDim = dim3(kQuadBlock);
            cfg.stream = stream;
            cudaLaunchAttribute cluster = {};
            cluster.id = cudaLaunchAttributeClusterDimension;
            cluster.val.clusterDim.x = ctas;
            cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
            cfg.attrs = &cluster;
            cfg.numAttrs = 1;
            return has_solid ? cudaLaunchKernelEx(&cfg, coarse_quads_kernel<true, 1, true>, g, state, solid, B, lanes,
                                                  groups, ctas, counts, rho, ux, uy)
                             : cudaLaunchKernelEx(&cfg, coarse_quads_kernel<false, 1, true>, g, state, solid, B, lanes,
                                                  groups, ctas, counts, rho, ux, uy);
        }
        auto launch = [&](auto kernel) {
            kernel<<<grid, kQuadBlock, 0, stream>>>(g, state, solid, B, lanes, groups, 1, counts, rho, ux, uy);
        };
        if (per == 4) has_solid ? launch(coarse_quads_kernel<true, 4>) : launch(coarse_quads_kernel<false, 4>);
        else if (per == 2) has_solid ? launch(coarse_quads_kernel<true, 2>) : launch(coarse_quads_kernel<false, 2>);
        else has_solid ? launch(coarse_quads_kernel<true, 1>) : launch(coarse_quads_kernel<false, 1>);
        return cudaGetLastError();
    }
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
