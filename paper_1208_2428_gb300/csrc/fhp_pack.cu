// fhp_pack.cu -- conversion between node bytes (arXiv:1208.2428 Section 2,
// Fig. 1: bits 0-5 movers, bit 6 rest, bit 7 solid) and bit-planes, and the
// obstacle map.
//
// Bytes and planes: a thread converts the 32 nodes of one word, 32 bytes
// against 8 plane words, as four 8 x 8 bit transposes done side by side in the
// bytes of 8 registers (three rounds of masked exchanges, 48 operations) and a
// byte transpose (16 permutes).  The byte side is one 32-byte access per
// thread, the plane side a 128-byte row segment per warp and plane, so both
// conversions run at the speed of memory: 8192 x 4096 nodes, 2 bytes moved
// per node, 10.6 us each way, against 138 us out and 177 us in for the warp
// ballots that convert one word per warp and load single bytes.  The ballot
// kernels remain for byte arrays that are not 32-byte aligned.
#include <cmath>

#include "fhp_device.cuh"
#include "fhp_internal.h"

namespace fhp {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kBlock = 256;

unsigned grid_for(size_t warps) {
    size_t blocks = (warps * 32 + kBlock - 1) / kBlock;
    if (blocks > 65535u * 16u) blocks = 65535u * 16u;  // grid-stride loop covers the rest
    return (unsigned)(blocks ? blocks : 1);
}

// Exchange of bits between two registers: those of `a` under mask << s with
// those of `b` under mask.
template <int S, uint32_t MASK>
__device__ __forceinline__ void exchange(uint32_t& a, uint32_t& b) {
    const uint32_t up = b << S, down = a >> S;
    a = (a & ~(MASK << S)) | (up & (MASK << S));
    b = (b & ~MASK) | (down & MASK);
}

// Transposes the 8 x 8 bit matrices held by equal bytes of r[0..7] (its own
// inverse).
__device__ __forceinline__ void transpose_bits(uint32_t (&r)[8]) {
#pragma unroll
    for (int i = 0; i < 8; i += 2) exchange<1, 0x55555555u>(r[i], r[i + 1]);
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (!(i & 2)) exchange<2, 0x33333333u>(r[i], r[i + 2]);
#pragma unroll
    for (int i = 0; i < 4; ++i) exchange<4, 0x0F0F0F0Fu>(r[i], r[i + 4]);
}

// Transposes the 4 x 4 byte matrix of four registers (its own inverse).
__device__ __forceinline__ void transpose_bytes(uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d) {
    const uint32_t ab = __byte_perm(a, b, 0x5140), cd = __byte_perm(c, d, 0x5140);
    const uint32_t ab2 = __byte_perm(a, b, 0x7362), cd2 = __byte_perm(c, d, 0x7362);
    a = __byte_perm(ab, cd, 0x5410);
    b = __byte_perm(ab, cd, 0x7632);
    c = __byte_perm(ab2, cd2, 0x5410);
    d = __byte_perm(ab2, cd2, 0x7632);
}

// Rows [0, rows) of a lattice whose pointers start at its first row; RAGGED:
// rows end in padding words.  Word n of the rows: byte 8g + k of the 32 bytes
// is node 8g + k; after the byte transpose register k holds nodes 8g + k in
// its byte g, after the bit transpose register b is plane b.
template <bool RAGGED>
__global__ void __launch_bounds__(kBlock) pack_words_kernel(int Wq, int Pq, uint32_t total, size_t plane_words,
                                                            const uint8_t* __restrict__ bytes,
                                                            uint32_t* __restrict__ state, uint32_t* __restrict__ solid,
                                                            unsigned int* any_solid) {
    const uint32_t item = blockIdx.x * (uint32_t)kBlock + threadIdx.x;   // word of the padded rows
    uint32_t r[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (item < total) {
        uint32_t word = item;   // word of the unpadded rows
        bool valid = true;
        if (RAGGED) {
            const uint32_t y = item / (uint32_t)Pq, w = item - y * (uint32_t)Pq;
            valid = w < (uint32_t)Wq;
            word = y * (uint32_t)Wq + w;
        }
        if (valid) {
            const uint8_t* src = bytes + (size_t)word * 32;
            asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[0]), "=r"(r[4]), "=r"(r[1]), "=r"(r[5]), "=r"(r[2]), "=r"(r[6]), "=r"(r[3]),
                           "=r"(r[7])
                         : "l"(src));
            transpose_bytes(r[0], r[1], r[2], r[3]);
            transpose_bytes(r[4], r[5], r[6], r[7]);
            transpose_bits(r);
        }
#pragma unroll
        for (int b = 0; b < 7; ++b) state[(size_t)b * plane_words + item] = r[b];
        solid[item] = r[7];
    }
    if (__syncthreads_or(r[7] != 0u) && threadIdx.x == 0) atomicOr(any_solid, 1u);
}

template <bool RAGGED>
__global__ void __launch_bounds__(kBlock) unpack_words_kernel(int Wq, int Pq, uint32_t total, size_t plane_words,
                                                              const uint32_t* __restrict__ state,
                                                              const uint32_t* __restrict__ solid,
                                                              uint8_t* __restrict__ bytes) {
    const uint32_t word = blockIdx.x * (uint32_t)kBlock + threadIdx.x;   // word of the unpadded rows
    if (word >= total) return;
    uint32_t item = word;   // word of the padded rows
    if (RAGGED) {
        const uint32_t y = word / (uint32_t)Wq;
        item = y * (uint32_t)Pq + (word - y * (uint32_t)Wq);
    }
    uint32_t r[8];
#pragma unroll
    for (int b = 0; b < 7; ++b) r[b] = state[(size_t)b * plane_words + item];
    r[7] = solid[item];
    transpose_bits(r);
    transpose_bytes(r[0], r[1], r[2], r[3]);
    transpose_bytes(r[4], r[5], r[6], r[7]);
    uint8_t* dst = bytes + (size_t)word * 32;
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(r[0]), "r"(r[4]), "r"(r[1]),
                 "r"(r[5]), "r"(r[2]), "r"(r[6]), "r"(r[3]), "r"(r[7])
                 : "memory");
}

// Rows per launch of the word kernels (their word indices have 32 bits).
int rows_per_launch(const Geometry& g) {
    const long long rows = ((1LL << 31) - kBlock) / g.Pq;
    return (int)(rows < g.H ? rows : g.H);
}

// Byte arrays that are not 32-byte aligned: one warp per word, lane j holds
// node 32w + j and __ballot_sync gathers bit b of the 32 nodes into plane b.
__global__ void __launch_bounds__(kBlock) pack_kernel(Geometry g, const uint8_t* __restrict__ bytes,
                                                      uint32_t* __restrict__ state,
                                                      uint32_t* __restrict__ solid,
                                                      unsigned int* __restrict__ any_solid) {
    const int lane = threadIdx.x & 31;
    const size_t nwarps = ((size_t)gridDim.x * blockDim.x) >> 5;
    const size_t total = (size_t)g.H * g.Pq;
    for (size_t item = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; item < total;
         item += nwarps) {
        const int y = (int)(item / g.Pq);
        const int w = (int)(item - (size_t)y * g.Pq);
        uint32_t v = 0;
        if (w < g.Wq) v = bytes[(size_t)y * g.W + 32 * w + lane];
        uint32_t mine = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t plane_word = __ballot_sync(kFull, (v >> b) & 1u);
            if (lane == b) mine = plane_word;
        }
        const size_t off = (size_t)y * g.Pq + w;
        if (lane < 7) state[(size_t)lane * g.plane_words + off] = mine;
        if (lane == 7) {
            solid[off] = mine;
            if (mine) atomicOr(any_solid, 1u);
        }
    }
}

__global__ void __launch_bounds__(kBlock) unpack_kernel(Geometry g, const uint32_t* __restrict__ state,
                                                        const uint32_t* __restrict__ solid,
                                                        uint8_t* __restrict__ bytes) {
    const int lane = threadIdx.x & 31;
    const size_t nwarps = ((size_t)gridDim.x * blockDim.x) >> 5;
    const size_t total = (size_t)g.H * g.Wq;
    for (size_t item = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; item < total;
         item += nwarps) {
        const int y = (int)(item / g.Wq);
        const int w = (int)(item - (size_t)y * g.Wq);
        const size_t off = (size_t)y * g.Pq + w;
        uint32_t byte = ((solid[off] >> lane) & 1u) << 7;
#pragma unroll
        for (int b = 0; b < 7; ++b) byte |= ((state[(size_t)b * g.plane_words + off] >> lane) & 1u) << b;
        bytes[(size_t)y * g.W + 32 * w + lane] = (uint8_t)byte;
    }
}

__global__ void __launch_bounds__(kBlock) obstacle_kernel(Geometry g, const uint8_t* __restrict__ mask,
                                                          uint32_t* __restrict__ state,
                                                          uint32_t* __restrict__ solid,
                                                          unsigned int* __restrict__ any_solid) {
    const int lane = threadIdx.x & 31;
    const size_t nwarps = ((size_t)gridDim.x * blockDim.x) >> 5;
    const size_t total = (size_t)g.H * g.Pq;
    for (size_t item = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; item < total;
         item += nwarps) {
        const int y = (int)(item / g.Pq);
        const int w = (int)(item - (size_t)y * g.Pq);
        bool s = false;
        if (w < g.Wq) s = mask[(size_t)y * g.W + 32 * w + lane] != 0;
        const uint32_t word = __ballot_sync(kFull, s);
        const size_t off = (size_t)y * g.Pq + w;
        if (lane < 7 && word) state[(size_t)lane * g.plane_words + off] &= ~word;
        if (lane == 7) {
            solid[off] = word;
            if (word) atomicOr(any_solid, 1u);
        }
    }
}

// item / pitch: by a 32-bit division (a quarter of the instructions) while the
// item has 32 bits.
__device__ __forceinline__ int row_of(size_t item, int pitch) {
    return (item >> 32) == 0 ? (int)((uint32_t)item / (uint32_t)pitch) : (int)(item / (size_t)pitch);
}

// The rounds of Philox4x32-10 after the first two.
__device__ __forceinline__ uint4 philox_from_round_2(uint4 c, Key2 k) {
    k.lo += 2u * 0x9E3779B9u;
    k.hi += 2u * 0xBB67AE85u;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const unsigned long long a = (unsigned long long)0xD2511F53u * c.x;
        const unsigned long long b = (unsigned long long)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(b >> 32) ^ c.y ^ k.lo, (uint32_t)b, (uint32_t)(a >> 32) ^ c.w ^ k.hi, (uint32_t)a);
        k.lo += 0x9E3779B9u;
        k.hi += 0xBB67AE85u;
    }
    return c;
}

// Generated initial state: for word w of row y and bit b, four Philox blocks
// (counter (w, y, b, j), j = 0..3, under the init key) give the 32 nodes'
// 16-bit uniforms -- node i takes block i / 8, output word (i mod 8) / 2,
// half i mod 2 -- and the node's bit b is set iff its uniform < P.  Solid
// nodes end without particles.
//
// The integer pipes bound it (28 blocks per word).  A word's blocks share
// their first two rounds' products: round 1 multiplies w and b, round 2 one
// value that depends on b alone and one that depends on j alone.  A uniform is
// compared in the upper half of a register: u < P is (u << 16) <= P * 2^16 - 1,
// which also holds for P = 2^16.  4096 x 4096: 38.5 us, 52 us without sharing.
__global__ void __launch_bounds__(kBlock) init_kernel(Geometry g, uint32_t* __restrict__ state,
                                                      const uint32_t* __restrict__ solid, bool has_solid,
                                                      Key2 key, uint32_t P) {
    const size_t total = (size_t)g.H * g.Pq;
    const uint32_t top = (P << 16) - 1u;
    for (size_t item = (size_t)blockIdx.x * blockDim.x + threadIdx.x; item < total;
         item += (size_t)gridDim.x * blockDim.x) {
        const int y = row_of(item, g.Pq);
        const int w = (int)(item - (size_t)y * g.Pq);
        if (w >= g.Wq || P == 0u) {
            for (int b = 0; b < 7; ++b) state[(size_t)b * g.plane_words + item] = 0u;
            continue;
        }
        const uint32_t fluid = has_solid ? ~solid[item] : 0xFFFFFFFFu;
        const unsigned long long a1 = (unsigned long long)0xD2511F53u * (uint32_t)w;
        unsigned long long b2[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j)
            b2[j] = (unsigned long long)0xCD9E8D57u * ((uint32_t)(a1 >> 32) ^ j ^ key.hi);
        const uint32_t k1_lo = key.lo + 0x9E3779B9u, k1_hi = key.hi + 0xBB67AE85u;
#pragma unroll 1
        for (uint32_t b = 0; b < 7; ++b) {
            const unsigned long long b1 = (unsigned long long)0xCD9E8D57u * b;
            const unsigned long long a2 =
                (unsigned long long)0xD2511F53u * ((uint32_t)(b1 >> 32) ^ (uint32_t)y ^ key.lo);
            uint32_t word = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 r = philox_from_round_2(
                    make_uint4((uint32_t)(b2[j] >> 32) ^ (uint32_t)b1 ^ k1_lo, (uint32_t)b2[j],
                               (uint32_t)(a2 >> 32) ^ (uint32_t)a1 ^ k1_hi, (uint32_t)a2), key);
                const uint32_t outs[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if ((outs[k] << 16) <= top) word |= 1u << (8 * j + 2 * k);
                    if (outs[k] <= top) word |= 2u << (8 * j + 2 * k);
                }
            }
            state[(size_t)b * g.plane_words + item] = word & fluid;
        }
    }
}

// Obstacles from shapes: one thread per word; a node is solid if any shape
// covers it (discs: squared distance in index coordinates, exact in 64-bit
// integers; row bands).  Only the words a disc's edge cuts test every node:
// the distances of a word's two ends decide the others.
__global__ void __launch_bounds__(kBlock) shape_kernel(Geometry g, ShapeList shapes, uint32_t* __restrict__ state,
                                                       uint32_t* __restrict__ solid, unsigned int* any_solid) {
    const size_t total = (size_t)g.H * g.Pq;
    for (size_t item = (size_t)blockIdx.x * blockDim.x + threadIdx.x; item < total;
         item += (size_t)gridDim.x * blockDim.x) {
        const int y = row_of(item, g.Pq);
        const int w = (int)(item - (size_t)y * g.Pq);
        uint32_t word = 0;
        if (w < g.Wq) {
            for (int k = 0; k < shapes.n; ++k) {
                const Shape sh = shapes.s[k];
                if (sh.kind == 2) {
                    if (y >= sh.a && y < sh.b) word = 0xFFFFFFFFu;
                } else if (sh.kind == 1) {
                    const long long dy = (long long)y - sh.b;
                    const long long r2 = (long long)sh.c * sh.c - dy * dy;
                    if (r2 < 0) continue;
                    const long long lo = (long long)(32 * w) - sh.a, hi = lo + 31;
                    if (lo > sh.c || hi < -(long long)sh.c) continue;
                    if (lo * lo <= r2 && hi * hi <= r2) {
                        word = 0xFFFFFFFFu;
                        continue;
                    }
                    if ((lo > 0 && lo * lo > r2) || (hi < 0 && hi * hi > r2)) continue;
                    for (int i = 0; i < 32; ++i) {
                        const long long dx = (long long)(32 * w + i) - sh.a;
                        if (dx * dx <= r2) word |= 1u << i;
                    }
                }
            }
        }
        const size_t off = (size_t)y * g.Pq + w;
        solid[off] = word;
        if (word) {
            for (int b = 0; b < 7; ++b) state[(size_t)b * g.plane_words + off] &= ~word;
            if (any_solid) atomicOr(any_solid, 1u);
        }
    }
}

}  // namespace

cudaError_t launch_obstacle_shapes(const Geometry& g, const ShapeList& shapes, uint32_t* state, uint32_t* solid,
                                   unsigned int* device_any_solid, cudaStream_t stream) {
    shape_kernel<<<grid_for((size_t)g.H * g.Pq / 32 + 1), kBlock, 0, stream>>>(g, shapes, state, solid,
                                                                               device_any_solid);
    return cudaGetLastError();
}

cudaError_t launch_init_random(const Geometry& g, uint32_t* state, const uint32_t* solid, bool has_solid,
                               uint64_t seed, double density, cudaStream_t stream) {
    const double scaled = density * 65536.0;
    uint32_t P;
    if (!(scaled > 0.0)) P = 0;
    else if (scaled >= 65536.0) P = 65536;
    else P = (uint32_t)std::nearbyint(scaled);  // nearest, ties to even
    const Key2 key{(uint32_t)seed ^ 0x9E3779B9u, (uint32_t)(seed >> 32) ^ 0x7F4A7C15u};
    init_kernel<<<grid_for((size_t)g.H * g.Pq / 32 + 1), kBlock, 0, stream>>>(g, state, solid, has_solid, key, P);
    return cudaGetLastError();
}

cudaError_t launch_pack(const Geometry& g, const uint8_t* bytes, uint32_t* state, uint32_t* solid,
                        unsigned int* device_any_solid, cudaStream_t stream) {
    if (((uintptr_t)bytes & 31u) != 0) {
        pack_kernel<<<grid_for((size_t)g.H * g.Pq), kBlock, 0, stream>>>(g, bytes, state, solid, device_any_solid);
        return cudaGetLastError();
    }
    const int step = rows_per_launch(g);
    for (int y = 0; y < g.H; y += step) {
        const uint32_t total = (uint32_t)(g.H - y < step ? g.H - y : step) * (uint32_t)g.Pq;
        const size_t off = (size_t)y * g.Pq;
        auto kernel = g.Wq == g.Pq ? pack_words_kernel<false> : pack_words_kernel<true>;
        kernel<<<(total + kBlock - 1) / kBlock, kBlock, 0, stream>>>(g.Wq, g.Pq, total, g.plane_words,
                                                                    bytes + (size_t)y * g.W, state + off, solid + off,
                                                                    device_any_solid);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_unpack(const Geometry& g, const uint32_t* state, const uint32_t* solid,
                          uint8_t* bytes, cudaStream_t stream) {
    if (((uintptr_t)bytes & 31u) != 0) {
        unpack_kernel<<<grid_for((size_t)g.H * g.Wq), kBlock, 0, stream>>>(g, state, solid, bytes);
        return cudaGetLastError();
    }
    const int step = rows_per_launch(g);
    for (int y = 0; y < g.H; y += step) {
        const uint32_t total = (uint32_t)(g.H - y < step ? g.H - y : step) * (uint32_t)g.Wq;
        const size_t off = (size_t)y * g.Pq;
        auto kernel = g.Wq == g.Pq ? unpack_words_kernel<false> : unpack_words_kernel<true>;
        kernel<<<(total + kBlock - 1) / kBlock, kBlock, 0, stream>>>(g.Wq, g.Pq, total, g.plane_words, state + off,
                                                                    solid + off, bytes + (size_t)y * g.W);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_load_obstacles(const Geometry& g, const uint8_t* mask, uint32_t* state,
                                  uint32_t* solid, unsigned int* device_any_solid,
                                  cudaStream_t stream) {
    obstacle_kernel<<<grid_for((size_t)g.H * g.Pq), kBlock, 0, stream>>>(g, mask, state, solid,
                                                                        device_any_solid);
    return cudaGetLastError();
}

}  // namespace fhp
