// fhp_internal.h -- layout and launcher declarations shared by the library's
// translation units (not part of the public ABI).
//
// Device layout of one lattice of W x H nodes (W multiple of 32, H even):
//   Wq = W / 32 words per row, nq = ceil(Wq / 4) quads of 4 words per row,
//   row pitch Pq = 4 * nq words (16-byte aligned rows; the words Wq..Pq-1 of
//   every row are padding and stay zero).  A plane is H * Pq words; a state
//   buffer is 7 consecutive planes (planes 0..5 movers along c_0..c_5,
//   plane 6 rest particles); the solid flags form one more plane.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace fhp {

struct Key2 {
    uint32_t lo, hi;
};

struct ForcingTable {
    unsigned long long q[33];
    // P + 1 with P = round(p * 2^32): Q_K <= K (P + 1), so u >= K (P + 1)
    // proves that none of K candidates is forced (cheap exact pre-check).
    unsigned long long p_plus_1;
    // The pre-check in 32 bits: u < K * pre is the same test for P + 1 <
    // 2^27 (32 candidates do not overflow); for larger P (p >= 1/32, where
    // most warps hold a forced node anyway) pre is 0 and dense is 1: every
    // quad then takes the exact walk.
    uint32_t pre;
    uint32_t dense;
    uint32_t inv;   // floor(2^32 / (P + 1)): (u * inv) >> 32 never exceeds the least g with u < Q_g, minus 1
};

struct Geometry {
    int W = 0, H = 0;
    int Wq = 0;         // words per row
    int nq = 0;         // quads per row
    int Pq = 0;         // row pitch in words (multiple of 4)
    size_t plane_words = 0;  // H * Pq
    int row_base = 0;   // lattice row of array row 0 (a strip of a larger lattice; even)
    int rules = 2;      // collision rule set: 2 = FHP-II, 1 = FHP-I, 3 = FHP-III (direct and ring kernels)
};

// Forcing thresholds of probability p (host): P = round-half-even(p * 2^32),
// computed from the integer and fraction parts of the exact double p * 2^32
// (independent of the floating-point rounding mode); S_0 = 2^32,
// S_g = floor(S_{g-1} (2^32 - P) / 2^32), Q_g = 2^32 - S_g (exact integers).
ForcingTable forcing_table(double p);

// Mask that enables the rest-particle rules of the bit-sliced scattering.
inline uint32_t rest_rules_mask(const Geometry& g) { return g.rules == 1 ? 0u : 0xFFFFFFFFu; }

Geometry make_geometry(int W, int H);

// SMs of the current device (0: unknown).
int sm_count();

// Arguments of one k = 1 step kernel launch.
struct StepArgs {
    const uint32_t* __restrict__ src;    // 7 planes of S_t
    uint32_t* __restrict__ dst;          // 7 planes of S_{t+1}
    const uint32_t* __restrict__ solid;  // solid plane (read only if has_solid)
    unsigned long long plane_words;
    int H, Wq, nq, Pq;
    int rows_per_warp;       // nq < 32: rows of one parity packed into a warp
    int groups_per_parity;   // nq < 32: warps per row parity
    int warps_per_row;       // nq >= 32: warps covering one row
    Key2 key;
    uint32_t t_lo, t_hi;
    unsigned int* err;       // set nonzero if a bounded device-side wait gives up
    int y_base = 0;          // added to the row index that keys the random words (strips)
    uint32_t rest_rules = 0xFFFFFFFFu;  // ones: FHP-II rest-particle rules on; zero: FHP-I
    ForcingTable ft;
};

// Row tiling of the bulk-copy step kernel: tiles of R full rows, staged in a
// ring of shared-memory buffers by cp.async.bulk.
struct TileArgs {
    int R;                         // rows per tile
    int ntiles;                    // ceil(H / R)
    unsigned long long nq_magic;   // ceil(2^32 / nq): j / nq == (j * nq_magic) >> 32 for small j
};

// Step kernel choice: automatic, direct register loads, or the bulk-copy ring
// (cp.async.bulk into shared memory; falls back to direct when a row does not
// fit a stage).
// kStepRun: the ring kernel running many steps in one cooperative launch
// (per-tile dependency counters instead of a launch per step).
// kStepResident: lattices that fit in the SMs' shared memory stay on chip for
// all steps of a call (fhp_resident.cu).
enum StepKernel { kStepAuto = 0, kStepDirect = 1, kStepRing = 2, kStepRun = 3, kStepResident = 4 };

// Launch one time step (motion, scattering, bounce-back, forcing).
// `err` (device word, may be NULL) is set nonzero if a bounded wait gives up.
cudaError_t launch_step(const Geometry& g, const uint32_t* src, uint32_t* dst,
                        const uint32_t* solid, bool has_solid, bool force,
                        const ForcingTable& ft, Key2 key, uint64_t t, cudaStream_t stream,
                        unsigned int* err = nullptr, int kernel = kStepAuto);

// The kernel fhp_step uses for `requested`: kStepDirect, kStepRing or kStepRun
// (launch_step itself runs single_step_kernel's for kStepRun: one step per
// launch).
int resolved_step_kernel(const Geometry& g, bool has_solid, bool force, int requested);

// The faster kernel of single steps: kStepDirect or kStepRing.
int single_step_kernel(const Geometry& g, bool has_solid, bool force);

// Tiles of the ring / multi-step kernels (0 if a row does not fit a stage);
// the multi-step kernel needs that many counter words of scratch.
int run_tiles(const Geometry& g, bool has_solid);

// n >= 1 steps from buf0 (state at t0) in one cooperative launch; the result
// is in buf0 if n is even, else in buf1.  `done` holds run_tiles() words of
// scratch (zeroed by the call on the stream).
cudaError_t launch_run(const Geometry& g, uint32_t* buf0, uint32_t* buf1, const uint32_t* solid,
                       bool has_solid, bool force, const ForcingTable& ft, Key2 key, uint64_t t0,
                       int nsteps, unsigned int* done, cudaStream_t stream, unsigned int* err);

// Shared-memory resident lattices (fhp_resident.cuh): `gh` is the number of
// steps between exchanges (1, 2 or 4), of which every strip computes gh ghost
// rows per side itself.  Supported when the strips fit in shared memory and the
// exchange fits `staging_bytes` of scratch (the lattice's byte-staging area).
// n >= 1 steps from buf0 (state at t0); the result is in buf1 if
// resident_flips(n, gh), else in buf0.
bool resident_supported(const Geometry& g, bool has_solid, size_t staging_bytes, int gh = 1);
// The interval expected to be fastest (0: not supported).
int resident_interval_for(const Geometry& g, bool has_solid, size_t staging_bytes, bool force);
// The least number of steps for which moving the lattice into shared memory and
// back pays (the direct kernel takes shorter calls of the automatic choice).
int resident_least_steps(const Geometry& g, bool force);
// Every strip loads its own rows and its neighbours' edge rows from buf0.  Only
// the first exchange of edge rows, after step gh, tells a strip that its
// neighbours have done so: a call of up to gh steps has none, and must not
// store into buf0 what a strip that starts late has yet to load.
constexpr bool resident_flips(int nsteps, int gh) { return nsteps % 2 != 0 || nsteps <= gh; }
cudaError_t launch_resident(const Geometry& g, uint32_t* buf0, uint32_t* buf1, const uint32_t* solid, bool has_solid,
                            bool force, const ForcingTable& ft, Key2 key, uint64_t t0, int nsteps, int gh,
                            uint32_t* halo, size_t halo_bytes, cudaStream_t stream, unsigned int* err);

// Temporal blocking: k (2, 4 or 8) steps from src (state at t0) to dst in one
// pass.  Supported when rows are whole quads (W multiple of 128), there are
// at least 4 quads per row and H >= 2k + 2.
bool block_supported(const Geometry& g, int k);
cudaError_t launch_block(const Geometry& g, const uint32_t* src, uint32_t* dst, const uint32_t* solid,
                         bool has_solid, bool force, const ForcingTable& ft, Key2 key, uint64_t t0, int k,
                         cudaStream_t stream, unsigned int* err);

// Temporal blocking inside batches (fhp_batch_block.cu): one launch applies
// pass `pass` (k = 2 or 4 steps) to every member with more passes than that
// in the call, tile by tile over a list of (member, row tile) records.  A
// member's tile holds R_out full rows (even; batch_block_rows, 0 if the
// member's rows are too wide); the kernel stages R_out + 2k rows of the
// member's pitch in each of 16 shared-memory planes of kBBPlaneWords words.
constexpr int kBBPlaneWords = 3072;
struct BlockMember {
    StepArgs a;              // geometry, solid plane, key, forcing, rules, err (src, dst, t: set per pass)
    uint32_t* buf[2];        // state buffers; buf[cur] holds the state at step t0
    unsigned long long t0;   // the member's step at the start of the call
    int cur;
    int passes;              // blocked passes of the member in the call
    int R_out;               // output rows per tile
    int force;               // forcing probability nonzero
    int y0, rows_out, active;  // per tile: filled in by the kernel in its shared-memory copy
    int pad;
};
struct BlockTile {
    int lattice;             // index into the member table
    int tile;                // row tile of the member
};
int batch_block_rows(const Geometry& g, int k);
cudaError_t configure_batch_block();   // kernel attributes of the current device (first use loads the kernel)
cudaError_t launch_batch_block(const BlockMember* d_members, const BlockTile* d_tiles, int ntiles, int pass, int k,
                               unsigned int* err, cudaStream_t stream);

// Temporal blocking by row wavefronts (fhp_wave.cu): k (2, 3 or 4) steps from
// src (state at t0) to dst in one pass over full-width row bands, the
// intermediate levels in shared-memory row rings.  Supported when a row of
// every level ring fits shared memory (about W <= 16,384 for k = 2 and 3,
// 8,192 for k = 4) and the rule set is FHP-I or FHP-II.
bool wave_supported(const Geometry& g, int k);
cudaError_t launch_wave(const Geometry& g, const uint32_t* src, uint32_t* dst, const uint32_t* solid,
                        bool has_solid, bool force, const ForcingTable& ft, Key2 key, uint64_t t0, int k,
                        cudaStream_t stream, unsigned int* err);

// Temporal blocking in registers (fhp_march.cu): `passes` passes of k (2 or 3)
// steps from src (state at t0); the result is in dst if `passes` is odd, else
// in src.  Every lane marches a quad column up a band of rows; all passes run
// in one cooperative launch, a warp waiting only for the warps around it.  Any
// rule set and row width; needs H >= 2k + 2 and planes of less than 4 GiB.
// `flags` is scratch of `flag_bytes` (a word per warp; too few: one launch per
// pass).
bool march_supported(const Geometry& g, int k);
// ... and whether one resident wave of the current device's warps holds a
// band's columns (rows of up to 7.0 million nodes for k = 3, 9.3 million for k =
// 2 on 152 SMs), without which launch_march refuses.
bool march_fits(const Geometry& g, int k, bool has_solid, bool force);
// Steps per pass for which register marching is the automatic choice (0: it
// is not).
int march_choice(const Geometry& g, const ForcingTable& ft, bool has_solid, bool force);
cudaError_t launch_march(const Geometry& g, uint32_t* src, uint32_t* dst, const uint32_t* solid, bool has_solid,
                         bool force, const ForcingTable& ft, Key2 key, uint64_t t0, int k, int passes,
                         unsigned int* flags, size_t flag_bytes, cudaStream_t stream, unsigned int* err);

struct MarchLayout {
    int pitch;      // chain positions per band (0: whole rows in a warp)
    int left;       // chain positions left of a band's quad 0
    int hl;         // halo lanes per side of a warp (chain)
    int per_warp;   // whole rows: bands per warp
};
MarchLayout march_layout(const Geometry& g, int k);
long long march_warps(const Geometry& g, const MarchLayout& l, int R);   // warps for bands of R rows
int march_rows(const Geometry& g, int k, int R);                         // band height allowed from R on

// Register marching of a batch (fhp_batch_march.cu): all passes of k (2 or 3)
// steps of up to kMarchJobs members in one cooperative launch.  The member
// table is a kernel parameter, and a CTA (kMarchCtaWarps warps) works for one
// member, so that its fields are uniform operands as in the single-lattice
// kernel (read from device memory into registers they spilled: 88 to 560 bytes
// a thread).
constexpr int kMarchJobs = 256;
constexpr int kMarchMaxCtas = 640;
constexpr int kMarchCtaWarps = 4;
struct MarchJob {
    uint32_t* src;             // state at t0; the result where `passes` is even
    uint32_t* dst;
    const uint32_t* solid;
    unsigned long long t0;
    unsigned long long P;      // round(p * 2^32)
    uint32_t plane_words;
    int H, Wq;
    Key2 key;
    uint32_t rest_rules;
    uint32_t pre, dense, inv;  // forcing (ForcingTable)
    MarchLayout lay;
    int R, nbands, nwarps, passes;
    int first_cta;             // the member's first CTA
};
struct MarchBatch {
    MarchJob job[kMarchJobs];
    uint8_t member[kMarchMaxCtas];   // CTA -> job
    unsigned int* flags;             // kMarchCtaWarps words per CTA: passes finished, counted from `epoch`
    unsigned int* err;
    unsigned int epoch;              // no word is above this at launch
};
static_assert(sizeof(MarchBatch) <= 32764, "kernel parameters are limited to 32,764 bytes");
// CTAs one launch may have (all must be resident; at most kMarchMaxCtas).
cudaError_t batch_march_ctas(int k, bool force, bool ragged, int* ctas);
cudaError_t launch_batch_march(const MarchBatch& t, int ctas, int k, bool force, bool ragged, cudaStream_t stream);

// Pack H x W node bytes (device) into 7 state planes + the solid plane.
// Sets *device_any_solid to a nonzero value if any node is solid.
cudaError_t launch_pack(const Geometry& g, const uint8_t* bytes, uint32_t* state,
                        uint32_t* solid, unsigned int* device_any_solid, cudaStream_t stream);

// Generated initial state: bits 0..6 of every fluid node set independently
// with probability round(density * 2^16) / 2^16 from counter-based draws of
// the lattice seed (solid nodes end empty).
cudaError_t launch_init_random(const Geometry& g, uint32_t* state, const uint32_t* solid, bool has_solid,
                               uint64_t seed, double density, cudaStream_t stream);

// Unpack 7 state planes + the solid plane into H x W node bytes (device).
cudaError_t launch_unpack(const Geometry& g, const uint32_t* state, const uint32_t* solid,
                          uint8_t* bytes, cudaStream_t stream);

// Replace the solid plane from an H x W byte mask (nonzero = solid) and clear
// the particles of solid nodes in `state`.
cudaError_t launch_load_obstacles(const Geometry& g, const uint8_t* mask, uint32_t* state,
                                  uint32_t* solid, unsigned int* device_any_solid,
                                  cudaStream_t stream);

// Obstacles from shapes (kinds as FHP_SHAPE_*): replaces the solid plane and
// clears the particles of solid nodes.  *device_any_solid (may be NULL) is
// set nonzero if any node is solid.
struct Shape {
    int kind, a, b, c;
};
struct ShapeList {
    Shape s[8];
    int n;
};
cudaError_t launch_obstacle_shapes(const Geometry& g, const ShapeList& shapes, uint32_t* state, uint32_t* solid,
                                   unsigned int* device_any_solid, cudaStream_t stream);

// Coarse-grain over B x B blocks (B multiple of 32 dividing W and H).
cudaError_t launch_coarse_grain(const Geometry& g, const uint32_t* state, const uint32_t* solid,
                                bool has_solid, int B, int32_t* counts, float* rho, float* ux,
                                float* uy, cudaStream_t stream);

// Record the calling thread's last error (returned by fhp_last_error(NULL)).
void set_thread_error(const char* message);

// Philox4x32-10 over n counters (diagnostic entry point).
cudaError_t launch_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, int64_t n,
                          cudaStream_t stream);

}  // namespace fhp
