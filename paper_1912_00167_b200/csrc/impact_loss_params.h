// Parameters of the loss kernels, shared by the host entry points and the translation units that instantiate kernels
// (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "impact.h"
#include "impact_device.cuh"
#include "impact_internal.h"

namespace impact {

using dev::LossScalars;

constexpr int kWsMaxStages = 24;      // stages of a persistent kernel's ring at most
// A workspace: 128 KB of spare slots for split launches of wide rows, the counter words, the tagged rows, the tiles' aggregates
// where there is room.
constexpr int kMaxGridBlocks = 4096;  // (32 bytes each of the first part)
constexpr long long kSpareSlots = kMaxGridBlocks * 32ll / 8;
constexpr size_t kCounterBytes = 256; // words: [0] unused, [1] error flag, [2] launch number
constexpr int kMaxTaggedRows = 1024;  // rows of eight (value, tag) pairs after the counter words: one per block of a persistent kernel
constexpr int kMinTileRows = 64;      // the smallest tile that tile_aggregates has room for

// How a batch is laid out over the grid (see impact_flat.cuh).
struct BatchGeometry {
    long long B, T;
    int nt;          // rows of a tile
    int ntiles;      // long: tiles per trajectory
    int tile_major;  // long: order of the grid's tiles
};

struct CatParams {
    const void* learner_logits;
    const void* target_logits;
    const float* worker_logp;
    const int32_t* actions;
    const float* rewards;
    const float* discounts;
    const float* values;
    const float* bootstrap;
    float* loss_terms;
    void* dlogits;
    float* dvalues;
    float* vtarget;
    float* advantage;
    unsigned int* counter;
    unsigned long long* tagged_rows;      // rows of (value, launch tag) pairs, see dev::publish_tagged
    unsigned long long* tile_aggregates;  // long launches: two (value, launch tag) pairs per tile (NULL = no room for them)
    unsigned long long* block_values;     // long launches of wide rows: see dev::value_from_later_tiles (NULL = no room)
    unsigned long long* spare_slots;      // kSpareSlots of the workspace's (NULL = a call without one)
    void* target_copy;  // where the target logits are written as well (NULL = nowhere)
    const impact_loss_inputs* indirect;  // device record that overrides the nine input pointers above (NULL = none)
    BatchGeometry geo;
    LossScalars k;
    int A;
};

struct GaussParams {
    const float* learner_mean;
    const float* learner_logstd;
    const float* target_mean;
    const float* target_logstd;
    const float* actions;
    const float* worker_logp;
    const float* rewards;
    const float* discounts;
    const float* values;
    const float* bootstrap;
    float* loss_terms;
    float* dmean;
    float* dlogstd;
    float* dvalues;
    float* vtarget;
    float* advantage;
    unsigned int* counter;
    unsigned long long* tagged_rows;
    unsigned long long* tile_aggregates;
    unsigned long long* spare_slots;
    BatchGeometry geo;
    LossScalars k;
    int D;
};

// The rest of a launch's shape.
struct LaunchForm {
    int nt, stages, in_flight, lanes, n_prefetch, prefetch_arrays;
    int log_lanes, passes, rot_shift, rot_mask;  // how rows are laid on lanes (see impact_categorical.cuh)
};

struct LossInputPointers {
    const void* learner_logits;
    const void* target_logits;
    const float* worker_logp;
    const int32_t* actions;
    const float* rewards;
    const float* discounts;
    const float* values;
    const float* bootstrap;
    void* target_copy;
};

// Picks the kernel for a categorical call (`p` complete except for geo.nt and what follows it) and launches it.  Every count
// up to 32 is compiled in, in two kinds of translation units: told at run time, a row of 1 to 16 actions takes a warp some 200
// to 350 instructions more for tests of what is there (926 000 steps of 7 actions in fp32 24.3 against 20.2 us, 2.1 million of
// 2 actions 46.9 against 30.1), one of 17 to 32 takes 1.1 to 1.2 times as long in fp32, 1.3 to 1.5 in bf16 (20 actions 21.2
// against 17.5 us, in bf16 21.5 against 15.6, with every switch 33.0 against 20.5).
constexpr bool is_compiled_count(int A) { return A <= 16 || A == 18; }
constexpr bool is_larger_count(int A) { return A <= 32; }
template <typename LT, typename GT>
int32_t run_compiled_count(const CatParams& p, const DeviceInfo* di, cudaStream_t stream);
template <typename LT, typename GT>
int32_t run_larger_count(const CatParams& p, const DeviceInfo* di, cudaStream_t stream);
template <typename LT, typename GT, int kV>  // more than 32 actions, of which kV are read at a time (1: odd counts)
int32_t run_runtime_width(const CatParams& p, const DeviceInfo* di, cudaStream_t stream);

int32_t run_gaussian(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <int kPart>  // (one specialisation per translation unit, see impact_gaussian.cu)
int32_t run_gaussian_part(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <> int32_t run_gaussian_part<0>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <> int32_t run_gaussian_part<1>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <> int32_t run_gaussian_part<2>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <> int32_t run_gaussian_part<3>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <> int32_t run_gaussian_part<4>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <> int32_t run_gaussian_part<5>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);
template <> int32_t run_gaussian_part<6>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream);

// Stages of a ring that a block has room for; 4 KB are left for static shared memory.
inline int stages_that_fit(size_t stage_bytes, int max_smem) { return (int)((size_t)(max_smem - 4096) / stage_bytes); }
// Tiles the producer keeps in flight and stages of the ring, for tiles of `tile_in_bytes` bytes of logits.
void ws_ring_shape(size_t stage_bytes, size_t tile_in_bytes, int groups, int max_smem, long long tiles_per_block,
                   int* stages, int* in_flight, bool cold = false);
// Does a companion (impact_prefetch.cu) pay for a categorical launch of `rows` steps of `row_bytes` inputs each?  (Where
// ws_plan finds its tiles large and few enough.)  Both sides measured, companion / none, in us, on inputs that come from HBM;
// where a program's inputs are still in L2 a companion can only cost (1024 x 128 of 18 actions 7.9 / 7.5, cold 7.5 / 7.9).
//   Rows wider than 32 actions: no.  It gains nothing with fp32 logits and doubles a launch with bf16 ones (27 / 14 at 65 536
//   steps).
//   Split trajectories: up to 28 MB.  Up to 18 actions they gain, their tiles being spread over the device (31 x 4000 steps of 9
//   actions 11.1 / 13.6, of 18 13.1 / 13.5, in bf16 12.8 / 14.8); where blocks have fewer than four and a half tiles only small
//   tiles gain without losing as much on inputs in L2 (16 x 4096 of 9 7.3 / 8.3, in L2 7.7 / 7.8; of 12 7.8 / 8.4 and 7.7 / 8.0;
//   of 18 8.5 / 8.8 but 9.1 / 8.4).  More actions: not at up to four tiles (16 x 4096 in bf16 of 24 actions 10.7 / 10.1, of 20
//   10.1 / 9.1; at 4.3 tiles 20 x 4096 of 24 in fp32 11.4 / 12.1).
//   Whole trajectories: not where a group has about a tile, all of which are asked for at once (600 x 100 of 12 5.6 / 5.5, in L2
//   5.6 / 4.8; of 24 in bf16 6.8 / 6.0 and 6.7 / 5.1); nor where tiles are small but for large batches (1024 x 128 of 9 6.7 / 7.0, in
//   L2 6.8 / 6.0; 2500 x 100 with every switch 10.2 / 11.1, in L2 10.4 / 10.4).
//   Otherwise by the tiles that a block has in flight, behind whose requests the next launch's companion puts its own: three and
//   more (fp32 logits of up to 23 actions) up to 25.5 MB (1024 x 128 of 20 7.8 / 8.2, 1180 x 128 10.4 / 9.1), with bf16 gradients
//   28 MB (8.1 / 8.5); two up to 22 MB (800 x 128 of 24 8.0 / 8.2, 900 x 128 10.9 / 9.0; 700 x 128 of 28 8.0 / 8.1, 800 x 128
//   10.7 / 8.7).
constexpr size_t kSmallTile = 12 * 1024 + 512;
inline bool companion_pays(int A, bool split, long long rows, size_t row_bytes, int nt, long long tiles,
                           long long grid, int in_flight, size_t grad_bytes) {
    if (A > 32) return false;
    const long long bytes = rows * (long long)row_bytes;
    const bool few_tiles = 2 * rows < 9 * grid * nt;
    if (split) return bytes <= 28000000 && (A > 18 ? tiles > 4 * grid : !few_tiles || nt * row_bytes <= 15 * 1024);
    if (few_tiles || (nt * row_bytes < kSmallTile && bytes < 20000000)) return false;
    return bytes <= (in_flight < 3 ? 22000000 : grad_bytes == 4 ? 25500000 : 28000000);
}
// How many tiles per block are asked for in L2 ahead of time, and by whom.
struct WsPlan {
    int prefetch_tiles;  // tiles per block asked for in L2 ahead of time
    bool companion;      // by a companion kernel enqueued before the loss kernel (else by the loss kernel's first warp)
};
WsPlan ws_plan(long long tiles, long long grid, size_t tile_bytes, int in_flight, bool allow_companion);

// What the first warp of a launch without a companion asks L2 for: the tiles that it is about to request, while the dependency
// resolves.  What is not done by then delays the tiles.  In us: nothing / rows of logits / the per-step arrays too.
//   Nothing where tiles are small: 2500 x 100 steps of 8 actions 9.2 / 9.4 / 10.1, 5243 x 50 of 18 in bf16 11.0 / 11.3 / 11.8,
//   Gaussian 8000 x 50 of 4 dimensions 14.3 / 16.0 / 16.4.
//   Nothing where a block has few tiles (fewer than `few` fifths of one) and they are not large: 300 x 50 of 12 3.7 / 4.0 / 4.4, of
//   18 4.0 / 4.1 / 4.4; 600 x 50 of 18 5.0 / 4.8 / 5.1, but with inputs in L2 4.0 and 5.3 with all; Gaussian 600 x 50 of 8
//   dimensions 5.7 / 5.8, in L2 4.7 / 5.5, though 512 x 128 7.4 / 6.8 and 5.5 / 6.3.
//   Rows of logits up to `all_from` bytes to a tile (categorical 16 KB, Gaussian 24): 2500 x 100 of 10 9.8 / 9.5 / 10.2, of 12
//   10.5 / 9.8 / 10.0, Gaussian 512 x 128 of 8 dimensions 7.4 / 6.7 / 6.8.
//   All beyond: 2500 x 100 of 32 in bf16 13.8 / 13.7 / 13.0, of 24 with every switch 17.8 / 19.0 / 16.5, 40 x 1000 of 64 12.1 / 11.2 / 10.3.
//   Split trajectories, whose tiles are asked for one by one: nothing up to 18 actions (16 x 4096 of 18 9.3 / 9.0 / 8.7, in L2 6.4 and 8.7
//   with all), all beyond (of 24 12.0 / 10.4, in bf16 12.0 / 9.8).
struct OwnRequests {
    int tiles;
    bool slabs_only;
};
inline OwnRequests own_requests(const WsPlan& plan, size_t tile_bytes, long long rows, long long grid, int nt, size_t all_from, int few) {
    const long long tile_rows = grid * nt;
    OwnRequests r = {plan.prefetch_tiles, tile_bytes < all_from};
    if (tile_bytes < kSmallTile || (5 * rows < few * tile_rows && tile_bytes < 30 * 1024)) r.tiles = 0;
    return r;
}

// The share of the SM's shared memory that a launch with a companion asks to have laid out as such, in percent, for blocks of
// `smem` bytes: room for a block of the next launch's companion beside one of its own (a kilobyte of either is the system's).
// By itself the driver picks the smallest layout that a block fits; where that leaves no room, the companion cannot become
// resident beside the launch: all its blocks start on the first SMs that come free, whose copy engines then ask L2 for the whole
// batch (16 actions in fp32, 16 x 4096 steps 16.2 us, 8.4 so; 1024 x 128 with every switch 24 and 8.5).  No more than that, and
// nothing without a companion, because the rest is the L1 that per-step arrays and split trajectories' aggregates are read
// through.  With all of it as shared memory: 31 x 4000 steps of 18 actions in bf16 13.4 us instead of 12.8, of 32 in fp32 22.8
// instead of 20.0 (no companion), 14 x 2091 of 64 with every switch 14.8 instead of 13.4, Gaussian 28 012 x 28 of 3 dimensions
// 19.3 instead of 18.9.
constexpr size_t kRingStepShared = 20 * 1024;  // of a one-warp block of the ring's step, which runs between loss launches
inline int percent_beside(size_t smem, size_t other, const DeviceInfo* di) {
    const size_t percent = (100 * (smem + other + 2048) + di->smem_per_sm - 1) / di->smem_per_sm;
    return percent < 100 ? (int)percent : 100;
}

// The companion of a categorical launch of `grid` blocks: asks L2 for each block's first `n_tiles` tiles.
int32_t launch_companion(const CatParams& p, int elem_bytes, bool is_long, int n_tiles, int grid, cudaStream_t stream);

}  // namespace impact
