// What the persistent loss kernels share: how a batch is laid out over the grid and its rows over lanes, the protocols
// between warps, row access, launch shape.
//
// One block per SM.  A producer warp streams the block's tiles -- consecutive steps of the row-major [B*T, A] logits --
// through a ring of shared-memory stages by bulk asynchronous copies; C consumer groups of four warps take every C-th
// tile as it lands, one thread per step for the recursion and 1 to 32 lanes per step for the row passes, and every
// warp sends its own gradient rows off by a bulk store while later tiles are still arriving.
//
// Two ways to lay the batch out over the grid:
//   flat  (kLong = false): a block owns a contiguous range of whole trajectories and walks its rows from the END, a tile
//         of NT rows at a time, with no regard to where trajectories begin: a step that ends its trajectory has the
//         affine map (0, b), so the recursion is cut there by itself.  Where a trajectory crosses a tile boundary, the
//         value at the later tile's first step passes to the earlier tile through a mailbox in shared memory; only that
//         one multiply-add per tile is serial.  (Packing whole trajectories into tiles instead leaves a fifth of the
//         lanes idle at T = 50 or 100.)
//   long  (kLong = true): tiles of one trajectory on neighbouring blocks, for few long trajectories; the recursion
//         crosses tiles through their affine aggregates, published in the workspace (see the kernel's carry step).
#pragma once

#include "impact_device.cuh"
#include "impact_internal.h"
#include "impact_loss_params.h"

namespace impact {

// ---- geometry ---------------------------------------------------------------------------------------------------
struct Tile {
    long long row0;  // first row of the tile (of the whole batch)
    int nrows;       // rows of the slab that are loaded
    int r;           // long: number of the tile counted from its trajectory's end
    long long traj;  // long: the trajectory
};
// What a block of a flat launch owns.
struct BlockRange {
    long long traj0, r0, r1;  // first trajectory, first row, end of rows
    long long base;           // row of the first tile's first slot: r0, or up to seven rows before it
    int tiles;
};
__host__ __device__ __forceinline__ BlockRange block_range(const BatchGeometry& g, unsigned int block, unsigned int blocks) {
    BlockRange b;
    const long long q = g.B / blocks, rem = g.B - q * blocks, x = block;
    b.traj0 = x * q + (x < rem ? x : rem);
    const long long ntraj = q + (x < rem ? 1 : 0);
    b.r0 = b.traj0 * g.T;
    b.r1 = b.r0 + ntraj * g.T;
    // tiles start on multiples of eight rows, where every row pitch is a multiple of 16 bytes, unless that costs a tile
    const int shift = (int)(b.r0 & 7);
    const long long rows = b.r1 - b.r0;
    const long long tiles = (rows + g.nt - 1) / g.nt;
    const bool fits = rows + shift <= tiles * g.nt;
    b.base = fits ? b.r0 - shift : b.r0;
    b.tiles = (int)tiles;
    return b;
}
// The block's n-th tile in the order in which it works on them.
template <bool kLong>
__host__ __device__ __forceinline__ Tile tile_at(const BatchGeometry& g, const BlockRange& b, int n, int nt,
                                                 unsigned int block, unsigned int blocks) {
    Tile t;
    if (kLong) {
        const long long x = (long long)block + (long long)n * blocks;
        if (g.tile_major) {  // the last tiles of all trajectories first, then the tiles before them, ...
            t.r = (int)((unsigned long long)x / (unsigned long long)g.B);
            t.traj = x - (long long)t.r * g.B;
        } else {  // trajectory by trajectory, each from its last tile backwards
            t.traj = (long long)((unsigned long long)x / (unsigned int)g.ntiles);
            t.r = (int)(x - t.traj * g.ntiles);
        }
        const long long t0 = (long long)(g.ntiles - 1 - t.r) * nt;
        const long long left = g.T - t0;
        t.nrows = left < nt ? (int)left : nt;
        t.row0 = t.traj * g.T + t0;
    } else {
        t.row0 = b.base + (long long)(b.tiles - 1 - n) * nt;
        const long long left = b.r1 - t.row0;
        t.nrows = left < nt ? (int)left : nt;
        t.r = 0;
        t.traj = 0;
    }
    return t;
}
__host__ __device__ __forceinline__ int tiles_of_block(const BatchGeometry& g, const BlockRange& b, bool is_long,
                                                       unsigned int block, unsigned int blocks) {
    if (!is_long) return b.tiles;
    const long long total = g.B * g.ntiles;
    return (int)((total - block + blocks - 1) / blocks);
}
// ... for the block that asks.
__device__ __forceinline__ BlockRange block_range(const BatchGeometry& g) { return block_range(g, blockIdx.x, gridDim.x); }
template <bool kLong>
__device__ __forceinline__ Tile tile_at(const BatchGeometry& g, const BlockRange& b, int n, int nt) {
    return tile_at<kLong>(g, b, n, nt, blockIdx.x, gridDim.x);
}
__device__ __forceinline__ int tiles_of_block(const BatchGeometry& g, const BlockRange& b, bool is_long) {
    return tiles_of_block(g, b, is_long, blockIdx.x, gridDim.x);
}

// Asks L2 for the block's first n_tiles tiles, lane a for array a's rows of `pitch` bytes (base NULL: none), tile after tile in
// the order in which the block wants them, so that the memory system sees the requests in that order too.  The first kSlabs
// arrays are those of logits; of the others, a few bytes to a step, all the tiles' rows are asked for at once where they are
// neighbours (flat launches): a request takes the copy engine some 35 ns whatever its size.  (A request to each array of each
// tile: 2500 x 100 steps of 10 actions 10.8 us instead of 10.2, of 12 10.3 instead of 10.0.)
template <bool kLong, int kSlabs>
__device__ __forceinline__ void ask_for_tiles(const BatchGeometry& g, const BlockRange& br, const void* base, long long pitch,
                                              int n_tiles, int nt, long long total_rows) {
    const bool at_once = !kLong && (int)(threadIdx.x & 31) >= kSlabs;
    for (int n = 0; n < n_tiles; ++n) {
        Tile t = tile_at<kLong>(g, br, n, nt);
        if (at_once) {
            if (n > 0) break;
            const Tile first = tile_at<kLong>(g, br, n_tiles - 1, nt);
            t.nrows += (int)(t.row0 - first.row0);
            t.row0 = first.row0;
        }
        if (base) dev::prefetch_range_l2(base, t.row0 * pitch, (uint32_t)(t.nrows * pitch), total_rows * pitch);
    }
}

// A consumer group's tile: which of its rows are the block's (flat) or exist at all (long) -- [lo, hi), empty for a group
// that has no tile -- and where its first row sits.
struct TileRows {
    long long row0, traj;
    int lo, hi, r;
};
template <bool kLong>
__host__ __device__ __forceinline__ TileRows tile_rows(const BatchGeometry& g, const BlockRange& b, int n, int n_tiles, int nt,
                                                       unsigned int block, unsigned int blocks) {
    const Tile t = tile_at<kLong>(g, b, n < n_tiles ? n : 0, nt, block, blocks);
    TileRows w;
    w.row0 = t.row0; w.traj = t.traj; w.r = t.r;
    w.lo = (!kLong && n == n_tiles - 1) ? (int)(b.r0 - b.base) : 0;
    w.hi = n < n_tiles ? t.nrows : 0;
    return w;
}
// (flat) How many steps follow a row in its trajectory, and the trajectory (counted from the block's first).  Counted in
// 32 bits (Steps) where trajectories are short enough, see fits_flat.
template <typename Steps>
struct StepPlace {
    Steps to_end;
    unsigned int traj;
};
template <typename Steps>
__host__ __device__ __forceinline__ StepPlace<Steps> step_place(const BlockRange& b, long long row, Steps T) {
    const unsigned long long rho = row > b.r0 ? (unsigned long long)(row - b.r0) : 0ull;
    const unsigned long long q = rho / T;
    StepPlace<Steps> s;
    s.to_end = T - 1u - (Steps)(rho - q * T);
    s.traj = (unsigned int)q;
    return s;
}
// The place `back` rows further back, back = back_traj * T + back_rest.
template <typename Steps>
__host__ __device__ __forceinline__ void step_back(StepPlace<Steps>& s, unsigned int back_traj, Steps back_rest, Steps T) {
    s.to_end += back_rest;
    const bool wrapped = s.to_end >= T || s.to_end < back_rest;
    s.to_end -= wrapped ? T : (Steps)0;
    s.traj -= back_traj + (wrapped ? 1u : 0u);
}
// (flat) Is every slot of tile n a row of the block's, and is the row behind the last one too?  Then its per-step arrays
// are read without a look at the row.  (A group without a tile, n >= n_tiles, stands on the block's first tile, whose rows
// may end anywhere: it reads none.)
__host__ __device__ __forceinline__ bool rows_unguarded(const TileRows& t, int n, int n_tiles) {
    return n > 0 && n < n_tiles && t.lo == 0;
}

// A slab in shared memory: nt rows of `row_bytes`, plus 32 bytes of padding, because a tile's rows sit at the same
// offset inside their 16-byte granule as in global memory (0..15 bytes after the slab's start) and the copy that
// brings them is widened to whole granules (see dev::widen_range).
__host__ __device__ constexpr size_t slab_pitch(size_t nt, size_t row_bytes) { return nt * row_bytes + 32; }
// ---- row access -------------------------------------------------------------------------------------------------
// kV neighbouring elements of a row in shared memory, in their storage type, as one access.
template <typename ST, int kV> struct Vec;
template <> struct Vec<float, 1> {
    static __device__ __forceinline__ void ld(const unsigned char* p, float* f) { f[0] = *reinterpret_cast<const float*>(p); }
    static __device__ __forceinline__ void st(unsigned char* p, const float* f) { *reinterpret_cast<float*>(p) = f[0]; }
};
template <> struct Vec<float, 2> {
    static __device__ __forceinline__ void ld(const unsigned char* p, float* f) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        f[0] = v.x; f[1] = v.y;
    }
    static __device__ __forceinline__ void st(unsigned char* p, const float* f) { *reinterpret_cast<float2*>(p) = make_float2(f[0], f[1]); }
};
template <> struct Vec<float, 4> {
    static __device__ __forceinline__ void ld(const unsigned char* p, float* f) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
    }
    static __device__ __forceinline__ void st(unsigned char* p, const float* f) {
        *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
    }
};
template <> struct Vec<__nv_bfloat16, 1> {
    static __device__ __forceinline__ void ld(const unsigned char* p, float* f) {
        f[0] = __uint_as_float((uint32_t)*reinterpret_cast<const unsigned short*>(p) << 16);
    }
    static __device__ __forceinline__ void st(unsigned char* p, const float* f) {
        *reinterpret_cast<__nv_bfloat16*>(p) = __float2bfloat16_rn(f[0]);
    }
};
template <> struct Vec<__nv_bfloat16, 2> {
    static __device__ __forceinline__ void ld(const unsigned char* p, float* f) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
        f[0] = __uint_as_float(w << 16); f[1] = __uint_as_float(w & 0xFFFF0000u);
    }
    static __device__ __forceinline__ void st(unsigned char* p, const float* f) {
        *reinterpret_cast<uint32_t*>(p) = dev::bf16_pair(f[0], f[1]);
    }
};
template <> struct Vec<__nv_bfloat16, 4> {
    static __device__ __forceinline__ void ld(const unsigned char* p, float* f) {
        const uint2 w = *reinterpret_cast<const uint2*>(p);
        f[0] = __uint_as_float(w.x << 16); f[1] = __uint_as_float(w.x & 0xFFFF0000u);
        f[2] = __uint_as_float(w.y << 16); f[3] = __uint_as_float(w.y & 0xFFFF0000u);
    }
    static __device__ __forceinline__ void st(unsigned char* p, const float* f) {
        *reinterpret_cast<uint2*>(p) = make_uint2(dev::bf16_pair(f[0], f[1]), dev::bf16_pair(f[2], f[3]));
    }
};
// Overwrites one element after vector stores to the same row; an explicit shared-memory store keeps it ordered behind
// them.
template <typename ST>
__device__ __forceinline__ void put_element(unsigned char* row, int col, float x) {
    if constexpr (sizeof(ST) == 4) {
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(dev::smem_addr(row) + (uint32_t)col * 4u), "f"(x) : "memory");
    } else {
        const unsigned short h = __bfloat16_as_ushort(__float2bfloat16_rn(x));
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(dev::smem_addr(row) + (uint32_t)col * 2u), "h"(h) : "memory");
    }
}
template <typename ST>
__device__ __forceinline__ float get_element(const unsigned char* row, int col) {
    float f;
    Vec<ST, 1>::ld(row + col * (int)sizeof(ST), &f);
    return f;
}

// ---- the recursion's scan ---------------------------------------------------------------------------------------
// Suffix composition of the lanes' affine maps: lane l ends up with f_l o f_{l+1} o ... o f_{l + limit}, where limit is
// what is left of the lane's trajectory (or of the warp): nothing of another trajectory enters, not even times zero.
__device__ __forceinline__ void warp_suffix_compose(float& a, float& b, int limit) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const float a2 = __shfl_down_sync(0xffffffffu, a, off);
        const float b2 = __shfl_down_sync(0xffffffffu, b, off);
        asm("{\n\t.reg .pred p;\n\tsetp.ge.s32 p, %4, %5;\n\t"
            "@p fma.rn.f32 %1, %0, %3, %1;\n\t"
            "@p mul.rn.f32 %0, %0, %2;\n\t}"
            : "+f"(a), "+f"(b) : "f"(a2), "f"(b2), "r"(limit), "r"(off));
    }
}

// Barrier protocol of the persistent kernels (S stages, at most W tiles in flight, lanes <= S - W):
//   full[s]     one arrival (a producer lane's, with the bytes the tile's two copies will deliver): stage s holds
//               the rows of its current tile.
//   empty[s]    one arrival per consumer warp, after that warp's stores have finished reading the stage.
// A wait names a phase by its PARITY, which is only unambiguous while the waiter is at most one phase ahead of the
// barrier: asked about phase k while phase k-1 is still open, the barrier answers "complete".  The producer
// therefore issues tiles STRICTLY in order, and tile n only after (a) tile n-W has landed and
// (b) every consumer warp has released tile n-S.  From that:
//   * consumer of tile n waits on full[n % S] for phase n/S.  It got there after consuming tile n-C, so n-C was
//     issued, so (in order) tile n-S+W <= n-C was issued, so by (a) tile n-S -- phase n/S - 1 of the same stage --
//     had landed: the barrier is in phase n/S or later.  It cannot be beyond n/S + 1 open, because tile n+S is not
//     issued before this consumer releases tile n (b).  (This is where S >= W + C is needed.)
//   * producer's look at full[(n-W) % S] for phase (n-W)/S: tile n-W was issued, so by (b) tile n-W-S was consumed,
//     hence had landed: phase (n-W)/S - 1 is complete; tile n-W+S > n is not issued yet.
//   * producer's look at empty[n % S] for phase n/S - 1: tile n-S was issued, so by (b) phase n/S - 2 is complete;
//     phase n/S needs the consumers of tile n, which is not issued yet.
// Without the in-order rule (lanes that found their own tile ready first went first) the first argument fails for
// tiles of one round: a consumer could be handed a stage whose previous tile had not landed, read stale rows,
// release the stage early, and the phases slipped until one of the bounded waits ran out.

// ---- waits ------------------------------------------------------------------------------------------------------
// The first look is inline (the barrier's own wait usually covers it); what follows is out of the way of the loop.
static __device__ __noinline__ bool stage_wait_rest(uint64_t* bar, uint32_t parity, int* abort_flag) {
    return dev::mbarrier_wait(bar, parity, abort_flag);
}
__device__ __forceinline__ bool stage_wait(uint64_t* bar, uint32_t parity, int* abort_flag) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(dev::smem_addr(bar)), "r"(parity) : "memory");
    return __all_sync(0xffffffffu, done) ? true : stage_wait_rest(bar, parity, abort_flag);
}
// A warp hands its part of a stage back, once its lane 0's bulk stores have read it.  The other lanes may have copied bytes
// of the stage themselves (dev::warp_send_bytes); the warp's barrier puts those reads before the arrival that lets the
// producer overwrite the stage.
__device__ __forceinline__ void hand_back_stage(uint64_t* empty, int lane) {
    dev::bulk_store_wait_read();
    __syncwarp();
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(dev::smem_addr(empty)), "r"((uint32_t)(lane == 0)) : "memory");
}

// ---- the mailbox of a flat launch -------------------------------------------------------------------------------
// The block's n-th tile leaves the value at its first step in slot n mod 32 as one 8-byte (value, n + 1) pair; tile
// n + 1 reads it there.  A slot is not written again before it has been read: tile n + 32 is requested only after
// tile n + 32 - S was handed back by its four warps, S <= 24 stages, tiles are requested in order, and a warp of tile
// n + 1 reads the mailbox before it hands its stage back; a block with no more tiles than stages never uses a slot twice.
constexpr int kMailSlots = 32;
static_assert(kWsMaxStages < kMailSlots, "see above");
__device__ __forceinline__ void mail_put(uint64_t* mail, int n, float value) {
    const uint64_t v = ((uint64_t)(uint32_t)(n + 1) << 32) | (uint64_t)__float_as_uint(value);
    asm volatile("st.volatile.shared.b64 [%0], %1;" ::"r"(dev::smem_addr(mail + (n & (kMailSlots - 1)))), "l"(v) : "memory");
}
// (a wait that gives up raises the workspace's error word: what is formed from the value it returns is not to be used)
static __device__ __noinline__ float mail_wait(uint32_t at, uint32_t tag, int* abort_flag, unsigned int* error_word) {
    uint64_t v = 0;
    for (unsigned int tries = 0; tries < (1u << 24); ++tries) {
        asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(v) : "r"(at) : "memory");
        if ((uint32_t)(v >> 32) == tag) return __uint_as_float((uint32_t)v);
        if (*reinterpret_cast<volatile int*>(abort_flag)) return 0.0f;
    }
    *reinterpret_cast<volatile int*>(abort_flag) = 1;
    atomicExch(error_word, 1u);
    return 0.0f;
}
__device__ __forceinline__ float mail_get(const uint64_t* mail, int n, int* abort_flag, unsigned int* error_word) {
    const uint32_t at = dev::smem_addr(mail + (n & (kMailSlots - 1)));
    uint64_t v;
    asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(v) : "r"(at) : "memory");
    const bool here = (uint32_t)(v >> 32) == (uint32_t)(n + 1);
    return __all_sync(0xffffffffu, here) ? __uint_as_float((uint32_t)v) : mail_wait(at, (uint32_t)(n + 1), abort_flag, error_word);
}

// Sends rows [lo, hi) of a warp's share [wrow, wrow + ntw) of a tile (`slab` and `out` point at the tile's first row in
// shared and in global memory).  Out of line: it serves the ends of a block's range and row pitches that do not keep a
// warp's rows on 16-byte boundaries.
static __device__ __noinline__ void send_rows_general(unsigned char* out, const unsigned char* slab, int pitch, int wrow,
                                                      int ntw, int lo, int hi, bool wrote) {
    lo = max(lo, wrow);
    hi = min(hi, wrow + ntw);
    const uint32_t bytes = hi > lo ? (uint32_t)(hi - lo) * (uint32_t)pitch : 0u;
    dev::warp_send_bytes(out + (long long)lo * pitch, slab + lo * pitch, bytes, wrote);
}

// How the rows of a batch are laid on lanes: rows of a tile, lanes per row, rotation of a lane's vectors.
struct RowLayout {
    int nt = 128, log_lanes = 0, passes = 1, rot_shift = 0, rot_mask = 0;
};

// Long trajectories go to neighbouring blocks where blocks that own whole ones would leave most of the device idle: the
// busiest of them has ceil(B / blocks) trajectories (and where the caller's scratch has room for the tiles' aggregates).
// A split launch pays for its exchange with up to half of a flat one's rate.  Measured in us, flat against split, by the
// share of the device that the flat launch keeps busy:
//   rows of one lane: 0.21 (A = 18, 31 x 4000) 16.3 / 14.6; 0.30 (18, 45 x 1000) 7.5 / 7.3; 0.40 (18, 59 x 4000) 17.1 /
//   25.6; 0.43 (20, 64 x 1000) 9.4 / 11.1; 0.47 (7, 69 x 4000) 18.2 / 23.6; 0.70 (18, 104 x 4000) 19.9 / 40.2
//   A trajectory of up to three tiles is done before the exchange would be: (18, 16 x 200) 3.8 / 4.8, (18, 44 x 256) 3.9 / 5.1,
//   (18, 16 x 300) 4.5 / 5.1, in bf16 4.4 / 5.0, 17 dimensions 4.9 / 5.7; of four either: (18, 4 x 400) 4.8 / 5.0, with every
//   switch 5.4 / 5.0; of five (18, 16 x 600) 5.8 / 4.8.  With every switch (not `plain`) one or two trajectories of three tiles are
//   split: (18, 1 x 300) 5.0 / 4.7, (18, 2 x 384) 5.0 / 4.8, (32, 1 x 300) 5.6 / 5.4, (6, 1 x 300) 4.2 / 4.2, 17 dimensions 5.7 / 5.3; but
//   (18, 4 x 300) 4.4 / 4.9, (6, 4 x 384) 3.6 / 4.3
//   rows of several lanes (`wide_row` elements, else 0) in tiles of nt rows, 128 / lanes, each of which takes a group some 0.65
//   us whatever the width: a flat launch takes as long as the busiest block's tiles, a split one twice its tiles per SM
//   (`slope` tenths) and 2.5 tiles more (`cost`): (64, 16 x 300) 6.6 / 5.6, (64, 32 x 300) 6.9 / 6.2, (64, 50 x 300) 7.5 / 7.8; with every
//   switch (60, 20 x 300) 9.1 / 6.4, (60, 38 x 500) 12.1 / 9.1; (40, 20 x 200) 5.1 / 5.1, (40, 40 x 200) 5.4 / 5.7; (60, 50 x 500) 10.3 /
//   8.4, in bf16 8.6 / 7.6; (64, 54 x 1000) 16.0 / 11.2, (64, 58 x 1000) 16.2 / 15.5, inputs in L2 13.6 / 14.4; (64, 62 x 2000) 29.2 /
//   26.1; (64, 66 x 4000) 54.3 / 48.8; (100, 40 x 100) 6.3 / 6.2; (100, 58 x 1000) 27.2 / 20.8; (180, 50 x 100) 7.3 / 7.6; (400, 40 x 50)
//   8.0 / 7.9; (64, 160 x 100) 6.0 / 7.7
inline long long split_tiles(const BatchGeometry& g, int nt) { return g.B * ((g.T + nt - 1) / nt); }
inline bool splits_trajectories(const BatchGeometry& g, bool aggregates, int nt, const DeviceInfo* di, int wide_row, int slope = 20,
                                int cost = 25, bool plain = true) {
    if (g.T <= nt || !aggregates) return false;
    const long long rounds = (g.B + di->sm_count - 1) / di->sm_count;
    if (wide_row) return 10 * ((rounds * g.T + nt - 1) / nt) * di->sm_count > slope * split_tiles(g, nt) + cost * di->sm_count;
    return g.T > (plain || g.B > 2 ? 3ll : 2ll) * nt && 100 * g.B < 30 * rounds * di->sm_count;
}
// Flat launches count a trajectory's steps in 32 bits, but for the form of the fewest actions with every switch compiled in.
inline bool fits_flat(const BatchGeometry& g) { return g.T < (1ll << 32) - 4096; }

// Where a warp's accesses of `access_bytes`, `group` neighbouring lanes to a row and the rows `stride` bytes apart, fall
// on the banks: `ways` accesses meet, and rows 2^shift apart are the first that do.
struct BankPattern {
    int ways, shift;
};
inline BankPattern bank_pattern(size_t stride, int group, int access_bytes) {
    const size_t window = (size_t)group * access_bytes;
    const size_t rows_at_once = 128 / window > 1 ? 128 / window : 1;
    size_t step = stride % 128;  // gcd(stride, 128)
    step = step ? (step & (~step + 1)) : 128;
    BankPattern b = {1, 0};
    for (size_t d = 128 / step; d > 1; d /= 2) ++b.shift;
    if (rows_at_once > 1 && step > window) b.ways = (int)(step / window);
    return b;
}

// The grid of a launch, its tiles, and the ring that streams them.  False: no valid shape.
struct LaunchShape {
    long long grid, tiles, tiles_per_block;
    int stages, in_flight, lanes;
};
inline bool launch_shape(BatchGeometry& g, int nt, bool is_long, size_t stage_bytes, size_t tile_in_bytes, int groups,
                         const DeviceInfo* di, LaunchShape* out, bool cold = false) {
    g.nt = nt;
    g.ntiles = is_long ? (int)((g.T + nt - 1) / nt) : 1;
    if (is_long) {
        out->tiles = g.B * g.ntiles;
        out->grid = out->tiles < di->sm_count ? out->tiles : di->sm_count;
        out->tiles_per_block = (out->tiles + out->grid - 1) / out->grid;
    } else {
        // a block per tile's worth of whole trajectories, or per trajectory, up to one per SM
        const long long per_tile = g.T < nt ? nt / g.T : 1;
        out->grid = (g.B + per_tile - 1) / per_tile;
        if (out->grid > di->sm_count) out->grid = di->sm_count;
        const long long trajs = (g.B + out->grid - 1) / out->grid;
        out->tiles_per_block = (trajs * g.T + nt - 1) / nt;
        out->tiles = out->tiles_per_block * out->grid;
    }
    if (out->grid > kMaxTaggedRows) return false;  // one tagged row per block
    // tile-major once every block has a trajectory of its own: the aggregates a tile needs are then a round old
    g.tile_major = (is_long && g.B >= out->grid) ? 1 : 0;
    ws_ring_shape(stage_bytes, tile_in_bytes, groups, di->max_smem_optin, out->tiles_per_block, &out->stages, &out->in_flight,
                  cold);
    if (out->stages < 1 || out->in_flight < 1) return false;
    const int spare = out->stages - out->in_flight;  // producer lanes that request tiles side by side
    out->lanes = spare < 4 ? (spare < 1 ? 1 : spare) : 4;
    return true;
}

}  // namespace impact
