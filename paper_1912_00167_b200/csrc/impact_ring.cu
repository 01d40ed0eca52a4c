// Circular buffer C(N, K) of device-resident train batches (Algorithm 1; Section 3.2), and
// the byte-exact copy / gather kernels behind it.
//
// Slot bookkeeping is a few integers per slot and lives on the host, where the learner loop
// that calls push / sample runs; the payload never leaves HBM.  A sample is normally
// zero-copy (the loss kernel reads the slot in place); the fused copy kernel serves pushes
// from device memory and the optional gather into caller buffers.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <vector>

#include "impact.h"
#include "impact_device.cuh"
#include "impact_internal.h"
#include "impact_pinned.h"
#include "impact_ring_copy.cuh"

namespace impact {
namespace {

constexpr int kMaxFields = 16;
constexpr size_t kFieldAlign = 256;

struct CopySegments {
    const char* src[kMaxFields];
    char* dst[kMaxFields];
    unsigned long long bytes[kMaxFields];
    unsigned long long vec_end[kMaxFields];  // running count of 16-byte units up to and including segment f
    int n;
};

// Copies up to kMaxFields byte ranges in one launch.  Every range is walked in 16-byte
// units; the last unit of a range whose length is not a multiple of 16 is copied bytewise.
// kHost: the sources are pinned host memory, read anew (never from what a cache kept of an earlier batch).
template <bool kHost>
__device__ __forceinline__ void copy_segments(const CopySegments& s) {
    const unsigned long long total = s.vec_end[s.n - 1];
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    unsigned long long v = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    constexpr int U = 4;
    while (v < total) {
        uint4 x[U];
        char* out[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned long long vu = v + u * stride;
            out[u] = nullptr;
            if (vu < total) {
                int f = 0;
                while (vu >= s.vec_end[f]) ++f;
                const unsigned long long off = (vu - (f ? s.vec_end[f - 1] : 0ull)) * 16ull;
                out[u] = s.dst[f] + off;
                if (off + 16ull <= s.bytes[f]) {
                    const uint4* const from = reinterpret_cast<const uint4*>(s.src[f] + off);
                    x[u] = kHost ? __ldcv(from) : __ldcs(from);
                } else {
                    const int tail = (int)(s.bytes[f] - off);
                    for (int i = 0; i < tail; ++i) out[u][i] = kHost ? __ldcv(s.src[f] + off + i) : s.src[f][off + i];
                    out[u] = nullptr;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (out[u]) __stcs(reinterpret_cast<uint4*>(out[u]), x[u]);
        v += U * stride;
    }
}
template <bool kHost>
__global__ void __launch_bounds__(256) multi_copy_kernel(const __grid_constant__ CopySegments s) {
    grid_dependency_wait();
    copy_segments<kHost>(s);
}

// dst[i, :] = src[idx[i], :], rows of `units` elements of type V, at least 16 bytes, and a destination on a 16-byte boundary.
//
// The destination is walked flat in granules of 16 bytes, a grid's width at a time, so that every lane has one whatever the
// row's width.  A granule is put together from elements of one row or, where a row ends inside it, of two; both rows'
// indices are asked for side by side.  A thread's row and place in it are carried along: from one of its granules to the
// next the row advances by stride_rows and the place by stride_rest; the one division is done while the kernel before this
// one drains.  Bound by HBM from 64-byte rows on (a granule at a time keeps 2048 threads' loads under way on every SM; two
// where granules are single loads, four are slower).  40 MB in rows of 17, 36, 132, 200, 1800 and 4096 bytes take 66, 21.4,
// 16.9, 16.1, 15.1 and 14.5 us, 4.2 MB in rows of 200 and 204 bytes 3.5 and 3.6; element by element (below) 72, 24.2, 22.1,
// 17.0, 16.5, 14.9, 4.5 and 5.7.
template <typename V, int U>
__global__ void __launch_bounds__(256, 8) gather_granules_kernel(const V* __restrict__ src, const int32_t* __restrict__ idx,
                                                                 unsigned int n, int n_src_rows, unsigned int units,
                                                                 unsigned int stride_rows, unsigned int stride_rest,
                                                                 V* __restrict__ dst) {
    constexpr int N = 16 / (int)sizeof(V);  // elements of a granule
    union Granule {
        uint4 all;
        V part[N];
    };
    const unsigned long long total = (unsigned long long)n * units;  // elements
    const unsigned long long granules = total / N;
    const unsigned int stride = gridDim.x * blockDim.x;
    unsigned long long v = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned int i = (unsigned int)(v * N / units), c = (unsigned int)(v * N - (unsigned long long)i * units);
    grid_dependency_wait();
    auto row_at = [&](unsigned int k) {
        const int r = __ldg(idx + k);
        return src + (unsigned long long)(unsigned int)min(max(r, 0), n_src_rows - 1) * units;
    };
    for (; v < granules; v += (unsigned long long)U * stride) {
        const V *first[U], *second[U];
        unsigned int left[U];  // elements of the granule that its first row still has
#pragma unroll
        for (int u = 0; u < U; ++u) {
            left[u] = units - c;
            first[u] = second[u] = src;
            if (v + (unsigned long long)u * stride < granules) {
                first[u] = row_at(i) + c;
                // (asked for in any case, the same index where the row goes on: no branch that waits for the first)
                if constexpr (N > 1) second[u] = row_at(left[u] < N ? i + 1 : i) - left[u];
            }
            i += stride_rows;
            c += stride_rest;
            if (c >= units) { c -= units; ++i; }
        }
        Granule x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (v + (unsigned long long)u * stride < granules) {
#pragma unroll
                for (int e = 0; e < N; ++e) x[u].part[e] = __ldg((e < (int)left[u] ? first[u] : second[u]) + e);
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (v + (unsigned long long)u * stride < granules)
                reinterpret_cast<uint4*>(dst)[v + (unsigned long long)u * stride] = x[u].all;
    }
    // what is left of the last granule (by threads that had none, in a grid of one round)
    const unsigned long long free_thread = blockIdx.x * blockDim.x + threadIdx.x - (granules + 16 <= stride ? granules : 0);
    if (free_thread < total - granules * N) {
        const unsigned long long at = granules * N + free_thread;
        const unsigned int k = (unsigned int)(at / units);
        dst[at] = __ldg(row_at(k) + (at - (unsigned long long)k * units));
    }
}

// The same element by element, for rows narrower than a granule, of which one would hold several, and destinations that lie
// on a smaller boundary; two elements of 8 bytes and more of a thread are under way, one of the narrower ones.  40 MB in rows
// of 12 bytes take 28.7 us.
template <typename V, int U>
__global__ void __launch_bounds__(256) gather_rows_kernel(const V* __restrict__ src, const int32_t* __restrict__ idx,
                                                          long long n, long long n_src_rows, long long units,
                                                          long long stride_rows, long long stride_rest,
                                                          V* __restrict__ dst) {
    grid_dependency_wait();
    const long long total = n * units, stride = (long long)gridDim.x * blockDim.x;
    long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long i = v / units, c = v - i * units;
    for (; v < total; v += U * stride) {
        long long from[U], at[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            from[u] = v + u * stride < total ? (long long)idx[i] : 0;
            at[u] = c;
            i += stride_rows;
            c += stride_rest;
            if (c >= units) { c -= units; ++i; }
        }
        V x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long r = from[u] < 0 ? 0 : (from[u] >= n_src_rows ? n_src_rows - 1 : from[u]);
            if (v + u * stride < total) x[u] = src[r * units + at[u]];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (v + u * stride < total) dst[v + u * stride] = x[u];
    }
}

// Reads `n_read` 16-byte units and writes `n_write` of them back out (n_write <= n_read): a loss launch's byte mix
// with no arithmetic in between.  What is read but not written is folded into one word per thread that is stored
// only if it has an impossible value, so that the loads cannot be dropped.
__global__ void __launch_bounds__(256) stream_copy_kernel(const uint4* __restrict__ src, unsigned long long n_read,
                                                          uint4* __restrict__ dst, unsigned long long n_write,
                                                          unsigned int* __restrict__ sink) {
    grid_dependency_wait();
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    unsigned int fold = 0;
    constexpr int U = 4;
    for (unsigned long long v = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; v < n_read; v += U * stride) {
        uint4 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            x[u] = (v + u * stride < n_read) ? __ldcs(src + v + u * stride) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (v + u * stride < n_write) dst[v + u * stride] = x[u];
            else fold |= x[u].x ^ x[u].y ^ x[u].z ^ x[u].w;
        }
    }
    if (fold == 0xFFFFFFFFu && n_read == 1) *sink = fold;  // (never: keeps the unwritten loads alive)
}

// ---- bookkeeping resident on the device ---------------------------------------------------------------------
// The same few integers per slot as on the host, in device memory, so that a learner iteration -- push a worker
// batch into a free slot, obtain a batch, loss and gradients -- can be enqueued (or captured into a CUDA graph)
// without the host ever seeing a slot number.  One warp does the bookkeeping; it is the protocol of
// impact_buffer_push / impact_buffer_sample statement by statement (docs/ring_protocol.md), so both modes give the
// same trace for the same seed.
struct RingDeviceHeader {
    int32_t write_cursor, read_cursor;
    uint32_t n_events, steps;  // steps: launches so far
    uint64_t draws, pushes;
};
static_assert(sizeof(RingDeviceHeader) == 32, "read as two 16-byte words");
constexpr int kEventLog = 4096;  // the most recent push / sample outcomes, for the host to read back
constexpr int kMaxDeviceSlots = 1024;  // slots a buffer may have for its bookkeeping to go to the device

// What every block of a step reads, in two copies of which a launch reads one and writes the other: the launch's number, odd
// or even, says which.  `tickets` goes up by 2^kTicketBits with every launch, whatever its grid, and by less with each of its
// blocks but the one that makes up for them: what it held when a block drew its ticket, shifted, is the launch's number.
struct RingDeviceState {
    RingDeviceHeader hd;
    uint32_t live[kMaxDeviceSlots / 32];  // the slots that hold a batch
};
constexpr int kTicketBits = 16;
struct RingDeviceShared {
    uint32_t tickets, failed, pad[2];  // failed: see copy_by_warp
    RingDeviceState state[2];
    // As the last launch that is complete left it, for the host.  (`tickets` goes up at a launch's start, the copy that it
    // writes is there at its end.)
    const RingDeviceState& current() const { return state[(int32_t)(state[1].hd.steps - state[0].hd.steps) > 0 ? 1 : 0]; }
};

struct RingDeviceView {
    RingDeviceShared* shared;
    int32_t* count;    // per slot: traversals; read and written by one block
    uint64_t* fresh;   // per slot: the extra pointer that came with the batch pushed into it
    int4* events;      // (op, status, slot, k_before); op 1 = push, 2 = sample
    char* storage;
    unsigned long long slot_stride;
    unsigned long long field_offset[kMaxFields], field_bytes[kMaxFields];
    int32_t N, K, n_fields, mode;
    uint64_t seed;
};

__device__ __forceinline__ uint64_t splitmix64_at_dev(uint64_t seed, uint64_t n) {
    uint64_t z = seed + (n + 1) * 0x9E3779B97F4A7C15ull;
    z ^= z >> 30; z *= 0xBF58476D1CE4E5B9ull;
    z ^= z >> 27; z *= 0x94D049BB133111EBull;
    z ^= z >> 31;
    return z;
}

// Bits of a set of at most kMaxDeviceSlots slots, word w with lane w of a warp: the first member at or after `from`
// in circular order (-1 = the set is empty).  Called by a whole warp.
__device__ __forceinline__ int32_t first_at_or_after(uint32_t word, int32_t from) {
    const int lane = threadIdx.x & 31, fw = from >> 5;
    const uint32_t later = lane < fw ? 0u : (lane == fw ? word & (0xFFFFFFFFu << (from & 31)) : word);
    const uint32_t none = 0xFFFFFFFFu;
    uint32_t at = __reduce_min_sync(0xFFFFFFFFu, later ? (uint32_t)(lane * 32 + __ffs((int)later) - 1) : none);
    if (at == none) at = __reduce_min_sync(0xFFFFFFFFu, word ? (uint32_t)(lane * 32 + __ffs((int)word) - 1) : none);
    return (int32_t)at;
}
// The j-th member (0-based) of the same set, which has more than j.
__device__ __forceinline__ int32_t nth_member(uint32_t word, uint32_t j) {
    const int lane = threadIdx.x & 31;
    uint32_t upto = (uint32_t)__popc(word);  // members in words 0 .. lane
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t below = __shfl_up_sync(0xFFFFFFFFu, upto, off);
        if (lane >= off) upto += below;
    }
    const int owner = __ffs((int)__ballot_sync(0xFFFFFFFFu, upto > j)) - 1;
    int32_t at = 0;
    if (lane == owner) {
        uint32_t rest = j - (upto - (uint32_t)__popc(word));
        uint32_t w = word;
        while (rest--) w &= w - 1;
        at = lane * 32 + __ffs((int)w) - 1;
    }
    return __shfl_sync(0xFFFFFFFFu, at, owner);
}

// One learner-side step of the bookkeeping: (1) if `sources` is given, the next candidate batch is copied into the
// first free slot at or after the write cursor (none free: nothing happens, the event says FULL); (2) a live slot is
// drawn and the inputs of the loss call are resolved into `inputs`.
//
// One launch does both.  Every block reads the state for itself (past L1: an earlier launch may have left an older version
// there) and works out the push's slot; the first block also works out the draw and writes the new state, over the copy that
// no block of this launch takes anything from, so no block waits for another.  The launch is a chain of latencies: its start,
// one trip to L2, its end.  So everything that it may need is asked for at once, where there is not too much of it: the
// candidates' pointers and what is kept with each slot.  (An iteration of 131 072 steps of 18 actions, K = 4, step and loss
// 12.0 us -> 11.0, of 1 600 steps 7.1 -> 6.2, of 16 384 steps of 9 with a push in each 8.4 -> 7.3; before, every block read all
// of the state and the one that drew the last ticket wrote it, in blocks of 512 threads.  Rings and tables of which there is too
// much take another trip: a step that pushes nothing on 128, 129, 512, 1024 slots 2.6, 2.7, 2.9, 2.9 us, then 3.3, 3.3, 3.4, 3.7;
// 126, 132, 510 pointers 2.6, 2.7, 2.7, then 3.4.  L2 asked for the drawn slot's fields from here: a grid is complete only when its requests are, 0.3 to 1 us more.)
//
// kThreads = 32: a warp per block and 16 KB of shared memory, so that the blocks become resident beside those of the loss
// launch before, and the loss launch behind beside them, where that leaves them kRingStepShared: neither's start adds to the
// chain then.  (It does but for 18 actions in fp32 in the default configuration, whose 12 stages take 217 KB of an SM.)  The copy
// goes through shared memory, which keeps 16 KB under way with a warp's registers; batches of more than 32 KB to a block, the
// 131 072 steps above among them, go to blocks of 512 threads (kStepThreads), which find no registers beside a loss launch's.
// (The next launch is let in behind the wait: before it, 0.1 to 0.4 us more.  The warp's copy through
// registers or by a loop over the segments: up to 1.2 us more where every step pushes.)
constexpr int kStepThreads = 512;
constexpr int kAheadSlots = 128;       // slots and candidates' pointers that are asked for before it is known which are needed
constexpr int kMostSmallUnits = 2048;  // of a block's part of a batch

template <int kThreads>
__global__ void __launch_bounds__(kThreads) ring_step_kernel(const __grid_constant__ RingDeviceView v, const impact_ring_field_map map,
                                                             const void* learner_logits, const float* values,
                                                             const float* bootstrap_values, const void* const* sources,
                                                             int32_t n_candidates, int32_t do_sample,
                                                             impact_loss_inputs* inputs) {
    constexpr bool kSmall = kThreads == 32;
    __shared__ __align__(8) uint64_t bar_s;
    if (kSmall && threadIdx.x == 0) {
        dev::mbarrier_init_nofence(&bar_s, 1);
        dev::fence_mbarrier_init();
    }
    grid_dependency_wait();
    __shared__ int32_t count_s[kAheadSlots];
    __shared__ unsigned long long fresh_s[kAheadSlots];
    __shared__ unsigned long long cand_s[kAheadSlots];
    __shared__ CopySegments plan_s;
    __shared__ __align__(16) uint4 buffer_s[kSmall ? kStepUnits : 1];
    const int tid = threadIdx.x, lane = tid & 31;
    const char* src = nullptr;  // of the lane's segment
    char* dst = nullptr;
    unsigned long long bytes = 0, seg_end = 0, units = 0;
    if (tid < 32) {
        const int width = v.n_fields + 1;  // pointers of a candidate
        const bool all_candidates = sources && (long long)n_candidates * width <= kAheadSlots, all_slots = v.N <= kAheadSlots;
        const bool writes = blockIdx.x == 0;
        unsigned int ticket = 0;
        if (lane == 0)
            asm volatile("atom.add.relaxed.gpu.global.u32 %0, [%1], %2;" : "=r"(ticket)
                         : "l"(&v.shared->tickets), "r"(writes ? (1u << kTicketBits) - (gridDim.x - 1u) : 1u) : "memory");
        // (both copies; the headers by every thread: one request)
        const uint4 *const q0 = reinterpret_cast<const uint4*>(&v.shared->state[0].hd), *const q1 = reinterpret_cast<const uint4*>(&v.shared->state[1].hd);
        const uint4 a0 = __ldcg(q0), b0 = __ldcg(q0 + 1), a1 = __ldcg(q1), b1 = __ldcg(q1 + 1);
        const uint32_t live0 = __ldcg(v.shared->state[0].live + lane), live1 = __ldcg(v.shared->state[1].live + lane);
        unsigned long long cand[kAheadSlots / 32], fresh[kAheadSlots / 32];
        int32_t count[kAheadSlots / 32];
#pragma unroll
        for (int i = 0; i < kAheadSlots / 32; ++i) {
            const int at = i * 32 + lane;
            cand[i] = all_candidates && at < n_candidates * width ? __ldcg(reinterpret_cast<const unsigned long long*>(sources) + at) : 0ull;
            const bool slot_there = writes && all_slots && at < v.N;
            count[i] = slot_there ? __ldcg(v.count + at) : 0;
            fresh[i] = slot_there ? __ldcg(reinterpret_cast<const unsigned long long*>(v.fresh) + at) : 0ull;
        }
#pragma unroll
        for (int i = 0; i < kAheadSlots / 32; ++i) {
            cand_s[i * 32 + lane] = cand[i];
            count_s[i * 32 + lane] = count[i];
            fresh_s[i * 32 + lane] = fresh[i];
        }
        const bool odd = ((__shfl_sync(0xFFFFFFFFu, ticket, 0) >> kTicketBits) & 1u) != 0u;
        const uint4 h0 = odd ? a1 : a0, h1 = odd ? b1 : b0;
        RingDeviceHeader hd;
        hd.write_cursor = (int32_t)h0.x; hd.read_cursor = (int32_t)h0.y; hd.n_events = h0.z; hd.steps = h0.w + 1u;
        hd.draws = ((uint64_t)h1.y << 32) | h1.x; hd.pushes = ((uint64_t)h1.w << 32) | h1.z;
        uint32_t live = odd ? live1 : live0;
        __syncwarp();
        const int32_t left = v.N - 32 * lane;  // slots that exist in this lane's word
        const uint32_t exist = left >= 32 ? 0xFFFFFFFFu : (left > 0 ? (1u << left) - 1u : 0u);
        int32_t slot = -1;
        int first_cand = 0;  // of the candidate's pointers in cand_s
        if (sources) slot = first_at_or_after(~live & exist, hd.write_cursor);
        if (slot >= 0) {
            const uint64_t c = hd.pushes % (uint64_t)n_candidates;
            if (all_candidates) first_cand = (int)c * width;
            else if (lane < width) cand_s[lane] = __ldcg(reinterpret_cast<const unsigned long long*>(sources) + c * (uint64_t)width + lane);
            __syncwarp();
            if (lane == (slot >> 5)) live |= 1u << (slot & 31);
        }
        if (slot >= 0) {
            const bool mine = lane < v.n_fields;
            src = mine ? reinterpret_cast<const char*>(cand_s[first_cand + lane]) : nullptr;
            bytes = src ? v.field_bytes[lane] : 0ull;
            dst = mine ? v.storage + (unsigned long long)slot * v.slot_stride + v.field_offset[lane] : nullptr;
            seg_end = (bytes + 15ull) / 16ull;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned long long below = __shfl_up_sync(0xFFFFFFFFu, seg_end, off);
                if (lane >= off) seg_end += below;
            }
            units = __shfl_sync(0xFFFFFFFFu, seg_end, 31);
            if (!kSmall && mine) {
                plan_s.src[lane] = src;
                plan_s.dst[lane] = dst;
                plan_s.bytes[lane] = bytes;
                plan_s.vec_end[lane] = seg_end;
            }
        }
        if (!kSmall && lane == 0) plan_s.n = units ? v.n_fields : 0;
        if (writes) {
            int32_t pick = -1;
            const uint32_t n_live = (uint32_t)__reduce_add_sync(0xFFFFFFFFu, (unsigned)__popc(live));
            if (do_sample && n_live > 0)
                pick = v.mode == IMPACT_SAMPLE_UNIFORM  // floor(u * live / 2^64)
                           ? nth_member(live, (uint32_t)__umul64hi(splitmix64_at_dev(v.seed, hd.draws), (uint64_t)n_live))
                           : first_at_or_after(live, hd.read_cursor);
            const unsigned long long pushed_fresh = slot >= 0 ? cand_s[first_cand + v.n_fields] : 0ull;
            if (sources) {
                if (slot >= 0) {
                    if (lane == 0) {
                        v.fresh[slot] = pushed_fresh;
                        v.count[slot] = 0;
                    }
                    hd.write_cursor = (slot + 1) % v.N;
                    hd.pushes += 1;
                }
                if (lane == 0) v.events[hd.n_events % kEventLog] = make_int4(1, slot >= 0 ? IMPACT_OK : IMPACT_ERR_FULL, slot, 0);
                hd.n_events += 1;
            }
            if (do_sample) {
                int32_t k_before = 0;
                unsigned long long kept = 0;
                if (pick >= 0) {
                    if (pick == slot) {  // (drawn as it is pushed)
                        kept = pushed_fresh;
                    } else {
                        k_before = all_slots ? count_s[pick] : __ldcg(v.count + pick);
                        kept = all_slots ? fresh_s[pick] : __ldcg(reinterpret_cast<const unsigned long long*>(v.fresh) + pick);
                    }
                    if (v.mode == IMPACT_SAMPLE_UNIFORM) hd.draws += 1;
                    else hd.read_cursor = (pick + 1) % v.N;
                    if (k_before + 1 >= v.K && lane == (pick >> 5)) live &= ~(1u << (pick & 31));
                }
                if (lane == 0) {
                    if (pick >= 0) {
                        v.count[pick] = k_before + 1;
                        const void* const fresh_at = reinterpret_cast<const void*>(kept);
                        auto field = [&](int32_t f) -> const void* {
                            return f >= 0 ? v.storage + (unsigned long long)pick * v.slot_stride + v.field_offset[f] : nullptr;
                        };
                        impact_loss_inputs in;
                        in.learner_logits = learner_logits;
                        in.values = values;
                        in.bootstrap_values = bootstrap_values;
                        in.actions = static_cast<const int32_t*>(field(map.actions));
                        in.rewards = static_cast<const float*>(field(map.rewards));
                        in.discounts = static_cast<const float*>(field(map.discounts));
                        in.worker_logp = static_cast<const float*>(field(map.worker_logp));
                        const void* in_slot = field(map.target_logits);
                        if (k_before == 0 && fresh_at && in_slot) {  // first traversal: the target network's output is appended now
                            in.target_logits = fresh_at;
                            in.target_logits_copy = const_cast<void*>(in_slot);
                        } else {
                            in.target_logits = in_slot;
                            in.target_logits_copy = nullptr;
                        }
                        in.status = IMPACT_OK;
                        in.slot = pick;
                        in.k_before = k_before;
                        in.pad = 0;
                        *inputs = in;
                    } else {
                        inputs->status = IMPACT_ERR_EMPTY;  // the pointers of the previous draw stay in place
                    }
                    v.events[hd.n_events % kEventLog] = make_int4(2, pick >= 0 ? IMPACT_OK : IMPACT_ERR_EMPTY, pick, k_before);
                }
                hd.n_events += 1;
            }
            RingDeviceState* const next = &v.shared->state[odd ? 0 : 1];
            next->live[lane] = live;
            if (lane == 0) next->hd = hd;
        }
    }
    if constexpr (kSmall) {
        if (units != 0 &&
            !copy_by_warp(src, dst, bytes, seg_end - (bytes + 15ull) / 16ull, units * blockIdx.x / gridDim.x,
                          units * (blockIdx.x + 1ull) / gridDim.x, buffer_s, &bar_s, kCopyTries) && lane == 0)
            atomicExch(&v.shared->failed, 1u);
    } else {
        __syncthreads();
        if (plan_s.n > 0) copy_segments<false>(plan_s);
    }
}

int blocks_for(unsigned long long work_items, int per_worker, const DeviceInfo* di, int workers = 256) {
    const unsigned long long per_block = (unsigned long long)workers * per_worker;
    unsigned long long blocks = (work_items + per_block - 1) / per_block;
    const unsigned long long cap = (unsigned long long)di->sm_count * 8ull;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

// n-th output of SplitMix64 (Steele, Lea, Flood 2014) for the stream that starts at `seed`:
// the additive state after n+1 steps, passed through the two multiply-xorshift rounds.
uint64_t splitmix64_at(uint64_t seed, uint64_t n) {
    uint64_t z = seed + (n + 1) * 0x9E3779B97F4A7C15ull;
    z ^= z >> 30; z *= 0xBF58476D1CE4E5B9ull;
    z ^= z >> 27; z *= 0x94D049BB133111EBull;
    z ^= z >> 31;
    return z;
}

struct StateHeader {
    uint32_t magic, version;
    int32_t N, K, n_fields, mode;
    int32_t write_cursor, read_cursor;
    uint64_t seed, draws;
};
constexpr uint32_t kStateMagic = 0x494D5043u;  // "IMPC"

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace
}  // namespace impact

using namespace impact;

struct impact_buffer {
    int32_t N = 0, K = 0, n_fields = 0, mode = 0;
    uint64_t seed = 0, draws = 0;
    int32_t write_cursor = 0, read_cursor = 0;
    std::vector<int32_t> valid, count;
    size_t field_bytes[kMaxFields] = {};
    size_t field_offset[kMaxFields] = {};
    size_t slot_stride = 0;
    char* storage = nullptr;
    bool owns_storage = false;
    // bookkeeping on the device (impact_buffer_device_begin): one allocation, laid out as
    // [RingDeviceShared | count N | fresh N | events]
    char* device_state = nullptr;
    bool device_mode = false;
    size_t device_state_bytes() const {
        return align_up16(sizeof(RingDeviceShared)) + align_up16(sizeof(int32_t) * (size_t)N) +
               align_up16(sizeof(uint64_t) * (size_t)N) + sizeof(int4) * (size_t)kEventLog;
    }
    static size_t align_up16(size_t x) { return (x + 15) / 16 * 16; }
    RingDeviceView view() const {
        RingDeviceView v;
        char* p = device_state;
        v.shared = reinterpret_cast<RingDeviceShared*>(p); p += align_up16(sizeof(RingDeviceShared));
        v.count = reinterpret_cast<int32_t*>(p); p += align_up16(sizeof(int32_t) * (size_t)N);
        v.fresh = reinterpret_cast<uint64_t*>(p); p += align_up16(sizeof(uint64_t) * (size_t)N);
        v.events = reinterpret_cast<int4*>(p);
        v.storage = storage;
        v.slot_stride = slot_stride;
        for (int f = 0; f < kMaxFields; ++f) { v.field_offset[f] = field_offset[f]; v.field_bytes[f] = field_bytes[f]; }
        v.N = N; v.K = K; v.n_fields = n_fields; v.mode = mode;
        v.seed = seed;
        return v;
    }

    char* field_ptr(int32_t slot, int32_t f) const {
        return storage + (size_t)slot * slot_stride + field_offset[f];
    }
};

static bool valid_fields(int32_t n_fields, const size_t* field_bytes) {
    if (n_fields < 1 || n_fields > kMaxFields || !field_bytes) return false;
    for (int f = 0; f < n_fields; ++f)
        if (field_bytes[f] == 0) return false;
    return true;
}

extern "C" size_t impact_buffer_storage_bytes(int32_t N, int32_t n_fields, const size_t* field_bytes) {
    if (N < 1 || !valid_fields(n_fields, field_bytes)) return 0;
    size_t stride = 0;
    for (int f = 0; f < n_fields; ++f) stride += align_up(field_bytes[f], kFieldAlign);
    return stride * (size_t)N;
}

extern "C" int32_t impact_buffer_create(int32_t N, int32_t K, int32_t n_fields, const size_t* field_bytes,
                                        uint64_t seed, int32_t sample_mode, void* storage,
                                        impact_buffer** out) {
    if (!out || N < 1 || K < 1 || !valid_fields(n_fields, field_bytes)) return IMPACT_ERR_INVALID_ARG;
    if (sample_mode != IMPACT_SAMPLE_UNIFORM && sample_mode != IMPACT_SAMPLE_ROUND_ROBIN)
        return IMPACT_ERR_INVALID_ARG;
    if (storage && (reinterpret_cast<uintptr_t>(storage) % kFieldAlign) != 0) return IMPACT_ERR_INVALID_ARG;
    impact_buffer* h = new (std::nothrow) impact_buffer();
    if (!h) return IMPACT_ERR_INVALID_ARG;
    h->N = N; h->K = K; h->n_fields = n_fields; h->mode = sample_mode; h->seed = seed;
    h->valid.assign((size_t)N, 0);
    h->count.assign((size_t)N, 0);
    size_t off = 0;
    for (int f = 0; f < n_fields; ++f) {
        h->field_bytes[f] = field_bytes[f];
        h->field_offset[f] = off;
        off += align_up(field_bytes[f], kFieldAlign);
    }
    h->slot_stride = off;
    if (storage) {
        h->storage = static_cast<char*>(storage);
    } else {
        void* mem = nullptr;
        cudaError_t e = cudaMalloc(&mem, off * (size_t)N);
        if (e != cudaSuccess) { delete h; return record_cuda_error(e); }
        h->storage = static_cast<char*>(mem);
        h->owns_storage = true;
    }
    *out = h;
    return IMPACT_OK;
}

extern "C" int32_t impact_buffer_destroy(impact_buffer* h) {
    if (!h) return IMPACT_ERR_INVALID_ARG;
    int32_t st = IMPACT_OK;
    if (h->owns_storage || h->device_state) {
        cudaError_t e = cudaDeviceSynchronize();
        if (e == cudaSuccess && h->owns_storage) e = cudaFree(h->storage);
        if (e == cudaSuccess && h->device_state) e = cudaFree(h->device_state);
        if (e != cudaSuccess) st = record_cuda_error(e);
    }
    delete h;
    return st;
}

// Enqueue one fused copy of the given segments.
template <bool kHost = false>
static int32_t launch_copy(const CopySegments& segs, cudaStream_t stream) {
    if (segs.n == 0) return IMPACT_OK;
    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;
    const unsigned long long total = segs.vec_end[segs.n - 1];
    // (from the host: a unit per thread, the trip over the bus is what takes the time)
    IMPACT_CUDA_TRY(launch_serialized(multi_copy_kernel<kHost>, dim3(blocks_for(total, kHost ? 1 : 4, di)), dim3(256), 0, stream, segs));
    return IMPACT_OK;
}

// A batch of up to this many bytes in pinned host memory is pushed by one kernel that reads it where it is, instead of a
// copy per field (four fields, a push of 26 KB 27.6 -> 16.4 us from the call to its end, 500 KB 33 -> 27; 1 MB 43 / 46: larger
// ones stay with the copy engine).
constexpr size_t kMostReadInPlace = 512 * 1024;
// Not in a capture either: what a graph copies at its replays stays a copy of the graph's.
static bool is_capturing(cudaStream_t stream) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return capture != cudaStreamCaptureStatusNone;
}

static void add_segment(CopySegments& s, const void* src, void* dst, size_t bytes) {
    const int f = s.n++;
    s.src[f] = static_cast<const char*>(src);
    s.dst[f] = static_cast<char*>(dst);
    s.bytes[f] = bytes;
    s.vec_end[f] = (f ? s.vec_end[f - 1] : 0ull) + (bytes + 15) / 16;
}

extern "C" int32_t impact_buffer_push(impact_buffer* h, const void* const* field_src, int32_t src_location,
                                      int32_t* slot_out, void* stream) {
    if (!h || !field_src || !slot_out || h->device_mode) return IMPACT_ERR_INVALID_ARG;
    if (src_location != IMPACT_SRC_DEVICE && src_location != IMPACT_SRC_HOST) return IMPACT_ERR_INVALID_ARG;
    if (src_location == IMPACT_SRC_DEVICE)
        for (int f = 0; f < h->n_fields; ++f)
            if (field_src[f] && !aligned16(field_src[f])) return IMPACT_ERR_INVALID_ARG;
    int32_t slot = -1;
    for (int32_t i = 0; i < h->N; ++i) {
        const int32_t s = (h->write_cursor + i) % h->N;
        if (!h->valid[s]) { slot = s; break; }
    }
    if (slot < 0) return IMPACT_ERR_FULL;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    if (src_location == IMPACT_SRC_DEVICE) {
        CopySegments segs;
        segs.n = 0;
        for (int f = 0; f < h->n_fields; ++f)
            if (field_src[f]) add_segment(segs, field_src[f], h->field_ptr(slot, f), h->field_bytes[f]);
        int32_t st = launch_copy(segs, cs);
        if (st != IMPACT_OK) return st;
    } else {
        CopySegments segs;
        segs.n = 0;
        size_t total = 0;
        bool in_place = true;
        for (int f = 0; f < h->n_fields; ++f)
            if (field_src[f]) { total += h->field_bytes[f]; in_place = in_place && aligned16(field_src[f]); }
        in_place = in_place && total <= kMostReadInPlace && !is_capturing(cs);
        for (int f = 0; f < h->n_fields && in_place; ++f) {
            if (!field_src[f]) continue;
            in_place = pinned_in_one_range(field_src[f], h->field_bytes[f]);
            if (in_place) add_segment(segs, field_src[f], h->field_ptr(slot, f), h->field_bytes[f]);
        }
        if (in_place) {
            const int32_t st = launch_copy<true>(segs, cs);
            if (st != IMPACT_OK) return st;
        } else {
            for (int f = 0; f < h->n_fields; ++f)
                if (field_src[f])
                    IMPACT_CUDA_TRY(cudaMemcpyAsync(h->field_ptr(slot, f), field_src[f], h->field_bytes[f],
                                                    cudaMemcpyHostToDevice, cs));
        }
    }
    h->valid[slot] = 1;
    h->count[slot] = 0;
    h->write_cursor = (slot + 1) % h->N;
    *slot_out = slot;
    return IMPACT_OK;
}

extern "C" int32_t impact_buffer_sample(impact_buffer* h, int32_t* slot_out, int32_t* k_before_out,
                                        void* const* gather_dst, void* stream) {
    if (!h || !slot_out || !k_before_out || h->device_mode) return IMPACT_ERR_INVALID_ARG;
    if (gather_dst)
        for (int f = 0; f < h->n_fields; ++f)
            if (gather_dst[f] && !aligned16(gather_dst[f])) return IMPACT_ERR_INVALID_ARG;
    int32_t live = 0;
    for (int32_t s = 0; s < h->N; ++s) live += h->valid[s] ? 1 : 0;
    if (live == 0) return IMPACT_ERR_EMPTY;
    int32_t pick = -1;
    uint64_t draws = h->draws;
    int32_t read_cursor = h->read_cursor;
    if (h->mode == IMPACT_SAMPLE_UNIFORM) {
        const uint64_t u = splitmix64_at(h->seed, draws++);
        // floor(u * live / 2^64): unbiased up to 2^-64, no modulo
        uint64_t j = (uint64_t)(((unsigned __int128)u * (uint64_t)live) >> 64);
        for (int32_t s = 0; s < h->N; ++s) {
            if (!h->valid[s]) continue;
            if (j == 0) { pick = s; break; }
            --j;
        }
    } else {
        for (int32_t i = 0; i < h->N; ++i) {
            const int32_t s = (read_cursor + i) % h->N;
            if (h->valid[s]) { pick = s; break; }
        }
        read_cursor = (pick + 1) % h->N;
    }
    if (gather_dst) {
        CopySegments segs;
        segs.n = 0;
        for (int f = 0; f < h->n_fields; ++f)
            if (gather_dst[f]) add_segment(segs, h->field_ptr(pick, f), gather_dst[f], h->field_bytes[f]);
        int32_t st = launch_copy(segs, static_cast<cudaStream_t>(stream));
        if (st != IMPACT_OK) return st;  // bookkeeping untouched on failure
    }
    h->draws = draws;
    h->read_cursor = read_cursor;
    *slot_out = pick;
    *k_before_out = h->count[pick];
    h->count[pick] += 1;
    if (h->count[pick] >= h->K) h->valid[pick] = 0;
    return IMPACT_OK;
}

extern "C" int32_t impact_buffer_append(impact_buffer* h, int32_t slot, int32_t field, const void* src,
                                        void* stream) {
    if (!h || !src || slot < 0 || slot >= h->N || field < 0 || field >= h->n_fields || !aligned16(src))
        return IMPACT_ERR_INVALID_ARG;
    CopySegments segs;
    segs.n = 0;
    add_segment(segs, src, h->field_ptr(slot, field), h->field_bytes[field]);
    return launch_copy(segs, static_cast<cudaStream_t>(stream));
}

extern "C" void* impact_buffer_slot_ptr(impact_buffer* h, int32_t slot, int32_t field) {
    if (!h || slot < 0 || slot >= h->N || field < 0 || field >= h->n_fields) return nullptr;
    return h->field_ptr(slot, field);
}

// A step's wait has run out, twice: the batch is whole, but copies that it had asked for may have come late.
static int32_t status_of(const RingDeviceShared& shared) {
    return shared.failed ? record_cuda_error(cudaErrorTimeout) : IMPACT_OK;
}

// Brings the host copy of the bookkeeping up to date with the device's (device mode only) whatever status_of says; synchronises
// `stream`.
static int32_t download_state(impact_buffer* h, cudaStream_t cs, bool* brought_back) {
    const RingDeviceView v = h->view();
    RingDeviceShared shared;
    IMPACT_CUDA_TRY(cudaMemcpyAsync(&shared, v.shared, sizeof(shared), cudaMemcpyDeviceToHost, cs));
    IMPACT_CUDA_TRY(cudaMemcpyAsync(h->count.data(), v.count, sizeof(int32_t) * (size_t)h->N, cudaMemcpyDeviceToHost, cs));
    IMPACT_CUDA_TRY(cudaStreamSynchronize(cs));
    *brought_back = true;
    const RingDeviceState& now = shared.current();
    for (int32_t i = 0; i < h->N; ++i) h->valid[i] = (int32_t)((now.live[i >> 5] >> (i & 31)) & 1u);
    h->write_cursor = now.hd.write_cursor;
    h->read_cursor = now.hd.read_cursor;
    h->draws = now.hd.draws;
    return status_of(shared);
}

extern "C" int32_t impact_buffer_device_begin(impact_buffer* h, void* stream) {
    if (!h || h->device_mode) return IMPACT_ERR_INVALID_ARG;
    if (h->N > kMaxDeviceSlots) return IMPACT_ERR_UNSUPPORTED;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    if (!h->device_state) {
        void* mem = nullptr;
        IMPACT_CUDA_TRY(cudaMalloc(&mem, h->device_state_bytes()));
        h->device_state = static_cast<char*>(mem);
    }
    IMPACT_CUDA_TRY(cudaMemsetAsync(h->device_state, 0, h->device_state_bytes(), cs));
    const RingDeviceView v = h->view();
    RingDeviceShared shared = {};
    RingDeviceState& first = shared.state[0];
    first.hd.write_cursor = h->write_cursor;
    first.hd.read_cursor = h->read_cursor;
    first.hd.draws = h->draws;
    for (int32_t i = 0; i < h->N; ++i) first.live[i >> 5] |= (h->valid[i] ? 1u : 0u) << (i & 31);
    // (pageable sources: the copies have read them when the calls return)
    IMPACT_CUDA_TRY(cudaMemcpyAsync(v.shared, &shared, sizeof(shared), cudaMemcpyHostToDevice, cs));
    IMPACT_CUDA_TRY(cudaMemcpyAsync(v.count, h->count.data(), sizeof(int32_t) * (size_t)h->N, cudaMemcpyHostToDevice, cs));
    h->device_mode = true;
    return IMPACT_OK;
}

extern "C" int32_t impact_buffer_device_end(impact_buffer* h, void* stream) {
    if (!h || !h->device_mode) return IMPACT_ERR_INVALID_ARG;
    bool brought_back = false;
    const int32_t st = download_state(h, static_cast<cudaStream_t>(stream), &brought_back);
    if (brought_back) h->device_mode = false;
    return st;
}

extern "C" int32_t impact_buffer_device_step(impact_buffer* h, const impact_ring_field_map* map,
                                             const void* learner_logits, const float* values,
                                             const float* bootstrap_values, const void* const* push_sources,
                                             int32_t n_candidates, impact_loss_inputs* inputs_out, void* stream) {
    if (!h || !h->device_mode) return IMPACT_ERR_INVALID_ARG;
    if (push_sources && (n_candidates < 1 || (reinterpret_cast<uintptr_t>(push_sources) & 7u) != 0)) return IMPACT_ERR_INVALID_ARG;
    impact_ring_field_map m = {-1, -1, -1, -1, -1};
    if (inputs_out) {
        if (!map || !aligned16(inputs_out)) return IMPACT_ERR_INVALID_ARG;
        m = *map;
        const int32_t* fs = &m.actions;
        for (int i = 0; i < 5; ++i)
            if (fs[i] < -1 || fs[i] >= h->n_fields) return IMPACT_ERR_INVALID_ARG;
    } else if (!push_sources) {
        return IMPACT_ERR_INVALID_ARG;  // nothing to do
    }
    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    const RingDeviceView v = h->view();
    int blocks = 1;
    bool small = true;
    if (push_sources) {
        unsigned long long units = 0;
        for (int f = 0; f < h->n_fields; ++f) units += (h->field_bytes[f] + 15) / 16;
        // (a block per SM: most steps find every slot live and copy nothing, and an empty launch should cost as little as
        // possible)
        small = units <= (unsigned long long)di->sm_count * kMostSmallUnits;
        blocks = blocks_for(units, 4, di, small ? 32 : kStepThreads);
        if (blocks > di->sm_count) blocks = di->sm_count;
    }
    IMPACT_CUDA_TRY(launch_laid_out(100, small ? ring_step_kernel<32> : ring_step_kernel<kStepThreads>, dim3(blocks),
                                    dim3(small ? 32 : kStepThreads), 0, cs, v, m, learner_logits, values, bootstrap_values, push_sources,
                                    n_candidates, inputs_out ? 1 : 0, inputs_out));
    return IMPACT_OK;
}

extern "C" int32_t impact_buffer_device_events(impact_buffer* h, int32_t* events_out, int32_t max_events,
                                               int32_t* n_out, void* stream) {
    if (!h || !h->device_mode || !events_out || !n_out || max_events < 1) return IMPACT_ERR_INVALID_ARG;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    const RingDeviceView v = h->view();
    RingDeviceShared shared;
    std::vector<int4> log((size_t)kEventLog);
    IMPACT_CUDA_TRY(cudaMemcpyAsync(&shared, v.shared, sizeof(shared), cudaMemcpyDeviceToHost, cs));
    IMPACT_CUDA_TRY(cudaMemcpyAsync(log.data(), v.events, sizeof(int4) * (size_t)kEventLog, cudaMemcpyDeviceToHost, cs));
    IMPACT_CUDA_TRY(cudaStreamSynchronize(cs));
    const RingDeviceHeader& hd = shared.current().hd;
    uint32_t have = hd.n_events < (uint32_t)kEventLog ? hd.n_events : (uint32_t)kEventLog;
    if (have > (uint32_t)max_events) have = (uint32_t)max_events;
    for (uint32_t i = 0; i < have; ++i) {  // oldest first
        const int4 e = log[(hd.n_events - have + i) % kEventLog];
        events_out[4 * i + 0] = e.x; events_out[4 * i + 1] = e.y; events_out[4 * i + 2] = e.z; events_out[4 * i + 3] = e.w;
    }
    *n_out = (int32_t)have;
    return status_of(shared);
}

extern "C" int32_t impact_buffer_live(const impact_buffer* h) {
    if (!h) return IMPACT_ERR_INVALID_ARG;
    if (h->device_mode) {
        bool brought_back = false;
        const int32_t st = download_state(const_cast<impact_buffer*>(h), nullptr, &brought_back);
        if (st != IMPACT_OK) return st;
    }
    int32_t live = 0;
    for (int32_t s = 0; s < h->N; ++s) live += h->valid[s] ? 1 : 0;
    return live;
}

extern "C" size_t impact_buffer_state_bytes(const impact_buffer* h) {
    if (!h) return 0;
    return sizeof(StateHeader) + 2 * sizeof(int32_t) * (size_t)h->N;
}

extern "C" int32_t impact_buffer_export_state(const impact_buffer* h, void* blob, size_t blob_bytes) {
    if (!h || !blob || blob_bytes < impact_buffer_state_bytes(h)) return IMPACT_ERR_INVALID_ARG;
    if (h->device_mode) {  // the device holds the truth: fetch it (default stream; synchronises)
        bool brought_back = false;
        const int32_t st = download_state(const_cast<impact_buffer*>(h), nullptr, &brought_back);
        if (st != IMPACT_OK) return st;
    }
    StateHeader hd;
    memset(&hd, 0, sizeof(hd));
    hd.magic = kStateMagic; hd.version = 1;
    hd.N = h->N; hd.K = h->K; hd.n_fields = h->n_fields; hd.mode = h->mode;
    hd.write_cursor = h->write_cursor; hd.read_cursor = h->read_cursor;
    hd.seed = h->seed; hd.draws = h->draws;
    char* out = static_cast<char*>(blob);
    memcpy(out, &hd, sizeof(hd));
    memcpy(out + sizeof(hd), h->valid.data(), sizeof(int32_t) * (size_t)h->N);
    memcpy(out + sizeof(hd) + sizeof(int32_t) * (size_t)h->N, h->count.data(), sizeof(int32_t) * (size_t)h->N);
    return IMPACT_OK;
}

extern "C" int32_t impact_buffer_import_state(impact_buffer* h, const void* blob, size_t blob_bytes) {
    if (!h || !blob || blob_bytes < impact_buffer_state_bytes(h) || h->device_mode) return IMPACT_ERR_INVALID_ARG;
    StateHeader hd;
    const char* in = static_cast<const char*>(blob);
    memcpy(&hd, in, sizeof(hd));
    if (hd.magic != kStateMagic || hd.version != 1 || hd.N != h->N || hd.K != h->K ||
        hd.n_fields != h->n_fields || (hd.mode != IMPACT_SAMPLE_UNIFORM && hd.mode != IMPACT_SAMPLE_ROUND_ROBIN))
        return IMPACT_ERR_INVALID_ARG;
    if (hd.write_cursor < 0 || hd.write_cursor >= h->N || hd.read_cursor < 0 || hd.read_cursor >= h->N)
        return IMPACT_ERR_INVALID_ARG;
    const int32_t* v = reinterpret_cast<const int32_t*>(in + sizeof(hd));
    const int32_t* c = v + h->N;
    for (int32_t s = 0; s < h->N; ++s)
        if ((v[s] != 0 && v[s] != 1) || c[s] < 0 || c[s] > h->K) return IMPACT_ERR_INVALID_ARG;
    h->mode = hd.mode; h->seed = hd.seed; h->draws = hd.draws;
    h->write_cursor = hd.write_cursor; h->read_cursor = hd.read_cursor;
    h->valid.assign(v, v + h->N);
    h->count.assign(c, c + h->N);
    return IMPACT_OK;
}

template <typename V, int U>
static int32_t launch_granules(const V* src, const int32_t* idx, unsigned int n, int n_src_rows, unsigned int units, V* dst,
                               const DeviceInfo* di, cudaStream_t cs) {
    constexpr unsigned int per = 16 / sizeof(V);
    const unsigned long long granules = (unsigned long long)n * units / per;
    const int blocks = blocks_for(granules + 16, U, di);  // (16: threads for what is left of the last granule)
    const unsigned long long stride = (unsigned long long)blocks * 256 * per;
    IMPACT_CUDA_TRY(launch_serialized(gather_granules_kernel<V, U>, dim3(blocks), dim3(256), 0, cs, src, idx, n, n_src_rows,
                                      units, (unsigned int)(stride / units), (unsigned int)(stride % units), dst));
    return IMPACT_OK;
}

template <typename V>
static int32_t launch_gather(const void* src, const int32_t* idx, int64_t n, int64_t n_src_rows, size_t row_bytes,
                             void* dst, const DeviceInfo* di, cudaStream_t cs) {
    const long long units = (long long)(row_bytes / sizeof(V));
    const V* const from = static_cast<const V*>(src);
    V* const to = static_cast<V*>(dst);
    constexpr long long most = 1ll << 31;  // (what the granules' counters hold)
    // (elements of 4 and 8 bytes: a fifth and more of the granules of rows below 32 bytes hold an end, 25.4 / 27.4 us at 20
    // bytes; narrower elements gain all the same, 45 / 40 at 18)
    const bool wide_enough = sizeof(V) == 4 || sizeof(V) == 8 ? row_bytes >= 32 : row_bytes >= 16;
    if (wide_enough && aligned16(dst) && n < most && n_src_rows < most && (long long)row_bytes < most) {
        if constexpr (sizeof(V) == 16)  // (two under way where a thread has more than one: 4 MB 4.3 us against 4.7; less 1.5 / 1.4)
            if (n * units > (long long)di->sm_count * 8 * 256)
                return launch_granules<V, 2>(from, idx, (unsigned int)n, (int)n_src_rows, (unsigned int)units, to, di, cs);
        return launch_granules<V, 1>(from, idx, (unsigned int)n, (int)n_src_rows, (unsigned int)units, to, di, cs);
    }
    constexpr int U = sizeof(V) >= 8 ? 2 : 1;
    const int blocks = blocks_for((unsigned long long)n * (unsigned long long)units, U, di);
    const long long stride = (long long)blocks * 256;
    IMPACT_CUDA_TRY(launch_serialized(gather_rows_kernel<V, U>, dim3(blocks), dim3(256), 0, cs, from, idx, (long long)n,
                                      (long long)n_src_rows, units, stride / units, stride % units, to));
    return IMPACT_OK;
}

extern "C" int32_t impact_gather_rows(const void* src, const int32_t* idx, int64_t n, int64_t n_src_rows,
                                      size_t row_bytes, void* dst, void* stream) {
    if (!src || !idx || !dst || n < 0 || n_src_rows < 1 || row_bytes == 0) return IMPACT_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(idx) & 3u) != 0) return IMPACT_ERR_INVALID_ARG;
    if (n == 0) return IMPACT_OK;
    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    const uintptr_t both = reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst) | row_bytes;
    // the widest element that every row of both tensors is aligned to
    if ((both & 15u) == 0) return launch_gather<uint4>(src, idx, n, n_src_rows, row_bytes, dst, di, cs);
    if ((both & 7u) == 0) return launch_gather<uint2>(src, idx, n, n_src_rows, row_bytes, dst, di, cs);
    if ((both & 3u) == 0) return launch_gather<uint32_t>(src, idx, n, n_src_rows, row_bytes, dst, di, cs);
    if ((both & 1u) == 0) return launch_gather<uint16_t>(src, idx, n, n_src_rows, row_bytes, dst, di, cs);
    return launch_gather<unsigned char>(src, idx, n, n_src_rows, row_bytes, dst, di, cs);
}

extern "C" int32_t impact_stream_copy(const void* src, size_t read_bytes, void* dst, size_t write_bytes, void* stream) {
    if (!src || !dst || !aligned16(src) || !aligned16(dst) || read_bytes == 0 || write_bytes > read_bytes ||
        (read_bytes & 15u) != 0 || (write_bytes & 15u) != 0 || write_bytes < 16)
        return IMPACT_ERR_INVALID_ARG;
    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;
    const unsigned long long n_read = read_bytes / 16, n_write = write_bytes / 16;
    IMPACT_CUDA_TRY(launch_serialized(stream_copy_kernel, dim3(blocks_for(n_read, 4, di)), dim3(256), 0,
                                      static_cast<cudaStream_t>(stream), static_cast<const uint4*>(src), n_read,
                                      static_cast<uint4*>(dst), n_write, reinterpret_cast<unsigned int*>(dst)));
    return IMPACT_OK;
}
