// Device building blocks of the fused IMPACT loss kernels (sm_100a): bulk copies and their barriers, fast
// exponentials, the importance weights and the surrogate, published aggregates and sums.
//
// Work decomposition shared by the loss kernels (see impact_flat.cuh):
//   * a tile is a number of consecutive steps ("rows") of the row-major [B*T, width] tensors, which is one contiguous
//     slab of global memory; each byte is read once;
//   * slabs reach shared memory by bulk asynchronous copies (one instruction per slab) and keep their dense layout;
//     gradients overwrite the staged rows in place and leave by bulk stores;
//   * sums are reduced in a fixed order: per thread, per warp, per block, and across blocks by one collecting group
//     that reads every block's tagged row.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace impact {
namespace dev {

constexpr int kNumSums = 7;  // surrogate, value, entropy, kl, clipped, rho-truncated, ratio

// Two fp32 values as a pair of bf16, rounded to nearest even.
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&h);
}

// ---- bulk asynchronous copies (the 1-D form of the tensor memory accelerator) -----------
// One elected thread moves a whole contiguous slab between global and shared memory; the
// other threads spend no instructions on staging.  Source, destination and size must be
// multiples of 16 bytes.  Loads signal an mbarrier in shared memory; stores are tracked by
// bulk async-groups.  No multicast and no cluster: every copy is local to the block.
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// Initialisation of many barriers: each without a fence, then one fence_mbarrier_init() by every
// initialising thread before the block-wide barrier that precedes their first use.
__device__ __forceinline__ void mbarrier_init_nofence(uint64_t* bar, uint32_t arrivals) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(arrivals) : "memory");
}
__device__ __forceinline__ void fence_mbarrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbarrier_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbarrier_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// One look at the barrier, without waiting: has the phase with the given parity completed?
__device__ __forceinline__ bool mbarrier_test(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return done != 0;
}
// Waits for the phase with the given parity to complete.  The wait is bounded: if the bytes never arrive the caller
// gets `false` instead of a hang.  It also gives up (at once) when `*abort_flag` is set, and sets it when it gives up
// itself, so that one wait that runs out ends every other wait of the block instead of each running out in turn.
__device__ __forceinline__ bool mbarrier_wait(uint64_t* bar, uint32_t parity, int* abort_flag) {
    const uint32_t addr = smem_addr(bar);
    // (no suspend hint and no sleep between tries: the wait sits between a tile's landing and the first
    // instruction that uses it, and a hinted try followed by a 64 ns sleep measured 0.1 us per launch slower)
    for (uint32_t tries = 0; tries < (1u << 24); ++tries) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (done) return true;
        if (*reinterpret_cast<volatile int*>(abort_flag)) return false;
    }
    *reinterpret_cast<volatile int*>(abort_flag) = 1;
    return false;
}
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gmem_src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(smem_dst)), "l"(__cvta_generic_to_global(gmem_src)), "r"(bytes),
                 "r"(smem_addr(bar)) : "memory");
}
// Asks L2 to fetch a contiguous range (16-byte aligned, a multiple of 16 bytes); nothing waits for it.
__device__ __forceinline__ void bulk_prefetch_l2(const void* gmem_src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(gmem_src)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_store(void* gmem_dst, const void* smem_src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 ::"l"(__cvta_generic_to_global(gmem_dst)), "r"(smem_addr(smem_src)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Shared memory written by ordinary stores becomes visible to the copy engine.
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// All bulk stores of this thread have finished READING shared memory (it may be reused).
__device__ __forceinline__ void bulk_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// ---- byte ranges that do not start or end on a 16-byte boundary ---------------------------
// A tile of a dense tensor starts wherever its first row does: for row pitches that are not a
// multiple of 16 bytes (A = 18 in bf16: 36 bytes) most tiles start and end inside a 16-byte
// granule, which a bulk copy cannot do.  Loads are therefore widened to the enclosing granules:
// the copy also brings the up to 15 bytes before the range and the up to 15 bytes after it (the
// tensor's own neighbouring rows) into the padding of the shared-memory slab, and the range
// itself lands at the same offset inside its granule as in global memory.  Only where the tensor
// ENDS inside the last granule is that granule fetched by ordinary loads instead.
struct WideRange {
    long long first;  // byte offset (in the tensor) of the first granule
    uint32_t span;    // bytes a bulk copy may move from there: a multiple of 16, possibly 0
    uint32_t tail;    // bytes after the span that belong to the tensor's last, partial granule (0..15)
};
__device__ __forceinline__ WideRange widen_range(long long byte0, uint32_t bytes, long long tensor_bytes) {
    WideRange w;
    const uint32_t m = (uint32_t)byte0 & 15u;
    w.first = byte0 - m;
    w.span = (m + bytes + 15u) & ~15u;
    w.tail = 0;
    if (w.first + (long long)w.span > tensor_bytes) {
        w.span -= 16u;
        w.tail = (uint32_t)(tensor_bytes - (w.first + (long long)w.span));
    }
    return w;
}
// Asks L2 for the granules of a byte range of a tensor whose base is 16-byte aligned (one request to the copy
// engine; nothing waits for it).  Ordinary per-line prefetch instructions were tried instead and slowed the
// launches down by half.
__device__ __forceinline__ void prefetch_range_l2(const void* base, long long byte0, uint32_t bytes, long long tensor_bytes) {
    const WideRange w = widen_range(byte0, bytes, tensor_bytes);
    if (w.span) bulk_prefetch_l2(static_cast<const unsigned char*>(base) + w.first, w.span);
}

// Run by a whole warp: sends `bytes` bytes of shared memory at `src` to global memory at `dst`, where src and
// dst agree modulo 16.  The whole granules in between leave by one bulk store (lane 0); the up to 15 bytes before
// the first whole granule and after the last one leave by byte stores, a lane each (a granule shared with a
// neighbouring range is written by both neighbours, each its own bytes).  `wrote`: the bytes were written by
// ordinary stores of this warp's threads, so they are fenced towards the copy engine first.  Lane 0 learns
// whether a bulk store was issued (its group is committed; see bulk_store_wait_read).
__device__ __forceinline__ bool warp_send_bytes(unsigned char* dst, const unsigned char* src, uint32_t bytes, bool wrote) {
    const uint32_t lane = threadIdx.x & 31u;
    if ((((uint32_t)reinterpret_cast<uintptr_t>(dst) | bytes) & 15u) == 0u) {  // whole granules only: the usual case
        if (wrote) fence_async_shared();
        __syncwarp();
        if (lane == 0 && bytes) {
            bulk_store(dst, src, bytes);
            return true;
        }
        return false;
    }
    uint32_t head = (16u - ((uint32_t)reinterpret_cast<uintptr_t>(dst) & 15u)) & 15u;
    if (head > bytes) head = bytes;
    const uint32_t body = (bytes - head) & ~15u;
    const uint32_t tail = bytes - head - body;
    if (wrote) fence_async_shared();
    __syncwarp();
    if (lane < head) dst[lane] = src[lane];
    if (lane >= 16u && lane - 16u < tail) dst[head + body + lane - 16u] = src[head + body + lane - 16u];
    if (lane == 0 && body) {
        bulk_store(dst + head, src + head, body);
        return true;
    }
    return false;
}

__device__ __forceinline__ float exp2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float log2_fast(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 1 / x for a normal x whose reciprocal is one too: the approximate reciprocal (an ulp off at most) and one step of
// Newton's iteration, which leaves the rounding of that step.  (The rounded reciprocal is a call with a path for every other
// x: 0.2 us on the shortest launches, 3 % on 926 000 steps of seven actions.)
__device__ __forceinline__ float reciprocal(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return fmaf(y, fmaf(-x, y, 1.0f), y);
}

// The larger of two; a NaN stays one.
__device__ __forceinline__ float max_or_nan(float x, float y) {
    float m;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(x), "f"(y));
    return m;
}

// Sum of one value over the warp, in every lane (fixed order).
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}
// Sums of four values over the warp in one butterfly of six shuffles: lanes 0-7 return the
// total of `a`, lanes 8-15 of `b`, lanes 16-23 of `c`, lanes 24-31 of `d` (fixed order).
__device__ __forceinline__ float warp_sum4(float a, float b, float c, float d) {
    const int lane = threadIdx.x & 31;
    const bool hi16 = (lane & 16) != 0, hi8 = (lane & 8) != 0;
    float k0 = hi16 ? c : a, k1 = hi16 ? d : b;
    const float s0 = hi16 ? a : c, s1 = hi16 ? b : d;
    k0 += __shfl_xor_sync(0xffffffffu, s0, 16);
    k1 += __shfl_xor_sync(0xffffffffu, s1, 16);
    float x = hi8 ? k1 : k0;
    const float y = hi8 ? k0 : k1;
    x += __shfl_xor_sync(0xffffffffu, y, 8);
    x += __shfl_xor_sync(0xffffffffu, x, 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x;
}

__device__ __forceinline__ void publish_tagged(unsigned long long* slot, float value, unsigned int tag);

// A tile's aggregate map, published as two (value, launch tag) pairs (see publish_tagged).
__device__ __forceinline__ void publish_tile_aggregate(unsigned long long* slot, float a, float b, unsigned int tag) {
    publish_tagged(slot, a, tag);
    publish_tagged(slot + 1, b, tag);
}

// The two slots of the aggregate of the tile `j` places later in this tile's trajectory (they lie j * stride
// before `mine`), as they are right now.  The values are not looked at here, so the load can be issued long before
// it is needed.
__device__ __forceinline__ void load_aggregate(const unsigned long long* mine, long long stride, int j,
                                               unsigned long long& va, unsigned long long& vb) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(va), "=l"(vb) : "l"(mine - (long long)j * stride) : "memory");
}

// A chunk's maps, the one that is applied first in lane 0, which gets the whole.
__device__ __forceinline__ void compose_in_time_order(float& a, float& b) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const float a2 = __shfl_down_sync(0xffffffffu, a, off);
        const float b2 = __shfl_down_sync(0xffffffffu, b, off);
        if (lane + off < 32) {  // (a, b) <- (a2, b2) o (a, b): the higher lane's map is applied later
            b = fmaf(a2, b, b2);
            a = a2 * a;
        }
    }
}

// Run by one warp: `mine` points at this tile's pair of slots; tile j (1 = the nearest later tile ... r = the
// trajectory's last) has its slots at mine - j * stride.  Reads their aggregates (a lane each, 32 at a time,
// waiting -- bounded -- until a pair carries this launch's tag), composes them in time order and returns the
// composition applied to 0: the value that enters this tile's last step.  A pair that never came raises the error word.  `peeked` / (pa, pb): lane l brings along
// what load_aggregate found earlier for tile r - l; it counts if it carries the tag.
__device__ __forceinline__ float compose_later_aggregates(const unsigned long long* mine, long long stride, int r,
                                                          unsigned int tag, int* abort_flag, unsigned int* error_word,
                                                          bool peeked, unsigned long long pa,
                                                          unsigned long long pb) {
    const int lane = threadIdx.x & 31;
    // the value flows from tile r down to tile 1: x <- agg_j(x).  Lanes take j = r - lane, r - lane - 32, ...:
    // chunk by chunk from the far end, lane 0 holding the map that is applied first.
    float x = 0.0f;
    for (int base = r; base > 0; base -= 32) {
        const int j = base - lane;
        float a = 1.0f, b = 0.0f;  // identity for lanes beyond the chunk
        if (j > 0) {
            unsigned long long va = pa, vb = pb;
            bool ok = peeked && base == r && ((unsigned int)(va >> 32) == tag) && ((unsigned int)(vb >> 32) == tag);
            for (int tries = 0; tries < (1 << 22) && !ok; ++tries) {
                load_aggregate(mine, stride, j, va, vb);
                ok = ((unsigned int)(va >> 32) == tag) && ((unsigned int)(vb >> 32) == tag);
                if (!ok && *reinterpret_cast<volatile int*>(abort_flag)) break;
            }
            if (!ok) {
                *reinterpret_cast<volatile int*>(abort_flag) = 1;
                atomicExch(error_word, 1u);
            }
            a = __uint_as_float((unsigned int)va);
            b = __uint_as_float((unsigned int)vb);
        }
        compose_in_time_order(a, b);
        const float ca = __shfl_sync(0xffffffffu, a, 0), cb = __shfl_sync(0xffffffffu, b, 0);
        x = fmaf(ca, x, cb);
    }
    return x;
}

// The same, with the same bits, for tiles of few rows, of which a trajectory has hundreds (a look at all later tiles takes a
// trip to L2 for every 32 of them: 11 of 375).  Tiles are counted from the trajectory's end, this one is number r; its blocks of
// 32 are the chunks above.  The last tile of a block leads it: it publishes the block's map, finds what enters the block -- a
// lane per earlier block, from the nearest whose value is known -- and publishes the value that leaves it.  The other tiles
// wait for the maps between them and their block's first and for the one value that enters it, so that a trajectory's tiles do
// not all ask for the same lines.  A block's maps are always composed as the one tree and applied to what leaves the block
// before, so the bits do not depend on what had been published by when.
// `blocks`: four slots per whole block of this trajectory -- the block's map, the value that leaves it, none.  (own_a, own_b):
// this tile's map, in lane 0.
// (A call of its own, out of the way of the row passes' registers: 16 x 4096 steps of 64 actions 16.3 us, inlined 17.2; 31 x 4000 of 40
// 18.2 / 20.0; 2 x 4000 of 512 17.4 / 18.3.)
static __device__ __noinline__ float value_from_later_tiles(const unsigned long long* mine, unsigned long long* blocks, int r,
                                                            float own_a, float own_b, unsigned int tag, int* abort_flag,
                                                            unsigned int* error_word) {
    const int lane = threadIdx.x & 31;
    const int block = r >> 5, part = r & 31;
    const bool leads = part == 31;
    auto tagged = [&](unsigned long long v) { return (unsigned int)(v >> 32) == tag; };  // (no tag is 0)
    auto number = [](unsigned long long v) { return __uint_as_float((unsigned int)v); };
    auto gave_up = [&]() {
        *reinterpret_cast<volatile int*>(abort_flag) = 1;
        if (lane == 0) atomicExch(error_word, 1u);
        return 0.0f;
    };
    // the block's maps in front of this tile's, and what enters the block
    const bool map = lane < part, value = lane == 31 && !leads && block > 0;
    const unsigned long long* const at = map ? mine - 2 * (part - lane) : blocks + 4 * (block - 1) + 2;
    unsigned long long va = 0, vb = 0;
    bool there = !map && !value, all = false;
    for (int tries = 0; tries < (1 << 22); ++tries) {
        if (!there) {
            load_aggregate(at, 0, 0, va, vb);
            there = tagged(va) && (value || tagged(vb));
        }
        all = __all_sync(0xffffffffu, there);
        if (all || __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(abort_flag))) break;
    }
    if (!all) return gave_up();
    float x = block > 0 && !leads ? number(__shfl_sync(0xffffffffu, va, 31)) : 0.0f;
    float a = map ? number(va) : 1.0f, b = map ? number(vb) : 0.0f;
    if (leads) {
        own_a = __shfl_sync(0xffffffffu, own_a, 0);
        own_b = __shfl_sync(0xffffffffu, own_b, 0);
        float ba = map ? a : own_a, bb = map ? b : own_b;
        compose_in_time_order(ba, bb);
        if (lane == 0) publish_tile_aggregate(blocks + 4 * block, ba, bb, tag);
        if (block > 0) {
            unsigned int needed = 0, have = 0, valued = 0;
            int known = lane >= block ? 2 : 0;  // 1: the map of the block, lane + 1 before this one, 2: the value that leaves it
            unsigned long long vx = 0, none = 0;
            for (int tries = 0; tries < (1 << 22); ++tries) {
                if (known < 2 && lane < block) {
                    load_aggregate(blocks + 4 * (block - 1 - lane), 0, 0, va, vb);
                    load_aggregate(blocks + 4 * (block - 1 - lane) + 2, 0, 0, vx, none);
                    known = tagged(vx) ? 2 : tagged(va) && tagged(vb) ? 1 : 0;
                }
                valued = __ballot_sync(0xffffffffu, known == 2);
                have = __ballot_sync(0xffffffffu, known != 0);
                needed = valued ^ (valued - 1u);  // lanes up to the first of those
                if (valued && (have & needed) == needed) break;
                if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(abort_flag))) break;
            }
            if (!valued || (have & needed) != needed) return gave_up();
            int n = __ffs((int)valued) - 1;
            x = n < block ? number(__shfl_sync(0xffffffffu, vx, n)) : 0.0f;
            while (--n >= 0) x = fmaf(number(__shfl_sync(0xffffffffu, va, n)), x, number(__shfl_sync(0xffffffffu, vb, n)));
        }
        if (lane == 0) publish_tagged(blocks + 4 * block + 2, fmaf(ba, x, bb), tag);
    }
    if (part == 0) return x;
    compose_in_time_order(a, b);
    return fmaf(__shfl_sync(0xffffffffu, a, 0), x, __shfl_sync(0xffffffffu, b, 0));
}

// Scalars of the loss that the kernels need; filled on the host.
struct LossScalars {
    float rho_bar, c_bar, clip_lo, clip_hi;
    float vf_coef, ent_coef, kl_coef, lambda_, log_rho_tw;
    float inv_M;
    // products and conversions of the above that a step would otherwise form for itself
    float ent_over_M, kl_over_M, dvalue_over_adv, log2_rho_tw;
    int is_source, ratio_mode, objective;
    double steps_total;  // M: the steps the means are taken over (this call's, or the whole batch's when it is split)
};

// Per-step quantities once the three log-probabilities are known.
struct StepIn {
    float l_theta, l_target, l_worker;  // may all be shifted by one common amount ...
    float l_shift = 0.0f;               // ... which is this: l_theta + l_shift is the true log-probability
    float reward, discount, value, value_next;
    bool last_step;  // t == T-1: the trace stops, V_{t+1} is the bootstrap value
    float rho = 0.0f;       // truncated importance weight of the step (set by recursion_map)
    float adv_next = 0.0f;  // A_{t+1} (set from the scan)
};

// exp of a log-probability difference.  Arguments are a few units at most, where the
// multiply-then-exp2 form stays within ~3e-7 relative of the correctly rounded result.
__device__ __forceinline__ float exp_of_logratio(float x) { return exp2_fast(x * 1.4426950408889634f); }

// Truncated importance weights and the affine map of the advantage recursion
// (Section 2.2; Section 3.1).  Returns whether exp(x) exceeded rho_bar.  kPlain: the default configuration
// (importance weights pi_target / pi_worker, ratio R3, clipped surrogate), without the run-time switches.
// (Products and sums are spelled out so that both forms give the same bits.)
template <bool kPlain>
__device__ __forceinline__ bool recursion_map(StepIn& s, const LossScalars& k, float& a, float& b) {
    const float x = ((!kPlain && k.is_source == 1) ? s.l_theta : s.l_target) - s.l_worker;
    const float w = (!kPlain && k.is_source == 2) ? 1.0f : exp_of_logratio(x);  // 2: plain GAE, no importance weights
    const float rho = fminf(k.rho_bar, w);
    s.rho = rho;
    const float c = fminf(k.c_bar, w);
    b = __fmul_rn(rho, __fadd_rn(fmaf(s.discount, s.value_next, s.reward), -s.value));
    a = s.last_step ? 0.0f : __fmul_rn(__fmul_rn(k.lambda_, s.discount), c);
    return w > k.rho_bar;
}

// Ratio of Section 4.1 and the eps-clipped surrogate of Appendix E.  Returns the weight
// adv * R of the policy-gradient term (0 where the clip removes it).
template <bool kPlain>
__device__ __forceinline__ float surrogate(const StepIn& s, const LossScalars& k, float adv,
                                           float& surr, float& ratio, bool& clipped) {
    if (!kPlain && k.objective == 1) {
        // IMPALA's actor update (Section 2.2): weight rho_t (r_t + gamma_t v_{t+1} - V_t) on
        // grad log pi_theta, v the V-trace target V + A (the bootstrap value after the last step)
        const float v_next = s.value_next + (s.last_step ? 0.0f : s.adv_next);
        const float w = __fmul_rn(s.rho, __fadd_rn(fmaf(s.discount, v_next, s.reward), -s.value));
        surr = __fmul_rn(w, s.l_theta + s.l_shift);
        ratio = s.rho;
        clipped = false;
        return w;
    }
    float d = fmaxf(s.l_target, s.l_worker - k.log_rho_tw);
    if (!kPlain) {
        if (k.ratio_mode == 1) d = s.l_target;
        else if (k.ratio_mode == 2) d = s.l_worker;
    }
    const float R = exp_of_logratio(s.l_theta - d);
    const float Rc = fminf(fmaxf(R, k.clip_lo), k.clip_hi);
    const float Ra = __fmul_rn(R, adv);
    surr = fminf(Ra, __fmul_rn(Rc, adv));
    clipped = (adv > 0.0f && R > k.clip_hi) || (adv < 0.0f && R < k.clip_lo);
    ratio = R;
    return clipped ? 0.0f : Ra;
}

// ---- sums published as tagged rows (persistent kernel) --------------------------------------
// Every launch that uses a workspace has a number, kept in the workspace's third counter word: the
// launch's tag is that word + 1 (never 0, which is what a cleared workspace holds), and the launch's
// collecting group stores the tag back as its last act.  A group's row is eight (value, tag) pairs,
// each written by ONE aligned 8-byte store, which the memory model makes indivisible: a reader that
// sees this launch's tag in a pair sees this launch's value beside it.  So rows need no fence, no
// atomic counter and no "last block" -- the collecting group simply reads every row until all its
// pairs carry the tag (a bounded wait), and adds them in index order.
__device__ __forceinline__ unsigned int launch_tag(const unsigned int* counter_words) {
    unsigned int n;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(counter_words + 2) : "memory");
    return n + 1u == 0u ? 1u : n + 1u;
}
__device__ __forceinline__ void publish_tagged(unsigned long long* slot, float value, unsigned int tag) {
    const unsigned long long v = ((unsigned long long)tag << 32) | (unsigned long long)__float_as_uint(value);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(slot), "l"(v) : "memory");
}

// The block's row of sums.  Every consumer warp, once its sums are final, leaves them in its row of shared memory
// -- [surrogate, value, entropy, kl, clipped, truncated, ratio, 0] -- and draws a ticket from a counter in shared
// memory; the producer warp draws one too, after it has left this launch's tag there.  Whoever draws the last
// ticket adds all rows in index order (so the result does not depend on who that is) and publishes the block's row
// of (value, tag) pairs.  A pair is one 8-byte store, so whoever reads the tag of this launch reads this launch's
// value with it: no fence, no round trip.  The tickets are acquire-release operations on one word: the last
// drawer sees every row and the tag.  (Before, the producer warp polled one barrier per group and published: its
// row left 0.35-0.5 us after the last group's sums were final.)
template <int C, int WPG>
__device__ __forceinline__ void draw_ticket_and_publish(unsigned int* tickets, const unsigned int* tag_s,
                                                        float (*red)[WPG][8], unsigned long long* tagged_rows) {
    const int lane = threadIdx.x & 31;
    unsigned int t = 0;
    __syncwarp();
    if (lane == 0)
        asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(t) : "r"(smem_addr(tickets)) : "memory");
    __syncwarp();
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t == (unsigned int)(C * WPG) && lane < 8) {  // C * WPG consumer warps and the producer warp: the last of C * WPG + 1
        float y = 0.0f;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            float yc = 0.0f;
#pragma unroll
            for (int w = 0; w < WPG; ++w) yc += red[c][w][lane];
            y = (c == 0) ? yc : y + yc;
        }
        publish_tagged(tagged_rows + (size_t)blockIdx.x * 8 + lane, y, *reinterpret_cast<const volatile unsigned int*>(tag_s));
    }
}
// A consumer warp's part (called by every thread of the warp): a butterfly into the warp's row, then the ticket.
template <int C, int WPG>
__device__ __forceinline__ void hand_over_warp_sums(float t_surr, float t_val, float t_ent, float t_ratio, float t_kl,
                                                    bool want_kl, int n_clip, int n_trunc, float* warp_row,
                                                    unsigned int* tickets, const unsigned int* tag_s,
                                                    float (*red)[WPG][8], unsigned long long* tagged_rows) {
    const int lane = threadIdx.x & 31;
    const float x = warp_sum4(t_surr, t_val, t_ent, t_ratio);
    const float xk = want_kl ? warp_sum(t_kl) : 0.0f;
    if ((lane & 7) == 0) warp_row[lane == 24 ? 6 : (lane >> 3)] = x;
    if (lane == 0) {
        warp_row[3] = xk;
        warp_row[4] = (float)n_clip;
        warp_row[5] = (float)n_trunc;
        warp_row[7] = 0.0f;
    }
    draw_ticket_and_publish<C, WPG>(tickets, tag_s, red, tagged_rows);
}

// Run by the NT threads of one group (`gtid` in the group, named barrier `bar_id`): waits for `nrows`
// tagged rows, adds them, writes the eight loss terms and advances the workspace's launch number.
// Thread t owns column t % 8 of rows t / 8, t / 8 + NT / 8, ...: a row is read by eight neighbouring
// lanes (64 contiguous bytes) and all of a thread's loads are in flight together, so a grid's worth of rows
// costs one trip to L2.  The rows, fp32 sums over a block's tiles, are added in S as trees in a fixed order: each thread
// its rows, then lanes, then warps.  Returns false if a row never showed up.
template <int NT, typename S>
__device__ __noinline__ bool reduce_tagged_rows(const unsigned long long* rows, int nrows, unsigned int tag,
                                                  unsigned int* counter_words, float* loss_terms, float vf_coef,
                                                  float ent_coef, float kl_coef, double M, int gtid, int bar_id,
                                                  int* abort_flag) {
    __shared__ S fred[NT / 32][8];
    constexpr int kStride = NT / 8, kU = 10;
    const int col = gtid & 7, rc = gtid >> 3;
    const double inv_m = 1.0 / M;  // (a long division: done while the rows are still on their way)
    auto tree = [](S* x, int n) {
#pragma unroll
        for (int w = 1; w < n; w *= 2)
#pragma unroll
            for (int u = 0; u + w < n; u += 2 * w) x[u] += x[u + w];
        return x[0];
    };
    S acc = 0;
    bool missing = false;
    for (int base = rc; base < nrows && !missing; base += kStride * kU) {
        unsigned long long v[kU];
        unsigned int have = 0;
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (base + kStride * u >= nrows) have |= 1u << u;  // beyond the last row: nothing to wait for
        for (int tries = 0; tries < (1 << 22) && have != (1u << kU) - 1u; ++tries) {
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (!(have & (1u << u)))
                    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];"
                                 : "=l"(v[u]) : "l"(rows + (size_t)(base + kStride * u) * 8 + col) : "memory");
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (!(have & (1u << u)) && (unsigned int)(v[u] >> 32) == tag) have |= 1u << u;
            if (have != (1u << kU) - 1u && *reinterpret_cast<volatile int*>(abort_flag)) break;
        }
        if (have != (1u << kU) - 1u) missing = true;
        S x[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) x[u] = base + kStride * u < nrows ? (S)__uint_as_float((unsigned int)v[u]) : (S)0;
        acc += tree(x, kU);
    }
    if (missing) *reinterpret_cast<volatile int*>(abort_flag) = 1;  // read back below, after the group's barrier
    const int lane = gtid & 31, warp = gtid >> 5;
    acc += __shfl_xor_sync(0xffffffffu, acc, 8);
    acc += __shfl_xor_sync(0xffffffffu, acc, 16);
    if (lane < 8) fred[warp][lane] = acc;
    asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "n"(NT) : "memory");
    // the last steps sit between the slowest block's row and the end of the launch: a lane per column
    if (gtid < 8) {
        S x[NT / 32];
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) x[w] = fred[w][gtid];
        const double t = (double)tree(x, NT / 32) * inv_m;  // columns: surrogate, value, entropy, kl, clipped, truncated, ratio
        const double t1 = __shfl_sync(0xffu, t, 1), t2 = __shfl_sync(0xffu, t, 2), t3 = __shfl_sync(0xffu, t, 3);
        if (gtid == 0) {
            loss_terms[0] = (float)(-t + (double)vf_coef * t1 - (double)ent_coef * t2 + (double)kl_coef * t3);
            counter_words[2] = tag;
        }
        if (gtid < kNumSums) loss_terms[gtid + 1] = (float)(gtid == 0 ? -t : t);
    }
    return *reinterpret_cast<volatile int*>(abort_flag) == 0;
}

}  // namespace dev
}  // namespace impact
