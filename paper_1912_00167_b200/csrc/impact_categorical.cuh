// The categorical IMPACT loss + gradient kernel and its launch rules (one kernel template for every action count).
//
// (Layout, protocols and launch shape: impact_flat.cuh.)
#pragma once

#include <type_traits>

#include "impact_flat.cuh"

namespace impact {

__host__ __device__ constexpr size_t cat_stage_bytes(size_t nt, size_t A, size_t in_elem, size_t out_elem) {
    const size_t raw = 2 * slab_pitch(nt, A * in_elem) + (in_elem == out_elem ? 0 : slab_pitch(nt, A * out_elem));
    return (raw + 127) / 128 * 128;
}

constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;

// ---- a step's scalars -------------------------------------------------------------------------------------------
// Log-probabilities are kept in base 2 (as the row passes form them): every exponential of a difference is then one
// instruction.  The worker's, which comes in natural units, is scaled inside the multiply-add that subtracts it: scaled by
// itself it would be rounded at its own size before the difference is taken, the largest error of a ratio where actions
// are few (dvalues' error against 64 bits, two to seven actions: 2.5e-7 to 3.2e-7 that way).
// (Products and sums are spelled out where the compiler could fuse them one way in one instantiation and another way in
// the next: every kernel that can serve a call gives the same bits, but for the KL term and its gradient, which flat launches
// of few actions form from exponentials that they keep and split ones do not; see kKeepTarget.)
struct Step {
    float l2_theta, l2_target, l_worker;
    float reward, discount, value, value_next;
    bool ends;              // last step of its trajectory: the trace stops, V_{t+1} is the bootstrap value
    float rho = 0.0f;       // truncated importance weight (set by recursion_map)
    float adv_next = 0.0f;  // A_{t+1} (set from the scan)
};
// Truncated importance weights and the affine map of the advantage recursion (Section 2.2; Section 3.1).  Returns
// whether the weight exceeded rho_bar.
template <bool kPlain>
__device__ __forceinline__ bool step_map(Step& s, const LossScalars& k, float& a, float& b) {
    const float x = fmaf(-s.l_worker, kLog2e, (!kPlain && k.is_source == 1) ? s.l2_theta : s.l2_target);
    const float w = (!kPlain && k.is_source == 2) ? 1.0f : dev::exp2_fast(x);  // 2: plain GAE, no importance weights
    const float rho = fminf(k.rho_bar, w);
    s.rho = rho;
    const float c = fminf(k.c_bar, w);
    b = __fmul_rn(rho, __fadd_rn(fmaf(s.discount, s.value_next, s.reward), -s.value));
    a = s.ends ? 0.0f : __fmul_rn(__fmul_rn(k.lambda_, s.discount), c);
    return w > k.rho_bar;
}
// Ratio of Section 4.1 and the eps-clipped surrogate of Appendix E.  Returns the weight adv * R of the policy-gradient
// term (0 where the clip removes it).
template <bool kPlain>
__device__ __forceinline__ float step_surrogate(const Step& s, const LossScalars& k, float adv, float& surr, float& ratio,
                                                bool& clipped) {
    if (!kPlain && k.objective == 1) {
        // IMPALA's actor update (Section 2.2): weight rho_t (r_t + gamma_t v_{t+1} - V_t) on
        // grad log pi_theta, v the V-trace target V + A (the bootstrap value after the last step)
        const float v_next = s.value_next + (s.ends ? 0.0f : s.adv_next);
        const float w = __fmul_rn(s.rho, __fadd_rn(fmaf(s.discount, v_next, s.reward), -s.value));
        surr = __fmul_rn(w, s.l2_theta * kLn2);
        ratio = s.rho;
        clipped = false;
        return w;
    }
    const float over_target = s.l2_theta - s.l2_target, over_worker = fmaf(-s.l_worker, kLog2e, s.l2_theta);
    float y = fminf(over_target, over_worker + k.log2_rho_tw);  // over the larger of the two
    if (!kPlain) {
        if (k.ratio_mode == 1) y = over_target;
        else if (k.ratio_mode == 2) y = over_worker;
    }
    const float R = dev::exp2_fast(y);
    const float Rc = fminf(fmaxf(R, k.clip_lo), k.clip_hi);
    const float Ra = __fmul_rn(R, adv);
    surr = fminf(Ra, __fmul_rn(Rc, adv));
    clipped = (adv > 0.0f && R > k.clip_hi) || (adv < 0.0f && R < k.clip_lo);
    ratio = R;
    return clipped ? 0.0f : Ra;
}

// ---- shape of the row passes ------------------------------------------------------------------------------------
// kA > 0: the action count, known at compile time (1 to 32); a row belongs to one lane, which keeps its exponentials.
// kA < 0: any count above 32; a row belongs to L = 2 ... 16 lanes with -kA vectors each (vector i of lane g is the row's
//   vector i L + g), known at compile time, of which the last one, for single pairs the last two, may not be there.  A warp
//   works on 32 / L rows at once, in one pass or in two; row q P + p of the warp is worked on in pass p of P by lanes
//   [q L, q L + L) and owned -- for everything that is per step -- by lane q L + p of them, so results never move between
//   lanes.  (Told at run time how many vectors a lane has, up to 32 elements, a warp took 2340 instructions for 32 rows of 64
//   actions in bf16; so 1760 in one pass, 1500 in two: a million steps 124 -> 86 -> 80 us.)
//
// Rows keep their dense layout in shared memory.  kV = 4 or 2: elements per access, where they divide the count.
// kV = 1 stands for odd counts: a row is then one element and pairs, the element in front where the row starts on an odd
// one (so that the pairs are aligned) and behind where it starts on an even one.  (fp32 and a count known at compile
// time: element by element -- such rows meet on no bank, their pairs on two; 250 000 steps of 9 actions with every
// switch in use take 11.8 us instead of 12.4.)  Where rows meet on the same banks
// (pitches with a large power of two), lanes take their vectors in rotated order; maxima and sums do not mind.
__host__ __device__ constexpr bool is_atari(int A) { return A == 4 || A == 6 || A == 9 || A == 18; }
// Trajectories of 2^32 steps and more that no room for aggregates lets split: with more actions than this they are wider
// than any device's memory.
constexpr int kLongestRows = 3;

// The record of impact_buffer_device_step, read past L1 (an earlier launch may have left an older version there).
__device__ __forceinline__ LossInputPointers fetch_loss_inputs(const impact_loss_inputs* rec) {
    const ulonglong2* q = reinterpret_cast<const ulonglong2*>(rec);
    const ulonglong2 a = __ldcg(q), b = __ldcg(q + 1), c = __ldcg(q + 2), d = __ldcg(q + 3);
    const unsigned long long e = __ldcg(reinterpret_cast<const unsigned long long*>(q + 4));
    LossInputPointers in;
    in.learner_logits = reinterpret_cast<const void*>(a.x);
    in.target_logits = reinterpret_cast<const void*>(a.y);
    in.worker_logp = reinterpret_cast<const float*>(b.x);
    in.actions = reinterpret_cast<const int32_t*>(b.y);
    in.rewards = reinterpret_cast<const float*>(c.x);
    in.discounts = reinterpret_cast<const float*>(c.y);
    in.values = reinterpret_cast<const float*>(d.x);
    in.bootstrap = reinterpret_cast<const float*>(d.y);
    in.target_copy = reinterpret_cast<void*>(e);
    return in;
}

// kPlain: the configuration of the paper's experiments -- no KL term, the clipped surrogate with the default ratio and
// importance weights, no optional outputs -- with those branches compiled out.
//
// kKeepLearner: the gradient pass finds the learner row's exponentials in registers, and there is one pass.  Else it forms them
// again, there may be two, and the forms with every switch have registers enough (with the exponentials kept: 0.82 to 0.9 of
// the rate).
template <typename LT, typename GT, int kA, int C, int kV, bool kPlain, bool kLong, bool kIndirect, bool kKeepLearner>
__global__ void __launch_bounds__(C * 128 + 32, 1)
impact_loss_categorical_kernel(const __grid_constant__ CatParams p, const __grid_constant__ LaunchForm sh) {
    constexpr bool kWide = kA < 0;
    constexpr bool kRotated = kV == 4 && (kWide || kA % 8 == 0);  // (rows of 4 and 12 actions meet on no bank)
    constexpr bool kSingles = kV == 1 && !kWide && sizeof(LT) == 4;  // rows element by element
    constexpr bool kOdd = kV == 1 && !kSingles;
    constexpr int VW = kV == 1 ? 2 : kV;  // elements of a vector
    constexpr int NV = kWide ? -kA : kA / VW;  // vectors per lane
    constexpr int NP = NV * VW / 2 + (kV == 1 ? 1 : 0);  // pairs: Blackwell's packed fp32 add / mul / fma work on two at once
    constexpr float kLowest = -3.402823466e38f;  // stands for an element that is not there: its exponential is 0
    constexpr int kSure = kWide ? (kV == 4 ? NV - 1 : NV - 2) : NV;  // vectors that are there whatever the lane
    static_assert(kWide || kA % VW == (kV == 1 ? 1 : 0), "whole vectors");
    // The KL term from the target row's own exponentials, kept for the gradient pass too, instead of formed twice again
    // (with the KL term, 100 MB: 7 actions in fp32 25.5 -> 24.9 us, 12 in bf16 20.7 -> 19.2, 14 19.9 -> 18.3).  Not where the
    // registers run short -- 96, the learner's exponentials among them: more actions, the split forms -- nor at 8 to 14
    // actions in fp32, where the term gains 0 to 3 % and calls without it lose as much.
    constexpr bool kKeepTarget = !kWide && !kPlain && !kLong && kA <= (sizeof(LT) == 2 ? 14 : 7);
    const int A = kWide ? p.A : kA;
    const int NT = kWide ? sh.nt : 128;
    const int NTW = NT >> 2;  // rows of a tile that one warp works on
    const int S = sh.stages, W = sh.in_flight;
    const int in_row = A * (int)sizeof(LT), out_row = A * (int)sizeof(GT);
    const int in_pitch = (int)slab_pitch(NT, in_row);
    const int stage_bytes = (int)cat_stage_bytes(NT, A, sizeof(LT), sizeof(GT));

    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kWsMaxStages], empty_bar[kWsMaxStages];
    __shared__ __align__(8) uint64_t mail[kMailSlots];
    __shared__ unsigned int tickets_s, tag_s;  // (see dev::draw_ticket_and_publish)
    __shared__ float2 warp_agg[C][2][4];       // (two sets, used in turn: a tile's scan has one barrier)
    __shared__ __align__(16) float red[C][4][8];
    __shared__ int abort_s;
    __shared__ float carry_s[C];

    const int tid = threadIdx.x, lane = tid & 31;
    const LossScalars& k = p.k;
    const BatchGeometry& g = p.geo;
    const BlockRange br = block_range(g);
    const int n_tiles = tiles_of_block(g, br, kLong);
    const long long total_rows = g.B * g.T;
    // The tensors this launch reads: the call's own arguments (kernel parameters, read where they are used), or --
    // kIndirect: the call names a record in device memory that an earlier kernel of the stream fills (the circular
    // buffer's bookkeeping on the device) -- that record's, fetched once the stream dependency has resolved and kept
    // in shared memory (the producer warp alone fetches the record, before the block-wide barrier that releases the
    // consumer warps: with every warp of the grid fetching it -- 3 000 warps asking one cache line at the same
    // moment -- the first tile was requested 3.6 us late)
    __shared__ LossInputPointers in_s;
#define IMPACT_IN(field) (kIndirect ? in_s.field : p.field)

    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (known to be the same for the whole warp)
    if (warp >= C * 4) {
        // ---- producer warp ----------------------------------------------------------------------------------
        const int n_first = n_tiles < W ? n_tiles : W;
        // First of all, while the kernel before this one on the stream is still finishing, the warp asks L2 for
        // the block's first tiles (logits and per-step scalars), unless the launch's companion kernel has done so
        // already: the pages are mapped and the bytes on their way when the dependency resolves.
        if (sh.n_prefetch > 0) {
            const void* base = nullptr;
            long long pitch = 4;
            if (lane == 0) { base = IMPACT_IN(learner_logits); pitch = in_row; }
            else if (lane == 1) { base = IMPACT_IN(target_logits); pitch = in_row; }
            else if (lane == 2) base = IMPACT_IN(actions);
            else if (lane == 3) base = IMPACT_IN(worker_logp);
            else if (lane == 4) base = IMPACT_IN(rewards);
            else if (lane == 5) base = IMPACT_IN(discounts);
            else if (lane == 6) base = IMPACT_IN(values);
            if (lane >= sh.prefetch_arrays) base = nullptr;
            ask_for_tiles<kLong, 2>(g, br, base, pitch, n_tiles < sh.n_prefetch ? n_tiles : sh.n_prefetch, NT, total_rows);
        }
        // then the barriers
        if (lane < S) {
            dev::mbarrier_init_nofence(&full_bar[lane], 1);
            dev::mbarrier_init_nofence(&empty_bar[lane], 4);  // one arrival per consumer warp
        }
        mail[lane] = 0ull;
        if (lane == 0) { abort_s = 0; tickets_s = 0u; }
        dev::fence_mbarrier_init();
        __syncwarp();

        // One slab of a tile into stage s: a bulk copy of the 16-byte granules that enclose the tile's rows
        // (dev::widen_range).  The lane with the learner's slab makes the barrier's one arrival, announcing the
        // bytes of both slabs; where the tensors end inside the last granule, it also fetches that granule's bytes
        // of both slabs by ordinary loads, fenced towards the copy engine because the consumers may send the target
        // rows on from the stage by a bulk store.
        const long long tensor_bytes = total_rows * in_row;
        struct SlabRequest {
            unsigned char* d0;        // the learner's slab of the stage (the target's lies in_pitch further)
            const unsigned char* gl;  // first granule of the tile in the learner's logits
            const unsigned char* gt;  // ... in the target's
            uint32_t span, tail;      // dev::WideRange
        };
        auto request_for = [&](int n, int s) {
            const Tile t = tile_at<kLong>(g, br, n, NT);
            const dev::WideRange w = dev::widen_range(t.row0 * (long long)in_row, (uint32_t)t.nrows * in_row, tensor_bytes);
            SlabRequest r;
            r.d0 = smem_raw + s * stage_bytes;  // the tile's first row starts (row0 * in_row) mod 16 bytes in
            r.gl = static_cast<const unsigned char*>(IMPACT_IN(learner_logits)) + w.first;
            r.gt = static_cast<const unsigned char*>(IMPACT_IN(target_logits)) + w.first;
            r.span = w.span;
            r.tail = w.tail;
            return r;
        };
        auto send_slab = [&](const SlabRequest& r, int s, bool target) {
            uint64_t* const bar = &full_bar[s];
            if (target) {
                if (r.span) dev::bulk_load(r.d0 + in_pitch, r.gt, r.span, bar);
                return;
            }
            if (r.tail) {
                for (uint32_t i = 0; i < r.tail; ++i) {
                    r.d0[r.span + i] = r.gl[r.span + i];
                    r.d0[in_pitch + r.span + i] = r.gt[r.span + i];
                }
                dev::fence_async_shared();
            }
            if (r.span) {
                dev::mbarrier_expect_tx(bar, 2 * r.span);
                dev::bulk_load(r.d0, r.gl, r.span, bar);
            } else {
                dev::mbarrier_arrive(bar);
            }
        };
        // Tiles leave in rounds: lane l < 16 owns the round's l-th tile and requests its learner slab, lane l + 16
        // requests the same tile's target slab, so that all requests of a round leave in the same few instructions
        // (one thread gets at most four bulk requests under way, and needs about a third of a microsecond per
        // tile; a lane per request reaches the HBM rate).
        const int sub = lane & 15;
        const bool second = lane >= 16;
        // the first W tiles need no wait (tile n goes to stage n): their requests are worked out now and leave the
        // moment the stream's previous kernel is done, before the rest of the block has even started
        SlabRequest first = request_for(sub < n_first ? sub : 0, sub);

        grid_dependency_wait();

        if (kIndirect) {  // (the addresses were not known before)
            if (lane == 0) in_s = fetch_loss_inputs(p.indirect);
            __syncwarp();
            first = request_for(sub < n_first ? sub : 0, sub);
        }
        if (sub < n_first) send_slab(first, sub, second);
        __syncthreads();  // the barriers are set up: the consumer warps may use them
        const unsigned int tag = dev::launch_tag(p.counter);  // (asked for now, needed after the last tile has left)
        // The rest.  Tile n goes to stage n % S once that stage's previous tile has left (the "empty" phase before
        // this one) and tile n - W has landed (at most W tiles in flight).  The owners look at their barriers side by
        // side (one thread taking tile after tile through blocking waits costs a third of a microsecond per tile, too
        // much for small tiles: measured 33 us against 25 us on a million steps of six actions), but a tile is sent
        // only when every earlier tile of the round has been sent or is sent in the same instruction: tiles leave in
        // order.
        const int lanes = sh.lanes;
        for (int base = n_first; base < n_tiles; base += lanes) {
            const int n = base + sub;
            bool pending = sub < lanes && n < n_tiles;
            const int cyc = n / S, s = n - cyc * S;
            const int wcyc = (n - W) / S, ws = (n - W) - wcyc * S;
            const SlabRequest req = request_for(pending ? n : 0, s);
            for (unsigned int spin = 0; spin < (1u << 22); ++spin) {
                const bool ready = !second && pending && (cyc == 0 || dev::mbarrier_test(&empty_bar[s], (uint32_t)(cyc - 1) & 1u)) &&
                                   dev::mbarrier_test(&full_bar[ws], (uint32_t)wcyc & 1u);
                const unsigned int waiting = __ballot_sync(0xffffffffu, !second && pending && !ready);
                bool go = ready && (waiting & ((1u << sub) - 1u)) == 0u;
                go = __shfl_sync(0xffffffffu, go, sub);  // the owner decides for both lanes of its tile
                if (go && pending) {
                    send_slab(req, s, second);
                    pending = false;
                }
                if (!__any_sync(0xffffffffu, pending)) break;
                if (*reinterpret_cast<volatile int*>(&abort_s)) break;
                __nanosleep(32);
            }
            if (__any_sync(0xffffffffu, pending)) {  // a stage never came back, or a tile never landed
                if (lane == 0) {
                    atomicExch(p.counter + 1, 1u);
                    *reinterpret_cast<volatile int*>(&abort_s) = 1;
                }
                break;
            }
        }
        __syncwarp();
        // ---- then it leaves this launch's tag for whoever publishes the block's sums, and draws its own ticket
        if (lane == 0) tag_s = tag;
        dev::draw_ticket_and_publish<C, 4>(&tickets_s, &tag_s, red, p.tagged_rows);
        return;
    }

    // ---- consumer groups ------------------------------------------------------------------
    // What is the same for a whole warp (the tile, the stage, addresses) is kept apart from what differs by lane, so
    // that it is worked out once per warp: a tile costs about as many instructions outside the row passes as in them.
    const int grp = warp >> 2, gwarp = warp & 3;
    const int gtid = gwarp * 32 + lane;
    const int bar_id = grp + 1;
    const int wrow = gwarp * NTW;  // the warp's first row in a tile
    const bool want_kl = !kPlain && (k.kl_coef != 0.0f);

    // the lane's part in the row passes (wide: see above), and the row of a tile that it owns
    const int log_l = kWide ? sh.log_lanes : 0;
    const int L = 1 << log_l;
    const int part = kWide ? (lane & (L - 1)) : 0;
    const int passes = kKeepLearner ? 1 : sh.passes;
    const int my_rows = wrow + (lane >> log_l) * passes;  // the rows that the lane works on: one in each pass
    const bool owner = part < passes;
    // (a lane that owns no row stands for the one after it: the identity map, in that row's trajectory)
    const int lrow = my_rows + (passes == 1 ? (owner ? 0 : 1) : min(part, passes));
    const int row_vecs = A / VW;  // vectors of a row (odd counts: and one element)
    const int rot = kRotated ? ((lane >> log_l) >> sh.rot_shift) & sh.rot_mask : 0;

    // The tile (in a flat launch only a block's first tile ends early, only its last one can begin late, and from one of
    // the group's tiles to its next, C tiles further back, every position changes by a constant).
    auto tile_now = [&](int n) { return tile_rows<kLong>(g, br, n, n_tiles, NT, blockIdx.x, gridDim.x); };
    const unsigned int back = (unsigned int)(C * NT);
    TileRows tl = tile_now(grp);
    // (flat) the place of the lane's step
    using Steps = typename std::conditional<!kWide && kA <= kLongestRows && !kPlain, unsigned long long, unsigned int>::type;
    const Steps Tn = (Steps)g.T;
    const unsigned int back_traj = kLong ? 0u : (unsigned int)(back / Tn);
    const Steps back_rest = kLong ? (Steps)0 : back - back_traj * Tn;
    StepPlace<Steps> at = {0, 0};
    if constexpr (!kLong) at = step_place(br, tl.row0 + lrow, Tn);
    auto to_next_tile = [&](int n_next) {
        if constexpr (kLong) {
            tl = tile_now(n_next);
        } else {
            tl.row0 -= back;
            tl.lo = n_next == n_tiles - 1 ? (int)(br.r0 - br.base) : 0;
            tl.hi = NT;
            step_back(at, back_traj, back_rest, Tn);
        }
    };
    auto is_mine = [&](const TileRows& t) { return owner && lrow >= t.lo && lrow < t.hi; };
    auto ends_here = [&](const TileRows& t) { return kLong ? (t.r == 0 && lrow == t.hi - 1) : at.to_end == 0; };

    struct StepRaw {
        int a;
        float l_worker, reward, discount, value, value_next;
    };
    auto load_scalars = [&](const TileRows& t, bool inner) {
        StepRaw x;
        // (loads that name the global space: a pointer taken from the device record is a generic one to the
        // compiler, and a generic load has to be complete before the next store to shared memory -- that put the
        // whole trip to L2 into every tile, 10.9 us a launch against 6.8)
        auto fetch = [&]() {
            x.a = __ldg(IMPACT_IN(actions) + t.row0 + lrow);
            x.l_worker = __ldg(IMPACT_IN(worker_logp) + t.row0 + lrow);
            x.reward = __ldg(IMPACT_IN(rewards) + t.row0 + lrow);
            x.discount = __ldg(IMPACT_IN(discounts) + t.row0 + lrow);
            const float* const v = IMPACT_IN(values) + t.row0 + lrow;
            x.value = __ldg(v);
            x.value_next = __ldg(ends_here(t) ? IMPACT_IN(bootstrap) + (kLong ? t.traj : br.traj0 + (long long)at.traj) : v + 1);
        };
        if (inner) {  // every row is there, and so is the one after the last
            fetch();
        } else {
            x.a = 0; x.l_worker = 0.0f; x.reward = 0.0f; x.discount = 0.0f; x.value = 0.0f; x.value_next = 0.0f;
            if (is_mine(t)) fetch();
        }
        return x;
    };
    // (a lane that owns no row reads that of the row it stands for, which may be the first of the next tile)
    auto is_inner = [&](const TileRows& t, int n) { return !kLong && !kWide && rows_unguarded(t, n, n_tiles); };

    float t_surr = 0.0f, t_val = 0.0f, t_ent = 0.0f, t_ratio = 0.0f, t_kl = 0.0f;
    int n_clip = 0, n_trunc = 0;
    // The group's sums, once final: a butterfly per warp into `red`, then the warp's ticket; the last ticket of
    // the block publishes its row (fixed order throughout).
    auto hand_over_sums = [&]() {
        dev::hand_over_warp_sums<C, 4>(t_surr, t_val, t_ent, t_ratio, t_kl, want_kl,
                                       __reduce_add_sync(0xffffffffu, n_clip), __reduce_add_sync(0xffffffffu, n_trunc),
                                       red[grp][gwarp], &tickets_s, &tag_s, red, p.tagged_rows);
    };

    const bool reuse = n_tiles > S;  // a block with no more tiles than stages never needs a stage back
    // a warp's rows of a whole tile lie on 16-byte boundaries (flat: tiles are nt rows apart)
    const uint32_t m_in0 = ((uint32_t)br.base * (uint32_t)in_row) & 15u, m_out0 = ((uint32_t)br.base * (uint32_t)out_row) & 15u;
    const bool rows_aligned = ((((kLong ? 0 : (int)(br.base & 15)) * out_row) | (NTW * out_row)) & 15) == 0 &&
                              (!kLong || ((g.T * out_row) & 15) == 0);

    grid_dependency_wait();
    StepRaw cur;
    if (!kIndirect) cur = load_scalars(tl, is_inner(tl, grp));
    __syncthreads();  // the producer warp has set up the barriers (and fetched the device record)
    if (kIndirect) cur = load_scalars(tl, is_inner(tl, grp));
    // (long, wide rows) this launch's tag, for the warps that exchange aggregates: asked for once, behind the first tile's
    // scalars (the word changes only after every block has handed its sums over).  Asked for where it is needed, a trip to L2
    // lies between a tile's scan and its aggregate and another before the later tiles' are looked at.  (Only here: the other
    // split forms have no register left for it and take up to a sixth longer; and asked for by every warp of the grid at the
    // start, the one line is served 2 us late.)
    constexpr bool kTagKept = kLong && kWide;
    const unsigned int kept_tag = kTagKept && gwarp == 0 ? dev::launch_tag(p.counter) : 0u;
    auto tag = [&]() { return kTagKept ? kept_tag : dev::launch_tag(p.counter); };
    int s = grp % S, s_prev = 0;
    uint32_t ph = (uint32_t)(grp / S) & 1u;
    int turn = 0;  // which of the group's two sets of warp aggregates this tile uses

    for (int n = grp; n < n_tiles; n += C) {
        // this warp's previous rows have left shared memory: hand the stage back.  (Only where stages are used
        // more than once: the wait for the store's reads sits between two tiles of the warp.)
        if (reuse && n != grp) hand_back_stage(&empty_bar[s_prev], lane);
        // (long) one early look at the aggregates of the later tiles of this tile's trajectory: with many
        // trajectories they were published a round ago, and reading them now keeps that trip to L2 off the path
        // between this tile's scan and its gradients (only where tiles are numbered tile-major; the values are first
        // looked at after the scan)
        const long long gtile = (long long)blockIdx.x + (long long)n * gridDim.x;
        const long long tile_stride = g.tile_major ? g.B : 1;  // from a tile to the one after it in time (and two slots to each)
        // (rows of several lanes are never split where there are as many trajectories as blocks)
        const bool peeked = kLong && !kWide && g.tile_major && gwarp == 0 && tl.r > lane;
        unsigned long long early_a = 0, early_b = 0;
        if (peeked) dev::load_aggregate(p.tile_aggregates + 2 * gtile, 2 * tile_stride, tl.r - lane, early_a, early_b);
        // every thread waits for the stage itself (a bounded wait: on a time-out the flag is set and the
        // thread goes on with whatever the stage holds, so that all barriers below still pair up)
        if (!stage_wait(&full_bar[s], ph, &abort_s)) atomicExch(p.counter + 1, 1u);

        // rows keep their place inside their 16-byte granule: the tile's first row starts (row0 * pitch) mod 16
        // bytes into the slab
        unsigned char* const stage = smem_raw + s * stage_bytes;
        // (flat: tiles are a multiple of eight rows apart, so this is the same for all of the block's)
        const uint32_t m_in = kLong ? ((uint32_t)tl.row0 * (uint32_t)in_row) & 15u : m_in0;
        const uint32_t m_out = (sizeof(LT) == sizeof(GT)) ? m_in : (kLong ? ((uint32_t)tl.row0 * (uint32_t)out_row) & 15u : m_out0);
        unsigned char* const s0 = stage + m_in;    // learner logits
        unsigned char* const s1 = s0 + in_pitch;   // target logits
        unsigned char* const so = (sizeof(LT) == sizeof(GT)) ? s0 : stage + 2 * in_pitch + m_out;
        // (first traversal of a batch) the target rows go to the circular buffer as well, each warp's rows
        // straight from the stage, which nothing writes to
        if (IMPACT_IN(target_copy))
            send_rows_general(static_cast<unsigned char*>(IMPACT_IN(target_copy)) + tl.row0 * (long long)in_row, s1,
                              in_row, wrow, NTW, tl.lo, tl.hi, false);

        // ---- row passes (every lane; rows that are not the tile's hold stale bytes and are masked)
        float2 e[kKeepLearner ? NP : 1];  // the learner row's exponentials, kept for the gradient pass
        float2 et[kKeepTarget ? NP : 1];  // (KL term) the target row's
        // Per row: log2 e times the largest logit (m2), log2 of the exponentials' sum (lg); learner: 1 / that sum and the
        // mean logit.  m2 and lg are kept apart: adding them first would round their sum, the largest of the numbers
        // that a log-probability is made of.
        float m2_t = 0.0f, lg_t = 0.0f, m2_l = 0.0f, lg_l = 0.0f, inv_s = 0.0f, mean_z = 0.0f, ent = 0.0f, kl = 0.0f, inv_t = 0.0f;
        // byte offset of the lane's i-th vector from the row's first (of `elem`-byte elements)
        auto vec_at = [&](int i, int elem) {
            const int step = (VW * elem) << log_l;
            return kRotated ? ((i * step) ^ (rot * step)) : i * step;
        };
        auto vec_there = [&](int i) { return i < kSure || (i << log_l) + part < row_vecs; };
        // (odd counts) does the row start on an odd element?  Tiles are an even number of rows apart.
        const uint32_t tile_odd = kOdd ? (uint32_t)(kLong ? tl.row0 : br.base) & 1u : 0u;
        auto first_of = [&](int r) { return kOdd ? (int)((tile_odd + (uint32_t)r) & 1u) : 0; };  // of the vectors
        auto single_of = [&](int r) { return first_of(r) ? 0 : A - 1; };                         // the element beside them
        auto load_row = [&](const unsigned char* slab, int r, float2 (&z)[NP]) {
            const unsigned char* const row = slab + r * in_row;
            const unsigned char* const at = row + (first_of(r) + part * VW) * (int)sizeof(LT);
            float f[2 * NP];
#pragma unroll
            for (int j = 0; j < 2 * NP; ++j) f[j] = kLowest;
            if constexpr (kSingles) {
#pragma unroll
                for (int j = 0; j < kA; ++j) f[j] = get_element<LT>(row, j);
            }
#pragma unroll
            for (int i = 0; i < NV && !kSingles; ++i) {
                // (a vector that is not there: the lane's first, read again and left out)
                const bool there = vec_there(i);
                Vec<LT, VW>::ld(at + (there ? vec_at(i, (int)sizeof(LT)) : 0), f + i * VW);
#pragma unroll
                for (int v = 0; v < VW; ++v) f[i * VW + v] = there ? f[i * VW + v] : kLowest;
            }
            if (kOdd && (!kWide || part == 0)) f[2 * NP - 2] = get_element<LT>(row, single_of(r));
#pragma unroll
            for (int j = 0; j < NP; ++j) z[j] = make_float2(f[2 * j], f[2 * j + 1]);
        };
        auto row_max = [&](const float2 (&z)[NP]) {
            float m0 = fmaxf(z[0].x, z[0].y), m1 = m0;
#pragma unroll
            for (int j = 1; j < NP; ++j) {
                if (j & 1) m1 = fmaxf(m1, fmaxf(z[j].x, z[j].y));
                else m0 = fmaxf(m0, fmaxf(z[j].x, z[j].y));
            }
            return fmaxf(m0, m1);
        };
        const float2 log2e2 = make_float2(kLog2e, kLog2e);
#pragma unroll 1
        for (int pass = 0; pass < passes; ++pass) {
            const int r = my_rows + pass;
            float2 z[NP];
            // target row
            load_row(s1, r, z);
            float m_t = row_max(z);
            if (kWide) for (int o = 1; o < L; o <<= 1) m_t = fmaxf(m_t, __shfl_xor_sync(0xffffffffu, m_t, o));
            const float m2t = __fmul_rn(m_t, kLog2e);
            float2 sum2 = make_float2(0.0f, 0.0f);
            {
                const float2 neg_m2 = make_float2(-m2t, -m2t);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 t2 = __ffma2_rn(z[j], log2e2, neg_m2);  // (z - m) log2 e
                    const float2 ex = make_float2(dev::exp2_fast(t2.x), dev::exp2_fast(t2.y));
                    sum2 = __fadd2_rn(sum2, ex);
                    if constexpr (kKeepTarget) et[j] = ex;
                }
            }
            float sum_t = sum2.x + sum2.y;
            // learner row: also sum_j e_j z_j
            load_row(s0, r, z);
            float m_l = row_max(z);
            if (kWide) for (int o = 1; o < L; o <<= 1) m_l = fmaxf(m_l, __shfl_xor_sync(0xffffffffu, m_l, o));
            const float m2 = __fmul_rn(m_l, kLog2e);
            sum2 = make_float2(0.0f, 0.0f);
            float2 sez2 = make_float2(0.0f, 0.0f);
            {
                const float2 neg_m2 = make_float2(-m2, -m2);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 t2 = __ffma2_rn(z[j], log2e2, neg_m2);
                    const float2 ex = make_float2(dev::exp2_fast(t2.x), dev::exp2_fast(t2.y));
                    sum2 = __fadd2_rn(sum2, ex);
                    sez2 = __ffma2_rn(ex, z[j], sez2);
                    if constexpr (kKeepLearner) e[j] = ex;
                }
            }
            float sum_l = sum2.x + sum2.y, sez = sez2.x + sez2.y;
            if (kWide) {
                for (int o = 1; o < L; o <<= 1) {
                    sum_t += __shfl_xor_sync(0xffffffffu, sum_t, o);
                    sum_l += __shfl_xor_sync(0xffffffffu, sum_l, o);
                    sez += __shfl_xor_sync(0xffffffffu, sez, o);
                }
            }
            const float lgt = dev::log2_fast(sum_t), lgl = dev::log2_fast(sum_l);
            const float is = dev::reciprocal(sum_l);
            float klr = 0.0f, ist = 0.0f;
            if (want_kl) {
                const unsigned char* const row = s1 + r * in_row;
                const unsigned char* const at = row + (first_of(r) + part * VW) * (int)sizeof(LT);
                auto target_vec = [&](int i, float (&zt)[VW]) {
                    if constexpr (kSingles) { zt[0] = get_element<LT>(row, 2 * i); zt[1] = get_element<LT>(row, 2 * i + 1); }
                    else Vec<LT, VW>::ld(at + vec_at(i, (int)sizeof(LT)), zt);
                };
                // (An action masked by the type's lowest value in both rows counts 0 times a finite difference in both forms; in
                // base 2 its log-probabilities overflow and the difference is no number.)
                if constexpr (kKeepTarget) {
                    // KL = sum_j e^t_j ((zt_j - m_t) - (zl_j - m_l)) / S_t + ln S_l - ln S_t.  What the logits of a row have in
                    // common cancels before anything is rounded at its size.  Differences are taken a sixteenth as large,
                    // which rounds nothing: where the learner alone masks actions by the type's lowest value they are as
                    // large as a float gets, and the sum of up to 14 of them, each times at most 1, has to stay one.
                    static_assert(!kKeepTarget || kA <= 16, "sixteenths");
                    constexpr float kPart = 1.0f / 16.0f;
                    float2 skl2 = make_float2(0.0f, 0.0f);
                    const float2 part2 = make_float2(kPart, kPart);
                    const float2 part_t2 = make_float2(-kPart * m_t, -kPart * m_t), part_l2 = make_float2(-kPart * m_l, -kPart * m_l);
                    auto add_kl = [&](const float2& zt, const float2& zl, int pair) {
                        const float2 dt = __ffma2_rn(zt, part2, part_t2), dl = __ffma2_rn(zl, part2, part_l2);
                        skl2 = __ffma2_rn(et[pair], __ffma2_rn(dl, make_float2(-1.0f, -1.0f), dt), skl2);
                    };
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        float zt[VW];
                        target_vec(i, zt);
#pragma unroll
                        for (int v = 0; v < VW; v += 2) add_kl(make_float2(zt[v], zt[v + 1]), z[(i * VW + v) / 2], (i * VW + v) / 2);
                    }
                    if (kV == 1)  // (the pair's other element is in neither row)
                        add_kl(make_float2(get_element<LT>(row, single_of(r)), kLowest), make_float2(z[NP - 1].x, kLowest), NP - 1);
                    ist = dev::reciprocal(sum_t);
                    klr = fmaf(skl2.x + skl2.y, __fmul_rn(ist, 1.0f / kPart), __fmul_rn(lgl - lgt, kLn2));
                } else {  // in natural units, action by action
                    const float lse_t = fmaf(lgt, kLn2, m_t), lse_l = fmaf(lgl, kLn2, m_l);
                    auto add_kl = [&](float zt, float zl) {
                        const float lpt = __fadd_rn(zt, -lse_t);
                        klr = fmaf(dev::exp2_fast(__fmul_rn(lpt, kLog2e)), __fadd_rn(lpt, -__fadd_rn(zl, -lse_l)), klr);
                    };
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        if (!vec_there(i)) continue;
                        float zt[VW];
                        target_vec(i, zt);
#pragma unroll
                        for (int v = 0; v < VW; v += 2) {
                            add_kl(zt[v], z[(i * VW + v) / 2].x);
                            add_kl(zt[v + 1], z[(i * VW + v) / 2].y);
                        }
                    }
                    if (kV == 1 && (!kWide || part == 0)) add_kl(get_element<LT>(row, single_of(r)), z[NP - 1].x);
                    if (kWide) for (int o = 1; o < L; o <<= 1) klr += __shfl_xor_sync(0xffffffffu, klr, o);
                }
            }
            if (kKeepLearner || part == pass) {
                m2_t = m2t; lg_t = lgt; m2_l = m2; lg_l = lgl; inv_s = is; mean_z = __fmul_rn(sez, is); kl = klr; inv_t = ist;
                // H = -sum_j pi_j lp_j = (m - sum_j e_j z_j / S) + ln S: what the logits have in common cancels first
                ent = fmaf(lgl, kLn2, __fadd_rn(m_l, -mean_z));
            }
        }
        // ---- the step's own scalars (its owner lane)
        const int act = min(max(cur.a, 0), A - 1);
        Step st;
        st.l_worker = cur.l_worker;
        st.reward = cur.reward;
        st.discount = cur.discount;
        st.value = cur.value;
        st.value_next = cur.value_next;
        st.ends = ends_here(tl);
        // (kept finite where the taken action is masked by the type's lowest value: its probability is 0 either way)
        st.l2_target = dev::max_or_nan(fmaf(get_element<LT>(s1 + (owner ? lrow : my_rows) * in_row, act), kLog2e, -m2_t) - lg_t, kLowest);
        st.l2_theta = dev::max_or_nan(fmaf(get_element<LT>(s0 + (owner ? lrow : my_rows) * in_row, act), kLog2e, -m2_l) - lg_l, kLowest);
        float fa, fb;
        const bool truncated = step_map<kPlain>(st, k, fa, fb);
        const bool mine = is_mine(tl);
        if (!mine) { fa = 1.0f; fb = 0.0f; }
        // (flat) the slot of the tile, or beyond, where the step's trajectory ends
        const int reach = lrow + (int)min(at.to_end, (Steps)1024);
        int limit = 31 - lane;
        if constexpr (!kLong) {
            const int left = reach - wrow;  // ... counted from the warp's first row
            limit = min(limit, (passes == 1 ? left << log_l : (left / passes << log_l) + left % passes) - lane);
        }

        // the next tile's scalars travel while this tile is worked on
        const TileRows here = tl;
        to_next_tile(n + C);
        if (n + C < n_tiles) cur = load_scalars(tl, is_inner(tl, n + C));

        // ---- the recursion: maps composed from the tile's end
        warp_suffix_compose(fa, fb, limit);
        if (lane == 0) warp_agg[grp][turn][gwarp] = make_float2(fa, fb);
        asm volatile("bar.sync %0, 128;" ::"r"(bar_id) : "memory");
        float adv, after;  // A of the step, and (lane 31) of the step after the warp's last
        if constexpr (!kLong) {
            // what follows the warp's last step, as far as the step's trajectory reaches
            float x = 0.0f;
            // (a lane that owns no row passes the value on to the one before it, as the advantage of the step after it)
            const bool goes_on = (owner ? mine : n > 0) && reach >= NT;
            if (__any_sync(0xffffffffu, goes_on)) {
                const float m = mail_get(mail, n - 1, &abort_s, p.counter + 1);
                x = goes_on ? m : 0.0f;
            }
#pragma unroll
            for (int w = 3; w > 0; --w) {
                const float2 f = warp_agg[grp][turn][w];
                if (w > gwarp && reach >= w * NTW) x = fmaf(f.x, x, f.y);
            }
            adv = fmaf(fa, x, fb);
            after = x;
            if (gtid == 0) mail_put(mail, n, adv);
        } else {
            // maps instead of values: (ma, mb) takes the value that enters the tile's last step to A of this step,
            // (la, lb) to A of the step after this warp's last
            float la = 1.0f, lb = 0.0f;
#pragma unroll
            for (int w = 3; w > 0; --w) {
                const float2 f = warp_agg[grp][turn][w];
                if (w > gwarp) { lb = fmaf(f.x, lb, f.y); la = f.x * la; }
            }
            const float ma = fa * la, mb = fmaf(fa, lb, fb);
            unsigned long long* const slots = p.tile_aggregates + 2 * gtile;
            if (gtid == 0) dev::publish_tile_aggregate(slots, ma, mb, tag());
            float carry = 0.0f;
            if (here.r > 0) {  // uniform over the group
                if (gwarp == 0) {
                    float c;
                    if (kWide && p.block_values)
                        c = dev::value_from_later_tiles(slots, p.block_values + 4 * (here.traj * (g.ntiles / 32)), here.r, ma, mb,
                                                        tag(), &abort_s, p.counter + 1);
                    else
                        c = dev::compose_later_aggregates(slots, 2 * tile_stride, here.r, tag(), &abort_s, p.counter + 1, peeked,
                                                          early_a, early_b);
                    if (lane == 0) carry_s[grp] = c;
                }
                asm volatile("bar.sync %0, 128;" ::"r"(bar_id) : "memory");
                carry = carry_s[grp];
            }
            adv = fmaf(ma, carry, mb);
            after = fmaf(la, carry, lb);
        }
        if constexpr (!kPlain) {
            const float below = __shfl_down_sync(0xffffffffu, adv, 1);
            st.adv_next = (lane == 31) ? after : below;
        }
        turn ^= 1;

        float surr, ratio;
        bool clipped;
        const float wpg = step_surrogate<kPlain>(st, k, adv, surr, ratio, clipped);
        if (mine) {
            t_surr += surr;
            t_val = fmaf(0.5f * adv, adv, t_val);
            t_ent += ent;
            t_ratio += ratio;
            if (!kPlain) t_kl += kl;
            n_clip += clipped ? 1 : 0;  // (per thread; added up over the warp when the sums are handed over)
            n_trunc += truncated ? 1 : 0;
        }
        // the group's sums are final after its last tile's scan: handed over here, they are published while
        // that tile's gradient pass runs
        if (n + C >= n_tiles) hand_over_sums();

        // ---- gradients: row_j = e_j (ga z_j + gb) [- kl_coef pi_target_j / M], then the taken action's entry
        float w1 = __fmul_rn(wpg, k.inv_M);
        if (kWide && kKeepLearner) w1 = __shfl_sync(0xffffffffu, w1, lane & ~(L - 1));  // (the owner's)
        const float ce = k.ent_over_M, ck = kPlain ? 0.0f : k.kl_over_M;
        const float ga = __fmul_rn(ce, inv_s), gb = __fmul_rn(__fadd_rn(fmaf(-ce, mean_z, w1), ck), inv_s);
#pragma unroll 1
        for (int pass = 0; pass < passes; ++pass) {
            const int r = my_rows + pass;
            float pga = ga, pgb = gb, pm2 = m2_l, plt = kPlain ? 0.0f : __fadd_rn(m2_t, lg_t);
            if (!kKeepLearner) {  // (its owner's)
                const int from = (lane & ~(L - 1)) + pass;
                pga = __shfl_sync(0xffffffffu, ga, from);
                pgb = __shfl_sync(0xffffffffu, gb, from);
                pm2 = __shfl_sync(0xffffffffu, m2_l, from);
                if (want_kl) plt = __shfl_sync(0xffffffffu, __fadd_rn(m2_t, lg_t), from);
            }
            const float2 ga2 = make_float2(pga, pga), gb2 = make_float2(pgb, pgb);
            const float2 neg_m2 = make_float2(-pm2, -pm2);
            const float2 neg_lse2 = make_float2(-plt, -plt), nck2 = make_float2(-ck, -ck);
            const float nckt = __fmul_rn(-ck, inv_t);
            const float2 nckt2 = make_float2(nckt, nckt);
            // the gradient of up to VW neighbouring elements: z and zt in, their places among the lane's elements
            auto grad_of = [&](const float2& z2, const float2& zt2, int pair) {
                float2 ex;
                if constexpr (kKeepLearner) {
                    ex = e[pair];
                } else {
                    const float2 t2 = __ffma2_rn(z2, log2e2, neg_m2);
                    ex = make_float2(dev::exp2_fast(t2.x), dev::exp2_fast(t2.y));
                }
                float2 gr = __fmul2_rn(ex, __ffma2_rn(z2, ga2, gb2));
                if (want_kl) {
                    if constexpr (kKeepTarget) {
                        gr = __ffma2_rn(nckt2, et[pair], gr);
                    } else {
                        const float2 tt = __ffma2_rn(zt2, log2e2, neg_lse2);
                        gr = __ffma2_rn(nck2, make_float2(dev::exp2_fast(tt.x), dev::exp2_fast(tt.y)), gr);
                    }
                }
                return gr;
            };
            const unsigned char* const zrow = s0 + r * in_row;
            const unsigned char* const trow = s1 + r * in_row;
            unsigned char* const grow = so + r * out_row;
            const int first = first_of(r) + part * VW;
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                if (!vec_there(i)) continue;
                float z[VW], o[VW], zt[VW];
#pragma unroll
                for (int v = 0; v < VW; ++v) zt[v] = 0.0f;
                if constexpr (kSingles) {
                    z[0] = get_element<LT>(zrow, 2 * i); z[1] = get_element<LT>(zrow, 2 * i + 1);
                    if (!kKeepTarget && want_kl) { zt[0] = get_element<LT>(trow, 2 * i); zt[1] = get_element<LT>(trow, 2 * i + 1); }
                } else {
                    Vec<LT, VW>::ld(zrow + first * (int)sizeof(LT) + vec_at(i, (int)sizeof(LT)), z);
                    if (!kKeepTarget && want_kl) Vec<LT, VW>::ld(trow + first * (int)sizeof(LT) + vec_at(i, (int)sizeof(LT)), zt);
                }
#pragma unroll
                for (int v = 0; v < VW; v += 2) {
                    const float2 gr = grad_of(make_float2(z[v], z[v + 1]), make_float2(zt[v], zt[v + 1]), (i * VW + v) / 2);
                    o[v] = gr.x;
                    o[v + 1] = gr.y;
                }
                if constexpr (kSingles) {
                    Vec<GT, 1>::st(grow + 2 * i * (int)sizeof(GT), o);
                    Vec<GT, 1>::st(grow + (2 * i + 1) * (int)sizeof(GT), o + 1);
                } else {
                    Vec<GT, VW>::st(grow + first * (int)sizeof(GT) + vec_at(i, (int)sizeof(GT)), o);
                }
            }
            if (kV == 1 && (!kWide || part == 0)) {
                const int c = single_of(r);
                const float z = get_element<LT>(zrow, c), zt = !kKeepTarget && want_kl ? get_element<LT>(trow, c) : 0.0f;
                put_element<GT>(grow, c, grad_of(make_float2(z, z), make_float2(zt, zt), NP - 1).x);
            }
        }
        const float pi_a = dev::exp2_fast(st.l2_theta);
        float g_a = fmaf(pi_a, fmaf(ce, fmaf(st.l2_theta, kLn2, ent), w1), -w1);
        if (want_kl) g_a = fmaf(ck, pi_a - dev::exp2_fast(st.l2_target), g_a);
        if (mine) {
            p.dvalues[here.row0 + lrow] = __fmul_rn(k.dvalue_over_adv, adv);  // V - Vhat = -A
            if (!kPlain) {
                if (p.vtarget) p.vtarget[here.row0 + lrow] = st.value + adv;
                if (p.advantage) p.advantage[here.row0 + lrow] = adv;
            }
        }
        if (kWide) __syncwarp();  // (other lanes wrote the row that this one corrects)
        if (owner) put_element<GT>(so + lrow * out_row, act, g_a);
        // ---- each warp sends its own rows: no barrier across the group
        {
            unsigned char* const out = static_cast<unsigned char*>(p.dlogits) + here.row0 * (long long)out_row;
            if (here.lo == 0 && here.hi == NT && rows_aligned) {  // whole granules: the usual case
                dev::fence_async_shared();
                __syncwarp();
                if (lane == 0) dev::bulk_store(out + wrow * out_row, so + wrow * out_row, (uint32_t)(NTW * out_row));
            } else {
                send_rows_general(out, so, out_row, wrow, NTW, here.lo, here.hi, true);
            }
        }
        s_prev = s;
        s += C;
        if (s >= S) { s -= S; ph ^= 1u; }  // (C <= S wherever a group has a second tile)
    }

    // a group without tiles still hands over its (zero) sums, so that every row of the grid is defined
    if (grp >= n_tiles) hand_over_sums();
    // ---- one group of the grid (block 0's, the one that runs out of tiles first and so is polling long before the
    // last rows appear) collects every block's row as it appears and writes the loss terms
    // (in fp64, but for the Atari action sets on trajectories that fit a tile or are split, which add in fp32 as they
    // always did: fp64 costs 0.15 to 0.3 us at the end of a launch)
    if (blockIdx.x == 0 && grp == n_tiles % C) {
        auto collect = [&](auto zero) {
            if (!dev::reduce_tagged_rows<128, decltype(zero)>(p.tagged_rows, (int)gridDim.x, dev::launch_tag(p.counter),
                                                              p.counter, p.loss_terms, k.vf_coef, k.ent_coef, k.kl_coef,
                                                              k.steps_total, gtid, bar_id, &abort_s))
                if (gtid == 0) atomicExch(p.counter + 1, 1u);
        };
        if (!is_atari(kA) || (!kLong && g.T > 128)) collect(0.0);
        else collect(0.0f);
    }
    if (lane == 0) dev::bulk_store_wait_read();  // shared memory must outlive the stores' reads
#undef IMPACT_IN
}

// ------------------------------------------------------------------------------------------
// Launch
// ------------------------------------------------------------------------------------------
template <typename LT, typename GT, int kA, int C, int kV, bool kPlain, bool kLong, bool kIndirect, bool kKeepLearner = true>
int32_t launch_categorical(CatParams p, const RowLayout& rl, const DeviceInfo* di, cudaStream_t stream) {
    const int nt = rl.nt;
    auto kernel = impact_loss_categorical_kernel<LT, GT, kA, C, kV, kPlain, kLong, kIndirect, kKeepLearner>;
    const size_t stage = cat_stage_bytes(nt, p.A, sizeof(LT), sizeof(GT));
    LaunchShape ls;
    if (!launch_shape(p.geo, nt, kLong, stage, 2 * (size_t)nt * p.A * sizeof(LT), C, di, &ls, kIndirect)) return IMPACT_ERR_UNSUPPORTED;
    if (kA < 0) p.geo.tile_major = 0;  // (a trajectory's tiles side by side, as value_from_later_tiles looks for them)
    LaunchForm sh = {};
    sh.nt = nt;
    sh.log_lanes = rl.log_lanes;
    sh.passes = rl.passes;
    sh.rot_shift = rl.rot_shift;
    sh.rot_mask = rl.rot_mask;
    sh.stages = ls.stages;
    sh.in_flight = ls.in_flight;
    sh.lanes = ls.lanes;
    const size_t smem = (size_t)sh.stages * stage;
    static thread_local int configured_device = -1;
    static thread_local size_t own_smem = 0;  // (the kernel's static arrays)
    if (configured_device != di->device) {  // once per device: room for the largest ring any window setting asks for
        IMPACT_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, di->max_smem_optin - 4096));
        cudaFuncAttributes a;
        IMPACT_CUDA_TRY(cudaFuncGetAttributes(&a, kernel));
        own_smem = a.sharedSizeBytes;
        configured_device = di->device;
    }
    const size_t row_bytes = 2 * p.A * sizeof(LT) + 20;
    WsPlan plan = ws_plan(ls.tiles, ls.grid, nt * row_bytes, sh.in_flight,
                          companion_pays(p.A, kLong, p.geo.B * p.geo.T, row_bytes, nt, ls.tiles, ls.grid, sh.in_flight, sizeof(GT)));
    if (kIndirect) { plan.companion = false; plan.prefetch_tiles = 0; }  // (addresses unknown on the host)
    if (plan.companion) {
        const int32_t st = launch_companion(p, (int)sizeof(LT), kLong, plan.prefetch_tiles, (int)ls.grid, stream);
        if (st != IMPACT_OK) return st;
    } else {
        const OwnRequests own = own_requests(plan, nt * row_bytes, p.geo.B * p.geo.T, ls.grid, nt, kLong ? 0 : 16 * 1024, kLong ? 0 : 21);
        sh.n_prefetch = kLong && kA > 0 && kA <= 18 ? 0 : own.tiles;
        sh.prefetch_arrays = own.slabs_only ? 2 : 7;
    }
    const int shared_percent = plan.companion ? percent_beside(smem + own_smem, 0, di)
                               : kIndirect    ? percent_beside(smem + own_smem, kRingStepShared, di) : -1;
    IMPACT_CUDA_TRY(launch_laid_out(shared_percent, kernel, dim3((unsigned)ls.grid), dim3(C * 128 + 32), smem, stream, p, sh));
    return IMPACT_OK;
}

// The configuration of the paper's experiments, for which the switches and optional outputs are compiled out.
inline bool is_plain(const CatParams& p) {
    return p.k.kl_coef == 0.0f && p.k.objective == IMPACT_OBJECTIVE_CLIPPED_SURROGATE &&
           p.k.is_source == IMPACT_IS_TARGET_OVER_WORKER && p.k.ratio_mode == IMPACT_RATIO_R3 && !p.vtarget && !p.advantage;
}

// Rows on 2^l lanes each: the rows of a tile, and the rotation that lanes of vectors of four elements take them in, from how a
// warp's rows meet on the banks.
template <typename LT, int kV>
void settle_rows(RowLayout& rl, int A, int l) {
    constexpr int VW = kV == 1 ? 2 : kV;
    rl.log_lanes = l;
    rl.nt = (128 >> l) * rl.passes;
    const int vecs = A / VW;
    const BankPattern b = bank_pattern(A * sizeof(LT) * rl.passes, 1 << l, VW * (int)sizeof(LT));
    rl.rot_mask = 0;
    rl.rot_shift = b.shift;
    if (kV == 4 && vecs % (1 << l) == 0) {
        const int per_lane = vecs >> l;
        while (2 * (rl.rot_mask + 1) <= b.ways && per_lane % (2 * (rl.rot_mask + 1)) == 0) rl.rot_mask = 2 * rl.rot_mask + 1;
    }
}

// Consumer groups: four with every switch compiled in; five in the default configuration; six there for small action
// sets, which are bound by arithmetic, not bytes.  One and two fewer where the rows' exponentials take 19 to 32 registers
// (128 to a thread with three groups, 96 with four).
template <typename LT, typename GT, int A>
int32_t run_fixed(const CatParams& p, const DeviceInfo* di, cudaStream_t stream) {
    constexpr int C = A <= 18 ? 4 : 3, CP = A <= 9 ? 6 : A <= 18 ? 5 : 4, kV = A % 4 == 0 ? 4 : A % 2 == 0 ? 2 : 1;
    const bool plain = is_plain(p), fits = fits_flat(p.geo);
    RowLayout rl;
    settle_rows<LT, kV>(rl, A, 0);
    if (p.indirect) {  // compiled for trajectories that fit a tile only
        if constexpr (is_atari(A)) {
            if (p.geo.T > 128) return IMPACT_ERR_UNSUPPORTED;
            return plain ? launch_categorical<LT, GT, A, CP, kV, true, false, true>(p, rl, di, stream)
                         : launch_categorical<LT, GT, A, C, kV, false, false, true>(p, rl, di, stream);
        }
        return IMPACT_ERR_UNSUPPORTED;
    }
    if (splits_trajectories(p.geo, p.tile_aggregates, 128, di, 0, 0, 0, plain) || (!fits && p.tile_aggregates)) {
        // Where three groups spill as well (100 bytes a thread and more: 30 and 31 actions with fp32 logits; 32 are read four
        // at a time and lose nothing by it) and nearly every block has four tiles, four groups have one each: 16 x 4096 steps of
        // 30 and 31 actions 12.1 and 12.5 us instead of 13.2 and 14.1, with bf16 gradients 11.9 and 12.9 instead of 13.3 and
        // 14.6.  With fewer tiles three have as much to do (14 x 4096 11.4 on four, 10.6 on three), with more they are faster
        // (20 x 4096 17.5 and 14.0).
        if constexpr (A >= 30 && kV < 4 && sizeof(LT) == 4) {
            const long long tiles = p.geo.B * ((p.geo.T + 127) / 128);
            if (5 * tiles > 16 * di->sm_count && tiles <= 4 * di->sm_count)
                return launch_categorical<LT, GT, A, 4, kV, false, true, false>(p, rl, di, stream);
        }
        return launch_categorical<LT, GT, A, C, kV, false, true, false>(p, rl, di, stream);
    }
    if (!fits && A > kLongestRows) return IMPACT_ERR_UNSUPPORTED;
    return plain && fits ? launch_categorical<LT, GT, A, CP, kV, true, false, false>(p, rl, di, stream)
                         : launch_categorical<LT, GT, A, C, kV, false, false, false>(p, rl, di, stream);
}

// How a row of more than 32 actions is laid on lanes: the fewest that hold it in up to 32 elements each (a row costs a lane
// some hundred instructions besides its elements'), and the vectors that this makes a lane's: 5 to 8 of four elements, or 10
// to 16, even numbers of them, of two.
struct WideWidth {
    int log_lanes, vectors;
};
constexpr int wide_elements(int A) { return A % 4 == 0 ? 4 : 2; }  // of a vector
constexpr WideWidth wide_width(int A) {
    const int most = 32 / wide_elements(A), step = most / 8, vecs = A / wide_elements(A);
    WideWidth w = {1, 5};
    while ((most << w.log_lanes) < vecs) ++w.log_lanes;
    while ((w.vectors * step << w.log_lanes) < vecs) ++w.vectors;
    w.vectors *= step;
    return w;
}
// Rows of a tile where a row takes more than a lane: those of one pass of a group's warps or of two, which share what a tile
// costs besides its rows.  Split launches, three groups: two passes where the tiles are enough for every SM (16 x 4096 steps of
// 64 actions in bf16 13.5 us instead of 17.5, of 80 in fp32 20.7 / 28.7; 20 x 300 of 100 7.3 / 6.8) and the ring has a stage for
// every group.  Whole trajectories, four groups: with two tiles to every SM (bf16, 50 actions: 8.0 us instead of 8.8 at 50 000
// steps, 30.8 / 34.6 at 400 000, but 7.0 / 6.4 at 25 000) and two stages more than groups.
inline int wide_tile_rows(const BatchGeometry& g, bool split, int A, size_t in_elem, size_t out_elem, const DeviceInfo* di) {
    const int one = 128 >> wide_width(A).log_lanes, two = 2 * one;
    const int fit = stages_that_fit(cat_stage_bytes(two, A, in_elem, out_elem), di->max_smem_optin);
    if (split) return fit >= 3 && split_tiles(g, two) >= di->sm_count ? two : one;
    return fit >= 6 && g.B * g.T >= 2ll * two * di->sm_count ? two : one;
}

template <typename LT, typename GT, int kV, int NV>
int32_t run_wide_form(const CatParams& p, const DeviceInfo* di, cudaStream_t stream) {
    constexpr int C = 4;
    const int log_lanes = wide_width(p.A).log_lanes, one_pass = 128 >> log_lanes;
    auto laid_out = [&](int rows) {
        RowLayout rl;
        rl.passes = rows / one_pass;
        settle_rows<LT, kV>(rl, p.A, log_lanes);
        return rl;
    };
    if (p.indirect) {
        if constexpr (kV == 4 && NV == 8) {
            if (p.A == 64 && p.geo.T <= 64)
                return launch_categorical<LT, GT, -NV, C, kV, false, false, true, false>(p, laid_out(one_pass), di, stream);
        }
        return IMPACT_ERR_UNSUPPORTED;
    }
    const bool fits = fits_flat(p.geo), plain = is_plain(p);
    // Tiles of few rows keep their maps and their blocks' values in the workspace's spare slots, as do blocks' values alone, where
    // there is room.  (A block of 32 tiles takes four slots.)
    const int nt = wide_tile_rows(p.geo, true, p.A, sizeof(LT), sizeof(GT), di);
    const long long tiles = split_tiles(p.geo, nt);
    const bool room = nt < kMinTileRows ? p.spare_slots && 3 * tiles <= kSpareSlots : p.tile_aggregates != nullptr;
    if (splits_trajectories(p.geo, room, one_pass, di, p.A) || (!fits && room)) {
        CatParams q = p;
        if (nt < kMinTileRows) q.tile_aggregates = p.spare_slots;
        q.block_values = nt < kMinTileRows ? p.spare_slots + 2 * tiles : tiles <= kSpareSlots ? p.spare_slots : nullptr;
        return launch_categorical<LT, GT, -NV, 3, kV, false, true, false, false>(q, laid_out(nt), di, stream);
    }
    if (!fits) return IMPACT_ERR_UNSUPPORTED;
    const int rows = wide_tile_rows(p.geo, false, p.A, sizeof(LT), sizeof(GT), di);
    if (!plain) return launch_categorical<LT, GT, -NV, C, kV, false, false, false, false>(p, laid_out(rows), di, stream);
    // (fp32 rows take as long as their bytes: one pass)
    if constexpr (sizeof(LT) == 2 && sizeof(GT) == 2) {
        if (rows > one_pass) return launch_categorical<LT, GT, -NV, C, kV, true, false, false, false>(p, laid_out(rows), di, stream);
    }
    return launch_categorical<LT, GT, -NV, C, kV, true, false, false, true>(p, laid_out(one_pass), di, stream);
}

template <typename LT, typename GT, int kV>
int32_t run_runtime_width(const CatParams& p, const DeviceInfo* di, cudaStream_t stream) {
    constexpr int kStep = kV == 4 ? 1 : 2;
    switch (wide_width(p.A).vectors) {
        case 5 * kStep: return run_wide_form<LT, GT, kV, 5 * kStep>(p, di, stream);
        case 6 * kStep: return run_wide_form<LT, GT, kV, 6 * kStep>(p, di, stream);
        case 7 * kStep: return run_wide_form<LT, GT, kV, 7 * kStep>(p, di, stream);
        case 8 * kStep: return run_wide_form<LT, GT, kV, 8 * kStep>(p, di, stream);
        default: return IMPACT_ERR_UNSUPPORTED;
    }
}

template <typename LT, typename GT>
int32_t run_compiled_count(const CatParams& p, const DeviceInfo* di, cudaStream_t stream) {
    switch (p.A) {
#define IMPACT_FIXED(n) case n: return run_fixed<LT, GT, n>(p, di, stream)
        IMPACT_FIXED(1); IMPACT_FIXED(2); IMPACT_FIXED(3); IMPACT_FIXED(4); IMPACT_FIXED(5); IMPACT_FIXED(6);
        IMPACT_FIXED(7); IMPACT_FIXED(8); IMPACT_FIXED(9); IMPACT_FIXED(10); IMPACT_FIXED(11); IMPACT_FIXED(12);
        IMPACT_FIXED(13); IMPACT_FIXED(14); IMPACT_FIXED(15); IMPACT_FIXED(16); IMPACT_FIXED(18);
        default: return IMPACT_ERR_UNSUPPORTED;
    }
}

template <typename LT, typename GT>
int32_t run_larger_count(const CatParams& p, const DeviceInfo* di, cudaStream_t stream) {
    switch (p.A) {
        IMPACT_FIXED(17); IMPACT_FIXED(19); IMPACT_FIXED(20); IMPACT_FIXED(21); IMPACT_FIXED(22); IMPACT_FIXED(23);
        IMPACT_FIXED(24); IMPACT_FIXED(25); IMPACT_FIXED(26); IMPACT_FIXED(27); IMPACT_FIXED(28); IMPACT_FIXED(29);
        IMPACT_FIXED(30); IMPACT_FIXED(31); IMPACT_FIXED(32);
#undef IMPACT_FIXED
        default: return IMPACT_ERR_UNSUPPORTED;
    }
}

}  // namespace impact
