// The diagonal-Gaussian IMPACT loss + gradient kernel and its launch rules (layout, protocols and launch shape:
// impact_flat.cuh; the categorical kernel beside it has the same skeleton).
//
// Five input slabs per tile (learner mean / log-std, target mean / log-std, actions), two output slabs (dmean, dlogstd)
// written over the learner's.  Rows are streamed from shared memory.  Tiles have as many rows, 128 to 8, as keep five of
// them in shared memory (at three dimensions: four), a warp works on a quarter of a tile's rows at once, and a row
// belongs to the 1 to 16 lanes that this leaves it: no lane has more than about 17 dimensions, and none waits for another pass.
#include "impact_flat.cuh"

namespace impact {

// Five stages, two tiles in flight and three being worked on; four, one of them in flight, at 71, 142 and 143 dimensions,
// where tiles of half the rows would make it five and take longer (143: 33 against 43 us on 100 MB, 142: 30 / 33).
constexpr size_t gauss_stage_cap = 45 * 1024;
__host__ __device__ constexpr size_t gauss_stage_bytes(size_t nt, size_t D) {
    return (5 * slab_pitch(nt, D * sizeof(float)) + 127) / 128 * 128;
}

namespace {

// exp(x).  The MuJoCo tasks' dimensions: one instruction and a rounded product in front of it, whose error grows with |x|.  Others:
// the accurate function, so that a small standard deviation (log-stds of -2 and less, as a trained policy has) costs its
// inverse nothing: dmean's error against 64 bits at log-stds of -3 to -2 and 5 dimensions is 5.6e-7 with it, 8.1e-7 without.
__host__ __device__ constexpr bool is_mujoco(int D) { return D == 3 || D == 6 || D == 17; }
template <bool kFast>
__device__ __forceinline__ float exp_of(float x) {
    return kFast ? dev::exp2_fast(x * 1.4426950408889634f) : expf(x);
}

// kD > 0: the dimension, known at compile time, 1 to 15 and 17: a row belongs to one lane.  kD < 0: -kD vectors per lane, of which a
// lane may lack the last.  Either keeps z and 1 / sigma where no switch is in use.  kV: dimensions per access to shared memory, where
// they divide the dimension.
template <int kD, int C, int kV, bool kPlain, bool kLong>
__global__ void __launch_bounds__(C * 128 + 32, 1)
impact_loss_gaussian_kernel(const __grid_constant__ GaussParams p, const __grid_constant__ LaunchForm sh) {
    constexpr bool kFixed = kD > 0, kFast = is_mujoco(kD);
    constexpr int kVecs = kFixed ? kD / kV : -kD;  // a lane's vectors
    constexpr float kHalfLog2Pi = 0.91893853320467274178f;
    const int D = kFixed ? kD : p.D;
    const int NT = kFixed ? 128 : sh.nt;
    const int NTW = NT >> 2;  // rows of a tile that one warp works on
    const int S = sh.stages, W = sh.in_flight;
    const int row_bytes = D * (int)sizeof(float);
    const int pitch = (int)slab_pitch(NT, row_bytes);
    const int stage_bytes = (int)gauss_stage_bytes(NT, D);

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
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (known to be the same for the whole warp)
    if (warp >= C * 4) {
        // ---- producer warp ----------------------------------------------------------------------------------
        const int n_first = n_tiles < W ? n_tiles : W;
        // First of all, while the kernel before this one on the stream is still finishing, the warp asks L2 for
        // the block's first tiles: the pages are mapped and the bytes on their way when the dependency resolves.  (By
        // itself: a companion kernel costs more of the copy engine's time than the earlier start gains, 10.7 us per
        // launch against 8.8 on 512 trajectories of 128 steps, D = 17.)
        const float* const src[5] = {p.learner_mean, p.learner_logstd, p.target_mean, p.target_logstd, p.actions};
        if (sh.n_prefetch > 0) {
            const void* base = nullptr;
            long long width = 4;
            if (lane < 5) { base = src[lane]; width = row_bytes; }
            else if (lane == 5) base = p.worker_logp;
            else if (lane == 6) base = p.rewards;
            else if (lane == 7) base = p.discounts;
            else if (lane == 8) base = p.values;
            if (lane >= sh.prefetch_arrays) base = nullptr;
            ask_for_tiles<kLong, 5>(g, br, base, width, n_tiles < sh.n_prefetch ? n_tiles : sh.n_prefetch, NT, total_rows);
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

        // One slab of a tile into stage s (protocol, widened copies and in-order issue as in impact_flat.cuh): lane l < 4
        // owns the round's l-th tile, requests its first slab, makes the barrier's arrival with the bytes of all five
        // slabs and fetches the bytes of a last, partial granule of the tensors; lanes l + 4, l + 8, l + 12, l + 16
        // request the tile's other slabs.
        const long long tensor_bytes = total_rows * row_bytes;
        struct SlabRequest {
            unsigned char* d;      // the stage
            long long first;       // byte offset of the tile's first granule in each of the five tensors
            uint32_t span, tail;   // dev::WideRange
        };
        auto request_for = [&](int n, int s) {
            const Tile t = tile_at<kLong>(g, br, n, NT);
            const dev::WideRange w = dev::widen_range(t.row0 * (long long)row_bytes, (uint32_t)t.nrows * row_bytes, tensor_bytes);
            SlabRequest r;
            r.d = smem_raw + s * stage_bytes;
            r.first = w.first;
            r.span = w.span;
            r.tail = w.tail;
            return r;
        };
        auto send_slab = [&](const SlabRequest& r, int s, int q) {
            uint64_t* const bar = &full_bar[s];
            const unsigned char* const gq = reinterpret_cast<const unsigned char*>(src[q]) + r.first;
            if (q == 0) {
                if (r.tail) {
#pragma unroll
                    for (int j = 0; j < 5; ++j) {
                        const unsigned char* const gj = reinterpret_cast<const unsigned char*>(src[j]) + r.first;
                        for (uint32_t i = 0; i < r.tail; ++i) r.d[j * pitch + r.span + i] = gj[r.span + i];
                    }
                    dev::fence_async_shared();
                }
                if (r.span) dev::mbarrier_expect_tx(bar, 5 * r.span);
                else dev::mbarrier_arrive(bar);
            }
            if (r.span) dev::bulk_load(r.d + q * pitch, gq, r.span, bar);
        };
        const int sub = lane & 3, q_lane = lane >> 2;
        const bool sends = q_lane < 5;
        const SlabRequest first = request_for(sub < n_first ? sub : 0, sub);

        grid_dependency_wait();

        // the first W tiles need no wait (tile n goes to stage n), four at a time
        if (sends && sub < n_first) send_slab(first, sub, q_lane);
        for (int base = 4; base < n_first; base += 4)
            if (sends && base + sub < n_first) send_slab(request_for(base + sub, base + sub), base + sub, q_lane);
        __syncthreads();  // the barriers are set up: the consumer warps may use them
        const unsigned int tag = dev::launch_tag(p.counter);  // (asked for now, needed after the last tile has left)
        const int lanes = sh.lanes;
        for (int base = n_first; base < n_tiles; base += lanes) {
            const int n = base + sub;
            bool pending = sends && sub < lanes && n < n_tiles;
            const int cyc = n / S, s = n - cyc * S;
            const int wcyc = (n - W) / S, ws = (n - W) - wcyc * S;
            const SlabRequest req = request_for(pending ? n : 0, s);
            for (unsigned int spin = 0; spin < (1u << 22); ++spin) {
                const bool ready = q_lane == 0 && pending && (cyc == 0 || dev::mbarrier_test(&empty_bar[s], (uint32_t)(cyc - 1) & 1u)) &&
                                   dev::mbarrier_test(&full_bar[ws], (uint32_t)wcyc & 1u);
                const unsigned int waiting = __ballot_sync(0xffffffffu, q_lane == 0 && pending && !ready);
                bool go = ready && (waiting & ((1u << sub) - 1u)) == 0u;
                go = __shfl_sync(0xffffffffu, go, sub);  // the owner decides for all lanes of its tile
                if (go && pending) {
                    send_slab(req, s, q_lane);
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
    const int grp = warp >> 2, gwarp = warp & 3;
    const int gtid = gwarp * 32 + lane;
    const int bar_id = grp + 1;
    const int wrow = gwarp * NTW;  // the warp's first row in a tile
    constexpr bool kKeep = kPlain;  // z and 1 / sigma of the row stay in registers for the gradient pass
    const bool want_kl = !kPlain && (k.kl_coef != 0.0f);

    // the lane's part in a row, and the row of a tile that it owns (the first lane of each row; a lane that owns none
    // stands for the row after it: the identity map, in that row's trajectory)
    const int log_l = kFixed ? 0 : sh.log_lanes;
    const int L = 1 << log_l;
    const int part = kFixed ? 0 : (lane & (L - 1));
    const int my_row = wrow + (kFixed ? lane : (lane >> log_l));
    const bool owner = part == 0;
    const int lrow = my_row + (owner ? 0 : 1);
    const int rot = (kV == 4 && !kFixed) ? ((lane >> log_l) >> sh.rot_shift) & sh.rot_mask : 0;

    // The tile (in a flat launch only a block's first tile ends early, only its last one can begin late, and from one of
    // the group's tiles to its next, C tiles further back, every position changes by a constant).
    auto tile_now = [&](int n) { return tile_rows<kLong>(g, br, n, n_tiles, NT, blockIdx.x, gridDim.x); };
    const unsigned int back = (unsigned int)(C * NT);
    TileRows tl = tile_now(grp);
    // (flat) the place of the lane's step
    using Steps = unsigned int;
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
        float l_worker, reward, discount, value, value_next;
    };
    auto load_scalars = [&](const TileRows& t, bool inner) {
        StepRaw x;
        auto fetch = [&]() {
            x.l_worker = __ldg(p.worker_logp + t.row0 + lrow);
            x.reward = __ldg(p.rewards + t.row0 + lrow);
            x.discount = __ldg(p.discounts + t.row0 + lrow);
            const float* const v = p.values + t.row0 + lrow;
            x.value = __ldg(v);
            x.value_next = __ldg(ends_here(t) ? p.bootstrap + (kLong ? t.traj : br.traj0 + (long long)at.traj) : v + 1);
        };
        if (inner) {  // every row is there, and so is the one after the last
            fetch();
        } else {
            x.l_worker = 0.0f; x.reward = 0.0f; x.discount = 0.0f; x.value = 0.0f; x.value_next = 0.0f;
            if (is_mine(t)) fetch();
        }
        return x;
    };
    // (a lane that owns no row reads that of the row it stands for, which may be the first of the next tile)
    auto is_inner = [&](const TileRows& t, int n) { return !kLong && kFixed && rows_unguarded(t, n, n_tiles); };

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
    const uint32_t m_in0 = ((uint32_t)br.base * (uint32_t)row_bytes) & 15u;
    const bool rows_aligned = ((((kLong ? 0 : (int)(br.base & 15)) * row_bytes) | (NTW * row_bytes)) & 15) == 0 &&
                              (!kLong || ((g.T * row_bytes) & 15) == 0);

    grid_dependency_wait();
    StepRaw cur = load_scalars(tl, is_inner(tl, grp));
    __syncthreads();  // the producer warp has set up the barriers
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
        const long long agg_stride = g.tile_major ? 2 * g.B : 2;  // slots between a tile's aggregate and that of the tile after it in time
        const bool peeked = kLong && g.tile_major && gwarp == 0 && tl.r > lane;
        unsigned long long early_a = 0, early_b = 0;
        if (peeked) dev::load_aggregate(p.tile_aggregates + 2 * gtile, agg_stride, tl.r - lane, early_a, early_b);
        // every thread waits for the stage itself (a bounded wait: on a time-out the flag is set and the
        // thread goes on with whatever the stage holds, so that all barriers below still pair up)
        if (!stage_wait(&full_bar[s], ph, &abort_s)) atomicExch(p.counter + 1, 1u);

        // rows keep their place inside their 16-byte granule: the tile's first row starts (row0 * pitch) mod 16
        // bytes into the slab
        unsigned char* const stage = smem_raw + s * stage_bytes;
        // (flat: tiles are a multiple of eight rows apart, so this is the same for all of the block's)
        const uint32_t m_in = kLong ? ((uint32_t)tl.row0 * (uint32_t)row_bytes) & 15u : m_in0;
        unsigned char* const slabs = stage + m_in;
        unsigned char* const mine_at = slabs + my_row * row_bytes + part * (kV * 4);
        auto vec_at = [&](int i) {
            const int step = (kV * 4) << log_l;
            return (kV == 4 && !kFixed) ? ((i * step) ^ (rot * step)) : i * step;
        };
        auto vec_there = [&](int i) { return kFixed || i < kVecs - 1 || (i << log_l) + part < D / kV; };

        // ---- row pass (every lane; rows that are not the tile's hold stale bytes and are masked).  Log-probabilities:
        // D-term sums of magnitude tens that end up in exponents, so they are accumulated in fp64.
        double lth = 0.0, ltg = 0.0;
        float ls_sum = 0.0f, kl = 0.0f;
        float z_kept[kKeep ? kVecs * kV : 1], inv_kept[kKeep ? kVecs * kV : 1];
        auto row_vec = [&](int i) {
            float mu[kV], ls[kV], mt[kV], lt[kV], ac[kV];
            const int off = vec_at(i);
            Vec<float, kV>::ld(mine_at + off, mu);
            Vec<float, kV>::ld(mine_at + pitch + off, ls);
            Vec<float, kV>::ld(mine_at + 2 * pitch + off, mt);
            Vec<float, kV>::ld(mine_at + 3 * pitch + off, lt);
            Vec<float, kV>::ld(mine_at + 4 * pitch + off, ac);
#pragma unroll
            for (int v = 0; v < kV; ++v) {
                const float inv_s = exp_of<kFast>(-ls[v]), inv_st = exp_of<kFast>(-lt[v]);
                const float z1 = (ac[v] - mu[v]) * inv_s;
                const float z2 = (ac[v] - mt[v]) * inv_st;
                lth += (double)fmaf(-0.5f * z1, z1, -ls[v]);
                ltg += (double)fmaf(-0.5f * z2, z2, -lt[v]);
                ls_sum += ls[v];
                if constexpr (kKeep) { z_kept[i * kV + v] = z1; inv_kept[i * kV + v] = inv_s; }
                if (want_kl) {  // KL(target || learner), per dimension
                    const float dm = (mt[v] - mu[v]) * inv_s;
                    const float sr = exp_of<kFast>(lt[v] - ls[v]);  // sigma_target / sigma_learner
                    kl += (ls[v] - lt[v]) + 0.5f * fmaf(sr, sr, dm * dm) - 0.5f;
                }
            }
        };
        // (lanes that share rows, every switch: eight dimensions at a time; all of them at once took 23.8 us instead of 22.5 at 64
        // dimensions, 26.4 / 23.2 at 30)
        constexpr int kUnroll = kFixed || kPlain ? 32 : 8 / kV;
#pragma unroll kUnroll
        for (int i = 0; i < kVecs; ++i)
            if (vec_there(i)) row_vec(i);
        if constexpr (!kFixed) {
            for (int o = 1; o < L; o <<= 1) {
                lth += __shfl_xor_sync(0xffffffffu, lth, o);
                ltg += __shfl_xor_sync(0xffffffffu, ltg, o);
                ls_sum += __shfl_xor_sync(0xffffffffu, ls_sum, o);
                if (want_kl) kl += __shfl_xor_sync(0xffffffffu, kl, o);
            }
        }
        const float ent = ls_sum + (float)D * (kHalfLog2Pi + 0.5f);
        // ---- the step's own scalars (its owner lane)
        dev::StepIn st;
        {
            const double shift = (double)cur.l_worker + (double)D * (double)kHalfLog2Pi;
            // everything downstream works on log-probabilities relative to the worker's
            st.l_theta = (float)(lth - shift);
            st.l_target = (float)(ltg - shift);
            st.l_worker = 0.0f;
            st.l_shift = cur.l_worker;
        }
        st.reward = cur.reward;
        st.discount = cur.discount;
        st.value = cur.value;
        st.value_next = cur.value_next;
        st.last_step = ends_here(tl);
        float fa, fb;
        const bool truncated = dev::recursion_map<kPlain>(st, k, fa, fb);
        const bool mine = is_mine(tl);
        if (!mine) { fa = 1.0f; fb = 0.0f; }
        // (flat) the slot of the tile, or beyond, where the step's trajectory ends
        const int reach = lrow + (int)min(at.to_end, (Steps)1024);
        int limit = 31 - lane;
        if constexpr (!kLong) limit = min(limit, ((reach - wrow) << log_l) - lane);  // (counted from the warp's first row)

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
            if (gtid == 0) dev::publish_tile_aggregate(p.tile_aggregates + 2 * gtile, ma, mb, dev::launch_tag(p.counter));
            float carry = 0.0f;
            if (here.r > 0) {  // uniform over the group
                if (gwarp == 0) {
                    const float c = dev::compose_later_aggregates(p.tile_aggregates + 2 * gtile, agg_stride, here.r,
                                                                  dev::launch_tag(p.counter), &abort_s, p.counter + 1,
                                                                  peeked, early_a, early_b);
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
        const float wpg = dev::surrogate<kPlain>(st, k, adv, surr, ratio, clipped);
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

        // ---- gradients, in place over the learner's slabs
        {
            float w1 = __fmul_rn(wpg, k.inv_M);
            if (!kFixed) w1 = __shfl_sync(0xffffffffu, w1, lane & ~(L - 1));  // (the owner's)
            const float ce = k.ent_over_M, ck = kPlain ? 0.0f : k.kl_over_M;
            auto grad_vec = [&](int i) {
                float mu[kV], ls[kV], ac[kV], mt[kV], lt[kV];
                const int off = vec_at(i);
                if (!kKeep || want_kl) {
                    Vec<float, kV>::ld(mine_at + off, mu);
                    Vec<float, kV>::ld(mine_at + pitch + off, ls);
                }
                if (!kKeep) Vec<float, kV>::ld(mine_at + 4 * pitch + off, ac);
                if (want_kl) {
                    Vec<float, kV>::ld(mine_at + 2 * pitch + off, mt);
                    Vec<float, kV>::ld(mine_at + 3 * pitch + off, lt);
                }
                float om[kV], os[kV];
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    float inv_s, z;
                    if constexpr (kKeep) {
                        inv_s = inv_kept[i * kV + v];
                        z = z_kept[i * kV + v];
                    } else {
                        inv_s = exp_of<kFast>(-ls[v]);
                        z = (ac[v] - mu[v]) * inv_s;  // (a - mu) / sigma
                    }
                    // d log pi / d mu = z / sigma ;  d log pi / d logstd = z^2 - 1 ;  d H / d logstd = 1
                    float gm = __fmul_rn(-w1, z);
                    float gs = fmaf(-w1, fmaf(z, z, -1.0f), -ce);
                    if (want_kl) {
                        // d KL / d mu = (mu - mu_t) / sigma^2 ; d KL / d logstd = 1 - (sigma_t^2 + (mu_t - mu)^2) / sigma^2
                        const float dm = (mu[v] - mt[v]) * inv_s;
                        const float sr = exp_of<kFast>(lt[v] - ls[v]);
                        gm = fmaf(ck, dm, gm);
                        gs = fmaf(ck, 1.0f - fmaf(sr, sr, dm * dm), gs);
                    }
                    om[v] = __fmul_rn(gm, inv_s);
                    os[v] = gs;
                }
                Vec<float, kV>::st(mine_at + off, om);
                Vec<float, kV>::st(mine_at + pitch + off, os);
            };
#pragma unroll kUnroll
            for (int i = 0; i < kVecs; ++i)
                if (vec_there(i)) grad_vec(i);
        }
        if (mine) {
            p.dvalues[here.row0 + lrow] = __fmul_rn(k.dvalue_over_adv, adv);  // V - Vhat = -A
            if (!kPlain) {
                if (p.vtarget) p.vtarget[here.row0 + lrow] = st.value + adv;
                if (p.advantage) p.advantage[here.row0 + lrow] = adv;
            }
        }
        // ---- each warp sends its own rows of both gradient slabs: no barrier across the group
        {
            unsigned char* const gm = reinterpret_cast<unsigned char*>(p.dmean) + here.row0 * (long long)row_bytes;
            unsigned char* const gs = reinterpret_cast<unsigned char*>(p.dlogstd) + here.row0 * (long long)row_bytes;
            if (here.lo == 0 && here.hi == NT && rows_aligned) {  // whole granules: the usual case
                dev::fence_async_shared();
                __syncwarp();
                if (lane == 0) {
                    dev::bulk_store(gm + wrow * row_bytes, slabs + wrow * row_bytes, (uint32_t)(NTW * row_bytes));
                    dev::bulk_store(gs + wrow * row_bytes, slabs + pitch + wrow * row_bytes, (uint32_t)(NTW * row_bytes));
                }
            } else {
                send_rows_general(gm, slabs, row_bytes, wrow, NTW, here.lo, here.hi, true);
                send_rows_general(gs, slabs + pitch, row_bytes, wrow, NTW, here.lo, here.hi, true);
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
    // (in fp64, but for the MuJoCo tasks' dimensions on trajectories that fit a tile or are split, which add in fp32 as they
    // always did: fp64 costs 0.15 to 0.3 us at the end of a launch)
    if (blockIdx.x == 0 && grp == n_tiles % C) {
        auto collect = [&](auto zero) {
            if (!dev::reduce_tagged_rows<128, decltype(zero)>(p.tagged_rows, (int)gridDim.x, dev::launch_tag(p.counter),
                                                              p.counter, p.loss_terms, k.vf_coef, k.ent_coef, k.kl_coef,
                                                              k.steps_total, gtid, bar_id, &abort_s))
                if (gtid == 0) atomicExch(p.counter + 1, 1u);
        };
        if (!kFast || (!kLong && g.T > 128)) collect(0.0);
        else collect(0.0f);
    }
    if (lane == 0) dev::bulk_store_wait_read();  // shared memory must outlive the stores' reads
}


template <int kD, int C, int kV, bool kPlain, bool kLong>
int32_t launch_gaussian(GaussParams p, const RowLayout& rl, const DeviceInfo* di, cudaStream_t stream) {
    auto kernel = impact_loss_gaussian_kernel<kD, C, kV, kPlain, kLong>;
    const int nt = rl.nt;
    const size_t stage = gauss_stage_bytes(nt, p.D);
    LaunchShape ls;
    if (!launch_shape(p.geo, nt, kLong, stage, stage, C, di, &ls)) return IMPACT_ERR_UNSUPPORTED;
    LaunchForm sh = {};
    sh.nt = nt;
    sh.stages = ls.stages;
    sh.in_flight = ls.in_flight;
    sh.lanes = ls.lanes;
    sh.log_lanes = rl.log_lanes;
    sh.rot_shift = rl.rot_shift;
    sh.rot_mask = rl.rot_mask;
    const size_t smem = (size_t)sh.stages * stage;
    static thread_local int configured_device = -1;
    if (configured_device != di->device) {  // once per device: room for the largest ring any window setting asks for
        IMPACT_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, di->max_smem_optin - 4096));
        configured_device = di->device;
    }
    const size_t tile_bytes = (size_t)nt * (5 * p.D * sizeof(float) + 16);
    const OwnRequests own = own_requests(ws_plan(ls.tiles, ls.grid, tile_bytes, sh.in_flight, false), tile_bytes, p.geo.B * p.geo.T,
                                         ls.grid, nt, 24 * 1024, 12);
    sh.n_prefetch = own.tiles;
    sh.prefetch_arrays = own.slabs_only ? 5 : 9;
    IMPACT_CUDA_TRY(launch_serialized(kernel, dim3((unsigned)ls.grid), dim3(C * 128 + 32), smem, stream, p, sh));
    return IMPACT_OK;
}

// What a split launch of lanes that share rows costs (see splits_trajectories): 48 x 200 steps of 100 dimensions 14.7 us
// flat, 13.0 split; 32 x 200 of 40 9.0 / 7.5, of 33 7.4 / 8.2; 10 x 80 of 40 5.1 / 5.6, of 100 7.0 / 5.9.
constexpr int kGaussSplitSlope = 24, kGaussSplitCost = 26;

template <int kD, int C, int CP, int CL, int kV>
int32_t run_gaussian_form(const GaussParams& p, const RowLayout& rl, const DeviceInfo* di, cudaStream_t stream) {
    const bool plain = p.k.kl_coef == 0.0f && p.k.objective == IMPACT_OBJECTIVE_CLIPPED_SURROGATE &&
                       p.k.is_source == IMPACT_IS_TARGET_OVER_WORKER && p.k.ratio_mode == IMPACT_RATIO_R3 && !p.vtarget && !p.advantage;
    // Tiles of few rows keep their maps in the workspace's spare slots, where there is room: 16 x 4096 steps of 40 dimensions take
    // 30 us, on one block per trajectory 88; of 100 61 / 196.
    const bool few_rows = rl.nt < kMinTileRows;
    const bool room = few_rows ? p.spare_slots && 2 * split_tiles(p.geo, rl.nt) <= kSpareSlots : p.tile_aggregates != nullptr;
    if (splits_trajectories(p.geo, room, rl.nt, di, rl.log_lanes ? p.D : 0, kGaussSplitSlope, kGaussSplitCost, plain) || !fits_flat(p.geo)) {
        if (!room) return IMPACT_ERR_UNSUPPORTED;
        GaussParams q = p;
        if (few_rows) q.tile_aggregates = p.spare_slots;
        return launch_gaussian<kD, CL, kV, false, true>(q, rl, di, stream);
    }
    if (plain) return launch_gaussian<kD, CP, kV, true, false>(p, rl, di, stream);
    // Lanes that share rows take four groups where these leave the ring two stages more, one where a vector is one dimension
    // (26 dimensions 23.2 us, three groups 24.2; 45 27.2 / 29.4; 60, five stages, 26.9 / 23.4).
    if constexpr (kD < 0) {
        if (stages_that_fit(gauss_stage_bytes(rl.nt, p.D), di->max_smem_optin) >= (kV == 1 ? 5 : 6))
            return launch_gaussian<kD, C + 1, kV, false, false>(p, rl, di, stream);
    }
    return launch_gaussian<kD, C, kV, false, false>(p, rl, di, stream);
}

// Lanes that share rows: the rows of a tile, the lanes of a row, the rotation that lanes of vectors of four take them in.
template <int kV>
RowLayout rows_on_lanes(int D) {
    RowLayout rl;
    while (rl.nt > 8 && gauss_stage_bytes(rl.nt, D) > gauss_stage_cap) rl.nt /= 2;
    while ((rl.nt / 4 << rl.log_lanes) < 32) ++rl.log_lanes;
    const BankPattern b = bank_pattern(D * sizeof(float), 1 << rl.log_lanes, kV * 4);
    rl.rot_shift = b.shift;
    const int vecs = D / kV;
    if (kV == 4 && vecs % (1 << rl.log_lanes) == 0)
        while (2 * (rl.rot_mask + 1) <= b.ways && (vecs >> rl.log_lanes) % (2 * (rl.rot_mask + 1)) == 0)
            rl.rot_mask = 2 * rl.rot_mask + 1;
    return rl;
}
template <int kV>
int vectors_of_a_lane(int D) {
    const int log_lanes = rows_on_lanes<kV>(D).log_lanes;
    return (D / kV + (1 << log_lanes) - 1) >> log_lanes;
}

}  // namespace

// The kernels are compiled in units of a few dimensions each, by files that say which and include this one: the first launch of
// a unit's kernels loads the whole unit (all dimensions in one took 45 ms).
#ifndef IMPACT_GAUSSIAN_PART
#define IMPACT_GAUSSIAN_PART 0
#endif
constexpr int kGaussPart = IMPACT_GAUSSIAN_PART;  // (0: this file by itself)

#if IMPACT_GAUSSIAN_PART < 3
// Consumer groups, with every switch, plain, split.  Where rows are short a tile's time is arithmetic: five (five with every
// switch up to five dimensions: 512 x 128 of 1 4.4 us, four 4.6; of 7 6.8 / 6.7).  Longer rows take three, whose ring has
// stages enough (8000 x 50 of 15 32.3 us, four 41.7), but four with every switch and split (4000 x 50 of 9 14.2, three 15.3;
// 16 x 4096 of 9 9.7 / 12.1, of 17 11.2 / 13.2).  The dimension known at run time: 2500 x 50 of 4 7.6 instead of 6.9, of
// 9 12.9 / 9.3, of 13 15.1 / 12.1, with every switch 4000 x 50 of 13 25.9 / 18.0.  16 is not among them: rows 64 bytes
// apart meet on the banks, and lanes that take their vectors in rotated order do not (35.2 us, 36.2 in order).
#define IMPACT_FIXED(n, full, plain, split) \
    case n: return run_gaussian_form<n, full, plain, split, n % 4 == 0 ? 4 : n % 2 == 0 ? 2 : 1>(p, RowLayout(), di, stream)
template <>
int32_t run_gaussian_part<kGaussPart>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream) {
    switch (p.D) {
#if IMPACT_GAUSSIAN_PART == 0
        IMPACT_FIXED(3, 5, 5, 5); IMPACT_FIXED(6, 4, 4, 4); IMPACT_FIXED(17, 3, 3, 4);
#elif IMPACT_GAUSSIAN_PART == 1
        IMPACT_FIXED(1, 5, 5, 4); IMPACT_FIXED(2, 5, 5, 4); IMPACT_FIXED(4, 5, 5, 4); IMPACT_FIXED(5, 5, 5, 4);
        IMPACT_FIXED(7, 4, 5, 4); IMPACT_FIXED(8, 4, 5, 4);
#else
        IMPACT_FIXED(9, 4, 3, 4); IMPACT_FIXED(10, 4, 3, 4); IMPACT_FIXED(11, 4, 3, 4); IMPACT_FIXED(12, 4, 3, 4);
        IMPACT_FIXED(13, 4, 3, 4); IMPACT_FIXED(14, 4, 3, 4); IMPACT_FIXED(15, 3, 3, 4);
#endif
        default: return IMPACT_ERR_UNSUPPORTED;
    }
}
#undef IMPACT_FIXED
#else
// A lane's vectors, the same for many dimensions, are compiled in.  Told at run time they took, on the bytes of 8000 x 50 steps of 17,
// 50.3 us instead of 38.5 at 19 dimensions, 51.8 / 35.8 at 37, 47.5 / 36.9 at 63, 35.5 / 35.4 at 32; with every switch on half of
// that 34.0 / 24.7 at 23, 23.7 / 22.5 at 64; 300 x 50 of 45 11.2 / 8.2; 16 x 4096 of 23 22.4 / 18.4, of 35 27.0 / 21.7.
#define IMPACT_VECS(n) case n: return run_gaussian_form<-(n), 3, 3, 4, kV>(p, rows_on_lanes<kV>(p.D), di, stream)
template <>
int32_t run_gaussian_part<kGaussPart>(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream) {
    constexpr int kV = kGaussPart == 3 ? 4 : kGaussPart == 4 ? 2 : 1;
    switch (vectors_of_a_lane<kV>(p.D)) {
#if IMPACT_GAUSSIAN_PART == 3
        IMPACT_VECS(3); IMPACT_VECS(4); IMPACT_VECS(5);
#elif IMPACT_GAUSSIAN_PART == 4
        IMPACT_VECS(5); IMPACT_VECS(6); IMPACT_VECS(7); IMPACT_VECS(8); IMPACT_VECS(9);
#elif IMPACT_GAUSSIAN_PART == 5
        IMPACT_VECS(10); IMPACT_VECS(11); IMPACT_VECS(12); IMPACT_VECS(13);
#else
        IMPACT_VECS(14); IMPACT_VECS(15); IMPACT_VECS(16); IMPACT_VECS(17); IMPACT_VECS(18);
#endif
        default: return IMPACT_ERR_UNSUPPORTED;  // (no dimension up to 256 gets here)
    }
}
#undef IMPACT_VECS
#endif

#if IMPACT_GAUSSIAN_PART == 0
int32_t run_gaussian(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream) {
    if (is_mujoco(p.D)) return run_gaussian_part<0>(p, di, stream);
    if (p.D <= 8) return run_gaussian_part<1>(p, di, stream);
    if (p.D <= 15) return run_gaussian_part<2>(p, di, stream);
    if (p.D % 4 == 0) return run_gaussian_part<3>(p, di, stream);
    if (p.D % 2 == 0) return run_gaussian_part<4>(p, di, stream);
    return vectors_of_a_lane<1>(p.D) <= 13 ? run_gaussian_part<5>(p, di, stream) : run_gaussian_part<6>(p, di, stream);
}
#endif

}  // namespace impact
