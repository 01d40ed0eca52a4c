// Fused IMPACT loss + gradient kernels and their host entry points.
//
// One launch per call does every step of the learner's "compute policy and value network
// gradients" (Algorithm 1): log-probabilities under learner and target, truncated
// importance weights, the backward V-trace GAE-lambda recursion (Section 3.1), the
// target-worker-clipped, eps-clipped surrogate (Section 3.1, Appendix E), value / entropy /
// KL terms, the gradients, and the batch means.  Each input byte is read from HBM once and
// each output byte written once; nothing on this path is a matrix product, so no tensor
// cores are involved -- the kernel is bound by HBM bandwidth.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include "impact.h"
#include "impact_device.cuh"
#include "impact_internal.h"
#include "impact_loss_params.h"

namespace impact {
namespace {

struct TileGeometry {
    int tile_major;  // long trajectories in a persistent kernel: order of the grid's tiles (see place_of)
    long long B, T;
    long long nchunks;  // units of block-level work
    int G;              // whole trajectories per chunk (T <= NT), else 1
    int ntiles;         // tiles per trajectory (T > NT), else 1
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
    float* partials;
    unsigned int* counter;
    unsigned long long* tagged_rows;
    unsigned long long* tile_aggregates;
    TileGeometry geo;
    LossScalars k;
    int D, Ds;
};

// Where a tile sits: its first global row, how many rows, and each thread's (b, t).
struct TileRows {
    long long row0;
    int nrows;
};

template <int NT>
__device__ __forceinline__ TileRows tile_rows(const TileGeometry& g, long long chunk, int tile) {
    TileRows r;
    if (g.ntiles > 1) {
        const long long t0 = (long long)tile * NT;
        const long long left = g.T - t0;
        r.nrows = (int)(left < NT ? left : NT);
        r.row0 = chunk * g.T + t0;
    } else {
        const long long traj0 = chunk * g.G;
        long long ntraj = g.B - traj0;
        if (ntraj > g.G) ntraj = g.G;
        r.nrows = (int)(ntraj * g.T);
        r.row0 = traj0 * g.T;
    }
    return r;
}

constexpr int kRegTileRows = 128;

// Where the n-th tile of a block of a persistent kernel sits: first row, rows, first trajectory, and (long
// trajectories) the tile's number counted from its trajectory's end.
struct Place {
    long long row0, traj;
    int nrows, r;
};
template <bool kLong, int NT>
__device__ __forceinline__ Place tile_place(const TileGeometry& g, int n, int rows_full, long long total_rows) {
    Place pl;
    const long long gt_ = (long long)blockIdx.x + (long long)n * gridDim.x;
    if (kLong) {
        if (g.tile_major) {  // the last tiles of all trajectories first, then the tiles before them, ...
            pl.r = (int)((unsigned long long)gt_ / (unsigned long long)g.B);
            pl.traj = gt_ - (long long)pl.r * g.B;
        } else {  // trajectory by trajectory, each from its last tile backwards
            pl.traj = (long long)((unsigned long long)gt_ / (unsigned int)g.ntiles);
            pl.r = (int)(gt_ - pl.traj * g.ntiles);
        }
        const long long t0 = (long long)(g.ntiles - 1 - pl.r) * NT;
        const long long left = g.T - t0;
        pl.nrows = left < NT ? (int)left : NT;
        pl.row0 = pl.traj * g.T + t0;
    } else {
        pl.row0 = gt_ * rows_full;
        pl.traj = gt_ * g.G;
        const long long left = total_rows - pl.row0;
        pl.nrows = left < rows_full ? (int)left : rows_full;
        pl.r = 0;
    }
    return pl;
}

// A slab of the persistent kernels in shared memory: NT rows of `row_bytes`, plus 32 bytes of padding, because a
// tile's rows sit at the same offset inside their 16-byte granule as in global memory (0..15 bytes after the
// slab's start) and the copy that brings them is widened to whole granules (see dev::widen_range).
__host__ __device__ constexpr size_t ws_slab_pitch(size_t nt, size_t row_bytes) { return nt * row_bytes + 32; }

// ------------------------------------------------------------------------------------------
// Diagonal-Gaussian policy
// ------------------------------------------------------------------------------------------
template <int NT>
__global__ void __launch_bounds__(NT) impact_loss_gaussian_kernel(const GaussParams p) {
    grid_dependency_wait();
    extern __shared__ __align__(16) float smem[];
    const int D = p.D, Ds = p.Ds;
    float* const s_mu = smem;                              // learner mean -> dmean
    float* const s_ls = s_mu + (size_t)NT * Ds;            // learner logstd -> dlogstd
    float* const s_mt = s_ls + (size_t)NT * Ds;            // target mean
    float* const s_lt = s_mt + (size_t)NT * Ds;            // target logstd
    float* const s_ac = s_lt + (size_t)NT * Ds;            // actions
    __shared__ float2 warp_agg[NT / 32];
    __shared__ float red[NT / 32][8];
    __shared__ float carry_s;

    const int tid = threadIdx.x;
    const LossScalars k = p.k;
    const TileGeometry g = p.geo;
    const float half_log_2pi = 0.91893853320467274178f;

    float acc[dev::kNumSums];
#pragma unroll
    for (int j = 0; j < dev::kNumSums; ++j) acc[j] = 0.0f;

    for (long long chunk = blockIdx.x; chunk < g.nchunks; chunk += gridDim.x) {
        float carry = 0.0f;
        for (int tile = g.ntiles - 1; tile >= 0; --tile) {
            const TileRows tr = tile_rows<NT>(g, chunk, tile);
            const long long base = tr.row0 * D;
            const int nelem = tr.nrows * D;
            __syncthreads();
            dev::stage_slab<float, NT>(s_mu, p.learner_mean, base, nelem, D, Ds);
            dev::stage_slab<float, NT>(s_ls, p.learner_logstd, base, nelem, D, Ds);
            dev::stage_slab<float, NT>(s_mt, p.target_mean, base, nelem, D, Ds);
            dev::stage_slab<float, NT>(s_lt, p.target_logstd, base, nelem, D, Ds);
            dev::stage_slab<float, NT>(s_ac, p.actions, base, nelem, D, Ds);
            __syncthreads();

            const bool active = tid < tr.nrows;
            const long long row = tr.row0 + tid;
            float* const r_mu = s_mu + tid * Ds;
            float* const r_ls = s_ls + tid * Ds;
            const float* const r_mt = s_mt + tid * Ds;
            const float* const r_lt = s_lt + tid * Ds;
            const float* const r_ac = s_ac + tid * Ds;
            dev::StepIn s;
            float fa = 1.0f, fb = 0.0f;
            float ent = 0.0f, kl = 0.0f;
            bool truncated = false;
            if (active) {
                long long b, t;
                if (g.ntiles > 1) { b = chunk; t = (long long)tile * NT + tid; }
                else { const int q = tid / (int)g.T; b = chunk * g.G + q; t = tid - q * (int)g.T; }
                // The log-probabilities are sums of D terms and reach magnitudes of tens; they
                // enter exponentials, so their absolute error is the relative error of the
                // ratios.  Accumulating them in fp64 (half-rate on this part, a few percent of
                // the pipe here) keeps that error at the level of the fp32 terms themselves.
                double lth = 0.0, ltg = 0.0;
                for (int j = 0; j < D; ++j) {
                    const float ls = r_ls[j], lt = r_lt[j], ac = r_ac[j];
                    const float inv_s = expf(-ls), inv_st = expf(-lt);
                    const float z1 = (ac - r_mu[j]) * inv_s;
                    const float z2 = (ac - r_mt[j]) * inv_st;
                    lth += (double)(fmaf(-0.5f * z1, z1, -ls) - half_log_2pi);
                    ltg += (double)(fmaf(-0.5f * z2, z2, -lt) - half_log_2pi);
                    ent += ls + (half_log_2pi + 0.5f);
                    if (k.kl_coef != 0.0f) {  // KL(target || learner), per dimension
                        const float dm = (r_mt[j] - r_mu[j]) * inv_s;
                        const float sr = expf(lt - ls);  // sigma_target / sigma_learner
                        kl += (ls - lt) + 0.5f * fmaf(sr, sr, dm * dm) - 0.5f;
                    }
                }
                // differences against the worker's log-probability are taken in fp64, then
                // everything continues in fp32 relative to it
                const float lw = p.worker_logp[row];
                s.l_theta = (float)(lth - (double)lw);
                s.l_target = (float)(ltg - (double)lw);
                s.l_worker = 0.0f;
                s.l_shift = lw;
                s.reward = p.rewards[row];
                s.discount = p.discounts[row];
                s.value = p.values[row];
                s.last_step = (t == g.T - 1);
                s.value_next = s.last_step ? p.bootstrap[b] : p.values[row + 1];
                asm volatile("" ::: "memory");
                truncated = dev::recursion_map(s, k, fa, fb);
            }
            const float adv = dev::suffix_affine_scan<NT>(fa, fb, carry, warp_agg, s.adv_next);
            if (tid == 0) carry_s = adv;

            float sums[dev::kNumSums];
#pragma unroll
            for (int j = 0; j < dev::kNumSums; ++j) sums[j] = 0.0f;
            if (active) {
                float surr, ratio;
                bool clipped;
                const float wpg = dev::surrogate(s, k, adv, surr, ratio, clipped);
                const float w1 = wpg * k.inv_M, ce = k.ent_coef * k.inv_M, ck = k.kl_coef * k.inv_M;
                for (int j = 0; j < D; ++j) {
                    const float ls = r_ls[j], lt = r_lt[j], mu = r_mu[j];
                    const float inv_s = expf(-ls);
                    const float z = (r_ac[j] - mu) * inv_s;       // (a - mu) / sigma
                    const float dm = (mu - r_mt[j]) * inv_s;      // (mu - mu_target) / sigma
                    const float sr = expf(lt - ls);
                    // d log pi / d mu = z / sigma ; d KL / d mu = dm / sigma
                    r_mu[j] = (ck * dm - w1 * z) * inv_s;
                    // d log pi / d logstd = z^2 - 1 ; d H / d logstd = 1 ;
                    // d KL / d logstd = 1 - (sigma_t^2 + (mu_t - mu)^2) / sigma^2
                    r_ls[j] = -w1 * fmaf(z, z, -1.0f) - ce + ck * (1.0f - fmaf(sr, sr, dm * dm));
                }
                p.dvalues[row] = -k.vf_coef * k.inv_M * adv;
                if (p.vtarget) p.vtarget[row] = s.value + adv;
                if (p.advantage) p.advantage[row] = adv;
                sums[0] = surr;
                sums[1] = 0.5f * adv * adv;
                sums[2] = ent;
                sums[3] = kl;
                sums[4] = clipped ? 1.0f : 0.0f;
                sums[5] = truncated ? 1.0f : 0.0f;
                sums[6] = ratio;
            }
            dev::block_sums_stage1<NT>(sums, red);
            __syncthreads();
            carry = carry_s;
            dev::unstage_slab<float, NT>(p.dmean, s_mu, base, nelem, D, Ds);
            dev::unstage_slab<float, NT>(p.dlogstd, s_ls, base, nelem, D, Ds);
            dev::block_sums_stage2<NT>(acc, red);
        }
    }
    dev::finish_loss_terms<NT>(acc, p.partials, p.counter, p.loss_terms, k,
                               k.steps_total);
}

// ------------------------------------------------------------------------------------------
// Diagonal-Gaussian policy, action dimension known at compile time
// ------------------------------------------------------------------------------------------
// Same structure as the register-resident categorical kernel: the five [tile, D] slabs
// (learner mean / log-std, target mean / log-std, actions) arrive by bulk copies, a thread
// walks its row with every loop unrolled, dmean / dlogstd replace the learner slabs in place and
// leave by two bulk stores.  One stage per block (five slabs are 43 KB at D = 17), four
// blocks per SM overlap each other's loads and arithmetic.
template <int D>
__global__ void __launch_bounds__(kRegTileRows, 4) impact_loss_gaussian_reg_kernel(const GaussParams p) {
    grid_dependency_wait();
    constexpr int NT = kRegTileRows;
    constexpr int kSlab = NT * D * (int)sizeof(float);
    constexpr float kLog2e = 1.4426950408889634f;
    constexpr float kHalfLog2Pi = 0.91893853320467274178f;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* const s_mu = reinterpret_cast<float*>(smem_raw);              // learner mean -> dmean
    float* const s_ls = reinterpret_cast<float*>(smem_raw + kSlab);      // learner log-std -> dlogstd
    const float* const s_mt = reinterpret_cast<const float*>(smem_raw + 2 * kSlab);
    const float* const s_lt = reinterpret_cast<const float*>(smem_raw + 3 * kSlab);
    const float* const s_ac = reinterpret_cast<const float*>(smem_raw + 4 * kSlab);
    __shared__ __align__(8) uint64_t bar;
    __shared__ float2 warp_agg[NT / 32];
    __shared__ float red[NT / 32][8];
    __shared__ float carry_s;
    __shared__ int is_last_s;

    const int tid = threadIdx.x;
    const LossScalars k = p.k;
    const TileGeometry g = p.geo;
    const bool want_kl = (k.kl_coef != 0.0f);
    const float* const src[5] = {p.learner_mean, p.learner_logstd, p.target_mean, p.target_logstd, p.actions};

    if (tid == 0) {
        dev::mbarrier_init(&bar, 1);
        is_last_s = 0;
    }
    __syncthreads();
    uint32_t parity = 0;

    float acc[dev::kNumSums], tsum[dev::kNumSums];
#pragma unroll
    for (int j = 0; j < dev::kNumSums; ++j) acc[j] = tsum[j] = 0.0f;

    for (long long chunk = blockIdx.x; chunk < g.nchunks; chunk += gridDim.x) {
        float carry = 0.0f;
        for (int tile = g.ntiles - 1; tile >= 0; --tile) {
            const bool final_tile = (tile == 0) && (chunk + gridDim.x >= g.nchunks);
            const TileRows tr = tile_rows<NT>(g, chunk, tile);
            const long long base = tr.row0 * D;
            const uint32_t bytes = (uint32_t)tr.nrows * D * (uint32_t)sizeof(float);
            uintptr_t align = bytes;
#pragma unroll
            for (int q = 0; q < 5; ++q) align |= reinterpret_cast<uintptr_t>(src[q] + base);
            const bool bulk_in = (align & 15u) == 0;
            const bool bulk_out = (((reinterpret_cast<uintptr_t>(p.dmean + base) |
                                     reinterpret_cast<uintptr_t>(p.dlogstd + base) | bytes) & 15u) == 0);
            if (bulk_in) {
                if (tid == 0) {
                    dev::mbarrier_expect_tx(&bar, 5 * bytes);
#pragma unroll
                    for (int q = 0; q < 5; ++q) dev::bulk_load(smem_raw + q * kSlab, src[q] + base, bytes, &bar);
                }
            } else {
                const int nelem = tr.nrows * D;
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    for (int e = tid; e < nelem; e += NT) reinterpret_cast<float*>(smem_raw + q * kSlab)[e] = src[q][base + e];
            }

            const bool active = tid < tr.nrows;
            const long long row = tr.row0 + tid;
            dev::StepIn s;
            float lw = 0.0f;
            if (active) {
                long long b, t;
                if (g.ntiles > 1) { b = chunk; t = (long long)tile * NT + tid; }
                else if (g.G == 1) { b = chunk; t = tid; }
                else { const int q = tid / (int)g.T; b = chunk * g.G + q; t = tid - q * (int)g.T; }
                lw = p.worker_logp[row];
                s.reward = p.rewards[row];
                s.discount = p.discounts[row];
                s.value = p.values[row];
                s.last_step = (t == g.T - 1);
                s.value_next = s.last_step ? p.bootstrap[b] : p.values[row + 1];
            }
            if (bulk_in) {
                if (tid < 32) {
                    if (!dev::mbarrier_wait(&bar, parity)) atomicExch(p.counter + 1, 1u);
                }
                parity ^= 1u;
            }
            __syncthreads();

            float* const r_mu = s_mu + tid * D;
            float* const r_ls = s_ls + tid * D;
            const float* const r_mt = s_mt + tid * D;
            const float* const r_lt = s_lt + tid * D;
            const float* const r_ac = s_ac + tid * D;
            float fa = 1.0f, fb = 0.0f, ent = 0.0f, kl = 0.0f;
            bool truncated = false;
            if (active) {
                // log-probabilities: D-term sums of magnitude tens that end up in exponents, so they
                // are accumulated in fp64 (half-rate here, a few percent of the pipe)
                double lth = 0.0, ltg = 0.0;
                float ls_sum = 0.0f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    const float ls = r_ls[j], lt = r_lt[j], ac = r_ac[j], mu = r_mu[j], mt = r_mt[j];
                    const float inv_s = dev::exp2_fast(-ls * kLog2e), inv_st = dev::exp2_fast(-lt * kLog2e);
                    const float z1 = (ac - mu) * inv_s;
                    const float z2 = (ac - mt) * inv_st;
                    lth += (double)fmaf(-0.5f * z1, z1, -ls);
                    ltg += (double)fmaf(-0.5f * z2, z2, -lt);
                    ls_sum += ls;
                    if (want_kl) {  // KL(target || learner), per dimension
                        const float dm = (mt - mu) * inv_s;
                        const float sr = dev::exp2_fast((lt - ls) * kLog2e);  // sigma_target / sigma_learner
                        kl += (ls - lt) + 0.5f * fmaf(sr, sr, dm * dm) - 0.5f;
                    }
                }
                ent = ls_sum + (float)D * (kHalfLog2Pi + 0.5f);
                const double shift = (double)lw + (double)D * (double)kHalfLog2Pi;
                // everything downstream works on log-probabilities relative to the worker's
                s.l_theta = (float)(lth - shift);
                s.l_target = (float)(ltg - shift);
                s.l_worker = 0.0f;
                s.l_shift = lw;
                truncated = dev::recursion_map(s, k, fa, fb);
            }
            const float adv = dev::suffix_affine_scan<NT>(fa, fb, carry, warp_agg, s.adv_next);
            if (tid == 0) carry_s = adv;

            float surr = 0.0f, ratio = 0.0f, wpg = 0.0f;
            bool clipped = false;
            if (active) wpg = dev::surrogate(s, k, adv, surr, ratio, clipped);
            // each thread keeps its own running sums over the block's tiles; they are added across
            // the block once, in the last tile, and published right away so that the round trip
            // hides behind the epilogue
            if (active) {
                tsum[0] += surr;
                tsum[1] = fmaf(0.5f * adv, adv, tsum[1]);
                tsum[2] += ent;
                tsum[3] += kl;
                tsum[4] += clipped ? 1.0f : 0.0f;
                tsum[5] += truncated ? 1.0f : 0.0f;
                tsum[6] += ratio;
            }
            unsigned int ticket = 0;
            if (final_tile) {
                dev::block_sums_stage1<NT>(tsum, red);
                __syncthreads();
                if (tid == 0) {
                    dev::block_sums_stage2<NT>(acc, red);
                    ticket = dev::publish_block_sums(acc, p.partials, p.counter);
                }
            }
            if (active) {
                const float w1 = wpg * k.inv_M, ce = k.ent_coef * k.inv_M, ck = k.kl_coef * k.inv_M;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    const float ls = r_ls[j], mu = r_mu[j];
                    const float inv_s = dev::exp2_fast(-ls * kLog2e);
                    const float z = (r_ac[j] - mu) * inv_s;  // (a - mu) / sigma
                    // d log pi / d mu = z / sigma ;  d log pi / d logstd = z^2 - 1 ;  d H / d logstd = 1
                    float gm = -w1 * z;
                    float gs = -w1 * fmaf(z, z, -1.0f) - ce;
                    if (want_kl) {
                        // d KL / d mu = (mu - mu_t) / sigma^2 ; d KL / d logstd = 1 - (sigma_t^2 + (mu_t - mu)^2) / sigma^2
                        const float dm = (mu - r_mt[j]) * inv_s;
                        const float sr = dev::exp2_fast((r_lt[j] - ls) * kLog2e);
                        gm = fmaf(ck, dm, gm);
                        gs = fmaf(ck, 1.0f - fmaf(sr, sr, dm * dm), gs);
                    }
                    r_mu[j] = gm * inv_s;
                    r_ls[j] = gs;
                }
                p.dvalues[row] = -k.vf_coef * k.inv_M * adv;
                if (p.vtarget) p.vtarget[row] = s.value + adv;
                if (p.advantage) p.advantage[row] = adv;
            }
            if (bulk_out) dev::fence_async_shared();
            if (tid == 0 && final_tile) is_last_s = (ticket == gridDim.x - 1) ? 1 : 0;
            __syncthreads();
            carry = carry_s;
            if (bulk_out) {
                if (tid == 0) {
                    dev::bulk_store(p.dmean + base, s_mu, bytes);
                    dev::bulk_store(p.dlogstd + base, s_ls, bytes);
                    if (!final_tile) dev::bulk_store_wait_read();
                }
            } else {
                const int nelem = tr.nrows * D;
                for (int i = tid; i < nelem; i += NT) {
                    p.dmean[base + i] = s_mu[i];
                    p.dlogstd[base + i] = s_ls[i];
                }
            }
            if (!final_tile) __syncthreads();
        }
    }
    if (is_last_s) dev::reduce_published_sums<NT>(p.partials, p.counter, p.loss_terms, k.vf_coef, k.ent_coef, k.kl_coef,
                                                   k.steps_total);
    if (tid == 0) dev::bulk_store_wait_read();
}

// ------------------------------------------------------------------------------------------
// Diagonal-Gaussian policy, persistent warp-specialised form (trajectories of at most 128 steps)
// ------------------------------------------------------------------------------------------
// The structure of impact_loss_categorical_ws_kernel with five input slabs per tile (learner mean /
// log-std, target mean / log-std, actions) and two output slabs (dmean, dlogstd, written over the
// learner's): a producer warp streams tiles through the ring, C consumer groups take them as they
// land, every warp stores its own rows, the block's sums leave as one tagged row.  Row arithmetic is
// that of impact_loss_gaussian_reg_kernel (log-probabilities accumulated in fp64).  kLong as in the
// categorical kernel: tiles of a long trajectory on neighbouring blocks, linked through their aggregates.
template <int D>
__host__ __device__ constexpr size_t gaussian_ws_stage_bytes() {
    return (5 * ws_slab_pitch(128, D * sizeof(float)) + 127) / 128 * 128;
}

template <int D, int C, bool kLong>
__global__ void __launch_bounds__(C * 128 + 32, 1)
impact_loss_gaussian_ws_kernel(const __grid_constant__ GaussParams p, const int S, const int W, const int lanes,
                               const int n_prefetch) {
    constexpr int NT = 128;
    constexpr int kRow = D * (int)sizeof(float);
    constexpr int kSlab = (int)ws_slab_pitch(NT, kRow);  // rows keep their place inside their 16-byte granule
    constexpr int kStageBytes = (int)gaussian_ws_stage_bytes<D>();
    constexpr float kLog2e = 1.4426950408889634f;
    constexpr float kHalfLog2Pi = 0.91893853320467274178f;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kWsMaxStages], empty_bar[kWsMaxStages];
    __shared__ unsigned int tickets_s, tag_s;
    __shared__ float2 warp_agg[C][NT / 32];
    __shared__ __align__(16) float red[C][NT / 32][8];
    __shared__ int abort_s;
    __shared__ float carry_s[C];

    const int tid = threadIdx.x, lane = tid & 31;
    const LossScalars& k = p.k;
    const TileGeometry& g = p.geo;
    const long long total_tiles = kLong ? g.nchunks * g.ntiles : g.nchunks;
    const int n_tiles = (int)((total_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x);
    const int rows_full = kLong ? NT : g.G * (int)g.T;
    const long long total_rows = g.B * g.T;
    const long long agg_stride = g.tile_major ? 2 * g.B : 2;  // slots between a tile's aggregate and that of the tile after it in time
    auto place_of = [&](int n) { return tile_place<kLong, NT>(g, n, rows_full, total_rows); };

    if (tid >= C * NT) {
        // ---- producer warp ----------------------------------------------------------------------------------
        const float* const src[5] = {p.learner_mean, p.learner_logstd, p.target_mean, p.target_logstd, p.actions};
        const int n_first = n_tiles < W ? n_tiles : W;
        const long long tensor_bytes = total_rows * kRow;
        // the block's first tiles are asked for in L2 before the stream dependency resolves, unless the launch's
        // companion kernel has done so already (see the categorical kernel): lane a takes array a
        if (n_prefetch > 0) {
            const void* base = nullptr;
            long long pitch = 4;
            if (lane < 5) { base = src[lane]; pitch = kRow; }
            else if (lane == 5) base = p.worker_logp;
            else if (lane == 6) base = p.rewards;
            else if (lane == 7) base = p.discounts;
            else if (lane == 8) base = p.values;
            const int n_pf = n_tiles < n_prefetch ? n_tiles : n_prefetch;
            for (int n = 0; n < n_pf; ++n) {
                const Place pc = place_of(n);
                if (base) dev::prefetch_range_l2(base, pc.row0 * pitch, (uint32_t)(pc.nrows * pitch), total_rows * pitch);
            }
        }
        if (lane < S) {
            dev::mbarrier_init_nofence(&full_bar[lane], 1);
            dev::mbarrier_init_nofence(&empty_bar[lane], NT / 32);
        }
        if (lane == 0) { abort_s = 0; tickets_s = 0u; }
        dev::fence_mbarrier_init();
        __syncwarp();

        // One slab of a tile into stage s (protocol, widened copies and in-order issue as in the categorical
        // kernel): lane l < 4 owns the round's l-th tile, requests its first slab, makes the barrier's arrival
        // with the bytes of all five slabs and fetches the bytes of a last, partial granule of the tensors; lanes
        // l + 4, l + 8, l + 12, l + 16 request the tile's other slabs.
        struct SlabRequest {
            unsigned char* d;      // the stage
            long long first;       // byte offset of the tile's first granule in each of the five tensors
            uint32_t span, tail;   // dev::WideRange
        };
        auto request_for = [&](const Place& pc, int s) {
            const dev::WideRange w = dev::widen_range(pc.row0 * (long long)kRow, (uint32_t)pc.nrows * kRow, tensor_bytes);
            SlabRequest r;
            r.d = smem_raw + s * kStageBytes;
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
                        for (uint32_t i = 0; i < r.tail; ++i) r.d[j * kSlab + r.span + i] = gj[r.span + i];
                    }
                    dev::fence_async_shared();
                }
                if (r.span) dev::mbarrier_expect_tx(bar, 5 * r.span);
                else dev::mbarrier_arrive(bar);
            }
            if (r.span) dev::bulk_load(r.d + q * kSlab, gq, r.span, bar);
        };
        const int sub = lane & 3, q_lane = lane >> 2;
        const bool sends = q_lane < 5;
        const SlabRequest first = request_for(place_of(sub < n_first ? sub : 0), sub);

        grid_dependency_wait();

        // the first W tiles need no wait (tile n goes to stage n), four at a time
        if (sends && sub < n_first) send_slab(first, sub, q_lane);
        for (int base = 4; base < n_first; base += 4)
            if (sends && base + sub < n_first) send_slab(request_for(place_of(base + sub), base + sub), base + sub, q_lane);
        __syncthreads();  // the barriers are set up: the consumer warps may use them
        const unsigned int tag = dev::launch_tag(p.counter);  // (asked for now, needed after the last tile has left)
        for (int base = n_first; base < n_tiles; base += lanes) {
            const int n = base + sub;
            bool pending = sends && sub < lanes && n < n_tiles;
            const int cyc = n / S, s = n - cyc * S;
            const int wcyc = (n - W) / S, ws = (n - W) - wcyc * S;
            const SlabRequest req = request_for(place_of(pending ? n : 0), s);
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
        // this launch's tag for whoever publishes the block's sums, and the warp's own ticket
        if (lane == 0) tag_s = tag;
        dev::draw_ticket_and_publish<C, NT / 32>(&tickets_s, &tag_s, red, p.tagged_rows);
        return;
    }

    // ---- consumer groups ------------------------------------------------------------------
    const int grp = tid >> 7, gtid = tid & (NT - 1), gwarp = gtid >> 5;
    const int bar_id = grp + 1;
    const bool want_kl = (k.kl_coef != 0.0f);

    int q = 0, ts = gtid;
    if (!kLong && g.G > 1) { q = gtid / (int)g.T; ts = gtid - q * (int)g.T; }
    struct Mine {
        long long row, traj;
        bool active, last_step;
        Place pc;
    };
    auto mine_in = [&](int n) {
        Mine m;
        m.pc = place_of(n < n_tiles ? n : 0);
        m.row = m.pc.row0 + gtid;
        m.traj = m.pc.traj + q;
        m.active = n < n_tiles && gtid < m.pc.nrows;
        m.last_step = kLong ? (m.pc.r == 0 && gtid == m.pc.nrows - 1) : (ts == (int)g.T - 1);
        return m;
    };

    struct StepRaw {
        float l_worker, reward, discount, value, value_next;
    };
    auto load_scalars = [&](const Mine& m) {
        StepRaw x;
        x.l_worker = 0.0f; x.reward = 0.0f; x.discount = 0.0f; x.value = 0.0f; x.value_next = 0.0f;
        if (m.active) {
            const long long r = m.row;
            x.l_worker = p.worker_logp[r];
            x.reward = p.rewards[r];
            x.discount = p.discounts[r];
            x.value = p.values[r];
            x.value_next = m.last_step ? p.bootstrap[m.traj] : p.values[r + 1];
        }
        return x;
    };

    float t_surr = 0.0f, t_val = 0.0f, t_ent = 0.0f, t_ratio = 0.0f, t_kl = 0.0f;
    int n_clip = 0, n_trunc = 0;
    auto hand_over_sums = [&]() {
        dev::hand_over_warp_sums<C, NT / 32>(t_surr, t_val, t_ent, t_ratio, t_kl, want_kl, n_clip, n_trunc, red[grp][gwarp],
                                             &tickets_s, &tag_s, red, p.tagged_rows);
    };
    bool pending = false;
    int pending_stage = 0;

    grid_dependency_wait();
    Mine me = mine_in(grp);
    StepRaw cur = load_scalars(me);
    __syncthreads();  // the producer warp has set up the barriers
    int s = grp % S;
    uint32_t ph = (uint32_t)(grp / S) & 1u;

    for (int n = grp; n < n_tiles; n += C) {
        const Mine me_next = mine_in(n + C);
        const StepRaw nxt = load_scalars(me_next);
        const bool active = me.active;
        const long long row = me.row;
        if (lane == 0 && pending) {
            dev::bulk_store_wait_read();
            dev::mbarrier_arrive(&empty_bar[pending_stage]);
            pending = false;
        }
        // (long trajectories) one early look at the aggregates of the later tiles of this tile's trajectory: with
        // many trajectories they were published a round ago, and reading them now keeps that trip to L2 off the
        // path between this tile's scan and its gradients
        // (only where tiles are numbered tile-major; the values are first looked at after the scan)
        const bool peeked = kLong && g.tile_major && gwarp == 0 && me.pc.r > lane;
        unsigned long long early_a = 0, early_b = 0;
        if (peeked)
            dev::load_aggregate(p.tile_aggregates + 2 * ((long long)blockIdx.x + (long long)n * gridDim.x), agg_stride,
                                me.pc.r - lane, early_a, early_b);
        if (!dev::mbarrier_wait(&full_bar[s], ph, &abort_s)) atomicExch(p.counter + 1, 1u);

        // the tile's first row starts (row0 * kRow) mod 16 bytes into each slab
        unsigned char* const stage = smem_raw + s * kStageBytes + ((uint32_t)(me.pc.row0 * kRow) & 15u);
        float* const r_mu = reinterpret_cast<float*>(stage) + gtid * D;              // learner mean -> dmean
        float* const r_ls = reinterpret_cast<float*>(stage + kSlab) + gtid * D;      // learner log-std -> dlogstd
        const float* const r_mt = reinterpret_cast<const float*>(stage + 2 * kSlab) + gtid * D;
        const float* const r_lt = reinterpret_cast<const float*>(stage + 3 * kSlab) + gtid * D;
        const float* const r_ac = reinterpret_cast<const float*>(stage + 4 * kSlab) + gtid * D;
        dev::StepIn st;
        st.reward = cur.reward;
        st.discount = cur.discount;
        st.value = cur.value;
        st.value_next = cur.value_next;
        st.last_step = me.last_step;

        // ---- row pass (every thread; rows beyond the tile hold stale bytes and are masked)
        float ent, kl = 0.0f;
        {
            // log-probabilities: D-term sums of magnitude tens that end up in exponents, so they are
            // accumulated in fp64
            double lth = 0.0, ltg = 0.0;
            float ls_sum = 0.0f;
#pragma unroll
            for (int j = 0; j < D; ++j) {
                const float ls = r_ls[j], lt = r_lt[j], ac = r_ac[j], mu = r_mu[j], mt = r_mt[j];
                const float inv_s = dev::exp2_fast(-ls * kLog2e), inv_st = dev::exp2_fast(-lt * kLog2e);
                const float z1 = (ac - mu) * inv_s;
                const float z2 = (ac - mt) * inv_st;
                lth += (double)fmaf(-0.5f * z1, z1, -ls);
                ltg += (double)fmaf(-0.5f * z2, z2, -lt);
                ls_sum += ls;
                if (want_kl) {  // KL(target || learner), per dimension
                    const float dm = (mt - mu) * inv_s;
                    const float sr = dev::exp2_fast((lt - ls) * kLog2e);
                    kl += (ls - lt) + 0.5f * fmaf(sr, sr, dm * dm) - 0.5f;
                }
            }
            ent = ls_sum + (float)D * (kHalfLog2Pi + 0.5f);
            const double shift = (double)cur.l_worker + (double)D * (double)kHalfLog2Pi;
            // everything downstream works on log-probabilities relative to the worker's
            st.l_theta = (float)(lth - shift);
            st.l_target = (float)(ltg - shift);
            st.l_worker = 0.0f;
            st.l_shift = cur.l_worker;
        }
        float fa, fb;
        const bool truncated = dev::recursion_map(st, k, fa, fb);
        if (!active) { fa = 1.0f; fb = 0.0f; }
        float adv;
        if (!kLong) {
            adv = dev::suffix_affine_scan_group<NT>(fa, fb, warp_agg[grp], st.adv_next, bar_id);
        } else {
            float ma, mb, la, lb;
            dev::suffix_affine_maps_group<NT>(fa, fb, warp_agg[grp], ma, mb, la, lb, bar_id);
            const long long gtile = (long long)blockIdx.x + (long long)n * gridDim.x;
            if (gtid == 0) dev::publish_tile_aggregate(p.tile_aggregates + 2 * gtile, ma, mb, dev::launch_tag(p.counter));
            float carry = 0.0f;
            if (me.pc.r > 0) {  // uniform over the group
                if (gwarp == 0) {
                    const float c = dev::compose_later_aggregates(p.tile_aggregates + 2 * gtile, agg_stride, me.pc.r,
                                                                  dev::launch_tag(p.counter), &abort_s, peeked,
                                                                  early_a, early_b);
                    if (lane == 0) carry_s[grp] = c;
                }
                asm volatile("bar.sync %0, 128;" ::"r"(bar_id) : "memory");
                carry = carry_s[grp];
            }
            adv = fmaf(ma, carry, mb);
            const float below = __shfl_down_sync(0xffffffffu, adv, 1);
            st.adv_next = (lane == 31) ? fmaf(la, carry, lb) : below;
        }

        float surr, ratio;
        bool clipped;
        const float wpg = dev::surrogate(st, k, adv, surr, ratio, clipped);
        if (active) {
            t_surr += surr;
            t_val = fmaf(0.5f * adv, adv, t_val);
            t_ent += ent;
            t_ratio += ratio;
            t_kl += kl;
        }
        n_clip += __popc(__ballot_sync(0xffffffffu, active && clipped));
        n_trunc += __popc(__ballot_sync(0xffffffffu, active && truncated));
        if (n + C >= n_tiles) hand_over_sums();

        // ---- gradients, in place over the learner's slabs
        {
            const float w1 = wpg * k.inv_M, ce = k.ent_coef * k.inv_M, ck = k.kl_coef * k.inv_M;
#pragma unroll
            for (int j = 0; j < D; ++j) {
                const float ls = r_ls[j], mu = r_mu[j];
                const float inv_s = dev::exp2_fast(-ls * kLog2e);
                const float z = (r_ac[j] - mu) * inv_s;  // (a - mu) / sigma
                // d log pi / d mu = z / sigma ;  d log pi / d logstd = z^2 - 1 ;  d H / d logstd = 1
                float gm = -w1 * z;
                float gs = -w1 * fmaf(z, z, -1.0f) - ce;
                if (want_kl) {
                    const float dm = (mu - r_mt[j]) * inv_s;
                    const float sr = dev::exp2_fast((r_lt[j] - ls) * kLog2e);
                    gm = fmaf(ck, dm, gm);
                    gs = fmaf(ck, 1.0f - fmaf(sr, sr, dm * dm), gs);
                }
                r_mu[j] = gm * inv_s;
                r_ls[j] = gs;
            }
            if (active) {
                p.dvalues[row] = -k.vf_coef * k.inv_M * adv;
                if (p.vtarget) p.vtarget[row] = st.value + adv;
                if (p.advantage) p.advantage[row] = adv;
            }
        }
        // ---- each warp sends its own 32 rows of both gradient slabs
        {
            const long long wrow0 = row - lane;
            const int left = me.pc.nrows - (gtid - lane);
            const int wrows = left > 32 ? 32 : (left > 0 ? left : 0);
            unsigned char* const gm = reinterpret_cast<unsigned char*>(p.dmean) + wrow0 * (long long)kRow;
            unsigned char* const gs = reinterpret_cast<unsigned char*>(p.dlogstd) + wrow0 * (long long)kRow;
            const unsigned char* const src_m = stage + (gtid - lane) * kRow;
            bool stored = dev::warp_send_bytes(gm, src_m, (uint32_t)wrows * kRow, true);
            if (dev::warp_send_bytes(gs, src_m + kSlab, (uint32_t)wrows * kRow, false)) stored = true;  // (fenced above)
            if (lane == 0) {
                if (stored) {
                    pending = n_tiles > S;  // a block with no more tiles than stages never needs a stage back
                    pending_stage = s;
                } else {
                    dev::mbarrier_arrive(&empty_bar[s]);
                }
            }
        }
        cur = nxt;
        me = me_next;
        s += C;
        while (s >= S) { s -= S; ph ^= 1u; }
    }

    if (grp >= n_tiles) hand_over_sums();
    if (blockIdx.x == 0 && grp == n_tiles % C) {
        if (!dev::reduce_tagged_rows<NT>(p.tagged_rows, (int)gridDim.x, dev::launch_tag(p.counter), p.counter,
                                         p.loss_terms, k.vf_coef, k.ent_coef, k.kl_coef, k.steps_total,
                                         gtid, bar_id, &abort_s))
            if (gtid == 0) atomicExch(p.counter + 1, 1u);
    }
    if (lane == 0) dev::bulk_store_wait_read();
}

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
// Long trajectories (T > 128 steps): two (value, tag) pairs per 128-step tile, after everything else.
size_t tile_aggregate_bytes(int64_t B, int64_t T) {
    if (T <= kMinTileRows) return 0;
    return (size_t)B * (size_t)((T + kMinTileRows - 1) / kMinTileRows) * 2 * sizeof(unsigned long long);
}

constexpr size_t kWorkspaceFixedBytes = (size_t)kMaxGridBlocks * 8 * sizeof(float) + kCounterBytes +
                                        (size_t)kMaxTaggedRows * 8 * sizeof(unsigned long long);

int pad_odd(int w) { return (w & 1) ? w : w + 1; }

// Threads per block = rows per tile: as many as keep a tile's staged slabs within
// `budget` bytes of shared memory, so that several blocks stay resident per SM.
int pick_nt(int width_padded, int n_slabs, size_t budget) {
    for (int nt : {128, 64}) {
        if ((size_t)nt * width_padded * n_slabs * sizeof(float) <= budget) return nt;
    }
    return 32;
}

TileGeometry make_geometry(int64_t B, int64_t T, int nt) {
    TileGeometry g;
    g.tile_major = 0;
    g.B = B;
    g.T = T;
    if (T <= nt) {
        g.G = (int)(nt / T);
        g.ntiles = 1;
        g.nchunks = (B + g.G - 1) / g.G;
    } else {
        g.G = 1;
        g.ntiles = (int)((T + nt - 1) / nt);
        g.nchunks = B;
    }
    return g;
}

bool bad_scalar(float x) { return !(x >= 0.0f); }  // negative or NaN

int32_t fill_scalars(LossScalars& k, float rho_bar, float c_bar, float clip_eps,
                     const impact_coefficients* coef, int64_t B, int64_t T) {
    if (bad_scalar(rho_bar) || bad_scalar(c_bar) || bad_scalar(clip_eps)) return IMPACT_ERR_INVALID_ARG;
    if (!(coef->rho_tw > 0.0f) || !isfinite(coef->vf_coef) || !isfinite(coef->ent_coef) ||
        !isfinite(coef->kl_coef) || !isfinite(coef->lambda_))
        return IMPACT_ERR_INVALID_ARG;
    if (coef->is_source < IMPACT_IS_TARGET_OVER_WORKER || coef->is_source > IMPACT_IS_NONE) return IMPACT_ERR_INVALID_ARG;
    if (coef->objective != IMPACT_OBJECTIVE_CLIPPED_SURROGATE && coef->objective != IMPACT_OBJECTIVE_VTRACE_PG)
        return IMPACT_ERR_INVALID_ARG;
    if (coef->ratio_mode < IMPACT_RATIO_R3 || coef->ratio_mode > IMPACT_RATIO_R2) return IMPACT_ERR_INVALID_ARG;
    k.rho_bar = rho_bar;
    k.c_bar = c_bar;
    k.clip_lo = 1.0f - clip_eps;
    k.clip_hi = 1.0f + clip_eps;
    k.vf_coef = coef->vf_coef;
    k.ent_coef = coef->ent_coef;
    k.kl_coef = coef->kl_coef;
    k.lambda_ = coef->lambda_;
    k.log_rho_tw = (float)log((double)coef->rho_tw);
    const double own = (double)B * (double)T;
    if (coef->global_steps != 0 && (double)coef->global_steps < own) return IMPACT_ERR_INVALID_ARG;
    k.steps_total = coef->global_steps != 0 ? (double)coef->global_steps : own;
    k.inv_M = (float)(1.0 / k.steps_total);
    k.ent_over_M = k.ent_coef * k.inv_M;
    k.kl_over_M = k.kl_coef * k.inv_M;
    k.dvalue_over_adv = -k.vf_coef * k.inv_M;
    k.log2_rho_tw = (float)log2((double)coef->rho_tw);
    k.is_source = coef->is_source;
    k.ratio_mode = coef->ratio_mode;
    k.objective = coef->objective;
    return IMPACT_OK;
}

// Blocks to launch: every chunk gets its own block while all of them can be resident at
// once; beyond that, a resident-sized grid walks the chunks.
template <typename Kernel>
int32_t grid_for(Kernel kernel, int nt, size_t smem, long long nchunks, const DeviceInfo* di, int* grid) {
    struct Key { const void* fn; size_t smem; int dev; int per_sm; };
    static thread_local Key cache[16];
    static thread_local int ncache = 0;
    int per_sm = -1;
    for (int i = 0; i < ncache; ++i)
        if (cache[i].fn == (const void*)kernel && cache[i].smem == smem && cache[i].dev == di->device)
            per_sm = cache[i].per_sm;
    if (per_sm < 0) {
        if (smem > 48 * 1024)
            IMPACT_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        IMPACT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, nt, smem));
        if (per_sm < 1) return IMPACT_ERR_UNSUPPORTED;
        if (ncache < 16) cache[ncache++] = Key{(const void*)kernel, smem, di->device, per_sm};
    }
    long long resident = (long long)per_sm * di->sm_count;
    if (resident > kMaxGridBlocks) resident = kMaxGridBlocks;
    *grid = (int)(nchunks < resident ? nchunks : resident);
    return IMPACT_OK;
}

}  // namespace

// Tiles the producer keeps in flight and stages of the ring, for tiles of `tile_in_bytes` bytes of logits.
// Bytes in flight per SM (IMPACT_OPT_WINDOW_BYTES; 0 = chosen here): 72 KB where a block streams many tiles (over
// 148 SMs that covers HBM's latency at full bandwidth; measured: 64 KB and more reach the copy rate, 48 KB stop at
// 0.9 of it), 48 KB where a block has only a few (a bigger first burst makes every tile of it land later, and the
// first tile's landing is what such a launch waits for).  Beyond the window there is room for the tiles being
// worked on and being stored.  The barrier protocol needs stages >= in_flight + groups, or exactly one stage per
// group (then the stage's previous tile is the one the same group worked on last); 0 stages = no valid shape.
void ws_ring_shape(size_t stage_bytes, size_t tile_in_bytes, int groups, int max_smem, long long tiles_per_block,
                   int* stages, int* in_flight) {
    size_t window = (size_t)option(IMPACT_OPT_WINDOW_BYTES);
    if (window == 0) window = tiles_per_block <= 8 ? 48 * 1024 : 72 * 1024;
    int w = (int)((window + tile_in_bytes - 1) / tile_in_bytes);
    if (w < 2) w = 2;
    if (w > 8) w = 8;
    int s = w + groups + 3;
    if (s > kWsMaxStages) s = kWsMaxStages;
    const int fit = (int)((size_t)(max_smem - 4096) / stage_bytes);  // 4 KB left for static shared memory
    if (s > fit) s = fit;
    if (tiles_per_block <= s) {
        // no stage is used twice: every barrier sees one phase only, and any number of tiles may be in flight
        if (w > s) w = s;
    } else if (s > groups) {
        if (w > s - groups) w = s - groups;
    } else if (s == groups) {
        if (w > s) w = s;
    } else {
        s = 0;
    }
    *stages = s;
    *in_flight = w;
}

// How a persistent kernel is launched for a batch of `tiles` tiles on `grid` blocks.
WsPlan ws_plan(long long tiles, long long grid, size_t tile_bytes, int in_flight, bool allow_companion) {
    WsPlan pl;
    const long long per_block = (tiles + grid - 1) / grid;
    const long long budget = option(IMPACT_OPT_PREFETCH_BYTES);
    long long pf = budget / (grid * (long long)tile_bytes);
    // Asking L2 for tiles ahead of time goes through the copy engine like the tiles themselves, so it pays only
    // where requests are large (measured: with 12-21 KB tiles a short launch gains half a microsecond from its
    // companion and a third from asking itself; with 3-9 KB tiles either costs 5-15 %).  The companion pays where a
    // launch is short: a block has a handful of tiles, all within the budget.  A long launch is bound by HBM either
    // way, and asking for many tiles far ahead of their use only competes with the tiles that are needed now.
    // Without a companion the loss kernel's first warp asks for the tiles it is about to request anyway (more than
    // that sits in the copy engine's queue ahead of the requests themselves).
    const bool large_tiles = tile_bytes >= 10 * 1024;
    // (measured on 18 actions: a gain from five tiles per block on -- 8.3 -> 7.6 us at seven --, nothing at three
    // to four, a loss of a quarter of a microsecond at two)
    pl.companion = allow_companion && large_tiles && option(IMPACT_OPT_EARLY_PREFETCH) != 0 && pf >= per_block &&
                   per_block >= 4 && per_block <= 8;
    if (!large_tiles) pf = 0;
    if (!pl.companion && pf > in_flight) pf = in_flight;
    if (pf > per_block) pf = per_block;
    pl.prefetch_tiles = (int)pf;
    return pl;
}

namespace {

template <int NT>
int32_t launch_gaussian(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream) {
    auto kernel = impact_loss_gaussian_kernel<NT>;
    const size_t smem = (size_t)5 * NT * p.Ds * sizeof(float);
    int grid = 0;
    int32_t st = grid_for(kernel, NT, smem, p.geo.nchunks, di, &grid);
    if (st != IMPACT_OK) return st;
    IMPACT_CUDA_TRY(launch_serialized(kernel, dim3(grid), dim3(NT), smem, stream, p));
    return IMPACT_OK;
}

constexpr int kWsGroupsGaussian = 3;  // consumer groups: five slabs per tile leave room for five stages at D = 17

template <int D, bool kLong>
int32_t launch_gaussian_ws(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream) {
    constexpr int C = kWsGroupsGaussian;
    auto kernel = impact_loss_gaussian_ws_kernel<D, C, kLong>;
    const size_t stage = gaussian_ws_stage_bytes<D>();
    const long long tiles = kLong ? p.geo.nchunks * p.geo.ntiles : p.geo.nchunks;
    long long grid = tiles < di->sm_count ? tiles : di->sm_count;
    if (grid > kMaxTaggedRows) grid = kMaxTaggedRows;  // one tagged row per block
    int S = 0, W = 0;
    ws_ring_shape(stage, stage, C, di->max_smem_optin, (tiles + grid - 1) / grid, &S, &W);
    if (S < 1 || W < 1) return IMPACT_ERR_UNSUPPORTED;
    const size_t smem = (size_t)S * stage;
    static thread_local int configured_device = -1;
    if (configured_device != di->device) {
        IMPACT_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, di->max_smem_optin - 4096));
        configured_device = di->device;
    }
    const int lanes = (S - W) < 4 ? ((S - W) < 1 ? 1 : (S - W)) : 4;  // tiles the producer requests side by side
    GaussParams q = p;
    q.geo.tile_major = (kLong && p.geo.B >= grid) ? 1 : 0;
    const int rows_full = kLong ? 128 : q.geo.G * (int)q.geo.T;
    // (no companion here: measured on B = 512, T = 128, D = 17 it costs more of the copy engine's time than the
    // earlier start gains: 10.7 us per launch with it, 8.8 us without)
    const WsPlan plan = ws_plan(tiles, grid, (size_t)rows_full * (5 * D * sizeof(float) + 16), W, false);
    IMPACT_CUDA_TRY(launch_serialized(kernel, dim3((unsigned)grid), dim3(C * 128 + 32), smem, stream, q, S, W, lanes,
                                      plan.prefetch_tiles));
    return IMPACT_OK;
}

template <int D>
int32_t launch_gaussian_reg(const GaussParams& p, const DeviceInfo* di, cudaStream_t stream) {
    if (p.geo.ntiles == 1) return launch_gaussian_ws<D, false>(p, di, stream);
    if (p.tile_aggregates) return launch_gaussian_ws<D, true>(p, di, stream);
    auto kernel = impact_loss_gaussian_reg_kernel<D>;
    const size_t smem = (size_t)5 * kRegTileRows * D * sizeof(float);
    int grid = 0;
    int32_t st = grid_for(kernel, kRegTileRows, smem, p.geo.nchunks, di, &grid);
    if (st != IMPACT_OK) return st;
    IMPACT_CUDA_TRY(launch_serialized(kernel, dim3(grid), dim3(kRegTileRows), smem, stream, p));
    return IMPACT_OK;
}

// Action dimensions with a compiled register-resident kernel (the MuJoCo tasks of Section 4.3).
constexpr bool has_gaussian_reg_kernel(int D) { return D == 3 || D == 6 || D == 17; }

}  // namespace
}  // namespace impact

using namespace impact;

extern "C" size_t impact_loss_workspace_bytes(int64_t B, int64_t T) {
    if (B <= 0 || T <= 0) return 0;
    return kWorkspaceFixedBytes + tile_aggregate_bytes(B, T);
}

extern "C" int32_t impact_loss_workspace_init(void* workspace, size_t workspace_bytes, void* stream) {
    if (!workspace || !aligned16(workspace) || workspace_bytes == 0) return IMPACT_ERR_INVALID_ARG;
    IMPACT_CUDA_TRY(cudaMemsetAsync(workspace, 0, workspace_bytes, static_cast<cudaStream_t>(stream)));
    return IMPACT_OK;
}

extern "C" int32_t impact_loss_workspace_status(const void* workspace, size_t workspace_bytes, int32_t* flag_out,
                                                void* stream) {
    if (!workspace || !flag_out || !aligned16(workspace)) return IMPACT_ERR_INVALID_ARG;
    if (workspace_bytes < impact_loss_workspace_bytes(1, 1)) return IMPACT_ERR_WORKSPACE_TOO_SMALL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const char* word = static_cast<const char*>(workspace) + (size_t)kMaxGridBlocks * 8 * sizeof(float) + sizeof(unsigned int);
    unsigned int flag = 0;
    IMPACT_CUDA_TRY(cudaMemcpyAsync(&flag, word, sizeof(flag), cudaMemcpyDeviceToHost, s));
    IMPACT_CUDA_TRY(cudaStreamSynchronize(s));
    *flag_out = (int32_t)flag;
    return IMPACT_OK;
}

static int32_t run_typed(const CatParams& p, bool logits_bf16, bool grads_bf16, const DeviceInfo* di, cudaStream_t s) {
    if (!logits_bf16 && !grads_bf16) return run_categorical<float, float>(p, di, s);
    if (!logits_bf16) return run_categorical<float, __nv_bfloat16>(p, di, s);
    if (!grads_bf16) return run_categorical<__nv_bfloat16, float>(p, di, s);
    return run_categorical<__nv_bfloat16, __nv_bfloat16>(p, di, s);
}

static int32_t loss_fwd_bwd_impl(
    const void* learner_logits, const void* target_logits, const float* worker_logp,
    const int32_t* actions, const float* rewards, const float* discounts, const float* values,
    const float* bootstrap_values, float rho_bar, float c_bar, float clip_eps,
    const impact_coefficients* coef, int64_t B, int64_t T, int32_t A, int32_t logits_dtype,
    float* loss_terms, void* dlogits, float* dvalues, float* vtarget, float* advantage,
    void* workspace, size_t workspace_bytes, void* target_logits_copy, const impact_loss_inputs* indirect, void* stream) {
    if (!coef || !loss_terms || !dlogits || !dvalues || !workspace) return IMPACT_ERR_INVALID_ARG;
    if (indirect) {  // the inputs come from a record in device memory: the pointers passed here are not looked at
        if (!aligned16(indirect)) return IMPACT_ERR_INVALID_ARG;
        learner_logits = target_logits = nullptr;
        worker_logp = rewards = discounts = values = bootstrap_values = nullptr;
        actions = nullptr;
        target_logits_copy = nullptr;
    } else if (!learner_logits || !target_logits || !worker_logp || !actions || !rewards || !discounts || !values ||
               !bootstrap_values) {
        return IMPACT_ERR_INVALID_ARG;
    }
    if (B <= 0 || T <= 0 || A <= 0) return IMPACT_ERR_INVALID_ARG;
    const void* ptrs[] = {learner_logits, target_logits, worker_logp, actions, rewards, discounts,
                          values, bootstrap_values, loss_terms, dlogits, dvalues, workspace};
    for (const void* q : ptrs)
        if (!aligned16(q)) return IMPACT_ERR_INVALID_ARG;
    if ((vtarget && !aligned16(vtarget)) || (advantage && !aligned16(advantage))) return IMPACT_ERR_INVALID_ARG;
    if (target_logits_copy && (!aligned16(target_logits_copy) || target_logits_copy == target_logits))
        return IMPACT_ERR_INVALID_ARG;
    if (logits_dtype != IMPACT_DTYPE_F32 && logits_dtype != IMPACT_DTYPE_BF16) return IMPACT_ERR_INVALID_ARG;
    if (coef->dlogits_dtype != IMPACT_DTYPE_F32 && coef->dlogits_dtype != IMPACT_DTYPE_BF16)
        return IMPACT_ERR_INVALID_ARG;
    if (A > 512) return IMPACT_ERR_UNSUPPORTED;
    if ((double)B * (double)T * (double)A >= 1099511627776.0 || (double)B * (double)T >= 4.0e12)
        return IMPACT_ERR_UNSUPPORTED;
    if (workspace_bytes < kWorkspaceFixedBytes) return IMPACT_ERR_WORKSPACE_TOO_SMALL;

    CatParams p = {};
    int32_t st = fill_scalars(p.k, rho_bar, c_bar, clip_eps, coef, B, T);
    if (st != IMPACT_OK) return st;
    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;

    p.learner_logits = learner_logits;
    p.target_logits = target_logits;
    p.worker_logp = worker_logp;
    p.actions = actions;
    p.rewards = rewards;
    p.discounts = discounts;
    p.values = values;
    p.bootstrap = bootstrap_values;
    p.loss_terms = loss_terms;
    p.dlogits = dlogits;
    p.dvalues = dvalues;
    p.vtarget = vtarget;
    p.advantage = advantage;
    p.counter = reinterpret_cast<unsigned int*>(static_cast<char*>(workspace) +
                                                (size_t)kMaxGridBlocks * 8 * sizeof(float));
    p.tagged_rows = reinterpret_cast<unsigned long long*>(static_cast<char*>(workspace) +
                                                          (size_t)kMaxGridBlocks * 8 * sizeof(float) + kCounterBytes);
    // room for the tiles' aggregates is optional: without it long trajectories are swept inside one block
    p.tile_aggregates = (T > kMinTileRows && workspace_bytes >= impact_loss_workspace_bytes(B, T))
                            ? reinterpret_cast<unsigned long long*>(static_cast<char*>(workspace) + kWorkspaceFixedBytes)
                            : nullptr;
    p.target_copy = target_logits_copy;
    p.indirect = indirect;
    p.A = A;
    p.geo.B = B;
    p.geo.T = T;
    return run_typed(p, logits_dtype == IMPACT_DTYPE_BF16, coef->dlogits_dtype == IMPACT_DTYPE_BF16, di,
                     static_cast<cudaStream_t>(stream));
}

extern "C" int32_t impact_loss_fwd_bwd(
    const void* learner_logits, const void* target_logits, const float* worker_logp,
    const int32_t* actions, const float* rewards, const float* discounts, const float* values,
    const float* bootstrap_values, float rho_bar, float c_bar, float clip_eps,
    const impact_coefficients* coef, int64_t B, int64_t T, int32_t A, int32_t logits_dtype,
    float* loss_terms, void* dlogits, float* dvalues, float* vtarget, float* advantage,
    void* workspace, size_t workspace_bytes, void* stream) {
    return loss_fwd_bwd_impl(learner_logits, target_logits, worker_logp, actions, rewards, discounts, values,
                             bootstrap_values, rho_bar, c_bar, clip_eps, coef, B, T, A, logits_dtype, loss_terms,
                             dlogits, dvalues, vtarget, advantage, workspace, workspace_bytes, nullptr, nullptr, stream);
}

extern "C" int32_t impact_loss_fwd_bwd_call(const impact_loss_call* c, void* stream) {
    if (!c) return IMPACT_ERR_INVALID_ARG;
    return loss_fwd_bwd_impl(c->learner_logits, c->target_logits, c->worker_logp, c->actions, c->rewards,
                             c->discounts, c->values, c->bootstrap_values, c->rho_bar, c->c_bar, c->clip_eps,
                             &c->coef, c->B, c->T, c->A, c->logits_dtype, c->loss_terms, c->dlogits,
                             c->dvalues, c->vtarget, c->advantage, c->workspace, c->workspace_bytes,
                             c->target_logits_copy, c->inputs_on_device, stream);
}

extern "C" int32_t impact_loss_fwd_bwd_gaussian(
    const float* learner_mean, const float* learner_logstd, const float* target_mean,
    const float* target_logstd, const float* worker_logp, const float* actions,
    const float* rewards, const float* discounts, const float* values,
    const float* bootstrap_values, float rho_bar, float c_bar, float clip_eps,
    const impact_coefficients* coef, int64_t B, int64_t T, int32_t D,
    float* loss_terms, float* dmean, float* dlogstd, float* dvalues, float* vtarget,
    float* advantage, void* workspace, size_t workspace_bytes, void* stream) {
    if (!learner_mean || !learner_logstd || !target_mean || !target_logstd || !worker_logp ||
        !actions || !rewards || !discounts || !values || !bootstrap_values || !coef || !loss_terms ||
        !dmean || !dlogstd || !dvalues || !workspace)
        return IMPACT_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || D <= 0) return IMPACT_ERR_INVALID_ARG;
    const void* ptrs[] = {learner_mean, learner_logstd, target_mean, target_logstd, worker_logp,
                          actions, rewards, discounts, values, bootstrap_values, loss_terms,
                          dmean, dlogstd, dvalues, workspace};
    for (const void* q : ptrs)
        if (!aligned16(q)) return IMPACT_ERR_INVALID_ARG;
    if ((vtarget && !aligned16(vtarget)) || (advantage && !aligned16(advantage))) return IMPACT_ERR_INVALID_ARG;
    if (coef->dlogits_dtype != IMPACT_DTYPE_F32) return IMPACT_ERR_INVALID_ARG;
    if (D > 256) return IMPACT_ERR_UNSUPPORTED;
    if ((double)B * (double)T * (double)D >= 1099511627776.0 || (double)B * (double)T >= 4.0e12)
        return IMPACT_ERR_UNSUPPORTED;
    if (workspace_bytes < kWorkspaceFixedBytes) return IMPACT_ERR_WORKSPACE_TOO_SMALL;

    GaussParams p;
    int32_t st = fill_scalars(p.k, rho_bar, c_bar, clip_eps, coef, B, T);
    if (st != IMPACT_OK) return st;
    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;

    p.learner_mean = learner_mean;
    p.learner_logstd = learner_logstd;
    p.target_mean = target_mean;
    p.target_logstd = target_logstd;
    p.actions = actions;
    p.worker_logp = worker_logp;
    p.rewards = rewards;
    p.discounts = discounts;
    p.values = values;
    p.bootstrap = bootstrap_values;
    p.loss_terms = loss_terms;
    p.dmean = dmean;
    p.dlogstd = dlogstd;
    p.dvalues = dvalues;
    p.vtarget = vtarget;
    p.advantage = advantage;
    p.partials = static_cast<float*>(workspace);
    p.counter = reinterpret_cast<unsigned int*>(static_cast<char*>(workspace) +
                                                (size_t)kMaxGridBlocks * 8 * sizeof(float));
    p.tagged_rows = reinterpret_cast<unsigned long long*>(static_cast<char*>(workspace) +
                                                          (size_t)kMaxGridBlocks * 8 * sizeof(float) + kCounterBytes);
    p.tile_aggregates = (T > kRegTileRows && workspace_bytes >= impact_loss_workspace_bytes(B, T))
                            ? reinterpret_cast<unsigned long long*>(static_cast<char*>(workspace) + kWorkspaceFixedBytes)
                            : nullptr;
    p.D = D;
    if (has_gaussian_reg_kernel(D)) {
        p.Ds = D;
        p.geo = make_geometry(B, T, kRegTileRows);
        cudaStream_t rs = static_cast<cudaStream_t>(stream);
        switch (D) {
            case 3: return launch_gaussian_reg<3>(p, di, rs);
            case 6: return launch_gaussian_reg<6>(p, di, rs);
            default: return launch_gaussian_reg<17>(p, di, rs);
        }
    }
    p.Ds = pad_odd(D);
    const int nt = pick_nt(p.Ds, 5, 100 * 1024);
    p.geo = make_geometry(B, T, nt);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    switch (nt) {
        case 128: return launch_gaussian<128>(p, di, s);
        case 64: return launch_gaussian<64>(p, di, s);
        default: return launch_gaussian<32>(p, di, s);
    }
}

// ------------------------------------------------------------------------------------------
// Variant for callers that must not allocate
// ------------------------------------------------------------------------------------------
namespace impact {
namespace {

constexpr int kStaticMaxBlocks = 1024;  // tiles (= blocks) the built-in scratch has room for
constexpr size_t kStaticScratchBytes = (size_t)kStaticMaxBlocks * 8 * sizeof(float) + kCounterBytes +
                                       (size_t)kMaxTaggedRows * 8 * sizeof(unsigned long long);

// Scratch that lives in the library image, laid out like a workspace: per-block sums, 256 bytes of
// counter words, the tagged rows of the persistent kernel.  Every device that loads the library
// carries its own copy.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

// Steps per tile that the limit on a call's size is counted in.
int static_scratch_tile_rows(int A, int64_t T, bool logits_bf16, bool grads_bf16) {
    if (A == 4 || A == 6 || A == 9 || A == 18) return 128;
    if (A == 64 && T <= 64) return 64;
    const size_t in = logits_bf16 ? 2 : 4, out = grads_bf16 ? 2 : 4;
    const size_t row = (size_t)A * (2 * in + (in == out ? 0 : out));
    return 128 * row <= 72 * 1024 ? 128 : 64;  // (A <= 64: 64 rows always fit)
}

// Device address of g_static_scratch on the current device.  In host code the symbol's name
// is only a handle, so the address is asked for once per device and remembered.
int32_t static_scratch_address(const DeviceInfo* di, unsigned char** out) {
    static unsigned char* address[64] = {};
    if (!address[di->device]) {
        void* p = nullptr;
        IMPACT_CUDA_TRY(cudaGetSymbolAddress(&p, g_static_scratch));
        address[di->device] = static_cast<unsigned char*>(p);
    }
    *out = address[di->device];
    return IMPACT_OK;
}

}  // namespace
}  // namespace impact

extern "C" int32_t impact_loss_fwd_bwd_static_scratch(
    const void* learner_logits, const void* target_logits, const float* worker_logp,
    const int32_t* actions, const float* rewards, const float* discounts, const float* values,
    const float* bootstrap_values, float rho_bar, float c_bar, float clip_eps,
    const impact_coefficients* coef, int64_t B, int64_t T, int32_t A, int32_t logits_dtype,
    float* loss_terms, void* dlogits, float* dvalues, float* vtarget, float* advantage,
    void* stream) {
    if (!learner_logits || !target_logits || !worker_logp || !actions || !rewards || !discounts ||
        !values || !bootstrap_values || !coef || !loss_terms || !dlogits || !dvalues)
        return IMPACT_ERR_INVALID_ARG;
    if (B <= 0 || T <= 0 || A <= 0) return IMPACT_ERR_INVALID_ARG;
    const void* ptrs[] = {learner_logits, target_logits, worker_logp, actions, rewards, discounts,
                          values, bootstrap_values, loss_terms, dlogits, dvalues};
    for (const void* q : ptrs)
        if (!aligned16(q)) return IMPACT_ERR_INVALID_ARG;
    if ((vtarget && !aligned16(vtarget)) || (advantage && !aligned16(advantage))) return IMPACT_ERR_INVALID_ARG;
    if (logits_dtype != IMPACT_DTYPE_F32 && logits_dtype != IMPACT_DTYPE_BF16) return IMPACT_ERR_INVALID_ARG;
    if (coef->dlogits_dtype != IMPACT_DTYPE_F32 && coef->dlogits_dtype != IMPACT_DTYPE_BF16)
        return IMPACT_ERR_INVALID_ARG;
    if (A > 64) return IMPACT_ERR_UNSUPPORTED;  // keeps the tile at 64 steps or more, which the limit below counts in

    CatParams p = {};
    int32_t st = fill_scalars(p.k, rho_bar, c_bar, clip_eps, coef, B, T);
    if (st != IMPACT_OK) return st;
    p.A = A;
    // the documented limit: 1024 tiles of 128 steps, or of 64 where rows are wider than 32 actions
    const bool logits_bf16 = logits_dtype == IMPACT_DTYPE_BF16, grads_bf16 = coef->dlogits_dtype == IMPACT_DTYPE_BF16;
    if (make_geometry(B, T, static_scratch_tile_rows(A, T, logits_bf16, grads_bf16)).nchunks > kStaticMaxBlocks)
        return IMPACT_ERR_WORKSPACE_TOO_SMALL;

    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;
    unsigned char* scratch = nullptr;
    st = static_scratch_address(di, &scratch);
    if (st != IMPACT_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the scratch keeps whatever the previous call left: the error word is sticky until
    // impact_loss_static_scratch_status clears it, and the launch number tells this call's rows from the previous call's
    unsigned char* counter = scratch + (size_t)kStaticMaxBlocks * 8 * sizeof(float);

    p.learner_logits = learner_logits;
    p.target_logits = target_logits;
    p.worker_logp = worker_logp;
    p.actions = actions;
    p.rewards = rewards;
    p.discounts = discounts;
    p.values = values;
    p.bootstrap = bootstrap_values;
    p.loss_terms = loss_terms;
    p.dlogits = dlogits;
    p.dvalues = dvalues;
    p.vtarget = vtarget;
    p.advantage = advantage;
    p.counter = reinterpret_cast<unsigned int*>(counter);
    p.tagged_rows = reinterpret_cast<unsigned long long*>(counter + kCounterBytes);
    p.tile_aggregates = nullptr;  // a long trajectory stays with one block
    p.target_copy = nullptr;
    p.geo.B = B;
    p.geo.T = T;
    // the same kernels, chosen the same way, as impact_loss_fwd_bwd
    return run_typed(p, logits_bf16, grads_bf16, di, s);
}

extern "C" int32_t impact_loss_static_scratch_status(int32_t* flag_out, int32_t clear, void* stream) {
    if (!flag_out) return IMPACT_ERR_INVALID_ARG;
    const DeviceInfo* di = current_device_info();
    if (!di) return IMPACT_ERR_CUDA;
    unsigned char* scratch = nullptr;
    const int32_t st = static_scratch_address(di, &scratch);
    if (st != IMPACT_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned char* word = scratch + (size_t)kStaticMaxBlocks * 8 * sizeof(float) + sizeof(unsigned int);
    unsigned int flag = 0;
    IMPACT_CUDA_TRY(cudaMemcpyAsync(&flag, word, sizeof(flag), cudaMemcpyDeviceToHost, s));
    IMPACT_CUDA_TRY(cudaStreamSynchronize(s));
    if (clear && flag != 0) IMPACT_CUDA_TRY(cudaMemsetAsync(word, 0, sizeof(unsigned int), s));
    *flag_out = (int32_t)flag;
    return IMPACT_OK;
}
