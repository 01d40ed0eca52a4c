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

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
// Trajectories longer than the smallest tile: two (value, tag) pairs per tile of 64 steps, after everything else.
size_t tile_aggregate_bytes(int64_t B, int64_t T) {
    if (T <= kMinTileRows) return 0;
    return (size_t)B * (size_t)((T + kMinTileRows - 1) / kMinTileRows) * 2 * sizeof(unsigned long long);
}

constexpr size_t kWorkspaceFixedBytes = (size_t)kMaxGridBlocks * 8 * sizeof(float) + kCounterBytes +
                                        (size_t)kMaxTaggedRows * 8 * sizeof(unsigned long long);

// Tiles of `nt` rows with whole trajectories packed into them, a trajectory longer than a tile counting as one: what the
// documented limit of the static scratch is counted in (the kernels lay rows out otherwise, see impact_flat.cuh).
long long packed_tiles(int64_t B, int64_t T, int nt) {
    if (T > nt) return B;
    const long long per_tile = nt / T;
    return (B + per_tile - 1) / per_tile;
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

}  // namespace

// Tiles the producer keeps in flight and stages of the ring, for tiles of `tile_in_bytes` bytes of logits.
// Bytes in flight per SM (IMPACT_OPT_WINDOW_BYTES; 0 = chosen here): 72 KB where a block streams many tiles (over
// 148 SMs that covers HBM's latency at full bandwidth; measured: 64 KB and more reach the copy rate, 48 KB stop at
// 0.9 of it), 48 KB where a block has only a few (a bigger first burst makes every tile of it land later, and the
// first tile's landing is what such a launch waits for).  Beyond the window there is room for the tiles being
// worked on and being stored.  The barrier protocol needs stages >= in_flight + groups, or exactly one stage per
// group (then the stage's previous tile is the one the same group worked on last); 0 stages = no valid shape.
// `cold`: 72 KB whatever the tiles -- no kernel has asked L2 for the inputs of a launch that finds them by a record, and a
// drawn batch comes from a ring larger than L2 (a step and a loss on 131 072 steps of 18 actions 11.0 us with 48 KB, 10.6 with
// 72, 11.1 with 96, 11.6 with 32).
void ws_ring_shape(size_t stage_bytes, size_t tile_in_bytes, int groups, int max_smem, long long tiles_per_block,
                   int* stages, int* in_flight, bool cold) {
    size_t window = (size_t)option(IMPACT_OPT_WINDOW_BYTES);
    if (window == 0) window = tiles_per_block <= 8 && !cold ? 48 * 1024 : 72 * 1024;
    int w = (int)((window + tile_in_bytes - 1) / tile_in_bytes);
    if (w < 2) w = 2;
    if (w > 8) w = 8;
    int s = w + groups + 3;
    if (s > kWsMaxStages) s = kWsMaxStages;
    const int fit = stages_that_fit(stage_bytes, max_smem);
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
    // companion; with 3-9 KB tiles it costs 5-15 %).  The companion pays where a
    // launch is short: a block has a handful of tiles, all within the budget.  A long launch is bound by HBM either
    // way, and asking for many tiles far ahead of their use only competes with the tiles that are needed now.
    // Without a companion the loss kernel's first warp asks for the tiles it is about to request anyway (more than
    // that sits in the copy engine's queue ahead of the requests themselves).
    const bool large_tiles = tile_bytes >= 10 * 1024;
    // (measured on 18 actions: a gain from five tiles per block on -- 8.3 -> 7.6 us at seven --, nothing at three
    // to four, a loss of a quarter of a microsecond at two; on small tiles up to as many as companion_pays' bytes hold: 2500 x
    // 100 steps of 9 actions with every switch 11.0 -> 10.1 us, of 10 9.7 -> 8.8)
    pl.companion = allow_companion && large_tiles && option(IMPACT_OPT_EARLY_PREFETCH) != 0 && pf >= per_block &&
                   per_block >= 4 && per_block <= 16;
    if (!large_tiles) pf = 0;
    if (!pl.companion && pf > in_flight) pf = in_flight;
    if (pf > per_block) pf = per_block;
    pl.prefetch_tiles = (int)pf;
    return pl;
}

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

template <typename LT, typename GT>
static int32_t run_categorical(const CatParams& p, const DeviceInfo* di, cudaStream_t s) {
    if (is_compiled_count(p.A)) return run_compiled_count<LT, GT>(p, di, s);
    if (is_larger_count(p.A)) return run_larger_count<LT, GT>(p, di, s);
    if (p.A % 4 == 0) return run_runtime_width<LT, GT, 4>(p, di, s);
    return p.A % 2 == 0 ? run_runtime_width<LT, GT, 2>(p, di, s) : run_runtime_width<LT, GT, 1>(p, di, s);
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
    p.spare_slots = static_cast<unsigned long long*>(workspace);
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

    GaussParams p = {};
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
    p.counter = reinterpret_cast<unsigned int*>(static_cast<char*>(workspace) +
                                                (size_t)kMaxGridBlocks * 8 * sizeof(float));
    p.tagged_rows = reinterpret_cast<unsigned long long*>(static_cast<char*>(workspace) +
                                                          (size_t)kMaxGridBlocks * 8 * sizeof(float) + kCounterBytes);
    p.tile_aggregates = (T > kMinTileRows && workspace_bytes >= impact_loss_workspace_bytes(B, T))
                            ? reinterpret_cast<unsigned long long*>(static_cast<char*>(workspace) + kWorkspaceFixedBytes)
                            : nullptr;
    p.spare_slots = static_cast<unsigned long long*>(workspace);
    p.D = D;
    p.geo.B = B;
    p.geo.T = T;
    return run_gaussian(p, di, static_cast<cudaStream_t>(stream));
}

// ------------------------------------------------------------------------------------------
// Variant for callers that must not allocate
// ------------------------------------------------------------------------------------------
namespace impact {
namespace {

constexpr int kStaticMaxBlocks = 1024;  // tiles that a call may have (packed_tiles)
constexpr size_t kStaticScratchBytes = (size_t)kStaticMaxBlocks * 8 * sizeof(float) + kCounterBytes +
                                       (size_t)kMaxTaggedRows * 8 * sizeof(unsigned long long);

// Scratch that lives in the library image, laid out like a workspace: an unused part, 256 bytes
// of counter words, the tagged rows.  Every device that loads the library
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
    if (packed_tiles(B, T, static_scratch_tile_rows(A, T, logits_bf16, grads_bf16)) > kStaticMaxBlocks)
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
