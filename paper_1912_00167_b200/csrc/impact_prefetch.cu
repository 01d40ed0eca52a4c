// The companion kernel that asks L2 for a categorical loss launch's first tiles while the kernel before it on the
// stream is still running.
#include "impact_flat.cuh"

namespace impact {
namespace {

// What a block of the loss kernel will read, as a list of row-major arrays: the first tiles of every block are asked
// for in L2 before the launch's stream dependency has resolved.  A prefetch changes nothing that a program can observe
// (L2 is where the device's writes meet, so a later write to these addresses is not lost); it only moves the wait for
// HBM from the start of this launch into the end of the one before it.
constexpr int kArrays = 7;
struct PrefetchList {
    const void* base[kArrays];
    int row_bytes[kArrays];
    int n_tiles_max;  // tiles of a block that are asked for (from its first)
    int is_long;
    BatchGeometry geo;
};

// Enqueued right before the loss launch and of as many blocks, it becomes resident next to the blocks of whatever
// kernel is still running on the stream (it needs one warp and no shared memory per block), asks L2 for the loss
// launch's first tiles -- tile after tile in the order the block will want them, lane a asking for array a's rows of
// the tile, so that the memory system sees the requests in that order too -- and only then waits for the stream's
// previous kernel, which keeps stream order exact for the loss kernel behind it, whose own dependency is this kernel.
__global__ void __launch_bounds__(32) impact_prefetch_kernel(const __grid_constant__ PrefetchList pf) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x;
    const BlockRange br = block_range(pf.geo);
    int n_tiles = tiles_of_block(pf.geo, br, pf.is_long != 0);
    if (n_tiles > pf.n_tiles_max) n_tiles = pf.n_tiles_max;
    const long long total_rows = pf.geo.B * pf.geo.T;
    const void* base = nullptr;
    long long pitch = 0;
#pragma unroll
    for (int a = 0; a < kArrays; ++a)
        if (lane == a) { base = pf.base[a]; pitch = pf.row_bytes[a]; }
    if (pf.is_long) ask_for_tiles<true, 2>(pf.geo, br, base, pitch, n_tiles, pf.geo.nt, total_rows);
    else ask_for_tiles<false, 2>(pf.geo, br, base, pitch, n_tiles, pf.geo.nt, total_rows);
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace

int32_t launch_companion(const CatParams& p, int elem_bytes, bool is_long, int n_tiles, int grid, cudaStream_t stream) {
    PrefetchList pf = {};
    const void* const bases[kArrays] = {p.learner_logits, p.target_logits, p.actions, p.worker_logp, p.rewards, p.discounts, p.values};
    for (int i = 0; i < kArrays; ++i) {
        pf.base[i] = bases[i];
        pf.row_bytes[i] = i < 2 ? p.A * elem_bytes : 4;
    }
    pf.n_tiles_max = n_tiles;
    pf.is_long = is_long ? 1 : 0;
    pf.geo = p.geo;
    IMPACT_CUDA_TRY(launch_serialized(impact_prefetch_kernel, dim3((unsigned)grid), dim3(32), 0, stream, pf));
    return IMPACT_OK;
}

}  // namespace impact
