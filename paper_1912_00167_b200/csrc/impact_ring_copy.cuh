// The copy of a pushed batch by blocks of one warp (see ring_step_kernel).
#pragma once

#include "impact_device.cuh"

namespace impact {

constexpr int kStepUnits = 1024;             // 16-byte units of a block's buffer
constexpr unsigned int kCopyTries = 1u << 22;  // looks at a barrier before its wait gives up, some seconds

// A segment's part of the units [u0, u1) of all segments, a segment to every lane, by bulk copies through `buffer` (kStepUnits
// units).  Where a round's bytes have not come after `limit` looks, ordinary loads bring them and all that is left: the step has
// counted on this copy by then, and so may the loss call behind it.  The copies asked for are waited for once more, because
// they write to the block's shared memory; returns false if they may be under way still.
__device__ __forceinline__ bool copy_by_warp(const char* src, char* dst, unsigned long long bytes, unsigned long long first,
                                             unsigned long long u0, unsigned long long u1, uint4* buffer, uint64_t* bar,
                                             unsigned int limit) {
    const int lane = threadIdx.x & 31;
    const unsigned long long whole_end = first + bytes / 16ull;  // (the last unit may be a part of one)
    uint32_t parity = 0;
    auto landed = [&](unsigned int looks) {
        bool there = false;
        for (unsigned int tries = 0; tries < looks && !there; ++tries) there = dev::mbarrier_test(bar, parity);
        return __all_sync(0xFFFFFFFFu, there) != 0;
    };
    bool none_left = true;
    for (unsigned long long base = u0; base < u1; base += kStepUnits, parity ^= 1u) {
        const unsigned long long end = base + kStepUnits < u1 ? base + kStepUnits : u1;
        const unsigned long long lo = base > first ? base : first, hi = end < whole_end ? end : whole_end;
        const uint32_t n = lo < hi ? (uint32_t)(hi - lo) * 16u : 0u;
        uint4* const at = buffer + (lo - base);
        if (n) dev::bulk_load(at, src + (lo - first) * 16ull, n, bar);
        const uint32_t all = __reduce_add_sync(0xFFFFFFFFu, n);
        if (lane == 0) dev::mbarrier_expect_tx(bar, all);
        if (!landed(limit)) {
            for (unsigned long long u = lo; u < u1 && u < whole_end; ++u)
                reinterpret_cast<uint4*>(dst)[u - first] = reinterpret_cast<const uint4*>(src)[u - first];
            none_left = landed(kCopyTries);
            break;
        }
        if (n) dev::bulk_store(dst + (lo - first) * 16ull, at, n);
        dev::bulk_store_wait_read();
        __syncwarp();
    }
    if (whole_end >= u0 && whole_end < u1)
        for (unsigned long long i = bytes & ~15ull; i < bytes; ++i) dst[i] = src[i];
    return none_left;
}

}  // namespace impact
