// What the host takes for the bookkeeping's present state at every moment of a step (no GPU).
// With an argument, the ring's step where its waits run out.  The copy of a batch whose wait is given no look at all: every byte of it is there and
// none beside it.  A handle whose step has said that copies may have come late: it is told, gets its bookkeeping back and
// goes on outside device mode.  Returns the number of checks that fail (255 at most).
#include "impact_ring.cu"

#include <stdio.h>

static int bad = 0;
static void check(bool ok, const char* what, long long x) {
    if (!ok && bad++ < 8) printf("%s %lld\n", what, x);
}

struct Segments {
    int n;
    const char* src[4];
    char* dst[4];
    unsigned long long bytes[4];
};

__global__ void __launch_bounds__(32) copy_batch(const Segments s, unsigned int limit, int* late) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ __align__(16) uint4 buffer[kStepUnits];
    if (threadIdx.x == 0) {
        dev::mbarrier_init_nofence(&bar, 1);
        dev::fence_mbarrier_init();
    }
    __syncwarp();
    const int lane = threadIdx.x;
    unsigned long long first = 0, units = 0;
    for (int f = 0; f < s.n; ++f) {
        if (f < lane) first += (s.bytes[f] + 15) / 16;
        units += (s.bytes[f] + 15) / 16;
    }
    const bool mine = lane < s.n;
    if (!copy_by_warp(mine ? s.src[lane] : nullptr, mine ? s.dst[lane] : nullptr, mine ? s.bytes[lane] : 0ull, first,
                      units * blockIdx.x / gridDim.x, units * (blockIdx.x + 1ull) / gridDim.x, buffer, &bar, limit) && lane == 0)
        atomicAdd(late, 1);
}

static void copies() {
    const size_t sizes[3][4] = {{7, 16, 4000, 33}, {100003, 64, 15, 20000}, {600001, 31, 300000, 16}};
    int* late;
    if (cudaMalloc(&late, 4) || cudaMemset(late, 0, 4)) { check(false, "late", 0); return; }
    for (auto& size : sizes)
        for (unsigned int limit : {0u, kCopyTries}) {
            Segments s = {};
            s.n = 4;
            std::vector<unsigned char> want[4], got;
            char* dst[4];
            for (int f = 0; f < 4; ++f) {
                want[f].resize(size[f] + 64, 0xA5);
                char* src;
                if (cudaMalloc(&src, size[f] + 64) || cudaMalloc(&dst[f], size[f] + 64) || cudaMemset(dst[f], 0xA5, size[f] + 64)) { check(false, "memory", f); return; }
                for (size_t i = 0; i < size[f]; ++i) want[f][i] = (unsigned char)(i * 7 + i / 251 + f);
                if (cudaMemcpy(src, want[f].data(), size[f], cudaMemcpyHostToDevice)) { check(false, "source", f); return; }
                s.src[f] = src;
                s.dst[f] = dst[f];
                s.bytes[f] = size[f];
            }
            copy_batch<<<9, 32>>>(s, limit, late);
            check(cudaDeviceSynchronize() == cudaSuccess, "copy", limit);
            for (int f = 0; f < 4; ++f) {
                got.resize(want[f].size());
                check(cudaMemcpy(got.data(), dst[f], got.size(), cudaMemcpyDeviceToHost) == cudaSuccess && got == want[f], "bytes", size[f]);
                cudaFree(const_cast<char*>(s.src[f]));
                cudaFree(dst[f]);
            }
        }
    int n = 9;
    check(cudaMemcpy(&n, late, 4, cudaMemcpyDeviceToHost) == cudaSuccess && n == 0, "copies under way at the end", n);
}

static void handle_that_was_told() {
    const size_t bytes[2] = {400, 24};
    impact_buffer* h = nullptr;
    check(impact_buffer_create(2, 9, 2, bytes, 1, IMPACT_SAMPLE_UNIFORM, nullptr, &h) == IMPACT_OK, "create", 0);
    char *src, *table, *record;
    if (cudaMalloc(&src, 512) || cudaMalloc(&table, 24) || cudaMalloc(&record, sizeof(impact_loss_inputs))) { check(false, "memory", 0); return; }
    const void* pointers[3] = {src, src, nullptr};
    check(cudaMemcpy(table, pointers, 24, cudaMemcpyHostToDevice) == cudaSuccess, "table", 0);
    for (int round = 0; round < 2; ++round) {  // (once told, once not)
        check(impact_buffer_device_begin(h, nullptr) == IMPACT_OK, "begin", round);
        const impact_ring_field_map map = {0, -1, -1, -1, -1};
        check(impact_buffer_device_step(h, &map, src, nullptr, nullptr, reinterpret_cast<const void* const*>(table), 1,
                                        reinterpret_cast<impact_loss_inputs*>(record), nullptr) == IMPACT_OK, "step", round);
        const uint32_t failed = round == 0 ? 1 : 0;
        check(cudaDeviceSynchronize() == cudaSuccess &&
                  cudaMemcpy(&h->view().shared->failed, &failed, 4, cudaMemcpyHostToDevice) == cudaSuccess, "flag", round);
        const int32_t want = failed ? IMPACT_ERR_CUDA : IMPACT_OK;
        int32_t events[16], n = 0;
        char state[256];
        check(impact_buffer_device_events(h, events, 4, &n, nullptr) == want && n == 2 && events[4 * 1 + 0] == 2, "events", n);
        check(impact_buffer_live(h) == (failed ? want : 2), "live", round);
        check(impact_buffer_export_state(h, state, sizeof(state)) == want, "state", round);
        check(impact_buffer_device_end(h, nullptr) == want, "end", round);
        check(!failed || impact_last_cuda_error() == cudaErrorTimeout, "last error", impact_last_cuda_error());
        check(impact_buffer_live(h) == round + 1 && h->count[0] + h->count[1] == round + 1, "bookkeeping", impact_buffer_live(h));
    }
    const void* fields[2] = {src, src};
    int32_t slot = -1, k = -1;
    check(impact_buffer_sample(h, &slot, &k, nullptr, nullptr) == IMPACT_OK && impact_buffer_push(h, fields, IMPACT_SRC_DEVICE, &slot, nullptr) == IMPACT_ERR_FULL, "calls afterwards", k);
    check(impact_buffer_destroy(h) == IMPACT_OK, "destroy", 0);
}

// Block 0 draws the ticket that makes up for the others' at any place among them, and writes the other copy at its end.
static void states() {
    for (uint32_t blocks : {1u, 2u, 148u})
        for (uint32_t first : {0u, 65534u, 0xFFFFFFFEu}) {
            RingDeviceShared s = {};
            s.tickets = first << kTicketBits;
            s.state[first & 1].hd.steps = first;
            s.state[~first & 1].hd.steps = first - 1;  // (a buffer of no steps has 0 in both)
            if (first == 0) s.state[1].hd.steps = 0;
            for (uint32_t n = first; n != first + 5; ++n) {
                const uint32_t odd = (s.tickets >> kTicketBits) & 1u;
                for (uint32_t place : {0u, blocks / 2, blocks - 1}) {  // block 0's among the tickets
                    RingDeviceShared at = s;
                    for (uint32_t i = 0; i < blocks; ++i) {
                        check(((at.tickets >> kTicketBits) & 1u) == odd, "copy that a block reads", n);
                        at.tickets += i == place ? (1u << kTicketBits) - (blocks - 1) : 1u;
                        check(at.current().hd.steps == n, "state in a step", n);
                    }
                }
                s.tickets += 1u << kTicketBits;
                s.state[odd ^ 1u].hd = s.state[odd].hd;
                s.state[odd ^ 1u].hd.steps += 1;
                check(s.current().hd.steps == n + 1, "state behind a step", n);
            }
        }
}

int main(int argc, char**) {
    states();
    if (argc > 1) {
        copies();
        handle_that_was_told();
    }
    printf("%d wrong\n", bad);
    return bad > 255 ? 255 : bad;
}
