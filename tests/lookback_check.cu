// What a tile of a split trajectory finds behind the tiles that come after it has the same bits whichever blocks of 32 tiles have
// published the value that leaves them by then, and the bits of the maps composed from the trajectory's end.  One warp per case,
// everything that it waits for in memory beforehand; what a case publishes has to be right too.  Returns the number of cases
// that differ (255 at most).
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "impact_device.cuh"

using namespace impact;

constexpr unsigned int kTag = 7;
constexpr int kTiles = 1313, kBlocks = kTiles / 32;

struct Case {
    int r;
    unsigned long long valued;  // the blocks whose values are there
};

__global__ void compose_all(const unsigned long long* maps, float* found, unsigned int* words) {
    __shared__ int abort_s;
    if (threadIdx.x == 0) abort_s = 0;
    __syncwarp();
    const int r = blockIdx.x;
    const float x = dev::compose_later_aggregates(maps + 2 * r, 2, r, kTag, &abort_s, words, false, 0ull, 0ull);
    if (threadIdx.x == 0) found[r] = x;
}

__global__ void look_back(const Case* cases, const unsigned long long* maps, unsigned long long* blocks, float* found, unsigned int* words) {
    __shared__ int abort_s;
    if (threadIdx.x == 0) abort_s = 0;
    __syncwarp();
    const int r = cases[blockIdx.x].r;
    const float a = __uint_as_float((unsigned int)maps[2 * r]), b = __uint_as_float((unsigned int)maps[2 * r + 1]);
    const float x = dev::value_from_later_tiles(maps + 2 * r, blocks + (size_t)blockIdx.x * 4 * kBlocks, r, a, b, kTag, &abort_s, words);
    if (threadIdx.x == 0) found[blockIdx.x] = x;
}

int main() {
    uint32_t state = 12345;
    auto next = [&]() { return (state = state * 1664525u + 1013904223u) >> 8; };
    auto uniform = [&]() { return (float)next() / 16777216.0f; };
    auto tagged = [](float x) {
        uint32_t u;
        memcpy(&u, &x, 4);
        return ((unsigned long long)kTag << 32) | u;
    };
    std::vector<unsigned long long> maps(2 * kTiles);
    for (int t = 0; t < kTiles; ++t) {
        maps[2 * t] = tagged(t == 0 ? 0.0f : 0.9f + 0.2f * uniform());
        maps[2 * t + 1] = tagged(uniform() - 0.5f);
    }
    // the blocks' leaders one after another first: what they publish is what the cases below find
    std::vector<Case> leaders, cases;
    for (int b = 0; b < kBlocks; ++b) leaders.push_back({32 * b + 31, 0});
    for (int r = 1; r < kTiles; ++r) {
        const int block = r / 32;
        const unsigned long long nearest = block ? 1ull << (block - 1) : 0ull;
        if (r % 32 != 31) {
            cases.push_back({r, nearest});
            continue;
        }
        // (a leader looks at 32 blocks: one of those is known, or the trajectory ends among them)
        const unsigned long long within = block > 31 ? 1ull << (block - 32 + next() % 32) : 0ull;
        for (unsigned long long valued : {0ull, ~0ull, 1ull, nearest, nearest >> 1, 0x30004ull, (unsigned long long)next(), (unsigned long long)next() << 20})
            cases.push_back({r, valued | within});
    }
    const int n = (int)cases.size();
    std::vector<unsigned long long> full(4 * kBlocks), blocks((size_t)n * 4 * kBlocks, 0);
    std::vector<float> all(kTiles), got(n);
    unsigned long long *d_maps, *d_blocks;
    Case* d_cases;
    float *d_all, *d_found;
    unsigned int *d_words, words[2] = {9, 9};
    if (cudaMalloc(&d_maps, maps.size() * 8) || cudaMalloc(&d_blocks, blocks.size() * 8) || cudaMalloc(&d_cases, n * sizeof(Case)) ||
        cudaMalloc(&d_all, kTiles * 4) || cudaMalloc(&d_found, n * 4) || cudaMalloc(&d_words, sizeof(words)) ||
        cudaMemset(d_words, 0, sizeof(words)) || cudaMemset(d_blocks, 0, full.size() * 8) ||
        cudaMemcpy(d_maps, maps.data(), maps.size() * 8, cudaMemcpyHostToDevice) ||
        cudaMemcpy(d_cases, leaders.data(), kBlocks * sizeof(Case), cudaMemcpyHostToDevice))
        return 255;
    compose_all<<<kTiles, 32>>>(d_maps, d_all, d_words);
    for (int b = 0; b < kBlocks; ++b) look_back<<<1, 32>>>(d_cases + b, d_maps, d_blocks, d_found, d_words);
    if (cudaDeviceSynchronize() || cudaMemcpy(all.data(), d_all, kTiles * 4, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(full.data(), d_blocks, full.size() * 8, cudaMemcpyDeviceToHost))
        return 255;
    for (int i = 0; i < n; ++i)
        for (int b = 0; 32 * b + 31 < cases[i].r; ++b) {
            unsigned long long* const at = &blocks[((size_t)i * kBlocks + b) * 4];
            at[0] = full[4 * b];
            at[1] = full[4 * b + 1];
            if ((cases[i].valued >> b) & 1u) at[2] = full[4 * b + 2];
        }
    if (cudaMemcpy(d_blocks, blocks.data(), blocks.size() * 8, cudaMemcpyHostToDevice) ||
        cudaMemcpy(d_cases, cases.data(), n * sizeof(Case), cudaMemcpyHostToDevice))
        return 255;
    look_back<<<n, 32>>>(d_cases, d_maps, d_blocks, d_found, d_words);
    std::vector<unsigned long long> after(blocks.size());
    if (cudaDeviceSynchronize() || cudaMemcpy(got.data(), d_found, n * 4, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(after.data(), d_blocks, after.size() * 8, cudaMemcpyDeviceToHost) ||
        cudaMemcpy(words, d_words, sizeof(words), cudaMemcpyDeviceToHost))
        return 255;
    int bad = words[0] ? 1 : 0;
    for (int b = 0; b < kBlocks; ++b)
        if (full[4 * b + 2] != tagged(all[32 * b + 32])) ++bad;  // (what leaves a block enters the tile behind it)
    for (int i = 0; i < n; ++i) {
        const int r = cases[i].r;
        if (r % 32 == 31)
            for (int k = 0; k < 3; ++k) blocks[((size_t)i * kBlocks + r / 32) * 4 + k] = full[4 * (r / 32) + k];
        const bool ok = memcmp(&got[i], &all[r], 4) == 0 &&
                        memcmp(&blocks[(size_t)i * 4 * kBlocks], &after[(size_t)i * 4 * kBlocks], 32 * kBlocks) == 0;
        if (!ok && bad++ < 8) printf("r=%d valued=%llx: %.9g, %.9g\n", r, cases[i].valued, got[i], all[r]);
    }
    printf("%d of %d differ, error word %u\n", bad, n, words[0]);
    return bad > 255 ? 255 : bad;
}
