// The depth ranges that the ranking's sample gives an env of n slots whose depths
// ascend with the slot (as they do along a Morton order that runs away from the
// camera), visible where bit j % 32 of mask[j / 32] is set: writes the number of
// visible records per range (at most `room` ranges) and returns the ranges.
#include <algorithm>
#include <vector>

#include "gs_internal.cuh"

extern "C" int rank_ranges(int n, const uint32_t* mask, uint32_t* per_range, int room) {
    using namespace gsb;
    std::vector<EnvInfo> envs(2);
    envs[0].n_local = (unsigned)n;
    const int words = (n + 31) / 32;
    std::vector<uint4> r3((size_t)n);
    for (int j = 0; j < n; ++j) r3[(size_t)j] = make_uint4(0u, 0u, 0x3f800000u + 7u * (uint32_t)j, (uint32_t)j);
    RankParams R = rank_sizes(words, 1, false);
    if (R.bins < 1 || R.bins > room) return -1;
    void *d_envs = nullptr, *d_mask = nullptr, *d_r3 = nullptr, *d_tab = nullptr;
    bool ok = cudaMalloc(&d_envs, sizeof(EnvInfo) * 2) == cudaSuccess && cudaMalloc(&d_mask, 4 * words) == cudaSuccess &&
              cudaMalloc(&d_r3, 16 * (size_t)n) == cudaSuccess &&
              cudaMalloc(&d_tab, rank_tables(R, 1, nullptr)) == cudaSuccess;
    if (ok) {
        ok = cudaMemcpy(d_envs, envs.data(), sizeof(EnvInfo) * 2, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(d_mask, mask, 4 * words, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(d_r3, r3.data(), 16 * (size_t)n, cudaMemcpyHostToDevice) == cudaSuccess;
        rank_tables(R, 1, static_cast<unsigned char*>(d_tab));
        R.envs = static_cast<EnvInfo*>(d_envs);
        R.mask = static_cast<uint32_t*>(d_mask);
        R.r3 = static_cast<uint4*>(d_r3);
        R.index_in_r3 = 1;
        std::vector<unsigned long long> split((size_t)R.bins);
        ok = ok && launch_rank_sample(R, 1, 0) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess &&
             cudaMemcpy(split.data(), R.split, 8 * (size_t)R.bins, cudaMemcpyDeviceToHost) == cudaSuccess;
        std::fill(per_range, per_range + R.bins, 0u);
        for (int j = 0; j < n && ok; ++j) {
            if (!((mask[j >> 5] >> (j & 31)) & 1u)) continue;
            const unsigned long long key = (unsigned long long)r3[(size_t)j].z << 32 | r3[(size_t)j].w;
            ++per_range[std::upper_bound(split.begin(), split.end() - 1, key) - split.begin()];
        }
    }
    for (void* p : {d_envs, d_mask, d_r3, d_tab}) cudaFree(p);
    return ok ? R.bins : -2;
}
