// Block-wide helpers shared by the binning, ranking and compositing kernels.
#pragma once

#include <algorithm>

#include "gs_internal.cuh"

namespace gsb {

// Resident CTAs of a kernel on the current device, looked up once per device.
struct PerDevice {
    int n[64] = {0};
    cudaError_t ctas(const void* fn, int threads, int* out) {
        int dev = 0, per_sm = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        if (n[dev] == 0) {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, 0);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            n[dev] = (per_sm < 1 ? 1 : per_sm) * sms;
        }
        *out = n[dev];
        return cudaSuccess;
    }
};

// Exclusive scan of one value per thread and its total; red holds NT/32 words.
template <int NT>
__device__ __forceinline__ uint32_t block_excl_scan_total(uint32_t v, uint32_t* red, uint32_t& total) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) red[warp] = x;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        const uint32_t r = red[w];
        if (w < warp) before += r;
        total += r;
    }
    __syncthreads();
    return before + x - v;
}

template <int NT>
__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t v, uint32_t* red) {
    uint32_t total;
    return block_excl_scan_total<NT>(v, red, total);
}

// Block-wide min and max of one u32 per thread; red holds 2 NT/32 words.
template <int NT>
__device__ __forceinline__ void block_minmax_u32(uint32_t& mn, uint32_t& mx, uint32_t* red) {
    constexpr int NW = NT / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) {
        red[warp] = mn;
        red[NW + warp] = mx;
    }
    __syncthreads();
    mn = red[0];
    mx = red[NW];
    for (int w = 1; w < NW; ++w) {
        mn = min(mn, red[w]);
        mx = max(mx, red[NW + w]);
    }
    __syncthreads();
}

// The visible record slots of mask words [w0, w1) of one env, one word per
// thread (w1 - w0 <= blockDim.x), listed block-wide in slot order in lst (at
// most 32 (w1 - w0) entries, slots relative to 32 w0); returns their number.
// One list per block spreads the visible records evenly over its warps,
// however unevenly visibility clusters in the storage order, and a two-pass
// kernel walks the same list in both passes.  wtot: one u32 per warp.
__device__ __forceinline__ int block_visible(const uint32_t* mask, int64_t w0, int64_t w1, uint16_t* lst,
                                             uint32_t* wtot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t w = w0 + threadIdx.x;
    uint32_t m = w < w1 ? __ldg(mask + w) : 0u;
    const uint32_t c = __popc(m);
    uint32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    uint32_t before = 0, total = 0;
    for (int i = 0; i < nw; ++i) {
        const uint32_t t = wtot[i];
        if (i < warp) before += t;
        total += t;
    }
    uint32_t pos = before + incl - c;
    while (m) {
        const int bit = __ffs(m) - 1;
        m &= m - 1u;
        lst[pos++] = (uint16_t)(threadIdx.x * 32 + bit);
    }
    __syncthreads();
    return (int)total;
}

// Sort key of the record in slot j: depth bits, then the caller's local index.
__device__ __forceinline__ unsigned long long rank_key(const RankParams& R, const uint4& q, uint32_t j) {
    const uint32_t i = R.index_in_r3 ? q.w : ((R.bg_index && j < R.n_bg) ? (uint32_t)__ldg(R.bg_index + j) : j);
    return ((unsigned long long)q.z << 32) | i;
}

// Depth range of a key: the number of splitters (split[0, bins - 1),
// ascending) that are <= key.  The key's depth cell bounds it to a few
// candidates (cell[c]: splitters before the cell); z0, shift: the cells.
__device__ __forceinline__ int rank_bin(const unsigned long long* split, const uint16_t* cell, int cells, int bins, uint32_t z0,
                                        int shift, unsigned long long key) {
    const uint32_t z = (uint32_t)(key >> 32);
    const uint32_t c = z <= z0 ? 0u : min((z - z0) >> shift, (uint32_t)(cells - 1));
    int lo = cell[c], hi = c + 1 < (uint32_t)cells ? (int)cell[c + 1] : bins - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (split[mid] <= key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

}  // namespace gsb
