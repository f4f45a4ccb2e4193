// (env, tile) intersection counting, prefix scan and bucketed scatter of
// depth ranks (steps A3 and A4).  The renderer of the paper (Sec. III-C
// "Throughput Scaling", built on gsplat) bins projected splats into screen
// tiles before compositing; this file is that binning, designed for many envs.
//
// Each splat's support box [i0,i1]x[j0,j1] (pixels) touches the tiles
// [i0/tw, i1/tw] x [j0/th, j1/th].  Counting and scattering first aggregate in
// a shared-memory histogram per (env, block of Gaussians), so global atomics
// are one per touched tile per block rather than one per intersection.  The
// order inside a bucket is arbitrary; the compositor orders each bucket by the
// records' unique depth ranks (gs_rank.cu).
#include "gs_internal.cuh"
#include "gs_block.cuh"

namespace gsb {

// Tile widths and heights are powers of two (8, 16 or 32; the API rejects
// other shapes), and box coordinates are non-negative, so the tile of a pixel
// coordinate is a shift of it: sx = log2(tile width), sy = log2(tile height).
__device__ __forceinline__ void tile_span(uint32_t rx, uint32_t ry, int sx, int sy, int& tx0, int& tx1, int& ty0,
                                          int& ty1) {
    tx0 = (int)((rx & 0xffffu) >> sx);
    tx1 = (int)((rx >> 16) >> sx);
    ty0 = (int)((ry & 0xffffu) >> sy);
    ty1 = (int)((ry >> 16) >> sy);
}

// f(t, tx, ty) for every tile t = ty ntx + tx of a record's span: rows
// ty0..ty1 of the columns tx0..tx1 in one flat loop (lanes with spans of
// different shapes then diverge only by their tile counts).  WRAP (LiDAR
// waves): a box with x0 > x1 covers the columns [x0, cols) and [0, x1] (a cone
// across azimuth 0), so its tile columns run tx0..ntx-1 and then 0..tx1.
template <bool WRAP, typename F>
__device__ __forceinline__ void for_span(uint32_t rx, uint32_t ry, int sx, int sy, int ntx, F&& f) {
    int tx0, tx1, ty0, ty1;
    tile_span(rx, ry, sx, sy, tx0, tx1, ty0, ty1);
    if (WRAP && (rx & 0xffffu) > (rx >> 16)) {
        const int nx = min(ntx, ntx - tx0 + tx1 + 1);
        const int n = nx * (ty1 - ty0 + 1);
        int tx = tx0, ty = ty0, row = ty0 * ntx, c = 0;
        for (int k = 0; k < n; ++k) {
            f(row + tx, tx, ty);
            if (++c == nx) {
                c = 0;
                tx = tx0;
                row += ntx;
                ++ty;
            } else if (++tx == ntx) {
                tx = 0;
            }
        }
        return;
    }
    const int n = (tx1 - tx0 + 1) * (ty1 - ty0 + 1);
    int tx = tx0, ty = ty0, t = ty0 * ntx + tx0;
    for (int k = 0; k < n; ++k) {
        f(t, tx, ty);
        if (tx == tx1) {
            tx = tx0;
            ++ty;
            t += ntx - (tx1 - tx0);
        } else {
            ++tx;
            ++t;
        }
    }
}

// A block's tile histogram of the boxes on a grid of ntx x nty tiles, in hist
// with a row pitch of ntx + 1.  DIFF: each box adds to the corners of a 2D
// difference array (ntx + 1) x (nty + 1), which block_sum2d then sums, so a box
// costs four atomics whatever its span: at 640x480 spans average 11 tiles and
// reach all 1200, and one lane walking a long span held its whole block up.
// On small grids (spans of one or two tiles) the walk is cheaper.
template <bool WRAP, bool DIFF>
__device__ __forceinline__ void add_box(uint32_t rx, uint32_t ry, int sx, int sy, int ntx, uint32_t* hist) {
    if constexpr (!DIFF) {
        for_span<WRAP>(rx, ry, sx, sy, ntx, [&](int, int tx, int ty) { atomicAdd(&hist[ty * (ntx + 1) + tx], 1u); });
    } else {
        static_assert(!WRAP, "wrapped boxes walk their spans");
        int tx0, tx1, ty0, ty1;
        tile_span(rx, ry, sx, sy, tx0, tx1, ty0, ty1);
        uint32_t* top = hist + ty0 * (ntx + 1);
        uint32_t* end = hist + (ty1 + 1) * (ntx + 1);
        atomicAdd(top + tx0, 1u);
        atomicAdd(top + tx1 + 1, ~0u);
        atomicAdd(end + tx0, ~0u);
        atomicAdd(end + tx1 + 1, 1u);
    }
}

// Sums a difference array along rows, then columns (block-wide).
__device__ __forceinline__ void block_sum2d(uint32_t* hist, int ntx, int nty) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    for (int y = warp; y < nty; y += nw) {  // a warp per row
        uint32_t* row = hist + y * (ntx + 1);
        uint32_t carry = 0;
        for (int x0 = 0; x0 < ntx; x0 += 32) {
            uint32_t v = x0 + lane < ntx ? row[x0 + lane] : 0u;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += o;
            }
            v += carry;
            if (x0 + lane < ntx) row[x0 + lane] = v;
            carry = __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < ntx; x += blockDim.x) {
        uint32_t run = 0;
        for (int y = 0; y < nty; ++y) hist[y * (ntx + 1) + x] = run += hist[y * (ntx + 1) + x];
    }
    __syncthreads();
}

// Words of a block's tile histogram.
__host__ __device__ __forceinline__ int hist_words(int ntx, int nty) { return (ntx + 1) * (nty + 1); }

// grid: (blocks over the largest env's visibility words, envs); block 256;
// dynamic smem: the env's splitters, depth cells and range counters, then the
// largest tile histogram.  Blocks past their env's words exit at once.  Counts
// the visible records of a block (block_visible's list; neighbouring threads
// take neighbouring records) per tile and per depth range of the env, and notes
// each record's range and place among the block's records of that range, so
// that the placement (gs_rank.cu) neither searches nor counts again.
template <bool WRAP, bool DIFF>
__global__ void __launch_bounds__(256) k_count(BinParams P, RankParams R) {
    extern __shared__ __align__(16) unsigned char csm[];
    __shared__ uint16_t lst[32 * kWordsPerBlock];
    __shared__ uint32_t wtot[32];
    unsigned long long* split = reinterpret_cast<unsigned long long*>(csm);
    uint16_t* cell = reinterpret_cast<uint16_t*>(split + R.bins);
    uint32_t* zhist = reinterpret_cast<uint32_t*>(cell + R.cells);
    uint32_t* hist = zhist + R.bins;
    const int el = P.e_begin + blockIdx.y;
    const EnvInfo E = P.envs[el];
    const int64_t words = (E.n_local + 31) / 32;
    const int64_t w0 = (int64_t)blockIdx.x * R.words_per_block;
    if (w0 >= words) return;
    const int64_t w1 = min(w0 + (int64_t)R.words_per_block, words);
    const int ntx = E.ntx, nty = E.T / ntx;
    for (int t = threadIdx.x; t < hist_words(ntx, nty); t += blockDim.x) hist[t] = 0;
    for (int b = threadIdx.x; b < R.bins; b += blockDim.x) {
        zhist[b] = 0u;
        split[b] = R.split[(size_t)el * R.bins + b];
    }
    const uint4* gc = reinterpret_cast<const uint4*>(R.cell + (size_t)el * R.cells);
    for (int c = threadIdx.x; c < R.cells / 8; c += blockDim.x) reinterpret_cast<uint4*>(cell)[c] = gc[c];
    const int nvis = block_visible(P.mask + E.mask_base, w0, w1, lst, wtot);
    const uint32_t z0 = R.bins ? (uint32_t)split[R.bins - 1] : 0u;
    const int zshift = R.bins ? (int)(split[R.bins - 1] >> 32) : 0;
    const uint4* r3 = P.r3 + E.rec_base;
    const int sx = __ffs(P.tile_w) - 1, sy = __ffs(P.tile_h) - 1;
    for (int i = threadIdx.x; i < nvis; i += blockDim.x) {
        const uint32_t j = (uint32_t)(w0 * 32) + lst[i];
        const uint4 q = r3[j];
        if (R.bins) {
            const uint32_t b = (uint32_t)rank_bin(split, cell, R.cells, R.bins, z0, zshift, rank_key(R, q, j));
            R.rank[E.rec_base + j] = b << 13 | atomicAdd(&zhist[b], 1u);
        }
        add_box<WRAP, DIFF>(q.x, q.y, sx, sy, ntx, hist);
    }
    if constexpr (DIFF) block_sum2d(hist, ntx, nty);
    else __syncthreads();
    uint32_t* cnt = P.counts + E.tile_base;
    for (int t = threadIdx.x; t < E.T; t += blockDim.x) {
        const uint32_t h = hist[t + t / ntx];
        if (h) {
            const uint32_t before = atomicAdd(cnt + t, h);
            if (P.tile_off) P.tile_off[((size_t)el * R.blocks + blockIdx.x) * P.tile_pitch + t] = before;
        }
    }
    uint32_t* zc = R.bin_cnt + (size_t)el * R.bins;
    uint32_t* bo = R.block_off + ((size_t)el * R.blocks + blockIdx.x) * R.bins;
    for (int b = threadIdx.x; b < R.bins; b += blockDim.x) {
        const uint32_t h = zhist[b];
        if (h) bo[b] = atomicAdd(zc + b, h);
    }
}

// The kernels' largest dynamic shared memory: the ranges and depth cells of a
// LiDAR scan's ranking and the histogram of the largest grid that the entry
// points take (kMaxTiles tiles of at least 8 pixels in images of at most 16384:
// 2048 x 8).  The attribute belongs to the function, not to the launch, so every
// launch sets this one value: with its own size, a launch failed when another
// thread set a smaller one in between.
constexpr int kMaxTiles = 16384;
constexpr size_t kMaxBinSmem = kRankBins * 12 + 4096 * 2 + (size_t)(kMaxTiles + 2048 + 8 + 1) * 4;

static cudaError_t opt_in_smem(const void* fn, size_t smem) {
    if (smem <= 30 * 1024) return cudaSuccess;  // plus at most 17.2 KB of static shared memory
    if (smem > kMaxBinSmem) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxBinSmem);
}

static_assert(kWordsPerBlock <= 256, "binning blocks: one visibility word per thread of 256, places below 2^13");

cudaError_t launch_count(const BinParams& P, const RankParams& R, int n_envs, int max_T, int max_hist,
                         cudaStream_t st) {
    if (n_envs == 0 || R.blocks == 0) return cudaSuccess;
    const bool diff = !P.wrap && max_T >= kDiffTiles;
    const size_t smem = (size_t)R.bins * 12 + (size_t)R.cells * 2 + (size_t)max_hist * 4;
    auto launch = [&](auto fn) -> cudaError_t {
        const cudaError_t e = opt_in_smem((const void*)fn, smem);
        if (e != cudaSuccess) return e;
        fn<<<dim3((unsigned)R.blocks, (unsigned)n_envs), 256, smem, st>>>(P, R);
        return cudaGetLastError();
    };
    if (P.wrap) return launch(k_count<true, false>);
    return diff ? launch(k_count<false, true>) : launch(k_count<false, false>);
}

// ---------------------------------------------------------------- scan

template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T* warp_tot, T& block_total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? warp_tot[lane] : T(0);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const T y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        if (lane < nw) warp_tot[lane] = w;  // inclusive
    }
    __syncthreads();
    const T before = warp == 0 ? T(0) : warp_tot[warp - 1];
    block_total = warp_tot[nw - 1];
    __syncthreads();
    return before + x - v;
}

// Bases of the envs, by one CTA: env_base[e] = sum_{e' < e} env_total[e'],
// env_base[We] = total; host_base (pinned host memory, or null) gets the same,
// with the env's longest bucket where that is asked for.
struct EnvBases {
    unsigned long long *total, *base, *host;
    unsigned int* ticket;  // CTAs done; 0 before and after the launch
    bool longest;          // total and host carry the longest bucket above kTotalBits bits
};
__device__ __forceinline__ void scan_bases(const EnvBases& B, int We) {
    __shared__ unsigned long long wt[32];
    unsigned long long carry = 0;
    for (int first = 0; first < We; first += blockDim.x) {
        const int e = first + threadIdx.x;
        const unsigned long long t = e < We ? __ldcg(B.total + e) : 0ull, v = t & ((1ull << kTotalBits) - 1ull);
        unsigned long long tot;
        const unsigned long long ex = block_exclusive_scan<unsigned long long>(v, wt, tot);
        if (e < We) {
            B.base[e] = carry + ex;
            if (B.host) B.host[e] = (carry + ex) | (t - v);
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        B.base[We] = carry;
        if (B.host) B.host[We] = carry;
        *B.ticket = 0u;
    }
}

// per env: off_local[t] = sum_{t' < t} counts[t'], total = sum.  With R
// (bins > 0), also the offsets of the env's depth ranges, the number of ranked
// records, and the window table: win[v] is the first range start >= v
// kRankStride, so a window is at most kRankStride plus its last range.  The CTA
// that finishes last scans the envs' totals (a kernel of its own for that cost a
// launch: one 128x96 view 104 -> 102 us, 8 without allocation 162 -> 158).
__global__ void __launch_bounds__(1024) k_scan_env(const EnvInfo* envs, const uint32_t* counts, uint32_t* off_local,
                                                   EnvBases B, int per, RankParams R) {
    __shared__ uint32_t wt[32];
    __shared__ bool last;
    __shared__ uint32_t longest;
    const int el = blockIdx.x;
    if (threadIdx.x == 0) longest = 0u;  // the scan's barriers come before its use
    uint32_t most = 0;
    const int T = envs[el].T * per;
    const uint32_t* c = counts + (size_t)envs[el].tile_base * per;
    uint32_t* o = off_local + (size_t)envs[el].tile_base * per;
    uint32_t carry = 0;
    for (int base = 0; base < T; base += blockDim.x) {
        const int t = base + threadIdx.x;
        const uint32_t v = t < T ? c[t] : 0u;
        most = max(most, v);
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<uint32_t>(v, wt, tot);
        if (t < T) o[t] = carry + ex;
        carry += tot;
    }
    if (B.longest) {
        most = __reduce_max_sync(0xffffffffu, most);
        if (most && (threadIdx.x & 31) == 0) atomicMax(&longest, most);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        B.total[el] = carry | (unsigned long long)min(longest, kTotalMost) << kTotalBits;
        __threadfence();
        last = atomicAdd(B.ticket, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (last) scan_bases(B, (int)gridDim.x);
    if (R.bins == 0) return;
    // two neighbouring ranges per thread
    const int b = 2 * threadIdx.x;
    const size_t eb = (size_t)el * R.bins + b;
    const uint2 c2 = b < R.bins ? *reinterpret_cast<const uint2*>(R.bin_cnt + eb) : make_uint2(0u, 0u);
    uint32_t nv;
    const uint32_t start = block_exclusive_scan<uint32_t>(c2.x + c2.y, wt, nv), mid = start + c2.x, end = mid + c2.y;
    if (b < R.bins) *reinterpret_cast<uint2*>(R.bin_off + eb) = make_uint2(start, mid);
    uint32_t* win = R.win + (size_t)el * R.win_pitch;
    if (b == 0) {
        R.nvis[el] = nv;
        win[0] = 0u;
        if (nv % kRankStride) win[nv / kRankStride + 1] = nv;
    }
    // the first range boundary at or after every multiple of the stride in
    // (start, mid] is mid, and in (mid, end] it is end
    if (b < R.bins) {
        uint32_t v = start / kRankStride + 1;
        for (; v * kRankStride <= mid; ++v) win[v] = mid;
        for (; v * kRankStride <= end; ++v) win[v] = end;
    }
}

static_assert(kRankBins <= 2048, "two depth ranges per thread of the scan");

cudaError_t launch_scan_ranks(const EnvInfo* envs, const uint32_t* counts, uint32_t* off_local,
                              unsigned long long* env_total, unsigned long long* env_base,
                              unsigned long long* host_base, bool longest, unsigned int* ticket, int We,
                              const RankParams& R, cudaStream_t st) {
    if (We == 0) return cudaSuccess;
    k_scan_env<<<We, 1024, 0, st>>>(envs, counts, off_local, EnvBases{env_total, env_base, host_base, ticket, longest}, 1, R);
    return cudaGetLastError();
}

cudaError_t launch_scan(const EnvInfo* envs, const uint32_t* counts, uint32_t* off_local,
                        unsigned long long* env_total, unsigned long long* env_base,
                        unsigned long long* host_base, unsigned int* ticket, int We, int per, cudaStream_t st) {
    if (We == 0) return cudaSuccess;
    k_scan_env<<<We, 1024, 0, st>>>(envs, counts, off_local, EnvBases{env_total, env_base, host_base, ticket, false}, per,
                                    RankParams{});
    return cudaGetLastError();
}

// ---------------------------------------------------------------- item order
// A warp composites a bucket of tens of thousands of keys in milliseconds, so
// a launch of a few items per warp ends on whichever long buckets were claimed
// last.  Claiming the long classes first fills the tail with short ones.  The
// lists keep the order of the environments within a class (up to the order of
// the blocks), so neighbouring tiles still share their records in L2.
__global__ void __launch_bounds__(256) k_item_order(const EnvInfo* envs, int e_begin, const uint32_t* counts,
                                                    const uint32_t* item_cnt, const uint32_t* item_off,
                                                    const unsigned long long* item_base, uint32_t* items,
                                                    uint32_t pitch, uint32_t* class_cnt) {
    const int el = e_begin + blockIdx.y, t = blockIdx.x * 256 + threadIdx.x;
    const int T = envs[el].T;
    if (blockIdx.x * 256 >= (unsigned)T) return;
    const uint32_t tile = envs[el].tile_base + (uint32_t)t;
    int cls = -1;
    uint32_t first = tile, cnt = 0;
    if (t < T) {
        const uint32_t n = counts[tile];
        cls = n >= 16384u ? 0 : n >= 4096u ? 1 : n >= 1024u ? 2 : 3;
        cnt = 1;
        if (item_cnt) {
            cnt = item_cnt[tile];
            first = (uint32_t)item_base[el] + item_off[tile];
        }
    }
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < kItemClasses; ++c) {  // one atomic per warp and class
        const uint32_t mine = cls == c ? cnt : 0u;
        uint32_t x = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, x, 31);
        if (total == 0u) continue;
        uint32_t at = 0;
        if (lane == 31) at = atomicAdd(class_cnt + c, total);
        at = __shfl_sync(0xffffffffu, at, 31) + x - mine;
        for (uint32_t k = 0; k < mine; ++k) items[(size_t)c * pitch + at + k] = first + k;
    }
}

cudaError_t launch_item_order(const EnvInfo* envs, int e_begin, int n_envs, int max_T, const uint32_t* counts,
                              const uint32_t* item_cnt, const uint32_t* item_off,
                              const unsigned long long* item_base, uint32_t* items, uint32_t pitch,
                              uint32_t* class_cnt, cudaStream_t st) {
    if (n_envs == 0 || max_T == 0) return cudaSuccess;
    k_item_order<<<dim3((unsigned)((max_T + 255) / 256), (unsigned)n_envs), 256, 0, st>>>(
        envs, e_begin, counts, item_cnt, item_off, item_base, items, pitch, class_cnt);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- scatter
// Where the blocks are those of k_count, the count has noted each block's place
// in every bucket it reaches.  Otherwise pass 1 rebuilds the block's histogram,
// and one global atomic per touched tile reserves the block's range of that
// bucket.  Then each rank is written at (bucket start + block range + shared
// cursor).  512 views of 128x128, 600,000 splats each: 1.20 ms with pass 1, 0.97
// with the noted places (bound by issue and by the latency of the records).  A key past the pair buffer's capacity (possible only for a
// launch planned with a fixed capacity) is dropped and flagged.

// The 8x8 subtiles of the tile (tx, ty) that a box reaches, one bit each,
// row-major.  lx, ly: log2 of the tile's subtile columns and rows (ly <= 1).
template <bool WRAP>
__device__ __forceinline__ uint32_t subtile_mask(uint32_t rx, uint32_t ry, int tx, int ty, int lx, int ly) {
    const int x0 = (int)(rx & 0xffffu) >> 3, x1 = (int)(rx >> 16) >> 3;
    const int ax = tx << lx, bx = ax + (1 << lx) - 1;
    uint32_t xm;
    if (WRAP && (rx & 0xffffu) > (rx >> 16)) {
        xm = (x0 <= bx ? (2u << (bx - ax)) - (1u << max(x0 - ax, 0)) : 0u) |
             (x1 >= ax ? (2u << min(x1 - ax, bx - ax)) - 1u : 0u);
    } else {
        xm = (2u << (min(x1, bx) - ax)) - (1u << max(x0 - ax, 0));
    }
    if (ly == 0) return xm;
    const int y0 = (int)(ry & 0xffffu) >> 3, y1 = (int)(ry >> 16) >> 3;
    return (y0 <= 2 * ty ? xm : 0u) | (y1 > 2 * ty ? xm << (1 << lx) : 0u);
}

constexpr int kLongSpan = 64;   // tiles: longer spans are walked by a warp
constexpr int kLongList = 512;  // of them listed at a time

template <bool WRAP, bool MASK, bool DIFF>
__global__ void __launch_bounds__(256, 6) k_scatter(BinParams P) {  // <= 42 registers: 6 CTAs/SM
    extern __shared__ uint32_t cur[];  // the block's histogram, then its next position per tile
    __shared__ uint16_t lst[32 * kWordsPerBlock];
    __shared__ uint16_t far[DIFF ? kLongList : 1];
    __shared__ uint32_t wtot[32];
    __shared__ uint32_t n_far;
    const int el = P.e_begin + blockIdx.y;
    const EnvInfo E = P.envs[el];
    const int64_t words = (E.n_local + 31) / 32;
    const int64_t w0 = (int64_t)blockIdx.x * P.words_per_block;
    if (w0 >= words) return;
    const int64_t w1 = min(w0 + (int64_t)P.words_per_block, words);
    const int ntx = E.ntx, nty = E.T / ntx;
    const uint32_t* off = P.off_local + E.tile_base;
    const bool known = !DIFF && P.tile_off;  // the count noted the block's place in each bucket
    if (known) {
        const uint32_t* mine = P.tile_off + ((size_t)el * gridDim.x + blockIdx.x) * P.tile_pitch;
        for (int t = threadIdx.x; t < E.T; t += blockDim.x) cur[t + t / ntx] = off[t] + mine[t];
    } else {
        for (int t = threadIdx.x; t < hist_words(ntx, nty); t += blockDim.x) cur[t] = 0;
    }
    if (threadIdx.x == 0) n_far = 0u;
    const int nvis = block_visible(P.mask + E.mask_base, w0, w1, lst, wtot);
    const uint4* r3 = P.r3 + E.rec_base + w0 * 32;
    const uint32_t* rank = P.rank + E.rec_base + w0 * 32;
    const int sx = __ffs(P.tile_w) - 1, sy = __ffs(P.tile_h) - 1;
    if (!known) {
        for (int i = threadIdx.x; i < nvis; i += blockDim.x) {
            const uint4 q = r3[lst[i]];
            add_box<WRAP, DIFF>(q.x, q.y, sx, sy, ntx, cur);
        }
        if constexpr (DIFF) block_sum2d(cur, ntx, nty);
        else __syncthreads();
        for (int t = threadIdx.x; t < E.T; t += blockDim.x) {
            uint32_t& c = cur[t + t / ntx];
            if (c) c = off[t] + atomicAdd(P.cursor + E.tile_base + t, c);
        }
        __syncthreads();
    }
    const unsigned long long eb = P.env_base[el] - P.pair_base;
    bool dropped = false;
    auto put = [&](const uint4& q, uint32_t key, int tx, int ty) {
        const unsigned long long pos = eb + atomicAdd(&cur[ty * (ntx + 1) + tx], 1u);
        const uint32_t v = MASK ? key << P.key_shift | subtile_mask<WRAP>(q.x, q.y, tx, ty, sx - 3, sy - 3) : key;
        if (pos < P.pair_cap) P.pairs[pos] = v;
        else dropped = true;
    };
    // Uniform trip count: the block drains its list of long spans together.  The
    // list's length for that decision is counted at the barrier and kept by every
    // thread; n_far only hands out places.  (Read after the barrier, n_far may
    // already hold places taken in the next round by warps that are ahead, and
    // warps that disagree on draining part at the barriers below.)
    uint32_t nf = 0;
    for (int i0 = 0; i0 < nvis; i0 += blockDim.x) {
        const int i = i0 + threadIdx.x;
        bool longer = false;
        if (i < nvis) {
            const uint4 q = r3[lst[i]];
            if constexpr (DIFF) {
                int tx0, tx1, ty0, ty1;
                tile_span(q.x, q.y, sx, sy, tx0, tx1, ty0, ty1);
                longer = (tx1 - tx0 + 1) * (ty1 - ty0 + 1) > kLongSpan;
                if (longer) far[atomicAdd(&n_far, 1u)] = (uint16_t)i;  // at most blockDim.x more per round
            }
            if (!longer) {
                const uint32_t key = rank[lst[i]];
                for_span<WRAP>(q.x, q.y, sx, sy, ntx, [&](int, int tx, int ty) { put(q, key, tx, ty); });
            }
        }
        if constexpr (DIFF) {
            nf += (uint32_t)__syncthreads_count(longer);
            if (nf + blockDim.x > (uint32_t)kLongList || (i0 + (int)blockDim.x >= nvis && nf)) {
                for (uint32_t k = threadIdx.x >> 5; k < nf; k += blockDim.x >> 5) {
                    const uint4 q = r3[lst[far[k]]];
                    const uint32_t key = rank[lst[far[k]]];
                    int tx0, tx1, ty0, ty1;
                    tile_span(q.x, q.y, sx, sy, tx0, tx1, ty0, ty1);
                    const int nx = tx1 - tx0 + 1, n = nx * (ty1 - ty0 + 1);
                    for (int t = threadIdx.x & 31; t < n; t += 32) put(q, key, tx0 + t % nx, ty0 + t / nx);
                }
                __syncthreads();
                if (threadIdx.x == 0) n_far = 0u;
                __syncthreads();
                nf = 0u;
            }
        }
    }
    if (__syncthreads_or(dropped) && threadIdx.x == 0) atomicOr(P.status, kStOverflow);
}

cudaError_t launch_scatter(const BinParams& P, int n_envs, int max_words, int max_T, int max_hist, cudaStream_t st) {
    if (n_envs == 0 || max_words == 0) return cudaSuccess;
    const bool diff = !P.wrap && max_T >= kDiffTiles, mask = P.key_shift > 0;
    const size_t smem = (size_t)max_hist * 4;
    auto launch = [&](auto fn) -> cudaError_t {
        const cudaError_t e = opt_in_smem((const void*)fn, smem);
        if (e != cudaSuccess) return e;
        fn<<<dim3((unsigned)((max_words + P.words_per_block - 1) / P.words_per_block), (unsigned)n_envs), 256, smem,
             st>>>(P);
        return cudaGetLastError();
    };
    if (P.wrap) return mask ? launch(k_scatter<true, true, false>) : launch(k_scatter<true, false, false>);
    if (diff) return mask ? launch(k_scatter<false, true, true>) : launch(k_scatter<false, false, true>);
    return mask ? launch(k_scatter<false, true, false>) : launch(k_scatter<false, false, false>);
}

}  // namespace gsb
