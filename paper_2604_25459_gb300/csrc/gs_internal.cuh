// Internal declarations shared by the CUDA translation units of libgsbatch.
//
// Device data layout (all in HBM):
//   Gaussians (scene-owned), background first (in the scene's Morton storage
//   order of the means) then link-major (storage index g):
//     p0[g] = {mean.x, mean.y, mean.z, opacity}
//     p1[g] = {F00, F01, F02, F10}      F = R diag(exp(s)), the factor of the 3D
//     p2[g] = {F11, F12, F20, F21}      covariance F F^T in the frame the mean lives
//     p3[g] = {F22, qstar, tr, link}    in (world for the background, link frame for
//                                       link Gaussians); qstar = 2 ln(255 o) (< 0
//                                       culls), tr = trace(F F^T), link = 0 for the
//                                       background, l+1 for link l (int bits)
//     sh plane-major: plane p holds values 4p..4p+3 (f32) or 8p..8p+7 (bf16/f16)
//     of the flattened [coefficient][channel] vector, for every g: sh[p][g].
//   Per wave of envs (scratch), env el described by EnvInfo envs[el]:
//     record slots: local index j = g for background Gaussians (padded to a
//       multiple of 32), then the env's link Gaussians in storage order; slot
//       (el, j) is slot s = envs[el].rec_base + j, valid where bit j%32 of
//       mask[envs[el].mask_base + j/32] is set; its first three 16-byte words
//       r0 = (u, v, log2 o, z), r1, r2 lie side by side at float4 index kRecStride s of one array
//       (the compositor gathers all three: two 32-byte sectors instead of
//       three half-used ones), its fourth word r3 at index s of another (the
//       binning reads only r3, coalesced across a warp).
//     rank[rec_base + j], order[rec_base + r]  the env's visible records in depth
//       order: sorted by (depth bits << 32 | i) with i the caller's local index
//       (background: its index before the Morton reordering; links: j), so equal
//       depths order by global index; rank[j] is record j's place and order[r]
//       the slot of place r.  nvis[el] records are ranked.
//     xf[envs[el].xf_base + f]  frame f = 0 background, f = 1 + (l - link_begin)
//     counts/off_local/cursor[envs[el].tile_base + t]  per (env, tile)
//     env_base[el]              exclusive scan of per-env intersection totals
//     pairs[...]                u32 ranks bucketed by (env, tile)
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "gsbatch.h"

namespace gsb {

// float4 stride between the r0 (r1, r2) words of consecutive record slots
// (r1 = r0 + 1, r2 = r0 + 2 in one array; see the layout above)
constexpr int kRecStride = 3;

// Stores the r0, r1, r2 words of a warp's 32 consecutive record slots
// (slot0 = the slot of lane 0) from the warp's staging buffer st (96 float4:
// word w of lane l at 3 l + w), with coalesced stores: lane l writes float4
// l, l + 32 and l + 64 of the slots' interleaved region, each where its record
// ((l + 32 k) / 3) is visible in m.  Direct per-lane stores at the 48-byte
// stride would write half sectors.  Call with every lane of the warp, after
// the lanes' staging writes and a __syncwarp().
__device__ __forceinline__ void store_records(float4* r0, size_t slot0, const float4* st, uint32_t m, int lane) {
    static_assert(kRecStride == 3, "three 16-byte words per record slot");
    float4* dst = r0 + (size_t)kRecStride * slot0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int i = lane + 32 * k;
        if ((m >> (i / 3)) & 1u) dst[i] = st[i];
    }
}

enum : uint32_t {
    kStBadPose = 1u,     // zero or non-finite link pose quaternion
    kStBadScene = 2u,    // zero or non-finite Gaussian quaternion at scene build
    kStOverflow = 4u,    // intersection keys beyond the capacity (planned launches) or a corrupted bucket
    kStBadRay = 8u,      // a ray direction outside its sensor's binning grid (or zero)
};

// Row-major rigid transform camera <- frame, plus the camera centre in that frame.
struct __align__(16) LinkXf {
    float4 r0;  // R00 R01 R02 t0
    float4 r1;  // R10 R11 R12 t1
    float4 r2;  // R20 R21 R22 t2
    float4 o;   // camera centre in the frame (x,y,z), unused
};

struct DevGaussians {
    int64_t n = 0;
    int64_t n_bg = 0;
    int n_links = 0;
    int sh_degree = 3;
    gs_dtype dtype = GS_F32;
    int sh_planes = 0;
    float4* p0 = nullptr;
    float4* p1 = nullptr;
    float4* p2 = nullptr;
    float4* p3 = nullptr;
    void* sh = nullptr;  // sh_planes * n * 16 bytes
};

inline int sh_values(int degree) { return 3 * (degree + 1) * (degree + 1); }
inline int sh_planes_for(int degree, gs_dtype dt) {
    int v = sh_values(degree);
    return dt == GS_F32 ? (v + 3) / 4 : (v + 7) / 8;
}

// One environment of a wave.
struct EnvInfo {
    unsigned long long rec_base;   // first record slot
    unsigned long long mask_base;  // first visibility word
    unsigned long long pix_base;   // first pixel of the env's image in the outputs
    long long pose_base;           // index (units of 7 floats) of the pose of link_begin
    unsigned int tile_base;        // first (env, tile) counter of the wave
    unsigned int n_local;          // record slots: padded background + the env's link Gaussians
    int xf_base;                   // first link-table entry
    int link_begin, n_links;       // links of the scene rendered in this env
    int W, H, ntx, T;              // image and tile grid
    int env;                       // index of the environment in the caller's batch
    long long g_link0;             // storage (= caller's) index of the env's first link Gaussian (slot bg_slots)
    float lim[4];                  // camera guard band: 1.3 cx/fx, 1.3 (W-cx)/fx, 1.3 cy/fy, 1.3 (H-cy)/fy
};

// A projection block: up to 256 consecutive Gaussians (thread t takes global
// index g_first + t, record slot local_first + t) for envs [e0, e1) of a wave;
// link frame of Gaussian with link field li is xf[envs[e].xf_base + li - lb].
struct ProjBlock {
    long long g_first;
    unsigned int local_first;  // multiple of 32
    int n;
    int e0, e1;
    int lb;
    int frame0;  // 1: every Gaussian of the block is background (link frame 0)
};

struct ProjParams {
    int64_t n_gauss;  // SH plane stride
    const float4* p0;
    const float4* p1;
    const float4* p2;
    const float4* p3;
    const void* sh;
    const ProjBlock* blocks;
    const EnvInfo* envs;
    const gs_camera* cams;  // per env of the wave
    const LinkXf* xf;
    float4* r0;
    float4* r1;
    float4* r2;
    uint4* r3;
    uint32_t* mask;
    float2* dbg_hxy;  // nullable, per record slot
    unsigned long long* nvis;  // nullable: visible (env, Gaussian) pair counter
    unsigned long long* nfp64; // nullable: counter of (env, Gaussian) pairs whose conic took the FP64 branch
    const gs_lidar* lidars;    // LiDAR projection only: per env of the wave
    const int* bg_index;       // nullable: caller's index of the background Gaussian in slot j (into r3.w)
    float cell_pad;            // LiDAR: grid boxes widened by this many cells (arbitrary rays: a ray
                               // anywhere in a cell, not only at its centre)
};

// Depth ranking of a wave's visible records (gs_rank.cu): per env a sample
// sort into `bins` key ranges, then windows of ranges sorted in shared memory.
struct RankParams {
    const EnvInfo* envs;
    const uint32_t* mask;
    const uint4* r3;
    long long max_slots;          // of the largest env
    int bins;                     // key ranges per env: a power of two, <= kRankBins; 0: envs are ranked whole
    int cells;                    // depth cells of the range lookup: a power of two
    int win_pitch;                // window table entries per env
    int words_per_block;          // of the count and of the placement (the same blocks)
    int blocks;                   // binning blocks per env
    unsigned long long* split;    // [We][bins]: splitters 0 .. bins-2, then the lookup's first depth and shift
    uint16_t* cell;               // [We][cells]: first range of each depth cell
    uint32_t* bin_cnt;            // [We][bins], zeroed
    uint32_t* bin_off;            // [We][bins]
    uint32_t* block_off;          // [We][blocks][bins]: keys of the range in earlier blocks
    uint32_t* win;                // [We][win_pitch]: window v holds positions [win[v], win[v+1])
    uint32_t* nvis;               // [We]
    unsigned long long* zkeys;    // [recs]: an env's keys from rec_base, grouped by range
    uint32_t* order;              // [recs]
    uint32_t* rank;               // [recs]; until the sort: range << 13 | place among the block's keys of it
    uint32_t* status;
    // the caller's local index of a record: camera records hold it in r3.w
    // (index_in_r3), LiDAR records map through bg_index (nullable: caller's
    // index of the background Gaussian in storage slot j < n_bg)
    int index_in_r3;
    const int* bg_index;
    const int* bg_slot;           // nullable: storage slot of the caller's background Gaussian i
    unsigned int n_bg;
};

struct BinParams {
    const EnvInfo* envs;
    const uint32_t* mask;
    const uint4* r3;
    int e_begin;             // first env (wave-local) handled by this launch
    int tile_w, tile_h;
    int words_per_block;     // of the scatter (the count shares the ranking's blocks)
    uint32_t* counts;
    const uint32_t* off_local;
    const unsigned long long* env_base;
    unsigned long long pair_base;   // env_base[e_begin], subtracted from absolute offsets
    unsigned long long pair_cap;    // keys the pair buffer holds
    uint32_t* cursor;
    uint32_t* pairs;
    const uint32_t* rank;
    uint32_t* status;
    int wrap;  // LiDAR: a box with x0 > x1 covers columns [x0, cols) and [0, x1]
    int key_shift;           // see CompParams
    // nullable: per env, block and tile (tile_pitch of them) the block's place in
    // the tile's bucket, where it has keys there; written by the count
    uint32_t* tile_off;
    unsigned int tile_pitch;
};

struct CompParams {
    const EnvInfo* envs;
    int e_begin, e_end;              // envs of this launch (wave-local)
    unsigned int item_begin, item_end;  // (env, tile) items: envs[e_begin].tile_base .. envs[e_end].tile_base
    int chunk;                       // items claimed per atomic
    unsigned int* work;              // work counter (zeroed before the launch)
    // nullable (warp form): the items in claiming order, kItemClasses lists of
    // class_cnt[c] items each, list c from items + c * item_pitch
    const uint32_t* items;
    const uint32_t* class_cnt;
    unsigned int item_pitch;
    unsigned int* team_work;  // nullable: the teams' work counter (zeroed before the launch)
    int team_classes;         // set by the launch: the first classes go to teams of four warps
    const float4* r0;                // records, r0, r1 and r2 side by side (kRecStride)
    const uint32_t* nvis;            // per env of the wave: ranked records
    const uint32_t* order;           // record slot of rank r at rec_base + r
    const uint32_t* counts;
    const uint32_t* off_local;
    const unsigned long long* env_base;
    unsigned long long pair_base;
    unsigned long long pair_cap;
    const uint32_t* pairs;
    unsigned long long* neval;       // nullable: composited (pixel, Gaussian) pair counter
    int tile_w, tile_h;
    int quad;       // camera images: the warp form (k_composite_warp)
    int even;       // no bucket of four times the average: no tail of long ones for teams
    // Keys of waves with envs in the warp form carry, below the rank, one bit
    // per 8x8 subtile of the tile that the record's box reaches (row-major): key
    // = rank << key_shift | mask.  key_shift = 0: no mask (plain ranks).
    int key_shift;
    float* rgb;     // images at envs[e].pix_base (x3 for rgb); unused when rgb8 is set
    float* depth;   // unused when depth16 is set
    float* alpha;   // nullable
    uint8_t* rgb8;        // nullable: observation RGB, 8 bits per channel, at pix_base (x3)
    uint16_t* depth16;    // nullable: observation depth, IEEE half bits, at pix_base
    const gs_appearance* appear;  // nullable: per env (wave-local index) for rgb8
    float* score;         // nullable: contribution pass (no images): score[g] += sum of alpha T
    unsigned int nbp;     // background slots (slot j < nbp is the background Gaussian stored at j)
    const int* bg_index;  // nullable: caller's index of the background Gaussian in slot j (contribution pass, debug)
    const gs_lidar* lidars;  // nullable: LiDAR scan (range in depth, hit in alpha), per env of the wave
    const uint4* r3;         // LiDAR scan: records' fourth word (|g2|)
    uint32_t* status;
    // Arbitrary rays (set with lidars): items are (env, tile, chunk of <= 64
    // rays); outputs are indexed by ray, at envs[e].pix_base + ray.
    const float* ray_dirs;         // [wave env][n_rays][3], sensor frame
    const uint32_t* ray_cell;      // [wave env][n_rays]: tile << 8 | cell in tile (row-major 16x16)
    const uint32_t* ray_list;      // [wave env][n_rays]: ray indices grouped by tile, then 4x4 quadrant
    const uint32_t* ray_cnt;       // per (env, tile, quadrant) at kRayGroups tile_base: its rays
    const uint32_t* ray_off;       // per (env, tile, quadrant): its first entry in the env's ray_list
    const uint32_t* item_off;      // per (env, tile): first item of the tile within its env
    const unsigned long long* item_base;  // per wave env (+1): first item of the env
    int n_rays;
};

// Launchers (return cudaGetLastError()).
// Input Gaussian i is stored at dst_offset + (place ? place[i] : i).
cudaError_t launch_prep(const float* mean, const float* quat, const void* log_scale, const void* opacity,
                        const void* sh, int64_t n, int64_t dst_offset, const int64_t* place, int link_mode,
                        const int64_t* link_offsets, int n_links, const DevGaussians& D, uint32_t* status,
                        cudaStream_t st);
// n_items = sum over envs of (1 + n_links); envs[We].xf_base must hold n_items.
cudaError_t launch_link_table(const float* poses, const gs_camera* cams, const EnvInfo* envs, int We, int n_items,
                              LinkXf* out, uint32_t* status, cudaStream_t st);
cudaError_t launch_project(const DevGaussians& D, const ProjParams& P, int n_blocks, cudaStream_t st);
// LiDAR records: r0 = (b, o), r1 = (g0, x-range), r2 = (g1, y-range), r3 =
// (x-range, y-range, distance bits, |g2| bits) with g_k the rows of
// diag(e^-s) R^T in the sensor frame and b = G mu; ranges over the
// (azimuth, beam) grid.
cudaError_t launch_project_lidar(const ProjParams& P, int n_blocks, cudaStream_t st);
// Arbitrary rays, per wave: the cell of every ray on its sensor's binning
// grid (zero and out-of-grid directions flagged and left out) and the rays per
// (env, tile); then the rays grouped by tile and the compositor's items
// (chunks of at most kRayChunk rays per tile).  ray_cnt and ray_cur are zeroed
// by the caller.
constexpr int kRayChunk = 64;
constexpr int kRayGroups = 16;  // 4x4 quadrants per tile, by which a tile's rays are grouped
cudaError_t launch_ray_count(const float* dirs, const gs_lidar* lidars, const EnvInfo* envs, int We, int n_rays,
                             uint32_t* cell, uint32_t* cnt, uint32_t* status, cudaStream_t st);
cudaError_t launch_ray_scatter(const EnvInfo* envs, int We, int n_rays, const uint32_t* cell, const uint32_t* off,
                               uint32_t* cur, uint32_t* list, const uint32_t* cnt, uint32_t* item_cnt,
                               unsigned int tiles, cudaStream_t st);
// max_T, max_hist: tiles and padded tile histogram ((ntx + 1) (nty + 1)) of the
// largest env.  The count also histograms the records over the env's depth
// ranges (R).
cudaError_t launch_count(const BinParams& P, const RankParams& R, int n_envs, int max_T, int max_hist,
                         cudaStream_t st);
// per: counters per tile (counts and off_local hold per T from per tile_base).
// host_base: pinned host memory that gets a copy of env_base, or null; ticket: a
// word that holds 0, and does so again afterwards.
cudaError_t launch_scan(const EnvInfo* envs, const uint32_t* counts, uint32_t* off_local,
                        unsigned long long* env_total, unsigned long long* env_base,
                        unsigned long long* host_base, unsigned int* ticket, int We, int per, cudaStream_t st);
// As launch_scan, with the scans of the depth ranges and their window tables.
// longest: host_base gets the keys of each env's longest bucket (at most
// kTotalMost) above its low kTotalBits bits.
constexpr int kTotalBits = 40;
constexpr uint32_t kTotalMost = (1u << (64 - kTotalBits)) - 1u;
cudaError_t launch_scan_ranks(const EnvInfo* envs, const uint32_t* counts, uint32_t* off_local,
                              unsigned long long* env_total, unsigned long long* env_base,
                              unsigned long long* host_base, bool longest, unsigned int* ticket, int We,
                              const RankParams& R, cudaStream_t st);
cudaError_t launch_scatter(const BinParams& P, int n_envs, int max_words, int max_T, int max_hist, cudaStream_t st);
// Lists a launch's items by the length of their buckets, longest class first
// (CompParams::items); class_cnt is zeroed by the caller.  Rays: item_cnt and
// item_off per (env, tile) and item_base per env give a tile's items.
constexpr int kWorkWords = 8;    // work counters of a launch (see run_wave)
constexpr int kItemClasses = 4;  // buckets of >= 16384, >= 4096, >= 1024 and fewer keys
cudaError_t launch_item_order(const EnvInfo* envs, int e_begin, int n_envs, int max_T, const uint32_t* counts,
                              const uint32_t* item_cnt, const uint32_t* item_off,
                              const unsigned long long* item_base, uint32_t* items, uint32_t pitch,
                              uint32_t* class_cnt, cudaStream_t st);
// Depth ranking: splitters before the count, ranks after the scan.
cudaError_t launch_rank_sample(const RankParams& R, int n_envs, cudaStream_t st);
cudaError_t launch_rank(const RankParams& R, int n_envs, int max_words, cudaStream_t st);
// grid = persistent CTAs; returns the grid size used through *ctas.  The warp
// form (launch_composite_warp) renders LiDAR scans and, with P.quad, images.
cudaError_t launch_composite(const CompParams& P, cudaStream_t st, int* ctas);
cudaError_t launch_composite_warp(const CompParams& P, cudaStream_t st, int* ctas);

constexpr int kWordsPerBlock = 256;  // binning block: at most one visibility word per thread of 256 (8192 slots)
constexpr int kRankBins = 2048;      // depth ranges per env, at most
constexpr int kRankStride = 768;     // ranks per window of the depth sort
// Depth ranges of an env of n record slots: one per 512 slots for cameras
// (which see a quarter of a room), one per 256 for LiDARs (which see all of it).
// Envs of at most this many slots are ranked whole, by one CTA each, as many keys
// as its shared memory sorts.  Calls by sampling / whole (us): 8 views of 128x96 of
// 3000 splats without allocation 98 / 79, 24 of 4000 120 / 105; 64 of 64x48 of 3000
// 135 / 128, 200 201 / 185; one of 300x250 of 4000 75 / 69.
constexpr int kSmallRank = 4096;
inline int rank_bins(long long n, bool lidar) {
    const int most = lidar ? kRankBins : kRankBins / 2;
    int b = 32;
    while (b < most && (long long)b * (lidar ? 256 : 512) < n) b *= 2;
    return b;
}
// Sizes the ranking of We envs of at most max_words visibility words.  Binning
// blocks: as few words as still give every SM a few blocks, but no fewer slots
// than two per range (a block keeps an offset per range).
inline RankParams rank_sizes(long long max_words, int We, bool lidar) {
    RankParams R{};
    R.max_slots = max_words * 32;
    R.bins = R.max_slots <= kSmallRank ? 0 : rank_bins(R.max_slots, lidar);
    R.cells = R.bins < 1024 ? 4 * R.bins : 4096;
    R.win_pitch = (int)(max_words * 32 / kRankStride) + 2;
    int w = kWordsPerBlock;
    while (w > 16 && w > R.bins / 16 && (max_words + w - 1) / w * We < 4 * 152) w /= 2;
    R.words_per_block = w;
    R.blocks = (int)((max_words + w - 1) / w);
    return R;
}
// Tile grids of at least this many tiles are counted by difference arrays
// (average spans at 128x128, 64 tiles, are 2.1 tiles; at 320x240, 300: 4.5; at
// 640x480: 11).
constexpr int kDiffTiles = 256;
// Bytes of the places that the count notes for the scatter (BinParams::tile_off);
// 0 where their blocks differ, and on grids counted by difference arrays.
inline size_t tile_off_bytes(const RankParams& R, int words_per_block, int We, int max_T, bool wrap) {
    if (words_per_block != R.words_per_block || (!wrap && max_T >= kDiffTiles)) return 0;
    return (size_t)We * R.blocks * max_T * 4;
}
// Visibility words per scatter block: many blocks per SM, as one block may hold
// a link that fills the image (at 640x480, 32 envs: 30 us per env with 256
// words, 13 with 32), and on large grids 64, whose writes stay in reach of the
// L2 (256 envs: 8.5 us per env with 256, 7.15 with 64, 8.6 with 32); on small
// grids the per-block tables weigh more (512 envs at 128x128: 2.3 us with 256,
// 2.7 with 64).
inline int scatter_words(long long max_words, int n_envs, int max_T) {
    int w = max_T >= kDiffTiles ? 64 : kWordsPerBlock;
    while (w > 16 && (max_words + w - 1) / w * n_envs < 62 * 152) w /= 2;
    return w;
}
// Bytes of the ranking's per-env tables (everything but bin_cnt, zkeys, order
// and rank) for We envs, and their layout from a 16-byte aligned base.
inline size_t rank_tables(RankParams& R, int We, unsigned char* base) {
    const size_t nb = (size_t)We * R.bins;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        unsigned char* p = base + o;
        o = (o + bytes + 15) & ~size_t(15);
        return p;
    };
    R.split = reinterpret_cast<unsigned long long*>(take(nb * 8));
    R.cell = reinterpret_cast<uint16_t*>(take((size_t)We * R.cells * 2));
    R.bin_off = reinterpret_cast<uint32_t*>(take(nb * 4));
    R.block_off = reinterpret_cast<uint32_t*>(take(nb * R.blocks * 4));
    R.win = reinterpret_cast<uint32_t*>(take((size_t)We * R.win_pitch * 4));
    R.nvis = reinterpret_cast<uint32_t*>(take((size_t)We * 4));
    return o;
}
// Depth-ordered window held in shared memory by the compositor.
constexpr int kCompCap = 768;
// Plain renders use the warp form of the compositor on 16x16 or 8x8 tiles when
// no image of the wave has more pixels than this.  Scatter + compositing, CTA
// form / warp form (us, the room): 400x300: 1 env 215 / 148, 4 586 / 307, 16
// 837 / 776, 64 2290 / 2152; 480x360: 160 / 174, 419 / 352, 835 / 833, 2617 /
// 2658; 640x480: 155 / 200, 379 / 475, 1007 / 1097, 3399 / 3859.
constexpr int kQuadMaxPixels = 140000;
// Envs of few slots have short buckets, which the CTA form sorts at once, without
// an item order.  Calls, warp / CTA form (us): 24 envs of 1500 splats at 64x48 106
// / 94, of 4000 at 128x96 132 / 123, of 6000 at 40x30 158 / 236; 64 of 3000 at 64x48
// 142 / 132; 200 of 1100 in the room at 32x24 130 / 118, of 2200 at 64x48 167 / 156,
// 200 even cubes of 2000 at 64x48 165 / 176.
constexpr long long kQuadMinSlots = 4097;
inline bool warp_form(int tile_w, int tile_h, long long most_pixels, long long most_slots) {
    return ((tile_w == 16 && tile_h == 16) || (tile_w == 8 && tile_h == 8)) && most_pixels <= kQuadMaxPixels &&
           most_slots >= kQuadMinSlots;
}
// Whether the warp form pays for images of `tiles` tiles with `keys` keys, the
// longest bucket `most` (of the envs that warp_form admits).  On buckets that are
// short on average, four warps that share a window beat four that each order
// their own, unless long buckets among them would leave a CTA behind alone, or
// the tiles are so few that latency counts.  Scatter + compositing, CTA form / warp
// form (us).  The room, where a tenth of the tiles holds most keys: 333x251, 32
// views of 9,000 slots (78 keys per tile) 180 / 227, of 30,000 (200) 315 / 289, of
// 600,000 (2233) 1112 / 1119; 128x96, 64 views of 600,000 (6396) 4591 / 1521.  An
// even cube: 300x250, 8 views of 120,000 (1209 per tile, 2432 tiles) 165 / 313; 128x96
// of 30,000 (1095): 64 views (3072 tiles) 347 / 427, 4 views (192) 119 / 77; of
// 120,000 (4361): 64 views 571 / 462.
constexpr unsigned long long kEvenTiles = 400;
inline bool even_buckets(unsigned long long tiles, unsigned long long keys, unsigned long long most) {
    return tiles >= kEvenTiles && most * tiles < 4 * keys;
}
inline bool warp_pays(unsigned long long tiles, unsigned long long keys, unsigned long long most) {
    return keys >= 100 * tiles && (!even_buckets(tiles, keys, most) || keys >= 3200 * tiles);
}
// Bits of the subtile mask below the ranks of the warp form's keys: one per 8x8
// subtile while they and the ranks of n_slots records fit 32 bits, else none.
inline int subtile_bits(int tile_w, int tile_h, unsigned long long n_slots) {
    const int n = (tile_w / 8) * (tile_h / 8);
    return n > 1 && (n_slots >> (32 - n)) == 0 ? n : 0;
}

// Read-only view of a scene's device data for entry points outside gs_api.cu.
struct SceneView {
    int device;
    DevGaussians D;
    uint32_t* status;
    int tile_w, tile_h;
    const int* bg_index;  // nullable: caller's index of the background Gaussian in storage slot j
    const int* bg_slot;   // nullable: storage slot of the caller's background Gaussian i
};
SceneView scene_view(gs_scene s);
// Set the thread-local message returned by gs_last_error and return st.
gs_status report(gs_status st, const char* msg);

// Host-side construction of a wave's tables (shared by all entry points).
struct EnvSpec {        // one env as requested by the caller
    const gs_camera* cam;
    int link_begin, link_end;
    long long pose_offset;    // pose index of link_begin
    long long pixel_offset;   // first pixel of the image
    int env = 0;              // its index in the caller's batch
};
int64_t bg_slots(int64_t n_bg);  // background slots padded to 32
// Fills envs (n+1 entries; the last holds the totals in rec_base, mask_base,
// tile_base and xf_base) and appends projection blocks; returns totals through
// the EnvInfo sentinel.  link_offsets: host copy of the scene's link offsets.
void build_wave_tables(const DevGaussians& D, const int64_t* link_offsets, const EnvSpec* specs, int n, int tile_w,
                       int tile_h, long long pix_rebase, EnvInfo* envs, ProjBlock* blocks, int* n_blocks,
                       int max_blocks);
int count_wave_blocks(const DevGaussians& D, const int64_t* link_offsets, const EnvSpec* specs, int n);

}  // namespace gsb
