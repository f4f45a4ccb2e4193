// The compositor's warp form: one warp composites one 8x8 subtile (or up to 64
// rays) on its own, from its tile's bucket to its pixels.  It renders camera
// images of low resolution and every LiDAR scan (paper Sec. III-C, Sec. III-E);
// gs_composite.cu holds the form for large images.
//
// At 128x128 a splat covers a few pixels and half of a view's keys fall in two
// or three tiles: the four warps of a 16x16 tile's CTA spent more time waiting
// for one another at each staged batch than on any other stall, and the chip
// drained on the longest buckets.  Here a subtile's warp shares nothing, so
// there is no barrier left; every lane stages one splat, tests it against the
// subtile in registers, and the records of the next 32 splats are copied
// (cp.async) while the current ones are blended.  The four warps of a tile each
// read the tile's bucket and keep the keys whose subtile bit is set.
//
// The bucket's keys are depth ranks (gs_rank.cu) in any order; windows of at
// most CAP ranks come in order from
//   - the whole bucket at once, if it is short;
//   - a histogram over kSortBins rank ranges, windows being runs of ranges
//     gathered from the bucket and sorted in shared memory (few keys per rank:
//     LiDAR scans rank every Gaussian around the sensor);
//   - a bitmap of the next 32768 ranks (many keys per rank), read back in order.
// Each pixel blends the same splats in the same order with the same arithmetic
// as in gs_composite.cu, so the images do not depend on the form.
#include "gs_blend.cuh"
#include "gs_block.cuh"

namespace gsb {

namespace {

constexpr uint32_t kAll = 0xffffffffu;
constexpr int kWarps = 4;         // warps per CTA (independent; one CTA per warp would cost 1 KB of shared memory each)
constexpr int kSortBins = 512;    // counters of the sort and of the histogram
constexpr int kCrowd = 32;        // longest range sorted by counting
constexpr int kWords = 1024;      // bitmap words
constexpr uint32_t kShort = 1024; // buckets gathered whole

// f(key, valid) for every key of the bucket L[0, n), by the whole warp: 16-byte
// loads, four in flight per lane.  Reads up to three words on either side of
// the bucket (the key buffer is padded); they come with valid = false.
template <typename F>
__device__ __forceinline__ void warp_keys(const uint32_t* L, uint32_t n, F&& f) {
    constexpr int U = 4;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t off = (uint32_t)((uintptr_t)L & 15u) >> 2, end = off + n;
    const uint4* V = reinterpret_cast<const uint4*>(L - off);
    for (uint32_t i = 0; i < end; i += 128 * U) {
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t x = i + 128 * u + 4 * lane;
            v[u] = x < end ? __ldg(V + (x >> 2)) : make_uint4(0u, 0u, 0u, 0u);
        }
        if (i >= off && i + 128 * U <= end) {  // no word outside the bucket
#pragma unroll
            for (int u = 0; u < U; ++u) {
                f(v[u].x, true);
                f(v[u].y, true);
                f(v[u].z, true);
                f(v[u].w, true);
            }
            continue;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t x = i + 128 * u;
            if (x >= end) break;
            const uint32_t y = x + 4 * lane - off;  // index in the bucket; wraps below it
            f(v[u].x, y < n);
            f(v[u].y, y + 1 < n);
            f(v[u].z, y + 2 < n);
            f(v[u].w, y + 3 < n);
        }
    }
}

// Sorts keys[0, m), distinct ranks in [lo, hi], m <= 512 (tmp: scratch).  One key per lane: a bitonic network in
// registers.  Otherwise a counting sort by kSortBins equal ranges,
// a rank's place in its range being the number of smaller ones, or, when a range holds more than kCrowd, a bitonic
// sort in shared memory.
__device__ __forceinline__ void warp_sort(uint32_t* keys, uint32_t* tmp, uint32_t* cnt, int m, uint32_t lo,
                                          uint32_t hi) {
    const int lane = threadIdx.x & 31;
    if (m <= 32) {
        uint32_t k = lane < m ? keys[lane] : kAll;
#pragma unroll
        for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                const uint32_t o = __shfl_xor_sync(kAll, k, stride);
                const bool up = (lane & size) == 0, low = (lane & stride) == 0;
                k = up == low ? min(k, o) : max(k, o);
            }
        keys[lane] = k;
        __syncwarp();
        return;
    }
    const uint32_t span = hi - lo;
    const int shift = (span >> 9) ? 23 - __clz(span) : 0;  // span >> shift < kSortBins
    uint4* c4 = reinterpret_cast<uint4*>(cnt);
#pragma unroll
    for (int j = 0; j < kSortBins / 128; ++j) c4[lane + 32 * j] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    for (int i = lane; i < m; i += 32) atomicAdd(&cnt[(keys[i] - lo) >> shift], 1u);
    __syncwarp();
    constexpr int PER = kSortBins / 32;
    uint32_t sum = 0, most = 0;
    uint4 q[PER / 4];
#pragma unroll
    for (int j = 0; j < PER / 4; ++j) {
        q[j] = c4[lane * (PER / 4) + j];
        sum += q[j].x + q[j].y + q[j].z + q[j].w;
        most = max(most, max(max(q[j].x, q[j].y), max(q[j].z, q[j].w)));
    }
    if (__any_sync(kAll, most > (uint32_t)kCrowd)) {
        int p = 64;
        while (p < m) p <<= 1;
        for (int i = m + lane; i < p; i += 32) keys[i] = kAll;
        for (int size = 2; size <= p; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                __syncwarp();
                for (int x = lane; x < p / 2; x += 32) {
                    const int i = 2 * x - (x & (stride - 1)), j = i + stride;
                    const uint32_t a = keys[i], b = keys[j];
                    if ((a > b) == ((i & size) == 0)) {
                        keys[i] = b;
                        keys[j] = a;
                    }
                }
            }
        __syncwarp();
        return;
    }
    uint32_t run = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kAll, run, d);
        if (lane >= d) run += y;
    }
    run -= sum;
#pragma unroll
    for (int j = 0; j < PER / 4; ++j) {
        uint4 r;
        r.x = run;
        r.y = r.x + q[j].x;
        r.z = r.y + q[j].y;
        r.w = r.z + q[j].z;
        run = r.w + q[j].w;
        c4[lane * (PER / 4) + j] = r;
    }
    __syncwarp();
    for (int i = lane; i < m; i += 32) {
        const uint32_t k = keys[i];
        tmp[atomicAdd(&cnt[(k - lo) >> shift], 1u)] = k;
    }
    __syncwarp();
    // cnt[b] is the end of range b now; a rank's place in its range is the
    // number of smaller ranks there
    for (int i = lane; i < m; i += 32) {
        const uint32_t k = tmp[i];
        const int b = (int)((k - lo) >> shift);
        const uint32_t e = cnt[b];
        uint32_t place = b ? cnt[b - 1] : 0u;
        for (uint32_t x = place; x < e; ++x) place += tmp[x] < k ? 1u : 0u;
        keys[place] = k;
    }
    __syncwarp();
}

// An item's place: the env, its first tile, the tile and (rays) the chunk of
// the tile's rays.  Carried from item to item.
struct Where {
    int el;
    unsigned int e_lo, e_hi;  // the env's tiles
    int t;
    uint32_t rchunk;
};

template <int MODE>
__device__ __forceinline__ void locate(const CompParams& P, unsigned int item, unsigned int t_env, Where& w) {
    if constexpr (MODE == 3) {
        int lo = P.e_begin, hi = P.e_end - 1;  // env: last e with item_base[e] <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&P.item_base[mid]) <= (unsigned long long)item) lo = mid; else hi = mid - 1;
        }
        w.el = lo;
        w.e_lo = __ldg(&P.envs[lo].tile_base);
        const uint32_t li = item - (uint32_t)__ldg(&P.item_base[lo]);
        int a = 0, b = __ldg(&P.envs[lo].T) - 1;  // tile: last t with item_off[t] <= li (empty tiles come before)
        while (a < b) {
            const int mid = (a + b + 1) >> 1;
            if (__ldg(&P.item_off[w.e_lo + mid]) <= li) a = mid; else b = mid - 1;
        }
        w.t = a;
        w.rchunk = li - __ldg(&P.item_off[w.e_lo + a]);
    } else {
        if (item < w.e_lo || item >= w.e_hi) {
            // uniform batches: by division
            w.el = min(P.e_begin + (int)((item - P.item_begin) / t_env), P.e_end - 1);
            w.e_lo = __ldg(&P.envs[w.el].tile_base);
            w.e_hi = w.e_lo + (unsigned)__ldg(&P.envs[w.el].T);
            if (item < w.e_lo || item >= w.e_hi) {
                int lo = P.e_begin, hi = P.e_end - 1;  // env: last e with tile_base <= item
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (__ldg(&P.envs[mid].tile_base) <= item) lo = mid; else hi = mid - 1;
                }
                w.el = lo;
                w.e_lo = __ldg(&P.envs[lo].tile_base);
                w.e_hi = w.e_lo + (unsigned)__ldg(&P.envs[lo].T);
            }
        }
        w.t = (int)(item - w.e_lo);
    }
}

// A lane's two pixels or rays.
struct Lane {
    bool in0, in1;
    float fpx;
    float2 fpy;           // camera: pixel centres (fpx, fpy.x) and (fpx, fpy.y)
    int cx0, cy0, cx1, cy1;  // pixels, or the rays' grid cells
    float3 dir0, dir1;    // LiDAR: unit directions
    int ray0, ray1;       // MODE 3: ray indices
    float near_range;
};

// Pixels (px, py) and (px, py + DY).
template <int MODE, int DY>
__device__ __forceinline__ void lane_pixels(const CompParams& P, int el, int W, int H, int px, int py, Lane& L) {
    L.in0 = px < W && py < H;
    L.in1 = px < W && py + DY < H;
    L.fpx = (float)px + 0.5f;
    L.fpy = make_float2((float)py + 0.5f, (float)(py + DY) + 0.5f);
    L.cx0 = L.cx1 = px;
    L.cy0 = py;
    L.cy1 = py + DY;
    if constexpr (MODE == 1) {
        const gs_lidar* Ld = P.lidars + el;
        const float em = __ldg(&Ld->elev_min), eM = __ldg(&Ld->elev_max);
        const float az0 = __ldg(&Ld->az_min), span = __ldg(&Ld->az_max) - az0;
        const float phi = az0 + span * L.fpx / (float)W;
        const float th0 = em + (eM - em) * L.fpy.x / (float)H, th1 = em + (eM - em) * L.fpy.y / (float)H;
        float sp, cp, s0, c0, s1, c1;
        sincosf(phi, &sp, &cp);
        sincosf(th0, &s0, &c0);
        sincosf(th1, &s1, &c1);
        L.dir0 = make_float3(c0 * cp, c0 * sp, s0);
        L.dir1 = make_float3(c1 * cp, c1 * sp, s1);
        L.near_range = __ldg(&Ld->near_range);
    }
}

// Rays k0 and k1 of the tile's list (grouped by quadrant); returns the subtile
// bits they lie in.
__device__ __forceinline__ uint32_t lane_rays(const CompParams& P, const Where& w, int tx, int ty, uint32_t k0,
                                              uint32_t k1, Lane& L) {
    const size_t renv = (size_t)w.el * (size_t)P.n_rays;
    const size_t rt = kRayGroups * (size_t)(w.e_lo + w.t), last = rt + kRayGroups - 1;
    const uint32_t first = __ldg(P.ray_off + rt), total = __ldg(P.ray_off + last) + __ldg(P.ray_cnt + last) - first;
    const uint32_t* list = P.ray_list + renv + first;
    L.in0 = k0 < total;
    L.in1 = k1 < total;
    L.near_range = __ldg(&P.lidars[w.el].near_range);
    L.ray0 = L.ray1 = -1;
    L.cx0 = L.cy0 = L.cx1 = L.cy1 = 0;
    L.dir0 = L.dir1 = make_float3(0.f, 0.f, 0.f);
    uint32_t subs = 0;
    auto take = [&](uint32_t k, int& ray, int& ci, int& cj, float3& d) {
        const uint32_t r = __ldg(list + k);
        ray = (int)r;
        const uint32_t c = __ldg(&P.ray_cell[renv + r]) & 255u;
        ci = tx * 16 + (int)(c & 15u);
        cj = ty * 16 + (int)(c >> 4);
        subs |= 1u << (((c >> 6) & 2u) | ((c >> 3) & 1u));
        const float* v = P.ray_dirs + (renv + r) * 3;
        const float x = v[0], y = v[1], z = v[2];
        const float inv = 1.0f / sqrtf(x * x + y * y + z * z);
        d = make_float3(x * inv, y * inv, z * inv);
    };
    if (L.in0) take(k0, L.ray0, L.cx0, L.cy0, L.dir0);
    if (L.in1) take(k1, L.ray1, L.cx1, L.cy1, L.dir1);
    return subs;
}

// LiDAR: alpha and t* of a staged Gaussian (b, o | g0 | g1 | g2) on each of the
// lane's two rays d: u = G d, q = |u x b|^2 / |u|^2, t* = u.b / |u|^2, with
// paired FP32 instructions (the reciprocal of |u|^2 by the fast division, ~2
// ulp, far inside the scan's tolerance).
__device__ __forceinline__ void ray_eval2(const Lane& L, const float4& A, const float4& B, const float4& C,
                                          const float4& D, float2& al, float2& ts) {
    const float2 dx = make_float2(L.dir0.x, L.dir1.x), dy = make_float2(L.dir0.y, L.dir1.y),
                 dz = make_float2(L.dir0.z, L.dir1.z);
    auto dot = [&](const float4& G) {
        return __ffma2_rn(make_float2(G.z, G.z), dz,
                          __ffma2_rn(make_float2(G.y, G.y), dy, __fmul2_rn(make_float2(G.x, G.x), dx)));
    };
    const float2 u0 = dot(B), u1 = dot(C), u2 = dot(D);
    const float2 aa = __ffma2_rn(u2, u2, __ffma2_rn(u1, u1, __fmul2_rn(u0, u0)));
    const float2 ab = __ffma2_rn(u2, make_float2(A.z, A.z),
                                 __ffma2_rn(u1, make_float2(A.y, A.y), __fmul2_rn(u0, make_float2(A.x, A.x))));
    const float2 c0 = __ffma2_rn(u1, make_float2(A.z, A.z), __fmul2_rn(u2, make_float2(-A.y, -A.y)));
    const float2 c1 = __ffma2_rn(u2, make_float2(A.x, A.x), __fmul2_rn(u0, make_float2(-A.z, -A.z)));
    const float2 c2 = __ffma2_rn(u0, make_float2(A.y, A.y), __fmul2_rn(u1, make_float2(-A.x, -A.x)));
    const float2 cc = __ffma2_rn(c2, c2, __ffma2_rn(c1, c1, __fmul2_rn(c0, c0)));
    const float2 inv = make_float2(__fdividef(1.0f, aa.x), __fdividef(1.0f, aa.y));
    const float2 q = __fmul2_rn(cc, inv);
    ts = __fmul2_rn(ab, inv);
    const float k = -0.72134752044448170f;  // -log2(e) / 2
    al.x = ts.x > L.near_range ? fminf(0.99f, A.w * ex2_approx(k * q.x)) : 0.0f;
    al.y = ts.y > L.near_range ? fminf(0.99f, A.w * ex2_approx(k * q.y)) : 0.0f;
}

// LiDAR: the third row of G, |g2| (g0 x g1) / (|g0| |g1|) (the rows are
// orthogonal).
__device__ __forceinline__ float4 third_row(const float4& q1, const float4& q2, float glen2) {
    const float gx = q1.y * q2.z - q1.z * q2.y, gy = q1.z * q2.x - q1.x * q2.z, gz = q1.x * q2.y - q1.y * q2.x;
    const float k = glen2 * rsqrtf((q1.x * q1.x + q1.y * q1.y + q1.z * q1.z) *
                                   (q2.x * q2.x + q2.y * q2.y + q2.z * q2.z));
    return make_float4(gx * k, gy * k, gz * k, 0.0f);
}

// LiDAR: a box across azimuth 0 (x0 > x1: columns [x0, cols) and [0, x1])
// becomes the hull of its parts in the 16 columns of tile column tx: the high
// part [max(x0, ta), tb] when x0 <= tb and the low part [ta, min(x1, tb)] when
// x1 >= ta.
__device__ __forceinline__ void unwrap_box(int tx, int& bx0, int& bx1) {
    if (bx0 <= bx1) return;
    const int ta = tx * 16, tb = ta + 15;
    const int h0 = max(bx0, ta), l1 = min(bx1, tb);
    bx0 = bx1 >= ta ? ta : h0;
    bx1 = h0 <= tb ? tb : l1;
}

__device__ __forceinline__ bool in_box(const int4& R, int x, int y) {
    return (unsigned)(x - R.x) <= (unsigned)R.y && (unsigned)(y - R.z) <= (unsigned)R.w;
}

// One tile's bucket.
struct Bucket {
    const uint32_t* keys;
    uint32_t n;
    uint32_t n_rank;        // ranks of the env; keys beyond them (a corrupted bucket's) are left out
    const uint32_t* order;  // record slot of each rank
    size_t recbase;
    uint32_t n_local;
};
__device__ __forceinline__ Bucket find_bucket(const CompParams& P, const Where& w, bool first_thread) {
    Bucket b;
    b.n = P.counts[w.e_lo + w.t];
    const unsigned long long start = __ldg(P.env_base + w.el) - P.pair_base + P.off_local[w.e_lo + w.t];
    if (start + b.n > P.pair_cap) {  // keys past a planned capacity were dropped: render nothing
        b.n = 0;
        if (first_thread) atomicOr(P.status, kStOverflow);
    }
    b.keys = P.pairs + start;
    b.recbase = (size_t)__ldg(&P.envs[w.el].rec_base);
    b.n_local = __ldg(&P.envs[w.el].n_local);
    b.order = P.order + b.recbase;
    b.n_rank = __ldg(P.nvis + w.el);
    return b;
}


// ------------------------------------------------------------------ teams
// A long bucket by the four warps of a CTA: a warp takes one 4x4 quadrant of
// the subtile (rays: a quarter of the chunk), they share the ordering and the
// staging, 128 splats at a time.  All four groups of eight lanes hold the same
// 16 pixels: a step takes the next four splats of the quadrant, group g
// evaluates splat g, the alphas go round by shuffles, every group follows the
// transmittance through all four, and group g keeps channel g of r, g, b, depth
// (LiDAR: every group keeps the range).  A step is 4 splats on 16 pixels where
// the warp form's is 2 splats on each of 4 quadrants: about 1.9 times the
// instructions per bucket, in a third of the time.  It pays where a launch
// would otherwise wait for its longest buckets (see launch_composite_warp).
constexpr int kTeamCap = 1024;    // ranks per window and per group of bitmap words
constexpr int kTeamWords = 4096;  // bitmap words: 128 groups of 32
template <bool LID>
struct TeamSmem {
    uint32_t keys[kTeamCap];
    uint32_t bm[kTeamWords];
    float4 raw[3][128];           // records of the next batch, in flight
    float4 st[3][128];            // camera: (u, v, log2 o, z), conic factor, (r, g, b, z); LiDAR: r0, r1, r2
    float4 sD[LID ? 128 : 1];
    int4 sR[128];                 // x0, x1 - x0, y0, y1 - y0
    uint32_t pre[129];
    uint32_t red[8];
    unsigned int claim;
};

template <int MODE>
__device__ __forceinline__ void team_item(const CompParams& P, TeamSmem<MODE == 1 || MODE == 3>& sm, const Where& w, int sub,
                                          int lx) {
    constexpr bool LID = MODE == 1 || MODE == 3;
    constexpr bool CNT = MODE != 0;
    constexpr int NT = 32 * kWarps;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grp = lane >> 3, l8 = lane & 7;
    const EnvInfo* Ep = P.envs + w.el;
    const int W = __ldg(&Ep->W), H = __ldg(&Ep->H), ntx = __ldg(&Ep->ntx);
    const unsigned long long pix_base = __ldg(&Ep->pix_base);
    const int tx = w.t % ntx, ty = w.t / ntx;
    const int sx0 = (tx * P.tile_w) + (sub & ((1 << lx) - 1)) * 8, sy0 = (ty * P.tile_h) + (sub >> lx) * 8;
    if (MODE != 3 && (sx0 >= W || sy0 >= H)) return;  // a subtile outside the image (uniform)
    Lane L;
    uint32_t submask = 1u << sub;
    int wx0 = sx0 + 4 * (warp & 1), wy0 = sy0 + 4 * (warp >> 1), wx1 = wx0 + 3, wy1 = wy0 + 3;  // the warp's pixels
    if constexpr (MODE == 3) {
        const uint32_t k0 = w.rchunk * (uint32_t)kRayChunk + (uint32_t)(16 * warp + l8);
        const uint32_t mine = __reduce_or_sync(kAll, lane_rays(P, w, tx, ty, k0, k0 + 8u, L));
        if (lane == 0) sm.red[warp] = mine;
        __syncthreads();
        submask = sm.red[0] | sm.red[1] | sm.red[2] | sm.red[3];
        const int big = 1 << 30;
        wx0 = __reduce_min_sync(kAll, min(L.in0 ? L.cx0 : big, L.in1 ? L.cx1 : big));
        wy0 = __reduce_min_sync(kAll, min(L.in0 ? L.cy0 : big, L.in1 ? L.cy1 : big));
        wx1 = __reduce_max_sync(kAll, max(L.in0 ? L.cx0 : -big, L.in1 ? L.cx1 : -big));
        wy1 = __reduce_max_sync(kAll, max(L.in0 ? L.cy0 : -big, L.in1 ? L.cy1 : -big));
    } else {
        lane_pixels<MODE, 2>(P, w.el, W, H, wx0 + (l8 & 3), wy0 + (l8 >> 2), L);
    }
    bool done0 = !L.in0, done1 = !L.in1;
    float2 Tp = make_float2(1.0f, 1.0f), acc = make_float2(0.0f, 0.0f);  // acc: channel grp (LiDAR: the range)
    uint32_t ncomp = 0;
    const Bucket bk = find_bucket(P, w, tid == 0);
    const int kshift = P.key_shift;
    const uint32_t any_sub = kshift == 0 ? 1u : 0u;
    bool finished = false;

    // The walk of one 32-splat chunk's quadrant mask.
    auto walk = [&](uint32_t q, int c) {
        while (q) {  // uniform
            const int n4 = min(4, __popc(q));
            int js[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                js[s] = s < n4 ? c + __ffs(q) - 1 : js[0];
                q &= q - 1u;  // stays 0
            }
            const int j = grp == 0 ? js[0] : grp == 1 ? js[1] : grp == 2 ? js[2] : js[3];
            const bool mine = grp < n4;
            float2 al, ts = make_float2(0.0f, 0.0f);
            bool h0 = mine && !done0, h1 = mine && !done1;
            if constexpr (LID) {
                const int4 R = sm.sR[j];
                h0 = h0 && in_box(R, L.cx0, L.cy0);
                h1 = h1 && in_box(R, L.cx1, L.cy1);
                ray_eval2(L, sm.st[0][j], sm.st[1][j], sm.st[2][j], sm.sD[j], al, ts);
            } else {
                al = splat_alpha2<true>(sm.st[0][j], sm.st[1][j], L.fpx, L.fpy);
            }
            const bool u0 = h0 && al.x >= (1.0f / 255.0f), u1 = h1 && al.y >= (1.0f / 255.0f);
            al = make_float2(u0 ? al.x : 0.0f, u1 ? al.y : 0.0f);
            if constexpr (LID) ts = make_float2(u0 ? ts.x : 0.0f, u1 ? ts.y : 0.0f);
            float2 a[4], x[4], T = Tp;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                a[s].x = __shfl_sync(kAll, al.x, 8 * s + l8);
                a[s].y = __shfl_sync(kAll, al.y, 8 * s + l8);
                x[s] = __fmul2_rn(a[s], T);
                T = __fadd2_rn(T, make_float2(-x[s].x, -x[s].y));
            }
            auto value = [&](int s) -> float2 {  // what splat s adds per unit of weight
                if constexpr (LID) {
                    return make_float2(__shfl_sync(kAll, ts.x, 8 * s + l8), __shfl_sync(kAll, ts.y, 8 * s + l8));
                } else {
                    const float v = reinterpret_cast<const float*>(&sm.st[2][js[s]])[grp];
                    return make_float2(v, v);
                }
            };
            const bool stop = T.x < 1e-4f || T.y < 1e-4f;  // the last transmittance is the smallest
            if (!__any_sync(kAll, stop)) {
#pragma unroll
                for (int s = 0; s < 4; ++s) acc = __ffma2_rn(x[s], value(s), acc);
                Tp = T;
                if constexpr (CNT)
                    if (grp == 0)
#pragma unroll
                        for (int s = 0; s < 4; ++s) ncomp += (uint32_t)(a[s].x > 0.0f) + (uint32_t)(a[s].y > 0.0f);
            } else {
#pragma unroll
                for (int s = 0; s < 4; ++s) {  // one splat at a time with the stop rule (blend2's arithmetic)
                    const bool v0 = !done0 && a[s].x > 0.0f, v1 = !done1 && a[s].y > 0.0f;
                    if constexpr (CNT)
                        if (grp == 0) ncomp += (uint32_t)v0 + (uint32_t)v1;
                    const float2 am = make_float2(v0 ? a[s].x : 0.0f, v1 ? a[s].y : 0.0f);
                    const float2 y = __fmul2_rn(am, Tp);
                    const float2 Tn = __fadd2_rn(Tp, make_float2(-y.x, -y.y));
                    const bool s0 = v0 && Tn.x < 1e-4f, s1 = v1 && Tn.y < 1e-4f;
                    done0 = done0 || s0;
                    done1 = done1 || s1;
                    acc = __ffma2_rn(make_float2(s0 ? 0.0f : y.x, s1 ? 0.0f : y.y), value(s), acc);
                    Tp = make_float2(s0 ? Tp.x : Tn.x, s1 ? Tp.y : Tn.y);
                }
            }
        }
    };

    // Composite the window keys[0, wn) (ranks in depth order).
    auto run_window = [&](uint32_t wn) {
        auto slot_of = [&](uint32_t i) -> uint32_t { return i < wn ? __ldg(bk.order + sm.keys[i]) : kAll; };
        auto fetch = [&](uint32_t g) {
            if (g < bk.n_local) {
                const float4* src = P.r0 + (size_t)kRecStride * (bk.recbase + g);
                copy16(&sm.raw[0][tid], src);
                copy16(&sm.raw[1][tid], src + 1);
                copy16(&sm.raw[2][tid], src + 2);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        uint32_t g = slot_of(tid), g_next = slot_of(NT + tid);
        fetch(g);
        for (uint32_t b = 0; b < wn; b += NT) {
            const int cnt_b = (int)min((uint32_t)NT, wn - b);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            int4 R = make_int4(1 << 20, -1, 1 << 20, -1);  // reaches nothing
            if (g < bk.n_local) {
                const float4 q0 = sm.raw[0][tid], q1 = sm.raw[1][tid], q2 = sm.raw[2][tid];
                const uint32_t rx = __float_as_uint(q1.w), ry = __float_as_uint(q2.w);
                int bx0 = (int)(rx & 0xffffu), bx1 = (int)(rx >> 16);
                const int by0 = (int)(ry & 0xffffu), by1 = (int)(ry >> 16);
                if constexpr (LID) {
                    unwrap_box(tx, bx0, bx1);
                    sm.st[0][tid] = q0;
                    sm.st[2][tid] = q2;
                    sm.sD[tid] = third_row(q1, q2, __uint_as_float(__ldg(&P.r3[bk.recbase + g].w)));
                } else {
                    sm.st[0][tid] = q0;
                    sm.st[2][tid] = make_float4(q2.x, q2.y, q2.z, q0.w);
                }
                sm.st[1][tid] = q1;
                R = make_int4(bx0, bx1 - bx0, by0, by1 - by0);
            }
            sm.sR[tid] = R;
            g = g_next;
            if (b + NT < wn) {
                fetch(g);
                g_next = slot_of(b + 2 * NT + tid);
            }
            __syncthreads();
            if (!__all_sync(kAll, done0 && done1))
                for (int c = 0; c < cnt_b; c += 32) {
                    const int4 B = sm.sR[c + lane];
                    const bool ov = B.x <= wx1 && B.x + B.y >= wx0 && B.z <= wy1 && B.z + B.w >= wy0;
                    walk(__ballot_sync(kAll, ov && c + lane < cnt_b), c);
                    if (__all_sync(kAll, done0 && done1)) break;
                }
            finished = __syncthreads_and(done0 && done1) != 0;
            if (finished) {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                break;
            }
        }
    };

    for (uint32_t r0 = 0; r0 < bk.n_rank && bk.n > 0 && !finished; r0 += (uint32_t)(kTeamWords * 32)) {
        for (int i = tid; i < kTeamWords / 4; i += NT) reinterpret_cast<uint4*>(sm.bm)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        const uint32_t k0 = r0 << kshift;
        const unsigned long long span = (unsigned long long)min((uint32_t)(kTeamWords * 32), bk.n_rank - r0) << kshift;
        auto set = [&](uint32_t k, bool valid) {
            const uint32_t d = k - k0;
            if (valid && d < span && ((k & submask) | any_sub) != 0u)
                atomicOr(&sm.bm[d >> (5 + kshift)], 1u << ((d >> kshift) & 31u));
        };
        {  // 16-byte loads, four in flight per thread
            constexpr int U = 4;
            const uint32_t off = (uint32_t)((uintptr_t)bk.keys & 15u) >> 2, end = off + bk.n;
            const uint4* V = reinterpret_cast<const uint4*>(bk.keys - off);
            for (uint32_t i = 4 * tid; i < end; i += 4 * NT * U) {
                uint4 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    v[u] = i + 4 * NT * u < end ? __ldg(V + ((i + 4 * NT * u) >> 2)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t y = i + 4 * NT * u - off;  // index in the bucket; wraps below it
                    set(v[u].x, y < bk.n);
                    set(v[u].y, y + 1 < bk.n);
                    set(v[u].z, y + 2 < bk.n);
                    set(v[u].w, y + 3 < bk.n);
                }
            }
        }
        __syncthreads();
        uint32_t c = 0;  // thread t counts group t
#pragma unroll 8
        for (int i = 0; i < 32; ++i) c += __popc(sm.bm[32 * tid + ((i + lane) & 31)]);
        uint32_t total;
        sm.pre[tid] = block_excl_scan_total<NT>(c, sm.red, total);
        if (tid == 0) sm.pre[128] = total;
        __syncthreads();
        for (int g0 = 0; g0 < 128 && !finished;) {
            const uint32_t base = sm.pre[g0];
            int lo = g0 + 1, hi = 128;  // last g1 with pre[g1] - base <= kTeamCap
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (sm.pre[mid] - base <= (uint32_t)kTeamCap) lo = mid; else hi = mid - 1;
            }
            const uint32_t wn = sm.pre[lo] - base;
            if (wn > 0) {
                for (int g = g0 + warp; g < lo; g += kWarps) {  // a warp reads a group's words back in order
                    uint32_t m = sm.bm[32 * g + lane];
                    const uint32_t pc = __popc(m);
                    uint32_t x = pc;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const uint32_t y = __shfl_up_sync(kAll, x, d);
                        if (lane >= d) x += y;
                    }
                    uint32_t at = sm.pre[g] - base + x - pc;
                    const uint32_t r = r0 + (uint32_t)(32 * g + lane) * 32u;
                    while (m) {
                        sm.keys[at++] = r + (uint32_t)(__ffs(m) - 1);
                        m &= m - 1u;
                    }
                }
                __syncthreads();
                run_window(wn);
            }
            g0 = lo;
        }
        __syncthreads();
    }

    if constexpr (CNT)
        if (P.neval) {
            const uint32_t c = __reduce_add_sync(kAll, ncomp);
            if (lane == 0 && c) atomicAdd(P.neval, (unsigned long long)c);
        }
    if constexpr (LID) {
        if (lane < 8) {
            const size_t o0 = pix_base + (MODE == 3 ? (size_t)L.ray0 : (size_t)L.cy0 * W + L.cx0);
            const size_t o1 = pix_base + (MODE == 3 ? (size_t)L.ray1 : (size_t)L.cy1 * W + L.cx1);
            const float a0 = 1.0f - Tp.x, a1 = 1.0f - Tp.y;
            if (L.in0) {
                P.depth[o0] = a0 > 0.0f ? acc.x / a0 : 0.0f;
                if (P.alpha) P.alpha[o0] = a0;
            }
            if (L.in1) {
                P.depth[o1] = a1 > 0.0f ? acc.y / a1 : 0.0f;
                if (P.alpha) P.alpha[o1] = a1;
            }
        }
    } else {
        float2 ch[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            ch[s].x = __shfl_sync(kAll, acc.x, 8 * s + l8);
            ch[s].y = __shfl_sync(kAll, acc.y, 8 * s + l8);
        }
        if (lane < 8) {
            const PixelStore store(P, w.el);
            if (L.in0) store.put(P, pix_base + (size_t)L.cy0 * W + L.cx0, Tp.x, ch[0].x, ch[1].x, ch[2].x, ch[3].x);
            if (L.in1) store.put(P, pix_base + (size_t)L.cy1 * W + L.cx1, Tp.y, ch[0].y, ch[1].y, ch[2].y, ch[3].y);
        }
    }
}

}  // namespace

// MODE 0: camera image or observation; 2: the same, also counting composited
// (pixel, splat) pairs into P.neval; 1: LiDAR scan on a grid (records of
// k_project_lidar; a "pixel" is a ray, the Gaussian evaluated at its closest
// approach); 3: LiDAR along arbitrary rays (an item is a chunk of at most 64
// rays of a 16x16 grid tile, grouped by 8x8 subtile; the culling box is that
// of the rays' cells).
//
// Lanes work in groups, a lane on two pixels: a group of four owns 2x4 pixels of
// the subtile (LiDAR grids: a group of two, 2x2 rays) and walks only the splats
// whose box reaches them, so the groups advance through different splats at
// once; a chunk of 32 splats takes as many steps as its fullest group.  At
// 128x128 a splat blends 5.6 of a subtile's 64 pixels: 443 steps of two splats
// for the whole subtile, 303 with 4x4 groups, 256 with 2x4, 241 with 2x2; a
// shared-memory load is split by quarter-warps, so two addresses in each cost
// nothing.  Compositing 512 views of 128x128 takes 6.37 ms with 4x4 groups,
// 6.33 with 4x2, 6.19 with 2x4 and 6.45 with 2x2 (more ballots per chunk, bank
// conflicts); 32 scans of 64 x 1024 rays 2.35, 2.13, 2.19 and 2.05.  (MODE 3:
// all lanes walk the same splats; groups with boxes of their own were slower on
// 128 envs, 8.1 instead of 7.5 ms, as the per-ray boxes cull whole steps).
template <int MODE>
__global__ void __launch_bounds__(32 * kWarps, MODE == 1 || MODE == 3 ? 5 : 6) k_composite_warp(CompParams P) {
    constexpr bool LID = MODE == 1 || MODE == 3;
    constexpr bool GROUPS = MODE != 3;
    constexpr int GPX = 2, GPY = LID ? 2 : 4, GL = GPX * GPY / 2;  // a group's pixels and lanes
    constexpr bool CNT = MODE != 0;
    constexpr int CAP = LID ? 512 : 256;   // ranks per window, and per group of bitmap words
    constexpr int GW = CAP / 32;           // words per group
    constexpr int NG = kWords / GW;        // groups
    struct Smem {                          // a warp's own
        uint32_t keys[CAP];                // the window's ranks
        uint32_t bm[kWords];               // bitmap | sort counters, then range starts
        float4 rec[2][3][32];              // records of this and the next 32 splats: r0, r1, r2; between windows sort scratch
        float4 sD[LID ? 32 : 1];           // LiDAR: third row of G
        int4 sR[LID ? 32 : 1];             // LiDAR: x0, x1 - x0, y0, y1 - y0
        uint32_t pre[NG + 1];              // ranks set before each group of the bitmap
    };
    static_assert(sizeof(Smem::rec) >= CAP * 4, "the sort scratch shares the records' memory");
    constexpr size_t BYTES = sizeof(Smem) * kWarps > sizeof(TeamSmem<LID>) ? sizeof(Smem) * kWarps : sizeof(TeamSmem<LID>);
    __shared__ __align__(16) unsigned char smem[BYTES];
    Smem& sm = reinterpret_cast<Smem*>(smem)[threadIdx.x >> 5];
    uint32_t* const keys = sm.keys;
    uint32_t* const bm = sm.bm;
    uint32_t* const pre = sm.pre;
    auto& rec = sm.rec;
    auto& sD = sm.sD;
    auto& sR = sm.sR;
    const int lane = threadIdx.x & 31;
    const int lx = __ffs(P.tile_w) - 4, ly = __ffs(P.tile_h) - 4;  // log2 of the tile's subtile columns, rows
    const int lsub = MODE == 3 ? 0 : lx + ly;
    const int grp = lane / GL, lg = lane % GL;
    Where w;
    w.el = P.e_begin;
    w.e_lo = __ldg(&P.envs[w.el].tile_base);
    w.e_hi = w.e_lo + (unsigned)__ldg(&P.envs[w.el].T);
    const unsigned int t_env = w.e_hi - w.e_lo;  // tiles of the first env
    const unsigned int end = (P.item_end - P.item_begin) << lsub;
    uint32_t cb[kItemClasses] = {0};  // items before each class of the claiming order
    if (P.items)
        for (int c = 1; c < kItemClasses; ++c) cb[c] = cb[c - 1] + __ldg(P.class_cnt + c - 1);
    auto item_at = [&](unsigned int it) -> unsigned int {
        const unsigned int q = it >> lsub;
        if (!P.items) return P.item_begin + q;
        const int c = q >= cb[3] ? 3 : q >= cb[2] ? 2 : q >= cb[1] ? 1 : 0;
        const uint32_t before = q >= cb[3] ? cb[3] : q >= cb[2] ? cb[2] : q >= cb[1] ? cb[1] : 0u;
        return __ldg(P.items + (size_t)c * P.item_pitch + (q - before));
    };
    // the long classes first, a CTA per item
    unsigned int n_team = 0;
    if (P.team_classes) {
        n_team = P.team_classes >= kItemClasses ? end : cb[P.team_classes] << lsub;
        TeamSmem<LID>& tm = *reinterpret_cast<TeamSmem<LID>*>(smem);
        for (;;) {
            if (threadIdx.x == 0) tm.claim = atomicAdd(P.team_work, 1u);
            __syncthreads();
            const unsigned int it = tm.claim;
            if (it >= n_team) break;
            locate<MODE>(P, item_at(it), t_env, w);
            team_item<MODE>(P, tm, w, (int)(it & ((1u << lsub) - 1u)), lx);
            __syncthreads();
        }
        __syncthreads();  // the warps' own memory from here on
    }
    unsigned int claim = 0;
    if (lane == 0) claim = n_team + atomicAdd(P.work, (unsigned)P.chunk);
    for (;;) {
    const unsigned int first = __shfl_sync(kAll, claim, 0);
    if (first >= end) break;
    if (lane == 0) claim = n_team + atomicAdd(P.work, (unsigned)P.chunk);  // the next claim, in flight meanwhile
    const unsigned int last = min(first + (unsigned)P.chunk, end);
    for (unsigned int it = first; it < last; ++it) {
    const int sub = (int)(it & ((1u << lsub) - 1u));
    locate<MODE>(P, item_at(it), t_env, w);
    const EnvInfo* Ep = P.envs + w.el;
    const int W = __ldg(&Ep->W), H = __ldg(&Ep->H), ntx = __ldg(&Ep->ntx);
    const unsigned long long pix_base = __ldg(&Ep->pix_base);
    const int tx = w.t % ntx, ty = w.t / ntx;
    int wx0 = (tx * P.tile_w) + (sub & ((1 << lx) - 1)) * 8, wy0 = (ty * P.tile_h) + (sub >> lx) * 8;
    if (MODE != 3 && (wx0 >= W || wy0 >= H)) continue;  // a subtile outside the image
    int wx1 = wx0 + 7, wy1 = wy0 + 7;
    Lane L;
    uint32_t submask = 1u << sub;  // subtile bits of the keys this warp takes
    if constexpr (MODE == 3) {
        const uint32_t k0 = w.rchunk * (uint32_t)kRayChunk + (uint32_t)lane;
        submask = __reduce_or_sync(kAll, lane_rays(P, w, tx, ty, k0, k0 + 32u, L));
        // the warp's culling box: the cells of its rays
        const int big = 1 << 30;
        wx0 = __reduce_min_sync(kAll, min(L.in0 ? L.cx0 : big, L.in1 ? L.cx1 : big));
        wy0 = __reduce_min_sync(kAll, min(L.in0 ? L.cy0 : big, L.in1 ? L.cy1 : big));
        wx1 = __reduce_max_sync(kAll, max(L.in0 ? L.cx0 : -big, L.in1 ? L.cx1 : -big));
        wy1 = __reduce_max_sync(kAll, max(L.in0 ? L.cy0 : -big, L.in1 ? L.cy1 : -big));
    } else {
        const int gx0 = wx0 + GPX * (grp % (8 / GPX)), gy0 = wy0 + GPY * (grp / (8 / GPX));
        lane_pixels<MODE, GPY / 2>(P, w.el, W, H, gx0 + lg % GPX, gy0 + lg / GPX, L);
    }
    bool done0 = !L.in0, done1 = !L.in1;
    // the lane's two pixels: .x = (px, py0), .y = (px, py1)
    float2 Tp = make_float2(1.0f, 1.0f), rp = make_float2(0.0f, 0.0f), gp = rp, bp = rp, dp = rp;
    uint32_t ncomp = 0;
    const Bucket bk = find_bucket(P, w, lane == 0);
    const int kshift = P.key_shift;
    // the rank of a key and whether this warp's pixels lie in its subtiles
    const uint32_t any_sub = kshift == 0 ? 1u : 0u;
    auto taken = [&](uint32_t k) { return ((k & submask) | any_sub) != 0u; };

    // Composite the ordered ranks keys[0, m).  True once every pixel of the warp
    // has terminated.
    auto run_window = [&](int m) -> bool {
        auto slot_of = [&](int i) -> uint32_t { return i < m ? __ldg(bk.order + keys[i]) : kAll; };
        auto fetch = [&](int buf, uint32_t s) {
            if (s < bk.n_local) {
                const float4* src = P.r0 + (size_t)kRecStride * (bk.recbase + s);
                copy16(&rec[buf][0][lane], src);
                copy16(&rec[buf][1][lane], src + 1);
                copy16(&rec[buf][2][lane], src + 2);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        uint32_t cur = slot_of(lane), nxt = slot_of(32 + lane);
        fetch(0, cur);
        for (int c = 0; c < m; c += 32) {
            const int b = (c >> 5) & 1;
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            const bool own = cur < bk.n_local;  // a splat of this chunk (every rank of a sound bucket has a slot)
            const uint32_t slot = cur;
            cur = nxt;
            if (c + 32 < m) fetch(b ^ 1, cur);
            nxt = slot_of(c + 64 + lane);
            float4* sA = rec[b][0];
            float4* sB = rec[b][1];
            float4* sC = rec[b][2];
            bool ov = false;
            int bx0 = 0, bx1 = -1, by0 = 0, by1 = -1;
            if (own) {
                const float4 q1 = sB[lane];
                const uint32_t rx = __float_as_uint(q1.w), ry = __float_as_uint(sC[lane].w);
                bx0 = (int)(rx & 0xffffu);
                bx1 = (int)(rx >> 16);
                by0 = (int)(ry & 0xffffu);
                by1 = (int)(ry >> 16);
                if constexpr (LID) {
                    sD[lane] = third_row(q1, sC[lane], __uint_as_float(__ldg(&P.r3[bk.recbase + slot].w)));
                    unwrap_box(tx, bx0, bx1);
                    sR[lane] = make_int4(bx0, bx1 - bx0, by0, by1 - by0);
                }
                ov = bx0 <= wx1 && bx1 >= wx0 && by0 <= wy1 && by1 >= wy0;
            }
            if constexpr (!LID) {
                // large splats: the exact ellipse (a box under 24 px in width + height
                // is kept as it is: it overstates the ellipse least)
                const bool big = ov && bx1 - bx0 + by1 - by0 >= 24;
                if (__any_sync(kAll, big)) {
                    if (big) {
                        const float4 A = sA[lane];
                        float4 B = sB[lane];
                        B.w = A.z + 7.9943534f;  // log2(255 o): alpha >= 1/255 iff q <= w
                        ov = reaches_rect(A, B, (float)wx0 + 0.5f, (float)wy0 + 0.5f);
                    }
                }
            }
            uint32_t m32;
            if constexpr (GROUPS) {  // per group: the splats whose box reaches it
                bool cx[8 / GPX], cy[8 / GPY];
#pragma unroll
                for (int i = 0; i < 8 / GPX; ++i)
                    cx[i] = ov && bx0 <= wx0 + GPX * i + GPX - 1 && bx1 >= wx0 + GPX * i;
#pragma unroll
                for (int i = 0; i < 8 / GPY; ++i) cy[i] = by0 <= wy0 + GPY * i + GPY - 1 && by1 >= wy0 + GPY * i;
                m32 = 0u;
#pragma unroll
                for (int g = 0; g < 32 / GL; ++g) {
                    const uint32_t b = __ballot_sync(kAll, cx[g % (8 / GPX)] && cy[g / (8 / GPX)]);
                    if (grp == g) m32 = b;
                }
                const uint32_t dm = __ballot_sync(kAll, done0 && done1);
                if ((~dm >> (GL * grp) & ((1u << GL) - 1u)) == 0u) m32 = 0u;
            } else {
                m32 = __ballot_sync(kAll, ov);
            }
            __syncwarp();  // the lanes' staged values
            // two splats per step: their four alpha evaluations are independent;
            // the blends then run in depth order
            while (GROUPS ? __any_sync(kAll, m32 != 0u) : m32 != 0u) {
                const bool one = !GROUPS || m32 != 0u;
                const int j1 = one ? __ffs(m32) - 1 : 0;
                m32 &= m32 - 1u;
                const bool two = m32 != 0u;
                const int j2 = two ? __ffs(m32) - 1 : j1;
                if (two) m32 &= m32 - 1u;
                // Camera pixels need no box test (a pixel outside a splat's support box
                // has q > q* (1 + 2e-4): its alpha falls below 1/255); LiDAR rays have
                // one (their grid box is a looser cone bound and a ray evaluation costs
                // more).
                bool h10 = one && !done0, h11 = one && !done1, h20 = two && !done0, h21 = two && !done1;
                if constexpr (LID) {
                    const int4 R1 = sR[j1];
                    const int4 R2 = sR[j2];
                    h10 = h10 && in_box(R1, L.cx0, L.cy0);
                    h11 = h11 && in_box(R1, L.cx1, L.cy1);
                    h20 = h20 && in_box(R2, L.cx0, L.cy0);
                    h21 = h21 && in_box(R2, L.cx1, L.cy1);
                    // Grid scans evaluate every lane's rays (no divergent branch, so the
                    // vote below sees every lane); along arbitrary rays the per-ray boxes
                    // cull so much that the branch pays.
                    if (MODE == 1 || h10 || h11 || h20 || h21) {
                        float2 al1, ts1, al2, ts2;
                        ray_eval2(L, sA[j1], sB[j1], sC[j1], sD[j1], al1, ts1);
                        ray_eval2(L, sA[j2], sB[j2], sC[j2], sD[j2], al2, ts2);
                        const bool u10 = h10 && al1.x >= (1.0f / 255.0f), u11 = h11 && al1.y >= (1.0f / 255.0f);
                        const bool v20 = h20 && al2.x >= (1.0f / 255.0f), v21 = h21 && al2.y >= (1.0f / 255.0f);
                        bool voted = false;
                        if constexpr (MODE == 1) {
                            // as in the camera form: both splats with selects unless a ray stops
                            const float2 am1 = make_float2(u10 ? al1.x : 0.0f, u11 ? al1.y : 0.0f);
                            const float2 x1 = __fmul2_rn(am1, Tp);
                            const float2 Tn1 = __fadd2_rn(Tp, make_float2(-x1.x, -x1.y));
                            const float2 am2 = make_float2(v20 ? al2.x : 0.0f, v21 ? al2.y : 0.0f);
                            const float2 x2 = __fmul2_rn(am2, Tn1);
                            const float2 Tn2 = __fadd2_rn(Tn1, make_float2(-x2.x, -x2.y));
                            const bool stop = Tn2.x < 1e-4f || Tn2.y < 1e-4f;  // Tn2 <= Tn1
                            if (!__any_sync(kAll, stop)) {
                                ncomp += (uint32_t)u10 + (uint32_t)u11 + (uint32_t)v20 + (uint32_t)v21;
                                dp = __ffma2_rn(x1, ts1, dp);
                                dp = __ffma2_rn(x2, ts2, dp);
                                Tp = Tn2;
                                voted = true;
                            }
                        }
                        if (!voted) {
                            const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (u10) {
                                ++ncomp;
                                blend(al1.x, none, ts1.x, Tp.x, rp.x, gp.x, bp.x, dp.x, done0);
                            }
                            if (u11) {
                                ++ncomp;
                                blend(al1.y, none, ts1.y, Tp.y, rp.y, gp.y, bp.y, dp.y, done1);
                            }
                            if (v20 && !done0) {
                                ++ncomp;
                                blend(al2.x, none, ts2.x, Tp.x, rp.x, gp.x, bp.x, dp.x, done0);
                            }
                            if (v21 && !done1) {
                                ++ncomp;
                                blend(al2.y, none, ts2.y, Tp.y, rp.y, gp.y, bp.y, dp.y, done1);
                            }
                        }
                    }
                } else {
                    // the arithmetic and the vote of the CTA form (gs_composite.cu)
                    const float4 A1 = sA[j1], B1 = sB[j1];
                    const float4 A2 = sA[j2], B2 = sB[j2];
                    const float2 a1 = splat_alpha2<true>(A1, B1, L.fpx, L.fpy);
                    const float2 a2 = splat_alpha2<true>(A2, B2, L.fpx, L.fpy);
                    const bool u10 = h10 && a1.x >= (1.0f / 255.0f);
                    const bool u11 = h11 && a1.y >= (1.0f / 255.0f);
                    const float2 am1 = make_float2(u10 ? a1.x : 0.0f, u11 ? a1.y : 0.0f);
                    const float2 x1 = __fmul2_rn(am1, Tp);
                    const float2 Tn1 = __fadd2_rn(Tp, make_float2(-x1.x, -x1.y));
                    const bool v20 = h20 && a2.x >= (1.0f / 255.0f);
                    const bool v21 = h21 && a2.y >= (1.0f / 255.0f);
                    const float2 am2 = make_float2(v20 ? a2.x : 0.0f, v21 ? a2.y : 0.0f);
                    const float2 x2 = __fmul2_rn(am2, Tn1);
                    const float2 Tn2 = __fadd2_rn(Tn1, make_float2(-x2.x, -x2.y));
                    const bool stop = Tn2.x < 1e-4f || Tn2.y < 1e-4f;
                    if (!__any_sync(kAll, stop)) {
                        if constexpr (CNT) ncomp += (uint32_t)u10 + (uint32_t)u11 + (uint32_t)v20 + (uint32_t)v21;
                        const float4 C1 = sC[j1], C2 = sC[j2];
                        rp = __ffma2_rn(x1, make_float2(C1.x, C1.x), rp);
                        gp = __ffma2_rn(x1, make_float2(C1.y, C1.y), gp);
                        bp = __ffma2_rn(x1, make_float2(C1.z, C1.z), bp);
                        dp = __ffma2_rn(x1, make_float2(A1.w, A1.w), dp);
                        rp = __ffma2_rn(x2, make_float2(C2.x, C2.x), rp);
                        gp = __ffma2_rn(x2, make_float2(C2.y, C2.y), gp);
                        bp = __ffma2_rn(x2, make_float2(C2.z, C2.z), bp);
                        dp = __ffma2_rn(x2, make_float2(A2.w, A2.w), dp);
                        Tp = Tn2;
                    } else {
                        if constexpr (CNT) ncomp += (uint32_t)u10 + (uint32_t)u11;
                        blend2(a1, u10, u11, sC[j1], A1.w, Tp, rp, gp, bp, dp, done0, done1);
                        const bool u20 = h20 && !done0 && a2.x >= (1.0f / 255.0f);
                        const bool u21 = h21 && !done1 && a2.y >= (1.0f / 255.0f);
                        if constexpr (CNT) ncomp += (uint32_t)u20 + (uint32_t)u21;
                        blend2(a2, u20, u21, sC[j2], A2.w, Tp, rp, gp, bp, dp, done0, done1);
                    }
                }
            }
            if (__all_sync(kAll, done0 && done1)) {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                __syncwarp();
                return true;
            }
        }
        return false;
    };

    // Appends the taken ranks in [lo, hi) of the bucket to keys (the first
    // CAP of them) and returns how many there are; wl, wh: their bounds.
    uint32_t wl = 0, wh = 0;
    auto gather = [&](uint32_t lo, uint32_t width) -> uint32_t {
        uint32_t have = 0, a = kAll, z = 0u;
        const uint32_t below = (1u << lane) - 1u;
        warp_keys(bk.keys, bk.n, [&](uint32_t k, bool valid) {
            const uint32_t r = k >> kshift;
            const bool in = valid && taken(k) && r - lo < width;
            const uint32_t b = __ballot_sync(kAll, in);
            if (in) {
                const uint32_t at = have + (uint32_t)__popc(b & below);
                if (at < (uint32_t)CAP) keys[at] = r;
                a = min(a, r);
                z = max(z, r);
            }
            have += (uint32_t)__popc(b);
        });
        wl = __reduce_min_sync(kAll, a);
        wh = __reduce_max_sync(kAll, z);
        __syncwarp();
        return have;
    };

    // how the windows come: the bucket at once, runs of histogram ranges, or bitmaps
    enum { kWhole, kRuns, kBitmap } how = kBitmap;
    uint32_t whole = 0;
    int hs = 0;            // histogram: log2 of the ranks per range
    uint32_t htotal = 0;
    int g0 = 0;            // next range or group
    uint32_t r0 = 0;       // next ranks of the bitmap
    bool loaded = false;   // a bitmap is set up
    if (bk.n <= kShort) {
        whole = bk.n ? gather(0u, bk.n_rank) : 0u;
        if (whole <= (uint32_t)CAP) how = kWhole;
    }
    if (how == kBitmap) {
        const uint32_t est = kshift ? bk.n / 2 : bk.n;
        if (est / CAP + 2 < bk.n_rank / (kWords * 32) + 1) {
            while (((bk.n_rank - 1u) >> hs) >= (uint32_t)kSortBins) ++hs;
            for (int i = lane; i < kSortBins; i += 32) bm[i] = 0u;
            __syncwarp();
            warp_keys(bk.keys, bk.n, [&](uint32_t k, bool valid) {
                const uint32_t r = k >> kshift;
                if (valid && taken(k) && r < bk.n_rank) atomicAdd(&bm[r >> hs], 1u);
            });
            __syncwarp();
            constexpr int PER = kSortBins / 32;
            uint32_t c[PER], sum = 0, most = 0;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                c[j] = bm[lane * PER + j];
                sum += c[j];
                most = max(most, c[j]);
            }
            uint32_t run = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(kAll, run, d);
                if (lane >= d) run += y;
            }
            htotal = __shfl_sync(kAll, run, 31);
            run -= sum;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                bm[kSortBins + lane * PER + j] = run;
                run += c[j];
            }
            __syncwarp();
            if (!__any_sync(kAll, most > (uint32_t)CAP)) how = kRuns;
        }
    }
    for (;;) {
        int wn = 0;
        if (how == kWhole) {
            wn = (int)whole;
            whole = 0;
            if (wn == 0) break;
        } else if (how == kRuns) {
            if (g0 >= kSortBins) break;
            const uint32_t* start_of = bm + kSortBins;
            auto begin = [&](int g) { return g < kSortBins ? start_of[g] : htotal; };
            const uint32_t base = begin(g0);
            if (base >= htotal) break;
            int lo = g0 + 1, hi = kSortBins;  // last g1 with begin(g1) - base <= CAP
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (begin(mid) - base <= (uint32_t)CAP) lo = mid; else hi = mid - 1;
            }
            wn = (int)(begin(lo) - base);
            const uint32_t a = (uint32_t)g0 << hs;
            g0 = lo;
            if (wn == 0) continue;
            gather(a, min((uint32_t)lo << hs, bk.n_rank) - a);
        } else {
            if (loaded && g0 >= NG) {
                loaded = false;
                r0 += (uint32_t)(kWords * 32);
            }
            if (!loaded) {
                if (r0 >= bk.n_rank || bk.n == 0) break;
                for (int i = lane; i < kWords / 4; i += 32)
                    reinterpret_cast<uint4*>(bm)[i] = make_uint4(0u, 0u, 0u, 0u);
                __syncwarp();
                const uint32_t k0 = r0 << kshift, span = min((uint32_t)(kWords * 32), bk.n_rank - r0) << kshift;
                warp_keys(bk.keys, bk.n, [&](uint32_t k, bool valid) {
                    const uint32_t d = k - k0;
                    if (valid && d < span && taken(k)) atomicOr(&bm[d >> (5 + kshift)], 1u << ((d >> kshift) & 31u));
                });
                __syncwarp();
                // ranks set before each group: a lane counts GPL groups
                constexpr int GPL = NG / 32;
                uint32_t c[GPL], run = 0;
#pragma unroll
                for (int k = 0; k < GPL; ++k) {
                    c[k] = 0u;
#pragma unroll
                    for (int i = 0; i < GW; ++i)  // rotated: neighbouring lanes hit different banks
                        c[k] += __popc(bm[(GPL * lane + k) * GW + ((i + lane) & (GW - 1))]);
                    run += c[k];
                }
                const uint32_t mine = run;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(kAll, run, d);
                    if (lane >= d) run += y;
                }
                if (lane == 31) pre[NG] = run;
                run -= mine;
#pragma unroll
                for (int k = 0; k < GPL; ++k) {
                    pre[GPL * lane + k] = run;
                    run += c[k];
                }
                __syncwarp();
                loaded = true;
                g0 = 0;
            }
            const uint32_t base = pre[g0];
            const uint32_t fit = base + (uint32_t)CAP;
            // groups whose end is within CAP of the window's start (ends ascend)
            int g1 = 0;
#pragma unroll
            for (int k = 0; k < NG / 32; ++k) g1 += __popc(__ballot_sync(kAll, pre[32 * k + lane + 1] <= fit));
            wn = (int)(pre[g1] - base);
            if (wn > 0) {
                // GW lanes read a group's words back in order
                const int word = lane & (GW - 1);
                for (int gb = g0; gb < g1; gb += 32 / GW) {
                    const int g = gb + lane / GW;
                    uint32_t w = g < g1 ? bm[g * GW + word] : 0u;
                    const uint32_t pc = __popc(w);
                    uint32_t x = pc;
#pragma unroll
                    for (int d = 1; d < GW; d <<= 1) {
                        const uint32_t y = __shfl_up_sync(kAll, x, d, GW);
                        if (word >= d) x += y;
                    }
                    if (w) {
                        uint32_t at = pre[g] - base + x - pc;
                        const uint32_t r = r0 + (uint32_t)(g * GW + word) * 32u;
                        while (w) {
                            keys[at++] = r + (uint32_t)(__ffs(w) - 1);
                            w &= w - 1u;
                        }
                    }
                }
                __syncwarp();
            }
            g0 = g1;
            if (wn == 0) continue;
        }
        if (how != kBitmap) warp_sort(keys, reinterpret_cast<uint32_t*>(&rec[0][0][0]), bm, wn, wl, wh);
        if (run_window(wn)) break;
        __syncwarp();
    }

    if (CNT && P.neval) {
        const uint32_t c = __reduce_add_sync(kAll, ncomp);
        if (lane == 0 && c) atomicAdd(P.neval, (unsigned long long)c);
    }
    if constexpr (LID) {  // range and hit per ray, at the ray's index or grid cell
        const size_t o0 = pix_base + (MODE == 3 ? (size_t)L.ray0 : (size_t)L.cy0 * W + L.cx0);
        const size_t o1 = pix_base + (MODE == 3 ? (size_t)L.ray1 : (size_t)L.cy1 * W + L.cx1);
        if (L.in0) {
            const float a = 1.0f - Tp.x;
            P.depth[o0] = a > 0.0f ? dp.x / a : 0.0f;
            if (P.alpha) P.alpha[o0] = a;
        }
        if (L.in1) {
            const float a = 1.0f - Tp.y;
            P.depth[o1] = a > 0.0f ? dp.y / a : 0.0f;
            if (P.alpha) P.alpha[o1] = a;
        }
    } else {
        const PixelStore store(P, w.el);
        if (L.in0) store.put(P, pix_base + (size_t)L.cy0 * W + L.cx0, Tp.x, rp.x, gp.x, bp.x, dp.x);
        if (L.in1) store.put(P, pix_base + (size_t)L.cy1 * W + L.cx1, Tp.y, rp.y, gp.y, bp.y, dp.y);
    }
    __syncwarp();
    }  // items of the claim
    }  // claims
}

template <int MODE>
static cudaError_t launch_warps(const CompParams& P, cudaStream_t st, int* ctas) {
    static PerDevice resident;
    int full = 0;
    const cudaError_t e = resident.ctas((const void*)k_composite_warp<MODE>, 32 * kWarps, &full);
    if (e != cudaSuccess) return e;
    const int subs = MODE == 3 ? 1 : (P.tile_w / 8) * (P.tile_h / 8);
    const unsigned long long items = (unsigned long long)(P.item_end - P.item_begin) * subs;
    if (items > 0xffffffffull) return cudaErrorInvalidValue;
    const unsigned long long claims = (items + P.chunk - 1) / P.chunk;
    CompParams Q = P;
    // Teams of four warps for the classes of long buckets, the fewer items there
    // are per resident warp to hide a long one behind.  Measured (us, teams for
    // the first 0 / 1 / 2 / 3 classes): 16 envs at 128x128 (1.1 items per warp)
    // 1615 / 855 / 800 / 804, 48 (3.4) 1987 / 1462 / 1153 / 1145, 128 (9) 2488 /
    // 2282 / 2369 / 2583, 256 (18) 3922 / 3842 / 4461 / 5229, 512 (36) 6249 /
    // 7251 / 8503 / -; spinning LiDAR 1 env (0.3) 1011 / 1008 / 517 / 486, 32
    // (11) 3984 / 3682 / 2853 / 3863, 128 (43) 8291 / 8697 / - / -.  Where items
    // are few per resident CTA, all go to teams (whole calls, us): one 128x96 view
    // of 16,384 splats (0.2 items per CTA) 57 -> 39, 8 of them (1.7) 145 -> 122,
    // 16 (3.4) 195 -> 173, but 2 views of 333x251 in the room (2.9) 351 -> 362 and
    // 4 rosettes (1.7) 1403 -> 1465.  Even scenes have no long buckets to wait for: whole
    // calls with teams for three classes / without (us), 64 views of 128x96 of an even
    // cube of 120,000 (3.4 items per warp) 1145 / 912, 24 of them (1.3) 508 / 484, 200 of
    // 64x48 (2.6) 2057 / 1803.
    constexpr bool LID = MODE == 1 || MODE == 3;
    Q.team_classes = 0;
    if (P.items && P.team_work) {
        const double per_warp = (double)items / ((double)kWarps * full);
        if (items * 2 <= (LID ? 2ull : 5ull) * full) Q.team_classes = kItemClasses;
        else if (P.even && per_warp > 1.0) Q.team_classes = 0;
        else if (per_warp <= 6.0) Q.team_classes = 3;
        else if (MODE == 1 || MODE == 3) Q.team_classes = per_warp <= 12.0 ? 2 : 0;
        else if (per_warp <= 20.0) Q.team_classes = 1;
    }
    // few claims: fewer warps per CTA, so that they spread over the SMs
    const int warps = Q.team_classes ? kWarps : (int)std::min((claims + full - 1) / full, (unsigned long long)kWarps);
    *ctas = (int)std::min((unsigned long long)full, Q.team_classes ? claims : (claims + warps - 1) / warps);
    k_composite_warp<MODE><<<*ctas, 32 * warps, 0, st>>>(Q);
    return cudaGetLastError();
}

cudaError_t launch_composite_warp(const CompParams& P, cudaStream_t st, int* ctas) {
    if (P.ray_list) return launch_warps<3>(P, st, ctas);
    if (P.lidars) return launch_warps<1>(P, st, ctas);
    if (P.neval) return launch_warps<2>(P, st, ctas);
    return launch_warps<0>(P, st, ctas);
}

}  // namespace gsb
