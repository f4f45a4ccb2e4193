// Per-tile front-to-back alpha compositing with early termination (step A5).
//
// The 3DGS forward pass (paper Sec. II-B; the batch renderer of Sec. III-C
// "Throughput Scaling" is built on it) blends, per pixel, the splats whose
// alpha = min(0.99, o exp(-q/2)) reaches 1/255, in depth order, until the
// transmittance would drop below 1e-4; Sec. III-A asks for RGB and depth.
//
// Persistent CTAs claim (env, tile) items; each warp owns an 8x8 pixel
// subtile and each lane two of its pixels.  The tile's bucket holds the depth
// ranks of its splats (gs_rank.cu), in any order; it is consumed in
// depth-ordered windows of at most kCompCap ranks, so ordering stops at the
// window where every pixel has terminated.  A short bucket is one window,
// sorted in shared memory by a counting sort.  A long one is ordered by setting
// a bit per rank in a bitmap of the next 65,536 ranks (128 groups of 512; fewer
// on tiles below 16x16) and reading the bits back in order: ranks are unique, so
// the bitmap is the sorted list, at one shared-memory OR per key.  A window's ranks are mapped to record
// slots; each warp then walks the window on its own, 32 splats at a time:
// a lane stages one of them (its record copied while the 32 before are
// blended) and tests it against the warp's subtile (box, then the exact
// ellipse for large splats), and the overlapping ones are blended two at a
// time, every lane evaluating both at its pixels with no branch inside a step.
// Warps of a tile meet at window ends only: batches of 128 splats staged by the
// whole CTA loaded each record once instead of four times, but a warp with few
// splats of a batch waited for the others (its top stall; 66 % of the issue
// slots used, now 72 %): 256 views of 640x480 11.0 -> 10.7 ms.  What bounds
// it is instruction issue: 72 steps of 2 splats x 64 pixels per subtile, 75
// instructions each.  Besides the image form the kernel has an observation
// form (8-bit colour after per-env appearance, half depth) and a contribution
// form (per-Gaussian blending weights, for pruning); images of low resolution
// and LiDAR scans are composited by gs_composite_warp.cu.
#include "gs_blend.cuh"
#include "gs_block.cuh"
#include <type_traits>

namespace gsb {

constexpr int kInsertMax = 32;   // longest rank range sorted by counting
constexpr int kGroupWords = 16;  // bitmap words per group (512 ranks)

// f(L[i]) for every i in [0, len), spread over the block: 16-byte loads of the
// aligned middle, two in flight per thread.
template <int NT, typename F>
__device__ __forceinline__ void for_ranks(const uint32_t* L, uint32_t len, F&& f) {
    const uint32_t tid = threadIdx.x;
    const uint32_t head = min(len, (uint32_t)((16u - ((uint32_t)(uintptr_t)L & 15u)) & 15u) >> 2);
    if (tid < head) f(L[tid]);
    const uint4* V = reinterpret_cast<const uint4*>(L + head);
    const uint32_t nv = (len - head) >> 2;
    for (uint32_t i = tid; i < nv; i += 2 * NT) {
        const uint4 a = V[i];
        const bool two = i + NT < nv;
        const uint4 b = two ? V[i + NT] : a;
        f(a.x);
        f(a.y);
        f(a.z);
        f(a.w);
        if (two) {
            f(b.x);
            f(b.y);
            f(b.z);
            f(b.w);
        }
    }
    const uint32_t done = head + 4u * nv;
    if (tid < len - done) f(L[done + tid]);
}

// Sorts keys[0, n), distinct ranks in [lo, hi] (tmp: scratch), and returns
// true: a counting sort by SB equal ranges, a rank's place in its range being
// the number of smaller ranks there.  Returns false, with keys untouched, when a range holds more than
// kInsertMax ranks.  c32 (kSortBins words) holds zeros on entry unless `dirty`
// is set (it is cleared here then); a successful sort leaves it zeroed again
// (each thread clears its own ranges after the last barrier; the next reader
// comes after the caller's next barriers).  red: 32 words.
template <int NT, int SB>
__device__ bool rank_sort(uint32_t* keys, uint32_t* tmp, uint32_t* c32, uint32_t* red, int n, uint32_t lo,
                          uint32_t hi, bool& dirty) {
    constexpr int PER = SB / NT;
    static_assert(SB % NT == 0, "ranges per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t span = hi - lo;
    constexpr int LB = SB == 1024 ? 10 : 9;
    const int shift = (span >> LB) ? 32 - LB - __clz(span) : 0;  // span >> shift < SB
    if (dirty) {
        for (int b = tid; b < SB; b += NT) c32[b] = 0u;
        __syncthreads();
        dirty = false;
    }
    for (int i = tid; i < n; i += NT) atomicAdd(&c32[(keys[i] - lo) >> shift], 1u);
    __syncthreads();
    uint32_t loc[PER];
    uint32_t sum = 0;
    bool crowded = false;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        loc[j] = c32[tid * PER + j];
        sum += loc[j];
        crowded |= loc[j] > (uint32_t)kInsertMax;
    }
    // exclusive scan of the per-thread sums; the warps' totals carry a crowded
    // range in bit 31 (a window holds at most kCompCap ranks)
    uint32_t x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    const bool wc = __any_sync(0xffffffffu, crowded);
    if (lane == 31) red[warp] = x | (wc ? 0x80000000u : 0u);
    __syncthreads();
    uint32_t before = 0;
    bool any = false;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        const uint32_t r = red[w];
        if (w < warp) before += r & 0x7fffffffu;
        any |= (r >> 31) != 0u;
    }
    if (any) {
        dirty = true;  // c32 keeps the counts
        __syncthreads();  // red is reused
        return false;
    }
    uint32_t run = before + x - sum;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        c32[tid * PER + j] = run;
        run += loc[j];
    }
    __syncthreads();
    for (int i = tid; i < n; i += NT) {
        const uint32_t k = keys[i];
        tmp[atomicAdd(&c32[(k - lo) >> shift], 1u)] = k;
    }
    __syncthreads();
    for (int i = tid; i < n; i += NT) {  // c32[b] is the end of range b now
        const uint32_t k = tmp[i];
        const uint32_t b = (k - lo) >> shift, e = c32[b];
        uint32_t place = b ? c32[b - 1] : 0u;
        for (uint32_t x = place; x < e; ++x) place += tmp[x] < k ? 1u : 0u;
        keys[place] = k;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; ++j) c32[tid * PER + j] = 0u;
    return true;
}

// Warp sum of one float per lane.
__device__ __forceinline__ float warp_sum(float v) {
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// Warp sums of a in lanes below 16 and of b above, in five exchanges (two
// warp_sum's take ten), adding in the order of warp_sum.  The contribution
// pass's composite, 16 views of 640x480, took 1.21 ms with two warp_sum's and
// takes 0.96 ms (bound by instruction issue, as the image form).
__device__ __forceinline__ float half_sums(float a, float b) {
    const bool high = (threadIdx.x & 16) != 0;
    const float got = __shfl_xor_sync(0xffffffffu, high ? a : b, 16);
    float v = (high ? b : a) + got;
    for (int d = 8; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// Persistent CTAs of TW*TH/2 threads claim (env, tile) items from a work
// counter, `chunk` consecutive items at a time (items run env-major, tiles
// row-major, so envs of any resolution mix in one launch).  For an item the
// CTA covers the TW x TH tile: warp w owns an 8x8 subtile and each lane two
// pixels of it, (x, y) and (x, y + 4), whose blend chains are independent.
//
// SC: contribution pass (pruning support): instead of writing images, add
// each blended (pixel, splat) weight alpha T to score[global index], summed
// per warp and splat before one atomic add.
// CNT: the camera form that also counts composited (pixel, splat) pairs into
// P.neval (the plain form leaves the count out of its blend loop).
template <int TW, int TH, bool SC = false, bool CNT = SC>
__global__ void __launch_bounds__(TW* TH / 2, (TW * TH >= 512 ? 4 : (TW * TH >= 256 ? 8 : (TW * TH >= 128 ? 12 : 24)))) k_composite(CompParams P) {
    constexpr int NT = TW * TH / 2;
    constexpr int CAP = NT == 32 ? 512 : kCompCap;
    constexpr int SB = NT == 32 ? 512 : 1024;      // rank ranges of the short-bucket sort
    constexpr int NG = NT > 128 ? 128 : NT;        // bitmap groups
    constexpr int BMW = NG * kGroupWords;          // bitmap words (32 ranks each)
    constexpr int NW = NT / 32;
    static_assert(BMW >= SB, "the short-bucket counters share the bitmap's memory");
    static_assert(CAP >= kGroupWords * 32, "a group's ranks fit a window");
    __shared__ uint32_t keys[CAP];                      // the window's ranks
    __shared__ float4 recs[NW][2][3][32];               // a warp's records of this and the next 32 splats | sort scratch
    __shared__ __align__(16) uint32_t bm[BMW];          // bitmap | counters of the short-bucket sort
    __shared__ uint32_t pre[NG + 1];                    // ranks set before each group of the bitmap
    __shared__ uint32_t red[32];
    static_assert(sizeof(recs) >= CAP * 4, "the sort scratch shares the records' memory");
    uint32_t* tmp = reinterpret_cast<uint32_t*>(recs);
    __shared__ unsigned int s_item;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto& rec = recs[warp];
    bool c32_dirty = true;  // the short-bucket sort's counters (bm) need clearing before use
    int el = P.e_begin;  // env of the current item, cached across items (uniform in the CTA)
    unsigned int e_lo = P.envs[el].tile_base, e_hi = e_lo + (unsigned)P.envs[el].T;
    if (tid == 0) s_item = atomicAdd(P.work, (unsigned)P.chunk);
    __syncthreads();
    for (;;) {
    const unsigned int first = P.item_begin + s_item;
    if (first >= P.item_end) break;
    const unsigned int last = min(first + (unsigned)P.chunk, P.item_end);
    for (unsigned int item = first; item < last; ++item) {
    if (item < e_lo || item >= e_hi) {
        int lo = P.e_begin, hi = P.e_end - 1;  // env: last e with tile_base <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&P.envs[mid].tile_base) <= item) lo = mid; else hi = mid - 1;
        }
        el = lo;
        e_lo = P.envs[el].tile_base;
        e_hi = e_lo + (unsigned)P.envs[el].T;
    }
    const int t = (int)(item - e_lo);
    const EnvInfo* Ep = P.envs + el;
    const int W = __ldg(&Ep->W), H = __ldg(&Ep->H), ntx = __ldg(&Ep->ntx);
    const unsigned int tile_base = e_lo;
    const unsigned int n_local = __ldg(&Ep->n_local);
    const unsigned long long pix_base = __ldg(&Ep->pix_base);
    const int tx = t % ntx, ty = t / ntx;
    constexpr int SWX = TW / 8;
    const int wx0 = tx * TW + (warp % SWX) * 8, wy0 = ty * TH + (warp / SWX) * 8;
    const int wx1 = wx0 + 7, wy1 = wy0 + 7;
    const int px = wx0 + (lane & 7), py0 = wy0 + (lane >> 3), py1 = py0 + 4;
    const bool in0 = px < W && py0 < H, in1 = px < W && py1 < H;
    const float fpx = (float)px + 0.5f, fpy0 = (float)py0 + 0.5f, fpy1 = (float)py1 + 0.5f;
    bool done0 = !in0, done1 = !in1;
    // the lane's two pixels: .x = (px, py0), .y = (px, py1)
    float2 Tp = make_float2(1.0f, 1.0f), rp = make_float2(0.0f, 0.0f), gp = rp, bp = rp, dp = rp;
    const float2 fpy = make_float2(fpy0, fpy1);
    uint32_t ncomp = 0;

    uint32_t n = P.counts[tile_base + t];
    const unsigned long long start = P.env_base[el] - P.pair_base + P.off_local[tile_base + t];
    if (start + n > P.pair_cap) {  // keys past a planned capacity were dropped: render nothing
        n = 0;
        if (tid == 0) atomicOr(P.status, kStOverflow);
    }
    const uint32_t* Lk = P.pairs + start;
    const size_t recbase = (size_t)__ldg(&Ep->rec_base);
    const uint32_t* order = P.order + recbase;  // record slot of each rank
    // contribution pass: record slot -> global Gaussian index
    const long long g_link0 = SC ? __ldg(&Ep->g_link0) : 0ll;
    auto score_index = [&](uint32_t j) -> long long {
        if (j < P.nbp) return P.bg_index ? (long long)__ldg(P.bg_index + j) : (long long)j;
        return g_link0 + (long long)(j - P.nbp);
    };
    bool finished = false;
    // Composite the window keys[0, wn) (ranks in depth order).  Sets
    // `finished` once every pixel of the tile has terminated.  Each warp walks
    // the window on its own: a lane copies (cp.async) the record of one of the
    // next 32 splats while the current 32 are blended.
    auto run_window = [&](uint32_t wn) {
        auto slot_of = [&](uint32_t i) -> uint32_t { return i < wn ? __ldg(order + keys[i]) : 0xffffffffu; };
        auto fetch = [&](int buf, uint32_t g) {
            if (g < n_local) {
                const float4* src = P.r0 + (size_t)kRecStride * (recbase + g);
                copy16(&rec[buf][0][lane], src);
                copy16(&rec[buf][1][lane], src + 1);
                copy16(&rec[buf][2][lane], src + 2);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        if (!__all_sync(0xffffffffu, done0 && done1)) {
            uint32_t g = slot_of(lane), g_next = slot_of(32 + lane);
            fetch(0, g);
            for (uint32_t c = 0; c < wn; c += 32) {
                const int buf = (int)(c >> 5) & 1;
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                __syncwarp();  // the other buffer is free
                const uint32_t slot = g;
                g = g_next;
                if (c + 32 < wn) fetch(buf ^ 1, g);
                g_next = slot_of(c + 64 + lane);
                float4* sA = rec[buf][0];  // u, v, log2 o, z
                float4* sB = rec[buf][1];  // scaled conic factor l00, l01, l11
                float4* sC = rec[buf][2];  // r, g, b
                {
                    // The lane's splat against the subtile: its box, then the exact
                    // ellipse for large splats (a box under 24 px in width + height is
                    // kept as it is: it overstates the ellipse least).
                    bool ov = false, bright = false;
                    if (slot < n_local) {
                        const float4 A = sA[lane];
                        float4 B = sB[lane];
                        const uint32_t rx = __float_as_uint(B.w), ry = __float_as_uint(sC[lane].w);
                        const int bx0 = (int)(rx & 0xffffu), bx1 = (int)(rx >> 16);
                        const int by0 = (int)(ry & 0xffffu), by1 = (int)(ry >> 16);
                        ov = bx0 <= wx1 && bx1 >= wx0 && by0 <= wy1 && by1 >= wy0;
                        bright = ov && A.z > -0.029146346f;  // log2(0.98)
                        if (ov && bx1 - bx0 + by1 - by0 >= 24) {
                            // alpha >= 1/255 iff q <= w = log2(255 o); the cull's 1e-3
                            // margin dwarfs the rounding of the constant
                            B.w = A.z + 7.9943534f;
                            ov = reaches_rect(A, B, (float)wx0 + 0.5f, (float)wy0 + 0.5f);
                        }
                    } else if (c + lane < wn) {  // never happens for a well-formed bucket
                        atomicOr(P.status, kStOverflow);
                    }
                    const uint32_t m = __ballot_sync(0xffffffffu, ov);
                    // Splats of opacity <= 0.98 never reach the 0.99 cap of alpha (o 2^-q
                    // with q >= 0), so a chunk without brighter splats walks a copy of the
                    // loop without the cap.
                    const bool clamp_chunk = __any_sync(0xffffffffu, bright);
                    // One step blends two splats (TWO): their four alpha evaluations are
                    // independent, the blends run in depth order; an odd last splat has a
                    // step of its own.  No per-pixel box test: a pixel outside a splat's
                    // support box has q > q* (1 + 2e-4), so its alpha falls below 1/255
                    // and the alpha test alone rejects it.
                    auto step = [&](auto clamp_tag, auto two_tag, int j1, int j2) {
                        constexpr bool CL = decltype(clamp_tag)::value, TWO = decltype(two_tag)::value;
                        const float4 A1 = sA[j1], B1 = sB[j1];
                        const float4 A2 = sA[j2], B2 = sB[j2];
                        const float2 a1 = splat_alpha2<CL>(A1, B1, fpx, fpy);
                        float2 a2 = make_float2(0.0f, 0.0f);
                        if constexpr (TWO) a2 = splat_alpha2<CL>(A2, B2, fpx, fpy);
                        const bool u10 = !done0 && a1.x >= (1.0f / 255.0f);
                        const bool u11 = !done1 && a1.y >= (1.0f / 255.0f);
                        float w1 = 0.0f, w2 = 0.0f;
                        // The blends with plain selects while no pixel of the warp stops at
                        // either splat (the common case); else one splat at a time with the
                        // stop rule.  Either way the arithmetic is that of blend2, so the
                        // images do not depend on the path taken.  Every lane of the warp
                        // reaches the vote: the camera path has no divergent branch around
                        // it (branches here measured slower than evaluating every lane's
                        // pixels).
                        const float2 am1 = make_float2(u10 ? a1.x : 0.0f, u11 ? a1.y : 0.0f);
                        const float2 x1 = __fmul2_rn(am1, Tp);
                        const float2 Tn1 = __fadd2_rn(Tp, make_float2(-x1.x, -x1.y));
                        float2 x2 = make_float2(0.0f, 0.0f), Tn2 = Tn1;
                        bool v20 = false, v21 = false;
                        if constexpr (TWO) {
                            v20 = !done0 && a2.x >= (1.0f / 255.0f);
                            v21 = !done1 && a2.y >= (1.0f / 255.0f);
                            const float2 am2 = make_float2(v20 ? a2.x : 0.0f, v21 ? a2.y : 0.0f);
                            x2 = __fmul2_rn(am2, Tn1);
                            Tn2 = __fadd2_rn(Tn1, make_float2(-x2.x, -x2.y));
                        }
                        // Tn2 = Tn1 - am2 Tn1 <= Tn1 (am2 >= 0, rounding is monotone),
                        // so a pixel that stops at either splat has Tn2 < 1e-4
                        const bool stop = Tn2.x < 1e-4f || Tn2.y < 1e-4f;
                        if (!__any_sync(0xffffffffu, stop)) {
                            if constexpr (CNT) ncomp += (uint32_t)u10 + (uint32_t)u11 + (uint32_t)v20 + (uint32_t)v21;
                            const float4 C1 = sC[j1];
                            rp = __ffma2_rn(x1, make_float2(C1.x, C1.x), rp);
                            gp = __ffma2_rn(x1, make_float2(C1.y, C1.y), gp);
                            bp = __ffma2_rn(x1, make_float2(C1.z, C1.z), bp);
                            dp = __ffma2_rn(x1, make_float2(A1.w, A1.w), dp);
                            if constexpr (TWO) {
                                const float4 C2 = sC[j2];
                                rp = __ffma2_rn(x2, make_float2(C2.x, C2.x), rp);
                                gp = __ffma2_rn(x2, make_float2(C2.y, C2.y), gp);
                                bp = __ffma2_rn(x2, make_float2(C2.z, C2.z), bp);
                                dp = __ffma2_rn(x2, make_float2(A2.w, A2.w), dp);
                            }
                            Tp = Tn2;
                            w1 = x1.x + x1.y;
                            w2 = x2.x + x2.y;
                        } else {
                            if constexpr (CNT) ncomp += (uint32_t)u10 + (uint32_t)u11;
                            w1 = blend2(a1, u10, u11, sC[j1], A1.w, Tp, rp, gp, bp, dp, done0, done1);
                            if constexpr (TWO) {
                                const bool u20 = !done0 && a2.x >= (1.0f / 255.0f);
                                const bool u21 = !done1 && a2.y >= (1.0f / 255.0f);
                                if constexpr (CNT) ncomp += (uint32_t)u20 + (uint32_t)u21;
                                w2 = blend2(a2, u20, u21, sC[j2], A2.w, Tp, rp, gp, bp, dp, done0, done1);
                            }
                        }
                        if constexpr (SC) {  // warp-uniform: the lanes add their weights
                            const bool high = TWO && lane >= 16;
                            const float v = TWO ? half_sums(w1, w2) : warp_sum(w1);
                            const uint32_t g = __shfl_sync(0xffffffffu, slot, high ? j2 : j1);
                            if ((lane == 0 || (TWO && lane == 16)) && v > 0.0f)
                                atomicAdd(P.score + score_index(g), v);
                        }
                    };
                    auto walk = [&](auto clamp_tag) {
                        uint32_t r = __brev(m);  // the first splat is the leading bit
                        while (r & (r - 1u)) {
                            const int k1 = __clz(r);
                            r ^= 0x80000000u >> k1;
                            const int k2 = __clz(r);
                            r ^= 0x80000000u >> k2;
                            step(clamp_tag, std::true_type{}, k1, k2);
                        }
                        if (r) {
                            const int k1 = __clz(r);
                            step(clamp_tag, std::false_type{}, k1, k1);
                        }
                    };
                    if (clamp_chunk) walk(std::true_type{});
                    else walk(std::false_type{});
                }
                if (__all_sync(0xffffffffu, done0 && done1)) break;
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        finished = __syncthreads_and(done0 && done1) != 0;
    };

    // The next window: its wn ranks in depth order in keys.
    uint32_t before = 0;          // ranks of the bucket in earlier windows
    bool whole = n <= (uint32_t)CAP;  // the bucket is one window, sorted at once
    bool loaded = false;          // a bitmap of the ranks [r0, r0 + 32 BMW) is set up
    uint32_t r0 = 0;
    int g0 = 0;                   // its next group
    while (before < n && !finished) {
        uint32_t wn = 0;
        if (whole) {
            uint32_t lo = 0xffffffffu, hi = 0u;
            for (uint32_t i = tid; i < n; i += NT) {
                const uint32_t k = Lk[i] >> P.key_shift;
                keys[i] = k;
                lo = min(lo, k);
                hi = max(hi, k);
            }
            block_minmax_u32<NT>(lo, hi, red);
            // (a rank beyond the env's, in a corrupted bucket: the bitmaps leave it out)
            whole = hi < __ldg(P.nvis + el) && rank_sort<NT, SB>(keys, tmp, bm, red, (int)n, lo, hi, c32_dirty);
            if (!whole) continue;  // crowded ranks: through bitmaps
            wn = n;
        } else {
            if (loaded && g0 >= NG) {
                loaded = false;
                r0 += (uint32_t)(BMW * 32);
                __syncthreads();  // bm is rewritten for the next ranks
            }
            if (!loaded) {
                const uint32_t n_rank = __ldg(P.nvis + el);  // read here: a register less through the blend loop
                if (r0 >= n_rank) {  // ranks beyond the env's: a corrupted bucket
                    if (tid == 0) atomicOr(P.status, kStOverflow);
                    break;
                }
                c32_dirty = true;
                for (int i = tid; i < BMW / 4; i += NT) reinterpret_cast<uint4*>(bm)[i] = make_uint4(0u, 0u, 0u, 0u);
                __syncthreads();
                for_ranks<NT>(Lk, n, [&](uint32_t k) {
                    const uint32_t d = (k >> P.key_shift) - r0;
                    if (d < (uint32_t)(BMW * 32)) atomicOr(&bm[d >> 5], 1u << (d & 31u));
                });
                __syncthreads();
                if (n_rank - r0 < (uint32_t)(BMW * 32)) {  // the env's last ranks: a bit beyond is a corrupted bucket's
                    bool stray = false;
                    for (uint32_t i = ((n_rank - r0) >> 5) + tid; i < (uint32_t)BMW; i += NT) {
                        const uint32_t first = r0 + 32u * i, m = bm[i];
                        const uint32_t keep = n_rank > first ? (1u << (n_rank - first)) - 1u : 0u;
                        stray |= (m & ~keep) != 0u;
                        bm[i] = m & keep;
                    }
                    if (stray) atomicOr(P.status, kStOverflow);
                    __syncthreads();
                }
                // ranks set before each group: thread t counts groups GPT t ..
                constexpr int GPT = NG < NT ? 1 : NG / NT;
                uint32_t c[GPT], sum = 0;
#pragma unroll
                for (int j = 0; j < GPT; ++j) {
                    const int g = tid * GPT + j;
                    c[j] = 0;
                    if (g >= NG) continue;
#pragma unroll
                    for (int i = 0; i < kGroupWords; ++i)  // rotated: neighbouring threads hit different banks
                        c[j] += __popc(bm[g * kGroupWords + ((i + tid) & (kGroupWords - 1))]);
                    sum += c[j];
                }
                uint32_t run = block_excl_scan_u32<NT>(sum, red);
#pragma unroll
                for (int j = 0; j < GPT; ++j) {
                    if (tid * GPT + j <= NG) pre[tid * GPT + j] = run;
                    run += c[j];
                }
                if (NG >= NT && tid == NT - 1) pre[NG] = run;
                __syncthreads();
                loaded = true;
                g0 = 0;
            }
            // a run of whole groups of at most CAP ranks
            const uint32_t base = pre[g0];
            int lo = g0 + 1, hi = NG;  // last g1 with pre[g1] - base <= CAP
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (pre[mid] - base <= (uint32_t)CAP) lo = mid; else hi = mid - 1;
            }
            const int g1 = lo;
            wn = pre[g1] - base;
            if (wn > 0) {
                // a half-warp reads a group's words back in order
                for (int gb = g0 + 2 * warp; gb < g1; gb += NT / 16) {
                    const int g = gb + (lane >> 4);
                    uint32_t w = g < g1 ? bm[g * kGroupWords + (lane & 15)] : 0u;
                    const uint32_t pc = __popc(w);
                    uint32_t x = pc;
#pragma unroll
                    for (int d = 1; d < 16; d <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d, 16);
                        if ((lane & 15) >= d) x += y;
                    }
                    if (w) {
                        uint32_t at = pre[g] - base + x - pc;
                        const uint32_t r = r0 + (uint32_t)(g * kGroupWords + (lane & 15)) * 32u;
                        while (w) {
                            keys[at++] = r + (uint32_t)(__ffs(w) - 1);
                            w &= w - 1u;
                        }
                    }
                }
                __syncthreads();
            }
            g0 = g1;
            if (wn == 0) continue;
        }
        run_window(wn);
        before += wn;
    }

    if (CNT && P.neval) {
        uint32_t c = ncomp;
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
        if (lane == 0 && c) atomicAdd(P.neval, (unsigned long long)c);
    }
    if constexpr (!SC) {
        const PixelStore store(P, el);
        if (in0) store.put(P, pix_base + (size_t)py0 * W + px, Tp.x, rp.x, gp.x, bp.x, dp.x);
        if (in1) store.put(P, pix_base + (size_t)py1 * W + px, Tp.y, rp.y, gp.y, bp.y, dp.y);
    }
    __syncthreads();  // shared staging is reused by the next item
    }  // items of the claim
    if (tid == 0) s_item = atomicAdd(P.work, (unsigned)P.chunk);  // every thread has read the last claim
    __syncthreads();
    }  // claims
}

template <int TW, int TH, bool SC = false, bool CNT = SC>
static cudaError_t launch_tiles(const CompParams& P, cudaStream_t st, int* ctas) {
    constexpr int NT = TW * TH / 2;
    static PerDevice resident;
    int full = 0;
    const cudaError_t e = resident.ctas((const void*)k_composite<TW, TH, SC, CNT>, NT, &full);
    if (e != cudaSuccess) return e;
    const unsigned claims = (P.item_end - P.item_begin + P.chunk - 1) / P.chunk;
    *ctas = (int)std::min((unsigned)full, claims);
    k_composite<TW, TH, SC, CNT><<<*ctas, NT, 0, st>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_composite(const CompParams& P, cudaStream_t st, int* ctas) {
    *ctas = 0;
    if (P.item_end <= P.item_begin) return cudaSuccess;
    if (P.lidars && (P.tile_w != 16 || P.tile_h != 16 || P.score)) return cudaErrorInvalidValue;
    if (P.lidars || P.quad) return launch_composite_warp(P, st, ctas);
    if (P.score) {  // the contribution pass runs on 16x16 tiles only
        if (P.tile_w != 16 || P.tile_h != 16) return cudaErrorInvalidValue;
        return launch_tiles<16, 16, true>(P, st, ctas);
    }
    if (P.neval) {  // counting pass
        if (P.tile_w == 16 && P.tile_h == 16) return launch_tiles<16, 16, false, true>(P, st, ctas);
        if (P.tile_w == 32 && P.tile_h == 16) return launch_tiles<32, 16, false, true>(P, st, ctas);
        if (P.tile_w == 8 && P.tile_h == 8) return launch_tiles<8, 8, false, true>(P, st, ctas);
        if (P.tile_w == 16 && P.tile_h == 8) return launch_tiles<16, 8, false, true>(P, st, ctas);
        return launch_tiles<32, 8, false, true>(P, st, ctas);
    }
    if (P.tile_w == 16 && P.tile_h == 16) return launch_tiles<16, 16>(P, st, ctas);
    if (P.tile_w == 32 && P.tile_h == 16) return launch_tiles<32, 16>(P, st, ctas);
    if (P.tile_w == 8 && P.tile_h == 8) return launch_tiles<8, 8>(P, st, ctas);
    if (P.tile_w == 16 && P.tile_h == 8) return launch_tiles<16, 8>(P, st, ctas);
    return launch_tiles<32, 8>(P, st, ctas);
}

}  // namespace gsb
