// Depth ranking: every visible record of an env gets its place in the env's
// front-to-back order (step A4's ordering, done once per record instead of
// once per (tile, record) intersection).  The renderer of the paper (Sec.
// III-C, built on gsplat) sorts its intersections by (tile, depth); a record
// reaches 2 tiles on average at 128x128 and 11 at 640x480, so ranking the
// records first sorts 2 to 11 times fewer keys, leaves 4-byte ranks to bin
// (instead of 8-byte depth keys), and turns the compositor's sort of a bucket
// into setting bits: ranks are unique and dense.
//
// A sample sort per env: k_rank_sample sorts a strided sample of the visible
// records' keys (depth bits << 32 | caller's index) and takes splitters; the
// count pass (gs_bin.cu) histograms the records over the ranges between them;
// k_rank_place groups the keys by range and k_rank_sort sorts windows of whole
// ranges in shared memory.  Splitters are whole keys, and keys are unique, so
// ranges stay balanced however the depths crowd (a wall at one depth included).
#include "gs_internal.cuh"
#include "gs_block.cuh"

namespace gsb {

namespace {

constexpr int kSampleLooks = 8;     // slots looked at per thread of k_rank_sample: a byte of bits
constexpr int kSortThreads = 256;
constexpr int kSortCap = 2048;      // keys of a window sorted in shared memory
constexpr int kSubBins = 1024;      // depth ranges of a window's counting sort
constexpr int kInsert = 128;        // longest range sorted by counting

// Ascending bitonic sort of NT * K keys by a block of NT threads, thread t
// holding elements K t .. K t + K - 1: exchanges stay in a thread or go by
// shuffles below 32 K keys, through smp (NT * K keys) above.
template <int NT, int K>
__device__ __forceinline__ void block_bitonic(unsigned long long (&v)[K], unsigned long long* smp) {
    const int tid = threadIdx.x;
    for (int size = 2; size <= NT * K; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= K) {
                unsigned long long o[K];
                if (stride >= 32 * K) {
                    __syncthreads();
#pragma unroll
                    for (int k = 0; k < K; ++k) smp[k * NT + tid] = v[k];
                    __syncthreads();
#pragma unroll
                    for (int k = 0; k < K; ++k) o[k] = smp[k * NT + (tid ^ (stride / K))];
                } else {
#pragma unroll
                    for (int k = 0; k < K; ++k) o[k] = __shfl_xor_sync(0xffffffffu, v[k], stride / K);
                }
                const bool low = (tid & (stride / K)) == 0;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const bool up = ((K * tid + k) & size) == 0;
                    v[k] = (v[k] < o[k]) == (up == low) ? v[k] : o[k];
                }
            } else {
#pragma unroll
                for (int d = K / 2; d > 0; d >>= 1)
                    if (stride == d) {
#pragma unroll
                        for (int k = 0; k < K; ++k) {
                            const int j = k ^ d;
                            if (j > k) {
                                const bool up = ((K * tid + k) & size) == 0;
                                const unsigned long long x = v[k], y = v[j];
                                if ((x > y) == up) {
                                    v[k] = y;
                                    v[j] = x;
                                }
                            }
                        }
                    }
            }
        }
}

}  // namespace

// One CTA of 1024 threads per env; K sampled keys per thread.  Bound by
// latency: a strided gather, a sort of the sample, then a search per depth cell.
// The whole sample is used however few ranges there are: with two samples per
// range, 8 views of 16,384 splats (32 ranges) had windows of over kSortCap keys
// and k_rank_sort took 28 us instead of 10.  bins is a power of two, so a
// splitter's place is a shift (640,000 slots, one env: 28 us with a 64-bit
// division, 21 with the shift).  The stride is odd, so it does not resonate with
// the 32-slot visibility words or the links' cluster sizes.  A thread numbers eight
// neighbouring looks, so that the visible ones are numbered in storage order and
// every n-th, which is kept, comes from all over it: numbered by threads with 1024
// looks between a thread's, views that see every slot kept each thread's first, the
// first eighth of the (Morton) order, and one range got up to half of the records
// (8 views of 120,000 splats: ranking after the scan 175 us, now 29).  The looks
// themselves are taken across the block, and the kept ones listed before one thread
// loads each: with both by the numbering thread the kernel took 11.3 us instead of
// 10.3 for 3,000 slots and 22.5 instead of 20.5 for 600,000.
template <int K>
__global__ void __launch_bounds__(1024) k_rank_sample(RankParams P) {
    constexpr int M = 1024 * K;
    __shared__ unsigned long long smp[M];
    __shared__ uint32_t red[32];
    __shared__ uint32_t words[32 * kSampleLooks];
    __shared__ uint16_t where[M];  // the kept looks
    const int el = blockIdx.x, tid = threadIdx.x;
    const EnvInfo E = P.envs[el];
    const uint32_t n = E.n_local;
    const int want = M;
    uint32_t step = (n + 1024 * kSampleLooks - 1) / (1024 * kSampleLooks);
    if (step > 1) step |= 1u;
#pragma unroll
    for (int k = 0; k < kSampleLooks; ++k) {  // bit i of the words: look i, slot i step, is visible
        const unsigned long long j = (unsigned long long)(tid + 1024 * k) * step;
        const uint32_t m =
            __ballot_sync(0xffffffffu, j < n && ((__ldg(P.mask + E.mask_base + (j >> 5)) >> (j & 31u)) & 1u));
        if ((tid & 31) == 0) words[32 * k + (tid >> 5)] = m;
    }
    __syncthreads();
    const uint32_t seen = reinterpret_cast<const uint8_t*>(words)[tid];  // looks kSampleLooks tid + k
    uint32_t total = 0;
    uint32_t at = block_excl_scan_total<1024>((uint32_t)__popc(seen), red, total);
    const uint32_t every = (total + (uint32_t)want - 1) / (uint32_t)want;
    const int kept = every ? (int)((total + every - 1) / every) : 0;
#pragma unroll
    for (int k = 0; k < K; ++k) smp[tid + 1024 * k] = ~0ull;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSampleLooks; ++k) {
        if (!((seen >> k) & 1u)) continue;
        if (at % every == 0) where[at / every] = (uint16_t)(kSampleLooks * tid + k);
        ++at;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (tid + 1024 * k < kept) {
            const uint32_t j = (uint32_t)where[tid + 1024 * k] * step;  // < n
            smp[tid + 1024 * k] = rank_key(P, P.r3[E.rec_base + j], j);
        }
    __syncthreads();
    // thread t holds elements K t .. K t + K - 1
    unsigned long long v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = smp[K * tid + k];
    block_bitonic<1024, K>(v, smp);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) smp[K * tid + k] = v[k];
    __syncthreads();
    unsigned long long* out = P.split + (size_t)el * P.bins;
    const int lb = __ffs(P.bins) - 1;  // bins are a power of two
    auto splitter = [&](int k) -> unsigned long long {
        return kept ? smp[min(kept - 1, (int)((uint32_t)((k + 1) * kept) >> lb))] : ~0ull;
    };
    for (int k = tid; k < P.bins - 1; k += 1024) out[k] = splitter(k);
    // the lookup: equal depth cells from the smallest sample
    const uint32_t z0 = kept ? (uint32_t)(smp[0] >> 32) : 0u;
    const uint32_t span = kept ? (uint32_t)(smp[kept - 1] >> 32) - z0 : 0u;
    int shift = 0;
    while ((span >> shift) >= (uint32_t)P.cells) ++shift;
    if (tid == 0) out[P.bins - 1] = (unsigned long long)shift << 32 | z0;
    uint16_t* cell = P.cell + (size_t)el * P.cells;
    for (int c = tid; c < P.cells; c += 1024) {
        int lo = 0, hi = c ? P.bins - 1 : 0;  // splitters below the cell's first key
        const unsigned long long first = ((unsigned long long)z0 + ((unsigned long long)c << shift)) << 32;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (splitter(mid) < first) lo = mid + 1; else hi = mid;
        }
        cell[c] = (uint16_t)lo;
    }
}

// Small envs, whole: one CTA per env sorts the visible keys of all K * 1024 slots
// and writes order, rank and the number of visible records; there are no depth
// ranges then (bins = 0), and the count and the scan skip theirs.  A counting sort
// by kSmallBins ranges of the depth bits, a key's place in its range being the
// number of smaller keys in it, or a bitonic sort when a range holds more than
// kSmallInsert (a wall seen head-on).  Bound by the latency of its ten barriers.
// The kernel on 200 views of 32x24, 1100 slots each: 25 us with the bitonic sort
// for all, now 9.  Calls without allocation (us; before records were ranked / by
// sampling / by the bitonic sort / now): one 64x48 view of 900 splats 73 / 94 / 71 /
// 71, 24 views of 1500 90 / 119 / 92 / 84.  K = 4 takes 16 us for 200 views.
constexpr int kSmallBins = 2048;
constexpr int kSmallInsert = 32;
template <int K>
__global__ void __launch_bounds__(1024) k_rank_small(RankParams P) {
    constexpr int NT = 1024;
    __shared__ unsigned long long smp[NT * K];
    __shared__ uint32_t cnt[kSmallBins];
    __shared__ uint32_t red[64];
    const int el = blockIdx.x, tid = threadIdx.x;
    const EnvInfo E = P.envs[el];
    auto put = [&](uint32_t place, unsigned long long key) {
        const uint32_t g = (uint32_t)key;
        const uint32_t slot = (P.bg_slot && g < P.n_bg) ? (uint32_t)__ldg(P.bg_slot + g) : g;
        P.order[E.rec_base + place] = slot;
        P.rank[E.rec_base + slot] = place;
    };
    unsigned long long v[K];
    uint32_t zl = 0xffffffffu, zh = 0u;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t j = (uint32_t)(k * NT + tid);
        v[k] = ~0ull;
        if (j < E.n_local && ((__ldg(P.mask + E.mask_base + (j >> 5)) >> (j & 31u)) & 1u)) {
            v[k] = rank_key(P, P.r3[E.rec_base + j], j);
            zl = min(zl, (uint32_t)(v[k] >> 32));
            zh = max(zh, (uint32_t)(v[k] >> 32));
        }
    }
    cnt[2 * tid] = 0u;
    cnt[2 * tid + 1] = 0u;
    block_minmax_u32<NT>(zl, zh, red);
    const uint32_t span = zh > zl ? zh - zl : 0u;
    const int shift = (span >> 11) ? 21 - __clz(span) : 0;  // span >> shift < kSmallBins
    uint32_t at[K];  // range << 16 | place in it
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (v[k] != ~0ull) {
            const uint32_t b = ((uint32_t)(v[k] >> 32) - zl) >> shift;
            at[k] = b << 16 | atomicAdd(&cnt[b], 1u);
        }
    __syncthreads();
    const uint32_t c0 = cnt[2 * tid], c1 = cnt[2 * tid + 1];
    const bool crowded = __syncthreads_or(max(c0, c1) > (uint32_t)kSmallInsert) != 0;
    uint32_t nv;
    const uint32_t start = block_excl_scan_total<NT>(c0 + c1, red, nv);
    if (tid == 0) P.nvis[el] = nv;
    if (crowded) {
        block_bitonic<NT, K>(v, smp);
#pragma unroll
        for (int k = 0; k < K; ++k)
            if ((uint32_t)(K * tid + k) < nv) put((uint32_t)(K * tid + k), v[k]);
        return;
    }
    cnt[2 * tid] = start;
    cnt[2 * tid + 1] = start + c0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (v[k] != ~0ull) smp[cnt[at[k] >> 16] + (at[k] & 0xffffu)] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (v[k] != ~0ull) {
            const uint32_t b = at[k] >> 16, s = cnt[b], e = b + 1 < (uint32_t)kSmallBins ? cnt[b + 1] : nv;
            uint32_t place = s;
            for (uint32_t x = s; x < e; ++x) place += smp[x] < v[k] ? 1u : 0u;
            put(place, v[k]);
        }
}

// Groups the env's keys by range: a record's range and place were noted by
// the count, whose blocks this kernel shares.  Streams the records once.
__global__ void __launch_bounds__(256) k_rank_place(RankParams P) {
    __shared__ uint32_t first[kRankBins];
    const int el = blockIdx.y, lane = threadIdx.x & 31;
    const EnvInfo E = P.envs[el];
    const uint32_t words = (E.n_local + 31) / 32;
    const uint32_t w0 = blockIdx.x * (uint32_t)P.words_per_block;
    if (w0 >= words) return;
    const uint32_t w1 = min(w0 + (uint32_t)P.words_per_block, words);
    const uint32_t* bo = P.block_off + ((size_t)el * P.blocks + blockIdx.x) * P.bins;
    for (int b = threadIdx.x; b < P.bins; b += 256) first[b] = P.bin_off[(size_t)el * P.bins + b] + bo[b];
    __syncthreads();
    constexpr int U = 4;  // words in flight per warp
    for (uint32_t w = w0 + (threadIdx.x >> 5); w < w1; w += 8 * U) {
        uint32_t at[U];
        uint4 q[U];
        bool vis[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            vis[u] = w + 8 * u < w1 && ((__ldg(P.mask + E.mask_base + w + 8 * u) >> lane) & 1u);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t j = E.rec_base + (w + 8 * u) * 32 + lane;
            if (vis[u]) {
                at[u] = P.rank[j];
                q[u] = P.r3[j];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (vis[u])
                P.zkeys[E.rec_base + first[at[u] >> 13] + (at[u] & 0x1fffu)] =
                    rank_key(P, q[u], (w + 8 * u) * 32 + lane);
    }
}

// Sorts an env's windows of whole ranges (positions [win[v], win[v+1])) and
// writes order and rank.  A window of at most kSortCap keys is sorted in
// shared memory: a counting sort by kSubBins ranges of its depth bits, a key's
// place in its range being the number of smaller keys in it (up to kInsert; a
// face seen head-on crowds hundreds of keys into few ranges), or a bitonic sort
// when a range holds more.  A larger window (a sample that missed a crowd) is
// cut into pieces of at most kSortCap keys by radix selection over its keys.
__global__ void __launch_bounds__(kSortThreads, 4) k_rank_sort(RankParams P) {
    constexpr int NT = kSortThreads;
    constexpr int PT = kSortCap / NT;  // keys per thread
    __shared__ unsigned long long tmp[kSortCap];
    __shared__ uint32_t cnt[kSubBins + 1];
    __shared__ uint32_t red[64];
    __shared__ unsigned long long sel_lo, sel_hi;
    __shared__ uint32_t sel_n;
    __shared__ int sel_state;
    const int tid = threadIdx.x, el = blockIdx.y;
    const EnvInfo E = P.envs[el];
    const uint32_t nv = P.nvis[el];
    const uint32_t nwin = (nv + kRankStride - 1) / kRankStride;
    const unsigned long long* Z = P.zkeys + E.rec_base;
    uint32_t* order = P.order + E.rec_base;
    uint32_t* rank = P.rank + E.rec_base;

    // sort src[0, m) (global keys, or tmp itself) and give the keys the places
    // first, first + 1, ...
    auto sort_out = [&](const unsigned long long* src, int m, uint32_t first) {
        auto put = [&](uint32_t place, unsigned long long key) {
            const uint32_t g = (uint32_t)key;
            const uint32_t slot = (P.bg_slot && g < P.n_bg) ? (uint32_t)__ldg(P.bg_slot + g) : g;
            if (slot < E.n_local) {  // always, for keys that the placement wrote
                order[place] = slot;
                rank[slot] = place;
            }
        };
        unsigned long long k[PT];
        uint32_t zl = 0xffffffffu, zh = 0u;
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            const int i = tid + u * NT;
            k[u] = i < m ? src[i] : ~0ull;
            if (i < m) {
                zl = min(zl, (uint32_t)(k[u] >> 32));
                zh = max(zh, (uint32_t)(k[u] >> 32));
            }
        }
        for (int b = tid; b < kSubBins; b += NT) cnt[b] = 0u;
        block_minmax_u32<NT>(zl, zh, red);
        const uint32_t span = zh - zl;
        const int shift = (span >> 10) ? 22 - __clz(span) : 0;  // span >> shift < kSubBins
        uint32_t at[PT];  // range << 16 | place in it
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            if (u * NT >= m) break;  // uniform
            if (tid + u * NT < m) {
                const uint32_t b = ((uint32_t)(k[u] >> 32) - zl) >> shift;
                at[u] = b << 16 | atomicAdd(&cnt[b], 1u);
            }
        }
        __syncthreads();
        constexpr int PER = kSubBins / NT;
        uint32_t loc[PER], sum = 0;
        bool crowded = false;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            loc[j] = cnt[tid * PER + j];
            sum += loc[j];
            crowded |= loc[j] > (uint32_t)kInsert;
        }
        if (__syncthreads_or(crowded)) {
            block_bitonic<NT, PT>(k, tmp);  // the keys in any order, ~0 beyond the last
#pragma unroll
            for (int u = 0; u < PT; ++u)
                if (PT * tid + u < m) put(first + (uint32_t)(PT * tid + u), k[u]);
            __syncthreads();
            return;
        }
        uint32_t run = block_excl_scan_u32<NT>(sum, red);
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            cnt[tid * PER + j] = run;
            run += loc[j];
        }
        if (tid == NT - 1) cnt[kSubBins] = run;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            if (u * NT >= m) break;
            if (tid + u * NT < m) tmp[cnt[at[u] >> 16] + (at[u] & 0xffffu)] = k[u];
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            if (u * NT >= m) break;
            if (tid + u * NT < m) {
                const uint32_t b = at[u] >> 16, s = cnt[b], e = cnt[b + 1];
                uint32_t place = s;
                for (uint32_t x = s; x < e; ++x) place += tmp[x] < k[u] ? 1u : 0u;
                put(first + place, k[u]);
            }
        }
        __syncthreads();
    };

    for (uint32_t v = blockIdx.x; v < nwin; v += gridDim.x) {
        const uint32_t a = P.win[(size_t)el * P.win_pitch + v], b = P.win[(size_t)el * P.win_pitch + v + 1];
        if (b <= a) continue;
        if (b - a <= (uint32_t)kSortCap) {
            sort_out(Z + a, (int)(b - a), a);
            continue;
        }
        // cut [a, b) into pieces: per piece the largest key bound below which
        // at most kSortCap of the remaining keys lie (8-bit digits of the
        // remaining key range; unique keys separate within eight levels)
        uint32_t used = 0;
        unsigned long long lo = 0ull;
        while (used < b - a) {
            if (tid == 0) {
                sel_lo = lo;
                sel_hi = ~0ull;
                sel_state = 0;
            }
            __syncthreads();
            for (int level = 0; level < 9; ++level) {
                const unsigned long long l = sel_lo, h = sel_hi, x = l ^ h;
                const int hb = x ? 63 - __clzll((long long)x) : 0;
                const int shift = hb > 7 ? hb - 7 : 0;
                for (int i = tid; i < 256; i += NT) cnt[i] = 0u;
                __syncthreads();
                for (uint32_t i = tid; i < b - a; i += NT) {
                    const unsigned long long k = Z[a + i];
                    if (k >= l && k <= h) atomicAdd(&cnt[(k >> shift) & 255u], 1u);
                }
                __syncthreads();
                if (tid == 0) {
                    const unsigned long long pre = (l >> shift >> 8) << 8 << shift;
                    int d = 0;
                    while (d < 255 && cnt[d] == 0u) ++d;
                    if (cnt[d] > (uint32_t)kSortCap) {
                        const unsigned long long bl = pre | ((unsigned long long)d << shift);
                        const unsigned long long bh = bl | ((1ull << shift) - 1ull);
                        sel_lo = bl > l ? bl : l;
                        sel_hi = bh < h ? bh : h;
                    } else {
                        uint32_t cum = 0;
                        while (d < 256 && cum + cnt[d] <= (uint32_t)kSortCap) cum += cnt[d++];
                        // keys up to and including sel_hi
                        sel_hi = d >= 256 ? h : min(h, (pre | ((unsigned long long)d << shift)) - 1ull);
                        sel_n = cum;
                        sel_state = 1;
                    }
                }
                __syncthreads();
                if (sel_state) break;
            }
            const unsigned long long bound = sel_hi;
            const uint32_t have = sel_n;
            const bool ok = sel_state != 0 && have > 0u;
            __syncthreads();
            if (!ok) {  // never for unique keys
                if (tid == 0) atomicOr(P.status, kStOverflow);
                break;
            }
            if (tid == 0) sel_n = 0u;
            __syncthreads();
            for (uint32_t i = tid; i < b - a; i += NT) {
                const unsigned long long k = Z[a + i];
                if (k >= lo && k <= bound) {
                    const uint32_t p = atomicAdd(&sel_n, 1u);
                    if (p < (uint32_t)kSortCap) tmp[p] = k;
                }
            }
            __syncthreads();
            sort_out(tmp, (int)have, a + used);
            used += have;
            lo = bound + 1ull;
        }
    }
}

static_assert(kSmallRank <= 4 * 1024 && kSmallBins == 2 * 1024, "small envs fit one CTA's keys and counters");

cudaError_t launch_rank_sample(const RankParams& R, int n_envs, cudaStream_t st) {
    if (n_envs == 0) return cudaSuccess;
    if (R.bins == 0) {
        if (R.max_slots <= 1024) k_rank_small<1><<<n_envs, 1024, 0, st>>>(R);
        else if (R.max_slots <= 2048) k_rank_small<2><<<n_envs, 1024, 0, st>>>(R);
        else k_rank_small<4><<<n_envs, 1024, 0, st>>>(R);
        return cudaGetLastError();
    }
    if (R.bins <= 512) k_rank_sample<1><<<n_envs, 1024, 0, st>>>(R);
    else if (R.bins <= 1024) k_rank_sample<2><<<n_envs, 1024, 0, st>>>(R);
    else k_rank_sample<4><<<n_envs, 1024, 0, st>>>(R);
    return cudaGetLastError();
}

cudaError_t launch_rank(const RankParams& R, int n_envs, int max_words, cudaStream_t st) {
    if (n_envs == 0 || max_words == 0 || R.bins == 0) return cudaSuccess;
    k_rank_place<<<dim3((unsigned)R.blocks, (unsigned)n_envs), 256, 0, st>>>(R);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // a CTA per window while an env's windows are few; the others loop
    const unsigned wins = (unsigned)std::min((long long)(max_words * 32ll + kRankStride - 1) / kRankStride, 160ll);
    k_rank_sort<<<dim3(wins, (unsigned)n_envs), kSortThreads, 0, st>>>(R);
    return cudaGetLastError();
}

}  // namespace gsb
