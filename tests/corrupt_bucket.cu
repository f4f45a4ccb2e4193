// Composites one 16x16 tile whose bucket holds the ranks 0 .. n-1 of an env of
// kVis ranked records and, with `bad`, one rank beyond them, by the CTA form
// (form 0), the warp form (1) or its teams (2).  Writes the alpha image and the
// status word.  The order array has kSlack more entries than ranks, all naming
// one opaque record, so the stray rank's place lies inside the array.
#include <string.h>

#include <vector>

#include "gs_internal.cuh"

namespace {
constexpr int kVis = 1500, kSlots = 2016, kSlack = 1 << 17;
template <typename T>
T* upload(const std::vector<T>& v, bool& ok) {
    T* p = nullptr;
    ok = ok && cudaMalloc((void**)&p, v.size() * sizeof(T)) == cudaSuccess &&
         cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) == cudaSuccess;
    return p;
}
}  // namespace

extern "C" int corrupt_bucket(int form, int n, int bad, float* alpha, uint32_t* status) {
    using namespace gsb;
    if (n < 1 || n > kVis) return -1;
    std::vector<EnvInfo> envs(2);
    envs[0].n_local = kSlots;
    envs[0].W = envs[0].H = 16;
    envs[0].ntx = envs[0].T = 1;
    envs[1].tile_base = 1;
    std::vector<float4> rec((size_t)kRecStride * kSlots);
    const uint32_t span = 15u << 16;
    float box;
    memcpy(&box, &span, 4);
    for (int s = 0; s < kSlots; ++s) {  // slot 0: opaque; the others: alpha 0.0045 over the whole tile
        rec[3 * s] = make_float4(8.0f, 8.0f, s ? -7.795859f : -0.1f, 1.0f + s);
        rec[3 * s + 1] = make_float4(0.001f, 0.0f, 0.001f, box);
        rec[3 * s + 2] = make_float4(0.5f, 0.5f, 0.5f, box);
    }
    std::vector<uint32_t> order(kVis + kSlack, 0u), keys((size_t)n + 8, 0u), counts(1, (uint32_t)(n + bad)), one(1, 0u),
        nvis(1, (uint32_t)kVis), work(kWorkWords, 0u);
    for (int r = 0; r < kVis; ++r) order[(size_t)r] = (uint32_t)r + 1u;
    for (int i = 0; i < n; ++i) keys[(size_t)i] = (uint32_t)(n - 1 - i) << 4 | 15u;
    if (bad) keys[(size_t)n] = (uint32_t)(kVis + 5) << 4 | 15u;
    std::vector<unsigned long long> base(2, 0ull);
    std::vector<float> img(16 * 16 * 5, -1.0f);
    bool ok = true;
    CompParams P{};
    P.envs = upload(envs, ok);
    P.e_end = 1;
    P.item_end = 1;
    P.chunk = 1;
    P.work = upload(work, ok);
    P.r0 = upload(rec, ok);
    P.nvis = upload(nvis, ok);
    P.order = upload(order, ok);
    P.counts = upload(counts, ok);
    P.off_local = upload(one, ok);
    P.env_base = upload(base, ok);
    P.pair_cap = keys.size();
    P.pairs = upload(keys, ok);
    P.tile_w = P.tile_h = 16;
    P.quad = form > 0;
    P.key_shift = 4;
    P.rgb = upload(img, ok);
    P.depth = P.rgb + 16 * 16 * 3;
    P.alpha = P.depth + 16 * 16;
    P.status = upload(one, ok);
    uint32_t* items = upload(std::vector<uint32_t>(kItemClasses, 0u), ok);
    if (ok && form == 2) {
        ok = launch_item_order(P.envs, 0, 1, 1, P.counts, nullptr, nullptr, nullptr, items, 1, P.work + 1, 0) ==
             cudaSuccess;
        P.items = items;
        P.class_cnt = P.work + 1;
        P.item_pitch = 1;
        P.team_work = P.work + 1 + kItemClasses;
    }
    int ctas = 0;
    ok = ok && launch_composite(P, 0, &ctas) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
    ok = ok && cudaMemcpy(alpha, P.alpha, 16 * 16 * 4, cudaMemcpyDeviceToHost) == cudaSuccess;
    ok = ok && cudaMemcpy(status, P.status, 4, cudaMemcpyDeviceToHost) == cudaSuccess;
    for (const void* p : {(const void*)P.envs, (const void*)P.work, (const void*)P.r0, (const void*)P.nvis,
                          (const void*)P.order, (const void*)P.counts, (const void*)P.off_local,
                          (const void*)P.env_base, (const void*)P.pairs, (const void*)P.rgb, (const void*)P.status,
                          (const void*)items})
        cudaFree((void*)p);
    return ok ? 0 : -2;
}
