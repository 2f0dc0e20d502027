// Forward over few query tiles: the parts that the CTAs of a cluster have formed of a 128-row tile, put together.
// Part k of a row: reference point m_k, sum l_k of exponentials and unnormalised O_k (f32), all relative to m_k.
//     m = max m_k,  f_k = 2^(m_k - m),  l = sum f_k l_k,  O = (sum f_k O_k) / l,  summed in the order of the parts
// A load from another SM's shared memory takes about a thousand clocks, so loads do not wait for one another: first one
// thread a row gathers the row's statistics, then D/4 threads a row its values, four parts at a time
// (a loop of dependent loads over the same: 16 heads of 64 queries over 512 keys in 20.4 us, 14.3 without dealing).
#pragma once
#include "umma.cuh"

namespace mgn {

constexpr int kMaxParts = 16;
constexpr uint32_t kPartsScratch = (kMaxParts + 2) * 128 * 4;

// Rows [first, last) of the tile, by the 256 threads t of named barrier `bar_id`.  stat(r, k, m, l): statistics of row r in
// part k (m = -inf: the part holds nothing that the row sees, and its O_k is not looked at).  O rows lie `pitch` bytes apart
// from `rows`, scratch is this CTA's; both addresses within a CTA.  emit(r, c, o, m, l): columns 4c .. 4c+3 of sum f_k O_k.
template <int D, typename Stat, typename Emit>
__device__ __forceinline__ void combine_parts(uint32_t rows, uint32_t pitch, uint32_t scratch, int parts, int first, int last, int t,
                                              uint32_t bar_id, Stat stat, Emit emit)
{
    constexpr int QUADS = D / 4;
    auto f_at = [&](int k, int r) { return scratch + (k * 128 + r) * 4; };
    for (int r = first + t; r < last; r += 256) {
        float m[kMaxParts], l[kMaxParts], top = -INFINITY, sum = 0.f;
#pragma unroll
        for (int k = 0; k < kMaxParts; ++k)
            if (k < parts) stat(r, k, m[k], l[k]);
#pragma unroll
        for (int k = 0; k < kMaxParts; ++k)
            if (k < parts) top = fmaxf(top, m[k]);
#pragma unroll
        for (int k = 0; k < kMaxParts; ++k)
            if (k < parts) {
                const bool none = m[k] == -INFINITY;
                const float f = ex2(m[k] - top);
                if (!none) sum = fmaf(l[k], f, sum);
                sts32(f_at(k, r), none ? -1.f : f);
            }
        sts32(f_at(kMaxParts, r), top);
        sts32(f_at(kMaxParts + 1, r), sum);
    }
    named_bar_sync(bar_id, 256);
    const int c = t % QUADS;
    for (int r = first + t / QUADS; r < last; r += 256 / QUADS) {
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k0 = 0; k0 < parts; k0 += 4) {
            float4 x[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = lds_cluster_128(cluster_map(rows + r * pitch + c * 16, min(k0 + e, parts - 1)));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (k0 + e >= parts) break;
                const float f = lds32f(f_at(k0 + e, r));
                if (f < 0.f) continue;
                o = make_float4(fmaf(x[e].x, f, o.x), fmaf(x[e].y, f, o.y), fmaf(x[e].z, f, o.z), fmaf(x[e].w, f, o.w));
            }
        }
        emit(r, c, o, lds32f(f_at(kMaxParts, r)), lds32f(f_at(kMaxParts + 1, r)));
    }
}

}  // namespace mgn
