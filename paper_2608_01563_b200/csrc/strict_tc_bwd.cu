// Strict backward on the tensor cores: dK + dV in one kernel, dQ in another (the split the paper lists in
// Section 3.3), f32 in and out, products as six bf16 partial products per f32 product (strict_tc.cuh).
// dK and dV, and dQ while one CTA walks over all keys of a query tile, are summed in a fixed order without
// floating-point atomics: bit-identical from run to run, and nothing has to be cleared first.  Where the keys of a tile
// are dealt to several CTAs (splits > 1), these add into a dQ that the caller has cleared, in no fixed order.  The price
// is that S and dP are formed twice (seven products per tile pair instead of five); a dQ partial formed beside dK and dV
// would need dS as a second, MN-major shared-memory operand of three parts, for which there is no room beside the split
// tiles.
//
// Both kernels: 512 threads, one CTA per SM.
//   warp 0   lane 0 issues the two score-shaped products      warp 1   lane 0 issues the row products
//   warps 2-4 and 5-7   split the two streamed tensors into shared memory (and stage row statistics)
//   warps 8-15          element-wise work: two threads per lane row, half of the columns each
// A wait costs an issuing lane more than an issue, so the conditions of a product share one barrier (see
// strict_tc_fwd.cu).  Results of the row products are added up in registers, tile by tile.
#include "strict_tc.cuh"

namespace mgn {
namespace {

using namespace stc;

constexpr int kThreads = 512, kBM = 128;
constexpr int kCompute = 256;
// 2 x 56 + 2 x 200 registers a thread over four warpgroups: the 512 that the CTA is launched with
constexpr int kRegsIssue = 56, kRegsCompute = 200;

// p = exp2(s - LSE log2 e): the row statistic as a sum of two floats.  P comes out larger by a share of 2 x 2^-24 (half
// of the largest error of the exponential), which gives back what the tensor core's truncation takes from the row
// products on average.
__device__ __forceinline__ void lse_log2(float lse, float& hi, float& lo) {
    constexpr float kLog2eLo = static_cast<float>(1.4426950408889634 - 1.4426950216293335);
    constexpr float kShare = static_cast<float>(2.0 * 0x1p-24 * 1.4426950408889634);
    hi = lse * kLog2e;
    lo = fmaf(lse, kLog2eLo, fmaf(lse, kLog2e, -hi)) - kShare;
}

// Flagged rows done again in plain f32 (see strict_tc.cuh).  Not inlined: the registers belong to the loops before it,
// and what a row needs is found again from the tile's first row (counted over all heads).
// dK and, where flagged in v_flags, dV rows over the queries of all G heads that see the key, into the exchange tiles.
template <int D>
__device__ __noinline__ void redo_dkv_rows(uint32_t flags, uint32_t v_flags, uint32_t ex, const float* Q, const float* K, const float* V,
                                           const float* dO, const float* LSE, const float* DELTA, size_t key0, int Sq, int Sk, int G,
                                           int causal, float scale)
{
    constexpr uint32_t PITCH = OwnRows<D>::PITCH;
    const int lane = threadIdx.x & 31;
    const size_t bhk = key0 / Sk;
    const int j0 = static_cast<int>(key0 - bhk * Sk);
    const float c2 = scale * kLog2e;
    for_flagged(flags, (static_cast<int>(threadIdx.x) >> 5) - 8, [&](uint32_t rows) {
        auto row = [&](int g) { return (rows >> (8 * g)) & 127u; };
        auto first = [&](int g) { return causal ? max(0, j0 + static_cast<int>(row(g)) - (Sk - Sq)) : 0; };     // query that sees it
        bool want_v[4];
        RowGroup<D> k, v, dk, dv;
        k.load(K + key0 * D, rows, lane);
        v.load(V + key0 * D, rows, lane);
        dk.clear();
        dv.clear();
#pragma unroll
        for (int g = 0; g < 4; ++g) want_v[g] = row_flagged(v_flags, row(g));
        // A query without an LSE makes every row that it sees NaN.
        const int from = first(0), to = max(max(first(0), first(1)), max(first(2), first(3)));  // rows rise: from is the least
        bool done = false;
        for (int g = 0; g < G; ++g)
            for (int i = to; i < Sq && !done; i += 32)
                done = __any_sync(0xffffffffu, isnan(__ldg(LSE + (bhk * G + g) * Sq + min(i + lane, Sq - 1))));
        if (done) {
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                dk.scale(g, NAN);
                dv.scale(g, NAN);
            }
        }
        for (int h = 0; h < G && !done; ++h) {
            const size_t head = (bhk * G + h) * Sq;
            for (int i = from; i < Sq && !done; i += 8) {
                const int n = min(8, Sq - i);
                const size_t at = head + i, mine = at + min(lane & 7, n - 1);
                const Streamed<D> q(Q + at * D, n, lane), d_o(dO + at * D, n, lane);
                const float p = ex2(fmaf(k.products(q, lane), c2, -(__ldg(LSE + mine) * kLog2e)));
                const float ds = p * (v.products(d_o, lane) - __ldg(DELTA + mine));
#pragma unroll
                for (int e = 0; e < 8; ++e)
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const float pe = __shfl_sync(0xffffffffu, p, 8 * g + e), se = __shfl_sync(0xffffffffu, ds, 8 * g + e);
                        if (i + e < first(g) || e >= n) continue;
                        dv.add(g, pe, d_o.r[e]);
                        dk.add(g, se, q.r[e]);
                    }
                bool nan = true;
#pragma unroll
                for (int g = 0; g < 4; ++g) nan = nan && dk.nan(g) && (dv.nan(g) || !want_v[g]);
                done = __all_sync(0xffffffffu, nan);
            }
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            dk.scale(g, scale);
            dk.store(g, ex, PITCH, rows, lane);
            if (want_v[g]) dv.store(g, ex + 128 * PITCH, PITCH, rows, lane);
        }
    });
}
// dQ rows over the keys of [j0, j1) that the query sees, into the exchange tile.
template <int D>
__device__ __noinline__ void redo_dq_rows(uint32_t flags, uint32_t ex, const float* Q, const float* K, const float* V, const float* dO,
                                          const float* LSE, const float* DELTA, size_t query0, int Sq, int Sk, int H, int G, int j0,
                                          int j1, int causal, float scale)
{
    const int lane = threadIdx.x & 31;
    const int bh = static_cast<int>(query0 / Sq), i0 = static_cast<int>(query0 - static_cast<size_t>(bh) * Sq);
    const size_t head = static_cast<size_t>((bh / H) * (H / G) + (bh % H) / G) * Sk;
    const float c2 = scale * kLog2e;
    for_flagged(flags, (static_cast<int>(threadIdx.x) >> 5) - 8, [&](uint32_t rows) {
        auto row = [&](int g) { return (rows >> (8 * g)) & 127u; };
        auto end = [&](int g) { return min(min(Sk, j1), causal ? i0 + static_cast<int>(row(g)) + Sk - Sq + 1 : Sk); };
        RowGroup<D> q, d_o, dq;
        q.load(Q + query0 * D, rows, lane);
        d_o.load(dO + query0 * D, rows, lane);
        dq.clear();
        const size_t mine = query0 + row(lane >> 3);
        const float lse2 = __ldg(LSE + mine) * kLog2e, delta = __ldg(DELTA + mine);
        const int to = end(3);                             // rows rise: the last one sees the most
        bool done = false;
        for (int j = j0; j < to && !done; j += 8) {
            const int n = min(8, to - j);
            const Streamed<D> k(K + (head + j) * D, n, lane), v(V + (head + j) * D, n, lane);
            const float p = ex2(fmaf(q.products(k, lane), c2, -lse2));
            const float ds = p * (d_o.products(v, lane) - delta);
#pragma unroll
            for (int e = 0; e < 8; ++e)
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float se = __shfl_sync(0xffffffffu, ds, 8 * g + e);
                    if (j + e < end(g)) dq.add(g, se, k.r[e]);
                }
            bool nan = true;
#pragma unroll
            for (int g = 0; g < 4; ++g) nan = nan && dq.nan(g);
            done = __all_sync(0xffffffffu, nan);
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            dq.scale(g, scale);
            dq.store(g, ex, OwnRows<D>::PITCH, rows, lane);
        }
    });
}

// ---------------------------------------------------------------------------------------------------------
// dK, dV.  A CTA owns 128 keys of one key/value head and walks over (query head of its group, query block);
// scores are transposed (lanes = keys).  Per block of R queries (c: the part of the score factor folded into Q):
//     S^T = K (c Q)^T    ->  P^T = exp2(S^T - LSE)       ->  dV += P^T dO
//     dP^T = V dO^T      ->  dS^T = P^T (dP^T - delta)   ->  dK += dS^T (c Q)
// While the element-wise warps form P^T(n) the tensor core runs dK(n-1) and dP^T(n), while they form dS^T(n)
// it runs dV(n) and S^T(n+1).  D = 64: K and V stay split in shared memory, blocks of 64 queries, all products
// stacked twice.  D = 128: V in tensor memory, K in shared memory, which leaves room for two stages of 32
// queries; scores are stacked three times, dK and dV results share one region.
template <int D>
struct KvCfg {
    static constexpr int R = D == 64 ? 64 : 32;
    static constexpr bool V_TMEM = D == 128, SHARED_Z = D == 128;
    static constexpr int ST = D == 64 ? 2 : 3, STZ = D == 64 ? 2 : 1;      // column sets of scores, of results
    static constexpr int STAGE = tile_bytes<D, R>();
    static constexpr int OFF_Q = 0, OFF_DO = 2 * STAGE, OFF_K = 4 * STAGE, OFF_V = OFF_K + tile_bytes<D, 128>();
    static constexpr int OFF_STAT = OFF_V + (V_TMEM ? 0 : tile_bytes<D, 128>());      // two stages of hi, lo, delta
    static constexpr int OFF_BAR = OFF_STAT + 2 * 3 * R * 4;
    static constexpr int SMEM = OFF_BAR + 256 + 1024;
    static_assert(SMEM <= 232448, "shared memory budget");
    static constexpr uint32_t X = x_cols<R, ST>();
    static constexpr uint32_t TM_V = 0, TM_X = V_TMEM ? 3 * D / 2 : 0, TM_Y = TM_X + X, TM_ZV = TM_Y + X,
                              TM_ZK = SHARED_Z ? TM_ZV : TM_ZV + STZ * D;
    static_assert(TM_ZK + STZ * D <= 512, "tensor memory budget");
    enum { S_GO = 0, P_GO = 2, V_GO = 4, K_GO = 6, S_DONE = 7, P_DONE = 8, V_DONE = 9, K_DONE = 10, KV = 12, COUNT = 13 };
};

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
strict_tc_dkv_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V,
                     const float* __restrict__ dO, const float* __restrict__ LSE, const float* __restrict__ DELTA,
                     float* __restrict__ dK, float* __restrict__ dV, int Sq, int Sk, int BHkv, int G, int Hg, int causal,
                     ScoreFactor c, float scale, unsigned* status)
{
    using C = KvCfg<D>;
    constexpr int R = C::R, HC = R / 2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* const smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t base = smem_u32(smem);
    const uint32_t bars = base + C::OFF_BAR, tmem_slot = bars + C::COUNT * 8;
    auto bar = [&](int i) { return bars + 8u * i; };
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    pdl_launch_dependents();                               // the dQ kernel may fill SMs as this one drains

    // First key blocks first: under a causal mask they see the most queries.
    int kb, bhk;
    item_of_block(static_cast<int>(blockIdx.x), (Sk + kBM - 1) / kBM, BHkv, Hg, kb, bhk);
    const int off = Sk - Sq;                               // causal: key j visible to query i iff j <= i + off
    const int j0 = kb * kBM;
    const int m0 = causal ? max(0, j0 - off) / R : 0;      // first query block that sees a key of this block
    const int n_m = (Sq + R - 1) / R - m0;
    const int n_blk = n_m * G;

    if (tid == 0) {
        for (int w = 0; w < 2; ++w) {
            mbar_init(bar(C::S_GO + w), kTeam + 1);           // Q split; P^T of the block before read
            mbar_init(bar(C::P_GO + w), kTeam + 1);           // dO split; dS^T of the block before read
            mbar_init(bar(C::V_GO + w), kTeam + kCompute);    // dO split; P^T written and the result region read
            mbar_init(bar(C::K_DONE + w), 1);
        }
        mbar_init(bar(C::K_GO), kCompute);                 // dS^T written and the result region read
        mbar_init(bar(C::S_DONE), 1);
        mbar_init(bar(C::P_DONE), 1);
        mbar_init(bar(C::V_DONE), 1);
        mbar_init(bar(C::KV), kCompute);
        fence_mbar_init();
    }
    __syncwarp();
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    if (tid == 32) sts32u(tmem_slot + 4, *reinterpret_cast<volatile unsigned*>(status));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, lds32u(tmem_slot), 0);
    if (lds32u(tmem_slot + 4) != 0) {                      // an earlier wait on this device gave up
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 512);
        return;
    }

    if (warp < 8) {
        reg_dealloc<kRegsIssue>();
        if (warp == 0) {
            const uint32_t leader = elect_one();       // the whole warp walks along, one lane issues
            // -------------------------------------------------------------- S^T and dP^T
            const uint64_t dQd = umma_smem_desc(base + C::OFF_Q, 16, 1024), dOd = umma_smem_desc(base + C::OFF_DO, 16, 1024);
            const uint64_t dKd = umma_smem_desc(base + C::OFF_K, 16, 1024);
            [[maybe_unused]] const uint64_t dVd = umma_smem_desc(base + C::OFF_V, 16, 1024);
            if (leader) mbar_arrive(bar(C::S_GO));
            if (leader) mbar_arrive(bar(C::P_GO));
            mbar_wait(bar(C::KV), 0, status);
#pragma unroll 1
            for (int n = 0; n < n_blk; ++n) {
                const int w = n & 1;
                const uint32_t ph = (n >> 1) & 1;
                const uint64_t so = static_cast<uint64_t>((w * C::STAGE) >> 4);
                mbar_wait(bar(C::S_GO + w), ph, status);
                tc_fence_after();
                issue_scores<true, D, R, C::ST>(leader, tmem + C::TM_X, dKd, dQd + so);
                umma_commit_warp(leader, bar(C::S_DONE));
                mbar_wait(bar(C::P_GO + w), ph, status);
                tc_fence_after();
                if constexpr (C::V_TMEM) issue_scores<false, D, R, C::ST>(leader, tmem + C::TM_Y, tmem + C::TM_V, dOd + so);
                else issue_scores<false, D, R, C::ST>(leader, tmem + C::TM_Y, dVd, dOd + so);
                umma_commit_warp(leader, bar(C::P_DONE));
            }
            __syncwarp();
        } else if (warp == 1) {
            const uint32_t leader = elect_one();       // the whole warp walks along, one lane issues
            // -------------------------------------------------------------- dV and dK results
            const uint64_t mQ = rows_desc<D, R>(base + C::OFF_Q), mO = rows_desc<D, R>(base + C::OFF_DO);
#pragma unroll 1
            for (int n = 0; n < n_blk; ++n) {
                const int w = n & 1;
                const uint64_t so = static_cast<uint64_t>((w * C::STAGE) >> 4);
                mbar_wait(bar(C::V_GO + w), (n >> 1) & 1, status);
                tc_fence_after();
                issue_rows<D, R, C::STZ>(leader, tmem + C::TM_ZV, tmem + C::TM_X, mO + so);
                umma_commit_warp(leader, bar(C::V_DONE));
                umma_commit_warp(leader, bar(C::S_GO + (w ^ 1)));
                mbar_wait(bar(C::K_GO), n & 1, status);
                tc_fence_after();
                issue_rows<D, R, C::STZ>(leader, tmem + C::TM_ZK, tmem + C::TM_Y, mQ + so);
                umma_commit_warp(leader, bar(C::K_DONE + w));       // both products of the block: its tiles are free too
                umma_commit_warp(leader, bar(C::P_GO + (w ^ 1)));
            }
            __syncwarp();
        } else {
            // ------------------------------------------------------------------ Q (and statistics), dO
            const bool is_q = warp < 5;
            const int t = tid - (is_q ? 64 : 160);
            const float* src = is_q ? Q : dO;
            const uint32_t stages = base + (is_q ? C::OFF_Q : C::OFF_DO);
            auto rows_of = [&](int n, int& g, int& i0) {   // n -> query head of the group, first query
                g = n / n_m;
                i0 = (m0 + n - g * n_m) * R;
            };
            Converter<D, R, true> cv(t, is_q ? c.hi : 1.f, is_q ? c.lo : 0.f);
            cv.run(n_blk,
                   [&](int n, int& rows) {
                       int g, i0;
                       rows_of(n, g, i0);
                       rows = Sq - i0;
                       return src + (static_cast<size_t>(bhk) * G + g) * Sq * D + static_cast<size_t>(i0) * D;
                   },
                   [&](int n) {
                       if (n >= 2) mbar_wait(bar(C::K_DONE + (n & 1)), ((n >> 1) & 1) ^ 1, status);
                       if (is_q) {
                           int g, i0;
                           rows_of(n, g, i0);
                           const size_t head = (static_cast<size_t>(bhk) * G + g) * Sq;
                           float* st = reinterpret_cast<float*>(smem + C::OFF_STAT) + (n & 1) * 3 * R;
                           if (t < R) {
                               float hi = INFINITY, lo = 0.f, dl = 0.f;       // past the end: P = 0
                               if (i0 + t < Sq) {
                                   lse_log2(__ldg(LSE + head + i0 + t), hi, lo);
                                   dl = __ldg(DELTA + head + i0 + t);
                               }
                               st[t] = -hi;
                               st[R + t] = -lo;
                               st[2 * R + t] = -dl;
                           }
                       }
                       return stages + (n & 1) * C::STAGE;
                   },
                   [&](int n) {
                       if (is_q) {
                           mbar_arrive(bar(C::S_GO + (n & 1)));
                       } else {
                           mbar_arrive(bar(C::P_GO + (n & 1)));
                           mbar_arrive(bar(C::V_GO + (n & 1)));
                       }
                   });
        }
    } else {
        // ------------------------------------------------------------------ element-wise
        reg_alloc<kRegsCompute>();
        const int h = (warp - 8) >> 2;                     // which half of the columns
        const int r = tid & 127;                           // key within the block = tensor-memory lane
        const uint32_t lane_base = static_cast<uint32_t>(r & ~31) << 16;
        const uint32_t tl = tmem + lane_base;
        const int j = j0 + r;
        const int t = tid - 256;
        const size_t own_at = (static_cast<size_t>(bhk) * Sk + j0) * D;
        {
            OwnRows<D> kr, vr;
            vr.load(V + own_at, Sk - j0, t);
            kr.load(K + own_at, Sk - j0, t);
            if constexpr (C::V_TMEM) {                     // by way of K's place
                vr.to_exchange(base + C::OFF_K, t);
                named_bar_sync(1, kCompute);
                OwnRows<D>::half_row_to_tmem(base + C::OFF_K, r, h, tl + C::TM_V);
                named_bar_sync(1, kCompute);
            } else {
                vr.to_tile(base + C::OFF_V, t);
            }
            kr.to_tile(base + C::OFF_K, t);
            fence_proxy_async_smem();
        }
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive(bar(C::KV));

        float accK[D / 2], accV[D / 2];
#pragma unroll
        for (int d = 0; d < D / 2; ++d) accK[d] = accV[d] = 0.f;
        auto add_result = [&](uint32_t z, float (&acc)[D / 2]) {
#pragma unroll
            for (int c = 0; c < D / 64; ++c) {
                float v[32];
                load_sets<32, C::STZ>(tl + z + h * (D / 2) + 32 * c, D, v);
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[32 * c + e] += v[e];
            }
            tc_fence_before();
        };

        const uint64_t pow2 = f2_pack(c.pow2, c.pow2);
        int m = 0;                                         // query block of the current head
#pragma unroll 1
        for (int n = 0; n < n_blk; ++n) {
            const uint32_t st = base + C::OFF_STAT + (n & 1) * 3 * R * 4 + h * HC * 4;
            const int i0 = (m0 + m) * R;
            if (++m == n_m) m = 0;
            const bool masked = causal && j0 + kBM - 1 > i0 + off;
            // ---- P^T
            mbar_wait(bar(C::S_DONE), n & 1, status);
            tc_fence_after();
            float p[HC];
            {
                uint32_t a[HC / 2], b[HC / 2], c[HC / 2];
                float s[HC];
                load_half<R, C::ST>(tl + C::TM_X, h, s);
#pragma unroll
                for (int e = 0; e < HC; e += 4) {
                    const U64x2 nh = lds128_pairs(st + e * 4), nl = lds128_pairs(st + R * 4 + e * 4);
                    float t0, t1, t2, t3;
                    f2_unpack(f2_add(f2_fma(f2_pack(s[e], s[e + 1]), pow2, nh.lo), nl.lo), t0, t1);
                    f2_unpack(f2_add(f2_fma(f2_pack(s[e + 2], s[e + 3]), pow2, nh.hi), nl.hi), t2, t3);
                    p[e] = ex2(t0);
                    p[e + 1] = ex2(t1);
                    p[e + 2] = ex2(t2);
                    p[e + 3] = ex2(t3);
                }
                if (masked) {
                    const int lim = j - off - i0 - h * HC;     // columns e >= lim see this key
#pragma unroll
                    for (int e = 0; e < HC; ++e)
                        if (e < lim) p[e] = 0.f;
                }
#pragma unroll
                for (int e = 0; e < HC; e += 2) split3(f2_pack(p[e], p[e + 1]), a[e / 2], b[e / 2], c[e / 2]);
                store_half_parts<R>(tl + C::TM_X, h, a, b, c);
            }
            if constexpr (C::SHARED_Z) {
                if (n > 0) {
                    mbar_wait(bar(C::K_DONE + ((n - 1) & 1)), ((n - 1) >> 1) & 1, status);
                    tc_fence_after();
                    add_result(C::TM_ZK, accK);
                }
            }
            tmem_st_wait();
            tc_fence_before();
            mbar_arrive(bar(C::V_GO + (n & 1)));
            if constexpr (!C::SHARED_Z) {
                if (n > 0) {
                    mbar_wait(bar(C::K_DONE + ((n - 1) & 1)), ((n - 1) >> 1) & 1, status);
                    tc_fence_after();
                    add_result(C::TM_ZK, accK);
                }
            }
            // ---- dS^T
            mbar_wait(bar(C::P_DONE), n & 1, status);
            tc_fence_after();
            {
                uint32_t a[HC / 2], b[HC / 2], c[HC / 2];
                float s[HC];
                load_half<R, C::ST>(tl + C::TM_Y, h, s);
#pragma unroll
                for (int e = 0; e < HC; e += 4) {
                    const U64x2 nd = lds128_pairs(st + 2 * R * 4 + e * 4);
                    split3(f2_mul(f2_pack(p[e], p[e + 1]), f2_add(f2_pack(s[e], s[e + 1]), nd.lo)),
                           a[e / 2], b[e / 2], c[e / 2]);
                    split3(f2_mul(f2_pack(p[e + 2], p[e + 3]), f2_add(f2_pack(s[e + 2], s[e + 3]), nd.hi)),
                           a[e / 2 + 1], b[e / 2 + 1], c[e / 2 + 1]);
                }
                store_half_parts<R>(tl + C::TM_Y, h, a, b, c);
            }
            if constexpr (!C::SHARED_Z) {
                tmem_st_wait();
                tc_fence_before();
                mbar_arrive(bar(C::K_GO));
            }
            mbar_wait(bar(C::V_DONE), n & 1, status);
            tc_fence_after();
            add_result(C::TM_ZV, accV);
            if constexpr (C::SHARED_Z) {
                tmem_st_wait();
                tc_fence_before();
                mbar_arrive(bar(C::K_GO));
            }
        }
        mbar_wait(bar(C::K_DONE + ((n_blk - 1) & 1)), ((n_blk - 1) >> 1) & 1, status);
        tc_fence_after();
        add_result(C::TM_ZK, accK);
        // every product has completed: the operand tiles are dead
        constexpr uint32_t EX = 128 * OwnRows<D>::PITCH;
        static_assert(2 * EX <= C::OFF_STAT, "two exchange tiles");
        const uint32_t ex = base + r * OwnRows<D>::PITCH + h * (D * 2), flags = tmem_slot + 8, v_flags = flags + 32;
        float bad_k = 0.f, bad_v = 0.f;                    // NaN once a result is not finite
#pragma unroll
        for (int d = 0; d < D / 2; ++d) {
            bad_k = fmaf(accK[d], 0.f, bad_k);
            bad_v = fmaf(accV[d], 0.f, bad_v);
        }
#pragma unroll
        for (int d = 0; d < D / 2; d += 4) {
            sts128f(ex + d * 4, accK[d] * c.grad * c.pow2, accK[d + 1] * c.grad * c.pow2, accK[d + 2] * c.grad * c.pow2,
                    accK[d + 3] * c.grad * c.pow2);
            sts128f(ex + EX + d * 4, accV[d], accV[d + 1], accV[d + 2], accV[d + 3]);
        }
        flag_rows(flags, warp - 8, j < Sk && (bad_k != 0.f || bad_v != 0.f));
        flag_rows(v_flags, warp - 8, bad_v != 0.f);
        named_bar_sync(1, kCompute);
        if (any_flagged(flags)) {
            redo_dkv_rows<D>(flags, v_flags, base, Q, K, V, dO, LSE, DELTA, own_at / D, Sq, Sk, G, causal, scale);
            named_bar_sync(1, kCompute);
        }
        OwnRows<D>::store(dK + own_at, Sk - j0, base, t);
        OwnRows<D>::store(dV + own_at, Sk - j0, base + EX, t);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------------------------------------
// dQ.  A CTA owns 128 query rows of one head (lanes = queries) and walks over key blocks of R keys:
//     S = (c Q) K^T,  dP = dO V^T   ->   dS = exp2(S - LSE) (dP - delta)   ->   dQ += dS K
// Two score regions, so that S(n+1) and dQ(n-1) run while the element-wise warps form dS(n).  D = 64: Q and dO
// split in shared memory, 64-key blocks.  D = 128: dO in tensor memory, 32-key blocks.
template <int D>
struct DqCfg {
    static constexpr int R = D == 64 ? 64 : 32;
    static constexpr bool DO_TMEM = D == 128;
    static constexpr int ST = 2, STZ = D == 64 ? 2 : 1;                    // column sets of scores, of results
    static constexpr int STAGE = tile_bytes<D, R>();
    static constexpr int OFF_K = 0, OFF_V = 2 * STAGE, OFF_Q = 4 * STAGE, OFF_DO = OFF_Q + tile_bytes<D, 128>();
    static constexpr int OFF_BAR = OFF_DO + (DO_TMEM ? 0 : tile_bytes<D, 128>());
    static constexpr int SMEM = OFF_BAR + 256 + 1024;
    static_assert(SMEM <= 232448, "shared memory budget");
    static constexpr uint32_t X = x_cols<R, ST>();
    static constexpr uint32_t TM_DO = 0, TM_X = DO_TMEM ? 3 * D / 2 : 0, TM_Y = TM_X + 2 * X, TM_Z = TM_Y + ST * R;
    static_assert(TM_Z + STZ * D <= 512, "tensor memory budget");
    enum { S_GO = 0, P_GO = 2, Q_GO = 4, S_DONE = 5, P_DONE = 7, Z_DONE = 8, QDO = 10, COUNT = 11 };
};

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
strict_tc_dq_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V,
                    const float* __restrict__ dO, const float* __restrict__ LSE, const float* __restrict__ DELTA,
                    float* __restrict__ dQ, int Sq, int Sk, int BH, int H, int G, int n_qt, int Hg, int splits, int causal,
                    ScoreFactor c, float scale, unsigned* status)
{
    using C = DqCfg<D>;
    constexpr int R = C::R, HC = R / 2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* const smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t base = smem_u32(smem);
    const uint32_t bars = base + C::OFF_BAR, tmem_slot = bars + C::COUNT * 8;
    auto bar = [&](int i) { return bars + 8u * i; };
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);

    // Heaviest (last) query tiles first when causal.
    const int item = static_cast<int>(blockIdx.x) / splits, part = static_cast<int>(blockIdx.x) % splits;
    int tile, bh;
    item_of_block(item, n_qt, BH, Hg, tile, bh);
    const int qt = n_qt - 1 - tile;
    const int bhk = (bh / H) * (H / G) + (bh % H) / G;     // key/value head of this query head
    const int off = Sk - Sq;                               // causal: key j visible to query i iff j <= i + off
    const int i0 = qt * kBM;
    const int i_last = min(i0 + kBM, Sq) - 1;
    // key blocks of this CTA: its share of those that the tile sees (the last share may be short, or empty)
    const int n_all = causal ? (i_last + off) / R + 1 : (Sk + R - 1) / R;
    const int share = (n_all + splits - 1) / splits, b0 = part * share;
    const int n_blk = min(share, n_all - b0);
    if (n_blk <= 0) {
        pdl_wait();
        return;
    }

    if (tid == 0) {
        for (int w = 0; w < 2; ++w) {
            mbar_init(bar(C::S_GO + w), kTeam + 1);           // K split; dS of two blocks back read
            mbar_init(bar(C::P_GO + w), kTeam + kCompute);    // V split; dP of the block before read
            mbar_init(bar(C::S_DONE + w), 1);
            mbar_init(bar(C::Z_DONE + w), 1);
        }
        mbar_init(bar(C::Q_GO), kCompute);                 // dS written and the last result read
        mbar_init(bar(C::P_DONE), 1);
        mbar_init(bar(C::QDO), kCompute);
        fence_mbar_init();
    }
    __syncwarp();
    if (warp == 0) tmem_alloc(tmem_slot, 512);
    if (tid == 32) sts32u(tmem_slot + 4, *reinterpret_cast<volatile unsigned*>(status));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, lds32u(tmem_slot), 0);
    if (lds32u(tmem_slot + 4) != 0) {                      // an earlier wait on this device gave up
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 512);
        pdl_wait();
        return;
    }

    if (warp < 8) {
        reg_dealloc<kRegsIssue>();
        if (warp == 0) {
            const uint32_t leader = elect_one();       // the whole warp walks along, one lane issues
            // -------------------------------------------------------------- S and dP
            const uint64_t dKd = umma_smem_desc(base + C::OFF_K, 16, 1024), dVd = umma_smem_desc(base + C::OFF_V, 16, 1024);
            const uint64_t dQd = umma_smem_desc(base + C::OFF_Q, 16, 1024);
            [[maybe_unused]] const uint64_t dOd = umma_smem_desc(base + C::OFF_DO, 16, 1024);
            if (leader) mbar_arrive(bar(C::S_GO));
            if (leader) mbar_arrive(bar(C::S_GO + 1));
            mbar_wait(bar(C::QDO), 0, status);
#pragma unroll 1
            for (int n = 0; n < n_blk; ++n) {
                const int w = n & 1;
                const uint32_t ph = (n >> 1) & 1;
                const uint64_t so = static_cast<uint64_t>((w * C::STAGE) >> 4);
                const uint32_t x = tmem + C::TM_X + w * C::X;
                mbar_wait(bar(C::S_GO + w), ph, status);
                tc_fence_after();
                issue_scores<true, D, R, C::ST>(leader, x, dQd, dKd + so);
                umma_commit_warp(leader, bar(C::S_DONE + w));
                mbar_wait(bar(C::P_GO + w), ph, status);
                tc_fence_after();
                if constexpr (C::DO_TMEM) issue_scores<false, D, R, C::ST>(leader, tmem + C::TM_Y, tmem + C::TM_DO, dVd + so);
                else issue_scores<false, D, R, C::ST>(leader, tmem + C::TM_Y, dOd, dVd + so);
                umma_commit_warp(leader, bar(C::P_DONE));
            }
            __syncwarp();
        } else if (warp == 1) {
            const uint32_t leader = elect_one();       // the whole warp walks along, one lane issues
            // -------------------------------------------------------------- dQ results
            const uint64_t mK = rows_desc<D, R>(base + C::OFF_K);
#pragma unroll 1
            for (int n = 0; n < n_blk; ++n) {
                const int w = n & 1;
                mbar_wait(bar(C::Q_GO), n & 1, status);
                tc_fence_after();
                issue_rows<D, R, C::STZ>(leader, tmem + C::TM_Z, tmem + C::TM_X + w * C::X,
                                    mK + static_cast<uint64_t>((w * C::STAGE) >> 4));
                umma_commit_warp(leader, bar(C::Z_DONE + w));       // S, dP (whose results it was formed from) and dQ: tiles free
                umma_commit_warp(leader, bar(C::S_GO + w));
            }
            __syncwarp();
        } else {
            // ------------------------------------------------------------------ K, V
            const bool is_k = warp < 5;
            const float* head = (is_k ? K : V) + static_cast<size_t>(bhk) * Sk * D;
            const uint32_t stages = base + (is_k ? C::OFF_K : C::OFF_V);
            const int go = is_k ? C::S_GO : C::P_GO;
            Converter<D, R> cv(tid - (is_k ? 64 : 160));
            cv.run(n_blk,
                   [&](int n, int& rows) {
                       rows = Sk - (b0 + n) * R;
                       return head + static_cast<size_t>(b0 + n) * R * D;
                   },
                   [&](int n) {
                       if (n >= 2) mbar_wait(bar(C::Z_DONE + (n & 1)), ((n >> 1) & 1) ^ 1, status);
                       return stages + (n & 1) * C::STAGE;
                   },
                   [&](int n) { mbar_arrive(bar(go + (n & 1))); });
        }
    } else {
        // ------------------------------------------------------------------ element-wise
        reg_alloc<kRegsCompute>();
        const int h = (warp - 8) >> 2;                     // which half of the columns
        const int r = tid & 127;                           // row within the tile = tensor-memory lane
        const uint32_t tl = tmem + (static_cast<uint32_t>(r & ~31) << 16);
        const int i = i0 + r;
        const bool row_ok = i < Sq;
        const int t = tid - 256;
        const size_t own_at = (static_cast<size_t>(bh) * Sq + i0) * D;
        mbar_arrive(bar(C::P_GO));                         // block 0 has no dP before it
        {
            OwnRows<D> qr, orr;
            orr.load(dO + own_at, Sq - i0, t);
            qr.load(Q + own_at, Sq - i0, t);
            if constexpr (C::DO_TMEM) {                    // by way of Q's place
                orr.to_exchange(base + C::OFF_Q, t);
                named_bar_sync(1, kCompute);
                OwnRows<D>::half_row_to_tmem(base + C::OFF_Q, r, h, tl + C::TM_DO);
                named_bar_sync(1, kCompute);
            } else {
                orr.to_tile(base + C::OFF_DO, t);
            }
            qr.scale(c.hi, c.lo);
            qr.to_tile(base + C::OFF_Q, t);
            fence_proxy_async_smem();
        }
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive(bar(C::QDO));

        float lse_hi = INFINITY, lse_lo = 0.f, dl = 0.f;   // past the end: P = 0
        if (row_ok) {
            lse_log2(__ldg(LSE + static_cast<size_t>(bh) * Sq + i), lse_hi, lse_lo);
            dl = __ldg(DELTA + static_cast<size_t>(bh) * Sq + i);
        }
        const uint64_t nh = f2_pack(-lse_hi, -lse_hi), nl = f2_pack(-lse_lo, -lse_lo), nd = f2_pack(-dl, -dl);
        const uint64_t pow2 = f2_pack(c.pow2, c.pow2);
        const int vis = min(Sk, causal ? i + off + 1 : Sk);    // keys this row sees
        float acc[D / 2];
#pragma unroll
        for (int d = 0; d < D / 2; ++d) acc[d] = 0.f;
        auto add_result = [&](int n) {
            mbar_wait(bar(C::Z_DONE + (n & 1)), (n >> 1) & 1, status);
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < D / 64; ++c) {
                float v[32];
                load_sets<32, C::STZ>(tl + C::TM_Z + h * (D / 2) + 32 * c, D, v);
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[32 * c + e] += v[e];
            }
        };

#pragma unroll 1
        for (int n = 0; n < n_blk; ++n) {
            const uint32_t x = tl + C::TM_X + (n & 1) * C::X;
            const int j0 = (b0 + n) * R;                   // first key of the block
            const bool masked = (causal && j0 + R - 1 > i0 + off) || j0 + R > Sk;
            float p[HC], s[HC];
            uint32_t a[HC / 2], b[HC / 2], c[HC / 2];
            mbar_wait(bar(C::S_DONE + (n & 1)), (n >> 1) & 1, status);
            tc_fence_after();
            load_half<R, C::ST>(x, h, s);
#pragma unroll
            for (int e = 0; e < HC; e += 2) {
                float t0, t1;
                f2_unpack(f2_add(f2_fma(f2_pack(s[e], s[e + 1]), pow2, nh), nl), t0, t1);
                p[e] = ex2(t0);
                p[e + 1] = ex2(t1);
            }
            if (masked) {
                const int lim = vis - j0 - h * HC;
#pragma unroll
                for (int e = 0; e < HC; ++e)
                    if (e >= lim) p[e] = 0.f;
            }
            mbar_wait(bar(C::P_DONE), n & 1, status);
            tc_fence_after();
            load_half<R, C::ST>(tl + C::TM_Y, h, s);
            tc_fence_before();
            mbar_arrive(bar(C::P_GO + ((n + 1) & 1)));     // dP of the next block may overwrite it
#pragma unroll
            for (int e = 0; e < HC; e += 2)
                split3(f2_mul(f2_pack(p[e], p[e + 1]), f2_add(f2_pack(s[e], s[e + 1]), nd)),
                       a[e / 2], b[e / 2], c[e / 2]);
            store_half_parts<R>(x, h, a, b, c);
            if (n > 0) add_result(n - 1);
            tmem_st_wait();
            tc_fence_before();
            mbar_arrive(bar(C::Q_GO));
        }
        add_result(n_blk - 1);
        // every product has completed: the operand tiles are dead
        const uint32_t ex = base + r * OwnRows<D>::PITCH + h * (D * 2), flags = tmem_slot + 8;
        float bad = 0.f;                                   // NaN once a result is not finite
#pragma unroll
        for (int d = 0; d < D / 2; ++d) bad = fmaf(acc[d], 0.f, bad);
#pragma unroll
        for (int d = 0; d < D / 2; d += 4)
            sts128f(ex + d * 4, acc[d] * scale, acc[d + 1] * scale, acc[d + 2] * scale, acc[d + 3] * scale);
        flag_rows(flags, warp - 8, row_ok && bad != 0.f);
        named_bar_sync(1, kCompute);
        if (any_flagged(flags)) {
            redo_dq_rows<D>(flags, base, Q, K, V, dO, LSE, DELTA, own_at / D, Sq, Sk, H, G, b0 * R, (b0 + n_blk) * R, causal, scale);
            named_bar_sync(1, kCompute);
        }
        if (splits == 1) OwnRows<D>::store(dQ + own_at, Sq - i0, base, t);
        else OwnRows<D>::add(dQ + own_at, Sq - i0, base, t);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
    pdl_wait();     // this grid must not complete before the one it may have started beside
}

template <int D>
cudaError_t launch(const Problem& p, const float* q, const float* k, const float* v, const float* d_o, const float* lse,
                   const float* delta, float* dq, float* dk, float* dv, int dq_splits, unsigned* status, cudaStream_t st)
{
    using KC = KvCfg<D>;
    using QC = DqCfg<D>;
    auto kv = strict_tc_dkv_kernel<D>;
    auto dqk = strict_tc_dq_kernel<D>;
    cudaError_t e = cudaFuncSetAttribute(kv, cudaFuncAttributeMaxDynamicSharedMemorySize, KC::SMEM);
    if (e != cudaSuccess) return MGN_FAIL(e, "strict_tc_dkv attributes");
    e = cudaFuncSetAttribute(dqk, cudaFuncAttributeMaxDynamicSharedMemorySize, QC::SMEM);
    if (e != cudaSuccess) return MGN_FAIL(e, "strict_tc_dq attributes");
    const long long kv_blocks = static_cast<long long>((p.Sk + kBM - 1) / kBM) * p.BHkv();
    const int n_qt = (p.Sq + kBM - 1) / kBM;
    const long long dq_blocks = static_cast<long long>(n_qt) * p.BH() * dq_splits;
    if (kv_blocks > 0x7fffffffLL || dq_blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const ScoreFactor c = score_factor(p.scale, D);
    kv<<<static_cast<unsigned>(kv_blocks), kThreads, KC::SMEM, st>>>(q, k, v, d_o, lse, delta, dk, dv, p.Sq, p.Sk, p.BHkv(),
                                                                     p.group(), head_group(8.0 * p.Sq * D * p.group(), p.BHkv()), p.causal, c, p.scale, status);
    e = cudaGetLastError();
    if (e != cudaSuccess) return MGN_FAIL(e, "strict_tc_dkv launch");
    return MGN_FAIL(launch_pdl(dqk, static_cast<unsigned>(dq_blocks), kThreads, QC::SMEM, st, q, k, v, d_o, lse, delta, dq, p.Sq,
                               p.Sk, p.BH(), p.H, p.group(), n_qt,
                               head_group(8.0 * p.Sk * D / p.group(), p.BH()), dq_splits, p.causal, c, p.scale, status),
                    "strict_tc_dq launch");
}

}  // namespace

cudaError_t launch_strict_tc_bwd(const Problem& p, const float* q, const float* k, const float* v, const float* d_o,
                                 const float* lse, const float* delta, float* dq, float* dk, float* dv, int dq_splits, unsigned* status,
                                 cudaStream_t st)
{
    return p.D == 64 ? launch<64>(p, q, k, v, d_o, lse, delta, dq, dk, dv, dq_splits, status, st)
                     : launch<128>(p, q, k, v, d_o, lse, delta, dq, dk, dv, dq_splits, status, st);
}

}  // namespace mgn
