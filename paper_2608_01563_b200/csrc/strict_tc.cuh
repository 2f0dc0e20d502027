// Strict (f32) products on the tensor cores: every f32 operand is split into three bf16 parts,
//     x = hi + mid + lo,   hi = bf16(x), mid = bf16(x - hi), lo = bf16(x - hi - mid),
// which together hold all 24 significant bits (the differences are exact in f32, the parts have f32's
// exponent range), and a product of two operands is the sum of the six partial products
//     lo*hi + hi*lo + mid*mid + mid*hi + hi*mid + hi*hi
// accumulated in f32.  What is left out (mid*lo, lo*mid, lo*lo) is at most 2^-24 of the product.  The tensor core adds
// into its accumulator with truncation, so chains are kept short: scores and dP over the D columns, row products over
// the R rows of one tile, results added up tile by tile in registers, rounded to nearest, where an FFMA kernel would
// chain its whole contraction.  Within a chain the small products come first, and the hi*hi products of a score have a
// column set to themselves (see term()).
//
// Operand tiles: R rows of D values in D/64 blocks of 64 columns, each block one part after the other
// (128-byte lines, 128-byte swizzle); the same tile serves as K-major and as MN-major operand.
//
// A 16-deep step of 128 rows takes about 50 clocks for 32 and for 64 columns, 64 to 72 for 128: its A operand
// has to be fetched whatever the width.  So steps are made wider by running one part of A against two or
// three adjacent parts of B at once ("stacked": 64 rows of hi followed by 64 rows of mid are a 128-row B
// operand); the column sets that come out are added in registers.  Stacked scores of 64 rows cost four
// steps of 228 clocks together per 16 columns of D instead of six of 300.  f32 tensors are read with plain 16-byte
// loads and split by converter warps.
//   The warp that issues walks along in step and one elected lane issues: with a single lane in a branch of its own the
// operands of every step went from that lane's registers to the uniform ones first, and a step took 80 to 110 clocks.
// Forward and backward, in us: (8,12,1024,64) causal 484 -> 458, (32,12,197,64) 281 -> 259, (4,32,1024,128) causal
// 1259 -> 1152.
#pragma once
#include "fast_items.cuh"
#include "kernels.h"
#include "umma.cuh"

namespace mgn {
namespace stc {

constexpr float kLog2e = 1.4426950408889634f;   // 1.4426950216293335 as a float
constexpr float kLn2 = 0.6931471805599453f, kLn2Lo = static_cast<float>(0.6931471805599453 - 0.6931471824645996);

// The factor between a product q k and a score in the log2 domain, c = scale log2 e (1 + bias): hi + lo is folded into
// Q before it is split, the power of two `pow2` multiplies the finished scores (exact, in the FMA that subtracts the
// row's reference).  pow2 takes the exponent of a factor below one, which would push c Q of a small scale to where its
// lower parts vanish (|scale| = 1e-36 over keys of 1e36); a large factor stays with Q, where it may lift a small Q.
//   The tensor core's truncation makes a score smaller by a fixed share on average -- measured on single-key problems,
// where LSE is the score: 0.93 x 2^-24 over 64 columns, 1.65 x 2^-24 over 128 -- which the bias gives back.
//   grad: what sums over the scaled Q are multiplied by, besides pow2, for sums over scale Q.
struct ScoreFactor { float hi, lo, pow2, grad; };
inline ScoreFactor score_factor(float scale, int D) {
    const double log2e = 1.4426950408889634 * (1.0 + (D == 64 ? 0.93 : 1.65) * 0x1p-24);
    int e = 0;
    double c = frexp(scale * log2e, &e);                   // in [0.5, 1)
    if (e > 0) {
        c = ldexp(c, e);
        e = 0;
    }
    const float hi = static_cast<float>(c);
    return {hi, static_cast<float>(c - hi), static_cast<float>(ldexp(1.0, e)), static_cast<float>(1.0 / log2e)};
}

// x * (c_hi + c_lo), rounded once.
__device__ __forceinline__ float scaled(float x, float c_hi, float c_lo) { return fmaf(x, c_hi, x * c_lo); }
__device__ __forceinline__ float4 scaled(float4 x, float c_hi, float c_lo) {
    return make_float4(scaled(x.x, c_hi, c_lo), scaled(x.y, c_hi, c_lo), scaled(x.z, c_hi, c_lo), scaled(x.w, c_hi, c_lo));
}

// A pair of f32 (a in the low half) -> three packed bf16 pairs.  hi saturates: a finite x near the end of the range
// (-3.4028e38 is a usual mask constant) keeps finite parts, the rest of it goes into mid; an infinite x gives
// (largest, infinite, NaN) and with that NaN in every product.
__device__ __forceinline__ void split3(uint64_t x, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    const uint64_t minus1 = f2_pack(-1.f, -1.f);
    float a, b;
    f2_unpack(x, a, b);
    hi = pack_bf16_sat(a, b);
    x = f2_fma(f2_pack(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), minus1, x);
    f2_unpack(x, a, b);
    mid = pack_bf16(a, b);
    x = f2_fma(f2_pack(__uint_as_float(mid << 16), __uint_as_float(mid & 0xffff0000u)), minus1, x);
    f2_unpack(x, a, b);
    lo = pack_bf16(a, b);
}

template <int R> __host__ __device__ constexpr uint32_t part_bytes() { return R * 128; }          // of one 64-column block
template <int R> __host__ __device__ constexpr uint32_t block_bytes() { return 3 * R * 128; }     // a 64-column block
template <int D, int R> __host__ __device__ constexpr uint32_t tile_bytes() { return D / 64 * 3 * R * 128; }

// Four consecutive f32 of a row -> the 8-byte pieces of the three parts of a split tile of R rows.  `at` is where
// the hi piece goes.
template <int R>
__device__ __forceinline__ uint32_t quad_offset(int r, int quad) {
    return (quad >> 4) * block_bytes<R>() + r * 128 + ((((quad >> 1) & 7) ^ (r & 7)) << 4) + (quad & 1) * 8;
}
template <int R>
__device__ __forceinline__ void store_quad(uint32_t at, const float4 x) {
    uint32_t h[2], m[2], l[2];
    split3(f2_pack(x.x, x.y), h[0], m[0], l[0]);
    split3(f2_pack(x.z, x.w), h[1], m[1], l[1]);
    sts64(at, h[0], h[1]);
    sts64(at + part_bytes<R>(), m[0], m[1]);
    sts64(at + 2 * part_bytes<R>(), l[0], l[1]);
}

// A team of kTeam threads turns a stream of R x D f32 tiles into split operand tiles, 2048 values at a time
// (a slot): six 16-byte quads a thread, each replaced by the same quad of the next slot as soon as it has
// been split and stored, so that global latency is covered by a whole slot of work.
// The loop is rolled over slots on purpose: every role of these kernels runs its own code on each scheduler,
// and larger unrolled bodies made instruction fetch the top stall (5.3 stalled warps per issue).  Staging the
// f32 values in shared memory is slower: a load from there queues behind the tensor core's operand traffic
// (512 queries over 4096 keys, D = 128: forward 0.239 ms against 0.169).
constexpr int kTeam = 96;

template <int D, int R, bool SCALED = false>
struct Converter {
    static constexpr int QUADS = D / 4;                                             // 16-byte quads of a row
    static constexpr int SLOT_ROWS = 2048 / D, SLOTS = R / SLOT_ROWS, STEP = kTeam / QUADS;
    static constexpr int NQ = (SLOT_ROWS + STEP - 1) / STEP;                        // quads of a thread in a slot
    static_assert(R % SLOT_ROWS == 0 && kTeam % QUADS == 0 && SLOT_ROWS % 8 == 0, "");

    float4 buf[NQ];
    uint32_t off[NQ];         // where they go in a slot of an operand tile
    int row, quad;
    float c_hi, c_lo;         // SCALED: what the values are multiplied by

    __device__ __forceinline__ explicit Converter(int t, float hi = 1.f, float lo = 0.f)
        : row(t / QUADS), quad(t % QUADS), c_hi(hi), c_lo(lo) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            off[k] = quad_offset<R>(row + k * STEP, quad);
        }
    }
    // Converts tiles 0 .. n-1.  src(i, rows) gives the first row of tile i and how many rows exist from there;
    // dst(i) waits until the tile's stage is free and returns its address; done(i) follows the stores.
    template <class Src, class Dst, class Done>
    __device__ __forceinline__ void run(int n, Src src, Dst dst, Done done) {
        int rows;
        const float* g = src(0, rows) + row * D + quad * 4;
        auto load = [&](int k) {
            const int r = row + k * STEP;
            buf[k] = r < min(rows, SLOT_ROWS) ? __ldg(reinterpret_cast<const float4*>(g + k * STEP * D))
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
        };
#pragma unroll
        for (int k = 0; k < NQ; ++k) load(k);
        uint32_t d = 0;
        int sl = 0, i = 0;
#pragma unroll 1
        while (i < n) {
            if (sl == 0) d = dst(i);
            if (sl == SLOTS - 1) {                       // the next slot is the first of the next tile
                if (i + 1 < n) g = src(i + 1, rows) + row * D + quad * 4;
                else rows = 0;
            } else {
                g += SLOT_ROWS * D;
                rows -= SLOT_ROWS;
            }
#pragma unroll
            for (int k = 0; k < NQ; ++k) {
                if (row + k * STEP < SLOT_ROWS) {
                    if constexpr (SCALED) buf[k] = scaled(buf[k], c_hi, c_lo);
                    store_quad<R>(d + off[k], buf[k]);
                }
                load(k);
            }
            d += SLOT_ROWS * 128;
            if (++sl == SLOTS) {
                fence_proxy_async_smem();
                done(i);
                ++i;
                sl = 0;
            }
        }
    }
};

// The 128 rows of D f32 that a CTA owns, read and written by its 256 element-wise threads (t) as 16-byte quads
// in row order: a thread per row instead touches 32 lines with each load or store, which alone took 4000
// clocks per tensor and CTA (dK+dV of a 197-token head: 10000 clocks to the first split tile, 5500 after the
// last product, of 41000).
template <int D>
struct OwnRows {
    static constexpr int NQ = 128 * D / 4 / 256, PITCH = D * 4 + 16;     // bytes of a row in the exchange tile
    float4 q[NQ];
    // src: the first row, of which `rows` exist
    __device__ __forceinline__ void load(const float* src, int rows, int t) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            const int u = t + 256 * k, r = u / (D / 4), c = u % (D / 4);
            q[k] = r < rows ? __ldg(reinterpret_cast<const float4*>(src + r * D + 4 * c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __device__ __forceinline__ void scale(float c_hi, float c_lo) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) q[k] = scaled(q[k], c_hi, c_lo);
    }
    // into a split tile of 128 rows
    __device__ __forceinline__ void to_tile(uint32_t tile, int t) const {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            const int u = t + 256 * k;
            store_quad<128>(tile + quad_offset<128>(u / (D / 4), u % (D / 4)), q[k]);
        }
    }
    // into the exchange tile
    __device__ __forceinline__ void to_exchange(uint32_t ex, int t) const {
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            const int u = t + 256 * k;
            sts128f(ex + (u / (D / 4)) * PITCH + (u % (D / 4)) * 16, q[k].x, q[k].y, q[k].z, q[k].w);
        }
    }
    // from the exchange tile to global memory
    static __device__ __forceinline__ void store(float* dst, int rows, uint32_t ex, int t) {
#pragma unroll 4
        for (int k = 0; k < NQ; ++k) {
            const int u = t + 256 * k, r = u / (D / 4), c = u % (D / 4);
            if (r < rows) *reinterpret_cast<float4*>(dst + r * D + 4 * c) = lds128(ex + r * PITCH + c * 16);
        }
    }
    // the same, added to what is there
    static __device__ __forceinline__ void add(float* dst, int rows, uint32_t ex, int t) {
#pragma unroll 4
        for (int k = 0; k < NQ; ++k) {
            const int u = t + 256 * k, r = u / (D / 4), c = u % (D / 4);
            const float4 x = lds128(ex + r * PITCH + c * 16);
            if (r < rows) red_add_v4(dst + r * D + 4 * c, x.x, x.y, x.z, x.w);
        }
    }
    // half h of row r of the exchange tile, split into tensor memory: part a at columns t + a * D / 2
    static __device__ __forceinline__ void half_row_to_tmem(uint32_t ex, int r, int h, uint32_t tm) {
#pragma unroll 1
        for (int c = 0; c < D / 64; ++c) {
            uint32_t p0[16], p1[16], p2[16];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 x = lds128(ex + r * PITCH + h * (D * 2) + c * 128 + e * 16);
                split3(f2_pack(x.x, x.y), p0[2 * e], p1[2 * e], p2[2 * e]);
                split3(f2_pack(x.z, x.w), p0[2 * e + 1], p1[2 * e + 1], p2[2 * e + 1]);
            }
            const uint32_t at = tm + h * (D / 4) + 16 * c;
            tmem_st16(at, p0);
            tmem_st16(at + D / 2, p1);
            tmem_st16(at + D, p2);
        }
    }
};

// The partial products as issued.  A term: part of A, first part of B, how many adjacent parts of B it runs
// against, and the column set that its first one goes to.
//  - Scores (the exponent of P): hi hi has a set of its own.  The forward and both backward kernels then round
//    a score alike whichever operand is A, and P = exp(s - LSE) is as good as a difference of two equally
//    rounded numbers even where both are large; with hi mid and mid hi split between the sets by operand, a
//    row that attends to one key (scores near 130 in the log2 domain) had 2.5e-5 of error in P instead of 8e-6.
//  - Everything else: smallest first, hi hi last.
struct Term { uint32_t a, b, n, set; };
template <bool SCORE, int ST> __device__ __forceinline__ Term term(int t) {
    if constexpr (SCORE && ST == 2) {        // hi [hi mid], mid hi, mid mid, lo hi, hi lo
        return {(0x02110u >> (4 * t)) & 3u, (0x20100u >> (4 * t)) & 3u, (0x11112u >> (4 * t)) & 3u, (0x11110u >> (4 * t)) & 3u};
    } else if constexpr (SCORE) {            // hi [hi mid lo], mid [hi mid], lo hi
        return {(0x210u >> (4 * t)) & 3u, 0u, (0x123u >> (4 * t)) & 3u, (0x210u >> (4 * t)) & 3u};
    } else if constexpr (ST == 1) {          // lo hi, hi lo, mid mid, mid hi, hi mid, hi hi
        return {(0x001102u >> (4 * t)) & 3u, (0x010120u >> (4 * t)) & 3u, 1u, 0u};
    } else if constexpr (ST == 2) {          // mid [hi mid], lo hi, hi lo, hi [hi mid]
        return {(0x0021u >> (4 * t)) & 3u, (0x0200u >> (4 * t)) & 3u, (0x2112u >> (4 * t)) & 3u, (0x0100u >> (4 * t)) & 3u};
    } else {                                 // mid [hi mid lo], lo hi, hi [hi mid lo]
        return {(0x021u >> (4 * t)) & 3u, 0u, (0x313u >> (4 * t)) & 3u, 0u};
    }
}
template <bool SCORE, int ST> __device__ constexpr int n_terms() {
    return SCORE && ST == 2 ? 5 : ST == 1 ? 6 : ST == 2 ? 4 : 3;
}

// A region of tensor memory that receives rows of N values in ST column sets (two or three) and is later overwritten
// by the three packed parts of what is formed from them.  The N/2 values of a half are worked on by one thread (or
// in one go) and its parts stay within the columns that held those values, so a half never overwrites values of the
// other half.
template <int N, int ST> __host__ __device__ constexpr uint32_t x_cols() { return ST * N; }
template <int N> __host__ __device__ constexpr uint32_t x_half_part_col(int half, int part) {
    return part == 2 ? N + half * (N / 2) : half * (N / 2) + part * (N / 4);
}
// columns of 16-value contraction step kk
template <int N> __device__ __forceinline__ uint32_t x_part_col(uint32_t part, int kk) {
    constexpr int SPH = N / 32;                          // steps per half
    return x_half_part_col<N>(kk / SPH, part) + (kk % SPH) * 8;
}

template <int N> __device__ __forceinline__ void tmem_load(uint32_t t, uint32_t (&v)[N]) {
    static_assert(N == 16 || N == 32, "");
    if constexpr (N == 32) tmem_ld32(t, v);
    else tmem_ld16(t, v);
}
// W f32 columns of this thread's lane, summed over ST sets `stride` columns apart (the hi hi set last).
template <int W, int ST> __device__ __forceinline__ void load_sets(uint32_t t, uint32_t stride, float (&v)[W]) {
    uint32_t s[ST][W];
#pragma unroll
    for (int i = 0; i < ST; ++i) tmem_load<W>(t + i * stride, s[i]);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < W; e += 2) {
        uint64_t x = f2_pack(__uint_as_float(s[ST - 1][e]), __uint_as_float(s[ST - 1][e + 1]));
#pragma unroll
        for (int i = ST - 2; i >= 0; --i) x = f2_add(x, f2_pack(__uint_as_float(s[i][e]), __uint_as_float(s[i][e + 1])));
        f2_unpack(x, v[e], v[e + 1]);
    }
}
// The values of one half of a region's row.
template <int N, int ST> __device__ __forceinline__ void load_half(uint32_t x, int half, float (&v)[N / 2]) {
    load_sets<N / 2, ST>(x + half * (N / 2), N, v);
}
// The packed parts of a half row (N/2 values) into its columns.
template <int N> __device__ __forceinline__ void store_half_parts(uint32_t x, int half, const uint32_t (&h)[N / 4],
                                                                          const uint32_t (&m)[N / 4], const uint32_t (&l)[N / 4]) {
    if constexpr (N == 64) {
        tmem_st16(x + x_half_part_col<N>(half, 0), h);
        tmem_st16(x + x_half_part_col<N>(half, 1), m);
        tmem_st16(x + x_half_part_col<N>(half, 2), l);
    } else {
        tmem_st8(x + x_half_part_col<N>(half, 0), h);
        tmem_st8(x + x_half_part_col<N>(half, 1), m);
        tmem_st8(x + x_half_part_col<N>(half, 2), l);
    }
}

// Unrolled over terms and steps: with uniform operands they are constants and a step is few instructions (forward and
// backward, terms rolled / unrolled: (8,12,1024,64) causal 449 / 444 us, (32,12,197,64) 258 / 254, (4,32,1024,128) causal
// 1134 / 1125).
// Sets of D[128 x R] = A B^T over D columns, at tensor-memory column d; B a split tile of R rows.  A in tensor
// memory (part p at a + p * D / 2) or a split tile of 128 rows (a: its descriptor).  SCORE: see term().
template <bool SCORE, int D, int R, int ST, typename A>
__device__ __forceinline__ void issue_scores(uint32_t leader, uint32_t d, A a_at, uint64_t b_desc) {
#pragma unroll
    for (int t = 0; t < n_terms<SCORE, ST>(); ++t) {
        const Term m = term<SCORE, ST>(t);
        const uint32_t idesc = umma_idesc_bf16(128, R, false, false) + (m.n - 1) * ((R >> 3) << 17);
        const uint64_t b = desc_at(b_desc, m.b * part_bytes<R>());
        const uint32_t dt = d + m.set * R;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
            const uint64_t bk = desc_at(b, (kk >> 2) * block_bytes<R>() + (kk & 3) * 32);
            const uint32_t add = (t > 0 || kk > 0) ? 1u : 0u;
            if constexpr (sizeof(A) == 4) umma_ts_warp(leader, dt, a_at + m.a * (D / 2) + kk * 8, bk, idesc, add);
            else umma_ss_warp(leader, dt, desc_at(a_at, m.a * part_bytes<128>() + (kk >> 2) * block_bytes<128>() + (kk & 3) * 32), bk, idesc, add);
        }
    }
}
// Sets of D[128 x D] = X B over the R rows of the split tile B (as MN-major operand, see rows_desc), X the parts
// in a region of scores.  Stacking (ST = 2) needs adjacent parts to be D columns apart: D = 64.
template <int D, int R> __device__ __forceinline__ uint64_t rows_desc(uint32_t tile) {
    return umma_smem_desc(tile, D == 64 ? part_bytes<R>() : block_bytes<R>(), 1024);
}
template <int D, int R, int ST>
__device__ __forceinline__ void issue_rows(uint32_t leader, uint32_t d, uint32_t x, uint64_t b_desc) {
    static_assert(ST == 1 || D == 64, "");
#pragma unroll
    for (int t = 0; t < n_terms<false, ST>(); ++t) {
        const Term m = term<false, ST>(t);
        const uint32_t idesc = umma_idesc_bf16(128, D, false, true) + (m.n - 1) * ((D >> 3) << 17);
        const uint64_t b = desc_at(b_desc, m.b * part_bytes<R>());
        const uint32_t dt = d + m.set * D;
#pragma unroll
        for (int kk = 0; kk < R / 16; ++kk)
            umma_ts_warp(leader, dt, x + x_part_col<R>(m.a, kk), desc_at(b, kk * 2048), idesc, (t > 0 || kk > 0) ? 1u : 0u);
    }
}

// ---------------------------------------------------------------------------------------------------------
// Rows done again in plain f32.  An infinite or NaN operand, or partial products that overflow with opposite signs
// (finite operands near 1e25 on both sides), leave NaN where f32 arithmetic has an infinity of one sign or nothing at
// all, so rows of results that are not finite are formed once more from the f32 tensors, over visible pairs only.
// The eight element-wise warps take up to four rows at a time and walk over eight streamed rows a step, so that a
// row fetched from L2 serves four: (1,4,4096,128) with one key at -inf, where no row of the backward is finite,
// 3.7 ms (11.3 with one row a warp; 2.2 FFMA kernels; 0.76 for finite inputs).  In a step lane 8 g + e holds the pair (row g of
// the group, streamed row e); in rows, a lane holds columns [lane D/32, (lane+1) D/32).
template <int D> struct Cols { float x[D / 32]; };
template <int D> __device__ __forceinline__ Cols<D> load_cols(const float* row, int lane) {
    Cols<D> c;
    if constexpr (D == 64) {
        const float2 t = __ldg(reinterpret_cast<const float2*>(row) + lane);
        c.x[0] = t.x; c.x[1] = t.y;
    } else {
        const float4 t = __ldg(reinterpret_cast<const float4*>(row) + lane);
        c.x[0] = t.x; c.x[1] = t.y; c.x[2] = t.z; c.x[3] = t.w;
    }
    return c;
}
// Eight streamed rows, n (1..8) of them there; the last one repeats.
template <int D> struct Streamed {
    Cols<D> r[8];
    __device__ __forceinline__ Streamed(const float* rows, int n, int lane) {
#pragma unroll
        for (int e = 0; e < 8; ++e) r[e] = load_cols<D>(rows + min(e, n - 1) * D, lane);
    }
};
// Four rows, one for each byte of `rows` (its number within the tile).
template <int D> struct RowGroup {
    Cols<D> c[4];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int e = 0; e < D / 32; ++e) c[g].x[e] = 0.f;
    }
    __device__ __forceinline__ void load(const float* tile, uint32_t rows, int lane) {
#pragma unroll
        for (int g = 0; g < 4; ++g) c[g] = load_cols<D>(tile + ((rows >> (8 * g)) & 127u) * D, lane);
    }
    // row g += w * b
    __device__ __forceinline__ void add(int g, float w, const Cols<D>& b) {
#pragma unroll
        for (int e = 0; e < D / 32; ++e) c[g].x[e] = fmaf(w, b.x[e], c[g].x[e]);
    }
    __device__ __forceinline__ void scale(int g, float f) {
#pragma unroll
        for (int e = 0; e < D / 32; ++e) c[g].x[e] *= f;
    }
    // this lane's columns of row g are all NaN: nothing can change them
    __device__ __forceinline__ bool nan(int g) const {
        bool r = true;
#pragma unroll
        for (int e = 0; e < D / 32; ++e) r = r && isnan(c[g].x[e]);
        return r;
    }
    // row g into an exchange tile whose rows are `pitch` bytes apart
    __device__ __forceinline__ void store(int g, uint32_t tile, uint32_t pitch, uint32_t rows, int lane) const {
        const uint32_t at = tile + ((rows >> (8 * g)) & 127u) * pitch + lane * (D / 8);
#pragma unroll
        for (int e = 0; e < D / 32; ++e) sts32(at + 4 * e, c[g].x[e]);
    }
    // Lane 8 g + e: row g times streamed row e.  Thirty-two partial sums a lane are reduced across the warp and dealt to
    // the lanes in one exchange of 16 + 8 + 4 + 2 + 1 values.
    __device__ __forceinline__ float products(const Streamed<D>& b, int lane) const {
        float s[32];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                s[8 * g + r] = c[g].x[0] * b.r[r].x[0];
#pragma unroll
                for (int e = 1; e < D / 32; ++e) s[8 * g + r] = fmaf(c[g].x[e], b.r[r].x[e], s[8 * g + r]);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int r = 0; r < o; ++r) {
                const float keep = up ? s[r + o] : s[r], send = up ? s[r] : s[r + o];
                s[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        return s[0];
    }
};
// A thread's flag for its row (the halves of a row may differ), as eight words in shared memory, one a warp.
__device__ __forceinline__ void flag_rows(uint32_t words, int warp8, bool flag) {
    const uint32_t word = __ballot_sync(0xffffffffu, flag);
    if ((threadIdx.x & 31) == 0) sts32u(words + 4 * warp8, word);
}
__device__ __forceinline__ uint32_t flagged_rows(uint32_t words, int w) { return lds32u(words + 4 * w) | lds32u(words + 16 + 4 * w); }
__device__ __forceinline__ bool row_flagged(uint32_t words, uint32_t row) { return (flagged_rows(words, row >> 5) >> (row & 31)) & 1u; }
__device__ __forceinline__ bool any_flagged(uint32_t words) {
    uint32_t m = 0;
#pragma unroll
    for (int w = 0; w < 4; ++w) m |= flagged_rows(words, w);
    return m != 0;
}
// Flagged rows, dealt to the eight warps one by one and handed over in fours (the last row of a short four repeats).
template <class Four> __device__ __forceinline__ void for_flagged(uint32_t words, int warp8, Four four) {
    uint32_t rows = 0;
    int n = 0, seen = 0;
    for (int w = 0; w < 4; ++w)
        for (uint32_t m = flagged_rows(words, w); m != 0; m &= m - 1) {
            if ((seen++ & 7) != warp8) continue;
            rows |= static_cast<uint32_t>(32 * w + __ffs(static_cast<int>(m)) - 1) << (8 * n);
            if (++n == 4) {
                four(rows);
                rows = 0;
                n = 0;
            }
        }
    if (n == 0) return;
    for (; n < 4; ++n) rows |= ((rows >> (8 * n - 8)) & 127u) << (8 * n);
    four(rows);
}

}  // namespace stc
}  // namespace mgn
