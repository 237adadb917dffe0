// Projection GEMMs of the forward for passes with many token rows (M > 128: verify steps of large
// batches, prefill passes): the same products and fused consumers as gemm_fused.cu, in the orientation
// that suits a tensor-bound product.
//
// Shape of the work.  Y[128 tokens][BNW features] = X[128 tokens][K] * W[BNW rows][K]^T: the token rows
// supply UMMA M (TMEM lanes), the weight rows UMMA N (TMEM columns, BNW = 128 or 256).  Activations are
// float32 values carried as (hi, lo) bf16 row pairs in the tile layout [TBL hi rows][TBL lo rows]; one TMA
// box brings both halves of a k-block, and the hi and the lo rows are two MMAs into the SAME accumulator,
// so the sum hi + lo costs no extra pass.  (With TBL < 128 the MMA's last lanes read rows that belong to
// something else; a lane's result depends on its own row only, and those lanes are never stored.)
//
// Persistent CTAs.  One CTA per SM walks the (feature tile, token tile) pairs blockIdx.x, + gridDim.x, ...
// with two accumulators in TMEM: while the eight epilogue warps drain tile j, the MMA warp already
// works on tile j + 1 in the other accumulator, and the TMA ring never stops between tiles.  A thread of
// the epilogue owns one token row (its TMEM lane) and 32 consecutive features per tcgen05.ld, so the
// row-wise consumers (RMS factor, RoPE pairs, sum of squares, row arg-max) need no exchange between threads.
//
// Pairs.  What bounds a tile is not the MMAs but what the SMs take in: a k-block of a 128 x 256 tile brings 64 KB (32 KB of
// token rows, hi and lo, and 32 KB of weights) for 1,024 cycles of MMA.  So where a product has 256-feature tiles for two token tiles or more, two CTAs form a pair
// (cta_group::2): one MMA of 256 token rows on both SMs' tensor cores, each CTA loading its own token rows and HALF of the
// weight rows, 48 KB per k-block.  The even CTA issues the MMAs and counts both CTAs' bytes on its barriers; the commits
// release stages and announce accumulators in both.
//   2,048 rows, 1,536 -> 17,920 features: 164 us before, 147 in pairs (tensor pipes 87 % busy), 140 with the epilogue below.
//
// Epilogue.  A thread holds 32 features of one row; 32 threads that each touch their own row make every access 32 lines, and
// at 2,048 rows the residual epilogue (nothing hides it in a grid of one wave) was longer than the MMAs of the O product.  A
// warp turns its 32 x 32 values around in shared memory first, so that eight lanes share a row: O and down together 162 ->
// 138 us, QKV 37 -> 34.
//
// Split-K.  A product with few output tiles and a long reduction (the down-projection, the narrow QKV and
// O matrices) runs as clusters of S CTAs instead: one tile per cluster, CTA r takes the r-th share of the
// k-blocks, parks its accumulator in its own shared memory (the ring is idle by then), and after a cluster
// barrier finishes every S-th 32-feature unit of the tile, adding the S copies in rank order
// (ld.shared::cluster).  No partial sum reaches global memory and the result does not depend on timing.
//
// Warp roles (320 threads): warps 0-7 epilogue (TMEM lane quarter w % 4; the two warps of a quarter split the
// tile's 32-column units, since one warp per scheduler leaves the epilogue bound by instruction latency),
// warp 8 TMA producer, warp 9 TMEM allocation + MMA issue.  Every mbarrier wait is bounded and gives up early once another role of the
// CTA has failed; a wait that runs out records TASC_ETIMEOUT, and the CTA frees its TMEM and returns.
#include "kernels.h"

#include <algorithm>
#include <map>
#include <mutex>

namespace tasc {

namespace {

constexpr int BK = 64;
constexpr int UMMA_K = 16;
constexpr int EPI_WARPS = 8;                 // two per TMEM lane quarter: they share the rows and split the 32-column units
constexpr int THREADS = (EPI_WARPS + 2) * 32;
constexpr int MAX_STAGES = 8;
constexpr int MAX_TT = 32;                   // token tiles of a prefill pass
constexpr int MAX_DYN_SMEM = 226 * 1024;
constexpr int STAGING_BYTES = EPI_WARPS * 32 * 32 * 4;        // behind the ring: the epilogue warps turn their rows around there

// CLUSTER: the arrivals may be another CTA's.
template <bool CLUSTER = false>
__device__ __forceinline__ bool wait_or_fail(uint32_t bar, uint32_t parity, volatile int* failed) {
    auto ready = [&]() { return CLUSTER ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
    if (ready()) return true;
    const long long t0 = clock64();
    for (;;) {
        if (ready()) return true;
        if (*failed) return false;
        if (clock64() - t0 > 1000000000ll) return false;
    }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}
// four consecutive values -> bf16; -> (hi, lo) bf16
__device__ __forceinline__ uint2 bf16x4(const float4& v) { return make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w)); }
__device__ __forceinline__ void hilo4(const float4& v, uint2& hi, uint2& lo) {
    split_bf16x2(v.x, v.y, hi.x, lo.x);
    split_bf16x2(v.z, v.w, hi.y, lo.y);
}
__device__ __forceinline__ void store_f32x32(float* p, const float (&v)[32]) {
#pragma unroll
    for (int e = 0; e < 32; e += 4) *reinterpret_cast<float4*>(p + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
}
// 32 accumulator columns of this thread's TMEM lane, as floats.
__device__ __forceinline__ void acc32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    tmem_ld32(taddr, r);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(r[e]);
}

// SPLIT: split-K clusters, one tile each, in place of persistent CTAs (or pairs).  Instances of their own: with the choice at run time
// every kernel carried both epilogues, 42 - 118 KB of code where it is 32 - 73 now, and the TMA lane worked out ring slots, tiles and rows by
// division at every k-block.  Step of the 0.5B + 8,192 tokens, 288 rows 1430 -> 1388 us; 1.5B, 448 rows 4242 -> 4181; prefill of 16 prompts of
// up to 1,024 tokens 77.5 -> 75.7 ms.
template <int EPI, bool PAIR, bool SPLIT>
__global__ void __launch_bounds__(THREADS, 1)
gemm_wide_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const FusedArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);

    __shared__ uint64_t s_bars[2 * MAX_STAGES + 4];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;              // a bounded wait ran out somewhere in this CTA
    volatile int* failed = &s_fail;

    const int BNW = a.BNW, TBL = a.TBL, stages = a.stages, num_kb = a.num_kb;
    const uint32_t a_bytes = (uint32_t)(2 * TBL) * 128u;        // one k-block of the token tile: TBL hi rows, TBL lo rows
    const uint32_t w_bytes = (uint32_t)(PAIR ? BNW / 2 : BNW) * 128u;   // (a pair's CTAs load half of the weight rows each)
    const uint32_t stage_bytes = a_bytes + w_bytes;
    const uint32_t bar_full = smem_u32(s_bars);
    const uint32_t bar_empty = bar_full + 8u * MAX_STAGES;
    const uint32_t bar_acc_full = bar_full + 16u * MAX_STAGES;  // [2]
    const uint32_t bar_acc_empty = bar_acc_full + 16u;          // [2]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    // Token tiles with rows in use, in s_tt.  (A ragged prefill's later passes are mostly padding: of 16 prompts of 512 to 1,024
    // tokens a quarter of all tiles.  1.5B: 85 ms with them, 79 without.)
    __shared__ int s_tt[MAX_TT];
    __shared__ int s_n_tt;
    const int S = SPLIT ? (int)cluster_nctarank() : 1;
    const int kb0 = SPLIT ? (int)((unsigned)(num_kb * rank) / (unsigned)S) : 0;
    const int nkb = SPLIT ? (int)((unsigned)(num_kb * (rank + 1)) / (unsigned)S) - kb0 : num_kb;      // k-blocks of this CTA (all of them when S = 1)
    constexpr int XPAD = 4;                                                 // floats: rows of the parked tile fall on distinct banks
    float* xch = reinterpret_cast<float*>(smem);                            // [128][BNW + XPAD], split-K only
    constexpr int FLD = 4 * 32 + XPAD;                                      // a CTA finishes at most four 32-column chunks of a split tile
    float* fin = xch + 128 * (BNW + XPAD);                                  // [128][FLD] the S copies of this CTA's chunks, added up
    uint32_t own_mask = 0u;                                                 // split-K: the tile's 32-column chunks that this CTA finishes
    const int FT = EPI == EPI_SWIGLU ? BNW / 2 : BNW;           // output features per tile
    float* stage = reinterpret_cast<float*>(smem + (size_t)stages * stage_bytes) + warp * 1024;      // the epilogue warps' 32 x 32 values (S = 1)
    auto fail = [&]() { set_status(a.status, TASC_ETIMEOUT); *failed = 1; };
#ifdef TASC_TIMELINE
    const unsigned long long g_t0 = global_ns();
    unsigned long long g_ta = 0, g_tb = 0, g_tc = 0, g_td = 0, g_te = 0, g_tf = 0;
#endif

    if (threadIdx.x == 0) {
        s_fail = 0;
        for (int s = 0; s < stages; ++s) {
            mbar_init(bar_full + 8u * s, 1);
            mbar_init(bar_empty + 8u * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar_acc_full + 8u * b, 1);
            mbar_init(bar_acc_empty + 8u * b, EPI_WARPS * 32 * (PAIR ? 2 : 1));
        }
        fence_barrier_init();
        tma_prefetch_desc(&tmW);
        tma_prefetch_desc(&tmX);
    }
    if (warp == EPI_WARPS + 1) {
        if (PAIR) tmem_alloc_pair(smem_u32(&s_tmem), (uint32_t)(2 * BNW)); else tmem_alloc(smem_u32(&s_tmem), (uint32_t)(2 * BNW));
    }
    if (warp == 0 && a.seq_rows) {
        if (!a.rows_early) griddep_wait();
        const bool live = lane < a.n_tt && rows_in_use(a.seq_rows, a.R, lane * TBL, min((lane + 1) * TBL, a.M));
        const uint32_t mask = __ballot_sync(0xFFFFFFFFu, live);
        if (live) s_tt[__popc(mask & ((1u << lane) - 1u))] = lane;
        if (lane == 0) s_n_tt = __popc(mask);
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();                                    // both CTAs' barriers are set up before either is signalled
    tc_fence_after();
    const uint32_t tmem_base = s_tmem;
    const int live_tt = a.seq_rows ? s_n_tt : a.n_tt;
    // the i-th of them; past the last one a tile without rows
    auto token_tile = [&](int i) { return i >= live_tt ? a.n_tt : a.seq_rows ? s_tt[i] : i; };
    const int n_tt = PAIR ? (live_tt + 1) / 2 : live_tt;        // token tiles, or pairs of them
    const int n_tiles = a.n_ft * n_tt;
    // S = 1: persistent, tiles blockIdx.x, + gridDim.x, ...   S > 1: the grid is S * n_tiles CTAs, one tile per cluster
    const int tile0 = PAIR ? (int)blockIdx.x / 2 : SPLIT ? (int)blockIdx.x / S : (int)blockIdx.x;
    const int tstep = PAIR ? (int)gridDim.x / 2 : SPLIT ? n_tiles : (int)gridDim.x;
    const int my_tiles = tile0 < n_tiles ? (n_tiles - tile0 + tstep - 1) / tstep : 0;

    if (warp == EPI_WARPS) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const uint64_t pol_w = a.n_tt > 1 ? policy_evict_last() : policy_evict_first();   // a weight tile is read once per token tile
            const uint64_t pol_x = policy_evict_last();                                       // token rows are read by every feature tile
            const int total = my_tiles * nkb;
            const uint32_t full0 = PAIR ? cluster_map(bar_full, 0u) : bar_full;      // a pair's bytes are counted by its even CTA
            auto expect = [&](int s) {
                if (!PAIR) mbar_expect_tx(bar_full + 8u * s, stage_bytes);
                else if (rank == 0) mbar_expect_tx(bar_full + 8u * s, 2u * stage_bytes);
            };
            // where the loads are: ring slot, k-block, tile (its first feature and first row of the activation buffer)
            struct At { int s, kb, tile, f0, row; };
            auto place = [&](At& c) {
                const int t = (int)((unsigned)c.tile / (unsigned)n_tt), i = c.tile - t * n_tt;
                c.f0 = t * FT;
                c.row = token_tile(PAIR ? 2 * i + rank : i) * 2 * TBL;
            };
            auto advance = [&](At& c) {
                if (++c.s == stages) c.s = 0;
                if (++c.kb == nkb) { c.kb = 0; c.tile += tstep; place(c); }
            };
            auto load_w = [&](const At& c) {
                const int f0 = c.f0, kc = (kb0 + c.kb) * BK;
                const uint32_t dst = smem_u32(smem + (size_t)c.s * stage_bytes) + a_bytes, bar = full0 + 8u * c.s;
                if (PAIR) {                                // 128 of the 256 weight rows: the gate rows or the up rows; the lower or the upper half
                    if (EPI == EPI_SWIGLU)
                        for (int r = 0; r < FT; r += 64) tma_load_2d_pair(dst + (uint32_t)r * 128u, &tmW, kc, rank * a.N + f0 + r, bar, pol_w);
                    else tma_load_2d_pair(dst, &tmW, kc, f0 + rank * 128, bar, pol_w);
                } else if (EPI == EPI_SWIGLU) {                   // FT gate rows, then the FT matching up rows (boxes of 64 rows)
                    for (int r = 0; r < FT; r += 64) {
                        tma_load_2d_hint(dst + (uint32_t)r * 128u, &tmW, kc, f0 + r, bar, pol_w);
                        tma_load_2d_hint(dst + (uint32_t)(FT + r) * 128u, &tmW, kc, a.N + f0 + r, bar, pol_w);
                    }
                } else {                                   // boxes of 128 rows
                    for (int r = 0; r < BNW; r += 128) tma_load_2d_hint(dst + (uint32_t)r * 128u, &tmW, kc, f0 + r, bar, pol_w);
                }
            };
            auto load_x = [&](const At& c) {
                const uint32_t dst = smem_u32(smem + (size_t)c.s * stage_bytes);
                if (PAIR) tma_load_2d_pair(dst, &tmX, c.kb * BK, c.row, full0 + 8u * c.s, pol_x);
                else tma_load_2d_hint(dst, &tmX, (kb0 + c.kb) * BK, c.row, bar_full + 8u * c.s, pol_x);
            };
            // The weights of the first stages depend on no earlier kernel: they are requested before the
            // preceding grid has finished, the token rows after it.
            const int pre = total < stages ? total : stages;
            At w = {0, 0, tile0, 0, 0};
            if (total > 0) place(w);
            At x = w;
#pragma unroll 1
            for (int i = 0; i < pre; ++i, advance(w)) {
                expect(w.s);
                load_w(w);
            }
            griddep_wait();
#pragma unroll 1
            for (int i = 0; i < pre; ++i, advance(x)) load_x(x);
            uint32_t parity = 0u;                          // of the stage's previous use
#pragma unroll 1
            for (int i = pre; i < total; ++i, advance(w)) {
                if (!wait_or_fail<PAIR>(bar_empty + 8u * w.s, parity, failed)) { fail(); break; }
                if (w.s == stages - 1) parity ^= 1u;
                expect(w.s);
                load_w(w);
                load_x(w);
            }
            griddep_launch_dependents();
        }
        __syncwarp();
    } else if (warp == EPI_WARPS + 1) {
        // ------------------------------------------------------------ MMA issue
        // (the whole warp, see umma_bf16_warp)
        if (!PAIR || rank == 0) {
            const uint32_t idesc = umma_idesc_bf16_f32(PAIR ? 256 : 128, BNW);
            const uint32_t ring = smem_u32(smem);
            auto mma = [&](uint32_t d, uint64_t da, uint64_t db, uint32_t acc) {
                if (PAIR) umma_bf16_pair_warp(d, da, db, idesc, acc);
                else umma_bf16_warp(d, da, db, idesc, acc);
            };
            auto commit = [&](uint32_t bar) { if (PAIR) umma_commit_pair_warp(bar); else umma_commit_warp(bar); };
            int s = 0;
            uint32_t round = 0;
            bool ok = true;
#pragma unroll 1
            for (int j = 0; j < my_tiles && ok; ++j) {
                const int b = j & 1;
                ok = __all_sync(0xFFFFFFFFu, wait_or_fail<PAIR>(bar_acc_empty + 8u * b, (((uint32_t)(j >> 1)) & 1u) ^ 1u, failed));
                if (!ok) { fail(); break; }
                tc_fence_after();
                const uint32_t d = tmem_base + (uint32_t)(b * BNW);
#pragma unroll 1
                for (int kb = 0; kb < nkb; ++kb) {
                    ok = __all_sync(0xFFFFFFFFu, wait_or_fail<PAIR>(bar_full + 8u * s, round & 1u, failed));
                    if (!ok) { fail(); break; }
                    tc_fence_after();
                    const uint32_t sa = ring + (uint32_t)s * stage_bytes;
                    const uint64_t hi = umma_desc_k_sw128(sa), lo = umma_desc_k_sw128(sa + (uint32_t)TBL * 128u), w = umma_desc_k_sw128(sa + a_bytes);
                    constexpr int STEP = UMMA_K * 2 / 16;            // (addresses in units of 16 bytes)
#pragma unroll
                    for (int kk = 0; kk < BK / UMMA_K; ++kk) mma(d, hi + kk * STEP, w + kk * STEP, (kb > 0 || kk > 0) ? 1u : 0u);
#pragma unroll
                    for (int kk = 0; kk < BK / UMMA_K; ++kk) mma(d, lo + kk * STEP, w + kk * STEP, 1u);
                    commit(bar_empty + 8u * s);
                    if (++s == stages) { s = 0; ++round; }
                }
                if (ok) commit(bar_acc_full + 8u * b);
            }
        }
        __syncwarp();
    }

    // ---------------------------------------------------------------- epilogue: one token row per thread (warps 0-7)
    const int quarter = warp & 3, wq = (warp >> 2) & 1;              // TMEM lane quarter; which of the quarter's two warps
    const int rowl = quarter * 32 + lane;                             // row within the token tile = TMEM lane
    const int XLD = BNW + XPAD;
    uint32_t peer[8];
    if (SPLIT) {
#pragma unroll
        for (int s = 0; s < 8; ++s) peer[s] = cluster_map(smem_u32(xch), (uint32_t)(s < S ? s : 0));
    }
    // Finishes tile `tile`.  `acc` = TMEM address of this thread's lane in the tile's accumulator.  With split-K the
    // 32-column units come from the S parked copies instead, added in rank order, and this CTA takes every S-th unit.
    auto finish_tile = [&](int tile, uint32_t acc) {
        const int ft = tile / n_tt, tt = token_tile(PAIR ? 2 * (tile % n_tt) + rank : tile % n_tt);
        const int f0 = ft * FT;
        const int m = tt * TBL + rowl;
        const bool rowok = rowl < TBL && m < a.M;
        auto get32 = [&](int col, float (&v)[32]) {
            if (!SPLIT) {
                acc32(acc + (uint32_t)col, v);
            } else {
                // the reduced columns of this CTA's units, packed in the order of their 32-column chunks
                const int jc = __popc(own_mask & ((1u << (col >> 5)) - 1u));
                const float* src = fin + (size_t)rowl * FLD + jc * 32;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 q = *reinterpret_cast<const float4*>(src + 4 * e);
                    v[4 * e] = q.x; v[4 * e + 1] = q.y; v[4 * e + 2] = q.z; v[4 * e + 3] = q.w;
                }
            }
        };
        // A thread has 32 values of ONE row; memory wants rows.  The 32 x 32 values of a warp go through shared memory (its own
        // swizzled 4 KB, or with split-K the reduced chunk they came from), and come back as emit(row within the quarter, column,
        // four values) with eight lanes to a row: 4 lines per access, where a thread per row touched 32.
        auto staged = [&](int col, int r, int c4) {
            return !SPLIT ? reinterpret_cast<float4*>(stage + r * 32 + ((c4 ^ (r & 7)) << 2))
                          : reinterpret_cast<float4*>(fin + (size_t)(quarter * 32 + r) * FLD + __popc(own_mask & ((1u << (col >> 5)) - 1u)) * 32 + 4 * c4);
        };
        auto rows_out = [&](int col, const float (&v)[32], auto&& emit) {
#pragma unroll
            for (int e = 0; e < 8; ++e) *staged(col, lane, e) = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) emit(4 * i + (lane >> 3), 4 * (lane & 7), *staged(col, 4 * i + (lane >> 3), lane & 7));
            __syncwarp();
        };
        const int q_row0 = quarter * 32, m0 = tt * TBL + q_row0;        // first row of the quarter in the tile, in the pass
        auto row_ok = [&](int r) { return q_row0 + r < TBL && m0 + r < a.M; };
        const size_t orow0 = (size_t)tt * (2 * TBL) + q_row0;
        auto store_hilo = [&](int r, int f, const float4& x) {
            uint2 h, l;
            hilo4(x, h, l);
            *reinterpret_cast<uint2*>(a.a_out + (orow0 + r) * a.N + f) = h;
            *reinterpret_cast<uint2*>(a.a_out + (orow0 + r + TBL) * a.N + f) = l;
        };
        int unit = 0;                                                 // running index of the tile's work units
        int owned = 0;                                                // ... of those of this CTA (every S-th)
        auto mine = [&]() {                                           // the quarter's two warps alternate over the CTA's units
            const bool own = !SPLIT || (unit++ % S) == rank;
            return own && (owned++ & 1) == wq;
        };
        float sc = 1.0f;
        if (a.ssq_in && rowok) {
            float ss = 0.f;
            const float4* sp = reinterpret_cast<const float4*>(a.ssq_in + (size_t)m * a.ssq_slots);
#pragma unroll 4
            for (int q = 0; q < a.ssq_slots / 4; ++q) { const float4 t = sp[q]; ss += (t.x + t.y) + (t.z + t.w); }
            sc = 1.0f / sqrtf(ss * a.inv_d + a.eps);
        }

        if (EPI == EPI_SWIGLU) {
#pragma unroll 1
            for (int c = 0; c < FT && f0 + c < a.N; c += 32) {
                if (!mine()) continue;
                float g[32], u[32];
                get32(c, g);
                get32(FT + c, u);
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const float g0 = g[e] * sc, u0 = u[e] * sc;
                    g[e] = __fdividef(g0, 1.0f + __expf(-g0)) * u0;
                }
                rows_out(c, g, [&](int r, int e, const float4& x) { if (row_ok(r)) store_hilo(r, f0 + c + e, x); });
            }
        } else if (EPI == EPI_RESID) {
            // ssq_out has one slot per 32 features here (a.ssq_out_slots of them, a multiple of four per 128 features)
#pragma unroll 1
            for (int c = 0; c < BNW && f0 + c < a.N; c += 32) {
                if (!mine()) continue;
                const int f = f0 + c;
                float v[32];
                float4 x[8];
                const int e0 = f + 4 * (lane & 7);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = 4 * i + (lane >> 3);
                    x[i] = row_ok(r) ? *reinterpret_cast<const float4*>(a.x + (size_t)(m0 + r) * a.N + e0) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                const float4 g4 = __ldg(reinterpret_cast<const float4*>(a.gain + e0));
                get32(c, v);
                int i = 0;
                rows_out(c, v, [&](int r, int, const float4& y) {
                    float4 t = x[i++];
                    t.x += y.x; t.y += y.y; t.z += y.z; t.w += y.w;
                    float ss = (t.x * t.x + t.y * t.y) + (t.z * t.z + t.w * t.w);
                    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 1);
                    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 2);
                    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 4);
                    if (!row_ok(r)) return;
                    *reinterpret_cast<float4*>(a.x + (size_t)(m0 + r) * a.N + e0) = t;
                    store_hilo(r, e0, make_float4(t.x * g4.x, t.y * g4.y, t.z * g4.z, t.w * g4.w));
                    if ((lane & 7) == 0) {
                        a.ssq_out[(size_t)(m0 + r) * a.ssq_out_slots + f / 32] = ss;
                        if (f + 32 >= a.N)                            // the slots past the last 32 features
#pragma unroll 1
                        for (int q = f / 32 + 1; q < a.ssq_out_slots; ++q) a.ssq_out[(size_t)(m0 + r) * a.ssq_out_slots + q] = 0.f;
                    }
                });
            }
        } else if (EPI == EPI_QKV) {
            const int hd = a.hd, half = hd >> 1;
            const int qd = a.n_q * hd, kvd = a.n_kv * hd;
            int pos = -1, page = -1;
            if (rowok) {
                pos = a.row_pos[m];
                if (pos >= a.max_positions) { set_status(a.status, TASC_EINVAL); pos = -1; }
                if (pos >= 0 && f0 + BNW > qd) {                      // the tile holds K or V heads
                    const int pslot = pos / a.page_size;
                    if (pslot < a.max_pages) page = a.block_table[(size_t)(m / a.R) * a.max_pages + pslot];
                    if (page < 0 || page >= a.n_pages) { set_status(a.status, TASC_ENOKV); page = -1; }
                }
            }
#pragma unroll 1
            for (int hc = 0; hc < BNW && f0 + hc < a.N; hc += hd) {
                const int fh = f0 + hc;                               // first feature of this head
                if (fh < qd + kvd) {
                    // a query or key head: rotate the pairs (i, i + half); a unit is 32 pairs
                    const bool is_q = fh < qd;
                    const long long kdst = !is_q && pos >= 0 && page >= 0
                        ? (long long)((((size_t)page * a.n_kv + (fh - qd) / hd) * a.page_size + pos % a.page_size) * hd) : -1ll;
#pragma unroll 1
                    for (int jj = 0; jj < half; jj += 32) {
                        if (!mine()) continue;
                        float lo[32], hi[32];
                        get32(hc + jj, lo);
                        get32(hc + half + jj, hi);
                        // (cos, sin) of the pair indices jj .. jj + 31 of this row's position: 64 floats, two units
                        if (pos >= 0) {
                            const float4* cs = reinterpret_cast<const float4*>(a.rope + (size_t)pos * half + jj);
#pragma unroll
                            for (int e = 0; e < 32; e += 2) {
                                const float4 t = cs[e >> 1];          // (cos, sin) of pair indices jj + e, jj + e + 1
                                const float a0 = lo[e] * sc, b0 = hi[e] * sc, a1 = lo[e + 1] * sc, b1 = hi[e + 1] * sc;
                                lo[e] = a0 * t.x - b0 * t.y;     hi[e] = b0 * t.x + a0 * t.y;
                                lo[e + 1] = a1 * t.z - b1 * t.w; hi[e + 1] = b1 * t.z + a1 * t.w;
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < 32; ++e) { lo[e] = 0.f; hi[e] = 0.f; }
                        }
                        auto put = [&](int col, int at, const float (&v)[32]) {
                            rows_out(col, v, [&](int r, int e, const float4& x) {
                                const long long dst = __shfl_sync(0xFFFFFFFFu, kdst, r);
                                if (is_q) { if (row_ok(r)) *reinterpret_cast<float4*>(a.qbuf + (size_t)(m0 + r) * qd + fh + at + e) = x; }
                                else if (dst >= 0) *reinterpret_cast<uint2*>(a.k_pages + dst + at + e) = bf16x4(x);
                            });
                        };
                        put(hc + jj, jj, lo);
                        put(hc + half + jj, half + jj, hi);
                    }
                } else {
                    // a value head
                    const long long vdst = pos >= 0 && page >= 0
                        ? (long long)((((size_t)page * a.n_kv + (fh - qd - kvd) / hd) * a.page_size + pos % a.page_size) * hd) : -1ll;
#pragma unroll 1
                    for (int c = 0; c < hd; c += 32) {
                        if (!mine()) continue;
                        float v[32];
                        get32(hc + c, v);
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] *= sc;
                        rows_out(hc + c, v, [&](int r, int e, const float4& x) {
                            const long long dst = __shfl_sync(0xFFFFFFFFu, vdst, r);
                            if (dst >= 0) *reinterpret_cast<uint2*>(a.v_pages + dst + c + e) = bf16x4(x);
                        });
                    }
                }
            }
        } else if (EPI == EPI_LM) {
            // the row's largest logit in this tile (smallest id on ties), merged across tiles by an atomic max on
            // the packed (value, id) word
            uint32_t bk = 0u, bi = 0xFFFFFFFFu;
#pragma unroll 1
            for (int c = 0; c < BNW && f0 + c < a.N; c += 32) {
                if (!mine()) continue;
                float v[32];
                get32(c, v);
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const uint32_t k = float_key(v[e]);
                    if (bi == 0xFFFFFFFFu || k > bk) { bk = k; bi = (uint32_t)(f0 + c + e); }
                }
                if (a.logits && rowok) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] *= sc;
                    store_f32x32(a.logits + (size_t)m * a.N + f0 + c, v);
                }
            }
            if (rowok && bi != 0xFFFFFFFFu)
                atomicMax(&a.argmax[m], ((unsigned long long)bk << 32) | (unsigned long long)(0xFFFFFFFFu - bi));
        }
    };

    if (warp < EPI_WARPS) {
        griddep_wait();
#ifdef TASC_TIMELINE
        g_ta = global_ns();
#endif
        const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const uint32_t acc_empty0 = PAIR ? cluster_map(bar_acc_empty, 0u) : bar_acc_empty;      // the MMAs are issued by the even CTA
        if (!SPLIT) {
#pragma unroll 1
            for (int j = 0; j < my_tiles; ++j) {
                const int b = j & 1;
                bool ok = wait_or_fail<PAIR>(bar_acc_full + 8u * b, ((uint32_t)(j >> 1)) & 1u, failed);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) { if (lane == 0) fail(); break; }
#ifdef TASC_TIMELINE
                if (j == 0) g_tb = global_ns();
                if (j == my_tiles - 1) g_tc = global_ns();
#endif
                tc_fence_after();
                finish_tile(tile0 + j * tstep, lane_base + (uint32_t)(b * BNW));
                tc_fence_before();
                if (PAIR) mbar_arrive_cluster(acc_empty0 + 8u * b); else mbar_arrive(bar_acc_empty + 8u * b);
            }
        } else if (my_tiles > 0) {
            // split-K, part 1: this CTA's partial tile -> its shared memory (zeros after a failed wait, so that the
            // peers read something defined)
            bool ok = nkb > 0 && wait_or_fail(bar_acc_full, 0u, failed);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok && nkb > 0 && lane == 0) fail();
#ifdef TASC_TIMELINE
            g_tb = global_ns();
#endif
            tc_fence_after();
#pragma unroll 1
            for (int c = 32 * wq; c < BNW; c += 64) {
                float v[32];
                if (ok) {
                    acc32(lane_base + (uint32_t)c, v);
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = 0.f;
                }
                store_f32x32(xch + (size_t)rowl * XLD + c, v);
            }
            tc_fence_before();
        }
    }
    if (SPLIT) {
        // every CTA's partial tile is in its shared memory (release / acquire at cluster scope)
#ifdef TASC_TIMELINE
        g_tc = global_ns();
#endif
        cluster_sync();
#ifdef TASC_TIMELINE
        g_td = global_ns();
#endif
        if (warp < EPI_WARPS && my_tiles > 0) {
            // split-K, part 2: the chunks of this CTA's units (every S-th unit of the tile, in the order finish_tile meets
            // them), summed over the S parked copies in rank order into `fin`.  A work item is one chunk of one lane
            // quarter (32 rows x 32 columns); eight consecutive lanes cover the 128 bytes of a row, so a warp-wide
            // remote read touches 4 rows, and the reads of all copies are in flight together.
            {
                const int f0 = (tile0 / n_tt) * FT;
                int unit = 0;
                auto take = [&](int c0, int c1) {
                    if ((unit++ % S) == rank) { own_mask |= 1u << (c0 >> 5); if (c1 >= 0) own_mask |= 1u << (c1 >> 5); }
                };
                if (EPI == EPI_QKV) {
                    const int hd = a.hd, half = hd >> 1, qkd = (a.n_q + a.n_kv) * hd;
                    for (int hc = 0; hc < BNW && f0 + hc < a.N; hc += hd) {
                        if (f0 + hc < qkd) { for (int jj = 0; jj < half; jj += 32) take(hc + jj, hc + half + jj); }
                        else { for (int c = 0; c < hd; c += 32) take(hc + c, -1); }
                    }
                } else {
                    for (int c = 0; c < BNW && f0 + c < a.N; c += 32) take(c, -1);
                }
            }
            const int n_own = __popc(own_mask);
#pragma unroll 1
            for (int idx = warp; idx < n_own * 4; idx += EPI_WARPS) {
                const int jc = idx >> 2, q = idx & 3;
                const int chunk = __fns(own_mask, 0, jc + 1);         // the jc-th chunk of the mask
                const uint32_t off = (uint32_t)((q * 32 + (lane >> 3)) * XLD + chunk * 32 + 4 * (lane & 7)) * 4u;
                float* dst = fin + (size_t)(q * 32 + (lane >> 3)) * FLD + jc * 32 + 4 * (lane & 7);
#pragma unroll 1
                for (int ib = 0; ib < 8; ib += 2) {                   // rows lane / 8 + 4 i, two i at a time: 2 S reads in flight
                    float4 u[8][2];
#pragma unroll
                    for (int s2 = 0; s2 < 8; ++s2)
                        if (s2 < S) {
                            u[s2][0] = ld_cluster_f4(peer[s2] + off + (uint32_t)(4 * ib * XLD) * 4u);
                            u[s2][1] = ld_cluster_f4(peer[s2] + off + (uint32_t)(4 * (ib + 1) * XLD) * 4u);
                        }
                    float4 t0 = u[0][0], t1 = u[0][1];
#pragma unroll
                    for (int s2 = 1; s2 < 8; ++s2)
                        if (s2 < S) {
                            t0.x += u[s2][0].x; t0.y += u[s2][0].y; t0.z += u[s2][0].z; t0.w += u[s2][0].w;
                            t1.x += u[s2][1].x; t1.y += u[s2][1].y; t1.z += u[s2][1].z; t1.w += u[s2][1].w;
                        }
                    *reinterpret_cast<float4*>(dst + (size_t)(4 * ib) * FLD) = t0;
                    *reinterpret_cast<float4*>(dst + (size_t)(4 * (ib + 1)) * FLD) = t1;
                }
            }
            asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");   // the eight epilogue warps
            finish_tile(tile0, 0u);
        }
#ifdef TASC_TIMELINE
        g_te = global_ns();
#endif
        // peers may still be reading this CTA's partial tile
        cluster_sync();
    }
#ifdef TASC_TIMELINE
    g_tf = global_ns();
#endif
    __syncthreads();
    if (s_fail && warp == EPI_WARPS && lane == 0) {
        // after a timeout: give this CTA's own tile loads that may still be in flight a bounded time to land
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) { }
    }
    __syncthreads();
    if (PAIR) cluster_sync();                                    // neither CTA leaves while the other may signal or read it
    if (warp == EPI_WARPS + 1) {
        tc_fence_after();
        if (PAIR) tmem_dealloc_pair(tmem_base, (uint32_t)(2 * BNW)); else tmem_dealloc(tmem_base, (uint32_t)(2 * BNW));
    }
#ifdef TASC_TIMELINE
    if (threadIdx.x == 0) ctalog_put(g_t0, g_ta, g_tb, 20 + EPI, g_tc, g_td, g_te, g_tf);
#endif
}

template <int EPI, bool PAIR, bool SPLIT>
tasc_status prepare_wide() {
    static std::mutex mu;
    static bool attr_done[64] = {false};
    int dev = 0;
    TASC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return TASC_EINVAL;
    std::lock_guard<std::mutex> lk(mu);
    if (!attr_done[dev]) {
        TASC_CUDA_TRY(cudaFuncSetAttribute(gemm_wide_kernel<EPI, PAIR, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM));
        attr_done[dev] = true;
    }
    return TASC_OK;
}

template <int EPI, bool PAIR, bool SPLIT>
tasc_status launch_wide(const CUtensorMap* tmW, const CUtensorMap* tmX, const FusedArgs& a, const FusedPlan& p, int kind,
                        cudaStream_t stream) {
    tasc_status pst = prepare_wide<EPI, PAIR, SPLIT>();
    if (pst != TASC_OK) return pst;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.grid, 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)p.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    int n = 0;
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
    if (PAIR || SPLIT) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = PAIR ? 2u : (unsigned)p.S;
        at[n].val.clusterDim.y = 1;
        at[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    ProfScope ps(kind, stream);
    TASC_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_wide_kernel<EPI, PAIR, SPLIT>, *tmW, *tmX, a));
    return TASC_OK;
}

// Clusters of S CTAs with `smem` bytes each that the device can hold at once (0 if the query fails).
template <int EPI>
int wide_clusters(int S, int smem) {
    if (prepare_wide<EPI, false, true>() != TASC_OK) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)S, 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)S;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_wide_kernel<EPI, false, true>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); return 0; }
    return n;
}

int wide_clusters_any(int epi, int S, int smem) {
    static std::mutex mu;
    static std::map<long long, int> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return 0; }
    const long long key = (((long long)dev * 8 + epi) * 32 + S) * (1ll << 20) + smem;
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int n = 0;
    switch (epi) {
        case EPI_QKV:    n = wide_clusters<EPI_QKV>(S, smem); break;
        case EPI_RESID:  n = wide_clusters<EPI_RESID>(S, smem); break;
        default: break;
    }
    cache[key] = n;
    return n;
}

int sm_count() {
    static std::mutex mu;
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return 148; }
    std::lock_guard<std::mutex> lk(mu);
    if (!cached[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) { (void)cudaGetLastError(); n = 148; }
        cached[dev] = n;
    }
    return cached[dev];
}

}  // namespace

bool plan_wide(int M, int N, int K, int epi, int hd, FusedPlan& p, int token_tile) {
    if ((M <= 128 && token_tile <= 0) || N % 32 || K % 8) return false;
    if (epi != EPI_QKV && epi != EPI_RESID && epi != EPI_SWIGLU && epi != EPI_LM) return false;
    if (epi == EPI_QKV && hd != 64 && hd != 128) return false;
    p.TBL = token_tile > 0 ? token_tile : gemm_token_tile(M, true, 3, true);
    p.TB = p.TBL;
    p.BN = 2 * p.TBL;
    p.m_tiles = (M + p.TBL - 1) / p.TBL;
    p.num_kb = (K + BK - 1) / BK;
    p.wide = 1;
    p.cta_pair = 0;
    const int sms = sm_count();
    // Tile width and k-splits, by a cost in SM cycles.  A k-block of a tile of `bnw` features is 8 MMAs of bnw / 2 cycles
    // and brings (2 TBL + bnw) rows of 128 bytes into shared memory, which an SM takes in at about 40 bytes per cycle
    // (measured: 0.97 us per k-block at 256 features, 0.70 us at 128).  A persistent grid (S = 1) pays one epilogue that
    // nothing hides; a split-K grid pays the parking of the tile, two cluster barriers and the pull of S copies.
    const bool may_split = epi == EPI_QKV || epi == EPI_RESID;
    double best_cost = -1.;
    for (int bnw = 256; bnw >= 128; bnw >>= 1) {
        const int ft = epi == EPI_SWIGLU ? bnw / 2 : bnw;
        const int tiles = ((N + ft - 1) / ft) * p.m_tiles;
        const int stage_bytes = (2 * p.TBL + bnw) * 128;
        const int st = std::max(2, std::min((192 * 1024) / stage_bytes, MAX_STAGES));
        const int data = std::max(st * stage_bytes + STAGING_BYTES, 128 * (bnw + 4) * 4 + 128 * (4 * 32 + 4) * 4);
        const int smem = std::min(std::max(1024 + data, 120 * 1024), MAX_DYN_SMEM);
        const double per_kb = std::max(4.0 * bnw, (2.0 * p.TBL + bnw) * 128.0 / 40.0);
        for (int S = 1; S <= (may_split ? 8 : 1); ++S) {
            if (S > p.num_kb || (S > 1 && tiles * S > sms)) break;
            if (S > 1) {
                const int fit = wide_clusters_any(epi, S, smem);
                if (fit <= 0 || tiles > fit) continue;
            }
            const int waves = S > 1 ? 1 : (tiles + sms - 1) / sms;
            const double cost = (double)waves * ((p.num_kb + S - 1) / S) * per_kb + (S > 1 ? 6000.0 + 10.0 * bnw : 12.0 * bnw);
            if (best_cost < 0. || cost < best_cost) {
                best_cost = cost;
                p.BNW = bnw; p.S = S; p.cta_pair = 0; p.out_tiles = (N + ft - 1) / ft; p.stages = st; p.data_bytes = data; p.smem_bytes = smem;
                p.grid = S > 1 ? tiles * S : std::min(tiles, sms);
            }
        }
    }
    // Pairs of CTAs on 256 features and two token tiles: half the weight rows per CTA.
    if (p.m_tiles >= 2 && sms % 2 == 0) {
        const int ft = epi == EPI_SWIGLU ? 128 : 256;
        const int out_tiles = (N + ft - 1) / ft, tiles = out_tiles * ((p.m_tiles + 1) / 2), pairs = sms / 2;
        const int stage_bytes = (2 * p.TBL + 128) * 128;
        const int st = std::min((192 * 1024) / stage_bytes, MAX_STAGES);
        // (a k-block takes a pair 0.92 of the time of a CTA alone, measured on 448 rows x 151,936 features; a lone last token
        // tile wastes half a pair: at 288 rows x 160,128 features, three token tiles, 174 us in pairs against 140)
        const double per_kb = std::max(4.0 * 256, 0.92 * (2.0 * p.TBL + 256) * 128.0 / 40.0);
        const double cost = (double)((tiles + pairs - 1) / pairs) * p.num_kb * per_kb + 12.0 * 256;
        if (cost < best_cost) {
            p.BNW = 256; p.S = 1; p.cta_pair = 1; p.out_tiles = out_tiles; p.stages = st; p.data_bytes = st * stage_bytes + STAGING_BYTES;
            p.smem_bytes = std::min(std::max(1024 + p.data_bytes, 120 * 1024), MAX_DYN_SMEM);
            p.grid = 2 * std::min(tiles, pairs);
        }
    }
    return best_cost >= 0.;
}

tasc_status launch_gemm_wide(int epi, const CUtensorMap* tmW, const CUtensorMap* tmX, FusedArgs a, const FusedPlan& p,
                             cudaStream_t stream) {
    a.num_kb = p.num_kb; a.BN = p.BN; a.TB = p.TB; a.TBL = p.TBL; a.stages = p.stages; a.pair = 1; a.data_bytes = p.data_bytes;
    a.BNW = p.BNW; a.n_ft = p.out_tiles; a.n_tt = p.m_tiles;
    if (a.n_tt > MAX_TT) a.seq_rows = nullptr;
    switch (epi) {                                                 // (gate/up and the LM head are never split: plan_wide)
        case EPI_QKV:    return p.cta_pair ? launch_wide<EPI_QKV, true, false>(tmW, tmX, a, p, K_GEMM, stream)
                              : p.S > 1    ? launch_wide<EPI_QKV, false, true>(tmW, tmX, a, p, K_GEMM, stream)
                                           : launch_wide<EPI_QKV, false, false>(tmW, tmX, a, p, K_GEMM, stream);
        case EPI_RESID:  return p.cta_pair ? launch_wide<EPI_RESID, true, false>(tmW, tmX, a, p, K_GEMM, stream)
                              : p.S > 1    ? launch_wide<EPI_RESID, false, true>(tmW, tmX, a, p, K_GEMM, stream)
                                           : launch_wide<EPI_RESID, false, false>(tmW, tmX, a, p, K_GEMM, stream);
        case EPI_SWIGLU: return p.cta_pair ? launch_wide<EPI_SWIGLU, true, false>(tmW, tmX, a, p, K_GEMM, stream)
                                           : launch_wide<EPI_SWIGLU, false, false>(tmW, tmX, a, p, K_GEMM, stream);
        case EPI_LM:     return p.cta_pair ? launch_wide<EPI_LM, true, false>(tmW, tmX, a, p, K_GEMM_LM, stream)
                                           : launch_wide<EPI_LM, false, false>(tmW, tmX, a, p, K_GEMM_LM, stream);
        default: return TASC_EINVAL;
    }
}

}  // namespace tasc
