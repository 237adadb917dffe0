// Verify and prefill attention for bf16 models on the 5th-generation tensor cores: the same job as attention_mma.cu (which see
// for the row and key order, the paged cache and the precision: Q and P as (hi, lo) bf16 pairs) for passes with enough rows
// and sequences.
//
// Bound: at 42 rows (7 rows x 6 query heads of a KV head) and 1,500 keys the warp-level kernel spent 5 us per 128 keys, on
// mma.sync pipes that half of its warps used and on barriers, while K and V could stream in a tenth of that.  Here S = Q K^T
// and P V are tcgen05 MMAs of 128 rows (M; the rows past the query tile cost nothing, the issue rate is the same) issued by
// one warp, S and O in TMEM, K and V staged by TMA, so that the softmax is what is left: a thread owns half of the keys
// of one row, registers hold its half of the row's O.  Per tile of TK keys
//   MMA warp       S(t + 1) while the softmax works on S(t); then P(t) V(t) into an O tile of its own
//   softmax warps  S(t) -> maximum (exchanged between the two threads of a row) -> P(t) as hi, lo, in TMEM in the place of S(t);
//                  then O += O tile (t - 1), rescaled: O is accumulated in registers, so a new maximum costs no pass over TMEM
//   TMA warp       K and V tiles, a ring of two or more
// P as the MMA's A operand in TMEM takes no pass through shared memory, does not wait for P(t - 1) to be used, and leaves the ring its
// memory, so that 128 keys make a tile for up to 128 rows too (64 before, and where the plan finds that better, see plan_attention_tc).  With up
// to 64 rows four of the eight softmax warps have any; two of the others are the TMA and the MMA warp then.
// Key ranges split over a cluster are merged as in attention_mma.cu.
//
// Measured, per layer: 1.5B at 64 sequences x 7 rows and up to 1,530 keys 61 -> 33 us (by stamps 2.2 us per 128 keys, 2.0
// with P in TMEM and the warps' places); 0.5B + 8,192 tokens at 32 x 9 rows, 640 keys 15.5 -> 13.4; prefill of 16 x 1,024 tokens
// on the 1.5B 72 -> 47 us per pass of 2,048 rows.  With P in TMEM, whole steps: 1.5B, 64 x 7 rows behind 1,500 keys 4,204 -> 4,190 us, and with
// the warps' places 4,094; 40 x 5 rows behind 1,400 2,859 -> 2,821, 2,736; 0.5B + 8,192 tokens 1,392 -> 1,370, 1,371; a prefill of
// 4 x 1,000 tokens of the 1.5B (96 rows) 19.68 -> 19.45 ms with tiles of 64 keys, 19.90 -> 19.47 with tiles of 128.
//
// A CTA with a few tiles waits for code that it executes as often, so there is one copy of everything (the first tile's scores, the last
// tile's O, both halves of a tile's load), ring slots are counted and rows divided by multiplication: 76 - 102 -> 47 - 66 KB.  A step
// of the 0.5B + 8,192 tokens at 288 rows 1476 -> 1448 us, a generation of the 0.5B with 8 sequences 57.5 -> 56.2 ms.
//
// Every wait is bounded; after one that ran out the loops run on without waiting, so that all barriers are still met.
#include "kernels.h"

#include <algorithm>
#include <mutex>

namespace tasc {

namespace {

constexpr int SM_WARPS = 8;                      // softmax: two per TMEM lane quarter, which share its rows
constexpr int PAGE = 16;
constexpr int MAX_PAGES = 1024;
constexpr int MAX_SMEM = 216 * 1024;
constexpr int MAX_RING = 4;

struct TcArgs {
    const float* q;
    const int32_t* block_table;
    int max_pages;
    long long n_pages;
    const int* seq_pos0;
    const int* seq_rows;
    __nv_bfloat16* out;
    int TB;
    int R, Rs, n_sub, n_q, n_kv, splits, stages;
    int g;                                                       // query heads of a KV head
    // split key ranges: query rows per CTA of the cluster, whose shares are stored into its shared memory; 0: fetched
    int push_rows;
    SmallDiv by_R, by_TB, by_splits, by_sub;
    int* status;
    float scale_log2e;
};

// 2^x; results below 2^-126 are zero here (.ftz)
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Shared-memory descriptor of an operand whose rows (128 bytes, swizzled) are steps along K and whose columns are M or N:
// 64 columns to a row block, `col_stride` bytes from one block of 64 columns to the next, 8 K-rows to 1,024 bytes.
__device__ __forceinline__ uint64_t umma_desc_mn_sw128(uint32_t smem_addr, uint32_t col_stride) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(col_stride >> 4) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// HD: head width, RP: rows of the query tile, TK: keys of a tile
template <int HD_, int RP_, int TK_> struct Tc {
    static constexpr int HD = HD_, RP = RP_, TK = TK_;
    static constexpr int HB = HD / 64;                           // blocks of 64 columns of a head
    // Query tiles of 64 rows have rows in the first two lane quarters: two warps of the others feed the tensor cores.  (Theirs are the other two
    // schedulers, and eight warps have more registers each than ten.)
    static constexpr int TMA_WARP = RP == 64 ? 2 : SM_WARPS, MMA_WARP = TMA_WARP + 1;
    static constexpr int WARPS = RP == 64 ? SM_WARPS : SM_WARPS + 2, THREADS = WARPS * 32, LOADERS = THREADS - 64;
    static constexpr int Q_BYTES = RP * HD * 2;                  // hi or lo
    static constexpr int KV_BYTES = TK * HD * 2;                 // K or V tile
    static constexpr int FIXED = 2 * Q_BYTES;
    static constexpr int S_COL = 0, O_COL = 2 * TK;              // TMEM columns: two S tiles, two O tiles
    static constexpr int COLS = 2 * TK + 2 * HD <= 256 ? 256 : 512;
    // A thread's share of a row of S, of O.  (128-wide heads and 128 rows: 40 bytes are spilled, ten warps have 168 registers each.  With S loaded 16
    // columns at a time 12 bytes, and slower: a prefill of 100 tokens of the 1.5B 1,581 -> 1,593 us, of 1,000 5,883 -> 5,899.)
    static constexpr int SC = TK / 2, OC = HD / 2;
    static int smem(int stages) { return 1024 + FIXED + stages * 2 * KV_BYTES; }
};

template <class C>
__global__ void __launch_bounds__(C::THREADS, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const TcArgs a) {
    constexpr int HD = C::HD, RP = C::RP, TK = C::TK, THREADS = C::THREADS, TMA_WARP = C::TMA_WARP, MMA_WARP = C::MMA_WARP;
    extern __shared__ uint8_t sm_raw[];
    uint8_t* sm = sm_raw + ((1024u - (smem_u32(sm_raw) & 1023u)) & 1023u);
    uint8_t* Qs = sm;                                            // hi, then lo: [HB][RP][128 bytes]
    uint8_t* ring = Qs + 2 * C::Q_BYTES;                         // [stages] K [HB][TK][128 bytes], V the same
    __shared__ int s_pages[MAX_PAGES];
    __shared__ float s_max[2][2][RP], s_sum[2][RP];
    __shared__ uint64_t s_bars[4 * MAX_RING + 9];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    volatile int* failed = &s_fail;

    const int sp = blockIdx.x, kh = blockIdx.y, b = a.by_sub.div(blockIdx.z), rb = ((int)blockIdx.z - b * a.n_sub) * a.Rs;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = a.g, R = a.Rs, G = g * R, h0 = kh * g, qd = a.n_q * HD;
#ifdef TASC_TIMELINE
    struct LogAtExit { unsigned long long t0, ta, tb, tc, td; __device__ ~LogAtExit() { if (threadIdx.x == 0) ctalog_put(t0, ta, tb, 11, tc, td); } } log_at_exit{global_ns(), 0, 0, 0, 0};
#endif
    // (the row plan, the block table and the committed K / V were written before the preceding grid started)
    const int seq_pos0 = a.seq_pos0[b];
    int rows = a.seq_rows[b] - rb;
    rows = rows < 0 ? 0 : (rows > R ? R : rows);
    const int pos0 = seq_pos0 + rb;
    auto head_of = [&](int rho) { return a.by_R.div(rho); };      // a query row's head, and its row of the sequence
    auto row_of = [&](int rho) { return rho - a.by_R.div(rho) * R; };
    auto out_row = [&](int rho) {
        const int m = b * a.R + rb + row_of(rho);
        return (size_t)(a.by_TB.div(m) * a.TB + m);
    };
    if (rows == 0) {
        griddep_wait();
        griddep_launch_dependents();
        // sequence not in this pass: its rows of the output are zero
        if (sp == 0) {
#pragma unroll 1
            for (int i = tid; i < G * (HD / 4); i += THREADS) {
                const int rho = i / (HD / 4), d4 = (i % (HD / 4)) * 4;
                const size_t row = out_row(rho), col = (size_t)(h0 + head_of(rho)) * HD + d4;
                *reinterpret_cast<uint2*>(a.out + row * qd + col) = make_uint2(0u, 0u);
                *reinterpret_cast<uint2*>(a.out + (row + a.TB) * qd + col) = make_uint2(0u, 0u);
            }
        }
        return;
    }
    if (a.push_rows) cluster_arrive();                           // (nothing is stored to a CTA that has not started)
    // this CTA's keys: the tiles are dealt out evenly over the splits
    const int total = pos0 + rows;
    const int tiles_all = (total + TK - 1) / TK, t_base = a.by_splits.div(tiles_all), t_rem = tiles_all - t_base * a.splits;
    // (no more keys than the staged pages hold: a sequence that is longer than its cache is reported by the append)
    const int n_tiles = min(t_base + (sp < t_rem ? 1 : 0), MAX_PAGES * PAGE / TK);
    const int k_begin = (sp * t_base + min(sp, t_rem)) * TK;
    const int k_end = min(total, k_begin + n_tiles * TK);
    const int pg_lo = k_begin / PAGE, n_pg = n_tiles > 0 ? (k_end - 1) / PAGE - pg_lo + 1 : 0;
    const int quarters = (G + 31) / 32;                          // TMEM lane quarters with rows: 2 softmax warps each
    const uint32_t arrivals = (uint32_t)quarters * 64u;

    const uint32_t bar_k_full = smem_u32(s_bars), bar_v_full = bar_k_full + 8u * MAX_RING;
    const uint32_t bar_k_empty = bar_v_full + 8u * MAX_RING, bar_v_empty = bar_k_empty + 8u * MAX_RING;
    const uint32_t bar_s_full = bar_v_empty + 8u * MAX_RING, bar_p_full = bar_s_full + 16u;
    const uint32_t bar_o_full = bar_p_full + 16u, bar_o_empty = bar_o_full + 16u, bar_q_full = bar_o_empty + 16u;
    if (warp == TMA_WARP) {
        // a barrier per lane, in the order of their addresses: the ring's, S full, P full, O full, O empty (two each), Q
        constexpr int RING = 4 * MAX_RING;
        if (lane < RING + 9)
            mbar_init(bar_k_full + 8u * lane, lane == RING + 8 ? (uint32_t)C::LOADERS : lane >= RING && ((lane - RING) & 2) ? arrivals : 1u);
        if (lane == 31) {
            s_fail = 0;
            tma_prefetch_desc(&tmK);
            tma_prefetch_desc(&tmV);
        }
        fence_barrier_init();
    }
#pragma unroll 1
    for (int i = tid; i < n_pg; i += THREADS) {
        const int pslot = pg_lo + i;
        int page = -1;
        if (pslot < a.max_pages) page = a.block_table[(size_t)b * a.max_pages + pslot];
        s_pages[i] = (page >= 0 && page < a.n_pages) ? page : -1;      // ids outside the pool are never used as addresses
    }
    if (warp == MMA_WARP) {
        tmem_alloc(smem_u32(&s_tmem), (uint32_t)C::COLS);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    auto wait = [&](uint32_t bar, uint32_t parity) {             // after a failure: no more waiting
        if (mbar_try_wait(bar, parity)) return;
        const long long t0 = clock64();
#pragma unroll 1
        while (!mbar_try_wait(bar, parity)) {
            if (*failed) return;
            if (clock64() - t0 > 1000000000ll) { set_status(a.status, TASC_ETIMEOUT); *failed = 1; return; }
        }
    };

    constexpr int OC = C::OC;
    float acc[OC];                                               // this thread's half of its row of O
    float m_run = -INFINITY, l_run = 0.f;
    const int quarter = warp & 3, half = (warp >> 2) & 1;
    const int rho = quarter * 32 + lane;                         // row of the query tile = TMEM lane
    const bool active = warp < SM_WARPS && warp != TMA_WARP && warp != MMA_WARP && quarter < quarters;

    if (warp == TMA_WARP) {
        // ------------------------------------------------------------ TMA
        // A tile is TK / 16 pages; a page of this KV head is one box (two for 128-wide heads) of K and one of V.  Rows past the
        // range re-read its last page, ids outside the pool read page 0: both are masked, and nothing unmapped is touched.
        // K and V have barriers of their own: K of a tile is free one softmax earlier than V.
        constexpr int BOXES = (TK / PAGE) * C::HB;
        // Tiles of committed positions are requested before the preceding grid has finished, the others after it.
        bool waited = false;
        int s = 0;                                               // ring slot of tile t; its parity is the one of its use before
        uint32_t used = 1u;
#pragma unroll 1
        for (int t = 0; t < n_tiles; ++t) {
            if (!waited && (t >= a.stages || k_begin + (t + 1) * TK > seq_pos0)) { griddep_wait(); waited = true; }
#pragma unroll 1
            for (int is_v = 0; is_v < 2; ++is_v) {
                if (t >= a.stages) wait((is_v ? bar_v_empty : bar_k_empty) + 8u * s, used);
                if (warp_failed(failed)) break;
                const uint32_t bar = (is_v ? bar_v_full : bar_k_full) + 8u * s;
                const uint32_t base = smem_u32(ring + (size_t)s * 2 * C::KV_BYTES) + (is_v ? C::KV_BYTES : 0);
                if (lane == 0) mbar_expect_tx(bar, C::KV_BYTES);
                __syncwarp();
                if (lane < BOXES) {
                    const int pg = lane / C::HB, h = lane % C::HB;
                    int key = k_begin + t * TK + pg * PAGE;
                    key = key < k_end ? key : k_end - 1;
                    int page = s_pages[key / PAGE - pg_lo];
                    page = page < 0 ? 0 : page;
                    tma_load_2d(base + h * (TK * 128) + pg * (PAGE * 128), is_v ? &tmV : &tmK, h * 64, (page * a.n_kv + kh) * PAGE, bar);
                }
                __syncwarp();
            }
            if (warp_failed(failed)) break;
            if (++s == a.stages) { s = 0; used ^= 1u; }
        }
        if (!waited) griddep_wait();
        __syncwarp();
    } else if (warp == MMA_WARP) {
        // ------------------------------------------------------------ MMA
        // (the whole warp, see umma_bf16_warp)
        if (n_tiles > 0) {
            const uint32_t qa = smem_u32(Qs), kv = smem_u32(ring);
            constexpr uint32_t idesc_s = umma_idesc_bf16_f32(128, TK);
            constexpr uint32_t idesc_o = umma_idesc_bf16_f32(128, HD) | (1u << 16);      // V: columns along N
            const uint64_t dq = umma_desc_k_sw128(qa);
            wait(bar_q_full, 0u);
            int sk = 0, sv = 0;                                  // ring slots of the next K and V tiles, and their parities
            uint32_t pk = 0u, pv = 0u;
#pragma unroll 1
            for (int t = -1; t < n_tiles; ++t) {
                if (t + 1 < n_tiles) {
                    const int u = t + 1;                         // S of the next tile
                    wait(bar_k_full + 8u * sk, pk);
                    // S and P of tile u - 2 were there: until P V of that tile is done.  (MMAs of one accumulator and shape follow one another;
                    // these have two accumulators, and the one reads what the other writes.)
                    if (u >= 2) wait(bar_o_full + 8u * (u & 1), (uint32_t)((u >> 1) - 1) & 1u);
                    tc_fence_after();
                    const uint64_t dk = umma_desc_k_sw128(kv + (uint32_t)sk * 2u * C::KV_BYTES);
                    const uint32_t d = tmem + C::S_COL + (uint32_t)(u & 1) * TK;
                    // (addresses in units of 16 bytes)
#pragma unroll
                    for (int p = 0; p < 2; ++p)                  // hi, lo
#pragma unroll
                        for (int ks = 0; ks < HD / 16; ++ks)
                            umma_bf16_warp(d, dq + (p * C::Q_BYTES + (ks >> 2) * (RP * 128) + (ks & 3) * 32) / 16,
                                           dk + ((ks >> 2) * (TK * 128) + (ks & 3) * 32) / 16, idesc_s, (p | ks) ? 1u : 0u);
                    umma_commit_warp(bar_s_full + 8u * (u & 1));
                    umma_commit_warp(bar_k_empty + 8u * sk);
                    if (++sk == a.stages) { sk = 0; pk ^= 1u; }
                }
                if (t < 0) continue;
                wait(bar_v_full + 8u * sv, pv);
                wait(bar_p_full + 8u * (t & 1), (uint32_t)(t >> 1) & 1u);
                if (t >= 2) wait(bar_o_empty + 8u * (t & 1), (uint32_t)((t >> 1) - 1) & 1u);
                tc_fence_after();
                const uint64_t dv = umma_desc_mn_sw128(kv + (uint32_t)sv * 2u * C::KV_BYTES + C::KV_BYTES, TK * 128);
                const uint32_t d = tmem + C::O_COL + (uint32_t)(t & 1) * HD;
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int kk = 0; kk < TK / 16; ++kk)
                        umma_bf16_ts_warp(d, tmem + C::S_COL + (uint32_t)((t & 1) * TK + p * (TK / 2) + kk * 8), dv + kk * (16 * 128 / 16), idesc_o,
                                          (p | kk) ? 1u : 0u);
                umma_commit_warp(bar_o_full + 8u * (t & 1));
                umma_commit_warp(bar_v_empty + 8u * sv);
                if (++sv == a.stages) { sv = 0; pv ^= 1u; }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ softmax
        griddep_wait();
#ifdef TASC_TIMELINE
        log_at_exit.ta = global_ns();
#endif
        griddep_launch_dependents();
        // Q rows, scaled, as (hi, lo) in shared memory; zeros where there is no row
        {
            constexpr int RPI = C::LOADERS / (HD / 4);           // rows of one reading of all threads; four readings under way together
            const int li = warp > MMA_WARP ? tid - 64 : tid, d4 = (li % (HD / 4)) * 4, chunk = (d4 & 63) >> 3;
#pragma unroll 1
            for (int r0 = li / (HD / 4); r0 < RP; r0 += 4 * RPI) {
                float4 qv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int r = r0 + j * RPI, hl = head_of(r), rr = r - hl * R;      // (rows past the tile: not stored)
                    qv[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r < G && rr < rows) qv[j] = *reinterpret_cast<const float4*>(a.q + (size_t)(b * a.R + rb + rr) * qd + (size_t)(h0 + hl) * HD + d4);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int r = r0 + j * RPI;
                    if (RP % (4 * RPI) && r >= RP) break;
                    uint2 h, l;
                    split_bf16x2(qv[j].x * a.scale_log2e, qv[j].y * a.scale_log2e, h.x, l.x);
                    split_bf16x2(qv[j].z * a.scale_log2e, qv[j].w * a.scale_log2e, h.y, l.y);
                    const uint32_t off = (uint32_t)((d4 >> 6) * (RP * 128) + r * 128 + ((chunk ^ (r & 7)) << 4) + (d4 & 7) * 2);
                    *reinterpret_cast<uint2*>(Qs + off) = h;
                    *reinterpret_cast<uint2*>(Qs + C::Q_BYTES + off) = l;
                }
            }
            fence_proxy_async_smem();
            mbar_arrive(bar_q_full);
        }
#ifdef TASC_TIMELINE
        log_at_exit.tc = global_ns();
#endif
#pragma unroll
        for (int e = 0; e < OC; ++e) acc[e] = 0.f;
        if (active) {
            const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
            const int lim = (rho < G && row_of(rho) < rows) ? min(pos0 + row_of(rho), k_end - 1) : -1;      // last visible key
            float al_o = 1.f;                                    // from acc's maximum to the one of the tile that is added next
            // O = O * al_o + the product of tile t.  (One copy of everything: a CTA with two or three tiles waits for code it executes
            // as often.)
            auto add_o = [&](int t) {
                wait(bar_o_full + 8u * (t & 1), (uint32_t)(t >> 1) & 1u);
                __syncwarp();                                    // (a lane waits by itself, TMEM is read by the warp as one)
                tc_fence_after();
#pragma unroll
                for (int c = 0; c < OC; c += 32) {
                    uint32_t r[32];
                    tmem_ld32(lane_base + C::O_COL + (uint32_t)((t & 1) * HD + half * OC + c), r);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; ++e) acc[c + e] = fmaf(acc[c + e], al_o, __uint_as_float(r[e]));
                }
                tc_fence_before();
                mbar_arrive(bar_o_empty + 8u * (t & 1));
            };
            constexpr int SC = C::SC;
            float s[SC];
#pragma unroll 1
            for (int t = 0; n_tiles > 0 && t <= n_tiles; ++t) {
                float al = 0.f;
                if (t < n_tiles) {
                    wait(bar_s_full + 8u * (t & 1), (uint32_t)(t >> 1) & 1u);
#ifdef TASC_TIMELINE
                    if (t == 0) log_at_exit.td = global_ns();
#endif
                    __syncwarp();
                    tc_fence_after();
#pragma unroll
                    for (int c = 0; c < SC; c += 32) {
                        uint32_t r[32];
                        tmem_ld32(lane_base + C::S_COL + (uint32_t)((t & 1) * TK + half * SC + c), r);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 32; ++e) s[c + e] = __uint_as_float(r[e]);
                    }
                    tc_fence_before();
                    const int k0 = k_begin + t * TK + half * SC;
                    if (k0 + SC - 1 > lim) {
#pragma unroll
                        for (int e = 0; e < SC; ++e) if (k0 + e > lim) s[e] = -INFINITY;
                    }
                    float m4[4] = {s[0], s[1], s[2], s[3]};          // (four chains: a warp has its scheduler nearly to itself)
#pragma unroll
                    for (int e = 4; e < SC; ++e) m4[e & 3] = fmaxf(m4[e & 3], s[e]);
                    const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
                    s_max[t & 1][half][rho] = mx;
                    asm volatile("bar.sync %0, 64;" ::"r"(1 + quarter) : "memory");      // the quarter's two warps
                    tc_fence_after();                                // (P goes where the other warp has read S)
                    const float mn = fmaxf(m_run, fmaxf(mx, s_max[t & 1][half ^ 1][rho])), mu = mn == -INFINITY ? 0.f : mn;
                    al = ex2(m_run - mu);                            // 0 while nothing was visible
                    m_run = mn;
                    float p4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int e = 0; e < SC; ++e) { s[e] = ex2(s[e] - mu); p4[e & 3] += s[e]; }
                    l_run = l_run * al + ((p4[0] + p4[1]) + (p4[2] + p4[3]));
                    // P, half row, in the place of S (which both threads of the row have read: the barrier above): hi, then lo
#pragma unroll
                    for (int c = 0; c < SC; c += 16) {
                        uint32_t h[8], l[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) split_bf16x2(s[c + 2 * e], s[c + 2 * e + 1], h[e], l[e]);
                        const uint32_t to = lane_base + C::S_COL + (uint32_t)((t & 1) * TK + (half * SC + c) / 2);
                        tmem_st8(to, h);
                        tmem_st8(to + TK / 2, l);
                    }
                    tmem_st_wait();
                    tc_fence_before();
                    mbar_arrive(bar_p_full + 8u * (t & 1));
                }
                if (t > 0) add_o(t - 1);
                al_o = al;
            }
            s_sum[half][rho] = l_run;
            asm volatile("bar.sync %0, 64;" ::"r"(1 + quarter) : "memory");
            l_run += s_sum[half ^ 1][rho];
        }
    }
#ifdef TASC_TIMELINE
    log_at_exit.tb = global_ns();
#endif
    // no copy and no MMA is under way any more (after a failure: give the copies a bounded time to land)
    tc_fence_before();
    __syncthreads();
    if (s_fail && tid == 0) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) { }
    }
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)C::COLS);
    }
    const int col0 = half * OC;
    if (a.splits == 1) {
        if (active && rho < G) {
            const float inv = l_run > 0.f && row_of(rho) < rows ? 1.0f / l_run : 0.f;
            const size_t row = out_row(rho), col = (size_t)(h0 + head_of(rho)) * HD + col0;
#pragma unroll
            for (int e = 0; e < OC; e += 8) {
                uint4 h, l;
                split_bf16x2(acc[e] * inv, acc[e + 1] * inv, h.x, l.x);
                split_bf16x2(acc[e + 2] * inv, acc[e + 3] * inv, h.y, l.y);
                split_bf16x2(acc[e + 4] * inv, acc[e + 5] * inv, h.z, l.z);
                split_bf16x2(acc[e + 6] * inv, acc[e + 7] * inv, h.w, l.w);
                *reinterpret_cast<uint4*>(a.out + row * qd + col + e) = h;
                *reinterpret_cast<uint4*>(a.out + (row + a.TB) * qd + col + e) = l;
            }
        }
        return;
    }
    // CTA r of the cluster merges the rows r, r + S, ...: the others' shares of them are stored into its shared memory, behind the ring.  Where there
    // is no room for that every CTA parks its rows in its own ring, and the mergers fetch them, which takes a barrier more and a trip on the chain: steps
    // of the 0.5B, 32 x 9 rows behind 1,000 keys, 1,409 -> 1,400 us, of the 1.5B, 24 x 7 rows, 2,411 -> 2,400.
    constexpr int XS = HD + 4;                                   // floats per row: O, maximum, sum, padding
    const int S = a.splits, rank = (int)cluster_ctarank(), push = a.push_rows;
    const uint32_t parked = smem_u32(ring), given = parked + (uint32_t)a.stages * 2u * C::KV_BYTES;      // given: [S][push_rows][XS]
    if (push) cluster_wait();
    if (active && rho < G) {
        if (push) {
            const int at = a.by_splits.div(rho);
            const uint32_t to = cluster_map(given + (uint32_t)((rank * push + at) * XS) * 4u, (uint32_t)(rho - at * S));
#pragma unroll
            for (int e = 0; e < OC; e += 4) st_cluster_f4(to + (uint32_t)(col0 + e) * 4u, make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]));
            if (half == 0) st_cluster_f2(to + HD * 4u, m_run, l_run);
        } else {
            float* to = reinterpret_cast<float*>(ring) + (size_t)rho * XS;
#pragma unroll
            for (int e = 0; e < OC; e += 4) *reinterpret_cast<float4*>(to + col0 + e) = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
            if (half == 0) *reinterpret_cast<float2*>(to + HD) = make_float2(m_run, l_run);
        }
    }
    cluster_sync();
#pragma unroll 1
    for (int at = tid / (HD / 4); at * S + rank < G; at += THREADS / (HD / 4)) {
        const int r = at * S + rank, d4 = (tid % (HD / 4)) * 4;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row_of(r) < rows) {
            float2 ml[8];
            float4 ov[8];
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (s < S) {                                     // all reads are issued before the first is used
                    const uint32_t from = push ? cluster_map(given + (uint32_t)((s * push + at) * XS) * 4u, (uint32_t)rank)
                                               : cluster_map(parked + (uint32_t)(r * XS) * 4u, (uint32_t)s);
                    ml[s] = ld_cluster_f2(from + HD * 4u);
                    ov[s] = ld_cluster_f4(from + (uint32_t)d4 * 4u);
                }
            float top = -INFINITY, den = 0.f;
#pragma unroll
            for (int s = 0; s < 8; ++s) if (s < S) top = fmaxf(top, ml[s].x);
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (s < S && ml[s].x != -INFINITY) {             // (a split without visible keys)
                    const float w = exp2f(ml[s].x - top);
                    den += w * ml[s].y;
                    o.x += w * ov[s].x; o.y += w * ov[s].y; o.z += w * ov[s].z; o.w += w * ov[s].w;
                }
            const float inv = den > 0.f ? 1.0f / den : 0.f;
            o.x *= inv; o.y *= inv; o.z *= inv; o.w *= inv;
        }
        const size_t row = out_row(r), col = (size_t)(h0 + head_of(r)) * HD + d4;
        uint2 h, l;
        split_bf16x2(o.x, o.y, h.x, l.x);
        split_bf16x2(o.z, o.w, h.y, l.y);
        *reinterpret_cast<uint2*>(a.out + row * qd + col) = h;
        *reinterpret_cast<uint2*>(a.out + (row + a.TB) * qd + col) = l;
    }
    if (push) return;                                            // (its shared memory is its own again)
    cluster_sync();                                            // peers may still be reading this CTA's rows
}

template <class C>
bool prepare() {
    static std::mutex mu;
    static int known[64] = {0};                                  // 1 yes, 2 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return false; }
    std::lock_guard<std::mutex> lk(mu);
    if (!known[dev]) {
        known[dev] = cudaFuncSetAttribute(attn_tc_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM) == cudaSuccess ? 1 : 2;
        if (known[dev] == 2) (void)cudaGetLastError();
    }
    return known[dev] == 1;
}

template <class C>
void config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&at)[2], int splits, int n_kv, int B, int stages) {
    cfg.gridDim = dim3((unsigned)splits, (unsigned)n_kv, (unsigned)B);
    cfg.blockDim = dim3(C::THREADS, 1, 1);
    cfg.dynamicSmemBytes = (size_t)C::smem(stages);
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)splits;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = splits > 1 ? 2 : 1;                           // the key-range splits of one (sequence, KV head) form a cluster
}

template <class C>
tasc_status launch_inst(const TcArgs& a, const CUtensorMap& tmK, const CUtensorMap& tmV, int B, cudaStream_t stream) {
    if (!prepare<C>()) return TASC_ECUDA;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    config<C>(cfg, at, a.splits, a.n_kv, B, a.stages);
    cfg.dynamicSmemBytes += (size_t)a.push_rows * a.splits * (C::HD + 4) * 4;
    cfg.stream = stream;
    ProfScope ps(K_ATT_SPLIT, stream);
    TASC_CUDA_TRY(cudaLaunchKernelEx(&cfg, attn_tc_kernel<C>, tmK, tmV, a));
    return TASC_OK;
}

template <class C> int ring_stages();
// Clusters of `splits` CTAs that the device holds at once (0: it cannot be asked).
template <class C>
int clusters(int splits) {
    static std::mutex mu;
    static int known[64][9] = {{0}};                             // + 1
    int dev = 0;
    if (!prepare<C>() || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return 0; }
    std::lock_guard<std::mutex> lk(mu);
    if (!known[dev][splits]) {
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[2];
        config<C>(cfg, at, splits, 1, 1, ring_stages<C>());
        cfg.attrs = at + 1;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, attn_tc_kernel<C>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
        known[dev][splits] = n + 1;
    }
    return known[dev][splits] - 1;
}
template <class C> int ring_stages() {
    int s = MAX_RING;
    while (s > 2 && C::smem(s) > MAX_SMEM) --s;
    return s;
}
// f(the instance for heads of hd, a query tile of up to 64 rows or more, tiles of `tile` keys)
template <class F>
auto with_instance(int hd, bool small, int tile, F f) {
    if (small) return hd == 64 ? f(Tc<64, 64, 128>{}) : f(Tc<128, 64, 128>{});
    if (tile == 64) return hd == 64 ? f(Tc<64, 128, 64>{}) : f(Tc<128, 128, 64>{});
    return hd == 64 ? f(Tc<64, 128, 128>{}) : f(Tc<128, 128, 128>{});
}

}  // namespace

// Splits by a cost in microseconds like plan_attention_mma's: T0 to start, `per_tile` for a tile of TK keys (taken for three
// quarters of the context and for all of it, half each: the tiles are large), as many waves as the occupancy of the launch
// dictates (one CTA per SM), the merge of split ranges.  The other kernel's cost is p.cost, and no less than what all its slabs
// take of the SMs' mma.sync pipes.  T0 as measured against the other kernel, which starts faster since its code was cut: a step
// of the 1.5B, 3 x 7 rows behind 400 keys, 1169 us here, 1121 there; 10 x 8 rows of the 0.5B 893 / 877; 1.5B 40 x 5 rows 2512 / 2549,
// 0.5B + 8,192 tokens 32 x 9 rows behind 640 keys 1441 / 1440.  (T0 was 3.9 and 2.8, a tile 1.8 and 1.4, before P was in TMEM: a step of the
// 0.5B, 32 x 9 rows behind 1,000 keys, was left with the other kernel then, 1445 us, 1409 here.  With T0 as it was the tiles' shorter times
// bring steps here that the other kernel is faster at: 0.5B, 2 x 7 rows behind 900 keys 675 us here, 630 there, 4 x 7 rows 740 / 698, 3 x 9
// behind 600 731 / 690.)  It pays for many (sequence, KV head) pairs with long contexts and three or
// more slabs of query rows, hardly ever at the 135M's 18 to 27 rows.
//   With 65 to 128 rows (prefill passes) tiles of 64 keys are weighed too: they start sooner and split finer, and two of them take longer
// than one of 128.  A prefill of one prompt with tiles of 128 / 64 keys and the splits that go with them, us: 1.5B, 48 tokens 1,181 / 1,156, 180
// 2,155 / 2,126, 256 2,284 / 2,258; but 100 1,571 / 1,598, 600 4,121 / 4,163, 1,000 5,929 / 6,003, 0.5B, 4 x 100 1,499 / 1,522.  A capacity of more than 64
// keys and a step's 16 rows, up to 144 (128 and 16), hardly ever means more than 128 keys, and one tile of 128 is the better one for them: 115 tokens
// 1,651 / 1,668, of the 0.5B 833 / 849.
bool plan_attention_tc(int B, int n_kv, int hd, int g, int rows, int max_ctx, int page_size, AttnPlan& p) {
    const int G = g * rows;
    if ((hd != 64 && hd != 128) || page_size != PAGE || G > 128 || max_ctx / PAGE > MAX_PAGES) return false;
    const bool small = G <= 64;
    const int groups = B * n_kv;
    const float pipes = (hd == 128 ? 0.6f : 0.3f) * (float)groups * (float)((G + 15) / 16) * (float)((max_ctx * 3 / 4 + 63) / 64) / 148.f;
    int best = 0, tile = 128;
    float best_cost = std::max(p.cost, 2.5f + pipes);
    for (int tk = 128; tk >= 64; tk -= 64) {
        if (tk == 64 && (small || (max_ctx > 64 + 16 && max_ctx <= 128 + 16))) break;
        const float T0 = hd == 128 ? (tk == 64 ? 3.8f : 4.3f) : (tk == 64 ? 3.1f : 3.2f);
        const float per_tile = hd == 128 ? (small ? 1.6f : tk == 64 ? 1.3f : 1.8f) : (small ? 1.2f : tk == 64 ? 0.95f : 1.4f);
        const int tiles_all = std::max(1, (max_ctx + tk - 1) / tk), tiles_34 = std::max(1, (max_ctx * 3 / 4 + tk - 1) / tk);
        for (int s = 1; s <= 8 && s <= tiles_all; ++s) {
            const int fit = with_instance(hd, small, tk, [&](auto c) { return clusters<decltype(c)>(s); });
            if (fit <= 0) continue;
            const int waves = (groups + fit - 1) / fit;
            const float tiles = 0.5f * (float)((tiles_all + s - 1) / s + (tiles_34 + s - 1) / s);
            // (merges and later waves as in the other kernel's plan: a layer of the 1.5B, 80 x 5 rows, 1,024 tokens of cache, 148.9 us whole
            // and 153.4 in 2 splits, 121.7 and 132.1 behind 170 of them; 48 x 3 rows, 4,096 tokens 137.8 whole, 137.9 in 4, 82.6 and 98.3 behind 680)
            const float cost = waves * (T0 + tiles * per_tile + (s > 1 ? 0.5f + 0.25f * s : 0.f)) + (waves - 1) * 1.0f + (groups * s > 128 ? 3.0f : 0.f);
            if (cost < best_cost - 1e-6f) { best_cost = cost; best = s; tile = tk; }
        }
    }
    if (!best) return false;
    p.tc = 1;
    p.heads = g;
    p.splits = best;
    p.tile = tile;
    const int share = (G + best - 1) / best;
    with_instance(hd, small, tile, [&](auto c) {
        using C = decltype(c);
        p.stages = ring_stages<C>();
        p.push_rows = best > 1 && C::smem(p.stages) + share * best * (hd + 4) * 4 <= MAX_SMEM ? share : 0;      // (one CTA per SM with or without it)
        return 0;
    });
    return true;
}

tasc_status launch_attention_tc(const float* qbuf, const CUtensorMap& tmK, const CUtensorMap& tmV, const int32_t* block_table, int max_pages,
                                long long n_pages, const RowPlan& rp, __nv_bfloat16* out, int TB, int B, int R, int n_q, int n_kv, int hd,
                                const AttnPlan& plan, int* status, cudaStream_t stream) {
    const int Rs = R <= 16 ? R : 16;
    if (R % Rs) return TASC_EINVAL;
    const int G = (n_q / n_kv) * Rs;
    if (G > 128 || (hd != 64 && hd != 128) || plan.splits < 1 || plan.splits > 8) return TASC_EINVAL;
    TcArgs a;
    a.q = qbuf; a.block_table = block_table; a.max_pages = max_pages; a.n_pages = n_pages;
    a.seq_pos0 = rp.seq_pos0; a.seq_rows = rp.seq_rows;
    a.out = out; a.TB = TB;
    a.R = R; a.Rs = Rs; a.n_sub = R / Rs; a.n_q = n_q; a.n_kv = n_kv; a.splits = plan.splits; a.stages = plan.stages;
    a.scale_log2e = 1.4426950408889634f / sqrtf((float)hd);
    a.status = status;
    a.g = n_q / n_kv;
    a.push_rows = plan.push_rows;
    a.by_R = SmallDiv(Rs); a.by_TB = SmallDiv(TB); a.by_splits = SmallDiv(plan.splits); a.by_sub = SmallDiv(a.n_sub);
    const int blocks = B * a.n_sub;
    return with_instance(hd, G <= 64, plan.tile, [&](auto c) { return launch_inst<decltype(c)>(a, tmK, tmV, blocks, stream); });
}

}  // namespace tasc
