// All decoder layers of a pass of few token rows as ONE persistent cooperative kernel (bf16 models).
//
// What bounds such a pass is not its bytes but its chain of dependent phases: QKV, attention, O, gate/up, down, five
// per layer, each of which needs the whole output of the one before.  As separate kernels (gemm_fused.cu,
// attention_mma.cu) a phase costs 4 - 8 us of launch hand-over, cluster exchange and tails around well under 1 us of
// work.  Here every SM runs one CTA for the whole pass and the phases are separated by a grid barrier (about 0.85 us
// from the last CTA's arrival until the last one is past it: one release increment per CTA on a counter in L2, one polling thread per CTA).
//
// Projections.  A CTA owns a block of output rows (1 / n_rb of them) for a block of T * 8 token rows and computes them
// over the whole reduction, so no partial sum leaves the CTA.  Its warps split the reduction; weights go from global
// memory straight into mma.sync fragments (the order of k inside a 32-wide chunk is a free choice as long as both
// operands use the same one: a lane's 16-byte load of 8 consecutive k is exactly one fragment half of two MMAs), so
// there is no shared-memory staging, and the first weights of a phase are requested BEFORE the barrier that precedes
// it.  16 weight rows are the MMA's M, 8 token rows its N; the hi and lo halves of an activation are two MMAs into one
// accumulator.  The warps' partial tiles meet in shared memory and are added in warp order (bitwise repeatable), and
// the stage that follows the product (RoPE + KV append, residual + next norm's input, SiLU * up) runs on the sums.
// The residual stream of a CTA's rows stays in its shared memory from the embedding to the last layer.
// A row's sum of squares for the RMSNorm comes from all CTAs, in any order: it is kept exact (ssq_word), so that a pass gives the
// same bits every time.  (In one double per row the order showed: rows built for it gave other logits in 39 of 40 passes.  A
// slot per CTA, added up in order by every reader, cost 0.3 us more per phase than eight words: 600 against 588 us at 135M, 6 rows.)
//
// Row pairs.  A tile's rows r and r + 8 are partners where the epilogue needs two features at once: the two halves of
// a rotary pair (QKV), a gate row and its up row (gate/up).
//
// Attention.  A unit is (sequence, KV head, 16 query rows, key range); all warps work on one tile of 128 keys, 16 per
// warp: S = Q K^T, the softmax statistics exchanged through shared memory, P as (hi, lo) in shared memory, O += P V with
// the warps splitting the head's columns.  K and V are staged by cp.async; the committed positions' are requested before
// the barrier.  Key ranges of one group are merged by the CTA that finishes last, in range order.
//
// Measured (one verify step, five kernels per layer / this kernel): 135M at 6 rows 747 / 594 us, 0.5B at 6 rows 746 / 650, 1.5B
// at 7 rows 1213 / 1144; more of it at persist_pays.  What is left, by stamps (which add about 0.3 us a phase): at 135M 3.0 - 3.5 us per
// projection, 0.8 - 1.0 of it the barrier, 0.7 - 1.0 the products behind their first fresh read, 1.5 the epilogue and the arrival;
// attention 6.6, 2.6 of it the merge of the key ranges.  At 1.5B the weights: gate/up 11.9 (products 8.2), down 7.9 (5.4), QKV 6.4 (CTAs
// start it 1.4 us apart), O 3.5, attention 9.5 (merge 3.9).
//
// Code is kept short, because a layer runs through more of it than the instruction cache holds: one copy of `decode` behind the
// products instead of two, two chunks in flight instead of four where they do not pay, loops of the attention not unrolled at one
// token tile, pairs split in two instructions: 64 -> 58 KB with heads of 64; 135M at 6 rows 577 -> 568 us, 0.5B 635 -> 628, 1.5B 1139 -> 1133.
//
// Every wait is bounded: a barrier that is not reached in about half a second records TASC_ETIMEOUT and the CTA
// leaves.  The limit holds for the first barrier too: a cooperative grid starts when all its CTAs can be resident, not one by
// one (measured: with another stream's kernel on one SM for 1.27 s the pass began behind it, without a time-out).
#include "kernels.h"

#include <algorithm>
#include <mutex>
#include <type_traits>

namespace tasc {

namespace {

constexpr int CHUNK = 64;                       // k per 32-byte load of a lane
constexpr int RED_N = 20;                       // floats per token of a parked 16-row tile (16 rows + padding: no bank conflicts)
constexpr int RED_TILE = 8 * RED_N;             // floats of a parked 16 x 8 tile
constexpr long long BARRIER_CYCLES = 1000000000ll;
constexpr int MAX_SMEM = 226 * 1024;

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// 32-byte loads at p + OFF: four lanes take a whole 128-byte line of a row.  ..._first: zero where `ok` is false;
// ..._next: the registers keep what they held there.  (The first load of a phase must define its registers, or their
// lifetime would reach around the whole layer loop.)
// Weights: read once by this SM, not kept in L1.
template <int OFF> __device__ __forceinline__ void ldg_stream_first(uint32_t (&v)[8], const void* p, bool ok) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t"
                 "mov.u32 %0, 0;\n\tmov.u32 %1, 0;\n\tmov.u32 %2, 0;\n\tmov.u32 %3, 0;\n\tmov.u32 %4, 0;\n\tmov.u32 %5, 0;\n\tmov.u32 %6, 0;\n\tmov.u32 %7, 0;\n\t"
                 "@q ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8 + %10];\n\t}"
                 : "=&r"(v[0]), "=&r"(v[1]), "=&r"(v[2]), "=&r"(v[3]), "=&r"(v[4]), "=&r"(v[5]), "=&r"(v[6]), "=&r"(v[7])
                 : "l"(p), "r"((uint32_t)ok), "n"(OFF));
}
template <int OFF> __device__ __forceinline__ void ldg_stream_next(uint32_t (&v)[8], const void* p, bool ok) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t"
                 "@q ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8 + %10];\n\t}"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
                 : "l"(p), "r"((uint32_t)ok), "n"(OFF));
}
// Activations another SM wrote before the last barrier (whose acquire has emptied this SM's L1): the warps that share
// a k range find them in L1.
template <int OFF> __device__ __forceinline__ void ldg_act_first(uint32_t (&v)[8], const void* p, bool ok) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t"
                 "mov.u32 %0, 0;\n\tmov.u32 %1, 0;\n\tmov.u32 %2, 0;\n\tmov.u32 %3, 0;\n\tmov.u32 %4, 0;\n\tmov.u32 %5, 0;\n\tmov.u32 %6, 0;\n\tmov.u32 %7, 0;\n\t"
                 "@q ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8 + %10];\n\t}"
                 : "=&r"(v[0]), "=&r"(v[1]), "=&r"(v[2]), "=&r"(v[3]), "=&r"(v[4]), "=&r"(v[5]), "=&r"(v[6]), "=&r"(v[7])
                 : "l"(p), "r"((uint32_t)ok), "n"(OFF) : "memory");
}
template <int OFF> __device__ __forceinline__ void ldg_act_next(uint32_t (&v)[8], const void* p, bool ok) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t"
                 "@q ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8 + %10];\n\t}"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
                 : "l"(p), "r"((uint32_t)ok), "n"(OFF) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
// Starts bringing `bytes` (a multiple of 16) into L2.
__device__ __forceinline__ void l2_prefetch(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_n(int n) {
    if (n) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float lds_f(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_f(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }

// Hides where a value comes from: what is derived from it is computed in this phase, not kept in registers over the
// whole layer loop (the compiler would otherwise hoist every phase's addresses out of it and spill them).
__device__ __forceinline__ int fresh(int v) {
    asm volatile("" : "+r"(v));
    return v;
}

// f(integral_constant 0), ..., f(integral_constant N - 1)
template <int N, int I = 0, typename F> __device__ __forceinline__ void for_each(F&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        for_each<N, I + 1>(f);
    }
}

enum { PH_QKV, PH_RESID, PH_GATEUP };

constexpr int MAX_PAGES = 1024;                 // pages of a key range
struct Unit { int b, kh, slab, sp, group, pos0, rows, k0, k1; };
constexpr int MAX_TOK = 32;                     // token rows per CTA
constexpr int WARPS = 8, LW = 3;                        // with 255 registers each: deep prefetch, and half the set-up work of sixteen

// One phase that is a projection: Y[rows of W][tokens] = W X^T and what follows it.
struct Phase {
    const __nv_bfloat16 *W, *X;
    int K, part;                       // reduction length; which partition of the rows (Shared::part)
    int kind;
    int lr;                            // log2 of the row groups the warps form
    int lh;                            // QKV: log2 of half a head; else 31
    int pair;                          // rows from a pair's first row to its second
    const float* gain;                 // residual phases
    const unsigned long long* ssq_in;
    unsigned long long* ssq_out;
    bool final_rows;
    __nv_bfloat16 *kp, *vp;
};

// What a CTA keeps for the whole pass, at the start of its dynamic shared memory.  (Behind a barrier's acquire a global
// load is a trip to L2, so everything that does not change between layers is read once and kept here.)
struct Shared {
    PersistArgs args;                  // for the routines that are not inlined (a reference to the kernel's parameters is slow there)
    long long koff[MAX_TOK];           // element offset of the token's slot in a layer's K or V pages, -1 = none
    LayerWeights layers[PERSIST_MAX_LAYERS];
    float rms[MAX_TOK];                // sums of squares of the current projection's input rows, or the RMS factors
    int pos[MAX_TOK];                  // positions, -1 = unused row
    int part[3][2];                    // first and last + 1 row (pair) of this CTA in the QKV, d-wide and gate/up products
    int m0;                            // its first token row
    Phase phase[2];                    // the current and the next projection (by parity)
    int stop;                          // a wait ran out
    int last;                          // this CTA merges the key ranges
    Unit unit;                         // the current attention unit
#ifdef TASC_TIMELINE
    unsigned long long tl[3];          // a phase of this CTA: start, past the barrier, products or key tiles done
#endif
    int pg[MAX_PAGES];                 // first pool rows of the pages of its key range, -1 outside the pool
};
constexpr int SHARED_BYTES = (sizeof(Shared) + 1023) / 1024 * 1024;
extern __shared__ __align__(1024) uint8_t dyn_smem[];
__device__ __forceinline__ Shared& sh() { return *reinterpret_cast<Shared*>(dyn_smem); }
__device__ __forceinline__ uint8_t* un() { return dyn_smem + SHARED_BYTES; }       // union: parked tiles / attention buffers

#ifdef TASC_TIMELINE
__device__ __forceinline__ void tl_stamp(int i) { if (threadIdx.x == 0) sh().tl[i] = global_ns(); }
__device__ __forceinline__ void tl_phase(int j) {
    if (threadIdx.x != 0) return;
    ctalog_put(sh().tl[0], sh().tl[1], sh().tl[2] ? sh().tl[2] : sh().tl[1], 30 + j);
    sh().tl[2] = 0;
    sh().tl[0] = global_ns();
}
#define TL_STAMP(i) tl_stamp(i)
#define TL_PHASE(j) tl_phase(j)
#else
#define TL_STAMP(i) do { } while (0)
#define TL_PHASE(j) do { } while (0)
#endif

// Grid barrier: arrival number `epoch` of every CTA completes barrier `epoch`.
__device__ __forceinline__ void grid_arrive(const PersistArgs& a) {
    __syncthreads();
    // everything this CTA has written is visible to whoever sees the counter
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
}
// false: the wait ran out.
__device__ __forceinline__ bool grid_wait(const PersistArgs& a, int epoch) {
    if (threadIdx.x == 0) {
        const unsigned target = (unsigned)epoch * gridDim.x;
        unsigned v;
        long long t0 = 0;
        for (int spin = 0;; ++spin) {
            // (an acquire on every poll: 0.28 us less per barrier than relaxed polls and a fence behind them)
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
            if (v >= target) break;
            if (spin == 64) t0 = clock64();
            if (spin > 64 && clock64() - t0 > BARRIER_CYCLES) { set_status(a.status, TASC_ETIMEOUT); sh().stop = 1; break; }
        }
    }
    __syncthreads();
    return sh().stop == 0;
}

// Starts bringing this CTA's rows of the projection that is phase j of layer l into L2.
template <int HD>
__device__ __noinline__ void prefetch_weights(int l, int j) {
    const PersistArgs& a = sh().args;
    const LayerWeights& lw = sh().layers[l];
    const int part = j == 0 ? 0 : j == 3 ? 2 : 1;
    const uint32_t row = (uint32_t)(j == 2 ? a.qd : j == 4 ? a.dff : a.d) * 2u;
    const uint8_t* W = reinterpret_cast<const uint8_t*>(j == 0 ? lw.wqkv : j == 2 ? lw.wo : j == 3 ? lw.w_gate_up : lw.w_down);
    int u = sh().part[part][0];
    const int u1 = sh().part[part][1];
    while (u < u1) {
        // a run of rows: all of them, or for QKV those of one head's half
        constexpr int half = HD / 2;
        const int e = j == 0 ? min(u1, (u / half + 1) * half) : u1;
        const uint8_t* p = W + (size_t)(j == 0 ? u + u / half * half : u) * row;
        l2_prefetch(p, (uint32_t)(e - u) * row);
        if (part != 1) l2_prefetch(p + (size_t)(j == 0 ? half : a.dff) * row, (uint32_t)(e - u) * row);
        u = e;
    }
}

// The projection of layer l that is the layer's phase j (0 QKV, 2 O, 3 gate/up, 4 down; 1 is the attention).
template <int HD>
__device__ __noinline__ void set_phase(int l, int j, Phase& ph) {
    const PersistArgs& a = sh().args;
    const LayerWeights& lw = sh().layers[l];
    ph.W = j == 0 ? lw.wqkv : j == 2 ? lw.wo : j == 3 ? lw.w_gate_up : lw.w_down;
    ph.X = j == 2 ? a.o : j == 4 ? a.act : a.h;
    ph.K = j == 2 ? a.qd : j == 4 ? a.dff : a.d;
    ph.kind = j == 0 ? PH_QKV : j == 3 ? PH_GATEUP : PH_RESID;
    ph.part = j == 0 ? 0 : j == 3 ? 2 : 1;
    ph.lr = a.lr[j == 0 ? 0 : j - 1];
    ph.lh = j == 0 ? (HD == 64 ? 5 : 6) : 31;
    ph.pair = j == 0 ? HD / 2 : a.dff;
    ph.gain = j == 2 ? lw.gain_mlp : lw.gain_next;
    ph.ssq_in = a.ssq + (2 * l + (j == 3 ? 1 : 0)) * (a.M * SSQ_WORDS);
    ph.ssq_out = a.ssq + (2 * l + (j == 2 ? 1 : 2)) * (a.M * SSQ_WORDS);
    ph.final_rows = j == 4 && l + 1 == a.n_layers;
    ph.kp = a.kv_pool + (size_t)l * 2 * a.kv_half;
    ph.vp = ph.kp + a.kv_half;
}

template <int HD, int T>
struct Cta {
    static constexpr int NW = WARPS, NT = NW * 32;
    static constexpr int LT = T == 4 ? 2 : T - 1;       // log2 T
    // chunks in flight per warp (64-wide heads: models whose rows are two or three chunks of a warp; four more of them are only code)
    static constexpr int D = T == 1 ? (HD == 64 ? 2 : 4) : (T == 2 ? 3 : 2);
    const PersistArgs& a;
    int epoch;                 // of the barrier that comes next

    // behind the union: the residual rows [nt_res][T][8][16], the rotary factors [nt_qkv][T][8][8] in the order of the QKV
    // epilogue
    __device__ __forceinline__ float* xs() const { return reinterpret_cast<float*>(un() + a.union_bytes); }
    __device__ __forceinline__ float2* s_cs() const { return reinterpret_cast<float2*>(un() + a.union_bytes + a.nt_res * (T * 512)); }
    // quotients of row numbers (below 2^16) by TBL and R without a division
    static __device__ __forceinline__ int div_r(const PersistArgs& a, int v) { return (int)__umulhi((unsigned)v, a.r_magic); }
    // Activations of width 64 * nch between the phases: blocks of 8 tokens x 64 features, hi then lo (1 KB each), so that
    // a warp's fragment load is one contiguous kilobyte.  Element offset of the hi value; lo is 512 elements further.
    static __device__ __forceinline__ unsigned act_at(int m, int f, int nch) {
        return (unsigned)((m >> 3) * nch + (f >> 6)) * 1024u + (unsigned)((m & 7) * 64 + (f & 63));
    }

    __device__ __forceinline__ float rms_factor(float ss) const { return 1.0f / sqrtf(ss * a.inv_d + a.eps); }
    // What one thread finishes: (row, token) of a tile -- for the pair phases both rows of the pair.
    struct Item {
        uint32_t p;            // shared address of the first parked copy this lane adds
        uint32_t xs;           // residual phases: shared address of the residual value
        float2 cs;             // QKV: rotary factors; residual phases: x = the next norm's gain
        uint8_t *out0, *out1;  // where the two results go (null: nowhere)
        int m;                 // token row
        bool lead;             // this lane stores
    };
    __device__ __forceinline__ Item decode(const Phase& ph, int idx, int lp, int tile0, uint32_t red, uint32_t stride, int u0, int u1, int m0) const {
        const bool resid = ph.kind == PH_RESID;
        const int lper = resid ? 4 : 3;
        const int part = (idx >> lper) & ((1 << lp) - 1), rest = idx >> (lper + lp), n = rest & 7;
        const int row = idx & ((1 << lper) - 1), hv = rest >> 3;
        const int tt = hv & (T - 1), tl = hv >> LT, tile = tile0 + tl, tok = tt * 8 + n;
        const int f = u0 + (tile << lper) + row;
        Item it;
        it.m = m0 + tok;
        it.p = red + (uint32_t)((tl * T + tt) * RED_TILE + n * RED_N + row) * 4u + (uint32_t)part * stride;
        it.lead = part == 0 && f < u1 && it.m < a.M;
        it.out0 = it.out1 = nullptr;
        it.xs = 0u;
        it.cs = make_float2(0.f, 0.f);
        if (resid) {
            it.xs = smem_u32(xs()) + (uint32_t)(((tile * T + tt) * 8 + n) * 16 + row) * 4u;
            if (it.lead) it.cs.x = __ldg(ph.gain + f);
            // the last rows go to the LM head: row-major layout tiles of TBL hi rows and TBL lo rows
            const unsigned at = ph.final_rows ? (unsigned)((int)__umulhi((unsigned)it.m, a.tbl_magic) * a.TBL + it.m) * a.d + f : act_at(it.m, f, a.d >> 6);
            it.out0 = reinterpret_cast<uint8_t*>(a.h + at);
            it.out1 = it.out0 + (ph.final_rows ? (unsigned)a.TBL * a.d : 512u) * 2u;
        } else if (ph.kind == PH_GATEUP) {
            it.out0 = reinterpret_cast<uint8_t*>(a.act + act_at(it.m, f, a.dff >> 6));
            it.out1 = it.out0 + 1024;
        } else {
            constexpr int half = HD / 2;
            const int head = f >> (HD == 64 ? 5 : 6), i = f & (half - 1);
            if (it.lead) it.cs = s_cs()[(tile * T + tt) * 64 + n * 8 + row];      // (1, 0) for value heads
            if (head < a.n_q) {
                it.out0 = reinterpret_cast<uint8_t*>(a.q + (size_t)it.m * a.qd + head * HD + i);
                it.out1 = it.out0 + half * 4;
            } else if (sh().koff[tok] >= 0) {
                const bool is_k = head < a.n_q + a.n_kv;
                it.out0 = reinterpret_cast<uint8_t*>((is_k ? ph.kp : ph.vp) + sh().koff[tok] + (((head - a.n_q - (is_k ? 0 : a.n_kv)) << a.page_shift) * HD) + i);
                it.out1 = it.out0 + half * 2;
            }
            it.xs = head < a.n_q ? 1u : 0u;                          // float results
        }
        return it;
    }

    // One projection phase: requests the first weights, passes the barrier, computes, finishes.  Everything that does not
    // depend on the phase before is done ahead of the barrier, where it costs nothing: behind it a hundred instructions
    // are 0.3 us on the critical path of the whole pass.  Returns false when the barrier timed out.
    __device__ __forceinline__ bool project(const Phase& ph, int next_l, int next_j, Phase& next) {
        const int tid = fresh(threadIdx.x), warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
        const int kind = ph.kind, lper = kind == PH_RESID ? 4 : 3, per = 1 << lper;      // rows (or pairs) per tile
        const int u0 = sh().part[ph.part][0], u1 = sh().part[ph.part][1], m0 = sh().m0;
        const int n_tiles = (u1 - u0 + per - 1) >> lper;
        // warps = row groups x k groups
        const int lr = ph.lr, lk = LW - lr, KG = 1 << lk, RG = 1 << lr, kg = warp >> lr, rg = warp & (RG - 1);
        const int chunks = ph.K >> 6;
        const int c0 = (chunks * kg) >> lk, n_ch = n_tiles > 0 ? ((chunks * (kg + 1)) >> lk) - c0 : 0;
        const int n_grp = (unsigned)(n_ch + D - 1) / (unsigned)D;      // this warp's chunks in groups of D
        const size_t k2 = (size_t)ph.K * 2;

        uint32_t w[D][2][8], b[D][T][2][8];
        const uint8_t *pw0, *pw1;                                      // of the group that is requested next
        const uint8_t* Wc = reinterpret_cast<const uint8_t*>(ph.W) + c0 * (CHUNK * 2) + t * 32;
        const uint8_t* Xc = reinterpret_cast<const uint8_t*>(ph.X) + ((size_t)(m0 >> 3) * chunks + c0) * 2048 + lane * 32;
        const size_t xt = (size_t)chunks * 2048;                       // to the next token tile
        auto point_w = [&](int tile) {
            // rows past the CTA's block repeat its last row (same addresses: no extra traffic); their sums are not used
            const int i = max(min(u0 + tile * per + g, u1 - 1), 0);
            pw0 = Wc + (i + ((i >> ph.lh) << ph.lh)) * k2;
            pw1 = kind == PH_RESID ? Wc + max(min(u0 + tile * per + g + 8, u1 - 1), 0) * k2 : pw0 + ph.pair * k2;
        };
        point_w(rg);
        for_each<D>([&](auto uc) {
            constexpr int u = decltype(uc)::value;
            ldg_stream_first<u * CHUNK * 2>(w[u][0], pw0, u < n_ch && rg < n_tiles);
            ldg_stream_first<u * CHUNK * 2>(w[u][1], pw1, u < n_ch && rg < n_tiles);
        });
        const uint32_t red = smem_u32(un());
        const int group = (unsigned)((a.park_bytes >> (lk + 2)) - 8) / (unsigned)(T * RED_TILE) & ~(RG - 1);      // tiles parked between two reductions
        const uint32_t stride = (uint32_t)(group * T * RED_TILE + 8) * 4u;      // bytes from one k group's parked tiles to the next one's
        // lanes that share an item's copies: where there are fewer items than threads
        auto items_of = [&](int tiles) { return tiles * T * 8 << lper; };
        int lp = 0;
        while (lp < 2 && lp < lk && (items_of(min(n_tiles, group)) << (lp + 1)) <= NT) ++lp;
        Item it = decode(ph, tid, lp, 0, red, stride, u0, u1, m0);
        const uint8_t* pb = Xc;
        if (tid == NT - 1 && next_l < a.n_layers) {
            set_phase<HD>(next_l, next_j, next);
            // HBM works ahead of the phases: O and gate/up start with QKV, down with O, the next layer's QKV with gate/up
            if (m0 == 0 && next_j != 0) {
                if (next_j == 3) prefetch_weights<HD>(next_l, 4);
                else {
                    const int pl = next_j == 2 ? next_l : next_l + 1;
                    if (pl < a.n_layers) prefetch_weights<HD>(pl, next_j == 2 ? 2 : 0);
                    if (next_j == 2) prefetch_weights<HD>(pl, 3);
                }
            }
        }
        if (!grid_wait(a, epoch)) return false;
        TL_STAMP(1);
        if (n_tiles == 0) return true;
        auto load_b = [&](auto first, auto uc, bool ok) {
            constexpr int u = decltype(uc)::value;
#pragma unroll
            for (int tt = 0; tt < T; ++tt) {
                if (decltype(first)::value) {
                    ldg_act_first<u * 2048>(b[u][tt][0], pb + tt * xt, ok);
                    ldg_act_first<u * 2048 + 1024>(b[u][tt][1], pb + tt * xt, ok);
                } else {
                    ldg_act_next<u * 2048>(b[u][tt][0], pb + tt * xt, ok);
                    ldg_act_next<u * 2048 + 1024>(b[u][tt][1], pb + tt * xt, ok);
                }
            }
        };
        // The sums of squares of the CTA's tokens, eight lanes each, for the RMS factors behind the products.  With four tiles they are
        // requested ahead of the activations, and the factors are ready made (48 rows of the 135M: 860 -> 848 us); with one the
        // two warps that add them up are on the critical path and do no more than that (6 rows: 588 -> 584).
        const bool sums = kind != PH_RESID && tid < T * 64;
        unsigned long long w8 = 0ull;
        auto load_sums = [&]() {
            if (sums && m0 + (tid >> 3) < a.M) asm volatile("ld.global.u64 %0, [%1];" : "=l"(w8) : "l"(ph.ssq_in + m0 * SSQ_WORDS + tid) : "memory");
        };
        if (T == 4) load_sums();
        for_each<D>([&](auto uc) { load_b(std::true_type{}, uc, decltype(uc)::value < n_ch); });
        if (T != 4) load_sums();
        if (sums) {
            const float ss = ssq_total(w8);
            if ((tid & 7) == 0) sh().rms[tid >> 3] = T == 4 ? rms_factor(ss) : ss;
        }
#pragma unroll 1
        for (int tile0 = 0; tile0 < n_tiles; tile0 += group) {
            const int tile1 = min(n_tiles, tile0 + group);
#pragma unroll 1
            for (int pt = tile0 + rg; pt < tile1; pt += RG) {
                float acc[T][2][4];                     // [1]: the lo halves (a second chain)
#pragma unroll
                for (int tt = 0; tt < T; ++tt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) { acc[tt][0][e] = 0.f; acc[tt][1][e] = 0.f; }
#pragma unroll 1
                for (int gi = 0; gi < n_grp; ++gi) {
                    // the next group: of this tile, or the first of the warp's next tile
                    const bool last = gi + 1 == n_grp;
                    const bool more = !last || pt + RG < n_tiles;
                    const int left = !more ? 0 : last ? n_ch : n_ch - (gi + 1) * D;
                    const int here = n_ch - gi * D;
                    if (more) {
                        if (last) { point_w(pt + RG); pb = Xc; }
                        else { pw0 += D * CHUNK * 2; pw1 += D * CHUNK * 2; pb += D * 2048; }
                    }
                    for_each<D>([&](auto uc) {
                        constexpr int u = decltype(uc)::value;
                        if (u < here) {
#pragma unroll
                            for (int j = 0; j < 8; j += 2)
#pragma unroll
                                for (int hl = 0; hl < 2; ++hl)
#pragma unroll
                                    for (int tt = 0; tt < T; ++tt)
                                        mma_bf16(acc[tt][hl], w[u][0][j], w[u][1][j], w[u][0][j + 1], w[u][1][j + 1], b[u][tt][hl][j], b[u][tt][hl][j + 1]);
                        }
                        if (more) {
                            ldg_stream_next<u * CHUNK * 2>(w[u][0], pw0, u < left);
                            ldg_stream_next<u * CHUNK * 2>(w[u][1], pw1, u < left);
                            if (n_grp > 1) load_b(std::false_type{}, uc, u < left);
                        }
                    });
                }
#pragma unroll
                for (int tt = 0; tt < T; ++tt) {
                    const uint32_t p = red + kg * stride + (uint32_t)(((pt - tile0) * T + tt) * RED_TILE + 2 * t * RED_N + g) * 4u;
                    sts_f(p, acc[tt][0][0] + acc[tt][1][0]);
                    sts_f(p + RED_N * 4, acc[tt][0][1] + acc[tt][1][1]);
                    sts_f(p + 32, acc[tt][0][2] + acc[tt][1][2]);
                    sts_f(p + RED_N * 4 + 32, acc[tt][0][3] + acc[tt][1][3]);
                }
            }
            __syncthreads();
            TL_STAMP(2);
            const int n_items = items_of(tile1 - tile0) << lp;
            bool decoded = tile0 == 0;
#pragma unroll 1
            for (int idx = tid; idx < n_items; idx += NT) {
                if (!decoded) it = decode(ph, idx, lp, tile0, red, stride, u0, u1, m0);
                decoded = false;
                float v0 = 0.f, v1 = 0.f;
                uint32_t p = it.p;
#pragma unroll (T == 1 ? 1 : 2)
                for (int k = KG >> lp; k > 0; --k, p += stride << lp) {
                    v0 += lds_f(p);
                    if (kind != PH_RESID) v1 += lds_f(p + 32);
                }
                if (lp >= 1) { v0 += __shfl_xor_sync(0xFFFFFFFFu, v0, per); v1 += __shfl_xor_sync(0xFFFFFFFFu, v1, per); }
                if (lp == 2) { v0 += __shfl_xor_sync(0xFFFFFFFFu, v0, 16); v1 += __shfl_xor_sync(0xFFFFFFFFu, v1, 16); }
                if (kind == PH_RESID) {
                    float ss = 0.f;
                    if (it.lead) {
                        const float x = lds_f(it.xs) + v0;
                        sts_f(it.xs, x);
                        ss = x * x;
                        uint32_t h, l;
                        split_bf16x2(x * it.cs.x, 0.f, h, l);
                        *reinterpret_cast<unsigned short*>(it.out0) = (unsigned short)h;
                        *reinterpret_cast<unsigned short*>(it.out1) = (unsigned short)l;
                    }
                    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 1);
                    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 2);
                    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 4);
                    ss += __shfl_xor_sync(0xFFFFFFFFu, ss, 8);
                    if (it.lead && (lane & 15) == 0) ssq_add(ph.ssq_out + it.m * SSQ_WORDS, ss);
                } else if (it.lead) {
                    float sc = sh().rms[it.m - m0];
                    if (T != 4) sc = rms_factor(sc);
                    v0 *= sc; v1 *= sc;
                    if (kind == PH_GATEUP) {
                        const float v = v0 / (1.0f + expf(-v0)) * v1;
                        __nv_bfloat16 h, l;
                        split_bf16(v, h, l);
                        *reinterpret_cast<__nv_bfloat16*>(it.out0) = h;
                        *reinterpret_cast<__nv_bfloat16*>(it.out1) = l;
                    } else if (it.out0) {
                        const float r0 = v0 * it.cs.x - v1 * it.cs.y, r1 = v1 * it.cs.x + v0 * it.cs.y;
                        if (it.xs) { *reinterpret_cast<float*>(it.out0) = r0; *reinterpret_cast<float*>(it.out1) = r1; }
                        else { *reinterpret_cast<__nv_bfloat16*>(it.out0) = __float2bfloat16_rn(r0); *reinterpret_cast<__nv_bfloat16*>(it.out1) = __float2bfloat16_rn(r1); }
                    }
                }
            }
            if (tile1 < n_tiles) __syncthreads();       // the parked tiles are overwritten by the next group
        }
        return true;
    }

    // ------------------------------------------------------------------------------------------------ attention
    static constexpr int KT = NW * 16;                  // keys per iteration
    static constexpr int CG = HD / 8;                   // column groups of the head
    static constexpr int NTW = CG / NW;                 // column groups per warp
    static constexpr int QS = HD + 8, PS = KT + 8;      // row strides of the Q and P tiles (elements)
    static constexpr int KV_BYTES = KT * HD * 2;
    static constexpr int ATT_BYTES = 2 * KV_BYTES + 2 * 16 * QS * 2 + 2 * 16 * PS * 2 + 2 * 16 * NW * 4;

    // Sets up unit u: what it is and the first pool row of every page of its key range.  Once per pass where every CTA has
    // at most one unit.
    static __device__ __noinline__ void prepare_unit(int u) {
        const PersistArgs& a = sh().args;
        __syncthreads();
        if (threadIdx.x == 0) {
            Unit r;
            r.sp = u % a.splits;
            r.group = u / a.splits;
            r.slab = r.group % a.n_slabs;
            const int bk = r.group / a.n_slabs;
            r.kh = bk % a.n_kv;
            r.b = bk / a.n_kv;
            r.pos0 = a.seq_pos0[r.b];
            r.rows = a.seq_rows[r.b];
            // keys the slab's rows can see: a slab inside one head ends at its last row, one that wraps sees every row
            const int first = r.slab * 16 - div_r(a, r.slab * 16) * a.R;
            const bool inside = first + 16 <= a.R;
            int total = r.rows > 0 ? r.pos0 + (inside ? min(r.rows, first + 16) : r.rows) : 0;
            if (inside && first >= r.rows) total = 0;
            const int per = ((total + a.splits - 1) / a.splits + 15) / 16 * 16;
            r.k0 = min(total, r.sp * per);
            // (no more keys than MAX_PAGES pages hold: a sequence that is longer than its cache is reported by the append)
            r.k1 = (int)min((long long)min(total, r.k0 + per), (long long)((r.k0 >> a.page_shift) + MAX_PAGES) << a.page_shift);
            sh().unit = r;
        }
        __syncthreads();
        const Unit& q = sh().unit;
        const int p0 = q.k0 >> a.page_shift, np = q.k1 > q.k0 ? ((q.k1 - 1) >> a.page_shift) - p0 + 1 : 0;
        for (int i = threadIdx.x; i < np; i += NT) {
            int page = -1;
            if (p0 + i < a.max_pages) page = a.block_table[(size_t)q.b * a.max_pages + p0 + i];
            sh().pg[i] = page < 0 || page >= a.n_pages ? -1 : (page * a.n_kv + q.kh) << a.page_shift;
        }
        __syncthreads();
    }

    // K or V rows of keys lo .. hi - 1 of the tile that starts at kb -> shared memory, 16-byte chunks XOR-ed with the row
    // (the eight rows of an ldmatrix phase on distinct banks); zeros past the unit's range and outside the pool.
    static __device__ __noinline__ void load_rows(const __nv_bfloat16* src, uint32_t dst, int kb, int lo, int hi) {
        const PersistArgs& a = sh().args;
        constexpr int CPR = HD / 8;
        const Unit& q = sh().unit;
        const int p0 = q.k0 >> a.page_shift, c = threadIdx.x % CPR;
#pragma unroll 1
        for (int key = lo + (int)threadIdx.x / CPR; key < hi; key += NT / CPR) {
            int row = key < q.k1 ? sh().pg[(key >> a.page_shift) - p0] : -1;
            const int bytes = row >= 0 ? 16 : 0;
            row = row >= 0 ? row + (key & (a.page_size - 1)) : 0;
            const int kr = key - kb;
            cp_async16(dst + (uint32_t)(kr * HD * 2 + ((c ^ (kr & 7)) << 4)), src + (size_t)row * HD + c * 8, bytes);
        }
    }

    // end of the rows a tile that starts at kb needs: whole blocks of 32 keys (the P V loop's step)
    static __device__ __forceinline__ int tile_end(int kb) { return kb + min(KT, (sh().unit.k1 - kb + 31) & ~31); }

    // One layer's attention.  Requests what it can of the first unit, passes the barrier, works through the units.
    __device__ __forceinline__ bool attention(const __nv_bfloat16* kp, const __nv_bfloat16* vp) {
        const int tid = fresh(threadIdx.x), warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
        __nv_bfloat16* Qh = reinterpret_cast<__nv_bfloat16*>(un() + 2 * KV_BYTES);
        __nv_bfloat16* Ph = Qh + 2 * 16 * QS;                     // Q and P: 16 hi rows, then 16 lo rows
        float* s_m = reinterpret_cast<float*>(Ph + 2 * 16 * PS);  // [16][NW] row maxima of the warps
        float* s_l = s_m + 16 * NW;                               // [16][NW] row sums of the warps
        const uint32_t ks = smem_u32(un()), vs = ks + KV_BYTES, qs = smem_u32(Qh), ps = smem_u32(Ph);
        // ldmatrix addresses of this lane: a 16 x 16 block of Q or P (row lane % 16, half lane / 16); for K the rows are keys
        const uint32_t qa = qs + (uint32_t)((lane & 15) * QS + (lane >> 4) * 8) * 2u, pa = ps + (uint32_t)((lane & 15) * PS + (lane >> 4) * 8) * 2u;
        const int kr = warp * 16 + (lane & 7) + ((lane >> 4) << 3), kc = (lane >> 3) & 1;
        const bool single = a.n_units <= (int)gridDim.x;          // the unit was set up before the first layer
        int u = fresh(blockIdx.x);
        if (!single && u < a.n_units) prepare_unit(u);
        const Unit& q = sh().unit;
        int from = 0;                                             // keys of the first tile that are on their way
        if (u < a.n_units && q.k0 < q.k1) {
            from = min(tile_end(q.k0), max(q.pos0, q.k0));
            load_rows(kp, ks, q.k0, q.k0, from);
            load_rows(vp, vs, q.k0, q.k0, from);
        }
        // this thread's share of the slab's query rows, and the last visible key of rows g and g + 8
        constexpr int NQ = 16 * (HD / 4) / NT;
        const int gq = a.n_q / a.n_kv, G = gq * a.R;
        const float* q_src[NQ];
        int lim[2];
        auto place = [&]() {
#pragma unroll
            for (int e = 0; e < NQ; ++e) {
                const int i = tid + e * NT, rho = q.slab * 16 + i / (HD / 4);
                const int hl = div_r(a, rho), rr = rho - hl * a.R;
                q_src[e] = rho < G && rr < q.rows ? a.q + (size_t)(q.b * a.R + rr) * a.qd + (size_t)(q.kh * gq + hl) * HD + (i % (HD / 4)) * 4 : nullptr;
            }
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int rho = q.slab * 16 + g + hf * 8, rr = rho - div_r(a, rho) * a.R;
                lim[hf] = rho < G && rr < q.rows ? min(q.pos0 + rr, q.k1 - 1) : -1;
            }
        };
        place();
        if (!grid_wait(a, epoch)) { cp_async_wait<0>(); return false; }
        TL_STAMP(1);
#pragma unroll 1
        for (; u < a.n_units; u += gridDim.x) {
            if (u != (int)blockIdx.x) { prepare_unit(u); from = q.k0; place(); }        // (its barriers: the previous unit's tiles are no longer read)
            float4 qv[NQ];
#pragma unroll
            for (int e = 0; e < NQ; ++e) qv[e] = q_src[e] ? __ldcg(reinterpret_cast<const float4*>(q_src[e])) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (const int end = tile_end(q.k0); q.k0 < q.k1 && from < end) {
                load_rows(kp, ks, q.k0, from, end);
                load_rows(vp, vs, q.k0, from, end);
            }
            cp_async_commit();
            // the query rows, scaled, as (hi, lo)
#pragma unroll
            for (int e = 0; e < NQ; ++e) {
                const int i = tid + e * NT, r = i / (HD / 4), d4 = (i % (HD / 4)) * 4;
                uint2 h, l;
                split_bf16x2(qv[e].x * a.scale_log2e, qv[e].y * a.scale_log2e, h.x, l.x);
                split_bf16x2(qv[e].z * a.scale_log2e, qv[e].w * a.scale_log2e, h.y, l.y);
                *reinterpret_cast<uint2*>(Qh + r * QS + d4) = h;
                *reinterpret_cast<uint2*>(Qh + (16 + r) * QS + d4) = l;
            }
            float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
            float oh[NTW][4], ol[NTW][4];                         // O from P's hi and lo halves: two MMA chains
#pragma unroll
            for (int i = 0; i < NTW; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) { oh[i][e] = 0.f; ol[i][e] = 0.f; }
            const int cg = warp * NTW;
#pragma unroll 1
            for (int kb = q.k0; kb < q.k1; kb += KT) {
                cp_async_wait_n(kb == q.k0 ? 0 : 1);              // K is there (after the first tile V may be on its way)
                __syncthreads();
                float s[2][4], sl[2][4];
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) { s[nt][e] = 0.f; sl[nt][e] = 0.f; }
                if (kb + warp * 16 < q.k1) {
#pragma unroll (T == 1 ? 2 : 4)
                    for (int j = 0; j < HD / 16; ++j) {
                        uint32_t ah[4], al[4], kf[4];
                        ldsm_x4(qa + j * 32, ah);
                        ldsm_x4(qa + 16 * QS * 2 + j * 32, al);
                        ldsm_x4(ks + (uint32_t)(kr * HD * 2 + (((2 * j + kc) ^ (kr & 7)) << 4)), kf);
                        mma_bf16(s[0], ah[0], ah[1], ah[2], ah[3], kf[0], kf[1]);
                        mma_bf16(s[1], ah[0], ah[1], ah[2], ah[3], kf[2], kf[3]);
                        mma_bf16(sl[0], al[0], al[1], al[2], al[3], kf[0], kf[1]);
                        mma_bf16(sl[1], al[0], al[1], al[2], al[3], kf[2], kf[3]);
                    }
                }
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    float mx = -INFINITY;
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int key = kb + warp * 16 + nt * 8 + 2 * t + e;
                            float& v = s[nt][2 * hf + e];
                            v = key > lim[hf] ? -INFINITY : v + sl[nt][2 * hf + e];
                            mx = fmaxf(mx, v);
                        }
                    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
                    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
                    if (t == 0) s_m[(g + 8 * hf) * NW + warp] = mx;
                }
                __syncthreads();
                const int next = kb + KT, end = tile_end(next);
                if (next < q.k1) load_rows(kp, ks, next, next, end);
                cp_async_commit();
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int row = g + 8 * hf;
                    float mn = m_run[hf];
#pragma unroll
                    for (int i = 0; i < NW; i += 4) {
                        const float4 x = *reinterpret_cast<const float4*>(s_m + row * NW + i);
                        mn = fmaxf(fmaxf(mn, fmaxf(x.x, x.y)), fmaxf(x.z, x.w));
                    }
                    const float mu = mn == -INFINITY ? 0.f : mn;
                    const float al = exp2f(m_run[hf] - mu);       // 0 while nothing was visible
                    m_run[hf] = mn;
                    float sum = 0.f;
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) {
                        const float e0 = exp2f(s[nt][2 * hf] - mu), e1 = exp2f(s[nt][2 * hf + 1] - mu);
                        sum += e0 + e1;
                        uint32_t h, l;
                        split_bf16x2(e0, e1, h, l);
                        const int col = warp * 16 + nt * 8 + 2 * t;
                        *reinterpret_cast<uint32_t*>(Ph + row * PS + col) = h;
                        *reinterpret_cast<uint32_t*>(Ph + (16 + row) * PS + col) = l;
                    }
                    l_run[hf] = l_run[hf] * al + sum;
#pragma unroll
                    for (int i = 0; i < NTW; ++i) {
                        oh[i][2 * hf] *= al; oh[i][2 * hf + 1] *= al;
                        ol[i][2 * hf] *= al; ol[i][2 * hf + 1] *= al;
                    }
                }
                cp_async_wait<1>();                               // this tile's V (the next K may be on its way)
                __syncthreads();
                const int kend = min(KT, q.k1 - kb);
#pragma unroll (T == 1 ? 1 : 2)
                for (int k32 = 0; k32 < kend; k32 += 32) {
                    uint32_t ah[2][4], al[2][4];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        ldsm_x4(pa + (k32 + j * 16) * 2, ah[j]);
                        ldsm_x4(pa + 16 * PS * 2 + (k32 + j * 16) * 2, al[j]);
                    }
                    const int vr = k32 + lane;
#pragma unroll
                    for (int i = 0; i < NTW; ++i) {
                        uint32_t vf[4];
                        ldsm_x4_trans(vs + (uint32_t)(vr * HD * 2 + (((cg + i) ^ (vr & 7)) << 4)), vf);
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            mma_bf16(oh[i], ah[j][0], ah[j][1], ah[j][2], ah[j][3], vf[2 * j], vf[2 * j + 1]);
                            mma_bf16(ol[i], al[j][0], al[j][1], al[j][2], al[j][3], vf[2 * j], vf[2 * j + 1]);
                        }
                    }
                }
                if (next < q.k1) {
                    __syncthreads();                              // every warp is past this V
                    load_rows(vp, vs, next, next, end);
                }
                cp_async_commit();
            }
            cp_async_wait<0>();
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                l_run[hf] += __shfl_xor_sync(0xFFFFFFFFu, l_run[hf], 1);
                l_run[hf] += __shfl_xor_sync(0xFFFFFFFFu, l_run[hf], 2);
                if (t == 0) s_l[(g + 8 * hf) * NW + warp] = l_run[hf];
            }
#pragma unroll
            for (int i = 0; i < NTW; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) oh[i][e] += ol[i][e];
            __syncthreads();
            float* part = a.part + (size_t)u * 16 * (HD + 2);
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int row = g + 8 * hf, rho = q.slab * 16 + row;
                float L = 0.f;
#pragma unroll
                for (int i = 0; i < NW; i += 4) {
                    const float4 x = *reinterpret_cast<const float4*>(s_l + row * NW + i);
                    L += (x.x + x.y) + (x.z + x.w);
                }
                if (a.splits == 1) {
                    const float inv = L > 0.f ? 1.0f / L : 0.f;
#pragma unroll
                    for (int i = 0; i < NTW; ++i) {
                        uint32_t h, l;
                        split_bf16x2(oh[i][2 * hf] * inv, oh[i][2 * hf + 1] * inv, h, l);
                        if (rho < G) {
                            __nv_bfloat16* p = a.o + out_at(a, q, rho, gq, (cg + i) * 8 + 2 * t);
                            *reinterpret_cast<uint32_t*>(p) = h;
                            *reinterpret_cast<uint32_t*>(p + 512) = l;
                        }
                    }
                } else {
                    // split key range: park (O, max, sum); the CTA that finishes last merges the ranges in order
#pragma unroll
                    for (int i = 0; i < NTW; ++i)
                        *reinterpret_cast<float2*>(part + row * HD + (cg + i) * 8 + 2 * t) = make_float2(oh[i][2 * hf], oh[i][2 * hf + 1]);
                    if (warp == 0 && t == 0) *reinterpret_cast<float2*>(part + 16 * HD + row * 2) = make_float2(m_run[hf], L);
                }
            }
            TL_STAMP(2);
            if (a.splits > 1) merge();
        }
        return true;
    }

    // element offset of a query row's column in the O-projection's input
    static __device__ __forceinline__ unsigned out_at(const PersistArgs& a, const Unit& q, int rho, int gq, int col) {
        const int hl = div_r(a, rho);
        return act_at(q.b * a.R + rho - hl * a.R, (q.kh * gq + hl) * HD + col, a.qd >> 6);
    }

    static __device__ __noinline__ void merge() {
        const PersistArgs& a = sh().args;
        const Unit& q = sh().unit;
        const int gq = a.n_q / a.n_kv, G = gq * a.R;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned old;
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(a.unit_ctr + q.group) : "memory");
            sh().last = old == (unsigned)(a.splits - 1);
            if (sh().last) a.unit_ctr[q.group] = 0u;              // everyone else has left this counter; visible by the next barrier
        }
        __syncthreads();
        if (!sh().last) return;
        const float* base = a.part + (size_t)q.group * a.splits * 16 * (HD + 2);
        // one trip to L2: every range of every item of this thread is requested before the first is used; a range without
        // visible keys has weight zero
        constexpr int NI = 16 * (HD / 4) / NT, NS = PERSIST_MAX_SPLITS;
        float2 ml[NI][NS];
        float4 o4[NI][NS];
#pragma unroll
        for (int e = 0; e < NI; ++e) {
            const int i = threadIdx.x + e * NT, r = i / (HD / 4), d4 = (i % (HD / 4)) * 4;
            const float *p = base + r * HD + d4, *pm = base + 16 * HD + r * 2;
#pragma unroll
            for (int sp = 0; sp < NS; ++sp) {
                ml[e][sp] = make_float2(-INFINITY, 0.f);
                o4[e][sp] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (sp < a.splits) {
                    ml[e][sp] = __ldcg(reinterpret_cast<const float2*>(pm + sp * (16 * (HD + 2))));
                    o4[e][sp] = __ldcg(reinterpret_cast<const float4*>(p + sp * (16 * (HD + 2))));
                }
            }
        }
#pragma unroll
        for (int e = 0; e < NI; ++e) {
            const int i = threadIdx.x + e * NT, r = i / (HD / 4), d4 = (i % (HD / 4)) * 4, rho = q.slab * 16 + r;
            float mn = -INFINITY, den = 0.f;
#pragma unroll
            for (int sp = 0; sp < NS; ++sp) mn = fmaxf(mn, ml[e][sp].x);
            const float mu = mn == -INFINITY ? 0.f : mn;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int sp = 0; sp < NS; ++sp) {
                const float wgt = exp2f(ml[e][sp].x - mu);
                den += wgt * ml[e][sp].y;
                acc.x += wgt * o4[e][sp].x; acc.y += wgt * o4[e][sp].y; acc.z += wgt * o4[e][sp].z; acc.w += wgt * o4[e][sp].w;
            }
            if (rho >= G) continue;
            const float inv = den > 0.f ? 1.0f / den : 0.f;
            uint2 h, l;
            split_bf16x2(acc.x * inv, acc.y * inv, h.x, l.x);
            split_bf16x2(acc.z * inv, acc.w * inv, h.y, l.y);
            __nv_bfloat16* dst = a.o + out_at(a, q, rho, gq, d4);
            *reinterpret_cast<uint2*>(dst) = h;
            *reinterpret_cast<uint2*>(dst + 512) = l;
        }
    }
};

template <int HD, int T>
__global__ void __launch_bounds__(WARPS * 32, 1) layers_kernel(const __grid_constant__ PersistArgs a) {
    constexpr int TOK = T * 8, NT = Cta<HD, T>::NT;
    static_assert(TOK <= MAX_TOK, "token rows per CTA");
    const int tid = threadIdx.x;
    const bool in_grid = (int)blockIdx.x < a.n_tb * a.n_rb;
    const int rb = blockIdx.x / a.n_tb, m0 = (blockIdx.x % a.n_tb) * TOK;
    Cta<HD, T> c{a, 1};
    if (tid == 0) { sh().stop = 0; sh().unit = Unit{}; sh().m0 = m0; }
    if (tid < 6) {
        const unsigned n = (tid >> 1) == 0 ? (unsigned)(a.qd / 2 + a.n_kv * HD) : (tid >> 1) == 1 ? (unsigned)a.d : (unsigned)a.dff;
        const int blocks = (tid >> 1) == 1 ? a.n_res : a.n_rb;
        sh().part[tid >> 1][tid & 1] = in_grid && rb < blocks ? (int)(n * (unsigned)(rb + (tid & 1)) / (unsigned)blocks) : 0;
    }
    if (tid < TOK) {
        const int m = m0 + tid;
        int pos = m < a.M ? a.row_pos[m] : -1;
        if (pos >= a.max_positions) { set_status(a.status, TASC_EINVAL); pos = -1; }
        long long off = -1;
        if (pos >= 0) {
            const int ps = pos / a.page_size;
            int page = -1;
            if (ps < a.max_pages) page = a.block_table[(size_t)(m / a.R) * a.max_pages + ps];
            if (page < 0 || page >= a.n_pages) set_status(a.status, TASC_ENOKV);
            else off = ((long long)page * a.n_kv * a.page_size + pos % a.page_size) * HD;
        }
        sh().pos[tid] = pos;
        sh().koff[tid] = off;
    }
    for (int i = tid; i < (int)(sizeof(PersistArgs) / 4); i += NT) reinterpret_cast<unsigned*>(&sh().args)[i] = reinterpret_cast<const unsigned*>(&a)[i];
#pragma unroll 1
    for (int i = tid; i < a.n_layers * (int)(sizeof(LayerWeights) / 8); i += NT)
        reinterpret_cast<unsigned long long*>(sh().layers)[i] = reinterpret_cast<const unsigned long long*>(a.layers)[i];
    __syncthreads();
    if ((int)blockIdx.x < a.n_units) c.prepare_unit(blockIdx.x);
    if (tid == 0) set_phase<HD>(0, 0, sh().phase[0]);
#pragma unroll 1
    for (int i = tid; i < a.nt_qkv * T * 64; i += NT) {
        const int row = i & 7, n = (i >> 3) & 7, tt = (i >> 6) % T, tile = i / (64 * T);
        const int f = sh().part[0][0] + tile * 8 + row, pos = sh().pos[tt * 8 + n];
        c.s_cs()[i] = f < sh().part[0][1] && f < (a.n_q + a.n_kv) * (HD / 2) && pos >= 0 ? a.rope[(size_t)pos * (HD / 2) + f % (HD / 2)] : make_float2(1.f, 0.f);
    }
#pragma unroll 1
    for (int i = tid; i < a.nt_res * T * 128; i += NT) {
        const int row = i & 15, n = (i >> 4) & 7, tt = (i >> 7) % T, tile = i / (128 * T);
        const int f = sh().part[1][0] + tile * 16 + row, m = m0 + tt * 8 + n;
        c.xs()[i] = f < sh().part[1][1] && m < a.M ? a.x0[(size_t)m * a.d + f] : 0.f;
    }
#ifdef TASC_TIMELINE
    if (tid == 0) { sh().tl[0] = global_ns(); sh().tl[2] = 0; }
#endif
    grid_arrive(a);                                               // (also makes the shared arrays visible to the CTA)
    // (one call of each routine: the layer loop has to stay within the instruction caches -- measured, an SM fetches code
    // that is not in its 32 KB cache at about five cycles per instruction, which is more than a phase's work)
    int slot = 0;
#pragma unroll 1
    for (int l = 0; l < a.n_layers; ++l) {
#pragma unroll 1
        for (int j = 0; j < 5; ++j) {
            if (j == 1) {
                __nv_bfloat16* kp = a.kv_pool + (size_t)l * 2 * a.kv_half;
                if (!c.attention(kp, kp + a.kv_half)) return;
            } else {
                if (!c.project(sh().phase[slot], l + (j == 4), j == 0 ? 2 : j == 4 ? 0 : j + 1, sh().phase[slot ^ 1])) return;
                if (l + 1 == a.n_layers && j == 4) { TL_PHASE(j); return; }
                slot ^= 1;
            }
            grid_arrive(a);
            TL_PHASE(j);
            ++c.epoch;
        }
    }
}

template <int HD, int T>
tasc_status launch_inst(const PersistArgs& a, const PersistPlan& p, cudaStream_t stream) {
    static std::mutex mu;
    static bool attr_done[64] = {false};
    int dev = 0;
    TASC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return TASC_EINVAL;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!attr_done[dev]) {
            TASC_CUDA_TRY(cudaFuncSetAttribute(layers_kernel<HD, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM));
            attr_done[dev] = true;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.grid, 1, 1);
    cfg.blockDim = dim3(WARPS * 32, 1, 1);
    cfg.dynamicSmemBytes = (size_t)p.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;                    // every CTA waits for every other: all must be resident
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ProfScope ps(K_LAYERS, stream);
    TASC_CUDA_TRY(cudaLaunchKernelEx(&cfg, layers_kernel<HD, T>, a));
    return TASC_OK;
}

}  // namespace

bool plan_persist(int n_layers, int M, int B, int R, int d, int qd, int n_q, int n_kv, int hd, int dff, int max_ctx, int page_size, PersistPlan& p) {
    if (n_layers > PERSIST_MAX_LAYERS || max_ctx / std::max(page_size, 1) > MAX_PAGES) return false;
    if (M < 1 || M > PERSIST_MAX_ROWS || (hd != 64 && hd != 128) || d % CHUNK || qd % CHUNK || dff % CHUNK) return false;
    if ((R > 16 && R % 16) || page_size < 1 || (page_size & (page_size - 1))) return false;
    static std::mutex mu;
    static int sms[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return false; }
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!sms[dev] && (cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms[dev] < 1)) {
            (void)cudaGetLastError();
            sms[dev] = 0;
            return false;
        }
        p.grid = sms[dev];
    }
    if (M > 16 && M <= 32) return false;             // (one block of four tiles: slower than kernels per phase, see persist_pays)
    p.T = M <= 8 ? 1 : (M <= 16 ? 2 : 4);
    p.n_tb = (M + p.T * 8 - 1) / (p.T * 8);
    p.n_rb = p.grid / p.n_tb;
    if (p.n_rb < 1) return false;
    // (blocks of a residual projection have 8 rows or more: each adds to the sums of squares of all token rows)
    p.n_res = std::min(p.n_rb, d / 8);
    p.nt_res = ((d + p.n_res - 1) / p.n_res + 15) / 16;
    if (p.n_res * p.nt_res > SSQ_MAX_ADDS) return false;
    const int qkv_pairs = qd / 2 + n_kv * hd;
    p.nt_qkv = ((qkv_pairs + p.n_rb - 1) / p.n_rb + 7) / 8;
    const int x_bytes = p.nt_res * p.T * 128 * 4 + p.nt_qkv * p.T * 64 * 8;      // residual rows, rotary factors
    p.union_bytes = hd == 64 ? Cta<64, 1>::ATT_BYTES : Cta<128, 1>::ATT_BYTES;                     // the parked tiles take what there is
    p.smem_bytes = SHARED_BYTES + p.union_bytes + x_bytes;
    if (p.smem_bytes > MAX_SMEM) return false;
    // how the warps of a CTA split a projection: row groups x k groups, by the longest chain of 64-wide chunks a warp walks
    const int rows[4] = {qkv_pairs, d, dff, d}, blocks[4] = {p.n_rb, p.n_res, p.n_rb, p.n_res}, per[4] = {8, 16, 8, 16}, red[4] = {d, qd, d, dff};
    for (int j = 0; j < 4; ++j) {
        const int tiles = ((rows[j] + blocks[j] - 1) / blocks[j] + per[j] - 1) / per[j], chunks = red[j] / CHUNK;
        int best = 1 << 30;
        for (int lr = 0; lr <= LW; ++lr) {
            const int rg = 1 << lr, kg = WARPS >> lr;
            const int steps = ((tiles + rg - 1) / rg) * ((chunks + kg - 1) / kg);
            if (steps < best) { best = steps; p.lr[j] = lr; }      // ties: fewer row groups, so that a warp's activations stay in registers
        }
    }
    // attention units: key ranges of about one tile each as long as that fills no more than one wave
    const int G = (n_q / n_kv) * R;
    p.n_slabs = (G + 15) / 16;
    const int groups = B * n_kv * p.n_slabs;
    const int want = std::max(1, (max_ctx + 127) / 128);
    p.splits = std::max(1, std::min({want, p.grid / groups, PERSIST_MAX_SPLITS}));
    p.n_units = groups * p.splits;
    if (groups > PERSIST_MAX_GROUPS || (p.splits > 1 && p.n_units > PERSIST_MAX_UNITS)) return false;
    return true;
}

tasc_status launch_persist(PersistArgs a, const PersistPlan& p, cudaStream_t stream) {
    a.n_tb = p.n_tb; a.n_rb = p.n_rb; a.nt_res = p.nt_res; a.nt_qkv = p.nt_qkv; a.park_bytes = p.union_bytes; a.n_res = p.n_res;
    for (int j = 0; j < 4; ++j) a.lr[j] = p.lr[j];
    a.r_magic = (unsigned)(((1ull << 32) + a.R - 1) / a.R);        // exact for quotients of numbers below 2^16
    a.tbl_magic = (unsigned)(((1ull << 32) + a.TBL - 1) / a.TBL);
    a.page_shift = 0;
    while ((1 << a.page_shift) < a.page_size) ++a.page_shift;
    a.union_bytes = p.union_bytes; a.splits = p.splits; a.n_slabs = p.n_slabs; a.n_units = p.n_units;
    if (a.hd == 64) return p.T == 1 ? launch_inst<64, 1>(a, p, stream) : p.T == 2 ? launch_inst<64, 2>(a, p, stream) : launch_inst<64, 4>(a, p, stream);
    return p.T == 1 ? launch_inst<128, 1>(a, p, stream) : p.T == 2 ? launch_inst<128, 2>(a, p, stream) : launch_inst<128, 4>(a, p, stream);
}

}  // namespace tasc
