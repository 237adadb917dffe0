// On-device n-gram drafter (TASC-draft): corpus tables p_corp, context model p_prompt, exact mixture argmax.
//
// Build (once per task): the windows (n context tokens, next token) of every order n = 1..n_max are counted exactly, in an
// open-addressing table whose 16-byte slots hold key, count and one position of the n-gram: a window's whole update is one
// 32-byte sector.  Order 1 is keyed by its two tokens, order n by the slot of its prefix in order n - 1's table and its
// last token, which is as exact and half as long.  A window can only reach p_min if the two windows of order n - 1 inside
// it have, so each order counts only what the order before left over.  Elements with count >= p_min are listed and moved
// into the final per-order structure: a context table (packed context -> offset, number of successors, total count) plus
// a flat successor array of (next, count).  Slot placement depends on thread timing, results do not: lookups return the
// same sets, and the export sorts canonically.
//
// Draft (every step): one CTA per sequence.  For each of the k drafts: warp-cooperative probes of the
// context tables of all orders at once (one warp per order, 32 slots per probe round; longest hit wins), a scan of the sequence's committed tokens for the
// longest matching suffix with its successor counts collected in a shared-memory hash, and the argmax
// of  lambda_num * c_corp(x) * T_prompt + (lambda_den - lambda_num) * c_prompt(x) * T_corp  in 64-bit
// integers with the smallest token id winning ties.
#include "kernels.h"
#include "ngram_table.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <vector>

struct CtxVal {
    unsigned long long offset;   // first successor in the order's successor array
    uint32_t n_succ;
    uint32_t total;              // sum of the surviving counts
};
struct Succ {
    int32_t next;
    uint32_t count;
};
struct OrderTable {
    uint64_t* keys;              // [cap][2]
    CtxVal* vals;                // [cap]
    Succ* succ;                  // [n_succ]
    uint64_t mask;               // cap - 1
    long long n_succ;
};
struct DeviceTables {
    OrderTable t[TASC_MAX_ORDER + 1];   // index = order n
    int n_max;
    int fallback;
};

struct tasc_drafter {
    DeviceTables dt;
    tasc::DeviceSlab slab[TASC_MAX_ORDER + 1];      // the memory of dt.t[n]
    int p_min, vocab, device;
};

namespace tasc {
namespace {

// ------------------------------------------------------------------------------------------- corpus
// What the host has to know about the documents before it can allocate.
struct CorpusCheck { unsigned long long pairs; long long tokens; int bad; };
__global__ void corpus_check_kernel(const int64_t* __restrict__ offsets, int64_t n_docs, CorpusCheck* out) {
    unsigned long long w = 0;
    bool bad = false;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < n_docs; d += step) {
        const int64_t len = offsets[d + 1] - offsets[d];
        if (len < 0) bad = true;
        else if (len > 1) w += (unsigned long long)(len - 1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xFFFFFFFFu, w, o);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd(&out->pairs, w);
    if (bad || (blockIdx.x == 0 && threadIdx.x == 0 && offsets[0] != 0)) out->bad = 1;
    if (blockIdx.x == 0 && threadIdx.x == 0) out->tokens = offsets[n_docs];
}
tasc_status check_corpus(const int64_t* offsets, int64_t n_docs, CorpusCheck& h, cudaStream_t stream) {
    DeviceSlab slab;
    const size_t o = slab.add(sizeof(CorpusCheck));
    if (!slab.allocate(stream)) return TASC_ENOMEM;
    TASC_CUDA_TRY(cudaMemsetAsync(slab.at<CorpusCheck>(o), 0, sizeof(h), stream));
    corpus_check_kernel<<<std::min(blocks_for((uint64_t)n_docs + 1, 256), 592u), 256, 0, stream>>>(offsets, n_docs, slab.at<CorpusCheck>(o));
    TASC_CUDA_TRY(cudaMemcpyAsync(&h, slab.at<CorpusCheck>(o), sizeof(h), cudaMemcpyDeviceToHost, stream));
    TASC_CUDA_TRY(cudaStreamSynchronize(stream));
    return h.bad || h.tokens < 0 ? TASC_EINVAL : TASC_OK;
}

// remaining[i] = number of tokens after position i inside its document, clamped to 255; and the histogram of the tokens.
// A block takes a run of the corpus, SCAN_POS positions at a time.  Its first warp searches the offsets for the run's first document, 32
// ways at once; from there the documents that begin in the next positions are set as bits, and a position's distance to the next
// bit is what remains.  The first tokens that fall on a line of the block's cache are counted there (a token can be per cents of
// the corpus), the others are an atomic each.  14 M tokens: 0.50 ms without that cache; 0.155 when two threads searched the documents
// of every SCAN_POS positions (18 dependent trips), every position searched among those, and the cache had 2,048 lines; 0.12 with
// bits and 2,048 lines, 0.089 with 4,096.
constexpr int SCAN_THREADS = 512, SCAN_PER = 8, SCAN_POS = SCAN_THREADS * SCAN_PER, SCAN_LINES = 4096;
__global__ void __launch_bounds__(SCAN_THREADS)
corpus_scan_kernel(const int32_t* __restrict__ tokens, const int64_t* __restrict__ offsets, int64_t n_docs, int64_t T, int vocab,
                   uint8_t* __restrict__ remaining, uint32_t* hist, int* status) {
    __shared__ uint32_t s_begin[SCAN_POS / 32];                  // documents begin here (or the corpus ends)
    __shared__ unsigned long long s_doc;                         // last document that begins at or before the next positions
    __shared__ int64_t s_end;                                    // end of the last position's document
    __shared__ int s_tok[SCAN_LINES];
    __shared__ uint32_t s_cnt[SCAN_LINES];
    for (int i = threadIdx.x; i < SCAN_LINES; i += SCAN_THREADS) { s_tok[i] = -1; s_cnt[i] = 0u; }
    const int64_t runs = (T + SCAN_POS - 1) / SCAN_POS, first = runs * blockIdx.x / gridDim.x, last = runs * (blockIdx.x + 1) / gridDim.x;
    if (threadIdx.x < 32 && first < last) {
        int64_t lo = 0, hi = n_docs;                             // last document in [lo, hi) that begins at or before the run
        while (hi - lo > 1) {
            const int64_t step = (hi - lo + 31) / 32, d = lo + threadIdx.x * step;
            const uint32_t yes = __ballot_sync(0xFFFFFFFFu, d < hi && offsets[d] <= first * SCAN_POS);
            lo += (31 - __clz(yes)) * step;
            hi = min(hi, lo + step);
        }
        if (threadIdx.x == 0) s_doc = (unsigned long long)lo;
    }
    for (int64_t r = first; r < last; ++r) {
        const int64_t p0 = r * SCAN_POS, p1 = p0 + SCAN_POS;
        int tok[SCAN_PER];
#pragma unroll
        for (int u = 0; u < SCAN_PER; ++u) {
            const int64_t i = p0 + u * SCAN_THREADS + threadIdx.x;
            tok[u] = i < T ? tokens[i] : 0;
        }
        if (threadIdx.x < SCAN_POS / 32) s_begin[threadIdx.x] = 0u;
        __syncthreads();
        const int64_t d0 = (int64_t)s_doc;
        __syncthreads();
        for (int64_t d = d0 + 1 + threadIdx.x;; d += SCAN_THREADS) {
            const int64_t o = d <= n_docs ? offsets[d] : p1 + 1;
            // the first document that begins behind the positions: its predecessor holds the last one
            if (o >= p1) {
                if (d <= n_docs ? d == d0 + 1 || offsets[d - 1] < p1 : false) s_end = o;
                if (o > p1) break;
            } else if (o > p0) atomicOr(&s_begin[(o - p0) >> 5], 1u << ((o - p0) & 31));
            if (d < n_docs) atomicMax(&s_doc, (unsigned long long)d);
            if (d >= n_docs) { if (o < p1) s_end = o; break; }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < SCAN_PER; ++u) {
            const int x = u * SCAN_THREADS + threadIdx.x;
            const int64_t i = p0 + x;
            if (i >= T) break;
            // the next beginning behind the position, within 256; else the document ends behind these positions
            int w = x >> 5;
            uint32_t bits = s_begin[w] & ~((2u << (x & 31)) - 1u);
            const int stop = min(w + 9, SCAN_POS / 32);
            while (!bits && ++w < stop) bits = s_begin[w];
            const int64_t end = bits ? p0 + w * 32 + __ffs(bits) - 1 : w < SCAN_POS / 32 ? i + 256 : s_end;
            remaining[i] = (uint8_t)min(end - i - 1, (int64_t)255);
            const int t = tok[u], line = t & (SCAN_LINES - 1);
            if (t < 0 || t >= vocab) { set_status(status, TASC_EINVAL); continue; }
            int have = *(volatile int*)&s_tok[line];
            if (have == -1) { have = atomicCAS(&s_tok[line], -1, t); if (have == -1) have = t; }
            if (have == t) atomicAdd(&s_cnt[line], 1u); else atomicAdd(&hist[t], 1u);
        }
        __syncthreads();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SCAN_LINES; i += SCAN_THREADS)
        if (s_cnt[i]) atomicAdd(&hist[s_tok[i]], s_cnt[i]);
}
inline unsigned scan_blocks(int64_t T) { return std::min(blocks_for((uint64_t)T, SCAN_POS), 4u * 148u); }
__global__ void hist_argmax_kernel(const uint32_t* __restrict__ hist, int vocab, unsigned long long* best) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long v = i < vocab ? ((unsigned long long)hist[i] << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)i) : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    if ((threadIdx.x & 31) == 0) atomicMax(best, v);
}

// ------------------------------------------------------------------------------------------- counting
// Two slots to a sector; a key is in the first pair from its home pair on that had room.  (Memory goes by sectors: one per
// window here, against two when keys of 16 bytes and counts were arrays of their own.  Filled to 4/5 at most, 1.25 slots per
// window: a table of a power of two had 2 to 4.)
struct __align__(16) CountSlot { unsigned long long key; uint32_t count, pos; };
struct CountTable { CountSlot* slots; uint32_t pairs; };
constexpr uint32_t NO_SLOT = 0xFFFFFFFFu;
inline uint64_t count_pairs(uint64_t windows) { return (windows + windows / 4) / 2 + 32; }

__device__ __forceinline__ uint64_t mix64(uint64_t k) {
    k ^= k >> 32; k *= 0xD6E8FEB86659FD93ull; k ^= k >> 29; k *= 0x9E3779B97F4A7C15ull; k ^= k >> 32;
    return k;
}
// Counts `add` occurrences of a window; its slot, or NO_SLOT when the table is full.
__device__ __forceinline__ uint32_t count_window(const CountTable& t, unsigned long long key, uint32_t pos, uint32_t add) {
    uint32_t pair = (uint32_t)__umul64hi(mix64(key), (uint64_t)t.pairs);
    for (uint32_t probe = 0; probe < t.pairs; ++probe) {
        CountSlot* s = t.slots + 2 * (size_t)pair;
        // (one request for both keys; what lies between them is not used)
        unsigned long long k0, k1;
        asm volatile("{\n\t.reg .b64 c0, c1;\n\tld.relaxed.gpu.global.v4.b64 {%0, c0, %1, c1}, [%2];\n\t}" : "=l"(k0), "=l"(k1) : "l"(s) : "memory");
        // (an empty slot is claimed whole: key, count and position in one atomic, where they were three requests.  A task of 200,000
        // documents 2067 -> 1999 us.)
        const Key slot = {key, (unsigned long long)add | ((unsigned long long)pos << 32)};
        if (k0 == 0ull) {
            k0 = cas128(reinterpret_cast<uint64_t*>(s), Key{0ull, 0ull}, slot).lo;
            if (k0 == 0ull) return 2 * pair;
        }
        if (k0 != key && k1 == 0ull) {
            k1 = cas128(reinterpret_cast<uint64_t*>(s + 1), Key{0ull, 0ull}, slot).lo;
            if (k1 == 0ull) return 2 * pair + 1;
        }
        if (k0 == key || k1 == key) {
            const int i = k0 == key ? 0 : 1;
            atomicAdd(&s[i].count, add);
            return 2 * pair + i;
        }
        pair = pair + 1 == t.pairs ? 0 : pair + 1;
    }
    return NO_SLOT;
}

// A block's own counts of the first keys it meets, one per line (the frequent ones are among them).  Text has windows that
// are a per cent of all: counted in the table directly, each is half a million atomics on one word, one after the other.
// 14 M tokens, per order: 1.6 ms without, 0.19 to 0.28 ms with it.  Two blocks of 64 KB fill an SM's threads.
constexpr int CACHE_LINES = 4096, COUNT_THREADS = 1024;
struct CountCache {
    unsigned long long key[CACHE_LINES];
    uint32_t slot[CACHE_LINES], count[CACHE_LINES];
    __device__ __forceinline__ void clear() {
        for (int i = threadIdx.x; i < CACHE_LINES; i += COUNT_THREADS) { key[i] = 0ull; slot[i] = NO_SLOT; count[i] = 0u; }
        __syncthreads();
    }
    __device__ __forceinline__ uint32_t add(const CountTable& t, unsigned long long k, uint32_t pos) {
        const uint32_t line = (uint32_t)(mix64(k) & (CACHE_LINES - 1));
        unsigned long long have = *(volatile unsigned long long*)&key[line];
        if (have == 0ull) {
            have = atomicCAS(&key[line], 0ull, k);
            if (have == 0ull) {                  // this thread brings the line in
                const uint32_t s = count_window(t, k, pos, 1u);
                *(volatile uint32_t*)&slot[line] = s;
                return s;
            }
        }
        if (have == k) {
            const uint32_t s = *(volatile uint32_t*)&slot[line];
            if (s != NO_SLOT) { atomicAdd(&count[line], 1u); return s; }
        }
        return count_window(t, k, pos, 1u);
    }
    __device__ __forceinline__ void flush(const CountTable& t) {
        __syncthreads();
        for (int i = threadIdx.x; i < CACHE_LINES; i += COUNT_THREADS)
            if (count[i]) atomicAdd(&t.slots[slot[i]].count, count[i]);
    }
};
// One window per position, n tokens of context and the next one.  Order 1 is keyed by its tokens; order n by prev[i], the slot
// of the order n - 1 window at i (NO_SLOT if there is none or it is too rare), and needs the one at i + 1 too.
// id[i] = the window's slot (id may be null).  Two blocks per SM stay for the whole corpus.
template <bool FIRST>
__global__ void __launch_bounds__(COUNT_THREADS, 2)
count_kernel(const int32_t* __restrict__ tokens, const uint8_t* __restrict__ remaining, int64_t T, int n, const uint32_t* __restrict__ prev,
             CountTable t, uint32_t* __restrict__ id, int* status) {
    extern __shared__ __align__(16) uint8_t count_smem[];
    CountCache& cache = *reinterpret_cast<CountCache*>(count_smem);
    cache.clear();
    const int64_t step = (int64_t)gridDim.x * COUNT_THREADS;
    for (int64_t i = (int64_t)blockIdx.x * COUNT_THREADS + threadIdx.x; i < T; i += step) {
        uint32_t slot = NO_SLOT;
        bool there = remaining[i] >= n;
        unsigned long long head = 0ull;
        if (FIRST) head = (unsigned long long)((uint32_t)tokens[i] & TOK_MASK);
        else if (there) {
            head = prev[i];
            there = prev[i] != NO_SLOT && prev[i + 1] != NO_SLOT;
        }
        if (there) {
            slot = cache.add(t, VALID_BIT | (head << TOK_BITS) | ((uint32_t)tokens[i + n] & TOK_MASK), (uint32_t)i);
            if (slot == NO_SLOT) set_status(status, TASC_ECAPACITY);
        }
        if (id) id[i] = slot;
    }
    cache.flush(t);
}
template <bool FIRST>
tasc_status launch_count(const int32_t* tokens, const uint8_t* remaining, int64_t T, int n, const uint32_t* prev, const CountTable& t, uint32_t* id,
                         int* status, cudaStream_t stream) {
    TASC_CUDA_TRY(cudaFuncSetAttribute(count_kernel<FIRST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CountCache)));
    const unsigned blocks = std::min(blocks_for((uint64_t)T, COUNT_THREADS), 2u * 148u);
    count_kernel<FIRST><<<blocks, COUNT_THREADS, sizeof(CountCache), stream>>>(tokens, remaining, T, n, prev, t, id, status);
    TASC_CUDA_TRY(cudaGetLastError());
    return TASC_OK;
}
// Takes the windows that stay below p_min out of id, and counts the positions where the next order has to look.  Which slots are
// frequent comes as bits (list_kernel): 2 MB of them for 14 M windows, which L2 answers, against a sector of a table of 280 MB per
// position.  (14 M positions, orders 1 / 2 / 3: 133 / 87 / 86 us with the counts looked up in the table, 42 / 30 / 29 with bits.)
constexpr int PRUNE_PER = 4;
__global__ void __launch_bounds__(256)
prune_kernel(uint32_t* __restrict__ id, const uint8_t* __restrict__ remaining, int64_t T, int n, const uint32_t* __restrict__ frequent, unsigned long long* n_next) {
    __shared__ uint32_t s_n;
    const int64_t p = ((int64_t)blockIdx.x * 256 + threadIdx.x) * PRUNE_PER;
    const bool whole = p + PRUNE_PER <= T;
    if (threadIdx.x == 0) s_n = 0;
    uint32_t v[PRUNE_PER + 1], rem = 0u;                     // one more: the position behind
    if (whole) {
        const uint4 x = *reinterpret_cast<const uint4*>(id + p);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        rem = *reinterpret_cast<const uint32_t*>(remaining + p);
    } else {
        for (int j = 0; j < PRUNE_PER; ++j) {
            v[j] = p + j < T ? id[p + j] : NO_SLOT;
            if (p + j < T) rem |= (uint32_t)remaining[p + j] << (8 * j);
        }
    }
    // (the warp behind may have taken it out already, which gives the same answer)
    v[PRUNE_PER] = (threadIdx.x & 31) == 31 && p + PRUNE_PER < T ? *(volatile const uint32_t*)(id + p + PRUNE_PER) : NO_SLOT;
#pragma unroll
    for (int j = 0; j <= PRUNE_PER; ++j)
        if (v[j] != NO_SLOT && !((frequent[v[j] >> 5] >> (v[j] & 31)) & 1u)) v[j] = NO_SLOT;
    const uint32_t behind = __shfl_down_sync(0xFFFFFFFFu, v[0], 1);
    if ((threadIdx.x & 31) != 31) v[PRUNE_PER] = behind;
    uint32_t next = 0u;
#pragma unroll
    for (int j = 0; j < PRUNE_PER; ++j)
        next += v[j] != NO_SLOT && v[j + 1] != NO_SLOT && (int)((rem >> (8 * j)) & 255u) >= n + 1 ? 1u : 0u;
    next = __reduce_add_sync(0xFFFFFFFFu, next);
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && next) atomicAdd(&s_n, next);
    if (whole) *reinterpret_cast<uint4*>(id + p) = make_uint4(v[0], v[1], v[2], v[3]);
    else for (int j = 0; j < PRUNE_PER; ++j) if (p + j < T) id[p + j] = v[j];
    __syncthreads();
    if (threadIdx.x == 0 && s_n) atomicAdd(n_next, (unsigned long long)s_n);
}

// ------------------------------------------------------------------------------------------- tables
struct Survivor { uint32_t pos, count; };
// Lists the n-grams that occur at least p_min times.  One reservation per block of LIST_SLOTS slots.  frequent: a bit per slot (or null).
constexpr int LIST_PER = 16, LIST_SLOTS = 256 * LIST_PER;
__global__ void __launch_bounds__(256)
list_kernel(CountTable t, uint32_t p_min, Survivor* __restrict__ list, unsigned long long* n_list, uint32_t* __restrict__ frequent) {
    __shared__ uint32_t s_n;
    __shared__ unsigned long long s_base;
    const uint64_t n_slots = 2 * (uint64_t)t.pairs, s0 = (uint64_t)blockIdx.x * LIST_SLOTS + threadIdx.x;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    Survivor v[LIST_PER];
    uint32_t at[LIST_PER];
#pragma unroll
    for (int u = 0; u < LIST_PER; ++u) {
        const uint64_t s = s0 + u * 256;
        v[u] = Survivor{0u, 0u};
        if (s < n_slots) {
            const uint4 x = *reinterpret_cast<const uint4*>(t.slots + s);
            v[u] = Survivor{x.w, x.z};
        }
    }
#pragma unroll
    for (int u = 0; u < LIST_PER; ++u) {
        const bool yes = v[u].count >= p_min;
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, yes);
        uint32_t base = 0;
        if ((threadIdx.x & 31) == 0 && frequent && s0 + u * 256 < n_slots) frequent[(s0 + u * 256) >> 5] = b;
        if ((threadIdx.x & 31) == 0 && b) base = atomicAdd(&s_n, (uint32_t)__popc(b));
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        at[u] = yes ? base + __popc(b & ((1u << (threadIdx.x & 31)) - 1u)) : NO_SLOT;
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_n) s_base = atomicAdd(n_list, (unsigned long long)s_n);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < LIST_PER; ++u)
        if (at[u] != NO_SLOT) list[s_base + at[u]] = v[u];
}

// The elements of one order: from the corpus (a list of positions), or packed (tasc_drafter_import).
struct CorpusElements {
    const int32_t* tokens;
    const Survivor* list;
    __device__ __forceinline__ void get(uint64_t i, int n, Key& ctx, int& next, uint32_t& count) const {
        const Survivor s = list[i];
        ctx = key_make(n);
        for (int j = 0; j < n; ++j) key_put(ctx, j, (uint32_t)tokens[(size_t)s.pos + j]);
        next = (int)((uint32_t)tokens[(size_t)s.pos + n] & TOK_MASK);
        count = s.count;
    }
};
struct PackedElements {
    const uint64_t* keys;
    const uint32_t* counts;
    __device__ __forceinline__ void get(uint64_t i, int n, Key& ctx, int& next, uint32_t& count) const {
        const Key e = {keys[2 * i], keys[2 * i + 1]};
        ctx = key_make(n);
        for (int j = 0; j < n; ++j) key_put(ctx, j, key_get(e, j));
        next = (int)key_get(e, n);
        count = counts[i];
    }
};
// place[i] = (slot of the element's context, its number among the context's successors)
template <typename Elements>
__global__ void __launch_bounds__(256) ctx_insert_kernel(Elements el, uint64_t n_el, int n, OrderTable t, uint2* __restrict__ place, int* status) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_el) return;
    Key ctx;
    int next;
    uint32_t count;
    el.get(i, n, ctx, next, count);
    const uint64_t slot = table_upsert(t.keys, t.mask, ctx);
    if (slot == ~0ull) { set_status(status, TASC_ECAPACITY); place[i] = make_uint2(NO_SLOT, 0u); return; }
    // (n_succ, total) as one word: n_succ stays below 2^32, so nothing is carried into the total
    const unsigned long long old = atomicAdd(reinterpret_cast<unsigned long long*>(&t.vals[slot].n_succ), ((unsigned long long)count << 32) | 1ull);
    place[i] = make_uint2((uint32_t)slot, (uint32_t)old);
}
// Every context's share of the successor array; one reservation per block.
__global__ void __launch_bounds__(256) assign_offsets_kernel(OrderTable t, unsigned long long* cursor) {
    __shared__ uint32_t s_warp[8];
    __shared__ unsigned long long s_base;
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n = i <= t.mask ? t.vals[i].n_succ : 0u;
    uint32_t x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) { if (w < warp) before += s_warp[w]; total += s_warp[w]; }
    if (threadIdx.x == 0 && total) s_base = atomicAdd(cursor, (unsigned long long)total);
    __syncthreads();
    if (n) t.vals[i].offset = s_base + before + x - n;
}
template <typename Elements>
__global__ void __launch_bounds__(256) succ_fill_kernel(Elements el, uint64_t n_el, int n, OrderTable t, const uint2* __restrict__ place, int* status) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_el || place[i].x == NO_SLOT) return;
    Key ctx;
    Succ s;
    el.get(i, n, ctx, s.next, s.count);
    const unsigned long long pos = t.vals[place[i].x].offset + place[i].y;
    if (pos >= (unsigned long long)t.n_succ) { set_status(status, TASC_ECAPACITY); return; }
    t.succ[pos] = s;
}
// The table of one order from its elements.  contexts: an upper bound of how many there are.
template <typename Elements>
tasc_status build_order(tasc_drafter* d, int n, const Elements& el, uint64_t n_el, uint64_t contexts, uint2* place, unsigned long long* cursor,
                        int* status, cudaStream_t stream) {
    OrderTable& t = d->dt.t[n];
    DeviceSlab& slab = d->slab[n];
    const uint64_t ccap = pow2_at_least(2 * std::min(n_el, contexts));
    const size_t o_keys = slab.add(ccap * 16), o_vals = slab.add(ccap * sizeof(CtxVal)), o_succ = slab.add(n_el * sizeof(Succ));
    if (!slab.allocate(stream)) return TASC_ENOMEM;
    t = OrderTable{slab.at<uint64_t>(o_keys), slab.at<CtxVal>(o_vals), slab.at<Succ>(o_succ), ccap - 1, (long long)n_el};
    TASC_CUDA_TRY(cudaMemsetAsync(t.keys, 0, o_succ, stream));         // keys and values
    TASC_CUDA_TRY(cudaMemsetAsync(cursor, 0, sizeof(unsigned long long), stream));
    ctx_insert_kernel<<<blocks_for(n_el, 256), 256, 0, stream>>>(el, n_el, n, t, place, status);
    assign_offsets_kernel<<<blocks_for(ccap, 256), 256, 0, stream>>>(t, cursor);
    succ_fill_kernel<<<blocks_for(n_el, 256), 256, 0, stream>>>(el, n_el, n, t, place, status);
    TASC_CUDA_TRY(cudaGetLastError());
    return TASC_OK;
}

// Order-1 model with one successor of count 1 per context: context token c -> table[c].
__global__ void bigram_insert_kernel(const int32_t* __restrict__ table, int vocab, OrderTable t, int* status) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= vocab) return;
    const int x = table[c];
    if (x < 0 || x >= vocab) { set_status(status, TASC_EINVAL); return; }
    Key key = key_make(1);
    key_put(key, 0, (uint32_t)c);
    const uint64_t slot = table_upsert(t.keys, t.mask, key);
    if (slot == ~0ull) { set_status(status, TASC_ECAPACITY); return; }
    CtxVal v;
    v.offset = (unsigned long long)c; v.n_succ = 1u; v.total = 1u;
    t.vals[slot] = v;
    Succ sc;
    sc.next = x; sc.count = 1u;
    t.succ[c] = sc;
}

// ------------------------------------------------------------------------------------------- corpus statistics
// The statistics are functions of the multiset of counts only, so the device first turns the counts into a histogram of
// count VALUES (how many bigrams occur c times), which is exact integer work whose result does not depend on where the
// hash table put anything; that histogram is then added up in a fixed order, from the largest count value down.
constexpr int CC_BITS = 20;                       // count values below 2^20 have a histogram bin of their own
constexpr uint32_t CC_BINS = 1u << CC_BITS;
constexpr int CC_OVERFLOW = 4096;                 // larger count values are listed individually
constexpr int CC_LOW = 1024;                      // ... and nearly all counts are below this: binned in shared memory first
constexpr int STATS_THREADS = 256, BIN_PER = 16, BIN_CHUNK = STATS_THREADS * BIN_PER, BIN_CHUNKS = (int)(CC_BINS / BIN_CHUNK);

// counts[i * stride], i < n.  scal: [0] distinct keys, [1] overflow entries, [2] sum of squared counts
__global__ void __launch_bounds__(STATS_THREADS)
count_values_kernel(const uint32_t* __restrict__ counts, int stride, uint64_t n, uint32_t* __restrict__ bins,
                    uint32_t* __restrict__ overflow, unsigned long long* __restrict__ scal, int* status) {
    __shared__ uint32_t low[CC_LOW];
    for (int i = threadIdx.x; i < CC_LOW; i += STATS_THREADS) low[i] = 0u;
    __syncthreads();
    unsigned long long sq = 0ull;
    unsigned int nz = 0u;
    const uint64_t step = (uint64_t)gridDim.x * STATS_THREADS;
#pragma unroll 8
    for (uint64_t i = (uint64_t)blockIdx.x * STATS_THREADS + threadIdx.x; i < n; i += step) {
        const uint32_t c = counts[i * stride];
        if (!c) continue;
        sq += (unsigned long long)c * c;
        ++nz;
        if (c < CC_LOW) atomicAdd(&low[c], 1u);
        else if (c < CC_BINS) atomicAdd(&bins[c], 1u);
        else {
            const unsigned long long at = atomicAdd(&scal[1], 1ull);
            if (at < CC_OVERFLOW) overflow[at] = c; else set_status(status, TASC_ECAPACITY);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
        nz += __shfl_xor_sync(0xFFFFFFFFu, nz, o);
    }
    if ((threadIdx.x & 31) == 0 && nz) {
        atomicAdd(&scal[0], (unsigned long long)nz);
        atomicAdd(&scal[2], sq);                   // integer sums: the order of the additions does not matter
    }
    __syncthreads();
    for (int i = threadIdx.x; i < CC_LOW; i += STATS_THREADS)
        if (low[i]) atomicAdd(&bins[i], low[i]);
}

struct CountSummary {
    unsigned long long n_total;      // sum of the counts
    unsigned long long n_distinct;
    unsigned long long sum_sq;
    unsigned long long n_for_cdf;    // smallest number of the largest counts that reach cdf_num / cdf_den of n_total
    double sum_c_log2_c;             // sum over all keys of c log2 c
};
struct BinSum { unsigned long long mass, keys; double lg; };

// A thread's BIN_PER bins of chunk `chunk` (chunk 0 has the largest count values, thread 0 the largest of a chunk).
__device__ __forceinline__ uint32_t bin_top(int chunk) { return CC_BINS - 1u - (uint32_t)chunk * BIN_CHUNK - (uint32_t)threadIdx.x * BIN_PER; }
// Sum of the block's values in thread 0, added in a fixed order.
__device__ __forceinline__ BinSum bin_reduce(BinSum v, BinSum* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.mass += __shfl_down_sync(0xFFFFFFFFu, v.mass, o);
        v.keys += __shfl_down_sync(0xFFFFFFFFu, v.keys, o);
        v.lg += __shfl_down_sync(0xFFFFFFFFu, v.lg, o);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int i = 1; i < STATS_THREADS / 32; ++i) { v.mass += red[i].mass; v.keys += red[i].keys; v.lg += red[i].lg; }
    return v;
}
// grid (BIN_CHUNKS, 2): the sums of a chunk of bins of the bigrams (y = 0) and the tokens (y = 1).  (One block that walked all
// bins of one histogram: 0.75 ms.)
__global__ void __launch_bounds__(STATS_THREADS) bin_sums_kernel(const uint32_t* __restrict__ bins, BinSum* __restrict__ sums) {
    __shared__ BinSum red[STATS_THREADS / 32];
    const uint32_t* b = bins + (size_t)blockIdx.y * CC_BINS;
    const uint32_t top = bin_top(blockIdx.x);
    uint32_t m[BIN_PER];
#pragma unroll
    for (int i = 0; i < BIN_PER; ++i) m[i] = b[top - i];
    BinSum v = {0ull, 0ull, 0.0};
#pragma unroll
    for (int i = 0; i < BIN_PER; ++i) {
        const uint32_t c = top - i;
        if (c && m[i]) { v.mass += (unsigned long long)m[i] * c; v.keys += m[i]; v.lg += (double)m[i] * ((double)c * log2((double)c)); }
    }
    v = bin_reduce(v, red);
    if (threadIdx.x == 0) sums[blockIdx.y * BIN_CHUNKS + blockIdx.x] = v;
}
// One block per histogram: adds up the overflow list and the chunks, and finds where the counts, from the largest down,
// reach the coverage target: in the list, or in one chunk, where the thread whose bins hold the crossing finishes the count.
__global__ void __launch_bounds__(STATS_THREADS)
count_summary_kernel(const uint32_t* __restrict__ bins, const BinSum* __restrict__ sums, const uint32_t* __restrict__ overflow_,
                     const unsigned long long* __restrict__ scal_, unsigned long long cdf_num_, unsigned long long cdf_den_, CountSummary* out_) {
    __shared__ BinSum s_sum[BIN_CHUNKS];
    __shared__ unsigned long long s_mass[STATS_THREADS], s_keys[STATS_THREADS];
    __shared__ uint32_t s_over[CC_OVERFLOW];
    __shared__ unsigned long long s_need, s_above, s_k;
    __shared__ int s_chunk;
    const int set = blockIdx.x, t = threadIdx.x;
    const uint32_t *b = bins + (size_t)set * CC_BINS, *overflow = overflow_ + (size_t)set * CC_OVERFLOW;
    const unsigned long long* scal = scal_ + 4 * set;
    const unsigned long long cdf_num = set ? 1ull : cdf_num_, cdf_den = set ? 1ull : cdf_den_;
    CountSummary* out = out_ + set;
    const int n_over = (int)min(scal[1], (unsigned long long)CC_OVERFLOW);
    // the overflow list, largest first: rank by counting (a few thousand entries at most)
    for (int i = t; i < n_over; i += STATS_THREADS) {
        const uint32_t c = overflow[i];
        int rank = 0;
        for (int j = 0; j < n_over; ++j) {
            const uint32_t o = overflow[j];
            rank += (o > c || (o == c && j < i)) ? 1 : 0;
        }
        s_over[rank] = c;
    }
    for (int i = t; i < BIN_CHUNKS; i += STATS_THREADS) s_sum[i] = sums[set * BIN_CHUNKS + i];
    __syncthreads();
    if (t == 0) {
        unsigned long long m = 0, k = (unsigned long long)n_over;
        double l = 0.0;
        for (int i = 0; i < n_over; ++i) { m += s_over[i]; l += (double)s_over[i] * log2((double)s_over[i]); }
        for (int i = 0; i < BIN_CHUNKS; ++i) { m += s_sum[i].mass; k += s_sum[i].keys; l += s_sum[i].lg; }
        out->n_total = m; out->n_distinct = k; out->sum_sq = scal[2]; out->sum_c_log2_c = l;
        out->n_for_cdf = 0;
        s_chunk = -1;
        // target: smallest run with run * den >= num * total.  128-bit products are not needed: total < 2^40, num, den <= 2^16.
        const unsigned long long need = (cdf_num * m + cdf_den - 1) / cdf_den;
        unsigned long long run = 0;
        k = 0;
        bool found = m == 0;
        for (int i = 0; i < n_over && !found; ++i) {
            run += s_over[i];
            ++k;
            if (run >= need) { out->n_for_cdf = k; found = true; }
        }
        for (int i = 0; i < BIN_CHUNKS && !found; ++i) {
            if (run + s_sum[i].mass >= need) { s_chunk = i; s_need = need; s_above = run; s_k = k; found = true; }
            run += s_sum[i].mass;
            k += s_sum[i].keys;
        }
    }
    __syncthreads();
    if (s_chunk < 0) return;
    const uint32_t top = bin_top(s_chunk);
    unsigned long long mass = 0, keys = 0;
    for (int i = 0; i < BIN_PER; ++i) {
        const uint32_t c = top - i, m = c ? b[c] : 0u;
        mass += (unsigned long long)m * c;
        keys += m;
    }
    s_mass[t] = mass; s_keys[t] = keys;
    __syncthreads();
    unsigned long long run = s_above, k = s_k;
    for (int i = 0; i < t; ++i) { run += s_mass[i]; k += s_keys[i]; }
    if (run >= s_need || run + mass < s_need) return;
    for (int i = 0; i < BIN_PER; ++i) {
        const uint32_t c = top - i, m = c ? b[c] : 0u;
        if (!m) continue;
        if (run + (unsigned long long)m * c >= s_need) { out->n_for_cdf = k + (s_need - run + c - 1) / c; return; }
        run += (unsigned long long)m * c;
        k += m;
    }
}

// ------------------------------------------------------------------------------------------- draft
// Bound: k times a chain of look-ups (slots and their values in one trip, then the successors), about 0.4 us a trip; what
// happens between the trips is kept short.  The suffix is matched against the context once per draft, every thread keeping the
// lengths of its positions; the few tokens that follow the longest matches are a list that is compared with directly.  Only
// lists beyond LIST_MAX are counted in the hash table, whose clearing and reading cost more than everything else (k = 6 behind
// 1,530 tokens: 33 us with it, 23 without; k = 8 behind 640: 33, 25; k = 5 behind 380: 18, 15.5; k = 4 behind 64: 9.6, 8.7).
constexpr int DRAFT_THREADS = 256;
constexpr int LIST_MAX = 64;
constexpr int POS_PER = 8;                       // positions whose match lengths a thread keeps; those of longer contexts are worked out again

struct Best { unsigned long long score; uint32_t id; };
__device__ __forceinline__ bool better(unsigned long long s, uint32_t id, const Best& b) {
    return s > b.score || (s == b.score && id < b.id);
}
__device__ __forceinline__ Best block_best(Best v, Best* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long s = __shfl_xor_sync(0xFFFFFFFFu, v.score, o);
        const uint32_t id = __shfl_xor_sync(0xFFFFFFFFu, v.id, o);
        if (better(s, id, v)) { v.score = s; v.id = id; }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    Best r = red[0];
    for (int i = 1; i < DRAFT_THREADS / 32; ++i)
        if (better(red[i].score, red[i].id, r)) r = red[i];
    return r;                                    // (the caller's next barrier comes before red is written again)
}

// Warp-cooperative lookup of a packed context: each round the 32 lanes test 32 consecutive slots.
__device__ __forceinline__ bool warp_lookup(const OrderTable& t, Key key, CtxVal& out) {
    if (!t.keys) return false;
    const int lane = threadIdx.x & 31;
    const uint64_t h = key_hash(key);
    for (uint64_t round = 0; round * 32 <= t.mask; ++round) {
        const uint64_t slot = (h + round * 32 + lane) & t.mask;
        const ulonglong2 kv = *reinterpret_cast<const ulonglong2*>(t.keys + 2 * slot);
        const uint4 v = *reinterpret_cast<const uint4*>(t.vals + slot);      // (the value of the slot that will match is among them)
        const uint32_t hit = __ballot_sync(0xFFFFFFFFu, kv.x == key.lo && kv.y == key.hi);
        const uint32_t hole = __ballot_sync(0xFFFFFFFFu, kv.x == 0 && kv.y == 0);
        if (hit) {
            const int src = __ffs(hit) - 1;
            out.offset = (unsigned long long)__shfl_sync(0xFFFFFFFFu, v.x, src) | ((unsigned long long)__shfl_sync(0xFFFFFFFFu, v.y, src) << 32);
            out.n_succ = __shfl_sync(0xFFFFFFFFu, v.z, src);
            out.total = __shfl_sync(0xFFFFFFFFu, v.w, src);
            // a hole before the hit cannot exist: insertion stops at the first free slot
            return true;
        }
        if (hole) return false;
    }
    return false;
}

__global__ void __launch_bounds__(DRAFT_THREADS)
draft_kernel(const DeviceTables dt, const int32_t* tokens, int64_t stride, const int32_t* len,
             int k, uint32_t lam_num, uint32_t lam_den, int32_t* __restrict__ drafts, int hs_mask) {
    extern __shared__ int32_t dsm[];
    int32_t* h_tok = dsm;                                          // [hs] token or -1
    uint32_t* h_cnt = reinterpret_cast<uint32_t*>(dsm + hs_mask + 1);   // [hs] count, bit 31 = seen in the corpus list
    int32_t* s_seq = dsm + 2 * (hs_mask + 1);                      // [L] the committed tokens
    __shared__ Best red[DRAFT_THREADS / 32];
    __shared__ int s_suffix[TASC_MAX_ORDER];     // last n_max tokens of the query, newest last
    __shared__ int s_best[DRAFT_THREADS / 32], s_tprompt;
    __shared__ int s_hit[TASC_MAX_ORDER];        // order n = index + 1 has a surviving context for the current suffix
    __shared__ CtxVal s_vals[TASC_MAX_ORDER];
    __shared__ int s_list[LIST_MAX], s_seen[LIST_MAX];

    const int b = blockIdx.x;
    const int tid = threadIdx.x, warp = tid >> 5;
    griddep_wait();
    griddep_launch_dependents();
    int L = len[b];
    L = L < 0 ? 0 : (L > stride ? (int)stride : L);
    const int n_max = dt.n_max;
    const bool use_corp = lam_num > 0, use_prompt = lam_num < lam_den;

    for (int i = tid; i < L; i += DRAFT_THREADS) s_seq[i] = tokens[(int64_t)b * stride + i];
    __syncthreads();
    const int32_t* seq = s_seq;
    if (tid < TASC_MAX_ORDER) {
        const int p = L - n_max + tid;             // suffix slot tid <-> position p (only the last n_max slots are used)
        s_suffix[tid] = (tid < n_max && p >= 0) ? seq[p] : -1;
    }
    if (tid == 0) s_tprompt = 0;
    __syncthreads();

    for (int j = 0; j < k; ++j) {
        const int Lq = L + j;                      // query length so far
        const int n_avail = Lq < n_max ? Lq : n_max;
        // ---------------------------------------------------------------- p_corp: all orders are probed at once, one warp
        // per order (warp w looks up the last w + 1 tokens); the longest order that matched wins the back-off
        if (warp < TASC_MAX_ORDER) {
            const int n = warp + 1;
            bool hit = false;
            CtxVal val = {0ull, 0u, 0u};
            if (use_corp && n <= n_avail) {
                Key key = key_make(n);
                for (int i = 0; i < n; ++i) key_put(key, i, (uint32_t)s_suffix[n_max - n + i]);
                hit = warp_lookup(dt.t[n], key, val);
            }
            if ((tid & 31) == 0) { s_hit[warp] = hit ? 1 : 0; s_vals[warp] = val; }
        }
        // ---------------------------------------------------------------- p_prompt: longest suffix match in the committed tokens
        int t_prompt_ = 0;
        bool listed = true;                        // the successors' list holds them all
        if (use_prompt) {
            auto match_len = [&](int p) {          // tokens before successor position p that agree with the query suffix
                int m = 0;
                const int lim = p < n_avail ? p : n_avail;
                while (m < lim && seq[p - 1 - m] == s_suffix[n_max - 1 - m]) ++m;
                return m;
            };
            int best = 0;
            uint32_t kept = 0u;                    // 4 bits per position: lengths are at most TASC_MAX_ORDER
            int i = 0;
            for (int p = 1 + tid; p < L; p += DRAFT_THREADS, ++i) {
                const int m = match_len(p);
                best = max(best, m);
                if (i < POS_PER) kept |= (uint32_t)m << (4 * i);
            }
            best = __reduce_max_sync(0xFFFFFFFFu, best);
            if ((tid & 31) == 0) s_best[warp] = best;
            __syncthreads();
            int nstar = 0;
#pragma unroll
            for (int w = 0; w < DRAFT_THREADS / 32; ++w) nstar = max(nstar, s_best[w]);
            auto matches = [&](int at, int p) { return (at < POS_PER ? (int)((kept >> (4 * at)) & 15u) : match_len(p)) == nstar; };
            if (nstar > 0) {
                i = 0;
                for (int p = 1 + tid; p < L; p += DRAFT_THREADS, ++i) {
                    if (!matches(i, p)) continue;
                    const int at = atomicAdd(&s_tprompt, 1);
                    if (at < LIST_MAX) { s_list[at] = seq[p]; s_seen[at] = 0; }
                }
            }
            __syncthreads();
            t_prompt_ = s_tprompt;
            listed = t_prompt_ <= LIST_MAX;
            if (!listed) {
                for (int q = tid; q <= hs_mask; q += DRAFT_THREADS) { h_tok[q] = -1; h_cnt[q] = 0u; }
                __syncthreads();
                i = 0;
                for (int p = 1 + tid; p < L; p += DRAFT_THREADS, ++i) {
                    if (!matches(i, p)) continue;
                    const int x = seq[p];
                    uint32_t slot = ((uint32_t)x * 2654435761u) & hs_mask;
                    for (int probe = 0; probe <= hs_mask; ++probe) {
                        const int old = atomicCAS(&h_tok[slot], -1, x);
                        if (old == -1 || old == x) { atomicAdd(&h_cnt[slot], 1u); break; }
                        slot = (slot + 1) & hs_mask;
                    }
                }
                __syncthreads();
            }
        } else {
            __syncthreads();
        }
        int found_n = 0;
        for (int n = n_max; n >= 1 && !found_n; --n)
            if (s_hit[n - 1]) found_n = n;
        const CtxVal cv = s_vals[found_n > 0 ? found_n - 1 : 0];
        const unsigned long long t_corp = cv.total;
        const unsigned long long t_prompt = (unsigned long long)t_prompt_;
        const bool has_corp = found_n > 0, has_prompt = t_prompt > 0;
        // ---------------------------------------------------------------- mixture argmax
        Best mine = {0ull, 0xFFFFFFFFu};
        bool any = false;
        auto offer = [&](unsigned long long score, uint32_t id) {
            if (!any || better(score, id, mine)) { mine.score = score; mine.id = id; any = true; }
        };
        if (has_corp) {
            const Succ* sl = dt.t[found_n].succ + cv.offset;
            const unsigned long long w_c = has_prompt ? (unsigned long long)lam_num * t_prompt : 1ull;
            const unsigned long long w_p = (unsigned long long)(lam_den - lam_num) * t_corp;
            for (uint32_t i = tid; i < cv.n_succ; i += DRAFT_THREADS) {
                const Succ s = sl[i];
                unsigned long long score = w_c * s.count;
                if (has_prompt && listed) {
                    uint32_t c = 0;
                    for (int e = 0; e < t_prompt_; ++e)
                        if (s_list[e] == s.next) { ++c; s_seen[e] = 1; }
                    score += w_p * c;
                } else if (has_prompt) {
                    uint32_t slot = ((uint32_t)s.next * 2654435761u) & hs_mask;
                    for (int probe = 0; probe <= hs_mask; ++probe) {
                        const int tk = h_tok[slot];
                        if (tk == -1) break;
                        if (tk == s.next) {
                            const uint32_t c = atomicOr(&h_cnt[slot], 0x80000000u) & 0x7FFFFFFFu;
                            score += w_p * c;
                            break;
                        }
                        slot = (slot + 1) & hs_mask;
                    }
                }
                offer(score, (uint32_t)s.next);
            }
            __syncthreads();     // the corpus pass has marked the shared successors
        }
        if (has_prompt) {
            const unsigned long long w_p = has_corp ? (unsigned long long)(lam_den - lam_num) * t_corp : 1ull;
            if (listed) {
                if (tid < t_prompt_ && !s_seen[tid]) {
                    const int tk = s_list[tid];
                    uint32_t c = 0;
                    for (int e = 0; e < t_prompt_; ++e) c += s_list[e] == tk;
                    offer(w_p * c, (uint32_t)tk);
                }
            } else {
                for (int i = tid; i <= hs_mask; i += DRAFT_THREADS) {
                    const int tk = h_tok[i];
                    const uint32_t c = h_cnt[i];
                    if (tk < 0 || (c & 0x80000000u)) continue;      // empty, or already scored with its corpus count
                    offer(w_p * c, (uint32_t)tk);
                }
            }
        }
        if (!any) { mine.score = 0ull; mine.id = 0xFFFFFFFFu; }
        const Best win = block_best(mine, red);
        const int draft = (has_corp || has_prompt) ? (int)win.id : dt.fallback;
        if (tid == 0) {
            drafts[(int64_t)b * k + j] = draft;
            for (int i = 0; i + 1 < n_max; ++i) s_suffix[i] = s_suffix[i + 1];
            s_suffix[n_max - 1] = draft;
            s_tprompt = 0;
        }
        __syncthreads();
    }
}

tasc_drafter* new_drafter(int n_max, int fallback, int p_min, int vocab) {
    tasc_drafter* d = new (std::nothrow) tasc_drafter();
    if (!d) return nullptr;
    for (int n = 0; n <= TASC_MAX_ORDER; ++n) d->dt.t[n] = OrderTable{nullptr, nullptr, nullptr, 0, 0};
    d->dt.n_max = n_max; d->dt.fallback = fallback; d->p_min = p_min; d->vocab = vocab;
    if (cudaGetDevice(&d->device) != cudaSuccess) (void)cudaGetLastError();
    return d;
}
// Frees the handle when nothing on its device reads the tables any more.
void free_drafter(tasc_drafter* d) {
    int dev = d->device;
    if (cudaGetDevice(&dev) != cudaSuccess) (void)cudaGetLastError();
    if (dev != d->device) cudaSetDevice(d->device);
    if (cudaDeviceSynchronize() != cudaSuccess) (void)cudaGetLastError();
    for (DeviceSlab& s : d->slab) s.release(nullptr);
    if (dev != d->device) cudaSetDevice(dev);
    delete d;
}

// Everything of tasc_drafter_build that can fail once the handle exists.
tasc_status build_from_corpus(tasc_drafter* d, const int32_t* tokens, const int64_t* offsets, int64_t n_docs, const CorpusCheck& c, cudaStream_t stream) {
    const int64_t T = c.tokens;
    if (T == 0) return TASC_OK;                  // (the fallback stays 0)
    if (T >= (1ll << 32) - 1 || count_pairs(c.pairs) >= (1ull << 31)) return TASC_ENOMEM;
    const int n_max = d->dt.n_max, p_min = d->p_min, vocab = d->vocab;
    // scalars: [0] histogram argmax, [1] n-grams listed, [2] positions left for the next order, [3] cursor, [4] status
    DeviceSlab slab;
    const uint64_t pairs1 = count_pairs(c.pairs), list_max = c.pairs / (uint64_t)p_min + 1;
    const size_t o_scal = slab.add(64), o_hist = slab.add((size_t)vocab * 4), o_slots = slab.add(pairs1 * 2 * sizeof(CountSlot)),
                 o_id0 = slab.add((size_t)T * 4), o_id1 = slab.add((size_t)T * 4), o_rem = slab.add((size_t)T),
                 o_bits = slab.add((2 * pairs1 + 31) / 32 * 4), o_list = slab.add(list_max * sizeof(Survivor)), o_place = slab.add(list_max * sizeof(uint2));
    if (!slab.allocate(stream)) return TASC_ENOMEM;
    unsigned long long* scal = slab.at<unsigned long long>(o_scal);
    int* status = reinterpret_cast<int*>(scal + 4);
    uint32_t *hist = slab.at<uint32_t>(o_hist), *id = slab.at<uint32_t>(o_id0), *prev = slab.at<uint32_t>(o_id1);
    uint8_t* remaining = slab.at<uint8_t>(o_rem);
    Survivor* list = slab.at<Survivor>(o_list);
    TASC_CUDA_TRY(cudaMemsetAsync(scal, 0, o_hist + (size_t)vocab * 4, stream));
    corpus_scan_kernel<<<scan_blocks(T), SCAN_THREADS, 0, stream>>>(tokens, offsets, n_docs, T, vocab, remaining, hist, status);
    hist_argmax_kernel<<<blocks_for(vocab, 256), 256, 0, stream>>>(hist, vocab, scal);
    unsigned long long h[5];
    uint64_t windows = c.pairs, contexts = (uint64_t)vocab;
    for (int n = 1; n <= n_max && windows; ++n) {
        const CountTable t = {slab.at<CountSlot>(o_slots), (uint32_t)count_pairs(windows)};
        TASC_CUDA_TRY(cudaMemsetAsync(t.slots, 0, (size_t)t.pairs * 2 * sizeof(CountSlot), stream));
        TASC_CUDA_TRY(cudaMemsetAsync(scal + 1, 0, 2 * sizeof(*scal), stream));
        const tasc_status cs = n == 1 ? launch_count<true>(tokens, remaining, T, n, nullptr, t, id, status, stream)
                                      : launch_count<false>(tokens, remaining, T, n, prev, t, id, status, stream);
        if (cs != TASC_OK) return cs;
        list_kernel<<<blocks_for(2 * (uint64_t)t.pairs, LIST_SLOTS), 256, 0, stream>>>(t, (uint32_t)p_min, list, scal + 1,
                                                                                                  n < n_max ? slab.at<uint32_t>(o_bits) : nullptr);
        if (n < n_max) prune_kernel<<<blocks_for((uint64_t)T, 256 * PRUNE_PER), 256, 0, stream>>>(id, remaining, T, n, slab.at<uint32_t>(o_bits), scal + 2);
        TASC_CUDA_TRY(cudaGetLastError());
        TASC_CUDA_TRY(cudaMemcpyAsync(h, scal, sizeof(h), cudaMemcpyDeviceToHost, stream));
        TASC_CUDA_TRY(cudaStreamSynchronize(stream));
        if ((int)h[4] != 0) return (int)h[4];                    // a token id outside [0, vocab)
        if (n == 1) d->dt.fallback = (int)(0xFFFFFFFFu - (uint32_t)(h[0] & 0xFFFFFFFFull));
        if (h[1] == 0) break;                                    // nor can anything longer be frequent
        const tasc_status rc = build_order(d, n, CorpusElements{tokens, list}, h[1], contexts, slab.at<uint2>(o_place), scal + 3, status, stream);
        if (rc != TASC_OK) return rc;
        windows = h[2];
        contexts = h[1];                                         // every context of the next order is one of these
        std::swap(id, prev);
    }
    if (c.pairs == 0) {
        TASC_CUDA_TRY(cudaMemcpyAsync(h, scal, sizeof(h), cudaMemcpyDeviceToHost, stream));
        TASC_CUDA_TRY(cudaStreamSynchronize(stream));
        if ((int)h[4] != 0) return (int)h[4];
        d->dt.fallback = (int)(0xFFFFFFFFu - (uint32_t)(h[0] & 0xFFFFFFFFull));
        return TASC_OK;
    }
    int st = 0;
    TASC_CUDA_TRY(cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, stream));
    TASC_CUDA_TRY(cudaStreamSynchronize(stream));
    return st;
}

}  // namespace
}  // namespace tasc

using namespace tasc;

extern "C" tasc_status tasc_drafter_build(const int32_t* corpus_tokens, const int64_t* doc_offsets, int64_t n_docs,
                                          int32_t n_max, int32_t p_min, int32_t vocab, tasc_stream stream_,
                                          tasc_drafter** out) {
    if (!out) return TASC_EINVAL;
    *out = nullptr;
    if (!doc_offsets || n_docs < 0 || n_max < 1 || n_max > TASC_MAX_ORDER || p_min < 1 || vocab < 1 ||
        vocab > (1 << TASC_VOCAB_BITS))
        return TASC_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    CorpusCheck c;
    tasc_status rc = check_corpus(doc_offsets, n_docs, c, stream);
    if (rc != TASC_OK) return rc;
    if (c.tokens > 0 && !corpus_tokens) return TASC_EINVAL;
    tasc_drafter* d = new_drafter(n_max, 0, p_min, vocab);
    if (!d) return TASC_ENOMEM;
    rc = build_from_corpus(d, corpus_tokens, doc_offsets, n_docs, c, stream);
    if (rc != TASC_OK) { free_drafter(d); return rc; }
    *out = d;
    return TASC_OK;
}

extern "C" tasc_status tasc_drafter_from_bigram(const int32_t* table, int32_t vocab, tasc_stream stream_, tasc_drafter** out) {
    if (!out) return TASC_EINVAL;
    *out = nullptr;
    if (!table || vocab < 1 || vocab > (1 << TASC_VOCAB_BITS)) return TASC_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    tasc_drafter* d = new_drafter(1, 0, 1, vocab);
    if (!d) return TASC_ENOMEM;
    OrderTable& t = d->dt.t[1];
    DeviceSlab& slab = d->slab[1];
    const uint64_t cap = pow2_at_least(2 * (uint64_t)vocab);
    const size_t o_status = slab.add(sizeof(int)), o_keys = slab.add(cap * 16), o_vals = slab.add(cap * sizeof(CtxVal)), o_succ = slab.add((size_t)vocab * sizeof(Succ));
    tasc_status rc = TASC_OK;
    if (!slab.allocate(stream)) rc = TASC_ENOMEM;
    if (rc == TASC_OK) {
        int* status = slab.at<int>(o_status);
        t = OrderTable{slab.at<uint64_t>(o_keys), slab.at<CtxVal>(o_vals), slab.at<Succ>(o_succ), cap - 1, vocab};
        cudaMemsetAsync(status, 0, o_succ, stream);                    // status, keys and values
        bigram_insert_kernel<<<blocks_for((uint64_t)vocab, 256), 256, 0, stream>>>(table, vocab, t, status);
        int st = 0;
        if (cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
            cudaStreamSynchronize(stream) != cudaSuccess) { (void)cudaGetLastError(); rc = TASC_ECUDA; }
        else if (st != 0) rc = st;
    }
    if (rc != TASC_OK) { free_drafter(d); return rc; }
    *out = d;
    return TASC_OK;
}

extern "C" tasc_status tasc_corpus_stats(const int32_t* corpus_tokens, const int64_t* doc_offsets, int64_t n_docs, int32_t vocab,
                                         int32_t cdf_num, int32_t cdf_den, tasc_stream stream_, tasc_corpus_statistics* out) {
    if (!out || !doc_offsets || n_docs < 0 || vocab < 1 || vocab > (1 << TASC_VOCAB_BITS) || cdf_den < 1 || cdf_den > 65536 ||
        cdf_num < 1 || cdf_num > cdf_den)
        return TASC_EINVAL;
    *out = tasc_corpus_statistics{};
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    CorpusCheck c;
    const tasc_status rc = check_corpus(doc_offsets, n_docs, c, stream);
    if (rc != TASC_OK) return rc;
    const int64_t T = c.tokens;
    if (T > 0 && !corpus_tokens) return TASC_EINVAL;
    if ((uint64_t)T >= (1ull << 40)) return TASC_EINVAL;
    if (T >= (1ll << 32) - 1 || count_pairs(c.pairs) >= (1ull << 31)) return TASC_ENOMEM;

    // scal: [0..2] bigram scalars, [4..6] token scalars, [8] status; behind it everything that starts as zero
    DeviceSlab slab;
    const CountTable empty = {nullptr, (uint32_t)count_pairs(c.pairs)};
    const size_t table_bytes = (size_t)empty.pairs * 2 * sizeof(CountSlot);
    const size_t o_scal = slab.add(9 * sizeof(unsigned long long)), o_hist = slab.add((size_t)vocab * 4), o_bins = slab.add(2 * (size_t)CC_BINS * 4),
                 o_slots = slab.add(table_bytes), o_over = slab.add(2 * (size_t)CC_OVERFLOW * 4), o_sums = slab.add(2 * BIN_CHUNKS * sizeof(BinSum)),
                 o_summ = slab.add(2 * sizeof(CountSummary)), o_rem = slab.add((size_t)T);
    if (!slab.allocate(stream)) return TASC_ENOMEM;
    unsigned long long* scal = slab.at<unsigned long long>(o_scal);
    int* status = reinterpret_cast<int*>(scal + 8);
    uint32_t *hist = slab.at<uint32_t>(o_hist), *bins = slab.at<uint32_t>(o_bins), *overflow = slab.at<uint32_t>(o_over);
    uint8_t* remaining = slab.at<uint8_t>(o_rem);
    const CountTable table = {slab.at<CountSlot>(o_slots), empty.pairs};
    const uint64_t n_slots = 2 * (uint64_t)table.pairs;
    TASC_CUDA_TRY(cudaMemsetAsync(scal, 0, o_slots + table_bytes, stream));
    if (T > 0) {
        corpus_scan_kernel<<<scan_blocks(T), SCAN_THREADS, 0, stream>>>(corpus_tokens, doc_offsets, n_docs, T, vocab, remaining, hist, status);
        // bigrams = the windows of the order-1 model before pruning: (token, next) inside one document
        const tasc_status cs = launch_count<true>(corpus_tokens, remaining, T, 1, nullptr, table, nullptr, status, stream);
        if (cs != TASC_OK) return cs;
    }
    constexpr unsigned VALUE_BLOCKS = 148 * 8;           // all resident
    count_values_kernel<<<std::min(blocks_for(n_slots, STATS_THREADS), VALUE_BLOCKS), STATS_THREADS, 0, stream>>>(
        &table.slots->count, (int)(sizeof(CountSlot) / 4), n_slots, bins, overflow, scal, status);
    count_values_kernel<<<std::min(blocks_for(vocab, STATS_THREADS), VALUE_BLOCKS), STATS_THREADS, 0, stream>>>(
        hist, 1, (uint64_t)vocab, bins + CC_BINS, overflow + CC_OVERFLOW, scal + 4, status);
    bin_sums_kernel<<<dim3(BIN_CHUNKS, 2), STATS_THREADS, 0, stream>>>(bins, slab.at<BinSum>(o_sums));
    count_summary_kernel<<<2, STATS_THREADS, 0, stream>>>(bins, slab.at<BinSum>(o_sums), overflow, scal, (unsigned long long)cdf_num,
                                                          (unsigned long long)cdf_den, slab.at<CountSummary>(o_summ));
    TASC_CUDA_TRY(cudaGetLastError());
    CountSummary h[2] = {};
    int st = 0;
    TASC_CUDA_TRY(cudaMemcpyAsync(h, slab.at<CountSummary>(o_summ), sizeof(h), cudaMemcpyDeviceToHost, stream));
    TASC_CUDA_TRY(cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, stream));
    TASC_CUDA_TRY(cudaStreamSynchronize(stream));
    if (st != 0) return st;
    // the closing arithmetic on a handful of scalars: H = log2 N - (sum c log2 c) / N;  H_2 = 2 log2 N - log2 sum c^2
    auto entropy = [](const CountSummary& c) { return c.n_total ? log2((double)c.n_total) - c.sum_c_log2_c / (double)c.n_total : 0.0; };
    out->n_tokens = T;
    out->n_bigrams = (int64_t)h[0].n_total;
    out->n_unique_tokens = (int64_t)h[1].n_distinct;
    out->n_unique_bigrams = (int64_t)h[0].n_distinct;
    out->bigrams_for_cdf = (int64_t)h[0].n_for_cdf;
    out->bigram_entropy_bits = entropy(h[0]);
    out->typical_set_size = exp2(out->bigram_entropy_bits);
    out->token_entropy_bits = entropy(h[1]);
    out->token_entropy_normalised = vocab > 1 ? out->token_entropy_bits / log2((double)vocab) : 0.0;
    out->token_renyi2_bits = h[1].n_total ? 2.0 * log2((double)h[1].n_total) - log2((double)h[1].sum_sq) : 0.0;
    return TASC_OK;
}

extern "C" tasc_status tasc_drafter_export(const tasc_drafter* d, tasc_ngram_entry* out, int64_t cap, int64_t* n_entries,
                                           int32_t* fallback_token) {
    if (!d || !n_entries || cap < 0 || (cap > 0 && !out)) return TASC_EINVAL;
    int64_t total = 0;
    for (int n = 1; n <= d->dt.n_max; ++n) total += d->dt.t[n].n_succ;
    *n_entries = total;
    if (fallback_token) *fallback_token = d->dt.fallback;
    if (cap < total) return cap == 0 ? TASC_OK : TASC_ECAPACITY;
    int64_t w = 0;
    for (int n = 1; n <= d->dt.n_max; ++n) {
        const OrderTable& t = d->dt.t[n];
        if (!t.keys) continue;
        const uint64_t ccap = t.mask + 1;
        std::vector<uint64_t> keys(ccap * 2);
        std::vector<CtxVal> vals(ccap);
        std::vector<Succ> succ((size_t)t.n_succ);
        TASC_CUDA_TRY(cudaMemcpy(keys.data(), t.keys, ccap * 16, cudaMemcpyDeviceToHost));
        TASC_CUDA_TRY(cudaMemcpy(vals.data(), t.vals, ccap * sizeof(CtxVal), cudaMemcpyDeviceToHost));
        TASC_CUDA_TRY(cudaMemcpy(succ.data(), t.succ, succ.size() * sizeof(Succ), cudaMemcpyDeviceToHost));
        for (uint64_t s = 0; s < ccap; ++s) {
            if (!(keys[2 * s + 1] & VALID_BIT)) continue;
            const Key k = {keys[2 * s], keys[2 * s + 1]};
            for (uint32_t i = 0; i < vals[s].n_succ; ++i) {
                const uint64_t pos = vals[s].offset + i;
                if (pos >= succ.size() || w >= total) return TASC_ECAPACITY;
                tasc_ngram_entry& e = out[w++];
                e.n = n;
                for (int j = 0; j < TASC_MAX_ORDER; ++j) e.ctx[j] = j < n ? (int32_t)key_get(k, j) : -1;
                e.next = succ[pos].next;
                e.count = succ[pos].count;
            }
        }
    }
    std::sort(out, out + w, [](const tasc_ngram_entry& a, const tasc_ngram_entry& b) {
        if (a.n != b.n) return a.n < b.n;
        for (int j = 0; j < TASC_MAX_ORDER; ++j)
            if (a.ctx[j] != b.ctx[j]) return a.ctx[j] < b.ctx[j];
        return a.next < b.next;
    });
    return w == total ? TASC_OK : TASC_ECAPACITY;
}

extern "C" tasc_status tasc_drafter_import(const tasc_ngram_entry* entries, int64_t n_entries, int32_t n_max, int32_t vocab,
                                           int32_t fallback_token, tasc_stream stream_, tasc_drafter** out) {
    if (!out) return TASC_EINVAL;
    *out = nullptr;
    if (n_entries < 0 || (n_entries > 0 && !entries) || n_max < 1 || n_max > TASC_MAX_ORDER || vocab < 1 ||
        vocab > (1 << TASC_VOCAB_BITS) || fallback_token < 0 || fallback_token >= vocab)
        return TASC_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    // the packed (context, next) keys and counts of every order, in the form the build's compaction kernels read
    std::vector<std::vector<uint64_t>> keys((size_t)n_max + 1);
    std::vector<std::vector<uint32_t>> counts((size_t)n_max + 1);
    for (int64_t i = 0; i < n_entries; ++i) {
        const tasc_ngram_entry& e = entries[i];
        if (e.n < 1 || e.n > n_max || e.next < 0 || e.next >= vocab || e.count < 1) return TASC_EINVAL;
        Key k = key_make(e.n);
        for (int j = 0; j < e.n; ++j) {
            if (e.ctx[j] < 0 || e.ctx[j] >= vocab) return TASC_EINVAL;
            key_put(k, j, (uint32_t)e.ctx[j]);
        }
        key_put(k, e.n, (uint32_t)e.next);
        keys[e.n].push_back(k.lo);
        keys[e.n].push_back(k.hi);
        counts[e.n].push_back(e.count);
    }
    tasc_drafter* d = new_drafter(n_max, fallback_token, 1, vocab);
    if (!d) return TASC_ENOMEM;
    uint64_t most = 0;
    for (const auto& v : counts) most = std::max<uint64_t>(most, v.size());
    DeviceSlab slab;
    const size_t o_scal = slab.add(16), o_keys = slab.add(most * 16), o_counts = slab.add(most * 4), o_place = slab.add(most * sizeof(uint2));
    auto fill = [&]() -> tasc_status {
        if (!slab.allocate(stream)) return TASC_ENOMEM;
        unsigned long long* scal = slab.at<unsigned long long>(o_scal);          // [0] cursor, [1] status
        int* status = reinterpret_cast<int*>(scal + 1);
        TASC_CUDA_TRY(cudaMemsetAsync(scal, 0, 16, stream));
        for (int n = 1; n <= n_max; ++n) {
            const uint64_t cnt = counts[n].size();
            if (cnt == 0) continue;
            const PackedElements el = {slab.at<uint64_t>(o_keys), slab.at<uint32_t>(o_counts)};
            TASC_CUDA_TRY(cudaMemcpyAsync(slab.at<uint64_t>(o_keys), keys[n].data(), cnt * 16, cudaMemcpyHostToDevice, stream));
            TASC_CUDA_TRY(cudaMemcpyAsync(slab.at<uint32_t>(o_counts), counts[n].data(), cnt * 4, cudaMemcpyHostToDevice, stream));
            const tasc_status rc = build_order(d, n, el, cnt, cnt, slab.at<uint2>(o_place), scal, status, stream);
            if (rc != TASC_OK) return rc;
        }
        int st = 0;
        TASC_CUDA_TRY(cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, stream));
        TASC_CUDA_TRY(cudaStreamSynchronize(stream));
        return st;
    };
    const tasc_status rc = fill();
    if (rc != TASC_OK) {
        cudaStreamSynchronize(stream);                               // the host arrays must outlive the copies
        free_drafter(d);
        return rc;
    }
    *out = d;
    return TASC_OK;
}

extern "C" tasc_status tasc_drafter_destroy(tasc_drafter* d) {
    if (!d) return TASC_EINVAL;
    free_drafter(d);
    return TASC_OK;
}

extern "C" tasc_status tasc_draft(const tasc_drafter* d, const int32_t* tokens, int64_t stride, const int32_t* len,
                                  int32_t B, int32_t k, int32_t lambda_num, int32_t lambda_den, int32_t* drafts,
                                  tasc_stream stream) {
    if (!d || !tokens || !len || !drafts || B < 1 || k < 1 || k > TASC_MAX_ROWS - 1 || stride < 1 || stride > 12288 ||
        lambda_den < 1 || lambda_den > 256 || lambda_num < 0 || lambda_num > lambda_den)
        return TASC_EINVAL;
    uint64_t hs = 64;
    while (hs * 3 < (uint64_t)stride * 4) hs <<= 1;      // load factor <= 3/4
    const size_t smem = hs * 8 + (size_t)stride * sizeof(int32_t);      // hash of the context successors + the tokens
    {
        // the attribute belongs to the device: set once per device, under a lock (two threads may make their first call together)
        static std::mutex mu;
        static bool attr_done[64] = {false};
        int dev = 0;
        TASC_CUDA_TRY(cudaGetDevice(&dev));
        if (dev < 0 || dev >= 64) return TASC_EINVAL;
        std::lock_guard<std::mutex> lk(mu);
        if (!attr_done[dev]) {
            TASC_CUDA_TRY(cudaFuncSetAttribute(draft_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 184 * 1024));
            attr_done[dev] = true;
        }
    }
    ProfScope ps(K_DRAFT, static_cast<cudaStream_t>(stream));
    TASC_CUDA_TRY(launch_ahead(draft_kernel, dim3(B), dim3(DRAFT_THREADS), smem, static_cast<cudaStream_t>(stream),
                               d->dt, tokens, stride, len, k, (uint32_t)lambda_num, (uint32_t)lambda_den, drafts, (int)(hs - 1)));
    return TASC_OK;
}
