// Tokenizer enrichment (TASC-tok, Section 4 of the paper) on the device.
//
// tasc_tok_enrich -- Algorithm 1: starting from the base vocabulary, every iteration counts the token n-grams
// (2 <= n <= n_max) of the task corpus as it is tokenised with the current vocabulary, scores each with the merge
// reward f_merge(t^n) = freq(t^n) * (n - 1) (Section 4.1), takes the argmax, adds it as one new token and replaces its
// occurrences (left to right, non-overlapping, inside each document) before the next iteration.  The prefix-collision
// test of the paper needs the tokens' strings; ids have none, so every candidate passes.
//   Counting is the drafter's machinery: one open-addressing table keyed by the full packing of (n, tokens), one
//   128-bit compare-and-swap per new n-gram.  The table is counted in full once and then kept up to date: a merge changes
//   the windows that overlap a replaced occurrence and no others, so only those are taken out and put back.  The argmax
//   is unique: largest reward, then the longer n-gram, then the one that occurs first; first occurrences are looked up
//   only in rounds where the first two tie.  Most rounds take it from a short list of the n-grams within a quarter of
//   the best, which every CTA reads for itself.  The documents stay at their original offsets and only get shorter.
//   All rounds run in one cooperative kernel without a host round trip.
// tasc_tok_init_rows -- Section 4.2: the embedding / LM-head row of an added token is the mean of its constituents'
//   rows (a constituent may itself be an added token): in order, by warps that wait for the rows they need.
// tasc_tok_encode -- Appendix on byte-pair encoding: text is encoded with the added tokens matched first and greedily
//   (the longest added token whose expansion into base tokens matches the upcoming base tokens).  The added tokens'
//   expansions form a trie stored as a hash of (node, token) -> child; a thread per document walks it.
#include "kernels.h"
#include "ngram_table.cuh"

#include <algorithm>
#include <cstring>
#include <vector>

namespace tasc {
namespace {

constexpr int MAX_N = TASC_TOK_MAX_N;            // longest n-gram (the key holds six ids)
constexpr int POS_BITS = 28;                     // window positions are below 2^28
constexpr int LEN_BITS = 3;

// What the merge loop shares across the grid.  Words that a later round uses again exist twice: one CTA prepares the one
// while all others still read the other.
struct TokState {
    unsigned long long used[2];                  // slots claimed
    unsigned long long first[2];                 // first position of the n-grams that tie, and the slot of the one that is there
    unsigned int n_cand[2];                      // entries of the candidates' list
    int rebuild;                                 // the round before which the table has to be counted again (0: the first)
    int n_merges, status;
    unsigned int bar;                            // arrivals at the grid barrier
};
// The best n-gram of a part of the table: its rank (reward and length), one slot that has it, and how many have it.
struct __align__(16) Best { unsigned long long rank; unsigned int slot, ties; };

// A slot's word: n-gram length (3 bits) and count (29 bits; positions are below 2^28).
constexpr uint32_t CNT_BITS = 29, CNT_MASK = (1u << CNT_BITS) - 1u;
// (reward, length) of a word, 0 for a count of zero: reward = count * (length - 1)
__device__ __forceinline__ unsigned long long tok_rank(uint32_t w) {
    const uint32_t c = w & CNT_MASK, n = w >> CNT_BITS;
    return c ? (((unsigned long long)c * (n - 1u)) << LEN_BITS) | n : 0ull;
}

constexpr int TOK_THREADS = 1024, TOK_WARPS = TOK_THREADS / 32;
constexpr int CHUNK_BITS = 7;                    // slots whose best n-gram is kept: 512 bytes of words, one load of a warp
constexpr unsigned int CAND_MAX = TOK_THREADS;   // candidates: one per thread
constexpr int TIED_MAX = 8;                      // n-grams that tie and are looked for by their tokens
constexpr long long TOK_BARRIER_CYCLES = 20000000000ll;           // (a document of millions of tokens is one warp's work)

struct TokArgs {
    int32_t* cur;                                // tokens at the documents' original offsets; -1 behind a document's end
    uint8_t* rem;                                // tokens that follow in the document (255 = more)
    uint8_t* mark;
    const int32_t* doc_of;
    const int64_t* offsets;
    int32_t *doc_len, *doc_round;                // length now; last round + 1 in which the n-gram was found
    int64_t n_docs, T;
    uint64_t* keys;
    uint32_t* words;
    uint8_t* dirty;                              // per chunk of slots: its best has to be looked up again
    Best *chunk_best, *cta_best;
    uint32_t* cand;                              // two lists of CAND_MAX slots
    uint64_t cap;
    TokState* st;
    int32_t* merges;
    int base_vocab, budget, n_max;
};

// The table's slots come in pairs of one 32-byte sector; a key is in the first pair of its own sequence that had room.  (With
// single slots one behind the other, the longest of the tens of thousands of look-ups of a round took over 30 trips to
// L2, 18 us; now about four.)
struct Probe {
    uint64_t pair, step, mask;
    __device__ __forceinline__ Probe(const TokArgs& a, const Key& key) {
        const uint64_t h = key_hash(key);
        mask = a.cap / 2 - 1;
        pair = h & mask;
        step = (h >> 36) | 1ull;
    }
    __device__ __forceinline__ void next() { pair = (pair + step) & mask; }
};
struct KeyPair { ulonglong2 k[2]; };
__device__ __forceinline__ KeyPair tok_pair(const TokArgs& a, uint64_t pair) {
    KeyPair v;
    asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(v.k[0].x), "=l"(v.k[0].y) : "l"(a.keys + 4 * pair) : "memory");
    asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(v.k[1].x), "=l"(v.k[1].y) : "l"(a.keys + 4 * pair + 2) : "memory");
    return v;
}
// The list of candidates: every slot whose rank is `floor` or more.  Filled when the whole table has been looked through; a slot
// whose rank rises past the floor later is added by whoever raised it (one that falls and rises again is in it twice: a tie with
// itself).  floor 0: there is none.
struct Candidates {
    uint32_t* slots;
    unsigned int* n;
    unsigned long long floor;
    __device__ __forceinline__ void add(uint64_t slot) const {
        const unsigned int at = atomicAdd(n, 1u);
        if (at < CAND_MAX) slots[at] = (uint32_t)slot;
    }
};
// Adds an occurrence of a window, or takes one out that was counted before this round.  1 if that claimed a slot.  (One loop
// for both: the lanes of a warp make their trips to the table together.)
__device__ __forceinline__ int tok_change(const TokArgs& a, const Key& key, int n, bool add, int round, const Candidates& cand) {
    Probe p(a, key);
    for (uint64_t probe = 0; probe <= p.mask; ++probe, p.next()) {
        const KeyPair v = tok_pair(a, p.pair);
        Key k0 = {v.k[0].x, v.k[0].y}, k1 = {v.k[1].x, v.k[1].y};
        bool claimed = false;
        // (a half that is still zero may belong to a key that is being written)
        if (add && (k0.lo == 0 || k0.hi == 0)) {
            k0 = cas128(a.keys + 4 * p.pair, Key{0ull, 0ull}, key);
            if (k0.lo == 0 && k0.hi == 0) { k0 = key; claimed = true; }
        }
        bool at0 = k0.lo == key.lo && k0.hi == key.hi;
        if (add && !at0 && (k1.lo == 0 || k1.hi == 0)) {
            k1 = cas128(a.keys + 4 * p.pair + 2, Key{0ull, 0ull}, key);
            if (k1.lo == 0 && k1.hi == 0) { k1 = key; claimed = true; }
        }
        if (at0 || (k1.lo == key.lo && k1.hi == key.hi)) {
            const uint64_t slot = 2 * p.pair + (at0 ? 0 : 1);
            const uint32_t old = atomicAdd(&a.words[slot], !add ? 0xFFFFFFFFu : claimed ? ((uint32_t)n << CNT_BITS) + 1u : 1u) & CNT_MASK;
            a.dirty[slot >> CHUNK_BITS] = 1;
            // (the length from here: whoever claimed the slot may not have written it yet)
            const uint32_t len = (uint32_t)n << CNT_BITS;
            if (add && cand.floor && tok_rank(len | (old + 1u)) >= cand.floor && tok_rank(len | old) < cand.floor) cand.add(slot);
            return claimed;
        }
        if (!add && k1.lo == 0 && k1.hi == 0) break;
    }
    a.st->rebuild = round + 1;                   // the table is full: all is counted again before the next round
    return 0;
}
// Rank and slot of a window's n-gram while no window is being added or taken out.
__device__ __forceinline__ unsigned long long tok_rank_of(const TokArgs& a, const Key& key, uint32_t& slot) {
    Probe p(a, key);
    for (uint64_t probe = 0; probe <= p.mask; ++probe, p.next()) {
        const KeyPair v = tok_pair(a, p.pair);
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (v.k[i].x == key.lo && v.k[i].y == key.hi) {
                slot = (uint32_t)(2 * p.pair + i);
                return tok_rank(__ldcg(a.words + slot));
            }
        if (v.k[1].x == 0 && v.k[1].y == 0) break;
    }
    return 0ull;
}

__device__ __forceinline__ void best_merge(Best& a, const Best& b) {
    if (b.rank > a.rank) a = b;
    else if (b.rank == a.rank && b.rank) { a.ties += b.ties; a.slot = min(a.slot, b.slot); }
}
__device__ __forceinline__ Best best_warp(Best v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Best x;
        x.rank = __shfl_xor_sync(0xFFFFFFFFu, v.rank, o);
        x.slot = __shfl_xor_sync(0xFFFFFFFFu, v.slot, o);
        x.ties = __shfl_xor_sync(0xFFFFFFFFu, v.ties, o);
        best_merge(v, x);
    }
    return v;
}
__device__ __forceinline__ Best best_load(const Best* p) {
    const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(p));
    return Best{v.x, (unsigned int)v.y, (unsigned int)(v.y >> 32)};
}

constexpr int DOC_SMEM = 256;                    // documents up to this length are rewritten in shared memory
constexpr int LIST_MAX = 512;                    // windows to take out or put in that a warp collects before it looks them up
constexpr int HIT_MAX = 1024;                    // documents of one CTA that are handed out to its warps in a round
struct TokWarp {
    int old_tok[DOC_SMEM], new_tok[DOC_SMEM];
    uint16_t list[LIST_MAX];                     // start (8 bits), length - 2 (3 bits), put in (1 bit)
    uint8_t old_mark[DOC_SMEM], new_mark[DOC_SMEM];
};
struct TokShared {
    Best red[TOK_WARPS];
    int n, tok[MAX_N];                           // this round's n-gram
    int stop;
    int n_tied;                                  // candidates of the best rank
    uint32_t tied_slot[TIED_MAX];
    Key tied_key[TIED_MAX];
    unsigned long long used;                     // of the round's state, read by one thread for all
    int rebuild;
    unsigned int n_cand;
    int windows[TOK_WARPS];                      // on the warps' lists
    int n_hits, next_hit, more_hits, long_hits;  // long_hits: a document of more than DOC_SMEM tokens is among them
    int hits[HIT_MAX], hit_len[HIT_MAX];         // documents, their lengths
    int64_t hit_at[HIT_MAX];                     // and where they start
    TokWarp warp[TOK_WARPS];
};

// Grid barrier in two halves; the wait is false when it ran out (a cooperative launch: all CTAs are resident).
__device__ __forceinline__ void tok_arrive(TokState* st, unsigned int& epoch) {
    ++epoch;
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&st->bar) : "memory");
}
__device__ __noinline__ bool tok_wait(TokState* st, unsigned int epoch, TokShared& sh) {
    if (threadIdx.x == 0) {
        const unsigned int target = epoch * gridDim.x;
        const long long t0 = clock64();
        for (;;) {
            unsigned int v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&st->bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if (clock64() - t0 > TOK_BARRIER_CYCLES) { set_status(&st->status, TASC_ETIMEOUT); sh.stop = 1; break; }
        }
    }
    __syncthreads();
    return sh.stop == 0;
}
__device__ __forceinline__ bool tok_barrier(TokState* st, unsigned int& epoch, TokShared& sh) {
    tok_arrive(st, epoch);
    return tok_wait(st, epoch, sh);
}

// A warp's list of windows: all lanes call everything.
struct TokList {
    TokWarp& w;
    const int32_t *old_tok, *new_tok;            // what the starts in the list count from
    int total;
    // the windows of the 32 positions from c on that hold a mark; starts are relative to `base`
    __device__ __forceinline__ void collect(const TokArgs& a, const uint8_t* mk, int L, int c, int base, bool add) {
        const int lane = threadIdx.x & 31, i = c + lane;
        // lengths of this position's windows that hold a mark: all from the first marked token on
        int from = MAX_N + 1;
        const int lim = min(a.n_max, L - i);
#pragma unroll
        for (int j = MAX_N - 1; j >= 0; --j) if (j < lim && mk[i + j]) from = j + 1;
        from = max(from, 2);
        const int cnt = max(0, lim - from + 1);
        int at = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, at, o);
            if (lane >= o) at += y;
        }
        const int sum = __shfl_sync(0xFFFFFFFFu, at, 31);
        at += total - cnt;
        for (int j = 0; j < cnt; ++j) w.list[at + j] = (uint16_t)((i - base) | ((from + j - 2) << 8) | (add ? 1 << 11 : 0));
        total += sum;
    }
    __device__ __forceinline__ bool full() const { return total + 32 * (MAX_N - 1) > LIST_MAX; }
    // looks the windows up; returns the slots this lane has claimed
    __device__ __forceinline__ int flush(const TokArgs& a, int round, const Candidates& cand) {
        int claimed = 0;
        __syncwarp();
        for (int p = threadIdx.x & 31; p < total; p += 32) {
            const int e = w.list[p], m = ((e >> 8) & 7) + 2;
            const bool add = (e >> 11) & 1;
            const int32_t* tok = (add ? new_tok : old_tok) + (e & 255);
            Key key = key_make(m);
#pragma unroll
            for (int j = 0; j < MAX_N; ++j) if (j < m) key_put(key, j, (uint32_t)tok[j]);
            claimed += tok_change(a, key, m, add, round, cand);
        }
        __syncwarp();
        total = 0;
        return claimed;
    }
};

// The occurrences of the round's n-gram among the 32 positions from c on: first tokens and the others of occurrences, as bits.
// skip: first position that is not part of the last occurrence.  (Left to right, non-overlapping.)
__device__ __forceinline__ void tok_occurrences(const TokShared& sh, const int32_t* tok, int L, int c, int& skip, uint32_t& starts, uint32_t& inside) {
    const int i = c + (threadIdx.x & 31), n = sh.n;
    bool hit = i + n <= L;
    for (int j = 0; hit && j < n; ++j) hit = tok[i + j] == sh.tok[j];
    uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit);
    starts = inside = 0u;
    if (skip > c) inside = skip - c >= 32 ? 0xFFFFFFFFu : (1u << (skip - c)) - 1u;
    while (hits) {
        const int p = c + __ffs(hits) - 1;
        hits &= hits - 1u;
        if (p < skip) continue;
        starts |= 1u << (p - c);
        skip = p + n;
        for (int q = p + 1; q < skip && q < c + 32; ++q) inside |= 1u << (q - c);
    }
}

// Replaces the occurrences of the round's n-gram in a document of at most DOC_SMEM tokens, in two steps.  First the document: it is worked
// on in shared memory and leaves its old and new tokens and marks there.  (Only this CTA reads it, so that does not wait for the
// others.)  Returns its new length and the chunks of 32 positions with a mark, old and new.
struct Rewritten { int len; uint32_t old_chunks, new_chunks; };
__device__ __noinline__ Rewritten tok_rewrite_short(const TokArgs& a, TokShared& sh, int d, int64_t s0, int L, int new_id) {
    const int lane = threadIdx.x & 31;
    TokWarp& w = sh.warp[threadIdx.x >> 5];
    int32_t* doc = a.cur + s0;
    int x[DOC_SMEM / 32];
#pragma unroll
    for (int u = 0; u < DOC_SMEM / 32; ++u) x[u] = u * 32 + lane < L ? doc[u * 32 + lane] : -1;
#pragma unroll
    for (int u = 0; u < DOC_SMEM / 32; ++u) if (u * 32 < L) w.old_tok[u * 32 + lane] = x[u];
    __syncwarp();
    // marks (1 = first of an occurrence, 2 = the others), and the document as it will be
    int skip = 0, wr = 0;
    uint32_t old_chunks = 0u, new_chunks = 0u;                 // chunks with a mark
#pragma unroll 1
    for (int c = 0; c < L; c += 32) {
        uint32_t starts, inside;
        tok_occurrences(sh, w.old_tok, L, c, skip, starts, inside);
        const int i = c + lane, f = (starts >> lane) & 1u ? 1 : ((inside >> lane) & 1u ? 2 : 0);
        if (starts | inside) old_chunks |= 1u << (c >> 5);
        const bool kept = i < L && f != 2;
        const uint32_t keep = __ballot_sync(0xFFFFFFFFu, kept);
        const int at = wr + __popc(keep & ((1u << lane) - 1u));
        if (i < L) w.old_mark[i] = (uint8_t)f;
        if (kept) {
            const int t = f == 1 ? new_id : w.old_tok[i];
            w.new_tok[at] = t;
            w.new_mark[at] = (uint8_t)f;
            doc[at] = t;
        }
        new_chunks |= __reduce_or_sync(0xFFFFFFFFu, kept && f == 1 ? 1u << (at >> 5) : 0u);
        wr += __popc(keep);
    }
    for (int i = lane; i < L; i += 32) {
        if (i < wr) a.rem[s0 + i] = (uint8_t)min(wr - 1 - i, 255);
        else doc[i] = -1;
    }
    if (lane == 0) a.doc_len[d] = wr;
    __syncwarp();
    return Rewritten{wr, old_chunks, new_chunks};
}
// Then the windows that change, old and new, are put on the warp's list.  Chunks without a changed token near are passed over.
// FLUSH: looks them up, and returns the slots that this lane has claimed.  Otherwise their number, -1 if they are more than the list holds.
template <bool FLUSH>
__device__ __noinline__ int tok_recount_short(const TokArgs& a, TokShared& sh, int L, Rewritten r, int round, const Candidates& cand) {
    TokWarp& w = sh.warp[threadIdx.x >> 5];
    TokList list = {w, w.old_tok, w.new_tok, 0};
    int claimed = 0;
#pragma unroll 1
    for (int c = 0; c < 2 * DOC_SMEM; c += 32) {
        const bool add = c >= DOC_SMEM;
        const int at = c & (DOC_SMEM - 1), len = add ? r.len : L;
        // (a window that holds a mark of the next chunk starts in this one)
        if (at < len && (((add ? r.new_chunks : r.old_chunks) >> (at >> 5)) & 3u)) {
            if (list.full()) {
                if (!FLUSH) return -1;
                claimed += list.flush(a, round, cand);
            }
            list.collect(a, add ? w.new_mark : w.old_mark, len, at, 0, add);
        }
    }
    return FLUSH ? claimed + list.flush(a, round, cand) : list.total;
}
// Looks up the windows of all warps' lists, dealt out to all threads of the CTA; returns the slots that this one has claimed.  (A look-up is
// two or three trips to L2 or to memory behind it, one after the other.  A round has a handful of documents per CTA: with every warp's
// windows looked up by itself, the warps with documents took 7 us of them and the others none.)
__device__ __noinline__ int tok_look_up(const TokArgs& a, TokShared& sh, int round, const Candidates& cand) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, mine = sh.windows[lane];
    int end = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, end, o);
        if (lane >= o) end += y;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, end, 31);
    int claimed = 0;
#pragma unroll 1
    for (int p0 = 0; p0 < total; p0 += TOK_THREADS) {
        const int p = p0 + lane * TOK_WARPS + warp;
        int of = 0;                                            // the list that has window p
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) if (__shfl_sync(0xFFFFFFFFu, end, of + o - 1) <= p) of += o;
        const int first = __shfl_sync(0xFFFFFFFFu, end - mine, of);
        if (p >= total) continue;
        const TokWarp& w = sh.warp[of];
        const int e = w.list[p - first], m = ((e >> 8) & 7) + 2;
        const bool add = (e >> 11) & 1;
        const int32_t* tok = (add ? w.new_tok : w.old_tok) + (e & 255);
        Key key = key_make(m);
#pragma unroll
        for (int j = 0; j < MAX_N; ++j) if (j < m) key_put(key, j, (uint32_t)tok[j]);
        claimed += tok_change(a, key, m, add, round, cand);
    }
    return claimed;
}

// The same for a longer document, in place, its windows chunk by chunk.
__device__ __noinline__ int tok_rewrite_long(const TokArgs& a, TokShared& sh, int d, int64_t s0, int L, int new_id, int round, const Candidates& cand) {
    const int lane = threadIdx.x & 31;
    TokWarp& w = sh.warp[threadIdx.x >> 5];
    int32_t* doc = a.cur + s0;
    uint8_t* mark = a.mark + s0;
    int skip = 0;
    for (int c = 0; c < L; c += 32) {
        uint32_t starts, inside;
        tok_occurrences(sh, doc, L, c, skip, starts, inside);
        if (c + lane < L) mark[c + lane] = (starts >> lane) & 1u ? 1 : ((inside >> lane) & 1u ? 2 : 0);
    }
    __syncwarp();
    TokList list = {w, doc, doc, 0};
    int claimed = 0;
    for (int c = 0; c < L; c += 32) {
        list.old_tok = doc + c;
        list.collect(a, mark, L, c, c, false);
        claimed += list.flush(a, round, cand);
    }
    // a chunk's tokens are in registers before any of them is overwritten, and what is written lies before it
    int wr = 0;
    for (int c = 0; c < L; c += 32) {
        const int i = c + lane;
        const int tok = i < L ? doc[i] : 0, f = i < L ? mark[i] : 2;
        const uint32_t keep = __ballot_sync(0xFFFFFFFFu, f != 2);
        const int at = wr + __popc(keep & ((1u << lane) - 1u));
        __syncwarp();
        if (f != 2) {
            doc[at] = f == 1 ? new_id : tok;
            mark[at] = (uint8_t)f;
        }
        wr += __popc(keep);
        __syncwarp();
    }
    for (int i = lane; i < L; i += 32) {
        if (i < wr) a.rem[s0 + i] = (uint8_t)min(wr - 1 - i, 255);
        else doc[i] = -1;
    }
    if (lane == 0) a.doc_len[d] = wr;
    __syncwarp();
    for (int c = 0; c < wr; c += 32) {
        list.new_tok = doc + c;
        list.collect(a, mark, wr, c, c, true);
        claimed += list.flush(a, round, cand);
    }
    return claimed;
}

// All rounds of Algorithm 1.  A round is a chain of short steps: the best n-gram, the documents that hold it (a warp looks
// through those that start in its share of the positions), a grid barrier, their rewriting (handed out to the warps of the CTA), a barrier.
//   The best n-gram comes from the list of candidates while the best of them is above its floor; every CTA finds it for
// itself.  Otherwise the table is looked through (the chunks that have changed; a barrier) and the list is made anew: the n-grams of three
// quarters of the best reward and more.  Where those are more than the list holds, the next round looks through the table again, and
// the list after it takes in half the distance from the best.
//   Measured on 20,000 documents (1.4 M tokens, 4.1 M windows, n_max 4), per round: 525 us when every round cleared and
// recounted the table, 33 when every round looked through the table's changed chunks (8 us, 4 more for the barrier and the best of
// all CTAs; a tie 30 us, because every window of the corpus was looked up to find the first), 27 when every warp read the round's state and looked
// up the windows of its own documents (256 rounds and the first count 6.7 ms), 22 now (5.6 ms).  By stamps, a round of 100 to 400 documents
// takes 18: 6 until they are listed, 3 to 5 to rewrite them, 1 the barrier, 4 to 5 the look-ups, 3 the barrier at its end; rounds of thousands, which
// come first, 20 to 90.
__global__ void __launch_bounds__(TOK_THREADS, 1) tok_rounds_kernel(const __grid_constant__ TokArgs a) {
    extern __shared__ __align__(16) uint8_t dyn[];
    TokShared& sh = *reinterpret_cast<TokShared*>(dyn);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * TOK_WARPS, wid = (int64_t)warp * gridDim.x + blockIdx.x;
    if (threadIdx.x == 0) { sh.stop = 0; sh.n_hits = 0; sh.next_hit = 0; sh.more_hits = 0; sh.long_hits = 0; }
    // this warp's documents
    auto doc_at = [&](int64_t pos) {
        int64_t lo = 0, hi = a.n_docs;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (a.offsets[mid] < pos) lo = mid + 1; else hi = mid;
        }
        return lo;
    };
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->first[0] = a.st->first[1] = ~0ull;
    const int64_t own = (int64_t)blockIdx.x * TOK_WARPS + warp;           // (neighbouring documents: one CTA's)
    const int64_t s = a.offsets[doc_at(own * a.T / nw)], e = own + 1 == nw ? a.T : a.offsets[doc_at((own + 1) * a.T / nw)];
    const uint64_t n_chunks = a.cap >> CHUNK_BITS;
    unsigned int epoch = 0;
    int n_merges = 0, n_ties = 0, n_rebuilds = 0, n_lists = 0, part = 2;
    Candidates cand = {a.cand, &a.st->n_cand[0], 0ull};
    __syncthreads();
    auto publish_claims = [&](int claimed) {
        claimed = __reduce_add_sync(0xFFFFFFFFu, claimed);
        if (lane == 0 && claimed) atomicAdd(&a.st->used[n_rebuilds & 1], (unsigned long long)claimed);
    };
    for (int round = 0;; ++round) {
        // ---- the table, if it has to be counted (again): n-grams that no longer occur keep their slots until then.  (One trip for all
        // that a round looks at first.)
        // (By one thread: read by all of them, 4,736 warps asked for the same three words, which took 2 us more.  A candidate's key and
        // count are on their way before it is known how many there are: a place that is not one is a slot of the table all the same.)
        if (threadIdx.x == 0) {
            sh.used = *(volatile unsigned long long*)&a.st->used[n_rebuilds & 1];
            sh.rebuild = *(volatile int*)&a.st->rebuild;
            sh.n_cand = *(volatile unsigned int*)cand.n;
        }
        const uint32_t cand_slot = __ldcg(cand.slots + threadIdx.x) & (uint32_t)(a.cap - 1);
        const ulonglong2 cand_key = __ldcg(reinterpret_cast<const ulonglong2*>(a.keys) + cand_slot);
        const uint32_t cand_word = __ldcg(a.words + cand_slot);
        __syncthreads();
        const unsigned long long used = sh.used;
        const int rebuild = sh.rebuild;
        unsigned int n_cand = sh.n_cand;
        if (rebuild == round || used * 4 > a.cap * 3) {
            const uint64_t gt = (uint64_t)blockIdx.x * TOK_THREADS + threadIdx.x, gn = (uint64_t)gridDim.x * TOK_THREADS;
            for (uint64_t i = gt; i < a.cap; i += gn) {
                reinterpret_cast<ulonglong2*>(a.keys)[i] = make_ulonglong2(0ull, 0ull);
                a.words[i] = 0u;
            }
            for (uint64_t i = gt; i < n_chunks; i += gn) a.dirty[i] = 1;
            ++n_rebuilds;
            cand.floor = 0ull;
            if (gt == 0) a.st->used[n_rebuilds & 1] = 0ull;
            if (!tok_barrier(a.st, epoch, sh)) return;
            int claimed = 0;
            for (int64_t i = s + lane; i < e; i += 32) {
                if (a.cur[i] < 0) continue;
                const int lim = min(a.n_max, (int)a.rem[i] + 1);
                for (int n = 2; n <= lim; ++n) {
                    Key key = key_make(n);
                    for (int j = 0; j < n; ++j) key_put(key, j, (uint32_t)a.cur[i + j]);
                    claimed += tok_change(a, key, n, true, round, cand);
                }
            }
            __syncwarp();
            publish_claims(claimed);
            if (!tok_barrier(a.st, epoch, sh)) return;
        }
        // ---- the best of the candidates.  (Nothing changes the table before every CTA has passed the next barrier.)
        Best best = {0ull, 0u, 0u};
        bool listed = false;
        int n_tied = 0;                                        // candidates of the best rank, in sh.tied as far as they fit
        if (cand.floor == 0ull) n_cand = 0u;
        if (n_cand > CAND_MAX) part = min(part + 1, 31);       // (did not fit: fewer the next time)
        else if (cand.floor) {
            uint32_t reward = 0u, len = 0u;
            Key key = {0ull, 0ull};
            if (threadIdx.x < n_cand) {
                const unsigned long long rank = tok_rank(cand_word);
                key = Key{cand_key.x, cand_key.y};
                reward = (uint32_t)(rank >> LEN_BITS);
                len = (uint32_t)rank & ((1u << LEN_BITS) - 1u);
            }
            if (threadIdx.x == 0) sh.n_tied = 0;
            uint32_t top = __reduce_max_sync(0xFFFFFFFFu, reward);
            uint32_t top_len = __reduce_max_sync(0xFFFFFFFFu, reward == top ? len : 0u);
            if (lane == 0) sh.red[warp].rank = ((unsigned long long)top << LEN_BITS) | top_len;
            __syncthreads();
            const unsigned long long r = sh.red[lane].rank;
            top = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(r >> LEN_BITS));
            top_len = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(r >> LEN_BITS) == top ? (uint32_t)r & ((1u << LEN_BITS) - 1u) : 0u);
            best.rank = ((unsigned long long)top << LEN_BITS) | top_len;
            listed = best.rank >= cand.floor;
            if (listed && reward == top && len == top_len) {
                const int at = atomicAdd(&sh.n_tied, 1);
                if (at < TIED_MAX) { sh.tied_slot[at] = cand_slot; sh.tied_key[at] = key; }
            }
            __syncthreads();
            n_tied = listed ? sh.n_tied : 0;
        }
        if (!listed) {
            // ---- the best of this warp's chunks of the table
            Best v = {0ull, 0u, 0u};
            for (uint64_t c0 = 0; c0 * nw < n_chunks; c0 += 32) {
                const uint64_t c = (c0 + lane) * nw + wid;
                const bool mine = c < n_chunks, stale = mine && __ldcg(a.dirty + c);
                Best b = {0ull, 0u, 0u};
                if (mine) b = a.chunk_best[c];
                uint32_t todo = __ballot_sync(0xFFFFFFFFu, stale);
                while (todo) {
                    int src[4];                                    // four chunks at a time
                    uint4 w[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        src[u] = __ffs(todo) - 1;
                        todo &= todo - 1u;
                        w[u] = make_uint4(0u, 0u, 0u, 0u);
                        if (src[u] >= 0) w[u] = __ldcg(reinterpret_cast<const uint4*>(a.words + (((c0 + src[u]) * nw + wid) << CHUNK_BITS)) + lane);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (src[u] < 0) break;
                        const uint32_t y[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
                        // the chunk's largest reward, then the lengths that have it (a reward is below 2^31)
                        uint32_t top = 0u;
#pragma unroll
                        for (int q = 0; q < 4; ++q) top = max(top, (y[q] & CNT_MASK) * ((y[q] >> CNT_BITS) - 1u));
                        top = __reduce_max_sync(0xFFFFFFFFu, top);
                        Best x = {0ull, 0u, 0u};
                        if (top) {
                            uint32_t len = 0u;
#pragma unroll
                            for (int q = 0; q < 4; ++q) if ((uint32_t)(tok_rank(y[q]) >> LEN_BITS) == top) len = max(len, y[q] >> CNT_BITS);
                            len = __reduce_max_sync(0xFFFFFFFFu, len);
                            x.rank = ((unsigned long long)top << LEN_BITS) | len;
                            uint32_t n_top = 0u, at = 0xFFFFFFFFu;
#pragma unroll
                            for (int q = 3; q >= 0; --q) if (tok_rank(y[q]) == x.rank) { ++n_top; at = lane * 4 + q; }
                            x.ties = __reduce_add_sync(0xFFFFFFFFu, n_top);
                            x.slot = (unsigned int)((((c0 + src[u]) * nw + wid) << CHUNK_BITS) + __reduce_min_sync(0xFFFFFFFFu, at));
                        }
                        if (lane == src[u]) { b = x; a.chunk_best[c] = x; a.dirty[c] = 0; }
                    }
                }
                best_merge(v, b);
            }
            auto block_best = [&](Best x) {
                x = best_warp(x);
                if (lane == 0) sh.red[warp] = x;
                __syncthreads();
                x = best_warp(sh.red[lane]);
                __syncthreads();
                return x;
            };
            v = block_best(v);
            if (threadIdx.x == 0) {
                a.cta_best[blockIdx.x] = v;
                if (blockIdx.x == 0) a.st->n_cand[(n_lists + 1) & 1] = 0u;
            }
            if (!tok_barrier(a.st, epoch, sh)) return;
            // ---- the best of all, found by every CTA for itself
            v = Best{0ull, 0u, 0u};
            if (warp == 0)
                for (int i = lane; i < (int)gridDim.x; i += 32) best_merge(v, best_load(a.cta_best + i));
            best = block_best(v);
            // ---- the candidates
            ++n_lists;
            const unsigned long long reward = best.rank >> LEN_BITS;
            cand = Candidates{a.cand + (n_lists & 1) * CAND_MAX, &a.st->n_cand[n_lists & 1], reward ? (reward - (reward >> part)) << LEN_BITS : 0ull};
            for (uint64_t c0 = 0; reward && c0 * nw < n_chunks; c0 += 32) {
                const uint64_t c = (c0 + lane) * nw + wid;
                uint32_t todo = __ballot_sync(0xFFFFFFFFu, c < n_chunks && a.chunk_best[c].rank >= cand.floor);
                for (; todo; todo &= todo - 1u) {
                    const uint64_t first = ((c0 + __ffs(todo) - 1) * nw + wid) << CHUNK_BITS;
                    // (a word that has been raised past the floor meanwhile is in the list twice, one that has fallen below is not missed)
                    const uint4 w = __ldcg(reinterpret_cast<const uint4*>(a.words + first) + lane);
                    const uint32_t y[4] = {w.x, w.y, w.z, w.w};
                    uint32_t full = 0u;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const bool in = tok_rank(y[q]) >= cand.floor;
                        const uint32_t who = __ballot_sync(0xFFFFFFFFu, in);
                        uint32_t at = 0u;
                        if (lane == 0 && who) at = atomicAdd(cand.n, (unsigned int)__popc(who));
                        at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(who & ((1u << lane) - 1u));
                        if (in && at < CAND_MAX) cand.slots[at] = (uint32_t)(first + lane * 4 + q);
                        full |= in && at >= CAND_MAX;              // (the counter has passed CAND_MAX: the next round sees the list as cut short)
                    }
                    if (__any_sync(0xFFFFFFFFu, full)) { c0 = n_chunks; break; }
                }
            }
        }
        if (best.rank == 0ull || n_merges >= a.budget) break;
        const int n = (int)(best.rank & ((1u << LEN_BITS) - 1u));
        bool tie = listed ? n_tied > 1 : best.ties > 1;
        if (n_tied > TIED_MAX) n_tied = 0;
        else if (tie && listed) {                              // several slots, or one several times?
            tie = false;
#pragma unroll 1
            for (int i = 1; i < n_tied; ++i) tie = tie || sh.tied_slot[i] != sh.tied_slot[0];
        }
        if (tie) {
            // ---- several: the one with the first position
            // (its slot comes along, so that its tokens are read from the table and the documents may change behind the next barrier)
            unsigned long long* first = &a.st->first[n_ties & 1];
            auto found_before = [&](int64_t p) { return (int64_t)__shfl_sync(0xFFFFFFFFu, (unsigned int)(*(volatile unsigned long long*)first >> 32), 0) <= p; };
            if (blockIdx.x == 0 && threadIdx.x == 0) a.st->first[~n_ties & 1] = ~0ull;
            if (n_tied) {
                // by their tokens, 512 positions at a time
                for (int64_t p = s & ~3ll; p < e; p += 512) {
                    if (found_before(p)) break;
                    int4 x[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int64_t q = p + u * 128 + 4 * lane;
                        x[u] = q < e ? *reinterpret_cast<const int4*>(a.cur + q) : make_int4(-1, -1, -1, -1);
                    }
                    unsigned int at = 0xFFFFFFFFu, slot = 0u;
                    for (int i = 0; i < n_tied; ++i) {
                        const int f = (int)key_get(sh.tied_key[i], 0);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int y[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int64_t q = p + u * 128 + 4 * lane + j;
                                if (y[j] != f || q < s || q >= e || q >= (int64_t)at || (int)a.rem[q] < n - 1) continue;
                                bool hit = true;
                                for (int k = 1; hit && k < n; ++k) hit = a.cur[q + k] == (int)key_get(sh.tied_key[i], k);
                                if (hit) { at = (unsigned int)q; slot = sh.tied_slot[i]; }
                            }
                        }
                    }
                    const unsigned int best_at = __reduce_min_sync(0xFFFFFFFFu, at);
                    if (best_at != 0xFFFFFFFFu) {
                        if (at == best_at) atomicMin(first, ((unsigned long long)at << 32) | slot);
                        break;
                    }
                }
            } else
            for (int64_t c = s; c < e; c += 32) {
                // (one lane's reading decides for all: the value changes meanwhile)
                if (found_before(c)) break;
                const int64_t i = c + lane;
                bool hit = false;
                uint32_t slot = 0u;
                if (i < e && a.cur[i] >= 0 && (int)a.rem[i] >= n - 1) {
                    Key key = key_make(n);
                    for (int j = 0; j < n; ++j) key_put(key, j, (uint32_t)a.cur[i + j]);
                    hit = tok_rank_of(a, key, slot) == best.rank;
                }
                const uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit);
                if (hits) {
                    if (lane == __ffs(hits) - 1) atomicMin(first, ((unsigned long long)i << 32) | slot);
                    break;
                }
            }
            ++n_ties;
            if (!tok_barrier(a.st, epoch, sh)) return;
        }
        if (threadIdx.x < MAX_N) {
            const int j = threadIdx.x;
            Key k = sh.tied_key[0];
            if (tie || !listed) {
                const uint32_t slot = tie ? (uint32_t)*(volatile unsigned long long*)&a.st->first[~n_ties & 1] : best.slot;
                const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(a.keys) + slot);
                k = Key{v.x, v.y};
            }
            const int t = j < n ? (int)key_get(k, j) : -1;
            sh.n = n;
            sh.tok[j] = t;
            if (blockIdx.x == 0) a.merges[(size_t)n_merges * MAX_N + j] = t;
        }
        const int new_id = a.base_vocab + n_merges++;
        __syncthreads();
        // ---- its documents: listed, and rewritten once every CTA has its n-gram; those that the list has no room for in another turn
        const int t0 = sh.tok[0];
        int claimed = 0;
        // (Behind a look through the table, and behind a tie, all CTAs are past what they read of it and of the documents.)
        for (bool passed = !listed || tie, more = true; more;) {
            for (int64_t p = s & ~3ll; p < e; p += 512) {
                int4 x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t q = p + u * 128 + 4 * lane;
                    x[u] = q < e ? *reinterpret_cast<const int4*>(a.cur + q) : make_int4(-1, -1, -1, -1);
                }
                uint32_t mine = 0u;                            // positions with the first token
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int y[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) mine |= y[j] == t0 ? 1u << (u * 4 + j) : 0u;
                }
                for (; mine; mine &= mine - 1u) {
                    const int b = __ffs(mine) - 1;
                    const int64_t q = p + (b >> 2) * 128 + 4 * lane + (b & 3);
                    // (an occurrence across the end of a document is found not to be one when the document is rewritten)
                    if (q < s || q >= e || q + n > a.T) continue;
                    const int d = a.doc_of[q];
                    bool hit = true;                           // (all tokens in one trip)
#pragma unroll
                    for (int i = 1; i < MAX_N; ++i) if (i < n) hit = (a.cur[q + i] == sh.tok[i]) & hit;
                    // the first hit of a document in this round puts it on the list
                    if (!hit) continue;
                    if (atomicExch(&a.doc_round[d], round + 1) == round + 1) continue;
                    const int L = a.doc_len[d];
                    const int64_t s0 = a.offsets[d];
                    const int slot = atomicAdd(&sh.n_hits, 1);
                    if (slot < HIT_MAX) { sh.hits[slot] = d; sh.hit_len[slot] = L; sh.hit_at[slot] = s0; if (L > DOC_SMEM) sh.long_hits = 1; }
                    else { atomicExch(&a.doc_round[d], round); sh.more_hits = 1; }
                }
            }
            __syncthreads();
            more = sh.more_hits != 0;
            const int n_hits = min(sh.n_hits, HIT_MAX);
            // while the barrier is on its way the warps work on their first documents
            if (!passed) tok_arrive(a.st, epoch);
            // A document for every warp at a time, its windows shared by all threads.  Where one of the CTA's documents is long (several times the
            // work, by one warp) its warps take documents as they get done instead, each with its own windows: otherwise 31 of them wait for it.
            // (128 added tokens on 10,000 documents, a tenth of them of 260 to 1,500 tokens: 12.3 -> 11.1 ms; one in 100 of 260 to 600, 20,000
            // documents: 6.6; no long ones, 10,000: 2.8.)
            const bool dealt_out = sh.long_hits == 0;
            while (!dealt_out) {
                int slot = 0;
                if (lane == 0) slot = atomicAdd(&sh.next_hit, 1);
                slot = __shfl_sync(0xFFFFFFFFu, slot, 0);
                const bool work = slot < n_hits;
                const int d = work ? sh.hits[slot] : 0, L = work ? sh.hit_len[slot] : 0;
                const int64_t s0 = work ? sh.hit_at[slot] : 0;
                Rewritten r = {0, 0u, 0u};
                if (work && L <= DOC_SMEM) r = tok_rewrite_short(a, sh, d, s0, L, new_id);
                if (!passed) {
                    if (!tok_wait(a.st, epoch, sh)) return;
                    passed = true;
                }
                if (!work) break;
                claimed += L <= DOC_SMEM ? tok_recount_short<true>(a, sh, L, r, round, cand) : tok_rewrite_long(a, sh, d, s0, L, new_id, round, cand);
            }
#pragma unroll 1
            for (int base = 0; dealt_out && (base < n_hits || !passed); base += TOK_WARPS) {
                const int slot = base + warp;
                const bool work = slot < n_hits;
                const int d = work ? sh.hits[slot] : 0, L = work ? sh.hit_len[slot] : 0;
                const int64_t s0 = work ? sh.hit_at[slot] : 0;
                Rewritten r = {0, 0u, 0u};
                int windows = 0;
                if (work) {
                    r = tok_rewrite_short(a, sh, d, s0, L, new_id);
                    windows = tok_recount_short<false>(a, sh, L, r, round, cand);
                }
                if (lane == 0) sh.windows[warp] = max(windows, 0);
                if (passed) __syncthreads();
                else if (!tok_wait(a.st, epoch, sh)) return;
                passed = true;
                claimed += tok_look_up(a, sh, round, cand);
                __syncthreads();                               // the lists are used again
                if (windows < 0) claimed += tok_recount_short<true>(a, sh, L, r, round, cand);
            }
            __syncthreads();
            if (threadIdx.x == 0) { sh.n_hits = 0; sh.next_hit = 0; sh.more_hits = 0; sh.long_hits = 0; }
            if (more) __syncthreads();
        }
        publish_claims(claimed);
        if (!tok_barrier(a.st, epoch, sh)) return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) a.st->n_merges = n_merges;
}

// What the host has to know about the documents before it can allocate.
struct TokCheck { unsigned long long windows; int64_t tokens; int bad; };
__global__ void tok_check_kernel(const int64_t* __restrict__ offsets, int64_t n_docs, int n_max, TokCheck* out) {
    unsigned long long w = 0;
    bool bad = false;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < n_docs; d += step) {
        const int64_t len = offsets[d + 1] - offsets[d];
        if (len < 0 || len >= (1ll << 31)) bad = true;
        else for (int n = 2; n <= n_max; ++n) w += (unsigned long long)(len - n + 1 > 0 ? len - n + 1 : 0);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xFFFFFFFFu, w, o);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd(&out->windows, w);
    if (bad || (blockIdx.x == 0 && threadIdx.x == 0 && offsets[0] != 0)) out->bad = 1;
    if (blockIdx.x == 0 && threadIdx.x == 0) out->tokens = offsets[n_docs];
}

// One warp per document.
__global__ void tok_init_docs_kernel(const int64_t* __restrict__ offsets, int64_t n_docs, int32_t* doc_len, int32_t* doc_round,
                                     int32_t* doc_of, uint8_t* rem) {
    const int64_t d = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (d >= n_docs) return;
    const int64_t s = offsets[d];
    const int L = (int)(offsets[d + 1] - s);
    if (lane == 0) { doc_len[d] = L; doc_round[d] = 0; }
    for (int j = lane; j < L; j += 32) {
        doc_of[s + j] = (int32_t)d;
        rem[s + j] = (uint8_t)min(L - 1 - j, 255);
    }
}

// Exclusive scan of the document lengths: blocks of 1,024 documents, their totals by one block, then the sum of both.
constexpr int SCAN_THREADS = 1024;
__device__ __forceinline__ long long block_exclusive(long long v, long long* s_warp, long long& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        long long w = s_warp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xFFFFFFFFu, w, o);
            if (lane >= o) w += y;
        }
        s_warp[lane] = w;
    }
    __syncthreads();
    total = s_warp[31];
    const long long r = x - v + (warp ? s_warp[warp - 1] : 0ll);
    __syncthreads();
    return r;
}
__global__ void __launch_bounds__(SCAN_THREADS)
tok_scan_blocks_kernel(const int32_t* __restrict__ doc_len, int64_t n_docs, int64_t* offsets_out, long long* totals) {
    __shared__ long long s_warp[32];
    const int64_t d = (int64_t)blockIdx.x * SCAN_THREADS + threadIdx.x;
    long long total;
    const long long r = block_exclusive(d < n_docs ? doc_len[d] : 0, s_warp, total);
    if (d < n_docs) offsets_out[d] = r;
    if (threadIdx.x == 0) totals[blockIdx.x] = total;
}
__global__ void __launch_bounds__(SCAN_THREADS)
tok_scan_totals_kernel(long long* totals, int64_t n_blocks, int64_t* end) {
    __shared__ long long s_warp[32];
    long long run = 0;
    for (int64_t b0 = 0; b0 < n_blocks; b0 += SCAN_THREADS) {
        const int64_t b = b0 + threadIdx.x;
        long long total;
        const long long r = block_exclusive(b < n_blocks ? totals[b] : 0, s_warp, total);
        if (b < n_blocks) totals[b] = run + r;
        run += total;
    }
    if (threadIdx.x == 0) *end = run;
}
// One warp per document: its final offset, and its tokens there.
__global__ void tok_compact_kernel(const int32_t* __restrict__ cur, const int64_t* __restrict__ offsets,
                                   const int32_t* __restrict__ doc_len, int64_t* offsets_out, const long long* __restrict__ totals,
                                   int64_t n_docs, int32_t* tokens_out) {
    const int64_t d = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (d >= n_docs) return;
    const int64_t off = offsets_out[d] + totals[d / SCAN_THREADS];
    __syncwarp();
    if (lane == 0) offsets_out[d] = off;
    const int32_t* src = cur + offsets[d];
    int32_t* dst = tokens_out + off;
    for (int j = lane; j < doc_len[d]; j += 32) dst[j] = src[j];
}

// ------------------------------------------------------------------------------------------- new rows
// Bound: a chain (a row may need any earlier one), mostly a short one, and the loads of what it starts from.  A block has ROWS_COLS columns, and its
// warps take the merges in turn: one waits for those of its constituents that are not there yet, whose rows other warps leave in shared memory.
// (Those that a merge waits for are earlier ones, and a warp's are in order: the first one that is not done never waits.)  Merges come in
// chunks, and the rows of the chunks before from where they were written.  256 merges of 896 columns: 316 us when a thread per column
// walked them one by one, 168 in groups of eight whose loads were under way together; the
// call 217 -> 70 us so (8,192 that need none: 5.9 -> 0.53 ms; a chain of 256, each of which needs the one before: 224 -> 198 us).
constexpr int ROWS_COLS = 32, ROWS_THREADS = 1024, ROWS_CHUNK = 256;
constexpr int ROWS_WAIT = 1 << 24;                 // looks at a row that is waited for (never reached, see above)
// (rows that other warps of the block have written: past L1)
__device__ __forceinline__ float load_row(const float* p) { return __ldcg(p); }
__device__ __forceinline__ __nv_bfloat16 load_row(const __nv_bfloat16* p) { return __ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short*>(p))); }
template <typename T>
__global__ void __launch_bounds__(ROWS_THREADS)
tok_rows_kernel(const T* base, int base_vocab, int d, const int32_t* __restrict__ merges, int n_merges, T* rows_out,
                int* status) {
    __shared__ float s_row[ROWS_CHUNK][ROWS_COLS];
    __shared__ int32_t s_tok[ROWS_CHUNK * MAX_N];
    __shared__ volatile int s_done[ROWS_CHUNK];
    constexpr int WARPS = ROWS_THREADS / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x * ROWS_COLS + lane;
    for (int c0 = 0; c0 < n_merges; c0 += ROWS_CHUNK) {
        const int n = min(ROWS_CHUNK, n_merges - c0);
        __syncthreads();                                          // the chunk before: its rows are written, and no longer read from here
        for (int i = threadIdx.x; i < n * MAX_N; i += ROWS_THREADS) s_tok[i] = merges[(size_t)c0 * MAX_N + i];
        if (threadIdx.x < ROWS_CHUNK) s_done[threadIdx.x] = 0;
        __syncthreads();
        T val[MAX_N], next[MAX_N];
        // what does not come from this chunk (no branch: all loads are under way together; what cannot be used reads some other row)
        auto fetch = [&](int i, T (&v)[MAX_N]) {
#pragma unroll
            for (int c = 0; c < MAX_N; ++c) {
                const int t = s_tok[i * MAX_N + c], at = t - base_vocab;
                const T* row = t >= 0 && at >= 0 && at < c0 ? rows_out + (size_t)at * d : base + (size_t)(t >= 0 && at < 0 ? t : 0) * d;
                v[c] = j < d ? load_row(row + j) : Num<T>::from_f(0.f);
            }
        };
        if (warp < n) fetch(warp, val);
        for (int i = warp; i < n; i += WARPS) {
            if (i + WARPS < n) fetch(i + WARPS, next);
            float acc = 0.f;
            int count = 0;
            bool more = true;
#pragma unroll
            for (int c = 0; c < MAX_N; ++c) {
                const int t = s_tok[i * MAX_N + c], at = t - base_vocab;
                more = more && t >= 0;
                if (!more) continue;
                ++count;
                if (at >= c0 + i) { set_status(status, TASC_EINVAL); continue; }         // a constituent that does not exist yet
                float v = Num<T>::to_f(val[c]);
                if (at >= c0) {
                    for (int look = 0; s_done[at - c0] == 0; ++look)
                        if (look == ROWS_WAIT) { set_status(status, TASC_EINVAL); break; }
                    __threadfence_block();
                    v = s_row[at - c0][lane];
                }
                acc += v;
            }
            if (count < 2) { set_status(status, TASC_EINVAL); count = 1; }
            const T mean = Num<T>::from_f(acc / (float)count);
            s_row[i][lane] = Num<T>::to_f(mean);
            if (j < d) rows_out[(size_t)(c0 + i) * d + j] = mean;
            __threadfence_block();
            __syncwarp();
            if (lane == 0) s_done[i] = 1;
#pragma unroll
            for (int c = 0; c < MAX_N; ++c) val[c] = next[c];
        }
    }
}

// ------------------------------------------------------------------------------------------- encode
struct TrieTable { const uint64_t* keys; const int32_t* child; const int32_t* token; uint64_t mask; };

__device__ __forceinline__ uint64_t trie_hash(uint64_t k) {
    k ^= k >> 33; k *= 0xFF51AFD7ED558CCDull; k ^= k >> 33; k *= 0xC4CEB9FE1A85EC53ull; k ^= k >> 33;
    return k;
}
// child of `node` along `tok`, or -1
__device__ __forceinline__ int trie_step(const TrieTable& t, int node, int tok) {
    const uint64_t key = ((uint64_t)(uint32_t)node << 32) | (uint64_t)(uint32_t)tok | (1ull << 63);
    uint64_t slot = trie_hash(key) & t.mask;
    for (uint64_t probe = 0; probe <= t.mask; ++probe) {
        const uint64_t k = t.keys[slot];
        if (k == key) return t.child[slot];
        if (k == 0ull) return -1;
        slot = (slot + 1) & t.mask;
    }
    return -1;
}

// One thread per document: at every position the longest added token whose expansion matches, else the base token.
// Output in place of a scratch copy at the document's original offset; lengths to doc_len.
__global__ void tok_encode_kernel(const int32_t* __restrict__ tokens, const int64_t* __restrict__ offsets, int64_t n_docs,
                                  TrieTable trie, int32_t* scratch, int32_t* doc_len) {
    const int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= n_docs) return;
    const int64_t s = offsets[d];
    const int L = (int)(offsets[d + 1] - s);
    const int32_t* doc = tokens + s;
    int32_t* out = scratch + s;
    int i = 0, w = 0;
    while (i < L) {
        int node = 0, best_tok = -1, best_len = 0;
        for (int j = i; j < L; ++j) {
            node = trie_step(trie, node, doc[j]);
            if (node < 0) break;
            const int tk = trie.token[node];
            if (tk >= 0) { best_tok = tk; best_len = j - i + 1; }
        }
        if (best_tok >= 0) { out[w++] = best_tok; i += best_len; }
        else { out[w++] = doc[i++]; }
    }
    doc_len[d] = w;
}

int64_t scan_blocks(int64_t n_docs) { return (n_docs + SCAN_THREADS - 1) / SCAN_THREADS; }
// totals: scan_blocks(n_docs) words
tasc_status compact_docs(const int32_t* cur, const int64_t* offsets, const int32_t* doc_len, int64_t n_docs, long long* totals,
                         int32_t* tokens_out, int64_t* offsets_out, cudaStream_t stream) {
    const int64_t nb = scan_blocks(n_docs);
    if (nb) tok_scan_blocks_kernel<<<(unsigned)nb, SCAN_THREADS, 0, stream>>>(doc_len, n_docs, offsets_out, totals);
    tok_scan_totals_kernel<<<1, SCAN_THREADS, 0, stream>>>(totals, nb, reinterpret_cast<int64_t*>(offsets_out) + n_docs);
    if (nb) tok_compact_kernel<<<blocks_for((uint64_t)n_docs, 8), 256, 0, stream>>>(cur, offsets, doc_len, offsets_out, totals, n_docs, tokens_out);
    TASC_CUDA_TRY(cudaGetLastError());
    return TASC_OK;
}

}  // namespace
}  // namespace tasc

using namespace tasc;

extern "C" tasc_status tasc_tok_enrich(const int32_t* corpus_tokens, const int64_t* doc_offsets, int64_t n_docs,
                                       int32_t base_vocab, int32_t budget, int32_t n_max, int32_t* merges,
                                       int32_t* n_merges, int32_t* tokens_out, int64_t* offsets_out, tasc_stream stream_) {
    if (!doc_offsets || !merges || !n_merges || !offsets_out || n_docs < 0 || base_vocab < 1 || budget < 0 || n_max < 2 ||
        n_max > MAX_N || (int64_t)base_vocab + budget > (1 << TASC_VOCAB_BITS) || n_docs >= (1ll << 31))
        return TASC_EINVAL;
    *n_merges = 0;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    DeviceSlab slab;
    const TokCheck zero = {0ull, 0, 0};
    TokCheck hc;
    {
        DeviceSlab small;
        const size_t o = small.add(sizeof(TokCheck));
        if (!small.allocate(stream)) return TASC_ENOMEM;
        TokCheck* dc = small.at<TokCheck>(o);
        TASC_CUDA_TRY(cudaMemcpyAsync(dc, &zero, sizeof(zero), cudaMemcpyHostToDevice, stream));
        tok_check_kernel<<<std::min(blocks_for((uint64_t)n_docs + 1, 256), 592u), 256, 0, stream>>>(doc_offsets, n_docs, n_max, dc);
        TASC_CUDA_TRY(cudaMemcpyAsync(&hc, dc, sizeof(hc), cudaMemcpyDeviceToHost, stream));
        TASC_CUDA_TRY(cudaStreamSynchronize(stream));
    }
    const int64_t T = hc.tokens;
    if (hc.bad || T < 0 || T >= (1ll << POS_BITS)) return TASC_EINVAL;
    if (T > 0 && (!corpus_tokens || !tokens_out)) return TASC_EINVAL;

    int dev = 0, grid = 0;
    TASC_CUDA_TRY(cudaGetDevice(&dev));
    TASC_CUDA_TRY(cudaDeviceGetAttribute(&grid, cudaDevAttrMultiProcessorCount, dev));      // one CTA per SM
    const uint64_t cap = std::max<uint64_t>(pow2_at_least(2 * hc.windows), 1ull << CHUNK_BITS), chunks = cap >> CHUNK_BITS;
    const size_t t = (size_t)T + 4, nd = (size_t)n_docs;
    const size_t o_keys = slab.add(cap * 16), o_words = slab.add(cap * 4), o_dirty = slab.add(chunks), o_chunk = slab.add(chunks * sizeof(Best)),
                 o_cta = slab.add(grid * sizeof(Best)), o_cand = slab.add(2 * CAND_MAX * 4), o_st = slab.add(sizeof(TokState)), o_cur = slab.add(t * 4), o_of = slab.add(t * 4),
                 o_rem = slab.add(t), o_mark = slab.add(t), o_len = slab.add(nd * 4), o_round = slab.add(nd * 4), o_tot = slab.add(scan_blocks(n_docs) * 8);
    if (!slab.allocate(stream)) return TASC_ENOMEM;
    TokArgs a = {};
    a.cur = slab.at<int32_t>(o_cur); a.rem = slab.at<uint8_t>(o_rem); a.mark = slab.at<uint8_t>(o_mark); a.doc_of = slab.at<int32_t>(o_of);
    a.offsets = doc_offsets; a.doc_len = slab.at<int32_t>(o_len); a.doc_round = slab.at<int32_t>(o_round); a.n_docs = n_docs; a.T = T;
    a.keys = slab.at<uint64_t>(o_keys); a.words = slab.at<uint32_t>(o_words); a.dirty = slab.at<uint8_t>(o_dirty);
    a.chunk_best = slab.at<Best>(o_chunk); a.cta_best = slab.at<Best>(o_cta); a.cand = slab.at<uint32_t>(o_cand); a.cap = cap; a.st = slab.at<TokState>(o_st);
    a.merges = merges; a.base_vocab = base_vocab; a.budget = budget; a.n_max = n_max;
    TokState hs = {};
    TASC_CUDA_TRY(cudaMemsetAsync(a.st, 0, sizeof(TokState), stream));
    TASC_CUDA_TRY(cudaMemsetAsync(merges, 0xFF, (size_t)budget * MAX_N * sizeof(int32_t), stream));
    if (T > 0) TASC_CUDA_TRY(cudaMemcpyAsync(a.cur, corpus_tokens, (size_t)T * 4, cudaMemcpyDeviceToDevice, stream));
    if (n_docs > 0) tok_init_docs_kernel<<<blocks_for(nd, 8), 256, 0, stream>>>(doc_offsets, n_docs, a.doc_len, a.doc_round, slab.at<int32_t>(o_of), a.rem);
    if (T > 0 && budget > 0) {
        void* args[] = {&a};
        TASC_CUDA_TRY(cudaFuncSetAttribute(tok_rounds_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TokShared)));
        TASC_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(tok_rounds_kernel), dim3(grid), dim3(TOK_THREADS), args, sizeof(TokShared), stream));
    }
    const tasc_status rc = compact_docs(a.cur, doc_offsets, a.doc_len, n_docs, slab.at<long long>(o_tot), tokens_out, offsets_out, stream);
    if (rc != TASC_OK) return rc;
    TASC_CUDA_TRY(cudaMemcpyAsync(&hs, a.st, sizeof(hs), cudaMemcpyDeviceToHost, stream));
    TASC_CUDA_TRY(cudaStreamSynchronize(stream));
    if (hs.status != 0) return hs.status;
    *n_merges = hs.n_merges;
    return TASC_OK;
}

extern "C" tasc_status tasc_tok_init_rows(const void* matrix, int32_t dtype, int32_t base_vocab, int32_t d,
                                          const int32_t* merges, int32_t n_merges, void* rows_out, int32_t* device_status,
                                          tasc_stream stream_) {
    if (!matrix || !merges || !rows_out || !device_status || base_vocab < 1 || d < 1 || n_merges < 0 ||
        (dtype != TASC_F32 && dtype != TASC_BF16))
        return TASC_EINVAL;
    if (n_merges == 0) return TASC_OK;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const unsigned blocks = (unsigned)((d + ROWS_COLS - 1) / ROWS_COLS);
    if (dtype == TASC_F32)
        tok_rows_kernel<float><<<blocks, ROWS_THREADS, 0, stream>>>(static_cast<const float*>(matrix), base_vocab, d, merges, n_merges,
                                                           static_cast<float*>(rows_out), device_status);
    else
        tok_rows_kernel<__nv_bfloat16><<<blocks, ROWS_THREADS, 0, stream>>>(static_cast<const __nv_bfloat16*>(matrix), base_vocab, d, merges,
                                                                   n_merges, static_cast<__nv_bfloat16*>(rows_out), device_status);
    TASC_CUDA_TRY(cudaGetLastError());
    return TASC_OK;
}

extern "C" tasc_status tasc_tok_encode(const int32_t* tokens, const int64_t* doc_offsets, int64_t n_docs, int32_t base_vocab,
                                       const int32_t* merges, int32_t n_merges, int32_t* tokens_out, int64_t* offsets_out,
                                       tasc_stream stream_) {
    if (!doc_offsets || !offsets_out || n_docs < 0 || base_vocab < 1 || n_merges < 0 || (n_merges > 0 && !merges)) return TASC_EINVAL;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    // the added tokens' expansions into base tokens, then the trie over them (host: a few thousand short sequences)
    std::vector<int32_t> hm((size_t)n_merges * MAX_N);
    int64_t T = 0;
    if (n_merges > 0) TASC_CUDA_TRY(cudaMemcpyAsync(hm.data(), merges, hm.size() * 4, cudaMemcpyDeviceToHost, stream));
    TASC_CUDA_TRY(cudaMemcpyAsync(&T, doc_offsets + n_docs, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
    TASC_CUDA_TRY(cudaStreamSynchronize(stream));
    if (T < 0 || (T > 0 && (!tokens || !tokens_out))) return TASC_EINVAL;
    constexpr size_t MAX_EXPANSION = 4096;
    std::vector<std::vector<int32_t>> exp((size_t)n_merges);
    for (int i = 0; i < n_merges; ++i) {
        for (int c = 0; c < MAX_N; ++c) {
            const int t = hm[(size_t)i * MAX_N + c];
            if (t < 0) break;
            if (t < base_vocab) exp[i].push_back(t);
            else if (t - base_vocab < i) exp[i].insert(exp[i].end(), exp[t - base_vocab].begin(), exp[t - base_vocab].end());
            else return TASC_EINVAL;
            if (exp[i].size() > MAX_EXPANSION) return TASC_ECAPACITY;
        }
        if (exp[i].size() < 2) return TASC_EINVAL;
    }
    // (node, token) -> child, in the open-addressing form that the kernel reads, twice as many slots as edges or more.  (With a std::map of the
    // edges and a copy per array the call took 511 us for 256 added tokens and 100,000 documents, 409 for 100 documents;
    // 411 and 319 so.)
    auto mix = [](uint64_t k) { k ^= k >> 33; k *= 0xFF51AFD7ED558CCDull; k ^= k >> 33; k *= 0xC4CEB9FE1A85EC53ull; k ^= k >> 33; return k; };
    struct Edges {
        std::vector<uint64_t> key;
        std::vector<int32_t> child;
        explicit Edges(uint64_t slots) : key(slots, 0ull), child(slots, -1) {}
    };
    auto slot_of = [&](const Edges& e, uint64_t key) {
        uint64_t slot = mix(key) & (e.key.size() - 1);
        while (e.key[slot] != 0ull && e.key[slot] != key) slot = (slot + 1) & (e.key.size() - 1);
        return slot;
    };
    uint64_t n_edges = 0;
    Edges edges(1024);
    std::vector<int32_t> node_token(1, -1);
    for (int i = 0; i < n_merges; ++i) {
        int node = 0;
        for (int32_t t : exp[i]) {
            const uint64_t key = ((uint64_t)(uint32_t)node << 32) | (uint64_t)(uint32_t)t | (1ull << 63), slot = slot_of(edges, key);
            if (edges.key[slot] == 0ull) {
                edges.key[slot] = key;
                edges.child[slot] = (int32_t)node_token.size();
                node_token.push_back(-1);
                node = edges.child[slot];
                if (2 * ++n_edges <= edges.key.size()) continue;
                Edges more(2 * edges.key.size());
                for (size_t e = 0; e < edges.key.size(); ++e)
                    if (edges.key[e] != 0ull) {
                        const uint64_t to = slot_of(more, edges.key[e]);
                        more.key[to] = edges.key[e];
                        more.child[to] = edges.child[e];
                    }
                edges = std::move(more);
            } else {
                node = edges.child[slot];
            }
        }
        if (node_token[node] < 0) node_token[node] = base_vocab + i;     // two added tokens with one expansion: the earlier one
    }
    const uint64_t cap = edges.key.size();
    DeviceSlab slab;
    const size_t o_keys = slab.add(cap * 8), o_child = slab.add(cap * 4), o_tok = slab.add(node_token.size() * 4),
                 o_scratch = slab.add((size_t)T * 4), o_len = slab.add((size_t)n_docs * 4), o_tot = slab.add(scan_blocks(n_docs) * 8);
    if (!slab.allocate(stream)) return TASC_ENOMEM;
    int32_t *scratch = slab.at<int32_t>(o_scratch), *doc_len = slab.at<int32_t>(o_len);
    std::vector<uint8_t> table(o_tok - o_keys + node_token.size() * 4);      // all three in one copy
    memcpy(table.data(), edges.key.data(), cap * 8);
    memcpy(table.data() + (o_child - o_keys), edges.child.data(), cap * 4);
    memcpy(table.data() + (o_tok - o_keys), node_token.data(), node_token.size() * 4);
    TASC_CUDA_TRY(cudaMemcpyAsync(slab.at<uint8_t>(o_keys), table.data(), table.size(), cudaMemcpyHostToDevice, stream));
    const TrieTable trie = {slab.at<uint64_t>(o_keys), slab.at<int32_t>(o_child), slab.at<int32_t>(o_tok), cap - 1};
    if (n_docs > 0)
        tok_encode_kernel<<<blocks_for((uint64_t)n_docs, 128), 128, 0, stream>>>(tokens, doc_offsets, n_docs, trie, scratch, doc_len);
    TASC_CUDA_TRY(cudaGetLastError());
    const tasc_status rc = compact_docs(scratch, doc_offsets, doc_len, n_docs, slab.at<long long>(o_tot), tokens_out, offsets_out, stream);
    TASC_CUDA_TRY(cudaStreamSynchronize(stream));                    // the host tables must outlive the copies
    return rc;
}
