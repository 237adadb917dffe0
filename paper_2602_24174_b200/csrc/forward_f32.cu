// The whole forward of a small float32 model as ONE kernel of one thread-block cluster.
//
// Bound: a chain of dependent steps, each a microsecond or less of work.  As one launch per stage (api.cu, forward_f32) a
// verify step of the two-layer, 128-wide configuration was 25 launches, 6 us each.  Sixteen SMs have room for the work and
// share a hardware barrier (about 0.25 us, against 1.3 us for one across the grid), so the stages run one after the other
// in one cluster: QKV + RoPE + KV append, attention, O + residual, norm + gate/up + SiLU * mul, down + residual, and the
// LM head with its arg-max.  What one stage hands to the next goes through L2; every CTA stages the rows it multiplies in
// its shared memory and works out their norms itself.
//
// Products: a warp owns a pair of weight rows (the halves of a rotary pair, a gate row and its up row) for all token rows,
// eight at a time; its lanes stride over k with 16-byte loads.  Attention: eight warps own a (row, query head), share its
// keys in blocks of eight (four lanes to a key for the scores, lanes = dimensions for P V) and merge their softmax states.
// (Blocks of 32 keys left most of the eight warps idle at 100 keys: 11 us per layer against 5.)
//
// Measured, draft + verify step of that configuration at one sequence: 174 us as a chain, 60 us so, 54 since it is set up while the
// draft runs and its stages are one copy of code (9 in the draft; replayed from a graph 52).
#include "kernels.h"

#include <algorithm>
#include <mutex>

namespace tasc {

namespace {

constexpr int CTAS = 16;                         // one non-portable cluster
constexpr int THREADS = 1024, WARPS = THREADS / 32;
constexpr int ROWS = 8;                          // token rows a warp multiplies at a time
constexpr int UNIT_WARPS = 8;                    // warps of an attention unit
constexpr int KEYS = 8;                          // keys of an attention step: four lanes to a key
constexpr int MAX_HD = 256;
constexpr int MAX_SMEM = 220 * 1024;

#ifdef TASC_TIMELINE
// A stage of a CTA: start, rows staged, work done, behind the barrier.
#define TL_STAGED() (tl_a = global_ns())
#define TL_END(tag) do { if (threadIdx.x == 0) ctalog_put(tl_0, tl_a, tl_b, tag); tl_0 = tl_a = global_ns(); } while (0)
#else
#define TL_STAGED() do { } while (0)
#endif

// Sums of eight values over the warp's lanes; lane l gets the sum of value l / 4.
__device__ __forceinline__ float sum8(float (&v)[ROWS]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const int o = 4 * h;
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float mine = up ? v[i + h] : v[i], theirs = up ? v[i] : v[i + h];
            v[i] = mine + __shfl_xor_sync(0xFFFFFFFFu, theirs, o);
        }
    }
    v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 2);
    v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 1);
    return v[0];
}
__device__ __forceinline__ float4 ldg_fresh(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }   // another CTA's result

// y[r] = dot(w0, x row r), z[r] = dot(w1, x row r) for eight rows; a, b: the lane's first weights, there already.
__device__ __forceinline__ void dot_pair(const float* __restrict__ w0, const float* __restrict__ w1, float4 a, float4 b, const float* x0, int K,
                                         float (&y)[ROWS], float (&z)[ROWS]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) y[r] = z[r] = 0.f;
#pragma unroll 1
    for (int k = 4 * lane; k < K;) {
        const int next = k + 128;
        float4 a2 = a, b2 = b;
        if (next < K) { a2 = __ldg(reinterpret_cast<const float4*>(w0 + next)); b2 = __ldg(reinterpret_cast<const float4*>(w1 + next)); }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const float4 x = *reinterpret_cast<const float4*>(x0 + r * K + k);
            y[r] = fmaf(a.x, x.x, fmaf(a.y, x.y, fmaf(a.z, x.z, fmaf(a.w, x.w, y[r]))));
            z[r] = fmaf(b.x, x.x, fmaf(b.y, x.y, fmaf(b.z, x.z, fmaf(b.w, x.w, z[r]))));
        }
        k = next; a = a2; b = b2;
    }
}

enum { ST_QKV, ST_ATTN, ST_O, ST_GATE_UP, ST_DOWN, ST_LM };      // the stages of a layer, and the LM head

// NJ: 32-wide pieces of a head.
template <int NJ>
__global__ void __launch_bounds__(THREADS, 1) forward_f32_kernel(const __grid_constant__ ForwardF32Args a) {
    extern __shared__ __align__(16) float sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = (int)cluster_ctarank();
    const int gw = warp * CTAS + cta;                            // neighbouring features on different SMs
    const int M = a.M, d = a.d, hd = a.hd, half = hd >> 1, qd = a.n_q * hd;
    float* xs = sm;                                              // [M rounded up to 8][widest input] rows of the running product
    float* part = xs + (size_t)((M + ROWS - 1) / ROWS * ROWS) * a.width;                      // [WARPS][hd + 4] attention states
    int* s_pos = reinterpret_cast<int*>(part + WARPS * (hd + 4));
    int* s_tok = s_pos + M;
    unsigned long long* s_best = reinterpret_cast<unsigned long long*>(s_tok + M);

#ifdef TASC_TIMELINE
    unsigned long long tl_0 = global_ns(), tl_a = tl_0, tl_b = tl_0;
    int tl_tag = 0;
#endif
    griddep_wait();
    griddep_launch_dependents();
    // ---- row plan: every CTA for itself, CTA 0 for the kernels behind
#pragma unroll 1
    for (int m = threadIdx.x; m < M; m += THREADS) {
        const int b = a.by_R.div(m), r = m - b * a.R, L = a.len[b];
        const bool len_ok = L >= 1 && L <= a.stride;
        if (!len_ok) set_status(a.status, TASC_EINVAL);
        int tok = 0, pos = -1, pos0 = 0, rows = 0;
        if (a.chunk < 0) {
            if (len_ok && !(a.stop_len && L >= a.stop_len[b])) {
                tok = r == 0 ? a.tokens[(int64_t)b * a.stride + L - 1] : a.drafts[b * (a.R - 1) + r - 1];
                pos = L - 1 + r;
                pos0 = L - 1;
                rows = a.R;
            }
        } else {
            pos0 = a.chunk * a.R;
            rows = len_ok ? max(0, min(a.R, L - 1 - pos0)) : 0;
            if (r < rows) {
                tok = a.tokens[(int64_t)b * a.stride + pos0 + r];
                pos = pos0 + r;
            }
        }
        if (tok < 0 || tok >= a.vocab) { set_status(a.status, TASC_EINVAL); tok = 0; }
        s_tok[m] = tok;
        s_pos[m] = pos;
        s_best[m] = 0ull;
        if (cta == 0) {
            a.rp.row_tok[m] = tok;
            a.rp.row_pos[m] = pos;
            if (r == 0) { a.rp.seq_pos0[b] = pos0; a.rp.seq_rows[b] = rows; }
            if (a.argmax) a.argmax[m] = 0ull;
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int m = warp; m < M; m += WARPS)                        // (row m by CTA m % CTAS)
        if (m % CTAS == cta)
            for (int j = 4 * lane; j < d; j += 128) *reinterpret_cast<float4*>(a.x + (size_t)m * d + j) = __ldg(reinterpret_cast<const float4*>(a.embed + (size_t)s_tok[m] * d + j));
    // One copy of a stage's code for all products (five copies: 114 - 128 KB of kernel, a third of the instruction-cache requests
    // missed and the kernel took 61 us under ncu; now 49 - 62 KB, 7 % and 50 us).  A stage's first weights, which depend on
    // nothing, are requested before the barrier that precedes it.
    int stage = ST_QKV, l = 0;
    LayerWeightsF32 lw = a.layers[0];
    bool first = true;
#pragma unroll 1
    for (;;) {
        if (stage == ST_LM && !a.lm_head) { if (!first) cluster_wait(); return; }
        if (stage != ST_ATTN) {
            const float* W = stage == ST_QKV ? lw.wqkv : stage == ST_O ? lw.wo : stage == ST_GATE_UP ? lw.w_gate_up : stage == ST_DOWN ? lw.w_down : a.lm_head;
            const int K = stage == ST_O ? qd : stage == ST_DOWN ? a.dff : d;
            const int n_pairs = stage == ST_QKV ? (a.n_q + 2 * a.n_kv) * half : stage == ST_GATE_UP ? a.dff : stage == ST_LM ? (a.vocab + 1) / 2 : d / 2;
            // a pair's weight rows: the halves of a rotary pair (value heads: the same pairs, not rotated), a gate row and its up row,
            // two neighbouring features
            auto rows_of = [&](int p, const float*& w0, const float*& w1) {
                int r0 = 2 * p, r1 = 2 * p + 1;
                if (stage == ST_QKV) { const int head = a.by_half.div(p); r0 = p + head * half; r1 = r0 + half; }
                else if (stage == ST_GATE_UP) { r0 = p; r1 = a.dff + p; }
                else if (stage == ST_LM) r1 = min(r1, a.vocab - 1);
                w0 = W + (size_t)r0 * K;
                w1 = W + (size_t)r1 * K;
            };
            const float *w0 = W, *w1 = W;
            float4 wa = make_float4(0.f, 0.f, 0.f, 0.f), wb = wa;
            if (gw < n_pairs) {
                rows_of(gw, w0, w1);
                if (4 * lane < K) { wa = __ldg(reinterpret_cast<const float4*>(w0 + 4 * lane)); wb = __ldg(reinterpret_cast<const float4*>(w1 + 4 * lane)); }
            }
            if (!first) cluster_wait();
#ifdef TASC_TIMELINE
            if (!first) TL_END(tl_tag);
#endif
            if (stage == ST_O || stage == ST_DOWN) {
                const float* src = stage == ST_O ? a.o : a.act;
#pragma unroll 1
                for (int i = threadIdx.x; i < M * (K / 4); i += THREADS) *reinterpret_cast<float4*>(xs + 4 * (size_t)i) = ldg_fresh(src + 4 * (size_t)i);
            } else {
                // rows of the residual stream -> RMS norm * gain in shared memory (first: straight from the embedding)
                const float* gain = stage == ST_QKV ? lw.attn_norm : stage == ST_GATE_UP ? lw.mlp_norm : a.final_norm;
#pragma unroll 1
                for (int m = warp; m < M; m += WARPS) {
                    const float* src = first ? a.embed + (size_t)s_tok[m] * d : a.x + (size_t)m * d;
                    float ss = 0.f;
#pragma unroll 1
                    for (int j = 4 * lane; j < d; j += 128) {
                        const float4 v = ldg_fresh(src + j);
                        *reinterpret_cast<float4*>(xs + (size_t)m * d + j) = v;
                        ss += (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
                    }
                    const float inv = 1.0f / sqrtf(warp_sum(ss) / (float)d + a.eps);
#pragma unroll 1
                    for (int j = 4 * lane; j < d; j += 128) {    // (a lane's own values)
                        float4 v = *reinterpret_cast<float4*>(xs + (size_t)m * d + j);
                        const float4 g = __ldg(reinterpret_cast<const float4*>(gain + j));
                        v.x *= inv * g.x; v.y *= inv * g.y; v.z *= inv * g.z; v.w *= inv * g.w;
                        *reinterpret_cast<float4*>(xs + (size_t)m * d + j) = v;
                    }
                }
            }
            first = false;
            __syncthreads();
            TL_STAGED();
            float* kp = a.kv_pool + (size_t)l * 2 * a.kv_half;
#pragma unroll 1
            for (int p = gw; p < n_pairs;) {
#pragma unroll 1
                for (int m0 = 0; m0 < M; m0 += ROWS) {
                    float y[ROWS], z[ROWS];
                    dot_pair(w0, w1, wa, wb, xs + (size_t)m0 * K, K, y, z);
                    float v0 = sum8(y), v1 = sum8(z);
                    const int m = m0 + (lane >> 2);
                    if ((lane & 3) != 0 || m >= M) continue;
                    if (stage == ST_O || stage == ST_DOWN) {
                        float2* x = reinterpret_cast<float2*>(a.x + (size_t)m * d + 2 * p);
                        float2 t = __ldcg(x);
                        t.x += v0; t.y += v1;
                        *x = t;
                    } else if (stage == ST_GATE_UP) {
                        a.act[(size_t)m * a.dff + p] = v0 / (1.0f + expf(-v0)) * v1;
                    } else if (stage == ST_LM) {
                        unsigned long long best = pack_argmax(v0, (uint32_t)(2 * p));
                        if (2 * p + 1 < a.vocab) best = max(best, pack_argmax(v1, (uint32_t)(2 * p + 1)));
                        atomicMax(&s_best[m], best);
                        if (a.logits) {
                            a.logits[(size_t)m * a.vocab + 2 * p] = v0;
                            if (2 * p + 1 < a.vocab) a.logits[(size_t)m * a.vocab + 2 * p + 1] = v1;
                        }
                    } else {
                        const int head = a.by_half.div(p), i = p - head * half, pos = s_pos[m];
                        float* out = a.q + (size_t)m * qd + head * hd;
                        if (pos < 0) {
                            if (head >= a.n_q) continue;
                            v0 = v1 = 0.f;
                        } else if (pos >= a.max_positions) {
                            set_status(a.status, TASC_EINVAL);
                            continue;
                        } else if (head < a.n_q + a.n_kv) {
                            const float2 c = a.rope[(size_t)pos * half + i];
                            const float r0 = v0 * c.x - v1 * c.y, r1 = v1 * c.x + v0 * c.y;
                            v0 = r0; v1 = r1;
                        }
                        if (head >= a.n_q) {
                            const int pslot = (int)((unsigned)pos / (unsigned)a.page_size);
                            int page = -1;
                            if (pslot < a.max_pages) page = a.block_table[(size_t)a.by_R.div(m) * a.max_pages + pslot];
                            if (page < 0 || page >= a.n_pages) { set_status(a.status, TASC_ENOKV); continue; }
                            const bool is_k = head < a.n_q + a.n_kv;
                            out = kp + (is_k ? 0 : a.kv_half) + (((size_t)page * a.n_kv + (head - a.n_q - (is_k ? 0 : a.n_kv))) * a.page_size + pos - pslot * a.page_size) * hd;
                        }
                        out[i] = v0;
                        out[i + half] = v1;
                    }
                }
                p += CTAS * WARPS;
                if (p < n_pairs) {
                    rows_of(p, w0, w1);
                    if (4 * lane < K) { wa = __ldg(reinterpret_cast<const float4*>(w0 + 4 * lane)); wb = __ldg(reinterpret_cast<const float4*>(w1 + 4 * lane)); }
                }
            }
            if (stage == ST_LM) {
                __syncthreads();
#ifdef TASC_TIMELINE
                tl_b = global_ns();
#endif
                for (int m = threadIdx.x; m < M; m += THREADS) atomicMax(&a.argmax[m], s_best[m]);
#ifdef TASC_TIMELINE
                TL_END(45);
#endif
                return;
            }
        } else {
            cluster_wait();
#ifdef TASC_TIMELINE
            TL_END(tl_tag);
#endif
            float* kp = a.kv_pool + (size_t)l * 2 * a.kv_half;
            float* vp = kp + a.kv_half;
            // ---- attention: unit = (token row, query head)
            const int n_units = M * a.n_q, g = a.n_q / a.n_kv, sub = warp / UNIT_WARPS, sw = warp % UNIT_WARPS;
#pragma unroll 1
            for (int u0 = cta; u0 < n_units; u0 += CTAS * (WARPS / UNIT_WARPS)) {
                const int u = u0 + sub * CTAS;
                const int m = u < n_units ? a.by_nq.div(u) : 0, h = u < n_units ? u - m * a.n_q : 0, b = a.by_R.div(m), kvh = h / g;
                const int n_keys = u < n_units ? s_pos[m] + 1 : 0;   // none for a row that is not in use
                const float* q = a.q + (size_t)m * qd + h * hd;
                float acc[NJ], mx = -INFINITY, den = 0.f;
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[j] = 0.f;
#pragma unroll 1
                for (int k0 = sw * KEYS; k0 < n_keys; k0 += UNIT_WARPS * KEYS) {
                    const int key = k0 + (lane >> 2);
                    const int pslot = (int)((unsigned)key / (unsigned)a.page_size);
                    int page = -1;
                    if (key < n_keys && pslot < a.max_pages) page = a.block_table[(size_t)b * a.max_pages + pslot];
                    const bool there = page >= 0 && page < a.n_pages;          // ids outside the pool read as zeros, never as memory
                    const uint32_t row = there ? (uint32_t)((page * a.n_kv + kvh) * a.page_size + key - pslot * a.page_size) : 0u;
                    // the values are on their way while the scores are worked out
                    float v[KEYS][NJ];
#pragma unroll
                    for (int t = 0; t < KEYS; ++t) {
                        const float* vr = vp + (size_t)__shfl_sync(0xFFFFFFFFu, row, 4 * t) * hd + lane;
#pragma unroll
                        for (int j = 0; j < NJ; ++j) v[t][j] = 32 * j + lane < hd ? __ldcg(vr + 32 * j) : 0.f;
                    }
                    float s = 0.f;
                    const float* kr = kp + (size_t)row * hd;
#pragma unroll 4
                    for (int j = 4 * (lane & 3); j < hd; j += 16) {
                        const float4 kv = ldg_fresh(kr + j), qv = ldg_fresh(q + j);
                        s = fmaf(qv.x, kv.x, fmaf(qv.y, kv.y, fmaf(qv.z, kv.z, fmaf(qv.w, kv.w, s))));
                    }
                    s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
                    s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
                    s = key < n_keys ? (there ? s * a.scale : 0.f) : -INFINITY;
                    const float mn = fmaxf(mx, warp_max(s)), al = expf(mx - mn), p = key < n_keys ? expf(s - mn) : 0.f;
                    den = den * al + warp_sum(p);                      // (four times the sum: four lanes to a key)
                    mx = mn;
#pragma unroll
                    for (int j = 0; j < NJ; ++j) acc[j] *= al;
                    const float pv = there ? p : 0.f;
#pragma unroll
                    for (int t = 0; t < KEYS; ++t) {
                        const float pt = __shfl_sync(0xFFFFFFFFu, pv, 4 * t);
#pragma unroll
                        for (int j = 0; j < NJ; ++j) acc[j] = fmaf(pt, v[t][j], acc[j]);
                    }
                }
                float* mine = part + (size_t)warp * (hd + 4);
#pragma unroll
                for (int j = 0; j < NJ; ++j) if (32 * j + lane < hd) mine[32 * j + lane] = acc[j];
                if (lane == 0) { mine[hd] = mx; mine[hd + 1] = 0.25f * den; }
                __syncthreads();
                if (sw == 0 && u < n_units) {
                    const float* p0 = part + (size_t)warp * (hd + 4);
                    float top = -INFINITY, sum = 0.f;
#pragma unroll 1
                    for (int w = 0; w < UNIT_WARPS; ++w) top = fmaxf(top, p0[w * (hd + 4) + hd]);
#pragma unroll 1
                    for (int w = 0; w < UNIT_WARPS; ++w)
                        if (p0[w * (hd + 4) + hd] != -INFINITY) sum += expf(p0[w * (hd + 4) + hd] - top) * p0[w * (hd + 4) + hd + 1];
#pragma unroll 1
                    for (int j = lane; j < hd; j += 32) {
                        float o = 0.f;
#pragma unroll 1
                        for (int w = 0; w < UNIT_WARPS; ++w)
                            if (p0[w * (hd + 4) + hd] != -INFINITY) o += expf(p0[w * (hd + 4) + hd] - top) * p0[w * (hd + 4) + j];
                        a.o[(size_t)m * qd + h * hd + j] = n_keys > 0 ? o / sum : 0.f;
                    }
                }
                __syncthreads();
            }
        }
#ifdef TASC_TIMELINE
        tl_b = global_ns();
        tl_tag = 40 + stage;
#endif
        cluster_arrive();
        if (stage == ST_DOWN) {
            if (++l == a.n_layers) stage = ST_LM;
            else { stage = ST_QKV; lw = a.layers[l]; }
        } else ++stage;
    }
}

size_t smem_bytes(int M, int width, int hd) {
    return ((size_t)((M + ROWS - 1) / ROWS * ROWS) * width + (size_t)WARPS * (hd + 4)) * 4 + (size_t)M * 16 + 16;
}

void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&at)[2], size_t smem) {
    cfg.gridDim = dim3(CTAS, 1, 1);
    cfg.blockDim = dim3(THREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CTAS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // (set up while the draft runs)
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}
// The kernel's attributes are set and the device takes its cluster.
template <int NJ>
bool cluster_available() {
    static std::mutex mu;
    static int known[64] = {0};                                  // 1 yes, 2 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return false; }
    std::lock_guard<std::mutex> lk(mu);
    if (!known[dev]) {
        int n = 0;
        bool ok = cudaFuncSetAttribute(forward_f32_kernel<NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM) == cudaSuccess &&
                  cudaFuncSetAttribute(forward_f32_kernel<NJ>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (ok) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[2];
            cluster_config(cfg, at, MAX_SMEM);
            ok = cudaOccupancyMaxActiveClusters(&n, forward_f32_kernel<NJ>, &cfg) == cudaSuccess && n > 0;
        }
        if (!ok) (void)cudaGetLastError();
        known[dev] = ok ? 1 : 2;
    }
    return known[dev] == 1;
}
template <int NJ>
tasc_status launch_inst(const ForwardF32Args& a, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    cluster_config(cfg, at, smem_bytes(a.M, a.width, a.hd));
    cfg.numAttrs = 2;
    cfg.stream = stream;
    ProfScope ps(K_LAYERS, stream);
    TASC_CUDA_TRY(cudaLaunchKernelEx(&cfg, forward_f32_kernel<NJ>, a));
    return TASC_OK;
}

}  // namespace

bool plan_forward_f32(int M, int d, int n_q, int n_kv, int hd, int dff, int max_ctx, double layer_mb) {
    if (M < 1 || d % 4 || dff % 4 || hd % 4 || hd > MAX_HD) return false;
    if (layer_mb > F32_CLUSTER_LAYER_MB || (long long)M * n_q * max_ctx > F32_CLUSTER_SCORES) return false;
    return smem_bytes(M, std::max({d, n_q * hd, dff}), hd) <= (size_t)MAX_SMEM &&
           (hd <= 32 ? cluster_available<1>() : hd <= 64 ? cluster_available<2>() : hd <= 128 ? cluster_available<4>() : cluster_available<8>());
}

tasc_status launch_forward_f32(ForwardF32Args a, cudaStream_t stream) {
    a.width = std::max({a.d, a.n_q * a.hd, a.dff});
    a.scale = 1.0f / sqrtf((float)a.hd);
    a.by_R = SmallDiv(a.R); a.by_half = SmallDiv(a.hd / 2); a.by_nq = SmallDiv(a.n_q);
    return a.hd <= 32 ? launch_inst<1>(a, stream) : a.hd <= 64 ? launch_inst<2>(a, stream) : a.hd <= 128 ? launch_inst<4>(a, stream) : launch_inst<8>(a, stream);
}

}  // namespace tasc
