// The end of a decoding step and the start of a request, as kernels of the launch chain: verification of the drafts,
// resampling, commit and the embedding of the next window; the state of a new request; the embedding of prompt tokens.
#include "xsm_proj.cuh"

namespace xsm {

constexpr int kTailThreads = 512, kTailWarps = kTailThreads / 32, kEmbedThreads = 256;
constexpr int kTailSmem = 200 * 1024;          // logits rows that the tail keeps in shared memory, at most
enum TailRows : int { kRowsAll = 0, kRowsOne = 1, kRowsNone = 2 };
constexpr int kMaxCand = 64;

__device__ __forceinline__ uint32_t rand24(const RunParams &R, int seq, uint32_t step, uint32_t slot, uint32_t purpose) {
    return philox_word0(step, slot, purpose, 0u, R.key0 ^ (uint32_t)seq, R.key1) >> 8;
}

// ---------------------------------------------------------------------------------------- embedding

// place in the cache of position pos of sequence b, for token row m (one thread)
static __device__ void place_row(const Dev &D, int m, int b, int pos, bool live) {
    RowInfo r;
    r.rp = row_in_page(D, pos);
    r.place = live ? ((long long)__ldcg(D.block_table + (size_t)b * D.max_blocks + page_of(D, pos)) * D.H * D.P + r.rp) * D.dh : -1;
    r.pad_ = 0;
    D.row_info[m] = r;
}

// 16 bytes of a row's embedding `e`, from column c on: master copy, the copy that the first projection reads (times the gain g
// of the first RMSNorm); returns their sum of squares
template <typename WT> static __device__ float embed_chunk(const Dev &D, int m, int Mp, int c, const uint4 &e_raw, const uint4 &g_raw) {
    constexpr int N = 16 / (int)sizeof(WT);
    const int d = D.d;
    const WT *e = reinterpret_cast<const WT *>(&e_raw), *g = reinterpret_cast<const WT *>(&g_raw);
    float v[N], ssq = 0.f;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        v[q] = to_f(e[q]);
        ssq += v[q] * v[q];
    }
#pragma unroll
    for (int q = 0; q < N; q += 4) *reinterpret_cast<float4 *>(D.h + (size_t)m * d + c + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
    if constexpr (sizeof(WT) == 2) {
        __align__(16) bf16 hi[N], lo[N];
#pragma unroll
        for (int q = 0; q < N; ++q) split_bf16(v[q] * to_f(g[q]), hi[q], lo[q]);
        bf16 *x = reinterpret_cast<bf16 *>(D.xa_) + (size_t)(m / kTokenTile) * 2 * Mp * d + plane_off(Mp, m % kTokenTile, c);
        *reinterpret_cast<uint4 *>(x) = *reinterpret_cast<const uint4 *>(hi);
        *reinterpret_cast<uint4 *>(x + kLo) = *reinterpret_cast<const uint4 *>(lo);
    } else {
        *reinterpret_cast<float4 *>(reinterpret_cast<float *>(D.xa_) + (size_t)m * d + c) =
            make_float4(v[0] * to_f(g[0]), v[1] * to_f(g[1]), v[2] * to_f(g[2]), v[3] * to_f(g[3]));
    }
    return ssq;
}
// 16 bytes of the embedding of `tok`, or of the gain of the first RMSNorm
template <typename WT> static __device__ uint4 embedding(const Dev &D, int tok, int c) {
    return __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const WT *>(D.E) + (size_t)min(max(tok, 0), D.V - 1) * D.d + c));
}
template <typename WT> static __device__ uint4 first_gain(const Dev &D, int c) {
    return __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const WT *>(D.gain_first) + c));
}
// the position's cosines and sines (first threads of the block), and the row's sum of squares from the threads' shares
static __device__ void embed_position(const Dev &D, int m, int pos) {
    const int half = D.dh >> 1;
    if ((int)threadIdx.x < half) D.row_cs[(size_t)m * half + threadIdx.x] = __ldg(D.rope_cs + (size_t)pos * half + threadIdx.x);
}
template <int THREADS> static __device__ void embed_sum(const Dev &D, int m, float ssq, float *sh) {
    ssq = warp_sum(ssq);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = ssq;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < THREADS / 32; ++w) s += sh[w];
        D.ss[(size_t)m * kShareLd] = s;      // the only share
    }
}

template <typename WT> __global__ void __launch_bounds__(kEmbedThreads) embed_rows_kernel(const Dev D, int t, int Mp, int pos0, int pos_end) {
    __shared__ float sh[kEmbedThreads / 32];
    chain_wait();
    chain_go();      // (only now: kernels further down may read what earlier chunks wrote before they wait themselves)
    const int b = blockIdx.x / t, j = blockIdx.x - b * t;
    int tok, pos;
    bool live = true;
    if (pos0 >= 0) {
        const int n = D.rp->prompt_len;
        live = pos0 + j < pos_end;
        pos = min(pos0 + j, pos_end);
        tok = pos0 + j < n ? D.prompt[(size_t)b * n + pos0 + j] : 0;
    } else {
        if (__ldcg(D.finished + b)) return;
        pos = __ldcg(D.len + b) + j;
        tok = __ldcg(D.window + b * t + j);
    }
    if (threadIdx.x == 0) place_row(D, blockIdx.x, b, pos, live);
    constexpr int N = 16 / (int)sizeof(WT);
    embed_position(D, blockIdx.x, pos);
    float ssq = 0.f;
    for (int c = threadIdx.x * N; c < D.d; c += kEmbedThreads * N) ssq += embed_chunk<WT>(D, blockIdx.x, Mp, c, embedding<WT>(D, tok, c), first_gain<WT>(D, c));
    embed_sum<kEmbedThreads>(D, blockIdx.x, ssq, sh);
}
cudaError_t launch_embed_rows(const Dev &D, int dtype, int t, int pos0, int pos_end, const ChainLaunch &L) {
    const void *fn = dtype == 1 ? (const void *)embed_rows_kernel<bf16> : (const void *)embed_rows_kernel<float>;
    const int Mp = D.B * t > kTokenTile ? kTokenTile : (D.B * t + 7) / 8 * 8;
    return L.launch(dim3(D.B * t), dim3(kEmbedThreads), 0, 1, fn, D, t, Mp, pos0, pos_end);
}

// ------------------------------------------------------------------------------------ block reductions

static __device__ float block_sum(float v, float *sh) {
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kTailWarps; ++w) s += sh[w];
    return s;
}
static __device__ float block_max(float v, float *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    float s = -INFINITY;
#pragma unroll
    for (int w = 0; w < kTailWarps; ++w) s = fmaxf(s, sh[w]);
    return s;
}
// (logit, token) as one 64-bit key whose unsigned order is the ranking: larger logit first, then smaller token.
// 0 is below every key ("no candidate").  -0.0 ranks with +0.0.
__device__ __forceinline__ uint32_t rank_bits(float z) {
    const uint32_t u = __float_as_uint(z + 0.0f);
    return u ^ ((uint32_t)((int)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ unsigned long long rank_key(uint32_t bits, int idx) {
    return ((unsigned long long)bits << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)idx);
}
__device__ __forceinline__ float key_logit(unsigned long long k) {
    uint32_t u = (uint32_t)(k >> 32);
    u ^= (u & 0x80000000u) ? 0x80000000u : 0xFFFFFFFFu;
    return __uint_as_float(u);
}
__device__ __forceinline__ int key_token(unsigned long long k) { return (int)(0xFFFFFFFFu - (uint32_t)k); }
// largest key over the warp; every lane gets it
__device__ __forceinline__ unsigned long long warp_best(unsigned long long k) {
    const unsigned hi = (unsigned)(k >> 32), m = __reduce_max_sync(0xffffffffu, hi);
    const unsigned l = __reduce_max_sync(0xffffffffu, hi == m ? (unsigned)k : 0u);
    return ((unsigned long long)m << 32) | l;
}

// ------------------------------------------------------------------------------- verify and resample

struct TailShared {
    float red[kTailWarps];
    unsigned long long best[kTailWarps * kMaxCand];      // the warps' ranked candidates
    float cv[kMaxCand], cw[kMaxCand];   // candidates, ranked: logits, sampling weights
    int ci[kMaxCand];
    int accepted[kMaxDraft];            // of the drafts (each CTA writes its own to all)
    int tok;                            // this slot's candidate
    int cand[kMaxDraft], win[kMaxDraft];      // cand: of all slots (each CTA writes its own to all)
    uint32_t r24;                       // this slot's random number
    int count, n_cand;                  // tokens ranked above the draft; tokens that may be among the best
    int old_win[kMaxDraft];
    int state[8];                       // len, n_gen, step_idx, n_blocks; new len, finished
    float tree_p[8];                    // probability tree: this head's best tokens
    int tree_t[8];
    double m[kMaxDraft * 8];            // the tree's tables (slot 1)
    int tk[kMaxDraft * 8];
};
__device__ __forceinline__ void st_cluster(uint32_t addr, int v) { asm volatile("st.shared::cluster.s32 [%0], %1;" :: "r"(addr), "r"(v) : "memory"); }

// acceptance of token x under backbone logits z, block-wide; every thread returns the same answer
static __device__ bool accept_token(const Dev &D, const RunParams &R, const float *z, int x, TailShared &sh) {
    const int V = D.V;
    if (x < 0 || x >= V) return false;
    if (R.verify_mode == 2) {     // p0(x) > delta
        float m = -INFINITY;
        for (int v = threadIdx.x; v < V; v += kTailThreads) m = fmaxf(m, z[v]);
        m = block_max(m, sh.red);
        float sum = 0.f;
        for (int v = threadIdx.x; v < V; v += kTailThreads) sum += expf(z[v] - m);
        sum = block_sum(sum, sh.red);
        return expf(z[x] - m) / sum > R.delta;
    }
    const int ka = R.verify_mode == 0 ? 1 : R.k_accept;
    const uint32_t ux = rank_bits(z[x]);
    int cnt = 0;
#pragma unroll 8
    for (int v = threadIdx.x; v < V; v += kTailThreads) {
        const uint32_t u = rank_bits(z[v]);
        cnt += u > ux || (u == ux && v < x) ? 1 : 0;
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0) atomicAdd(&sh.count, cnt);
    __syncthreads();
    return sh.count < ka;
}

// The k best (logit, token) pairs of z, ranked, left in sh.cv, sh.ci.  Three to sixteen (one for each warp): the k-th largest of the
// warps' maxima bounds the k-th best of all from below; what is not below it, a dozen or two as a rule, is listed and ranked by
// counting.  False: too many are not below it (equal logits).
static __device__ bool best_by_bound(const Dev &D, const float *z, int k, TailShared &sh) {
    const int V = D.V, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t top = 0u;
#pragma unroll 8
    for (int v = threadIdx.x; v < V; v += kTailThreads) top = max(top, rank_bits(z[v]));
    const uint32_t best = __reduce_max_sync(0xffffffffu, top);
    uint32_t *maxima = reinterpret_cast<uint32_t *>(sh.cw);
    if (lane == 0) maxima[warp] = best;
    __syncthreads();
    const uint32_t mine = lane < kTailWarps ? maxima[lane] : 0u;
    int above = 0;
#pragma unroll
    for (int w = 0; w < kTailWarps; ++w) {
        const uint32_t o = maxima[w];
        above += o > mine || (o == mine && w < lane) ? 1 : 0;
    }
    const unsigned at = __ballot_sync(0xffffffffu, lane < kTailWarps && above == k - 1);
    const uint32_t bound = __shfl_sync(0xffffffffu, mine, __ffs(at) - 1);
    if (top >= bound)
        for (int v = threadIdx.x; v < V; v += kTailThreads) {
            const uint32_t u = rank_bits(z[v]);
            if (u >= bound) {
                const int n = atomicAdd(&sh.n_cand, 1);
                if (n < kTailThreads) sh.best[n] = rank_key(u, v);
            }
        }
    __syncthreads();
    const int n = sh.n_cand;
    if (n > kTailThreads) return false;
    if ((int)threadIdx.x < n) {
        const unsigned long long key = sh.best[threadIdx.x];
        int rank = 0;
        for (int i = 0; i < n; ++i) rank += sh.best[i] > key ? 1 : 0;
        if (rank < k) { sh.cv[rank] = key_logit(key); sh.ci[rank] = key_token(key); }
    }
    __syncthreads();
    return true;
}
// Any k: every warp ranks the k best of its share, the first warp merges the lists (a pick is two warp reductions; block-wide picks
// with two barriers each took a microsecond for two).
static __device__ void top_candidates(const Dev &D, const float *z, int k, TailShared &sh) {
    if (k > 2 && k <= kTailWarps && k <= D.V && best_by_bound(D, z, k, sh)) return;
    const int V = D.V, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the two best of this thread's elements below `limit` (its elements come in ascending order: of equal ones the first stays)
    auto scan = [&](unsigned long long limit, unsigned long long &first, unsigned long long &second) {
        const uint32_t ul = (uint32_t)(limit >> 32);
        const int il = key_token(limit);
        uint32_t u1 = 0u, u2 = 0u;
        int i1 = -1, i2 = -1;
#pragma unroll 8
        for (int v = threadIdx.x; v < V; v += kTailThreads) {
            const uint32_t u = rank_bits(z[v]);
            if (u < ul || (u == ul && v > il)) {
                if (u > u1 || i1 < 0) { u2 = u1; i2 = i1; u1 = u; i1 = v; }
                else if (u > u2 || i2 < 0) { u2 = u; i2 = v; }
            }
        }
        first = i1 < 0 ? 0ull : rank_key(u1, i1);
        second = i2 < 0 ? 0ull : rank_key(u2, i2);
    };
    unsigned long long mine, next;
    scan(0xFFFFFFFF00000000ull, mine, next);      // (all are below)
    bool known = true;                   // next is what follows mine
    for (int j = 0; j < k; ++j) {
        const unsigned long long win = warp_best(mine);
        if (lane == 0) sh.best[warp * kMaxCand + j] = win;
        if (win == mine && win != 0ull && j + 1 < k) {      // mine was picked
            if (known) { mine = next; known = false; }
            else { scan(win, mine, next); known = true; }
        }
    }
    __syncthreads();
    if (warp == 0) {
        // lane l reads list l / 2, every second entry from l % 2 on
        const unsigned long long *list = sh.best + (lane >> 1) * kMaxCand;
        int at = lane & 1;
        unsigned long long head = at < k ? list[at] : 0ull;
        for (int j = 0; j < k; ++j) {
            const unsigned long long win = warp_best(head);
            if (lane == 0) { sh.cv[j] = key_logit(win); sh.ci[j] = key_token(win); }
            if (win == head) {
                at += 2;
                head = at < k ? list[at] : 0ull;
            }
        }
    }
    __syncthreads();
}

// one candidate by inverse CDF over the ranked best (thread 0's answer counts)
static __device__ int pick_candidate(const RunParams &R, int k, uint32_t r24, const TailShared &sh) {
    if (R.sample_mode == 0) return sh.ci[0];
    float total = 0.f;
    for (int j = 0; j < k; ++j) total += sh.cw[j];
    const float u = (float)r24 * (1.0f / 16777216.0f);
    float cum = 0.f;
    for (int j = 0; j < k; ++j) {
        cum += sh.cw[j];
        if (cum > u * total) return sh.ci[j];
    }
    return sh.ci[k - 1];
}

// Top-K_s probability tree over the decoding heads (Appendix, Ablation of Sampling Strategies): the leaves are the
// K_s^K paths in lexicographic order of the heads' ranked candidates, a path weighs the product of its tokens'
// full-vocabulary probabilities, paths whose product falls below 1e-5 are pruned, and the first leaf whose cumulative
// weight exceeds u * total is drawn (the last surviving leaf if rounding keeps the sum below; the most probable token of
// every head if no path survives).  m: [K][8] in shared memory.
static __device__ double leaf_weight(int K, int ks, int n_leaves, const double *m, int idx) {
    double w = 1.0;
    int div = n_leaves;
    for (int d = 0; d < K; ++d) {
        div /= ks;
        const int k = idx / div;
        idx -= k * div;
        w *= m[d * 8 + k];
        if (w < 1e-5) return 0.0;
    }
    return w;
}
// One warp; `known`: the leaves' weights, or null.  Returns the leaf's index.
static __device__ int tree_pick(int K, int ks, int n_leaves, const double *m, const double *known, double u) {
    const int lane = threadIdx.x & 31;
    auto weight = [&](int idx) -> double { return idx >= n_leaves ? 0.0 : known != nullptr ? known[idx] : leaf_weight(K, ks, n_leaves, m, idx); };
    double total = 0.0;
    for (int base = 0; base < n_leaves; base += 32) total += weight(base + lane);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    if (!(total > 0.0)) return 0;
    const double target = u * total;
    double cum = 0.0;
    int last = 0;
    for (int base = 0; base < n_leaves; base += 32) {
        const double w = weight(base + lane);
        double c = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double up = __shfl_up_sync(0xffffffffu, c, o);
            if (lane >= o) c += up;
        }
        c += cum;
        const unsigned alive = __ballot_sync(0xffffffffu, w > 0.0), hit = __ballot_sync(0xffffffffu, w > 0.0 && c > target);
        if (hit) return base + __ffs(hit) - 1;
        if (alive) last = base + 31 - __clz(alive);
        cum = __shfl_sync(0xffffffffu, c, 31);
    }
    return last;
}

static __device__ void draw_initial_drafts(const Dev &D, const RunParams &R, int b, int *win) {
    for (int i = 1; i <= D.K; ++i) {
        const unsigned long long m = rand24(R, b, 0u, (uint32_t)i, 1u);
        win[i] = (int)((m * (unsigned long long)D.V) >> 24);
    }
}

// pages for positions < len + K + 1 of sequence b (one thread)
static __device__ void reserve_pages(const Dev &D, int b, int len, int held) {
    const int need = page_of(D, len + D.K1 + D.P - 1);
    int nb = held;
    while (nb < need) {
        const int idx = atomicSub(D.n_free, 1) - 1;
        if (idx < 0 || nb >= D.max_blocks) {
            atomicAdd(D.n_free, 1);
            atomicExch(D.status, XSM_STATUS_CAPACITY);
            break;
        }
        __stcg(D.block_table + (size_t)b * D.max_blocks + nb, __ldcg(D.free_stack + idx));
        ++nb;
    }
    if (nb != held) __stcg(D.n_blocks + b, nb);
}

// Algorithm 1 lines 7-12 for one sequence by a cluster of K + 1 CTAs, one per window row and slot: CTA j < K decides on
// the draft behind row j; with the accept length a known to all, CTA i draws candidate i from row a of the backbone (i = 0)
// or of head i; every CTA works out the commit, CTA 0 writes it down, and CTA i embeds row i of the next window.
// A chain of short steps (copies, scans, two or three cluster barriers of 0.5 us, the embedding's way from memory): every row that
// may become row a is copied to shared memory at once, so that the candidates' scan starts when a is known.  `rows`: all of them,
// or, where they are too many, the two that are needed one after the other, or none.
template <typename WT> __global__ void __launch_bounds__(kTailThreads) tail_kernel(const Dev D, int stage, int rows) {
    extern __shared__ __align__(128) float row_buf[];
    __shared__ TailShared sh;
    __shared__ __align__(8) uint64_t bars[2];                // the row to verify, the candidates' rows
    const int K1 = D.K1, K = D.K, V = D.V, ld = D.ldv, tid = threadIdx.x;
    const int b = blockIdx.x / K1, slot = blockIdx.x - b * K1;
    chain_go();
    const RunParams &R = *D.rp;
    // (the kernel before it fills the SMs, so this one starts when that ends: everything is asked for at once)
    if (K > 0) cluster_arrive_relaxed();      // "this CTA runs": peers may write to its shared memory after cluster_wait
    if (tid == 0) {
        mbar_init(smem_u32(&bars[0]), 1u);
        mbar_init(smem_u32(&bars[1]), 1u);
        mbar_init_fence();
        sh.count = 0;
        sh.n_cand = 0;
    }
    if (tid == 32) sh.state[0] = __ldcg(D.len + b);
    if (tid == 64) sh.state[1] = __ldcg(D.n_gen + b);
    if (tid == 96) sh.state[2] = (int)__ldcg(D.step_idx + b);
    if (tid == 128) sh.state[3] = __ldcg(D.n_blocks + b);
    if (tid == 160) sh.state[4] = __ldcg(D.finished + b);
    if (tid >= 192 && tid < 192 + K1) sh.old_win[tid - 192] = __ldcg(D.window + b * K1 + tid - 192);
    __syncthreads();      // (warps that come to the wait together leave it sooner)
    if (K > 0) cluster_wait();
    chain_wait();
    if (sh.state[4]) {
        if (slot == 0 && tid == 0) __stcg(D.step_n_new + b, 0);
        return;
    }
    trace_mark(D, 1 + 2 * stage);
    const float *verify = D.logits0 + (size_t)(b * K1 + slot) * ld;
    const float *cands = slot == 0 ? D.logits0 + (size_t)b * K1 * ld : D.hlogits + ((size_t)(slot - 1) * D.M + b * K1) * ld;
    const uint32_t row_bytes = (uint32_t)ld * 4u, to_verify = smem_u32(&bars[0]), to_pick = smem_u32(&bars[1]), buf = smem_u32(row_buf);
    auto wait_rows = [&](uint32_t bar) { mbar_wait(bar, 0u, D.mbar_limit, D.status); };
    if (rows == kRowsAll && tid < 32) {
        if (tid == 0) mbar_arrive_expect_tx(to_pick, (uint32_t)K1 * row_bytes);
        __syncwarp();
        if (tid == K1 && slot > 0 && slot < K) {
            mbar_arrive_expect_tx(to_verify, row_bytes);
            bulk_g2s(buf + (uint32_t)K1 * row_bytes, verify, row_bytes, to_verify);
        }
        if (tid < K1) bulk_g2s(buf + (uint32_t)tid * row_bytes, cands + (size_t)tid * ld, row_bytes, to_pick);
    } else if (rows == kRowsOne && tid == 0 && slot < K) {
        mbar_arrive_expect_tx(to_verify, row_bytes);
        bulk_g2s(buf, verify, row_bytes, to_verify);
    }
    if (tid == kTailThreads - 32) sh.r24 = rand24(R, b, (uint32_t)sh.state[2], (uint32_t)slot, 0u);      // (while the rows come)
    // (requested here and looked at in the end: nothing waits for it)
    const int raised = slot == 0 && tid == kTailThreads - 1 ? __ldcg(D.status) : 0;
    int a = 0;
    if (K > 0) {
        if (slot < K) {
            const float *row = verify;
            if (rows != kRowsNone) {
                wait_rows(rows == kRowsAll && slot == 0 ? to_pick : to_verify);
                row = row_buf + (rows == kRowsAll && slot > 0 ? (size_t)K1 * ld : 0);
            }
            const bool ok = accept_token(D, R, row, sh.old_win[slot + 1], sh);
            if (tid < K1) st_cluster(map_rank(smem_u32(&sh.accepted[slot]), (uint32_t)tid), ok ? 1 : 0);
        }
        __syncthreads();
        cluster_arrive();
        cluster_wait();
        const int lane = tid & 31;
        const unsigned no = __ballot_sync(0xffffffffu, lane < K && sh.accepted[min(lane, K - 1)] == 0);
        a = no ? __ffs(no) - 1 : K;
    }
    // candidate of this slot
    const float *z = cands + (size_t)a * ld;
    if (rows == kRowsAll) {
        wait_rows(to_pick);
        z = row_buf + (size_t)a * ld;
    } else if (rows == kRowsOne) {
        // (every thread has read the row that was verified; slot 0 has row 0 already)
        if (!(slot == 0 && a == 0 && K > 0)) {
            if (tid == 0) {
                mbar_arrive_expect_tx(to_pick, row_bytes);
                bulk_g2s(buf, z, row_bytes, to_pick);
            }
            wait_rows(to_pick);
        }
        z = row_buf;
    }
    const bool tree = R.sample_mode == 2 && slot > 0;
    const int k = tree ? min(max(R.k_sample, 1), min(V, 8)) : R.sample_mode == 0 ? 1 : min(max(R.k_sample, 1), min(V, kMaxCand));
    top_candidates(D, z, k, sh);
    if (!tree) {
        if (R.sample_mode != 0) {
            if (tid < k) sh.cw[tid] = expf((sh.cv[tid] - sh.cv[0]) / R.temperature);
            __syncthreads();
        }
        if (tid == 0) sh.tok = pick_candidate(R, k, sh.r24, sh);
    } else {
        // probability tree: this head's K_s best tokens and their probabilities, for slot 1, which draws one path for all heads
        const float mx = sh.cv[0];
        float sum = 0.f;
        for (int v = tid; v < V; v += kTailThreads) sum += expf(z[v] - mx);
        sum = block_sum(sum, sh.red);
        if (tid < k) {
            sh.tree_t[tid] = sh.ci[tid];
            sh.tree_p[tid] = expf(sh.cv[tid] - mx) / sum;
        }
    }
    if (R.sample_mode == 2 && K > 0) {
        __syncthreads();
        cluster_arrive();
        cluster_wait();
        if (slot == 1) {
            const int ks = k;
            for (int i = tid; i < K * ks; i += kTailThreads) {
                const int d = i / ks, j = i - d * ks;
                sh.m[d * 8 + j] = (double)ld_cluster_f32(map_rank(smem_u32(&sh.tree_p[j]), (uint32_t)(d + 1)));
                asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(sh.tk[d * 8 + j]) : "r"(map_rank(smem_u32(&sh.tree_t[j]), (uint32_t)(d + 1))) : "memory");
            }
            int n_leaves = 1;
            for (int d = 0; d < K; ++d) n_leaves *= ks;
            __syncthreads();
            // (the rows' place is free: the leaves' weights, by all threads)
            double *known = rows != kRowsNone && (size_t)n_leaves * 8 <= (size_t)row_bytes ? reinterpret_cast<double *>(row_buf) : nullptr;
            if (known != nullptr) {
                for (int i = tid; i < n_leaves; i += kTailThreads) known[i] = leaf_weight(K, ks, n_leaves, sh.m, i);
                __syncthreads();
            }
            if (tid < 32) {
                const double u = (double)sh.r24 * (1.0 / 16777216.0);
                int leaf = tree_pick(K, ks, n_leaves, sh.m, known, u), div = n_leaves;
                for (int d = 0; d < K; ++d) {
                    div /= ks;
                    const int kk = leaf / div;
                    leaf -= kk * div;
                    if (tid < K1) st_cluster(map_rank(smem_u32(&sh.cand[d + 1]), (uint32_t)tid), sh.tk[d * 8 + kk]);
                }
            }
        }
    }
    __syncthreads();
    if (K > 0) {
        if (tid < K1 && (R.sample_mode != 2 || slot == 0)) st_cluster(map_rank(smem_u32(&sh.cand[slot]), (uint32_t)tid), sh.tok);
        cluster_arrive();
        cluster_wait();
    } else {
        if (tid == 0) sh.cand[0] = sh.tok;
        __syncthreads();
    }
    // (the embedding is on its way while the commit is worked out, which changes it only where drafts are scripted)
    constexpr int N = 16 / (int)sizeof(WT);
    static_assert(kTailThreads * 4 >= 2048, "a thread embeds 16 bytes at most");
    const int col = tid * N, guess = sh.cand[slot];
    uint4 e_raw, g_raw;
    if (col < D.d) {
        e_raw = embedding<WT>(D, guess, col);
        g_raw = first_gain<WT>(D, col);
    }
    // commit x_{s+1..s*}, s <- s*, next window <- candidates: worked out by every CTA, written by CTA 0 (one warp, a lane a token)
    if (tid < 32) {
        const bool w = slot == 0;
        const int len = sh.state[0] + a + 1, n_gen = sh.state[1];
        // scripted drafts: the token at the first rejected position is the script's as well, so that a near-tie
        // of the backbone's two best logits cannot take the run off the script for good
        const int first = R.script != nullptr && len < R.script_n ? R.script[(size_t)b * R.script_n + len] : sh.cand[0];
        const int tok = tid < a ? sh.old_win[min(tid + 1, K)] : first;
        int n_out = max(0, min(a + 1, R.max_new - n_gen));
        const unsigned ends = __ballot_sync(0xffffffffu, D.eos >= 0 && tid < n_out && tok == D.eos);
        if (ends) n_out = __ffs(ends);
        const int fin = ends != 0u || n_gen + n_out >= R.max_new || len > D.max_seq_len ? 1 : 0;
        int next = tid == 0 ? first : tid < K1 ? sh.cand[tid] : 0;
        if (R.script != nullptr && tid > 0 && tid < K1) {
            // scripted drafts: the next window drafts the script's tokens; the first `keep` stay as they
            // are, the others are made wrong (a forced accept length for a backbone that reproduces the script)
            const long long t = (long long)sh.state[2] + 1;
            const int keep = (int)((((t + 1) * R.script_acc) >> 10) - ((t * R.script_acc) >> 10)), pos = len + tid;
            next = pos < R.script_n ? R.script[(size_t)b * R.script_n + pos] : 0;
            if (tid > keep) next = next + 1 < D.V ? next + 1 : 0;
        }
        if (tid < K1) sh.win[tid] = next;
        if (tid == 0) sh.state[5] = fin;
        if (w) {
            if (tid < n_out) __stcg(D.tok_log + (size_t)b * D.tok_ld + n_gen + tid, tok);
            if (tid < K1) {
                __stcg(D.step_tokens + b * K1 + tid, tid < n_out ? tok : -1);
                __stcg(D.window + b * K1 + tid, next);
            }
            if (tid == 0) {
                __stcg(D.step_n_new + b, n_out);
                __stcg(D.n_gen + b, n_gen + n_out);
                __stcg(D.step_idx + b, (uint32_t)sh.state[2] + 1u);
                D.hist[(size_t)b * (kMaxDraft + 1) + a] += 1ull;
                D.steps[b] += 1ull;
                __stcg(D.len + b, len);
                if (!fin) reserve_pages(D, b, len, sh.state[3]);
            }
            if (fin) {
                __threadfence_system();      // (every lane's tokens are out before the host is told)
                __syncwarp();
                if (tid == 0) {
                    __stcg(D.finished + b, 1);
                    if (atomicSub(D.n_active, 1) == 1) {      // the last one: tell the host that its call is done
                        __threadfence_system();
                        *reinterpret_cast<volatile int *>(D.host_done) = R.call;
                    }
                }
            }
        }
    }
    __syncthreads();
    const int new_len = sh.state[0] + a + 1;
    if (slot == 0 && tid >= kTailThreads - 32 && tid - (kTailThreads - 32) < K1)      // (the last warp: the embedding needs the first ones)
        place_row(D, b * K1 + tid - (kTailThreads - 32), b, new_len + tid - (kTailThreads - 32), !sh.state[5]);
    if (!sh.state[5]) {
        embed_position(D, b * K1 + slot, new_len + slot);
        float ssq = 0.f;
        if (col < D.d) {
            if (sh.win[slot] != guess) e_raw = embedding<WT>(D, sh.win[slot], col);
            ssq = embed_chunk<WT>(D, b * K1 + slot, D.Mp, col, e_raw, g_raw);
        }
        embed_sum<kTailThreads>(D, b * K1 + slot, ssq, sh.red);
    }
    // a wait of this request ran out, or its pages: more steps are of no use (the host reads the status word itself)
    if (raised != 0) *reinterpret_cast<volatile int *>(D.host_done) = R.call;
    trace_mark(D, 2 + 2 * stage);
}

cudaError_t launch_tail(const Dev &D, int dtype, int stage, const ChainLaunch &L) {
    const void *fn = dtype == 1 ? (const void *)tail_kernel<bf16> : (const void *)tail_kernel<float>;
    // All rows, where two CTAs' share an SM or there is one for every CTA: a cluster more would be a second wave.
    const size_t row = (size_t)D.ldv * 4, all = row * (D.K > 0 ? D.K1 + 1 : 1);
    const bool fits = all <= kTailSmem / 2 || (all <= kTailSmem && (D.K == 0 || (D.K1 <= 8 && D.B <= resident_clusters(D.K1))));
    const int rows = fits ? kRowsAll : row <= kTailSmem ? kRowsOne : kRowsNone, smem = fits ? (int)all : row <= kTailSmem ? (int)row : 16;
    cudaError_t e = open_kernel(fn, smem, D.K1 > 8);
    if (e != cudaSuccess) return e;
    return L.launch(dim3(D.B * D.K1), dim3(kTailThreads), smem, D.K1, fn, D, stage, rows);
}

// --------------------------------------------------------------------------------- start of a request

// Algorithm 1 line 1: the pool, the run's parameters, and per sequence s = prompt_len - 1, its pages, the first window.
__global__ void begin_pool_kernel(const Dev D, const RunParams R) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < D.n_pages) D.free_stack[i] = D.n_pages - 1 - i;
    if (i == 0) { *D.n_free = D.n_pages; *D.n_active = D.B; *D.status = 0; *D.stage_word = 0; *D.rp = R; }
}
__global__ void begin_seq_kernel(const Dev D) {
    const int b = blockIdx.x;
    const RunParams &R = *D.rp;
    const int len = R.prompt_len - 1;
    if (threadIdx.x <= kMaxDraft) D.hist[(size_t)b * (kMaxDraft + 1) + threadIdx.x] = 0ull;
    if (threadIdx.x == 0) {
        int win[kMaxDraft];
        D.len[b] = len; D.finished[b] = 0; D.n_gen[b] = 0; D.n_blocks[b] = 0; D.step_idx[b] = 0u;
        D.steps[b] = 0ull; D.step_n_new[b] = 0;
        win[0] = D.prompt[(size_t)b * R.prompt_len + len];
        draw_initial_drafts(D, R, b, win);
        for (int j = 0; j < D.K1; ++j) D.window[b * D.K1 + j] = win[j];
        reserve_pages(D, b, len, 0);
    }
}
cudaError_t launch_begin(const Dev &D, const RunParams &R, cudaStream_t st) {
    begin_pool_kernel<<<(D.n_pages + 255) / 256, 256, 0, st>>>(D, R);
    begin_seq_kernel<<<D.B, 32, 0, st>>>(D);
    return cudaGetLastError();
}
// bounded: after D.spin_limit polls the status word is raised
__global__ void stage_gate_kernel(const Dev D, int stage) {
    for (unsigned n = 0; n < D.spin_limit; ++n)
        if (__ldcg(D.stage_word) == stage) return;
    atomicExch(D.status, XSM_STATUS_TIMEOUT);
}
__global__ void stage_mark_kernel(const Dev D, int done) { *D.stage_word = done; }
cudaError_t launch_stage_gate(const Dev &D, int stage, cudaStream_t st) {
    stage_gate_kernel<<<1, 1, 0, st>>>(D, stage);
    return cudaGetLastError();
}
cudaError_t launch_stage_mark(const Dev &D, int done, cudaStream_t st) {
    stage_mark_kernel<<<1, 1, 0, st>>>(D, done);
    return cudaGetLastError();
}
// The token limit of the steps that follow and the call that they are for, which is told at once if it needs none.
__global__ void set_limit_kernel(const Dev D, int max_new, int call) {
    D.rp->max_new = max_new;
    D.rp->call = call;
    if (*D.n_active == 0 || *D.status != 0) *reinterpret_cast<volatile int *>(D.host_done) = call;
}
cudaError_t launch_set_limit(const Dev &D, int max_new, int call, cudaStream_t st) {
    set_limit_kernel<<<1, 1, 0, st>>>(D, max_new, call);
    return cudaGetLastError();
}
__global__ void set_script_kernel(const Dev D, const int *script, int n, int acc) {
    D.rp->script = script;
    D.rp->script_n = n;
    D.rp->script_acc = acc;
}
cudaError_t launch_set_script(const Dev &D, const int *script, int n, int acc, cudaStream_t st) {
    set_script_kernel<<<1, 1, 0, st>>>(D, script, n, acc);
    return cudaGetLastError();
}

}  // namespace xsm
