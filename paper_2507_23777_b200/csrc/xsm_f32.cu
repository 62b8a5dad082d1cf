// The kernels of the launch chain for fp32 models (the parity configuration: at most kF32Rows token rows, plain FMA).
// Activations are [token row][column] floats; the cache holds fp32 tiles.
#include "xsm_proj.cuh"

namespace xsm {

constexpr int kF32Warps = 8, kF32Threads = kF32Warps * 32;

// Folds N values of every lane over the warp (lanes that differ in bits of at least `last`): each exchange halves the values
// that a lane keeps, so N values cost N - 1 + a few shuffles of 38 cycles instead of 5 N.  Lane l gets value l / (32 / N); the
// order of a sum is that of warp_sum.
template <int N, typename Op> __device__ __forceinline__ float fold(float (&v)[N], Op op, int last) {
    const int lane = threadIdx.x & 31;
    int k = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n /= 2, k /= 2) {
        const bool up = lane & k;
#pragma unroll
        for (int i = 0; i < N / 2; ++i)
            if (i < n) {
                const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
                v[i] = op(keep, __shfl_xor_sync(0xffffffffu, send, k));
            }
    }
    for (; k >= last; k /= 2) v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], k));
    return v[0];
}
struct Add { __device__ __forceinline__ float operator()(float a, float b) const { return a + b; } };
struct Max { __device__ __forceinline__ float operator()(float a, float b) const { return fmaxf(a, b); } };

// ------------------------------------------------------------------------------------ projections

// A warp owns units (a row, or a pair of rows: rotation partners, gate and up), its lanes the columns.  The weights of the
// first unit are in registers before the wait; the activations are staged in shared memory, a chunk of columns at a time.
// MT: token rows that a warp accumulates (at least A.rows).
template <int MT, int EPI0, int EPI1>
__global__ void __launch_bounds__(kF32Threads) proj_f32_kernel(const Dev D, const ProjArgs A) {
    extern __shared__ __align__(16) float xs[];       // [rows][chunk]
    __shared__ float s_inv[MT];
    constexpr bool PAIRS = EPI0 == PE_QKV || EPI0 == PE_GATEUP;
    constexpr int R = PAIRS ? 2 : 1, AHEAD = PAIRS ? 4 : 8;       // rows of a unit; quads of columns fetched before the wait
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (A.pos0 < 0 && !A.late_go && __ldcg(D.n_active) == 0) {      // every sequence has ended in an earlier step
        chain_wait();
        return;
    }
    if (!A.late_go) chain_go();
    const int job = A.x_jobs ? blockIdx.x / A.ctas : 0, cta = A.x_jobs ? blockIdx.x - job * A.ctas : blockIdx.x;
    const int units = EPI0 == PE_QKV ? A.g[0].units >> 1 : A.g[0].units + (EPI1 >= 0 ? A.g[1].units * A.g[1].jobs : 0);
    const int K = A.kdim, M = A.rows, half = D.dh >> 1, chunk = A.chunk;
    // weight row r (0, 1) of a unit; u and j become its place in its group
    auto weights = [&](int unit, int r, int &u, int &j, bool &second) -> const float * {
        u = unit; j = job; second = false;
        if (EPI0 == PE_QKV) {
            const int hd = D.d >> 1, sec = unit / hd, i = unit - sec * hd, head = i / half;
            u = sec * D.d + head * D.dh + (i - head * half);
            return reinterpret_cast<const float *>(A.g[0].w) + (size_t)(u + r * half) * K;
        }
        if (EPI0 == PE_GATEUP) return reinterpret_cast<const float *>(A.g[r].w) + (size_t)unit * K;
        if (EPI1 >= 0 && u >= A.g[0].units) {
            u -= A.g[0].units;
            j = u / A.g[1].units;
            u -= j * A.g[1].units;
            second = true;
            return reinterpret_cast<const float *>(A.g[1].w) + (size_t)j * A.g[1].w_stride + (size_t)u * K;
        }
        return reinterpret_cast<const float *>(A.g[0].w) + (size_t)job * A.g[0].w_stride + (size_t)u * K;
    };
    const int first = cta * kF32Warps + warp, step = A.ctas * kF32Warps;
    int u, j;
    bool second;
    const float *w[R];
    float4 wa[R][AHEAD];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        w[r] = weights(min(first, units - 1), r, u, j, second);
#pragma unroll
        for (int q = 0; q < AHEAD; ++q)
            if (q * 128 + lane * 4 < min(chunk, K)) wa[r][q] = __ldg(reinterpret_cast<const float4 *>(w[r] + q * 128 + lane * 4));
    }
    if (A.stage == 0) trace_mark(D, 0);
    __syncthreads();      // (warps that come to the wait together leave it sooner)
    chain_wait();
    if (A.late_go) chain_go();
    trace_mark(D, 1 + 2 * A.stage);
    const float *x = reinterpret_cast<const float *>(A.x) + (A.x_jobs ? (size_t)job * M * K : 0);
    auto stage = [&](int k0) {      // columns [k0, k0 + chunk) of all token rows
        const int n4 = min(chunk, K - k0) >> 2;
        __syncthreads();
        for (int i = tid; i < M * n4; i += kF32Threads) {
            const int m = i / n4, c = i - m * n4;
            reinterpret_cast<float4 *>(xs + m * chunk)[c] = __ldcg(reinterpret_cast<const float4 *>(x + (size_t)m * K + k0) + c);
        }
        __syncthreads();
    };
    // 1/rms of the token rows (their shares are requested before the activations, and added up behind them)
    constexpr int SHARES = (kShareLd + 31) / 32, MINE = (MT + kF32Warps - 1) / kF32Warps;
    float share[MINE][SHARES];
#pragma unroll
    for (int i = 0; i < MINE; ++i)
#pragma unroll
        for (int p = 0; p < SHARES; ++p) {
            const int m = warp + i * kF32Warps;
            share[i][p] = m < M && p * 32 + lane < A.ss_parts ? __ldcg(D.ss + (size_t)m * kShareLd + p * 32 + lane) : 0.f;
        }
    if (chunk >= K) {
        const int n4 = K >> 2;
        for (int i = tid; i < M * n4; i += kF32Threads) {
            const int m = i / n4, c = i - m * n4;
            reinterpret_cast<float4 *>(xs + m * chunk)[c] = __ldcg(reinterpret_cast<const float4 *>(x + (size_t)m * K) + c);
        }
    }
    if (A.ss_parts > 0) {
#pragma unroll
        for (int i = 0; i < MINE; ++i) {
            if (warp + i * kF32Warps >= M) break;
            float ss = 0.f;
#pragma unroll
            for (int p = 0; p < SHARES; ++p) ss += share[i][p];
            ss = warp_sum(ss);
            if (lane == 0) s_inv[warp + i * kF32Warps] = 1.0f / sqrtf(ss / (float)D.d + D.eps);
        }
    }
    __syncthreads();
    constexpr int ROWS = MT < 8 ? MT : 8, WIDTH = 32 / (ROWS * R);      // token rows folded at a time, lanes that share a value
    float ssq_mine[MT / ROWS];      // PE_ADD: the squares of a lane's token rows over the warp's units
#pragma unroll
    for (int c = 0; c < MT / ROWS; ++c) ssq_mine[c] = 0.f;
    for (int base = cta * kF32Warps; base < units; base += step) {      // (all warps of the CTA together: they share the staged columns)
        const int unit = base + warp;
        float acc[R][MT];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int m = 0; m < MT; ++m) acc[r][m] = 0.f;
        const bool mine = unit < units;
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = weights(min(unit, units - 1), r, u, j, second);
        for (int k0 = 0; k0 < K; k0 += chunk) {
            if (chunk < K) stage(k0);
            if (!mine) continue;
            const int n = min(chunk, K - k0);
            auto columns = [&](int c, const float4 (&wv)[R]) {
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    if (m < M) {
                        const float4 xv = *reinterpret_cast<const float4 *>(xs + m * chunk + c);
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            acc[r][m] = fmaf(wv[r].x, xv.x, fmaf(wv[r].y, xv.y, fmaf(wv[r].z, xv.z, fmaf(wv[r].w, xv.w, acc[r][m]))));
                    }
                }
            };
            int q0 = 0;
            if (unit == first && k0 == 0) {
#pragma unroll
                for (int q = 0; q < AHEAD; ++q) {
                    float4 wv[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) wv[r] = wa[r][q];
                    if (q * 128 + lane * 4 < n) columns(q * 128 + lane * 4, wv);
                }
                q0 = AHEAD;
            }
            for (int c = q0 * 128 + lane * 4; c < n; c += 128) {
                float4 wv[R];
#pragma unroll
                for (int r = 0; r < R; ++r) wv[r] = __ldg(reinterpret_cast<const float4 *>(w[r] + k0 + c));
                columns(c, wv);
            }
        }
        if (!mine) continue;
        // sums over the lanes, ROWS token rows (both rows of a pair) at a time
#pragma unroll
        for (int ch = 0; ch < MT / ROWS; ++ch) {
        if (ch * ROWS >= M) break;
        float part[ROWS * R];
#pragma unroll
        for (int i = 0; i < ROWS; ++i)
#pragma unroll
            for (int r = 0; r < R; ++r) part[i * R + r] = acc[r][ch * ROWS + i];
        float v = fold(part, Add(), 1), v2 = PAIRS ? __shfl_xor_sync(0xffffffffu, v, WIDTH) : 0.f;
        const int m = ch * ROWS + lane / (WIDTH * R);
        if (lane % (WIDTH * R) != 0 || m >= M) continue;
        const float inv = A.ss_parts > 0 ? s_inv[m] : 1.f;
        if (EPI0 == PE_ADD) {
            const float h = __ldcg(D.h + (size_t)m * D.d + u) + v;
            D.h[(size_t)m * D.d + u] = h;
            reinterpret_cast<float *>(A.g[0].out)[(size_t)m * A.g[0].ld + u] = h * __ldg(reinterpret_cast<const float *>(A.gain) + u);
            ssq_mine[ch] += h * h;
        } else if (EPI0 == PE_QKV) {
            v *= inv;
            v2 *= inv;
            const int sec = u >= D.d ? (u >= 2 * D.d ? 2 : 1) : 0, c = u - sec * D.d, head = c / D.dh, e = c - head * D.dh;
            const float2 cs = __ldcg(D.row_cs + (size_t)m * half + e);
            const long long place = __ldcg(reinterpret_cast<const long long *>(D.row_info + m));
            const float o1 = sec < 2 ? v * cs.x - v2 * cs.y : v, o2 = sec < 2 ? v2 * cs.x + v * cs.y : v2;
            if (sec == 0) {
                float *q = reinterpret_cast<float *>(A.q) + (size_t)m * D.d + c;
                q[0] = o1 * A.scale;
                q[half] = o2 * A.scale;
            } else if (place >= 0) {
                float *tile = kv_tile<float>(D, D.kv_pool, D.n_pages, A.layer, sec - 1, 0, head) + place + e;
                tile[0] = o1;
                tile[half] = o2;
            }
        } else if (EPI0 == PE_GATEUP) {
            reinterpret_cast<float *>(A.g[0].out)[(size_t)m * A.g[0].ld + u] = silu_f(v * inv) * (v2 * inv);
        } else if (EPI0 == PE_QUERY || (EPI1 == PE_QUERY && second)) {
            reinterpret_cast<float *>(A.q)[((size_t)j * M + m) * D.d + u] = v * inv * A.scale;
        } else if (EPI0 == PE_HEADADD || (EPI1 == PE_HEADY && second)) {
            const float g = __ldcg(D.h + (size_t)m * D.d + u) * inv * __ldg(reinterpret_cast<const float *>(A.gain) + u);
            const ProjGroup &G = A.g[EPI1 >= 0 ? 1 : 0];
            reinterpret_cast<float *>(G.out)[((size_t)j * M + m) * G.ld + u] = g + (EPI0 == PE_HEADADD ? v : silu_f(v * inv));
        } else {
            A.g[0].logits[((size_t)j * D.M + m) * A.g[0].ld + u] = A.norm ? v * inv : v;
        }
        }
    }
    if (EPI0 == PE_ADD) {
        // the CTA's shares of the sums of squares
        __syncthreads();
#pragma unroll
        for (int ch = 0; ch < MT / ROWS; ++ch)
            if (lane % WIDTH == 0) xs[warp * MT + ch * ROWS + lane / WIDTH] = ssq_mine[ch];
        __syncthreads();
        if (tid < M) {
            float s = 0.f;
            for (int q = 0; q < kF32Warps; ++q) s += xs[q * MT + tid];
            D.ss[(size_t)tid * kShareLd + cta] = s;
        }
    }
    trace_mark(D, 2 + 2 * A.stage);
}

// -------------------------------------------------------------------------------------- attention

// One CTA per (sequence, head): 128 keys and values at a time in shared memory (those that the step does not write are
// fetched before the wait), two threads score a key against all t rows, then the threads sum the values of a column each,
// a share of the keys each, and the shares are added in order.
constexpr int kF32Keys = kF32Threads / 2;
template <int T>
__global__ void __launch_bounds__(kF32Threads) attn_f32_kernel(const Dev D, const AttnArgs A) {
    extern __shared__ __align__(16) float sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, dh = D.dh, ld = dh + 4;
    const int h = blockIdx.y, b = blockIdx.z % D.B, set = blockIdx.z / D.B;
    const bool cross = A.cross != 0;
    float *ks = sm, *vs = ks + kF32Keys * ld, *qs = vs + kF32Keys * ld;
    float *p = qs + T * dh, *o = p + T * kF32Threads, *red = o + T * dh;      // weights [T][keys] (then shares), output, per-warp values
    float *m_run = red + kF32Warps * T, *l_run = m_run + T, *f_run = l_run + T;
    chain_go();
    const bool dead = A.pos0 < 0 && __ldcg(D.finished + b) != 0;
    const int start = cross ? 0 : A.pos0 >= 0 ? A.pos0 : __ldcg(D.len + b);      // (the state was written by an earlier step)
    const int n_keys = cross ? D.C : A.pos0 >= 0 ? min(start + A.t, A.pos_end) : start + A.t, n_old = cross ? D.C : start;
    auto fetch = [&](int k0, int lo, int hi) {      // keys and values [lo, hi) into the places of the chunk at k0
        const int c4 = dh >> 2, n = (hi - lo) * c4;
        for (int i = tid; i < n; i += kF32Threads) {
            const int kk = i / c4, c = i - kk * c4, key = lo + kk, pg = page_of(D, key);
            const int page = cross ? b * D.cpages + pg : __ldcg(D.block_table + (size_t)b * D.max_blocks + pg);
            const int pages = cross ? D.B * D.cpages : D.n_pages, lay = cross && A.sets > 1 ? set : A.layer;
            const size_t off = (size_t)row_in_page(D, key) * dh + 4 * c;
            const float4 kv = __ldcg(reinterpret_cast<const float4 *>(kv_tile<float>(D, const_cast<void *>(A.pool), pages, lay, 0, page, h) + off));
            const float4 vv = __ldcg(reinterpret_cast<const float4 *>(kv_tile<float>(D, const_cast<void *>(A.pool), pages, lay, 1, page, h) + off));
            *reinterpret_cast<float4 *>(ks + (key - k0) * ld + 4 * c) = kv;
            *reinterpret_cast<float4 *>(vs + (key - k0) * ld + 4 * c) = vv;
        }
    };
    if (!dead) fetch(0, 0, min(kF32Keys, n_old));
    __syncthreads();
    chain_wait();
    if (dead) return;
    trace_mark(D, 1 + 2 * A.stage);
    const float *q = reinterpret_cast<const float *>(A.q) + ((size_t)set * A.rows + (size_t)b * A.t) * D.d + h * dh;
    for (int i = tid; i < T * dh; i += kF32Threads) {
        const int r = i / dh;
        qs[i] = r < A.t ? __ldcg(q + (size_t)r * D.d + i - r * dh) : 0.f;
        o[i] = 0.f;
    }
    if (tid < T) { m_run[tid] = kNegBig; l_run[tid] = 0.f; }
    for (int k0 = 0; k0 < n_keys; k0 += kF32Keys) {
        const int n = min(kF32Keys, n_keys - k0), key = k0 + (tid >> 1), part = tid & 1;
        fetch(k0, k0 == 0 ? min(kF32Keys, n_old) : k0, k0 + n);
        __syncthreads();
        float s[T];
#pragma unroll
        for (int r = 0; r < T; ++r) s[r] = 0.f;
        if (key < n_keys) {
            const float *kr = ks + (tid >> 1) * ld + part * (dh >> 1), *qr = qs + part * (dh >> 1);
#pragma unroll 4
            for (int c = 0; c < (dh >> 1); c += 4) {
                const float4 kv = *reinterpret_cast<const float4 *>(kr + c);
#pragma unroll
                for (int r = 0; r < T; ++r) {
                    const float4 qv = *reinterpret_cast<const float4 *>(qr + r * dh + c);
                    s[r] = fmaf(kv.x, qv.x, fmaf(kv.y, qv.y, fmaf(kv.z, qv.z, fmaf(kv.w, qv.w, s[r]))));
                }
            }
        }
        // running maximum of every row, weights relative to it
        constexpr int ROWS = T < 8 ? T : 8;
#pragma unroll
        for (int r = 0; r < T; ++r) {
            s[r] += __shfl_xor_sync(0xffffffffu, s[r], 1);
            if (key >= n_keys || (!cross && key > start + r)) s[r] = -INFINITY;
        }
#pragma unroll
        for (int r0 = 0; r0 < T; r0 += ROWS) {
            float v[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) v[r] = s[r0 + r];
            const float m = fold(v, Max(), 2);
            if (lane % (32 / ROWS) == 0) red[warp * T + r0 + lane / (32 / ROWS)] = m;
        }
        __syncthreads();
        if (tid < T) {
            float m = m_run[tid];
            for (int w = 0; w < kF32Warps; ++w) m = fmaxf(m, red[w * T + tid]);
            f_run[tid] = exp2f(m_run[tid] - m);
            m_run[tid] = m;
        }
        __syncthreads();
#pragma unroll
        for (int r0 = 0; r0 < T; r0 += ROWS) {
            float v[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const float e = exp2f(s[r0 + r] - m_run[r0 + r]);
                if (part == 0) p[(r0 + r) * kF32Keys + (tid >> 1)] = e;
                v[r] = part == 0 ? e : 0.f;
            }
            const float l = fold(v, Add(), 1);
            if (lane % (32 / ROWS) == 0) red[warp * T + r0 + lane / (32 / ROWS)] = l;
        }
        __syncthreads();
        if (tid < T) {
            float l = l_run[tid] * f_run[tid];
            for (int w = 0; w < kF32Warps; ++w) l += red[w * T + tid];
            l_run[tid] = l;
        }
        // values: column c, keys share, share + shares, ...; every share its own place, added in order
        const int shares = kF32Threads / dh, c = tid % dh, share = tid / dh;
        float acc[T];
#pragma unroll
        for (int r = 0; r < T; ++r) acc[r] = 0.f;
#pragma unroll 4
        for (int k = share; k < n; k += shares) {
            const float v = vs[k * ld + c];
#pragma unroll
            for (int r = 0; r < T; ++r) acc[r] = fmaf(p[r * kF32Keys + k], v, acc[r]);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < T; ++r) p[r * kF32Threads + tid] = acc[r];
        __syncthreads();
        for (int i = tid; i < T * dh; i += kF32Threads) {
            const int r = i / dh, cc = i - r * dh;
            float v = o[i] * f_run[r];
            for (int k = 0; k < shares; ++k) v += p[r * kF32Threads + k * dh + cc];
            o[i] = v;
        }
    }
    __syncthreads();
    float *out = reinterpret_cast<float *>(A.out) + ((size_t)set * A.rows + (size_t)b * A.t) * D.d + h * dh;
    for (int i = tid; i < A.t * dh; i += kF32Threads) {
        const int r = i / dh;
        out[(size_t)r * D.d + i - r * dh] = o[i] / l_run[r];
    }
    trace_mark(D, 2 + 2 * A.stage);
}

// ---------------------------------------------------------------------------------------- launches

template <int MT, int EPI0, int EPI1>
static cudaError_t launch_proj_instance(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) {
    void (*fn)(const Dev, const ProjArgs) = proj_f32_kernel<MT, EPI0, EPI1>;
    cudaError_t e = open_kernel((const void *)fn, smem, false);
    if (e != cudaSuccess) return e;
    return L.launch(dim3(A.x_jobs ? A.ctas * A.g[0].jobs : A.ctas), dim3(kF32Threads), smem, 1, (const void *)fn, D, A);
}
template <int MT>
static cudaError_t launch_proj_rows(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) {
#define XSM_EPI(a, b) if (A.epi0 == a && A.epi1 == b) return launch_proj_instance<MT, a, b>(D, A, smem, L)
    XSM_EPI(PE_QKV, -1);
    XSM_EPI(PE_ADD, -1);
    XSM_EPI(PE_QUERY, -1);
    XSM_EPI(PE_GATEUP, -1);
    XSM_EPI(PE_LOGITS, -1);
    XSM_EPI(PE_LOGITS, PE_HEADY);
    XSM_EPI(PE_LOGITS, PE_QUERY);
    XSM_EPI(PE_HEADADD, -1);
#undef XSM_EPI
    return cudaErrorInvalidValue;
}
cudaError_t launch_proj_f32(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) {
    if (A.rows <= 4) return launch_proj_rows<4>(D, A, smem, L);
    if (A.rows <= 8) return launch_proj_rows<8>(D, A, smem, L);
    return launch_proj_rows<kF32Rows>(D, A, smem, L);
}

template <int T>
static cudaError_t launch_attn_rows(const Dev &D, const AttnArgs &A, const ChainLaunch &L) {
    void (*fn)(const Dev, const AttnArgs) = attn_f32_kernel<T>;
    const int smem = (2 * kF32Keys * (D.dh + 4) + 2 * T * D.dh + T * kF32Threads + kF32Warps * T + 3 * T) * 4;
    cudaError_t e = open_kernel((const void *)fn, smem, false);
    if (e != cudaSuccess) return e;
    return L.launch(dim3(1, D.H, D.B * A.sets), dim3(kF32Threads), smem, 1, (const void *)fn, D, A);
}
cudaError_t launch_attn_f32(const Dev &D, const AttnArgs &A, const ChainLaunch &L) {
    if (A.t <= 4) return launch_attn_rows<4>(D, A, L);
    if (A.t <= 8) return launch_attn_rows<8>(D, A, L);
    return launch_attn_rows<kF32Rows>(D, A, L);
}

}  // namespace xsm
