// Projections over few token rows of narrow bf16 models (plan_few), as kernels of the launch chain.
//
// A CTA owns a run of weight rows at full width.  Its rows are on their way to shared memory before the kernel waits for
// its predecessor (bulk copies by a producer warp, tiles of 16 rows x one pass of columns).  Then every warp fetches the
// activations of its own blocks of 32 columns straight into operand registers (one round trip to L2, nothing is staged),
// multiplies all tiles with mma.sync.m16n8k16 (weight rows on M; on N the hi parts of four token rows and their lo parts
// beside them, or eight token rows and a product for each part), and parks its partial sums; after one barrier the sums over the
// warps are finished and stored.  Latency is all that counts here (a step has about a hundred of these kernels in a row, 0.1 to 9 MB
// of weights each): no cluster, no exchange.
#pragma once
#include "xsm_proj.cuh"

namespace xsm {

// NW: multiplying warps; NT: tiles of eight token rows; PACK: at most four token rows, hi and lo parts side by side in one product,
// else in products of their own; MAXB: blocks of 32 columns that a warp holds in registers (a pass is NW * MAXB blocks at most)
template <int NW, int NT, bool PACK, int MAXB, int EPI0, int EPI1>
__global__ void __launch_bounds__((NW + 1) * 32, NW == 8 && NT == 1 && (PACK || MAXB == 4) ? 2 : 1) proj_few_kernel(const Dev D, const ProjArgs A) {
    extern __shared__ __align__(128) char smem[];
    __shared__ __align__(8) uint64_t full[kProjRing], empty[kProjRing];
    __shared__ float s_inv[NT * 8];
    constexpr int kOutThreads = NW * 32, LDM = NT * 8 + 1;      // (odd pitch: neighbouring rows in other banks)
    constexpr bool PAIRS = EPI0 == PE_QKV || EPI0 == PE_GATEUP;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (!A.late_go) chain_go();
    // sequences that still run: looked at just before the wait, when the weights are on their way
    const int active = A.pos0 < 0 && !A.late_go ? __ldcg(D.n_active) : 1;
    // this CTA's units: rows, or pairs of rows (rotation partners; gate and up)
    const int job = A.x_jobs ? blockIdx.x / A.ctas : 0, cta = A.x_jobs ? blockIdx.x - job * A.ctas : blockIdx.x;
    const int all_units = EPI0 == PE_QKV ? A.g[0].units >> 1 : A.g[0].units + (EPI1 >= 0 ? A.g[1].units * A.g[1].jobs : 0);
    const int lo = cta * A.upc, n_units = min(A.upc, all_units - lo), n_rows = PAIRS ? 2 * n_units : n_units;
    const int tiles = (n_rows + 15) >> 4, kdim = A.kdim, chunk = A.chunk, passes = (kdim + chunk - 1) / chunk;
    const uint32_t pitch = (uint32_t)chunk * 2u + 64u, slot_bytes = (uint32_t)A.slot_rows * pitch, ring = smem_u32(smem);
    const int half = D.dh >> 1, M = A.rows;
    // rows of pair p of q, k, v: p and its rotation partner half a head further
    auto qkv_row = [&](int p) {
        const int hd = D.d >> 1, sec = p / hd, i = p - sec * hd, head = i / half;
        return sec * D.d + head * D.dh + (i - head * half);
    };
    // the producer warp owns the barriers and the ring: stage s is a pass of a tile, tile by tile within a pass
    const int stages = tiles * passes;
    auto issue = [&](int s, int sl) {
        const int pass = s / tiles, tile = s - pass * tiles, r = tile * 16 + lane, rows = min(16, n_rows - tile * 16);
        const uint32_t bytes = (uint32_t)min(chunk, kdim - pass * chunk) * 2u, f = smem_u32(&full[sl]);
        if (lane == 0) mbar_arrive_expect_tx(f, bytes * (uint32_t)rows);
        __syncwarp();
        if (lane < rows) {
            const bf16 *src;
            if (EPI0 == PE_QKV) {
                src = A.g[0].w + (size_t)(qkv_row(lo + (r >> 1)) + (r & 1) * half) * kdim;
            } else if (EPI0 == PE_GATEUP) {
                src = A.g[r & 1].w + (size_t)(lo + (r >> 1)) * kdim;
            } else {
                int u = lo + r;
                if (EPI1 >= 0 && u >= A.g[0].units) {
                    u -= A.g[0].units;
                    const int j = u / A.g[1].units;
                    src = A.g[1].w + (size_t)j * A.g[1].w_stride + (size_t)(u - j * A.g[1].units) * kdim;
                } else {
                    src = A.g[0].w + (size_t)job * A.g[0].w_stride + (size_t)u * kdim;
                }
            }
            bulk_g2s(ring + (uint32_t)sl * slot_bytes + (uint32_t)lane * pitch, src + (size_t)pass * chunk, bytes, f);
        }
        __syncwarp();
    };
    if (tid < A.slots) {
        mbar_init(smem_u32(&full[tid]), 1u);
        mbar_init(smem_u32(&empty[tid]), (uint32_t)NW);
        mbar_init_fence();
    }
    __syncthreads();
    if (warp == NW) {
        for (int s = 0; s < min(stages, A.slots); ++s) issue(s, s);
    }
    if (A.stage == 0) trace_mark(D, 0);

    // Everything that does not depend on the step is worked out before the wait, so that little is left to issue after it (a
    // warp gets an instruction off every 8 cycles here): this thread's first output and where it goes, the places of the
    // warp's activations.
    constexpr int MP = NT * 8;                     // rows of a plane
    constexpr bool HEAD = EPI0 == PE_HEADADD || EPI1 == PE_HEADY;
    int lpt = 8;                                   // PE_ADD: lanes per token row
    if (EPI0 == PE_ADD)
        while (lpt < A.upc) lpt <<= 1;
    const int per_m = EPI0 == PE_ADD ? lpt : n_units;
    float *const red = reinterpret_cast<float *>(smem + (size_t)A.slots * slot_bytes);     // [tile][warp][16][LDM]
    struct Out {
        int m, r, grp, sec, e;                     // token row, unit or row of the CTA, group; section of q, k, v, element of the head
        const float *sum;                          // the warps' partial sums
        char *p;                                   // where the output goes (keys and values: head and section in page 0, row 0)
        const float *h;                            // residual stream
        float gain;
        RowInfo row;                               // q, k, v: place in the cache, cosine and sine
        float2 cs;
    };
    auto locate = [&](int e, Out &o) {
        o.m = e / per_m;
        o.r = e - o.m * per_m;
        o.grp = 0;
        const int lr = PAIRS ? 2 * o.r : o.r;
        o.sum = red + (size_t)((lr >> 4) * NW * 16 + (lr & 15)) * LDM + o.m;
        int u = lo + o.r, j = job;
        if (EPI0 == PE_QKV) {
            u = qkv_row(u);
            o.sec = u >= D.d ? (u >= 2 * D.d ? 2 : 1) : 0;
            u -= o.sec * D.d;
            const int head = u / D.dh;
            o.e = u - head * D.dh;
            if (o.sec > 0) o.p = reinterpret_cast<char *>(kv_tile<__half>(D, D.kv_pool, D.n_pages, A.layer, o.sec - 1, 0, head) + (o.e & 7));
        }
        if (EPI1 >= 0 && u >= A.g[0].units) {
            u -= A.g[0].units;
            j = u / A.g[1].units;
            u -= j * A.g[1].units;
            o.grp = 1;
        }
        const int epi = EPI1 >= 0 && o.grp ? EPI1 : EPI0;
        if (epi == PE_QKV || epi == PE_QUERY) {
            if (EPI0 != PE_QKV || o.sec == 0) o.p = reinterpret_cast<char *>(A.q + ((size_t)j * 2 * MP + o.m) * D.d + u);
        } else if (epi == PE_LOGITS) {
            o.p = reinterpret_cast<char *>(A.g[0].logits + ((size_t)j * D.M + o.m) * A.g[0].ld + u);
        } else {
            const ProjGroup &G = A.g[EPI1 >= 0 ? 1 : 0];
            o.p = reinterpret_cast<char *>(G.out + (size_t)j * 2 * MP * G.ld + plane_off(MP, o.m, u));
        }
        u = min(u, D.d - 1);
        o.h = D.h + (size_t)min(o.m, kMaxTokens - 1) * D.d + u;
        if (EPI0 == PE_ADD || HEAD) o.gain = to_f(__ldg(reinterpret_cast<const bf16 *>(A.gain) + u));
    };
    auto position = [&](Out &o) {
        o.row = *reinterpret_cast<const RowInfo *>(&(const int4 &)__ldcg(reinterpret_cast<const int4 *>(D.row_info + o.m)));
        o.cs = __ldcg(D.row_cs + (size_t)o.m * half + o.e);
    };
    Out o1;
    locate(tid, o1);
    const bool has = warp < NW && tid < M * per_m && o1.r < n_units;
    if (EPI0 == PE_QKV && has && !A.late_go) position(o1);
    const int g = lane >> 2, t4 = lane & 3;
    // the warp's blocks are warp + NW i.  PACK: lanes 0..15 hi parts of token rows g & 3, the others lo parts.  Lanes past the last
    // token row read the first one of their tile again (what they multiply goes nowhere).
    const bf16 *x0[2], *x_last[2];      // first (of two tiles) and last tile
#pragma unroll
    for (int q = 0; q < 2; ++q) {      // (odd NW: the blocks of a warp alternate between the halves of a 64-column block)
        const int blk = warp + NW * q, m = PACK ? ((g & 3) < M ? g & 3 : 0) : (NT - 1) * 8 + g < M ? g : 0, chunk8 = (blk & 1) * 4 + t4;
        const bf16 *base = A.x + (A.x_jobs ? (size_t)job * 2 * MP * kdim : 0) + (size_t)(blk >> 1) * (128 * MP);
        x0[q] = base + g * 64 + ((chunk8 ^ g) << 3);
        x_last[q] = base + (NT - 1) * 1024 + m * 64 + ((chunk8 ^ m) << 3) + (PACK ? (g >> 2) * kLo : 0);
    }
    const uint32_t full0 = smem_u32(&full[0]);
    const char *w0 = smem + (size_t)g * pitch + t4 * 16 + warp * 64;
    float *dst0 = red + (size_t)(warp * 16 + g) * LDM + 2 * t4;
#pragma unroll
    for (int q = 0; q < 2; ++q) { if (NT > 1) settle(x0[q]); settle(x_last[q]); }
    settle(o1.sum); settle(o1.p); settle(o1.h); settle(w0); settle(dst0);
    if (EPI0 == PE_ADD || HEAD) settle(o1.gain);
    if (warp < NW) bar_sync<NW * 32>(1);           // (warps that come to the wait together leave it sooner: 0.3 us a kernel)
    chain_wait();
    if (active == 0) {                             // every sequence has ended in an earlier step
        if (warp == NW)
            for (int s = 0; s < min(stages, A.slots); ++s) mbar_wait(smem_u32(&full[s]), 0u, D.mbar_limit, D.status);
        return;
    }
    if (A.late_go) {
        chain_go();
        if (EPI0 == PE_QKV && has) position(o1);
    }
    trace_mark(D, 1 + 2 * A.stage);

    float h_old = 0.f;
    auto park = [&](float *dst, const float (&c0)[NT][4], const float (&c1)[NT][4], bool first) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float v = c0[nt][q] + c1[nt][q];
                if (PACK) v += __shfl_xor_sync(0xffffffffu, v, 2);      // columns 0..3: hi parts, 4..7: lo parts of the same rows
                if (!PACK || t4 < 2) {
                    float *o = dst + (q >> 1) * 8 * LDM + nt * 8 + (q & 1);
                    *o = first ? v : *o + v;
                }
            }
    };
    if (warp < NW) {
        int sl = 0;
        uint32_t par = 0;
        for (int pass = 0; pass < passes; ++pass) {
            const int nb = min(chunk, kdim - pass * chunk) >> 5;      // blocks of 32 columns
            const size_t xp = (size_t)(pass * (chunk >> 6)) * (128 * MP);
            uint4 x[MAXB][NT], xl[MAXB][NT];      // PACK: both parts; else hi parts, lo parts
#pragma unroll
            for (int i = 0; i < MAXB; ++i)
                if (warp + NW * i < nb) {
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const int q = (NW & 1) ? i & 1 : 0;
                        const bf16 *p = (nt < NT - 1 ? x0[q] : x_last[q]) + xp + (size_t)((NW & 1) ? (i >> 1) * NW : i * (NW / 2)) * (128 * MP);
                        x[i][nt] = __ldcg(reinterpret_cast<const uint4 *>(p));
                        if (!PACK) xl[i][nt] = __ldcg(reinterpret_cast<const uint4 *>(p + kLo));
                    }
                }
            if ((EPI0 == PE_ADD || HEAD) && pass == 0 && has) h_old = __ldcg(o1.h);
            float *dst = dst0;
            for (int tile = 0; tile < tiles; ++tile) {
                const bool two = n_rows - tile * 16 > 8;
                mbar_wait(full0 + 8u * (uint32_t)sl, par, D.mbar_limit, D.status);
                const char *ws = w0 + (size_t)sl * slot_bytes;
                float c0[NT][4], c1[NT][4];      // PACK: even and odd steps of 16 columns; else hi parts, lo parts
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int q = 0; q < 4; ++q) c0[nt][q] = c1[nt][q] = 0.f;
#pragma unroll
                for (int i = 0; i < MAXB; ++i) {
                    if (warp + NW * i < nb) {
                        const uint4 a = *reinterpret_cast<const uint4 *>(ws + NW * i * 64);
                        uint4 c = make_uint4(0u, 0u, 0u, 0u);
                        if (two) c = *reinterpret_cast<const uint4 *>(ws + 8 * pitch + NW * i * 64);
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            mma16816_bf16(c0[nt], a.x, c.x, a.y, c.y, x[i][nt].x, x[i][nt].y);
                            if (PACK) {
                                mma16816_bf16(c1[nt], a.z, c.z, a.w, c.w, x[i][nt].z, x[i][nt].w);
                            } else {
                                mma16816_bf16(c1[nt], a.x, c.x, a.y, c.y, xl[i][nt].x, xl[i][nt].y);
                                mma16816_bf16(c0[nt], a.z, c.z, a.w, c.w, x[i][nt].z, x[i][nt].w);
                                mma16816_bf16(c1[nt], a.z, c.z, a.w, c.w, xl[i][nt].z, xl[i][nt].w);
                            }
                        }
                    }
                }
                if (A.slots < tiles * passes) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&empty[sl]));
                }
                if (++sl == A.slots) { sl = 0; par ^= 1u; }
                park(dst, c0, c1, pass == 0);
                dst += NW * 16 * LDM;
            }
        }
    } else {
        // the producer warp adds up the shares of the sums of squares: four lanes per token row, every fourth quad each
        if (A.ss_parts > 0) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const float4 *sh = reinterpret_cast<const float4 *>(D.ss + (size_t)min(nt * 8 + g, M - 1) * kShareLd) + t4;
            float4 v[kShareLd / 16];
#pragma unroll
            for (int q = 0; q < kShareLd / 16; ++q) v[q] = 16 * q + 4 * t4 < A.ss_parts ? __ldcg(sh + 4 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
            float ss = 0.f;
#pragma unroll
            for (int q = 0; q < kShareLd / 16; ++q) {
                const int n = A.ss_parts - 16 * q - 4 * t4;      // (the last quad may hold shares that nobody writes)
                ss += (v[q].x + (n > 1 ? v[q].y : 0.f)) + ((n > 2 ? v[q].z : 0.f) + (n > 3 ? v[q].w : 0.f));
            }
            ss += __shfl_xor_sync(0xffffffffu, ss, 1);
            ss += __shfl_xor_sync(0xffffffffu, ss, 2);
            if (t4 == 0) s_inv[nt * 8 + g] = 1.0f / sqrtf(ss / (float)D.d + D.eps);
        }
        }
        // then the rest of the weights, as their slots become free
        int sl = 0;
        uint32_t par = 0;
        for (int s = A.slots; s < stages; ++s) {
            mbar_wait(smem_u32(&empty[sl]), par, D.mbar_limit, D.status);
            __syncwarp();
            issue(s, sl);
            if (++sl == A.slots) { sl = 0; par ^= 1u; }
        }
    }
    __syncthreads();
    if (warp == NW) return;
    auto total = [&](const float *p) {
        float v[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) v[w] = p[w * 16 * LDM];
#pragma unroll
        for (int n = 1; n < NW; n *= 2)
#pragma unroll
            for (int w = 0; w + n < NW; w += 2 * n) v[w] += v[w + n];
        return v[0];
    };
    auto put_bf16 = [&](char *p, float v) {
        bf16 hi, lo_;
        split_bf16(v, hi, lo_);
        reinterpret_cast<bf16 *>(p)[0] = hi;
        reinterpret_cast<bf16 *>(p)[kLo] = lo_;
    };
    auto put_query = [&](char *p, float v) {
        __half hi, lo_;
        split_f16(v * A.scale, hi, lo_);
        reinterpret_cast<__half *>(p)[0] = hi;
        reinterpret_cast<__half *>(p)[(size_t)MP * D.d] = lo_;
    };
    const int outputs = EPI0 == PE_ADD ? (M * per_m + 31) & ~31 : M * per_m;      // (PE_ADD: whole warps, which shuffle)
    for (int e = tid; e < outputs; e += kOutThreads) {
        if (e != tid) {
            locate(e, o1);
            if (EPI0 == PE_QKV) position(o1);
            if (EPI0 == PE_ADD || HEAD) h_old = __ldcg(o1.h);
        }
        const float inv = A.ss_parts > 0 ? s_inv[o1.m] : 1.f;
        if (EPI0 == PE_ADD) {
            float h = 0.f;
            if (o1.r < n_units && o1.m < M) {
                h = h_old + total(o1.sum);
                *const_cast<float *>(o1.h) = h;
                put_bf16(o1.p, h * o1.gain);
            }
            float ssq = h * h;
            for (int k = lpt >> 1; k > 0; k >>= 1) ssq += __shfl_xor_sync(0xffffffffu, ssq, k);
            if (o1.r == 0 && o1.m < M) D.ss[(size_t)o1.m * kShareLd + cta] = ssq;
        } else if (EPI0 == PE_QKV) {
            const float v = total(o1.sum) * inv, v2 = total(o1.sum + LDM) * inv;
            if (o1.sec == 0) {
                put_query(o1.p, v * o1.cs.x - v2 * o1.cs.y);
                put_query(o1.p + half * 2, v2 * o1.cs.x + v * o1.cs.y);
            } else if (o1.row.place >= 0) {
                __half *p = reinterpret_cast<__half *>(o1.p) + o1.row.place;
                const int sw = row_swz(o1.row.rp, D.dh);
                p[((o1.e >> 3) ^ sw) << 3] = from_f<__half>(o1.sec == 1 ? v * o1.cs.x - v2 * o1.cs.y : v);
                p[(((o1.e + half) >> 3) ^ sw) << 3] = from_f<__half>(o1.sec == 1 ? v2 * o1.cs.x + v * o1.cs.y : v2);
            }
        } else if (EPI0 == PE_GATEUP) {
            put_bf16(o1.p, silu_f(total(o1.sum) * inv) * (total(o1.sum + LDM) * inv));
        } else if (EPI0 == PE_QUERY || (EPI1 == PE_QUERY && o1.grp)) {
            put_query(o1.p, total(o1.sum) * inv);
        } else if (EPI0 == PE_HEADADD) {
            put_bf16(o1.p, h_old * inv * o1.gain + total(o1.sum));
        } else if (EPI1 == PE_HEADY && o1.grp) {
            put_bf16(o1.p, h_old * inv * o1.gain + silu_f(total(o1.sum) * inv));
        } else {
            const float v = total(o1.sum);
            *reinterpret_cast<float *>(o1.p) = A.norm ? v * inv : v;
        }
    }
    trace_mark(D, 2 + 2 * A.stage);
}

template <int NW, int NT, bool PACK, int MAXB, int EPI0, int EPI1>
static cudaError_t launch_few_instance(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) {
    void (*fn)(const Dev, const ProjArgs) = proj_few_kernel<NW, NT, PACK, MAXB, EPI0, EPI1>;
    cudaError_t e = open_kernel((const void *)fn, smem, false);
    if (e != cudaSuccess) return e;
    return L.launch(dim3(A.x_jobs ? A.ctas * A.g[0].jobs : A.ctas), dim3((NW + 1) * 32), smem, 1, (const void *)fn, D, A);
}

template <int NW, int NT, bool PACK, int MAXB>
static cudaError_t launch_few(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) {
#define XSM_EPI(a, b) if (A.epi0 == a && A.epi1 == b) return launch_few_instance<NW, NT, PACK, MAXB, a, b>(D, A, smem, L)
    XSM_EPI(PE_ADD, -1);
    if constexpr (NW == 8 && MAXB == 4) {      // (rows of more than 1024 columns: the down projection's only)
        XSM_EPI(PE_QUERY, -1);
        XSM_EPI(PE_QKV, -1);
        XSM_EPI(PE_GATEUP, -1);
        XSM_EPI(PE_LOGITS, -1);
        XSM_EPI(PE_LOGITS, PE_HEADY);
        XSM_EPI(PE_LOGITS, PE_QUERY);
        XSM_EPI(PE_HEADADD, -1);
    }
#undef XSM_EPI
    return cudaErrorInvalidValue;
}

}  // namespace xsm
