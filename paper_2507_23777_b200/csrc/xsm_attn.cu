// Attention of bf16 models over the paged fp16 caches, as a kernel of the launch chain.
//
// A cluster of up to S CTAs serves one (sequence, head): they cut the keys by pages, a producer warp streams (page, head)
// tiles of keys and values through a ring in shared memory, eight or sixteen warps attend with mma.sync over 32 keys at a
// time (a unit).  How many of the S take part depends on the keys of the step (one CTA for every 384, 192 in heads of 128,
// 128 where the rows form tiles: the rule and its figures stand at plan_attn).  Each of them finishes a share of the rows:
// the others send it their partial results by counted stores into its shared memory, and it adds them up in rank order.
// The keys and values of the rows themselves have been written to the cache by the projection before, so self-attention
// is the same walk with a causal limit per row.  Pages that the step does not write (and the condition's) are fetched
// before the kernel waits for its predecessor.
//
// Few rows (at most eight, every step of a batch of any size with up to seven heads): the product is transposed,
// S^T = K Q^T and O^T = V^T P^T, so that the 16 keys of a product sit on its M side and the rows on its 8-wide N side;
// all warps take different keys.  More rows (chunks of a prompt, many heads): tiles of 16 rows on the M side; the
// warps are divided over the row tiles first and over the keys with what is left.
#include "xsm_proj.cuh"

namespace xsm {

constexpr int kAttnSlots = 16;

// ------------------------------------------------------------------- 32 keys against at most eight rows

template <int DH> struct FewState {
    float o[DH / 16][4];          // rows 16 dp + g (0, 1) and + 8 (2, 3) of O^T; columns 2t (0, 2) and 2t + 1 (1, 3)
    float m[2], l[2];             // rows 2t, 2t + 1; l: this thread's keys only until the state is parked
};

// lim: last key of the unit that row 2t (2t + 1) sees
template <int DH>
__device__ __forceinline__ void few_unit(const unsigned (&qh)[DH / 8], const unsigned (&ql)[DH / 8], uint32_t k_tile, uint32_t v_tile, int key0,
                                         int lim0, int lim1, FewState<DH> &ws) {
    constexpr int RB = DH * 2;
    const int lane = threadIdx.x & 31, g = lane >> 2;
    float s[2][4], sl[2][4];       // products with the hi and lo parts of the queries
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
        s[kt][0] = s[kt][1] = s[kt][2] = s[kt][3] = 0.f;
        sl[kt][0] = sl[kt][1] = sl[kt][2] = sl[kt][3] = 0.f;
    }
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks) {
#pragma unroll
        for (int kt = 0; kt < 2; ++kt) {
            const int row = key0 + kt * 16 + (lane & 7) + (((lane >> 3) & 1) << 3);
            const int chunk = 2 * ks + (lane >> 4);
            unsigned ka[4];
            ldmatrix_x4(ka, k_tile + (uint32_t)row * RB + (uint32_t)swz(row, chunk, RB) * 16u);
            mma16816_f16(s[kt], ka[0], ka[1], ka[2], ka[3], qh[2 * ks], qh[2 * ks + 1]);
            mma16816_f16(sl[kt], ka[0], ka[1], ka[2], ka[3], ql[2 * ks], ql[2 * ks + 1]);
        }
    }
#pragma unroll
    for (int kt = 0; kt < 2; ++kt)
#pragma unroll
        for (int q = 0; q < 4; ++q) s[kt][q] += sl[kt][q];
    float mx0 = kNegBig, mx1 = kNegBig;
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
        const int r0 = kt * 16 + g, r1 = r0 + 8;
        if (r0 > lim0) s[kt][0] = -INFINITY;
        if (r0 > lim1) s[kt][1] = -INFINITY;
        if (r1 > lim0) s[kt][2] = -INFINITY;
        if (r1 > lim1) s[kt][3] = -INFINITY;
        mx0 = fmaxf(mx0, fmaxf(s[kt][0], s[kt][2]));
        mx1 = fmaxf(mx1, fmaxf(s[kt][1], s[kt][3]));
    }
#pragma unroll
    for (int o = 4; o <= 16; o <<= 1) {
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
    }
    const float m0 = fmaxf(ws.m[0], mx0), m1 = fmaxf(ws.m[1], mx1);
    const float c0 = ex2(ws.m[0] - m0), c1 = ex2(ws.m[1] - m1);
    ws.m[0] = m0; ws.m[1] = m1;
    float l0 = 0.f, l1 = 0.f;
    unsigned pb[2][2];             // P^T as B fragments of the 16-key steps (fp16: weights in [0, 1])
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
        const float p0 = ex2(s[kt][0] - m0), p1 = ex2(s[kt][1] - m1);
        const float p2 = ex2(s[kt][2] - m0), p3 = ex2(s[kt][3] - m1);
        l0 += p0 + p2; l1 += p1 + p3;
        pb[kt][0] = movmatrix_trans(pack_f16x2(p0, p1));      // keys 0..7 of the step
        pb[kt][1] = movmatrix_trans(pack_f16x2(p2, p3));      // keys 8..15
    }
    ws.l[0] = ws.l[0] * c0 + l0;
    ws.l[1] = ws.l[1] * c1 + l1;
    if (__any_sync(0xffffffffu, c0 != 1.f || c1 != 1.f)) {     // a new maximum somewhere in the warp's columns
#pragma unroll
        for (int dp = 0; dp < DH / 16; ++dp) { ws.o[dp][0] *= c0; ws.o[dp][1] *= c1; ws.o[dp][2] *= c0; ws.o[dp][3] *= c1; }
    }
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
#pragma unroll
        for (int dp = 0; dp < DH / 16; ++dp) {   // value columns 16dp .. 16dp+15 (chunks 2dp, 2dp+1) are rows of O^T
            const int row = key0 + kt * 16 + (lane & 7) + ((lane >> 4) << 3);
            const int chunk = 2 * dp + ((lane >> 3) & 1);
            unsigned va[4];
            ldmatrix_x4_trans(va, v_tile + (uint32_t)row * RB + (uint32_t)swz(row, chunk, RB) * 16u);
            mma16816_f16(ws.o[dp], va[0], va[1], va[2], va[3], pb[kt][0], pb[kt][1]);
        }
    }
}

// ------------------------------------------------------------------------ 32 keys against sixteen rows

template <int DH> struct RowsState {
    float o[DH / 8][4];
    float m[2], l[2];             // rows g, g + 8
};

template <int DH>
__device__ __forceinline__ void rows_unit(const unsigned (&qh)[DH / 16][4], const unsigned (&ql)[DH / 16][4], uint32_t k_tile, uint32_t v_tile,
                                          int key0, int lim0, int lim1, RowsState<DH> &ws) {
    constexpr int RB = DH * 2;
    const int lane = threadIdx.x & 31, t = lane & 3;
    float s[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks) {
#pragma unroll
        for (int np = 0; np < 2; ++np) {      // key tiles 2np, 2np+1 (8 keys each)
            const int row = key0 + np * 16 + (lane & 7) + ((lane >> 4) << 3);
            const int chunk = 2 * ks + ((lane >> 3) & 1);
            unsigned kb[4];
            ldmatrix_x4(kb, k_tile + (uint32_t)row * RB + (uint32_t)swz(row, chunk, RB) * 16u);
            mma16816_f16(s[2 * np], qh[ks][0], qh[ks][1], qh[ks][2], qh[ks][3], kb[0], kb[1]);
            mma16816_f16(s[2 * np], ql[ks][0], ql[ks][1], ql[ks][2], ql[ks][3], kb[0], kb[1]);
            mma16816_f16(s[2 * np + 1], qh[ks][0], qh[ks][1], qh[ks][2], qh[ks][3], kb[2], kb[3]);
            mma16816_f16(s[2 * np + 1], ql[ks][0], ql[ks][1], ql[ks][2], ql[ks][3], kb[2], kb[3]);
        }
    }
    float mx0 = kNegBig, mx1 = kNegBig;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int k0 = nt * 8 + 2 * t;
        if (k0 > lim0) s[nt][0] = -INFINITY;
        if (k0 + 1 > lim0) s[nt][1] = -INFINITY;
        if (k0 > lim1) s[nt][2] = -INFINITY;
        if (k0 + 1 > lim1) s[nt][3] = -INFINITY;
        mx0 = fmaxf(mx0, fmaxf(s[nt][0], s[nt][1]));
        mx1 = fmaxf(mx1, fmaxf(s[nt][2], s[nt][3]));
    }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1)); mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float m0 = fmaxf(ws.m[0], mx0), m1 = fmaxf(ws.m[1], mx1);
    const float c0 = ex2(ws.m[0] - m0), c1 = ex2(ws.m[1] - m1);
    ws.m[0] = m0; ws.m[1] = m1;
    float l0 = 0.f, l1 = 0.f;
    unsigned ph[2][4];             // P as A fragments of the two 16-key steps (fp16: weights in [0, 1])
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const float p0 = ex2(s[nt][0] - m0), p1 = ex2(s[nt][1] - m0);
        const float p2 = ex2(s[nt][2] - m1), p3 = ex2(s[nt][3] - m1);
        l0 += p0 + p1; l1 += p2 + p3;
        const int kk = nt >> 1, hi2 = (nt & 1) * 2;     // a0,a1 from the even key tile, a2,a3 from the odd one
        ph[kk][hi2] = pack_f16x2(p0, p1); ph[kk][hi2 + 1] = pack_f16x2(p2, p3);
    }
    ws.l[0] = ws.l[0] * c0 + l0;
    ws.l[1] = ws.l[1] * c1 + l1;
    if (__any_sync(0xffffffffu, c0 != 1.f || c1 != 1.f)) {     // a new maximum somewhere in the warp's rows
#pragma unroll
        for (int dn = 0; dn < DH / 8; ++dn) { ws.o[dn][0] *= c0; ws.o[dn][1] *= c0; ws.o[dn][2] *= c1; ws.o[dn][3] *= c1; }
    }
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
        for (int dp = 0; dp < DH / 16; ++dp) {   // value columns 16dp .. 16dp+15 (chunks 2dp, 2dp+1)
            const int row = key0 + kk * 16 + (lane & 7) + (((lane >> 3) & 1) << 3);
            const int chunk = 2 * dp + (lane >> 4);
            unsigned vb[4];
            ldmatrix_x4_trans(vb, v_tile + (uint32_t)row * RB + (uint32_t)swz(row, chunk, RB) * 16u);
            mma16816_f16(ws.o[2 * dp], ph[kk][0], ph[kk][1], ph[kk][2], ph[kk][3], vb[0], vb[1]);
            mma16816_f16(ws.o[2 * dp + 1], ph[kk][0], ph[kk][1], ph[kk][2], ph[kk][3], vb[2], vb[3]);
        }
    }
}

// n partial results of a row, `step` floats apart, as one: columns c and c + 1 of [columns .., maximum, sum].  Eight at a time,
// all their loads together (one by one, each behind the last one's: large model, batch 1 1680 -> 1648 us a step).
__device__ __forceinline__ void merge_states(const float *src, int dh, int c, int n, int step, float &m, float &l, float &o0, float &o1) {
    m = kNegBig;
    l = o0 = o1 = 0.f;
#pragma unroll 1
    for (; n > 0; n -= 8, src += 8 * step) {
        float mv[8], lv[8];
        float2 ov[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            mv[w] = kNegBig;
            lv[w] = 0.f;
            ov[w] = make_float2(0.f, 0.f);
            if (w < n) {
                const float2 ml = *reinterpret_cast<const float2 *>(src + w * step + dh);
                mv[w] = ml.x;
                lv[w] = ml.y;
                ov[w] = *reinterpret_cast<const float2 *>(src + w * step + c);
            }
        }
        const float before = m;
#pragma unroll
        for (int w = 0; w < 8; ++w) m = fmaxf(m, mv[w]);
        const float f0 = ex2(before - m);
        l *= f0; o0 *= f0; o1 *= f0;
#pragma unroll
        for (int w = 0; w < 8; ++w)
            if (w < n) {
                const float f = ex2(mv[w] - m);
                o0 += f * ov[w].x;
                o1 += f * ov[w].y;
                l += f * lv[w];
            }
    }
}

// ------------------------------------------------------------------------------------------- kernel

__device__ __forceinline__ unsigned ldcg_u32(const void *p) { return __ldcg(reinterpret_cast<const unsigned *>(p)); }

// QP (cross-attention of a step, few rows): the kernel projects the queries of its head itself, from the normalised residual
// stream (every warp multiplies all rows over its share of the columns, as in the projections over few token rows), instead
// of a kernel of its own: 630 against 650 us a step at width 1024.  The head's rows of the projection and the pages are requested
// before the wait; a CTA (544 threads of 96 registers) shares an SM with none of the projections, but the out-projection before it
// holds 64 of 148, so the sixteen CTAs of a sequence start some 7 us before it ends.  4.0 us after the wait: 0.6 until the
// activations come, 1.3 products (128 KB of weights through shared memory), 0.4 sums, 1.1 keys, 0.6 merge and output.
constexpr int kQueryBlocks = 4;      // blocks of 32 columns per warp: d_model up to 1024
//
// NW: warps that attend, beside the producer.  A unit of 32 keys is some 300 dependent instructions, 1 us for a warp on its
// own, so sixteen warps where a CTA has many units (and where the queries are projected); eight otherwise, of which two
// CTAs share an SM when a batch has more (sequence, head) pairs than there are SMs.
// CL: several CTAs to a (sequence, head), a cluster.
template <int DH, bool FEW, bool QP, int NW, bool CL>
__global__ void __launch_bounds__(NW * 32 + 32, FEW && DH <= 64 && NW == 8 ? 2 : 1) attn_kernel(const Dev D, const AttnArgs A) {
    constexpr int kThreads = NW * 32 + 32, RB = DH * 2;
    extern __shared__ __align__(128) char smem[];
    __shared__ __align__(8) uint64_t full[kAttnSlots], empty[kAttnSlots], w_full, recv_bar;
    __shared__ float s_inv[8];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // (tiles of a sequence's rows: those that see the most keys first)
    const int rank = CL ? blockIdx.x : 0, h = blockIdx.y, b = blockIdx.z % D.B, zz = blockIdx.z / D.B, set = zz % A.sets;
    const int q0 = (A.qt - 1 - zz / A.sets) * kTokenTile, t_rows = min(A.t - q0, kTokenTile);
    const int P = D.P, upp = P >> 5, slots = A.slots;
    const bool cross = A.cross != 0;
    const int first = cross ? 0 : A.pos0 >= 0 ? A.pos0 : __ldcg(D.len + b);      // (the state was written by an earlier step)
    const int start = first + q0, n_keys = cross ? D.C : A.pos0 >= 0 ? min(start + t_rows, A.pos_end) : start + t_rows;
    const int S = CL ? min(A.S, (n_keys + A.split - 1) / A.split) : 1;           // CTAs that take part
    if (CL && rank >= S) {
        cluster_arrive_relaxed();
        cluster_wait();
        return;
    }
    // few rows: a warp looks only at the pages whose units it owns when the units of 1, 2 or 4 pages fill a round of the
    // warps (the ring is a whole number of rounds, so a warp meets every fill of its slots)
    const bool owned = FEW && NW == 8 && (upp == 1 || upp == 2 || upp == 4);
    if (tid == 0) {
        for (int i = 0; i < kAttnSlots; ++i) {
            mbar_init(smem_u32(&full[i]), 1u);
            mbar_init(smem_u32(&empty[i]), owned ? (uint32_t)upp : (uint32_t)NW);
        }
        if (QP) mbar_init(smem_u32(&w_full), 1u);
        mbar_init(smem_u32(&recv_bar), 1u);
        mbar_init_fence();
        // (rows rank, rank + S, .. are finished here; may be none)
        const int my_rows = (t_rows - rank + S - 1) / S;
        if (CL && S > 1 && my_rows > 0) mbar_arrive_expect_tx(smem_u32(&recv_bar), (uint32_t)(S * my_rows * (DH + 2)) * 4u);
    }
    __syncthreads();
    chain_go();
    if (CL) { cluster_arrive_relaxed(); cluster_wait(); }      // the peers run: what is sent to them has a place
    const bool dead = A.pos0 < 0 && __ldcg(D.finished + b) != 0;
    if (dead) {
        chain_wait();
        return;
    }
    const int np = page_of(D, n_keys + P - 1), p_lo = rank * np / S, p_hi = (rank + 1) * np / S;
    const uint32_t tile_bytes = (uint32_t)P * DH * 2u, ring = smem_u32(smem);
    // Few rows: where all pages fit the ring (of the last one only the units that hold keys), nothing is waited for but the page
    // of a unit, and nothing is given back.
    const int pages = p_hi - p_lo, last_rows = min(P, (n_keys - (p_hi - 1) * P + 31) & ~31);
    const bool all_in = FEW && pages > 0 && pages <= kAttnSlots && (uint32_t)(pages - 1) * 2u * tile_bytes + (uint32_t)last_rows * 2u * RB <= (uint32_t)A.ring;
    const int n_units = pages > 0 ? (pages - 1) * upp + (last_rows >> 5) : 0;
    const int qt_n = FEW ? 1 : (t_rows + 15) >> 4;                       // row tiles
    int wq = 1;                                                       // warps that share the keys between them: NW / wq
    if (!FEW)
        while (wq < qt_n) wq <<= 1;
    const int kg_n = NW / wq;            // (few rows: warps, at most; those without a unit leave nothing)
    // parked states of the warps [NW][rows][DH + 2]; they reuse the ring
    constexpr int LD = DH + 2;
    const int srows = FEW ? t_rows : 16;
    float *st = reinterpret_cast<float *>(smem);
    // QP, behind the ring: the head's weight rows; in their place later partial sums [row tile][8][16][9], queries hi, lo [8][DH + 8]
    constexpr int LDQ = DH + 8;
    const uint32_t w_pitch = (uint32_t)D.d * 2u + 64u;
    char *const w_rows = smem + A.ring;
    float *const q_sum = reinterpret_cast<float *>(w_rows);
    __half *const q_hi = reinterpret_cast<__half *>(q_sum + (DH / 16) * 8 * 16 * 9), *const q_lo = q_hi + 8 * LDQ;

    // A.warm: the attending warps run everything below twice.  The first time they wait for nothing and store nothing; it
    // brings the code into the SM's instruction caches while the predecessor still runs (each instruction is executed about
    // once per stage, and a cold one costs as much again: measured on the merge, 1900 against 1000 cycles).  Self-attention
    // of one sequence 3.5 -> 3.0 us; slower where the first run ends after the wait would have (two CTAs to an SM) or costs
    // registers (QP, heads of 128).
    constexpr bool WARM = FEW && !QP && !CL && DH <= 64 && NW == 8;
#pragma unroll 1
    for (int round = WARM && A.warm && warp < NW ? 0 : 1; round < 2; ++round) {
    int real = 1;
    if (WARM) { real = round; settle(real); }
    if (warp == NW) {
        if (QP) {
            const uint32_t bytes = (uint32_t)D.d * 2u, f = smem_u32(&w_full);
            if (lane == 0) mbar_arrive_expect_tx(f, bytes * DH);
            __syncwarp();
            for (int r = lane; r < DH; r += 32) bulk_g2s(smem_u32(w_rows) + (uint32_t)r * w_pitch, A.wq + (size_t)(h * DH + r) * D.d, bytes, f);
            __syncwarp();
        }
        // (QP: 1/rms of the rows, once the predecessor is done)
        auto scales = [&]() {
            const int m = lane >> 2, t4 = lane & 3;
            const float4 *sh = reinterpret_cast<const float4 *>(D.ss + (size_t)(b * A.t + min(m, t_rows - 1)) * kShareLd) + t4;
            chain_wait();
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
            if (t4 == 0) s_inv[m] = 1.0f / sqrtf(ss / (float)D.d + D.eps);
            asm volatile("bar.arrive 2, %0;" :: "n"(kThreads) : "memory");
        };
        bool scaled = !QP;
        const int n_old = cross ? np : page_of(D, first);         // pages that nobody writes in this step
        bool waited = false;
        int looked_up = 0;      // page p_lo + i with i % 32 == lane (one after the other the look-ups took 0.4 us each)
        for (int i = 0, pg = p_lo; pg < p_hi; ++pg, ++i) {
            if (!cross && (i & 31) == 0) looked_up = pg + lane < p_hi ? __ldcg(D.block_table + (size_t)b * D.max_blocks + pg + lane) : 0;
            const int page = cross ? b * D.cpages + pg : __shfl_sync(0xffffffffu, looked_up, i & 31);
            const int sl = all_in ? i : i % slots, rows = all_in && pg == p_hi - 1 ? last_rows : P;
            const uint32_t part = (uint32_t)rows * RB;
            if (QP && !all_in && i == slots) {      // (due before a slot is free again)
                scales();
                scaled = true;
            }
            if (lane != 0) continue;
            if (!all_in && i >= slots) mbar_wait(smem_u32(&empty[sl]), (uint32_t)((i / slots - 1) & 1), D.mbar_limit, D.status);
            const int pool_pages = cross ? D.B * D.cpages : D.n_pages, lay = cross && A.sets > 1 ? set : A.layer;
            const __half *kt = kv_tile<__half>(D, const_cast<void *>(A.pool), pool_pages, lay, 0, page, h);
            const __half *vt = kv_tile<__half>(D, const_cast<void *>(A.pool), pool_pages, lay, 1, page, h);
            uint32_t f = smem_u32(&full[sl]), dst = ring + (uint32_t)sl * 2u * tile_bytes;
            mbar_arrive_expect_tx(f, 2u * part);
            if (!waited && pg >= n_old) {
                settle(kt); settle(vt); settle(f); settle(dst);
                chain_wait();
                waited = true;
            }
            bulk_g2s(dst, kt, part, f);
            bulk_g2s(dst + part, vt, part, f);
        }
        __syncwarp();
        if (!scaled) scales();
        chain_wait();
        __syncthreads();                 // (1) every page has been consumed
    } else {
        const int g = lane >> 2, t4 = lane & 3;
        // this lane's part of the queries: row g of the first row tile of the warp
        const int row_tile = FEW ? 0 : warp & (wq - 1);
        const __half *qhi = A.q + (size_t)set * 2 * A.qp * D.d + (size_t)(b * A.t + q0 + row_tile * 16 + g) * D.d + h * DH + 2 * t4;
        const __half *qlo = qhi + (size_t)A.qp * D.d;
        // QP: of the residual stream, columns 8 t4 .. of the warp's first block of 32 for token row g (the last rows: the first one again)
        const int xm = b * A.t + (g < t_rows ? g : 0);
        const bf16 *xp = nullptr;
        if (QP) xp = A.x + (size_t)((warp & 7) >> 1) * (128 * A.Mp) + (xm >> 3) * 1024 + (xm & 7) * 64 + ((((warp & 1) * 4 + t4) ^ (xm & 7)) << 3);
        settle(qhi); settle(qlo); settle(xp);
        if (real) {
            bar_sync<NW * 32>(1);      // (warps that come to the wait together leave it sooner)
            chain_wait();
            trace_mark(D, 1 + 2 * A.stage);
        }
        if (FEW) {
            // Warps without keys leave no state, and fetch no queries (where the kernel projects them itself all warps take part in
            // that): 5 rows of width 768 33.87 -> 33.57 ms a request, of width 1024 56.71 -> 56.48, 20 rows 37.37 -> 36.98, 7 rows of
            // width 2048 58.72 -> 58.05.
            const bool busy = !all_in || warp < n_units;
            unsigned qh[DH / 8], ql[DH / 8];
            if constexpr (QP) {
                constexpr int TILES = DH / 32;       // row tiles of a warp: eight warps share the columns, two such groups the rows
                const int nb = D.d >> 5, kg = warp & 7, t0 = (warp >> 3) * TILES;
                uint4 xh[kQueryBlocks], xl[kQueryBlocks];
#pragma unroll
                for (int i = 0; i < kQueryBlocks; ++i)
                    if (kg + 8 * i < nb) {
                        const bf16 *p = xp + (size_t)i * 4 * (128 * A.Mp);
                        xh[i] = __ldcg(reinterpret_cast<const uint4 *>(p));
                        xl[i] = __ldcg(reinterpret_cast<const uint4 *>(p + kLo));
                    }
                if (real) mbar_wait(smem_u32(&w_full), 0u, D.mbar_limit, D.status);
                float ah[TILES][4], al[TILES][4];
#pragma unroll
                for (int tile = 0; tile < TILES; ++tile) {
                    const char *w = w_rows + (size_t)((t0 + tile) * 16 + g) * w_pitch + t4 * 16 + kg * 64;
#pragma unroll
                    for (int q = 0; q < 4; ++q) ah[tile][q] = al[tile][q] = 0.f;
#pragma unroll
                    for (int i = 0; i < kQueryBlocks; ++i)
                        if (kg + 8 * i < nb) {
                            const uint4 a = *reinterpret_cast<const uint4 *>(w + i * 512);
                            const uint4 c = *reinterpret_cast<const uint4 *>(w + 8 * w_pitch + i * 512);
                            mma16816_bf16(ah[tile], a.x, c.x, a.y, c.y, xh[i].x, xh[i].y);
                            mma16816_bf16(al[tile], a.x, c.x, a.y, c.y, xl[i].x, xl[i].y);
                            mma16816_bf16(ah[tile], a.z, c.z, a.w, c.w, xh[i].z, xh[i].w);
                            mma16816_bf16(al[tile], a.z, c.z, a.w, c.w, xl[i].z, xl[i].w);
                        }
                }
                bar_sync<NW * 32>(1);                // the weights' place is free
#pragma unroll
                for (int tile = 0; tile < TILES; ++tile) {
                    float *o = q_sum + (size_t)(((t0 + tile) * 8 + kg) * 16 + g) * 9 + 2 * t4;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (real) o[(q >> 1) * 8 * 9 + (q & 1)] = ah[tile][q] + al[tile][q];
                }
                if (real) bar_sync<kThreads>(2);     // (and the producer's scales)
                for (int i = tid; i < DH * 8; i += NW * 32) {
                    const int m = i / DH, e = i - m * DH;
                    const float *p = q_sum + (size_t)((e >> 4) * 8 * 16 + (e & 15)) * 9 + m;
                    float v = 0.f;
#pragma unroll
                    for (int w = 0; w < 8; ++w) v += p[w * 16 * 9];
                    v = m < t_rows ? v * s_inv[m] * A.scale : 0.f;
                    __half vh, vl;
                    split_f16(v, vh, vl);
                    if (real) { q_hi[m * LDQ + e] = vh; q_lo[m * LDQ + e] = vl; }
                }
                bar_sync<NW * 32>(1);
#pragma unroll
                for (int c = 0; c < DH / 8; ++c) {
                    qh[c] = *reinterpret_cast<const unsigned *>(q_hi + g * LDQ + 8 * c + 2 * t4);
                    ql[c] = *reinterpret_cast<const unsigned *>(q_lo + g * LDQ + 8 * c + 2 * t4);
                }
            } else
#pragma unroll
            for (int c = 0; c < DH / 8; ++c) {
                qh[c] = g < t_rows && busy ? ldcg_u32(qhi + 8 * c) : 0u;
                ql[c] = g < t_rows && busy ? ldcg_u32(qlo + 8 * c) : 0u;
            }
            FewState<DH> ws;
#pragma unroll
            for (int i = 0; i < DH / 16; ++i) ws.o[i][0] = ws.o[i][1] = ws.o[i][2] = ws.o[i][3] = 0.f;
            ws.m[0] = ws.m[1] = kNegBig;
            ws.l[0] = ws.l[1] = 0.f;
            const int row_lim0 = cross ? D.C - 1 : start + 2 * t4, row_lim1 = cross ? D.C - 1 : row_lim0 + 1;
            if (all_in || !real) {
                for (int u = real ? warp : 0; u < (real ? n_units : 1); u += NW) {
                    const int i = u / upp, uu = u - i * upp, base = (p_lo + i) * P + uu * 32;
                    if (real) mbar_wait(smem_u32(&full[i]), 0u, D.mbar_limit, D.status);
                    const uint32_t kt = ring + (uint32_t)i * 2u * tile_bytes, vt = kt + (uint32_t)(i == pages - 1 ? last_rows : P) * RB;
                    few_unit<DH>(qh, ql, kt, vt, uu * 32, row_lim0 - base, row_lim1 - base, ws);
                }
            } else {
                const int stride = owned ? NW / upp : 1;
                for (int i = owned ? warp / upp : 0; i < p_hi - p_lo; i += stride) {
                    const int sl = i % slots;
                    mbar_wait(smem_u32(&full[sl]), (uint32_t)((i / slots) & 1), D.mbar_limit, D.status);
                    const uint32_t kt = ring + (uint32_t)sl * 2u * tile_bytes;
                    for (int uu = owned ? warp % upp : 0; uu < upp; uu += owned ? upp : 1) {
                        if (!owned && ((i * upp + uu) & (NW - 1)) != warp) continue;
                        const int base = (p_lo + i) * P + uu * 32;
                        if (base < n_keys) few_unit<DH>(qh, ql, kt, kt + tile_bytes, uu * 32, row_lim0 - base, row_lim1 - base, ws);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&empty[sl]));
                }
            }
            if (real) __syncthreads();   // (1)
#pragma unroll
            for (int o = 4; o <= 16; o <<= 1) {
                ws.l[0] += __shfl_xor_sync(0xffffffffu, ws.l[0], o);
                ws.l[1] += __shfl_xor_sync(0xffffffffu, ws.l[1], o);
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int r = 2 * t4 + c;
                if (real && busy && r < t_rows) {
                    float *dst = st + (warp * srows + r) * LD;
#pragma unroll
                    for (int dp = 0; dp < DH / 16; ++dp) {
                        dst[16 * dp + g] = ws.o[dp][c];
                        dst[16 * dp + g + 8] = ws.o[dp][2 + c];
                    }
                    if (g == 0) { dst[DH] = ws.m[c]; dst[DH + 1] = ws.l[c]; }
                }
            }
        } else {
            const int qt = row_tile, kg = warp / wq;
            const int r0 = qt * 16 + g, r1 = r0 + 8;
            unsigned qh[DH / 16][4], ql[DH / 16][4];
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int r = (q & 1) ? r1 : r0;
                    const size_t o = (size_t)((q & 1) * 8) * D.d + ks * 16 + (q >> 1) * 8;
                    qh[ks][q] = r < t_rows ? ldcg_u32(qhi + o) : 0u;
                    ql[ks][q] = r < t_rows ? ldcg_u32(qlo + o) : 0u;
                }
            }
            RowsState<DH> ws;
#pragma unroll
            for (int i = 0; i < DH / 8; ++i) ws.o[i][0] = ws.o[i][1] = ws.o[i][2] = ws.o[i][3] = 0.f;
            ws.m[0] = ws.m[1] = kNegBig;
            ws.l[0] = ws.l[1] = 0.f;
            const int row_lim0 = cross ? D.C - 1 : start + r0, row_lim1 = cross ? D.C - 1 : start + r1;
            const int last = cross ? D.C - 1 : start + min(qt * 16 + 15, t_rows - 1);      // last key of the row tile
            for (int i = 0; i < p_hi - p_lo; ++i) {
                const int sl = i % slots;
                mbar_wait(smem_u32(&full[sl]), (uint32_t)((i / slots) & 1), D.mbar_limit, D.status);
                const uint32_t kt = ring + (uint32_t)sl * 2u * tile_bytes;
                for (int uu = 0; uu < upp; ++uu) {
                    const int base = (p_lo + i) * P + uu * 32;
                    if (((i * upp + uu) & (kg_n - 1)) != kg || base > last || qt >= qt_n) continue;
                    rows_unit<DH>(qh, ql, kt, kt + tile_bytes, uu * 32, row_lim0 - base, row_lim1 - base, ws);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&empty[sl]));
            }
            __syncthreads();             // (1)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                ws.l[c] += __shfl_xor_sync(0xffffffffu, ws.l[c], 1);
                ws.l[c] += __shfl_xor_sync(0xffffffffu, ws.l[c], 2);
                const int r = c ? r1 : r0;
                if (r < t_rows) {
                    float *dst = st + (warp * 16 + g + 8 * c) * LD;
#pragma unroll
                    for (int dn = 0; dn < DH / 8; ++dn) {
                        dst[8 * dn + 2 * t4] = ws.o[dn][2 * c];
                        dst[8 * dn + 2 * t4 + 1] = ws.o[dn][2 * c + 1];
                    }
                    if (t4 == 0) { dst[DH] = ws.m[c]; dst[DH + 1] = ws.l[c]; }
                }
            }
        }
    }
    if (real) __syncthreads();
    // the warps' states of a row -> the output, or this CTA's partial result.  Two neighbouring columns a thread.
    bf16 *out = A.out + (size_t)set * 2 * A.Mp * D.d;
    const int states = FEW && all_in ? min(NW, n_units) : kg_n;
    const int n_pairs = t_rows * (DH / 2), step = (FEW ? srows : wq * 16) * LD;
    const float *const recv = reinterpret_cast<const float *>(smem + A.recv);      // [sender][row of this CTA][DH + 2]
    auto store = [&](int r, int c, float v0, float v1) {
        bf16 h0, l0, h1, l1;
        split_bf16(v0, h0, l0);
        split_bf16(v1, h1, l1);
        const int row = b * A.t + q0 + r;
        bf16 *p = out + (size_t)(row / kTokenTile) * 2 * A.Mp * D.d + plane_off(A.Mp, row % kTokenTile, h * DH + c);
        if (real) {
            *reinterpret_cast<__nv_bfloat162 *>(p) = __nv_bfloat162(h0, h1);
            *reinterpret_cast<__nv_bfloat162 *>(p + kLo) = __nv_bfloat162(l0, l1);
        }
    };
    for (int e = tid; e < n_pairs; e += kThreads) {
        const int r = e / (DH / 2), c = (e - r * (DH / 2)) * 2;
        float m, o0, o1, l;
        merge_states(st + r * LD, DH, c, states, step, m, l, o0, o1);      // (row r of a row tile: the tiles of the first kg follow each other)
        if (!CL || S == 1) {
            const float inv = 1.f / l;
            store(r, c, o0 * inv, o1 * inv);
        } else if (real) {
            const uint32_t slot = (uint32_t)(r / S), owner = (uint32_t)r - slot * S, rows = (uint32_t)((t_rows - (int)owner + S - 1) / S);
            const uint32_t dst = map_rank(smem_u32(recv) + ((uint32_t)rank * rows + slot) * (uint32_t)(LD * 4), owner), bar = map_rank(smem_u32(&recv_bar), owner);
            st_async_v2(dst + (uint32_t)c * 4u, o0, o1, bar);
            if (c == 0) st_async_v2(dst + DH * 4u, m, l, bar);
        }
    }
    // The CTAs of a (sequence, head) are a cluster: each takes the partial results of its share of the rows from all of them, in
    // shared memory, by counted stores, and adds them up in rank order.  (Through global memory, with a counter that told the
    // last CTA to merge, the two fences and the round trips cost 4 to 5 us.)
    if (CL && S > 1 && real && rank < t_rows) {
        const int my_rows = (t_rows - rank + S - 1) / S;
        if (!mbar_wait(smem_u32(&recv_bar), 0u, D.mbar_limit, D.status)) mbar_wait(smem_u32(&recv_bar), 0u, D.mbar_limit, D.status);
        __syncwarp();
        for (int e = tid; e < my_rows * (DH / 2); e += kThreads) {
            const int i = e / (DH / 2), c = (e - i * (DH / 2)) * 2;
            float m, o0, o1, l;
            merge_states(recv + i * LD, DH, c, S, my_rows * LD, m, l, o0, o1);
            const float inv = 1.f / l;
            store(rank + i * S, c, o0 * inv, o1 * inv);
        }
    }
    }
    trace_mark(D, 2 + 2 * A.stage);
}

// shared memory for the partial results of the cluster's CTAs: s senders, ceil(t / s) rows, for any s up to S that takes part
int attn_recv(const Dev &D, int S, int t) { return S > 1 ? (min(t, kTokenTile) + S - 1) * (D.dh + 2) * 4 : 0; }
// shared memory that the states of the warps take when the pages are done with
int attn_park(const Dev &D, int t, int warps) { return warps * (t <= 8 ? t : 16) * (D.dh + 2) * 4; }
// shared memory beside the ring of a stage whose queries the kernel projects itself; 0: not possible
int attn_query_smem(const Dev &D, int t) {
    if (t > 8 || D.d > kQueryBlocks * 8 * 32 || D.dh > 64) return 0;
    const int weights = D.dh * (D.d * 2 + 64), later = (D.dh / 16) * 8 * 16 * 9 * 4 + 2 * 8 * (D.dh + 8) * 2;
    return weights > later ? weights : later;
}

template <int DH, bool FEW, bool QP, int NW, bool CL>
static cudaError_t launch_instance(const Dev &D, const AttnArgs &args, const ChainLaunch &L) {
    void (*fn)(const Dev, const AttnArgs) = attn_kernel<DH, FEW, QP, NW, CL>;
    AttnArgs A = args;
    A.recv = A.ring + (QP ? attn_query_smem(D, A.t) : 0);
    const int smem = A.recv + attn_recv(D, A.S, A.t);
    cudaError_t e = open_kernel((const void *)fn, smem, false);
    if (e != cudaSuccess) return e;
    return L.launch(dim3(A.S, D.H, D.B * A.sets * A.qt), dim3(NW * 32 + 32), smem, A.S, (const void *)fn, D, A);
}

template <int DH, bool CL>
static cudaError_t launch_heads(const Dev &D, const AttnArgs &A, const ChainLaunch &L) {
    if (A.t > 8) return launch_instance<DH, false, false, 8, CL>(D, A, L);
    if constexpr (DH <= 64) {
        if (A.wq != nullptr) return launch_instance<DH, true, true, 16, CL>(D, A, L);
        if (A.warps == 16) return launch_instance<DH, true, false, 16, CL>(D, A, L);
    }
    return launch_instance<DH, true, false, 8, CL>(D, A, L);
}
cudaError_t launch_attn(const Dev &D, const AttnArgs &A, const ChainLaunch &L) {
    if (A.S > 1) return D.dh == 32 ? launch_heads<32, true>(D, A, L) : D.dh == 64 ? launch_heads<64, true>(D, A, L) : launch_heads<128, true>(D, A, L);
    return D.dh == 32 ? launch_heads<32, false>(D, A, L) : D.dh == 64 ? launch_heads<64, false>(D, A, L) : launch_heads<128, false>(D, A, L);
}

}  // namespace xsm
