// Projections of bf16 models on the tensor cores of the 5th generation (tcgen05), as kernels of the launch chain.
//
// y[m][u] = W[u] . x[m] for the token rows m of a step (or of a chunk of the prompt).  The weight rows are the M side of the
// product (128 rows a tile, one accumulator lane each), the token rows the N side, twice: the activations are fp32 values
// split into bf16 hi + lo, published by their writer as two planes, and the two products are added after the fact, so
// nothing of the activations is lost and a weight tile serves all token rows in one pass.  A tile's columns are cut over
// the S CTAs of a cluster (a step has at most 128 token rows, so the row tiles alone would leave most of the chip idle).
// Each of them hands the partial sums of a share of the token rows to the CTA that finishes those rows, straight from the
// accumulator (asynchronous stores that count on the receiver's barrier), and they are added in rank order: results do not
// depend on timing.
//
// A chunk of a prompt has more token rows: tiles of 128 of them, two CTAs to an SM, so that one's products run under the
// other's epilogue.
//
// Weights do not depend on the rest of the step: their copies start before the kernel waits for its predecessor.
#include "xsm_proj.cuh"

#include <cuda.h>

#include <atomic>

namespace xsm {

// CL: a tile's columns are cut over a cluster.  256 or 384 threads (plan_proj) of at most 80 registers, so that the SM has room for the next kernel's
// CTA as well (with 512 of 67 to 103 the next kernel's barriers, tensor memory and first copies came after this one's end: 20
// token rows of width 1024 961 -> 908 us a step, 80 rows 1391 -> 1397).  Without a cluster two CTAs of 512 to an SM.
constexpr int kBlockK = 64;                        // columns of one operand block (128 bytes: one swizzled row)
constexpr int kABytes = 128 * kBlockK * 2;         // weight block

struct __align__(64) ProjMaps { CUtensorMap w0, w1; };      // group 0 (or gate), group 1 (or up)

// Where a kernel starts late (its shared memory does not fit beside its predecessor's), everything up to the wait is on the step's
// way: barriers by the lanes of two warps, one cluster barrier and none of the CTA, weights requested at once, no divisions, no
// load waited for.  20 token rows of width 1024 908 -> 766 us a step, 80 rows 1397 -> 1274, 28 rows of width 2048 2453 -> 2071 (with
// the products issued by an elected lane and six shuffles for the sums of squares of four rows).
//
// A chain of instructions bounds it at few token rows (nine cycles each): where every operand block has a place of its own, the
// activations count on one barrier and the issuing warp adds to two descriptors; with a barrier and two commits a block, a block
// took 0.28 us, eight of them more than the weights' way from memory (5 rows of width 1024 683 -> 631 us a step).
// G: token rows of a group that is sent and finished together (plan_proj).
// MANY: the CTA's blocks are added up in accumulators of A.chain blocks each, side by side in tensor memory, and these in fp32 here
// (plan_proj).  The price is code as much as work: 5 rows of width 1024 611 -> 615 us a step, 7 of width 2048 1647 -> 1691.  Fetching
// one while the tensor core fills the next, two at a time, or sending each by itself is 1.5 to 4 % slower.
template <int EPI0, int EPI1, bool CL, int G, bool MANY>
__global__ void __launch_bounds__(CL ? kClusterThreads : kTileThreads, 2) proj_umma_kernel(const Dev D, const ProjArgs A, const __grid_constant__ ProjMaps T) {
    extern __shared__ char smem_raw[];
    char *const smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);      // (swizzled tiles: 1024-byte boundaries)
    __shared__ __align__(8) uint64_t bars[4 * kProjRing + 1];      // A full, A empty, B full, B empty, done
    __shared__ __align__(8) uint64_t recv_bar;                      // the peers' shares of this CTA's token rows
    __shared__ uint32_t tmem_slot;
    __shared__ float s_inv[kTokenTile];
    __shared__ RowInfo s_row[kTokenTile];
    static_assert(sizeof(bars) + sizeof(s_inv) >= kProjDeclared, "plan_proj counts on that much");
    static_assert(sizeof(bars) + sizeof(recv_bar) + sizeof(s_inv) + (EPI0 == PE_QKV ? sizeof(s_row) : 0) + 64 + proj_smem_max(EPI0) <= kCtaSmem,
                  "a ring that is as large as plan_proj allows has to fit");
    constexpr bool TWO = EPI0 == PE_GATEUP;
    const int threads = CL && G == 1 ? (int)blockDim.x : CL ? kClusterThreads : kTileThreads;
    // Of eight warps the first four fetch, multiply and set up (and take the second part of an accumulator of two, more than eight token
    // rows); the others take its first part and the first token rows.  Of twelve the first four do both.
    const bool apart = CL && G == 1 && threads == 256;
    const int tmem_warp = apart ? 3 : (threads >> 5) - 1;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;      // (the warp's number: uniform, also to the compiler)
    const int S = CL ? A.S : 1, rank = CL ? (int)cluster_rank() : 0, Mp = A.Mp;
    // sequences that still run: looked at just before the wait, when the weights are on their way
    const int active = A.pos0 < 0 && !A.late_go ? __ldcg(D.n_active) : 1;
    // a tile of weight rows and a tile of token rows: neighbours share the weights
    // (divisions only where there is something to divide: 90 cycles each, on the way of a kernel that starts late)
    int tile = CL ? (int)cluster_index() : (int)blockIdx.x, token_tile = 0, plane = 0, job = 0, z = A.layer, grp = 0;
    if (A.tt > 1) {
        const int t = tile / A.tt;
        token_tile = tile - t * A.tt;
        tile = t;
        plane = token_tile * A.tok / Mp;
    }
    const int mb = token_tile * A.tok, rows = min(A.tok, A.rows - mb), pm = mb - plane * Mp, Nt = min(A.tok, Mp - pm);      // plane set, first row there; rows with padding
    if (EPI1 >= 0 && tile >= A.g[0].tiles) {
        tile -= A.g[0].tiles;
        grp = 1;
    }
    const ProjGroup &W = A.g[grp];
    if (EPI1 >= 0 || A.z_jobs) {          // the matrices of a group (one per decoding head) share its map, one behind the other
        z = job = grp == 1 || A.z_jobs ? tile / W.job_tiles : 0;
        tile -= job * W.job_tiles;
    }
    const int u0 = tile * (TWO ? 64 : 128);
    const int nblk = A.kdim / kBlockK, k_lo = (int)((uint32_t)(rank * nblk) * A.inv_s >> 16), n = (int)((uint32_t)((rank + 1) * nblk) * A.inv_s >> 16) - k_lo;
    const int na = A.na, nb = A.nb;
    const bool flat = na >= n && nb >= n;      // every block has a place of its own: the activations count on one barrier, nothing is given back
    const int qps = A.tps / G, m0 = rank * A.tps, nm = min(A.tps, rows - m0);      // token rows that this CTA finishes (nm may be <= 0)
    const uint32_t b_bytes = (uint32_t)(2 * Nt) * kBlockK * 2u, b_pitch = (uint32_t)(2 * A.tok) * kBlockK * 2u;
    // operand rings; behind them (one CTA to a tile: in their place, when the products are done) the partial sums
    const uint32_t sa = smem_u32(smem), sb = sa + (uint32_t)na * kABytes, srecv = CL ? sb + (uint32_t)nb * b_pitch : sa;
    float *recv = reinterpret_cast<float *>(smem + (srecv - sa));
    auto bar = [&](int kind, int i) { return smem_u32(&bars[kind * kProjRing + i]); };
    const uint32_t done = smem_u32(&bars[4 * kProjRing]);
    const void *wmap = grp == 1 ? &T.w1 : &T.w0;
    auto load_a = [&](int i, int slot) {
        const uint32_t dst = sa + (uint32_t)slot * kABytes, b = bar(0, slot);
        const int x = (k_lo + i) * kBlockK;
        mbar_arrive_expect_tx(b, kABytes);
        if (TWO) {
            tma_box(dst, &T.w0, x, u0, z, b);
            tma_box(dst + kABytes / 2, &T.w1, x, u0, z, b);
        } else {
            tma_box(dst, wmap, x, u0, z, b);
        }
    };
    // Barriers by the lanes of two warps, tensor memory by a third.  (The tensor memory is taken before the next kernel may start:
    // kernels further down the chain can then never hold columns that this one still waits for.)
    if (warp == 0) {
        if (lane < na) { mbar_init(bar(0, lane), 1u); mbar_init(bar(1, lane), 1u); }
        mbar_init_fence();
    } else if (warp == 1) {
        if (lane < nb) { mbar_init(bar(2, lane), 1u); mbar_init(bar(3, lane), 1u); }
        if (lane == 31) {
            mbar_init(done, (uint32_t)(threads >> 5) - 1u);      // the last products, and what the epilogue needs to know (warps 2 and up)
            mbar_init(smem_u32(&recv_bar), 1u);
        }
        mbar_init_fence();
        if (CL && lane == 31 && nm > 0) mbar_arrive_expect_tx(smem_u32(&recv_bar), (uint32_t)(S * ((nm + G - 1) / G)) * (512u * G));
    } else if (warp == tmem_warp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&tmem_slot)), "r"(A.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        if (!A.late_go) chain_go();
    }
    __syncwarp();
    // "this CTA runs": its barriers are there (mbar_init_fence), and peers may write to its shared memory, after cluster_wait.  A release
    // would wait for the load above, and hold back the weights' copies, which a kernel that starts late waits for: 5 rows of width 768
    // 33.91 -> 33.57 ms a request, of width 1024 57.23 -> 56.48, 20 rows 38.21 -> 36.98, 7 rows of width 2048 58.89 -> 58.05.
    if (CL) cluster_arrive_relaxed();
    if (warp == 0 && elect_one())      // the weights' way is the longest: it begins as early as that
        for (int i = 0; i < min(n, na); ++i) load_a(i, i);
    __syncwarp();
    if (A.stage == 0) trace_mark(D, 0);
    const bf16 *x = A.x + (size_t)(A.x_jobs ? job : plane) * 2 * Mp * A.kdim;
    const bf16 *xb = x + (size_t)k_lo * (128 * Mp) + (size_t)pm * 128;      // this CTA's blocks of the activations
    const uint32_t idesc = umma_idesc(128, 2 * Nt), full_a = bar(0, 0), full_b = bar(2, 0);
    settle(xb);
    constexpr int ROWS = TWO ? 64 : 128;
    const int sides = threads / ROWS;
    constexpr bool HEAD = EPI0 == PE_HEADADD || EPI1 == PE_HEADY;
    const int place = apart ? tid ^ 128 : tid;
    const int row = tid & (ROWS - 1), side = place / ROWS, u_row = u0 + row, half = D.dh >> 1, e = row & (D.dh - 1);
    const bool live_row = u_row < W.units;
    const uint32_t gain_bits = (EPI0 == PE_ADD || HEAD) && u_row < D.d ? ld_early_u16(reinterpret_cast<const bf16 *>(A.gain) + u_row) : 0u;
    // where this thread's weight row goes
    const int sec = EPI0 == PE_QKV ? (u_row >= D.d ? (u_row >= 2 * D.d ? 2 : 1) : 0) : 0, col = u_row - sec * D.d, head = EPI0 == PE_QKV ? col >> (31 - __clz(D.dh)) : 0;      // (d_head is 32, 64 or 128)
    __half *qrow = A.q + ((size_t)job * 2 * A.qp + mb) * D.d + (EPI0 == PE_QKV ? col : u_row);
    bf16 *xrow = W.out + (size_t)(job + plane) * 2 * Mp * W.ld + (size_t)(u_row >> 6) * (128 * Mp) + (size_t)pm * 128 + (u_row & 7);
    const int xchunk = (u_row >> 3) & 7;
    float *lrow = W.logits + ((size_t)job * D.M + mb) * W.ld + u_row;
    __half *crow = reinterpret_cast<__half *>(D.kv_pool) + ((size_t)(A.layer * 2 + (sec == 2 ? 1 : 0)) * D.n_pages * D.H + head) * (size_t)D.P * D.dh + (e & 7);
    settle(qrow); settle(xrow); settle(lrow); settle(crow);
    // Accumulator -> the CTA that finishes the token rows: [sender][group][weight row][G].  This thread's lane of the accumulator
    // is its weight row; eight token rows at a time, from c0 on.
    constexpr int GROUPS = 8 / G;
    const int lanes = warp & 3, arow = lanes * 32 + lane, c0 = place >> 7;
    const uint32_t recv_b = smem_u32(&recv_bar);
    uint32_t dst[GROUPS], dst_bar[GROUPS];
    auto where = [&](int c) {
#pragma unroll
        for (int q = 0; q < GROUPS; ++q) {
            if (CL && G > 1 && (GROUPS * c + q) * G >= rows) continue;      // (token rows one by one: the branch costs more than it saves)
            const int group = GROUPS * c + q, owner = (int)((uint32_t)group * A.inv_q >> 16), place = rank * qps + group - owner * qps;      // (group / qps: both are below 33)
            dst[q] = CL ? map_rank(srecv + (uint32_t)(place * 128 + arow) * (4u * G), (uint32_t)min(owner, S - 1)) : (uint32_t)(group * 128 + arow) * (4u * G);
            dst_bar[q] = CL ? map_rank(recv_b, (uint32_t)min(owner, S - 1)) : recv_b;
        }
    };
    where(c0);
#pragma unroll
    for (int q = 0; q < GROUPS; ++q) { settle(dst[q]); settle(dst_bar[q]); }
    tcgen05_before_sync();
    if (CL) cluster_wait();            // the peers run: their barriers and shared memory are there
    else __syncthreads();
    tcgen05_after_sync();
    if (warp > 0) asm volatile("bar.sync 1, %0;" :: "r"(threads - 32) : "memory");      // (warps that come to the wait together leave it sooner)
    chain_wait();
    if (active == 0) {      // every sequence has ended in an earlier step
        if (tid == 0)
            for (int i = 0; i < min(n, na); ++i) mbar_wait(bar(0, i), 0u, D.mbar_limit, D.status);
        __syncthreads();
        if (warp == tmem_warp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_slot), "r"(A.tmem_cols) : "memory");
        return;
    }
    if (A.late_go) chain_go();
    trace_mark(D, 1 + 2 * A.stage);
    if (warp == 0) {
        // (written by ordinary stores of an earlier kernel, which has completed: nothing to order)
        if (flat) {
            if (lane == 0) mbar_arrive_expect_tx(full_b, (uint32_t)n * b_bytes);
            __syncwarp();
        }
        if (lane < min(n, nb)) {
            const uint32_t f = flat ? full_b : full_b + 8u * (uint32_t)lane;
            if (!flat) mbar_arrive_expect_tx(f, b_bytes);
            bulk_g2s(sb + (uint32_t)lane * b_pitch, xb + (size_t)lane * (128 * Mp), b_bytes, f);
        }
        __syncwarp();
        if (elect_one()) {
            int slot = 0, a_slot = 0;
            uint32_t par = 0u, a_par = 0u;
            for (int i = flat ? n : min(na, nb); i < n; ++i) {
                if (i >= nb) {
                    mbar_wait(bar(3, slot), par, D.mbar_limit, D.status);
                    mbar_arrive_expect_tx(full_b + 8u * (uint32_t)slot, b_bytes);
                    bulk_g2s(sb + (uint32_t)slot * b_pitch, xb + (size_t)i * (128 * Mp), b_bytes, full_b + 8u * (uint32_t)slot);
                    if (++slot == nb) { slot = 0; par ^= 1u; }
                }
                if (i >= na) {
                    mbar_wait(bar(1, a_slot), a_par, D.mbar_limit, D.status);
                    load_a(i, a_slot);
                    if (++a_slot == na) { a_slot = 0; a_par ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // (the whole warp waits and one elected lane issues: a branch on the thread's number would keep the descriptors out of the
        // uniform registers that the instruction takes them from)
        const bool leader = elect_one();
        const uint64_t da = umma_desc_sw128(sa), db = umma_desc_sw128(sb);
        auto products = [&](uint32_t sum, int ia, int ib, bool add) {
            const uint64_t a = da + (uint64_t)(ia * (kABytes >> 4)), b = db + (uint64_t)((uint32_t)ib * (b_pitch >> 4));
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) umma_mma(sum, a + 2 * ks, b + 2 * ks, idesc, (add || ks > 0) ? 1u : 0u);
        };
        // (one loop with a counter: a loop for each accumulator around one for its blocks costs 2 % of a step where rings are refilled)
        uint32_t sum = tmem_slot;
        int held = 0;      // blocks in the accumulator
        auto next_sum = [&]() {
            if (!MANY) held = 1;
            else if (++held == A.chain) { held = 0; sum += (uint32_t)(2 * Nt); }
        };
        if (flat) {
            mbar_wait(full_b, 0u, D.mbar_limit, D.status);
            for (int i = 0; i < n; ++i) {
                mbar_wait(full_a + 8u * (uint32_t)i, 0u, D.mbar_limit, D.status);
                tcgen05_after_sync();
                if (leader) products(sum, i, i, held > 0);
                next_sum();
            }
        } else {
            const uint32_t empty_a = bar(1, 0), empty_b = bar(3, 0);
            int ia = 0, ib = 0;
            uint32_t pa = 0u, pb = 0u;
            for (int i = 0; i < n; ++i) {
                mbar_wait(full_a + 8u * (uint32_t)ia, pa, D.mbar_limit, D.status);
                mbar_wait(full_b + 8u * (uint32_t)ib, pb, D.mbar_limit, D.status);
                tcgen05_after_sync();
                if (leader) {
                    products(sum, ia, ib, held > 0);
                    if (i + na < n) umma_commit(empty_a + 8u * (uint32_t)ia);
                    if (i + nb < n) umma_commit(empty_b + 8u * (uint32_t)ib);
                }
                next_sum();
                if (++ia == na) { ia = 0; pa ^= 1u; }
                if (++ib == nb) { ib = 0; pb ^= 1u; }
                __syncwarp();      // (a lane two fills of a slot behind the leader would wait for a phase that has gone by)
            }
        }
        if (leader) umma_commit(done);
        __syncwarp();
    }
    // meanwhile: what the epilogue needs to know of the token rows that this CTA finishes
    if (warp >= 2) {
        for (int i = tid - 64; i < nm; i += threads - 64) {
            const int m = m0 + i;
            float inv = 1.f;
            if (A.ss_parts > 0) {
                float ss = 0.f;
                const float4 *sh = reinterpret_cast<const float4 *>(D.ss + (size_t)(mb + m) * kShareLd);
                for (int p0 = 0; p0 < A.ss_parts; p0 += 32) {        // 32 shares in flight, added in order
                    float4 v[8];
#pragma unroll
                    for (int p = 0; p < 8; ++p) v[p] = p0 + 4 * p < A.ss_parts ? __ldcg(sh + (p0 >> 2) + p) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        const int k = A.ss_parts - p0 - 4 * p;       // (the last quad may hold shares that nobody writes)
                        ss += (v[p].x + (k > 1 ? v[p].y : 0.f)) + ((k > 2 ? v[p].z : 0.f) + (k > 3 ? v[p].w : 0.f));
                    }
                }
                inv = 1.0f / sqrtf(ss / (float)D.d + D.eps);
            }
            s_inv[i] = inv;
            if (EPI0 == PE_QKV) *reinterpret_cast<int4 *>(&s_row[i]) = __ldcg(reinterpret_cast<const int4 *>(D.row_info + mb + m));
        }
    }
    // The epilogue: thread = weight row, the token rows of this CTA are dealt out to the `sides` threads of a weight row in groups of
    // G, which lie side by side in shared memory: up to 24 rows one by one, else four (one 16-byte load for each sender; four single
    // ones met four-way bank conflicts, half of an epilogue's time at 80 token rows); what it reads from memory is requested before
    // the products are waited for, or a round ahead.
    float hn[G];
    float2 csn[G];
    auto request = [&](int group) {
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const int i = G * group + q;
            if ((EPI0 == PE_ADD || HEAD) && i < nm && live_row && u_row < D.d) hn[q] = __ldcg(D.h + (size_t)(mb + m0 + i) * D.d + u_row);
            if (EPI0 == PE_QKV && i < nm) csn[q] = __ldcg(D.row_cs + (size_t)(mb + m0 + i) * half + (e < half ? e : e - half));
        }
    };
    __syncwarp();
    if (warp >= 2 && lane == 0) mbar_arrive(done);
    const float gain = __uint_as_float(gain_bits << 16);
    request(side);
    // (warps with neither a part of the accumulator nor token rows wait for nothing more: 5 rows of width 768 33.94 -> 33.57 ms a request,
    // of width 1024 56.93 -> 56.48, 20 rows 37.23 -> 36.98, 7 rows of width 2048 58.42 -> 58.05)
    const bool part = !CL || (c0 << 3) < Nt || G * side < nm;
    const bool done_ok = !part || mbar_wait(done, 0u, D.mbar_limit, D.status);
    __syncwarp();
    tcgen05_after_sync();
    const uint32_t tmem = tmem_slot;      // (its warp has arrived at `done`)
    for (int c = c0; c < (Nt >> 3); c += threads >> 7) {      // hi and lo parts added
        uint32_t v[16];
        tmem_ld16(v, tmem + ((uint32_t)(lanes * 32) << 16) + (uint32_t)c * 16u);
        if (c != c0) where(c);
        tmem_wait_ld();
        float sums[8];
        if constexpr (MANY) {
#pragma unroll
            for (int j = 0; j < 8; ++j) sums[j] = __uint_as_float(v[j]) + __uint_as_float(v[8 + j]);
            uint32_t at = tmem + ((uint32_t)(lanes * 32) << 16) + (uint32_t)c * 16u;
#pragma unroll 1
            for (int k = A.chain; k < n; k += A.chain) {
                at += (uint32_t)(2 * Nt);
                tmem_ld16(v, at);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) sums[j] += __uint_as_float(v[j]) + __uint_as_float(v[8 + j]);
            }
        }
#pragma unroll
        for (int q = 0; q < GROUPS; ++q) {
            if ((GROUPS * c + q) * G < rows) {
                float f[G];
#pragma unroll
                for (int j = 0; j < G; ++j) f[j] = MANY ? sums[G * q + j] : __uint_as_float(v[G * q + j]) + __uint_as_float(v[8 + G * q + j]);
                if constexpr (G == 1) {
                    if (done_ok) st_async_f32(dst[q], f[0], dst_bar[q]);      // (a peer that gave up waiting may have left)
                } else {
                    if (!CL) *reinterpret_cast<float4 *>(smem + (srecv - sa) + dst[q]) = make_float4(f[0], f[1], f[2], f[3]);
                    else if (done_ok) st_async_v4(dst[q], f, dst_bar[q]);
                }
            }
        }
    }
    tcgen05_before_sync();
    // The tensor memory goes back while the shares are on their way (at the kernel's end it kept the next one waiting: 5 rows of width
    // 768 35.14 -> 33.57 ms a request, of width 1024 58.04 -> 56.48, 20 rows 38.24 -> 36.98, 7 rows of width 2048 58.95 -> 58.05).  Behind the
    // barrier every product has been issued.  This warp waits for them itself: it may not have done so before, and others may have
    // given up waiting (and have raised the status), and another CTA must not get columns that products are still added to.  (0 to 0.3 %
    // of a request; with the status raised here as well, which is code for nothing, to 0.6 %.)
    if (warp != tmem_warp) {
        asm volatile("bar.arrive 2, %0;" :: "r"(threads) : "memory");
    } else {
        asm volatile("bar.sync 2, %0;" :: "r"(threads) : "memory");
        for (unsigned i = 0; !mbar_try_wait(done, 0u) && i < D.mbar_limit; ++i);
        __syncwarp();
        tcgen05_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(A.tmem_cols) : "memory");
    }
    // One CTA to a tile: a barrier.  In a cluster every CTA waits for all shares of its rows, its own among them, so none leaves
    // before what is sent to it has come: no barrier at the end, whose wait for all stores took 1600 to 2400 cycles.
    if (!CL) __syncthreads();
    else if (G * side < nm && !mbar_wait(recv_b, 0u, D.mbar_limit, D.status)) mbar_wait(recv_b, 0u, D.mbar_limit, D.status);
    __syncwarp();
    // sums over the cluster in rank order, epilogue
    auto total = [&](int group, int r, float (&v)[G]) {
        constexpr int kMost = CL ? 8 : 1;
        if constexpr (G == 1) {
            const float *p = recv + group * 128 + r;
            float part[kMost];
#pragma unroll
            for (int s = 0; s < kMost; ++s) part[s] = s < S ? p[s * qps * 128] : 0.f;
            v[0] = part[0];
#pragma unroll
            for (int s = 1; s < kMost; ++s) v[0] += part[s];
        } else {
            const float4 *p = reinterpret_cast<const float4 *>(recv) + group * 128 + r;
            float4 part[kMost];
#pragma unroll
            for (int s = 0; s < kMost; ++s) part[s] = s < S ? p[s * qps * 128] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int s = 1; s < kMost; ++s) { part[0].x += part[s].x; part[0].y += part[s].y; part[0].z += part[s].z; part[0].w += part[s].w; }
            v[0] = part[0].x; v[1] = part[0].y; v[2] = part[0].z; v[3] = part[0].w;
        }
    };
    auto put_x = [&](int m, float v) {
        bf16 hi, lo;
        split_bf16(v, hi, lo);
        bf16 *p = xrow + (m >> 3) * 1024 + (m & 7) * 64 + ((xchunk ^ (m & 7)) << 3);
        p[0] = hi;
        p[512] = lo;
    };
    auto put_q = [&](int m, float v) {
        __half hi, lo;
        split_f16(v * A.scale, hi, lo);
        qrow[(size_t)m * D.d] = hi;
        qrow[(size_t)(A.qp + m) * D.d] = lo;
    };
    for (int group = side; G * group < nm; group += sides) {
        float h[G];
        float2 cs[G];
#pragma unroll
        for (int q = 0; q < G; ++q) { h[q] = hn[q]; cs[q] = csn[q]; }
        request(group + sides);
        float sum[G], other[G];      // other: the rotation partner's, or up's
        total(group, row, sum);
        if (TWO) total(group, row + 64, other);
        if (EPI0 == PE_QKV) total(group, e < half ? row + half : row - half, other);
        if (EPI0 == PE_ADD) {
            float o[G];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                const int i = G * group + q, m = m0 + i;
                o[q] = live_row && i < nm ? h[q] + sum[q] : 0.f;
                if (live_row && i < nm) {
                    D.h[(size_t)(mb + m) * D.d + u_row] = o[q];
                    put_x(m, o[q] * gain);
                }
                o[q] *= o[q];
            }
            if constexpr (G == 1) {
                const float v = warp_sum(o[0]);
                if (lane == 0) D.ss[(size_t)(mb + m0 + group) * kShareLd + tile * 4 + (row >> 5)] = v;
            } else {
                // the warp's sums of the four rows: a lane keeps two of them after the first exchange, one after the second (six
                // shuffles instead of twenty, 38 cycles each); lane 8 r has row r
                const bool up = lane & 16, mid = lane & 8;
                float a = up ? o[2] : o[0], b = up ? o[3] : o[1];
                a += __shfl_xor_sync(0xffffffffu, up ? o[0] : o[2], 16);
                b += __shfl_xor_sync(0xffffffffu, up ? o[1] : o[3], 16);
                float v = mid ? b : a;
                v += __shfl_xor_sync(0xffffffffu, mid ? a : b, 8);
#pragma unroll
                for (int k = 4; k > 0; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
                const int i = G * group + (lane >> 3);
                if ((lane & 7) == 0 && i < nm) D.ss[(size_t)(mb + m0 + i) * kShareLd + tile * 4 + (row >> 5)] = v;
            }
        } else
#pragma unroll
        for (int q = 0; q < G; ++q) {
            const int i = G * group + q, m = m0 + i;
            if (i >= nm) break;
            const float v = sum[q];
            if (live_row) {
                const float inv = s_inv[i], x1 = v * inv;
                if (EPI0 == PE_QKV) {
                    const float x2 = other[q] * inv, o = sec == 2 ? x1 : e < half ? x1 * cs[q].x - x2 * cs[q].y : x1 * cs[q].x + x2 * cs[q].y;
                    if (sec == 0) put_q(m, o);
                    else if (s_row[i].place >= 0) crow[s_row[i].place + (((e >> 3) ^ row_swz(s_row[i].rp, D.dh)) << 3)] = from_f<__half>(o);
                } else if (TWO) {
                    put_x(m, silu_f(x1) * (other[q] * inv));
                } else if (EPI0 == PE_QUERY || (EPI1 == PE_QUERY && grp == 1)) {
                    put_q(m, x1);
                } else if (EPI0 == PE_HEADADD) {
                    put_x(m, h[q] * inv * gain + v);
                } else if (EPI1 == PE_HEADY && grp == 1) {
                    put_x(m, h[q] * inv * gain + silu_f(x1));
                } else {
                    lrow[(size_t)m * W.ld] = A.norm ? x1 : v;
                }
            }
        }
    }
    if (D.trace != nullptr) {
        __syncthreads();
        trace_mark(D, 2 + 2 * A.stage);
    }
}

template <int EPI0, int EPI1, bool CL, int G, bool MANY>
static cudaError_t launch_instance(const Dev &D, const ProjArgs &A, const ProjMaps &T, int smem, const ChainLaunch &L) {
    void (*fn)(const Dev, const ProjArgs, const ProjMaps) = proj_umma_kernel<EPI0, EPI1, CL, G, MANY>;
    cudaError_t e = open_kernel((const void *)fn, smem, false);
    if (e != cudaSuccess) return e;
    const int tiles = A.g[0].tiles + (EPI1 >= 0 ? A.g[1].tiles : 0);
    return L.launch(dim3(tiles * A.tt * A.S), dim3(A.threads), smem, A.S, (const void *)fn, D, A, T);
}

template <int EPI0, int EPI1, bool MANY>
static cudaError_t launch_sums(const Dev &D, const ProjArgs &A, const ProjMaps &T, int smem, const ChainLaunch &L) {
    if (A.S == 1) return launch_instance<EPI0, EPI1, false, 4, MANY>(D, A, T, smem, L);
    return A.group == 1 ? launch_instance<EPI0, EPI1, true, 1, MANY>(D, A, T, smem, L) : launch_instance<EPI0, EPI1, true, 4, MANY>(D, A, T, smem, L);
}
template <int EPI0, int EPI1>
static cudaError_t launch_cut(const Dev &D, const ProjArgs &A, const ProjMaps &T, int smem, const ChainLaunch &L) {
    return A.many ? launch_sums<EPI0, EPI1, true>(D, A, T, smem, L) : launch_sums<EPI0, EPI1, false>(D, A, T, smem, L);
}

// (asked for once per device: the answer does not change, and asking takes longer than the rest of a context's creation)
int resident_clusters(int size) {
    static std::atomic<int> known[kMaxDevices][9];      // the answer + 1
    int dev = 0;
    if (size < 2 || size > 8 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
    if (const int k = known[dev][size].load()) return k - 1;
    const void *fn = (const void *)proj_umma_kernel<PE_ADD, -1, true, 4, false>;
    constexpr int smem = 200 * 1024;
    int n = 0;
    cudaLaunchConfig_t c = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)size;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    c.gridDim = dim3(size);
    c.blockDim = dim3(kClusterThreads);
    c.dynamicSmemBytes = smem;
    c.attrs = &at;
    c.numAttrs = 1;
    if (open_kernel(fn, smem, false) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, fn, &c) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    known[dev][size].store(n + 1);
    return n;
}

cudaError_t launch_proj_umma(const Dev &D, const ProjArgs &A, const void *maps, int smem, const ChainLaunch &L) {
    const ProjMaps &T = *reinterpret_cast<const ProjMaps *>(maps);
#define XSM_EPI(a, b) if (A.epi0 == a && A.epi1 == b) return launch_cut<a, b>(D, A, T, smem, L)
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

}  // namespace xsm
