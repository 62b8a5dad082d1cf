// Device helpers shared by the kernels of the launch chain: PTX wrappers, number formats, the random numbers, cache tiles.
#pragma once
#include "xsm_internal.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

namespace xsm {

typedef __nv_bfloat16 bf16;

constexpr int XSM_STATUS_TIMEOUT = 5, XSM_STATUS_CAPACITY = 3;
constexpr float kNegBig = -1.0e30f;            // "no key seen yet" (finite, so that differences of two of them are zero)

// ------------------------------------------------------------------------------ chain of launches

// Every kernel of the chain is launched with programmatic stream serialization: it may start while its predecessor
// still runs, does what does not depend on it (barriers, weights on their way to shared memory), and calls chain_wait
// before the first access to anything that an earlier kernel of the step writes or still reads.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// lets the next kernel of the chain be launched as soon as every CTA of this one has said so
__device__ __forceinline__ void chain_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// barrier `id` (not 0) of the first N threads of a block
template <int N> __device__ __forceinline__ void bar_sync(int id) { asm volatile("bar.sync %0, %1;" :: "r"(id), "n"(N) : "memory"); }
// Keeps a value from being computed later than here (the compiler would put address arithmetic behind the wait, where it is
// on the step's critical path).
template <typename T> __device__ __forceinline__ void settle(T *&p) { asm volatile("" : "+l"(p)); }
__device__ __forceinline__ void settle(int &v) { asm volatile("" : "+r"(v)); }
__device__ __forceinline__ void settle(uint32_t &v) { asm volatile("" : "+r"(v)); }
__device__ __forceinline__ void settle(float &v) { asm volatile("" : "+f"(v)); }
// sixteen bits that no kernel writes, requested here and not later (and, unlike with settle, not waited for)
__device__ __forceinline__ uint32_t ld_early_u16(const void *p) {
    uint16_t v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// true in one lane of the warp
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// ------------------------------------------------------------------------- shared memory, barriers

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Waits for the phase of the given parity, bounded: when `limit` tries run out the status word is raised and the caller goes
// on (its results are then void; the host reports the timeout).
// (false: the limit ran out)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned limit, int *status) {
    if (mbar_try_wait(bar, parity)) return true;
    for (unsigned n = 0; n < limit; ++n)
        if (mbar_try_wait(bar, parity)) return true;
    atomicExch(status, XSM_STATUS_TIMEOUT);
    return false;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// 16 bytes into the shared memory of a CTA of the cluster, counted on a barrier there
__device__ __forceinline__ void st_async_v4(uint32_t dst, const float (&v)[4], uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 :: "r"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async_v2(uint32_t dst, float a, float b, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];"
                 :: "r"(dst), "f"(a), "f"(b), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async_f32(uint32_t dst, float v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" :: "r"(dst), "f"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

constexpr int kTraceCtas = 256;      // columns of a step's timeline
// timeline of a step (inspection): one thread notes the time in the CTA's column
__device__ __forceinline__ void trace_mark(const Dev &D, int row) {
    if (D.trace == nullptr || threadIdx.x != 0) return;
    const unsigned cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    if (cta < (unsigned)kTraceCtas) D.trace[(size_t)row * kTraceCtas + cta] = global_ns();
}

// ------------------------------------------------------------------------------- thread-block clusters

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_index() {
    uint32_t r;
    asm volatile("mov.u32 %0, %clusterid.x;" : "=r"(r));
    return r;
}
// For threads that have written nothing that others read, barriers made known by mbar_init_fence apart: a release waits for all
// that the thread has under way, loads from memory among it.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// shared-memory address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

// ------------------------------------------------------------------------------------- number formats

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(bf16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_f(__half v) { return __half2float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ __half from_f<__half>(float v) { return __float2half_rn(fminf(fmaxf(v, -65504.f), 65504.f)); }

// (bf16 models keep cached keys and values in fp16: the same two bytes, eleven bits of mantissa instead of eight; they are
// normalised activations times small weights, far inside the fp16 range; stores saturate.  Rounding of the cache is the
// largest error of the whole path.)
__device__ __forceinline__ float silu_f(float v) { return v / (1.0f + expf(-v)); }
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// x = hi + lo with hi, lo bf16: 16 mantissa bits of x survive, products with bf16 weights stay exact in fp32.
__device__ __forceinline__ void split_bf16(float x, bf16 &hi, bf16 &lo) {
    hi = __float2bfloat16_rn(x);
    lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}
// x = hi + lo with hi, lo fp16 (operands of the attention products)
__device__ __forceinline__ void split_f16(float x, __half &hi, __half &lo) {
    hi = from_f<__half>(x);
    lo = __float2half_rn(x - __half2float(hi));
}
// 2^x for the online softmax (x <= 0 or -inf): the hardware approximation, 2 ulp
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// two values rounded to fp16, first in the low half
__device__ __forceinline__ unsigned pack_f16x2(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const unsigned *>(&h);
}

// ------------------------------------------------------------------------- warp-level matrix products

__device__ __forceinline__ void mma16816_bf16(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma16816_f16(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4(unsigned (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(unsigned (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ unsigned movmatrix_trans(unsigned a) {
    unsigned d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}

// --------------------------------------------------------------------------------------- tcgen05

// K-major operand tile with the 128-byte swizzle: rows of 64 bf16 (128 bytes), 8-row groups 1024 bytes apart (stride byte
// offset), leading byte offset unused (1), descriptor version of sm_100, layout type 2.  The tile starts on a 1024-byte
// boundary; a K = 16 step inside the 64 columns is 32 bytes further.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, both K-major, N and M of the tile
__device__ __forceinline__ uint32_t umma_idesc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_mma(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 :: "r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
// one arrival at the barrier when every product issued by this thread so far has completed
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(bar) : "memory");
}
// box {columns, rows, 1} of a tensor map -> shared memory (swizzled as the map says), completion on an mbarrier
__device__ __forceinline__ void tma_box(uint32_t dst, const void *tmap, int x, int y, int z, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 :: "r"(dst), "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
__device__ __forceinline__ void tcgen05_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tcgen05_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// sixteen consecutive accumulator columns of this thread's lane
__device__ __forceinline__ void tmem_ld16(uint32_t (&v)[16], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                   "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------------- random numbers

// Philox4x32-10 (Salmon et al., SC'11): returns word 0.
__device__ __forceinline__ uint32_t philox_word0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                                 uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t h0 = __umulhi(0xD2511F53u, c0), l0 = 0xD2511F53u * c0;
        uint32_t h1 = __umulhi(0xCD9E8D57u, c2), l1 = 0xCD9E8D57u * c2;
        uint32_t n0 = h1 ^ c1 ^ k0, n2 = h0 ^ c3 ^ k1;
        c0 = n0; c1 = l1; c2 = n2; c3 = l0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    return c0;
}

// -------------------------------------------------------------------------------------- cache tiles

// One (page, head) tile holds P rows (positions) of dh elements.  16-bit tiles are stored with their 16-byte chunks
// permuted so that ldmatrix over 8 consecutive rows touches every bank once; fp32 tiles are stored plain.
template <typename KVT>
__device__ __forceinline__ KVT *kv_tile(const Dev &D, void *pool, int pool_pages, int layer, int kv, int page, int head) {
    return reinterpret_cast<KVT *>(pool) + ((((size_t)layer * 2 + kv) * pool_pages + page) * D.H + head) * (size_t)D.P * D.dh;
}
// physical 16-byte chunk of logical chunk c of row r, rows of row_bytes
__device__ __forceinline__ int swz(int r, int c, int row_bytes) {
    return row_bytes >= 128 ? (c ^ (r & 7)) : (c ^ ((r >> 1) & 3));
}
// element offset of (row r, element e) inside a tile
template <typename KVT> __device__ __forceinline__ size_t tile_off(int r, int e, int dh);
template <> __device__ __forceinline__ size_t tile_off<float>(int r, int e, int dh) { return (size_t)r * dh + e; }
template <> __device__ __forceinline__ size_t tile_off<__half>(int r, int e, int dh) {
    return (size_t)r * dh + (size_t)swz(r, e >> 3, dh * 2) * 8 + (e & 7);
}

// chunk permutation of a row of 16-bit elements
__device__ __forceinline__ int row_swz(int rp, int dh) { return dh >= 64 ? rp & 7 : (rp >> 1) & 3; }

// page and row inside the page of a position (pages of a power of two of positions need no division)
__device__ __forceinline__ int page_of(const Dev &D, int pos) { return D.p_shift >= 0 ? pos >> D.p_shift : pos / D.P; }
__device__ __forceinline__ int row_in_page(const Dev &D, int pos) { return D.p_shift >= 0 ? pos & (D.P - 1) : pos % D.P; }

}  // namespace xsm
