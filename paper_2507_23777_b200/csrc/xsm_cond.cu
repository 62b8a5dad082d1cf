// Prefill: keys and values of the condition under the layers' (or the decoding heads') projections, bf16 models, tcgen05.
//
// A plain dense contraction, out[c][r] = W[r] . cond[c]: 128 weight rows on the M side, up to 128 condition latents on the N
// side (the latents of a sequence cut evenly into as few tiles as that allows), blocks of 64 columns of both by TMA through
// a ring, one warp issuing the products, the accumulator stored as fp16 cache tiles.  Bound by the tensor cores while the
// products run; a tile is short (16 blocks at d_cond 1024), so two CTAs share an SM and one's stores run under the
// other's products.  257 x 1024 latents through 48 projections of 1024 x 1024: 304 us with operands staged by threads,
// one block at a time; see kCondRing for what the ring holds.
#include "xsm_chain.cuh"

#include <cuda.h>

namespace xsm {

constexpr int kCondThreads = 192;              // a warp that fetches, one that multiplies, four that store
constexpr int kCondRing = 3;                   // blocks in flight: 96 KB, two CTAs to an SM
constexpr int kCondBlock = 128 * 128;          // bytes of 128 rows x 64 columns

struct __align__(64) CondMaps { CUtensorMap wk, wv, cond; };

__global__ void __launch_bounds__(kCondThreads) cond_kv_kernel(const Dev D, const __grid_constant__ CondMaps T, int tile_n, void *pool) {
    extern __shared__ char smem_raw[];
    char *const smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ __align__(8) uint64_t full[kCondRing], empty[kCondRing], done;
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int z = blockIdx.z, b = z % D.B, kv = (z / D.B) % 2, set = z / (2 * D.B);
    const int c0 = blockIdx.x * tile_n, r0 = blockIdx.y * 128, n = (D.dc + 63) / 64;
    if (tid == 0) {
        for (int i = 0; i < kCondRing; ++i) { mbar_init(smem_u32(&full[i]), 1u); mbar_init(smem_u32(&empty[i]), 1u); }
        mbar_init(smem_u32(&done), 1u);
        mbar_init_fence();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&tmem_slot)), "n"(128) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tcgen05_before_sync();
    __syncthreads();
    tcgen05_after_sync();
    const uint32_t sm = smem_u32(smem);
    if (tid == 0) {
        for (int i = 0; i < n; ++i) {
            const int s = i % kCondRing;
            const uint32_t a = sm + (uint32_t)s * 2u * kCondBlock, f = smem_u32(&full[s]);
            if (i >= kCondRing) mbar_wait(smem_u32(&empty[s]), (uint32_t)((i / kCondRing - 1) & 1), D.mbar_limit, D.status);
            mbar_arrive_expect_tx(f, (uint32_t)(kCondBlock + tile_n * 128));
            tma_box(a, kv == 0 ? &T.wk : &T.wv, i * 64, r0, set, f);
            tma_box(a + kCondBlock, &T.cond, i * 64, c0, b, f);
        }
    } else if (tid == 32) {
        const uint32_t idesc = umma_idesc(128, tile_n), tmem = tmem_slot;
        for (int i = 0; i < n; ++i) {
            const int s = i % kCondRing;
            mbar_wait(smem_u32(&full[s]), (uint32_t)((i / kCondRing) & 1), D.mbar_limit, D.status);
            tcgen05_after_sync();
            const uint64_t da = umma_desc_sw128(sm + (uint32_t)s * 2u * kCondBlock), db = umma_desc_sw128(sm + (uint32_t)s * 2u * kCondBlock + kCondBlock);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) umma_mma(tmem, da + 2 * ks, db + 2 * ks, idesc, (i > 0 || ks > 0) ? 1u : 0u);
            umma_commit(smem_u32(&empty[s]));
        }
        umma_commit(smem_u32(&done));
    }
    __syncwarp();
    if (warp >= 2) {
        mbar_wait(smem_u32(&done), 0u, D.mbar_limit, D.status);
        __syncwarp();
        tcgen05_after_sync();
        const int lanes = warp & 3, r = r0 + lanes * 32 + lane, head = r / D.dh, e = r - head * D.dh;      // thread = weight row
        const uint32_t tbase = tmem_slot + ((uint32_t)(lanes * 32) << 16);
        for (int n0 = 0; n0 < tile_n; n0 += 16) {
            uint32_t v[16];
            tmem_ld16(v, tbase + (uint32_t)n0);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int c = c0 + n0 + j;
                if (n0 + j < tile_n && c < D.C && r < D.d) {
                    __half *tile = kv_tile<__half>(D, pool, D.B * D.cpages, set, kv, b * D.cpages + page_of(D, c), head);
                    tile[tile_off<__half>(row_in_page(D, c), e, D.dh)] = from_f<__half>(__uint_as_float(v[j]));
                }
            }
        }
    }
    tcgen05_before_sync();
    __syncthreads();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_slot), "n"(128) : "memory");
}

int cond_tile(int n_cond) {      // latents of a tile: a multiple of 16, at most 128
    const int tiles = (n_cond + 127) / 128;
    return ((n_cond + tiles - 1) / tiles + 15) / 16 * 16;
}

cudaError_t launch_cond_kv(const Dev &D, const void *maps, void *pool, int n_sets, cudaStream_t st) {
    const CondMaps &T = *reinterpret_cast<const CondMaps *>(maps);
    const int tile_n = cond_tile(D.C), smem = kCondRing * 2 * kCondBlock + 1024;
    cudaError_t e = open_kernel((const void *)cond_kv_kernel, smem, false);
    if (e != cudaSuccess) return e;
    cond_kv_kernel<<<dim3((D.C + tile_n - 1) / tile_n, (D.d + 127) / 128, n_sets * 2 * D.B), kCondThreads, smem, st>>>(D, T, tile_n, pool);
    return cudaGetLastError();
}

}  // namespace xsm
