// The kernels around the decoding step: prefill (keys and values of the condition), inspection, export.
#include "xsm_common.cuh"

namespace xsm {

// ------------------------------------------------------------------------------- prefill kernels

// Cross-attention keys and values of the condition (computed once per mesh):
// out[c][r] = sum_k W[r][k] * cond[b][c][k], stored as cache tiles.
__global__ void __launch_bounds__(256) cross_kv_kernel(const Dev D, const float *Wall, const size_t *wkc_off,
                                                       const size_t *wvc_off, const float *cond, void *pool) {
    constexpr int T = 64, KT = 16;
    __shared__ float As[KT][T + 1], Bs[KT][T + 1];
    const int z = blockIdx.z, b = z % D.B, kv = (z / D.B) % 2, layer = z / (2 * D.B);
    const float *W = Wall + (kv == 0 ? wkc_off[layer] : wvc_off[layer]);
    const float *A = cond + (size_t)b * D.C * D.dc;
    const int c0 = blockIdx.x * T, r0 = blockIdx.y * T;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < D.dc; k0 += KT) {
        for (int i = threadIdx.x; i < T * KT; i += 256) {
            const int rr = i / KT, kk = i % KT;
            As[kk][rr] = (c0 + rr < D.C && k0 + kk < D.dc) ? to_f(A[(size_t)(c0 + rr) * D.dc + k0 + kk]) : 0.f;
            Bs[kk][rr] = (r0 + rr < D.d && k0 + kk < D.dc) ? to_f(W[(size_t)(r0 + rr) * D.dc + k0 + kk]) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < KT; ++kk) {
            float av[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { av[i] = As[kk][ty * 4 + i]; bv[i] = Bs[kk][tx * 4 + i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + ty * 4 + i, r = r0 + tx * 4 + j;
            if (c < D.C && r < D.d) {
                const int page = b * D.cpages + c / D.P, head = r / D.dh, e = r % D.dh;
                float *tile = kv_tile<float>(D, pool, D.B * D.cpages, layer, kv, page, head);
                tile[tile_off<float>(c % D.P, e, D.dh)] = acc[i][j];
            }
        }
}

cudaError_t launch_cross_kv(const Dev &D, const void *W, const size_t *wkc_off, const size_t *wvc_off, const void *cond, void *pool, int n_sets,
                            cudaStream_t st) {
    dim3 grid((D.C + 63) / 64, (D.d + 63) / 64, n_sets * 2 * D.B);
    cross_kv_kernel<<<grid, 256, 0, st>>>(D, (const float *)W, wkc_off, wvc_off, (const float *)cond, pool);
    return cudaGetLastError();
}

template <typename KVT>
__global__ void gather_kv_kernel(const Dev D, int layer, int seq, int pos0, int n, float *out_k, float *out_v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * D.d) return;
    const int p = pos0 + i / D.d, r = i % D.d, head = r / D.dh, e = r % D.dh;
    const int page = D.block_table[(size_t)seq * D.max_blocks + p / D.P];
    const KVT *kt = kv_tile<KVT>(D, D.kv_pool, D.n_pages, layer, 0, page, head);
    const KVT *vt = kv_tile<KVT>(D, D.kv_pool, D.n_pages, layer, 1, page, head);
    out_k[i] = to_f(kt[tile_off<KVT>(p % D.P, e, D.dh)]);
    out_v[i] = to_f(vt[tile_off<KVT>(p % D.P, e, D.dh)]);
}
cudaError_t launch_gather_kv(const Dev &D, int dtype, int layer, int seq, int pos0, int n, float *out_k,
                             float *out_v, cudaStream_t st) {
    const int total = n * D.d;
    if (dtype == 1) gather_kv_kernel<__half><<<(total + 255) / 256, 256, 0, st>>>(D, layer, seq, pos0, n, out_k, out_v);
    else gather_kv_kernel<float><<<(total + 255) / 256, 256, 0, st>>>(D, layer, seq, pos0, n, out_k, out_v);
    return cudaGetLastError();
}

__global__ void export_kernel(const Dev D, int max_new, int *tokens, int *lengths) {
    const int b = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = min(D.n_gen[b], max_new);
    if (i < max_new && tokens) tokens[(size_t)b * max_new + i] = i < n ? D.tok_log[(size_t)b * D.tok_ld + i] : -1;
    if (i == 0 && lengths) lengths[b] = n;
}
cudaError_t launch_export(const Dev &D, int max_new, int *d_tokens, int *d_lengths, cudaStream_t st) {
    dim3 grid((max_new + 255) / 256, D.B);
    export_kernel<<<grid, 256, 0, st>>>(D, max_new, d_tokens, d_lengths);
    return cudaGetLastError();
}

}  // namespace xsm
