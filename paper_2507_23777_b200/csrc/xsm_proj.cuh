// What the projection kernels have in common: the layout of activations and the last step of every output.
#pragma once
#include "xsm_chain.cuh"

namespace xsm {

// Activations that a projection reads: fp32 values as bf16 hi + lo, in the image that the tensor core's operand tile has in
// shared memory.  A block is 64 columns of all rows: for every 8 token rows the 8 rows of hi parts, then the 8 of lo parts,
// rows of 128 bytes whose 16-byte chunks are permuted by the row (the 128-byte swizzle); 2 Mp * 128 consecutive bytes: one
// bulk copy, no tensor map.
__device__ __forceinline__ size_t plane_off(int Mp, int m, int k) {
    return (size_t)(k >> 6) * (size_t)(128 * Mp) + (size_t)((m >> 3) * 1024 + (m & 7) * 64 + ((((k >> 3) & 7) ^ (m & 7)) << 3) + (k & 7));
}
constexpr int kLo = 512;           // elements from a hi part to its lo part
// hi and lo of one value
__device__ __forceinline__ void store_split(bf16 *x, int Mp, int m, int k, float v) {
    bf16 hi, lo;
    split_bf16(v, hi, lo);
    bf16 *p = x + plane_off(Mp, m, k);
    p[0] = hi;
    p[kLo] = lo;
}
constexpr int kShareLd = 160;      // shares of a row's sum of squares: [row][kShareLd]

// Asks L2 for this CTA's share of the weights that a later kernel reads (one warp).  The kernels of a step are short against
// the latency of HBM and its weights' transfer; with what is needed 32 MB further on already on its way, memory is read at
// an even rate and a kernel's own copies come from L2.
__device__ __forceinline__ void fetch_ahead(const ProjArgs &A, unsigned cta, unsigned n_ctas) {
    constexpr unsigned kPiece = 4096;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const unsigned pieces = (A.ahead_bytes[q] + kPiece - 1) / kPiece;
        for (unsigned i = cta + n_ctas * (threadIdx.x & 31); i < pieces; i += n_ctas * 32) {
            const unsigned off = i * kPiece, n = min(kPiece, A.ahead_bytes[q] - off);
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(A.ahead[q] + off), "r"(n) : "memory");
        }
    }
}

}  // namespace xsm
