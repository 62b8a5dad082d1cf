// What the projection kernels have in common: the layout of activations and the last step of every output.
#pragma once
#include "xsm_chain.cuh"

namespace xsm {

// Activations that a projection reads: fp32 values as bf16 hi + lo, in the image that the tensor core's operand tile has in
// shared memory.  A block is 64 columns of all rows: for every 8 token rows the 8 rows of hi parts, then the 8 of lo parts,
// rows of 128 bytes whose 16-byte chunks are permuted by the row (the 128-byte swizzle); 2 Mp * 128 consecutive bytes: one
// bulk copy, no tensor map.
// (element k of token row m < kTokenTile)
__device__ __forceinline__ size_t plane_off(int Mp, int m, int k) {
    return (size_t)(k >> 6) * (size_t)(128 * Mp) + (size_t)((m >> 3) * 1024 + (m & 7) * 64 + ((((k >> 3) & 7) ^ (m & 7)) << 3) + (k & 7));
}
constexpr int kLo = 512;           // elements from a hi part to its lo part

}  // namespace xsm
