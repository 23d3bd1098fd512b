// The weights in the form the tensor-core products read: fp32 -> bf16 in both orientations, all hidden layers.
#pragma once

#include "common.cuh"
#include "internal.h"

namespace gear {

// A block of 256 threads takes a tile of 32 x 32 weights through shared memory, so that both copies are written with coalesced rows;
// block blk of `blocks` (a.blocks() of them) also clears its share of the gradient.  Bound: two trips to memory.
// PLANES 1: rounded to bf16 (bf16 heads); 3: split into three planes, fan_in * fan_out elements apart (fp32 heads).
template <int PLANES>
__device__ __forceinline__ void round_weights_block(const RoundArgs& a, int blk, int blocks) {
    __shared__ __nv_bfloat16 tile[PLANES][32][33];
    const int l = blk < a.tiles[0] ? 0 : 1, t = l ? blk - a.tiles[0] : blk;
    const int fan_in = a.fan_in[l], fan_out = a.fan_out[l], across = (fan_out + 31) / 32;
    const int64_t stride = (int64_t)fan_in * fan_out;
    const int r0 = t / across * 32, c0 = t % across * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    float w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {                        // all loads ahead of the stores, which might alias them
        const int r = r0 + ty + 8 * k, c = c0 + tx;
        w[k] = r < fan_in && c < fan_out ? __ldg(a.W[l] + (int64_t)r * fan_out + c) : 0.f;
    }
    for (int64_t i = (int64_t)blk * 256 + threadIdx.x; i < a.n_grad; i += (int64_t)blocks * 256) a.grad[i] = 0.f;
    if (a.loss && blk == 0 && threadIdx.x == 0) *a.loss = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = r0 + ty + 8 * k, c = c0 + tx;
        if (r < fan_in && c < fan_out) {
            float rest = w[k];
#pragma unroll
            for (int p = 0; p < PLANES; ++p) {
                const __nv_bfloat16 v = __float2bfloat16_rn(rest);
                a.wb[l][p * stride + (int64_t)r * fan_out + c] = v;
                tile[p][ty + 8 * k][tx] = v;
                rest -= __bfloat162float(v);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c = c0 + ty + 8 * k, r = r0 + tx;
        if (r < fan_in && c < fan_out)
#pragma unroll
            for (int p = 0; p < PLANES; ++p) a.wbt[l][p * stride + (int64_t)c * fan_in + r] = tile[p][tx][ty + 8 * k];
    }
}

}  // namespace gear
