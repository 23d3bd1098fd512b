// Forward products of fp32 heads: H = ReLU(X W + b) with fp32 multiply-adds, every output one chain over the reduction
// in ascending order.
//
// The backward products run on the tensor cores (head_tc3.cu); the forward ones stay on the ordinary lanes because the sign of
// a pre-activation decides a ReLU branch: a view's gradient depends on it as a whole, so a value that is rounded in another
// order, however accurately, shows in the gradients wherever it lies within rounding of zero (about one unit in ten
// million; a batch of 32768 views has 12 million).
//
// Operands are fp32 (the head input and the hidden activations are kept in fp32 beside their planes for this, the weights
// are the caller's).
#include "f32_chain.cuh"
#include "internal.h"

namespace gear {

// WVEC: the weights may be read 16 bytes at a time (the head input and the activations always can).
template <int BM, int BN, int TM, int TN, int BK, int DEPTH, int AHEAD, int MIN_BLOCKS, bool WVEC>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), MIN_BLOCKS)
fwd_kernel(int M, int N, int K, const float* __restrict__ A, const float* __restrict__ W, const float* __restrict__ bias,
           __nv_bfloat16* __restrict__ H, int64_t h_stride, float* __restrict__ Hf) {
    wait_for_predecessor();
    using T = ChainTile<BM, BN, TM, TN, BK, DEPTH, AHEAD>;
    __shared__ __align__(16) typename T::Smem smem;
    const int m0 = (int)(blockIdx.y + gridDim.y * blockIdx.z) * BM, n0 = blockIdx.x * BN;
    if (m0 >= M) return;                                            // (the last layer of more row tiles than a grid dimension takes)
    typename T::Acc acc;
#pragma unroll
    for (int i = 0; i < TM * TN / 2; ++i) acc[i] = 0ull;
    T::product(acc, K, smem, [&](int r, int k) { return load4<true>(A + (int64_t)(m0 + r) * K + k, m0 + r < M ? K - k : 0); },
               [&](int k, int c) { return load4<WVEC>(W + (int64_t)k * N + n0 + c, k < K ? N - (n0 + c) : 0); });
#pragma unroll
    for (int j = 0; j < TN / 4; ++j) {
        const int n = n0 + T::col(j);
        if (n >= N) continue;                                       // N is a multiple of 8: whole strips
        const float b0 = __ldg(bias + n), b1 = __ldg(bias + n + 1), b2 = __ldg(bias + n + 2), b3 = __ldg(bias + n + 3);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const int m = m0 + T::row(i);
            if (m >= M) continue;
            const float4 h = make_float4(fmaxf(T::value(acc, i, 4 * j) + b0, 0.f), fmaxf(T::value(acc, i, 4 * j + 1) + b1, 0.f),
                                         fmaxf(T::value(acc, i, 4 * j + 2) + b2, 0.f), fmaxf(T::value(acc, i, 4 * j + 3) + b3, 0.f));
            uint2 p[3];
            split3_pair_relu(h.x, h.y, p[0].x, p[1].x, p[2].x);
            split3_pair_relu(h.z, h.w, p[0].y, p[1].y, p[2].y);
            const int64_t at = (int64_t)m * N + n;
#pragma unroll
            for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2*>(H + q * h_stride + at) = p[q];
            if (Hf) st_f4(Hf + at, h);
        }
    }
}

// The chain over the reduction cannot be split, so a product takes as long as its fullest SM: the smallest tiles while they are one
// wave, then the next larger ones, whose blocks have an SM to themselves and fetch further ahead; large tiles, which issue
// multiply-adds in half of the cycles, from three waves of 64 x 64 on, where their last wave no longer counts.  Measured on
// either side of each line (us, the form below the line / above it):
//   16 x 32 | 32 x 32   one wave of 16 x 32:    256 x 256 outputs, depth 192 (0.86 waves) 9.1 / 10.8; 512 x 256 (1.73) 10.7 / 10.9
//   32 x 32 | 32 x 64   one wave of 32 x 32:    512 x 256 (0.86) 10.9 / 11.2, depth 1632 39.4 / 41.4; 1024 x 256 (1.73) 12.8 / 10.7,
//                                               depth 1632 53.7 / 42.2; 1536 x 128 (1.30) 12.7 / 10.8
//   32 x 64 | 64 x 128  three waves of 64 x 64: 5632 x 256 (2.4) 27.1 / 29.9, depth 1632 171 / 196; 7168 x 256 (3.0) 31.3 / 31.3, depth
//                                               1632 207 / 199; 9472 x 256 (4.0) 35.6 / 31.8; 16384 x 128 (3.5) 35.2 / 31.1
// (8 x 4, 8 x 8 and 16 x 4 outputs per thread, pairs along rows or columns, doubled operands in shared memory made no other
// difference to the large ones: 32768 views, 192-256-128: 139 us.)
cudaError_t launch_fwd_f32(const gear_ctx_impl& c, int M, int N, int K, const float* A, const float* W, const float* bias,
                           const Planes& H, float* Hf, cudaStream_t st) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    KernelScope ks(&c.prof, "f32_gemm_fwd", st);
    const bool wvec = (reinterpret_cast<uintptr_t>(W) & 15u) == 0;
    auto tiles = [&](int bm, int bn) { return ceil_div(M, bm) * ceil_div(N, bn); };
    auto grid = [&](int bm, int bn) {
        const int64_t rows = ceil_div(M, bm), y = rows < 65535 ? rows : 65535;
        return dim3((unsigned)ceil_div(N, bn), (unsigned)y, (unsigned)ceil_div(rows, y));
    };
#define GEAR_FWD(BM, BN, TM, TN, BK, DEPTH, AH, MB) \
    (wvec ? launch_dependent(fwd_kernel<BM, BN, TM, TN, BK, DEPTH, AH, MB, true>, grid(BM, BN), \
                             dim3((BM / TM) * (BN / TN)), 0, st, M, N, K, A, W, bias, H.p, H.stride, Hf) \
          : launch_dependent(fwd_kernel<BM, BN, TM, TN, BK, DEPTH, AH, MB, false>, grid(BM, BN), \
                             dim3((BM / TM) * (BN / TN)), 0, st, M, N, K, A, W, bias, H.p, H.stride, Hf))
    if (tiles(16, 32) <= sm_count()) return GEAR_FWD(16, 32, 2, 4, 32, 2, 3, 2);
    if (tiles(32, 32) <= sm_count()) return GEAR_FWD(32, 32, 2, 4, 32, 2, 3, 2);
    if (tiles(64, 64) < 3 * sm_count()) return GEAR_FWD(32, 64, 4, 4, 32, 4, 2, 1);
    return GEAR_FWD(64, 128, 16, 4, 16, 1, 1, 4);
#undef GEAR_FWD
}

}  // namespace gear
