// Forward products of fp32 heads: H = ReLU(X W + b) with fp32 multiply-adds, every output one chain over the reduction
// in ascending order.
//
// The backward products run on the tensor cores (head_tc3.cu); the forward ones stay on the ordinary lanes because the sign of
// a pre-activation decides a ReLU branch: a view's gradient depends on it as a whole, so a value that is rounded in another
// order, however accurately, shows in the gradients wherever it lies within rounding of zero (about one unit in ten
// million; a batch of 32768 views has 12 million).
//
// Operands are fp32 (the head input and the hidden activations are kept in fp32 beside their planes for this, the weights
// are the caller's).  Multiply-adds are issued in pairs (fma.rn.f32x2: two independent fp32 multiply-adds, each rounded like
// fmaf), which leaves issue slots for the shared-memory reads.  Bound: the fp32 lanes (128 multiply-adds per SM and cycle).
#include "common.cuh"
#include "internal.h"

namespace gear {

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 dup2(float a) { f32x2 r; asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a)); return r; }
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 unpack2(f32x2 v) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v)); return r; }

// 4 consecutive values of a row; VEC: the row is 16-byte aligned (and n a multiple of 4)
template <bool VEC> __device__ __forceinline__ float4 load4(const float* __restrict__ p, bool ok) {
    if (!ok) return make_float4(0.f, 0.f, 0.f, 0.f);
    if (VEC) return __ldg(reinterpret_cast<const float4*>(p));
    return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}

// A block computes BM x BN outputs, a thread TM x TN of them: rows in strips of 4, BM / (TM / 4) apart, columns likewise; a
// warp reads 4 row strips and 8 column strips per step of the reduction, one 128-byte wavefront each.  Operand tiles are
// fetched one step ahead into registers and pass through two shared-memory buffers.  The A tile is transposed on its way in:
// neighbouring lanes fetch a row's FW_BK values, and the row index is XORed so that the 32 stores of a warp hit 32 banks.
// WVEC: the weights may be read 16 bytes at a time.
template <int BM, int BN, int TM, int TN, int FW_BK, int MIN_BLOCKS, bool WVEC>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), MIN_BLOCKS)
fwd_kernel(int M, int N, int K, const float* __restrict__ A, const float* __restrict__ W, const float* __restrict__ bias,
           __nv_bfloat16* __restrict__ H, int64_t h_stride, float* __restrict__ Hf) {
    wait_for_predecessor();
    constexpr int THREADS = (BM / TM) * (BN / TN), TX = BN / TN, KQ = FW_BK / 4;
    constexpr int A_PIECES = BM * KQ / THREADS, B_PIECES = FW_BK * (BN / 4) / THREADS;      // 4-value pieces per thread
    static_assert(A_PIECES >= 1 && B_PIECES >= 1 && A_PIECES * THREADS == BM * KQ && B_PIECES * THREADS == FW_BK * (BN / 4), "whole pieces");
    static_assert(TM % 4 == 0 && TN % 4 == 0 && BM % 32 == 0 && (KQ == 2 || KQ == 4 || KQ == 8), "strips of four");
    constexpr int SW = 32 / KQ;                                     // rows a warp's store covers per k: the XOR's unit
    __shared__ __align__(16) float As[2][FW_BK][BM];
    __shared__ __align__(16) float Bs[2][FW_BK][BN];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    f32x2 acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
    float4 ra[A_PIECES], rb[B_PIECES];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int q = 0; q < A_PIECES; ++q) {
            const int p = tid + q * THREADS, m = m0 + p / KQ, k = k0 + 4 * (p % KQ);
            ra[q] = load4<true>(A + (int64_t)m * K + k, m < M && k < K);
        }
#pragma unroll
        for (int q = 0; q < B_PIECES; ++q) {
            const int p = tid + q * THREADS, n = n0 + 4 * (p % (BN / 4)), k = k0 + p / (BN / 4);
            rb[q] = load4<WVEC>(W + (int64_t)k * N + n, n < N && k < K);
        }
    };
    auto stash = [&](int buf) {
#pragma unroll
        for (int q = 0; q < A_PIECES; ++q) {
            const int p = tid + q * THREADS, kq = p % KQ, m = (p / KQ) ^ (kq * SW);
            As[buf][4 * kq][m] = ra[q].x; As[buf][4 * kq + 1][m] = ra[q].y;
            As[buf][4 * kq + 2][m] = ra[q].z; As[buf][4 * kq + 3][m] = ra[q].w;
        }
#pragma unroll
        for (int q = 0; q < B_PIECES; ++q) {
            const int p = tid + q * THREADS;
            st_f4(&Bs[buf][p / (BN / 4)][4 * (p % (BN / 4))], rb[q]);
        }
    };
    fetch(0);
    stash(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += FW_BK) {
        const bool more = k0 + FW_BK < K;
        if (more) fetch(k0 + FW_BK);
#pragma unroll
        for (int k = 0; k < FW_BK; ++k) {
            float a[TM];
            f32x2 b[TN / 2];
#pragma unroll
            for (int i = 0; i < TM / 4; ++i) {
                const float4 t = ld_f4(&As[buf][k][(i * (BM / (TM / 4)) + ty * 4) ^ ((k / 4) * SW)]);
                a[4 * i] = t.x; a[4 * i + 1] = t.y; a[4 * i + 2] = t.z; a[4 * i + 3] = t.w;
            }
#pragma unroll
            for (int j = 0; j < TN / 4; ++j) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(&Bs[buf][k][j * (BN / (TN / 4)) + tx * 4]);
                b[2 * j] = t.x; b[2 * j + 1] = t.y;
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const f32x2 aa = dup2(a[i]);
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], aa, b[j]);
            }
        }
        if (more) {
            stash(buf ^ 1);                                         // the other buffer: nobody reads it during this step
            __syncthreads();
            buf ^= 1;
        }
    }
#pragma unroll
    for (int j = 0; j < TN / 4; ++j) {
        const int n = n0 + j * (BN / (TN / 4)) + tx * 4;
        if (n >= N) continue;                                       // N is a multiple of 8: whole strips
        const float b0 = __ldg(bias + n), b1 = __ldg(bias + n + 1), b2 = __ldg(bias + n + 2), b3 = __ldg(bias + n + 3);
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const int m = m0 + (i / 4) * (BM / (TM / 4)) + ty * 4 + i % 4;
            if (m >= M) continue;
            const float2 lo = unpack2(acc[i][2 * j]), hi = unpack2(acc[i][2 * j + 1]);
            const float4 h = make_float4(fmaxf(lo.x + b0, 0.f), fmaxf(lo.y + b1, 0.f), fmaxf(hi.x + b2, 0.f), fmaxf(hi.y + b3, 0.f));
            uint2 p[3];
            split3_pair(h.x, h.y, p[0].x, p[1].x, p[2].x);
            split3_pair(h.z, h.w, p[0].y, p[1].y, p[2].y);
            const int64_t at = (int64_t)m * N + n;
#pragma unroll
            for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2*>(H + q * h_stride + at) = p[q];
            if (Hf) st_f4(Hf + at, h);
        }
    }
}

// The chain over the reduction cannot be split, so a small batch is spread over as many SMs as it has tiles.  Measured (us;
// 64 x 64 tiles with 8 x 4 outputs per thread | 32 x 64 with 4 x 4 | 32 x 32 with 4 x 4): 32768 x 128 x 256: 53 | 65 | 70;
// 8192 x 128 x 192: 14.5 | 16.5 | 18.6; 4015 x 184 x 128 (189 | 378 | 756 tiles): 11.0 | 10.4 | 10.4; 1024 x 256 x 1632 (64 | 128
// | 256 tiles): 70 | 42 | 44; 1024 x 64 x 256 (16 | 32 | 64): 14.5 | 10.4 | 8.4.
cudaError_t launch_fwd_f32(const gear_ctx_impl& c, int M, int N, int K, const float* A, const float* W, const float* bias,
                           const Planes& H, float* Hf, cudaStream_t st) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    KernelScope ks(&c.prof, "f32_gemm_fwd", st);
    const bool wvec = (reinterpret_cast<uintptr_t>(W) & 15u) == 0;
    auto tiles = [&](int bm, int bn) { return ceil_div(M, bm) * ceil_div(N, bn); };
#define GEAR_FWD(BM, BN, TM, TN, BK) \
    (wvec ? launch_dependent(fwd_kernel<BM, BN, TM, TN, BK, 4, true>, dim3((unsigned)ceil_div(N, BN), (unsigned)ceil_div(M, BM)), \
                             dim3((BM / TM) * (BN / TN)), 0, st, M, N, K, A, W, bias, H.p, H.stride, Hf) \
          : launch_dependent(fwd_kernel<BM, BN, TM, TN, BK, 4, false>, dim3((unsigned)ceil_div(N, BN), (unsigned)ceil_div(M, BM)), \
                             dim3((BM / TM) * (BN / TN)), 0, st, M, N, K, A, W, bias, H.p, H.stride, Hf))
    if (2 * tiles(64, 64) >= 3 * sm_count()) return GEAR_FWD(64, 64, 8, 4, 16);
    if (5 * tiles(32, 64) >= 4 * sm_count()) return GEAR_FWD(32, 64, 4, 4, 32);
    return GEAR_FWD(32, 32, 4, 4, 32);
#undef GEAR_FWD
}

}  // namespace gear
