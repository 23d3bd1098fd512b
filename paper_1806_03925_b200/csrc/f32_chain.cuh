// Products of fp32 matrices with one ascending chain of multiply-adds per output (head_fwd.cu, dense.cu).
//
// Multiply-adds are issued in pairs (fma.rn.f32x2: two independent fp32 multiply-adds, each rounded like fmaf), which
// leaves issue slots for the shared-memory reads.  Bound: the fp32 lanes (128 multiply-adds per SM and cycle) for large
// products, the length of the chain for small ones.
#pragma once

#include "common.cuh"

namespace gear {

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 dup2(float a) { f32x2 r; asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a)); return r; }
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 unpack2(f32x2 v) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v)); return r; }

// 4 consecutive values of a row; VEC: one 16-byte load, else one by one, `left` of them within the row
template <bool VEC> __device__ __forceinline__ float4 load4(const float* __restrict__ p, int left) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (left <= 0) return v;
    if (VEC) return __ldg(reinterpret_cast<const float4*>(p));
    v.x = __ldg(p);
    if (left > 1) v.y = __ldg(p + 1);
    if (left > 2) v.z = __ldg(p + 2);
    if (left > 3) v.w = __ldg(p + 3);
    return v;
}

// A block of (BM / TM) * (BN / TN) threads computes BM x BN outputs, a thread TM x TN of them: rows in strips of
// ChainTile::RS, BM / (TM / RS) apart, columns in strips of four, BN / (TN / 4) apart, so that shared-memory reads are wide
// and free of bank conflicts.  Operand tiles are fetched DEPTH steps ahead into registers and pass through two shared-memory
// buffers.  (One step ahead, a block that is alone on its SM waited for the L2 in half of its cycles: 1024 x 256 x 1632 took 66 us.)
// The A tile is transposed on its way in: neighbouring lanes fetch a row's BK values, and the row index is XORed so
// that the 32 stores of a warp hit 32 banks.  A step's values are read from shared memory AHEAD multiply-add rounds early.
template <int BM, int BN, int TM, int TN, int BK, int DEPTH, int AHEAD> struct ChainTile {
    static constexpr int THREADS = (BM / TM) * (BN / TN), TX = BN / TN, KQ = BK / 4;
    static constexpr int A_PIECES = BM * KQ / THREADS, B_PIECES = BK * (BN / 4) / THREADS;      // 4-value pieces per thread
    static constexpr int RS = TM < 4 ? TM : 4;
    static constexpr int SW = 32 / KQ < 4 ? 4 : 32 / KQ;             // the XOR's unit: rows a warp's store covers per k
    static_assert(A_PIECES >= 1 && B_PIECES >= 1 && A_PIECES * THREADS == BM * KQ && B_PIECES * THREADS == BK * (BN / 4), "whole pieces");
    static_assert(TM % RS == 0 && (RS == 2 || RS == 4) && TN % 4 == 0 && BM % 16 == 0 && (KQ == 2 || KQ == 4 || KQ == 8), "strips");
    struct Smem { float a[2][BK][BM]; float b[2][BK][BN]; };
    // A multiply-add takes a pair of neighbouring outputs: of a row, or, in tall tiles, of a column, where fewer values have to be
    // doubled for it (two moves each: 64 x 64 tiles with 8 x 4 outputs were bound by them).
    static constexpr bool TALL = TM > TN;
    typedef f32x2 Acc[TM * TN / 2];
    static __device__ __forceinline__ float value(const Acc& acc, int i, int j) {
        const float2 v = unpack2(TALL ? acc[(i / 2) * TN + j] : acc[i * (TN / 2) + j / 2]);
        return (TALL ? i : j) & 1 ? v.y : v.x;
    }
    static __device__ __forceinline__ int swizzle(int kq) { return (kq * SW) % BM; }
    // row / first column of the tile that output (i, 4 j) of this thread stands for
    static __device__ __forceinline__ int row(int i) { return (i / RS) * (BM / (TM / RS)) + (int)(threadIdx.x / TX) * RS + i % RS; }
    static __device__ __forceinline__ int col(int j) { return j * (BN / (TN / 4)) + (int)(threadIdx.x % TX) * 4; }

    // acc += A . B over k < K; load_a(row of the tile, k), load_b(k, column of the tile): four consecutive values (along k / the
    // columns), zeros where there are none
    template <typename LoadA, typename LoadB>
    static __device__ __forceinline__ void product(Acc& acc, int K, Smem& s, LoadA load_a, LoadB load_b) {
        const int tid = threadIdx.x;
        float4 ra[DEPTH][A_PIECES], rb[DEPTH][B_PIECES];
        auto fetch = [&](int d, int k0) {
#pragma unroll
            for (int q = 0; q < A_PIECES; ++q) { const int p = tid + q * THREADS; ra[d][q] = load_a(p / KQ, k0 + 4 * (p % KQ)); }
#pragma unroll
            for (int q = 0; q < B_PIECES; ++q) { const int p = tid + q * THREADS; rb[d][q] = load_b(k0 + p / (BN / 4), 4 * (p % (BN / 4))); }
        };
        auto stash = [&](int d, int buf) {
#pragma unroll
            for (int q = 0; q < A_PIECES; ++q) {
                const int p = tid + q * THREADS, kq = p % KQ, m = (p / KQ) ^ swizzle(kq);
                const float4 v = ra[d][q];
                s.a[buf][4 * kq][m] = v.x; s.a[buf][4 * kq + 1][m] = v.y; s.a[buf][4 * kq + 2][m] = v.z; s.a[buf][4 * kq + 3][m] = v.w;
            }
#pragma unroll
            for (int q = 0; q < B_PIECES; ++q) {
                const int p = tid + q * THREADS;
                st_f4(&s.b[buf][p / (BN / 4)][4 * (p % (BN / 4))], rb[d][q]);
            }
        };
#pragma unroll
        for (int d = 0; d < DEPTH; ++d) if (d * BK < K) fetch(d, d * BK);
        stash(0, 0);
        __syncthreads();
        int buf = 0;
        for (int k0 = 0; k0 < K; k0 += DEPTH * BK) {
#pragma unroll
            for (int d = 0; d < DEPTH; ++d) {                            // register set d held step k0 / BK + d
                const int at = k0 + d * BK;
                if (at >= K) break;
                if (at + DEPTH * BK < K) fetch(d, at + DEPTH * BK);
                f32x2 av[AHEAD + 1][TM / 2], bv[AHEAD + 1][TN / 2];
                auto read = [&](int k) {
                    const int f = k % (AHEAD + 1);
#pragma unroll
                    for (int i = 0; i < TM / RS; ++i) {
                        const float* p = &s.a[buf][k][row(i * RS) ^ swizzle(k / 4)];
                        if constexpr (RS == 4) {
                            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
                            av[f][2 * i] = t.x; av[f][2 * i + 1] = t.y;
                        } else av[f][i] = *reinterpret_cast<const f32x2*>(p);
                    }
#pragma unroll
                    for (int j = 0; j < TN / 4; ++j) {
                        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(&s.b[buf][k][col(j)]);
                        bv[f][2 * j] = t.x; bv[f][2 * j + 1] = t.y;
                    }
                };
#pragma unroll
                for (int k = 0; k < AHEAD; ++k) read(k);
#pragma unroll
                for (int k = 0; k < BK; ++k) {
                    if (k + AHEAD < BK) read(k + AHEAD);
                    const f32x2 (&a)[TM / 2] = av[k % (AHEAD + 1)];
                    const f32x2 (&b)[TN / 2] = bv[k % (AHEAD + 1)];
#pragma unroll
                    for (int x = 0; x < (TALL ? TN : TM); ++x) {
                        const float2 v = unpack2(TALL ? b[x / 2] : a[x / 2]);
                        const f32x2 vv = dup2(x & 1 ? v.y : v.x);
#pragma unroll
                        for (int y = 0; y < (TALL ? TM : TN) / 2; ++y) {
                            if (TALL) fma2(acc[y * TN + x], a[y], vv);
                            else fma2(acc[x * (TN / 2) + y], vv, b[y]);
                        }
                    }
                }
                if (at + BK < K) {
                    stash((d + 1) % DEPTH, buf ^ 1);                    // the other buffer: nobody reads it during this step
                    __syncthreads();
                    buf ^= 1;
                }
            }
        }
    }
};

}  // namespace gear
