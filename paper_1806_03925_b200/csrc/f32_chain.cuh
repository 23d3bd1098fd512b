// Products of fp32 matrices with one ascending chain of multiply-adds per output (head_fwd.cu, dense.cu).
//
// Multiply-adds are issued in pairs (fma.rn.f32x2: two independent fp32 multiply-adds, each rounded like fmaf), which
// leaves issue slots for the shared-memory reads.  A 16-byte read costs a warp about four clocks of the SM's 128 bytes per clock
// however many of its lanes ask for the same words (1 x 8 outputs per lane: 4.6 measured), so a step of the reduction costs a warp
// TM + TN clocks there and TM * TN / 4 in the multiply-add lanes.  Bound: 8 x 8 outputs per lane wait for the multiply-add pipe first
// (shared memory 58 % of its rate; 37888 x 128 x 2048: 54 TFLOP/s, of 65 to 69 that multiply-adds on registers alone reach; 16 x 4,
// as before: 40); 4 x 4 with a warp per scheduler, of products too small for more, for shared memory and their own latencies.
#pragma once

#include "common.cuh"

namespace gear {

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 dup2(float a) { f32x2 r; asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a)); return r; }
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 unpack2(f32x2 v) { float2 r; asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v)); return r; }

// 4-byte asynchronous copy global -> shared, for rows that are not 16-byte aligned; src_bytes = 0 fills with zero
__device__ __forceinline__ void cp_async_4(uint32_t smem_dst, const void* gsrc, int src_bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" :: "r"(smem_dst), "l"(gsrc), "r"(src_bytes) : "memory");
}

// WR x WC warps of LR x LC lanes; a lane computes TM x TN outputs: rows LR apart, columns in strips of four, 4 LC apart.
// Operand tiles of BK steps travel through a ring of STAGES buffers by asynchronous copies, rows of A as they lie in memory
// (a lane reads four steps of a row at a time; the pitch of BK + 4 words puts the rows of a warp in different banks).
template <int TM_, int TN_, int LR, int LC, int WR_, int WC_, int BK_, int STAGES_> struct ChainTile {
    static constexpr int TM = TM_, TN = TN_, WR = WR_, WC = WC_, BK = BK_, STAGES = STAGES_, LANES_C = LC, LANES_R = LR;
    static constexpr int BM = TM * LR * WR, BN = TN * LC * WC, THREADS = 32 * WR * WC;
    static constexpr int PITCH = BK + 4, A_WORDS = BM * PITCH, B_WORDS = BK * BN, STAGE_WORDS = A_WORDS + B_WORDS;
    static constexpr int SMEM = STAGES * STAGE_WORDS * 4;
    static constexpr int A_QUADS = BM * (BK / 4), B_QUADS = BK * (BN / 4);          // 4-value pieces of a step
    static constexpr int A_PIECES = (A_QUADS + THREADS - 1) / THREADS, B_PIECES = (B_QUADS + THREADS - 1) / THREADS;
    static_assert(LR * LC == 32 && TN % 4 == 0 && BK % 4 == 0 && STAGES >= 2, "shape");
    static_assert(B_QUADS % THREADS == 0, "whole pieces");
    typedef f32x2 Acc[TM][TN / 2];
    static __device__ __forceinline__ float value(const Acc& acc, int i, int j) { const float2 v = unpack2(acc[i][j / 2]); return j & 1 ? v.y : v.x; }
    static __device__ __forceinline__ int warp_row() { return (int)(threadIdx.x / 32) / WC; }
    static __device__ __forceinline__ int warp_col() { return (int)(threadIdx.x / 32) % WC; }
    // row / first column of the tile that outputs (i, 4 j ..) of this thread stand for
    static __device__ __forceinline__ int row(int i) { return warp_row() * (TM * LR) + i * LR + (int)(threadIdx.x % 32) / LC; }
    static __device__ __forceinline__ int col(int j) { return warp_col() * (TN * LC) + j * (4 * LC) + (int)(threadIdx.x % LC) * 4; }

    // acc = A . B over k < K.  a_row(r): row r of the tile in memory, or null (zeros); b: element (0, first column of the tile),
    // rows ldb apart, n_cols columns exist.  AVEC / BVEC: A's rows / B's rows may be read 16 bytes at a time (lengths and strides
    // are multiples of four then).  smem: SMEM bytes, free when the block enters and when it leaves.
    template <bool AVEC, bool BVEC, typename ARow>
    static __device__ __forceinline__ void product(Acc& acc, int K, float* smem, ARow a_row, const float* __restrict__ b, int64_t ldb, int n_cols) {
        const int tid = threadIdx.x;
        const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem);
        // What a copy that fills with zeros names as its source: that has to be aligned to the copy's size also where nothing is read.  (A
        // pointer to A in its place, one more register pair in the loop: 32 x 256 tiles 8 % slower.)
        const float* none = AVEC && !BVEC ? reinterpret_cast<const float*>(reinterpret_cast<uintptr_t>(b) & ~(uintptr_t)15) : b;
        const float* pa[A_PIECES];
#pragma unroll
        for (int q = 0; q < A_PIECES; ++q) {
            const int p = tid + q * THREADS;
            const float* r = p < A_QUADS ? a_row(p / (BK / 4)) : nullptr;
            pa[q] = r ? r + 4 * (p % (BK / 4)) : nullptr;
        }
        auto fetch = [&](int stage, int k0) {
            const uint32_t sa = s0 + (uint32_t)(stage * STAGE_WORDS) * 4u, sb = sa + (uint32_t)A_WORDS * 4u;
#pragma unroll
            for (int q = 0; q < A_PIECES; ++q) {
                const int p = tid + q * THREADS;
                if (A_QUADS % THREADS != 0 && p >= A_QUADS) break;
                const int k = k0 + 4 * (p % (BK / 4));
                const uint32_t dst = sa + (uint32_t)((p / (BK / 4)) * PITCH + 4 * (p % (BK / 4))) * 4u;
                if (AVEC) { const bool on = pa[q] && k < K; cp_async_16(dst, on ? pa[q] + k0 : none, on ? 16 : 0); }
                else
#pragma unroll
                    for (int e = 0; e < 4; ++e) { const bool on = pa[q] && k + e < K; cp_async_4(dst + 4u * e, on ? pa[q] + k0 + e : none, on ? 4 : 0); }
            }
#pragma unroll
            for (int q = 0; q < B_PIECES; ++q) {
                const int p = tid + q * THREADS, k = p / (BN / 4), c = 4 * (p % (BN / 4));
                const uint32_t dst = sb + (uint32_t)(k * BN + c) * 4u;
                const float* src = b + (int64_t)(k0 + k) * ldb + c;
                if (BVEC) { const bool on = k0 + k < K && c < n_cols; cp_async_16(dst, on ? src : b, on ? 16 : 0); }
                else
#pragma unroll
                    for (int e = 0; e < 4; ++e) { const bool on = k0 + k < K && c + e < n_cols; cp_async_4(dst + 4u * e, on ? src + e : b, on ? 4 : 0); }
            }
        };
        const int steps = (K + BK - 1) / BK;
#pragma unroll
        for (int s = 0; s < STAGES - 1; ++s) { if (s < steps) fetch(s, s * BK); cp_async_commit(); }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
        const int a_at = row(0) * PITCH, b_at = col(0);
        int stage = 0, next = STAGES - 1;
        for (int s = 0; s < steps; ++s) {
            cp_async_wait<STAGES - 2>();
            __syncthreads();                                     // step s is there for all; the buffer filled next has been read by all
            if (s + STAGES - 1 < steps) fetch(next, (s + STAGES - 1) * BK);
            cp_async_commit();
            next = next + 1 == STAGES ? 0 : next + 1;
            const float* sa = smem + stage * STAGE_WORDS + a_at;
            const float* sb = smem + stage * STAGE_WORDS + A_WORDS + b_at;
            stage = stage + 1 == STAGES ? 0 : stage + 1;
            float4 av[2][TM];
            f32x2 bv[2][TN / 2];
            auto read_a = [&](int f, int kq) {
#pragma unroll
                for (int i = 0; i < TM; ++i) av[f][i] = *reinterpret_cast<const float4*>(sa + i * (LR * PITCH) + 4 * kq);
            };
            auto read_b = [&](int f, int k) {
#pragma unroll
                for (int j = 0; j < TN / 4; ++j) {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(sb + k * BN + j * (4 * LC));
                    bv[f][2 * j] = t.x; bv[f][2 * j + 1] = t.y;
                }
            };
            read_a(0, 0); read_b(0, 0);
#pragma unroll
            for (int k = 0; k < BK; ++k) {
                if (k % 4 == 0 && k + 4 < BK) read_a((k / 4 + 1) & 1, k / 4 + 1);
                if (k + 1 < BK) read_b((k + 1) & 1, k + 1);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const float4 v = av[(k / 4) & 1][i];
                    const f32x2 vv = dup2(k % 4 == 0 ? v.x : k % 4 == 1 ? v.y : k % 4 == 2 ? v.z : v.w);
#pragma unroll
                    for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], vv, bv[k & 1][j]);
                }
            }
        }
        cp_async_wait<0>();
        __syncthreads();                                         // the buffers are free again
    }
};

}  // namespace gear
