// Forward products of fp32 heads: H = ReLU(X W + b) with fp32 multiply-adds, every output one chain over the reduction
// in ascending order; the top layer takes the output unit along.
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
template <class T, int MIN_BLOCKS, bool WVEC>
__global__ void __launch_bounds__(T::THREADS, MIN_BLOCKS)
fwd_kernel(int M, int N, int K, const float* __restrict__ A, const float* __restrict__ W, const float* __restrict__ bias,
           __nv_bfloat16* __restrict__ H, int64_t h_stride, float* __restrict__ Hf) {
    wait_for_predecessor();
    if (gridDim.x * gridDim.y <= FEW_BLOCKS) let_successor_start();
    extern __shared__ float4 dyn_smem[];
    const int m0 = (int)(blockIdx.y + gridDim.y * blockIdx.z) * T::BM, n0 = blockIdx.x * T::BN;
    if (m0 >= M) return;                                            // (the last layer of more row tiles than a grid dimension takes)
    typename T::Acc acc;
    T::template product<true, WVEC>(acc, K, reinterpret_cast<float*>(dyn_smem),
                                    [&](int r) -> const float* { return m0 + r < M ? A + (int64_t)(m0 + r) * K : nullptr; }, W + n0, N, N - n0);
#pragma unroll
    for (int j = 0; j < T::TN / 4; ++j) {
        const int n = n0 + T::col(j);
        if (n >= N) continue;                                       // N is a multiple of 8: whole strips
        const float b0 = __ldg(bias + n), b1 = __ldg(bias + n + 1), b2 = __ldg(bias + n + 2), b3 = __ldg(bias + n + 3);
#pragma unroll
        for (int i = 0; i < T::TM; ++i) {
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

// The top hidden layer (its columns are one tile) with all that hangs off it:
//   h = ReLU(A W + bias);  z = h . w_out + b_out;  p = sigmoid(z);  BCE in its overflow-safe form;  dz = (p - y) / M;
//   dA[b][j] = dz * w_out[j] where h[b][j] > 0, else 0 (in planes);  gw_out[j] += sum_b h dz;  gb_top[j] += sum_b dA
// h goes nowhere: nothing after this reads it.  Blocks walk the row tiles, so that the sums of a block leave it once.
template <class T, int MIN_BLOCKS, bool WVEC>
__global__ void __launch_bounds__(T::THREADS, MIN_BLOCKS)
fwd_top_kernel(int M, int N, int K, const float* __restrict__ A, const float* __restrict__ W, const float* __restrict__ bias,
               __nv_bfloat16* __restrict__ dA, int64_t stride, const TopArgs top) {
    wait_for_predecessor();
    if (gridDim.x * gridDim.y <= FEW_BLOCKS) let_successor_start();
    extern __shared__ float4 dyn_smem[];
    static_assert(T::TM <= T::LANES_C, "a lane per row of a thread's outputs");
    constexpr int WARPS = T::WR * T::WC;
    __shared__ float s_gw[T::WR][T::BN], s_gb[T::WR][T::BN];        // column sums, a row per row of warps
    __shared__ float s_z[T::WC][T::BM], s_part[2][WARPS];
    const int lane = (int)lane_id(), lc = lane % T::LANES_C, wr = T::warp_row(), wc = T::warp_col();
    for (int i = threadIdx.x; i < T::WR * T::BN; i += T::THREADS) { (&s_gw[0][0])[i] = 0.f; (&s_gb[0][0])[i] = 0.f; }
    float loss = 0.f, dz_sum = 0.f;
    const float b_out = __ldg(top.b_out);
    const int m_tiles = (M + T::BM - 1) / T::BM;
    for (int mt = blockIdx.x; mt < m_tiles; mt += gridDim.x) {
        const int m0 = mt * T::BM;
        typename T::Acc acc;
        T::template product<true, WVEC>(acc, K, reinterpret_cast<float*>(dyn_smem),
                                        [&](int r) -> const float* { return m0 + r < M ? A + (int64_t)(m0 + r) * K : nullptr; }, W, N, N);
        // activations; a lane's part of its rows' dot products
        float z[T::TM];
#pragma unroll
        for (int i = 0; i < T::TM; ++i) z[i] = 0.f;
        float h[T::TM][T::TN];
#pragma unroll
        for (int c = 0; c < T::TN; ++c) {
            const int n = T::col(c / 4) + c % 4;
            const bool on = n < N;
            const float b = on ? __ldg(bias + n) : 0.f, w = on ? __ldg(top.w_out + n) : 0.f;
#pragma unroll
            for (int i = 0; i < T::TM; ++i) {
                const float v = fmaxf(T::value(acc, i, c) + b, 0.f);
                h[i][c] = v >= 0x1.ffp127f ? __int_as_float(0x7f800000) : v;       // beyond the largest bf16 value: as infinite as in planes
                if (on) z[i] = fmaf(h[i][c], w, z[i]);
            }
        }
#pragma unroll
        for (int s = 1; s < T::LANES_C; s <<= 1)
#pragma unroll
            for (int i = 0; i < T::TM; ++i) z[i] += __shfl_xor_sync(0xffffffffu, z[i], s);
        if (T::WC > 1) {
            if (lc == 0)
#pragma unroll
                for (int i = 0; i < T::TM; ++i) s_z[wc][T::row(i)] = z[i];
            __syncthreads();
#pragma unroll
            for (int i = 0; i < T::TM; ++i) {
                z[i] = s_z[0][T::row(i)];
#pragma unroll
                for (int q = 1; q < T::WC; ++q) z[i] += s_z[q][T::row(i)];
            }
        }
        // lane lc of a row group works out row lc: sigmoid, loss, dz
        float zz = z[0];
        int m = m0 + T::row(0);
#pragma unroll
        for (int i = 1; i < T::TM; ++i) if (lc == i) { zz = z[i]; m = m0 + T::row(i); }
        zz += b_out;
        const float y = m < M ? __ldg(top.label + m) : 0.f;
        const float p = 1.0f / (1.0f + expf(-zz));
        const float dz = m < M ? (p - y) / (float)M : 0.f;
        if (lc < T::TM && wc == 0 && m < M) {
            loss += fmaxf(zz, 0.f) - zz * y + log1pf(expf(-fabsf(zz)));
            dz_sum += dz;
            if (top.prob) top.prob[m] = p;
        }
        float g[T::TM];
#pragma unroll
        for (int i = 0; i < T::TM; ++i) g[i] = __shfl_sync(0xffffffffu, dz, (lane - lc) + i);
#pragma unroll
        for (int j = 0; j < T::TN / 4; ++j) {
            const int n = T::col(j);
            float gw[4], gb[4], w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) { gw[e] = gb[e] = 0.f; w[e] = n < N ? __ldg(top.w_out + n + e) : 0.f; }
#pragma unroll
            for (int i = 0; i < T::TM; ++i) {
                const int row = m0 + T::row(i);
                if (row >= M || n >= N) continue;                    // N is a multiple of 8: whole strips
                float d[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float v = h[i][4 * j + e];
                    gw[e] = fmaf(v, g[i], gw[e]);
                    d[e] = v > 0.f ? g[i] * w[e] : 0.f;
                    gb[e] += d[e];
                }
                uint2 q[3];
                split3_pair(d[0], d[1], q[0].x, q[1].x, q[2].x);
                split3_pair(d[2], d[3], q[0].y, q[1].y, q[2].y);
#pragma unroll
                for (int t = 0; t < 3; ++t) *reinterpret_cast<uint2*>(dA + t * stride + (int64_t)row * N + n) = q[t];
            }
#pragma unroll
            for (int s = T::LANES_C; s < 32; s <<= 1)
#pragma unroll
                for (int e = 0; e < 4; ++e) { gw[e] += __shfl_xor_sync(0xffffffffu, gw[e], s); gb[e] += __shfl_xor_sync(0xffffffffu, gb[e], s); }
            if (lane < T::LANES_C)                                  // the warp's own words: nobody else adds to them
#pragma unroll
                for (int e = 0; e < 4; ++e) { s_gw[wr][n + e] += gw[e]; s_gb[wr][n + e] += gb[e]; }
        }
    }
    loss = warp_sum(loss);
    dz_sum = warp_sum(dz_sum);
    if (lane == 0) { s_part[0][threadIdx.x / 32] = loss; s_part[1][threadIdx.x / 32] = dz_sum; }
    __syncthreads();
    for (int n = threadIdx.x; n < N; n += T::THREADS) {
        float gw = s_gw[0][n], gb = s_gb[0][n];
#pragma unroll
        for (int q = 1; q < T::WR; ++q) { gw += s_gw[q][n]; gb += s_gb[q][n]; }
        atomicAdd(top.gw_out + n, gw);
        atomicAdd(top.gb_top + n, gb);
    }
    if (threadIdx.x == 0) {
        float l = 0.f, t = 0.f;
        for (int q = 0; q < WARPS; ++q) { l += s_part[0][q]; t += s_part[1][q]; }
        top.loss_part[blockIdx.x] = l;
        atomicAdd(top.gb_out, t);
    }
}

// Shared memory a block asks for: so much, where `even`, that no SM takes more of them than an even spread gives it.
constexpr int SM_SMEM = 228 * 1024, EVEN_SMEM_MAX = SM_SMEM / 2 - 512;
template <auto Kernel> static int even_smem(int own, int threads, int64_t blocks, bool even) {
    static const int fit = [&] { int n = 0; return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, Kernel, threads, own) == cudaSuccess ? n : 0; }();
    const int64_t per = ceil_div(blocks, sm_count());
    return even && per < fit ? (int)(SM_SMEM / (per + 1)) - 512 : own;                   // (a block takes 1 KB more than it asks for)
}

template <class T, int MIN_BLOCKS, bool WVEC>
static cudaError_t launch_form(bool even, int M, int N, int K, const float* A, const float* W, const float* bias, const Planes& H, float* Hf,
                               cudaStream_t st) {
    constexpr auto kernel = fwd_kernel<T, MIN_BLOCKS, WVEC>;
    static_assert(T::SMEM <= EVEN_SMEM_MAX, "two blocks per SM");
    if (const cudaError_t e = allow_smem<kernel>(EVEN_SMEM_MAX)) return e;
    const int64_t rows = ceil_div(M, T::BM), y = rows < 65535 ? rows : 65535;
    return launch_dependent(kernel, dim3((unsigned)ceil_div(N, T::BN), (unsigned)y, (unsigned)ceil_div(rows, y)), dim3(T::THREADS),
                            (size_t)even_smem<kernel>(T::SMEM, T::THREADS, rows * ceil_div(N, T::BN), even), st, M, N, K, A, W, bias, H.p, H.stride, Hf);
}

template <class T, int MIN_BLOCKS, bool WVEC>
static cudaError_t launch_top_form(bool even, int M, int N, int K, const float* A, const float* W, const float* bias, const Planes& dA,
                                   const TopArgs& top, int slots, int* n_part, cudaStream_t st) {
    constexpr auto kernel = fwd_top_kernel<T, MIN_BLOCKS, WVEC>;
    static_assert(T::SMEM <= EVEN_SMEM_MAX, "two blocks per SM");
    if (const cudaError_t e = allow_smem<kernel>(EVEN_SMEM_MAX)) return e;
    const int64_t tiles = ceil_div(M, T::BM), resident = (int64_t)sm_count() * MIN_BLOCKS;
    const int64_t most = resident < slots ? resident : slots;
    *n_part = (int)(tiles < most ? tiles : most);
    return launch_dependent(kernel, dim3((unsigned)*n_part), dim3(T::THREADS), (size_t)even_smem<kernel>(T::SMEM, T::THREADS, *n_part, even), st, M, N, K, A, W, bias, dA.p, dA.stride, top);
}

// Forms of a tile: outputs per lane, lanes, warps, steps per buffer, buffers.
typedef ChainTile<2, 4, 4, 8, 2, 1, 32, 4> F16x32;
typedef ChainTile<4, 4, 8, 4, 1, 2, 32, 4> F32x32;
typedef ChainTile<8, 8, 4, 8, 2, 2, 32, 2> F64x128;
typedef ChainTile<2, 4, 4, 8, 1, 2, 32, 4> F8x64;
typedef ChainTile<4, 4, 4, 8, 1, 2, 32, 4> F16x64;
typedef ChainTile<8, 8, 4, 8, 2, 1, 32, 2> F64x64;
typedef ChainTile<2, 4, 4, 8, 1, 4, 32, 3> F8x128;
typedef ChainTile<4, 4, 4, 8, 1, 4, 32, 3> F16x128;
typedef ChainTile<4, 4, 4, 8, 1, 8, 32, 3> F16x256;
typedef ChainTile<8, 8, 4, 8, 1, 4, 32, 2> F32x256;

// What a product takes in a form, in ns: per step of the reduction `alone` while no SM has more than one block, `shared` per block of the
// fullest SM where that is longer (blocks count in multiples of `unit`); `once` besides, of which what is beyond 1.5 us comes again
// with every round of tiles that `resident` blocks per SM walk.  The chain over the reduction cannot be split, so a product
// takes as long as its fullest SM.  Measured in a loop at depths of 96, 224, 608 and 1632, twelve batches of 64 to 16384 views and 32
// to 256 columns: the form that the sum names is within 5 % of the fastest at every one of them, the way (below) within 2.5 us.  A few of
// them (us, 1632 deep): 1024 x 128 in 16 x 32 tiles 22.0, in 32 x 32 26.4, in 64 x 128 82.6; 4096 x 256: 128, 96, 83.5.
struct Form {
    int bm, bn;
    float alone, shared, once;
    int unit, resident;
    // (sms: on so many SMs)
    float cost(int M, int N, int K, int sms) const {
        const int64_t tiles = ceil_div(M, bm) * ceil_div(N, bn), blocks = ceil_div(ceil_div(tiles, sms), unit) * unit;
        const float step = (float)blocks * shared, rounds = resident ? (float)ceil_div(tiles, (int64_t)resident * sm_count()) : 1.f;
        return 1500.f + (once - 1500.f) * rounds + (float)K * (step > alone ? step : alone);
    }
    // All blocks of a wave are placed within a microsecond, on the SMs that are free at that moment: 256 of them went to 75 SMs, four each,
    // while the ID sort and the expiry scan had begun on the other 73 (4096 x 1632 x 256: 164 us instead of 97, step 265 us instead of
    // 197; 1024 x 1632 x 256: 46 us and 32).  They are spread evenly where half of the SMs would take 8 us longer.  Elsewhere that
    // costs more than it gives, since the sort then waits for room (128 blocks of 16 x 32 outputs, 1632 deep: step 59.5 us as it comes,
    // 65.3 spread; of 8 x 64, 608 deep: 37.0, 39.3).
    bool even(int M, int N, int K) const { return cost(M, N, K, (sm_count() + 1) / 2) - cost(M, N, K, sm_count()) >= 8000.f; }
};
constexpr Form LOW[] = {{16, 32, 10.2f, 6.f, 1300.f, 1, 0}, {32, 32, 15.7f, 8.f, 1500.f, 1, 0}, {64, 128, 50.5f, 46.5f, 2700.f, 1, 0},
                        {64, 64, 51.f, 24.5f, 3100.f, 2, 0}};
constexpr Form TOP[] = {{16, 32, 12.f, 6.5f, 2300.f, 1, 4}, {32, 32, 17.5f, 10.2f, 2700.f, 1, 4},
                        {8, 64, 15.2f, 11.f, 2400.f, 1, 4}, {16, 64, 20.3f, 10.8f, 2600.f, 1, 4}, {64, 64, 50.5f, 25.f, 5000.f, 1, 4},
                        {8, 128, 21.7f, 15.f, 2400.f, 1, 3}, {16, 128, 24.8f, 17.8f, 2700.f, 1, 3}, {64, 128, 54.5f, 48.f, 4600.f, 1, 3},
                        {16, 256, 39.6f, 33.2f, 3100.f, 1, 2}, {32, 256, 61.5f, 55.f, 4600.f, 1, 2}};
// the cheapest of the forms of at least `cols` and less than 2 * max(cols, 32) columns (0: of any)
template <int COUNT> static int cheapest(const Form (&forms)[COUNT], int cols, int M, int N, int K, float* cost) {
    int best = -1;
    for (int f = 0; f < COUNT; ++f) {
        if (cols && (forms[f].bn < cols || forms[f].bn >= 2 * (cols > 32 ? cols : 32))) continue;
        const float c = forms[f].cost(M, N, K, sm_count());
        if (best < 0 || c < *cost) { best = f; *cost = c; }
    }
    return best;
}

// A tile over all columns takes longer for a step than a small one, and there are fewer of them: a deep layer is done sooner in small tiles
// with the output unit (head_out_kernel, 4 to 11 us) behind it.  Steps of the two ways, the output unit in the product / behind it (us):
// 1632 deep, 256 columns, 256 views 87.8 / 47.2, 1024 views 92 / 84; 608 deep, 136 columns, 256 views 47.4 / 35.1; 96 deep, 64 + 256
// columns, 1024 views 37.8 / 41.2.
bool fwd_top_fused_f32(int M, int N, int K) {
    if (N > F32_TOP_N) return false;
    float low, top;
    cheapest(LOW, 0, M, N, K, &low);
    cheapest(TOP, N, M, N, K, &top);
    return top <= low + 5000.f + (float)M * (0.25f + 0.0007f * (float)N);
}

cudaError_t launch_fwd_f32(const gear_ctx_impl& c, const char* name, int M, int N, int K, const float* A, const float* W, const float* bias,
                           const Planes& H, float* Hf, cudaStream_t st) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    KernelScope ks(&c.prof, name, st);
    const bool wvec = (reinterpret_cast<uintptr_t>(W) & 15u) == 0;
    float cost;
#define GEAR_FWD(T, MB) (wvec ? launch_form<T, MB, true>(even, M, N, K, A, W, bias, H, Hf, st) : launch_form<T, MB, false>(even, M, N, K, A, W, bias, H, Hf, st))
    const int f = cheapest(LOW, 0, M, N, K, &cost);
    const bool even = LOW[f].even(M, N, K);
    switch (f) {
    case 0: return GEAR_FWD(F16x32, 4);
    case 1: return GEAR_FWD(F32x32, 4);
    case 2: return GEAR_FWD(F64x128, 3);
    default: return GEAR_FWD(F64x64, 4);
    }
#undef GEAR_FWD
}

cudaError_t launch_fwd_top_f32(const gear_ctx_impl& c, int M, int N, int K, const float* A, const float* W, const float* bias,
                               const Planes& dA, const TopArgs& top, int* n_part, cudaStream_t st) {
    KernelScope ks(&c.prof, "f32_gemm_top", st);
    const bool wvec = (reinterpret_cast<uintptr_t>(W) & 15u) == 0;
    const int slots = c.ws.loss_slots;
    float cost;
#define GEAR_TOP(T, MB) (wvec ? launch_top_form<T, MB, true>(even, M, N, K, A, W, bias, dA, top, slots, n_part, st) \
                              : launch_top_form<T, MB, false>(even, M, N, K, A, W, bias, dA, top, slots, n_part, st))
    const int f = cheapest(TOP, N, M, N, K, &cost);
    const bool even = TOP[f].even(M, N, K);
    switch (f) {
    case 0: return GEAR_TOP(F16x32, 4);
    case 1: return GEAR_TOP(F32x32, 4);
    case 2: return GEAR_TOP(F8x64, 4);
    case 3: return GEAR_TOP(F16x64, 4);
    case 4: return GEAR_TOP(F64x64, 4);
    case 5: return GEAR_TOP(F8x128, 3);
    case 6: return GEAR_TOP(F16x128, 3);
    case 7: return GEAR_TOP(F64x128, 3);
    case 8: return GEAR_TOP(F16x256, 2);
    default: return GEAR_TOP(F32x256, 2);
    }
#undef GEAR_TOP
}

}  // namespace gear
