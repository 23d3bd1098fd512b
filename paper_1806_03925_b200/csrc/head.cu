// The Sparse Part's head (event 4): the order of its products, the output unit with the loss, and the weights' copies in
// the form the tensor-core products read.
//   forward        H_l    = ReLU(H_{l-1} W_l + b_l)
//   input gradient dH_{l-1} = (dA_l W_l^T) masked by H_{l-1} > 0
//   weight gradient dW_l  = H_{l-1}^T dA_l           (reduction over the batch, split over blocks)
// GEAR_BF16 heads: operands rounded to bf16 (head_tc.cu).  GEAR_F32 heads: every fp32 matrix is held as three bf16 planes
// whose sum it is for the backward products on the tensor cores (head_tc3.cu), and in fp32 for the forward ones (head_fwd.cu).
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "weights.cuh"

namespace gear {

struct F32x3 {};       // tag: fp32 values held as three bf16 planes

// Eight consecutive activations as they sit in memory (kept in registers between the two passes over a row).
template <typename TX> struct Raw8;
template <> struct Raw8<F32x3> {
    uint4 t[3];
    __device__ __forceinline__ void load(const __nv_bfloat16* p, int64_t stride) {
#pragma unroll
        for (int q = 0; q < 3; ++q) t[q] = *reinterpret_cast<const uint4*>(p + q * stride);
    }
    __device__ __forceinline__ void clear() { t[0] = t[1] = t[2] = make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ void unpack(float* v) const {
        const uint32_t a[4] = {t[0].x, t[0].y, t[0].z, t[0].w}, b[4] = {t[1].x, t[1].y, t[1].z, t[1].w}, c[4] = {t[2].x, t[2].y, t[2].z, t[2].w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {                      // both additions are exact
            v[2 * k] = (__uint_as_float(a[k] << 16) + __uint_as_float(b[k] << 16)) + __uint_as_float(c[k] << 16);
            v[2 * k + 1] = (__uint_as_float(a[k] & 0xffff0000u) + __uint_as_float(b[k] & 0xffff0000u)) + __uint_as_float(c[k] & 0xffff0000u);
        }
    }
};
template <> struct Raw8<__nv_bfloat16> {
    uint4 t;
    __device__ __forceinline__ void load(const __nv_bfloat16* p, int64_t) { t = *reinterpret_cast<const uint4*>(p); }
    __device__ __forceinline__ void clear() { t = make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ void unpack(float* v) const {
        const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) { v[2 * k] = __uint_as_float(w[k] << 16); v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u); }
    }
};

// stores 8 values in the head's form and leaves them as stored (rounded for bf16)
template <typename TX> __device__ __forceinline__ void store8(__nv_bfloat16* p, int64_t stride, float* v) {
    if constexpr (std::is_same<TX, F32x3>::value) {
        uint4 q0, q1, q2;
        split3_pair(v[0], v[1], q0.x, q1.x, q2.x); split3_pair(v[2], v[3], q0.y, q1.y, q2.y);
        split3_pair(v[4], v[5], q0.z, q1.z, q2.z); split3_pair(v[6], v[7], q0.w, q1.w, q2.w);
        *reinterpret_cast<uint4*>(p) = q0;
        *reinterpret_cast<uint4*>(p + stride) = q1;
        *reinterpret_cast<uint4*>(p + 2 * stride) = q2;
    } else {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
            w[k] = *reinterpret_cast<uint32_t*>(&h2);
            v[2 * k] = __uint_as_float(w[k] << 16);
            v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
        }
        *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Output unit, loss and everything that hangs off the top hidden layer:
//   z = h . w_out + b_out;  p = sigmoid(z);  BCE in its overflow-safe form;  dz = (p - y) / B
//   dA_top[b][j] = dz * w_out[j] where h[b][j] > 0, else 0            (stored in the head's form, planes `stride` apart)
//   gw_out[j] += sum_b h[b][j] dz[b];  gb_top[j] += sum_b dA_top[b][j];  gb_out += sum_b dz[b]
// A warp takes ROWS views at a time; a lane owns NQ = ceil(H / 256) chunks of 8 columns (128-bit loads and stores)
// and keeps its part of the ROWS rows in registers, so the top activations are read once.  The ROWS dot products
// are reduced together (a shuffle transpose-reduction: lane l ends up with the sum of row l >> (5 - log2 ROWS)),
// and sigmoid, loss and dz of the ROWS views are then worked out side by side, one view per group of lanes.
template <typename TX, int NQ, int ROWS>
__global__ void __launch_bounds__(256, NQ == 4 ? 1 : 2)
head_out_kernel(int B, int H, const __nv_bfloat16* __restrict__ h, int64_t stride, const float* __restrict__ w_out,
                const float* __restrict__ b_out, const float* __restrict__ label, float* __restrict__ prob,
                __nv_bfloat16* __restrict__ dA, float* __restrict__ loss_part,
                float* __restrict__ gw_out, float* __restrict__ gb_top, float* __restrict__ gb_out) {
    wait_for_predecessor();
    constexpr int LG = ROWS == 8 ? 3 : ROWS == 4 ? 2 : ROWS == 2 ? 1 : 0;
    static_assert((1 << LG) == ROWS, "ROWS is 1, 2, 4 or 8");
    __shared__ float part[8], gpart[8];
    __shared__ float s_gw[1024], s_gb[1024];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    for (int j = threadIdx.x; j < H; j += 256) { s_gw[j] = 0.f; s_gb[j] = 0.f; }
    float w[NQ][8], gw[NQ][8], gb[NQ][8];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int c0 = (lane + 32 * q) * 8;
#pragma unroll
        for (int k = 0; k < 8; ++k) { w[q][k] = c0 < H ? w_out[c0 + k] : 0.f; gw[q][k] = 0.f; gb[q][k] = 0.f; }
    }
    float local = 0.f, gsum = 0.f;
    const float bias = b_out[0];
    const int my_row = (int)(lane >> (5 - LG));            // the row of a batch whose sum this lane ends up with
    const bool my_first = (lane & ((32u >> LG) - 1u)) == 0u;   // one lane per row records the row's scalars
    __syncthreads();
    for (int b0 = (blockIdx.x * 8 + warp) * ROWS; b0 < B; b0 += gridDim.x * 8 * ROWS) {
        Raw8<TX> raw[ROWS][NQ];
        // the label of this lane's view: asked for first, so that its latency passes while the rows are summed
        const float y = b0 + my_row < B ? __ldg(label + b0 + my_row) : 0.f;
#pragma unroll
        for (int j = 0; j < ROWS; ++j)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int c0 = (lane + 32 * q) * 8;
                if (b0 + j < B && c0 < H) raw[j][q].load(h + (int64_t)(b0 + j) * H + c0, stride);
                else raw[j][q].clear();
            }
        float z[ROWS];
#pragma unroll
        for (int j = 0; j < ROWS; ++j) {
            z[j] = 0.f;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                float v[8];
                raw[j][q].unpack(v);
#pragma unroll
                for (int k = 0; k < 8; ++k) z[j] = fmaf(v[k], w[q][k], z[j]);
            }
        }
        // rows still held: ROWS, ROWS / 2, ..., 1; each round hands half of them to the lane 16, 8, 4 away
#pragma unroll
        for (int r = 0; r < LG; ++r) {
            const int s = 16 >> r, half = ROWS >> (r + 1);
            const bool upper = (lane & s) != 0;
#pragma unroll
            for (int i = 0; i < half; ++i) {
                const float send = upper ? z[i] : z[i + half];
                const float keep = upper ? z[i + half] : z[i];
                z[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
            }
        }
        float zz = z[0];
#pragma unroll
        for (int s = 16 >> LG; s >= 1; s >>= 1) zz += __shfl_xor_sync(0xffffffffu, zz, s);
        zz += bias;
        const int b = b0 + my_row;
        const bool live = b < B;
        const float p = 1.0f / (1.0f + expf(-zz));
        const float g = live ? (p - y) / (float)B : 0.f;
        if (live && my_first) {
            local += fmaxf(zz, 0.f) - zz * y + log1pf(expf(-fabsf(zz)));
            gsum += g;
            if (prob) prob[b] = p;
        }
#pragma unroll
        for (int j = 0; j < ROWS; ++j) {
            const float gj = __shfl_sync(0xffffffffu, g, j << (5 - LG));
            if (b0 + j >= B) continue;                        // warp-uniform
            __nv_bfloat16* drow = dA + (int64_t)(b0 + j) * H;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int c0 = (lane + 32 * q) * 8;
                if (c0 >= H) continue;
                float v[8], d[8];
                raw[j][q].unpack(v);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    gw[q][k] = fmaf(v[k], gj, gw[q][k]);
                    d[k] = v[k] > 0.f ? gj * w[q][k] : 0.f;
                }
                store8<TX>(drow + c0, stride, d);
#pragma unroll
                for (int k = 0; k < 8; ++k) gb[q][k] += d[k];
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int c0 = (lane + 32 * q) * 8;
        if (c0 >= H) continue;
#pragma unroll
        for (int k = 0; k < 8; ++k) { atomicAdd(&s_gw[c0 + k], gw[q][k]); atomicAdd(&s_gb[c0 + k], gb[q][k]); }
    }
    local = warp_sum(local);                 // one lane per row of a batch held that row's terms
    gsum = warp_sum(gsum);
    if (lane == 0) { part[warp] = local; gpart[warp] = gsum; }
    __syncthreads();
    for (int j = threadIdx.x; j < H; j += 256) { atomicAdd(gw_out + j, s_gw[j]); atomicAdd(gb_top + j, s_gb[j]); }
    if (threadIdx.x == 0) {
        float s = 0.f, t = 0.f;
        for (int k = 0; k < 8; ++k) { s += part[k]; t += gpart[k]; }
        loss_part[blockIdx.x] = s;
        atomicAdd(gb_out, t);
    }
}

// The weights' copies by themselves: of fp32 heads, and of an empty batch, which has no gather.
template <int PLANES>
__global__ void __launch_bounds__(256)
round_weights_kernel(const __grid_constant__ RoundArgs a) {
    wait_for_predecessor();
    round_weights_block<PLANES>(a, (int)blockIdx.x, (int)gridDim.x);
}

struct HeadParams {
    const float* W[MAX_LAYERS]; const float* b[MAX_LAYERS];
    float* gW[MAX_LAYERS]; float* gb[MAX_LAYERS];
    const float* w_out; const float* b_out; float* gw_out; float* gb_out;
    int fan[MAX_LAYERS + 1];
};

static HeadParams split_params(const gear_ctx_impl& c, float* grad) {
    HeadParams p;
    const float* base = c.buf.head_params;
    int64_t pos = 0;
    p.fan[0] = c.d_in;
    for (int l = 0; l < c.cfg.n_hidden; ++l) {
        const int h = c.cfg.hidden[l];
        p.W[l] = base + pos; p.gW[l] = grad + pos; pos += (int64_t)p.fan[l] * h;
        p.b[l] = base + pos; p.gb[l] = grad + pos; pos += h;
        p.fan[l + 1] = h;
    }
    p.w_out = base + pos; p.gw_out = grad + pos; pos += p.fan[c.cfg.n_hidden];
    p.b_out = base + pos; p.gb_out = grad + pos;
    return p;
}

// Where the parameters' gradient is put together.  The copy engine adds the weight gradients to it in 16-byte pieces; an fp32
// head may be handed a less aligned array: its gradient is then put together in the workspace and copied.
static float* grad_array(const gear_ctx_impl& c, const gear_step_out& o) {
    return (reinterpret_cast<uintptr_t>(o.head_grad) & 15u) == 0 ? o.head_grad : c.at<float>(c.ws.head_grad);
}

// bf16 copies or planes of the hidden layers' weights in both orientations (what the tensor-core products read).  Clears
// head_grad on the way.
RoundArgs round_args(const gear_ctx_impl& c, const gear_step_out& o) {
    RoundArgs ra = {};
    ra.grad = grad_array(c, o); ra.n_grad = c.n_params; ra.loss = o.loss;     // the loss of a batch is written after this
    int fan = c.d_in;
    int64_t pos = 0;
    for (int l = 0; l < c.cfg.n_hidden; ++l) {
        const int h = c.cfg.hidden[l];
        ra.fan_in[l] = fan; ra.fan_out[l] = h; ra.W[l] = c.buf.head_params + pos;
        ra.wb[l] = c.at<__nv_bfloat16>(c.ws.wb[l]); ra.wbt[l] = c.at<__nv_bfloat16>(c.ws.wbt[l]);
        ra.tiles[l] = (int)(ceil_div(fan, 32) * ceil_div(h, 32));
        pos += (int64_t)fan * h + h;
        fan = h;
    }
    return ra;
}
cudaError_t launch_round_weights(const gear_ctx_impl& c, const gear_step_out& o, cudaStream_t st) {
    const RoundArgs ra = round_args(c, o);
    KernelScope ks(&c.prof, "round_weights", st);
    return launch_dependent(c.cfg.head_dtype == GEAR_BF16 ? round_weights_kernel<1> : round_weights_kernel<3>,
                            dim3((unsigned)ra.blocks()), dim3(256), 0, st, ra);
}

// The head's matrices in the form the products take: bf16, or planes of an fp32 matrix
static Planes matrix_at(const gear_ctx_impl& c, size_t off, int64_t elems) { return Planes{c.at<__nv_bfloat16>(off), elems}; }

template <typename TX>
static cudaError_t run_head(const gear_ctx_impl& c, const gear_batch& bt, const gear_step_out& o, cudaStream_t st,
                            const HeadHooks& hooks) {
    constexpr bool BF = std::is_same<TX, __nv_bfloat16>::value;
    const int L = c.cfg.n_hidden, B = bt.B;
    float* grad = grad_array(c, o);
    const HeadParams p = split_params(c, grad);
    auto finish = [&]() -> cudaError_t {
        return grad != o.head_grad ? enqueue_copy(o.head_grad, grad, sizeof(float) * c.n_params, hooks.dw_stream) : cudaSuccess;
    };
    if (B <= 0) return finish();
    cudaError_t err = cudaSuccess;

    const int64_t max_b = c.cfg.max_batch;
    Planes H[MAX_LAYERS + 1], dA[MAX_LAYERS + 1] = {}, W[MAX_LAYERS], Wt[MAX_LAYERS];      // Wt: [out][in]
    H[0] = matrix_at(c, c.ws.x, max_b * p.fan[0]);
    for (int l = 0; l < L; ++l) {
        H[l + 1] = matrix_at(c, c.ws.h[l], max_b * p.fan[l + 1]);
        dA[l + 1] = matrix_at(c, c.ws.da[l], max_b * p.fan[l + 1]);
        W[l] = matrix_at(c, c.ws.wb[l], (int64_t)p.fan[l] * p.fan[l + 1]);
        Wt[l] = matrix_at(c, c.ws.wbt[l], (int64_t)p.fan[l] * p.fan[l + 1]);
    }
    float* loss_part = c.at<float>(c.ws.loss_part);

    // forward
    const int HT = p.fan[L];
    // a top layer whose columns are one tile of its product takes the output unit along (fp32: where that is the shorter way)
    const bool top_fused = BF ? HT <= TC_TOP_N : fwd_top_fused_f32(B, HT, p.fan[L - 1]);
    int n_part = 0;                                       // partial losses it leaves
    for (int l = 0; l < L; ++l) {
        const int K = p.fan[l], N = p.fan[l + 1];
        if (top_fused && l + 1 == L) {
            const TopArgs top{p.w_out, p.b_out, bt.label, o.prob, loss_part, p.gw_out, p.gb[l], p.gb_out};
            if constexpr (BF) err = tc_gemm_top(c, "tc_gemm_top", B, N, K, H[l].p, K, Wt[l].p, K, p.b[l], dA[L].p, top, &n_part, st);
            else err = launch_fwd_top_f32(c, B, N, K, c.at<float>(c.ws.xf[l]), p.W[l], p.b[l], dA[L], top, &n_part, st);
        } else if constexpr (BF)
            err = tc_gemm_kmajor(c, "tc_gemm_fwd", B, N, K, H[l].p, K, Wt[l].p, K, 0, H[l + 1].p, N, p.b[l], nullptr, 0, nullptr, LossSum{}, st);
        else
            err = launch_fwd_f32(c, top_fused ? "f32_gemm_low" : "f32_gemm_fwd", B, N, K, c.at<float>(c.ws.xf[l]), p.W[l], p.b[l], H[l + 1], l + 1 < L ? c.at<float>(c.ws.xf[l + 1]) : nullptr, st);
        if (err != cudaSuccess) return err;
    }
    if (!top_fused) {
        KernelScope ks(&c.prof, "head_out", st);
        const int nq = (int)ceil_div(HT, 256);
        // rows per warp and pass, as many as the registers hold.  (Up to 256 columns, one chunk a lane: fp32 heads only)
        const int rows = nq <= 1 ? 4 : nq == 2 && BF ? 2 : 1;
        // every warp gets the same number of passes where the batch allows it
        const int64_t batches = ceil_div(B, rows);
        const int64_t passes = ceil_div(batches, (int64_t)c.ws.loss_blocks * 8);
        const int blocks = n_part = (int)ceil_div(batches, 8 * passes);
#define GEAR_HEAD_OUT(NQ, ROWS) launch_dependent(head_out_kernel<TX, NQ, ROWS>, dim3(blocks), dim3(256), 0, st, B, HT, H[L].p, H[L].stride, p.w_out, p.b_out, bt.label, \
        o.prob, dA[L].p, loss_part, p.gw_out, p.gb[L - 1], p.gb_out)
        if (nq > 2) err = GEAR_HEAD_OUT(4, 1);
        else if constexpr (BF) err = GEAR_HEAD_OUT(2, 2);
        else err = nq <= 1 ? GEAR_HEAD_OUT(1, 4) : GEAR_HEAD_OUT(2, 1);
#undef GEAR_HEAD_OUT
        if (err != cudaSuccess) return err;
    }
    // dW_l = H_l^T dA_{l+1}, on the stream the hooks name
    const bool beside = hooks.dw_stream != st;
    auto weight_grad = [&](int l) -> cudaError_t {
        const int K = p.fan[l], N = p.fan[l + 1];
        if (beside) {
            err = enqueue_record(hooks.dw_ev[l], st);
            if (err == cudaSuccess) err = enqueue_wait(hooks.dw_stream, hooks.dw_ev[l]);
            if (err != cudaSuccess) return err;
        }
        if constexpr (BF) return tc_gemm_mnmajor(c, "tc_gemm_dw", K, N, B, H[l].p, K, dA[l + 1].p, N, p.gW[l], N, hooks.dw_stream);
        else return tc3_gemm_mnmajor(c, "tc3_gemm_dw", K, N, B, H[l], K, dA[l + 1], N, p.gW[l], N, hooks.dw_stream);
    };
    // backward.  The weight gradients run on a stream of their own, where the caller has one: as soon as dA_{l+1} exists, or after
    // dX, beside what the caller does with dX.  On one stream the gradient that the layers below wait for (dA_l, at the bottom
    // dX) comes first: once dX exists the caller's hook may start the embedding scatter on another stream.  The bias gradient of a lower layer is summed in the epilogue of the product
    // that makes its dA (the top layer's came with the output unit).
    for (int l = L - 1; l >= 0; --l) {
        const int K = p.fan[l], N = p.fan[l + 1];
        if (beside && !hooks.dw_last && (err = weight_grad(l)) != cudaSuccess) return err;
        const LossSum loss = l == L - 1 ? LossSum{loss_part, n_part, B, o.loss} : LossSum{};      // the product behind the output unit
        if constexpr (BF) {
            if (l > 0) err = tc_gemm_kmajor(c, "tc_gemm_dh", B, K, N, dA[l + 1].p, N, W[l].p, N, 1, dA[l].p, K, nullptr, H[l].p, K, p.gb[l - 1], loss, st);
            else err = tc_gemm_kmajor(c, "tc_gemm_dx", B, K, N, dA[l + 1].p, N, W[l].p, N, 2, o.dX, K, nullptr, nullptr, 0, nullptr, loss, st);
        } else {
            if (l > 0) err = tc3_gemm_kmajor(c, "tc3_gemm_dh", B, K, N, dA[l + 1], N, W[l], N, dA[l], nullptr, K, H[l].p, K, p.gb[l - 1], loss, st);
            else err = tc3_gemm_kmajor(c, "tc3_gemm_dx", B, K, N, dA[l + 1], N, W[l], N, Planes{}, o.dX, K, nullptr, 0, nullptr, loss, st);
        }
        if (err != cudaSuccess) return err;
        if (l == 0 && hooks.after_dx && (err = hooks.after_dx(hooks.arg)) != cudaSuccess) return err;
        if (!beside && (err = weight_grad(l)) != cudaSuccess) return err;
    }
    for (int l = 0; beside && hooks.dw_last && l < L; ++l)
        if ((err = weight_grad(l)) != cudaSuccess) return err;
    return finish();
}

cudaError_t launch_head(const gear_ctx_impl& c, const gear_batch& b, const gear_step_out& o, cudaStream_t st, const HeadHooks& hooks) {
    return c.cfg.head_dtype == GEAR_BF16 ? run_head<__nv_bfloat16>(c, b, o, st, hooks) : run_head<F32x3>(c, b, o, st, hooks);
}

}  // namespace gear
