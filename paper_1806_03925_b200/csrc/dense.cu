// The Slowgear side beyond the gradient store: a linear Dense Part and the optimiser of the paper's experiments.
//
//   dense forward   Section 3, events 2 and 3: the Dense Part turns an image's raw data into its Dense Feature Vector.
//                   Here the smallest Dense Part there is: DFV[id] = raw[id] . Wd  (raw [img_vocab][R], Wd [R][D]).
//   dense backward  Section 3, event 6, second half; Eq. 1, right factor: the averaged gradient of every completed
//                   group goes back through the Dense Part.  For the linear map dDFV[id][c] / dWd[r][c] = raw[id][r]:
//                   G[r][c] += sum over emissions e of raw[id_e][r] * avg_e[c].
//   Adam            Section 4: the optimiser of the paper's experiments, for dense parameter vectors (head, Wd) and for
//                   the rows of an embedding table that received a gradient in this step.
//
// The two products are fp32 FMA products with one operand gathered by Image ID (the tolerance is 1e-5).
#include "common.cuh"
#include "f32_chain.cuh"
#include "internal.h"

namespace gear {

constexpr int DT = 64;     // tile edge
constexpr int DK = 16;     // tile depth

// rows[k][c] = sum_r raw[ids[k]][r] * Wd[r][c],  k < min(n, *d_n),  c < D.  An ID outside [0, vocab) gives a zero row.
// A chain of R multiply-adds per output cannot be cut, so small tiles spread the live rows over the SMs (2500 rows of 1536
// values, 64 columns: 40 blocks of 64 x 64 took 242 us), and blocks walk the tiles so that a capacity far above the live
// count costs nothing.  32 x 32 tiles, 4 x 4 outputs per lane: bound by shared-memory reads (2 x 4 outputs in 16 x 64: 57 us for
// those rows, this 29, the same rows over and over; 38 in a loop pass, whose rows are other ones of a large table each time).  AVEC / BVEC: raw rows / Wd rows may be read 16 bytes at a time.
typedef ChainTile<4, 4, 8, 4, 1, 2, 32, 4> DenseTile;
template <bool AVEC, bool BVEC>
__global__ void __launch_bounds__(DenseTile::THREADS)
dense_forward_kernel(const float* __restrict__ raw, int64_t vocab, int R, const float* __restrict__ Wd, int D,
                     const int32_t* __restrict__ ids, int64_t n, const int64_t* __restrict__ d_n,
                     float* __restrict__ rows, int64_t ld, DevState* __restrict__ state) {
    wait_for_predecessor();
    constexpr int BM = DenseTile::BM, BN = DenseTile::BN;
    extern __shared__ float4 dyn_smem[];
    __shared__ int64_t row_of[BM];
    if (d_n) { const int64_t live = *d_n; n = live < n ? (live < 0 ? 0 : live) : n; }
    // Column tiles of a row tile are neighbours in the order, and the live tiles the first blocks', which sit on different SMs (with
    // a grid dimension for the columns the live blocks of its second half piled up four to an SM: 29 us became 57)
    const int n_tiles = (D + BN - 1) / BN;
    const int64_t tiles = (n + BM - 1) / BM * n_tiles;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t m0 = t / n_tiles * BM;
        const int n0 = (int)(t % n_tiles) * BN;
        __syncthreads();                                          // the tile before this one has been read
        if (threadIdx.x < BM) {
            int64_t id = -1;
            if (m0 + threadIdx.x < n) {
                id = ids[m0 + threadIdx.x];
                if (id < 0 || id >= vocab) { id = -1; atomicOr(&state->status, GEAR_DEV_BAD_ID); }
            }
            row_of[threadIdx.x] = id;
        }
        __syncthreads();
        // the tile's rows are random lines of a large table: all of them on their way at once, so that the steps of the chain wait
        // for the L2 only
        for (int q = threadIdx.x; q < BM * (int)ceil_div(R, 32); q += DenseTile::THREADS) {
            const int64_t id = row_of[q % BM];
            if (id >= 0) asm volatile("prefetch.global.L2 [%0];" :: "l"(raw + id * R + 32 * (q / BM)));
        }
        DenseTile::Acc acc;
        DenseTile::product<AVEC, BVEC>(acc, R, reinterpret_cast<float*>(dyn_smem),
                                       [&](int r) -> const float* { const int64_t id = row_of[r]; return id >= 0 ? raw + id * R : nullptr; },
                                       Wd + n0, D, D - n0);
#pragma unroll
        for (int i = 0; i < DenseTile::TM; ++i) {
            const int64_t m = m0 + DenseTile::row(i);
#pragma unroll
            for (int j = 0; j < DenseTile::TN / 4; ++j) {
                const int c = n0 + DenseTile::col(j);
                if (m >= n || c >= D) continue;                   // D is a multiple of 8: whole strips
                float* dst = rows + m * ld + c;
#pragma unroll
                for (int e = 0; e < 4; ++e) dst[e] = DenseTile::value(acc, i, 4 * j + e);
            }
        }
    }
}

// G[r][c] += sum over e in this block's slice of raw[ids[e]][r] * avg[e][c].  blockIdx.z walks slices of e_chunk emissions.
__global__ void __launch_bounds__(256)
dense_backward_kernel(const float* __restrict__ raw, int64_t vocab, int R, int D, const int32_t* __restrict__ ids,
                      const float* __restrict__ avg, int64_t ld_avg, int64_t n, const int64_t* __restrict__ d_n,
                      int e_chunk, float* __restrict__ G, DevState* __restrict__ state) {
    wait_for_predecessor();
    if (d_n) { const int64_t live = *d_n; n = live < n ? (live < 0 ? 0 : live) : n; }
    const int64_t e_begin = (int64_t)blockIdx.z * e_chunk;
    if (e_begin >= n) return;
    const int64_t e_end = min(n, e_begin + (int64_t)e_chunk);
    __shared__ float As[DK][DT + 4];       // [emission][r]
    __shared__ float Bs[DK][DT + 4];       // [emission][c]
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int r0 = blockIdx.y * DT, c0 = blockIdx.x * DT;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    int flags = 0;
    // a step's values travel while the one before it is added up (one after the other, an ID, its raw row and two barriers a step: a loop
    // pass of 1024 views with 256 emissions of 1536 values was 3 to 4 us longer)
    float ra[4], rb[4];
    auto fetch = [&](int64_t e0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int idx = tid + q * 256;
            const int k = idx >> 6, x = idx & 63;                  // both operands: emission slow, row / column fast
            const int64_t e = e0 + k;
            int64_t id = -1;
            if (e < e_end) {
                id = ids[e];
                if (id < 0 || id >= vocab) { id = -1; flags |= GEAR_DEV_BAD_ID; }
            }
            ra[q] = (id >= 0 && r0 + x < R) ? __ldg(raw + id * R + r0 + x) : 0.f;
            rb[q] = (id >= 0 && c0 + x < D) ? __ldg(avg + e * ld_avg + c0 + x) : 0.f;
        }
    };
    fetch(e_begin);
    for (int64_t e0 = e_begin; e0 < e_end; e0 += DK) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int idx = tid + q * 256;
            As[idx >> 6][idx & 63] = ra[q]; Bs[idx >> 6][idx & 63] = rb[q];
        }
        __syncthreads();
        if (e0 + DK < e_end) fetch(e0 + DK);
#pragma unroll
        for (int k = 0; k < DK; ++k) {
            const float4 a4 = *reinterpret_cast<const float4*>(&As[k][ty * 4]);
            const float4 b4 = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
            const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    if (flags) atomicOr(&state->status, flags);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + ty * 4 + i;
        if (r >= R) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + tx * 4 + j;
            if (c < D) atomicAdd(G + (int64_t)r * D + c, acc[i][j]);
        }
    }
}

cudaError_t launch_dense_forward(const gear_ctx_impl& c, const float* raw, int R, const float* Wd, const int32_t* ids,
                                 int64_t n, const int64_t* d_n, float* rows, int64_t ld, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    KernelScope k(&c.prof, "dense_forward", st);
    const int64_t want = ceil_div(n, DenseTile::BM) * ceil_div(c.cfg.dfv_dim, DenseTile::BN), cap = (int64_t)sm_count() * 4;
    const dim3 grid((unsigned)(want < cap ? want : cap));
    const bool avec = (R & 3) == 0 && (reinterpret_cast<uintptr_t>(raw) & 15u) == 0, bvec = (reinterpret_cast<uintptr_t>(Wd) & 15u) == 0;
    static_assert(DenseTile::SMEM + DenseTile::BM * 8 <= 48 * 1024, "a launch may have this much without asking");
#define GEAR_DF(A, B) launch_dependent(dense_forward_kernel<A, B>, grid, dim3(DenseTile::THREADS), (size_t)DenseTile::SMEM, st, raw, c.cfg.img_vocab, R, Wd, c.cfg.dfv_dim, ids, n, d_n, rows, ld, c.state())
    return avec ? (bvec ? GEAR_DF(true, true) : GEAR_DF(true, false)) : (bvec ? GEAR_DF(false, true) : GEAR_DF(false, false));
#undef GEAR_DF
}

cudaError_t launch_dense_backward(const gear_ctx_impl& c, const float* raw, int R, const int32_t* ids, const float* avg,
                                  int64_t ld_avg, int64_t n, const int64_t* d_n, float* G, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    KernelScope k(&c.prof, "dense_backward", st);
    // slices of the emission list: enough of them to fill the GPU a few times over, each at least 64 emissions long (the list's
    // live count is usually far below n: 256 of 1024 emissions were one slice of 24 blocks, 32 us)
    const int64_t tiles = ceil_div(c.cfg.dfv_dim, DT) * ceil_div(R, DT);
    int64_t slices = ceil_div((int64_t)sm_count() * 8, tiles);
    const int64_t max_slices = ceil_div(n, 64);
    if (slices > max_slices) slices = max_slices;
    if (slices < 1) slices = 1;
    if (slices > 65535) slices = 65535;
    const int e_chunk = (int)(ceil_div(ceil_div(n, slices), DK) * DK);
    const dim3 grid((unsigned)ceil_div(c.cfg.dfv_dim, DT), (unsigned)ceil_div(R, DT), (unsigned)ceil_div(n, e_chunk));
    return launch_dependent(dense_backward_kernel, grid, dim3(256), 0, st, raw, c.cfg.img_vocab, R, c.cfg.dfv_dim, ids, avg, ld_avg,
                            n, d_n, e_chunk, G, c.state());
}

// ---------------------------------------------------------------- Adam (Kingma and Ba 2015, Algorithm 1)
struct AdamCoef { float lr, b1, b2, eps, inv_c1, inv_c2; };      // inv_c1 = 1 / (1 - b1^t), inv_c2 = 1 / (1 - b2^t)

__device__ __forceinline__ void adam_update(float& p, float g, float& m, float& v, const AdamCoef& a) {
    m = a.b1 * m + (1.f - a.b1) * g;
    v = a.b2 * v + (1.f - a.b2) * g * g;
    p -= a.lr * (m * a.inv_c1) / (sqrtf(v * a.inv_c2) + a.eps);
}

__global__ void __launch_bounds__(256)
adam_dense_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                  int64_t n, const AdamCoef a) {
    wait_for_predecessor();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float pi = p[i], mi = m[i], vi = v[i];
        adam_update(pi, g[i], mi, vi, a);
        p[i] = pi; m[i] = mi; v[i] = vi;
    }
}

static AdamCoef adam_coef(const gear_adam& cfg, int64_t t) {
    const double c1 = 1.0 - pow((double)cfg.beta1, (double)t), c2 = 1.0 - pow((double)cfg.beta2, (double)t);
    return AdamCoef{cfg.lr, cfg.beta1, cfg.beta2, cfg.eps, (float)(1.0 / c1), (float)(1.0 / c2)};
}

cudaError_t launch_adam_dense(Profiler* prof, float* p, const float* g, float* m, float* v, int64_t n, int64_t t,
                              const gear_adam& cfg, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    KernelScope k(prof, "adam_dense", st);
    const int64_t want = ceil_div(n, 256), cap = (int64_t)sm_count() * 8;
    return launch_dependent(adam_dense_kernel, dim3((unsigned)(want < cap ? want : cap)), dim3(256), 0, st, p, g, m, v, n,
                            adam_coef(cfg, t));
}

// ---------------------------------------------------------------- Adam on the embedding rows a step touched
// The summed gradient of every distinct ID of the batch sits in a compact buffer, in the row of the sorted position
// at which the ID's run starts (emb_scatter.cu).  One lane group per sorted position: a position that starts a run
// takes the Adam step of its ID's table row and moment rows; the others have nothing to do.
template <int NQ>
__global__ void __launch_bounds__(256)
emb_adam_rows_kernel(const EmbAdamTable t0, const EmbAdamTable t1, int n, int E, int lpr, const AdamCoef a) {
    wait_for_predecessor();
    const EmbAdamTable& t = blockIdx.y == 0 ? t0 : t1;
    const int64_t gthread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t p = gthread / lpr;
    const int c = (int)(gthread % lpr);
    if (p >= n) return;
    const uint32_t key = t.ks[p];
    if (key >= t.vocab || (p > 0 && t.ks[p - 1] == key)) return;
    const int n_chunks = E / 4;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int ch = c + q * lpr;
        if (ch >= n_chunks) continue;
        const float4 g = ld_f4(t.gsum + p * (int64_t)E + ch * 4);
        float* prow = t.table + (int64_t)key * E + ch * 4;
        float* mrow = t.m + (int64_t)key * E + ch * 4;
        float* vrow = t.v + (int64_t)key * E + ch * 4;
        float4 pv = ld_f4(prow), mv = ld_f4(mrow), vv = ld_f4(vrow);
        adam_update(pv.x, g.x, mv.x, vv.x, a); adam_update(pv.y, g.y, mv.y, vv.y, a);
        adam_update(pv.z, g.z, mv.z, vv.z, a); adam_update(pv.w, g.w, mv.w, vv.w, a);
        st_f4(prow, pv); st_f4(mrow, mv); st_f4(vrow, vv);
    }
}

cudaError_t launch_emb_adam_rows(const gear_ctx_impl& c, const EmbAdamTable& t0, const EmbAdamTable& t1, int32_t B,
                                 int64_t t, const gear_adam& cfg, cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    const int E = c.cfg.emb_dim, n_chunks = E / 4;
    int lpr = 1;
    while (lpr < n_chunks && lpr < 32) lpr <<= 1;
    const int nq = (int)ceil_div(n_chunks, lpr);
    const dim3 grid((unsigned)ceil_div((int64_t)B * lpr, 256), 2);
    const AdamCoef a = adam_coef(cfg, t);
    KernelScope ks(&c.prof, "emb_adam_rows", st);
#define GEAR_EA_LAUNCH(NQ) launch_dependent(emb_adam_rows_kernel<NQ>, grid, dim3(256), 0, st, t0, t1, (int)B, E, lpr, a)
    if (nq <= 1) return GEAR_EA_LAUNCH(1);
    if (nq <= 2) return GEAR_EA_LAUNCH(2);
    if (nq <= 4) return GEAR_EA_LAUNCH(4);
    return GEAR_EA_LAUNCH(8);
#undef GEAR_EA_LAUNCH
}

}  // namespace gear
