// Backward matrix products of fp32 heads (GEAR_F32) on the 5th-generation tensor cores.
//
// Every fp32 operand is held as three bf16 matrices ("planes"): a = a0 + a1 + a2 with a0 = bf16(a), a1 = bf16(a - a0),
// a2 = bf16(a - a0 - a1), each rounded to nearest.  The three hold 24 significant bits, so the sum is the fp32 value itself
// (|a| < 3.38e38; parts below 2^-133 are lost).  A product of two operands is the six tensor-core products
//     a0 b0  +  (a0 b1 + a1 b0 + a1 b1 + a0 b2 + a2 b0),
// each exact, added in fp32; what is left out (a1 b2, a2 b1, a2 b2) is below 2^-26 of |a b|, a quarter of the rounding
// unit of one fp32 multiply-add.  The leading product and the other five have an accumulator each: the accumulator of
// the small terms rounds at 2^-8 of the scale, and the leading one sees one addition per 16 products where an fp32
// multiply-add chain rounds after every one.
//
// Bound: six bf16 products per fp32 product, against 128 fp32 multiply-adds per SM and cycle on the ordinary lanes.
//
// One persistent kernel, one CTA per SM, the same roles as the bf16 products (head_tc.cu): warp 0 streams operand tiles
// with TMA (all three planes of a 128 x 32 or BN x 32 box in one copy), warp 1 issues tcgen05.mma, warps 2-9 drain one pair
// of accumulators while the next tile fills the other.  Tiles are 32 deep so that three stages of two operands with three
// planes each (48 KB) fit beside the output blocks.  Epilogues: ReLU mask, split into planes again (matrices stay in planes
// between the products; masked outputs also sum their columns, the bias gradient of the layer below); plain fp32 (dX); fp32 added to memory by the copy engine (weight gradients, reduction over the batch
// split across CTAs).  Every wait is bounded.
#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace gear {

constexpr int T3_BK = 32;                 // 32 bf16 = 64 bytes = one row of the 64-byte swizzle
constexpr int T3_EW = 8;                  // epilogue warps
constexpr int T3_THREADS = 64 + 32 * T3_EW;
constexpr int T3_MAX_N = 1024;

enum { T3_MASK = 1, T3_F32 = 2, T3_RED = 3 };

template <int BN, int EPI> struct T3Cfg {
    static constexpr bool PLANES_OUT = EPI == T3_MASK;
    static constexpr int A_PLANE = TC_BM * T3_BK * 2, A_BYTES = 3 * A_PLANE;
    static constexpr int B_PLANE = BN * T3_BK * 2, B_BYTES = 3 * B_PLANE;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int OUT_BLOCK = PLANES_OUT ? 3 * 32 * 64 : 32 * 128;     // a warp's 32 x 32 block on its way out
    static constexpr int OUT_BYTES = T3_EW * OUT_BLOCK;
    static constexpr int VEC_BYTES = PLANES_OUT ? T3_MAX_N * 4 : 0;           // the CTA's column sums
    static constexpr int FIXED = 1024 /*alignment slack*/ + 256 /*barriers*/ + VEC_BYTES + OUT_BYTES;
    static constexpr int ROOM = (227 * 1024 - FIXED) / STAGE_BYTES;
    static constexpr int STAGES = ROOM > 6 ? 6 : ROOM;
    static constexpr int SMEM = STAGES * STAGE_BYTES + FIXED;
    static constexpr int TMEM_COLS = 4 * BN;                                  // two buffers of two accumulators
    static_assert(STAGES >= 3, "operand ring too short");
    static_assert(SMEM > 116 * 1024 && SMEM <= 227 * 1024, "one CTA per SM");
};

struct T3Args {
    int M, N, K;
    int m_tiles, n_tiles, k_splits, kb_per_split;   // kb = blocks of T3_BK along K
    const __nv_bfloat16* mask; int64_t ldm;         // T3_MASK: leading plane of the activations (positive where they are)
    float* colsum;                                  // T3_MASK: colsum[n] += column sums of the masked output (may be null)
    int32_t* err;
    LossSum loss;             // the loss to finish
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
                 :: "r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(0) : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
                 :: "l"(map), "r"(src), "r"(x), "r"(y), "r"(0) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// A finished 32 x 32 block (rows m0 + lane, columns n0 ..) of an epilogue warp on its way out.
template <int EPI>
__device__ __forceinline__ void t3_emit(const T3Args& g, const CUtensorMap* map_out, float (&v)[32], const uint4 (&mk)[4], int m0,
                                        int n0, int lane, float* s_vec, uint32_t out_buf, uint64_t keep_policy) {
    if (EPI == T3_MASK) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t w[4] = {mk[j].x, mk[j].y, mk[j].z, mk[j].w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {                       // activations are >= 0: positive means any bit is set
                v[8 * j + 2 * q] = (w[q] & 0x7fffu) ? v[8 * j + 2 * q] : 0.f;
                v[8 * j + 2 * q + 1] = (w[q] & 0x7fff0000u) ? v[8 * j + 2 * q + 1] : 0.f;
            }
        }
    }
    if (lane == 0) tma_store_wait_read<0>();                    // the block's previous contents have left
    __syncwarp();
    if (EPI == T3_MASK) {
        const uint32_t row_addr = out_buf + (uint32_t)lane * 64u, swz = ((uint32_t)lane >> 1) & 3u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint4 p0, p1, p2;
            split3_pair(v[8 * j + 0], v[8 * j + 1], p0.x, p1.x, p2.x);
            split3_pair(v[8 * j + 2], v[8 * j + 3], p0.y, p1.y, p2.y);
            split3_pair(v[8 * j + 4], v[8 * j + 5], p0.z, p1.z, p2.z);
            split3_pair(v[8 * j + 6], v[8 * j + 7], p0.w, p1.w, p2.w);
            const uint32_t at = row_addr + ((((uint32_t)j) ^ swz) << 4);
            sts_u4(at, p0); sts_u4(at + 2048u, p1); sts_u4(at + 4096u, p2);
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) tma_store_3d(map_out, out_buf, n0, m0);
        if (EPI == T3_MASK && g.colsum != nullptr) {
            // sums over the block's 32 rows (one per lane): each round hands half of the columns still held to the lane
            // 16, 8, 4, 2, 1 away; lane l ends up with column l.  Rows past M are zero.
#pragma unroll
            for (int r = 0; r < 5; ++r) {
                const int s = 16 >> r;
                const bool upper = (lane & s) != 0;
#pragma unroll
                for (int i = 0; i < s; ++i) {
                    const float send = upper ? v[i] : v[i + s], keep = upper ? v[i + s] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
                }
            }
            if (n0 + lane < g.N) atomicAdd(&s_vec[n0 + lane], v[0]);
        }
    } else {
        const uint32_t row_addr = out_buf + (uint32_t)lane * 128u, swz = (uint32_t)(lane & 7);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            sts_u4(row_addr + (((uint32_t)j ^ swz) << 4),
                   make_uint4(__float_as_uint(v[4 * j]), __float_as_uint(v[4 * j + 1]), __float_as_uint(v[4 * j + 2]), __float_as_uint(v[4 * j + 3])));
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
            if (EPI == T3_RED) tma_reduce_add_2d(map_out, out_buf, n0, m0);
            else tma_store_2d_hint(map_out, out_buf, n0, m0, keep_policy);      // dX is read again right after
        }
    }
}

template <int EPI>
__device__ __forceinline__ void t3_load_mask(const T3Args& g, uint4 (&mk)[4], int m, int n0) {
    if (EPI != T3_MASK) return;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        mk[j] = (m < g.M && n0 + 8 * j < g.N) ? ldg_u4(g.mask + (int64_t)m * g.ldm + n0 + 8 * j) : make_uint4(0u, 0u, 0u, 0u);
}

// SEG: the reduction is cut into segments of T3_SEG tiles; every segment has accumulators of its own and the epilogue warps
// add the segments up in registers (fp32, rounded to nearest).  A tensor-core accumulator loses the bits below its last
// one at every addition, so its error grows with the number of additions; 16 per segment keep it below what a chain of
// fp32 multiply-adds over the same terms collects.
constexpr int T3_SEG = 8;                 // 8 * 32 terms: 16 additions

template <int BN, bool MN_MAJOR, int EPI, bool SEG>
__global__ void __maxnreg__(SEG ? 168 : 128)
t3_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_out, const T3Args g) {
    using Cfg = T3Cfg<BN, EPI>;
    constexpr int STAGES = Cfg::STAGES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;
    const uint32_t out_blocks = tiles + STAGES * Cfg::STAGE_BYTES;
    const uint32_t bars = out_blocks + Cfg::OUT_BYTES;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
    auto acc_full = [&](int a) { return bars + 8u * (2 * STAGES + a); };
    auto acc_empty = [&](int a) { return bars + 8u * (2 * STAGES + 2 + a); };
    const uint32_t tmem_word = bars + 8u * (2 * STAGES + 4);
    volatile uint32_t* tmem_word_ptr = reinterpret_cast<volatile uint32_t*>(smem_raw + (tmem_word - raw));
    float* s_vec = reinterpret_cast<float*>(smem_raw + (bars + 256u - raw));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total_tiles = g.m_tiles * g.n_tiles * g.k_splits;
    const int total_kb = (g.K + T3_BK - 1) / T3_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(acc_full(a), 1); mbar_init(acc_empty(a), 32 * T3_EW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&map_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&map_b) : "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&map_out) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tmem_word), "r"((uint32_t)Cfg::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (EPI == T3_MASK)
        for (int n = threadIdx.x; n < T3_MAX_N; n += T3_THREADS) s_vec[n] = 0.f;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_word_ptr;
    wait_for_predecessor();
    if (EPI != T3_F32 && gridDim.x <= FEW_BLOCKS) let_successor_start();

    if (warp == 0) {
        // ---------------- TMA producer
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x) {
                const int nt = t % g.n_tiles, mt = (t / g.n_tiles) % g.m_tiles, ks = t / (g.m_tiles * g.n_tiles);
                const int kb0 = ks * g.kb_per_split, kb1 = min(total_kb, kb0 + g.kb_per_split);
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const int s = it % STAGES;
                    if (!(ok = mbar_wait(empty_bar(s), ((it / STAGES) & 1u) ^ 1u, g.err, 11))) break;
                    const uint32_t a_dst = tiles + s * Cfg::STAGE_BYTES, b_dst = a_dst + Cfg::A_BYTES;
                    mbar_expect_tx(full_bar(s), Cfg::STAGE_BYTES);
                    if (!MN_MAJOR) {
                        tma_load_3d(a_dst, &map_a, full_bar(s), kb * T3_BK, mt * TC_BM);     // 3 planes of 128 rows x 32 k
                        tma_load_3d(b_dst, &map_b, full_bar(s), kb * T3_BK, nt * BN);
                    } else {
                        // 3 planes of 32 k-rows x 64 columns per box: the slabs of one operand sit 12 KB apart
#pragma unroll
                        for (int j = 0; j < TC_BM / 64; ++j)
                            tma_load_3d(a_dst + j * 12288, &map_a, full_bar(s), mt * TC_BM + j * 64, kb * T3_BK);
#pragma unroll
                        for (int j = 0; j < BN / 64; ++j)
                            tma_load_3d(b_dst + j * 12288, &map_b, full_bar(s), nt * BN + j * 64, kb * T3_BK);
                    }
                }
            }
            if (*reinterpret_cast<volatile int32_t*>(g.err) != 0) {
                // leaving early: let the copies already issued land before the CTA gives its shared memory back
                const uint32_t first = it > (uint32_t)STAGES ? it - STAGES : 0u;
                for (uint32_t j = first; j < it; ++j)
                    for (uint32_t spin = 0; spin < (1u << 16) && !mbar_try(full_bar(j % STAGES), (j / STAGES) & 1u); ++spin)
                        __nanosleep(64);
            }
        }
        if (blockIdx.x == 0) { __syncwarp(); sum_loss(g.loss, lane); }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc = instr_desc(BN, MN_MAJOR);
            uint32_t it = 0, unit = 0;             // unit: a tile, or a segment of one
            bool ok = true;
            for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x) {
                const int ks = t / (g.m_tiles * g.n_tiles);
                const int kb0 = ks * g.kb_per_split, kb1 = min(total_kb, kb0 + g.kb_per_split);
                for (int s0 = kb0; s0 < kb1 && ok; s0 = SEG ? s0 + T3_SEG : kb1, ++unit) {
                const int s1 = SEG ? min(kb1, s0 + T3_SEG) : kb1;
                const int a = unit & 1;
                if (!(ok = mbar_wait(acc_empty(a), ((unit >> 1) & 1u) ^ 1u, g.err, 12))) break;
                tc_fence_after();
                const uint32_t d_hi = tmem_base + (uint32_t)(a * 2 * BN), d_lo = d_hi + BN;
                for (int kb = s0; kb < s1; ++kb, ++it) {
                    const int s = it % STAGES;
                    if (!(ok = mbar_wait(full_bar(s), (it / STAGES) & 1u, g.err, 13))) break;
                    tc_fence_after();
                    const uint32_t a_src = tiles + s * Cfg::STAGE_BYTES, b_src = a_src + Cfg::A_BYTES;
#pragma unroll
                    for (int k = 0; k < T3_BK / 16; ++k) {
                        uint64_t da[3], db[3];
#pragma unroll
                        for (int p = 0; p < 3; ++p) {
                            if (!MN_MAJOR) {
                                da[p] = smem_desc<64>(a_src + p * Cfg::A_PLANE + k * 32, 16, 512);
                                db[p] = smem_desc<64>(b_src + p * Cfg::B_PLANE + k * 32, 16, 512);
                            } else {
                                da[p] = smem_desc<128>(a_src + p * 4096 + k * 2048, 12288, 1024);
                                db[p] = smem_desc<128>(b_src + p * 4096 + k * 2048, 12288, 1024);
                            }
                        }
                        const uint32_t more = (kb > s0 || k > 0) ? 1u : 0u;
                        tc_mma(d_lo, da[0], db[2], idesc, more);
                        tc_mma(d_lo, da[2], db[0], idesc, 1u);
                        tc_mma(d_lo, da[1], db[1], idesc, 1u);
                        tc_mma(d_lo, da[0], db[1], idesc, 1u);
                        tc_mma(d_lo, da[1], db[0], idesc, 1u);
                        tc_mma(d_hi, da[0], db[0], idesc, more);
                    }
                    tc_commit(empty_bar(s));
                }
                if (ok) tc_commit(acc_full(a));
                }
            }
        }
    } else {
        // ---------------- epilogue warps
        const uint32_t out_buf = out_blocks + (uint32_t)((warp - 2) * Cfg::OUT_BLOCK);
        const uint64_t keep_policy = l2_policy_evict_last();
        constexpr int COLS = BN / 2, CHUNKS = COLS / 32;       // a warp: 32 rows of the tile, half of its columns
        const int quarter = warp & 3, part = (warp - 2) >> 2;
        uint32_t unit = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x) {
            const int nt = t % g.n_tiles, mt = (t / g.n_tiles) % g.m_tiles, ks = t / (g.m_tiles * g.n_tiles);
            const int kb0 = ks * g.kb_per_split, kb1 = min(total_kb, kb0 + g.kb_per_split);
            const int m0 = mt * TC_BM + quarter * 32, col0 = nt * BN + part * COLS;
            float sum[SEG ? CHUNKS : 1][32];
            for (int s0 = kb0; s0 < kb1; s0 = SEG ? s0 + T3_SEG : kb1, ++unit) {
                const int a = unit & 1;
                if (!(ok = mbar_wait(acc_full(a), (unit >> 1) & 1u, g.err, 14))) break;
                tc_fence_after();
                const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * 2 * BN + part * COLS);
                if constexpr (SEG) {
#pragma unroll
                    for (int h = 0; h < 2 * CHUNKS; ++h) {
                        uint32_t hi[16], lo[16];
                        tc_ld16(t_row + (uint32_t)(h * 16), hi);
                        tc_ld16(t_row + (uint32_t)(BN + h * 16), lo);
                        tc_wait_ld(hi);
                        tc_wait_ld(lo);
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float x = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
                            float& y = sum[h / 2][(h & 1) * 16 + i];
                            y = s0 == kb0 ? x : y + x;
                        }
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < CHUNKS; ++c) {
                        uint32_t hi[32], lo[32];
                        uint4 mk[4];
                        tc_ld32(t_row + (uint32_t)(c * 32), hi);
                        tc_ld32(t_row + (uint32_t)(BN + c * 32), lo);
                        t3_load_mask<EPI>(g, mk, m0 + lane, col0 + c * 32);
                        tc_wait_ld(hi);
                        tc_wait_ld(lo);
                        if (col0 + c * 32 >= g.N || m0 >= g.M) continue;            // warp-uniform
#pragma unroll
                        for (int i = 0; i < 32; ++i) sum[0][i] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
                        t3_emit<EPI>(g, &map_out, sum[0], mk, m0, col0 + c * 32, lane, s_vec, out_buf, keep_policy);
                    }
                }
                tc_fence_before();
                mbar_arrive_relaxed(acc_empty(a));
            }
            if constexpr (SEG) {
                if (!ok) break;
#pragma unroll
                for (int c = 0; c < CHUNKS; ++c) {
                    if (col0 + c * 32 >= g.N || m0 >= g.M) continue;
                    uint4 mk[4];
                    t3_load_mask<EPI>(g, mk, m0 + lane, col0 + c * 32);
                    t3_emit<EPI>(g, &map_out, sum[c], mk, m0, col0 + c * 32, lane, s_vec, out_buf, keep_policy);
                }
            }
        }
        if (lane == 0) tma_store_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    if (EPI == T3_MASK && g.colsum != nullptr)
        for (int n = threadIdx.x; n < g.N; n += T3_THREADS) {
            const float v = s_vec[n];
            if (v != 0.f) atomicAdd(g.colsum + n, v);
        }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     :: "r"(tmem_base), "r"((uint32_t)Cfg::TMEM_COLS) : "memory");
    }
}

// ---------------------------------------------------------------- host side
template <int BN, bool MN, int EPI, bool SEG>
static cudaError_t t3_launch_as(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mo, const T3Args& g, cudaStream_t st) {
    using Cfg = T3Cfg<BN, EPI>;
    constexpr auto kernel = t3_gemm_kernel<BN, MN, EPI, SEG>;
    if (const cudaError_t e = allow_smem<kernel>(Cfg::SMEM)) return e;
    const int tiles = g.m_tiles * g.n_tiles * g.k_splits;
    return launch_dependent(kernel, dim3(tiles < sm_count() ? tiles : sm_count()), dim3(T3_THREADS), (size_t)Cfg::SMEM, st, ma, mb, mo, g);
}

// Segments where a tile's reduction is more than two of them long.
template <int BN, bool MN, int EPI>
static cudaError_t t3_launch(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mo, const T3Args& g, cudaStream_t st) {
    return g.kb_per_split > 2 * T3_SEG ? t3_launch_as<BN, MN, EPI, true>(ma, mb, mo, g, st) : t3_launch_as<BN, MN, EPI, false>(ma, mb, mo, g, st);
}

// Column tiles of 128, or of 64 where the output is narrow or 128-wide tiles would leave more than half of the SMs idle
// (small batches: the time of a product is then its longest tile's).
static int t3_bn(const T3Args& g) {
    return g.N <= 64 || ceil_div(g.M, TC_BM) * ceil_div(g.N, 128) * 2 <= sm_count() ? 64 : 128;
}

cudaError_t tc3_gemm_kmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const Planes& A, int64_t lda,
                            const Planes& W, int64_t ldw, const Planes& out_planes, float* out_f32, int64_t ldo,
                            const __nv_bfloat16* mask, int64_t ldm, float* colsum, const LossSum& loss, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    T3Args g{};
    g.M = M; g.N = N; g.K = K; g.loss = loss;
    const int bn = t3_bn(g);
    g.m_tiles = (int)ceil_div(M, TC_BM); g.n_tiles = (int)ceil_div(N, bn);
    g.k_splits = 1; g.kb_per_split = (int)ceil_div(K, T3_BK);
    g.mask = mask; g.ldm = ldm; g.colsum = colsum; g.err = &c.state()->tc_error;
    if (N > T3_MAX_N && mask) return cudaErrorInvalidValue;
    CUtensorMap ma, mb, mo;
    if (!c.tma->get(&ma, TmaSpec{A.p, M, K, lda, A.stride, 3, TC_BM, T3_BK, 0, 64}) ||
        !c.tma->get(&mb, TmaSpec{W.p, N, K, ldw, W.stride, 3, bn, T3_BK, 0, 64}) ||
        !c.tma->get(&mo, mask ? TmaSpec{out_planes.p, M, N, ldo, out_planes.stride, 3, 32, 32, 0, 64}
                              : TmaSpec{out_f32, M, N, ldo, 0, 1, 32, 32, 1, 128}))
        return cudaErrorInvalidValue;
    KernelScope ks(&c.prof, name, st);
    if (mask) return bn == 128 ? t3_launch<128, false, T3_MASK>(ma, mb, mo, g, st) : t3_launch<64, false, T3_MASK>(ma, mb, mo, g, st);
    return bn == 128 ? t3_launch<128, false, T3_F32>(ma, mb, mo, g, st) : t3_launch<64, false, T3_F32>(ma, mb, mo, g, st);
}

cudaError_t tc3_gemm_mnmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const Planes& A, int64_t lda,
                             const Planes& Bm, int64_t ldb, float* out, int64_t ldo, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    T3Args g{};
    g.M = M; g.N = N; g.K = K;
    const int bn = N <= 64 ? 64 : 128;
    g.m_tiles = (int)ceil_div(M, TC_BM); g.n_tiles = (int)ceil_div(N, bn);
    // as many slices of the reduction as fit in one wave of CTAs, each at least two stages long
    const int total_kb = (int)ceil_div(K, T3_BK);
    int splits = sm_count() / (g.m_tiles * g.n_tiles);
    if (splits > total_kb / 2) splits = total_kb / 2;
    if (splits < 1) splits = 1;
    g.kb_per_split = (int)ceil_div(total_kb, splits);
    g.k_splits = (int)ceil_div(total_kb, g.kb_per_split);
    g.err = &c.state()->tc_error;
    CUtensorMap ma, mb, mo;
    if (!c.tma->get(&ma, TmaSpec{A.p, K, M, lda, A.stride, 3, T3_BK, 64, 0, 128}) ||
        !c.tma->get(&mb, TmaSpec{Bm.p, K, N, ldb, Bm.stride, 3, T3_BK, 64, 0, 128}) ||
        !c.tma->get(&mo, TmaSpec{out, M, N, ldo, 0, 1, 32, 32, 1, 128}))
        return cudaErrorInvalidValue;
    KernelScope ks(&c.prof, name, st);
    return bn == 128 ? t3_launch<128, true, T3_RED>(ma, mb, mo, g, st) : t3_launch<64, true, T3_RED>(ma, mb, mo, g, st);
}

}  // namespace gear
