// bf16 matrix products of the head on the 5th-generation tensor cores (sm_100a):
// tcgen05.mma with fp32 accumulators in tensor memory, operands staged in shared memory by TMA.
//
// One persistent kernel, one CTA per SM (two where tiles are 64 columns wide), three roles:
//   warp 0     TMA producer: streams 128 x 64 (A) and BN x 64 (B) bf16 tiles through a ring of
//              shared-memory stages (128-byte swizzle), one mbarrier pair per stage;
//   warp 1     MMA issuer: one elected lane issues tcgen05.mma (M 128, N BN, K 16) into one of two
//              accumulator buffers in tensor memory and commits each stage back to the producer;
//   warps 2-9  epilogue: tcgen05.ld the finished accumulator (32 lanes x 32 columns per instruction),
//              apply bias+ReLU / ReLU mask / nothing, and store; meanwhile the MMA warp already fills
//              the other accumulator buffer with the next tile.  Two warps share each quarter of the
//              tensor-memory lanes and split the tile's columns; the read of the next 32 columns and
//              the loads of the bias are in flight while the current 32 columns are processed; the ReLU
//              mask of a 32 x 32 block arrives by TMA, requested two blocks ahead of its use.
//              The ReLU-mask epilogue also sums its output columns (the bias gradient of the layer
//              below): each lane adds up two columns of the block staged for the store; per-CTA partials
//              in shared memory.
// Two operand layouts:
//   K-major   C[M][N] = A[M][K] . W[N][K]^T     (activations x weights; K contiguous in both)
//   MN-major  C[M][N] += A[K][M]^T . B[K][N]    (weight gradients: the reduction runs over the batch,
//                                                split across CTAs; a CTA's partial tile leaves like any
//                                                fp32 output, in 32 x 32 blocks through shared memory, but
//                                                as a TMA reduction: the copy engine adds it to the matrix)
// No cluster launch and no multicast.  Every wait is bounded: on a timeout the kernel records an error
// code, leaves its loops, frees its tensor memory and returns.
#include <new>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace gear {

constexpr int TC_BK = 64;                 // 64 bf16 = 128 bytes = one swizzle row
// Epilogue warps per CTA (a multiple of four: each warp reaches one quarter of the tensor-memory lanes).
constexpr int tc_threads(int ew) { return 64 + 32 * ew; }
constexpr int TC_MAX_N = 1024;            // widest output the column-sum partials cover
constexpr int TC_MASK_BLOCK = 32 * 64;    // a warp's ReLU-mask block for 32 columns: 32 rows of 64 bytes (two per warp)

enum { TC_EPI_BIAS_RELU = 0, TC_EPI_MASK = 1, TC_EPI_F32 = 2, TC_EPI_RED = 3, TC_EPI_TOP = 4 };

constexpr int TC_OUT_BLOCK = 32 * 128;   // a warp's output block on its way to a TMA store: 32 rows of 128 bytes

struct TopSmem {                          // the top hidden layer's epilogue
    float w[TC_TOP_N], bias[TC_TOP_N], gw[TC_TOP_N], gb[TC_TOP_N];     // output weights, the layer's bias; column sums
    float z[2][2][TC_BM];                 // [tile parity][column half] a row's part of the dot product
    float g[8][32];                       // per epilogue warp: dz of its rows
    float part[2][8];                     // per epilogue warp: loss, sum of dz
};

template <int BN, int EW, int EPI> struct TcCfg {
    static constexpr int A_BYTES = TC_BM * TC_BK * 2;            // 16 KB
    static constexpr int B_BYTES = BN * TC_BK * 2;               // 32 KB or 16 KB
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    // one output block per epilogue warp; the top layer's epilogue holds a warp's whole part of the tile
    // (64-column tiles in bf16: blocks of 64 bytes a row, one mask block)
    static constexpr bool NARROW = BN == 64;
    static constexpr int OUT_BYTES = EW * TC_OUT_BLOCK * (EPI == TC_EPI_TOP ? BN / (EW / 4) / 64 : 1) / (NARROW && (EPI == TC_EPI_BIAS_RELU || EPI == TC_EPI_MASK) ? 2 : 1);
    static constexpr int MASK_BYTES = EPI == TC_EPI_MASK ? EW * (NARROW ? 1 : 2) * TC_MASK_BLOCK : 0;
    // per-CTA column sums of the masked product; the top layer's vectors and sums
    static constexpr int COLSUM_BYTES = EPI == TC_EPI_MASK ? TC_MAX_N * 4 : EPI == TC_EPI_TOP ? (int)sizeof(TopSmem) : 0;
    static constexpr int FIXED = 1024 /*alignment slack*/ + 512 /*barriers*/ + COLSUM_BYTES + OUT_BYTES + MASK_BYTES;
    static constexpr int ROOM = (227 * 1024 - FIXED) / STAGE_BYTES;
    // Tiles of 64 columns take half an SM's shared memory: the next product's CTA is set up beside this one's (4096 views: the step
    // 54.3 -> 52.1 us, 3001 views: 51.2 -> 48.4).
    static constexpr int MOST = BN == 256 ? 4 : NARROW ? 3 : 6;
    static constexpr int STAGES = ROOM > MOST ? MOST : ROOM;
    static constexpr int SMEM = STAGES * STAGE_BYTES + FIXED;
    static constexpr int TMEM_COLS = BN == 192 ? 512 : 2 * BN;   // two accumulator buffers (a power of two is allocated)
    static_assert(STAGES >= 3, "operand ring too short");
    static_assert(NARROW || SMEM > 116 * 1024, "one CTA per SM: two CTAs would both ask for tensor memory");
    static_assert(!NARROW || SMEM <= 112 * 1024, "two CTAs per SM");
    static_assert(SMEM <= 227 * 1024, "shared memory budget");
};

struct TcArgs {
    int M, N, K;              // output rows, output columns, reduction length
    int m_tiles, n_tiles, k_splits, kb_per_split;   // kb = blocks of TC_BK along K
    void* out; int64_t ldo;
    const float* bias;
    const __nv_bfloat16* mask; int64_t ldm;
    float* colsum;            // ReLU-mask epilogue: colsum[n] += sum over rows of the stored output (may be null)
    int32_t* err;             // device word that receives a non-zero code on a timeout
    TopArgs top;              // top layer only
    LossSum loss;             // the loss to finish
    int let_next;             // the next kernel in the stream may be set up beside this one
};

// Epilogue of one finished accumulator buffer `a`, as run by one of the epilogue warps: warp w reads
// tensor-memory lanes 32 * (w % 4) .. + 31 (its rows of the tile); the EW / 4 warps of a lane quarter split the
// tile's columns evenly (warps 2..5 take the first share, 6..9 the second, ...).
//
// Output leaves through the copy engine: a lane owns a row of the accumulator, so it writes its row's 128 bytes
// (64 bf16 or 32 fp32 columns) into a 32-row block in shared memory, 16-byte pieces XOR-swizzled by the row number
// (conflict-free 128-bit writes, and the layout a 128-byte-swizzle tensor map expects); one lane then hands the
// block to a TMA store, which writes whole rows of it, drops what lies past the matrix edge and needs no register
// or issue slot of the warp while it runs.  `out_buf` is the shared-memory address of this warp's block(s).
// The ReLU mask of a warp's 32 x 32 blocks travels by TMA, two blocks ahead of their use: block c goes to the warp's
// half-buffer c % 2 (32 rows of 64 bytes, 64-byte swizzle) and reports to that half's mbarrier; as soon as the lanes
// have read a half, the block two further on (of this tile or the next) is requested into it.
struct MaskPipe {
    const CUtensorMap* map;
    uint32_t buf, bar;         // shared-memory addresses of the warp's two half-buffers / two mbarriers
    uint32_t parity;           // bit h: phase the next wait on half h looks for
    uint32_t pending;          // bit h: a copy into half h has been issued and not yet waited for
    int next_m0, next_col0;    // first row / column of this warp's part of the CTA's next tile (-1: there is none)
};
__device__ __forceinline__ void mask_request(MaskPipe& mp, int h, int x, int y, int lane) {
    __syncwarp();                                             // every lane has read the half's previous contents
    if (lane == 0) {
        fence_async_smem();
        const uint32_t bar = mp.bar + 8u * h;
        mbar_expect_tx(bar, TC_MASK_BLOCK);
        tma_load_2d(mp.buf + (uint32_t)h * TC_MASK_BLOCK, mp.map, bar, x, y);
    }
    mp.pending |= 1u << h;
}

template <int BN, int EPI, int EW>
__device__ __forceinline__ void epilogue_tile(const TcArgs& g, const CUtensorMap* map_out, uint32_t tmem_base, int a, int mt,
                                              int nt, int warp, int lane, float* s_colsum, MaskPipe& mp, uint32_t out_buf,
                                              uint64_t keep_policy) {
    const int quarter = warp & 3;
    const int part = (warp - 2) >> 2;
    constexpr int COLS = BN / (EW / 4);                   // columns per warp and tile
    constexpr int CHUNKS = COLS / 32;                     // 32-column chunks per warp and tile
    // bf16 output leaves in blocks of 64 columns (chunks 2k and 2k+1), or, where a warp has one chunk only, of 32 (then a CTA
    // has one tile: the next tile's mask is not asked for)
    constexpr bool NARROW = CHUNKS == 1;
    static_assert(EPI == TC_EPI_F32 || EPI == TC_EPI_RED || NARROW || CHUNKS % 2 == 0, "whole blocks of 64 columns");
    const int m0 = mt * TC_BM + quarter * 32;         // first row of this warp's block
    const int rows = min(32, max(0, g.M - m0));
    const int col0 = nt * BN + part * COLS;
    const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * BN + part * COLS);
    const uint32_t swz = (uint32_t)(lane & 7);
    uint32_t r[2][32];
    tc_ld32(t_row, r[0]);
#pragma unroll
    for (int c = 0; c < CHUNKS; ++c) {
        const int n0 = col0 + c * 32;
        const bool chunk_ok = n0 < g.N;               // warp-uniform; N is a multiple of 8
        // what this chunk's epilogue reads from memory, requested while the tensor-memory read is in flight
        float4 bias4[EPI == TC_EPI_BIAS_RELU ? 8 : 1];
        uint4 mask4[EPI == TC_EPI_MASK ? 4 : 1];
        if (EPI == TC_EPI_BIAS_RELU) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                bias4[j] = (n0 + 4 * j < g.N) ? ldg_f4(g.bias + n0 + 4 * j) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        tc_wait_ld(r[c & 1]);
        if (c + 1 < CHUNKS) tc_ld32(t_row + (uint32_t)((c + 1) * 32), r[(c + 1) & 1]);
        if (EPI == TC_EPI_MASK) {
            // this block's mask has been on its way since two blocks ago; a lane reads its own row (rows and columns past
            // the matrix edge arrive as zeros), then the half is free for the block two further on
            const int h = c & 1;
            mbar_wait(mp.bar + 8u * h, (mp.parity >> h) & 1u, g.err, 6);
            mp.parity ^= 1u << h;
            mp.pending &= ~(1u << h);
            const uint32_t row_addr = mp.buf + (uint32_t)h * TC_MASK_BLOCK + (uint32_t)lane * 64u;
            const uint32_t sw = ((uint32_t)lane >> 1) & 3u;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];"
                             : "=r"(mask4[j].x), "=r"(mask4[j].y), "=r"(mask4[j].z), "=r"(mask4[j].w)
                             : "r"(row_addr + ((((uint32_t)j) ^ sw) << 4)) : "memory");
            if (c + 2 < CHUNKS) mask_request(mp, h, n0 + 64, m0, lane);
            else if (!NARROW && mp.next_m0 >= 0) mask_request(mp, h, mp.next_col0 + (c + 2 - CHUNKS) * 32, mp.next_m0, lane);
        }
        if (!chunk_ok || rows == 0) continue;
        uint32_t (&acc)[32] = r[c & 1];
        if (EPI == TC_EPI_BIAS_RELU || EPI == TC_EPI_MASK) {
            uint32_t pk[16];
            if (EPI == TC_EPI_BIAS_RELU) {
                float v[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(acc[i]);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[4 * j + 0] = fmaxf(v[4 * j + 0] + bias4[j].x, 0.f);
                    v[4 * j + 1] = fmaxf(v[4 * j + 1] + bias4[j].y, 0.f);
                    v[4 * j + 2] = fmaxf(v[4 * j + 2] + bias4[j].z, 0.f);
                    v[4 * j + 3] = fmaxf(v[4 * j + 3] + bias4[j].w, 0.f);
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
                    pk[q] = *reinterpret_cast<uint32_t*>(&h2);
                }
            } else {
                // two columns at a time: round the pair, then clear the halves whose activation was not positive (a
                // packed compare of the two activations against zero gives all-ones per passing half)
                const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t w[4] = {mask4[j].x, mask4[j].y, mask4[j].z, mask4[j].w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(acc[8 * j + 2 * q]), __uint_as_float(acc[8 * j + 2 * q + 1]));
                        const unsigned int keep = __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&w[q]), zero2);
                        pk[4 * j + q] = *reinterpret_cast<uint32_t*>(&h2) & keep;
                    }
                }
            }
            {
                // chunks 2k and 2k+1 fill the left and right half of one 64-column block
                const int half = NARROW ? 0 : c & 1;
                const uint32_t row_addr = out_buf + (uint32_t)lane * (NARROW ? 64u : 128u);
                const uint32_t sw_out = NARROW ? ((uint32_t)lane >> 1) & 3u : swz;      // 64- or 128-byte swizzle
                if (half == 0) {
                    if (lane == 0) tma_store_wait_read<0>();          // the block's previous contents have been read
                    __syncwarp();
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    sts_u4(row_addr + ((((uint32_t)(4 * half + j)) ^ sw_out) << 4),
                           make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]));
                if (NARROW || half == 1 || n0 + 32 >= g.N) {
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) tma_store_2d(map_out, out_buf, n0 - 32 * half, m0);
                    if (EPI == TC_EPI_MASK && g.colsum != nullptr) {
                        // column sums of what was stored (the rounded values), read back from the block: lane l owns
                        // columns 2l and 2l + 1 of the 64, one word per row (rows past M hold zeros: their operand rows
                        // and mask were read as zeros)
                        // (a block of 32 columns has 16 words a row: lanes 16 .. 31 take its lower 16 rows)
                        const uint32_t word = NARROW ? (uint32_t)lane & 15u : (uint32_t)lane;
                        const int nb = n0 - 32 * half + 2 * (int)word;
                        float s_lo = 0.f, s_hi = 0.f;
#pragma unroll
                        for (int i = 0; i < (NARROW ? 16 : 32); ++i) {
                            const int rr = NARROW ? i + (lane & 16) : i;
                            uint32_t wv;
                            const uint32_t addr = out_buf + (uint32_t)rr * (NARROW ? 64u : 128u) +
                                                  (((word >> 2) ^ (NARROW ? ((uint32_t)rr >> 1) & 3u : (uint32_t)(rr & 7))) << 4) + ((word & 3u) << 2);
                            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(wv) : "r"(addr) : "memory");
                            s_lo += __uint_as_float(wv << 16);
                            s_hi += __uint_as_float(wv & 0xffff0000u);
                        }
                        if (nb < g.N) { atomicAdd(&s_colsum[nb], s_lo); atomicAdd(&s_colsum[nb + 1], s_hi); }
                    }
                }
            }
        } else {
            // fp32 output (dX): one block per 32 columns; it is read again right
            // after (embedding and DFV gradients): ask the L2 to keep it
            const uint32_t buf = out_buf;
            if (lane == 0) tma_store_wait_read<0>();                  // the block's previous contents have been read
            __syncwarp();
            const uint32_t row_addr = buf + (uint32_t)lane * 128u;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                sts_u4(row_addr + (((uint32_t)j ^ swz) << 4), make_uint4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]));
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                // a slice's partial tile of a weight gradient is added to the matrix by the copy engine
                if (EPI == TC_EPI_RED) tma_reduce_add_2d(map_out, buf, n0, m0);
                else tma_store_2d_hint(map_out, buf, n0, m0, keep_policy);
            }
        }
    }
}

// The top hidden layer's tile (its columns are one tile of the product) with all that hangs off it:
//   h = ReLU(acc + bias) rounded to bf16;  z = h . w_out + b_out;  p = sigmoid(z);  BCE in its overflow-safe form;
//   dz = (p - y) / M;  out[b][j] = dz * w_out[j] where h[b][j] > 0, else 0;  gw_out[j] += sum_b h dz;  gb_top[j] += sum_b out
// A lane first walks its row of the accumulator (dot product; h to the warp's blocks in shared memory, after which the buffer
// goes back to the MMA warp); the two warps of a lane quarter add their halves of z; then a lane owns two columns of a block and
// walks its 32 rows: column sums, h replaced by out in place.  h itself goes nowhere: nothing after this reads it.
// (Bound by instructions, about 15 per 2 elements in the second walk.  In a launch of its own, which read h and wrote out again,
// the output unit took 11 us for 4096 x 128 and 23 us for 65536 x 256.)
template <int BN> struct TopSums { float gw[BN / 128][2], gb[BN / 128][2], loss, dz; };

template <int BN>
__device__ __forceinline__ void epilogue_top(const TcArgs& g, const CUtensorMap* map_out, uint32_t tmem_base, int a, int mt, int parity,
                                             int warp, int lane, TopSmem& s, TopSums<BN>& sums, uint32_t out_buf, uint32_t empty_bar) {
    constexpr int COLS = BN / 2, BLOCKS = COLS / 64;
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const int m0 = mt * TC_BM + quarter * 32, b = m0 + lane;
    const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * BN + part * COLS);
    const uint32_t swz = (uint32_t)(lane & 7);
    const float y = b < g.M ? __ldg(g.top.label + b) : 0.f;
    float z = 0.f;
    uint32_t r[2][32];
    tc_ld32(t_row, r[0]);
    if (lane == 0) tma_store_wait_read<0>();                          // the blocks' previous contents have been read
    __syncwarp();
#pragma unroll
    for (int c = 0; c < COLS / 32; ++c) {
        const int n0 = part * COLS + c * 32;
        tc_wait_ld(r[c & 1]);
        if (c + 1 < COLS / 32) tc_ld32(t_row + (uint32_t)((c + 1) * 32), r[(c + 1) & 1]);
        if (n0 >= g.N) continue;                                      // warp-uniform; N is a multiple of 64
        const uint32_t row_addr = out_buf + (uint32_t)(c >> 1) * TC_OUT_BLOCK + (uint32_t)lane * 128u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t pk[4];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float4 bi = *reinterpret_cast<const float4*>(&s.bias[n0 + 8 * j + 4 * k]);
                const float4 w = *reinterpret_cast<const float4*>(&s.w[n0 + 8 * j + 4 * k]);
                const uint32_t* acc = &r[c & 1][8 * j + 4 * k];
                __nv_bfloat162 h01 = __floats2bfloat162_rn(fmaxf(__uint_as_float(acc[0]) + bi.x, 0.f), fmaxf(__uint_as_float(acc[1]) + bi.y, 0.f));
                __nv_bfloat162 h23 = __floats2bfloat162_rn(fmaxf(__uint_as_float(acc[2]) + bi.z, 0.f), fmaxf(__uint_as_float(acc[3]) + bi.w, 0.f));
                pk[2 * k] = *reinterpret_cast<uint32_t*>(&h01);
                pk[2 * k + 1] = *reinterpret_cast<uint32_t*>(&h23);
                z = fmaf(__uint_as_float(pk[2 * k] << 16), w.x, z);
                z = fmaf(__uint_as_float(pk[2 * k] & 0xffff0000u), w.y, z);
                z = fmaf(__uint_as_float(pk[2 * k + 1] << 16), w.z, z);
                z = fmaf(__uint_as_float(pk[2 * k + 1] & 0xffff0000u), w.w, z);
            }
            sts_u4(row_addr + ((((uint32_t)(4 * (c & 1) + j)) ^ swz) << 4), make_uint4(pk[0], pk[1], pk[2], pk[3]));
        }
    }
    tc_fence_before();
    mbar_arrive_relaxed(empty_bar);                                   // all epilogue threads arrive: the buffer returns to the MMA warp
    s.z[parity][part][quarter * 32 + lane] = z;
    // the two warps of the quarter meet; two tiles on, z[parity] is written again only behind the next tile's meeting
    asm volatile("bar.sync %0, 64;" :: "r"(1 + quarter) : "memory");
    const float zz = s.z[parity][0][quarter * 32 + lane] + s.z[parity][1][quarter * 32 + lane] + __ldg(g.top.b_out);
    const float p = 1.0f / (1.0f + expf(-zz));
    const float dz = b < g.M ? (p - y) / (float)g.M : 0.f;            // rows past the edge add nothing
    if (part == 0 && b < g.M) {
        sums.loss += fmaxf(zz, 0.f) - zz * y + log1pf(expf(-fabsf(zz)));
        sums.dz += dz;
        if (g.top.prob) g.top.prob[b] = p;
    }
    s.g[warp - 2][lane] = dz;
    __syncwarp();
    const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < BLOCKS; ++k) {
        const int nb = part * COLS + 64 * k;
        if (nb >= g.N) break;
        const uint32_t blk = out_buf + (uint32_t)k * TC_OUT_BLOCK + (((uint32_t)lane & 3u) << 2);
        const float2 w = *reinterpret_cast<const float2*>(&s.w[nb + 2 * lane]);
#pragma unroll
        for (int r4 = 0; r4 < 8; ++r4) {
            const float4 g4 = *reinterpret_cast<const float4*>(&s.g[warp - 2][4 * r4]);
            const float gr[4] = {g4.x, g4.y, g4.z, g4.w};
            uint32_t h[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(h[i]) : "r"(blk + (uint32_t)(4 * r4 + i) * 128u + ((((uint32_t)lane >> 2) ^ (uint32_t)((4 * r4 + i) & 7)) << 4)) : "memory");
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                sums.gw[k][0] = fmaf(__uint_as_float(h[i] << 16), gr[i], sums.gw[k][0]);
                sums.gw[k][1] = fmaf(__uint_as_float(h[i] & 0xffff0000u), gr[i], sums.gw[k][1]);
                __nv_bfloat162 d2 = __floats2bfloat162_rn(gr[i] * w.x, gr[i] * w.y);
                const uint32_t dv = *reinterpret_cast<uint32_t*>(&d2) & __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&h[i]), zero2);
                asm volatile("st.shared.b32 [%0], %1;" :: "r"(blk + (uint32_t)(4 * r4 + i) * 128u + ((((uint32_t)lane >> 2) ^ (uint32_t)((4 * r4 + i) & 7)) << 4)), "r"(dv) : "memory");
                sums.gb[k][0] += __uint_as_float(dv << 16);
                sums.gb[k][1] += __uint_as_float(dv & 0xffff0000u);
            }
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) tma_store_2d(map_out, out_buf + (uint32_t)k * TC_OUT_BLOCK, nb, m0);
    }
}

// After the last tile (all threads of the CTA): sums to memory.
__device__ __forceinline__ void finish_top(const TcArgs& g, TopSmem& s) {
    for (int n = threadIdx.x; n < g.N; n += blockDim.x) { atomicAdd(g.top.gw_out + n, s.gw[n]); atomicAdd(g.top.gb_top + n, s.gb[n]); }
    if (threadIdx.x == 0) {
        float l = 0.f, t = 0.f;
        for (int k = 0; k < 8; ++k) { l += s.part[0][k]; t += s.part[1][k]; }
        g.top.loss_part[blockIdx.x] = l;
        atomicAdd(g.top.gb_out, t);
    }
}

// ---------------------------------------------------------------- the kernel
template <int BN, bool MN_MAJOR, int EPI, int EW>
__device__ __forceinline__ void tc_gemm_body(const CUtensorMap& map_a, const CUtensorMap& map_b, const CUtensorMap& map_out,
                                             const CUtensorMap& map_mask, const TcArgs& g) {
    using Cfg = TcCfg<BN, EW, EPI>;
    constexpr int STAGES = Cfg::STAGES;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;                  // operand stages, 1024-byte aligned
    const uint32_t out_blocks = tiles + STAGES * Cfg::STAGE_BYTES;  // output blocks of the epilogue warps, 1024-byte aligned
    const uint32_t mask_blocks = out_blocks + Cfg::OUT_BYTES;       // ReLU-mask blocks of the epilogue warps, 1024-byte aligned
    const uint32_t bars = mask_blocks + Cfg::MASK_BYTES;            // mbarriers, then the tmem address word
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
    auto acc_full = [&](int a) { return bars + 8u * (2 * STAGES + a); };
    auto acc_empty = [&](int a) { return bars + 8u * (2 * STAGES + 2 + a); };
    const uint32_t tmem_word = bars + 8u * (2 * STAGES + 4);
    volatile uint32_t* tmem_word_ptr =
        reinterpret_cast<volatile uint32_t*>(smem_raw + (tmem_word - raw));
    auto mask_bar = [&](int w, int h) { return bars + 8u * (24 + 2 * w + h); };     // two per epilogue warp
    float* s_colsum = reinterpret_cast<float*>(smem_raw + (bars + 512u - raw));     // [TC_MAX_N] per-CTA column sums
    TopSmem& top = *reinterpret_cast<TopSmem*>(s_colsum);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int total_tiles = g.m_tiles * g.n_tiles * g.k_splits;
    const int total_kb = (g.K + TC_BK - 1) / TC_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(acc_full(a), 1); mbar_init(acc_empty(a), 32 * EW); }
        if (EPI == TC_EPI_MASK)
            for (int w = 0; w < EW; ++w) { mbar_init(mask_bar(w, 0), 1); mbar_init(mask_bar(w, 1), 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&map_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&map_b) : "memory");
        asm volatile("prefetch.tensormap [%0];" :: "l"(&map_out) : "memory");
        if (EPI == TC_EPI_MASK) asm volatile("prefetch.tensormap [%0];" :: "l"(&map_mask) : "memory");
    }
    if (EPI == TC_EPI_MASK && g.colsum != nullptr)
        for (int n = threadIdx.x; n < TC_MAX_N; n += tc_threads(EW)) s_colsum[n] = 0.f;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(tmem_word), "r"((uint32_t)Cfg::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_word_ptr;
    wait_for_predecessor();      // barriers, tensor memory and descriptors are set up while the previous kernel drains
    if (g.let_next) let_successor_start();

    if (warp == 0) {
        // ---------------- TMA producer
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x) {
                // column tiles of one row tile are neighbours in the order: CTAs that run side by side read the same rows of A,
                // which then come from memory once
                const int nt = t % g.n_tiles, mt = (t / g.n_tiles) % g.m_tiles, ks = t / (g.m_tiles * g.n_tiles);
                const int kb0 = ks * g.kb_per_split, kb1 = min(total_kb, kb0 + g.kb_per_split);
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const int s = it % STAGES;
                    if (!(ok = mbar_wait(empty_bar(s), ((it / STAGES) & 1u) ^ 1u, g.err, 1))) break;
                    const uint32_t a_dst = tiles + s * Cfg::STAGE_BYTES, b_dst = a_dst + Cfg::A_BYTES;
                    mbar_expect_tx(full_bar(s), Cfg::STAGE_BYTES);
                    if (!MN_MAJOR) {
                        tma_load_2d(a_dst, &map_a, full_bar(s), kb * TC_BK, mt * TC_BM);     // 128 rows x 64 k
                        tma_load_2d(b_dst, &map_b, full_bar(s), kb * TC_BK, nt * BN);        // BN rows x 64 k
                    } else {
                        // 64 k-rows x 64 columns per box; the slabs of one operand sit 8 KB apart
#pragma unroll
                        for (int j = 0; j < TC_BM / 64; ++j)
                            tma_load_2d(a_dst + j * 8192, &map_a, full_bar(s), mt * TC_BM + j * 64, kb * TC_BK);
#pragma unroll
                        for (int j = 0; j < BN / 64; ++j)
                            tma_load_2d(b_dst + j * 8192, &map_b, full_bar(s), nt * BN + j * 64, kb * TC_BK);
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
            uint32_t it = 0, tile_it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x, ++tile_it) {
                const int ks = t / (g.m_tiles * g.n_tiles);
                const int kb0 = ks * g.kb_per_split, kb1 = min(total_kb, kb0 + g.kb_per_split);
                const int a = tile_it & 1;
                if (!(ok = mbar_wait(acc_empty(a), ((tile_it >> 1) & 1u) ^ 1u, g.err, 2))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(a * BN);
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const int s = it % STAGES;
                    if (!(ok = mbar_wait(full_bar(s), (it / STAGES) & 1u, g.err, 3))) break;
                    tc_fence_after();
                    const uint32_t a_src = tiles + s * Cfg::STAGE_BYTES, b_src = a_src + Cfg::A_BYTES;
#pragma unroll
                    for (int k = 0; k < TC_BK / 16; ++k) {
                        uint64_t da, db;
                        if (!MN_MAJOR) {
                            da = smem_desc(a_src + k * 32, 16, 1024);
                            db = smem_desc(b_src + k * 32, 16, 1024);
                        } else {
                            da = smem_desc(a_src + k * 2048, 8192, 1024);
                            db = smem_desc(b_src + k * 2048, 8192, 1024);
                        }
                        tc_mma(d_tmem, da, db, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
                    }
                    tc_commit(empty_bar(s));            // the stage may be refilled once these MMAs have read it
                }
                if (ok) tc_commit(acc_full(a));          // accumulator complete
            }
        }
    } else {
        // ---------------- epilogue warps
        const uint32_t out_buf = out_blocks + (uint32_t)((warp - 2) * (Cfg::OUT_BYTES / EW));
        const uint64_t keep_policy = l2_policy_evict_last();
        uint32_t tile_it = 0;
        bool ok = true;
        constexpr int COLS = BN / (EW / 4);
        // where this warp's part of tile t starts
        auto part_m0 = [&](int t) { return ((t / g.n_tiles) % g.m_tiles) * TC_BM + (warp & 3) * 32; };
        auto part_col0 = [&](int t) { return (t % g.n_tiles) * BN + ((warp - 2) >> 2) * COLS; };
        MaskPipe mp{&map_mask, mask_blocks + (uint32_t)((warp - 2) * (Cfg::MASK_BYTES / EW)), mask_bar(warp - 2, 0), 0u, 0u, -1, -1};
        if (EPI == TC_EPI_MASK && (int)blockIdx.x < total_tiles) {
            // the masks of the first tile's first two blocks (after the wait for the previous kernel, which wrote them)
            mask_request(mp, 0, part_col0(blockIdx.x), part_m0(blockIdx.x), lane);
            if (COLS > 32) mask_request(mp, 1, part_col0(blockIdx.x) + 32, part_m0(blockIdx.x), lane);
        }
        if constexpr (EPI == TC_EPI_TOP) {
            TopSums<BN> sums = {};
            for (int n = threadIdx.x - 64; n < TC_TOP_N; n += 32 * EW) {
                top.w[n] = n < g.N ? __ldg(g.top.w_out + n) : 0.f;
                top.bias[n] = n < g.N ? __ldg(g.bias + n) : 0.f;
                top.gw[n] = 0.f; top.gb[n] = 0.f;
            }
            asm volatile("bar.sync 5, %0;" :: "n"(32 * EW) : "memory");
            // A wait that gave up does not leave the loop (the two warps of a quarter meet in every tile; from then on all waits
            // return at once): the error word tells the host that the results are void.
            for (int t = blockIdx.x; t < total_tiles; t += gridDim.x, ++tile_it) {
                const int a = tile_it & 1;
                mbar_wait(acc_full(a), (tile_it >> 1) & 1u, g.err, 4);
                __syncwarp();
                tc_fence_after();
                epilogue_top<BN>(g, &map_out, tmem_base, a, t, (int)(tile_it & 1u), warp, lane, top, sums, out_buf, acc_empty(a));
            }
#pragma unroll
            for (int k = 0; k < BN / 128; ++k) {
                const int n = ((warp - 2) >> 2) * COLS + 64 * k + 2 * lane;
                atomicAdd(&top.gw[n], sums.gw[k][0]); atomicAdd(&top.gw[n + 1], sums.gw[k][1]);
                atomicAdd(&top.gb[n], sums.gb[k][0]); atomicAdd(&top.gb[n + 1], sums.gb[k][1]);
            }
            const float l = warp_sum(sums.loss), d = warp_sum(sums.dz);
            if (lane == 0) { top.part[0][warp - 2] = l; top.part[1][warp - 2] = d; }
        } else
        for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x, ++tile_it) {
            const int nt = t % g.n_tiles, mt = (t / g.n_tiles) % g.m_tiles;
            const int a = tile_it & 1;
            if (EPI == TC_EPI_MASK) {
                const int tn = t + (int)gridDim.x;
                mp.next_m0 = tn < total_tiles ? part_m0(tn) : -1;
                mp.next_col0 = tn < total_tiles ? part_col0(tn) : -1;
            }
            if (!(ok = mbar_wait(acc_full(a), (tile_it >> 1) & 1u, g.err, 4))) break;
            tc_fence_after();
            epilogue_tile<BN, EPI, EW>(g, &map_out, tmem_base, a, mt, nt, warp, lane, s_colsum, mp, out_buf, keep_policy);
            tc_fence_before();
            mbar_arrive_relaxed(acc_empty(a));                   // all epilogue threads arrive: the buffer returns to the MMA warp
        }
        if (lane == 0) tma_store_wait_all();   // this warp's stores have left shared memory and landed
        if (EPI == TC_EPI_MASK && mp.pending) {
            // leaving early: let the mask copies already issued land before the CTA gives its shared memory back
            for (int h = 0; h < 2; ++h)
                if (mp.pending & (1u << h))
                    for (uint32_t spin = 0; spin < (1u << 16) && !mbar_try(mp.bar + 8u * h, (mp.parity >> h) & 1u); ++spin)
                        __nanosleep(64);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (EPI == TC_EPI_MASK && g.colsum != nullptr)
        for (int n = threadIdx.x; n < g.N && n < TC_MAX_N; n += tc_threads(EW)) {
            const float v = s_colsum[n];
            if (v != 0.f) atomicAdd(g.colsum + n, v);
        }
    if constexpr (EPI == TC_EPI_TOP) finish_top(g, top);
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     :: "r"(tmem_base), "r"((uint32_t)Cfg::TMEM_COLS) : "memory");
    }
}

// Eight epilogue warps, at most 128 registers per thread: a CTA (320 threads) then fits on an SM beside a block of
// the ID sort.  One CTA per SM follows from the shared-memory footprint; of 64-column tiles two fit, in registers too.
template <int BN, bool MN_MAJOR, int EPI>
__global__ void __maxnreg__(BN == 64 ? 88 : 128)
tc_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_mask, const TcArgs g) {
    tc_gemm_body<BN, MN_MAJOR, EPI, 8>(map_a, map_b, map_out, map_mask, g);
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

bool TmaCache::get(CUtensorMap* out, const TmaSpec& k) {
    for (int i = 0; i < used_; ++i)
        if (key_[i] == k) { *out = map_[i]; return true; }
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t esz = k.f32 ? 4 : 2;
    cuuint64_t dims[3] = {(cuuint64_t)k.cols, (cuuint64_t)k.rows, (cuuint64_t)k.planes};
    cuuint64_t strides[2] = {(cuuint64_t)k.ld * esz, (cuuint64_t)k.plane_stride * esz};
    cuuint32_t box[3] = {(cuuint32_t)k.box_cols, (cuuint32_t)k.box_rows, (cuuint32_t)k.planes};
    cuuint32_t estr[3] = {1, 1, 1};
    if (fn(out, k.f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, k.planes > 1 ? 3 : 2,
           const_cast<void*>(k.ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
           k.swizzle == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    const int i = used_ < N ? used_++ : (next_ = (next_ + 1) % N);
    key_[i] = k; map_[i] = *out;
    return true;
}

TmaCache* new_tma_cache() { return new (std::nothrow) TmaCache; }
void delete_tma_cache(TmaCache* t) { delete t; }

// bf16 matrix in boxes of box_rows x 64 columns; fp32 matrix in boxes of 32 x 32 (both 128 bytes a row); the ReLU mask, a
// bf16 matrix in boxes of 32 x 32 (64 bytes a row)
static bool make_map(const gear_ctx_impl& c, CUtensorMap* m, const void* ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    return c.tma->get(m, TmaSpec{ptr, rows, cols, ld, 0, 1, box_rows, 64, 0, 128});
}
static bool make_map_f32(const gear_ctx_impl& c, CUtensorMap* m, const void* ptr, int64_t rows, int64_t cols, int64_t ld) {
    return c.tma->get(m, TmaSpec{ptr, rows, cols, ld, 0, 1, 32, 32, 1, 128});
}
static bool make_map_mask(const gear_ctx_impl& c, CUtensorMap* m, const void* ptr, int64_t rows, int64_t cols, int64_t ld) {
    return c.tma->get(m, TmaSpec{ptr, rows, cols, ld, 0, 1, 32, 32, 0, 64});
}

template <int BN, bool MN, int EPI, int EW>
static cudaError_t launch_variant(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mo, const CUtensorMap& mm,
                                  TcArgs g, cudaStream_t st) {
    using Cfg = TcCfg<BN, EW, EPI>;
    static_assert(EW == 8, "one kernel entry point: eight epilogue warps");
    constexpr auto kernel = tc_gemm_kernel<BN, MN, EPI>;
    if (const cudaError_t e = allow_smem<kernel>(Cfg::SMEM)) return e;
    const int tiles = g.m_tiles * g.n_tiles * g.k_splits;
    const int grid = tiles < sm_count() ? tiles : sm_count();
    // (Larger products gain nothing, and CTAs that wait on an SM keep the kernels of other streams from it: 65 k views, all products:
    // step 369 -> 373 us.  dX: its successor is the store, which would keep the weight gradients out.)
    if (BN == 64 && EPI != TC_EPI_F32 && !MN) g.let_next = 1;
    return launch_dependent(kernel, dim3(grid), dim3(tc_threads(EW)), (size_t)Cfg::SMEM, st, ma, mb, mo, mm, g);
}

template <bool MN, int EPI, int EW = 8>
static cudaError_t launch_bn(int bn, const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mo, const CUtensorMap& mm,
                             const TcArgs& g, cudaStream_t st) {
    return bn == 256   ? launch_variant<256, MN, EPI, EW>(ma, mb, mo, mm, g, st)
           : bn == 128 ? launch_variant<128, MN, EPI, EW>(ma, mb, mo, mm, g, st)
                       : launch_variant<64, MN, EPI, EW>(ma, mb, mo, mm, g, st);
}

cudaError_t tc_gemm_kmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const __nv_bfloat16* A, int64_t lda,
                           const __nv_bfloat16* W, int64_t ldw, int epi, void* out, int64_t ldo, const float* bias,
                           const __nv_bfloat16* mask, int64_t ldm, float* colsum, const LossSum& loss, cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    // column tiles of 256 or 128; the fp32 output (dX) also has 192, which fits a width like 384 without a half-empty tile
    int bn = N > 128 ? 256 : 128;
    if (epi == TC_EPI_F32 && N > 128 && ceil_div(N, 192) * 192 < ceil_div(N, 256) * 256) bn = 192;
    // Where narrower tiles still are no more than the SMs, a tile's epilogue is what a product waits for: a warp then has one
    // block of 32 columns instead of four (4096 x 256 x 192: 10.7 -> 9.1 us a launch).
    const int64_t m_tiles = ceil_div(M, TC_BM);
    if (m_tiles * ceil_div(N, 64) <= sm_count()) bn = 64;
    else if (m_tiles * ceil_div(N, 128) <= sm_count()) bn = 128;
    CUtensorMap ma, mb, mo;
    if (!make_map(c, &ma, A, M, K, lda, TC_BM) || !make_map(c, &mb, W, N, K, ldw, bn)) return cudaErrorInvalidValue;
    // the output leaves in boxes of 32 rows x 128 bytes (bf16 output of 64-column tiles: 64 bytes)
    if (!(epi == TC_EPI_F32 ? make_map_f32(c, &mo, out, M, N, ldo)
          : bn == 64        ? make_map_mask(c, &mo, out, M, N, ldo)
                            : make_map(c, &mo, out, M, N, ldo, 32)))
        return cudaErrorInvalidValue;
    TcArgs g = {};
    g.M = M; g.N = N; g.K = K; g.loss = loss;
    g.m_tiles = (int)m_tiles; g.n_tiles = (int)ceil_div(N, bn); g.k_splits = 1;
    g.kb_per_split = (int)ceil_div(K, TC_BK);
    g.out = out; g.ldo = ldo; g.bias = bias; g.mask = mask; g.ldm = ldm; g.err = &c.state()->tc_error;
    g.colsum = (epi == TC_EPI_MASK && N <= TC_MAX_N) ? colsum : nullptr;
    if (epi == TC_EPI_MASK && colsum != nullptr && g.colsum == nullptr) return cudaErrorInvalidValue;
    KernelScope ks(&c.prof, name, st);
    switch (epi) {
    case TC_EPI_BIAS_RELU: return launch_bn<false, TC_EPI_BIAS_RELU>(bn, ma, mb, mo, ma /*unused*/, g, st);
    case TC_EPI_MASK: {
        CUtensorMap mm;
        if (!mask || !make_map_mask(c, &mm, mask, M, N, ldm)) return cudaErrorInvalidValue;
        return launch_bn<false, TC_EPI_MASK>(bn, ma, mb, mo, mm, g, st);
    }
    default:
        if (bn == 192) return launch_variant<192, false, TC_EPI_F32, 8>(ma, mb, mo, ma /*unused*/, g, st);
        return launch_bn<false, TC_EPI_F32>(bn, ma, mb, mo, ma /*unused*/, g, st);
    }
}

cudaError_t tc_gemm_top(const gear_ctx_impl& c, const char* name, int M, int N, int K, const __nv_bfloat16* A, int64_t lda,
                        const __nv_bfloat16* W, int64_t ldw, const float* bias, __nv_bfloat16* dA, const TopArgs& top, int* n_part, cudaStream_t st) {
    const int bn = N > 128 ? 256 : 128;
    CUtensorMap ma, mb, mo;
    if (!make_map(c, &ma, A, M, K, lda, TC_BM) || !make_map(c, &mb, W, N, K, ldw, bn) || !make_map(c, &mo, dA, M, N, N, 32))
        return cudaErrorInvalidValue;
    TcArgs g = {};
    g.M = M; g.N = N; g.K = K;
    g.m_tiles = (int)ceil_div(M, TC_BM); g.n_tiles = 1; g.k_splits = 1;
    g.kb_per_split = (int)ceil_div(K, TC_BK);
    g.bias = bias; g.err = &c.state()->tc_error; g.top = top;
    *n_part = g.m_tiles < sm_count() ? g.m_tiles : sm_count();          // one per CTA
    KernelScope ks(&c.prof, name, st);
    return bn == 256 ? launch_variant<256, false, TC_EPI_TOP, 8>(ma, mb, mo, ma /*unused*/, g, st)
                     : launch_variant<128, false, TC_EPI_TOP, 8>(ma, mb, mo, ma /*unused*/, g, st);
}

cudaError_t tc_gemm_mnmajor(const gear_ctx_impl& c, const char* name, int M, int N, int K, const __nv_bfloat16* A, int64_t lda,
                            const __nv_bfloat16* Bm, int64_t ldb, float* out, int64_t ldo,
                            cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    const int total_kb = (int)ceil_div(K, TC_BK);
    // Tile width and number of slices, by what a CTA's time is made of (in clocks): its operand loads (50 bytes a clock), its
    // epilogue, and the copy engines' additions of all slices to the matrix (1500 bytes a clock for the whole GPU).  Long
    // reductions take wide tiles, whose operands are read fewer times (65536 rows, 384 x 512: 24 slices of 256 columns, 30 us),
    // short ones few slices of narrow tiles (4096 rows, 192 x 256: 11.2 -> 10.0 us a launch against 64 slices of 256 columns).
    int bn = 256, splits = 1;
    double best = 1e30;
    for (int w = N > 128 ? 256 : 128; w >= 64; w >>= 1) {
        const int tiles = (int)(ceil_div(M, TC_BM) * ceil_div(N, w));
        // as many slices of the reduction as fit in one wave of CTAs (one more would leave a second, nearly empty wave)
        for (int s = sm_count() / tiles > 1 ? sm_count() / tiles : 1; s >= 1; s >>= 1) {
            const int kb = (int)ceil_div(total_kb, s < total_kb ? s : total_kb), n = (int)ceil_div(total_kb, kb);
            const double t = ceil_div((int64_t)tiles * n, sm_count()) * (kb * (TC_BM + w) * 2.56 + w * 8.0) + (double)n * M * N * 4 / 1500.0;
            if (t < best) { best = t; bn = w; splits = n; }
        }
    }
    CUtensorMap ma, mb, mo;
    if (!make_map(c, &ma, A, K, M, lda, 64) || !make_map(c, &mb, Bm, K, N, ldb, 64) || !make_map_f32(c, &mo, out, M, N, ldo))
        return cudaErrorInvalidValue;
    TcArgs g = {};
    g.M = M; g.N = N; g.K = K;
    g.m_tiles = (int)ceil_div(M, TC_BM); g.n_tiles = (int)ceil_div(N, bn);
    g.kb_per_split = (int)ceil_div(total_kb, splits);
    g.k_splits = (int)ceil_div(total_kb, g.kb_per_split);
    g.out = out; g.ldo = ldo; g.bias = nullptr; g.mask = nullptr; g.ldm = 0; g.colsum = nullptr; g.err = &c.state()->tc_error;
    KernelScope ks(&c.prof, name, st);
    return launch_bn<true, TC_EPI_RED>(bn, ma, mb, mo, ma /*unused*/, g, st);
}

}  // namespace gear
