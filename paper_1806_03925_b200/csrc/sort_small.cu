// Key sort of small ID arrays (at most 32768 entries each), and the accumulate call's plan for the image array behind it.
//
// A cluster of eight blocks (one block for arrays of one tile) per array: the pairs stay in registers and shared memory over
// all passes of a stable radix sort (digits of up to 10 bits, so that a vocabulary of a million takes two passes).  A block
// owns a tile of consecutive entries, a warp 32 * ITEMS of them; it finds equal digits with match_any, sums the warps' digit
// counts column by column, reads the other blocks' counts through distributed shared memory and writes its pairs straight
// into the shared memory of the block that owns their new place.  Two cluster barriers per pass instead of grid barriers and
// trips through the L2.  Bound: latency of the barriers, and instructions: about 500 per 32 entries, which is why the
// work is spread over eight SMs (one block of 1024 threads took 75 us for 12 k entries).
//
// The cluster that sorts the image IDs goes on to plan the accumulate call (plan.cuh) from the keys it holds.
#include <cooperative_groups.h>

#include "common.cuh"
#include "internal.h"
#include "plan.cuh"

namespace gear {

namespace cg = cooperative_groups;

constexpr int SS_THREADS = 512;
constexpr int SS_WARPS = SS_THREADS / 32;
constexpr int SS_MAX_BITS = 10;
constexpr int SS_RADIX = 1 << SS_MAX_BITS;
constexpr int SS_CLUSTER = 8;

template <int ITEMS> constexpr int ss_smem() { return SS_THREADS * ITEMS * 8 + 2 * SS_RADIX * 4 + SS_WARPS * SS_RADIX * 2; }

// A block's place in the cluster and its views of its shared memory (dyn: ss_smem<ITEMS>() bytes; scratch: 2 * SS_WARPS + 2 words)
template <int ITEMS, int CL> struct SmallSort {
    static constexpr int TILE = SS_THREADS * ITEMS;
    uint32_t *skey, *sval;                                                  // the block's tile of the current order
    uint32_t *tot, *base;                                                   // [RADIX] the tile's digit counts (read by the cluster);
                                                                            // where the tile's entries of a digit go
    uint16_t* wcnt;                                                         // [SS_WARPS][RADIX]
    uint32_t* scratch;
    int cr, tile0;

    __device__ __forceinline__ SmallSort(uint32_t* dyn, uint32_t* scr)
        : skey(dyn), sval(dyn + TILE), tot(dyn + 2 * TILE), base(tot + SS_RADIX), wcnt(reinterpret_cast<uint16_t*>(base + SS_RADIX)), scratch(scr) {
        if constexpr (CL == 1) cr = 0; else cr = (int)cg::this_cluster().block_rank();
        tile0 = cr * TILE;
    }
    static __device__ __forceinline__ void sync_cluster() { if constexpr (CL == 1) __syncthreads(); else cg::this_cluster().sync(); }
    template <typename T> static __device__ __forceinline__ T* peer(T* p, int r) {
        if constexpr (CL == 1) return p; else return cg::this_cluster().map_shared_rank(p, r);
    }

    // Sorts n entries of the job; the result is in its first buffer pair, and the block's tile of it in skey / sval.
    __device__ __forceinline__ void sort(const SortJob& j, int n) {
        const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
        const int seg0 = tile0 + warp * 32 * ITEMS;
        const int passes = (j.bits + SS_MAX_BITS - 1) / SS_MAX_BITS, width = (j.bits + passes - 1) / passes;
        const uint32_t mask = (1u << width) - 1u, lt = (1u << lane) - 1u;
        uint32_t key[ITEMS], val[ITEMS];
        bool bad = false;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const int i = seg0 + it * 32 + lane;
            key[it] = 0u; val[it] = (uint32_t)i;
            if (i < n) {
                const int32_t id = __ldg(j.ids + i);
                const bool ok = id >= 0 && (uint32_t)id < j.sentinel;
                bad |= !ok;
                key[it] = ok ? (uint32_t)id : j.sentinel;
                if (j.src) val[it] = (uint32_t)__ldg(j.src + i);
            }
        }
        if (bad && j.status) atomicOr(j.status, GEAR_DEV_BAD_ID);
        for (int pass = 0; pass < passes; ++pass) {
            const int shift = pass * width;
            for (int q = threadIdx.x; q < SS_WARPS * SS_RADIX / 8; q += SS_THREADS) reinterpret_cast<uint4*>(wcnt)[q] = make_uint4(0u, 0u, 0u, 0u);
            __syncthreads();
            uint16_t* mine = wcnt + warp * SS_RADIX;
            uint32_t rank[ITEMS];
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                rank[it] = 0;
                if (seg0 + it * 32 < n) {                                       // warp-uniform
                    const bool valid = seg0 + it * 32 + lane < n;
                    const uint32_t d = valid ? (key[it] >> shift) & mask : 0xffffu;
                    const uint32_t peers = __match_any_sync(0xffffffffu, d);
                    const int leader = __ffs(peers) - 1;
                    uint32_t old = 0;
                    if (valid && lane == leader) {
                        old = mine[d];
                        mine[d] = (uint16_t)(old + __popc(peers));
                    }
                    rank[it] = __shfl_sync(0xffffffffu, old, leader) + __popc(peers & lt);
                    __syncwarp();
                }
            }
            __syncthreads();
            for (int d = threadIdx.x; d < SS_RADIX; d += SS_THREADS) {
                uint32_t total = 0;
                if (d <= (int)mask) {
                    uint32_t c[SS_WARPS];
#pragma unroll
                    for (int w = 0; w < SS_WARPS; ++w) c[w] = wcnt[w * SS_RADIX + d];
#pragma unroll
                    for (int w = 0; w < SS_WARPS; ++w) { wcnt[w * SS_RADIX + d] = (uint16_t)total; total += c[w]; }
                }
                tot[d] = total;
            }
            sync_cluster();                                                     // every tile's counts are there; every tile is in registers
            {
                // a thread owns two adjacent digits
                uint32_t all[2] = {0u, 0u}, before[2] = {0u, 0u};
                if (2 * (int)threadIdx.x <= (int)mask) {
#pragma unroll
                    for (int r = 0; r < CL; ++r) {
                        const uint2 t = *reinterpret_cast<const uint2*>(peer(tot, r) + 2 * threadIdx.x);
                        all[0] += t.x; all[1] += t.y;
                        if (r < cr) { before[0] += t.x; before[1] += t.y; }
                    }
                }
                const uint32_t start = block_exclusive_scan(all[0] + all[1], scratch, nullptr);
                base[2 * threadIdx.x] = start + before[0];
                base[2 * threadIdx.x + 1] = start + all[0] + before[1];
            }
            __syncthreads();
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                if (seg0 + it * 32 + lane < n) {
                    const uint32_t d = (key[it] >> shift) & mask;
                    const uint32_t pos = base[d] + mine[d] + rank[it];
                    const int r = CL == 1 ? 0 : (int)(pos / TILE);
                    const uint32_t at = pos - (uint32_t)r * TILE;
                    peer(skey, r)[at] = key[it];
                    peer(sval, r)[at] = val[it];
                }
            }
            sync_cluster();
            if (pass + 1 < passes) {
#pragma unroll
                for (int it = 0; it < ITEMS; ++it) {
                    const int i = seg0 + it * 32 + lane;
                    if (i < n) { key[it] = skey[i - tile0]; val[it] = sval[i - tile0]; }
                }
            }
        }
        const int live = min(max(n - tile0, 0), TILE);
        for (int i = threadIdx.x; i < live; i += SS_THREADS) { j.keys[0][tile0 + i] = skey[i]; j.vals[0][tile0 + i] = sval[i]; }
    }
};

template <int ITEMS, int CL>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(SS_THREADS)
sort_small_kernel(const SortBatch batch, const PlanArgs plan) {
    wait_for_predecessor();
    extern __shared__ uint32_t dyn[];
    __shared__ uint32_t scratch[2 * SS_WARPS + 2];
    __shared__ int xchg[4];                                                 // plan: last run head; groups, complete groups
    using S = SmallSort<ITEMS, CL>;
    constexpr int TILE = S::TILE;
    S s(dyn, scratch);
    const int job = (int)blockIdx.x / CL, n = (int)batch.job[job].n_max, tile0 = s.tile0, cr = s.cr;
    s.sort(batch.job[job], n);
    if (plan.totals && job == batch.n_jobs - 1) {
        auto key_at = [&](int i) -> uint32_t {
            if (CL == 1 || (unsigned)(i - tile0) < (unsigned)TILE) return s.skey[i - tile0];
            return S::peer(s.skey, i / TILE)[i % TILE];
        };
        plan_tile<ITEMS, SS_WARPS>(plan, n, tile0, key_at, [&](int i) { return s.sval[i - tile0]; }, reinterpret_cast<int*>(scratch),
            [&](int last_head) -> int {                                     // run heads of the tiles before this one
                if (CL == 1) return -1;
                if (threadIdx.x == 0) xchg[0] = last_head;
                S::sync_cluster();
                int run0 = -1;
                for (int r = 0; r < cr; ++r) run0 = max(run0, *S::peer(xchg, r));
                return run0;
            },
            [&](uint32_t g, uint32_t f, uint32_t& g0, uint32_t& f0) {       // groups in the tiles before this one
                g0 = f0 = 0;
                if (threadIdx.x == 0) { xchg[1] = (int)g; xchg[2] = (int)f; }
                S::sync_cluster();
                for (int r = 0; r < cr; ++r) { const int* x = S::peer(xchg, r); g0 += (uint32_t)x[1]; f0 += (uint32_t)x[2]; }
                if (cr == CL - 1 && threadIdx.x == 0) { *plan.totals = make_uint2(g0 + g, f0 + f); plan.state->plan_base = plan.state->q_count; }
            });
        S::sync_cluster();                                                     // nobody leaves while its keys may still be read
    }
}

// Hand-over of a queue that several calls fed (accumulate.cu): reports the count, checks the caller's capacity and, if the queue
// is out of order and short enough, sorts its IDs here.  state->sort_n: 0 nothing to sort, -1 sorted here (first buffer pair),
// n > 0 left to the multi-block sort.  (One launch instead of a count, a key copy and a multi-block sort: 52 us for 1500 entries.)
constexpr int64_t SS_MAX_N = (int64_t)SS_CLUSTER * SS_THREADS * 8;

__global__ void __cluster_dims__(SS_CLUSTER, 1, 1) __launch_bounds__(SS_THREADS)
collect_sort_kernel(const SortJob j, int64_t cap, int64_t* __restrict__ d_n, DevState* __restrict__ state) {
    wait_for_predecessor();
    extern __shared__ uint32_t dyn[];
    __shared__ uint32_t scratch[2 * SS_WARPS + 2];
    SmallSort<8, SS_CLUSTER> s(dyn, scratch);
    const int64_t n = state->q_count;
    const bool sort = n <= cap && state->q_calls > 1, here = sort && n <= SS_MAX_N;       // the same for the whole cluster
    if (s.cr == 0 && threadIdx.x == 0) {
        if (d_n) *d_n = n;
        if (n > cap) atomicOr(&state->status, GEAR_DEV_OUT_CAPACITY);
        state->collect_n = n > cap ? -1 : n;
        state->direct_done = 0;                 // (left by a reduce pass whose hand-over was never enqueued)
        state->sort_n = here ? -1 : sort ? n : 0;
    }
    if (here) s.sort(j, (int)n);
}

cudaError_t launch_collect_sort(const gear_ctx_impl& c, const SortJob& job, int64_t cap, int64_t* d_n, cudaStream_t st) {
    KernelScope k(&c.prof, "collect_sort", st);
    cudaError_t e = cudaFuncSetAttribute(collect_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ss_smem<8>());
    return e == cudaSuccess ? launch_dependent(collect_sort_kernel, dim3(SS_CLUSTER), dim3(SS_THREADS), ss_smem<8>(), st, job, cap, d_n, c.state()) : e;
}
int64_t sort_small_max() { return SS_MAX_N; }

bool sort_small_fits(const SortBatch& batch) {
    for (int j = 0; j < batch.n_jobs; ++j)
        if (batch.job[j].n_max > SS_MAX_N || !batch.job[j].ids || batch.job[j].n_dev) return false;
    return true;
}

// Sorts every job of the batch into its first buffer pair; plan (totals not null): the last job's accumulate plan.
cudaError_t launch_sort_small(const gear_ctx_impl& c, const SortBatch& batch, const PlanArgs& plan, cudaStream_t st) {
    int64_t n = 0;
    for (int j = 0; j < batch.n_jobs; ++j) n = batch.job[j].n_max > n ? batch.job[j].n_max : n;
    KernelScope k(&c.prof, batch.name, st);
    auto launch = [&](auto kernel, int smem, int cl) -> cudaError_t {
        cudaError_t e = smem > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) : cudaSuccess;
        return e == cudaSuccess ? launch_dependent(kernel, dim3(batch.n_jobs * cl), dim3(SS_THREADS), smem, st, batch, plan) : e;
    };
    // one block while a tile holds the longest array (no cluster barriers); tiles of 2048 entries, then of 4096
    if (n <= SS_THREADS * 4) return launch(sort_small_kernel<4, 1>, ss_smem<4>(), 1);
    if (n <= SS_CLUSTER * SS_THREADS * 4) return launch(sort_small_kernel<4, SS_CLUSTER>, ss_smem<4>(), SS_CLUSTER);
    return launch(sort_small_kernel<8, SS_CLUSTER>, ss_smem<8>(), SS_CLUSTER);
}

}  // namespace gear
