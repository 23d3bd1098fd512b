// Stable LSD radix sort of (key, value) pairs and small scan helpers.
//
// One cooperative, persistent kernel sorts up to three independent arrays ("jobs") in one launch.  A job has blocks of its
// own, and a block a chunk of consecutive tiles.  Per pass (digits of up to 9 bits):
//   counts    every block counts the digits of its chunk; grid barrier;
//   totals    a warp per digit turns the blocks' counts into running totals; grid barrier;
//   scatter   a block knows where its first entry of every digit goes and carries that along its tiles: a tile's keys are
//             ranked (a warp owns 32 * ITEMS consecutive elements and finds equal digits with ballots, which keeps equal keys
//             in index order), the pairs put in digit order in shared memory and written out position by position, so that
//             neighbouring threads write neighbouring words; grid barrier.
// (A single pass over the keys with per-tile descriptors and look-back, which saves reading the keys twice, took 22 us per
// tile and block, 8 us of them for the look-back and 5 for match_any: 205 us per pass over 16 M pairs.)
// The first pass can read raw int32 IDs and map out-of-range ones to a sentinel key that sorts last, so no
// separate key-building launch is needed.  Arrays whose live size (known only on the device) fits a few
// tiles are sorted by block 0 alone, with block-level barriers only.
//
// The grid barrier is a monotonically increasing 64-bit arrival counter: barrier k of a launch completes
// when the counter reaches base + grid * (k + 1), where the host knows `base` (it adds up what every
// earlier launch contributes).  The kernel is launched cooperatively, so all blocks are resident; the spin is bounded all
// the same, and a block that gives up records an error and makes every later wait of the launch fall through.
#include "common.cuh"

namespace gear {

constexpr uint32_t GRID_SPIN_LIMIT = 1u << 22;
constexpr int RS_SOLO_TILES = 3;        // live tiles (all jobs) up to which block 0 sorts alone
__device__ __forceinline__ int64_t effective_n(int64_t n_max, const int64_t* n_dev) {
    if (!n_dev) return n_max;
    int64_t n = __ldcg(n_dev);
    return n < n_max ? (n < 0 ? 0 : n) : n_max;
}

// All threads of every participating block call this.  Returns false once the launch has been abandoned.
__device__ __forceinline__ bool grid_barrier(unsigned long long* ctr, unsigned long long target, int32_t* err) {
    __shared__ int ok_flag;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        __threadfence();
        atomicAdd(ctr, 1ull);
        uint32_t spin = 0;
        while (*reinterpret_cast<volatile unsigned long long*>(ctr) < target) {
            if (++spin > GRID_SPIN_LIMIT) { atomicCAS(err, 0, 100); ok = 0; break; }
            if ((spin & 1023u) == 1023u && *reinterpret_cast<volatile int32_t*>(err) != 0) { ok = 0; break; }
        }
        __threadfence();
        ok_flag = ok;
    }
    __syncthreads();
    return ok_flag != 0;
}

__device__ __forceinline__ uint32_t load_key(const SortJob& j, int pass, int64_t i, int src) {
    if (pass == 0 && j.ids) {
        const int32_t id = __ldcg(j.ids + i);
        return (id >= 0 && (uint32_t)id < j.sentinel) ? (uint32_t)id : j.sentinel;
    }
    return __ldcg(j.keys[src] + i);
}

// Dynamic shared memory of a block: a tile's (key, value) pairs in digit order on their way out.
template <int ITEMS> constexpr int rs_stage_bytes() { return RS_THREADS * ITEMS * 8; }

struct SortShared {
    uint32_t scratch[33];
    uint32_t base[RS_BUCKETS];                         // where the next entry of each digit goes (of this block's chunk)
    uint32_t lstart[RS_BUCKETS];                       // where each digit starts in the tile's own digit order
    uint32_t wcnt[RS_THREADS / 32][RS_BUCKETS];
};

// One job, block b of nb.  sync(): barrier over everything that works on the batch; false once it has been abandoned.
template <int ITEMS, typename Sync>
__device__ __forceinline__ bool sort_job(const SortJob& j, int64_t n, int passes, int b, int nb, uint32_t* stage, SortShared& sh, Sync sync) {
    constexpr int TILE = RS_THREADS * ITEMS, WARPS = RS_THREADS / 32, DPT = RS_BUCKETS / RS_THREADS;      // adjacent digits owned by a thread
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const uint32_t mask = (1u << j.width) - 1u, lt = (1u << lane) - 1u;
    const int64_t tiles = ceil_div(n, TILE), per = ceil_div(tiles, nb);
    const int64_t t0 = b * per, t1 = min(tiles, t0 + per);
    for (int pass = 0; pass < passes; ++pass) {
        const int src = pass & 1, dst = src ^ 1, shift = pass * j.width;
        // ---- how many entries of each digit the block's chunk holds
        for (int i = threadIdx.x; i < WARPS * RS_BUCKETS; i += RS_THREADS) (&sh.wcnt[0][0])[i] = 0;
        __syncthreads();
        bool bad = false;
        for (int64_t t = t0; t < t1; ++t) {
            uint32_t key[ITEMS];
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {                    // all loads of the tile in flight before the first is used
                const int64_t i = t * TILE + it * RS_THREADS + threadIdx.x;
                key[it] = i < n ? load_key(j, pass, i, src) : 0u;
            }
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                if (t * TILE + it * RS_THREADS + threadIdx.x < n) {
                    bad |= key[it] == j.sentinel;
                    atomicAdd(&sh.wcnt[warp][(key[it] >> shift) & mask], 1u);
                }
            }
        }
        if (pass == 0 && bad && j.ids && j.status) atomicOr(j.status, GEAR_DEV_BAD_ID);
        __syncthreads();
        for (int d = threadIdx.x; d <= (int)mask; d += RS_THREADS) {
            uint32_t c = 0;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) c += sh.wcnt[w][d];
            __stcg(j.hist + (int64_t)d * nb + b, c);
        }
        if (!sync()) return false;
        // ---- a warp per digit: the counts of the job's blocks become running totals
        for (int d = b * WARPS + warp; d <= (int)mask; d += nb * WARPS) {
            uint32_t run = 0;
            for (int i0 = 0; i0 < nb; i0 += 128) {
                uint32_t v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) { const int i = i0 + q * 32 + lane; v[q] = i < nb ? __ldcg(j.hist + (int64_t)d * nb + i) : 0u; }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int i = i0 + q * 32 + lane;
                    const uint32_t inc = warp_inclusive_scan(v[q]);
                    if (i < nb) __stcg(j.hist + (int64_t)d * nb + i, run + inc - v[q]);
                    run += __shfl_sync(0xffffffffu, inc, 31);
                }
            }
            if (lane == 0) __stcg(j.tot + d, run);
        }
        if (!sync()) return false;
        // ---- where the block's entries of each digit go: digits before it in the whole array, blocks before this one
        {
            uint32_t gtot[DPT], mine = 0;
#pragma unroll
            for (int q = 0; q < DPT; ++q) {
                const int d = threadIdx.x * DPT + q;
                gtot[q] = d <= (int)mask ? __ldcg(j.tot + d) : 0u;
                mine += gtot[q];
            }
            uint32_t ex = block_exclusive_scan(mine, sh.scratch, nullptr);
#pragma unroll
            for (int q = 0; q < DPT; ++q) {
                const int d = threadIdx.x * DPT + q;
                sh.base[d] = ex + (d <= (int)mask ? __ldcg(j.hist + (int64_t)d * nb + b) : 0u);
                ex += gtot[q];
            }
        }
        for (int64_t t = t0; t < t1; ++t) {
            const int64_t seg0 = t * TILE + (int64_t)warp * (32 * ITEMS);
            const bool identity = pass == 0 && j.identity_vals;
            uint32_t key[ITEMS], rank[ITEMS], val[ITEMS];
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {                    // keys and values of the tile: one trip to memory
                const int64_t i = seg0 + it * 32 + lane;
                key[it] = i < n ? load_key(j, pass, i, src) : 0u;
                val[it] = identity ? (j.src && i < n ? (uint32_t)__ldcg(j.src + i) : (uint32_t)i) : (i < n ? __ldcg(j.vals[src] + i) : 0u);
            }
            for (int i = threadIdx.x; i < WARPS * RS_BUCKETS; i += RS_THREADS) (&sh.wcnt[0][0])[i] = 0;
            __syncthreads();
            // equal digits in index order: one ballot per digit bit (match_any takes about a hundred cycles of the SM per warp)
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                const bool valid = seg0 + it * 32 + lane < n;
                const uint32_t d = (key[it] >> shift) & mask;
                uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
                for (int q = 0; q < RS_RADIX_BITS; ++q)
                    if (q < j.width) {                              // uniform
                        const bool one = (d >> q) & 1u;
                        const uint32_t ones = __ballot_sync(0xffffffffu, one);
                        peers &= one ? ones : ~ones;
                    }
                const int leader = __ffs(peers) - 1;                // (of a lane past the end: unused)
                uint32_t old = 0;
                if (valid && lane == leader) {
                    old = sh.wcnt[warp][d];
                    sh.wcnt[warp][d] = old + __popc(peers);
                }
                rank[it] = __shfl_sync(0xffffffffu, old, leader & 31) + __popc(peers & lt);
                __syncwarp();
            }
            __syncthreads();
            // per digit: the warps' counts become running offsets, the tile's counts are scanned into lstart
            uint32_t tot[DPT];
            {
                uint32_t mine = 0;
#pragma unroll
                for (int q = 0; q < DPT; ++q) {
                    const int d = threadIdx.x * DPT + q;
                    uint32_t run = 0;
#pragma unroll
                    for (int w = 0; w < WARPS; ++w) {
                        const uint32_t c = sh.wcnt[w][d];
                        sh.wcnt[w][d] = run;
                        run += c;
                    }
                    tot[q] = run;
                    mine += run;
                }
                uint32_t ex = block_exclusive_scan(mine, sh.scratch, nullptr);
#pragma unroll
                for (int q = 0; q < DPT; ++q) { sh.lstart[threadIdx.x * DPT + q] = ex; ex += tot[q]; }
            }
            __syncthreads();
            // The pairs are first put in digit order inside the tile (shared memory), then written out position by
            // position: neighbouring threads write neighbouring words of a digit's run, so the stores of a warp fall
            // into a few full sectors instead of 32 different ones.
            uint32_t* skey = stage;
            uint32_t* sval = stage + TILE;
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                if (seg0 + it * 32 + lane < n) {
                    const uint32_t d = (key[it] >> shift) & mask;
                    const uint32_t lp = sh.lstart[d] + sh.wcnt[warp][d] + rank[it];
                    skey[lp] = key[it];
                    sval[lp] = val[it];
                }
            }
            __syncthreads();
            const int in_tile = (int)min((int64_t)TILE, n - t * TILE);
            for (int lp = threadIdx.x; lp < in_tile; lp += RS_THREADS) {
                const uint32_t k = skey[lp];
                const uint32_t d = (k >> shift) & mask;
                const uint32_t pos = sh.base[d] + ((uint32_t)lp - sh.lstart[d]);
                __stcg(j.keys[dst] + pos, k);
                __stcg(j.vals[dst] + pos, sval[lp]);
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < DPT; ++q) sh.base[threadIdx.x * DPT + q] += tot[q];
        }
        if (pass + 1 < passes && !sync()) return false;
    }
    return true;
}

// At most 80 registers per thread (three blocks' worth per SM): a sort block then leaves room for a CTA of the
// tensor-core head beside it, which matters because the ID sort of a step runs next to the gather and the head.
template <int ITEMS>
__global__ void __launch_bounds__(RS_THREADS, 3)
coop_sort_kernel(const SortBatch batch) {
    extern __shared__ uint32_t stage[];                // [TILE] keys, then [TILE] values
    __shared__ SortShared sh;
    __shared__ int64_t live_n[3];
    constexpr int TILE = RS_THREADS * ITEMS;
    if (threadIdx.x < 3) live_n[threadIdx.x] = (int)threadIdx.x < batch.n_jobs ? effective_n(batch.job[threadIdx.x].n_max, batch.job[threadIdx.x].n_dev) : 0;
    __syncthreads();
    int64_t live_tiles = 0;
    for (int q = 0; q < batch.n_jobs; ++q) live_tiles += ceil_div(live_n[q], TILE);
    if (live_tiles <= RS_SOLO_TILES) {
        // a few tiles in all: block 0 sorts everything without a grid barrier (and advances the arrival counter on behalf of all)
        if (blockIdx.x != 0) return;
        for (int q = 0; q < batch.n_jobs; ++q)
            if (live_n[q] > 0)
                sort_job<ITEMS>(batch.job[q], live_n[q], batch.passes, 0, 1, stage, sh, [] { __syncthreads(); return true; });
        if (threadIdx.x == 0) {
            // the host has already booked this launch's arrivals: deliver them
            __threadfence();
            atomicAdd(batch.barrier_ctr, (unsigned long long)gridDim.x * (unsigned long long)batch.n_barriers);
        }
        return;
    }
    unsigned long long target = batch.barrier_base;
    int q = 0;
    while (q + 1 < batch.n_jobs && (int)blockIdx.x >= batch.job[q + 1].block0) ++q;
    sort_job<ITEMS>(batch.job[q], live_n[q], batch.passes, (int)blockIdx.x - batch.job[q].block0, batch.job[q].n_blocks, stage, sh, [&]() -> bool {
        target += gridDim.x;
        return grid_barrier(batch.barrier_ctr, target, batch.err);
    });
}

template <int ITEMS> static int coop_grid_limit() {
    static const int limit = [] {
        int per_sm = 0;
        cudaFuncSetAttribute(coop_sort_kernel<ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, rs_stage_bytes<ITEMS>());
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, coop_sort_kernel<ITEMS>, RS_THREADS, rs_stage_bytes<ITEMS>());
        const int n = sm_count() * (per_sm < 1 ? 1 : per_sm > 3 ? 3 : per_sm);
        return n < RS_MAX_BLOCKS ? n : RS_MAX_BLOCKS;
    }();
    return limit;
}

template <int ITEMS> static cudaError_t launch_sort(SortBatch& batch, GridBarrierState* gbs, cudaStream_t st) {
    // every job gets blocks in proportion to its tiles, at least one and at most one per tile
    const int limit = coop_grid_limit<ITEMS>();
    int64_t tiles[3], total = 0;
    for (int j = 0; j < batch.n_jobs; ++j) {
        tiles[j] = ceil_div(batch.job[j].n_max, RS_THREADS * ITEMS);
        if (tiles[j] < 1) tiles[j] = 1;
        total += tiles[j];
    }
    int grid = 0, big = 0;
    for (int j = 0; j < batch.n_jobs; ++j) {
        int64_t nb = total <= limit ? tiles[j] : limit * tiles[j] / total;
        batch.job[j].n_blocks = (int)(nb < 1 ? 1 : nb);
        grid += batch.job[j].n_blocks;
        if (batch.job[j].n_blocks > batch.job[big].n_blocks) big = j;
    }
    if (grid > limit) { batch.job[big].n_blocks -= grid - limit; grid = limit; }      // (very small jobs beside a very large one)
    for (int j = 0, at = 0; j < batch.n_jobs; ++j) { batch.job[j].block0 = at; at += batch.job[j].n_blocks; }
    batch.n_barriers = 3 * batch.passes - 1;            // per pass: counts, running totals, the next order
    batch.barrier_ctr = gbs->device_counter;
    batch.barrier_base = gbs->host_base;
    gbs->host_base += (unsigned long long)grid * (unsigned long long)batch.n_barriers;
    return launch_as(Op::COOPERATIVE, coop_sort_kernel<ITEMS>, dim3(grid), dim3(RS_THREADS), rs_stage_bytes<ITEMS>(), st, batch);
}

int sort_jobs(SortBatch& batch, GridBarrierState* gbs, cudaStream_t st, Profiler* prof, cudaError_t* err_out) {
    int passes = 1;
    int64_t n = 0;
    for (int j = 0; j < batch.n_jobs; ++j) {
        const int p = (batch.job[j].bits + RS_RADIX_BITS - 1) / RS_RADIX_BITS;
        if (p > passes) passes = p;
        n += batch.job[j].n_max;
    }
    for (int j = 0; j < batch.n_jobs; ++j) batch.job[j].width = (batch.job[j].bits + passes - 1) / passes;
    batch.passes = passes;
    KernelScope k(prof, batch.name ? batch.name : "coop_sort", st);
    // smaller tiles while the larger ones would leave blocks idle
    *err_out = n <= (int64_t)RS_THREADS * 8 * coop_grid_limit<8>() ? launch_sort<8>(batch, gbs, st) : launch_sort<16>(batch, gbs, st);
    return passes & 1;
}

// ---------------------------------------------------------------- scan of counter pairs
__global__ void __launch_bounds__(1024)
scan_pairs_kernel(uint2* __restrict__ data, int64_t m, uint2* __restrict__ total) {
    wait_for_predecessor();
    __shared__ uint32_t scratch[33];
    uint32_t ca = 0, cb = 0;
    for (int64_t base = 0; base < m; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        uint2 v = i < m ? data[i] : make_uint2(0u, 0u);
        uint32_t ta, tb;
        uint32_t ea = block_exclusive_scan(v.x, scratch, &ta);
        uint32_t eb = block_exclusive_scan(v.y, scratch, &tb);
        if (i < m) data[i] = make_uint2(ca + ea, cb + eb);
        ca += ta;
        cb += tb;
    }
    if (threadIdx.x == 0) *total = make_uint2(ca, cb);
}

void scan_pairs(uint2* data, int64_t m, uint2* total, cudaStream_t st, Profiler* prof) {
    KernelScope k(prof, "scan_pairs", st);
    launch_dependent(scan_pairs_kernel, dim3(1), dim3(1024), 0, st, data, m, total);
}

}  // namespace gear
