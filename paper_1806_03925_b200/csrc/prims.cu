// Stable LSD radix sort of (key, value) pairs.
//
// One cooperative, persistent kernel sorts up to three independent arrays ("jobs") in one launch.  A job has blocks of its
// own, and a block a chunk of consecutive tiles.  Per pass (digits of up to 9 bits):
//   counts    every block counts the digits of its chunk; grid barrier;
//   totals    a warp per digit turns the blocks' counts into running totals; grid barrier;
//   scatter   a block knows where its first entry of every digit goes and carries that along its tiles: a tile's keys are
//             ranked (a warp owns 32 * ITEMS consecutive elements, equal keys stay in index order), the pairs put in digit order in shared memory and written out position by position, so that
//             neighbouring threads write neighbouring words; grid barrier.
// (A single pass over the keys with per-tile descriptors and look-back, which saves reading the keys twice, took 22 us per
// tile and block, 8 us of them for the look-back and 5 for match_any: 205 us per pass over 16 M pairs.)
// The first pass can read raw int32 IDs and map out-of-range ones to a sentinel key that sorts last, so no
// separate key-building launch is needed.  Arrays whose live size (known only on the device) fits a few
// tiles are sorted by block 0 alone, with block-level barriers only.
//
// The grid barrier is an arrival counter: barrier k of a launch completes when it reaches grid * (k + 1); the last block to
// leave the launch puts it back to zero, so that a launch needs nothing from the host and may be replayed.  The kernel is
// launched cooperatively, so all blocks are resident; the spin is bounded all the same, and a block that gives up records an
// error and makes every later wait of the launch fall through.
#include <type_traits>

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
__device__ __forceinline__ bool grid_barrier(unsigned int* ctr, unsigned int target, int32_t* err) {
    __shared__ int ok_flag;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        __threadfence();
        atomicAdd(ctr, 1u);
        uint32_t spin = 0;
        while (*reinterpret_cast<volatile unsigned int*>(ctr) < target) {
            if (++spin > GRID_SPIN_LIMIT) { atomicCAS(err, 0, 100); ok = 0; break; }
            if ((spin & 1023u) == 1023u && *reinterpret_cast<volatile int32_t*>(err) != 0) { ok = 0; break; }
        }
        __threadfence();
        ok_flag = ok;
    }
    __syncthreads();
    return ok_flag != 0;
}

// Dynamic shared memory of a block, in words (R = 2^width buckets in use).
struct SortSmem {
    uint32_t *skey, *sval;        // [TILE] a tile's pairs in digit order on their way out
    uint32_t *base, *lstart;      // [R] where the next entry of each digit goes; where it starts in the tile's own order
    uint32_t *wcnt, *peers;       // [WARPS][R] counts per warp; [WARPS][R][KEYS] lanes with equal digits (zero between uses)
};
template <int ITEMS> constexpr int rs_smem_bytes(int width, int keys) {
    return (2 * RS_THREADS * ITEMS + (2 + (1 + keys) * (RS_THREADS / 32)) * (1 << width)) * 4;
}
// Keys a lane ranks at a time: two, where the words for that leave room for two blocks on an SM.
constexpr int rs_keys(int width) { return width <= 8 ? 2 : 1; }

// One job, block b of nb.  sync(): barrier over everything that works on the batch; false once it has been abandoned.
template <int ITEMS, int KEYS, typename Sync>
__device__ __forceinline__ bool sort_job(const SortJob& j, int64_t n, int passes, int b, int nb, uint32_t* dyn, uint32_t* scratch, Sync sync) {
    constexpr int TILE = RS_THREADS * ITEMS, WARPS = RS_THREADS / 32;
    static_assert(RS_THREADS >= RS_BUCKETS, "a thread per digit");
    const int R = 1 << j.width, tid = (int)threadIdx.x, lane = (int)lane_id(), warp = tid >> 5;
    const uint32_t mask = (uint32_t)R - 1u, lt = (1u << lane) - 1u;
    SortSmem sh;
    sh.skey = dyn; sh.sval = sh.skey + TILE; sh.base = sh.sval + TILE; sh.lstart = sh.base + R; sh.peers = sh.lstart + R; sh.wcnt = sh.peers + KEYS * WARPS * R;
    uint32_t* my_cnt = sh.wcnt + warp * R;
    uint32_t* my_peers = sh.peers + KEYS * warp * R;
    const int64_t tiles = ceil_div(n, TILE), per = ceil_div(tiles, nb);
    const int64_t t0 = b * per, t1 = min(tiles, t0 + per);
    for (int i = tid; i < KEYS * WARPS * R; i += RS_THREADS) sh.peers[i] = 0;
    for (int pass = 0; pass < passes; ++pass) {
        const int src = pass & 1, dst = src ^ 1, shift = pass * j.width;
        // The first pass may read raw IDs: an ID out of range (a negative one is a large unsigned word) becomes the sentinel, when the
        // key is used and not where it is loaded, where the loads would be waited for (first pass over 16 M IDs: 228 -> 135 us).
        const bool raw = pass == 0 && j.ids;
        const uint32_t* __restrict__ from = raw ? reinterpret_cast<const uint32_t*>(j.ids) : j.keys[src];
        const uint32_t most = raw ? j.sentinel : 0xffffffffu;
        // ---- how many entries of each digit the block's chunk holds
        for (int i = tid; i < WARPS * R; i += RS_THREADS) sh.wcnt[i] = 0;
        __syncthreads();
        bool bad = false;
        for (int64_t t = t0; t < t1; ++t) {
            uint32_t key[ITEMS];
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {                    // all loads of the tile in flight before the first is used
                const int64_t i = t * TILE + it * RS_THREADS + tid;
                key[it] = i < n ? __ldcg(from + i) : 0u;
            }
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                key[it] = min(key[it], most);
                if (t * TILE + it * RS_THREADS + tid < n) {
                    bad |= key[it] == j.sentinel;
                    atomicAdd(&my_cnt[(key[it] >> shift) & mask], 1u);
                }
            }
        }
        if (pass == 0 && bad && j.ids && j.status) atomicOr(j.status, GEAR_DEV_BAD_ID);
        __syncthreads();
        if (tid < R) {
            uint32_t c = 0;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) c += sh.wcnt[w * R + tid];
            __stcg(j.hist + (int64_t)tid * nb + b, c);
        }
        if (!sync()) return false;
        // ---- a warp per digit: the counts of the job's blocks become running totals
        for (int d = b * WARPS + warp; d < R; d += nb * WARPS) {
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
        const bool identity = pass == 0 && j.identity_vals;
        uint32_t key[ITEMS], val[ITEMS];
        auto load = [&](int64_t t) {
            const int64_t seg0 = t * TILE + (int64_t)warp * (32 * ITEMS);
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {                    // keys and values of the tile: one trip to memory
                const int64_t i = seg0 + it * 32 + lane;
                key[it] = i < n ? __ldcg(from + i) : 0u;
                val[it] = identity ? (j.src && i < n ? (uint32_t)__ldcg(j.src + i) : (uint32_t)i) : (i < n ? __ldcg(j.vals[src] + i) : 0u);
            }
        };
        if (t0 < t1) load(t0);
        {
            const uint32_t mine = tid < R ? __ldcg(j.tot + tid) : 0u, chunk = tid < R ? __ldcg(j.hist + (int64_t)tid * nb + b) : 0u;
            const uint32_t ex = block_exclusive_scan(mine, scratch, nullptr);
            if (tid < R) sh.base[tid] = ex + chunk;
        }
        // Four barriers per tile: a warp goes on to rank the next tile's keys while others still write this one out, so what it
        // then touches is its own (its row of counts) or is written behind the next tile's first barrier.
        for (int i = lane; i < R; i += 32) my_cnt[i] = 0;
        __syncwarp();
        uint32_t tot = 0;                                           // the tile's entries of digit tid
        for (int64_t t = t0; t < t1; ++t) {
            const int64_t seg0 = t * TILE + (int64_t)warp * (32 * ITEMS);
            // Lanes with equal digits find one another through a word per warp and digit: every lane sets its bit, then reads
            // the word; the last one puts it back to zero and moves the count on.  (match_any, and a ballot per digit bit, took
            // three times as long.)  With two keys per lane at a
            // time, a word each, half as many trips through shared memory.
            uint32_t rank[ITEMS];
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) key[it] = min(key[it], most);
#pragma unroll
            for (int it = 0; it < ITEMS; it += KEYS) {
                const bool va = seg0 + it * 32 + lane < n;
                const uint32_t da = (key[it] >> shift) & mask;
                if constexpr (KEYS == 1) {
                    if (va) atomicOr(&my_peers[da], 1u << lane);
                    __syncwarp();
                    const uint32_t peers = va ? my_peers[da] : 0u, old = my_cnt[da];
                    rank[it] = old + __popc(peers & lt);
                    __syncwarp();
                    if (peers >> lane == 1u) {                      // the highest lane of its digit
                        my_cnt[da] = old + __popc(peers);
                        my_peers[da] = 0u;
                    }
                } else {
                    const bool vb = seg0 + (it + 1) * 32 + lane < n;
                    const uint32_t db = (key[it + 1] >> shift) & mask;
                    if (va) atomicOr(&my_peers[2 * da], 1u << lane);
                    if (vb) atomicOr(&my_peers[2 * db + 1], 1u << lane);
                    __syncwarp();
                    const uint2 pa = va ? *reinterpret_cast<const uint2*>(my_peers + 2 * da) : make_uint2(0u, 0u);
                    const uint2 pb = vb ? *reinterpret_cast<const uint2*>(my_peers + 2 * db) : make_uint2(0u, 0u);
                    const uint32_t ca = my_cnt[da], cb = my_cnt[db];
                    rank[it] = ca + __popc(pa.x & lt);
                    rank[it + 1] = cb + __popc(pb.x) + __popc(pb.y & lt);
                    __syncwarp();
                    if (pa.x >> lane == 1u) {                       // the highest lane of its digit among the first keys
                        if (pa.y == 0u) my_cnt[da] = ca + __popc(pa.x);
                        my_peers[2 * da] = 0u;
                    }
                    if (pb.y >> lane == 1u) {                       // ... and among the second ones
                        my_cnt[db] = cb + __popc(pb.x) + __popc(pb.y);
                        my_peers[2 * db + 1] = 0u;
                    }
                }
                __syncwarp();
            }
            __syncthreads();
            // per digit: the warps' counts become running offsets, the tile's counts are scanned into lstart
            if (tid < R) sh.base[tid] += tot;                       // the previous tile has been written out
            tot = 0;
            if (tid < R) {
#pragma unroll
                for (int w = 0; w < WARPS; ++w) {
                    const uint32_t c = sh.wcnt[w * R + tid];
                    sh.wcnt[w * R + tid] = tot;
                    tot += c;
                }
            }
            const uint32_t inc = warp_inclusive_scan(tot);
            if (lane == 31) scratch[warp] = inc;
            __syncthreads();
            const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? scratch[lane] : 0u);
            if (tid < R) sh.lstart[tid] = before + inc - tot;
            __syncthreads();
            // The pairs are first put in digit order inside the tile (shared memory), then written out position by
            // position: neighbouring threads write neighbouring words of a digit's run, so the stores of a warp fall
            // into a few full sectors instead of 32 different ones.
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                if (seg0 + it * 32 + lane < n) {
                    const uint32_t d = (key[it] >> shift) & mask;
                    const uint32_t lp = sh.lstart[d] + my_cnt[d] + rank[it];
                    sh.skey[lp] = key[it];
                    sh.sval[lp] = val[it];
                }
            }
            __syncthreads();
            for (int i = lane; i < R; i += 32) my_cnt[i] = 0;
            if (t + 1 < t1) load(t + 1);                            // travels while this tile is written out
            const int in_tile = (int)min((int64_t)TILE, n - t * TILE);
#pragma unroll 4
            for (int lp = tid; lp < in_tile; lp += RS_THREADS) {
                const uint32_t k = sh.skey[lp];
                const uint32_t d = (k >> shift) & mask;
                const uint32_t pos = sh.base[d] + ((uint32_t)lp - sh.lstart[d]);
                __stcg(j.keys[dst] + pos, k);
                __stcg(j.vals[dst] + pos, sh.sval[lp]);
            }
            __syncwarp();
        }
        if (pass + 1 < passes && !sync()) return false;
    }
    return true;
}

template <int ITEMS, int KEYS>
__global__ void __launch_bounds__(RS_THREADS, 2)
coop_sort_kernel(const SortBatch batch) {
    extern __shared__ uint32_t dyn[];
    __shared__ uint32_t scratch[33];
    __shared__ int64_t live_n[3];
    constexpr int TILE = RS_THREADS * ITEMS;
    if (threadIdx.x < 3) live_n[threadIdx.x] = (int)threadIdx.x < batch.n_jobs ? effective_n(batch.job[threadIdx.x].n_max, batch.job[threadIdx.x].n_dev) : 0;
    __syncthreads();
    int64_t live_tiles = 0;
    for (int q = 0; q < batch.n_jobs; ++q) live_tiles += ceil_div(live_n[q], TILE);
    if (live_tiles <= RS_SOLO_TILES) {
        // a few tiles in all: block 0 sorts everything without a grid barrier
        if (blockIdx.x != 0) return;
        for (int q = 0; q < batch.n_jobs; ++q)
            if (live_n[q] > 0) {
                __syncthreads();
                sort_job<ITEMS, KEYS>(batch.job[q], live_n[q], batch.passes, 0, 1, dyn, scratch, [] { __syncthreads(); return true; });
            }
        return;
    }
    unsigned int target = 0;             // at most 512 blocks * 12 barriers
    int q = 0;
    while (q + 1 < batch.n_jobs && (int)blockIdx.x >= batch.job[q + 1].block0) ++q;
    sort_job<ITEMS, KEYS>(batch.job[q], live_n[q], batch.passes, (int)blockIdx.x - batch.job[q].block0, batch.job[q].n_blocks, dyn, scratch, [&]() -> bool {
        target += gridDim.x;
        return grid_barrier(batch.barrier, target, batch.err);
    });
    // nobody arrives or looks any more once all have come here (a block that gave up too): the counts start again from zero
    __syncthreads();
    if (threadIdx.x == 0 && atomicInc(batch.barrier + 1, gridDim.x - 1) == gridDim.x - 1) batch.barrier[0] = 0u;
}

template <int ITEMS, int KEYS> constexpr int coop_smem() { return rs_smem_bytes<ITEMS>(KEYS == 2 ? 8 : RS_RADIX_BITS, KEYS); }      // of the widest digit
template <int ITEMS, int KEYS> static int coop_grid_limit() {
    static const int limit = [] {
        int per_sm = 0;
        constexpr int smem = coop_smem<ITEMS, KEYS>();
        allow_smem<coop_sort_kernel<ITEMS, KEYS>>(smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, coop_sort_kernel<ITEMS, KEYS>, RS_THREADS, smem);
        const int n = sm_count() * (per_sm < 1 ? 1 : per_sm > 2 ? 2 : per_sm);
        return n < RS_MAX_BLOCKS ? n : RS_MAX_BLOCKS;
    }();
    return limit;
}

template <int ITEMS, int KEYS> static cudaError_t launch_sort(SortBatch& batch, int width, cudaStream_t st) {
    // every job gets blocks in proportion to its tiles, at least one and at most one per tile
    const int limit = coop_grid_limit<ITEMS, KEYS>();
    if (const cudaError_t e = allow_smem<coop_sort_kernel<ITEMS, KEYS>>(coop_smem<ITEMS, KEYS>())) return e;
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
    return launch_as(Op::COOPERATIVE, coop_sort_kernel<ITEMS, KEYS>, dim3(grid), dim3(RS_THREADS), rs_smem_bytes<ITEMS>(width, KEYS), st, batch);
}

int sort_jobs(SortBatch& batch, cudaStream_t st, Profiler* prof, cudaError_t* err_out) {
    int passes = 1;
    int64_t n = 0;
    for (int j = 0; j < batch.n_jobs; ++j) {
        const int p = (batch.job[j].bits + RS_RADIX_BITS - 1) / RS_RADIX_BITS;
        if (p > passes) passes = p;
        n += batch.job[j].n_max;
    }
    int width = 1;
    for (int j = 0; j < batch.n_jobs; ++j) {
        batch.job[j].width = (batch.job[j].bits + passes - 1) / passes;
        width = batch.job[j].width > width ? batch.job[j].width : width;
    }
    batch.passes = passes;
    KernelScope k(prof, batch.name ? batch.name : "coop_sort", st);
    // smaller tiles while the larger ones would leave blocks idle
    auto launch = [&](auto keys) {
        constexpr int K = decltype(keys)::value;
        return n <= (int64_t)RS_THREADS * 4 * coop_grid_limit<4, K>() ? launch_sort<4, K>(batch, width, st) : launch_sort<8, K>(batch, width, st);
    };
    *err_out = rs_keys(width) == 2 ? launch(std::integral_constant<int, 2>{}) : launch(std::integral_constant<int, 1>{});
    return passes & 1;
}

}  // namespace gear
