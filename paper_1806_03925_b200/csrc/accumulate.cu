// Event 5 and event 6 of the step: the gradient store.
//
// Rule (Section 1 of the paper, "accumulated to M"; Section 3, event 6): gradients of one image are kept
// until M have arrived; their average is then handed on and the store for that image starts over.  Rows
// are taken to arrive in index order, so a call that brings k rows for an image holding c0 earlier ones
// completes floor((c0 + k) / M) groups, split exactly at every M-th arrival, and leaves (c0 + k) mod M.
//
// Plan on the device, nothing is read back:
//   1. keys = Image IDs (out-of-range -> sentinel that sorts last); stable radix sort with the row index
//      as value, so rows of one image are contiguous and still in arrival order.
//   2. flag pass: position i of the sorted array starts a group if it is the first row of its image or if
//      (c0 + rank within image) is a multiple of M; a group is complete if the image has enough further
//      rows to reach the next multiple.  Per-tile counts of (groups, complete groups).
//   3. every block of the plan pass adds up the counts before its tile (sections of 64 tiles, then tiles).
//   4. plan pass: the flags again, now with their global prefix: group g starts at grp_start[g]; complete
//      groups get consecutive ready-queue slots (a counter-threshold stream compaction: ballot-free block
//      scan of the "count reaches M" predicate).
//      Arrays of at most 32768 rows are sorted and planned by one kernel instead (sort_small.cu).
//   5. reduce pass: a warp sums the rows of each of its groups (fp32, arrival order, whole rows staged through
//      shared memory by asynchronous copies, addressed through the sort permutation) and either writes the
//      average to its queue slot or, for the open group, the running sum and count back to the table.  The
//      warp that owns the first group of an image also settles what the image's last, still open group
//      leaves in the table, so no two warps touch one table row.
//   6. commit (by the reduce pass): the queue length grows by the number of
//      complete groups (or the call is dropped whole if the queue would overflow).
// HBM bound: the reduce pass reads every gradient row once and reads/writes one accumulator row per
// distinct image; the sort and flag passes move 4-byte keys only.
#include "common.cuh"
#include "internal.h"

namespace gear {

constexpr int AF_THREADS = 256;
constexpr int AF_ITEMS = 4;
constexpr int AF_TILE = AF_THREADS * AF_ITEMS;
constexpr int AF_WARPS = AF_THREADS / 32;

__device__ __forceinline__ uint32_t warp_inclusive_max(uint32_t v) {
    const unsigned lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= (unsigned)o) v = max(v, t);
    }
    return v;
}

// The AF_ITEMS consecutive words a thread owns (a 16-byte load away from the array's end).
__device__ __forceinline__ void load_items(uint32_t (&v)[AF_ITEMS], const uint32_t* __restrict__ p, uint32_t i0, uint32_t n, uint32_t pad) {
    static_assert(AF_ITEMS == 4, "one 16-byte load");
    if (i0 + AF_ITEMS <= n) {
        const uint4 q = __ldg(reinterpret_cast<const uint4*>(p + i0));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        return;
    }
#pragma unroll
    for (int t = 0; t < AF_ITEMS; ++t) v[t] = i0 + t < n ? p[i0 + t] : pad;
}

// Flags of the AF_ITEMS consecutive sorted positions a thread owns.
struct TileFlags {
    uint32_t key[AF_ITEMS];
    bool head[AF_ITEMS];       // starts a group
    bool first[AF_ITEMS];      // ... and is the first row of its image in this call
    bool complete[AF_ITEMS];   // ... and the group reaches M
    int c0[AF_ITEMS];          // rows the image already holds in the table
    int seq[AF_ITEMS];         // group heads: how many groups of the image this call completes before this one
    uint32_t i0;               // first position owned by this thread (positions are below 2^31: 32-bit arithmetic throughout)
};

// smem: AF_WARPS + 1 words, not to be written again before the block's next barrier.  Every thread of the block must call this.
// (One barrier here and one in each pass: with a block scan per count, nine and fifteen of them, the passes waited at barriers
// for half of their time.)
// run_end (optional): run_end[first position of an image's run] = one past its last position.
__device__ __forceinline__ void tile_flags(TileFlags& f, const uint32_t* __restrict__ ks, uint32_t n, uint32_t vocab,
                                           const DivM& div, const int32_t* __restrict__ cnt, uint32_t* smem,
                                           DevState* __restrict__ state, uint32_t* __restrict__ run_end = nullptr) {
    const uint32_t tile0 = blockIdx.x * (uint32_t)AF_TILE;
    f.i0 = tile0 + threadIdx.x * (uint32_t)AF_ITEMS;
    uint32_t prev = vocab;   // key just before this thread's first position
    if (f.i0 < n && f.i0 > 0) prev = ks[f.i0 - 1];
    load_items(f.key, ks, f.i0, n, vocab);

    // start of the image's run that covers the tile's first position (the run may begin in an earlier tile).  Warp 0
    // searches backwards with all its lanes at once: first one round of probes at distances 1, 2, 4, ... brackets the
    // start, then rounds of 32 evenly spaced probes narrow the bracket by a factor of 32 each, so that even a run of
    // millions of rows (a hot image) costs a handful of trips to memory, and the usual short run one.
    if (threadIdx.x < 32) {
        const int lane0 = (int)threadIdx.x;
        const uint32_t key0 = __shfl_sync(0xffffffffu, f.key[0], 0);
        uint32_t start = tile0;
        const bool spans = tile0 > 0 && tile0 < n && ks[tile0 - 1] == key0;      // the same words for every lane
        if (spans) {
            int64_t hi = (int64_t)tile0 - 1;                         // ks[hi] == key0
            const int64_t far = hi - ((int64_t)1 << lane0);
            const bool same = lane0 < 31 && far >= 0 && ks[far] == key0;
            const int k = __popc(__ballot_sync(0xffffffffu, same));  // probes 0 .. k-1 still lie inside the run
            int64_t lo = hi - ((int64_t)1 << k);                     // ks[lo] != key0, or lo < 0
            if (lo < -1) lo = -1;
            if (k > 0) hi -= (int64_t)1 << (k - 1);
            while (hi - lo > 1) {
                const int64_t step = (hi - lo + 31) / 32;
                const int64_t p = hi - (int64_t)(lane0 + 1) * step;
                const bool in = p > lo && ks[p] == key0;
                const int m = __popc(__ballot_sync(0xffffffffu, in));
                hi -= (int64_t)m * step;
                const int64_t below = hi - step;
                if (below > lo) lo = below;                          // the first probe that failed (it lies above the old lo)
            }
            start = (uint32_t)hi;
        }
        if (lane0 == 0) smem[AF_WARPS] = start;
    }
    // rows the images already hold: asked for ahead of the barrier
#pragma unroll
    for (int t = 0; t < AF_ITEMS; ++t)
        f.c0[t] = f.i0 + t < n && f.key[t] < vocab && (t == 0 || f.key[t] != f.key[t > 0 ? t - 1 : 0]) ? __ldg(cnt + f.key[t]) : 0;
    // run start of every position: inclusive max-scan of "index if run head"
    uint32_t local_max = 0;
    uint32_t run_start[AF_ITEMS];
#pragma unroll
    for (int t = 0; t < AF_ITEMS; ++t) {
        const uint32_t before = t == 0 ? prev : f.key[t - 1];
        const bool run_head = (f.i0 + t < n) && (f.i0 + t == 0 || f.key[t] != before);
        if (run_head) { local_max = f.i0 + t + 1u; }   // +1 so that 0 means "none"
        run_start[t] = local_max;
    }
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    uint32_t inc = warp_inclusive_max(local_max);
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    uint32_t before_thread = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) before_thread = 0;
    before_thread = max(before_thread, __reduce_max_sync(0xffffffffu, lane < warp ? smem[lane] : 0u));
    const uint32_t carry = smem[AF_WARPS];

#pragma unroll
    for (int t = 0; t < AF_ITEMS; ++t) {
        const uint32_t i = f.i0 + t;
        f.head[t] = f.first[t] = f.complete[t] = false;
        f.seq[t] = 0;
        if (i >= n || f.key[t] >= vocab) continue;
        uint32_t rs = max(run_start[t], before_thread);
        const uint32_t start = rs ? rs - 1 : carry;
        const uint32_t j = i - start;                // rank of this row among the call's rows of its image
        if (t > 0 && f.key[t] == f.key[t > 0 ? t - 1 : 0]) f.c0[t] = f.c0[t > 0 ? t - 1 : 0];
        const int c0 = f.c0[t];
        const uint32_t x = (uint32_t)c0 + j, full = div(x);
        const uint32_t rem = x - full * (uint32_t)div.M;
        if (j == 0 || rem == 0) {
            f.head[t] = true;
            f.first[t] = (j == 0);
            f.seq[t] = (int)full;           // c0 < M: the first group of the image gets 0
            const uint32_t last = i + ((uint32_t)div.M - rem) - 1u;  // the row that brings the count to M
            f.complete[t] = last < n && ks[last] == f.key[t];
        }
        const uint32_t after = i + 1 < n ? ks[i + 1] : vocab;
        if (after >= vocab) state->n_valid = i + 1;                     // exactly one thread sees this
        if (run_end && after != f.key[t]) run_end[start] = i + 1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && (n == 0 || ks[0] >= vocab)) state->n_valid = 0;   // no valid row at all
}

// Counts of (groups, complete groups, in the upper word): per tile, and per section of AF_SECTION tiles (zero before a plan).
struct PlanCounts { uint2* tile; unsigned long long* section; };
constexpr int AF_SECTION = 64;

__global__ void __launch_bounds__(AF_THREADS)
acc_flag_kernel(const uint32_t* __restrict__ ks, uint32_t n, uint32_t vocab, const DivM div, const int32_t* __restrict__ cnt,
                const PlanCounts counts, DevState* __restrict__ state) {
    wait_for_predecessor();
    __shared__ uint32_t smem[AF_WARPS + 1], s_cnt[AF_WARPS];
    TileFlags f;
    tile_flags(f, ks, n, vocab, div, cnt, smem, state);
    uint32_t gc = 0;                                                // groups, complete groups (upper half): at most AF_TILE each
#pragma unroll
    for (int t = 0; t < AF_ITEMS; ++t) gc += (uint32_t)f.head[t] | ((uint32_t)f.complete[t] << 16);
    gc = __reduce_add_sync(0xffffffffu, gc);
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    if (lane == 0) s_cnt[warp] = gc;
    __syncthreads();
    if (warp == 0) {
        gc = __reduce_add_sync(0xffffffffu, lane < AF_WARPS ? s_cnt[lane] : 0u);
        const uint32_t tg = gc & 0xffffu, tc = gc >> 16;
        if (lane == 0) {
            counts.tile[blockIdx.x] = make_uint2(tg, tc);
            if (tg) atomicAdd(counts.section + blockIdx.x / AF_SECTION, (unsigned long long)tg | ((unsigned long long)tc << 32));
        }
    }
}

__global__ void __launch_bounds__(AF_THREADS)
acc_plan_kernel(const uint32_t* __restrict__ ks, uint32_t n, uint32_t vocab, const DivM div, const int32_t* __restrict__ cnt,
                const PlanCounts counts, uint2* __restrict__ totals, uint4* __restrict__ grp_rec, uint32_t* __restrict__ blk_first, uint32_t* __restrict__ run_end,
                int span, DevState* __restrict__ state) {
    wait_for_predecessor();
    __shared__ uint32_t smem[AF_WARPS + 1], s_cnt[AF_WARPS], s_g[AF_WARPS], s_c[AF_WARPS];
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    // groups in the sections and tiles before this one: a thread's share of both counts in one word (each stays below 2^30)
    const int section = (int)blockIdx.x / AF_SECTION;
    unsigned long long before = 0;
    for (int q = threadIdx.x; q < section; q += AF_THREADS) before += counts.section[q];
    const int q = section * AF_SECTION + (int)threadIdx.x;
    if (threadIdx.x < AF_SECTION && q < (int)blockIdx.x) { const uint2 v = counts.tile[q]; before += (unsigned long long)v.x | ((unsigned long long)v.y << 32); }
    TileFlags f;
    tile_flags(f, ks, n, vocab, div, cnt, smem, state, run_end);
    uint32_t gc = 0;                                                // groups, complete groups (upper half): at most AF_TILE each
#pragma unroll
    for (int t = 0; t < AF_ITEMS; ++t) gc += (uint32_t)f.head[t] | ((uint32_t)f.complete[t] << 16);
    const uint32_t inc = warp_inclusive_scan(gc);
    const uint32_t bg = __reduce_add_sync(0xffffffffu, (uint32_t)before), bc = __reduce_add_sync(0xffffffffu, (uint32_t)(before >> 32));
    if (lane == 31) { s_cnt[warp] = inc; s_g[warp] = bg; s_c[warp] = bc; }
    __syncthreads();
    const uint32_t of_warp = lane < AF_WARPS ? s_cnt[lane] : 0u;
    const uint32_t g0 = __reduce_add_sync(0xffffffffu, lane < AF_WARPS ? s_g[lane] : 0u), c0 = __reduce_add_sync(0xffffffffu, lane < AF_WARPS ? s_c[lane] : 0u);
    const uint32_t rank = __reduce_add_sync(0xffffffffu, lane < warp ? of_warp : 0u) + inc - gc, tile = __reduce_add_sync(0xffffffffu, of_warp);
    uint32_t gi = g0 + (rank & 0xffffu), ci = c0 + (rank >> 16);
    const int64_t q_base = state->q_count;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) { *totals = make_uint2(g0 + (tile & 0xffffu), c0 + (tile >> 16)); state->plan_base = q_base; }
#pragma unroll
    for (int t = 0; t < AF_ITEMS; ++t) {
        // the reduce pass hands out spans of 2^span sorted positions: index of the first group that starts in each
        if (((f.i0 + t) & ((1 << span) - 1)) == 0 && f.i0 + t < n && f.key[t] < vocab) blk_first[(f.i0 + t) >> span] = gi;
        if (!f.head[t]) continue;
        // one 16-byte record per group: start position (top bit: first group of its image in this call), image ID,
        // ready-queue slot (-1: the group stays open), and for the image's first group the rows the image already held,
        // for a later one its number among the groups of the image that this call completes
        grp_rec[gi] = make_uint4((f.i0 + t) | (f.first[t] ? 0x80000000u : 0u), f.key[t],
                                 (uint32_t)(f.complete[t] ? (int32_t)(q_base + ci) : -1),
                                 (uint32_t)(f.first[t] ? f.c0[t] : f.seq[t]));
        ++gi;
        ci += f.complete[t];
    }
}

// Where the row of sorted position p lives and what it is scaled by: pmeta[p] = (source row, scale bits); or, where the call
// names neither source rows nor scales, row perm[p] as it is.
struct RowGather {
    const float* grads; int64_t ld;
    const int2* pmeta; const uint32_t* perm;
};

// What a lane knows about "its" group of a span: own rows [start, start + len), then zlen rows from zstart.
struct LaneGroup {
    uint32_t start, key, zstart;
    int slot, c0, len, zlen, items;      // items = rows the warp stages for the group (0: nothing to do)
    int seq;                             // number of the group among those of its image that the call completes
    bool first;
};

// Where the averages of the groups a call completes go when they bypass the ready queue: the caller's own lists
// (gear_accumulate_collect).  All null: the groups join the queue.  cap < 0: the host has checked that the queue is empty
// and that the lists can take every group the call could complete.  cap >= 0: the kernel decides: the lists are used if
// the queue is empty and the call completes at most cap groups, else the groups join the queue and the hand-over pass
// that the host has enqueued behind this kernel deals with them.
struct EmitTarget { int32_t* ids; int32_t* seq; float* avg; int64_t* d_n; int64_t cap; };

// One row to stage, as the copy side sees it (where the row starts; bit 0 of the address word is set if the item
// exists) and as the adding side sees it (what the row is scaled by and
// meta = group lane << 2 | last item of the group << 1 | last of the group's own rows).
struct ItemDesc { uint32_t addr_lo, addr_hi; float scale; int meta; };

// The reduce pass.  A warp takes spans of 2^span_log2 (at most ACC_SPAN) sorted positions, span w, w + W, w + 2W, ... (W = warps of
// the grid); the groups that start inside a span (at most ACC_SPAN, one per lane) are walked as one flat
// sequence of items -- for every group first the image's accumulator row if it holds anything, then its
// gradient rows in arrival order; the first group of an image, if it completes, is followed by the rows of
// the image's trailing open group, so that one warp alone reads and writes the image's accumulator row.
// Items are staged through a per-warp ring of S row-sized shared-memory slots with asynchronous copies
// (cp.async, 16 bytes per lane, whole rows): the copy of item i + S - 1 is issued before item i is added,
// across group boundaries, so a warp keeps S - 1 rows in flight whatever the group sizes are -- most
// groups hold a single row, and registers alone cannot keep enough of those in flight.  What to copy is
// worked out 32 items at a time, one item per lane (a search over the groups' item counts, the position
// record fetched by the lane), one batch ahead of the copies; the inner loop only broadcasts a lane's
// descriptor, copies and adds.  The group records of the next span are requested while the current span
// streams.  Sums are fp32, in arrival order, starting from the stored partial sum.
// FULL: a row is exactly NQ * 512 bytes, so no lane is ever idle.  PLAIN: the caller's rows as they are (a store of 16 M rows
// then needs no 128 MB of records).
template <int NQ, int S, bool FULL, bool PLAIN>
__global__ void __launch_bounds__(256, NQ <= 2 ? 3 : 2)
acc_reduce_kernel(RowGather rg, int D, const DivM div, int span_log2, int64_t ready_cap, const uint2* __restrict__ plan_totals, const uint4* __restrict__ grp_rec,
                  const uint32_t* __restrict__ blk_first, const uint32_t* __restrict__ run_end,
                  float* __restrict__ gsum, int32_t* __restrict__ gcnt,
                  int32_t* __restrict__ q_id, float* __restrict__ q_avg, const EmitTarget direct,
                  unsigned long long* __restrict__ sections, int n_sections, DevState* __restrict__ state) {
    wait_for_predecessor();
    // the plan's section counts are not needed any more: zero for the next plan
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); i < n_sections; i += (int)(gridDim.x * blockDim.x)) sections[i] = 0ull;
    extern __shared__ float4 ring_mem[];                          // [warps][S][NQ * 32] float4
    const uint2 totals = *plan_totals;
    const int64_t n_groups = totals.x, q_base = state->plan_base;
    // Averages go to the ready queue, or (the queue being empty, so that queue slot k is also entry k of the hand-over)
    // straight into the caller's lists, whose capacity the host has checked against the row count.
    const bool to_caller = direct.avg != nullptr &&
                           (direct.cap < 0 || (q_base == 0 && (int64_t)totals.y <= direct.cap));
    int32_t* __restrict__ e_id = to_caller ? direct.ids : q_id;
    float* __restrict__ e_avg = to_caller ? direct.avg : q_avg;
    const bool dropped = !to_caller && q_base + (int64_t)totals.y > ready_cap;
    // Step 6 of the plan (commit), by one thread: every block goes by the queue length that the plan noted.  (The block that
    // found itself last did it before, behind a fence and a ticket that the call's end waited for.)
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state->direct_done = (to_caller && direct.cap >= 0) ? 1 : 0;
        if (to_caller) { if (direct.d_n) *direct.d_n = totals.y; }
        else if (dropped) atomicOr(&state->status, GEAR_DEV_READY_OVERFLOW);
        else if (totals.y > 0) { state->q_count = q_base + totals.y; state->q_calls += 1; }
    }
    if (dropped) return;                                             // the whole call is dropped
    const int64_t n_valid = state->n_valid;
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const int n_chunks = D / 4;
    const float m_f = (float)div.M;
    const int64_t W = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t n_spans = (n_valid + (1 << span_log2) - 1) >> span_log2;
    float4* my_ring = ring_mem + (size_t)warp * S * (NQ * 32);
    const uint32_t ring_addr = (uint32_t)__cvta_generic_to_shared(my_ring);
    constexpr uint32_t SLOT_BYTES = NQ * 32 * 16;

    // group range of a span: lane 0 holds the first group, lane 1 one past the last
    auto load_range = [&](int64_t span) -> uint32_t {
        uint32_t v = 0;
        if (span < n_spans && lane < 2) {
            const int64_t w = span + lane;
            v = w < n_spans ? __ldg(blk_first + w) : (uint32_t)n_groups;
        }
        return v;
    };
    auto load_group = [&](int64_t g_lo, int64_t g_hi) -> LaneGroup {
        LaneGroup r{0u, 0u, 0u, -1, 0, 0, 0, 0, 0, false};
        const int64_t g = g_lo + lane;
        if (g < g_hi) {
            const uint4 rec = __ldg(grp_rec + g);
            const uint32_t end = (g + 1 < n_groups) ? (__ldg(&grp_rec[g + 1].x) & 0x7fffffffu) : (uint32_t)n_valid;
            r.start = rec.x & 0x7fffffffu; r.first = rec.x >> 31; r.key = rec.y; r.slot = (int)rec.z;
            r.c0 = r.first ? (int)rec.w : 0;
            r.seq = r.first ? 0 : (int)rec.w;
            r.len = (int)(end - r.start);
        }
        return r;
    };

    int64_t span = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    uint32_t range_cur = load_range(span), range_nxt = load_range(span + W);
    LaneGroup G = load_group(__shfl_sync(0xffffffffu, range_cur, 0), __shfl_sync(0xffffffffu, range_cur, 1));

    for (; span < n_spans; span += W) {
        // ---- look-ahead: group records of the next span, group range of the one after it
        const LaneGroup G_nxt = load_group(__shfl_sync(0xffffffffu, range_nxt, 0), __shfl_sync(0xffffffffu, range_nxt, 1));
        const uint32_t range_nxt2 = load_range(span + 2 * W);

        // ---- complete this lane's group
        if (G.first && G.slot >= 0) {
            // what the image's remaining rows leave in the table: the rows of its trailing open group
            const uint32_t run_stop = __ldg(run_end + G.start);
            const uint32_t rows = (uint32_t)G.c0 + (run_stop - G.start);
            G.zlen = (int)(rows - div(rows) * (uint32_t)div.M);
            G.zstart = run_stop - (uint32_t)G.zlen;
        }
        // an image's trailing open group itself (not first, no queue slot) is skipped here
        if (G.len > 0 && (G.first || G.slot >= 0)) G.items = (G.c0 > 0 ? 1 : 0) + G.len + G.zlen;
        const int incl = (int)warp_inclusive_scan((uint32_t)G.items);      // items of the groups in lanes 0 .. lane
        const int total_items = __shfl_sync(0xffffffffu, incl, 31);
        if (total_items > 0) {
            // descriptor of item base + lane
            auto make_desc = [&](int base) -> ItemDesc {
                const int i = base + lane;
                int l = 0;                                      // group lane: the first one with incl > i
#pragma unroll
                for (int step = ACC_SPAN / 2; step >= 1; step >>= 1) {
                    const int v = __shfl_sync(0xffffffffu, incl, l + step - 1);
                    if (v <= i) l += step;
                }
                const int incl_l = __shfl_sync(0xffffffffu, incl, l), items_l = __shfl_sync(0xffffffffu, G.items, l);
                const int c0_l = __shfl_sync(0xffffffffu, G.c0, l), len_l = __shfl_sync(0xffffffffu, G.len, l);
                const uint32_t start_l = __shfl_sync(0xffffffffu, G.start, l);
                const uint32_t zstart_l = __shfl_sync(0xffffffffu, G.zstart, l);
                const uint32_t key_l = __shfl_sync(0xffffffffu, G.key, l);
                const int k = i - (incl_l - items_l);           // item number within the group
                const int tab = c0_l > 0 ? 1 : 0, own_end = tab + len_l;
                const bool ok = i < total_items, is_tab = k < tab;
                const int64_t p = k < own_end ? (int64_t)start_l + (k - tab) : (int64_t)zstart_l + (k - own_end);
                int2 pm = make_int2(0, __float_as_int(1.f));
                if (ok && !is_tab) {
                    if constexpr (PLAIN) pm.x = (int)__ldg(rg.perm + p); else pm = __ldg(rg.pmeta + p);
                }
                const float* row = (ok && is_tab) ? gsum + (int64_t)key_l * D : rg.grads + (int64_t)pm.x * rg.ld;
                const uint64_t a = reinterpret_cast<uint64_t>(row) | (ok ? 1ull : 0ull);      // rows are 16-byte aligned
                ItemDesc d;
                d.addr_lo = (uint32_t)a; d.addr_hi = (uint32_t)(a >> 32);
                d.scale = __int_as_float(pm.y);
                d.meta = (l << 2) | (k + 1 == items_l ? 2 : 0) | (k + 1 == own_end ? 1 : 0);
                return d;
            };

            float4 acc[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);

            // acc holds the group's own rows (own_done) and/or everything the warp adds for it (all_done)
            auto settle = [&](int l, bool own_done, bool all_done) {
                const uint32_t key = __shfl_sync(0xffffffffu, G.key, l);
                const int slot = __shfl_sync(0xffffffffu, G.slot, l);
                float* srow = gsum + (int64_t)key * D;
                if (own_done && slot >= 0) {                    // the group reached M: its average joins the queue
                    float* qrow = e_avg + (int64_t)slot * D;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const int ch = lane + 32 * q;
                        if (FULL || ch < n_chunks)
                            st_f4(qrow + ch * 4, make_float4(acc[q].x / m_f, acc[q].y / m_f, acc[q].z / m_f, acc[q].w / m_f));
                        acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    if (lane == 0) e_id[slot] = (int32_t)key;
                    if (to_caller) {
                        const int seq = __shfl_sync(0xffffffffu, G.seq, l);
                        if (lane == 0) direct.seq[slot] = seq;
                    }
                }
                if (all_done) {
                    const int c0 = __shfl_sync(0xffffffffu, G.c0, l), len = __shfl_sync(0xffffffffu, G.len, l);
                    const int zlen = __shfl_sync(0xffffffffu, G.zlen, l);
                    const bool first = __shfl_sync(0xffffffffu, (int)G.first, l) != 0;
                    // the table row: the open group (this one if it did not complete, else the image's trailing one)
                    const bool write_row = first && (slot < 0 || zlen > 0 || c0 > 0);
                    if (write_row) {
#pragma unroll
                        for (int q = 0; q < NQ; ++q) {
                            const int ch = lane + 32 * q;
                            if (FULL || ch < n_chunks) st_f4(srow + ch * 4, acc[q]);
                        }
                        if (lane == 0) gcnt[key] = slot < 0 ? c0 + len : zlen;
                    }
#pragma unroll
                    for (int q = 0; q < NQ; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            };

            // cur / nxt: the items being added (base .. base + 31) and the batch after them; icur / inxt: the same for the
            // copies, which run S - 1 items ahead (lane j of icur is item base + j + S - 1)
            ItemDesc cur = make_desc(0), nxt = make_desc(32), icur = make_desc(S - 1), inxt = make_desc(32 + S - 1);
            int islot = 0, cslot = 0;
            auto advance = [](int slot) { return (S & (S - 1)) == 0 ? ((slot + 1) & (S - 1)) : (slot + 1 == S ? 0 : slot + 1); };
            // copy of the item in lane j of descriptor batch d (an empty copy if the item does not exist)
            auto issue = [&](const ItemDesc& d, int j) {
                const uint32_t lo = __shfl_sync(0xffffffffu, d.addr_lo, j), hi = __shfl_sync(0xffffffffu, d.addr_hi, j);
                const float* src = reinterpret_cast<const float*>(((uint64_t)hi << 32) | (lo & ~15u));
                const int bytes = (int)(lo & 1u) << 4;
                const uint32_t dst = ring_addr + (uint32_t)islot * SLOT_BYTES;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int ch = lane + 32 * q;
                    const bool on = FULL || ch < n_chunks;          // lanes past the end of a narrow row copy nothing
                    cp_async_16(dst + (uint32_t)ch * 16u, src + (on ? ch * 4 : 0), on ? bytes : 0);
                }
                cp_async_commit();
                islot = advance(islot);
            };

            // ---- the pipeline: S - 1 items ahead
            __syncwarp();
#pragma unroll
            for (int i = 0; i < S - 1; ++i) issue(cur, i);
            for (int base = 0; base < total_items; base += 32) {
                const int n_in = min(32, total_items - base);
                for (int j = 0; j < n_in; ++j) {
                    __syncwarp();                                 // every lane is done with the slot refilled next
                    issue(icur, j);
                    cp_async_wait<S - 1>();
                    __syncwarp();                                 // ... and sees the other lanes' copies of item base + j
                    const float scale = __shfl_sync(0xffffffffu, cur.scale, j);
                    const int meta = __shfl_sync(0xffffffffu, cur.meta, j);
                    const float4* row = my_ring + (size_t)cslot * (NQ * 32);
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const float4 v = row[lane + 32 * q];
                        // in the indirect form the scaled row is never stored: the product joins the sum with one rounding
                        acc[q].x = fmaf(scale, v.x, acc[q].x); acc[q].y = fmaf(scale, v.y, acc[q].y);
                        acc[q].z = fmaf(scale, v.z, acc[q].z); acc[q].w = fmaf(scale, v.w, acc[q].w);
                    }
                    if (meta & 3) settle(meta >> 2, (meta & 1) != 0, (meta & 2) != 0);
                    cslot = advance(cslot);
                }
                cur = nxt; icur = inxt;
                nxt = make_desc(base + 64);
                inxt = make_desc(base + 64 + S - 1);
            }
            cp_async_wait<0>();
        }
        G = G_nxt; range_nxt = range_nxt2;
    }
}

// Steps 2-4 of the plan over the sorted keys ks (flag pass, plan pass).
static cudaError_t enqueue_plan(const gear_ctx_impl& c, const uint32_t* ks, int64_t n, cudaStream_t st) {
    const int64_t vocab = c.cfg.img_vocab;
    const DivM div = make_div(c.cfg.M);
    DevState* state = c.state();
    const int64_t n_tiles = ceil_div(n, AF_TILE);
    uint2* tile_cnt = c.at<uint2>(c.ws.tile_cnt);
    const PlanCounts counts{tile_cnt, c.at<unsigned long long>(c.ws.plan_sections)};
    // the reduce pass puts the sections back to zero; a plan that never got there left them
    if (c.plan_sections_dirty) {
        cudaError_t me = enqueue_memset(counts.section, sizeof(unsigned long long) * (size_t)c.plan_sections_dirty, st);
        if (me != cudaSuccess) return me;
    }
    c.plan_sections_dirty = (int)ceil_div(n_tiles, AF_SECTION);
    cudaError_t e;
    { KernelScope k(&c.prof, "acc_flag", st);
    e = launch_dependent(acc_flag_kernel, dim3((unsigned)n_tiles), dim3(AF_THREADS), 0, st, ks, (uint32_t)n, (uint32_t)vocab, div, c.buf.dfv_gcnt, counts, state); }
    if (e != cudaSuccess) return e;
    KernelScope k(&c.prof, "acc_plan", st);
    return launch_dependent(acc_plan_kernel, dim3((unsigned)n_tiles), dim3(AF_THREADS), 0, st, ks, (uint32_t)n, (uint32_t)vocab, div, c.buf.dfv_gcnt, counts, tile_cnt + n_tiles,
                            c.at<uint4>(c.ws.grp_rec), c.at<uint32_t>(c.ws.blk_first),
                            c.at<uint32_t>(c.ws.run_end), acc_span_log2(n), state);
}

// The plan for the image occurrences of the batch gear_forward_backward has just sorted, enqueued ahead of the
// accumulate call that will use it (on the side stream, beside the head): it depends on the sorted IDs, the counts in
// the table and the queue length only, none of which changes before that call unless another accumulate or collect
// comes first -- those calls drop the plan.
cudaError_t launch_accumulate_plan_ahead(const gear_ctx_impl& c, int64_t n, cudaStream_t st) {
    c.plan_ready = false;
    if (n <= 0 || !c.img_sorted || !c.img_sort_valid || c.cfg.accum_mode != GEAR_ACC_SORT) return cudaSuccess;
    SortJob sb = c.sort_job(gear_ctx_impl::SORT_IMG);
    cudaError_t e = enqueue_plan(c, sb.keys[c.img_sorted_buf], n, st);
    if (e == cudaSuccess) note_plan(c, n, nullptr, nullptr);
    return e;
}
// Where every sorted row lives and what it is scaled by, one 8-byte record each, resolved through the sort permutation once, so
// that the reduce pass reads both with one coalesced load (resolving there, 32 rows ahead of the copies, made it wait: 71 -> 79 us
// for the store of 65 k views).
__global__ void __launch_bounds__(256)
plan_resolve_kernel(int n, const DevState* __restrict__ state, const uint32_t* __restrict__ perm, const int32_t* __restrict__ src_row,
                    const float* __restrict__ scale, int2* __restrict__ pmeta) {
    wait_for_predecessor();
    const int i = (int)(blockIdx.x * 256 + threadIdx.x);
    if (i >= min(n, (int)state->n_valid)) return;          // rows without a valid image have no record
    int src = (int)__ldg(perm + i);
    if (src_row) src = __ldg(src_row + src);
    // (below zero: as in plan_tile)
    pmeta[i] = make_int2(max(src, 0), __float_as_int(src < 0 ? 0.f : scale ? __ldg(scale + src) : 1.f));
}
static cudaError_t launch_plan_resolve(const gear_ctx_impl& c, const uint32_t* perm, int64_t n, const int32_t* src_row, const float* scale, cudaStream_t st) {
    KernelScope k(&c.prof, "plan_resolve", st);
    return launch_dependent(plan_resolve_kernel, dim3((unsigned)ceil_div(n, 256)), dim3(256), 0, st, (int)n, (const DevState*)c.state(), perm,
                            src_row, scale, c.at<int2>(c.ws.pmeta));
}
cudaError_t launch_accumulate_resolve_ahead(const gear_ctx_impl& c, int64_t n, const int32_t* src_row, const float* scale, cudaStream_t st) {
    if (!c.plan_ready) return cudaSuccess;
    note_plan(c, n, src_row, scale);
    return launch_plan_resolve(c, c.sort_job(gear_ctx_impl::SORT_IMG).vals[c.img_sorted_buf], n, src_row, scale, st);
}
void note_plan(const gear_ctx_impl& c, int64_t n, const int32_t* src_row, const float* scale) {
    c.plan_ready = true; c.plan_n = n; c.plan_src_row = src_row; c.plan_scale = scale;
}
PlanArgs plan_args(const gear_ctx_impl& c, int64_t n, const int32_t* src_row, const float* scale) {
    return PlanArgs{c.at<uint2>(c.ws.tile_cnt) + ceil_div(n, AF_TILE), (uint32_t)c.cfg.img_vocab, c.buf.dfv_gcnt, c.at<uint4>(c.ws.grp_rec), src_row, scale,
                    c.at<int2>(c.ws.pmeta), c.at<uint32_t>(c.ws.blk_first), c.at<uint32_t>(c.ws.run_end), c.state(), make_div(c.cfg.M), acc_span_log2(n)};
}

// to_caller (optional): the caller's lists; only valid while the ready queue is known to be empty and the lists hold
// at least n entries (gear_accumulate_collect checks both on the host)
static cudaError_t launch_accumulate_to(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld,
                                        const int32_t* src_row, const float* scale, int64_t n, const EmitTarget& to_caller,
                                        cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int64_t vocab = c.cfg.img_vocab;
    const int D = c.cfg.dfv_dim, M = c.cfg.M;
    SortJob sb = c.sort_job(gear_ctx_impl::SORT_IMG);
    DevState* state = c.state();
    bool planned = !img_id && c.plan_ready && c.plan_n == n && c.plan_src_row == src_row && c.plan_scale == scale;
    c.plan_ready = false;
    // "the batch of the last gear_forward_backward" after a call with explicit IDs has used the sort buffers: sort again
    const bool resort_batch = !img_id && !c.img_sort_valid;
    if (resort_batch) img_id = c.last_img_id;
    int cur = c.img_sorted_buf;
    if (img_id) {
        SortBatch batch = c.sort_batch();
        batch.n_jobs = 1;
        batch.job[0] = sb;
        batch.job[0].ids = img_id;
        batch.job[0].sentinel = (uint32_t)vocab;
        batch.job[0].n_max = n;
        batch.job[0].bits = bits_for(vocab);
        cudaError_t se;
        batch.name = "sort_img";
        planned = sort_small_fits(batch);
        if (planned) { se = launch_sort_small(c, batch, plan_args(c, n, src_row, scale), st); cur = 0; }
        else cur = sort_jobs(batch, st, &c.prof, &se);
        if (se != cudaSuccess) return se;
        c.img_sort_valid = resort_batch;
        if (resort_batch) c.img_sorted_buf = cur;
    }
    const uint32_t* ks = sb.keys[cur];
    if (!planned) {
        cudaError_t pe = enqueue_plan(c, ks, n, st);
        if (pe == cudaSuccess && (src_row || scale)) pe = launch_plan_resolve(c, sb.vals[cur], n, src_row, scale, st);
        if (pe != cudaSuccess) return pe;
    }
    uint4* grp_rec = c.at<uint4>(c.ws.grp_rec);
    const bool plain = !src_row && !scale;
    RowGather rg{grads, ld, c.at<int2>(c.ws.pmeta), sb.vals[cur]};
    uint32_t* blk_first = c.at<uint32_t>(c.ws.blk_first);
    uint32_t* run_end = c.at<uint32_t>(c.ws.run_end);

    const int nq = (int)ceil_div(D / 4, 32);
    const int span = acc_span_log2(n);
    const int64_t want = ceil_div(ceil_div(n, 1 << span), 8);
    const int resident = sm_count() * (nq <= 2 ? 3 : 2);          // every block stays resident
    const int grid = (int)(want < resident ? (want < 1 ? 1 : want) : resident);
    cudaError_t le = cudaSuccess;
    { KernelScope k(&c.prof, "acc_reduce", st);
    auto launch = [&](auto kernel, int slot_bytes, int slots) {
        const int smem = 8 * slots * slot_bytes;
        le = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (le != cudaSuccess) return;
        le = launch_dependent(kernel, dim3(grid), dim3(256), (size_t)smem, st, rg, D, make_div(M), span, c.ws.ready_cap, c.at<uint2>(c.ws.tile_cnt) + ceil_div(n, AF_TILE), grp_rec, blk_first, run_end,
                                        c.buf.dfv_gsum, c.buf.dfv_gcnt, c.at<int32_t>(c.ws.q_id),
                                        c.at<float>(c.ws.q_avg), to_caller, c.at<unsigned long long>(c.ws.plan_sections), c.plan_sections_dirty, state);
    };
    // ring depth: as many row slots as about 96 KB per block (two blocks per SM) allow, at most 8.
    // FULL only when a row fills the instantiated width exactly (D == NQ * 128): every lane then owns a chunk of every
    // row; any other width (also 384, 640, 768, 896, which round up to the next instantiation) keeps the per-chunk guard
#define GEAR_ACC_LAUNCH(NQ, S) \
    do { \
        if (D == NQ * 128) { if (plain) launch(acc_reduce_kernel<NQ, S, true, true>, NQ * 512, S); else launch(acc_reduce_kernel<NQ, S, true, false>, NQ * 512, S); } \
        else if (plain) launch(acc_reduce_kernel<NQ, S, false, true>, NQ * 512, S); \
        else launch(acc_reduce_kernel<NQ, S, false, false>, NQ * 512, S); \
    } while (0)
    if (nq <= 1) GEAR_ACC_LAUNCH(1, 8);
    else if (nq <= 2) GEAR_ACC_LAUNCH(2, 8);
    else if (nq <= 4) GEAR_ACC_LAUNCH(4, 5);
    else GEAR_ACC_LAUNCH(8, 3);
#undef GEAR_ACC_LAUNCH
    }
    if (le != cudaSuccess) return le;
    c.plan_sections_dirty = 0;
    if (!to_caller.avg) ++c.acc_calls_pending;                    // a call that bypasses the queue leaves it empty (a call
                                                                  // that may or may not bypass it: see launch_accumulate_collect)
    return cudaGetLastError();
}

cudaError_t launch_accumulate(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld,
                              const int32_t* src_row, const float* scale, int64_t n, cudaStream_t st) {
    return launch_accumulate_to(c, img_id, grads, ld, src_row, scale, n, EmitTarget{nullptr, nullptr, nullptr, nullptr, -1}, st);
}

// Events 5 and 6 in one call.  When the host knows the ready queue to be empty (no accumulate call since a collect that
// could not be refused) and the caller's lists can take every group the n rows could complete, the reduce pass writes
// ids, emission numbers and averages straight into the caller's lists and its first thread reports the count: no
// hand-over pass, and the averages cross memory once.  Otherwise: accumulate into the queue, then hand the queue over.
cudaError_t launch_accumulate_collect(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld,
                                      const int32_t* src_row, const float* scale, int64_t n, int32_t* ids, int32_t* seq,
                                      float* avg, int64_t cap, int64_t* d_n, cudaStream_t st) {
    const bool queue_empty = c.cfg.accum_mode == GEAR_ACC_SORT && c.acc_calls_pending == 0 && n > 0;
    if (queue_empty && cap >= n)
        return launch_accumulate_to(c, img_id, grads, ld, src_row, scale, n, EmitTarget{ids, seq, avg, d_n, -1}, st);
    if (queue_empty && cap > 0) {
        // the lists may or may not be long enough for what this call completes: the reduce pass finds out, and the
        // hand-over pass behind it moves the queue only if the reduce pass had to use it
        cudaError_t de = launch_accumulate_to(c, img_id, grads, ld, src_row, scale, n, EmitTarget{ids, seq, avg, d_n, cap}, st);
        if (de != cudaSuccess) return de;
        c.acc_calls_pending = 1;
        return launch_collect_ready(c, ids, seq, avg, cap, d_n, st);
    }
    cudaError_t e = cudaSuccess;
    if (n > 0)
        e = c.cfg.accum_mode == GEAR_ACC_ATOMIC
                ? launch_accumulate_atomic(c, img_id ? img_id : c.last_img_id, grads, ld, src_row, scale, n, st)
                : launch_accumulate(c, img_id, grads, ld, src_row, scale, n, st);
    if (e != cudaSuccess) return e;
    return launch_collect_ready(c, ids, seq, avg, cap, d_n, st);
}

// ---------------------------------------------------------------- GEAR_ACC_ATOMIC: the store without arrival order
// Rows are added to the accumulator rows with fp32 reductions in whatever order the hardware takes them, so
// which arrivals share a group is not defined; what is defined (and equal to the ordered path) is every
// image's count and its number of emissions.  After all rows of the call have been added, every image that
// was touched and now holds k >= M gradients emits floor(k / M) averages, each the mean of all k pooled
// gradients, and keeps k mod M gradients' worth of that mean, so that nothing is lost or counted twice.
// Under heavy skew the reductions of a hot image serialise on its accumulator row; that is the cost the
// sorted path avoids.
constexpr int32_t ACC_TOUCHED = 0x40000000;      // bit of dfv_gcnt[id] while a call is in flight: id is on the touched list

// A block takes 256 rows at a time, puts them in ID order (bitonic sort of 64-bit words in registers and, for the longer
// exchanges, shared memory) and a warp adds up the rows of each ID in its 32 positions before one reduction per ID goes to memory.
// Bound by the reductions on the hottest image otherwise: one row's 512 bytes take about 5 ns, and with Zipf(1.3) IDs a quarter
// of the rows are one image's (99.7 k rows: 118 us with a reduction per row).
__global__ void __launch_bounds__(256)
acc_atomic_add_kernel(const int32_t* __restrict__ img_id, int64_t n, int64_t vocab, const float* __restrict__ grads,
                      int64_t ld, const int32_t* __restrict__ src_row, const float* __restrict__ scale, int D,
                      float* __restrict__ gsum, int32_t* __restrict__ gcnt, int32_t* __restrict__ touched,
                      int64_t ready_cap, DevState* __restrict__ state) {
    wait_for_predecessor();
    // a call completes at most n groups: refuse it whole if the queue could not take them
    const bool drop = state->q_count + n > ready_cap;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state->pad[3] = drop ? 1 : 0;
        state->n_copies = 0;
        if (drop) atomicOr(&state->status, GEAR_DEV_READY_OVERFLOW);
    }
    if (drop) return;
    __shared__ unsigned long long xchg[256];
    const int lane = (int)lane_id(), tid = (int)threadIdx.x;
    int flags = 0;
    for (int64_t r0 = (int64_t)blockIdx.x * 256; r0 < n; r0 += (int64_t)gridDim.x * 256) {
        int32_t id = -1;
        if (r0 + tid < n) {
            id = __ldg(img_id + r0 + tid);
            if (id < 0 || id >= vocab) { flags |= GEAR_DEV_BAD_ID; id = -1; }
        }
        unsigned long long w = ((unsigned long long)(uint32_t)id << 32) | (uint32_t)tid;       // invalid rows sort last
#pragma unroll
        for (int k = 2; k <= 256; k <<= 1)
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                unsigned long long o;
                if (j >= 32) {
                    __syncthreads();
                    xchg[tid] = w;
                    __syncthreads();
                    o = xchg[tid ^ j];
                } else o = __shfl_xor_sync(0xffffffffu, w, j);
                const bool keep_min = ((tid & j) == 0) == ((tid & k) == 0);
                w = keep_min == (o < w) ? o : w;
            }
        id = (int32_t)(uint32_t)(w >> 32);
        const bool live = id >= 0;
        const int64_t r = r0 + (int64_t)(uint32_t)(w & 0xffffffffu);
        int64_t src = 0;
        float sc = 0.f;
        if (live) {
            src = src_row ? (int64_t)__ldg(src_row + r) : r;
            sc = scale ? __ldg(scale + src) : 1.f;
        }
        // ends[j]: position j is the last of its ID among the warp's
        const int32_t next = __shfl_down_sync(0xffffffffu, id, 1);
        const bool end = live && (lane == 31 || next != id);
        const uint32_t ends = __ballot_sync(0xffffffffu, end);
        const int m = __popc(__ballot_sync(0xffffffffu, live));
        if (end) {
            const uint32_t below = ends & ((1u << lane) - 1u);
            const int len = lane - (below ? 31 - __clz(below) : -1);
            const int32_t before = atomicOr(&gcnt[id], ACC_TOUCHED);
            atomicAdd(&gcnt[id], len);
            const bool fresh = !(before & ACC_TOUCHED);
            const uint32_t fr = __ballot_sync(ends, fresh);          // (the lanes of `ends` are the ones here)
            unsigned long long pos = 0;
            const int leader = __ffs(ends) - 1;
            if (lane == leader && fr) pos = atomicAdd(reinterpret_cast<unsigned long long*>(&state->pad[2]), (unsigned long long)__popc(fr));
            pos = __shfl_sync(ends, pos, leader);
            if (fresh) touched[pos + __popc(fr & ((1u << lane) - 1u))] = id;
        }
        __syncwarp();
        for (int c0 = 0; c0 < D / 4; c0 += 32) {
            const int ch = c0 + lane;
            const bool on = ch < D / 4;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int p0 = 0; p0 < m; p0 += 8) {
                float4 v[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int64_t s = __shfl_sync(0xffffffffu, src, p0 + t);
                    v[t] = on && p0 + t < m ? ld_stream_f4(grads + s * ld + ch * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const float f = __shfl_sync(0xffffffffu, sc, p0 + t);
                    const int32_t to = __shfl_sync(0xffffffffu, id, p0 + t);
                    acc.x = fmaf(f, v[t].x, acc.x); acc.y = fmaf(f, v[t].y, acc.y);
                    acc.z = fmaf(f, v[t].z, acc.z); acc.w = fmaf(f, v[t].w, acc.w);
                    if ((ends >> (p0 + t)) & 1u) {
                        if (on) red_add_f4(gsum + (int64_t)to * D + ch * 4, acc);
                        acc = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            }
        }
    }
    if (flags) atomicOr(&state->status, flags);
}

// An image may emit one average many times (hot ones: a quarter of a call's rows / M).  The warp that settles it writes the first
// SETTLE_COPIES; the others are written by a launch of their own, a warp per 32 of them.  (One warp wrote 25 thousand copies of the
// hottest image's average: M = 1, 99.7 k rows, 569 us for the call.)
constexpr int SETTLE_COPIES = 32;
struct CopyList { uint32_t* src; uint32_t* first; uint32_t* count; };      // queue slots [first, first + count) repeat slot src

// A warp takes 4 to 32 touched images, as few as the grid allows: a lane settles the count of one, the warp together the rows of
// those that emit.
__global__ void __launch_bounds__(256)
acc_atomic_settle_kernel(const int32_t* __restrict__ touched, int D, const DivM div, float* __restrict__ gsum,
                         int32_t* __restrict__ gcnt, int32_t* __restrict__ q_id, float* __restrict__ q_avg, const CopyList copies,
                         DevState* __restrict__ state) {
    wait_for_predecessor();
    if (state->pad[3] != 0) return;                            // the call was dropped
    const int64_t n_touched = state->pad[2];
    const int lane = (int)lane_id();
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    if (blockIdx.x == 0 && threadIdx.x == 0)                   // emission order is not ID order: collect has to sort
        atomicAdd(reinterpret_cast<unsigned long long*>(&state->q_calls), 2ull);
    const int per = (int)min((int64_t)32, max((int64_t)4, (n_touched + warps - 1) / warps));
    for (int64_t t0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per; t0 < n_touched; t0 += warps * per) {
        int32_t id = 0, k = 0, e = 0, rest = 0;
        if (lane < per && t0 + lane < n_touched) {
            id = touched[t0 + lane];
            k = gcnt[id] & ~ACC_TOUCHED;
            e = (int32_t)div((uint32_t)k);
            rest = k - e * div.M;
            gcnt[id] = rest;
        }
        uint32_t todo = __ballot_sync(0xffffffffu, e > 0);
        if (!todo) continue;
        // queue slots for all of them with one addition
        const uint32_t incl = warp_inclusive_scan((uint32_t)e), total = __shfl_sync(0xffffffffu, incl, 31);
        unsigned long long slot0 = 0;
        if (lane == 0) slot0 = atomicAdd(reinterpret_cast<unsigned long long*>(&state->q_count), (unsigned long long)total);
        slot0 = __shfl_sync(0xffffffffu, slot0, 0);
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            const int32_t id_l = __shfl_sync(0xffffffffu, id, l), e_l = __shfl_sync(0xffffffffu, e, l);
            const unsigned long long slot = slot0 + (__shfl_sync(0xffffffffu, incl, l) - (uint32_t)e_l);
            const float kf = (float)__shfl_sync(0xffffffffu, k, l), rf = (float)__shfl_sync(0xffffffffu, rest, l);
            const int32_t here = min(e_l, SETTLE_COPIES);
            float* row = gsum + (int64_t)id_l * D;
            for (int ch = lane; ch < D / 4; ch += 32) {
                const float4 sum = ld_f4(row + ch * 4);
                const float4 avg = make_float4(sum.x / kf, sum.y / kf, sum.z / kf, sum.w / kf);
                for (int32_t j = 0; j < here; ++j) st_f4(q_avg + (int64_t)(slot + j) * D + ch * 4, avg);
                st_f4(row + ch * 4, make_float4(avg.x * rf, avg.y * rf, avg.z * rf, avg.w * rf));
            }
            if (lane < here) q_id[slot + lane] = id_l;
            if (e_l > here) {
                const uint32_t n_rec = (uint32_t)(e_l - here + 31) / 32u;
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&state->n_copies, n_rec);
                at = __shfl_sync(0xffffffffu, at, 0);
                for (uint32_t r = lane; r < n_rec; r += 32) {
                    copies.src[at + r] = (uint32_t)slot;
                    copies.first[at + r] = (uint32_t)slot + (uint32_t)here + 32u * r;
                    copies.count[at + r] = min(32u, (uint32_t)(e_l - here) - 32u * r);
                }
            }
        }
    }
}

__global__ void __launch_bounds__(256)
acc_atomic_copy_kernel(int D, const CopyList copies, int32_t* __restrict__ q_id, float* __restrict__ q_avg, const DevState* __restrict__ state) {
    wait_for_predecessor();
    const uint32_t n = state->n_copies, lane = lane_id();
    for (uint32_t r = blockIdx.x * 8 + (threadIdx.x >> 5); r < n; r += gridDim.x * 8) {
        const uint32_t src = copies.src[r], first = copies.first[r], count = copies.count[r];
        if (lane < count) q_id[first + lane] = q_id[src];
        for (int ch = (int)lane; ch < D / 4; ch += 32) {
            const float4 v = ld_f4(q_avg + (int64_t)src * D + ch * 4);
            for (uint32_t j = 0; j < count; ++j) st_f4(q_avg + (int64_t)(first + j) * D + ch * 4, v);
        }
    }
}

cudaError_t launch_accumulate_atomic(const gear_ctx_impl& c, const int32_t* img_id, const float* grads, int64_t ld,
                                     const int32_t* src_row, const float* scale, int64_t n, cudaStream_t st) {
    c.plan_ready = false;
    if (n <= 0) return cudaSuccess;
    DevState* state = c.state();
    int32_t* touched = c.at<int32_t>(c.ws.pmeta);               // the sorted path's scratch is free in this mode
    // (at most n emissions, so far fewer records than the sort buffers, which this mode does not use, have words)
    const SortJob free_buffers = c.sort_job(gear_ctx_impl::SORT_IMG);
    const CopyList copies{free_buffers.keys[0], free_buffers.vals[0], free_buffers.keys[1]};
    cudaError_t e = enqueue_memset(&state->pad[2], sizeof(int64_t), st);
    if (e != cudaSuccess) return e;
    const int resident = sm_count() * 8;
    auto grid = [&](int64_t want) { return dim3((unsigned)(want < resident ? (want < 1 ? 1 : want) : resident)); };
    { KernelScope k(&c.prof, "acc_atomic_add", st);
    e = launch_dependent(acc_atomic_add_kernel, grid(ceil_div(n, 256)), dim3(256), 0, st, img_id, n, c.cfg.img_vocab, grads, ld, src_row, scale, c.cfg.dfv_dim,
                         c.buf.dfv_gsum, c.buf.dfv_gcnt, touched, c.ws.ready_cap, state); }
    if (e != cudaSuccess) return e;
    // at most n images are touched; a warp that finds nothing to do costs nothing, so the grid follows n
    { KernelScope k(&c.prof, "acc_atomic_settle", st);
    e = launch_dependent(acc_atomic_settle_kernel, grid(ceil_div(n, 256)), dim3(256), 0, st, touched, c.cfg.dfv_dim, make_div(c.cfg.M), c.buf.dfv_gsum, c.buf.dfv_gcnt,
                         c.at<int32_t>(c.ws.q_id), c.at<float>(c.ws.q_avg), copies, state); }
    if (e != cudaSuccess) return e;
    if ((n + c.cfg.M - 1) / c.cfg.M > SETTLE_COPIES) {          // else no image can emit more than the settle pass writes
        KernelScope k(&c.prof, "acc_atomic_copy", st);
        e = launch_dependent(acc_atomic_copy_kernel, grid(ceil_div(n, (int64_t)c.cfg.M * 256)), dim3(256), 0, st, c.cfg.dfv_dim, copies,
                             c.at<int32_t>(c.ws.q_id), c.at<float>(c.ws.q_avg), (const DevState*)state);
    }
    if (e != cudaSuccess) return e;
    c.acc_calls_pending += 2;
    return cudaGetLastError();
}

// ---------------------------------------------------------------- event 6b: hand the ready queue over
// Output entry k comes from queue slot perm[k] (or k itself when the queue is already in order); its emission
// number is its rank among equal IDs.  IDs and emission numbers: one thread per entry.  Rows: a warp copies
// eight rows at a time, 16 bytes per lane, all loads issued before the first store.
__global__ void __launch_bounds__(256)
collect_move_kernel(const uint32_t* __restrict__ keys_small, const uint32_t* __restrict__ perm_small,
                    const uint32_t* __restrict__ keys_large, const uint32_t* __restrict__ perm_large, const int32_t* __restrict__ q_id, const float* __restrict__ q_avg,
                    int D, DevState* __restrict__ state, int32_t* __restrict__ ids, int32_t* __restrict__ seq,
                    float* __restrict__ avg, int solo, int64_t cap, int64_t* __restrict__ d_n) {
    wait_for_predecessor();
    // solo: this launch is the whole hand-over (a queue fed by one accumulate call is in order already): it checks
    // the caller's capacity itself.  Either way the last block to finish empties the queue.
    const int64_t n = solo ? state->q_count : state->collect_n;
    if (solo) {
        if (state->direct_done != 0) {
            // the reduce pass in front of this launch has written the caller's lists and the count itself: nothing to
            // move; the block that leaves last takes the mark down
            __shared__ int last_out;
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                last_out = atomicInc(&state->pad32, gridDim.x - 1) == gridDim.x - 1;
                if (last_out) state->direct_done = 0;
            }
            return;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            if (d_n) *d_n = n;
            if (n > cap) atomicOr(&state->status, GEAR_DEV_OUT_CAPACITY);
        }
        if (n > cap) return;                            // nothing is consumed
    }
    const int64_t sort_n = solo ? 0 : state->sort_n;
    const bool in_order = sort_n == 0;                 // the queue itself is sorted: no permutation
    const uint32_t* ks = in_order ? reinterpret_cast<const uint32_t*>(q_id) : sort_n < 0 ? keys_small : keys_large;
    const uint32_t* sorted_perm = sort_n < 0 ? perm_small : perm_large;
    const int64_t threads = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += threads) {
        const uint32_t id = ks[k];
        // first index of this ID's run: gallop backwards, then bisect
        int64_t hi = k, step = 1, lo = k - 1;                  // ks[hi] == id
        while (lo >= 0 && ks[lo] == id) { hi = lo; step <<= 1; lo = max(hi - step, (int64_t)-1); }
        int64_t l = lo + 1, h = hi;                            // answer in [l, h]; ks[h] == id, ks[lo] != id
        while (l < h) {
            const int64_t mid = (l + h) >> 1;
            if (ks[mid] == id) h = mid; else l = mid + 1;
        }
        ids[k] = (int32_t)id;
        seq[k] = (int32_t)(k - l);
    }
    const unsigned lane = lane_id();
    const int64_t warps = threads >> 5;
    const int chunks = D / 4;
    constexpr int R = 8;
    for (int64_t k0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k0 < n; k0 += R * warps) {
        int64_t src[R];
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int64_t k = k0 + t * warps;
            src[t] = k < n ? (in_order ? k : (int64_t)sorted_perm[k]) : -1;
        }
        for (int ch = lane; ch < chunks; ch += 32) {
            float4 v[R];
#pragma unroll
            for (int t = 0; t < R; ++t)
                v[t] = src[t] >= 0 ? ld_stream_f4(q_avg + src[t] * D + ch * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int t = 0; t < R; ++t)
                if (src[t] >= 0) st_f4(avg + (k0 + t * warps) * D + ch * 4, v[t]);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicInc(&state->pad32, gridDim.x - 1) == gridDim.x - 1 && n >= 0) { state->q_count = 0; state->q_calls = 0; }
    }
}

cudaError_t launch_collect_ready(const gear_ctx_impl& c, int32_t* ids, int32_t* seq, float* avg, int64_t cap,
                                 int64_t* d_n, cudaStream_t st) {
    DevState* state = c.state();
    c.plan_ready = false;                                    // a plan made ahead counted on the queue length of before
    SortJob sb = c.sort_job(gear_ctx_impl::SORT_READY);
    const int64_t n_max = c.ws.ready_cap;
    const int64_t resident = (int64_t)sm_count() * 8;       // blocks of 256 threads that fit the GPU at once
    // A queue fed by at most one accumulate call is in (id, group) order already.  The host knows an upper bound
    // of the number of feeding calls; only when that exceeds one are the sort kernels enqueued at all (the device
    // then still decides from the exact count whether there is anything to re-order).
    const bool solo = c.acc_calls_pending <= 1;
    int cur = 0;
    cudaError_t e = cudaSuccess;
    if (!solo) {
        sb.ids = c.at<int32_t>(c.ws.q_id);
        sb.bits = bits_for(c.cfg.img_vocab);
        e = launch_collect_sort(c, sb, cap, d_n, st);
        if (e != cudaSuccess) return e;
        if (n_max > sort_small_max()) {                      // the queue may be longer than that launch can sort
            SortBatch batch = c.sort_batch();
            batch.n_jobs = 1;
            batch.job[0] = sb;
            batch.job[0].n_max = n_max;
            batch.job[0].n_dev = &state->sort_n;
            batch.name = "sort_ready";
            cur = sort_jobs(batch, st, &c.prof, &e);
            if (e != cudaSuccess) return e;
        }
    }
    if (cap >= c.ws.ready_cap) c.acc_calls_pending = 0;      // this collect cannot be refused: the queue will be empty
    const int64_t want = ceil_div(n_max, 8);
    KernelScope k(&c.prof, "collect_move", st);
    return launch_dependent(collect_move_kernel, dim3((unsigned)(want > resident ? resident : want)), dim3(256), 0, st, sb.keys[0], sb.vals[0],
                            sb.keys[cur], sb.vals[cur], c.at<int32_t>(c.ws.q_id), c.at<float>(c.ws.q_avg), c.cfg.dfv_dim, state, ids, seq, avg,
                            solo ? 1 : 0, cap, d_n);
}

}  // namespace gear
