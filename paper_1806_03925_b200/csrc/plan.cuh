// The accumulate call's plan over sorted Image IDs, one tile of positions at a time (steps 2-4 of accumulate.cu).
#pragma once

#include "common.cuh"
#include "internal.h"

namespace gear {

// Positions tile0 .. of the n sorted ones; a warp owns 32 * ITEMS consecutive positions of the tile, so that every load and
// store is coalesced and counts come from ballots.
//   key_at(i), perm_at(i)   sorted keys / permutation (key_at: any position of the array)
//   run_before(last_head)   last_head: where the tile's last run starts (-1: none starts in it); returns where the run that
//                           covers tile0 starts, if it starts before tile0
//   base(g, f, g0, f0)      g groups start in the tile, f of them complete; sets how many there are in the tiles before it
// s_warp: 2 * WARPS words of shared memory.  Every thread of the block must call this.
template <int ITEMS, int WARPS, typename KeyAt, typename PermAt, typename RunBefore, typename Base>
__device__ __forceinline__ void plan_tile(const PlanArgs& p, int n, int tile0, KeyAt key_at, PermAt perm_at, int* s_warp, RunBefore run_before, Base base) {
    const int lane = (int)lane_id(), warp = (int)(threadIdx.x >> 5);
    const int seg0 = tile0 + warp * 32 * ITEMS;
    const uint32_t lt = (1u << lane) - 1u;
    // rows the images already hold: all loads of the thread in flight at once
    int c0[ITEMS];
    int last_head = -1;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int i = seg0 + it * 32 + lane;
        const uint32_t key = i < n ? key_at(i) : p.vocab;
        c0[it] = key < p.vocab ? __ldg(p.cnt + key) : 0;
        const uint32_t heads = __ballot_sync(0xffffffffu, i < n && (i == 0 || key != key_at(i - 1)));
        if (heads) last_head = seg0 + it * 32 + 31 - __clz(heads);
    }
    if (lane == 0) s_warp[warp] = last_head;
    __syncthreads();
    // where the run that covers the warp's first position starts
    const int heads_of = lane < WARPS ? s_warp[lane] : -1;
    const int run0 = run_before(__reduce_max_sync(0xffffffffu, heads_of));
    int carry = max(run0, __reduce_max_sync(0xffffffffu, lane < warp ? heads_of : -1));
    __syncthreads();
    uint32_t head_bits = 0, full_bits = 0;
    int rank[ITEMS], groups = 0, full = 0;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int i = seg0 + it * 32 + lane;
        const uint32_t key = i < n ? key_at(i) : p.vocab;
        const uint32_t heads = __ballot_sync(0xffffffffu, i < n && (i == 0 || key != key_at(i - 1)));
        const uint32_t mine = heads & (lt | (1u << lane));
        const int start = mine ? seg0 + it * 32 + 31 - __clz(mine) : carry;
        if (heads) carry = seg0 + it * 32 + 31 - __clz(heads);
        rank[it] = i - start;
        bool head = false, complete = false;
        if (key < p.vocab) {
            const uint32_t x = (uint32_t)c0[it] + (uint32_t)rank[it], rem = x - p.div(x) * (uint32_t)p.div.M;
            head = rank[it] == 0 || rem == 0;
            if (head) {
                const int64_t last = (int64_t)i + (p.div.M - (int64_t)rem) - 1;          // the row that brings the count to M
                complete = last < n && key_at((int)last) == key;
            }
            const uint32_t after = i + 1 < n ? key_at(i + 1) : p.vocab;
            if (after >= p.vocab) p.state->n_valid = i + 1;                          // exactly one thread sees this
            if (after != key) p.run_end[start] = (uint32_t)(i + 1);
        }
        if (i == 0 && key >= p.vocab) p.state->n_valid = 0;                // no valid row at all
        head_bits |= (uint32_t)head << it;
        full_bits |= (uint32_t)complete << it;
        groups += __popc(__ballot_sync(0xffffffffu, head));
        full += __popc(__ballot_sync(0xffffffffu, complete));
    }
    if (lane == 0) { s_warp[warp] = groups; s_warp[WARPS + warp] = full; }
    __syncthreads();
    const int g_warp = lane < WARPS ? s_warp[lane] : 0, f_warp = lane < WARPS ? s_warp[WARPS + lane] : 0;
    uint32_t g0, f0;
    base(__reduce_add_sync(0xffffffffu, (uint32_t)g_warp), __reduce_add_sync(0xffffffffu, (uint32_t)f_warp), g0, f0);
    // where the gradient row of every sorted position lives and what it is scaled by (one 8-byte record), where the call names
    // either; every level of the chain is requested for all positions at once.  A source row below zero (an occurrence that no page
    // view of a malformed batch covers): row 0 times zero.
    if (p.src_row || p.scale) {
        int src[ITEMS];
        float scale[ITEMS];
        uint32_t live = 0;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const int i = seg0 + it * 32 + lane;
            const bool on = i < n && key_at(i) < p.vocab;                            // a row without a valid image has no record
            live |= (uint32_t)on << it;
            src[it] = on ? (int)perm_at(i) : -1;
        }
        if (p.src_row)
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) if (src[it] >= 0) src[it] = __ldg(p.src_row + src[it]);
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) scale[it] = src[it] < 0 ? 0.f : p.scale ? __ldg(p.scale + src[it]) : 1.f;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it)
            if ((live >> it) & 1u) p.pmeta[seg0 + it * 32 + lane] = make_int2(max(src[it], 0), __float_as_int(scale[it]));
    }
    uint32_t gi = g0 + __reduce_add_sync(0xffffffffu, (uint32_t)(lane < warp ? g_warp : 0));
    uint32_t ci = f0 + __reduce_add_sync(0xffffffffu, (uint32_t)(lane < warp ? f_warp : 0));
    const int64_t q_base = p.state->q_count;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int i = seg0 + it * 32 + lane;
        const bool head = (head_bits >> it) & 1u, complete = (full_bits >> it) & 1u;
        const uint32_t hb = __ballot_sync(0xffffffffu, head), fb = __ballot_sync(0xffffffffu, complete);
        const uint32_t key = i < n ? key_at(i) : p.vocab;
        if (key < p.vocab) {
            const uint32_t g = gi + __popc(hb & lt);
            // the reduce pass hands out spans of 2^span sorted positions: index of the first group that starts in each
            if ((i & ((1 << p.span) - 1)) == 0) p.blk_first[i >> p.span] = g;
            if (head) {
                // one 16-byte record per group: start position (top bit: first group of its image in this call), image ID,
                // ready-queue slot (-1: the group stays open), and for the image's first group the rows the image already held,
                // for a later one its number among the groups of the image that this call completes
                const bool first = rank[it] == 0;
                p.grp_rec[g] = make_uint4((uint32_t)i | (first ? 0x80000000u : 0u), key,
                                          (uint32_t)(complete ? (int32_t)(q_base + ci + __popc(fb & lt)) : -1),
                                          first ? (uint32_t)c0[it] : p.div((uint32_t)c0[it] + (uint32_t)rank[it]));
            }
        }
        gi += __popc(hb);
        ci += __popc(fb);
    }
}

}  // namespace gear
