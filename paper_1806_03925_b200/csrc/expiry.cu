// Inference-expired time (Section 1, second point; Section 3: the workers drop expired inference
// results continuously): list every image whose cached DFV is older than the expiry time.
//
// Two launches, none waits on another block:
//   mark   streams the int64 timestamp table once (the only HBM-sized traffic: 8 bytes per image),
//          evaluates now - ts >= expire, packs the predicate 32 entries to a word with a warp ballot and counts per
//          2048-entry tile and, with one atomic per tile, per section of 64 tiles;
//   write  every block adds up the sections and tiles before its own, checks the caller's capacity against the total,
//          re-reads only the bitmap (1 bit per image), ranks the set bits with popc + block scan and writes the ascending ID
//          list; listed entries are restamped on request.
// (A scan kernel between the two took 7 us for 20 M images, and one kernel that keeps the bits in shared memory and waits for
// the counts of the blocks before it read the table at 2.8 TB/s instead of 5.7: too few loads in flight.)
#include "common.cuh"
#include "internal.h"

namespace gear {

constexpr int EXP_THREADS = 256;
constexpr int EXP_MARK_ITEMS = EXP_MARK_TILE / EXP_THREADS;
static_assert(EXP_TILE == EXP_THREADS * 32, "one bitmap word per thread in the write pass");
static_assert(EXP_MARK_TILE % (EXP_THREADS * 1) == 0 && EXP_TILE % EXP_MARK_TILE == 0, "mark tiles nest in write tiles");

// Per-tile counts, then the sections' counts twice over: a scan adds to one set and clears the other for the next scan.  Which
// set it is stands in the device state, so that a scan that is replayed, or was written down and never ran, leaves nothing
// behind: the mark pass reads scan_next and notes it in scan_set, the write pass reads that and turns scan_next over.
struct ExpiryCounts {
    uint32_t* tile; uint32_t* section;
    int64_t n_tiles, n_sections;
};
constexpr int EXP_SECTION = 64;           // mark tiles per section

// One block per EXP_MARK_TILE timestamps.  All of a thread's loads are issued before the first ballot, so a
// block keeps its whole 16 KB tile in flight; the small tiles leave the balancing to the block scheduler.
__global__ void __launch_bounds__(EXP_THREADS)
expiry_mark_kernel(const int64_t* __restrict__ ts, int64_t vocab, int64_t now, int64_t expire,
                   uint32_t* __restrict__ bits, const ExpiryCounts cnt, DevState* __restrict__ state) {
    wait_for_predecessor();
    const uint32_t set = state->scan_next & 1u;
    __shared__ uint32_t warp_cnt[EXP_THREADS / 32];
    const int64_t tile0 = (int64_t)blockIdx.x * EXP_MARK_TILE;
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    int64_t t[EXP_MARK_ITEMS];
#pragma unroll
    for (int it = 0; it < EXP_MARK_ITEMS; ++it) {
        const int64_t i = tile0 + (int64_t)it * EXP_THREADS + threadIdx.x;
        t[it] = i < vocab ? __ldcs(reinterpret_cast<const long long*>(ts) + i) : 0;
    }
    uint32_t count = 0;
#pragma unroll
    for (int it = 0; it < EXP_MARK_ITEMS; ++it) {
        const int64_t i = tile0 + (int64_t)it * EXP_THREADS + threadIdx.x;
        const bool expired = i < vocab && now - t[it] >= expire;
        const uint32_t word = __ballot_sync(0xffffffffu, expired);
        if (lane == 0) {
            const int64_t w = (tile0 + (int64_t)it * EXP_THREADS) / 32 + warp;
            if (w * 32 < vocab) bits[w] = word;
            count += __popc(word);
        }
    }
    if (lane == 0) warp_cnt[warp] = count;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t total = 0;
#pragma unroll
        for (int w = 0; w < EXP_THREADS / 32; ++w) total += warp_cnt[w];
        cnt.tile[blockIdx.x] = total;
        if (total) atomicAdd(cnt.section + set * cnt.n_sections + blockIdx.x / EXP_SECTION, total);
        if (blockIdx.x % EXP_SECTION == 0) cnt.section[(set ^ 1u) * cnt.n_sections + blockIdx.x / EXP_SECTION] = 0u;
        if (blockIdx.x == 0) state->scan_set = set;
    }
}

// One block per EXP_TILE entries: re-reads the bitmap only.  Every block compares the total with the
// caller's capacity itself; block 0 reports the count and raises the status bit.
__global__ void __launch_bounds__(EXP_THREADS)
expiry_write_kernel(const uint32_t* __restrict__ bits, int64_t vocab, const ExpiryCounts cnt, int64_t cap,
                    int64_t* __restrict__ d_n, DevState* __restrict__ state, int64_t now, int restamp, int64_t* __restrict__ ts,
                    int32_t* __restrict__ ids) {
    wait_for_predecessor();
    __shared__ uint32_t scratch[33];
    const int64_t w = (int64_t)blockIdx.x * EXP_THREADS + threadIdx.x;
    uint32_t word = (w * 32 < vocab) ? bits[w] : 0u;
    const int64_t my_tile = (int64_t)blockIdx.x * (EXP_TILE / EXP_MARK_TILE), my_section = my_tile / EXP_SECTION;
    const uint32_t set = state->scan_set & 1u;
    uint32_t before = 0, after = 0;                         // this thread's share
    for (int64_t s = threadIdx.x; s < cnt.n_sections; s += EXP_THREADS) {
        const uint32_t v0 = cnt.section[s], v1 = cnt.section[cnt.n_sections + s], v = set ? v1 : v0;     // (no load waits for `set`)
        if (s < my_section) before += v; else after += v;
    }
    const int64_t t = my_section * EXP_SECTION + threadIdx.x;
    if (threadIdx.x < EXP_SECTION && t < my_tile) { const uint32_t v = cnt.tile[t]; before += v; after -= v; }
    uint32_t n_before, n_after;
    block_exclusive_scan(before, scratch, &n_before);
    block_exclusive_scan(after, scratch, &n_after);
    const int64_t total = (int64_t)(n_before + n_after);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state->scan_next = set ^ 1u;                        // the mark pass behind this one finds that set cleared
        if (d_n) *d_n = total;
        if (total > cap) atomicOr(&state->status, GEAR_DEV_OUT_CAPACITY);
    }
    if (total > cap) return;                                // capacity too small: nothing listed, nothing restamped
    int64_t out = (int64_t)n_before + block_exclusive_scan(__popc(word), scratch, nullptr);
    while (word) {
        const int bit = __ffs(word) - 1;
        word &= word - 1;
        const int64_t id = w * 32 + bit;
        ids[out++] = (int32_t)id;
        if (restamp) ts[id] = now;
    }
}

// The two launches of one scan over scratch (bits, counts, state).  prof may be null.
static cudaError_t enqueue_expiry_scan(int64_t* ts, int64_t vocab, int64_t expire, int64_t now, int restamp,
                                       int32_t* ids, int64_t cap, int64_t* d_n, uint32_t* bits, const ExpiryCounts& cnt,
                                       DevState* state, Profiler* prof, cudaStream_t st) {
    const int64_t n_write = ceil_div(vocab, EXP_TILE);
    cudaError_t e;
    { KernelScope k(prof, "expiry_mark", st);
    e = launch_dependent(expiry_mark_kernel, dim3((unsigned)cnt.n_tiles), dim3(EXP_THREADS), 0, st, ts, vocab, now, expire, bits, cnt, state); }
    if (e != cudaSuccess) return e;
    KernelScope k(prof, "expiry_write", st);
    return launch_dependent(expiry_write_kernel, dim3((unsigned)n_write), dim3(EXP_THREADS), 0, st, bits, vocab, cnt, cap, d_n, state, now,
                            restamp, ts, ids);
}

// counts: [n_tiles] tile counts, then two sets of section counts; the set that scan_next names is zero before the scan
static ExpiryCounts expiry_counts(uint32_t* counts, int64_t vocab) {
    const int64_t n = ceil_div(vocab, EXP_MARK_TILE);
    return ExpiryCounts{counts, counts + n, n, ceil_div(n, EXP_SECTION)};
}

cudaError_t launch_collect_expired(const gear_ctx_impl& c, int64_t now, int restamp, int32_t* ids, int64_t cap,
                                   int64_t* d_n, cudaStream_t st) {
    const ExpiryCounts cnt = expiry_counts(c.at<uint32_t>(c.ws.exp_cnt), c.cfg.img_vocab);
    if (c.scan_cut_off) {                                   // a mark pass may have run whose write pass did not
        const cudaError_t e = enqueue_memset(cnt.section, 2 * sizeof(uint32_t) * (size_t)cnt.n_sections, st);
        if (e != cudaSuccess) return e;
        c.scan_cut_off = false;
    }
    return enqueue_expiry_scan(c.buf.dfv_ts, c.cfg.img_vocab, c.cfg.expire, now, restamp, ids, cap, d_n, c.at<uint32_t>(c.ws.exp_bits),
                               cnt, c.state(), &c.prof, st);
}

}  // namespace gear

// ---------------------------------------------------------------------------------------------------
// gear_collect_expired_static: the same scan for callers that cannot allocate device memory.
//
// Some hosts of this library run it where cudaMalloc is off limits: inside a serving process whose memory
// pool was carved up at start-up and is policed, from a plug-in that is handed buffers but no allocator,
// or on a path that must not touch the allocator because an allocation may synchronise the device.  Such a
// caller cannot provide the workspace a gear_ctx needs.  This entry point therefore keeps the scan's
// scratch (expired bitmap, per-tile counts, a small state block) in a fixed array that is part of the
// library image: every GPU that loads libgear holds GEAR_STATIC_EXPIRY_SCRATCH_BYTES of it until the
// process exits.  The price is a bound on the table size and one shared scratch per device.
// ---------------------------------------------------------------------------------------------------
#include <mutex>
#include <new>

namespace gear {

constexpr int64_t STATIC_MAX_VOCAB = GEAR_STATIC_EXPIRY_MAX_VOCAB;
constexpr size_t STATIC_STATE_BYTES = 256;
constexpr size_t STATIC_BITS_BYTES = (size_t)(STATIC_MAX_VOCAB / 32) * 4;
constexpr size_t STATIC_CNT_BYTES = ((size_t)(STATIC_MAX_VOCAB / EXP_MARK_TILE) + 1) * 8;     // tile and section counts
constexpr size_t STATIC_SCRATCH_BYTES = STATIC_STATE_BYTES + STATIC_BITS_BYTES + ((STATIC_CNT_BYTES + 255) / 256) * 256;
static_assert(sizeof(DevState) <= STATIC_STATE_BYTES, "state block");
static_assert(STATIC_SCRATCH_BYTES == GEAR_STATIC_EXPIRY_SCRATCH_BYTES, "the header states the size of the array");

// In host code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_static_expiry_scratch[STATIC_SCRATCH_BYTES];

constexpr int STATIC_MAX_DEVICES = 64;
static std::mutex g_static_mutex;
static unsigned char* g_static_ptr[STATIC_MAX_DEVICES];     // device address of the scratch, per device ordinal

// Device address of the scratch on the current device (looked up once per device).
static cudaError_t static_scratch(unsigned char** out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= STATIC_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_expiry_scratch);
        if (e != cudaSuccess) return e;
        g_static_ptr[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_static_ptr[dev];
    return cudaSuccess;
}

}  // namespace gear

extern "C" int gear_collect_expired_static(int64_t* dfv_ts, int64_t img_vocab, int64_t expire, int64_t now, int restamp,
                                           int32_t* ids, int64_t cap, int64_t* d_n, int64_t* h_n, void* stream) {
    using namespace gear;
    if (!dfv_ts || img_vocab < 1 || expire < 0 || cap < 0 || (cap > 0 && !ids)) return GEAR_ERR_ARG;
    if (img_vocab > STATIC_MAX_VOCAB) return GEAR_ERR_CAPACITY;      // the fixed scratch cannot hold the bitmap
    unsigned char* base = nullptr;
    if (static_scratch(&base) != cudaSuccess) return GEAR_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    DevState* state = reinterpret_cast<DevState*>(base);
    uint32_t* bits = reinterpret_cast<uint32_t*>(base + STATIC_STATE_BYTES);
    uint32_t* counts = reinterpret_cast<uint32_t*>(base + STATIC_STATE_BYTES + STATIC_BITS_BYTES);

    // the array keeps what the previous call left: the state block and the section counts have to start from zero, the
    // bitmap words and tile counts of this table size are all rewritten by the mark pass
    const ExpiryCounts cnt = expiry_counts(counts, img_vocab);
    if (enqueue_memset(state, STATIC_STATE_BYTES, st) != cudaSuccess) return GEAR_ERR_CUDA;
    if (enqueue_memset(cnt.section, sizeof(uint32_t) * (size_t)cnt.n_sections, st) != cudaSuccess) return GEAR_ERR_CUDA;
    int64_t* d_cnt = d_n ? d_n : &state->pad[1];
    try {                                            // (a launch is written down in host memory, which may run out)
        if (enqueue_expiry_scan(dfv_ts, img_vocab, expire, now, restamp, ids, cap, d_cnt, bits, cnt, state, nullptr, st) != cudaSuccess)
            return GEAR_ERR_CUDA;
    } catch (const std::bad_alloc&) { return GEAR_ERR_CUDA; }
    if (h_n) {
        if (cudaMemcpyAsync(h_n, d_cnt, sizeof(int64_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return GEAR_ERR_CUDA;
        if (*h_n > cap) return GEAR_ERR_CAPACITY;
    }
    return GEAR_OK;
}
