// Shared device helpers and the internal host-side declarations of libgear.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cfloat>
#include <stdint.h>

#include <atomic>
#include <utility>
#include <vector>

#include "../../include/gear.h"
#include "enqueue.cuh"

namespace gear {

// ---------------------------------------------------------------- device state
// Lives at the start of the workspace.  Counters are device-resident so that no
// call has to synchronise to learn a size produced by an earlier kernel.
struct DevState {
    int32_t status;        // GEAR_DEV_* bits, sticky
    int32_t tc_error;      // non-zero: a bounded wait of the tensor-core head gave up (code of the wait)
    int64_t q_count;       // averages waiting in the ready queue
    int64_t n_valid;       // accumulate: rows with an in-range ID (sorted prefix length)
    int64_t direct_done;   // accumulate + collect as one call: 1 while the hand-over pass that follows has nothing to do
                           // (the reduce pass wrote the averages straight into the caller's lists)
    int64_t plan_base;     // accumulate: length of the ready queue that the plan goes by
    uint32_t scan_next;    // expiry scan: which set of section counts the next mark pass adds to (written by the write pass)
    uint32_t scan_set;     // ... and which one the last mark pass added to (written by that pass)
    int64_t collect_n;     // collect_ready: entries moved by the running call
    unsigned int barrier_arrived;      // the cooperative sort's grid barrier: arrivals; blocks that have left the launch
    unsigned int barrier_left;         // (both zero between launches)
    unsigned int n_copies; // order-free store: records of repeated averages still to be written
    unsigned int pad32;                // blocks of a solo collect_move_kernel that have finished (wraps to 0)
    int64_t q_calls;       // accumulate calls that added to the ready queue since the last collect
    int64_t sort_n;        // collect_ready: entries the queue sort has to order (0: the queue is already in order)
    int64_t pad[5];
};
static_assert(sizeof(DevState) == 128, "DevState layout");

// ---------------------------------------------------------------- small helpers
__host__ __device__ inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// SMs of the current device (host side; 148 on a B200)
inline int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 148;
    }
    return n;
}

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ uint32_t warp_inclusive_scan(uint32_t v) {
    const unsigned lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= (unsigned)o) v += t;
    }
    return v;
}

// Exclusive scan over the threads of a block (blockDim.x a multiple of 32, <= 1024).
// `scratch` needs 33 words of shared memory.  Returns the exclusive prefix; *total gets the block sum.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* scratch, uint32_t* total) {
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    uint32_t inc = warp_inclusive_scan(v);
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nwarp ? scratch[lane] : 0u;
        uint32_t winc = warp_inclusive_scan(w);
        scratch[lane] = winc - w;
        if (lane == 31) scratch[32] = winc;
    }
    __syncthreads();
    uint32_t res = scratch[warp] + inc - v;
    if (total) *total = scratch[32];
    __syncthreads();
    return res;
}

__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

__device__ __forceinline__ float4 ld_f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st_f4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

// 128-bit load that does not allocate in L1 (streamed data read once)
__device__ __forceinline__ float4 ld_stream_f4(const float* p) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

// An fp32 matrix held as three bf16 matrices `stride` elements apart, whose sum it is (head_tc3.cu)
struct Planes { __nv_bfloat16* p; int64_t stride; };

// two fp32 values as three packed pairs of bf16 (each part rounded to nearest; the three parts of a value sum to it).  Values that
// round to infinity come out as NaN (the second part is inf - inf): see split3_pair_any.
__device__ __forceinline__ void split3_rest(float rx, float ry, uint32_t& p1, uint32_t& p2) {
    const __nv_bfloat162 h1 = __floats2bfloat162_rn(rx, ry);
    p1 = *reinterpret_cast<const uint32_t*>(&h1);
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(rx - __uint_as_float(p1 << 16), ry - __uint_as_float(p1 & 0xffff0000u));
    p2 = *reinterpret_cast<const uint32_t*>(&h2);
}
__device__ __forceinline__ void split3_pair(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(x, y);
    p0 = *reinterpret_cast<const uint32_t*>(&h0);
    split3_rest(x - __uint_as_float(p0 << 16), y - __uint_as_float(p0 & 0xffff0000u), p1, p2);
}
// The same for activations (x, y >= 0): one that rounds to infinity comes out as infinity.  (A branch instead: the forward products
// of 32 k views 69.7 -> 72.7 us; like this 70.3.)
__device__ __forceinline__ void split3_pair_relu(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(x, y);
    p0 = *reinterpret_cast<const uint32_t*>(&h0);
    // rests of values in range are below 2^120; those of inf - inf and x - inf become a finite number, which infinity swallows
    split3_rest(fmaxf(x - __uint_as_float(p0 << 16), -0x1p120f), fmaxf(y - __uint_as_float(p0 & 0xffff0000u), -0x1p120f), p1, p2);
}
// The same for any value: one that rounds to infinity has its leading part cut off instead; an infinity or NaN is its leading
// part alone.
__device__ __forceinline__ void split3_pair_any(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(x, y);
    p0 = *reinterpret_cast<const uint32_t*>(&h0);
    float rx = x - __uint_as_float(p0 << 16), ry = y - __uint_as_float(p0 & 0xffff0000u);
    if (!(fabsf(rx) + fabsf(ry) <= FLT_MAX)) {               // the rests of values in range are below 2^120
        const float hx = fabsf(x) <= FLT_MAX ? __uint_as_float(__float_as_uint(x) & 0xffff0000u) : x;
        const float hy = fabsf(y) <= FLT_MAX ? __uint_as_float(__float_as_uint(y) & 0xffff0000u) : y;
        const __nv_bfloat162 cut = __floats2bfloat162_rn(hx, hy);
        p0 = *reinterpret_cast<const uint32_t*>(&cut);
        rx = fabsf(x) <= FLT_MAX ? x - hx : 0.f; ry = fabsf(y) <= FLT_MAX ? y - hy : 0.f;
    }
    split3_rest(rx, ry, p1, p2);
}

// vector reduction: *p += v without a return value (sm_90+)
__device__ __forceinline__ void red_add_f4(float* p, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};"
                 :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// L2 eviction priorities: data that is read again soon is kept (evict_last), data touched once is let go first
// (evict_first), so that a streamed table does not push a reused matrix out of the L2.
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void st_f4_hint(float* p, float4 v, uint64_t policy) {
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1,%2,%3,%4}, %5;"
                 :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "l"(policy) : "memory");
}

// 16-byte asynchronous copy global -> shared; src_bytes = 0 reads nothing and fills the 16 bytes with zeros
__device__ __forceinline__ void cp_async_16(uint32_t smem_dst, const void* gsrc, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" :: "r"(smem_dst), "l"(gsrc), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory");
}

// ---------------------------------------------------------------- programmatic dependent launch
// The step is a chain of two dozen short kernels on one stream.  Launched this way, the blocks of a kernel may be
// set up on SMs that the previous kernel in the stream has already left while its last blocks still run; every
// such kernel calls wait_for_predecessor() before it touches memory, which returns once the previous kernel has
// completed and its writes are visible.  That takes the launch latency out of the gaps between kernels.  Every
// block of such a kernel must make the call, first thing, or the chain of completions would break.
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The next kernel in the stream may be set up beside this one from here on.  It still waits for this one to complete, and, since this
// is called behind wait_for_predecessor(), for all before it.  For launches that leave a third of the SMs to it: elsewhere, blocks
// which only wait keep the kernels of other streams out.  Steps in fp32 with this line at 128 blocks / at 98 / at 74 (us): 4096 views,
// 256 + 64 units 61.8 / 59.6 / 59.6, 256 + 200 units 80.4 / 76.2 / 76.2; 1024 views, 64 to 256 units 33.3 / 33.0 / 33.0; 780 views,
// 256 + 64 units 39.2 / 39.1 / 40.7, 128 + 128 units 37.1 / 35.4 / 36.1; 256 views no difference.
constexpr unsigned FEW_BLOCKS = 98;
__device__ __forceinline__ void let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_as(Op::Attr attr, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    OpList local;
    OpList& l = t_ops ? *t_ops : local;
    l.kernel(reinterpret_cast<const void*>(kernel), grid, block, smem, attr, st);
    auto push = [&l](const auto& v) { l.arg(&v, sizeof(v)); return 0; };
    (push(static_cast<const KArgs&>(KArgs(args))), ...);
    return t_ops ? cudaSuccess : launch_list_kernel(l.ops.back(), l, st);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    return launch_as(Op::DEPENDENT, kernel, grid, block, smem, st, std::forward<Args>(args)...);
}

// Lets a kernel take `bytes` of dynamic shared memory beside its static one.  The attribute belongs to the kernel on one device: it is
// asked for once on each, again where that failed.
template <auto Kernel> inline cudaError_t allow_smem(int bytes) {
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
    if (e != cudaSuccess || (done.load(std::memory_order_relaxed) & bit)) return e;
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

// ---------------------------------------------------------------- launch accounting / per-kernel timing
// Every kernel launch of the library goes through a KernelScope: it counts the launch and, when profiling is on, has it
// bracketed with a pair of CUDA events on its stream (read back by gear_profile_read): by the player where the
// launch is being written down, by the scope itself otherwise.
struct Profiler {
    struct Rec { const char* name; cudaEvent_t start, stop; };
    bool on = false;
    bool keep_streams = false;     // timeline mode: events are recorded but the library keeps its side stream
    int64_t launches = 0;
    std::vector<Rec> recs;
    std::vector<cudaEvent_t> pool;
    cudaEvent_t get() {
        if (!pool.empty()) { cudaEvent_t e = pool.back(); pool.pop_back(); return e; }
        cudaEvent_t e = nullptr;
        cudaEventCreate(&e);
        return e;
    }
    void clear() {
        for (auto& r : recs) { pool.push_back(r.start); pool.push_back(r.stop); }
        recs.clear();
    }
    ~Profiler() {
        clear();
        for (auto e : pool) cudaEventDestroy(e);
    }
};

struct KernelScope {
    Profiler* p; cudaStream_t st; cudaEvent_t stop = nullptr;
    KernelScope(Profiler* prof, const char* name, cudaStream_t s) : p(prof), st(s) {
        if (!p) return;
        ++p->launches;
        if (t_ops) t_ops->next_name = name;
        else if (p->on) {
            Profiler::Rec r{name, p->get(), p->get()};
            stop = r.stop;
            cudaEventRecord(r.start, st);
            p->recs.push_back(r);
        }
    }
    ~KernelScope() { if (stop) cudaEventRecord(stop, st); }
};

// Sorted positions per unit of work (span) of the accumulate's reduce pass: 16, or as few as 2 while longer spans would leave more
// than half of the warps idle (12 k rows in spans of 16 kept 768 of 3552 warps busy, each with a serial chain of 16 rows; in spans of
// 2 a warp went through the latencies of a span's start twice: step of 4096 views 52.1 us, spans of 4: 50.6, of 8: 51.1).  Against
// spans that leave no warp idle, stores of 5000 to 56000 rows of 512 bytes to 4 KB: 0 to 7 % shorter; the one range that is longer
// is 40 to 50 thousand rows of 1 KB and more with uniform IDs, 1 to 4 % (Zipf IDs there: 0 to 6 % shorter).
// The workspace holds one word per span.
constexpr int ACC_SPAN = 16;
constexpr int64_t ACC_WARPS = 3552;        // warps of a full reduce grid: 148 SMs x 3 blocks x 8
inline int acc_span_log2(int64_t n) {
    int s = 4;
    while (s > 1 && (n >> s) < ACC_WARPS / 2) --s;
    return s;
}
// words of the span table for any n up to n_max
inline int64_t acc_max_spans(int64_t n_max) {
    const int64_t small = n_max < (ACC_WARPS << 5) ? n_max : (ACC_WARPS << 5);
    const int64_t a = ceil_div(n_max, ACC_SPAN), b = ceil_div(small, 2);
    return (a > b ? a : b) + 2;
}

// x / M for x < M + 2^30: a multiplication and a shift (division by an invariant integer, Granlund and Montgomery, PLDI 1994:
// exact for x < 2^31 with the factor ceil(2^(31 + s) / M), s = ceil(log2 M)); from M = 2^30 on the quotient is 0 or 1.
struct DivM {
    int M; uint32_t factor; int shift;
    __host__ __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
        return M >= (1 << 30) ? (uint32_t)(x >= (uint32_t)M) : (uint32_t)(((uint64_t)x * factor) >> shift);
    }
};
inline DivM make_div(int M) {
    int s = 0;
    while (s < 31 && (1ll << s) < M) ++s;
    return DivM{M, (uint32_t)(((1ull << (31 + s)) + M - 1) / M), 31 + s};
}

// ---------------------------------------------------------------- radix sort / scans (prims.cu)
constexpr int RS_THREADS = 512;
constexpr int RS_RADIX_BITS = 9;
constexpr int RS_BUCKETS = 1 << RS_RADIX_BITS;
constexpr int RS_MAX_BLOCKS = 512;        // of the sort's grid (two per SM)

// most blocks a job can get: one per tile of RS_THREADS * 4 entries
inline int64_t sort_max_blocks(int64_t n_max) {
    const int64_t tiles = ceil_div(n_max, RS_THREADS * 4);
    return tiles < 1 ? 1 : tiles < RS_MAX_BLOCKS ? tiles : RS_MAX_BLOCKS;
}

// One array to sort: (key, value) pairs ordered by the low `bits` bits of the key, equal keys in input order.
struct SortJob {
    const int32_t* ids;     // if set, pass 0 reads these: key = id if 0 <= id < sentinel, else sentinel
    uint32_t sentinel;      // key of out-of-range IDs (sorts last when bits covers it)
    int32_t* status;        // device status word that gets GEAR_DEV_BAD_ID when a sentinel key is met (may be null)
    uint32_t* keys[2];      // without ids the input keys are keys[0]
    uint32_t* vals[2];      // with identity_vals the value of element i is i, else vals[0][i]
    uint32_t* hist;         // [RS_BUCKETS][blocks of the job] digit counts of the blocks' chunks
    uint32_t* tot;          // [RS_BUCKETS] digit counts of the array
    int64_t n_max;          // element count (or its upper bound when n_dev is given)
    const int64_t* n_dev;   // optional device-resident count, capped at n_max
    int bits;
    int identity_vals;
    const int32_t* src;     // with identity_vals: the value of element i is src[i] instead, if set
    int width, block0, n_blocks;     // filled in by sort_jobs
};

struct SortBatch {
    SortJob job[3];
    int n_jobs;
    const char* name;                 // host only: the name the launch is timed under
    int passes;                       // filled in by sort_jobs
    unsigned int* barrier;            // two device words, zero before and after every launch: arrivals, blocks that have left
    int32_t* err;                     // device word that receives a non-zero code when a grid barrier gives up
};

// Sorts every job of the batch in one cooperative launch.  Returns the index (0 or 1) of the keys/vals
// buffer pair that holds the sorted result of every job.
int sort_jobs(SortBatch& batch, cudaStream_t st, Profiler* prof, cudaError_t* err_out);

inline int bits_for(int64_t max_key_inclusive) {
    int b = 1;
    while (b < 32 && (int64_t(1) << b) <= max_key_inclusive) ++b;
    return b;
}

}  // namespace gear
