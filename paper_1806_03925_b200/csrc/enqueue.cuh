// How the calls of the library reach the GPU.
//
// A call first writes down what it wants enqueued -- kernels with their arguments, memsets, copies, events between
// streams -- in an OpList, and the list is then played.  Played directly, every entry is one runtime call (about 2 us each:
// a step of 20 kernels on three streams cost the host 80 us, more than the GPU needs for a few thousand views).  A list whose
// shape (which kernels, on which streams, in which order) has come up GRAPH_AFTER times, in a row or not, is captured into a
// CUDA graph once; from then on a call compares its entries with those of the call before, sets the parameters of the
// nodes that differ (pointers, sizes, grids of a new batch) and launches the graph with one call.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <vector>

#include "../../include/gear.h"

namespace gear {

struct Profiler;

struct Op {
    enum Kind : uint8_t { KERNEL, MEMSET, COPY, RECORD, WAIT };
    enum Attr : uint8_t { PLAIN, DEPENDENT, COOPERATIVE };       // DEPENDENT: programmatic stream serialisation
    Kind kind;
    Attr attr;
    uint8_t role;                  // which of the list's streams
    const void* func;              // KERNEL; MEMSET / COPY: source (or null)
    void* ptr;                     // MEMSET / COPY: destination; RECORD / WAIT: the event
    size_t bytes;                  // KERNEL: dynamic shared memory; MEMSET / COPY: length
    dim3 grid, block;
    uint32_t arg0, n_args, blob0, blob1;
    const char* name;              // KERNEL: what its time is booked under
    bool same_shape(const Op& o) const {
        return kind == o.kind && attr == o.attr && role == o.role && n_args == o.n_args && (kind == KERNEL ? func == o.func : true) &&
               ((kind != RECORD && kind != WAIT) || ptr == o.ptr);
    }
};

class OpList {
public:
    static constexpr int MAX_STREAMS = 3 * GEAR_MAX_LOCAL_RANKS + 1;
    cudaStream_t streams[MAX_STREAMS] = {};      // [0] the caller's stream
    int n_streams = 0;
    int n_kernels = 0;
    std::vector<Op> ops;
    std::vector<uint8_t> blob;                   // kernel arguments
    std::vector<uint32_t> arg_off;               // where each argument starts in the blob
    const char* next_name = nullptr;

    void clear() { ops.clear(); blob.clear(); arg_off.clear(); n_streams = 0; n_kernels = 0; next_name = nullptr; }
    Op& add(Op::Kind kind, cudaStream_t st) {
        ops.emplace_back();
        Op& o = ops.back();
        memset(static_cast<void*>(&o), 0, sizeof(o));
        o.kind = kind;
        int r = 0;
        while (r < n_streams && streams[r] != st) ++r;
        if (r == n_streams) { streams[r] = st; ++n_streams; }
        o.role = (uint8_t)r;
        return o;
    }
    void kernel(const void* func, dim3 grid, dim3 block, size_t smem, Op::Attr attr, cudaStream_t st) {
        Op& o = add(Op::KERNEL, st);
        o.func = func; o.grid = grid; o.block = block; o.bytes = smem; o.attr = attr;
        o.arg0 = (uint32_t)arg_off.size(); o.blob0 = o.blob1 = (uint32_t)blob.size();
        o.name = next_name ? next_name : "kernel";
        ++n_kernels;
    }
    void arg(const void* p, size_t bytes) {
        const size_t at = (blob.size() + 15) & ~(size_t)15;
        blob.resize(at + bytes);
        memcpy(blob.data() + at, p, bytes);
        arg_off.push_back((uint32_t)at);
        Op& o = ops.back();
        ++o.n_args; o.blob1 = (uint32_t)blob.size();
    }
};

// The list that the calling thread is filling (null: launches go straight to their stream).
extern thread_local OpList* t_ops;

cudaError_t enqueue_memset(void* p, size_t bytes, cudaStream_t st);                       // zeros
cudaError_t enqueue_copy(void* dst, const void* src, size_t bytes, cudaStream_t st);      // cudaMemcpyDefault
cudaError_t enqueue_record(cudaEvent_t ev, cudaStream_t st);
cudaError_t enqueue_wait(cudaStream_t st, cudaEvent_t ev);
cudaError_t launch_list_kernel(const Op& o, OpList& l, cudaStream_t st);

// Plays lists for one ctx and keeps its graphs (at most MAX_GRAPHS shapes; given back with the ctx).
class Player {
public:
    ~Player();
    // Enqueues what `l` holds; the list's contents are undefined afterwards.
    cudaError_t play(OpList& l, Profiler* prof);
    OpList list;                                 // scratch of the call that is being written down

private:
    static constexpr int MAX_GRAPHS = 6;
    static constexpr int GRAPH_AFTER = 3;        // a graph costs a few direct calls to make: not for a shape seen once or twice
    static constexpr int MIN_KERNELS = 3;        // shorter lists gain nothing
    struct Entry {
        OpList last;                             // what the graph's nodes hold (or the shape seen, while exec is null)
        std::vector<cudaGraphNode_t> node;       // per op; null for events
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        int seen = 0;
        uint64_t used = 0;
    };
    Entry entry_[MAX_GRAPHS];
    uint64_t clock_ = 0;
    cudaStream_t capture_ = nullptr;

    static void drop(Entry& e);
    cudaError_t direct(OpList& l, Profiler* prof);
    bool build(Entry& e, OpList& l);
    bool update(Entry& e, OpList& l);
};

// Fills the player's list for the duration of a call.
class Recording {
public:
    explicit Recording(Player& p, cudaStream_t st) : p_(p), outer_(t_ops) {
        if (outer_) return;                      // a call inside a call adds to the outer one's list
        p_.list.clear();
        p_.list.streams[0] = st; p_.list.n_streams = 1;
        t_ops = &p_.list;
    }
    ~Recording() { if (!outer_) t_ops = nullptr; }
    // Ends the recording and enqueues it (nothing to do in an inner call).
    cudaError_t play(Profiler* prof) {
        if (outer_) return cudaSuccess;
        t_ops = nullptr;
        return p_.play(p_.list, prof);
    }
private:
    Player& p_;
    OpList* outer_;
};

}  // namespace gear
