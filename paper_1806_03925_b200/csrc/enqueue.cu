// Direct and graph play of what a call wrote down (enqueue.cuh).
#include "enqueue.cuh"
#include "common.cuh"

namespace gear {

thread_local OpList* t_ops = nullptr;

cudaError_t enqueue_memset(void* p, size_t bytes, cudaStream_t st) {
    if (!t_ops) return cudaMemsetAsync(p, 0, bytes, st);
    Op& o = t_ops->add(Op::MEMSET, st);
    o.ptr = p; o.bytes = bytes;
    return cudaSuccess;
}
cudaError_t enqueue_copy(void* dst, const void* src, size_t bytes, cudaStream_t st) {
    if (!t_ops) return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, st);
    Op& o = t_ops->add(Op::COPY, st);
    o.ptr = dst; o.func = src; o.bytes = bytes;
    return cudaSuccess;
}
cudaError_t enqueue_record(cudaEvent_t ev, cudaStream_t st) {
    if (!t_ops) return cudaEventRecord(ev, st);
    t_ops->add(Op::RECORD, st).ptr = ev;
    return cudaSuccess;
}
cudaError_t enqueue_wait(cudaStream_t st, cudaEvent_t ev) {
    if (!t_ops) return cudaStreamWaitEvent(st, ev, 0);
    t_ops->add(Op::WAIT, st).ptr = ev;
    return cudaSuccess;
}

static constexpr int MAX_ARGS = 32;

static int gather_args(const Op& o, OpList& l, void** params) {
    if (o.n_args > (uint32_t)MAX_ARGS) return -1;
    for (uint32_t i = 0; i < o.n_args; ++i) params[i] = l.blob.data() + l.arg_off[o.arg0 + i];
    return (int)o.n_args;
}

cudaError_t launch_list_kernel(const Op& o, OpList& l, cudaStream_t st) {
    void* params[MAX_ARGS];
    if (gather_args(o, l, params) < 0) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = o.grid; cfg.blockDim = o.block; cfg.dynamicSmemBytes = o.bytes; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (o.attr != Op::PLAIN) {
        attr[0].id = o.attr == Op::DEPENDENT ? cudaLaunchAttributeProgrammaticStreamSerialization : cudaLaunchAttributeCooperative;
        if (o.attr == Op::DEPENDENT) attr[0].val.programmaticStreamSerializationAllowed = 1;
        else attr[0].val.cooperative = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
    }
    return cudaLaunchKernelExC(&cfg, o.func, params);
}

static cudaError_t play_op(const Op& o, OpList& l, cudaStream_t st) {
    switch (o.kind) {
    case Op::KERNEL: return launch_list_kernel(o, l, st);
    case Op::MEMSET: return cudaMemsetAsync(o.ptr, 0, o.bytes, st);
    case Op::COPY: return cudaMemcpyAsync(o.ptr, o.func, o.bytes, cudaMemcpyDefault, st);
    case Op::RECORD: return cudaEventRecord(static_cast<cudaEvent_t>(o.ptr), st);
    default: return cudaStreamWaitEvent(st, static_cast<cudaEvent_t>(o.ptr), 0);
    }
}

cudaError_t Player::direct(OpList& l, Profiler* prof) {
    cudaError_t first = cudaSuccess;
    for (const Op& o : l.ops) {
        const cudaStream_t st = l.streams[o.role];
        // after a failure only the events are still played, so that streams that were forked are joined again
        if (first != cudaSuccess && o.kind != Op::RECORD && o.kind != Op::WAIT) continue;
        cudaError_t e;
        if (o.kind == Op::KERNEL && prof && prof->on) {
            Profiler::Rec r{o.name, prof->get(), prof->get()};
            cudaEventRecord(r.start, st);
            e = play_op(o, l, st);
            cudaEventRecord(r.stop, st);
            prof->recs.push_back(r);
        } else e = play_op(o, l, st);
        if (e != cudaSuccess && first == cudaSuccess) first = e;
    }
    return first;
}

void Player::drop(Entry& e) {
    if (e.exec) cudaGraphExecDestroy(e.exec);
    if (e.graph) cudaGraphDestroy(e.graph);
    e.exec = nullptr; e.graph = nullptr; e.seen = 0;
    e.node.clear();
}

Player::~Player() {
    for (Entry& e : entry_) drop(e);
    if (capture_) cudaStreamDestroy(capture_);
}

static bool same_shape(const OpList& a, const OpList& b) {
    if (a.ops.size() != b.ops.size() || a.n_streams != b.n_streams) return false;
    for (int r = 1; r < a.n_streams; ++r) if (a.streams[r] != b.streams[r]) return false;
    for (size_t i = 0; i < a.ops.size(); ++i) if (!a.ops[i].same_shape(b.ops[i])) return false;
    return true;
}

// The list captured into a graph (nothing is enqueued).  The caller's stream is stood in for by a stream of the player's
// own, since the default stream cannot be captured.
bool Player::build(Entry& e, OpList& l) {
    e.node.assign(l.ops.size(), nullptr);                // (nothing below allocates: a capture that has begun is ended)
    if (!capture_ && cudaStreamCreateWithFlags(&capture_, cudaStreamNonBlocking) != cudaSuccess) return false;
    if (cudaStreamBeginCapture(capture_, cudaStreamCaptureModeRelaxed) != cudaSuccess) return false;
    bool ok = true;
    for (size_t i = 0; i < l.ops.size() && ok; ++i) {
        const Op& o = l.ops[i];
        const cudaStream_t st = o.role == 0 ? capture_ : l.streams[o.role];
        ok = play_op(o, l, st) == cudaSuccess;
        if (ok && (o.kind == Op::KERNEL || o.kind == Op::MEMSET || o.kind == Op::COPY)) {
            cudaStreamCaptureStatus status;
            const cudaGraphNode_t* deps = nullptr;
            size_t n_deps = 0;
            const cudaGraphEdgeData* edges = nullptr;
            ok = cudaStreamGetCaptureInfo_v3(st, &status, nullptr, nullptr, &deps, &edges, &n_deps) == cudaSuccess &&
                 status == cudaStreamCaptureStatusActive && n_deps == 1;
            if (ok) e.node[i] = deps[0];                 // the node just added: what a next entry of this stream would wait for
        }
    }
    if (cudaStreamEndCapture(capture_, &e.graph) != cudaSuccess) ok = false;
    if (ok) ok = cudaGraphInstantiate(&e.exec, e.graph, 0) == cudaSuccess;
    if (!ok) { cudaGetLastError(); drop(e); }
    return ok;
}

// Brings the graph's nodes up to date with the list.
bool Player::update(Entry& e, OpList& l) {
    for (size_t i = 0; i < l.ops.size(); ++i) {
        const Op& o = l.ops[i];
        const Op& p = e.last.ops[i];
        if (o.kind == Op::KERNEL) {
            const bool same = o.grid.x == p.grid.x && o.grid.y == p.grid.y && o.grid.z == p.grid.z && o.block.x == p.block.x &&
                              o.bytes == p.bytes && o.blob1 - o.blob0 == p.blob1 - p.blob0 &&
                              memcmp(l.blob.data() + o.blob0, e.last.blob.data() + p.blob0, o.blob1 - o.blob0) == 0;
            if (same) continue;
            void* params[MAX_ARGS];
            if (gather_args(o, l, params) < 0) return false;
            cudaKernelNodeParams kp = {};
            kp.func = const_cast<void*>(o.func); kp.gridDim = o.grid; kp.blockDim = o.block;
            kp.sharedMemBytes = (unsigned)o.bytes; kp.kernelParams = params;
            if (cudaGraphExecKernelNodeSetParams(e.exec, e.node[i], &kp) != cudaSuccess) return false;
        } else if (o.kind == Op::MEMSET) {
            if (o.ptr == p.ptr && o.bytes == p.bytes) continue;
            cudaMemsetParams mp = {};
            mp.dst = o.ptr; mp.elementSize = 1; mp.width = o.bytes; mp.height = 1;
            if (cudaGraphExecMemsetNodeSetParams(e.exec, e.node[i], &mp) != cudaSuccess) return false;
        } else if (o.kind == Op::COPY) {
            if (o.ptr == p.ptr && o.func == p.func && o.bytes == p.bytes) continue;
            if (cudaGraphExecMemcpyNodeSetParams1D(e.exec, e.node[i], o.ptr, o.func, o.bytes, cudaMemcpyDefault) != cudaSuccess) return false;
        }
    }
    return true;
}

cudaError_t Player::play(OpList& l, Profiler* prof) {
    if (l.ops.empty()) return cudaSuccess;
    if (prof && prof->on) return direct(l, prof);
    if (l.n_kernels < MIN_KERNELS) return direct(l, prof);
    // a stream that its owner is capturing is left to the owner's graph (the legacy default stream cannot be captured)
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (l.streams[0] && (cudaStreamIsCapturing(l.streams[0], &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone)) return direct(l, prof);
    Entry* e = nullptr;
    for (Entry& x : entry_)
        if (x.seen && same_shape(x.last, l)) { e = &x; break; }
    if (!e) {
        e = &entry_[0];
        for (Entry& x : entry_) if (x.used < e->used) e = &x;
        drop(*e);
    }
    e->used = ++clock_;
    if (!e->exec) {
        if (++e->seen <= GRAPH_AFTER || !build(*e, l)) {
            const cudaError_t r = direct(l, prof);
            if (!e->seen) e->seen = 1;
            std::swap(e->last, l);
            return r;
        }
        std::swap(e->last, l);
        return cudaGraphLaunch(e->exec, e->last.streams[0]);
    }
    if (!update(*e, l)) {
        cudaGetLastError();
        drop(*e);
        return direct(l, prof);
    }
    std::swap(e->last, l);
    return cudaGraphLaunch(e->exec, e->last.streams[0]);
}

}  // namespace gear
