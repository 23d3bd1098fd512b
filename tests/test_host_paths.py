"""Host code of libgear without a GPU: the library's own objects, linked against a stand-in for the CUDA runtime
(fake_cudart.cpp) that writes down what is enqueued and can make a chosen call fail.  What the kernels compute is not tested here."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STREAM = 0x5000                  # the caller's stream


class Host:
    """The linked library, and contexts on addresses that nothing ever reads."""

    def __init__(self, lib, gb):
        self.lib, self.gb = lib, gb
        lib.fake_unfinished.restype = C.c_int
        lib.fake_calls.restype = lib.fake_live.restype = lib.fake_log.restype = lib.fake_news.restype = C.c_long
        lib.fake_fail_at.argtypes = lib.fake_no_memory_at.argtypes = [C.c_long]
        lib.fake_device.argtypes = [C.c_int]
        lib.fake_user_capture.argtypes = [C.c_void_p, C.c_int]
        self.next = 1 << 40
        self.keep = []

    def address(self, n=1 << 24):
        self.next += n
        return self.next - n

    def log(self):
        buf = C.create_string_buffer(1 << 20)
        assert self.lib.fake_log(buf, len(buf)) >= 0
        return [line.split() for line in buf.value.decode().splitlines()]

    def ctx(self, batch=64, nnz=512, hidden=(64,), head=0, M=4, mode=0, img_vocab=1000, max_batch=None, max_nnz=None):
        gb = self.gb
        cfg = gb.make_config(1000, 1000, img_vocab, 16, 64, 0, head, list(hidden), M, 10, max_batch or batch, max_nnz or nnz, 0, mode)
        words = C.c_size_t()
        assert self.lib.gear_workspace_bytes(C.byref(cfg), C.byref(words)) == 0
        b = gb.gear_buffers()
        for name in ("user_emb", "url_emb", "dfv", "dfv_gsum", "dfv_gcnt", "dfv_ts", "head_params"):
            setattr(b, name, self.address())
        b.workspace, b.workspace_bytes = self.address(1 << 34), words.value
        out = C.c_void_p()
        assert self.lib.gear_init_tables(C.byref(out), C.byref(cfg), C.byref(b), 0, 0, 0, STREAM) == 0
        return out

    def out(self, **more):
        o = self.gb.gear_step_out()
        for name in ("loss", "prob", "head_grad", "dX", "row_view", "inv_n"):
            setattr(o, name, self.address())
        for name, v in more.items():
            setattr(o, name, v)
        return o

    def lists(self, cap=512):
        s = self.gb.gear_step_lists()
        for name in ("ids", "seq", "avg", "d_n", "expired"):
            setattr(s, name, self.address())
        s.d_expired, s.cap, s.expired_cap = s.d_n + 8, cap, 1000
        return s

    def shard(self, world=2, batch=64, nnz=512, arrivals=100, head=0):
        """A plan, its batches (host arrays), the contexts; `arrivals` is what every owner finds in the staging buffer's counts."""
        gb, lib = self.gb, self.lib
        owners = [self.ctx(batch * world, nnz * world, head=head, img_vocab=100_000) for _ in range(world)]
        workers = [self.ctx(batch, nnz, head=head, mode=gb.GEAR_ACC_ATOMIC, img_vocab=100_000) for _ in range(world)]
        words = C.c_int64()
        assert lib.gear_shard_host_words(world, batch, nnz, C.byref(words)) == 0
        stage = (C.c_int32 * words.value)(*([arrivals] * (words.value - 4 * world)))          # (the owners' results: zeros)
        dX, rows = self.address(), self.address(1 << 30)
        outs = (gb.gear_step_out * world)(*(self.out(dX=dX + 4 * s * batch * 96, dfv_grad=rows + 4 * s * nnz * 64) for s in range(world)))
        lists = (gb.gear_step_lists * world)(*(self.lists(nnz * world) for _ in range(world)))
        ctxs = [(C.c_void_p * world)(*(c.value for c in side)) for side in (owners, workers)]
        plan = gb.gear_shard_plan(world, batch, nnz, ctxs[0], ctxs[1], C.addressof(stage), self.address(1 << 30), self.address(), outs, lists)
        batches = (gb.gear_host_batch * world)()
        zeros = (C.c_int32 * (batch + nnz))()
        for b in batches:
            b.B, b.nnz = batch, nnz
            for name in ("user_id", "url_id", "img_off", "img_id", "label"):
                setattr(b, name, C.addressof(zeros))
        self.keep += [stage, outs, lists, ctxs, zeros]
        return plan, batches, owners + workers

    def shard_step(self, plan, batches, now=1, mean=1):
        counts = (C.c_int64 * (2 * plan.world))()
        return self.lib.gear_shard_step(C.byref(plan), batches, 0.1, now, mean, counts, STREAM)

    def batch(self, B=64, nnz=200):
        b = self.gb.gear_batch()
        for name in ("user_id", "url_id", "img_off", "img_id", "label"):
            setattr(b, name, self.address())
        b.B, b.nnz = B, nnz
        return b


@pytest.fixture(scope="module")
def linked(tmp_path_factory):
    from paper_1806_03925_b200 import binding, build
    build.build()
    d = tmp_path_factory.mktemp("host")
    so = str(d / "libgear_host.so")
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    cuda = os.path.dirname(os.path.dirname(build._nvcc()))
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                           os.path.join(ROOT, "tests", "fake_cudart.cpp")] + objs + ["-o", so])
    lib_path, lib = binding.LIB_PATH, binding._lib
    try:                                                         # the binding's prototypes, on the linked library
        binding.LIB_PATH, binding._lib = so, None
        return binding.load(), binding
    finally:
        binding.LIB_PATH, binding._lib = lib_path, lib


@pytest.fixture()
def host(linked):
    linked[0].fake_reset()
    return Host(*linked)


def test_image_occurrences_without_page_views_are_refused(host):
    """A batch of no views with image IDs: the occurrences' rows exist nowhere.  Refused before anything is enqueued."""
    gb = host.gb
    for mode in (gb.GEAR_ACC_SORT, gb.GEAR_ACC_ATOMIC):
        ctx = host.ctx(mode=mode)
        host.log()
        rc = host.lib.gear_step(ctx, host.batch(B=0, nnz=5), 0.1, host.out(), host.lists(), 1, 1, 1, None, STREAM)
        assert rc == gb.GEAR_ERR_STATE and host.log() == []
        assert host.lib.gear_step(ctx, host.batch(B=0, nnz=0), 0.1, host.out(), host.lists(), 1, 1, 1, None, STREAM) == 0
        assert host.lib.gear_destroy(ctx) == 0
    plan, batches, ctxs = host.shard()
    assert host.shard_step(plan, batches) == 0
    host.log()
    batches[1].B = 0
    assert host.shard_step(plan, batches) == gb.GEAR_ERR_ARG and host.log() == []
    batches[1].nnz = 0
    assert host.shard_step(plan, batches) == 0
    for c in ctxs:
        assert host.lib.gear_destroy(c) == 0


def _store_call(host, ctx, n=40_001, ids=None, grads=None):
    lists = host.lists(cap=n)
    return host.lib.gear_accumulate_collect(ctx, ids or host.address(), grads or host.address(), 64, None, None, n, lists.ids, lists.seq,
                                            lists.avg, n, lists.d_n, None, STREAM)


def test_a_capturing_stream_gets_kernels_also_of_a_shape_with_a_graph(host):
    """Its owner's graph holds the call's own kernels, and the call's graph is left as it was."""
    ctx = host.ctx(nnz=50_000, max_nnz=50_000)
    kernels = []
    for call in range(6):
        host.log()
        assert _store_call(host, ctx) == 0
        seen = [line[0] for line in host.log()]
        assert ("graph" in seen) == (call >= 3), (call, seen)
    host.lib.fake_user_capture(STREAM, 1)
    assert _store_call(host, ctx) == 0
    host.lib.fake_user_capture(None, 0)
    log = host.log()
    assert all(line[0] == "node" and line[1] == "%x" % STREAM for line in log), log
    kernels = [line[2] for line in log]
    assert len(kernels) == 4 and "coop_sort_kernel" in kernels[0] and "acc_reduce_kernel" in kernels[3]
    assert _store_call(host, ctx) == 0
    assert [line[0] for line in host.log()].count("graph") == 1
    assert host.lib.gear_destroy(ctx) == 0


def test_an_expiry_scan_that_was_cut_off_leaves_no_counts(host):
    """A mark pass without its write pass: the next scan clears the counts first; one that ran whole costs nothing more."""
    lib, ctx = host.lib, host.ctx()
    scan = lambda: lib.gear_collect_expired(ctx, 1, 1, host.address(), 1000, host.address(), None, STREAM)
    names = lambda: [("expiry_" + line[2].split("expiry_")[1].split("_")[0]) if line[0] == "launch" else line[0] for line in host.log()]
    host.log()
    assert scan() == 0 and scan() == 0
    assert names() == ["expiry_mark", "expiry_write"] * 2
    lib.fake_fail_at(2)
    assert scan() == host.gb.GEAR_ERR_CUDA
    lib.fake_fail_at(-1)
    assert names() == ["expiry_mark", "FAIL"]
    assert scan() == 0 and scan() == 0
    assert names() == ["memset", "expiry_mark", "expiry_write", "expiry_mark", "expiry_write"]
    assert lib.gear_destroy(ctx) == 0


def _failing_call(host, call, k):
    host.lib.fake_fail_at(k)
    rc = call()
    hit = host.lib.fake_calls() >= k
    host.lib.fake_fail_at(-1)
    return rc, hit


@pytest.mark.parametrize("warm", [0, 5])                       # one launch after the other; as graphs
@pytest.mark.parametrize("arrivals,nnz", [(100, 512), (40_000, 25_000)])
def test_a_partitioned_step_that_fails_leaves_nothing_running(host, arrivals, nnz, warm):
    """Whichever of its calls to the runtime fails: when gear_shard_step has returned, no stream holds work that the host has not
    waited for (the caller may free the tables or use the staging buffer again), and the next step goes through."""
    gb, lib = host.gb, host.lib
    live, failed, k, hit = lib.fake_live(), 0, 0, True
    while hit:
        k += 1
        plan, batches, ctxs = host.shard(nnz=nnz, arrivals=arrivals)
        for _ in range(warm):
            assert host.shard_step(plan, batches) == 0, lib.gear_last_error()
            assert lib.fake_unfinished() == 0
        rc, hit = _failing_call(host, lambda: host.shard_step(plan, batches), k)
        failed += rc != 0                                        # (a graph that cannot be updated is played launch by launch)
        assert rc in (0, gb.GEAR_ERR_CUDA) and lib.fake_unfinished() == 0, k
        assert host.shard_step(plan, batches) == 0 and lib.fake_unfinished() == 0, k
        for c in ctxs:
            assert lib.gear_destroy(c) == 0
        host.log()
    assert failed > (5 if warm else 50) and lib.fake_live() == live


@pytest.mark.parametrize("warm", [0, 5])
@pytest.mark.parametrize("head,B,nnz", [(0, 64, 200), (1, 5000, 40_000)])
def test_a_step_that_fails_is_joined_to_its_stream(host, head, B, nnz, warm):
    """Whichever of its calls to the runtime fails: the caller's stream covers what was enqueued, and the next step does not take
    the ready queue to be empty."""
    lib = host.lib
    failed, k, hit = 0, 0, True
    while hit:
        k += 1
        ctx = host.ctx(B, nnz, hidden=(128, 64), head=head)
        out, lists = host.out(), host.lists(nnz)
        step = lambda: lib.gear_step(ctx, host.batch(B, nnz), 0.1, out, lists, 1, 1, 1, None, STREAM)
        for _ in range(warm):
            assert step() == 0
        rc, hit = _failing_call(host, step, k)
        lib.cudaStreamSynchronize(C.c_void_p(STREAM))
        assert lib.fake_unfinished() == 0, k
        host.log()
        assert step() == 0
        log = " ".join(" ".join(line) for line in host.log())
        if rc != 0:
            failed += 1
            assert "collect_sort" in log and "collect_move" in log, k         # whatever the queue holds is handed over, in order
        assert lib.gear_destroy(ctx) == 0
    assert failed > (0 if warm else 30)


@pytest.mark.parametrize("warm", [0, 3, 5])                    # ... where the graph is made; with it
def test_no_call_throws_when_the_host_is_out_of_memory(host, warm):
    """Whichever allocation of a call fails, the call returns GEAR_ERR_CUDA (an exception would end the process here), the caller's
    stream covers what was enqueued, and the calls that follow go through."""
    gb, lib = host.gb, host.lib
    calls = {
        "step": lambda c: lib.gear_step(c, host.batch(5000, 40_000), 0.1, host.out(), host.lists(40_000), 1, 1, 1, None, STREAM),
        "forward_backward": lambda c: lib.gear_forward_backward(c, host.batch(), 0.1, host.out(), STREAM),
        "collect_expired": lambda c: lib.gear_collect_expired(c, 1, 1, host.address(), 1000, None, None, STREAM),
        "refresh": lambda c: lib.gear_refresh_dfv(c, host.address(), host.address(), 64, 10, None, 1, STREAM),
        "fetch": lambda c: lib.gear_fetch_rows(c, 0, host.address(), 10, host.address(), STREAM),
        "dense_forward": lambda c: lib.gear_dense_forward(c, host.address(), 32, host.address(), host.address(), 10, None, host.address(), 64, STREAM),
        "dense_backward": lambda c: lib.gear_dense_backward(c, host.address(), 32, host.address(), host.address(), 10, None, host.address(), STREAM),
        "adam": lambda c: lib.gear_adam_dense(host.address(), host.address(), host.address(), host.address(), 10, 1, C.byref(gb.make_adam()), STREAM),
        "expired_static": lambda c: lib.gear_collect_expired_static(host.address(), 1000, 1, 1, 1, host.address(), 1000, None, None, STREAM),
    }
    for name, call in calls.items():
        failed, k, hit = 0, 0, True
        while hit:
            k += 1
            ctx = host.ctx(5000, 40_000, hidden=(128, 64))
            for _ in range(warm):
                assert call(ctx) == 0, (name, lib.gear_last_error())
            lib.fake_no_memory_at(k)
            rc = call(ctx)
            hit = lib.fake_news() >= k
            lib.fake_no_memory_at(-1)
            assert rc == (gb.GEAR_ERR_CUDA if hit else 0), (name, k)
            failed += hit
            lib.cudaStreamSynchronize(C.c_void_p(STREAM))
            assert lib.fake_unfinished() == 0, (name, k)
            for _ in range(2):
                assert call(ctx) == 0, (name, k)
            assert lib.gear_destroy(ctx) == 0
            host.log()
        assert failed > 0 or (warm and name in ("step", "forward_backward")), name
    plan, batches, ctxs = host.shard(nnz=25_000, arrivals=40_000)
    for _ in range(warm):
        assert host.shard_step(plan, batches) == 0
    k, hit = 0, True
    while hit:
        k += 1
        lib.fake_no_memory_at(k)
        rc = host.shard_step(plan, batches)
        hit = lib.fake_news() >= k
        lib.fake_no_memory_at(-1)
        assert rc == (gb.GEAR_ERR_CUDA if hit else 0) and lib.fake_unfinished() == 0, k
    for c in ctxs:
        assert lib.gear_destroy(c) == 0


def test_kernels_get_their_shared_memory_on_every_device(host):
    """Contexts on a second device of the process: what a kernel may take beyond 48 KB is asked for there too."""
    lib = host.lib
    for device in (0, 1):
        lib.fake_device(device)
        for head in (0, 1):
            for hidden in ((64,), (128, 64), (256, 192), (512, 256), (512, 320)) + (((24,), (256, 136)) if head == 0 else ()):
                for B, nnz in ((64, 200), (1200, 3600), (2400, 7000), (8000, 40_000), (60_000, 600_000)):
                    ctx = host.ctx(B, nnz, hidden=hidden, head=head)
                    rc = lib.gear_step(ctx, host.batch(B, nnz), 0.1, host.out(), host.lists(nnz), 1, 1, 1, None, STREAM)
                    assert rc == 0, (device, head, hidden, B, lib.gear_last_error())
                    assert lib.gear_dense_forward(ctx, host.address(), 32, host.address(), host.address(), 10, None, host.address(), 64, STREAM) == 0
                    assert lib.gear_dense_forward(ctx, host.address(), 33, host.address() + 4, host.address(), 10, None, host.address(), 64, STREAM) == 0
                    assert lib.gear_destroy(ctx) == 0
    lib.fake_device(0)


@pytest.mark.parametrize("head", [0, 1])
def test_batches_of_millions_of_views_fit_every_grid(host, head):
    """65536 row tiles of 64 views and one more: no launch has a second or third dimension above 65535."""
    B = 65_536 * 64 + 1
    ctx = host.ctx(B, 2 * B, hidden=(128,), head=head)
    assert host.lib.gear_step(ctx, host.batch(B, 2 * B), 0.1, host.out(), host.lists(2 * B), 1, 1, 1, None, STREAM) == 0
    assert host.lib.gear_destroy(ctx) == 0


def test_a_context_costs_no_pinned_memory_before_a_count_is_waited_for(host):
    """One clear besides the tables', no page-locked block; the block comes with the first h_n, and a partitioned step needs none
    (its counts lie in the plan's staging buffer)."""
    lib = host.lib
    plan, batches, ctxs = host.shard()
    log = [line[0] for line in host.log()]
    assert "pinned" not in log and log.count("memset") == len(ctxs)
    for _ in range(5):
        assert host.shard_step(plan, batches) == 0
    assert "pinned" not in [line[0] for line in host.log()]
    n = C.c_int64()
    for k in range(3):
        assert lib.gear_collect_expired(ctxs[0], 1, 1, host.address(), 1000, None, C.byref(n), STREAM) == 0
    assert [line[0] for line in host.log()].count("pinned") == 1
    for c in ctxs:
        assert lib.gear_destroy(c) == 0
