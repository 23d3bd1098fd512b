"""Sizes at which a kernel changes its tiles or a call its path: sorts, both stores, replayed steps, host batches, chains.

The store's rule is restated here in numpy (fp64) for one array of (ID, row) pairs."""
import numpy as np
import pytest
import torch

from paper_1806_03925_b200 import workloads
from paper_1806_03925_b200.workloads import BF16, F32, PRESETS, Batch, BatchSource

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _store_session(vocab, D, M, n, atomic=False):
    from paper_1806_03925_b200.session import GearSession
    p = PRESETS["skew"].scaled(img_vocab=vocab, dfv_dim=D, M=M, user_vocab=64, url_vocab=64, expire=1 << 40)
    return GearSession(p, np.zeros(p.n_params, np.float32), max_batch=8, max_nnz=max(n, 1), seed=1, expired_cap=1,
                       ready_cap=2 * n + vocab, accum_mode=1 if atomic else 0)


def _ids(vocab, n, seed):
    """A tenth of the rows on three hot images, a few IDs out of range, the rest uniform."""
    rng = np.random.default_rng(seed)
    ids = rng.integers(0, vocab, n)
    hot = rng.random(n) < 0.1
    ids[hot] = rng.choice(np.array([0, vocab // 2, vocab - 1]), int(hot.sum()))
    bad = rng.random(n) < 0.01
    ids[bad] = rng.choice(np.array([-1, vocab, 2 ** 31 - 1, -2 ** 31]), int(bad.sum()))
    return ids.astype(np.int32)


# one block's radix sort up to 2048 rows, a cluster's up to 16384 (tiles of 2048) and 32768 (4096); then the multi-block sort, tiles
# of 2048 while those are no more than its blocks (2 * 148), else of 4096.  A vocabulary of 150000 takes two digits of 9 bits
# (ranked one key at a time), 60000 two of 8 (two keys), 1000 two of 5.
@pytest.mark.parametrize("n,vocab,M", [
    (1, 1000, 1), (31, 1000, 3), (2048, 60_000, 4), (2049, 60_000, 4), (16_384, 1000, 7), (16_385, 150_000, 2),
    (32_768, 60_000, 5), (32_769, 60_000, 5), (40_001, 150_000, 4), (606_208, 60_000, 8), (606_209, 60_000, 8),
    (700_001, 150_000, 16), (620_000, 3_000_000, 2),
])
def test_sorted_store_at_sort_and_plan_edges(n, vocab, M):
    """Two calls, so that the second finds partial sums.  A sum of fewer than M values in (-1, 1), added one by one in fp32, is off
    by at most M * 2^-24 * M; the division adds a rounding."""
    D = 8
    s = _store_session(vocab, D, M, n)
    try:
        rng = np.random.default_rng(n)
        held, count = np.zeros((vocab, D)), np.zeros(vocab, np.int64)
        for call in range(2):
            ids, rows = _ids(vocab, n, 10 * n + call), rng.uniform(-1, 1, (n, D)).astype(np.float32)
            got = s.accumulate_collect_rows(torch.from_numpy(ids).cuda(), torch.from_numpy(rows).cuda())
            ok = (ids >= 0) & (ids < vocab)
            order = np.flatnonzero(ok)[np.argsort(ids[ok], kind="stable")]
            key = ids[order]
            first = np.r_[True, key[1:] != key[:-1]] if key.size else np.zeros(0, bool)
            start = np.flatnonzero(first)
            rank = np.arange(key.size) - np.repeat(start, np.diff(np.r_[start, key.size])) + count[key]
            group = rank // M                                        # 0: the group that was open before the call
            new = first | (rank % M == 0)
            g0 = np.flatnonzero(new)
            sums = np.add.reduceat(rows[order].astype(np.float64), g0, axis=0) if g0.size else np.zeros((0, D))
            gkey, ggroup = key[g0], group[g0]
            sums[ggroup == 0] += held[gkey[ggroup == 0]]
            total = count + np.bincount(key, minlength=vocab)
            done = ggroup < total[gkey] // M
            assert got == int(done.sum())
            tol = M * M * 2.0 ** -24 + 2.0 ** -23
            assert np.array_equal(s.ready_ids[:got].cpu().numpy(), gkey[done])
            assert np.array_equal(s.ready_seq[:got].cpu().numpy(), ggroup[done])
            np.testing.assert_allclose(s.ready_avg[:got].cpu().numpy(), sums[done] / M, rtol=0, atol=tol)
            touched = np.unique(key)
            held[touched] = 0.0
            held[gkey[~done]] = sums[~done]
            count = total % M
            assert np.array_equal(s.dfv_gcnt.cpu().numpy(), count)
            open_ = np.flatnonzero(count)
            np.testing.assert_allclose(s.dfv_gsum[torch.from_numpy(open_).cuda()].cpu().numpy(), held[open_], rtol=0, atol=tol)
    finally:
        s.close()


# sorted and planned by one block, by one cluster (bf16: beside the gather, the rows put in behind both), by the multi-block sort
@pytest.mark.parametrize("head,B", [(F32, 300), (BF16, 300), (F32, 1500), (BF16, 1500), (BF16, 12_000)])
def test_occurrences_that_no_page_view_covers(head, B):
    """Two views with offsets beyond the batch: their occurrences' entries of row_view stay what they were (-1).  The rows count as
    zeros, the others as always: k values of an image, each rounded once, added one by one in fp32, are off by at most (k + 1) * 2^-24
    of the sum of their sizes."""
    from paper_1806_03925_b200 import binding as gb
    from paper_1806_03925_b200.session import DeviceBatch, GearSession
    p = PRESETS["medium"].scaled(batch=B, user_vocab=500, url_vocab=500, img_vocab=2000, M=50_000, dfv_dim=72, dfv_dtype=head, head_dtype=head,
                                 hidden=(64,))
    b = BatchSource(p, 3).batch(0, B)
    lo, hi = int(b.img_off[B // 2]), int(b.img_off[B // 2 + 2])
    b.img_off[B // 2 + 1] = b.nnz + 100                                  # view B / 2 ends past the batch, the next one starts there
    s = GearSession(p, workloads.head_params(p, 0), max_batch=B, max_nnz=b.nnz, seed=3)
    try:
        for now in (1, 2):
            s.row_view.fill_(-1)
            s.dfv_gsum.zero_()
            s.dfv_gcnt.zero_()
            s.step(DeviceBatch.from_host(b), now)
            torch.cuda.synchronize()
            assert s.status()[1] == gb.GEAR_DEV_BAD_CSR
            view = s.row_view[:b.nnz].cpu().numpy()
            assert (view[lo:hi] == -1).all() and (np.delete(view, np.arange(lo, hi)) >= 0).all()
            g = s.dX[:, 2 * p.emb_dim:].double().cpu().numpy()[view] * s.inv_n.double().cpu().numpy()[view][:, None] * (view >= 0)[:, None]
            want, size = np.zeros((2, p.img_vocab, p.dfv_dim))
            np.add.at(want, b.img_id, g)
            np.add.at(size, b.img_id, np.abs(g))
            k = np.bincount(b.img_id, minlength=p.img_vocab)
            assert np.array_equal(s.dfv_gcnt.cpu().numpy(), k)
            assert np.all(np.abs(s.dfv_gsum.cpu().numpy() - want) <= (k + 1)[:, None] * 2.0 ** -24 * size + 1e-37)
    finally:
        s.close()


# blocks take 256 rows, warps 32 of them; rows of 72 columns leave lanes idle, of 136 take a second round
@pytest.mark.parametrize("n,vocab,M,D", [(1, 1000, 1, 8), (255, 1000, 4, 72), (256, 5, 3, 128), (257, 1000, 2, 136), (20_011, 3, 64, 72),
                                         (33_000, 40_000, 1, 64)])
def test_order_free_store_at_block_edges(n, vocab, M, D):
    """k rows for an image of an empty store: floor(k / M) copies of their mean leave, k mod M times the mean stays (k < M: the sum).
    k values in (-1, 1) added in any order in fp32 are off by at most k * 2^-24 * k."""
    s = _store_session(vocab, D, M, n, atomic=True)
    try:
        ids, rows = _ids(vocab, n, n), np.random.default_rng(n).uniform(-1, 1, (n, D)).astype(np.float32)
        got = s.accumulate_collect_rows(torch.from_numpy(ids).cuda(), torch.from_numpy(rows).cuda())
        ok = (ids >= 0) & (ids < vocab)
        k = np.bincount(ids[ok], minlength=vocab)
        total = np.zeros((vocab, D))
        np.add.at(total, ids[ok], rows[ok].astype(np.float64))
        want = np.repeat(np.arange(vocab), k // M)
        assert got == want.size
        assert np.array_equal(s.ready_ids[:got].cpu().numpy(), want)
        assert np.array_equal(s.dfv_gcnt.cpu().numpy(), k % M)
        mean = total / np.maximum(k, 1)[:, None]
        tol = (k.max() * 2.0 ** -24 + 2.0 ** -22) * max(M, 1)
        np.testing.assert_allclose(s.ready_avg[:got].cpu().numpy(), mean[want], rtol=0, atol=tol)
        stay = np.where((k < M)[:, None], total, mean * (k % M)[:, None])
        np.testing.assert_allclose(s.dfv_gsum.cpu().numpy(), stay, rtol=0, atol=tol)
    finally:
        s.close()


@pytest.mark.parametrize("head", [F32, BF16])
def test_replayed_steps_follow_sizes_and_pointers(head):
    """Twenty steps over batches of changing sizes (three of the same shape make a graph of them) against the same calls one by one.
    The sums of embedding rows and weight gradients are added in no fixed order: 1e-5, bf16 1e-2, as everywhere."""
    from gpu_harness import _np, assert_close
    from paper_1806_03925_b200.session import DeviceBatch, GearSession
    p = PRESETS["medium"].scaled(batch=640, user_vocab=5000, url_vocab=5000, img_vocab=20_011, expire=3, M=3, dfv_dtype=head,
                                 head_dtype=head, hidden=(128, 64))
    sizes = [640, 640, 640, 640, 640, 640, 1, 639, 640, 33, 640, 1, 639, 200, 201, 202, 203, 640, 5, 640]
    batches = [BatchSource(p, 7 + k).batch(k, n) for k, n in enumerate(sizes)]
    nnz = max(b.nnz for b in batches)
    a, c = (GearSession(p, workloads.head_params(p, 3), max_batch=p.batch, max_nnz=nnz, seed=3, expired_cap=p.img_vocab) for _ in range(2))
    tol = 1e-5 if head == F32 else 1e-2
    try:
        for now, b in enumerate(batches, 1):
            d = DeviceBatch.from_host(b)
            n_ready, n_exp = a.step(d, now, sync=now % 2 == 0)
            torch.cuda.synchronize()
            if n_ready is None:
                n_ready, n_exp = (int(x) for x in a.d_counts[:2].tolist())
            c.forward_backward(d)
            assert c.accumulate_collect_from_step(d) == n_ready
            assert c.collect_expired(now) == n_exp
            for name, m in (("ready_ids", n_ready), ("ready_seq", n_ready), ("expired_ids", n_exp)):
                assert np.array_equal(_np(getattr(a, name)[:m]), _np(getattr(c, name)[:m])), (now, name)
            assert torch.equal(a.dfv_gcnt, c.dfv_gcnt) and torch.equal(a.dfv_ts, c.dfv_ts)
            assert_close(_np(a.ready_avg[:n_ready]), _np(c.ready_avg[:n_ready]), tol, "averages")
            assert_close(_np(a.loss), _np(c.loss), tol, "loss")
            assert_close(_np(a.head_grad), _np(c.head_grad), tol, "head_grad")
            assert_close(_np(a.user_emb), _np(c.user_emb), tol, "user rows")
        assert a.status()[1] == 0 and c.status()[1] == 0
    finally:
        a.close()
        c.close()


@pytest.mark.parametrize("fast", [False, True])
def test_host_batch_arrives_as_it_is(fast):
    """Slices of one copy, also of arrays that are not contiguous; a batch without images; the C struct follows replaced tensors."""
    from paper_1806_03925_b200.session import DeviceBatch, GearSession
    rng = np.random.default_rng(5)
    for B, nnz in ((1, 0), (7, 13), (300, 1001)):
        cut = np.sort(rng.integers(0, nnz + 1, B - 1)) if B > 1 else np.zeros(0, np.int64)
        off = np.r_[0, cut, nnz].astype(np.int32)
        b = Batch(rng.integers(0, 99, 2 * B).astype(np.int32)[::2], rng.integers(0, 99, B).astype(np.int32), off,
                  rng.integers(0, 99, nnz).astype(np.int32), rng.random(B).astype(np.float32),
                  rng.random((B, 12)).astype(np.float32) if fast else None)
        d = DeviceBatch.from_host(b)
        assert d.B == B and d.nnz == nnz
        for name in ("user_id", "url_id", "img_off", "img_id", "label") + (("fast",) if fast else ()):
            got, want = getattr(d, name), getattr(b, name)
            assert got.is_cuda and got.is_contiguous() and np.array_equal(got.cpu().numpy(), want), name
            assert str(got.dtype) == "torch." + want.dtype.name
        c = GearSession._c_batch(d)
        assert c.user_id == d.user_id.data_ptr() and c.label == d.label.data_ptr() and c.img_off == d.img_off.data_ptr()
        assert (c.fast or 0) == (d.fast.data_ptr() if fast else 0)
        d.label = d.label.clone()
        assert GearSession._c_batch(d).label == d.label.data_ptr()


# tiles of 32 rows x 32 columns, up to three of the ring's four buffers of 32 values (deeper: test_dense_forward_of_unaligned_operands) or,
# 129 values, five; rows that are no multiple of 16 bytes
@pytest.mark.parametrize("n,R,D", [(1, 1, 8), (16, 32, 64), (17, 33, 72), (15, 64, 8), (40, 31, 136), (33, 96, 64), (2400, 129, 64)])
def test_dense_forward_at_tile_edges(n, R, D):
    """Against fp64; R products of values in (-1, 1) added one by one in fp32 are off by at most R * 2^-24 * R."""
    s = _store_session(500, D, 4, 8)
    try:
        rng = np.random.default_rng(R)
        raw, Wd = rng.uniform(-1, 1, (500, R)).astype(np.float32), rng.uniform(-1, 1, (R, D)).astype(np.float32)
        ids = rng.integers(0, 500, n).astype(np.int32)
        rows = torch.full((n, D), 7.0, device="cuda")
        s.dense_forward(torch.from_numpy(raw).cuda(), torch.from_numpy(Wd).cuda(), torch.from_numpy(ids).cuda(), rows, n=n)
        want = raw[ids].astype(np.float64) @ Wd.astype(np.float64)
        np.testing.assert_allclose(rows.cpu().numpy(), want, rtol=0, atol=R * R * 2.0 ** -24)
    finally:
        s.close()


def _replays(call, *sessions):
    """The call captured on its owner's graph, as a function that replays it."""
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g.replay


# one cluster's sort, the multi-block sort with its grid barrier
@pytest.mark.parametrize("n,vocab", [(1000, 500), (40_001, 60_000)])
def test_a_captured_store_call_can_be_replayed(n, vocab):
    """Replays with new rows, other calls between them, against the same calls one by one: the order of a sum is fixed, so the
    results are the same numbers."""
    M, D = 3, 8
    a, c = (_store_session(vocab, D, M, n) for _ in range(2))
    try:
        ids, rows = torch.zeros(n, dtype=torch.int32, device="cuda"), torch.zeros((n, D), device="cuda")

        def fresh(seed):
            ids.copy_(torch.from_numpy(_ids(vocab, n, seed)))
            rows.copy_(torch.from_numpy(np.random.default_rng(seed).uniform(-1, 1, (n, D)).astype(np.float32)))
        fresh(0)
        for k in range(5):                                   # past the point where the call has a graph of its own
            for s in (a, c):
                s.accumulate_collect_rows(ids, rows)
        replay = _replays(lambda: a.accumulate_collect_rows(ids, rows, sync=False))
        for k in range(1, 7):
            fresh(k)
            if k % 3 == 0:
                a.accumulate_collect_rows(ids, rows)
            else:
                replay()
            want = c.accumulate_collect_rows(ids, rows)
            torch.cuda.synchronize()
            assert int(a.d_counts[0]) == want, k
            for name in ("ready_ids", "ready_seq", "ready_avg"):
                assert torch.equal(getattr(a, name)[:want], getattr(c, name)[:want]), (k, name)
            assert torch.equal(a.dfv_gcnt, c.dfv_gcnt) and torch.equal(a.dfv_gsum, c.dfv_gsum), k
        assert a.status()[1] & ~1 == 0                       # (the IDs out of range were noted)
    finally:
        a.close()
        c.close()


def test_a_captured_expiry_scan_can_be_replayed():
    """A scan adds to one of two sets of section counts (64 tiles of 2048 timestamps) and clears the other: replays, the same scan
    over and over, with scans of a step's kind between them, against the timestamps on the host."""
    from paper_1806_03925_b200.session import GearSession
    V, T = 300_007, 5
    p = PRESETS["tiny"].scaled(user_vocab=64, url_vocab=64, img_vocab=V, expire=T)
    s = GearSession(p, workloads.head_params(p, 0), max_batch=8, max_nnz=32)
    try:
        replay = None
        for k in range(8):
            ts = np.random.default_rng(k).integers(-9, 10, V)
            if k == 2:
                replay = _replays(lambda: s.collect_expired(10, restamp=True, sync=False))
            s.dfv_ts.copy_(torch.from_numpy(ts))
            if k in (0, 1, 5):
                s.collect_expired(10, restamp=True)
            else:
                replay()
            torch.cuda.synchronize()
            want = np.flatnonzero(10 - ts >= T)
            assert int(s.d_counts[1]) == want.size, k
            assert np.array_equal(s.expired_ids[:want.size].cpu().numpy(), want), k
            ts[want] = 10
            assert np.array_equal(s.dfv_ts.cpu().numpy(), ts), k
        assert s.status()[1] == 0
    finally:
        s.close()


def test_a_host_batch_may_be_used_on_any_stream():
    """Made on a stream that is busy for some milliseconds; its tensors read, or the batch handed to a session, on another one."""
    from paper_1806_03925_b200.session import DeviceBatch, GearSession
    p = PRESETS["tiny"]
    b = BatchSource(p, 3).batch(0)
    names = ("user_id", "url_id", "img_off", "img_id", "label")
    busy, other = torch.cuda.Stream(), torch.cuda.Stream()
    a, c = (GearSession(p, workloads.head_params(p, 3), max_nnz=b.nnz, seed=3) for _ in range(2))
    try:
        DeviceBatch.from_host(b)                                         # (the pools have their blocks)
        torch.cuda.synchronize()
        with torch.cuda.stream(busy):
            torch.cuda._sleep(20_000_000)
            read, used, mixed = (DeviceBatch.from_host(b) for _ in range(3))
            mixed.label = 1 - torch.from_numpy(b.label).cuda()
        with torch.cuda.stream(other):
            got = {name: getattr(read, name).clone() for name in names}
            n_ready, n_exp = a.step(used, 1, sync=True)
            assert GearSession._c_batch(mixed).label == mixed.label.data_ptr()
        torch.cuda.synchronize()
        for name, t in got.items():
            assert np.array_equal(t.cpu().numpy(), getattr(b, name)), name
        assert np.array_equal(mixed.label.cpu().numpy(), 1 - b.label) and np.array_equal(mixed.img_id.cpu().numpy(), b.img_id)
        assert (n_ready, n_exp) == c.step(DeviceBatch(*(torch.from_numpy(getattr(b, n)).cuda() for n in names), b.B, b.nnz), 1, sync=True)
        assert torch.equal(a.prob, c.prob)
    finally:
        a.close()
        c.close()


def test_a_step_writes_to_the_lists_a_session_has_now():
    """A program that keeps a step's lists and puts fresh ones in their place."""
    from paper_1806_03925_b200.session import DeviceBatch, GearSession
    p = PRESETS["tiny"].scaled(expire=1, M=1)
    batches = [DeviceBatch.from_host(BatchSource(p, 3).batch(k)) for k in range(2)]
    a, c = (GearSession(p, workloads.head_params(p, 3), max_nnz=max(b.nnz for b in batches), seed=3) for _ in range(2))
    try:
        names = ("ready_ids", "ready_seq", "ready_avg", "expired_ids", "d_counts")
        assert a.step(batches[0], 1, sync=True) == c.step(batches[0], 1, sync=True)
        kept = {n: getattr(a, n) for n in names}
        held = {n: t.clone() for n, t in kept.items()}
        for n in names:
            setattr(a, n, torch.full_like(kept[n], -3))
        got = a.step(batches[1], 2, sync=True)
        assert got == c.step(batches[1], 2, sync=True) and got[0] == batches[1].nnz and got[1] == p.img_vocab
        assert a.d_counts.tolist() == list(got)
        for n, m in (("ready_ids", got[0]), ("ready_seq", got[0]), ("ready_avg", got[0]), ("expired_ids", got[1])):
            assert torch.equal(getattr(a, n)[:m], getattr(c, n)[:m]), n
        for n in names:
            assert torch.equal(kept[n], held[n]), n
    finally:
        a.close()
        c.close()
