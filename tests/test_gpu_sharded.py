"""The step with the tables partitioned by ID and all ranks in this process: the native call (gear_shard_step) against the same step
exchange by exchange, which goes by the same rules through other calls."""
import numpy as np
import pytest
import torch

from paper_1806_03925_b200 import workloads
from paper_1806_03925_b200.workloads import BF16, PRESETS, Batch, BatchSource

pytestmark = pytest.mark.gpu

TABLES = ("user_emb", "url_emb", "dfv_gsum", "dfv_gcnt", "dfv_ts")


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _exchange(world):
    """An in-process exchange with a method of its own: the step goes through its calls."""
    from paper_1806_03925_b200.sharded import LoopbackExchange

    class Counting(LoopbackExchange):
        routed = 0

        def route(self, ids):
            self.routed += 1
            return super().route(ids)
    return Counting(world)


def _jobs(p, world, max_batch, max_nnz, **more):
    from paper_1806_03925_b200.sharded import LoopbackExchange, ShardedGear
    return [ShardedGear(p, workloads.head_params(p, 2), ex, max_batch_local=max_batch, max_nnz_local=max_nnz, seed=5, **more)
            for ex in (LoopbackExchange(world), _exchange(world))]


def _small(world, **more):
    p = PRESETS["tiny"].scaled(user_vocab=501, url_vocab=400, img_vocab=603, batch=60, expire=3, **more)
    return p, [BatchSource(p, 3 + r).batch(0) for r in range(world)]


def _same(a, c, tol):
    from gpu_harness import _np, assert_close
    for oa, oc in zip(a.owners, c.owners):
        for name in TABLES:
            x, y = _np(getattr(oa, name)), _np(getattr(oc, name))
            assert np.array_equal(x, y) if x.dtype.kind == "i" else assert_close(x, y, tol, name) is None, name


def test_an_exchange_with_methods_of_its_own_is_used():
    p, batches = _small(2)
    native, by_hand = _jobs(p, 2, p.batch, p.batch * p.img_hi)
    try:
        assert native.step(batches, 1) == by_hand.step(batches, 1)
        assert by_hand.ex.routed == 3 and by_hand._in_process is None
        _same(native, by_hand, 1e-5)
    finally:
        native.close()
        by_hand.close()


def test_a_step_needs_a_batch_for_every_rank_and_whole_arrays():
    p, batches = _small(3)
    (native, by_hand) = _jobs(p, 3, p.batch, p.batch * p.img_hi)
    try:
        for job in (native, by_hand):
            job.step(batches, 1)
            with pytest.raises(IndexError):
                job.step(batches[:2], 2)
        whole = batches[1]
        for name in ("url_id", "img_off", "label"):
            cut = Batch(whole.user_id, whole.url_id, whole.img_off, whole.img_id, whole.label)
            setattr(cut, name, getattr(whole, name)[:-1])
            with pytest.raises(ValueError):
                native.step([batches[0], cut, batches[2]], 2)
        assert native.step(batches, 2) == by_hand.step(batches, 2)
    finally:
        native.close()
        by_hand.close()


def test_ids_beyond_int32_are_not_wrapped_around():
    """An int64 list with an ID of 2^32 + 6: no shard holds it, its row counts as zeros.  (As int32 it would be ID 6.)"""
    p, batches = _small(2)
    native, by_hand = _jobs(p, 2, p.batch, p.batch * p.img_hi)
    try:
        wide = batches[0].user_id.astype(np.int64)
        wide[:] = 2 ** 32 + 6
        odd = Batch(wide, batches[0].url_id, batches[0].img_off, batches[0].img_id, batches[0].label)
        before = native.owners[0].user_emb.clone()
        quiet = Batch(np.full_like(batches[1].user_id, 7), *(getattr(batches[1], n) for n in ("url_id", "img_off", "img_id", "label")))
        assert native.step([odd, quiet], 1) == by_hand.step([odd, quiet], 1)
        assert torch.equal(native.owners[0].user_emb, before)              # (the other rank names ID 7, of owner 1)
        _same(native, by_hand, 1e-5)
        # 64-bit lists that int32 can hold take the short way
        narrow = Batch(batches[0].user_id.astype(np.int64), *(getattr(batches[0], n) for n in ("url_id", "img_off", "img_id", "label")))
        assert native.step([narrow, batches[1]], 2) == by_hand.step([narrow, batches[1]], 2)
        assert native._in_process is not None
        _same(native, by_hand, 1e-5)
    finally:
        native.close()
        by_hand.close()


def test_stores_of_any_m_are_taken():
    """Workers keep no store: what a store of their kind could not take (M from 2^29 on) does not matter to them."""
    p, batches = _small(2, M=1 << 30)
    native, by_hand = _jobs(p, 2, p.batch, p.batch * p.img_hi)
    try:
        got = native.step(batches, 1)
        assert got == by_hand.step(batches, 1) and all(n_ready == 0 for n_ready, _ in got)
        _same(native, by_hand, 1e-5)
        assert sum(int(o.dfv_gcnt.sum()) for o in native.owners) == sum(b.nnz for b in batches)
    finally:
        native.close()
        by_hand.close()


def test_a_closed_job_is_refused():
    from paper_1806_03925_b200 import binding as gb
    p, batches = _small(2)
    for job in _jobs(p, 2, p.batch, p.batch * p.img_hi):
        job.step(batches, 1)
        job.owners[1].close()
        with pytest.raises(gb.GearError) as e:
            job.step(batches, 2)
        assert e.value.code == gb.GEAR_ERR_STATE
        job.close()
        with pytest.raises(gb.GearError) as e:
            job.step(batches, 2)
        assert e.value.code == gb.GEAR_ERR_STATE


@pytest.mark.parametrize("name,world,batch,vocab,mean", [
    ("tiny", 2, 300, 2003, True),               # every sort in one cluster
    ("medium", 2, 12_000, 50_021, True),        # about 38 000 occurrences arrive at an owner: the multi-block sort
    ("medium", 3, 700, 1501, False),
])
def test_seven_steps_against_the_exchange_form(name, world, batch, vocab, mean):
    """The fourth step of a shape makes graphs, the ones after it replay them; a few IDs lie outside every shard.  Sums are taken in
    no fixed order on either side: 1e-5 in fp32, bf16 heads 1e-2."""
    from gpu_harness import _np, assert_close
    p = PRESETS[name].scaled(user_vocab=vocab, url_vocab=vocab - 300, img_vocab=vocab + 11, batch=batch, expire=3, M=3)
    tol = 1e-2 if p.head_dtype == BF16 else 1e-5
    steps = []
    for s in range(7):
        bs = [BatchSource(p, 10 * s + r).batch(0, batch - (31 * r if s != 5 else 17)) for r in range(world)]
        for b in bs:
            b.user_id[:3] = -1, p.user_vocab, -2 ** 31
            b.img_id[5:8] = p.img_vocab, -7, 2 ** 31 - 1
        steps.append(bs)
    native, by_hand = _jobs(p, world, batch, max(b.nnz for bs in steps for b in bs))
    try:
        for s, bs in enumerate(steps):
            got, want = native.step(bs, s + 1, mean_head_grad=mean), by_hand.step(bs, s + 1, mean_head_grad=mean)
            assert got == want, s
            for wa, wc in zip(native.workers, by_hand.workers):
                assert_close(_np(wa.loss), _np(wc.loss), tol, "loss")
                assert_close(_np(wa.head_grad), _np(wc.head_grad), tol, "head_grad")
            for (n_ready, n_exp), oa, oc in zip(got, native.owners, by_hand.owners):
                for field, m in (("ready_ids", n_ready), ("ready_seq", n_ready), ("expired_ids", n_exp)):
                    assert torch.equal(getattr(oa, field)[:m], getattr(oc, field)[:m]), (s, field)
                assert_close(_np(oa.ready_avg[:n_ready]), _np(oc.ready_avg[:n_ready]), tol, "averages")
            _same(native, by_hand, tol)
        from paper_1806_03925_b200 import binding as gb
        for job in (native, by_hand):
            bits = {o.status()[1] for o in job.owners}
            assert gb.GEAR_DEV_BAD_ID in bits and bits <= {0, gb.GEAR_DEV_BAD_ID}
        if mean:
            for w in native.workers[1:]:
                assert torch.equal(w.head_grad, native.workers[0].head_grad)
    finally:
        native.close()
        by_hand.close()
