"""Performance cases of the Gear Training step: what a user of the package has it do, over the range of sizes.

Kinds of case (the "kind" key):

  step   GearSession.step on batches that are in HBM: events 1, 3, 4 (gather, head forward and backward, embedding
         update), 5 and 6 (gradient store, hand-over of completed groups) and the expiry scan.
  train  a training program around the step: the batch comes from host arrays, the embedding rows and the head take
         Adam steps, the two counts of the step are read back.
  loop   the whole gear loop with a linear Dense Part on the same device: the expiry scan's images are recomputed and
         refreshed, the step runs, the averaged gradients go back through the Dense Part, its weights take an Adam step.
  store  the gradient store alone: (Image ID, gradient row) pairs in, averages of completed groups out.
  shard  the step with the tables partitioned by Image ID, all ranks in this process (host batches, as that API takes).

Every state holds several batches and a pass takes the next one, as a training program does.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1806_03925_b200 import binding as gb
from paper_1806_03925_b200 import workloads
from paper_1806_03925_b200.session import DeviceBatch, GearSession
from paper_1806_03925_b200.sharded import LoopbackExchange, ShardedGear
from paper_1806_03925_b200.workloads import Batch, GearPreset, ZipfIds

N_BATCHES = 4


# ------------------------------------------------------------------------------------------------ the cases
def _step(name, batch, user_vocab, url_vocab, img_vocab, emb_dim, dfv_dim, dtype, hidden1, hidden2, M, expire,
          zipf, zipf_img, img_dist, img_lo, img_hi, img_lambda=0.0, fast_dim=0, kind="step", **more):
    return dict(name=name, kind=kind, batch=batch, user_vocab=user_vocab, url_vocab=url_vocab, img_vocab=img_vocab,
                emb_dim=emb_dim, dfv_dim=dfv_dim, dtype=dtype, hidden1=hidden1, hidden2=hidden2, M=M, expire=expire,
                zipf=zipf, zipf_img=zipf_img, img_dist=img_dist, img_lo=img_lo, img_hi=img_hi, img_lambda=img_lambda,
                fast_dim=fast_dim, **more)


def _store(name, rows, img_vocab, dfv_dim, M, zipf_img, mode):
    return dict(name=name, kind="store", rows=rows, img_vocab=img_vocab, dfv_dim=dfv_dim, M=M, zipf_img=zipf_img, mode=mode)


def listed():
    return [
        # the smallest configuration (preset "tiny"): a handful of page views per step, where launches count
        _step("step_tiny_f32", 256, 10_000, 10_000, 5_000, 16, 64, "f32", 64, 0, 4, 1000, 1.1, 1.1, "uniform", 1, 4),
        # an ordinary step (preset "medium"): bf16 vectors and head
        _step("step_medium_bf16", 4096, 1_000_000, 1_000_000, 1_000_000, 32, 128, "bf16", 256, 128, 16, 100, 1.05, 1.05,
              "poisson", 1, 8, 3.0),
        # the largest step (preset "large"): the configuration the headline is quoted on
        _step("step_large_bf16", 65_536, 50_000_000, 20_000_000, 20_000_000, 64, 256, "bf16", 512, 256, 32, 100, 1.05, 1.05,
              "poisson", 1, 16, 4.0),
        # fp32 vectors and head, image IDs so skewed that a hundred images take most gradients (preset "skew")
        _step("step_skew_f32", 32_768, 1_000_000, 1_000_000, 4_000_000, 32, 128, "f32", 256, 128, 64, 10, 1.05, 1.3,
              "poisson", 1, 8, 3.0),
        # a model whose widths fit no tile and the ragged last batch of an epoch, bf16
        _step("step_ragged_bf16", 3001, 30_011, 20_021, 40_009, 20, 200, "bf16", 320, 192, 3, 50, 1.05, 1.05,
              "poisson", 1, 8, 3.0),
        # the same in fp32, one hidden layer
        _step("step_ragged_f32", 1237, 50_021, 50_023, 50_033, 24, 72, "f32", 136, 0, 8, 10, 1.05, 1.3, "poisson", 1, 8, 3.0),
        # a training program on preset "medium": host batches, Adam on embeddings and head, counts read every step
        _step("train_medium_bf16", 4096, 1_000_000, 1_000_000, 1_000_000, 32, 128, "bf16", 256, 128, 16, 100, 1.05, 1.05,
              "poisson", 1, 8, 3.0, kind="train"),
        # the shape of the paper's CIFAR100 experiment (preset "split_image"): the top half of a 32x32x3 image (1536 values)
        # is the Fastgear side's own input, the bottom half (1536 values) goes through the Dense Part
        _step("loop_split_image_f32", 1024, 10_000, 10_000, 50_000, 16, 64, "f32", 256, 64, 4, 20, 1.1, 1.05, "uniform", 1, 1,
              fast_dim=1536, kind="loop", raw_dim=1536),
        # the accumulate-only benchmark: 16M gradient rows, Zipf IDs, M = 8
        _store("store_zipf_16m", 1 << 24, 1 << 22, 128, 8, 1.1, "sort"),
        # a million rows, uniform IDs, few completed groups
        _store("store_uniform_1m", 1_000_003, 1 << 22, 128, 64, 0.0, "sort"),
        # the order-free store under contention: the rows of one step of preset "skew"
        _store("store_atomic_skew", 99_700, 4_000_000, 128, 64, 1.3, "atomic"),
        # tables partitioned by ID over two ranks, preset "medium"
        _step("shard_medium_2ranks", 4096, 1_000_000, 1_000_000, 1_000_000, 32, 128, "bf16", 256, 128, 16, 100, 1.05, 1.05,
              "poisson", 1, 8, 3.0, kind="shard", world=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: bf16 steps up to preset "large", fp32 steps up to preset "skew"."""
    kind = rng.choice(["step", "step", "step", "step", "train", "loop", "store", "store", "shard"])
    if kind == "store":
        dim = 8 * rng.randint(8, 32)
        mode = rng.choice(["sort", "sort", "atomic"])
        rows = _log_int(rng, 1000, min(1 << 24, (1 << 31) // dim) if mode == "sort" else 1 << 20)
        c = _store("", rows, _log_int(rng, 10_000, 1 << 22), dim, _log_int(rng, 1, 1024) if rows < 1 << 20 else _log_int(rng, 8, 1024),
                   rng.choice([0.0, 1.05, 1.1, 1.3]), mode)
    else:
        bf16 = kind == "shard" or rng.random() < 0.6
        loop = kind == "loop"
        wide = kind == "step" and bf16
        q = 64 if bf16 else 8                                   # hidden widths: multiples the head takes
        h1, h2 = q * rng.randint(1, (512 if wide else 256) // q), q * rng.randint(1, (256 if wide else 128) // q)
        vmax = 20_000_000 if wide else 4_000_000 if kind == "step" else 1_000_000
        lam = rng.choice([0.0, 3.0, 4.0] if wide else [0.0, 3.0])
        c = _step("", _log_int(rng, 64, 65_536 if wide else 32_768 if kind == "step" else 4096),
                  _log_int(rng, 5000, 2 * vmax), _log_int(rng, 5000, vmax), _log_int(rng, 2000, 50_000) if loop else _log_int(rng, 5000, vmax),
                  4 * rng.randint(2, 16 if wide else 8), 8 * rng.randint(6, 32 if wide else 16), "bf16" if bf16 else "f32",
                  h1, rng.choice([0, h2]), _log_int(rng, 1, 64), rng.randint(5, 200), rng.choice([1.05, 1.1]),
                  rng.choice([1.05, 1.1, 1.3]), "poisson" if lam else "uniform", 1, 16 if lam == 4.0 else 8 if lam else 4, lam,
                  fast_dim=1536 if loop else 0, kind=kind)
        if loop:
            c["raw_dim"] = 1536
        if kind == "shard":
            c["world"] = rng.randint(2, 4)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=12)
def _zipf(vocab, s):
    return ZipfIds(vocab, s)


@functools.lru_cache(maxsize=6)
def _zipf_cdf(vocab, s):
    return torch.from_numpy(_zipf(vocab, s)._table()).cuda()


def _ids(vocab, s, n, gen):
    """n IDs on the GPU, Zipf(s) over the vocabulary with the hot ones scattered (ZipfIds' mapping); s = 0: uniform."""
    if s == 0.0:
        return torch.randint(0, vocab, (n,), generator=gen, device="cuda", dtype=torch.int32)
    u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    rank = torch.searchsorted(_zipf_cdf(vocab, s), u).clamp_(max=vocab - 1)
    z = _zipf(vocab, s)
    return ((rank * z.a + z.c) % vocab).to(torch.int32)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & (2**63 - 1))
    return g


def _batches(c, seed, count):
    """Page views in CSR form on the GPU: IDs Zipf, images per view uniform or clipped Poisson, one label in twenty."""
    gen, out = _gen(seed), []
    for _ in range(count):
        B = c["batch"]
        if c["img_dist"] == "uniform":
            n = torch.randint(c["img_lo"], c["img_hi"] + 1, (B,), generator=gen, device="cuda")
        else:
            n = torch.poisson(torch.full((B,), c["img_lambda"], device="cuda"), generator=gen).clamp_(c["img_lo"], c["img_hi"])
        off = torch.zeros(B + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(n.to(torch.int64), 0, out=off[1:])
        nnz = int(off[-1])
        fast = torch.rand((B, c["fast_dim"]), generator=gen, device="cuda") - 0.5 if c["fast_dim"] else None
        out.append(DeviceBatch(_ids(c["user_vocab"], c["zipf"], B, gen), _ids(c["url_vocab"], c["zipf"], B, gen),
                               off.to(torch.int32), _ids(c["img_vocab"], c["zipf_img"], nnz, gen),
                               (torch.rand(B, generator=gen, device="cuda") < 0.05).to(torch.float32), B, nnz, fast))
    return out


def _on_host(b):
    f = lambda t: None if t is None else t.cpu().numpy()
    return Batch(f(b.user_id), f(b.url_id), f(b.img_off), f(b.img_id), f(b.label), f(b.fast))


def _preset(c):
    return GearPreset(name=c["kind"], batch=c["batch"], steps=1, user_vocab=c["user_vocab"], url_vocab=c["url_vocab"],
                      img_vocab=c["img_vocab"], emb_dim=c["emb_dim"], dfv_dim=c["dfv_dim"], dfv_dtype=c["dtype"],
                      head_dtype=c["dtype"], hidden=(c["hidden1"], c["hidden2"]) if c["hidden2"] else (c["hidden1"],),
                      M=c["M"], expire=c["expire"], zipf_user=c["zipf"], zipf_url=c["zipf"], zipf_img=c["zipf_img"],
                      img_dist=c["img_dist"], img_lo=c["img_lo"], img_hi=c["img_hi"], img_lambda=c["img_lambda"],
                      fast_dim=c["fast_dim"])


def _views_mean(c):
    lo, hi, lam = c["img_lo"], c["img_hi"], c["img_lambda"]
    if c["img_dist"] == "uniform":
        return (lo + hi) / 2
    total, mean, k, pk = 0.0, 0.0, 0, math.exp(-lam)
    while k < 100:
        mean += pk * min(max(k, lo), hi)
        total += pk
        k += 1
        pk *= lam / k
    return mean + (1 - total) * hi


def _max_nnz(c):
    """Image occurrences the program makes room for: a tenth above the mean of a batch, and a little for small batches."""
    return int(1.1 * _views_mean(c) * c["batch"]) + 256


class _State:
    """What the program keeps between passes; the session's ctx goes with it."""

    def __init__(self, kind):
        self.kind, self.now, self.session = kind, 0, None

    def next(self):
        """The pass's time step and batch."""
        self.now += 1
        return self.now, self.batches[(self.now - 1) % len(self.batches)]

    def __del__(self):
        if self.session is not None:
            self.session.close()


def prepare(case, seed):
    c, st = case, _State(case["kind"])
    if st.kind == "store":
        gen = _gen(seed)
        st.batches = [_ids(c["img_vocab"], c["zipf_img"], c["rows"], gen) for _ in range(2)]
        p = workloads.PRESETS["skew"].scaled(img_vocab=c["img_vocab"], dfv_dim=c["dfv_dim"], M=c["M"], user_vocab=64,
                                             url_vocab=64, expire=1 << 40)
        # room for every group that can complete: all full groups plus one for each image with an open one
        cap = 2 * c["rows"] if c["mode"] == "atomic" else c["rows"] // c["M"] + min(c["rows"], c["img_vocab"])
        st.session = GearSession(p, np.zeros(p.n_params, np.float32), max_batch=8, max_nnz=c["rows"], ready_cap=cap, seed=seed,
                                 expired_cap=1, accum_mode=gb.GEAR_ACC_ATOMIC if c["mode"] == "atomic" else gb.GEAR_ACC_SORT)
        st.grads = torch.empty((c["rows"], c["dfv_dim"]), device="cuda")
        gb.gear_fill_uniform(st.grads, seed=seed, tag=gb.GEAR_TAG_GRAD, amp=1.0)
        return st
    p, params = _preset(c), workloads.head_params(_preset(c), seed)
    if st.kind == "shard":
        W = c["world"]
        bs = [_on_host(b) for b in _batches(c, seed, W * N_BATCHES)]
        st.batches = [bs[i * W:(i + 1) * W] for i in range(N_BATCHES)]
        st.session = ShardedGear(p, params, LoopbackExchange(W), max_batch_local=p.batch, max_nnz_local=_max_nnz(c), seed=seed)
        return st
    st.batches = _batches(c, seed, N_BATCHES)
    st.adam = gb.make_adam()
    s = st.session = GearSession(p, params, max_batch=p.batch, max_nnz=_max_nnz(c), seed=seed,
                                 adam=st.adam if st.kind == "train" else None)
    if st.kind == "train":
        st.batches = [_on_host(b) for b in st.batches]
        st.m, st.v = torch.zeros_like(s.head_params), torch.zeros_like(s.head_params)
    if st.kind == "loop":
        gen, R = _gen(seed + 1), c["raw_dim"]
        st.raw = torch.rand((p.img_vocab, R), generator=gen, device="cuda") - 0.5        # "pixels", as in BatchSource
        st.Wd = (torch.rand((R, p.dfv_dim), generator=gen, device="cuda") - 0.5) * (2 * math.sqrt(3.0 / R))
        st.m, st.v, st.Wd_grad = torch.zeros_like(st.Wd), torch.zeros_like(st.Wd), torch.zeros_like(st.Wd)
        st.rows = torch.zeros((p.img_vocab, p.dfv_dim), device="cuda")
    return st


# ------------------------------------------------------------------------------------------------ one pass
def _results(s):
    """The step's outputs and the tables it updates."""
    return dict(loss=s.loss, prob=s.prob, head_grad=s.head_grad, dX=s.dX, user_emb=s.user_emb, url_emb=s.url_emb,
                gsum=s.dfv_gsum, gcnt=s.dfv_gcnt, ts=s.dfv_ts, counts=s.d_counts, ready_ids=s.ready_ids,
                ready_seq=s.ready_seq, ready_avg=s.ready_avg, expired_ids=s.expired_ids)


def run(state):
    s, kind = state.session, state.kind
    now, batch = state.next()
    if kind == "step":
        s.step(batch, now)
        return _results(s)
    if kind == "train":
        s.step(DeviceBatch.from_host(batch), now, sync=True)
        gb.gear_adam_dense(s.head_params, s.head_grad, state.m, state.v, now, state.adam)
        return dict(_results(s), user_m=s.user_m, user_v=s.user_v, url_m=s.url_m, url_v=s.url_v,
                    params=s.head_params, params_m=state.m, params_v=state.v)
    if kind == "loop":
        V = s.p.img_vocab
        s.collect_expired(now, restamp=True, sync=False)
        s.dense_forward(state.raw, state.Wd, s.expired_ids, state.rows, n=V, d_n=s.d_counts[1:2])
        s.refresh_dfv(s.expired_ids, state.rows, now, n=V, d_n=s.d_counts[1:2])
        s.forward_backward(batch)
        s.accumulate_collect_from_step(batch, sync=False)
        state.Wd_grad.zero_()
        s.dense_backward(state.raw, batch.nnz, state.Wd_grad, d_n=s.d_counts[0:1])
        gb.gear_adam_dense(state.Wd, state.Wd_grad, state.m, state.v, now, state.adam)
        return dict(_results(s), dfv=s.dfv, Wd=state.Wd, Wd_grad=state.Wd_grad, Wd_m=state.m, Wd_v=state.v)
    if kind == "store":
        s.accumulate_collect_rows(batch, state.grads, sync=False)
        return dict(gsum=s.dfv_gsum, gcnt=s.dfv_gcnt, count=s.d_counts[0:1], ids=s.ready_ids, seq=s.ready_seq, avg=s.ready_avg)
    counts = s.step(batch, now)
    keep = ("user_emb", "url_emb", "dfv_gsum", "dfv_gcnt", "dfv_ts", "ready_ids", "ready_seq", "ready_avg", "expired_ids")
    return dict(counts=counts, owners=[{k: getattr(o, k) for k in keep} for o in s.owners],
                workers=[dict(loss=w.loss, prob=w.prob, head_grad=w.head_grad) for w in s.workers])


# ------------------------------------------------------------------------------------------------ work, tolerance
@functools.lru_cache(maxsize=64)
def _distinct(vocab, s, n):
    """Expected number of distinct IDs among n draws."""
    if s == 0.0:
        return vocab * -math.expm1(n * math.log1p(-1.0 / vocab)) if vocab > 1 else 1.0
    p = np.diff(_zipf(vocab, s)._table(), prepend=0.0)
    return float(-np.expm1(n * np.log1p(-np.minimum(p, 1 - 1e-12))).sum())


def work(case):
    """Bytes: every table row, input and output of the pass once (a row that is updated: read and written); the head's
    intermediate matrices are not counted.  Flops: the head's products, forward and backward, and the Dense Part's."""
    c = case
    if c["kind"] == "store":
        n, D = c["rows"], c["dfv_dim"]
        return {"bytes": n * (D * 4 + 4) + _distinct(c["img_vocab"], c["zipf_img"], n) * (D * 4 + 4) * 2 + n / c["M"] * (D * 4 + 8), "flops": n * D}
    p, W = _preset(c), c.get("world", 1)
    B, E, D, nnz = p.batch * W, p.emb_dim, p.dfv_dim, _views_mean(c) * p.batch * W
    dsz = 2 if c["dtype"] == "bf16" else 4
    u_emb = _distinct(p.user_vocab, p.zipf_user, B) + _distinct(p.url_vocab, p.zipf_url, B)
    u_img = _distinct(p.img_vocab, p.zipf_img, int(nnz))
    expired = p.img_vocab / max(p.expire, 1)
    out = {"bytes": B * (4 * 4 + p.fast_dim * 4) + nnz * 4 + u_img * D * dsz                             # views, vectors
                    + u_emb * E * 4 * (6 if c["kind"] == "train" else 2)                                 # embeddings, moments
                    + W * p.n_params * 4 * (8 if c["kind"] == "train" else 2)                            # head
                    + B * (p.d_in * 4 + 4) + nnz * 4 + B * 4                                             # dX, prob, row_view, 1/n
                    + u_img * (D * 4 + 4) * 2 + nnz / p.M * (D * 4 + 8)                                  # store, averages
                    + p.img_vocab * 8 + expired * 12,                                                    # expiry scan
           "flops": 6.0 * B * sum(a * b for a, b in zip((p.d_in,) + p.hidden, p.hidden + (1,)))}
    if c["kind"] == "loop":
        R, emitted = c["raw_dim"], nnz / p.M
        out["bytes"] += expired * (R * 4 + D * dsz) + emitted * R * 4 + R * D * 4 * 7
        out["flops"] += 2.0 * R * D * (expired + emitted)
    return out


def tolerance(case):
    """Sums in fp32: 1e-5; products with bf16 operands: 1e-2.  A hidden unit whose pre-activation is within rounding of
    zero may take either branch of the ReLU, which moves its view's gradient as a whole; in fp32 that is one unit in about
    2^22, so a norm moves by sqrt(2 * 2^-21) = 1e-3 once a batch has enough units for one to be expected.  "max" is wide
    for the same reason, and because most rows of a table are ones the pass never touched (zero), so that an entry is
    measured against itself, cancellation included."""
    if case["kind"] == "store":
        return {"rel": 1e-5}
    if case["dtype"] == "bf16":
        return {"rel": 1e-2, "max": 0.9}
    units = case["batch"] * (case["hidden1"] + case["hidden2"])
    return {"rel": 1e-3 if units > 1 << 16 else 1e-5, "max": 0.9}
