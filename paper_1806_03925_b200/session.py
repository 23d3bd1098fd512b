"""Device-memory plumbing around the C calls: allocates the tables, the
workspace and the per-step outputs as torch tensors and issues the calls of one
step in order.  No arithmetic of the method happens here.
"""
from __future__ import annotations

from dataclasses import dataclass, field
from typing import Dict, Optional

import numpy as np
import torch

from . import binding as gb
from .workloads import BF16, Batch, GearPreset


_WORD = np.dtype(np.int32)
_NAMES = ("user_id", "url_id", "img_off", "img_id", "label", "fast")
_FAST_FIRST = ("fast",) + _NAMES[:5]                  # the order of a host batch's copy
_TORCH = {np.dtype(np.int32): torch.int32, np.dtype(np.float32): torch.float32}


@dataclass
class DeviceBatch:
    user_id: torch.Tensor
    url_id: torch.Tensor
    img_off: torch.Tensor
    img_id: torch.Tensor
    label: torch.Tensor
    B: int
    nnz: int
    fast: Optional[torch.Tensor] = field(default_factory=lambda: None)       # [B][fast_dim] fp32: the views' own dense input

    # A batch whose copy to the device is still on its way (from_host) has no tensors yet, only what they are made from, in _arriving:
    # whoever asks for one waits for the copy and may use it on any stream; GearSession asks for none and is ordered behind the
    # copy by its stream.
    def __getattr__(self, name):                      # (called for what is not there yet)
        if name in _NAMES and "_arriving" in self.__dict__:
            self._arrive()
        try:
            return self.__dict__[name]
        except KeyError:
            raise AttributeError(name) from None

    def _arrive(self):
        arriving = self.__dict__.get("_arriving")
        if arriving is None:
            return
        raw_stream, there, sizes, dtypes, fast_shape = arriving
        torch.cuda.ExternalStream(raw_stream, there.device).synchronize()
        parts = [t if d == _WORD else t.view(_TORCH.get(d) or getattr(torch, d.name))
                 for d, t in zip(dtypes, there.split_with_sizes(sizes))]
        parts.append(parts.pop(0).view(fast_shape) if fast_shape is not None else None)
        self.__dict__["_c_struct"] = self.__dict__["_c_struct"][0], tuple(parts)
        for name, t in zip(_NAMES, parts):
            self.__dict__.setdefault(name, t)
        self.__dict__.pop("_arriving", None)          # last: a second thread may come here meanwhile

    @staticmethod
    def from_host(b: Batch, device="cuda") -> "DeviceBatch":
        """The batch's arrays on the device: put side by side in pinned memory (torch's pool of it), one copy, and slices of
        what arrives, which is waited for when a tensor is asked for.  (Five copies from pageable memory, each a synchronisation,
        took 80 us for 4096 views.)"""
        arrays = [b.user_id, b.url_id, b.img_off, b.img_id, b.label]
        if b.fast is not None:
            arrays.insert(0, b.fast)                  # first: its rows are read 16 bytes at a time
        if torch.device(device).type != "cuda" or any(a.dtype.itemsize != 4 for a in arrays):
            f = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(device)
            return DeviceBatch(f(b.user_id), f(b.url_id), f(b.img_off), f(b.img_id), f(b.label), b.B, b.nnz,
                               None if b.fast is None else f(b.fast))
        sizes = [a.size for a in arrays]
        host = torch.empty(sum(sizes), dtype=torch.int32, pin_memory=True)
        np.concatenate([(a if a.flags.c_contiguous else np.ascontiguousarray(a)).reshape(-1).view(_WORD) for a in arrays],
                       out=host.numpy())
        there = host.to(device, non_blocking=True)
        # the C struct of the batch: the pointers follow from where the copy went
        c, at = gb.gear_batch(), there.data_ptr()
        for name, n in zip(_NAMES if b.fast is None else _FAST_FIRST, sizes):
            setattr(c, name, at)
            at += 4 * n
        out = DeviceBatch.__new__(DeviceBatch)
        out.__dict__.update(B=b.B, nnz=b.nnz, _c_struct=(c, None),
                            _arriving=(torch._C._cuda_getCurrentRawStream(there.get_device()), there, sizes, [a.dtype for a in arrays],
                                       None if b.fast is None else b.fast.shape))
        return out


class GearSession:
    """Tables + ctx + output buffers for one configuration on one GPU."""

    GUARD_I = -7
    GUARD_F = 12345.0

    def __init__(self, p: GearPreset, head_params: np.ndarray, max_batch: Optional[int] = None,
                 max_nnz: Optional[int] = None, seed: int = 0, fill: bool = True, now: int = 0,
                 tables: Optional[Dict[str, np.ndarray]] = None, ready_cap: int = 0, device: str = "cuda",
                 want_emb_grad: bool = False, want_debug: bool = False, expired_cap: Optional[int] = None,
                 accum_mode: int = gb.GEAR_ACC_SORT, adam: Optional["gb.gear_adam"] = None,
                 scalars: Optional[torch.Tensor] = None):
        """tables: initial contents of user_emb, url_emb, dfv (bf16 as uint16) and ts; a device tensor is used as it is.
        scalars: where the loss and the two counts go (3 x int64), e.g. a part of a larger buffer."""
        gb.load()
        self.p = p
        self.dev = torch.device(device)
        self.max_batch = int(max_batch or p.batch)
        self.max_nnz = int(max_nnz or self.max_batch * p.img_hi)
        self.d_in = p.d_in
        dfv_t = torch.bfloat16 if p.dfv_dtype == BF16 else torch.float32
        self.cfg = gb.make_config(p.user_vocab, p.url_vocab, p.img_vocab, p.emb_dim, p.dfv_dim,
                                  gb.GEAR_BF16 if p.dfv_dtype == BF16 else gb.GEAR_F32,
                                  gb.GEAR_BF16 if p.head_dtype == BF16 else gb.GEAR_F32,
                                  list(p.hidden), p.M, p.expire, self.max_batch, self.max_nnz, ready_cap, accum_mode,
                                  fast_dim=p.fast_dim)
        dev = self.dev
        if tables is None:
            self.user_emb = torch.empty((p.user_vocab, p.emb_dim), dtype=torch.float32, device=dev)
            self.url_emb = torch.empty((p.url_vocab, p.emb_dim), dtype=torch.float32, device=dev)
            self.dfv = torch.empty((p.img_vocab, p.dfv_dim), dtype=dfv_t, device=dev)
            self.dfv_ts = torch.zeros(p.img_vocab, dtype=torch.int64, device=dev)
        else:
            fill = False
            own = lambda t: t if torch.is_tensor(t) else torch.from_numpy(t).to(dev)
            self.user_emb = own(tables["user_emb"])
            self.url_emb = own(tables["url_emb"])
            dfv = tables["dfv"]
            if dfv.dtype == np.uint16:
                self.dfv = torch.from_numpy(dfv.view(np.int16)).to(dev).view(torch.bfloat16)
            else:
                self.dfv = own(dfv)
            assert self.dfv.dtype == dfv_t
            self.dfv_ts = own(tables["ts"])
        self.dfv_gsum = torch.zeros((p.img_vocab, p.dfv_dim), dtype=torch.float32, device=dev)
        self.dfv_gcnt = torch.zeros(p.img_vocab, dtype=torch.int32, device=dev)
        self.head_params = torch.from_numpy(np.ascontiguousarray(head_params, dtype=np.float32)).to(dev)
        assert self.head_params.numel() == p.n_params
        self.workspace = torch.empty(gb.gear_workspace_bytes(self.cfg), dtype=torch.uint8, device=dev)
        self.ctx = gb.gear_init_tables(self.cfg, self.user_emb, self.url_emb, self.dfv, self.dfv_gsum, self.dfv_gcnt,
                                       self.dfv_ts, self.head_params, self.workspace, seed=seed, fill=fill, now=now)
        B, nnz = self.max_batch, self.max_nnz
        # loss and the two counts share one small buffer, so that a caller can read them back with a single copy
        self.scalars = torch.zeros(3, dtype=torch.int64, device=dev) if scalars is None else scalars
        self.loss = self.scalars[0:1].view(torch.float32)[0:1]
        self.prob = torch.zeros(B, dtype=torch.float32, device=dev)
        self.head_grad = torch.zeros(p.n_params, dtype=torch.float32, device=dev)
        self.dX = torch.zeros((B, self.d_in), dtype=torch.float32, device=dev)
        self.row_view = torch.zeros(nnz, dtype=torch.int32, device=dev)
        self.inv_n = torch.zeros(B, dtype=torch.float32, device=dev)
        self.x_debug = (torch.zeros((B, self.d_in), dtype=torch.bfloat16 if p.head_dtype == BF16 else torch.float32,
                                    device=dev) if want_debug else None)
        # event 5's rows in materialised form (what a worker would send to the owners of the images); with want_debug
        self.dfv_grad = torch.zeros((nnz, p.dfv_dim), dtype=torch.float32, device=dev) if want_debug else None
        self.user_grad = torch.zeros_like(self.user_emb) if want_emb_grad else None
        self.url_grad = torch.zeros_like(self.url_emb) if want_emb_grad else None
        # Section 4's optimiser for the embedding tables: first and second moments per table row
        self.adam = adam
        self.adam_step = 0
        self.user_m = torch.zeros_like(self.user_emb) if adam is not None else None
        self.user_v = torch.zeros_like(self.user_emb) if adam is not None else None
        self.url_m = torch.zeros_like(self.url_emb) if adam is not None else None
        self.url_v = torch.zeros_like(self.url_emb) if adam is not None else None
        # every output list is followed by one guard entry the library must never write (guards_intact checks them)
        self.ready_cap = int(ready_cap or nnz)
        self._ready_ids_g = torch.full((self.ready_cap + 1,), self.GUARD_I, dtype=torch.int32, device=dev)
        self._ready_seq_g = torch.full((self.ready_cap + 1,), self.GUARD_I, dtype=torch.int32, device=dev)
        self._ready_avg_g = torch.zeros((self.ready_cap + 1, p.dfv_dim), dtype=torch.float32, device=dev)
        self._ready_avg_g[self.ready_cap].fill_(self.GUARD_F)
        self.ready_ids, self.ready_seq = self._ready_ids_g[:self.ready_cap], self._ready_seq_g[:self.ready_cap]
        self.ready_avg = self._ready_avg_g[:self.ready_cap]
        self.expired_cap = int(expired_cap if expired_cap is not None else p.img_vocab)
        self._expired_ids_g = torch.full((self.expired_cap + 1,), self.GUARD_I, dtype=torch.int32, device=dev)
        self.expired_ids = self._expired_ids_g[:self.expired_cap]
        self.d_counts = self.scalars[1:3]
        self._step_out = self._step_lists = self._lists_at = None

    # ---- the four calls of a step ---------------------------------------------------------------
    def forward_backward(self, b: DeviceBatch, lr: Optional[float] = None):
        o = self._step_out or self._make_step_out()
        if self.adam is not None:
            self.adam_step += 1
            o.adam_step = self.adam_step
        return gb.gear_forward_backward_structs(self.ctx, self._c_batch(b), self.p.lr if lr is None else lr, o)

    # structs are made once: a step's outputs never change, a batch only in its counts
    def _make_step_out(self):
        self._step_out = gb.make_step_out(self.loss, self.head_grad, self.dX, prob=self.prob, row_view=self.row_view,
                                              inv_n=self.inv_n, x_debug=self.x_debug, user_grad=self.user_grad,
                                              url_grad=self.url_grad, dfv_grad=self.dfv_grad, adam=self.adam, user_m=self.user_m,
                                              user_v=self.user_v, url_m=self.url_m, url_v=self.url_v)
        return self._step_out

    def _lists(self):
        """The struct of the output lists, made anew when a program has put other tensors in their place."""
        at = (self.ready_ids.data_ptr(), self.ready_seq.data_ptr(), self.ready_avg.data_ptr(), self.ready_cap,
              self.expired_ids.data_ptr(), self.expired_cap, self.d_counts.data_ptr())
        if at != self._lists_at:
            self._step_lists = gb.make_step_lists(self.ready_ids, self.ready_seq, self.ready_avg, self.ready_cap, self.expired_ids,
                                                  self.expired_cap, d_n=self.d_counts[0:1], d_expired=self.d_counts[1:2])
            self._lists_at = at
        return self._step_lists

    @staticmethod
    def _c_batch(b: DeviceBatch):
        if "_arriving" in b.__dict__:
            if len(b.__dict__) == 4 and b.__dict__["_arriving"][0] == gb._raw_stream(None):      # no tensor has been put in its place
                bt = b.__dict__["_c_struct"][0]
                bt.B, bt.nnz = b.B, b.nnz
                return bt
            b._arrive()
        bt, of = b.__dict__.get("_c_struct", (None, None))
        if bt is None or not (of[0] is b.user_id and of[1] is b.url_id and of[2] is b.img_off and of[3] is b.img_id and
                              of[4] is b.label and of[5] is b.fast):
            of = (b.user_id, b.url_id, b.img_off, b.img_id, b.label, b.fast)
            bt = gb.make_batch(*of[:5], fast=b.fast)
            b.__dict__["_c_struct"] = bt, of
        bt.B, bt.nnz = b.B, b.nnz
        return bt

    def accumulate_from_step(self, b: DeviceBatch, reuse_sorted_ids: bool = True):
        """Event 5 in its indirect form: row r of the batch is dX[row_view[r], 2E:] * inv_n[row_view[r]].
        With reuse_sorted_ids the image IDs sorted during forward_backward are used (img_id = NULL)."""
        if b.nnz == 0:
            return 0
        ptr = self.dX.data_ptr() + 4 * 2 * self.p.emb_dim
        return gb.gear_accumulate_dfv_grad(self.ctx, None if reuse_sorted_ids else b.img_id, ptr, self.d_in,
                                           self.row_view, self.inv_n, b.nnz)

    def accumulate_rows(self, img_id: torch.Tensor, grads: torch.Tensor):
        assert grads.dtype == torch.float32 and grads.shape[1] == self.p.dfv_dim
        return gb.gear_accumulate_dfv_grad(self.ctx, img_id, grads.data_ptr(), grads.stride(0), None, None,
                                           int(img_id.shape[0]))

    def accumulate_collect_from_step(self, b: DeviceBatch, sync: bool = True, reuse_sorted_ids: bool = True):
        """Events 5 and 6 of a step as one call: the batch's gradient rows (indirect form, as in
        accumulate_from_step) are added and the averages of the completed groups handed over."""
        ptr = self.dX.data_ptr() + 4 * 2 * self.p.emb_dim
        return gb.gear_accumulate_collect(self.ctx, None if (reuse_sorted_ids and b.nnz > 0) else b.img_id, ptr, self.d_in,
                                          self.row_view, self.inv_n, b.nnz, self.ready_ids, self.ready_seq,
                                          self.ready_avg, self.ready_cap, d_n=self.d_counts[0:1], sync=sync)

    def accumulate_collect_rows(self, img_id: torch.Tensor, grads: torch.Tensor, sync: bool = True):
        assert grads.dtype == torch.float32 and grads.shape[1] == self.p.dfv_dim
        return gb.gear_accumulate_collect(self.ctx, img_id, grads.data_ptr(), grads.stride(0) if grads.shape[0] else
                                          self.p.dfv_dim, None, None, int(img_id.shape[0]), self.ready_ids, self.ready_seq,
                                          self.ready_avg, self.ready_cap, d_n=self.d_counts[0:1], sync=sync)

    def collect_ready(self, sync: bool = True):
        return gb.gear_collect_ready(self.ctx, self.ready_ids, self.ready_seq, self.ready_avg, self.ready_cap,
                                     d_n=self.d_counts[0:1], sync=sync)

    def collect_expired(self, now: int, restamp: bool = True, sync: bool = True):
        return gb.gear_collect_expired(self.ctx, now, restamp, self.expired_ids, self.expired_cap,
                                       d_n=self.d_counts[1:2], sync=sync)

    def refresh_dfv(self, ids: torch.Tensor, rows: torch.Tensor, now: int, n: Optional[int] = None, d_n=None):
        """Recomputed DFVs replace cached ones (rows fp32) and restart their clocks."""
        return gb.gear_refresh_dfv(self.ctx, ids, rows, int(ids.shape[0]) if n is None else n, now, d_n=d_n)

    # ---- a linear Dense Part on the same device ---------------------------------------------------
    def dense_forward(self, raw: torch.Tensor, Wd: torch.Tensor, ids: torch.Tensor, rows: torch.Tensor, n=None, d_n=None):
        return gb.gear_dense_forward(self.ctx, raw, Wd, ids, int(ids.shape[0]) if n is None else n, rows, d_n=d_n)

    def dense_backward(self, raw: torch.Tensor, n: int, Wd_grad: torch.Tensor, d_n=None):
        """Back-propagation of the averages just handed over (ready_ids, ready_avg) through the Dense Part."""
        return gb.gear_dense_backward(self.ctx, raw, self.ready_ids, self.ready_avg, n, Wd_grad, d_n=d_n)

    def step(self, b: DeviceBatch, now: int, sync: bool = False, expiry_beside: Optional[bool] = None):
        """One pass of the whole hot path over one batch (gear_step).  The expiry scan depends on nothing the training
        calls produce and runs beside them (expiry_beside=False: behind them)."""
        beside = True if expiry_beside is None else expiry_beside
        o, lists = self._step_out or self._make_step_out(), self._lists()
        if self.adam is not None:
            self.adam_step += 1
            o.adam_step = self.adam_step
        return gb.gear_step_structs(self.ctx, self._c_batch(b), self.p.lr, o, lists, now, True, beside, sync)

    def status(self):
        return gb.gear_status(self.ctx)

    def guards_intact(self) -> bool:
        """The entry after the end of each output list still holds the value it was created with."""
        return bool(int(self._ready_ids_g[-1]) == self.GUARD_I and int(self._ready_seq_g[-1]) == self.GUARD_I and
                    int(self._expired_ids_g[-1]) == self.GUARD_I and
                    bool((self._ready_avg_g[-1] == self.GUARD_F).all()))

    def close(self):
        if self.ctx is not None:
            gb.gear_destroy(self.ctx)
            self.ctx = None
