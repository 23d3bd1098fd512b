"""Products of the head at the edges of their tiles, against the oracle: fp32 heads (three bf16 planes per matrix) at the fp32
tolerance (1e-5 of the largest value of a tensor), bf16 heads at theirs."""
import numpy as np
import pytest
import torch

from paper_1806_03925_b200.workloads import BF16, F32, PRESETS, BatchSource

pytestmark = pytest.mark.gpu


# row tiles are 128 views, column tiles 64 or 128 wide, the reduction goes in steps of 32 and is cut into segments of 256
# terms from 544 on; weight gradients reduce over the batch
@pytest.mark.parametrize("B,E,D,hidden", [
    (1, 4, 8, (8,)),                        # one view, narrowest layers: one tile, most of it past the edge
    (127, 12, 40, (64,)), (129, 12, 48, (72, 8)),          # one row short of / past a tile; 64 and 72 columns
    (256, 16, 480, (136, 120)),             # head input 512 wide: two segments' worth in one, columns one step past 128
    (640, 16, 512, (128, 64)),              # head input 544 wide: the first width that is cut into segments
    (20_000, 4, 24, (1024,)),               # widest layer, a long reduction over the batch
    # one hidden layer, and two of changing width, around whole numbers of blocks per SM in the forward products
    (1184, 4, 16, (64,)), (1185, 4, 16, (64, 40)), (1889, 8, 88, (128,)), (7105, 4, 24, (120, 136)),
    (2368, 4, 24, (64,)), (2369, 4, 24, (64, 40)), (14_144, 4, 24, (128,)), (14_145, 4, 24, (120, 136)),
])
def test_fp32_products_at_tile_edges(B, E, D, hidden):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_harness import Pair
    p = PRESETS["skew"].scaled(emb_dim=E, dfv_dim=D, dfv_dtype=F32, head_dtype=F32, hidden=hidden, M=3, user_vocab=3000,
                               url_vocab=2000, img_vocab=4000, expire=2)
    batch = BatchSource(p, B).batch(0, B)
    pair = Pair(p, [batch], seed=1, want_emb_grad=True)
    try:
        pair.step_and_compare(batch, now=1)
    finally:
        pair.close()


# the same in a shallow layer (one step of the operand ring), around whole numbers of blocks per SM in tiles of 8 to 64 rows and 32 to 256
# columns, where the forms of a tile change; more than 256 columns: the output unit in a launch of its own
@pytest.mark.parametrize("B,hidden", [
    (4736, (24,)), (4737, (32,)), (9472, (64,)), (9473, (40,)), (1184, (128,)), (1185, (72,)), (7104, (128, 120)), (7105, (128, 72)),
    (3552, (256,)), (3553, (136,)), (300, (264,)), (14_208, (64, 8)), (14_209, (64, 16)),
])
def test_fp32_forward_forms(B, hidden):
    test_fp32_products_at_tile_edges(B, 4, 24, hidden)


def _off_by_one_float(t):
    out = torch.empty(t.numel() + 1, device=t.device)[1:].view(t.shape)
    assert out.data_ptr() % 16 == 4
    return out.copy_(t)


def _with_params_off(s):
    """The session's ctx made anew with head parameters that start 4 bytes past a 16-byte boundary (fp32 heads take any address)."""
    from paper_1806_03925_b200 import binding as gb
    gb.gear_destroy(s.ctx)
    s.head_params = _off_by_one_float(s.head_params)
    s.ctx = gb.gear_init_tables(s.cfg, s.user_emb, s.url_emb, s.dfv, s.dfv_gsum, s.dfv_gcnt, s.dfv_ts, s.head_params, s.workspace, fill=False)


# Every form of a forward tile, 304 terms deep (nine and a half steps of the operand ring), on batches that end inside a tile:
# weights read 16 bytes at a time and one by one.
@pytest.mark.parametrize("off", [False, True])
@pytest.mark.parametrize("B,hidden", [
    (33, (24,)), (7107, (32,)), (1001, (64,)), (1193, (40,)), (11_847, (64,)), (1001, (128,)), (1193, (72,)), (7107, (128,)),     # with the output unit
    (1777, (256,)), (7107, (256,)),
    (301, (136,)), (1777, (136,)), (11_363, (136,)), (10_061, (256,)),                                                # the output unit behind it
    (300, (64, 8)), (1889, (128, 8)), (14_213, (128, 8)), (16_579, (64, 8)),                                          # a layer above
])
def test_fp32_forward_forms_in_deep_layers(B, hidden, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_harness import Pair
    p = PRESETS["skew"].scaled(emb_dim=4, dfv_dim=296, dfv_dtype=F32, head_dtype=F32, hidden=hidden, M=3, user_vocab=3000,
                               url_vocab=2000, img_vocab=4000, expire=2)
    batch = BatchSource(p, B).batch(0, B)
    pair = Pair(p, [batch], seed=1, want_emb_grad=True)
    try:
        if off:
            _with_params_off(pair.gpu)
        pair.step_and_compare(batch, now=1)
    finally:
        pair.close()


# the Dense Part's products over more steps than the ring of four has buffers, with rows and weights off a 16-byte boundary or not
@pytest.mark.parametrize("raw_off,w_off", [(False, False), (False, True), (True, False), (True, True)])
@pytest.mark.parametrize("n,R,D", [(33, 300, 72), (2401, 288, 64), (31, 301, 8)])
def test_dense_forward_of_unaligned_operands(n, R, D, raw_off, w_off):
    """Against fp64; R products of values in (-1, 1) added one by one in fp32 are off by at most R * 2^-24 * R.  An ID out of range
    gives a row of zeros."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_03925_b200 import workloads
    from paper_1806_03925_b200.session import GearSession
    p = PRESETS["tiny"].scaled(user_vocab=64, url_vocab=64, img_vocab=500, dfv_dim=D)
    s = GearSession(p, workloads.head_params(p, 0), max_batch=8, max_nnz=32)
    try:
        rng = np.random.default_rng(R)
        raw, Wd = rng.uniform(-1, 1, (500, R)).astype(np.float32), rng.uniform(-1, 1, (R, D)).astype(np.float32)
        ids = rng.integers(0, 500, n).astype(np.int32)
        ids[::7] = -1
        ids[5] = 500
        at = lambda a, off: _off_by_one_float(torch.from_numpy(a).cuda()) if off else torch.from_numpy(a).cuda()
        rows = torch.full((n, D), 7.0, device="cuda")
        s.dense_forward(at(raw, raw_off), at(Wd, w_off), torch.from_numpy(ids).cuda(), rows, n=n)
        ok = (ids >= 0) & (ids < 500)
        want = raw[np.where(ok, ids, 0)].astype(np.float64) @ Wd.astype(np.float64) * ok[:, None]
        np.testing.assert_allclose(rows.cpu().numpy(), want, rtol=0, atol=R * R * 2.0 ** -24)
        assert s.status()[1] == 1
    finally:
        s.close()


# column tiles are 64 wide while 64-column tiles are no more than the SMs (148), then 128, then 256 (dX: 192 where that fits);
# weight gradients take 64 to 256 columns and cut the batch into slices
@pytest.mark.parametrize("B,E,D,hidden", [
    (1, 4, 8, (64,)), (127, 12, 40, (512,)), (129, 12, 48, (64, 128)),     # one view; a row short of / past a tile
    (4736, 16, 96, (256, 192)), (4737, 16, 96, (256, 192)),                # 37 row tiles x 4 = 148 tiles of 64 columns, and more
    (9472, 32, 128, (256, 64)), (9473, 32, 128, (256, 64)),                # the same at 128 columns; dX 192 wide
    (18_945, 4, 24, (128, 64)), (20_000, 64, 256, (1024,)),                # several tiles per block
])
def test_bf16_products_at_tile_edges(B, E, D, hidden):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_harness import Pair
    p = PRESETS["medium"].scaled(emb_dim=E, dfv_dim=D, dfv_dtype=BF16, head_dtype=BF16, hidden=hidden, M=3, user_vocab=3000,
                                 url_vocab=2000, img_vocab=4000, expire=2)
    batch = BatchSource(p, B).batch(0, B)
    pair = Pair(p, [batch], seed=1, want_emb_grad=True)
    try:
        pair.step_and_compare(batch, now=1)
    finally:
        pair.close()


@pytest.mark.parametrize("bias", [float("inf"), 3.4e38, -float("inf")])
@pytest.mark.parametrize("head", [F32, BF16])
def test_units_beyond_the_largest_value(head, bias):
    """One unit of the top layer saturated by its bias: infinite, or finite but above the largest bf16 value (3.39e38), which counts
    as infinite.  The views' probabilities and all gradients but the unit's own output weight are finite: 1e-5 of
    the largest value against fp64, bf16 1e-2."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_03925_b200 import workloads
    from paper_1806_03925_b200.session import DeviceBatch, GearSession
    p = PRESETS["tiny"].scaled(dfv_dtype=head, head_dtype=head, hidden=(128, 64))
    b = BatchSource(p, 3).batch(0)
    params = workloads.head_params(p, 3)
    n0, n1 = p.d_in * 128 + 128, 128 * 64
    params[n0 + n1 + 5] = bias
    w_out = params[n0 + n1 + 64:-1]
    w_out[5] = 1e-38
    s = GearSession(p, params, max_nnz=b.nnz, seed=3, want_debug=True, want_emb_grad=True)
    try:
        s.forward_backward(DeviceBatch.from_host(b))
        t = [torch.from_numpy(a.astype(np.float64)).requires_grad_() for a in
             (params[:n0 - 128].reshape(p.d_in, 128), params[n0 - 128:n0], params[n0:n0 + n1].reshape(128, 64),
              params[n0 + n1:n0 + n1 + 64], w_out, params[-1:])]
        rnd = (lambda v: v) if head == F32 else (lambda v: v + (v.to(torch.bfloat16).to(torch.float64) - v).detach().nan_to_num(0.0))
        x = s.x_debug.double().cpu().requires_grad_()
        h = rnd(torch.relu(x @ rnd(t[0]) + t[1]))
        h = rnd(torch.relu(h @ rnd(t[2]) + t[3]))
        h = torch.where(h > 3.39e38, torch.full_like(h, float("inf")), h)
        z = h @ t[4] + t[5]
        y = torch.from_numpy(b.label).double()
        prob = torch.sigmoid(z)
        dz = ((prob - y) / b.B).detach()
        z.backward(dz)                                               # dLoss/dz is p - y, also where the loss is not finite
        tol = 1e-5 if head == F32 else 1e-2
        close = lambda got, want: np.testing.assert_allclose(got, want, rtol=0, atol=tol * max(np.abs(want).max(), 1e-30))
        close(s.prob[:b.B].cpu().numpy(), prob.detach().numpy())
        grads = [a.grad.numpy().ravel() for a in t]
        got = s.head_grad.cpu().numpy()
        own = n0 + n1 + 64 + 5
        assert np.isfinite(got[own]) == np.isfinite(grads[4][5])
        if np.isfinite(got[own]):
            np.testing.assert_allclose(got[own], grads[4][5], rtol=1e-4 if head == F32 else 1e-2)
        want = np.concatenate(grads)
        got[own] = want[own] = 0.0
        for lo, hi in ((0, n0 - 128), (n0 - 128, n0), (n0, n0 + n1), (n0 + n1, n0 + n1 + 64), (n0 + n1 + 64, want.size)):
            close(got[lo:hi], want[lo:hi])
        close(s.dX[:b.B].cpu().numpy(), x.grad.numpy())
    finally:
        s.close()
