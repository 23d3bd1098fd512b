"""Products of the head at the edges of their tiles, against the oracle: fp32 heads (three bf16 planes per matrix) at the fp32
tolerance (1e-5 of the largest value of a tensor), bf16 heads at theirs."""
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
    # forward tiles of 16 x 32 up to 148 of them, 32 x 32, 32 x 64 from 119 of those, 64 x 128 from 222 tiles of 64 x 64
    (1184, 4, 16, (64,)), (1185, 4, 16, (64, 40)), (1889, 8, 88, (128,)), (7105, 4, 24, (120, 136)),
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
