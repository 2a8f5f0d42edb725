"""Gradients around the key tiles of batches of unequal lengths, which are taken by their distance from the end of the
sequence, and at head size 64 around the product kernel's tiles: 128 keys per block, 64 query rows per step, one and many
steps per block, and sink key tiles whose query range is cut into chunks (bounds as in test_prefill_backward_gpu)."""
import pytest

from paper_2512_10411_b200 import inputs
from test_prefill_backward_gpu import run_forward_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seqlens,Hq,Hkv,W,S,full", [
    ((127, 128, 129, 1), 2, 1, 1, 0, True),
    ((63, 64, 65, 256), 8, 2, 64, 4, False),
    ((191, 193), 3, 1, 128, 130, False),
    ((2500,), 2, 1, 100, 4, False),
])
def test_backward_d64_tile_edges(seqlens, Hq, Hkv, W, S, full):
    run_forward_backward(inputs.PrefillConfig(f"bwd64{seqlens}", seqlens, Hq, Hkv, 64, W, S, full, seed=500 + W))


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("W,S,full", [(100, 300, False), (400, 4, False), (1, 0, True)])
def test_backward_unequal_lengths(D, W, S, full):
    # 18, 3, 2, 1, 1 and 0 key tiles; with 300 sink keys three of them are cut into chunks, all of the shorter sequences'
    cfg = inputs.PrefillConfig(f"bwdlen{D}", (130, 2200, 257, 1, 128, 0), 2, 2, D, W, S, full, seed=700 + W)
    run_forward_backward(cfg)
