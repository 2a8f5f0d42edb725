"""GPU parity of the prefill kernel's work items where they can go wrong: sequences around the size that is packed into
one item per kv head, batches of more sequences than one look of the scheduler covers, tiles that join band and sink
keys, a few sink keys in a tile of their own, and scores that outgrow the exponent range of the reference within one tile
(the item is then run again)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_10411_b200 import inputs
from helpers import check_against_oracle
from test_prefill_chunked_gpu import make, run_chunked
from test_prefill_gpu import run_prefill

pytestmark = pytest.mark.gpu


def _check(lq, lk, Hq, Hkv, D, W, S, full, seed, scale=0.0):
    q, k, v = make(lq, lk, Hq, Hkv, D, seed)
    out, lse, status = run_chunked(q, k, v, lq, lk, W, S, full, scale)
    assert status == 0
    ref = oracle.prefill_chunked(*(inputs.to_f32_numpy(t) for t in (q, k, v)), np.concatenate([[0], np.cumsum(lq)]),
                                 np.concatenate([[0], np.cumsum(lk)]), W, S, full, scale=scale if scale > 0 else None)
    check_against_oracle(out, ref["out"], f"{lq[:4]} {lk[:4]} Hq={Hq} Hkv={Hkv} D={D} W={W} S={S} full={full}")
    np.testing.assert_allclose(lse.cpu().numpy().T, ref["lse"], rtol=0, atol=2e-3)


@pytest.mark.parametrize("Hq,Hkv,D", [(2, 2, 128), (4, 2, 64), (7, 1, 128), (16, 2, 128), (128, 1, 64), (130, 1, 128)])
def test_sequences_around_the_packed_size(Hq, Hkv, D):
    n = 128 // (Hq // Hkv)  # tokens that fill an item's rows (0: never packed)
    lq = (max(n - 1, 1), max(n, 1), n + 1, 1, 1)
    lk = (max(n - 1, 1), max(n, 1) + 300, n + 1 + 77, 1, 513)
    for W, S, full in ((1, 0, True), (128, 4, False), (100, 20, False), (33, 140, False), (1, 1, False)):
        _check(lq, lk, Hq, Hkv, D, W, S, full, seed=40 + n)


def test_more_sequences_than_one_look_of_the_scheduler():
    rng = np.random.default_rng(3)
    lq = tuple(int(x) for x in rng.integers(1, 200, 70))
    lk = tuple(a + int(x) for a, x in zip(lq, rng.integers(0, 200, 70)))
    _check(lq, lk, 4, 2, 128, 100, 4, False, seed=60)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("S", [1, 16, 31, 32, 33, 160])
def test_few_sink_keys_in_a_tile_of_their_own(D, S):
    # window 128: the band fills its two tiles exactly, so the sink keys start one; 160 leaves 32 for the second.  The
    # large scale makes them outgrow the reference of the band keys.
    lens = (300, 129, 517, 40)
    q, k, v = make(lens, lens, 3, 1, D, 90 + S)
    cu = np.concatenate([[0], np.cumsum(lens)])
    for W, scale in ((128, 0.0), (128, 4.0), (112, 0.0)):
        out, lse, status = run_prefill(q, k, v, torch.tensor(cu, dtype=torch.int32, device="cuda"), max(lens), W, S, False, scale)
        assert status == 0
        ref = oracle.prefill(*(inputs.to_f32_numpy(t) for t in (q, k, v)), cu, W, S, False, scale=scale if scale > 0 else None)
        check_against_oracle(out, ref["out"], f"D={D} W={W} S={S} scale={scale}")
        np.testing.assert_allclose(lse.cpu().numpy().T, ref["lse"], rtol=0, atol=2e-3)


@pytest.mark.parametrize("Hq,Hkv", [(24, 8), (32, 8), (12, 12), (9, 3)])  # with 13 tiles at most: two heads per item but for 9
@pytest.mark.parametrize("D", [64, 128])
def test_one_and_two_heads_per_item(Hq, Hkv, D):
    lq, lk = (300, 1, 129, 128, 517), (300, 70, 400, 128, 600)
    for W, S, full in ((1, 0, True), (128, 4, False), (200, 130, False)):
        _check(lq, lq, Hq, Hkv, D, W, S, full, seed=120 + Hq)
        _check(lq, lk, Hq, Hkv, D, W, S, full, seed=121 + Hq)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("scale", [4.0, 30.0])
def test_scores_that_leave_the_exponent_range_of_the_reference(D, scale):
    # |scaled scores| reach 4 * 45 = 180 and 30 * 45 = 1350: from one key tile to the next the largest one of a row grows
    # by far more than 60 in log2 units.  Tolerances as everywhere: the products are exact in fp32 to 2^-23 * 1350 = 2e-4.
    for lq, lk in (((700,), (700,)), ((1, 30, 129), (900, 430, 1000))):
        for W, S, full in ((1, 0, True), (300, 4, False)):
            _check(lq, lk, 4, 1, D, W, S, full, seed=80 + D, scale=scale)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("bits,v_exp", [(40, 95), (100, 0), (100, 95), (118, 0)])
@pytest.mark.parametrize("lq,lk,Hq,Hkv", [((1024,), (1024,), 2, 1), ((640, 30, 1), (1024, 900, 700), 4, 1), ((2560,), (2560,), 16, 2)])
def test_scores_that_grow_within_one_tile(D, lq, lk, Hq, Hkv, bits, v_exp):
    """A key in an unmasked tile whose score lies 2^bits above all before it: taken as it comes with the reference raised behind
    it (40, 100), past what is taken that way (118), and with values around 2^95, whose products stay below 2^127 only
    against a reference that follows the scores."""
    q, k, v = (t.float() for t in make(lq, lk, Hq, Hkv, D, 70))
    u = q[0, 0] / q[0, 0].norm()
    q = 0.2 * q + 16.0 * u
    k = 0.2 * k
    for a in np.concatenate([[0], np.cumsum(lk)[:-1]]):
        k[a + 300] += u * (bits * 0.6931 * D ** 0.5 / 16.0)
    q, k = q.to(torch.bfloat16), k.to(torch.bfloat16)
    v = (v * 2.0 ** v_exp).to(torch.bfloat16)
    out, lse, status = run_chunked(q, k, v, lq, lk, 1, 0, True)
    assert status == 0
    rows = np.unique(np.linspace(0, sum(lq) - 1, 400).astype(np.int64))
    rh = (rows % Hq).astype(np.int32)
    cu_q, cu_k = (np.concatenate([[0], np.cumsum(n)]) for n in (lq, lk))
    ref = oracle.prefill_chunked(*(inputs.to_f32_numpy(t) for t in (q, k, v * 2.0 ** -v_exp)), cu_q, cu_k, 1, 0, True, rows=(rows, rh))
    got = out[torch.as_tensor(rows, device="cuda"), torch.as_tensor(rh.astype(np.int64), device="cuda")] * 2.0 ** -v_exp
    check_against_oracle(got, ref["out"], f"{lq} {lk} D={D}")
    np.testing.assert_allclose(lse.cpu().numpy()[rh, rows], ref["lse"], rtol=0, atol=2e-3)
