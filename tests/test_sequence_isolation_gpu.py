"""What a sequence must not see does not reach its results: keys and values of its neighbours in a packed batch that hold
NaN, and those of later tokens in a key tile that earlier ones do not reach."""
import numpy as np
import pytest
import torch

import paper_2512_10411_b200 as swaa
from test_prefill_chunked_gpu import make, run_chunked
from test_prefill_gpu import run_prefill

pytestmark = pytest.mark.gpu


def _cu(lens):
    return torch.tensor(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32), device="cuda")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("W,S,full", [(64, 4, False), (100, 0, False), (100, 20, False), (1, 0, True)])
def test_forward_next_to_a_sequence_of_nan_keys_and_values(D, W, S, full):
    # key lengths that end on a tile: no key tile on the grid of whole tiles holds keys of two sequences
    for lq, lk in (((256, 128), (256, 128)), ((256, 128, 77), (640, 256, 77)), ((3, 256, 40), (256, 384, 40))):
        q, k, v = make(lq, lk, 4, 2, D, 50 + W)
        want, want_lse, _ = run_chunked(q, k, v, lq, lk, W, S, full)
        n_q, n_k = sum(lq[:-1]), sum(lk[:-1])
        k[n_k:] = float("nan")
        v[n_k:] = float("nan")
        outs = [run_chunked(q, k, v, lq, lk, W, S, full)]
        if lq == lk:
            outs.append(run_prefill(q, k, v, _cu(lq), max(lq), W, S, full))
        for out, lse, status in outs:
            assert status == 0
            assert torch.equal(out[:n_q], want[:n_q]) and torch.equal(lse[:, :n_q], want_lse[:, :n_q]), (lq, lk)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("W,S,full", [(100, 0, False), (100, 20, False), (1, 0, True)])
@pytest.mark.parametrize("lq,lk", [((3, 2), (256, 300)), ((1, 4, 3), (2500, 2304, 130)), ((1, 3, 60), (144, 2512, 2600))])
def test_generated_tokens_next_to_a_sequence_of_nan_keys_and_values(D, W, S, full, lq, lk):
    q, k, v = make(lq, lk, 4, 2, D, 80 + W)
    want, want_lse, _ = run_chunked(q, k, v, lq, lk, W, S, full)
    # lists that end inside a tile; tokens alone also inside a group of 16 keys (next to a prompt a few short lists are the prefill
    # kernel's, which reads keys in such groups)
    for bad in range(len(lk)):
        kk, vv = k.clone(), v.clone()
        rows = slice(sum(lk[:bad]), sum(lk[:bad + 1]))
        kk[rows] = vv[rows] = float("nan")
        out, lse, status = run_chunked(q, kk, vv, lq, lk, W, S, full)
        assert status == 0
        for b in range(len(lq)):
            mine = slice(sum(lq[:b]), sum(lq[:b + 1]))
            if b != bad and lq[b] <= 4:
                assert torch.equal(out[mine], want[mine]) and torch.equal(lse[:, mine], want_lse[:, mine]), (bad, b)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("L0", [64, 100, 192, 256])
def test_backward_next_to_a_sequence_of_nan_keys(D, L0):
    lens, Hq, Hkv, W, S = (L0, 200), 4, 2, 100, 4
    q, k, v = make(lens, lens, Hq, Hkv, D, 60 + L0)
    out, lse, _ = run_prefill(q, k, v, _cu(lens), max(lens), W, S, False)
    dout = make(lens, lens, Hq, Hkv, D, 61 + L0)[0]
    ws = torch.empty(swaa.prefill_backward_workspace_size(2, sum(lens), Hq, Hkv, D, S), dtype=torch.uint8, device="cuda")

    def grads(kk):
        g = [torch.full_like(t, float("nan")) for t in (q, k, v)]
        swaa.swaa_prefill_backward(q, kk, v, out, dout, lse, _cu(lens), max(lens), W, S, False, *g, ws)
        assert swaa.last_device_status() == 0
        return g

    want = grads(k)
    for bad, kept in ((slice(L0, None), slice(0, L0)), (slice(0, L0), slice(L0, None))):
        kk = k.clone()
        kk[bad] = float("nan")
        for got, w, name in zip(grads(kk), want, ("dq", "dk", "dv")):
            err = (got[kept].double() - w[kept].double()).norm() / w[kept].double().norm()
            assert err.item() <= 1e-3, (name, bad)  # the order of the fp32 sums into dq varies: bf16 roundings that flip


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("len_q,first_bad", [(2, 128), (8, 128), (8, 133)])
@pytest.mark.parametrize("other", [(3, 300), (40, 3000), (40, 300)])  # tokens alone; behind a prompt; with the prompt, packed
def test_values_of_later_tokens_in_a_tile_of_their_own(D, bad, len_q, first_bad, other):
    # one query head per kv head, so that several tokens are rows of one item; the keys from 128 on are its second tile
    lq, lk = (len_q, other[0]), (129 if len_q == 2 else 134, other[1])
    q, k, v = make(lq, lk, 4, 4, D, 70)
    want, want_lse, _ = run_chunked(q, k, v, lq, lk, 1, 0, True)
    k[first_bad:lk[0]], v[first_bad:lk[0]] = float("nan"), bad
    out, lse, status = run_chunked(q, k, v, lq, lk, 1, 0, True)
    n = 128 - (lk[0] - len_q)  # queries that see the first tile only
    assert status == 0 and n > 0
    assert torch.equal(out[:n], want[:n]) and torch.equal(lse[:, :n], want_lse[:, :n])
    assert torch.equal(out[len_q:], want[len_q:])
