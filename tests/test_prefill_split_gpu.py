"""Long key lists of generated tokens cut into parts (chunked and paged prefill with a workspace) against the float64 oracle:
key counts around the smallest part, more parts than one round of the merge takes and the most there are, every group size,
tokens alone and next to prompts, which kernel takes them, and whose memory the scratch is."""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_10411_b200 as swaa
from paper_2512_10411_b200 import binding, inputs
from helpers import check_against_oracle
from test_prefill_chunked_gpu import _cu, make

pytestmark = pytest.mark.gpu

BATCHES = [
    # new tokens, context lengths
    ((1,), (1025,)),                                 # one tile more than a part: two parts
    ((1, 1), (1024, 9000)),                          # not cut, and many parts
    ((3, 200, 1, 2), (5000, 700, 4481, 2049)),       # several rows per token group next to a chunk
    (tuple([1] * 40), tuple(range(300, 300 + 40 * 150, 150))),  # more than 32 sequences: two groups of the scheduler
    ((1, 90, 1), (20500, 130, 4000)),                # 21 parts where there is one kv head: two rounds of the merge
    ((1,), (41000,)),                                # 321 tiles: 32 parts, the most, of ten and eleven tiles
]


def _run(paged, q, k, v, lq, lk, W, S, full, full_seq, stream=None):
    """The call, on `stream` (a torch stream, or the address of one) behind all that the current one has been given."""
    out = torch.full_like(q, float("nan"))
    lse = torch.full((q.shape[1], q.shape[0]), float("nan"), device="cuda")
    fs = None if full_seq is None else torch.tensor(full_seq, dtype=torch.uint8, device="cuda")
    if not paged:
        cu_q, cu_k = _cu(lq), _cu(lk)
        call = lambda: swaa.swaa_prefill_chunked(q, k, v, out, cu_q, cu_k, max(lq), max(lk), W, S, full, lse=lse, is_full_seq=fs, stream=stream)
    else:
        page, Hkv, D = 128, k.shape[1], k.shape[2]
        used = [-(-n // page) for n in lk]
        order = torch.randperm(sum(used), generator=torch.Generator().manual_seed(3))
        kp = torch.full((sum(used), page, Hkv, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        vp, table, n, pos = kp.clone(), torch.zeros(len(lk), max(used), dtype=torch.int32), 0, 0
        for b, L in enumerate(lk):
            for i in range(used[b]):
                m = min(page, L - i * page)
                kp[order[n], :m], vp[order[n], :m] = k[pos + i * page:pos + i * page + m], v[pos + i * page:pos + i * page + m]
                table[b, i] = order[n]
                n += 1
            pos += L
        cu_q, len_k, table = _cu(lq), torch.tensor(lk, dtype=torch.int32, device="cuda"), table.cuda()
        call = lambda: swaa.swaa_prefill_paged(q, kp, vp, out, cu_q, len_k, table, max(lq), W, S, full, lse=lse, is_full_seq=fs, stream=stream)
    torch_stream = _torch_stream(stream)
    torch_stream.wait_stream(torch.cuda.current_stream())
    call()
    assert swaa.last_device_status(stream) == 0  # waits for the call
    return out, lse


def _torch_stream(stream):
    if stream is None:
        return torch.cuda.current_stream()
    if isinstance(stream, int):
        return torch.cuda.ExternalStream(stream) if stream else torch.cuda.default_stream()
    return stream


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("heads,D", [((4, 1), 128), ((16, 2), 64), ((6, 6), 128)])
@pytest.mark.parametrize("batch", range(len(BATCHES)))
def test_split_items_against_the_oracle(batch, heads, D, paged):
    lq, lk = BATCHES[batch]
    Hq, Hkv = heads
    q, k, v = make(lq, lk, Hq, Hkv, D, 900 + batch)
    k[::97] *= 6  # scores that outgrow the reference in the middle of a part
    qh, kh, vh = (inputs.to_f32_numpy(t) for t in (q, k, v))
    for W, S, full, full_seq in ((1, 0, True, None), (2500, 4, False, None), (100, 20, False, [b % 2 for b in range(len(lq))])):
        out, lse = _run(paged, q, k, v, lq, lk, W, S, full, full_seq)
        kw = {} if full_seq is None else {"is_full_seq": np.array(full_seq, dtype=np.uint8)}
        ref = oracle.prefill_chunked(qh, kh, vh, _cu(lq).cpu().numpy(), _cu(lk).cpu().numpy(), W, S, full, **kw)
        check_against_oracle(out, ref["out"], f"split {batch} {heads} D={D} paged={paged} W={W} S={S} full={full}")
        np.testing.assert_allclose(lse.cpu().numpy().T, ref["lse"], rtol=0, atol=2e-3)


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 6, 7, 8])
def test_group_sizes(G, paged):
    """As many tokens as fill the rows (8 // G), one, and lists that end inside a tile; the tokens have the same bits alone (one kernel, which
    waits for what is before it) and next to a prompt (behind the prefill kernel)."""
    most, Hkv, W, S = 8 // G, 2, 300, 20
    lq, lk = (most, 1, most), (2500, 1111, 77)
    q, k, v = make(lq, lk, G * Hkv, Hkv, 64, 920 + G)
    for full, full_seq in ((True, None), (False, None), (False, [1, 0, 1])):
        out, lse = _run(paged, q, k, v, lq, lk, W, S, full, full_seq)
        kw = {} if full_seq is None else {"is_full_seq": np.array(full_seq, dtype=np.uint8)}
        ref = oracle.prefill_chunked(*(inputs.to_f32_numpy(t) for t in (q, k, v)), _cu(lq).cpu().numpy(), _cu(lk).cpu().numpy(), W, S, full, **kw)
        check_against_oracle(out, ref["out"], f"G={G} paged={paged} full={full} {full_seq}")
        np.testing.assert_allclose(lse.cpu().numpy().T, ref["lse"], rtol=0, atol=2e-3)
        if not full and full_seq is None:
            continue  # few short lists: next to a prompt they are not the token kernel's
        # the prompt in front: 150 queries of 2900 keys
        p, pk, pv = make((150,), (2900,), G * Hkv, Hkv, 64, 930 + G)
        both, both_lse = _run(paged, torch.cat([p, q]), torch.cat([pk, k]), torch.cat([pv, v]), (150, *lq), (2900, *lk), W, S, full,
                              None if full_seq is None else [0, *full_seq])
        assert torch.equal(both[150:], out) and torch.equal(both_lse[:, 150:], lse)


def test_calls_that_the_library_would_cut_ask_it():
    """What the binding tells without the library, over random calls: none that the library has a workspace size for goes without."""
    rng, lib, cut = np.random.default_rng(0), binding.load_library(), 0
    for _ in range(2000):
        G, Hkv, B = (int(x) for x in (rng.choice([1, 2, 3, 4, 7, 8, 16]), rng.choice([1, 2, 8]), rng.integers(1, 40)))
        max_k, window = (int(np.exp(rng.uniform(np.log(lo), np.log(5000)))) for lo in (100, 1))
        n_sink, full = int(rng.choice([0, 4, 200])), bool(rng.integers(2))
        q = torch.empty((B, G * Hkv, 64), dtype=torch.bfloat16, device="cuda")  # a token each
        nbytes = lib.swaa_prefill_split_workspace_size(B, max_k, G * Hkv, Hkv, 64, window, n_sink, int(full), None)
        ws = binding._split_workspace(lib, q, None, B, 1, max_k, Hkv, window, n_sink, full) if max_k > binding._UNCUT_KEYS else None
        assert (0 if ws is None else ws.numel()) == nbytes
        cut += nbytes > 0
    assert 200 < cut < 1800


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("lq,lk,heads,kernels", [
    ((1, 2, 1), (1281, 70, 9), (8, 2), 1),                           # tokens alone: the token kernel
    ((100, 1, 1), (1280, 1280, 700), (8, 2), 1),                     # lists of ten tiles stay with the prompts
    ((100, 1, 1), (1281, 1280, 700), (8, 2), 2),                     # of eleven do not
    ((20,) + (1,) * 36, (90,) + (100,) * 36, (8, 8), 1),             # two tiles per SM in all (37 lists of one, eight heads)
    ((20,) + (1,) * 37, (90,) + (100,) * 37, (8, 8), 2),             # one more
    ((60, 70), (2000, 1500), (8, 2), 1),                             # no room for a token
    ((70, 2, 0), (2000, 1500, 0), (6, 2), 2),
    ((70, 3), (2000, 1500), (32, 2), 1),                             # sixteen heads to a group
])
def test_which_kernels_take_the_tokens(lq, lk, heads, kernels, paged):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines are those of 148 SMs")
    q, k, v = make(lq, lk, *heads, 64, 950)
    qh, kh, vh = (inputs.to_f32_numpy(t) for t in (q, k, v))
    before = swaa.kernel_launch_count()
    out, lse = _run(paged, q, k, v, lq, lk, 1, 0, True, None)
    assert swaa.kernel_launch_count() - before == kernels
    ref = oracle.prefill_chunked(qh, kh, vh, _cu(lq).cpu().numpy(), _cu(lk).cpu().numpy(), 1, 0, True)
    check_against_oracle(out, ref["out"], f"{lq} {lk} {heads} paged={paged}")
    np.testing.assert_allclose(lse.cpu().numpy().T, ref["lse"], rtol=0, atol=2e-3)


def test_split_calls_on_other_streams_and_in_a_graph():
    """A stream of its own (object and address), and a capture, where the call goes without a workspace."""
    lq, lk, W, S = (1, 1, 70), (6000, 1300, 900), 64, 4
    q, k, v = make(lq, lk, 8, 2, 128, 77)
    want, _ = _run(False, q, k, v, lq, lk, W, S, True, None)
    side = torch.cuda.Stream()
    for stream in (side, side.cuda_stream, 0):
        got, _ = _run(False, q, k, v, lq, lk, W, S, True, None, stream=stream)
        assert torch.equal(got, want)
    lib = binding.load_library()
    assert lib.swaa_prefill_split_workspace_size(3, 6000, 8, 2, 128, W, S, 1, None) > 0
    assert lib.swaa_prefill_split_workspace_size(3, 1024, 8, 2, 128, W, S, 1, None) == 0
    assert lib.swaa_prefill_split_workspace_size(3, 6000, 8, 2, 128, W, S, 0, None) == 0  # windows of 64 keys
    cu_q, cu_k, out = _cu(lq), _cu(lk), torch.full_like(q, float("nan"))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        assert lib.swaa_prefill_split_workspace_size(3, 6000, 8, 2, 128, W, S, 1, torch.cuda.current_stream().cuda_stream) == 0
        swaa.swaa_prefill_chunked(q, k, v, out, cu_q, cu_k, max(lq), max(lk), W, S, True)
    g.replay()
    torch.cuda.synchronize()
    assert (out.float() - want.float()).norm() / want.float().norm() < 1e-2  # two correct splits: bf16 outputs differ by 2e-3


@pytest.mark.parametrize("by", ["stream", "address", "zero"])
def test_scratch_is_not_a_block_that_another_stream_still_uses(by):
    """A block of the scratch's size, freed on the current stream with its reader still queued behind slow work, stays what it is
    while a call on another stream runs, and the call's result is the usual one."""
    lq, lk, W, S = (1, 1, 70), (6000, 1300, 900), 64, 4
    q, k, v = make(lq, lk, 8, 2, 128, 77)
    want, _ = _run(False, q, k, v, lq, lk, W, S, True, None)
    side = torch.cuda.Stream()
    stream = {"stream": side, "address": side.cuda_stream, "zero": 0}[by]
    nbytes = binding.load_library().swaa_prefill_split_workspace_size(3, 6000, 8, 2, 128, W, S, 1, None)
    work, kept, out = torch.zeros(1 << 28, device="cuda"), torch.zeros(nbytes, dtype=torch.uint8, device="cuda"), torch.zeros_like(q)
    cu_q, cu_k = _cu(lq), _cu(lk)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):  # the current stream of the caller
        for _ in range(2):
            block = torch.full((nbytes,), 7, dtype=torch.uint8, device="cuda")
            for _ in range(40):  # 2 GiB each: over 10 ms
                work.add_(1.0)
            kept.copy_(block)
            del block
            swaa.swaa_prefill_chunked(q, k, v, out, cu_q, cu_k, max(lq), max(lk), W, S, True, stream=stream)
            torch.cuda.synchronize()
            assert torch.equal(out, want) and bool((kept == 7).all())
            kept.zero_()
            out.zero_()
            torch.cuda.synchronize()
