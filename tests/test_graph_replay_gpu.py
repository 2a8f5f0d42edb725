"""Calls captured in a CUDA graph and replayed with other inputs in the same buffers give what a plain call gives for those
inputs: decode with items cut into two and into many parts (the workspace then holds what the replay before left there),
a serving step of prompt chunks and generated tokens, and a training step."""
import numpy as np
import pytest
import torch

import paper_2512_10411_b200 as swaa
from paper_2512_10411_b200 import inputs

pytestmark = pytest.mark.gpu


def _capture(call):
    call()  # first call outside the capture: kernel attributes and static scratch are set up here
    assert swaa.last_device_status() == 0
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        call()
    return graph


def _replay_and_compare(call, graph, out, refill, steps=4):
    want = []
    for step in range(steps):
        refill(step)
        call()
        want.append(out.clone())
    # replays in a row, with nothing but new inputs between them: each finds what the one before left in the workspace
    for rep in range(2):
        for step in range(steps):
            refill(step)
            out.fill_(float("nan"))
            graph.replay()
            assert swaa.last_device_status() == 0
            assert torch.equal(out, want[step]), f"replay {rep}, inputs {step}"


@pytest.mark.parametrize("form", ["dense", "paged", "partial", "static"])
@pytest.mark.parametrize("lens,Hq,Hkv,D", [
    ((640,) * 20, 16, 8, 128),       # 10 tiles per item over groups that own 12 of the list: items in two parts
    ((20000,), 8, 2, 64),            # one sequence over all blocks: items in many parts
    ((9000, 70, 3001, 1), 32, 8, 128),
])
def test_decode(form, lens, Hq, Hkv, D):
    cfg = inputs.DecodeConfig("replay", len(lens), -(-max(lens) // 64) * 64, Hq, Hkv, D, 200, 4, seed=31, seqlens=lens)
    q, kc, vc, sl = inputs.make_decode_inputs(cfg, "cuda")
    B, W, S, full = cfg.B, cfg.window, cfg.n_sink, True
    out = torch.empty_like(q)
    if form == "paged":
        nb = cfg.Lmax // 64
        table = torch.arange(B * nb, dtype=torch.int32, device="cuda").view(B, nb)
        ws = torch.empty(swaa.decode_paged_workspace_size(B, Hq, Hkv, D, nb, 64, W, S, full), dtype=torch.uint8, device="cuda")
        kp, vp = (t.view(B * nb, 64, Hkv, D) for t in (kc, vc))
        call = lambda: swaa.swaa_decode_paged(q, kp, vp, out, table, sl, W, S, full, ws)
    elif form == "partial":
        out = torch.empty((B, Hq, D + 2), dtype=torch.float32, device="cuda")
        ws = torch.empty(swaa.decode_partial_workspace_size(B, Hq, Hkv, D, cfg.Lmax, W, S, full), dtype=torch.uint8, device="cuda")
        call = lambda: swaa.swaa_decode_partial(q, kc, vc, out, sl, 0, W, S, full, ws)
    elif form == "static":
        call = lambda: swaa.swaa_decode_static(q, kc, vc, out, sl, W, S, full)
    else:
        ws = torch.empty(swaa.decode_workspace_size(B, Hq, Hkv, D, cfg.Lmax, W, S, full), dtype=torch.uint8, device="cuda")
        call = lambda: swaa.swaa_decode(q, kc, vc, out, sl, W, S, full, ws)

    def refill(step):
        g = torch.Generator(device="cuda").manual_seed(500 + step)
        q.copy_(torch.randn(q.shape, generator=g, device="cuda"))
        kc.copy_(torch.randn(kc.shape, generator=g, device="cuda"))
        sl.copy_(torch.tensor([max(n - 37 * step, 1) for n in lens], dtype=torch.int32))

    _replay_and_compare(call, _capture(call), out, refill)


@pytest.mark.parametrize("workspace", [False, True])
@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("Hq,Hkv,D", [(8, 2, 128), (16, 2, 64)])
@pytest.mark.parametrize("tokens_only", [False, True])
def test_serving_step(tokens_only, Hq, Hkv, D, paged, workspace):
    """Generated tokens whose key lists a plain call cuts over several SMs.  Captured with a workspace the call has the bits of the
    plain one (whatever the replay before left there); captured without, those of a call that cuts no list."""
    lq = (1, 1, 1, 1) if tokens_only else (70, 1, 1, 1)
    caps, W, S, page = (1500, 9000, 41000, 1100), 200, 4, 128  # the third list: the most parts, 32
    B, Tq, nb = len(lq), sum(lq), -(-max(caps) // page)
    q = torch.empty((Tq, Hq, D), dtype=torch.bfloat16, device="cuda")
    out, lse = torch.empty_like(q), torch.empty((Hq, Tq), device="cuda")
    n_pages = sum(-(-n // page) for n in caps)
    kv = [torch.empty((n_pages * page if paged else sum(caps), Hkv, D), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    pages = [t.view(n_pages, page, Hkv, D) if paged else None for t in kv]
    cu_q = torch.tensor(np.concatenate([[0], np.cumsum(lq)]).astype(np.int32), device="cuda")
    cu_k, lens = torch.zeros(B + 1, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
    full_seq = torch.tensor([0, 1, 1, 0], dtype=torch.uint8, device="cuda")
    table, n = torch.zeros((B, nb), dtype=torch.int32), 0
    for b, c in enumerate(caps):
        table[b, :-(-c // page)] = torch.arange(n, n + -(-c // page), dtype=torch.int32).flip(0)
        n += -(-c // page)
    table = table.cuda()

    def call(ws=None):
        if paged:
            swaa.swaa_prefill_paged(q, *pages, out, cu_q, lens, table, max(lq), W, S, False, lse=lse, is_full_seq=full_seq, workspace=ws)
        else:
            swaa.swaa_prefill_chunked(q, *kv, out, cu_q, cu_k, max(lq), max(caps), W, S, False, lse=lse, is_full_seq=full_seq, workspace=ws)

    nbytes = swaa.prefill_split_workspace_size(B, nb * page if paged else max(caps), Hq, Hkv, D, W, S, True)
    assert nbytes > 0
    own = torch.full((nbytes,), 255, dtype=torch.uint8, device="cuda") if workspace else None

    def refill(step):
        g = torch.Generator(device="cuda").manual_seed(700 + step)
        for t in (q, *kv):
            t.copy_(torch.randn(t.shape, generator=g, device="cuda"))
        lens.copy_(torch.tensor([c - 300 * step for c in caps], dtype=torch.int32))
        cu_k[1:] = lens.cumsum(0)

    refill(0)
    graph, want = _capture(lambda: call(own)), []
    for step in range(3):
        refill(step)
        call(None if workspace else q.new_empty(0, dtype=torch.uint8))
        want.append((out.clone(), lse.clone()))
    for rep in range(2):
        for step in range(3):
            refill(step)
            out.fill_(float("nan"))
            lse.fill_(float("nan"))
            graph.replay()
            assert swaa.last_device_status() == 0
            assert torch.equal(out, want[step][0]) and torch.equal(lse, want[step][1]), f"replay {rep}, inputs {step}"


def test_plain_call_on_another_stream_during_a_capture():
    """The call is not part of the graph, and the capture goes on."""
    q, kv = torch.randn((2, 8, 128), device="cuda").bfloat16(), torch.randn((6000, 2, 128), device="cuda").bfloat16()
    cu_q, cu_k = (torch.tensor(x, dtype=torch.int32, device="cuda") for x in ([0, 1, 2], [0, 3000, 6000]))
    want, out, x, side = torch.empty_like(q), torch.empty_like(q), torch.zeros(10, device="cuda"), torch.cuda.Stream()
    call = lambda o, **kw: swaa.swaa_prefill_chunked(q, kv, kv, o, cu_q, cu_k, 1, 3000, 1, 0, True, **kw)
    call(want, workspace=q.new_empty(0, dtype=torch.uint8))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        x.add_(1.0)
        call(out, stream=side)
        x.add_(1.0)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    out.zero_()
    x.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert bool((x == 2).all()) and bool((out == 0).all())


def test_a_workspace_that_is_too_small_is_refused():
    q, kv = torch.zeros((2, 8, 128), dtype=torch.bfloat16, device="cuda"), torch.zeros((6000, 2, 128), dtype=torch.bfloat16, device="cuda")
    cu_q, cu_k = (torch.tensor(x, dtype=torch.int32, device="cuda") for x in ([0, 1, 2], [0, 3000, 6000]))
    nbytes = swaa.prefill_split_workspace_size(2, 3000, 8, 2, 128, 1, 0, True)
    with pytest.raises(swaa.SwaaError, match="SWAA_ERR_WORKSPACE"):
        swaa.swaa_prefill_chunked(q, kv, kv, torch.empty_like(q), cu_q, cu_k, 1, 3000, 1, 0, True,
                                  workspace=torch.empty(nbytes - 1, dtype=torch.uint8, device="cuda"))
    with pytest.raises(TypeError, match="workspace"):
        swaa.swaa_prefill_chunked(q, kv, kv, torch.empty_like(q), cu_q, cu_k, 1, 3000, 1, 0, True,
                                  workspace=torch.empty(nbytes, dtype=torch.float32, device="cuda"))


@pytest.mark.parametrize("D", [64, 128])
def test_training_step(D):
    # 2300 tokens: the query range of the sink key tile is cut into chunks, whose accumulators a memset node clears
    cfg = inputs.PrefillConfig("replay", (2300, 130), 4, 2, D, 100, 4, False, seed=32)
    q, k, v, cu = inputs.make_prefill_inputs(cfg, "cuda")
    T, Hq, Hkv = cfg.T, cfg.Hq, cfg.Hkv
    out, lse, dout = torch.empty_like(q), torch.empty((Hq, T), device="cuda"), torch.randn_like(q)
    dq, dk, dv = torch.empty_like(q), torch.empty_like(k), torch.empty_like(v)
    ws = torch.empty(swaa.prefill_backward_workspace_size(2, T, Hq, Hkv, D, 4), dtype=torch.uint8, device="cuda")

    def call():
        swaa.swaa_prefill(q, k, v, out, cu, 2300, 100, 4, False, lse=lse)
        swaa.swaa_prefill_backward(q, k, v, out, dout, lse, cu, 2300, 100, 4, False, dq, dk, dv, ws)

    graph = _capture(call)
    g = torch.Generator(device="cuda").manual_seed(6)
    for _ in range(3):
        for t in (q, k, v, dout):
            t.copy_(torch.randn(t.shape, generator=g, device="cuda"))
        call()
        want = [t.clone() for t in (out, lse, dq, dk, dv)]
        for t in (out, lse, dq, dk, dv):
            t.fill_(float("nan"))
        graph.replay()
        assert swaa.last_device_status() == 0
        assert torch.equal(out, want[0]) and torch.equal(lse, want[1])
        for t, w in zip((dq, dk, dv), want[2:]):  # fp32 sums in an order that differs from run to run, rounded to bf16
            assert ((t.double() - w.double()).norm() <= 1e-3 * w.double().norm()).item()
