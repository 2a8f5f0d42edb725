"""The work that a user of the library has it do, as cases that can be timed and compared.

A case is one call (for training: one forward and one backward call) of the public entry points, at sizes taken from
the benchmark's workloads and the tests, or generic: decode steps of one user and of a full batch, dense and paged;
prompts short and long, one and many in a packed batch, under the sliding-window mask with sinks and under full
attention; the mixed step of a serving engine (prompt chunks next to generated tokens, paged cache); training steps.
Head sizes 64 and 128 and both mask policies occur in each direction.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2512_10411_b200 as swaa

# (query heads, key/value heads)
HEADS = ((4, 2), (16, 4), (32, 8), (28, 4), (64, 8))
MAX_FLOPS = 2.0e13  # of a drawn case; the packed batch of long prompts has about this many
MAX_BYTES = 4.5e9   # the full-batch decode step over 64k-entry caches


def listed():
    """
    prefill_tiny            one short prompt of a small model: launch latency
    prefill_long_swa        a 32k prompt in an SWA layer (the benchmark's headline workload)
    prefill_long_full       a 32k prompt in a full-attention layer of the interleaved stack
    prefill_varlen          packed batch of ragged long prompts, 8 query heads per kv head
    serve_mixed_paged       one step of a serving engine: prompt chunks under the SWA mask next to generated tokens under
                            full attention (FA decode), keys and values in pages
    decode_fa_batch         FA decode of a batch at 64k context
    decode_swa_batch        the same step in an SWA layer without FA decode
    decode_fa_one           one user, long context, full attention
    decode_swa_one          one user, SWA: the smallest decode step
    decode_paged_ragged     FA decode of many users with contexts of very different lengths, paged cache
    train_long              forward and backward of a long-context fine-tuning sample under the SWA mask
    train_packed_d64        forward and backward of short samples packed to one batch, head size 64
    """
    ragged = "22655,26778,2743,26868,16451,17879,21409,10827"
    return [
        {"name": "prefill_tiny", "kind": "prefill", "lens": "1024", "Hq": 4, "Hkv": 2, "D": 64, "window": 128, "n_sink": 4, "full": False},
        {"name": "prefill_long_swa", "kind": "prefill", "lens": "32768", "Hq": 32, "Hkv": 8, "D": 128, "window": 2048, "n_sink": 4, "full": False},
        {"name": "prefill_long_full", "kind": "prefill", "lens": "32768", "Hq": 32, "Hkv": 8, "D": 128, "window": 2048, "n_sink": 4, "full": True},
        {"name": "prefill_varlen", "kind": "prefill", "lens": ragged, "Hq": 64, "Hkv": 8, "D": 128, "window": 4096, "n_sink": 4, "full": False},
        {"name": "serve_mixed_paged", "kind": "mixed", "Hq": 32, "Hkv": 8, "D": 128, "window": 4096, "n_sink": 4, "page": 128,
         "chunks": "2048,2048,1500,500", "ctx": "2048,16384,31000,500", "decodes": 24, "decode_lo": 1024, "decode_hi": 32768, "lens_seed": 7},
        {"name": "decode_fa_batch", "kind": "decode", "lens": ",".join(["65536"] * 16), "Lmax": 65536, "Hq": 32, "Hkv": 8, "D": 128, "window": 4096, "n_sink": 4, "full": True},
        {"name": "decode_swa_batch", "kind": "decode", "lens": ",".join(["65536"] * 16), "Lmax": 65536, "Hq": 32, "Hkv": 8, "D": 128, "window": 4096, "n_sink": 4, "full": False},
        {"name": "decode_fa_one", "kind": "decode", "lens": "65536", "Lmax": 65536, "Hq": 32, "Hkv": 8, "D": 128, "window": 4096, "n_sink": 4, "full": True},
        {"name": "decode_swa_one", "kind": "decode", "lens": "20011", "Lmax": 32768, "Hq": 16, "Hkv": 4, "D": 64, "window": 2048, "n_sink": 4, "full": False},
        {"name": "decode_paged_ragged", "kind": "decode_paged", "batch": 64, "lo": 512, "hi": 32768, "lens_seed": 11, "page": 64, "Hq": 64, "Hkv": 8, "D": 128,
         "window": 4096, "n_sink": 4, "full": True},
        {"name": "train_long", "kind": "train", "lens": "16384", "Hq": 32, "Hkv": 8, "D": 128, "window": 2048, "n_sink": 4, "full": False},
        {"name": "train_packed_d64", "kind": "train", "lens": "4096,700,1333,2048,3001,511,2500,2195", "Hq": 16, "Hkv": 4, "D": 64, "window": 1024, "n_sink": 4, "full": False},
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _one(rng: random.Random) -> dict:
    kind = rng.choice(("prefill", "prefill", "mixed", "decode", "decode_paged", "train"))
    Hq, Hkv = rng.choice(HEADS)
    c = {"kind": kind, "Hq": Hq, "Hkv": Hkv, "D": rng.choice((64, 128, 128)), "window": _log_int(rng, 128, 8192), "n_sink": rng.choice((0, 4, 4, 64)),
         "full": rng.random() < 0.35}
    if kind in ("prefill", "train"):
        total = _log_int(rng, 256, 65536 if kind == "prefill" else 32768)
        n = rng.choice((1, 1, 2, 5, 8))
        cuts = sorted(rng.randrange(1, total) for _ in range(n - 1))
        c["lens"] = ",".join(str(b - a) for a, b in zip([0] + cuts, cuts + [total]) if b > a)
    elif kind == "mixed":
        del c["full"]  # chunks run under the SWA mask, generated tokens under full attention
        chunks = [_log_int(rng, 64, 4096) for _ in range(rng.randint(1, 5))]
        c.update(page=rng.choice((128, 256)), chunks=",".join(map(str, chunks)), ctx=",".join(str(n + rng.choice((0, _log_int(rng, 128, 32768)))) for n in chunks),
                 decodes=rng.randint(0, 48), decode_lo=_log_int(rng, 64, 2048), decode_hi=_log_int(rng, 4096, 32768), lens_seed=rng.randrange(1 << 20))
    elif kind == "decode":
        n = _log_int(rng, 1, 64)
        hi = _log_int(rng, 1024, 65536)
        c["lens"] = ",".join(str(hi if n == 1 or rng.random() < 0.5 else _log_int(rng, max(1, hi // 16), hi)) for _ in range(n))
        c["Lmax"] = hi + rng.choice((0, 1, 200))
    else:
        c.update(batch=_log_int(rng, 1, 128), lo=_log_int(rng, 64, 2048), hi=_log_int(rng, 4096, 65536), lens_seed=rng.randrange(1 << 20), page=rng.choice((64, 128, 256)))
    return c


def draw(rng: random.Random) -> dict:
    """One more case of the same ranges; one that would cost more than the largest listed one is drawn again."""
    while True:
        c = _one(rng)
        w = work(c)
        if w["flops"] <= MAX_FLOPS and w["bytes"] <= MAX_BYTES and _cache_bytes(c) <= MAX_BYTES:
            return c


# ------------------------------------------------------------------------------------------ lengths
def _ints(text: str) -> list:
    return [int(x) for x in text.split(",")]


def _spread(n: int, lo: int, hi: int, seed: int) -> list:
    """n lengths, even over the logarithm of [lo, hi]."""
    r = np.random.default_rng(seed)
    return [int(x) for x in np.exp(r.uniform(math.log(lo), math.log(hi), n)).round()]


def _sequences(c: dict) -> list:
    """[(new tokens, context length including them, full attention)] of a case, in batch order."""
    if c["kind"] == "mixed":
        seqs = [(q, k, False) for q, k in zip(_ints(c["chunks"]), _ints(c["ctx"]))]
        return seqs + [(1, k, True) for k in _spread(c["decodes"], c["decode_lo"], c["decode_hi"], c["lens_seed"])]
    if c["kind"] == "decode_paged":
        return [(1, k, c["full"]) for k in _spread(c["batch"], c["lo"], c["hi"], c["lens_seed"])]
    if c["kind"] == "decode":
        return [(1, k, c["full"]) for k in _ints(c["lens"])]
    return [(n, n, c["full"]) for n in _ints(c["lens"])]


def _pairs_and_keys(c: dict) -> tuple:
    """(visible query/key pairs, keys that some query of the call sees), summed over the sequences."""
    pairs = keys = 0
    W, S = c["window"], c["n_sink"]
    for nq, nk, full in _sequences(c):
        i = np.arange(nk - nq, nk, dtype=np.int64)
        if full:
            pairs += int((i + 1).sum())
            keys += nk
        else:
            before = np.maximum(i + 1 - W, 0)  # keys before the window
            pairs += int((i + 1 - before + np.minimum(before, S)).sum())
            first = max(0, nk - nq + 1 - W)
            keys += nk - first + min(S, first)
    return pairs, keys


def _cache_bytes(c: dict) -> int:
    """Bytes of the keys and values that the caller holds."""
    per = c["Hkv"] * c["D"] * 4
    if c["kind"] == "decode":
        return len(_ints(c["lens"])) * c["Lmax"] * per
    return sum(nk for _, nk, _ in _sequences(c)) * per


def work(c: dict) -> dict:
    pairs, keys = _pairs_and_keys(c)
    tokens = sum(nq for nq, _, _ in _sequences(c))
    rows, kv = tokens * c["Hq"] * c["D"] * 2, keys * c["Hkv"] * c["D"] * 4
    if c["kind"] == "train":  # forward: q, k, v -> out, lse; backward: those and dout -> dq, dk, dv
        return {"bytes": 6 * rows + 3 * kv + 2 * tokens * c["Hq"] * 4, "flops": 14 * c["D"] * c["Hq"] * pairs}
    return {"bytes": 2 * rows + kv, "flops": 4 * c["D"] * c["Hq"] * pairs}


def tolerance(c: dict) -> dict:
    """Relative 2-norm of an output against the same path in float64: 2.1e-3 for bf16 outputs, 2.6e-3 for bf16 gradients
    (measured at both head sizes, both masks); four times that is what another split or order of the sums may show."""
    return {"rel": 1e-2}


# ------------------------------------------------------------------------------------------- inputs
def _randn(gen: torch.Generator, *shape) -> torch.Tensor:
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)


def _int32(values) -> torch.Tensor:
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _packed(lengths) -> torch.Tensor:
    return _int32([0] + np.cumsum(lengths).tolist())


def _with_sinks(k: torch.Tensor, starts, gen: torch.Generator) -> None:
    """Shifts the first key of every sequence along a random direction, so that it draws attention as a sink does."""
    u = torch.randn(k.shape[-2:], generator=gen, device="cuda")
    u = (3.0 * u / u.norm(dim=-1, keepdim=True)).to(k.dtype)
    flat = k.view(-1, *k.shape[-2:])
    flat[torch.tensor(list(starts), device="cuda")] += u


def prepare(case: dict, seed: int) -> dict:
    c = dict(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    seqs = _sequences(c)
    Hq, Hkv, D = c["Hq"], c["Hkv"], c["D"]
    n_q, n_k = [s[0] for s in seqs], [s[1] for s in seqs]
    B, T = len(seqs), sum(n_q)
    s = {"case": c, "q": _randn(gen, T, Hq, D), "out": torch.empty(T, Hq, D, dtype=torch.bfloat16, device="cuda")}
    if c["kind"] in ("prefill", "train"):
        s.update(k=_randn(gen, T, Hkv, D), v=_randn(gen, T, Hkv, D), cu=_packed(n_q), max_len=max(n_q))
        _with_sinks(s["k"], s["cu"][:-1].tolist(), gen)
        if c["kind"] == "train":
            nbytes = swaa.prefill_backward_workspace_size(B, T, Hq, Hkv, D, c["n_sink"])
            s.update(lse=torch.empty(Hq, T, device="cuda"), dout=_randn(gen, T, Hq, D), dq=torch.empty_like(s["q"]), dk=torch.empty_like(s["k"]),
                     dv=torch.empty_like(s["v"]), ws=torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
    elif c["kind"] == "decode":
        s.update(k=_randn(gen, B, c["Lmax"], Hkv, D), v=_randn(gen, B, c["Lmax"], Hkv, D), lens=_int32(n_k))
        _with_sinks(s["k"], [b * c["Lmax"] for b in range(B)], gen)
        nbytes = swaa.decode_workspace_size(B, Hq, Hkv, D, c["Lmax"], c["window"], c["n_sink"], c["full"])
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    else:  # pages of all sequences in a common pool, in random order
        page = c["page"]
        used = [-(-n // page) for n in n_k]
        order = torch.randperm(sum(used), generator=gen, device="cuda").to(torch.int32)
        table = torch.zeros(B, max(used), dtype=torch.int32, device="cuda")
        first = 0
        for b, n in enumerate(used):
            table[b, :n] = order[first:first + n]
            first += n
        s.update(k=_randn(gen, first, page, Hkv, D), v=_randn(gen, first, page, Hkv, D), table=table, lens=_int32(n_k))
        _with_sinks(s["k"], (table[:, 0].long() * page).tolist(), gen)
        if c["kind"] == "mixed":
            s.update(cu=_packed(n_q), max_len=max(n_q), full_seq=torch.tensor([int(f) for _, _, f in seqs], dtype=torch.uint8, device="cuda"))
        else:
            nbytes = swaa.decode_paged_workspace_size(B, Hq, Hkv, D, max(used), page, c["window"], c["n_sink"], c["full"])
            s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    return s


def run(s: dict):
    c = s["case"]
    W, S = c["window"], c["n_sink"]
    if c["kind"] == "prefill":
        swaa.swaa_prefill(s["q"], s["k"], s["v"], s["out"], s["cu"], s["max_len"], W, S, c["full"])
        return s["out"]
    if c["kind"] == "mixed":
        swaa.swaa_prefill_paged(s["q"], s["k"], s["v"], s["out"], s["cu"], s["lens"], s["table"], s["max_len"], W, S, False, is_full_seq=s["full_seq"])
        return s["out"]
    if c["kind"] == "decode":
        swaa.swaa_decode(s["q"], s["k"], s["v"], s["out"], s["lens"], W, S, c["full"], s["ws"])
        return s["out"]
    if c["kind"] == "decode_paged":
        swaa.swaa_decode_paged(s["q"], s["k"], s["v"], s["out"], s["table"], s["lens"], W, S, c["full"], s["ws"])
        return s["out"]
    swaa.swaa_prefill(s["q"], s["k"], s["v"], s["out"], s["cu"], s["max_len"], W, S, c["full"], lse=s["lse"])
    swaa.swaa_prefill_backward(s["q"], s["k"], s["v"], s["out"], s["dout"], s["lse"], s["cu"], s["max_len"], W, S, c["full"], s["dq"], s["dk"], s["dv"], s["ws"])
    return {"out": s["out"], "lse": s["lse"], "dq": s["dq"], "dk": s["dk"], "dv": s["dv"]}
