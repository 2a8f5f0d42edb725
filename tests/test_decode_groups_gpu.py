"""GPU parity of the decode kernel where heads are streamed in step by groups of blocks: kv head counts that do and do
not divide the SMs well, more items per sequence than SMs, ragged lengths, runs that end inside sequences."""
import pytest

import oracle
import paper_2512_10411_b200 as swaa
import torch
from paper_2512_10411_b200 import inputs
from helpers import check_against_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D", [(7, 7, 64), (40, 40, 64), (160, 160, 64), (24, 1, 128), (34, 2, 128), (13, 13, 128)])
@pytest.mark.parametrize("lens", [(1, 700, 64, 65, 3000), (4096,) * 3])
def test_decode_heads_in_step(Hq, Hkv, D, lens):
    cfg = inputs.DecodeConfig("groups", len(lens), max(lens), Hq, Hkv, D, 200, 4, seed=21, seqlens=lens)
    q, kc, vc, sl = inputs.make_decode_inputs(cfg, "cuda")
    for full in (True, False):
        ws = torch.empty(swaa.decode_workspace_size(cfg.B, Hq, Hkv, D, cfg.Lmax, 200, 4, full), dtype=torch.uint8, device="cuda")
        out = torch.full_like(q, float("nan"))
        swaa.swaa_decode(q, kc, vc, out, sl, 200, 4, full, ws)
        assert swaa.last_device_status() == 0
        ref = oracle.decode(*(inputs.to_f32_numpy(t) for t in (q, kc, vc)), lens, 200, 4, full)
        check_against_oracle(out, ref["out"], f"{lens} Hq={Hq} Hkv={Hkv} D={D} full={full}")
