"""The decode step's front end with sequences whose features are NaN: they pick k distinct experts all the same,
and the other sequences' results do not notice them."""
import pytest
import torch

from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,k", [(3, 2), (40, 8), (64, 8), (256, 2)])
def test_nan_features_stay_in_their_sequence(B, k):
    cfg = synth.LayerConfig("nan", "bf16", B, 1, 64, 1, 16, 16, 1, 16, k, 64, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=90)
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    ok = torch.arange(B) % 4 == 0
    ws = torch.empty(sb.swimba_decode_workspace_bytes(h, B), dtype=torch.uint8, device="cuda")
    got = []
    for bad in (False, True):
        u = inp["u"][:, 0].clone()
        if bad:
            u[~ok] = float("nan")
        ws.fill_(0xff)                       # (rows nobody writes are NaN)
        state, y = hp.dev(inp["h0"]), torch.empty(B, 1, 16, dtype=torch.bfloat16, device="cuda")
        idx = torch.empty(B, k, dtype=torch.int32, device="cuda")
        sb.swimba_decode_step(h, w, u.cuda(), hp.dev(inp["x"][:, 0]), hp.dev(inp["dt"][:, 0]), state, B, y, idx, None, ws)
        assert sb.swimba_status(h) == 0
        got.append((y.cpu()[ok], state.cpu()[ok], idx.cpu()[ok]))
        srt = idx.cpu().sort(dim=1).values
        assert srt.min() >= 0 and srt.max() < 16 and (srt[:, 1:] != srt[:, :-1]).all()
    assert all(torch.equal(a, b) for a, b in zip(*got))
    sb.swimba_destroy(h)
