"""Routing and projection with tokens whose features are NaN, in each router: they pick k distinct experts, so that
the lists hold what they are sized for, and the other tokens' streams do not notice them."""
import pytest
import torch

from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


# one warp per token; tensor cores fed from registers; streaming; fp32
@pytest.mark.parametrize("dtype,T,F,E,k", [("bf16", 700, 72, 5, 2), ("bf16", 900, 128, 16, 3), ("bf16", 28500, 64, 4, 2),
                                           ("fp32", 300, 64, 9, 4)])
def test_nan_features_stay_in_their_token(dtype, T, F, E, k):
    cfg = synth.LayerConfig("nan", dtype, 1, T, F, 1, 16, 16, 1, E, k, 64)
    inp = synth.make_inputs(cfg, seed=95)
    h = hp.create_handle(cfg, None, sb.FLAG_CHECK_INDICES)
    w, keep = hp.device_weights(inp)
    ok = torch.arange(T) % 4 == 0
    ws = torch.empty(sb.swimba_workspace_bytes(h, 1, T), dtype=torch.uint8, device="cuda")
    got = []
    for bad in (False, True):
        u = inp["u"][0].clone()
        if bad:
            u[~ok] = float("nan")
        bc = torch.empty(T, cfg.S, dtype=u.dtype, device="cuda")
        idx = torch.empty(T, k, dtype=torch.int32, device="cuda")
        wt = torch.empty(T, k, device="cuda")
        sb.swimba_route_mix(h, w, u.cuda(), T, bc, idx, wt, ws)
        assert sb.swimba_status(h) == 0, sb.swimba_last_error(h)
        got.append((bc.cpu()[ok], idx.cpu()[ok], wt.cpu()[ok]))
        srt = idx.cpu().sort(dim=1).values
        assert srt.min() >= 0 and srt.max() < E and (srt[:, 1:] != srt[:, :-1]).all()
        assert not bad or torch.isnan(bc.cpu()[~ok]).all()
    assert all(torch.equal(a, b) for a, b in zip(*got))
    sb.swimba_destroy(h)
