"""The decode step's front end where its forms meet: up to four tokens (one kernel), more (two), feature
counts that eight warps do not share evenly, more than two experts per token (slots), rows of state that the
early reads cover and not; two steps in a row, the second reading what the first wrote."""
import pytest
import torch

import oracle
from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,F,H,P,N,G,E,k", [(1, 64, 1, 64, 128, 1, 2, 1), (4, 96, 3, 64, 128, 1, 16, 4), (5, 96, 2, 64, 128, 1, 8, 2),
                                             (7, 832, 4, 64, 128, 2, 5, 3), (40, 288, 40, 64, 128, 1, 4, 2),
                                             (3, 2080, 2, 13, 48, 1, 8, 2), (2, 160, 2, 32, 160, 1, 3, 2), (256, 32, 1, 16, 16, 1, 16, 5)])
def test_two_decode_steps_match_oracle(B, F, H, P, N, G, E, k):
    cfg = synth.LayerConfig("front", "bf16", B, 1, F, H, P, N, G, E, k, 64, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=40 + B)
    h = hp.create_handle(cfg, None, sb.FLAG_CHECK_INDICES)
    w, keep = hp.device_weights(inp)
    state, raw = hp.with_canary((B, H, P, N), torch.float32, 0.0)
    state.copy_(inp["h0"])
    ref_state = synth.f64(inp["h0"]).copy()
    ws, ws_raw = hp.with_canary((sb.swimba_decode_workspace_bytes(h, B),), torch.uint8, 0)
    gen = torch.Generator().manual_seed(41)
    for step in range(2):
        s = synth.make_decode_step_inputs(cfg, gen)
        y = torch.full((B, H, P), float("nan"), dtype=torch.bfloat16, device="cuda")
        idx = torch.full((B, k), -1, dtype=torch.int32, device="cuda")
        wt = torch.full((B, k), float("nan"), device="cuda")
        sb.swimba_decode_step(h, w, hp.dev(s["u"]), hp.dev(s["x"]), hp.dev(s["dt"]), state, B, y, idx, wt, ws)
        assert sb.swimba_status(h) == 0, sb.swimba_last_error(h)
        one = dict(inp, u=s["u"][:, None], x=s["x"][:, None], dt=s["dt"][:, None])
        hp.check_routing(cfg, one, idx.cpu(), wt.cpu())
        r = oracle.router(synth.f64(s["u"]), synth.f64(inp["W_r"]), k)
        fw = torch.gather(torch.from_numpy(r["pi"]), 1, idx.cpu().long()).numpy()
        ref = oracle.swimba_decode_step(synth.f64(s["u"]), synth.f64(s["x"]), synth.f64(s["dt"]), synth.f64(inp["W_r"]),
                                        synth.f64(inp["W_e"]), synth.f64(inp["A"]), synth.f64(inp["dt_bias"]), synth.f64(inp["D"]),
                                        k, ref_state, G=G, forced_idx=idx.cpu().numpy(), forced_w=fw)
        # fp32 throughout, except y's store: 2^-8 of it
        assert hp.max_rel(y.cpu().double().numpy(), ref["y"]) <= 2.0 ** -8 + 1e-4
        assert hp.per_head_rel(state.cpu().double().numpy(), ref_state, 1) <= 1e-4
    assert hp.canary_intact(raw) and hp.canary_intact(ws_raw)
    sb.swimba_destroy(h)
