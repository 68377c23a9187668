"""Every form in which calls reach the SSD kernel for six tiles and more, small: segments (a ragged last one, given
states), slots that add to what the first one left (odd heads, leading tiles, segments), states updated in place,
shards; with heads that decay too fast for one reference per tile.  That a case goes to that kernel follows from its
rule: a block walks one of the sequence's segments, which are equal but for the last one."""
import pytest
import torch

import oracle
from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp
import test_gpu_general as tg
import test_gpu_sharded as ts
from test_gpu_strong_decay import strong_inputs

pytestmark = pytest.mark.gpu

RUN_TILES = 6


def layer(B, L, H, G=1, E=4, k=2):
    return synth.LayerConfig("forms", "bf16", B, L, 32, H, 64, 128, G, E, k, 128, h0_std=0.2)


def tiles_walked(cfg, L=None):
    h = hp.create_handle(cfg)
    segments = sb.swimba_ssd_segments(h, cfg.B, L or cfg.L)
    sb.swimba_destroy(h)
    return -(-(-(-(L or cfg.L) // 128)) // segments), segments


@pytest.mark.parametrize("B,L,H,G", [(1, 5000, 38, 2), (3, 6000, 12, 1)])
def test_segments(B, L, H, G):
    cfg = layer(B, L, H, G)
    tiles, segments = tiles_walked(cfg)
    assert tiles >= RUN_TILES and segments > 1
    inp = strong_inputs(cfg, 90, True)
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))


@pytest.mark.parametrize("B,L,H,G", [(25, 769, 6, 1), (1, 5000, 38, 2)])
def test_in_place_states(B, L, H, G):
    cfg = layer(B, L, H, G)
    assert tiles_walked(cfg)[0] >= RUN_TILES
    inp = strong_inputs(cfg, 91, True)
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    state, y = hp.dev(inp["h0"]), torch.empty_like(hp.dev(inp["x"]))
    idx, wt = torch.empty(B, L, 2, dtype=torch.int32, device="cuda"), torch.empty(B, L, 2, device="cuda")
    ws = torch.empty(sb.swimba_workspace_bytes(h, B, L), dtype=torch.uint8, device="cuda")
    sb.swimba_forward(h, w, hp.dev(inp["u"]), hp.dev(inp["x"]), hp.dev(inp["dt"]), state, B, L, y, state, idx, wt, ws)
    assert sb.swimba_status(h) == 0
    sb.swimba_destroy(h)
    got = dict(y=y.cpu(), h_final=state.cpu(), idx=idx.cpu(), w=wt.cpu())
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))


# 75 pairs of heads (leading tiles), 150 pairs, segments
@pytest.mark.parametrize("B,L,H,G,k", [(25, 769, 6, 1, 2), (50, 769, 5, 1, 3), (1, 5000, 38, 2, 2)])
def test_slots(B, L, H, G, k):
    cfg = layer(B, L, H, G, E=3, k=k)
    assert tiles_walked(cfg)[0] >= RUN_TILES
    inp = strong_inputs(cfg, 92, True)
    xe = torch.randn(B, L, 3, H, cfg.P, generator=torch.Generator().manual_seed(93)).to(torch.bfloat16)
    y, hf, idx, wt = tg.run_general(cfg, inp, xe, h0=inp["h0"])
    hp.check_routing(cfg, inp, idx, wt)
    BCe = oracle.expert_streams(synth.f64(inp["u"]).reshape(B * L, cfg.F), synth.f64(inp["W_e"]))
    y_ref, h_ref = oracle.mixed_general(synth.f64(xe), BCe.reshape(B, L, 3, cfg.S), tg.dense_pi(cfg, inp, idx),
                                        synth.f64(inp["dt"]), synth.f64(inp["A"]), synth.f64(inp["dt_bias"]),
                                        h0=synth.f64(inp["h0"]), G=G)
    hp.check_outputs(cfg, inp, y, hf, dict(y=y_ref, h_final=h_ref), *hp.tolerances(cfg))


def test_shards():
    cfg = layer(40, 1700, 4)
    assert tiles_walked(cfg, 800)[0] >= RUN_TILES
    inp = strong_inputs(cfg, 94, True)
    got = ts.sharded_forward(cfg, inp, [900, 800], h0=inp["h0"])
    got["h_final"] = got["ends"][-1]
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
