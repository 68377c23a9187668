"""The general form on the tile kernel where its launches differ: one token, segmented sequences, split
launches (two CTAs per head pair), two B/C groups; every slot behind the first is added in place."""
import pytest
import torch

import oracle
from paper_2603_06938_b200 import synth

import helpers as hp
import test_gpu_general as tg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,H,G,E,k", [(2, 1, 3, 1, 4, 2), (1, 1290, 3, 1, 4, 2), (20, 640, 8, 1, 3, 2),
                                         (2, 390, 6, 2, 4, 3)])
def test_slots_on_the_tile_kernel_match_the_state_equation(B, L, H, G, E, k):
    cfg = synth.LayerConfig("slots", "bf16", B, L, 64, H, 64, 128, G, E, k, 128, h0_std=0.3)
    inp = synth.make_inputs(cfg, seed=91)
    gen = torch.Generator(device="cpu").manual_seed(92)
    xe = torch.randn(B, L, E, H, cfg.P, generator=gen).to(torch.bfloat16)
    y, hf, idx, wt = tg.run_general(cfg, inp, xe, h0=inp["h0"])
    hp.check_routing(cfg, inp, idx, wt)
    BCe = oracle.expert_streams(synth.f64(inp["u"]).reshape(B * L, cfg.F), synth.f64(inp["W_e"]))
    y_ref, h_ref = oracle.mixed_general(synth.f64(xe), BCe.reshape(B, L, E, cfg.S), tg.dense_pi(cfg, inp, idx),
                                        synth.f64(inp["dt"]), synth.f64(inp["A"]), synth.f64(inp["dt_bias"]),
                                        h0=synth.f64(inp["h0"]), G=G)
    tol_y, tol_h = hp.tolerances(cfg)
    hp.check_outputs(cfg, dict(inp, D=None), y, hf, dict(y=y_ref, h_final=h_ref), tol_y, tol_h)
