"""The forward's front end for up to 256 tokens at its edges (column tiles of 8 and passes of 32 tokens per
expert, feature counts that eight warps do not share evenly, the first call size beyond it), and the
whole forward behind it with and without an initial state."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,F,G,E,k", [(1, 32, 1, 2, 1), (9, 96, 1, 3, 2), (33, 288, 2, 16, 2), (255, 64, 1, 2, 2), (256, 2080, 1, 5, 1),
                                       (257, 96, 1, 4, 2)])
def test_short_streams_match_oracle(T, F, G, E, k):
    cfg = synth.LayerConfig("short", "bf16", 1, T, F, 2 * G, 64, 128, G, E, k, 64, h0_std=0.2 if T % 2 else 0.0)
    inp = synth.make_inputs(cfg, seed=70 + T)
    h = hp.create_handle(cfg, None, sb.FLAG_CHECK_INDICES)
    w, keep = hp.device_weights(inp)
    BC, raw = hp.with_canary((T, cfg.S), torch.bfloat16, float("nan"))
    idx = torch.full((T, k), -1, dtype=torch.int32, device="cuda")
    wt = torch.full((T, k), float("nan"), device="cuda")
    ws = torch.empty(sb.swimba_workspace_bytes(h, 1, T), dtype=torch.uint8, device="cuda")
    sb.swimba_route_mix(h, w, hp.dev(inp["u"][0]), T, BC, idx, wt, ws)
    assert sb.swimba_status(h) == 0, sb.swimba_last_error(h)
    assert hp.canary_intact(raw)
    sb.swimba_destroy(h)
    u, W_e = synth.f64(inp["u"][0]), synth.f64(inp["W_e"])
    ii, ww = idx.cpu().numpy(), wt.cpu().double().numpy()
    slots = ww[..., None] * np.take_along_axis(oracle.expert_streams(u, W_e), ii[..., None].astype(np.int64), 1)
    # a stored bf16 value is off by up to 2^-8 of it: one slot is stored once, of two each is and their sum is;
    # fp32 sums of F products: F 2^-24 of the sum of their absolute values, at most sqrt(F) typical entries
    bound = 1.01 * 2.0 ** -8 * (np.abs(slots.sum(1)) + (np.abs(slots).sum(1) if k > 1 else 0.0)) \
        + F ** 1.5 * 2.0 ** -24 * np.abs(slots).max()
    assert np.all(np.abs(BC.cpu().double().numpy() - slots.sum(1)) <= bound)
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))
