"""The SSD kernel for long runs of tiles at its edges: six tiles (the fewest it takes) and one more token, odd head
counts, two groups, leading tiles, given states (and segments of two tiles, which the other kernel works: longer ones are in
test_gpu_run_forms.py); heads that decay too fast for one reference per tile
(2^-176 and more over its 128 tokens), and for products of factors at all (2^-96 over 32)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,H,G,fast", [(25, 768, 5, 1, False), (38, 769, 4, 2, True), (25, 769, 6, 1, True),
                                          (13, 1537, 17, 1, True), (1, 5000, 12, 2, True), (76, 768, 4, 1, False)])
def test_long_runs_match_oracle(B, L, H, G, fast):
    cfg = synth.LayerConfig("runs", "bf16", B, L, 32, H, 64, 128, G, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=60 + H)
    if fast:
        # log2 decay over n tokens: 16 step n / ln 2 -- 250 a tile, 63 a block for the first head, 110 a block (+- a
        # few) for the last one
        for head, step in ((0, 0.085), (H - 1, 0.149)):
            inp["A"][head] = -16.0
            inp["dt_bias"][head] = math.log(math.expm1(step))
        inp["dt"] *= 0.1
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))


def test_vanishing_steps_in_front_of_fast_tokens():
    """Eight tokens of step size 0 lead every 32-token block of two heads, the others decay by 2^-99 in all: of one
    warp's rows some have decayed by nothing, some by more than 2^-96."""
    B, L, H = 25, 769, 6
    cfg = synth.LayerConfig("runs", "bf16", B, L, 32, H, 64, 128, 1, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=70)
    for head in (0, H - 1):
        inp["A"][head] = -16.0
        inp["dt_bias"][head] = math.log(math.expm1(0.179))
        inp["dt"][..., head] = 0.0
        inp["dt"][:, torch.arange(L) % 32 < 8, head] = -200.0
    got = hp.gpu_forward(cfg, inp)
    hp.compare_forward(cfg, inp, got, *hp.tolerances(cfg))


def test_leading_tiles_hand_over_the_state_of_fast_heads():
    """75 pairs of heads of 60 tiles: some 23 leading tiles are evaluated for their end state alone.  In every tile of two
    heads 32 tokens in the middle decay by 2^-14800 and inject nothing: the rows behind the last leading tile read what its
    last tokens left, whose weights refer to the end of a count of 340000.  Where the count is off by its rounding (2 % and
    more in some of ten sequences and heads), all of those rows are off by one factor.  Inside a tile l is rounded to
    2^-11 at each of 48 additions: 1.4e-3 on that factor if they are independent."""
    B, L, H = 5, 7680, 30
    cfg = synth.LayerConfig("runs", "bf16", B, L, 32, H, 64, 128, 1, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=75)
    inp["D"] = None
    middle = (torch.arange(L) % 128 >= 48) & (torch.arange(L) % 128 < 80)
    noise = torch.randn(B, int(middle.sum()), generator=torch.Generator().manual_seed(77))
    for head in (0, H - 1):
        inp["A"][head], inp["dt_bias"][head] = -16.0, 0.0
        inp["dt"][..., head] = -5.0
        inp["dt"][:, middle, head] = 20.0 + noise
        inp["x"][:, middle, head] = 0
    bc = (0.3 * torch.randn(B, L, cfg.S, generator=torch.Generator().manual_seed(76))).to(torch.bfloat16)
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    assert sb.swimba_ssd_segments(h, B, L) == 1
    y, hf = torch.empty(B, L, H, 64, dtype=torch.bfloat16, device="cuda"), torch.empty(B, H, 64, 128, device="cuda")
    ws = torch.empty(sb.swimba_workspace_bytes(h, B, L), dtype=torch.uint8, device="cuda")
    sb.swimba_ssd(h, w, hp.dev(inp["x"]), hp.dev(bc), hp.dev(inp["dt"]), hp.dev(inp["h0"]), B, L, y, hf, ws)
    assert sb.swimba_status(h) == 0
    sb.swimba_destroy(h)
    heads = [0, 13, H - 1]
    sub = dict(inp, **{n: inp[n][..., heads].contiguous() for n in ("A", "dt_bias", "dt")},
               x=inp["x"][:, :, heads].contiguous(), h0=inp["h0"][:, heads].contiguous())
    y_ref, h_ref = oracle.ssm_recurrence(*(synth.f64(t) for t in (sub["x"], bc, sub["dt"], sub["A"], sub["dt_bias"])),
                                         None, synth.f64(sub["h0"]))
    hp.check_outputs(cfg, sub, y.cpu()[:, :, heads], hf.cpu()[:, heads], dict(y=y_ref, h_final=h_ref), *hp.tolerances(cfg))
    for i in (0, 2):
        for b in range(B):
            got, ref = (a[b, :, i].reshape(L // 128, 128, 64)[1:, :48].reshape(L // 128 - 1, -1)
                        for a in (y.cpu()[:, :, heads].double().numpy(), y_ref))
            assert np.abs((got * ref).sum(1) / (ref * ref).sum(1) - 1.0).max() <= 8e-3


@pytest.mark.parametrize("bc_scale,x_scale", [(2.0 ** 10, 2.0 ** 4), (2.0 ** -17, 1.0)])
def test_range_of_magnitudes(bc_scale, x_scale):
    """Readouts of some 2^25, and entries C.B Delta of some 2^-35: heads whose factors are the furthest apart, at 2^-100 to
    2^-372 a tile (2^-93 a block), on the kernel for six tiles and more."""
    B, L, H = 38, 900, 8
    cfg = synth.LayerConfig("runs", "bf16", B, L, 32, H, 64, 128, 1, 4, 2, 128)
    inp = synth.make_inputs(cfg, seed=78)
    inp["D"] = None
    inp["A"][:] = -16.0
    step = torch.tensor([100.0, 140.0, 172.0, 180.0, 187.0, 190.0, 300.0, 372.0]) * (math.log(2.0) / (16 * 128))
    inp["dt_bias"] = torch.log(torch.expm1(step))
    inp["dt"] *= 0.01
    inp["x"] *= x_scale
    bc = (bc_scale * torch.randn(B, L, cfg.S, generator=torch.Generator().manual_seed(79))).to(torch.bfloat16)
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    assert sb.swimba_ssd_segments(h, B, L) == 1
    y, hf = torch.empty(B, L, H, 64, dtype=torch.bfloat16, device="cuda"), torch.empty(B, H, 64, 128, device="cuda")
    ws = torch.empty(sb.swimba_workspace_bytes(h, B, L), dtype=torch.uint8, device="cuda")
    sb.swimba_ssd(h, w, hp.dev(inp["x"]), hp.dev(bc), hp.dev(inp["dt"]), None, B, L, y, hf, ws)
    assert sb.swimba_status(h) == 0
    sb.swimba_destroy(h)
    y_ref, h_ref = oracle.ssm_recurrence(*(synth.f64(t) for t in (inp["x"], bc, inp["dt"], inp["A"], inp["dt_bias"])))
    hp.check_outputs(cfg, inp, y.cpu(), hf.cpu(), dict(y=y_ref, h_final=h_ref), *hp.tolerances(cfg))
