"""The CUDA-core recurrence (fp32, and bf16 shapes without a tensor-core kernel) is causal for any input bits:
infinities and NaN in a token's x, B or C stay out of the outputs of the tokens before it and of other
sequences, and are in its own."""
import pytest
import torch

from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth

import helpers as hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("t", [1, 2, 3, 38, 63, 64, 291])
def test_no_token_sees_a_later_one(dtype, t):
    cfg = synth.LayerConfig("causal", dtype, 2, 292, 64, 2, 32, 16, 1, 4, 2, 128, h0_std=0.2)
    inp = synth.make_inputs(cfg, seed=80)
    h = hp.create_handle(cfg)
    w, keep = hp.device_weights(inp)
    B, L, td = cfg.B, cfg.L, synth.torch_dtype(dtype)
    gen = torch.Generator().manual_seed(81)
    x, bc, h0 = hp.dev(inp["x"]), torch.randn(B, L, 2 * cfg.N, generator=gen).to(td).cuda(), hp.dev(inp["h0"])
    ws = torch.empty(sb.swimba_workspace_bytes(h, B, L), dtype=torch.uint8, device="cuda")

    def run(x, bc):
        y = torch.zeros_like(x)
        sb.swimba_ssd(h, w, x, bc, hp.dev(inp["dt"]), h0, B, L, y, torch.empty_like(h0), ws)
        assert sb.swimba_status(h) == 0
        return y

    clean = run(x, bc)
    assert torch.isfinite(clean).all()
    for bad in (float("inf"), float("nan")):
        for where in ("x", "B", "C"):
            x2, bc2 = x.clone(), bc.clone()
            if where == "x":
                x2[0, t] = bad
            else:
                bc2[0, t, (0 if where == "B" else cfg.N):(cfg.N if where == "B" else 2 * cfg.N)] = bad
            y = run(x2, bc2)
            assert torch.equal(y[0, :t], clean[0, :t]) and torch.equal(y[1], clean[1]), (bad, where)
            assert not torch.isfinite(y[0, t]).any(), (bad, where)
    sb.swimba_destroy(h)
