"""The calls whose speed counts: what a program built on this library has it do, through
paper_2603_06938_b200.binding, over the range of shapes the kernels serve.

A case names one call pattern ("kind") and its sizes:
  forward    swimba_forward: prefill of B sequences of L tokens (bf16 tensor-core shapes, or fp32)
  decode     swimba_decode_step: one token for each of B running sequences
  packed     swimba_forward_packed: prompts of different lengths, decode tokens riding along
  block      swimba_block_forward: the whole block around the mixer
  backward   swimba_backward_weights: a training step's gradients of router and expert matrices
  slots      swimba_route_project_slots + swimba_ssd_slots: experts with their own SSM inputs
A program keeps the layer's handle, its weights, the workspace and the output buffers from call to
call; the inputs are new.  Distributions are those of synth.py (Mamba-2 style initialisation).
"""
import math
import random
import weakref

import torch

from paper_2603_06938_b200 import binding as sb
from paper_2603_06938_b200 import synth


def _layer(name):
    """Layer sizes of one of the repository's workloads."""
    c = synth.CONFIGS[name]
    return dict(dtype=c.dtype, F=c.F, H=c.H, P=c.P, N=c.N, G=c.G, E=c.E, k=c.k, chunk=c.Q)


def listed():
    return [
        # the fp32 path at the smallest workload: debugging, numerics references
        dict(name="forward_tiny_fp32", kind="forward", B=1, L=256, h0=False, **_layer("tiny_fp32")),
        # one short prompt (a chat turn) in a top-1 layer of four experts: latency and launches
        dict(name="forward_short", kind="forward", B=1, L=93, h0=True,
             **dict(_layer("small_lm"), E=4, k=1)),
        # the prefill / training-forward workloads
        dict(name="forward_small_lm", kind="forward", B=8, L=2048, h0=False, **_layer("small_lm")),
        dict(name="forward_mid", kind="forward", B=4, L=8192, h0=False, **_layer("mid")),
        # one long document
        dict(name="forward_long_seq", kind="forward", B=1, L=65536, h0=False, **_layer("long_seq")),
        # chunked prefill of a few ragged sequences, two B/C groups, four experts per token
        dict(name="forward_ragged", kind="forward", B=3, L=1531, h0=True,
             **dict(_layer("small_lm"), F=1152, H=36, G=2, E=16, k=4)),
        # decoding: one user, and a full serving batch
        dict(name="decode_one", kind="decode", B=1, **_layer("decode")),
        dict(name="decode_batch", kind="decode", B=128, **_layer("decode")),
        # continuous batching: prompts of mixed lengths with decode tokens between them
        dict(name="packed_serving", kind="packed", prompts=7, longest=4000, decode=57, mix=3, **_layer("mid")),
        # the whole block, forward
        dict(name="block_mid", kind="block", B=4, L=8192, d_conv=4, **_layer("mid")),
        # one step of training router and experts
        dict(name="backward_mid", kind="backward", B=4, L=8192, **_layer("mid")),
        # experts with their own inputs
        dict(name="slots_small_lm", kind="slots", B=8, L=2048, **_layer("small_lm")),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["forward", "forward", "forward", "fp32", "decode", "decode", "packed", "packed", "block",
                       "backward", "slots"])
    if kind == "fp32":
        E = rng.choice([2, 4, 8])
        return dict(kind="forward", dtype="fp32", B=rng.randint(1, 4), L=_log_int(rng, 24, 700),
                    F=8 * _log_int(rng, 12, 64), H=rng.randint(2, 16), P=rng.choice([32, 64]),
                    N=rng.choice([16, 32, 64]), G=1, E=E, k=rng.randint(1, min(3, E)), chunk=64,
                    h0=rng.random() < 0.5)
    G = rng.choice([1, 1, 1, 2])
    E = rng.choice([4, 8, 8, 16])
    c = dict(kind=kind, dtype="bf16", F=64 * _log_int(rng, 8, 32), H=G * _log_int(rng, 12 // G, 64 // G), P=64,
             N=128, G=G, E=E, k=rng.choice([1, 2, 2, 2, 3]), chunk=rng.choice([128, 256]))
    if kind == "decode":
        return dict(c, B=_log_int(rng, 1, 200))
    if kind == "packed":
        return dict(c, prompts=_log_int(rng, 1, 24), longest=_log_int(rng, 60, 6000), decode=_log_int(rng, 1, 96),
                    mix=rng.randrange(1000))
    # tokens of the call, over the logarithm, then how many sequences they come as; the widest layers
    # with the most tokens are left to the listed cases
    top = {"forward": 32768, "block": 16384, "backward": 16384, "slots": 12288}[kind]
    low = {"forward": 40, "block": 300, "backward": 1500, "slots": 300}[kind]
    tokens = _log_int(rng, low, top)
    B = min(_log_int(rng, 1, 16), max(1, tokens // 40))
    c.update(B=B, L=max(1, tokens // B))
    if kind == "forward":
        c["h0"] = rng.random() < 0.5
    if kind == "block":
        c["d_conv"] = rng.choice([4, 4, 4, 3, 2])
    return c


def _lengths(case):
    """Lengths of a packed batch: prompts spread over the logarithm up to the longest (the first
    one), decode tokens of one token each, shuffled."""
    r = random.Random(case["mix"])
    lens = [case["longest"]] + [_log_int(r, min(20, case["longest"]), case["longest"])
                                for _ in range(case["prompts"] - 1)]
    lens += [1] * case["decode"]
    r.shuffle(lens)
    return lens


class State:
    """A layer as a program holds it, with one call's inputs and outputs."""


def _workspace(nbytes):
    return torch.empty(max(int(nbytes), 16), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    kind, F, H, P, N, G, E, k = (case[n] for n in ("kind", "F", "H", "P", "N", "G", "E", "k"))
    S = 2 * G * N
    td = synth.torch_dtype(case["dtype"])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def randn(*shape, std=1.0, dtype=td):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32).mul_(std).to(dtype)

    def rand(*shape):
        return torch.rand(*shape, generator=gen, device="cuda")

    def empty(*shape, dtype=td):
        return torch.empty(*shape, dtype=dtype, device="cuda")

    s = State()
    s.kind = kind
    s.h = sb.swimba_create(F, H, P, N, G, E, k, case["chunk"],
                           sb.DTYPE_FP32 if case["dtype"] == "fp32" else sb.DTYPE_BF16)
    weakref.finalize(s, sb.swimba_destroy, s.h)
    A = -torch.exp(rand(H) * math.log(16.0))
    dt0 = torch.exp(rand(H) * math.log(100.0) + math.log(1e-3))
    dt_bias = dt0 + torch.log(-torch.expm1(-dt0))
    D = 1.0 + randn(H, std=0.1, dtype=torch.float32)
    s.w = sb.make_weights(randn(E, F, std=0.25 / math.sqrt(F)), randn(E, S, F, std=0.02), A, dt_bias, D)
    s.ints, s.floats = dict(dtype=torch.int32), dict(dtype=torch.float32)

    if kind == "decode":
        B = s.B = case["B"]
        s.u, s.x, s.dt = randn(B, F), randn(B, H, P), randn(B, H, std=0.5, dtype=torch.float32)
        s.state = randn(B, H, P, N, std=0.1, dtype=torch.float32)
        s.y, s.idx, s.tw = empty(B, H, P), empty(B, k, **s.ints), empty(B, k, **s.floats)
        s.ws = _workspace(sb.swimba_decode_workspace_bytes(s.h, B))
        return s

    if kind == "packed":
        s.cu = [0]
        for n in _lengths(case):
            s.cu.append(s.cu[-1] + n)
        T, nseq = s.cu[-1], len(s.cu) - 1
        s.u, s.x, s.dt = randn(T, F), randn(T, H, P), randn(T, H, std=0.5, dtype=torch.float32)
        s.h0 = randn(nseq, H, P, N, std=0.1, dtype=torch.float32)
        s.y, s.idx, s.tw = empty(T, H, P), empty(T, k, **s.ints), empty(T, k, **s.floats)
        s.hf = torch.empty_like(s.h0)
        s.ws = _workspace(sb.swimba_packed_workspace_bytes(s.h, s.cu))
        return s

    B, L = s.B, s.L = case["B"], case["L"]
    s.u = randn(B, L, F)
    s.idx, s.tw = empty(B, L, k, **s.ints), empty(B, L, k, **s.floats)
    s.hf = empty(B, H, P, N, **s.floats)
    if kind == "block":
        Dn, C = H * P, H * P + S
        W_in = randn(2 * Dn + H, F, std=1.0 / math.sqrt(F))
        W_in[2 * Dn:].mul_(0.25)        # the step-size rows are small, as a trained projection's are
        s.bw = sb.make_block_weights(W_in,
                                     randn(C, case["d_conv"], std=0.5, dtype=torch.float32),
                                     randn(C, std=0.1, dtype=torch.float32),
                                     1.0 + randn(Dn, std=0.1, dtype=torch.float32),
                                     randn(F, Dn, std=1.0 / math.sqrt(Dn)), case["d_conv"])
        s.conv_in, s.conv_out = randn(B, case["d_conv"] - 1, C), empty(B, case["d_conv"] - 1, C)
        s.h0 = randn(B, H, P, N, std=0.1, dtype=torch.float32)
        s.out = empty(B, L, F)
        s.ws = _workspace(sb.swimba_block_workspace_bytes(s.h, B, L))
        return s

    s.dt = randn(B, L, H, std=0.5, dtype=torch.float32)
    if kind == "slots":
        s.x = randn(k, B, L, H, P)
        s.bc, s.y = empty(B * L, k, S), empty(B, L, H, P)
        s.ws = _workspace(sb.swimba_workspace_bytes(s.h, B, L))
        s.ws2 = _workspace(sb.swimba_ssd_slots_workspace_bytes(s.h, B, L))
        return s

    s.x = randn(B, L, H, P)
    if kind == "backward":
        s.dy = randn(B, L, H, P)
        s.dWr, s.dWe = empty(E, F, **s.floats), empty(E, S, F, **s.floats)
        s.ws = _workspace(sb.swimba_backward_workspace_bytes(s.h, B, L))
        return s

    s.h0 = randn(B, H, P, N, std=0.1, dtype=torch.float32) if case["h0"] else None
    s.y = empty(B, L, H, P)
    s.ws = _workspace(sb.swimba_workspace_bytes(s.h, B, L))
    return s


def run(s):
    if s.kind == "forward":
        sb.swimba_forward(s.h, s.w, s.u, s.x, s.dt, s.h0, s.B, s.L, s.y, s.hf, s.idx, s.tw, s.ws)
        return dict(y=s.y, h=s.hf, idx=s.idx, w=s.tw)
    if s.kind == "decode":
        sb.swimba_decode_step(s.h, s.w, s.u, s.x, s.dt, s.state, s.B, s.y, s.idx, s.tw, s.ws)
        return dict(y=s.y, h=s.state, idx=s.idx, w=s.tw)
    if s.kind == "packed":
        sb.swimba_forward_packed(s.h, s.w, s.u, s.x, s.dt, s.h0, s.cu, s.y, s.hf, s.idx, s.tw, s.ws)
        return dict(y=s.y, h=s.hf, idx=s.idx, w=s.tw)
    if s.kind == "block":
        sb.swimba_block_forward(s.h, s.w, s.bw, s.u, s.conv_in, s.h0, s.B, s.L, s.out, s.conv_out, s.hf, s.idx, s.tw,
                                s.ws)
        return dict(out=s.out, conv=s.conv_out, h=s.hf, idx=s.idx, w=s.tw)
    if s.kind == "backward":
        sb.swimba_backward_weights(s.h, s.w, s.u, s.x, s.dt, None, s.dy, s.B, s.L, s.dWr, s.dWe, s.idx, s.ws)
        return dict(dW_router=s.dWr, dW_expert=s.dWe, idx=s.idx)
    sb.swimba_route_project_slots(s.h, s.w, s.u, s.B * s.L, s.bc, s.idx, s.tw, s.ws)
    sb.swimba_ssd_slots(s.h, s.w, s.x, s.bc, s.dt, None, s.B, s.L, s.y, s.hf, s.ws2)
    return dict(y=s.y, h=s.hf, idx=s.idx, w=s.tw, bc=s.bc)


def work(case):
    kind, F, H, P, N, G, E, k = (case[n] for n in ("kind", "F", "H", "P", "N", "G", "E", "k"))
    es = 4 if case["dtype"] == "fp32" else 2
    S, Dn = 2 * G * N, H * P
    if kind == "decode":
        B, T = case["B"], case["B"]
    elif kind == "packed":
        lens = _lengths(case)
        B, T = len(lens), sum(lens)
    else:
        B, T = case["B"], case["B"] * case["L"]
    state = B * H * P * N * 4
    weights = E * F * es + min(E, T * k) * S * F * es + 3 * H * 4
    routing = T * k * 8
    # per token: router logits, the k active projections, and the recurrence with one state of N per
    # channel: one multiply-add to advance every state entry and one to read it out
    proj, scan = 2 * T * k * F * S, 4 * T * H * P * N
    nbytes = T * F * es + T * H * 4 + weights + routing
    flops = 2 * T * F * E + proj + scan
    if kind == "decode":
        nbytes += 2 * T * Dn * es + 2 * state
    elif kind == "packed":
        nbytes += 2 * T * Dn * es + 2 * state
    elif kind == "forward":
        nbytes += 2 * T * Dn * es + state + (state if case["h0"] else 0)
    elif kind == "block":
        C = Dn + S
        nbytes += T * F * es - T * H * 4 + 2 * state + 2 * B * (case["d_conv"] - 1) * C * es
        nbytes += (2 * Dn + H) * F * es + F * Dn * es + C * (case["d_conv"] + 1) * 4 + Dn * 4
        flops += 2 * T * F * (2 * Dn + H) + 2 * T * Dn * F + 2 * T * C * case["d_conv"]
    elif kind == "backward":
        # x and dy in, gradients out; the projections serve the mix and dpi, the outer products
        # dW_expert; the recurrence runs forwards for dC and backwards for dB
        nbytes += 2 * T * Dn * es - T * k * 4 + E * S * F * 4 + E * F * 4
        flops += proj + scan + 2 * T * F * E
    else:
        nbytes += (k + 1) * T * Dn * es + T * k * S * es + state
        flops += (k - 1) * 2 * T * H * P * N
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the error measured against the same mathematics in 64 bits (per-timestep
    recurrence, autograd for the gradients) at a few hundred tokens.  fp32: 3e-7 on y and h, where
    sums in another order (chunks instead of single steps) stay below 1e-5.  bf16: y 1.7e-3 (its
    own rounding), end state up to 3.1e-3, gradients 4.0e-3, y without the skip term and the block's
    output 4.4e-3; the largest single deviations 5e-2 on a state, 7e-2 on y without the skip term.
    Routing may differ where two logits are closer than their rounding."""
    if case["dtype"] == "fp32":
        return {"rel": 1e-5, "max": 2e-4, "differ": 1e-4}
    if case["kind"] == "decode":
        return {"rel": 7e-3, "max": 3e-2, "differ": 1e-4}
    if case["kind"] in ("forward", "packed"):
        return {"rel": 1.2e-2, "max": 0.2, "differ": 1e-4}
    return {"rel": 1.6e-2, "max": 0.28, "differ": 1e-4}
