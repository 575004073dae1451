"""The work a user of this library has it do, as a list of measured cases.

Every case goes through the public calls of ``paper_2605_13473_b200``.  Shapes are those of the benchmark
configurations (the 340M layer: 8 heads of 128, rows of 2048 tokens; the 1.3B layer: 16 heads, rows of 4096;
packed rows of 131072 tokens) and of the decode, fp32 and channel-gate tests.  ``draw`` gives further cases
of the same ranges: batches, lengths that are no multiple of the 64-token chunk, heads, head sizes.

A case: ``path`` (which calls), ``B`` sequences of ``T`` tokens (``packed``: T tokens in ``nseq`` sequences),
``H`` heads, ``D`` = dk = dv, ``io`` dtype, and ``setting``, the layer variant and its value distributions:

  gated     the gate is the retention as well, step 0.003: after a few tokens the preconditioner rests
            on the lower face of its box
  mixture   the same with gates that are mostly near zero and now and then strong (the 1.3B configuration)
  moving    step 0.3, sparse keys, a retention of its own: the preconditioner moves at every token
  ungated   g = 0, retention near 0.999, non-beta-aware step (the paper's ungated 1.3B setting)
  channel   one gate per key channel, constant retention 0.999 (OSKDA)
"""
from __future__ import annotations

import math

import torch

from paper_2605_13473_b200 import (make_params, osdn_bwd, osdn_decode_step, osdn_fwd, osdn_precond_update,
                                   osdn_workspace_bytes)
from paper_2605_13473_b200.binding import (FLAG_RESIDUALS_VALID, FLAG_SAVE_RESIDUALS, osdn_kda_bwd, osdn_kda_fwd,
                                           osdn_kda_workspace_bytes)
from paper_2605_13473_b200.synth import OsdnHyper, varlen_lengths

HYPER = {
    "gated": OsdnHyper(eta=0.003, apf_mode=1),
    "mixture": OsdnHyper(eta=0.003, apf_mode=1),
    "moving": OsdnHyper(eta=0.3, apf_mode=2),
    "ungated": OsdnHyper(eta=0.003, apf_mode=2, beta_aware=0),
    "channel": OsdnHyper(eta=0.003, apf_mode=2, channel_gate=1),
}


def _case(path, B, T, H, D, io, setting, **more):
    return dict(path=path, B=B, T=T, H=H, D=D, io=io, setting=setting, **more)


def listed():
    return [
        # one user's generation, one token: latency of a single call
        dict(name="decode_1_seq", **_case("decode", 1, 1, 8, 128, "bf16", "gated")),
        # a serving batch, one token each: the cached states stream through the chip once
        dict(name="decode_512_seqs", **_case("decode", 512, 1, 8, 128, "bf16", "gated")),
        # the prompt of one request (2048 tokens), whose state and preconditioner go to the decode cache
        dict(name="prefill_1x2048", **_case("fwd", 1, 2048, 8, 128, "bf16", "gated")),
        # the 340M layer's forward over a batch: evaluation, prefill of a batch
        dict(name="fwd_340m", **_case("fwd", 8, 2048, 8, 128, "bf16", "gated")),
        # the 340M layer's training step, the headline benchmark
        dict(name="train_340m", **_case("train", 8, 2048, 8, 128, "bf16", "gated")),
        # the 1.3B layer's training step
        dict(name="train_1p3b", **_case("train", 4, 4096, 16, 128, "bf16", "mixture")),
        # packed training rows: eight documents of 976 to 32768 tokens, none a multiple of the chunk but the longest
        dict(name="train_packed_131k", **_case("train", 1, 131072, 8, 128, "bf16", "gated", nseq=8, lens_seed=4)),
        # training with a preconditioner that really moves
        dict(name="train_moving_340m", **_case("train", 8, 2048, 8, 128, "bf16", "moving")),
        # the ungated 1.3B setting
        dict(name="train_ungated_1p3b", **_case("train", 4, 4096, 16, 128, "bf16", "ungated")),
        # the channel-gate extension at the 340M layer's training shape
        dict(name="train_oskda_340m", **_case("oskda", 8, 2048, 8, 128, "bf16", "channel")),
        # fp32 training at the small head size, lengths with a ragged last chunk (gradient checks, small models)
        dict(name="train_fp32_d64", **_case("train", 4, 1000, 4, 64, "fp32", "gated")),
        # phase 1 alone with its write keys, for a caller that runs its own delta-rule kernel
        dict(name="precond_update_340m", **_case("precond", 8, 2048, 8, 128, "bf16", "moving")),
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], even over its logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    path = rng.choice(["decode", "decode", "fwd", "fwd", "train", "train", "train", "packed", "packed",
                       "oskda", "fp32", "precond"])
    H = rng.choice([2, 3, 4, 6, 8, 8, 12, 16])
    if path == "decode":      # a few tokens per call: speculative or multi-token steps
        return _case("decode", _log_int(rng, 1, 512), rng.choice([1, 1, 1, 2, 4, 7, 16]), H,
                     rng.choice([128, 128, 128, 64]), rng.choice(["bf16", "bf16", "fp32"]),
                     rng.choice(["gated", "moving"]))
    if path == "packed":      # documents of very different lengths; the tokens of the listed row at most
        return _case("train", 1, _log_int(rng, 3000, 131072), min(H, 8), 128, "bf16", "gated",
                     nseq=rng.randint(5, 24), lens_seed=rng.randrange(1 << 20))
    if path == "fp32":        # the CUDA-core family
        T = _log_int(rng, 60, 1500)
        return _case("train", _log_int(rng, 1, max(1, 24000 // (T * H))), T, H, rng.choice([64, 64, 128]), "fp32",
                     rng.choice(["gated", "moving"]))
    most = 131072             # token-heads of the listed 340M shape
    if path == "fwd":
        T = _log_int(rng, 50, 8192)
        setting = rng.choice(["gated", "gated", "mixture", "moving", "ungated"])
    elif path == "train":
        T, most = _log_int(rng, 100, 4096), 2 * most
        setting = rng.choice(["gated", "gated", "mixture", "moving", "ungated"])
    elif path == "precond":
        T, setting = _log_int(rng, 100, 4096), rng.choice(["gated", "moving", "ungated"])
    else:
        T, setting = _log_int(rng, 60, 2048), "channel"
    B = _log_int(rng, 1, min(64, max(1, most // (T * H))))
    return _case(path, B, T, H, 128, "bf16", setting)


def _lengths(case):
    if "nseq" not in case:
        return [case["T"]] * case["B"]
    total = case["T"]
    return varlen_lengths(case["lens_seed"], case["nseq"], max(1, total // 256), total // 4, total)


def prepare(case, seed):
    """Inputs, output buffers, parameters and the workspace of one case on the GPU."""
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    path, setting, B, T, H, D = (case[x] for x in ("path", "setting", "B", "T", "H", "D"))
    hy = HYPER[setting]
    io = torch.bfloat16 if case["io"] == "bf16" else torch.float32
    N, S = B * T, case.get("nseq", B)

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device=dev)

    def rand(*shape):
        return torch.rand(*shape, generator=gen, device=dev)

    def unit(x):
        return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-12)

    s = dict(path=path)
    k = randn(N, H, D)
    if setting == "moving":   # about a tenth of a key's coordinates, one at least
        k = k * (rand(N, H, D) < 0.10).logical_or_(rand(N, H, D).argmax(-1, keepdim=True) == torch.arange(D, device=dev))
    s["k"] = unit(k).to(io)
    s["beta"] = torch.sigmoid(randn(N, H))
    if setting == "mixture":
        gate = torch.where(rand(N, H) < 0.10, -3.0 + 2.0 * rand(N, H), -0.005 * randn(N, H).abs())
    elif setting == "ungated":
        gate = torch.zeros(N, H, device=dev)
    else:
        gate = -0.1 * torch.nn.functional.softplus(randn(N, H))
    if setting == "channel":
        gate = gate.unsqueeze(-1) * (0.25 + 1.5 * rand(N, H, D))
    s["gate"] = gate
    s["log_ret"] = None
    if setting == "channel":
        s["log_ret"] = torch.full((N, H), math.log(0.999), device=dev)
    elif setting in ("moving", "ungated"):
        s["log_ret"] = torch.nn.functional.logsigmoid(randn(N, H) + (7.0 if setting == "ungated" else 5.0))

    cu = None
    if "nseq" in case:
        cu = torch.tensor([0] + _lengths(case), dtype=torch.int32).cumsum(0, dtype=torch.int32).to(dev)
        s["cu"] = cu
    shape = dict(B=B, T=T, H=H, K=D, V=D, io_dtype=case["io"], hyper=hy, cu_seqlens=cu)
    s["p"] = make_params(**shape)

    if path == "precond":
        s["precond_in"] = hy.d_min + (hy.d_max - hy.d_min) * rand(S, H, D)
        s["k_tilde"] = torch.empty(N, H, D, device=dev, dtype=io)
        s["precond_out"] = torch.empty(S, H, D, device=dev)
        return s

    s["q"] = unit(randn(N, H, D)).to(io)
    s["v"] = randn(N, H, D).to(io)
    s["out"] = torch.empty(N, H, D, device=dev, dtype=io)
    if path == "decode":      # the caches that earlier tokens of each sequence have left
        s["state"] = 0.5 * randn(B, H, D, D)
        s["precond"] = hy.d_min + (hy.d_max - hy.d_min) * rand(B, H, D)
        return s

    s["final_state"] = torch.empty(S, H, D, D, device=dev)
    s["precond_out"] = torch.empty(S, H, D, device=dev)
    train = path != "fwd"
    nbytes = (osdn_kda_workspace_bytes if path == "oskda" else osdn_workspace_bytes)(s["p"], train)
    s["workspace"] = torch.empty(nbytes, device=dev, dtype=torch.uint8)
    if train:
        s["p"] = make_params(**shape, flags=FLAG_SAVE_RESIDUALS)
        s["p_bwd"] = make_params(**shape, flags=FLAG_RESIDUALS_VALID)
        s["dout"] = randn(N, H, D).to(io)
        for name in ("dq", "dk", "dv"):
            s[name] = torch.empty(N, H, D, device=dev, dtype=io)
        s["dbeta"] = torch.empty(N, H, device=dev)
        s["dgate"] = torch.empty_like(s["gate"])
        s["dlog_ret"] = None if s["log_ret"] is None else torch.empty_like(s["log_ret"])
        s["dinit_state"] = torch.empty(S, H, D, D, device=dev)
        s["dprecond_in"] = torch.empty(S, H, D, device=dev)
    return s


_FWD_OUT = ("out", "final_state", "precond_out")
_BWD_OUT = ("dq", "dk", "dv", "dbeta", "dgate", "dlog_ret", "dinit_state", "dprecond_in")


def run(s):
    path = s["path"]
    if path == "decode":
        osdn_decode_step(s["p"], s["q"], s["k"], s["v"], s["beta"], s["gate"], s["log_ret"], s["state"],
                         s["precond"], s["out"])
        return [s["out"], s["state"], s["precond"]]
    if path == "precond":
        osdn_precond_update(s["p"], s["k"], s["beta"], s["log_ret"] if s["log_ret"] is not None else s["gate"],
                            s["precond_in"], s["k_tilde"], s["precond_out"])
        return [s["k_tilde"], s["precond_out"]]
    fwd, bwd = (osdn_kda_fwd, osdn_kda_bwd) if path == "oskda" else (osdn_fwd, osdn_bwd)
    fwd(s["p"], s["q"], s["k"], s["v"], s["beta"], s["gate"], s["log_ret"], None, None, s["out"], s["final_state"],
        s["precond_out"], s["workspace"])
    if path == "fwd":
        return [s[x] for x in _FWD_OUT]
    bwd(s["p_bwd"], s["q"], s["k"], s["v"], s["beta"], s["gate"], s["log_ret"], None, None, s["dout"], None, None,
        s["dq"], s["dk"], s["dv"], s["dbeta"], s["dgate"], s["dlog_ret"], s["dinit_state"], s["dprecond_in"],
        s["workspace"])
    return [s[x] for x in _FWD_OUT + _BWD_OUT if s[x] is not None]


def work(case):
    """Every input read once and every output written once; the operations of the token recurrence: per token
    and head one product with the state each for the read, the write and the output (forward), four more each
    for the adjoint with the state replayed by its read and its write (backward)."""
    path, D = case["path"], case["D"]
    nh = case["B"] * case["T"] * case["H"]
    sh = case.get("nseq", case["B"]) * case["H"]
    e = 2 if case["io"] == "bf16" else 4
    ret = 4 if HYPER[case["setting"]].apf_mode == 2 else 0
    gate = 4 * D if path == "oskda" else 4
    if path == "precond":
        return dict(bytes=nh * (2 * e * D + 8) + sh * 8 * D, flops=nh * 8 * D)
    if path == "decode":
        return dict(bytes=nh * (4 * e * D + 4 + gate + ret) + sh * (8 * D * D + 8 * D), flops=nh * (6 * D * D + 8 * D))
    fwd = nh * (4 * e * D + 4 + gate + ret) + sh * (4 * D * D + 4 * D)
    if path == "fwd":
        return dict(bytes=fwd, flops=nh * (6 * D * D + 8 * D))
    bwd = nh * (4 * e * D + 4 + gate + ret) + sh * (4 * D * D + 4 * D)
    return dict(bytes=fwd + bwd, flops=nh * (22 * D * D + 24 * D))


def tolerance(case):
    """Outputs against those of another correct implementation at the same precision."""
    if case["io"] == "fp32":
        return {"rel": 1e-4}      # fp32 sums through a chunk's unit-triangular system and a long recurrence
    if case["path"] in ("decode", "precond", "oskda"):
        return {"rel": 5e-3}      # fp32 arithmetic, results stored in bf16
    return {"rel": 1e-2}          # bf16 operands, fp32 accumulation
