"""The kernels' dispatch rules and block edges: sizes on both sides of every line, against the oracle.

Tolerances are the suite's: 1e-4 of the largest value for fp32 arithmetic (parity.TOL for bf16 results)."""
import copy

import numpy as np
import pytest
import torch

import oracle
import parity
from paper_2605_13473_b200 import binding, run_inputs_bwd
from paper_2605_13473_b200.synth import OsdnHyper, draw

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("K", [64, 128])
@pytest.mark.parametrize("eta,keys,apf,clamp", [(0.3, "sparse", 2, 1), (0.003, "gauss", 2, 1), (0.05, "gauss", 1, 0), (0.3, "sparse", 3, 1)])
@pytest.mark.parametrize("L", [1, 31, 32, 33, 300])
def test_standalone_update_at_block_edges(L, eta, keys, apf, clamp, K):
    """Blocks of 32 tokens: the smallest sequence, one short of, at and past a block, more blocks than the ring holds."""
    hy = OsdnHyper(eta=eta, apf_mode=apf, clamp=clamp)
    inp = draw(f"edge_{L}", 7000 + L, [L, L], 2, K, K, "fp32", dense_B=2, hyper=hy, key_kind=keys,
               with_log_ret=apf >= 2, with_state=True)
    b = binding.DeviceBundle(inp, DEV, need_bwd=False)
    kt, d = torch.empty_like(b.k), torch.empty(2, 2, K, device=DEV)
    binding.osdn_precond_update(b.params, b.k, b.beta, b.log_ret if apf >= 2 else b.gate, b.precond_in, kt, d)
    ref = oracle.precond_update(hy, inp.seq_lens, inp.k, inp.beta, inp.gate, inp.log_ret, inp.precond_in)
    assert parity.err(d.cpu().numpy(), ref["precond_out"]) <= 1e-5
    assert parity.err(kt.cpu().numpy(), ref["ktil"]) <= 1e-5


def _all_outputs(inp, label, **kw):
    got = run_inputs_bwd(inp, **kw)
    ref = parity.oracle_all(inp, True, got["projection_masks"])
    parity.compare(got, ref, inp.io_dtype, parity.FWD_KEYS + parity.BWD_KEYS, label,
                   tensor_core=inp.io_dtype == "bf16" and inp.K == 128)


INF = float("inf")


@pytest.mark.parametrize("box", [(0.5, INF), (-INF, 2.0), (-INF, INF), (0.5, 3e38), (-1e4, 1e4), (-1.0, 2.0), (0.0, 2.0), (0.7, 0.7), (0.5, 0.5 + 2.0 ** -24)],
                         ids=lambda b: f"{b[0]:g}_{b[1]:g}")
@pytest.mark.parametrize("L,eta,apf", [(20, 0.3, 2), (300, 0.3, 2), (300, 0.3, 3), (300, 0.003, 1)])
def test_boxes_of_any_shape(box, L, eta, apf):
    """Open, wide, negative and empty boxes: the sums are taken in d itself there, and no bits are lost to d - d_min.
    Short sequences are walked, long ones go through the blocks; with the small step d rests on the lower face."""
    hy = OsdnHyper(eta=eta, apf_mode=apf, d_min=box[0], d_max=box[1])
    inp = draw(f"box_{L}", 7500 + L + apf, [L], 2, 64, 64, "fp32", dense_B=1, hyper=hy, key_kind="sparse" if eta > 0.1 else "gauss",
               with_dout=True, with_log_ret=apf >= 2, with_state_cotangents=True)
    _all_outputs(inp, f"box_{box}_{L}")
    b = binding.DeviceBundle(inp, DEV, need_bwd=False)
    kt, d = torch.empty_like(b.k), torch.empty(1, 2, 64, device=DEV)
    binding.osdn_precond_update(b.params, b.k, b.beta, b.log_ret if apf >= 2 else b.gate, None, kt, d)
    ref = oracle.precond_update(hy, inp.seq_lens, inp.k, inp.beta, inp.gate, inp.log_ret, None)
    assert parity.err(d.cpu().numpy(), ref["precond_out"]) <= 1e-5
    assert parity.err(kt.cpu().numpy(), ref["ktil"]) <= 1e-5


@pytest.mark.parametrize("beta", [1e-2, 1e-3, 1e-4, 1e-6])
def test_small_write_strengths_in_the_reverse_blocks(beta):
    """beta so small that the coupling of a block's tokens vanishes: lambda stands after one round, but the gradients of
    the write strengths and keys need the sums <lambda, k^2> of that lambda.  Bound: about ten fp32 roundings (2e-6)."""
    hy = OsdnHyper(eta=0.3, apf_mode=2)
    inp = draw("small_beta", 7600, [300], 2, 64, 64, "fp32", dense_B=1, hyper=hy, key_kind="sparse", with_dout=True,
               with_log_ret=True, with_state_cotangents=True)
    inp.beta = torch.full_like(inp.beta, beta)
    got = run_inputs_bwd(inp)
    ref = parity.oracle_all(inp, True, got["projection_masks"])
    for key in ("dbeta", "dk", "dlog_ret"):
        assert parity.err(got[key], ref[key], norm="l2") <= 2e-6, key


@pytest.mark.parametrize("shift", [3.0, 7.0])
@pytest.mark.parametrize("lens", [[2300], [700, 64, 0, 33, 1, 1500]])
def test_lists_of_processed_tokens(lens, shift):
    """Retention near one without a gate: runs off the face, then tokens that leave it one at a time, so that the passes
    work on dense runs, on lists with jumps and on short lists; more than one group of 2048 tokens, ragged packing."""
    hy = OsdnHyper(eta=0.003, apf_mode=2, beta_aware=0)
    inp = draw("lists", 7100 + int(shift), lens, 1, 64, 64, "fp32", dense_B=len(lens) == 1, hyper=hy, gate_kind="zero",
               with_dout=True, with_log_ret=True, log_ret_shift=shift, with_state_cotangents=True)
    _all_outputs(inp, f"lists_{len(lens)}_{shift}")


@pytest.mark.parametrize("io,K", [("bf16", 128), ("fp32", 128), ("fp32", 64)])
@pytest.mark.parametrize("apf,eta,shift", [(2, 0.3, 5.0), (2, 0.003, 7.0), (3, 0.3, 3.0), (1, 0.003, 5.0)])
def test_more_chains_than_sms(io, K, apf, eta, shift):
    """Beyond one chain per SM the preconditioner passes share SMs: bit for bit what the few chains compute, and the
    oracle's write keys.  300 tokens: walked lists, blocks, more blocks than the short ring holds, a ragged last one."""
    hy = OsdnHyper(eta=eta, apf_mode=apf, beta_aware=int(shift != 7.0))
    few = draw("many", 7800 + apf, [300, 300], 4, K, K, io, dense_B=2, hyper=hy, key_kind="sparse" if eta > 0.1 else "gauss",
               gate_kind="zero" if shift == 7.0 else "softplus", with_log_ret=apf >= 2, log_ret_shift=shift, with_state=True)
    results = {}
    for rep in (1, 20):   # 8 and 160 chains
        more = lambda x: None if x is None else x.repeat(rep, *[1] * (x.dim() - 1)).contiguous()
        big = copy.copy(few)
        big.seq_lens, big.dense_B = few.seq_lens * rep, 2 * rep
        for name in ("q", "k", "v", "beta", "gate", "log_ret", "init_state", "precond_in"):
            setattr(big, name, more(getattr(few, name)))
        b = binding.DeviceBundle(big, DEV, need_bwd=True)
        b.fwd(save=True)
        kt, d, ratio = torch.empty_like(b.k), torch.empty_like(b.precond_out), torch.empty_like(b.beta)
        ret = b.log_ret if apf >= 2 else b.gate
        binding.osdn_precond_update(b.params, b.k, b.beta, ret, b.precond_in, kt, d)
        binding.osdn_residual_ratio(b.params, b.k, b.beta, ret, b.precond_in, ratio, None)
        torch.cuda.synchronize()
        assert b.device_status() == 0
        results[rep] = [kt, d, ratio, b.precond_out, b.projection_masks()]
    for x, y in zip(results[1], results[20]):
        assert torch.equal(y, x.repeat(20, *[1] * (x.dim() - 1)))
    ref = oracle.precond_update(hy, few.seq_lens, few.k, few.beta, few.gate, few.log_ret, few.precond_in)
    assert parity.err(results[1][1].cpu().numpy(), ref["precond_out"]) <= 1e-5
    assert parity.err(results[1][0].float().cpu().numpy(), ref["ktil"]) <= (1e-5 if io == "fp32" else 2.0 ** -8)


@pytest.mark.parametrize("io,flags", [("bf16", 0), ("fp32", 0), ("bf16", binding.FLAG_FORCE_SIMT)])
def test_built_in_scratch_takes_8192_token_heads(io, flags):
    """osdn_fwd_static at 1024 tokens, 8 heads of 128, in every kernel family: the results of osdn_fwd, bit for bit."""
    inp = draw("static", 7700, [1024], 8, 128, 128, io, dense_B=1, with_state=True)
    b = binding.DeviceBundle(inp, DEV, need_bwd=False, flags=flags)
    b.fwd()
    want = [b.out.clone(), b.final_state.clone(), b.precond_out.clone()]
    for x in (b.out, b.final_state, b.precond_out):
        x.zero_()
    rc = binding.osdn_fwd_static(b.params, b.q, b.k, b.v, b.beta, b.gate, None, b.init_state, b.precond_in, b.out, b.final_state, b.precond_out)
    torch.cuda.synchronize()
    assert rc == 0 and binding.osdn_read_static_status() == 0
    for x, y in zip(want, (b.out, b.final_state, b.precond_out)):
        assert torch.equal(x, y)


@pytest.mark.parametrize("io,K", [("fp32", 64), ("fp32", 128), ("bf16", 64)])
def test_chains_in_wide_slices(io, K):
    """Enough chains for the wide slices of the CUDA-core state chains (the other cases have few and take the narrow ones)."""
    hy = OsdnHyper(eta=0.003, apf_mode=1)
    inp = draw("wide", 7200 + K, [70] * 50, 6, K, 64, io, dense_B=50, hyper=hy, with_dout=True, with_state=True,
               with_state_cotangents=True)
    _all_outputs(inp, f"wide_{io}_{K}")


@pytest.mark.parametrize("io,cg,gates", [("fp32", 0, "softplus"), ("bf16", 0, "softplus"), ("fp32", 1, "softplus"), ("fp32", 1, "strong"), ("bf16", 1, "mixture")])
def test_chains_in_wide_slices_of_128_rows(io, cg, gates):
    """K = V = 128 in wide slices, two to a chain (from 38 chains on): scalar and channel gates, weak and strong."""
    hy = OsdnHyper(eta=0.003, apf_mode=2, channel_gate=cg)
    inp = draw("wide128", 7250 + cg, [150] * 8, 5, 128, 128, io, dense_B=8, hyper=hy, gate_kind=gates, with_dout=True,
               with_log_ret=True, with_state=True, with_state_cotangents=True)
    got = run_inputs_bwd(inp, flags=binding.FLAG_FORCE_SIMT)
    ref = parity.oracle_all(inp, True, got["projection_masks"])
    parity.compare(got, ref, io, parity.FWD_KEYS + parity.BWD_KEYS, f"wide128_{io}_{cg}_{gates}")


@pytest.mark.parametrize("B,L", [(37, 150), (38, 150), (37, 64), (9, 129)])
@pytest.mark.parametrize("cg", [0, 1])
def test_chains_on_both_sides_of_the_slice_rule(B, L, cg):
    """K = V = 128: the most chains that narrow slices take (four waves), one more, one chunk only, one token past two chunks."""
    hy = OsdnHyper(eta=0.003, apf_mode=2, channel_gate=cg)
    inp = draw(f"slices_{B}_{L}", 7270 + B + cg, [L] * B, 1, 128, 128, "fp32", dense_B=B, hyper=hy, with_dout=True,
               with_log_ret=True, with_state=True, with_state_cotangents=True)
    _all_outputs(inp, f"slices_{B}_{L}_{cg}")


def test_backward_twice_on_the_same_residuals():
    """The backward leaves its tile queue as it found it."""
    hy = OsdnHyper(eta=0.003, apf_mode=1)
    inp = draw("twice", 7300, [200, 200], 2, 128, 128, "bf16", dense_B=2, hyper=hy, with_dout=True)
    b = binding.DeviceBundle(inp, DEV, need_bwd=True)
    b.fwd(save=True)
    seen = []
    for _ in range(2):
        for x in (b.dq, b.dk, b.dv):
            x.fill_(float("nan"))
        b.bwd(residuals_valid=True)
        torch.cuda.synchronize()
        assert b.device_status() == 0
        seen.append([x.clone() for x in (b.dq, b.dk, b.dv)])
    for x, y in zip(*seen):
        assert not torch.isnan(x.float()).any() and torch.equal(x, y)


@pytest.mark.parametrize("kind", ["gated", "moving", "mixture"])
@pytest.mark.parametrize("lens", [[1], [63, 65], [64, 64], [129, 0, 191]], ids=str)
def test_backward_tiles_at_their_edges(lens, kind):
    """Chunk-local backward on the tensor cores: tiles of 1, 63, 64 tokens and a remainder, every step skipped, some and none;
    twice on the same residuals, bit for bit (the second time every counter, flag and staging area has been used)."""
    hy = OsdnHyper(eta=0.3 if kind == "moving" else 0.003, apf_mode=2 if kind == "moving" else 1)
    inp = draw(f"tiles_{kind}", 7900 + len(lens), lens, 2, 128, 128, "bf16", dense_B=len(lens) if len(set(lens)) == 1 else 0, hyper=hy,
               key_kind="sparse" if kind == "moving" else "gauss", gate_kind="mixture" if kind == "mixture" else "softplus",
               with_dout=True, with_log_ret=kind == "moving", with_state=True, with_state_cotangents=True)
    got = run_inputs_bwd(inp)
    ref = parity.oracle_all(inp, True, got["projection_masks"])
    parity.compare(got, ref, "bf16", parity.BWD_KEYS, f"tiles_{kind}_{lens}", tensor_core=True)
    b = binding.DeviceBundle(inp, DEV, need_bwd=True)
    b.fwd(save=True)
    seen = []
    for _ in range(2):
        for x in (b.dq, b.dk, b.dv):
            x.fill_(float("nan"))
        b.bwd(residuals_valid=True)
        torch.cuda.synchronize()
        assert b.device_status() == 0
        seen.append([x.clone() for x in (b.dq, b.dk, b.dv)])
    for x, y in zip(*seen):
        assert not torch.isnan(x.float()).any() and torch.equal(x, y)


def _follows(call, spoil, outputs):
    """What `call` writes to `outputs` with its kernels held apart (the library's stage events stand between them), against one
    call right behind `spoil`, which leaves other valid results everywhere, and one replayed from a graph behind it."""
    spoil()
    binding.stage_timing_enable(True)
    call()
    torch.cuda.synchronize()
    binding.stage_timing_enable(False)
    want = [x.clone() for x in outputs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for run in (call, graph.replay) * 2:
        spoil()
        torch.cuda.synchronize()
        assert not any(torch.equal(x, y) for x, y in zip(want, outputs))
        run()
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(want, outputs))


@pytest.mark.parametrize("io,K,cg,lens", [("bf16", 128, 0, [130, 130]), ("bf16", 128, 0, [70, 0, 200]), ("bf16", 128, 0, [70] * 60), ("fp32", 64, 0, [130, 130]),
                                          ("fp32", 64, 0, [70, 0, 200]), ("fp32", 128, 0, [130] * 24), ("fp32", 64, 1, [130])])
def test_calls_follow_the_work_before_them(io, K, cg, lens):
    """Every kernel of a call, the first one too, may be launched while the one before it in the stream runs.  Outputs and
    workspace hold the results of other inputs when the call is enqueued, behind the kernels that write its own: a kernel that
    does not wait for the one before it reads them."""
    hy = OsdnHyper(eta=0.3, apf_mode=2, channel_gate=cg)
    inp, other = (draw(f"follow_{io}_{cg}", 7950 + x + len(lens), lens, 2, K, K, io, dense_B=len(lens) if len(set(lens)) == 1 else 0, hyper=hy, key_kind="sparse",
                       with_dout=True, with_log_ret=True, with_state=True, with_state_cotangents=True) for x in (0, 100))
    b, o = binding.DeviceBundle(inp, DEV), binding.DeviceBundle(other, DEV)
    names = ("q", "k", "v", "beta", "gate", "log_ret", "init_state", "precond_in", "dout", "dfinal_state", "dprecond_out")
    kept = {x: getattr(b, x).clone() for x in names}

    def run(src):
        for x in names:
            torch.mul(src[x], 1, out=getattr(b, x))
        b.fwd(save=True)
        b.bwd(residuals_valid=True)

    _follows(lambda: run(kept), lambda: run({x: getattr(o, x) for x in names}),
             [b.out, b.final_state, b.precond_out, b.dq, b.dk, b.dv, b.dbeta, b.dgate, b.dlog_ret, b.dinit_state, b.dprecond_in])
    assert b.device_status() == 0


@pytest.mark.parametrize("B", [2, 90])
def test_standalone_update_follows_the_work_before_it(B):
    """As above, the stand-alone update with its chains one and three to an SM."""
    inp, other = (draw("follow_update", 7970 + x, [100] * B, 2, 128, 128, "bf16", dense_B=B, hyper=OsdnHyper(eta=0.3, apf_mode=2), key_kind="sparse",
                       with_log_ret=True, with_state=True) for x in (0, 100))
    b, o = (binding.DeviceBundle(x, DEV, need_bwd=False) for x in (inp, other))
    kt, d = torch.empty_like(b.k), torch.empty_like(b.precond_in)
    names = ("k", "beta", "log_ret", "precond_in")
    kept = {x: getattr(b, x).clone() for x in names}

    def run(src):
        for x in names:
            torch.mul(src[x], 1, out=getattr(b, x))
        binding.osdn_precond_update(b.params, b.k, b.beta, b.log_ret, b.precond_in, kt, d)

    _follows(lambda: run(kept), lambda: run({x: getattr(o, x) for x in names}), [kt, d])


@pytest.mark.parametrize("B,H,L", [(49, 3, 8), (37, 4, 9), (191, 1, 1), (192, 1, 1), (50, 3, 17), (103, 1, 1), (104, 1, 1), (103, 1, 9), (52, 2, 9)])
@pytest.mark.parametrize("io,K,V,apf", [("bf16", 128, 128, 1), ("fp32", 64, 128, 2), ("fp32", 128, 64, 3)])
def test_decode_on_both_sides_of_its_dispatch(B, H, L, io, K, V, apf):
    """103 / 104 chains, with one token and several (and well beyond); blocks of eight tokens: at, one past, two and one past."""
    hy = OsdnHyper(eta=0.3, apf_mode=apf)
    inp = draw(f"dec_{B}_{L}", 7400 + B + L, [L] * B, H, K, V, io, dense_B=B, hyper=hy, with_log_ret=apf >= 2, with_state=True)
    p = binding.make_params(B=B, T=L, H=H, K=K, V=V, io_dtype=io, hyper=hy)
    dt = torch.bfloat16 if io == "bf16" else torch.float32
    q, k, v = (x.to(DEV, dt).contiguous() for x in (inp.q, inp.k, inp.v))
    beta, gate = inp.beta.float().to(DEV), inp.gate.float().to(DEV)
    lr = None if inp.log_ret is None else inp.log_ret.float().to(DEV)
    S, d = inp.init_state.float().to(DEV).clone(), inp.precond_in.float().to(DEV).clone()
    out = torch.empty(B * L, H, V, device=DEV, dtype=dt)
    binding.osdn_decode_step(p, q, k, v, beta, gate, lr, S, d, out)
    ref = oracle.fwd_inputs(inp)
    assert parity.err(S.cpu().numpy(), ref["final_state"]) <= 1e-4
    assert parity.err(d.cpu().numpy(), ref["precond_out"]) <= 1e-4
    assert parity.err(out.float().cpu().numpy(), ref["out"]) <= parity.TOL[io]


def test_beta_gradient_takes_the_scores_in_fp32():
    """One chunk whose operands are small integers, exact in bf16, and whose score gradients (up to eleven bits) are not: keys
    one-hot and shared by two tokens each, beta 1/2, no gate, d = 1.  Sums of 128 integers are exact in fp32, so dbeta is."""
    inp = draw("exact_beta", 7990, [64], 2, 128, 128, "bf16", dense_B=1, hyper=OsdnHyper(eta=0.0, apf_mode=0, scale=1.0), with_dout=True)
    gen = torch.Generator().manual_seed(7991)
    inp.q = inp.k = torch.nn.functional.one_hot(torch.arange(64) // 2, 128).float()[:, None].expand(64, 2, 128).contiguous()
    inp.v, inp.dout = (torch.randint(-15, 16, (64, 2, 128), generator=gen).float() for _ in range(2))
    inp.beta = torch.full((64, 2), 0.5)
    inp.gate = torch.zeros(64, 2)
    got = run_inputs_bwd(inp)
    ref = oracle.bwd_inputs(inp)
    assert float(np.abs(ref["dbeta"][1::2]).max()) > 256.0
    assert parity.err(got["dbeta"], ref["dbeta"]) <= 1e-6
