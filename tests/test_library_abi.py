"""CPU-side checks of the C ABI: the library builds, loads, exports every declared symbol,
and validates its arguments before touching a device."""
import ctypes
import os
import re

import pytest

import paper_2605_13473_b200 as osdn
from paper_2605_13473_b200 import binding
from paper_2605_13473_b200.build import build
from paper_2605_13473_b200.synth import OsdnHyper

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build()
    return osdn.load_library()


def test_exports_every_declared_symbol(lib):
    header = open(os.path.join(ROOT, "include", "osdn.h")).read()
    header = re.sub(r"/\*.*?\*/", "", header, flags=re.S)
    declared = set(re.findall(r"\b(osdn_[a-z_]+)\s*\(", header))
    assert declared == set(binding.EXPORTS), declared ^ set(binding.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_workspace_sizes_and_validation(lib):
    hy = OsdnHyper()
    p = osdn.make_params(B=8, T=2048, H=8, K=128, V=128, io_dtype="bf16", hyper=hy)
    fwd_bytes = osdn.osdn_workspace_bytes(p, False)
    bwd_bytes = osdn.osdn_workspace_bytes(p, True)
    assert 0 < fwd_bytes < bwd_bytes < 8 << 30
    assert osdn.osdn_host_staging_bytes(p, True) > bwd_bytes
    for bad in (dict(K=96), dict(V=32), dict(T=0)):
        kw = dict(B=1, T=64, H=1, K=64, V=64)
        kw.update(bad)
        q = osdn.make_params(io_dtype="fp32", hyper=hy, **kw)
        assert osdn.osdn_workspace_bytes(q, False) == 0
    q = osdn.make_params(B=1, T=64, H=1, K=64, V=64, io_dtype="fp32", hyper=hy)
    q.chunk = 32
    assert osdn.osdn_workspace_bytes(q, False) == 0


@pytest.mark.parametrize("K", [64, 128])
@pytest.mark.parametrize("V", [64, 128])
def test_forward_workspace_has_a_ceiling(lib, K, V):
    """The forward's scratch is at most the write keys, two 64 x 64 tiles, W, U, dU and the chunk states side by side (with
    two scalars per token-head, the flags and the table), whatever the shape: what fits the built-in scratch stays accepted."""
    up = lambda n: -(-n // 256) * 256
    for B, T, nseq in ((1, 1, 0), (1, 64, 0), (3, 65, 0), (25, 1, 0), (1, 1024, 0), (8, 2048, 0), (1, 1024, 9)):
        for H in (1, 3, 8):
            for io in ("fp32", "bf16"):
                p = osdn.make_params(B=B, T=T, H=H, K=K, V=V, io_dtype=io, hyper=OsdnHyper())
                if nseq:
                    p.nseq, p.cu_seqlens = nseq, 0x1000   # never dereferenced
                S, n = nseq or B, B * T
                nt = n // 64 + S if nseq else B * (-(-T // 64))
                regions = [256, 4 * (4 * S + 1 + 6 * nt + 4), 4 * n * H, 4 * n * H, 8 * nt * H, 4 * n * H * K] + [4 * nt * H * 4096] * 2
                regions += [4 * nt * H * 64 * K] + [4 * nt * H * 64 * V] * 2 + [4 * nt * H * K * V]
                assert osdn.osdn_workspace_bytes(p, False) <= sum(map(up, regions)), (B, T, H, io, nseq)
    p = osdn.make_params(B=1, T=1024, H=8, K=128, V=128, io_dtype="bf16", hyper=OsdnHyper())
    assert osdn.osdn_workspace_bytes(p, False) <= binding.STATIC_SCRATCH_BYTES


def test_calls_reject_bad_arguments_before_any_launch(lib):
    hy = OsdnHyper()
    p = osdn.make_params(B=1, T=64, H=1, K=64, V=64, io_dtype="fp32", hyper=hy)
    null = ctypes.c_void_p(None)
    rc = lib.osdn_fwd(ctypes.byref(p), *([null] * 11), null, ctypes.c_size_t(0), null)
    assert rc == -1 and osdn.status_string(rc) == "invalid argument"
    fake = ctypes.c_void_p(0x1000)      # never dereferenced: validation fails first
    odd = ctypes.c_void_p(0x1004)
    rc = lib.osdn_fwd(ctypes.byref(p), odd, fake, fake, fake, fake, null, null, null, fake, null, null,
                      fake, ctypes.c_size_t(1 << 30), null)
    assert rc == -3
    rc = lib.osdn_fwd(ctypes.byref(p), fake, fake, fake, fake, fake, null, null, null, fake, null, null,
                      fake, ctypes.c_size_t(16), null)
    assert rc == -4
    p.apf_mode = 2
    rc = lib.osdn_fwd(ctypes.byref(p), fake, fake, fake, fake, fake, null, null, null, fake, null, null,
                      fake, ctypes.c_size_t(1 << 30), null)
    assert rc == -1                     # separate retention requested but not given
    p.apf_mode = 3
    rc = lib.osdn_fwd(ctypes.byref(p), fake, fake, fake, fake, fake, null, null, null, fake, null, null,
                      fake, ctypes.c_size_t(1 << 30), null)
    assert rc == -1                     # vector retention requested but not given
    p.apf_mode = 4
    assert osdn.osdn_workspace_bytes(p, False) == 0   # no such retention mode
    p.apf_mode = 1
    p.nseq = 3                          # var-len without cu_seqlens
    rc = lib.osdn_precond_update(ctypes.byref(p), fake, fake, fake, null, null, fake, null)
    assert rc == -1
    assert osdn.status_string(-2) == "unsupported shape"
    # the residual-ratio diagnostic: no output requested, misaligned output
    pr = osdn.make_params(B=1, T=64, H=1, K=64, V=64, io_dtype="fp32", hyper=hy)
    rc = lib.osdn_residual_ratio(ctypes.byref(pr), fake, fake, fake, null, null, null, null, null)
    assert rc == -1
    rc = lib.osdn_residual_ratio(ctypes.byref(pr), fake, fake, fake, null, odd, null, null, null)
    assert rc == -3
    # the recurrent step: missing cache, misaligned pointer, missing separate retention, packed batch
    p = osdn.make_params(B=2, T=1, H=1, K=128, V=128, io_dtype="bf16", hyper=hy)
    rc = lib.osdn_decode_step(ctypes.byref(p), fake, fake, fake, fake, fake, null, null, fake, fake, null)
    assert rc == -1
    rc = lib.osdn_decode_step(ctypes.byref(p), fake, fake, fake, fake, fake, null, odd, fake, fake, null)
    assert rc == -3
    p.apf_mode = 2
    rc = lib.osdn_decode_step(ctypes.byref(p), fake, fake, fake, fake, fake, null, fake, fake, fake, null)
    assert rc == -1
    p.apf_mode = 1
    p.K = 96
    rc = lib.osdn_decode_step(ctypes.byref(p), fake, fake, fake, fake, fake, null, fake, fake, fake, null)
    assert rc == -2


def test_calls_refuse_what_is_no_params_or_no_memory(lib):
    """Through the marshalled entry: an exception, and never the end of the process (hence the child)."""
    import subprocess
    import sys
    code = """
import ctypes, torch, paper_2605_13473_b200 as osdn
from paper_2605_13473_b200 import binding
p = osdn.make_params(B=1, T=1, H=1, K=64, V=64, io_dtype="fp32")
def refused(kind, *args):
    try:
        binding.osdn_decode_step(*args)
    except kind as e:
        print("refused", type(e).__name__, flush=True)
x = torch.empty(64)
refused(TypeError, bytes(p), x, x, x, x, x, None, x, x, x)     # the right number of bytes
refused(TypeError, None, x, x, x, x, x, None, x, x, x)
refused(TypeError, p, 5, x, x, x, x, None, x, x, x)
refused(ValueError, p, torch.empty(64, 2).t(), x, x, x, x, None, x, x, x)
class Sub(binding.OsdnParams):
    _fields_ = [("more", ctypes.c_int)]
refused(RuntimeError, Sub(), None, x, x, x, x, None, x, x, x)  # taken as params (all zero): refused further down
def inside(t):
    refused(RuntimeError, p, t, x, x, x, x, None, x, x, x)     # a wrapped tensor has no memory of its own
    return t.sum()
torch.func.vmap(inside)(torch.empty(3, 64))
torch.func.grad(inside)(torch.empty(64))
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.count("refused") == 7, (r.returncode, r.stdout, r.stderr[-2000:])


def test_extension_belongs_to_this_interpreter_and_torch(lib):
    """Another interpreter does not find it, another torch has it built again."""
    import importlib
    import sysconfig

    import torch
    from paper_2605_13473_b200 import build as b
    module = importlib.import_module("paper_2605_13473_b200._osdn_call")
    assert module.__file__ == b.CALL_LIB and b.CALL_LIB.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert os.path.join(os.path.dirname(torch.__file__), "version.py") in b.call_inputs()
    assert os.path.getmtime(b.CALL_LIB) >= max(map(os.path.getmtime, b.call_inputs()))


def test_missing_library_fails_loudly(tmp_path):
    with pytest.raises(RuntimeError, match="no fallback"):
        osdn.load_library(str(tmp_path / "libosdn.so"))
