"""What the warp roles of the tensor-core kernels owe one another, read from the source: a missing wait or an unbounded one
shows in no result, and a test that ran into it would hang the device."""
import os
import re

import pytest

import paper_2605_13473_b200

CSRC = os.path.join(os.path.dirname(paper_2605_13473_b200.__file__), "csrc")


def role(name, file="osdn_tc.cu"):
    """The body of a function of a kernel file, without its comments."""
    with open(os.path.join(CSRC, file)) as f:
        text = f.read()
    body = re.search(r"\n__(?:device__ __forceinline__|global__) [^\n]*\b" + name + r"\(.*?\n\{\n(.*?)\n\}\n", text, re.S).group(1)
    return re.sub(r"//[^\n]*", "", body)


@pytest.mark.parametrize("name", ["chain_fwd_role", "chain_bwd_role", "chunk_bwd_role"])
def test_roles_meet_at_bounded_waits_only(name):
    """A warp whose wait runs out leaves its loop by itself.  Between the barrier that starts the roles and the one behind
    them the others must not meet it at a hardware barrier, which has no limit."""
    parts = re.split(r"__syncthreads(?:_\w+)?\(", role(name))
    roles = max(parts, key=len)
    assert roles.count("mbar_wait(") >= 5 and roles.count("break;") >= 5
    assert not re.findall(r"named_sync\w*\(|\bbar\.|barrier\.", roles)
    assert all("mbar_wait(" not in p for p in parts if p is not roles)


def test_epilogue_waits_for_the_copies_that_it_reads():
    """Chunk-local backward, full tiles: each operand that the epilogue warps read from shared memory has been waited for by
    them on the barrier that its copy completes on."""
    epilogue = role("chunk_bwd_role").split("const uint32_t offT", 1)[1]
    epilogue = re.sub(r"\n {12}if \(len < CH\) \{.*?\n {12}\}", "", epilogue, flags=re.S)
    for bar, regions in {"bar_tok": ("R_Q", "R_K", "R_KT"), "bar_v": ("R_V",), "bar_s": ("R_S", "R_DS")}.items():
        for region in regions:
            at = re.search(r"s0 \+ " + region + r" \+", epilogue).start()
            assert "mbar_wait(&" + bar + "," in epilogue[:at], (region, bar)


@pytest.mark.parametrize("name", ["chunk_fwd_tile", "chain_fwd_role", "chain_bwd_role", "chunk_bwd_role"])
def test_roles_leave_no_copy_or_product_behind(name):
    """However a role ends, the copies that it has asked for have landed and its products are complete (both waits bounded, and
    deaf to the status word) before the memory they work on is used again or given back."""
    body = role(name)
    targets = set(re.findall(r"(?:bulk_load|tma_load_2d|load_tok)\([^;]*&(?:gs\.)?(bar_\w+)", body))
    assert targets
    for bar in targets:
        assert re.search(r"mbar_drain\(&" + bar + r"\b", body), bar
    assert re.search(r"mma_commit\(&(gs\.)?bar_drain, lead\);\s*mbar_drain\(&(gs\.)?bar_drain, 0\);", body)


def test_wide_chain_slices_leave_no_copy_behind():
    """The two stage copies that may be on their way when a wide slice of a CUDA-core chain gives up: the one that was waited
    for (a status code ends a wait early) and the one behind it."""
    give_up = role("chain_wide_kernel", "osdn_simt.cuh").split("if (!__syncthreads_and(ok)) {", 1)[1].split("break;", 1)[0]
    assert re.search(r"for \(int x = j; x <= j \+ 1 && x < w\.n; \+\+x\) umma::mbar_drain\(&s\.full\[x & 1\], \(x >> 1\) & 1\);", give_up)
