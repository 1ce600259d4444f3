"""Rules of the dependent launches and of the bounded waits, checked on the CUDA sources (no GPU needed).

A kernel launched with programmatic stream serialization is resident while the kernels before it still write.  What
such a kernel reads through the non-coherent path (``__ldg``, ``const ... __restrict__`` parameters) must not change
while it is resident, and the compiler may move those loads above ``pdl_wait()``: they are for data that no kernel of a
pass writes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_03311_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))

# weights and gains; tables of the store; what is copied to the device, or finished before a wait of the host, ahead of
# the first dependent launch (packed offsets and order, a build's or selection's token records, score tiles)
CONSTANT = {"embed", "gain", "head", "w1", "b1", "w2", "slot_row", "slot_m", "tok_off", "perm", "tok_pair", "tok_pos",
            "pair_slot", "units", "a_off"}
CONSTANT_LDG = ("xn_gain", "cs", "wgt")  # the next norm's gains, the RoPE table's entries, the q/k norm gains


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _block(text, start):
    """The brace-delimited block that begins at or after `start`."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def _kernels(text):
    """(name, parameter list, body) of every __global__ function defined in the text."""
    for m in re.finditer(r"__global__\b", text):
        sig = re.compile(r"(\bk_\w+)\s*\(").search(text, m.end())
        depth, i = 1, sig.end()
        while depth:
            depth += (text[i] == "(") - (text[i] == ")")
            i += 1
        yield sig.group(1), text[sig.end():i - 1], _block(text, i)


def _call_args(text, name):
    for m in re.finditer(r"\b%s\s*\(" % name, text):
        depth, i = 1, m.end()
        while depth:
            depth += (text[i] == "(") - (text[i] == ")")
            i += 1
        yield text[m.end():i - 1]


@pytest.mark.parametrize("name", SOURCES)
def test_non_coherent_loads_are_of_constant_data(name):
    text = _source(name)
    for arg in _call_args(text, "__ldg"):
        assert any(re.search(r"\b%s\b" % c, arg) for c in CONSTANT_LDG), f"{name}: __ldg({arg})"
    for kernel, params, body in _kernels(text):
        if "pdl_wait()" not in body:
            continue
        for p in params.split(","):
            if re.search(r"\bconst\b", p) and "__restrict__" in p:
                assert p.split()[-1] in CONSTANT, f"{name}: {kernel} reads {p.split()[-1]} through the non-coherent path"


def test_the_rule_sees_the_dependent_kernels():
    found = {k for s in SOURCES for k, _, body in _kernels(_source(s)) if "pdl_wait()" in body}
    assert {"k_embed", "k_gemm_pair", "k_gemm_few", "k_attn", "k_attn_tc", "k_attn_tc_long", "k_sal_tc", "k_sal_colstat",
            "k_sal_topk", "k_sal_gather", "k_score", "k_score_mlp", "k_score_mlp_sum", "k_gather_score_rows",
            "k_prefix_store", "k_commit_scores"} <= found


def test_waits_before_work_of_the_whole_warp_are_the_whole_warps():
    # A lane that gives up by itself at the time limit leaves the others in a shuffle or a tensor memory access that
    # waits for it.  Single-lane waits stay where the block meets right after (k_attn) and in the one-thread probe.
    for name in SOURCES:
        single = list(_call_args(_source(name), "mbar_wait")) + list(_call_args(_source(name), "mbar_wait_cluster"))
        allowed = {"k_attn.cu": 2, "k_rows.cu": 1, "k_gemm.cu": 1}.get(name, 0)  # k_gemm: inside wait_all_lanes
        assert len(single) == allowed, (name, single)


def test_the_few_row_launch_beside_a_wide_one_passes_its_gate_before_it_reads():
    # The launch beside does not wait for the kernel before it until its end; what that kernel waited for reaches it
    # through the gate: a release after the wide launch's wait, an acquire and a proxy fence before the first read.
    bodies = {k: body for k, _, body in _kernels(_source("k_gemm.cu"))}
    wide, few = bodies["k_gemm_pair"], bodies["k_gemm_few"]
    assert wide.index("pdl_wait()") < wide.index("gate_open(") < wide.index("pdl_trigger()")
    passed = few.index("gate_wait_warp(")
    assert passed < few.index("fence_proxy_async_global()") < few.index("__syncthreads()") < few.index("tma_load_")
    assert passed < few.index("epilogue_prefetch<") and "if (!gate_passed) total = 0;" in few
    # without a gate every warp waits for the kernel before, and a launch beside does so at its end
    assert few.count("if (!p.beside) pdl_wait();") == 1 and few.count("if (warp != 0 && !p.beside) pdl_wait();") == 1
    assert few.index("if (p.beside) pdl_wait();") > few.index("epilogue_tile<") and few.count("pdl_wait()") == 3
