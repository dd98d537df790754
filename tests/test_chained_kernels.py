"""Kernels that are resident while their predecessors still run (launch_chained): what their source has
to say for their reads to be ordered, and evaluations repeated until a disorder would show."""
import os
import re

import numpy as np
import pytest

from paper_2103_11595_gb300 import ajf, workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_11595_gb300", "csrc")
DESCRIPTORS = {"StepDev", "PermDev", "FinalDev"}  # uploaded before a chain starts, written by no kernel


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def restrict_params(text, function):
    """Pointee types of the __restrict__ parameters of `function` where it is defined."""
    found = [re.search(r"\b%s\(([^)]*)\)\s*\{" % function, text)]
    assert found[0], function
    return [t for t in re.findall(r"(\w+)\s*\*\s*__restrict__", found[0].group(1))]


@pytest.mark.parametrize("name", ["kernels.cu", "dg_gemm.cu", "tc_gemm.cu"])
def test_chained_kernels_promise_nothing_about_others_data(name):
    """A __restrict__ pointer to data that a predecessor writes allows non-coherent loads, and loads
    above the wait."""
    text = source(name)
    kernels = {k for call in re.findall(r"launch_chained\(([^;]*);", text) for k in re.findall(r"\bk_\w+", call)}
    assert kernels
    for k in sorted(kernels):
        assert set(restrict_params(text, k)) <= DESCRIPTORS, k


def test_a_kernel_lets_its_successor_start_after_its_own_wait():
    """So that at most two kernels of a chain are resident: the trigger is only ever issued behind the wait."""
    found = 0
    for name in sorted(os.listdir(CSRC)):
        text = source(name)
        for m in re.finditer(r"griddepcontrol\.launch_dependents", text):
            found += 1
            assert "griddepcontrol.wait" in text[:m.start()].rsplit("{", 1)[1], name
    assert found == 1


def test_shared_bodies_promise_nothing_about_others_data():
    for name in ("bodies.cuh", "dg_gemm.cu"):
        text = source(name)
        for body in sorted(set(re.findall(r"\b(\w+_body|perm_tiles_\w+)\(const \w+[&*]", text))):
            assert set(restrict_params(text, body)) <= DESCRIPTORS, body


def test_epilogue_lanes_read_behind_a_warp_barrier():
    """No lane of the GEMM's epilogue reads scales or accumulators on another lane's word alone (a shuffle
    orders no memory): a warp barrier stands behind each wait."""
    epilogue = source("tc_gemm_dev.cuh").split("} else if (warp >= kEpiWarp0) {")[1].split("if (mine) {")[0]
    waits = epilogue.split("mbar_wait(")[1:]
    assert len(waits) == 2
    for w in waits:
        w = w[:w.index("if (!ok) break;")]
        assert "__syncwarp();" in w[w.index("__shfl_sync("):]


def test_scales_are_given_back_across_the_proxies():
    """The scaled fp16 epilogue reads its scales through the generic proxy, and the issuer overwrites them
    with a bulk copy once the buffer's barrier has been arrived at: a proxy fence stands between."""
    epilogue = source("tc_gemm_dev.cuh").split("} else if (warp >= kEpiWarp0) {")[1].split("mbar_arrive(sh.acce0")[0]
    last_read = epilogue.rindex("(sbv + c0 + j)")
    assert "if (kKind == 2) asm volatile(\"fence.proxy.async.shared::cta;\"" in epilogue[last_read:]


def test_warp_operations_name_their_lanes():
    """A shuffle or vote over whichever lanes happen to be together drops the others' values: the masks
    come from the conditions that the lanes are under."""
    for name in os.listdir(CSRC):
        assert "__activemask" not in source(name), name


def test_drain_commits_from_the_lane_that_issued():
    """A commit tracks the MMAs of the thread that executes it: wherever an elected lane issues them, an
    elected lane commits them, also in the drain after an abort."""
    drain = source("tc_gemm_dev.cuh").split("void tc_drain_after_abort(")[1]
    issuer = drain[:drain.index("mma_commit(")].rsplit("else if", 1)[1]
    assert "warp == 1 && elect_one()" in issuer and "lane" not in issuer
    for name in ("tc_gemm.cu", "queue.cu"):  # and every lane of the warp is there to elect it
        assert re.search(r"if \(__any_sync\(0xffffffffu, \*sh\.abort_flag != 0\)\)\s*tc_drain_after_abort", source(name))


@pytest.mark.gpu
@pytest.mark.parametrize("seed", range(10))
def test_repeated_scaled_fp16_evaluations_are_bitwise_equal(seed):
    """The mode whose epilogue also reads per-block scales that the GEMM copies in; the chain without and
    with a graph, and a new context's first evaluation among the repeated ones."""
    inst = W.mid(seed)
    seen = set()
    for k in range(4):
        with ajf.Context(0) as c:
            ajf.load_instance(c.handle, inst)
            ajf.ajf_plan(c.handle, 2, precision="f16x3", trials=8, use_graph=k % 2 == 1)
            seen |= {ajf.ajf_fidelity_alg2(c.handle)["S"] for _ in range(25)}
    assert len(seen) == 1


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["f64", "f32", "bf16x6", "tf32x3", "f16x3"])
def test_first_evaluations_are_bitwise_equal(precision):
    """New contexts, one evaluation each, the launches enqueued one by one."""
    for seed in (0, 3):
        inst = W.mid(seed)
        seen = set()
        for _ in range(25):
            with ajf.Context(0) as c:
                ajf.load_instance(c.handle, inst)
                ajf.ajf_plan(c.handle, 2, precision=precision, trials=8)
                seen.add(ajf.ajf_fidelity_alg2(c.handle)["S"])
        assert len(seen) == 1


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["f64", "f32", "bf16x6", "tf32x3", "bf16x3"])
def test_repeated_evaluations_are_bitwise_equal(precision):
    """The same plan and inputs, enqueued one by one and from a graph, always give the same bits (every
    kernel sums in a fixed order), also with several circuits' chains side by side."""
    insts = [W.mid(s) for s in (0, 3, 7)]
    ctxs = [ajf.Context(0) for _ in insts]
    try:
        for graph in (False, True):
            for c, inst in zip(ctxs, insts):
                ajf.load_instance(c.handle, inst)
                ajf.ajf_plan(c.handle, 2, precision=precision, trials=8, use_graph=graph)
            first = [ajf.ajf_fidelity_alg2(c.handle)["S"] for c in ctxs]
            for _ in range(40):
                assert [ajf.ajf_fidelity_alg2(c.handle)["S"] for c in ctxs] == first
            for _ in range(40):
                assert [r["S"] for r in ajf.ajf_fidelity_batch([c.handle for c in ctxs], 2)] == first
    finally:
        for c in ctxs:
            c.close()


@pytest.mark.gpu
def test_repeated_traces_are_bitwise_equal():
    """A chain of short launches (small steps, split-K sums), each of which lets the next one start."""
    inst = W.batching_circuit(1)
    with ajf.Context(0) as c:
        ajf.load_instance(c.handle, inst)
        ajf.ajf_plan(c.handle, 1, trials=8)
        n = inst.n_combinations()
        ajf.ajf_fidelity_alg1(c.handle)
        first = ajf.ajf_alg1_traces(c.handle, n)
        for _ in range(100):
            ajf.ajf_fidelity_alg1(c.handle)
            assert np.array_equal(ajf.ajf_alg1_traces(c.handle, n), first)
