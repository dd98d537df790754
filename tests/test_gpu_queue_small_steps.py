"""Small steps in the step interpreter: its body threads run two of a launch's 128-thread blocks at a time."""
import pytest

from paper_2103_11595_gb300 import ajf, workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [3, 8])
def test_small_steps_share_the_body_threads(seed):
    """Tasks of the small launches: at most half the steps, rounded up per launch (every step of these
    networks has at most 128 outputs, and with one step per task half the threads have none), and the
    bits of the per-context path."""
    with ajf.Context(0) as c:
        ajf.load_instance(c.handle, W.tiny(seed))
        info = ajf.ajf_plan(c.handle, 2, trials=4)
        assert info["n_gemm_steps"] == 0 and info["width"] <= 7
        small = sum(1 for l in ajf.ajf_plan_launches(c.handle) if l["kind"] == "small")
        ref = ajf.ajf_fidelity_alg2(c.handle)
        ajf.ajf_profile_enable(c.handle, True)
        got = ajf.ajf_fidelity_batch_queue([c.handle], 2)[0]
        tasks = ajf.ajf_queue_profile(c.handle)["small"]["tasks"]
        ajf.ajf_profile_enable(c.handle, False)
    assert got == ref
    assert small <= tasks <= (info["n_steps"] + small) // 2
