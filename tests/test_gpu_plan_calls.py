"""Plan calls around the step on the GPU: launch timing and launch counts."""
import pytest
import torch

import workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

PRECS = {"fp32": 0, "bf16": 1, "bf16x3": 2}  # DION_PREC_*


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_13728_gb300 import build

    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def make_plan(shapes, rank, prec, g_dtype="bf16"):
    import paper_2512_13728_gb300 as cd

    w = wl.scaled(wl.WORKLOADS["gpt160m_block_r192"], "calls", shapes, rank=rank, g_dtype=g_dtype)
    st = gu.make_state(w)
    gu.write_gradients(st, 1)
    return cd.Plan(st.X, st.M, st.Q, st.G, st.taus, PRECS[prec])


@pytest.mark.parametrize("prec", ["fp32", "bf16", "bf16x3"])
def test_finished_timing_outlives_a_step_of_another_mode(prec):
    """Steps after the requested number are not recorded, whatever their gate mode and launch count; a
    change of the launch sequence while recording starts the recording again."""
    import paper_2512_13728_gb300 as cd

    plan = make_plan([(200, 136), (136, 200)], 16, prec)
    try:
        steps = iter(range(1, 20))

        def run(mode, n):
            for _ in range(n):
                plan.step(cd.hparams(step=next(steps), gate_mode=mode))
            return plan.launches_per_step()

        cd.native.dion_timing_enable(plan.handle, 2)
        always = run(cd.DION_GATE_ALWAYS, 2)
        gated = run(cd.DION_GATE_PER_LAYER, 2)
        assert always != gated and plan.launches_per_step() == gated
        recorded, launches = cd.native.dion_timing_read(plan.handle)
        names = [name for name, _ in launches]
        assert recorded == 2 and len(names) == always and "local" not in names and names[-1] == "finalize"
        assert all(ms > 0 for _, ms in launches)
        # the recording begins again after a read: one step of each mode, of which the last sequence counts
        run(cd.DION_GATE_ALWAYS, 1)
        run(cd.DION_GATE_PER_LAYER, 3)
        recorded, launches = cd.native.dion_timing_read(plan.handle)
        assert recorded == 2 and len(launches) == gated and "local" in [name for name, _ in launches]
    finally:
        plan.close()


@pytest.mark.parametrize("prec,shapes,rank", [("fp32", [(200, 136)], 16), ("bf16", [(200, 136)], 16),
                                              ("bf16", [(400, 500)], 300), ("bf16x3", [(200, 136)], 16),
                                              ("bf16", [(520, 300), (300, 200), (400, 700), (200, 64)], 300)])
@pytest.mark.parametrize("g_dtype", ["bf16", "fp32"])
def test_launch_count_before_the_first_step(prec, shapes, rank, g_dtype):
    """Before the first step the count is that of an ALWAYS step, also where the first pass's Cholesky takes
    two launches (ranks on both sides of 256)."""
    import paper_2512_13728_gb300 as cd

    plan = make_plan(shapes, rank, prec, g_dtype)
    try:
        before = plan.launches_per_step()
        plan.step(cd.hparams(step=1))
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        assert plan.launches_per_step() == before
    finally:
        plan.close()


@pytest.mark.parametrize("prec,rank", [("fp32", 500), ("bf16", 500), ("bf16", 256), ("bf16x3", 256)])
def test_a_plan_of_smaller_rank_leaves_others_usable(prec, rank):
    """Two plans in one process: creating the second, of a smaller rank, takes nothing from the first."""
    import paper_2512_13728_gb300 as cd

    shapes = [(600, 520), (520, 600)]
    a = make_plan(shapes, rank, prec)
    b = make_plan(shapes, 8, prec)
    try:
        for plan in (a, b, a):
            plan.step(cd.hparams(step=1))
            torch.cuda.synchronize()
            assert plan.device_status() == 0
    finally:
        a.close()
        b.close()
