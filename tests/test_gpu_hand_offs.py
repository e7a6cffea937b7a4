"""Hand-offs inside the kernels: the same step from the same state gives the same bits every time.

A hand-off that is not ordered (a warp's lanes through shared memory, the two CTAs of a pair) shows up
as a result that depends on the timing.  Each case repeats one step, between other work on the GPU so
that the timing differs, and compares every output bit for bit.
"""
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


def repeat(w, prec, times):
    import paper_2512_13728_gb300 as cd

    st = gu.make_state(w)
    gu.write_gradients(st, 1)
    start = [t.clone() for t in st.X + st.M + st.Q]
    plan = cd.Plan(st.X, st.M, st.Q, st.G, st.taus, PRECS[prec])
    noise = torch.ones(1 << 22, device="cuda")
    first = None
    try:
        for k in range(times):
            for dst, src in zip(st.X + st.M + st.Q, start):
                dst.copy_(src)
            plan.prev_norm.zero_()
            plan.refresh()
            for _ in range(k % 4):
                noise.mul_(1.0)
            plan.step(cd.hparams(step=1))
            torch.cuda.synchronize()
            assert plan.device_status() == 0
            out = [t.clone() for t in st.X + st.M + st.Q] + [plan.rmmc.clone(), plan.rmmc_eq1.clone()]
            first = first or out
            assert all(torch.equal(a, b) for a, b in zip(out, first)), k
    finally:
        plan.close()


@pytest.mark.parametrize("prec,rank", [("fp32", 96), ("fp32", 250), ("bf16", 33), ("bf16", 192), ("bf16", 300),
                                       ("bf16x3", 130)])
def test_cholesky_blocks_repeat_bitwise(prec, rank):
    """The three Cholesky kernels, whose two warps per diagonal block pass columns through shared memory."""
    w = wl.scaled(wl.WORKLOADS["gpt160m_block_r192"], "lanes", [(520, 300), (300, 520)] * 8, rank=rank)
    repeat(w, prec, 24)


@pytest.mark.parametrize("prec,rank,g_dtype", [("bf16", 48, "bf16"), ("bf16", 300, "bf16"), ("bf16x3", 64, "bf16"),
                                               ("bf16x3", 256, "fp32")])
def test_pair_hand_offs_repeat_bitwise(prec, rank, g_dtype):
    """Converted operand boxes that the pair's other CTA has multiplied: the fused buffer kernel (bf16,
    bf16 gradients) and the Gram and solve with split operands, over many chunks and tiles per pair,
    with an empty second row tile and partial chunks."""
    w = wl.scaled(wl.WORKLOADS["gpt160m_block_r192"], "pairs", [(1160, 1100), (640, 2056), (2056, 640)] * 12, rank=rank,
                  g_dtype=g_dtype)
    repeat(w, prec, 24)
