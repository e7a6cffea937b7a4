"""Orthogonalize on hard P: how far P^T P is from the identity, read from the library itself.

One data-parallel worker runs the four phases; between ORTHO and UPDATE it replaces R by columns of the
identity, so that Q_t is those columns and the update leaves X = -eta sqrt(m/n) [P | 0]: P as the
update's operands hold it.
"""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

PRECS = {"fp32": 0, "bf16": 1, "bf16x3": 2}  # DION_PREC_*


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_13728_gb300 import build

    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def spectrum_layer(m, n, r, power, zero_rows, seed):
    """B with singular values k^-power and its first rows zero (dead or padded rows), random unit-column Q."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def basis(a, b):
        return torch.linalg.qr(torch.randn((a, b), generator=g, device="cuda", dtype=torch.float64))[0]

    k = min(m, n)
    s = torch.arange(1, k + 1, device="cuda", dtype=torch.float64) ** -power
    B = (basis(m, k) * s) @ basis(n, k).T
    B[:zero_rows] = 0
    Q = torch.randn((n, r), generator=g, device="cuda", dtype=torch.float64)
    return B.float(), (Q / Q.norm(dim=0)).float()


def orthonormal_p(B, Q, prec, copies):
    """P of the first of `copies` equal layers, in fp64."""
    import paper_2512_13728_gb300 as cd

    m, n, r = B.shape[0], B.shape[1], Q.shape[1]
    X = [torch.zeros_like(B) for _ in range(copies)]
    G = [torch.zeros(B.shape, device="cuda", dtype=torch.bfloat16) for _ in range(copies)]
    plan = cd.Plan(X, [B.clone() for _ in range(copies)], [Q.clone() for _ in range(copies)], G, [1.0] * copies, PRECS[prec])
    hp = cd.hparams(step=1, eta=1.0)
    try:
        for phase in (cd.DION_PHASE_NORMS, cd.DION_PHASE_POWER, cd.DION_PHASE_ORTHO):
            plan.step_phase(phase, hp)
        ldp = (r + 7) // 8 * 8
        R = plan.exchange(cd.DION_PHASE_ORTHO)[: n * ldp].view(n, ldp)
        R.zero_()
        R[:r, :r].fill_diagonal_(1.0)
        plan.step_phase(cd.DION_PHASE_UPDATE, hp)
        torch.cuda.synchronize()
        assert plan.device_status() == 0
        return X[0][:, :r].double() / -math.sqrt(m / n)
    finally:
        plan.close()


# Passes 1 and 2 take the first-order factor while 1.5 ||E||_2 is below 6e-2 (bf16) or 1e-3 (bf16x3), E = X^T X - I,
# and then leave -F F - F F^T - F^T F^T with F + F^T = E: 3 ||E||^2 at most, 4.8e-3 or 1.3e-6.  On top of it come
# the solve's operands and P's own halves: tf32 (2^-10 on each factor) and bf16 in bf16 mode, 2.2e-3 to 3.3e-3 in
# a model of these roundings with every factor exact; 2^-17 in bf16x3.
DEFECT = {"bf16": 8e-3, "bf16x3": 3e-5}
# Two plans that add S up in another order: the Q factor of the same P in arithmetic of 2^-22 moves by as
# much times the condition of P (the range of 3xTF32 products and fp32 sums).
ORDER = 2.0 ** -22


@pytest.mark.parametrize("prec", ["bf16", "bf16x3"])
@pytest.mark.parametrize("m,n,r,power,zero_rows", [(256, 512, 16, 2.0, 0), (256, 512, 16, 2.5, 32), (256, 512, 32, 2.0, 32),
                                                   (256, 512, 32, 2.5, 0), (3072, 768, 32, 2.0, 0)])
def test_hard_p_with_a_split_gram(m, n, r, power, zero_rows, prec):
    """A plan of one layer splits the layer's Gram into row ranges, whose partial sums the Cholesky
    kernels add up; hard P make the second pass decide by its estimate of ||X^T X - I||_2.  P comes out
    orthonormal, and as in a plan of 152 such layers, whose Grams are whole."""
    worst = 0.0
    for seed in range(8):
        B, Q = spectrum_layer(m, n, r, power, zero_rows, seed)
        P = orthonormal_p(B, Q, prec, 1)
        defect = torch.linalg.matrix_norm(P.T @ P - torch.eye(r, device="cuda", dtype=torch.float64), 2).item()
        worst = max(worst, defect)
        if m < 1000 and seed < 3:
            apart = torch.linalg.matrix_norm(P - orthonormal_p(B, Q, prec, 152), 2).item()
            cond = torch.linalg.cond(B.double() @ Q.double()).item()
            print("apart", apart, "condition", cond)
            assert apart <= DEFECT[prec] + ORDER * cond
    print("defect", worst)
    assert worst <= DEFECT[prec]


@pytest.mark.parametrize("r", [16, 40])
@pytest.mark.parametrize("gram", [2e38, 1.0, 1e-39, 1e-41])
def test_gram_at_the_ends_of_fp32(gram, r):
    """Pivots at the largest fp32 values and among the subnormal ones (whose reciprocals overflow), in FP32
    mode.  A Gram of 1e-41 keeps 13 bits, which pass 1 makes up for: 3 (1e-3 / 1.5)^2 = 1.3e-6 is the most
    that the first-order factor leaves, and the fp32 solve adds about r 2^-24."""
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    B = torch.randn((256, 320), generator=g, device="cuda") * math.sqrt(gram / 256)
    Q = torch.linalg.qr(torch.randn((320, r), generator=g, device="cuda"))[0].contiguous()
    P = orthonormal_p(B, Q, "fp32", 1)
    defect = torch.linalg.matrix_norm(P.T @ P - torch.eye(r, device="cuda", dtype=torch.float64), 2).item()
    print("defect", defect)
    assert defect <= 1e-5
