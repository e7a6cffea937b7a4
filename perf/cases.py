"""Workloads whose time and results are measured: optimizer steps over stacks of matrix layers.

A case is one training setup: the shapes of its layers, the rank, the precision mode, the
gradient type, the gate and the entry point a training loop calls.  `prepare` makes the state
such a loop has in hand before a step (parameters, momentum, right factors, gradients, the plan),
`run` is one optimizer step, `exact` the same step in plain float64 torch.

The state is that of an early step of a run: momentum that has taken in a few gradients (noise
and a rank-8 part that the gradients share), unit-column right factors, and the norm of the last
buffer.  Repeated steps on one state keep the branch each layer takes: the gradients stay, the
gated cases' thresholds are far from the RMMC values that follow.
"""
from __future__ import annotations

import math

import torch

import paper_2512_13728_gb300 as cd

PRECISIONS = {"fp32": cd.DION_PREC_FP32, "bf16": cd.DION_PREC_BF16, "bf16x3": cd.DION_PREC_BF16X3}
GATES = {"always": cd.DION_GATE_ALWAYS, "global": cd.DION_GATE_GLOBAL, "per_layer": cd.DION_GATE_PER_LAYER}
MU, ETA, DECAY, EPS = 0.95, 0.01, 0.01, 1e-8
SIGMA = 1e-3  # gradient noise
SIGNAL_RANK = 8


def block(d: int, f: int) -> str:
    """The matrices of one transformer block: four d x d, d x f and f x d."""
    return f"{d}x{d} {d}x{d} {d}x{d} {d}x{d} {d}x{f} {f}x{d}"


def case_of(name, shapes, repeat, rank, precision="bf16", grad="bf16", gate="always", sync=1.0, via="step"):
    """sync: the share of the layers that synchronizes under a per-layer gate."""
    c = dict(shapes=shapes, repeat=repeat, rank=rank, precision=precision, grad=grad, gate=gate, sync=sync, via=via)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small fp32 matrix with fp32 gradients, a layer optimized by itself: launches and latency
        case_of("matrix_fp32", "256x512", 1, 16, "fp32", "fp32"),
        # the same on the tensor cores with split operands
        case_of("matrix_bf16x3", "256x512", 1, 16, "bf16x3", "fp32"),
        # one block of a 160M-parameter GPT (d = 768, rank fraction 1/4)
        case_of("block160m_r192", block(768, 3072), 1, 192),
        # its whole stack, 72 matrices, at rank fractions 1/16 and 1/4
        case_of("stack160m_r48", block(768, 3072), 12, 48),
        case_of("stack160m_r192", block(768, 3072), 12, 192),
        # the same stack as a data-parallel worker steps it: four phases, global gate
        case_of("stack160m_r192_phases", block(768, 3072), 12, 192, gate="global", via="phases"),
        # widths and a rank that no tile divides, bf16 mode
        case_of("ragged_r101", block(771, 2055), 2, 101),
        # 350M-parameter stack under the per-layer gate: the steps between synchronizations
        case_of("stack350m_r256_local", block(1024, 4096), 24, 256, gate="per_layer", sync=0.0),
        # and a step in which half of the layers synchronize
        case_of("stack350m_r256_mixed", block(1024, 4096), 24, 256, gate="per_layer", sync=0.5),
        # the same stack with fp32-class arithmetic, every layer synchronizing: tensor cores, CUDA cores
        case_of("stack350m_r256_bf16x3", block(1024, 4096), 24, 256, "bf16x3"),
        case_of("stack350m_r256_fp32", block(1024, 4096), 24, 256, "fp32"),
        # the 1.3B-parameter stack, 144 matrices at rank fraction 1/4
        case_of("stack1p3b_r512", block(2048, 8192), 24, 512),
    ]


def draw(rng):
    """A stack of blocks, or of single matrices, of a width between 96 and 2048, with a rank
    fraction between 1/16 and 1/4, in one of the modes above; at most the 1.3B stack's elements,
    fewer where the contractions run on CUDA cores."""
    precision = rng.choice(["bf16", "bf16", "bf16", "bf16x3", "fp32"])
    via, gate, sync = "step", "always", 1.0
    kind = rng.random()
    if kind < 0.2:
        gate, sync = "per_layer", rng.choice([0.0, 0.0, 0.25, 0.5])
    elif kind < 0.35:
        gate = "global"
        via = rng.choice(["step", "phases"])
    elif kind < 0.45:
        via = "host"
    d = int(round(math.exp(rng.uniform(math.log(96), math.log(2048)))))
    if rng.random() < 0.6:
        d = max(96, d // 64 * 64)
    f = int(d * rng.uniform(1.0, 4.0))
    if rng.random() < 0.6:
        f = max(d, f // 64 * 64)
    rank = max(4, int(d * math.exp(rng.uniform(math.log(1 / 16), math.log(1 / 4)))))
    if rng.random() < 0.6:
        rank = max(8, rank // 16 * 16)
    if precision == "bf16x3":
        rank = min(rank, 256)
    shapes = block(d, f) if rng.random() < 0.7 else rng.choice([f"{d}x{f}", f"{f}x{d}", f"{d}x{f} {f}x{d}"])
    per = sum(m * n for m, n in parse(shapes))
    most = 302_000_000 if precision != "bf16" or via == "host" else 1_200_000_000
    repeat = int(round(math.exp(rng.uniform(0.0, math.log(24)))))
    repeat = max(1, min(repeat, most // per))
    grad = "fp32" if rng.random() < (0.4 if precision != "bf16" else 0.15) else "bf16"
    return case_of(None, shapes, repeat, rank, precision, grad, gate, sync, via)


def parse(text):
    return [tuple(int(v) for v in s.split("x")) for s in text.split()]


def layers_of(case):
    return parse(case["shapes"]) * case["repeat"]


def up8(v):
    return (v + 7) // 8 * 8


def packed(dims, dtype, device, pin=False):
    """One zeroed buffer and a row-major view per matrix, rows padded to 8 elements."""
    sizes = [m * up8(n) for m, n in dims]
    flat = torch.zeros(sum(sizes), dtype=dtype, device=device, pin_memory=pin)
    views, at = [], 0
    for (m, n), size in zip(dims, sizes):
        views.append(flat[at:at + size].view(m, up8(n))[:, :n])
        at += size
    return flat, views


def syncs(case, i):
    """Whether layer i takes the synchronized branch."""
    if case["gate"] != "per_layer":
        return True
    return math.floor((i + 1) * case["sync"]) > math.floor(i * case["sync"])


def inputs(case, seed):
    """X, M, Q, G and the norm of the last buffer for every layer, from the seed alone."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) & ((1 << 62) - 1))

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=dev)

    dims = layers_of(case)
    gdt = torch.float32 if case["grad"] == "fp32" else torch.bfloat16
    s = {"dims": dims}
    s["X"], s["Xs"] = packed(dims, torch.float32, dev)
    s["M"], s["Ms"] = packed(dims, torch.float32, dev)
    s["Q"], s["Qs"] = packed([(n, min(case["rank"], m, n)) for m, n in dims], torch.float32, dev)
    s["G"], s["Gs"] = packed(dims, gdt, dev)
    for (m, n), X, M, Q, G in zip(dims, s["Xs"], s["Ms"], s["Qs"], s["Gs"]):
        k = min(SIGNAL_RANK, m, n)
        signal = (normal(m, k) / math.sqrt(m)) @ (normal(k, n) * (4 * SIGMA * math.sqrt(max(m, n)) / math.sqrt(n)))
        X.copy_(normal(m, n) * 0.02)
        M.copy_(normal(m, n) * (2 * SIGMA) + 3 * signal)
        G.copy_(normal(m, n) * SIGMA + signal)
        q = normal(*Q.shape)
        Q.copy_(q / torch.linalg.vector_norm(q, dim=0, keepdim=True))
    norms = torch.stack([torch.linalg.vector_norm(M.double()) for M in s["Ms"]])
    s["prev_norm"] = norms * 0.9 if case["gate"] == "per_layer" else norms * 0.5
    return s


def prepare(case, seed):
    s = inputs(case, seed)
    dims = s["dims"]
    # a layer that synchronizes under the per-layer gate does so on any change of the norm
    taus = [0.0 if case["gate"] == "per_layer" and syncs(case, i) else 10.0 for i in range(len(dims))]
    s["plan"] = cd.Plan(s["Xs"], s["Ms"], s["Qs"], s["Gs"], taus, PRECISIONS[case["precision"]])
    s["plan"].prev_norm.copy_(s["prev_norm"])
    s["t"] = 0
    s["via"], s["gate"] = case["via"], GATES[case["gate"]]
    if case["via"] == "host":
        s["host"], s["host_G"] = packed(dims, s["G"].dtype, "cpu", pin=True)
        s["host"].copy_(s["G"])
        s["plan"].enable_host_gradients()
    return s


def run(state):
    plan = state["plan"]
    state["t"] += 1
    # tau_global 0: a data-parallel run that synchronizes on any change, as in its spiky phases
    hp = cd.hparams(mu=MU, eta=ETA, eps_rmmc=EPS, eps_col=EPS, tau_global=0.0, gate_mode=state["gate"],
                    step=state["t"], weight_decay=DECAY)
    if state["via"] == "step":
        plan.step(hp)
    elif state["via"] == "host":
        plan.step_host(hp, state["host_G"])
    else:  # one data-parallel worker: its reductions between the phases are the identity
        for phase in (cd.DION_PHASE_NORMS, cd.DION_PHASE_POWER, cd.DION_PHASE_ORTHO, cd.DION_PHASE_UPDATE):
            plan.step_phase(phase, hp)
    return {"X": state["X"], "M": state["M"], "Q": state["Q"], "prev_norm": plan.prev_norm, "rmmc": plan.rmmc,
            "rmmc_eq1": plan.rmmc_eq1, "flags": plan.flags, "global_flag": plan.global_flag}


def exact(case, seed):
    """Algorithm 2's step in float64: B = M + G, RMMC, then per layer either P = qf(B Q) with a
    positive-diagonal triangular factor, R = B^T P, M = B - (1 - mu) P R^T, Q = R with unit
    columns, X = X (1 - eta decay) - eta sqrt(m / n) P Q^T; or M = B, X = X (1 - eta decay) - eta G."""
    s = inputs(case, seed)
    dev = s["X"].device
    mu, eta, decay, eps = (torch.tensor(v, dtype=torch.float32).double().item() for v in (MU, ETA, DECAY, EPS))
    L = len(s["dims"])
    out = {}
    out["X"], Xs = packed(s["dims"], torch.float64, dev)
    out["M"], Ms = packed(s["dims"], torch.float64, dev)
    out["Q"], Qs = packed([tuple(q.shape) for q in s["Qs"]], torch.float64, dev)
    out["prev_norm"] = torch.zeros(L, dtype=torch.float64, device=dev)
    out["rmmc"], out["rmmc_eq1"] = torch.zeros_like(out["prev_norm"]), torch.zeros_like(out["prev_norm"])
    for i, (m, n) in enumerate(s["dims"]):
        M, G, Q = s["Ms"][i].double(), s["Gs"][i].double(), s["Qs"][i].double()
        B = M + G
        before, norm, prev = torch.linalg.vector_norm(M), torch.linalg.vector_norm(B), s["prev_norm"][i]
        out["prev_norm"][i] = norm
        out["rmmc"][i] = (norm - prev).abs() / (prev + eps)
        X = s["Xs"][i].double() * (1 - eta * decay)
        if syncs(case, i):
            P = B @ Q
            for _ in range(2):  # Cholesky QR twice: the Q factor of a well-conditioned P to float64 rounding
                low = torch.linalg.cholesky(P.T @ P)
                P = torch.linalg.solve_triangular(low, P.T, upper=False).T
            R = B.T @ P
            Q = R / (torch.linalg.vector_norm(R, dim=0, keepdim=True) + eps)
            B -= (1 - mu) * (P @ R.T)
            X -= eta * math.sqrt(m / n) * (P @ Q.T)
        else:
            X -= eta * G
        out["rmmc_eq1"][i] = (torch.linalg.vector_norm(B) - before).abs() / (before + eps)
        Xs[i].copy_(X)
        Ms[i].copy_(B)
        Qs[i].copy_(Q)
    out["flags"] = out["global_flag"] = None  # whole numbers
    return out


def work(case):
    """Each of X, M read and written and G read once; per synchronized layer Q read and written
    once, and the multiply-adds of B Q, one Q factor (m r^2), B^T P, P R^T and P Q_t^T."""
    g = 4 if case["grad"] == "fp32" else 2
    nbytes = flops = 0
    for i, (m, n) in enumerate(layers_of(case)):
        r = min(case["rank"], m, n)
        nbytes += m * n * (16 + g)
        if syncs(case, i):
            nbytes += 8 * n * r
            flops += 8 * m * n * r + 2 * m * r * r
        else:
            flops += 4 * m * n
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the largest error of any output against `exact` (that of Q_t, which the
    operands' rounding reaches undamped): 3.1e-3 in bf16, 7.4e-6 with split operands, 1e-6 in fp32."""
    return {"bf16": {"rel": 1.3e-2}, "bf16x3": {"rel": 3e-5}, "fp32": {"rel": 1e-5}}[case["precision"]]
