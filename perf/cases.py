"""The calls that users of this library make, as cases that can be timed and checked.

Each case is a dict of plain values.  Kinds:

  gemm      C <- alpha A B + beta C through a Plan on device operands (default
            fixed-rule depth unless the case names one), any of the four
            precisions, optionally on views of wider buffers (row strides)
  static    the allocation-free entry point (M, N, K <= 1024)
  batched   independent uneven products bound by one BatchedPlan
  host      a Plan on operands in pinned host memory, copies in and out inside
  residual  the Freivalds check r = C x - A (B x) of a product in hand, in
            float64 accumulation (in float32 its result is rounding noise)
  train     one full-batch training step of the planner's cost model

Operands are drawn on the GPU from the seed alone.
"""
import math

import torch

from paper_1205_2927_gb300 import fmm, inputs

NPARAM = fmm.NPARAM


def listed():
    return [
        # latency-bound callers that cannot allocate: small, odd in every dimension
        dict(name="static_700", kind="static", M=700, N=515, K=901, alpha=1.0, beta=0.0, dist="uniform"),
        # the single n = 1024 call at depth 2 (leaves of 256)
        dict(name="fp32_1024_depth2", kind="gemm", precision="fp32", M=1024, N=1024, K=1024, depth=2, pad=0,
             alpha=1.0, beta=0.0, dist="uniform"),
        # an ordinary ragged product on views of wider buffers, accumulated into C
        dict(name="fp32_ragged_views", kind="gemm", precision="fp32", M=1900, N=3101, K=1503, depth=-1, pad=13,
             alpha=0.75, beta=0.5, dist="normal"),
        # square products at the sizes of the size sweep: one, two and three levels
        dict(name="fp32_4096", kind="gemm", precision="fp32", M=4096, N=4096, K=4096, depth=-1, pad=0, alpha=1.0,
             beta=0.0, dist="normal"),
        dict(name="fp32_8192", kind="gemm", precision="fp32", M=8192, N=8192, K=8192, depth=-1, pad=0, alpha=1.0,
             beta=0.0, dist="uniform"),
        # the headline call
        dict(name="fp32_16384", kind="gemm", precision="fp32", M=16384, N=16384, K=16384, depth=-1, pad=0, alpha=1.0,
             beta=0.0, dist="uniform"),
        # split precision: the large rectangular product, and wide magnitudes in scaled fp16
        dict(name="bf16x3_19000x15000x12000", kind="gemm", precision="bf16x3", M=19000, N=15000, K=12000, depth=-1,
             pad=0, alpha=1.0, beta=0.0, dist="normal"),
        dict(name="fp16x3_8192", kind="gemm", precision="fp16x3", M=8192, N=8192, K=8192, depth=-1, pad=0, alpha=1.0,
             beta=0.0, dist="loguniform"),
        # 512 uneven products, one persistent launch
        dict(name="batched_512", kind="batched", precision="fp32", count=512, shapes=20260400, lo=128, hi=4096,
             multiple=4),
        # operands in pinned host memory, streamed
        dict(name="host_8192", kind="host", precision="fp32", M=8192, N=8192, K=8192, alpha=1.0, beta=0.0,
             dist="uniform"),
        # the check of a product: odd, rectangular
        dict(name="residual_12000x9001", kind="residual", M=12000, N=9001, K=10500, dist="uniform"),
        # the cost model's training on 20000 timings, one of its full-batch steps
        dict(name="train_20000", kind="train", batch=20000, step=200),
    ]


def _size(rng, lo, hi):
    """Log-uniform in [lo, hi]; half of them odd, the rest multiples of 4."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    n = n | 1 if rng.random() < 0.5 else n // 4 * 4
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "gemm", "gemm", "static", "batched", "host", "residual", "train"])
    dist = rng.choice(["uniform", "normal", "loguniform"])
    ab = rng.choice([(1.0, 0.0), (1.0, 0.0), (0.75, 0.5), (-1.0, 0.0), (1.0, -0.25)])
    if kind == "gemm":
        precision = rng.choice(["fp32", "fp32", "fp32", "bf16x3", "fp16x3", "tf32"])
        while True:
            M, N, K = _size(rng, 256, 16384), _size(rng, 256, 16384), _size(rng, 256, 16384)
            if M * N * K <= 12000 ** 3:
                break
        small = max(M, N, K) <= 2048 and min(M, N, K) >= 512
        return dict(kind=kind, precision=precision, M=M, N=N, K=K, depth=2 if small and rng.random() < 0.5 else -1,
                    pad=rng.choice([0, 0, 8, 13]), alpha=ab[0], beta=ab[1], dist=dist)
    if kind == "static":
        return dict(kind=kind, M=_size(rng, 64, 1024), N=_size(rng, 64, 1024), K=_size(rng, 64, 1024), alpha=ab[0],
                    beta=ab[1], dist=dist)
    if kind == "batched":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp32", "bf16x3", "fp16x3", "tf32"]),
                    count=_size(rng, 16, 512), shapes=rng.randrange(1 << 30), lo=128, hi=rng.choice([1024, 2048, 4096]),
                    multiple=rng.choice([1, 4]))
    if kind == "host":
        return dict(kind=kind, precision="fp32", M=_size(rng, 2048, 8192), N=_size(rng, 2048, 8192),
                    K=_size(rng, 2048, 8192), alpha=ab[0], beta=ab[1], dist=dist)
    if kind == "residual":
        return dict(kind=kind, M=_size(rng, 1024, 16384), N=_size(rng, 1024, 16384), K=_size(rng, 1024, 16384),
                    dist="uniform")
    return dict(kind=kind, batch=_size(rng, 256, 26000), step=rng.randrange(1, 2000))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _matrix(g, rows, cols, dist):
    if dist == "normal":
        return torch.randn((rows, cols), generator=g, device="cuda")
    x = torch.rand((rows, cols), generator=g, device="cuda")
    if dist == "uniform":
        return x.mul_(2).sub_(1)
    # sign * 10^U(-3, 3)
    sign = torch.rand((rows, cols), generator=g, device="cuda").sub_(0.5).sign_()
    return x.mul_(6 * math.log(10)).sub_(3 * math.log(10)).exp_().mul_(sign)


def _operands(case, seed):
    """A, B and the C that a beta reads, with `pad` unused columns beyond each row."""
    g, pad = _gen(seed), int(case.get("pad", 0))
    M, N, K, dist = case["M"], case["N"], case["K"], case["dist"]
    A = _matrix(g, M, K + pad, dist)[:, :K]
    B = _matrix(g, K, N + pad, dist)[:, :N]
    C = _matrix(g, M, N + pad, "normal")[:, :N] if case["beta"] else torch.zeros((M, N + pad), device="cuda")[:, :N]
    return A, B, C


def _batched_shapes(case):
    return inputs.batched_shapes(case["count"], case["shapes"], case["lo"], case["hi"], case["multiple"])


def _carve(shapes):
    """One buffer holding a matrix of each shape, every one on a 256-byte boundary."""
    starts, at = [], 0
    for r, c in shapes:
        starts.append(at)
        at += -(-(r * c) // 64) * 64
    return starts, at


def _batched_operands(case, seed):
    g, shapes = _gen(seed), _batched_shapes(case)
    out = []
    for pick in (lambda m, k, n: (m, k), lambda m, k, n: (k, n), lambda m, k, n: (m, n)):
        dims = [pick(*s) for s in shapes]
        starts, total = _carve(dims)
        flat = torch.zeros(total, device="cuda") if len(out) == 2 else _matrix(g, 1, total, "uniform").view(-1)
        out.append((flat, [flat[s: s + r * c].view(r, c) for s, (r, c) in zip(starts, dims)]))
    return out


def _train_inputs(case, seed):
    g, n = _gen(seed), case["batch"]
    u = torch.rand((n, 3), generator=g, device="cuda") * 5 + 7                       # log2 of M, K, N
    depth = torch.randint(0, 5, (n,), generator=g, device="cuda").float()
    tile = 2.0 ** torch.randint(0, 3, (n,), generator=g, device="cuda").float()
    prec = torch.randint(0, 4, (n,), generator=g, device="cuda").float()
    X = torch.cat([u, depth[:, None], tile[:, None], prec[:, None]], 1)
    # log milliseconds: work that a level cuts by 7/8, launches that it adds, measurement noise
    T = torch.log(2.0 ** (u.sum(1) - 38) * (7 / 8) ** depth * (1 + 0.2 * tile) + 0.02 + 0.01 * depth)
    T = T + 0.05 * torch.randn(n, generator=g, device="cuda")
    X = (X - X.mean(0)) / X.std(0)
    p = torch.zeros(NPARAM, device="cuda")
    p[:384] = torch.randn(384, generator=g, device="cuda") * math.sqrt(2 / 6)
    p[448:4544] = torch.randn(4096, generator=g, device="cuda") * math.sqrt(2 / 64)
    p[4608:4672] = torch.randn(64, generator=g, device="cuda") * math.sqrt(1 / 64)
    m = torch.randn(NPARAM, generator=g, device="cuda") * 1e-2                       # moments of a run under way
    v = torch.rand(NPARAM, generator=g, device="cuda") * 1e-3 + 1e-4
    return X.contiguous(), T.contiguous(), p, m, v


def _residual_inputs(case, seed):
    """A, B, a product in hand that carries split-precision rounding, and the +-1 probe."""
    g = _gen(seed)
    A, B = _matrix(g, case["M"], case["K"], case["dist"]), _matrix(g, case["K"], case["N"], case["dist"])
    C = A @ B
    C.mul_(torch.rand(C.shape, generator=g, device="cuda").mul_(2e-5).add_(1 - 1e-5))
    x = torch.rand(case["N"], generator=g, device="cuda").sub_(0.5).sign_()
    return A, B, C, x


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B, C = _operands(case, seed)
        pad = case["pad"]
        plan = fmm.Plan(case["M"], case["N"], case["K"], case["K"] + pad, case["N"] + pad, case["N"] + pad,
                        depth=case["depth"], precision=case["precision"])
        return dict(case=case, plan=plan, A=A, B=B, C=C)
    if kind == "static":
        A, B, C = _operands(case, seed)
        return dict(case=case, A=A, B=B, C=C)
    if kind == "batched":
        (_, As), (_, Bs), (flat, Cs) = _batched_operands(case, seed)
        return dict(case=case, plan=fmm.BatchedPlan(As, Bs, Cs, precision=case["precision"]), flat=flat)
    if kind == "host":
        A, B, C = (torch.empty(t.shape, pin_memory=True).copy_(t) for t in _operands(case, seed))
        plan = fmm.Plan(case["M"], case["N"], case["K"], precision=case["precision"], host_operands=1)
        return dict(case=case, plan=plan, A=A, B=B, C=C)
    if kind == "residual":
        A, B, C, x = _residual_inputs(case, seed)
        return dict(case=case, A=A, B=B, C=C, x=x)
    X, T, p, m, v = _train_inputs(case, seed)
    ws = torch.empty(fmm.mlp_workspace_bytes(case["batch"]), dtype=torch.uint8, device="cuda")
    return dict(case=case, X=X, T=T, p=p, m=m, v=v, ws=ws, grad=torch.empty_like(p),
                loss=torch.zeros(1, device="cuda"))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("gemm", "host"):
        return state["plan"](state["A"], state["B"], state["C"], alpha=case["alpha"], beta=case["beta"])
    if kind == "static":
        return fmm.fmm_gemm_static(state["A"], state["B"], state["C"], alpha=case["alpha"], beta=case["beta"])
    if kind == "batched":
        state["plan"].run()
        return state["flat"]
    if kind == "residual":
        return fmm.fmm_residual(state["A"], state["B"], state["C"], state["x"], fp64=True)
    fmm.fmm_mlp_train_step(state["p"], state["m"], state["v"], case["step"], 3e-3, state["X"], state["T"],
                           state["ws"], grad_out=state["grad"], loss_out=state["loss"])
    return dict(params=state["p"], m=state["m"], v=state["v"], grad=state["grad"], loss=state["loss"])


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    kind = case["kind"]
    if kind in ("gemm", "static", "host"):
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=4.0 * (M * K + K * N + M * N * (2 if case["beta"] else 1)), flops=2.0 * M * N * K)
    if kind == "batched":
        s = _batched_shapes(case)
        return dict(bytes=4.0 * sum(m * k + k * n + m * n for m, k, n in s), flops=2.0 * sum(m * k * n for m, k, n in s))
    if kind == "residual":
        M, N, K = case["M"], case["N"], case["K"]
        e = float(M * K + K * N + M * N)
        return dict(bytes=4.0 * e + 4.0 * N + 8.0 * M, flops=2.0 * e)
    n = case["batch"]   # forward, both backward products of the hidden layer, every gradient
    return dict(bytes=4.0 * (7 * n + 7 * NPARAM), flops=2.0 * n * (3 * 64 * 64 + 2 * 6 * 64 + 3 * 64))


# ------------------------------------------------------------------ in 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind in ("gemm", "static", "host"):
        A, B, C = _operands(case, seed)
        if 2.0 * case["M"] * case["N"] * case["K"] > 1e13:
            return None
        out = torch.matmul(A.double(), B.double()).mul_(case["alpha"])
        if case["beta"]:
            out.add_(C.double(), alpha=case["beta"])
        return out.cpu() if kind == "host" else out
    if kind == "batched":
        (_, As), (_, Bs), (flat, Cs) = _batched_operands(case, seed)
        starts, total = _carve([tuple(c.shape) for c in Cs])
        out = torch.zeros(total, dtype=torch.float64, device="cuda")
        for s, A, B in zip(starts, As, Bs):
            n = A.shape[0] * B.shape[1]
            out[s: s + n] = torch.matmul(A.double(), B.double()).view(-1)
        return out
    if kind == "residual":
        A, B, C, x = _residual_inputs(case, seed)
        xd = x.double()
        return torch.mv(C.double(), xd) - torch.mv(A.double(), torch.mv(B.double(), xd))
    X, T, p, m, v = (t.double() for t in _train_inputs(case, seed))
    n, step = case["batch"], case["step"]
    W1, b1, W2 = p[:384].view(64, 6), p[384:448], p[448:4544].view(64, 64)
    b2, w3, b3 = p[4544:4608], p[4608:4672], p[4672]
    h1 = torch.relu(X @ W1.T + b1)
    h2 = torch.relu(h1 @ W2.T + b2)
    r = h2 @ w3 + b3 - T
    dy = r / n
    d2 = dy[:, None] * w3 * (h2 > 0)
    d1 = (d2 @ W2) * (h1 > 0)
    grad = torch.cat([(d1.T @ X).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), dy @ h2, dy.sum()[None]])
    m = 0.9 * m + 0.1 * grad
    v = 0.999 * v + 0.001 * grad * grad
    p = p - 3e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    return dict(params=p, m=m, v=v, grad=grad, loss=(0.5 * (r * r).mean())[None])
