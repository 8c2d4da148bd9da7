"""The work that programs have this library do, as timed cases.

Families (the `kind` of a case):

* "qr": the R factor of a new matrix on a kept factorization handle (plan and
  workspace made once, `refactor_async` per matrix). R is scaled to a positive
  diagonal, which makes it unique.
* "qr_q": the same and Q itself (square matrices).
* "fit": a new matrix is factored (unless `kept`) and a block of right-hand
  sides is projected on its column space: Q^T B, the rows past N set to zero,
  Q times that. Both directions of Q in one pass.
* "ls": a least-squares plan over one or many problems, run on what the
  buffers hold (mixed precision with refinement for FP32 matrices, plain QR
  for FP64 ones).
* "gels": the one-shot solve with tolerance-stopped refinement.

`dtype` is the storage type ("f64", "f32"); `tensor` puts FP32 tiles of 128 on
the tensor-core kernels.
"""
import math

import torch

from paper_1110_1553_gb300 import hqr, workloads

DEVICE = "cuda"
TREES = ("flat", "binary", "greedy", "fibonacci")


def _qr(kind, dtype, tensor, M, N, nb, ib, a, p, low, high, **more):
    c = dict(kind=kind, dtype=dtype, tensor=tensor, M=M, N=N, nb=nb, ib=ib, a=a, p=p, low=low, high=high)
    c.update(more)
    return c


def listed():
    cases = {
        # the smallest calls: a small ragged regression, one launch deep, all latency
        "qr64_130x70": _qr("qr", "f64", False, 130, 70, 32, 16, 4, 1, "greedy", "greedy"),
        # latency of one small square factorization with Q formed, flat tree
        "qr64_q_512": _qr("qr_q", "f64", False, 512, 512, 64, 16, 8, 1, "flat", "flat"),
        # an ordinary square FP64 matrix whose size is no multiple of the tile
        "qr64_2000": _qr("qr", "f64", False, 2000, 2000, 128, 32, 4, 4, "fibonacci", "flat"),
        # the tall-skinny FP64 setting of the benchmark at a quarter of its height
        "qr64_tall_32768x2048": _qr("qr", "f64", False, 32768, 2048, 256, 32, 4, 16, "greedy", "fibonacci"),
        # square FP32 on the tensor cores, bound by the chain of panels
        "qr32tc_6144": _qr("qr", "f32", True, 6144, 6144, 128, 128, 16, 1, "greedy", "greedy"),
        # tall FP32 on the tensor cores, bound by the updates; ragged in both directions
        "qr32tc_tall_65000x2000": _qr("qr", "f32", True, 65000, 2000, 128, 128, 8, 8, "greedy", "greedy"),
        # plain FP32 (CUDA cores): factor and project a few right-hand sides
        "fit32_2500x1700": _qr("fit", "f32", False, 2500, 1700, 128, 16, 4, 2, "binary", "binary", nrhs=40, kept=False),
        # many new right-hand sides on kept tensor-core factors
        "fit32tc_8192x1024": _qr("fit", "f32", True, 8192, 1024, 128, 128, 8, 4, "greedy", "fibonacci", nrhs=300,
                                 kept=True),
        # an ill-conditioned square system, FP32 QR refined to FP64 accuracy
        "ls_mixed_4096": dict(kind="ls", dtype="f32", tensor=True, M=4096, N=4096, count=1, kappa=1e6, iters=40, tol=1e-12),
        # a batch of uneven least-squares problems, mixed precision
        "ls_batch_mixed_160": dict(kind="ls", dtype="f32", tensor=True, M=8192, N=512, count=160, kappa=0.0, iters=5,
                                   tol=0.0),
        # the same in plain FP64
        "ls_batch_f64_48": dict(kind="ls", dtype="f64", tensor=False, M=8192, N=512, count=48, kappa=0.0, iters=0,
                                tol=0.0),
        # one small solve from scratch, nothing kept by the caller
        "gels_300x40": dict(kind="gels", dtype="f32", tensor=True, M=300, N=40, iters=30, tol=1e-12),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["qr64", "qr64", "qr32tc", "qr32tc", "qr_q", "fit32", "fit32tc", "ls_mixed", "ls_batch", "ls_batch64",
                       "gels"])
    low, high = rng.choice(TREES), rng.choice(TREES)
    a, p = rng.choice([1, 2, 4, 8, 16]), rng.choice([1, 1, 2, 4, 16])
    if kind in ("qr64", "qr32tc"):
        f64 = kind == "qr64"
        most = 2.0 * 32768 * 2048 ** 2 if f64 else 2.0 * 65000 * 2000 ** 2  # flops of the largest listed ones
        while True:
            M, N = _log_int(rng, 64, 32768 if f64 else 65000), _log_int(rng, 32, 2048 if f64 else 6144)
            if M >= N and 2.0 * M * N * N <= most:
                break
        if not f64:
            return _qr("qr", "f32", True, M, N, 128, 128, a, p, low, high)
        nb = rng.choice([32, 64] if N <= 192 else [64, 128] if N <= 1024 else [128, 256])
        return _qr("qr", "f64", False, M, N, nb, 32 if nb >= 128 else 16, a, p, low, high)
    if kind == "qr_q":
        n = _log_int(rng, 64, 1024)
        return _qr("qr_q", "f64", False, n, n, 64, 16, a, p, low, high)
    if kind in ("fit32", "fit32tc"):
        N = _log_int(rng, 100, 1700)
        M = _log_int(rng, N + N // 8 + 1, min(8192, 5 * N))
        nrhs = _log_int(rng, 1, 300)
        if kind == "fit32":
            nb = rng.choice([32, 64, 128])
            return _qr("fit", "f32", False, M, N, nb, 16, a, p, low, high, nrhs=nrhs, kept=rng.random() < 0.5)
        return _qr("fit", "f32", True, M, N, 128, 128, a, p, low, high, nrhs=nrhs, kept=rng.random() < 0.5)
    if kind == "ls_mixed":
        N = _log_int(rng, 256, 4096)
        M = min(_log_int(rng, N, 4 * N), max(N, 2 ** 24 // N))
        return dict(kind="ls", dtype="f32", tensor=rng.random() < 0.75, M=M, N=N, count=1,
                    kappa=10.0 ** rng.uniform(2, 6), iters=40, tol=1e-12)
    if kind == "ls_batch":
        return dict(kind="ls", dtype="f32", tensor=rng.random() < 0.75, M=8192, N=512, count=_log_int(rng, 4, 160),
                    kappa=0.0, iters=5, tol=0.0)
    if kind == "ls_batch64":
        return dict(kind="ls", dtype="f64", tensor=False, M=8192, N=512, count=_log_int(rng, 2, 48), kappa=0.0, iters=0,
                    tol=0.0)
    N = _log_int(rng, 8, 400)
    return dict(kind="gels", dtype=rng.choice(["f32", "f32", "f64"]), tensor=rng.random() < 0.75, M=_log_int(rng, N, 8 * N + 64),
                N=N, iters=30, tol=1e-12)


# ------------------------------------------------------------------ inputs --

def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(11101553 + 7919 * int(seed))
    return g


def _gaussian(M, N, dtype, g):
    return torch.randn((N, M), dtype=dtype, device=DEVICE, generator=g).t()


def _shapes(case):
    """Sizes of a plan's problems: one, or `count` uneven ones up to M x N."""
    if case["count"] == 1:
        return [(case["M"], case["N"])]
    return workloads.uneven_shapes(case["count"], seed=case["count"], mmax=case["M"], nmax=case["N"])


def _ls_inputs(case, seed):
    """(A, b) of every problem of a least-squares case: b = A x_true plus noise."""
    g = _generator(seed)
    out = []
    for M, N in (_shapes(case) if case["kind"] == "ls" else [(case["M"], case["N"])]):
        if case.get("kappa", 0.0) > 0.0:
            A = workloads.conditioned(torch, M, N, case["kappa"], seed=int(seed), device=DEVICE)
            noise = 1e-8
        else:
            A = _gaussian(M, N, _dtype(case), g)
            noise = 0.1
        b = A.double() @ torch.randn(N, dtype=torch.float64, device=DEVICE, generator=g)
        b += noise * torch.randn(M, dtype=torch.float64, device=DEVICE, generator=g)
        out.append((A, b))
    return out


def _qr_inputs(case, seed):
    g = _generator(seed)
    A = _gaussian(case["M"], case["N"], _dtype(case), g)
    B = _gaussian(case["M"], case["nrhs"], _dtype(case), g) if case["kind"] == "fit" else None
    return A, B


def prepare(case, seed):
    if case["kind"] == "gels":
        A, b = _ls_inputs(case, seed)[0]
        return {"case": case, "A": A, "b": b}
    if case["kind"] == "ls":
        problems = _ls_inputs(case, seed)
        x = torch.zeros(sum(A.shape[1] for A, _ in problems), dtype=torch.float64, device=DEVICE)
        views, at = [], 0
        for A, b in problems:
            views.append((A, b, x[at:at + A.shape[1]]))
            at += A.shape[1]
        plan = hqr.LSPlan(views, refine_iters=case["iters"], tensor=case["tensor"], tol=case["tol"] or None)
        return {"case": case, "plan": plan, "x": x}
    M, N, nb = case["M"], case["N"], case["nb"]
    A, B = _qr_inputs(case, seed)
    records = hqr.elim_list(-(-M // nb), -(-N // nb), case["a"], case["p"], case["low"], case["high"])
    state = {"case": case, "A": A, "F": hqr.geqrf(A, nb, case["ib"], records, tensor=case["tensor"])}
    if case["kind"] == "qr_q":
        state["eye"] = torch.eye(M, dtype=A.dtype, device=DEVICE)
        state["Q"] = hqr.empty_colmajor(M, M, dtype=A.dtype)
    if B is not None:
        state["B"] = B
        state["P"] = hqr.empty_colmajor(M, case["nrhs"], dtype=A.dtype)
    return state


# -------------------------------------------------------------------- runs --

def run(state):
    case = state["case"]
    if case["kind"] == "gels":
        return hqr.gels(state["A"], state["b"], tol=case["tol"], max_iter=case["iters"], tensor=case["tensor"])[0]
    if case["kind"] == "ls":
        state["plan"].run()
        return state["x"]
    F = state["F"]
    if case["kind"] == "fit":
        if not case["kept"]:
            F.refactor_async(state["A"])
        P = state["P"]
        P.copy_(state["B"])
        F.apply_q(P, trans=True)
        P[case["N"]:] = 0
        F.apply_q(P, trans=False)
        return P
    F.refactor_async(state["A"])
    R = F.R()
    sign = torch.sign(torch.diagonal(R))
    if case["kind"] == "qr":
        return R.mul_(sign.unsqueeze(1))
    Q = state["Q"]
    Q.copy_(state["eye"])
    F.apply_q(Q, trans=False)
    return [R.mul_(sign.unsqueeze(1)), Q * sign]


def work(case):
    es = 8 if case["dtype"] == "f64" else 4

    def qr_flops(M, N):
        return 2.0 * M * N * N - 2.0 / 3.0 * N ** 3

    if case["kind"] in ("gels", "ls"):
        shapes = _shapes(case) if case["kind"] == "ls" else [(case["M"], case["N"])]
        return {"bytes": sum(es * M * N + 8 * (M + N) for M, N in shapes), "flops": sum(qr_flops(M, N) for M, N in shapes)}
    M, N = case["M"], case["N"]
    if case["kind"] == "fit":
        n = case["nrhs"]
        flops = 2 * (4.0 * M * N - 2.0 * N * N) * n + (0.0 if case["kept"] else qr_flops(M, N))
        return {"bytes": es * (M * N + 2 * M * n), "flops": flops}
    if case["kind"] == "qr_q":
        return {"bytes": es * (M * N + N * N + M * M), "flops": qr_flops(M, N) + (4.0 * M * N - 2.0 * N * N) * M}
    return {"bytes": es * (M * N + N * N), "flops": qr_flops(M, N)}


def tolerance(case):
    """About four times the distance from `exact` seen on the ranges above: FP64
    factors 3e-15 (Q: 6e-15), FP64 solutions 1e-15, FP32 R 2.5e-6, FP32
    projections 2e-6 and with the tensor-core factors 1e-5. Refined solutions
    are asked for 1e-12, or take a fixed number of rounds that leave no more
    than 1e-13."""
    f64 = case["dtype"] == "f64"
    if case["kind"] in ("gels", "ls"):
        if f64 and not case["tol"]:
            return {"rel": 1e-14}
        return {"rel": 1e-12 if case["tol"] else 1e-13}
    if f64:
        return {"rel": 4e-14 if case["kind"] == "qr_q" else 2e-14}
    return {"rel": 4e-5 if case["kind"] == "fit" and case["tensor"] else 1e-5}


# ------------------------------------------------------------------- exact --

def _halves(a):
    c = 134217729.0 * a
    hi = c - (c - a)
    return hi, a - hi


def _dot_rows(A, x, extra):
    """sum(extra) - A x with products split into exact parts and summed in
    twice the working precision (pairwise TwoSum)."""
    out = torch.empty(A.shape[0], dtype=torch.float64, device=A.device)
    xh, xl = _halves(x)
    step = max(1, 2 ** 24 // A.shape[1])
    for r in range(0, A.shape[0], step):
        a = A[r:r + step]
        terms = [-(a * xh), -(a * xl)]
        if A.dtype == torch.float64:
            ah, al = _halves(a)
            terms = [-(ah * xh), -(ah * xl), -(al * xh), -(al * xl)]
        s = torch.cat(terms + [e[r:r + step].unsqueeze(1) for e in extra], dim=1)
        c = torch.zeros_like(s)
        while s.shape[1] > 1:
            if s.shape[1] % 2:
                s, c = (torch.nn.functional.pad(t, (0, 1)) for t in (s, c))
            p, q = s[:, 0::2], s[:, 1::2]
            t = p + q
            z = t - p
            c = c[:, 0::2] + c[:, 1::2] + ((p - (t - z)) + (q - z))
            s = t
        out[r:r + step] = (s + c)[:, 0]
    return out


def _least_squares(A, b):
    """min ||b - A x|| in 64 bits: QR and three steps of refinement of the
    augmented system with its residuals in twice that."""
    A64 = A.double()
    Q, R = torch.linalg.qr(A64)

    def back(v):
        return torch.linalg.solve_triangular(R, v.unsqueeze(1), upper=True)[:, 0]

    x = back(Q.t() @ b)
    r = _dot_rows(A64, x, [b])
    for _ in range(3):
        f1 = _dot_rows(A64, x, [b, -r])
        f2 = _dot_rows(A64.t().contiguous(), r, [])
        d = Q.t() @ f1 - torch.linalg.solve_triangular(R.t(), f2.unsqueeze(1), upper=False)[:, 0]
        x = x + back(d)
        r = r + f1 - Q @ d
    return x


def exact(case, seed):
    if case["kind"] in ("gels", "ls"):
        x = [_least_squares(A, b) for A, b in _ls_inputs(case, seed)]
        return x[0] if case["kind"] == "gels" else torch.cat(x)
    A, B = _qr_inputs(case, seed)
    Q, R = torch.linalg.qr(A.double(), mode="r" if case["kind"] == "qr" else "reduced")
    if case["kind"] == "fit":
        return Q @ (Q.t() @ B.double())
    sign = torch.sign(torch.diagonal(R))
    R = R * sign.unsqueeze(1)
    return R if case["kind"] == "qr" else [R, Q * sign]
