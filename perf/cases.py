"""Performance cases of the out-of-core GEMM library.

Each case is one call (or one factorization) through the public binding, on operands where a
user has them: pinned host memory for the out-of-core entry points, device memory for the
in-core one.  Sizes are those of the repository's smoke run, tests and benchmark
configurations, the large ones scaled down to passes well under a second with the same
proportions and the same ratio of operands to device budget.
"""
import math

import numpy as np
import torch

import paper_1808_05056_gb300 as ooc

MIB = 1 << 20
FORMS = {"fp64": ooc.OOC_FORM_FP64, "ozaki": ooc.OOC_FORM_OZAKI, "bf16x3": ooc.OOC_FORM_BF16X3}


def _gemm(name, form, ta, tb, M, N, K, alpha, beta, dist, budget):
    return {"name": name, "op": "gemm", "form": form, "ta": ta, "tb": tb, "M": M, "N": N, "K": K, "alpha": alpha,
            "beta": beta, "dist": dist, "budget": budget}


def listed():
    return [
        # the smoke run's product: the smallest out-of-core call, all overhead and a few tiles
        _gemm("dgemm_smallest", "fp64", "N", "N", 384, 320, 256, 1.5, 0.5, "uniform", 1 * MIB),
        # the paper-sized small configuration: 1024^3 under a 4 MiB budget, many small blocks
        _gemm("dgemm_1024", "fp64", "N", "N", 1024, 1024, 1024, 1.0, 0.0, "uniform", 4 * MIB),
        # the default workload's kind of call (FP64, alpha and beta, operands six times the budget),
        # ragged and with a transposed operand
        _gemm("dgemm_large_ragged", "fp64", "T", "N", 6000, 5003, 7001, 1.5, 0.5, "normal", 152 * MIB),
        # the in-core device call of an outer algorithm (the paper's runtime DGEMM)
        {"name": "dgemm_device", "op": "device", "ta": "N", "tb": "T", "M": 1536, "N": 1000, "K": 2000,
         "alpha": -1.0, "beta": 1.0},
        # FP64-accurate products on the tensor cores: a mid-size ragged call ...
        _gemm("ozaki_ragged", "ozaki", "N", "T", 2500, 3100, 1900, 1.0, 0.5, "logspread", 64 * MIB),
        # ... and the benchmark's 4 : 4 : 1 shape, wide exponent spread, operands 3.5 times the budget
        _gemm("ozaki_large", "ozaki", "N", "N", 10240, 10240, 2560, 1.0, 0.0, "logspread", 400 * MIB),
        # FP32-accurate products: mid-size ragged, transposed
        _gemm("sgemm_ragged", "bf16x3", "T", "N", 3000, 2001, 2502, 1.5, 0.5, "uniform", 24 * MIB),
        # FP32-accurate square product that reads and writes C, operands six times the budget
        _gemm("sgemm_large", "bf16x3", "N", "N", 12288, 12288, 12288, 1.0, 0.5, "uniform", 288 * MIB),
        # a stream of uneven FP64 products in one captured graph (the batched benchmark, scaled down)
        {"name": "batched_uneven", "op": "batched", "count": 20, "lo": 256, "hi": 2048, "shapes": 1234,
         "budget": 256 * MIB, "graph": True},
        # the solves and factorizations built on the product
        {"name": "trsm", "op": "trsm", "form": "ozaki", "side": "L", "uplo": "L", "ta": "N", "diag": "N", "M": 4096,
         "N": 3000, "alpha": 1.0, "budget": 64 * MIB},
        {"name": "potrf", "op": "potrf", "form": "fp64", "uplo": "L", "N": 4096, "budget": 64 * MIB},
        {"name": "getrf", "op": "getrf", "form": "fp64", "N": 4096, "budget": 64 * MIB},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the operations of listed(), sizes log-uniform between its smallest and largest."""
    op = rng.choice(["fp64", "fp64", "ozaki", "ozaki", "bf16x3", "bf16x3", "device", "batched", "trsm", "potrf",
                     "getrf"])
    if op in FORMS:
        hi, cap = {"fp64": (7000, 4.2e11), "ozaki": (10240, 5.3e11), "bf16x3": (12288, 3.7e12)}[op]
        while True:
            M, N, K = (_log_int(rng, 256, hi) for _ in range(3))
            if 2.0 * M * N * K <= cap:
                break
        es = 4 if op == "bf16x3" else 8
        foot = es * (M * K + K * N + M * N)
        budget = max(4 * MIB, int(foot * rng.uniform(0.16, 0.6)))
        if op != "fp64":  # the split planes of the smallest whole-tile plan fit with room
            budget = max(budget, 24 * MIB, 2 * 128 * es * 6 * K)
        c = _gemm("", op, rng.choice("NT"), rng.choice("NT"), M, N, K, rng.choice([1.0, 1.5, -1.0]),
                  rng.choice([0.0, 0.5]),
                  {"fp64": "normal", "ozaki": rng.choice(["logspread", "normal"]), "bf16x3": "uniform"}[op], budget)
        del c["name"]
        return c
    if op == "device":
        M, N, K = (2 * _log_int(rng, 32, 1500) for _ in range(3))
        return {"op": "device", "ta": rng.choice("NT"), "tb": rng.choice("NT"), "M": M, "N": N, "K": K,
                "alpha": rng.choice([1.0, -1.0]), "beta": rng.choice([0.0, 1.0])}
    if op == "batched":
        hi = _log_int(rng, 512, 2048)
        return {"op": "batched", "count": rng.randint(4, 24), "lo": rng.randint(128, 256), "hi": hi,
                "shapes": rng.randrange(1 << 20), "budget": 256 * MIB, "graph": rng.random() < 0.7}
    n = _log_int(rng, 600, 4096)
    form = rng.choice(["fp64", "ozaki"])
    budget = max(64 * MIB, 8 * n * n // 3)
    if op == "trsm":
        left = rng.random() < 0.5
        v = _log_int(rng, 600, 4096)
        return {"op": "trsm", "form": form, "side": "L" if left else "R", "uplo": rng.choice("LU"),
                "ta": rng.choice("NT"), "diag": "N", "M": n if left else v, "N": v if left else n, "alpha": 1.0,
                "budget": budget}
    if op == "potrf":
        return {"op": "potrf", "form": form, "uplo": rng.choice("LU"), "N": n, "budget": budget}
    return {"op": "getrf", "form": form, "N": n, "budget": budget}


# ------------------------------------------------------------------ inputs --
def _values(gen, rows, cols, dist, dtype):
    """A rows x cols device tensor of the named distribution."""
    kw = {"generator": gen, "device": "cuda", "dtype": torch.float64}
    if dist == "normal":
        x = torch.randn(rows, cols, **kw)
    elif dist == "uniform":
        x = torch.rand(rows, cols, **kw).mul_(2.0).sub_(1.0)
    else:  # sign * 10^U(-4, 4)
        x = torch.rand(rows, cols, **kw).mul_(8.0).sub_(4.0).mul_(math.log(10.0)).exp_()
        x.mul_(torch.randint(0, 2, (rows, cols), generator=gen, device="cuda").mul_(2).sub_(1))
    return x.to(dtype)


def _pin(x):
    h = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
    h.copy_(x)
    return h


def _stored(rows, cols, t):
    return (rows, cols) if t == "N" else (cols, rows)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _gemm_inputs(case, seed):
    g = _gen(seed)
    dt = torch.float32 if case["form"] == "bf16x3" else torch.float64
    A = _values(g, *_stored(case["M"], case["K"], case["ta"]), case["dist"], dt)
    B = _values(g, *_stored(case["K"], case["N"], case["tb"]), case["dist"], dt)
    C = _values(g, case["M"], case["N"], case["dist"], dt)
    return A, B, C


def _device_inputs(case, seed):
    g = _gen(seed)
    return (_values(g, *_stored(case["M"], case["K"], case["ta"]), "normal", torch.float64),
            _values(g, *_stored(case["K"], case["N"], case["tb"]), "normal", torch.float64),
            _values(g, case["M"], case["N"], "normal", torch.float64))


def _batch_shapes(case):
    """M, N, K of each problem, log-uniform as in the batched benchmark; a quarter use a transposed B."""
    r = np.random.RandomState(case["shapes"])
    mnk = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), (case["count"], 3))).round().astype(int)
    return [(int(m), int(n), int(k), "T" if 4 * i >= 3 * case["count"] else "N") for i, (m, n, k) in enumerate(mnk)]


def _batch_inputs(case, seed):
    g = _gen(seed)
    out = []
    for m, n, k, tb in _batch_shapes(case):
        out.append((_values(g, m, k, "normal", torch.float64), _values(g, *_stored(k, n, tb), "normal", torch.float64),
                    _values(g, m, n, "normal", torch.float64), tb))
    return out


def _trsm_inputs(case, seed):
    """A well-conditioned triangular matrix (dominant diagonal) and the right-hand sides."""
    g = _gen(seed)
    n = case["M"] if case["side"] == "L" else case["N"]
    A = _values(g, n, n, "normal", torch.float64)
    A.div_(math.sqrt(n))
    A.diagonal().add_(4.0)
    return A, _values(g, case["M"], case["N"], "normal", torch.float64)


def _potrf_input(case, seed):
    """Symmetric, entries N(0, 1/2) plus a diagonal that makes it positive definite."""
    g = _gen(seed)
    n = case["N"]
    X = _values(g, n, n, "normal", torch.float64)
    A = X.add(X.t()).mul_(0.5)
    A.diagonal().add_(2.0 * math.sqrt(n))
    return A


def _getrf_input(case, seed):
    return _values(_gen(seed), case["N"], case["N"], "normal", torch.float64)


def prepare(case, seed):
    op = case["op"]
    if op == "gemm":
        A, B, C = (_pin(x) for x in _gemm_inputs(case, seed))
        return {"case": case, "A": A, "B": B, "C": C, "opts": ooc.make_opts(form=FORMS[case["form"]])}
    if op == "device":
        A, B, C = _device_inputs(case, seed)
        return {"case": case, "A": A, "B": B, "C": C, "C0": C.clone()}
    if op == "batched":
        mats = [(_pin(A), _pin(B), _pin(C), tb) for A, B, C, tb in _batch_inputs(case, seed)]
        descs = [ooc.gemm_desc("N", tb, A, B, C, alpha=1.0, beta=0.5) for A, B, C, tb in mats]
        opts = ooc.make_opts(flags=ooc.OOC_BATCH_GRAPH if case["graph"] else 0)
        return {"case": case, "mats": mats, "descs": descs, "opts": opts}
    opts = ooc.make_opts(form=FORMS[case["form"]])
    if op == "trsm":
        A, B = (_pin(x) for x in _trsm_inputs(case, seed))
        return {"case": case, "A": A, "B0": B, "B": torch.empty_like(B, pin_memory=True), "opts": opts}
    A = _pin(_potrf_input(case, seed) if op == "potrf" else _getrf_input(case, seed))
    s = {"case": case, "A0": A, "A": torch.empty_like(A, pin_memory=True), "opts": opts}
    if op == "getrf":
        s["ipiv"] = np.zeros(case["N"], dtype=np.int64)
    return s


def _ok(rc, what):
    if rc != ooc.OOC_OK:
        raise RuntimeError("%s: %s (%d)" % (what, ooc.ooc_last_error(), rc))


def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "gemm":
        f = ooc.sgemm if case["form"] == "bf16x3" else ooc.dgemm
        f(state["A"], state["B"], state["C"], alpha=case["alpha"], beta=case["beta"], budget=case["budget"],
          transA=case["ta"], transB=case["tb"], opts=state["opts"])
        return state["C"]
    if op == "device":
        C = state["C"]
        if case["beta"] != 0.0:  # an update of a fresh C on each pass
            C.copy_(state["C0"])
        _ok(ooc.ooc_dgemm_device(case["ta"], case["tb"], case["M"], case["N"], case["K"], case["alpha"], state["A"],
                                 state["A"].shape[1], state["B"], state["B"].shape[1], case["beta"], C, C.shape[1],
                                 torch.cuda.current_stream().cuda_stream), "ooc_dgemm_device")
        return C
    if op == "batched":
        _ok(ooc.ooc_dgemm_batched(state["descs"], case["budget"], state["opts"]), "ooc_dgemm_batched")
        return [m[2] for m in state["mats"]]
    # the solves and factorizations overwrite their operand: a fresh copy for each pass
    if op == "trsm":
        B = state["B"]
        B.copy_(state["B0"])
        _ok(ooc.ooc_dtrsm(case["side"], case["uplo"], case["ta"], case["diag"], case["M"], case["N"], case["alpha"],
                          state["A"], state["A"].shape[1], B, case["N"], case["budget"], state["opts"]), "ooc_dtrsm")
        return B
    A = state["A"]
    A.copy_(state["A0"])
    if op == "potrf":
        rc, info = ooc.ooc_dpotrf(case["uplo"], case["N"], A, case["N"], case["budget"], state["opts"])
        _ok(rc, "ooc_dpotrf")
        return {"factor": A, "info": info}
    rc, info = ooc.ooc_dgetrf(case["N"], A, case["N"], state["ipiv"], case["budget"], state["opts"])
    _ok(rc, "ooc_dgetrf")
    return {"lu": A, "ipiv": state["ipiv"], "info": info}


# ------------------------------------------------------------- accounting --
def work(case):
    op = case["op"]
    if op in ("gemm", "device"):
        M, N, K = case["M"], case["N"], case["K"]
        es = 4 if case.get("form") == "bf16x3" else 8
        c = 2 if case["beta"] != 0.0 else 1
        return {"bytes": es * (M * K + K * N + c * M * N), "flops": 2 * M * N * K}
    if op == "batched":
        s = _batch_shapes(case)
        return {"bytes": sum(8 * (m * k + k * n + 2 * m * n) for m, n, k, _ in s),
                "flops": sum(2 * m * n * k for m, n, k, _ in s)}
    if op == "trsm":
        M, N = case["M"], case["N"]
        n, v = (M, N) if case["side"] == "L" else (N, M)
        return {"bytes": 8 * (n * n // 2 + 2 * n * v), "flops": n * n * v}
    n = case["N"]
    if op == "potrf":
        return {"bytes": 8 * n * n, "flops": n ** 3 // 3}
    return {"bytes": 16 * n * n, "flops": 2 * n ** 3 // 3}


def _op(x, t):
    return x if t == "N" else x.t()


def exact(case, seed):
    """The outputs of run() on a new state, in 64 bits by plain torch."""
    op = case["op"]
    if op in ("gemm", "device"):
        A, B, C = (_gemm_inputs if op == "gemm" else _device_inputs)(case, seed)
        R = torch.mm(_op(A.double(), case["ta"]), _op(B.double(), case["tb"])).mul_(case["alpha"])
        if case["beta"] != 0.0:
            R.add_(C.double(), alpha=case["beta"])
        return R
    if op == "batched":
        return [torch.mm(A, _op(B, tb)).add_(C, alpha=0.5) for A, B, C, tb in _batch_inputs(case, seed)]
    if op == "trsm":
        A, B = _trsm_inputs(case, seed)
        T = torch.tril(A) if case["uplo"] == "L" else torch.triu(A)
        upper = (case["uplo"] == "U") != (case["ta"] == "T")
        return torch.linalg.solve_triangular(_op(T, case["ta"]), case["alpha"] * B, upper=upper,
                                             left=case["side"] == "L")
    if op == "potrf":
        A = _potrf_input(case, seed)
        F = torch.linalg.cholesky(A)
        if case["uplo"] == "L":
            return {"factor": torch.tril(F) + torch.triu(A, 1), "info": None}
        return {"factor": torch.triu(F.t()) + torch.tril(A, -1), "info": None}
    LU, _ = torch.linalg.lu_factor(_getrf_input(case, seed))
    return {"lu": LU, "ipiv": None, "info": None}
