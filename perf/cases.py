"""Performance cases: dense solves as a user of this library runs them.

Each case is one pass through the public entry points of
``paper_2108_09337_gb300.cf``: factor a matrix and solve with the factors (FP64),
a mixed-precision refined solve, or a batch of small factorizations or solves.
Sizes, precisions, shifts and numbers of right-hand sides follow the library's
benchmark and test configurations; inputs are made on the GPU from the seed.
"""
import math

import torch

from paper_2108_09337_gb300 import cf


def listed():
    return [
        # A small system solved in FP64: what a simulation step calls many times; latency and launches count.
        {"name": "lu_f64_300", "kind": "lu64", "n": 300, "nrhs": 1},
        # The plain FP64 configuration at N = 2048 (uniform entries, the row pivoting of the paper), and its Cholesky.
        {"name": "lu_f64_2048", "kind": "lu64", "n": 2048, "nrhs": 1},
        {"name": "chol_f64_2048", "kind": "chol64", "n": 2048, "nrhs": 1},
        # FP64 at the smallest of the paper-like sizes, and a ragged Cholesky near it with a few right-hand sides.
        {"name": "lu_f64_8192", "kind": "lu64", "n": 8192, "nrhs": 1},
        {"name": "chol_f64_7777", "kind": "chol64", "n": 7777, "nrhs": 3},
        # The headline mixed solves: N = 32768, 16 (LU) and 8 (Cholesky) right-hand sides, FP16 updates.
        {"name": "lu_f16_32768", "kind": "lu_mixed", "n": 32768, "nrhs": 16, "prec": "f16", "shifted": True},
        {"name": "chol_f16_32768", "kind": "chol_mixed", "n": 32768, "nrhs": 8, "prec": "f16"},
        # A ragged mid-size mixed LU with BF16 updates.
        {"name": "lu_bf16_10001", "kind": "lu_mixed", "n": 10001, "nrhs": 5, "prec": "bf16", "shifted": True},
        # An unshifted uniform matrix: worse conditioned, split-BF16 factors, the refinement works harder.
        {"name": "lu_bf16x3_4096_unshifted", "kind": "lu_mixed", "n": 4096, "nrhs": 16, "prec": "bf16x3", "shifted": False},
        # Cholesky with FP8 updates (8 right-hand sides), at a size whose inputs are quick to make.
        {"name": "chol_fp8_16384", "kind": "chol_mixed", "n": 16384, "nrhs": 8, "prec": "fp8"},
        # Uneven batches, n = 16..512, half LU and half Cholesky: FP64 factors in place, and FP32 factors refined to FP64.
        {"name": "batch_f64_2000", "kind": "batch_factor", "count": 2000, "lo": 16, "hi": 512},
        {"name": "batch_mixed_2000", "kind": "batch_mixed", "count": 2000, "lo": 16, "hi": 512},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["lu64", "chol64", "lu_mixed", "chol_mixed", "batch_factor", "batch_mixed"])
    if kind in ("lu64", "chol64"):
        return {"kind": kind, "n": _log_int(rng, 100, 8192), "nrhs": rng.choice([1, 2, 3, 8, 16])}
    if kind == "lu_mixed":
        shifted = rng.random() < 0.75
        prec = rng.choice(["f16", "bf16", "bf16x3"]) if shifted else "bf16x3"
        return {"kind": kind, "n": _log_int(rng, 512, 32768 if shifted else 4096), "nrhs": rng.randint(1, 16),
                "prec": prec, "shifted": shifted}
    if kind == "chol_mixed":
        return {"kind": kind, "n": _log_int(rng, 512, 32768), "nrhs": rng.randint(1, 16),
                "prec": rng.choice(["f16", "bf16", "bf16x3", "fp8"])}
    return {"kind": kind, "count": _log_int(rng, 60, 2000), "lo": 16, "hi": _log_int(rng, 40, 512)}


# ---------------------------------------------------------------------------------------------------------------------
# Inputs


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + stream)
    return g


def _uniform(n, seed, shift):
    """U[-1, 1] entries, plus a diagonal shift; column-major."""
    a = torch.rand((n, n), generator=_generator(seed, 0), device="cuda", dtype=torch.float64).mul_(2.0).sub_(1.0)
    if shift:
        a.diagonal().add_(shift)
    return a.t()


def _gram(n, seed, alpha):
    """G G^T / n + alpha I with G ~ N(0, 1), formed in FP32 and held in FP64, exactly symmetric."""
    g = torch.randn((n, n), generator=_generator(seed, 0), device="cuda", dtype=torch.float32)
    low = (g @ g.t()).div_(n).tril_()
    del g
    a = low.to(torch.float64)
    a += low.tril(-1).t()
    a.diagonal().add_(alpha)
    return a.t()


def _normal(n, nrhs, seed):
    return torch.randn((nrhs, n), generator=_generator(seed, 1), device="cuda", dtype=torch.float64).t()


def _matrix(case, seed):
    n, kind = case["n"], case["kind"]
    if kind == "lu64":
        return _uniform(n, seed, 0.0)
    if kind == "chol64":
        return _gram(n, seed, 1.0)
    if kind == "lu_mixed":
        return _uniform(n, seed, 2.0 * math.sqrt(n) if case["shifted"] else 0.0)
    return _gram(n, seed, 0.04)       # condition number about 1e2


def _sizes(case):
    """The batch's sizes belong to the workload, not to its values: the same for every seed."""
    g = torch.Generator()
    g.manual_seed(7)
    return torch.randint(case["lo"], case["hi"] + 1, (case["count"],), generator=g).tolist()


def _batch(case, seed):
    """An uneven batch: odd matrices U[-1, 1] (LU), even ones G G^T / n + I (Cholesky)."""
    sizes = _sizes(case)
    batch = cf.Batch(sizes, kinds=[1 - i % 2 for i in range(len(sizes))])
    batch.data.copy_(torch.rand(batch.data.shape, generator=_generator(seed, 0), device="cuda", dtype=torch.float64))
    batch.data.mul_(2.0).sub_(1.0)
    for i in range(0, len(sizes), 2):
        m = batch.matrix(i)
        s = (m @ m.t()).mul_(3.0 / sizes[i])      # variance of U[-1, 1] is 1/3
        m.copy_(s.tril() + s.tril(-1).t())
        m.diagonal().add_(1.0)
    return batch


def _batch_x(batch, seed):
    return torch.randn(batch.vec_total, generator=_generator(seed, 1), device="cuda", dtype=torch.float64)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch_factor", "batch_mixed"):
        batch = _batch(case, seed)
        if kind == "batch_factor":
            plan = cf.BatchedPlan(batch, kind="factor")
            return {"case": case, "plan": plan, "source": batch.data.clone()}
        plan = cf.BatchedPlan(batch, kind="mixed")
        x = _batch_x(batch, seed)
        for n, o, i in zip(batch.sizes, batch.vec_offsets, range(len(batch.sizes))):
            torch.mv(batch.matrix(i), x[o:o + n], out=plan.B[o:o + n])
        return {"case": case, "plan": plan}
    a = _matrix(case, seed)
    b = cf.to_fortran(a @ _normal(case["n"], case["nrhs"], seed))
    if kind in ("lu64", "chol64"):
        return {"case": case, "a": a, "b": b, "w": cf.to_fortran(a).clone(), "x": b.clone()}
    return {"case": case, "a": a, "b": b}


# ---------------------------------------------------------------------------------------------------------------------
# One pass


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lu64":
        w, x = state["w"], state["x"]
        w.copy_(state["a"])
        x.copy_(state["b"])
        ipiv, info = cf.getrf(w)
        cf.getrs(w, ipiv, x)
        return {"lu": w, "ipiv": ipiv, "info": info, "x": x}
    if kind == "chol64":
        w, x = state["w"], state["x"]
        w.copy_(state["a"])
        x.copy_(state["b"])
        info = cf.potrf(w)
        cf.potrs(w, x)
        return {"l": w, "info": info, "x": x}
    if kind == "lu_mixed":
        x, info, _, _ = cf.gesv_mixed(state["a"], state["b"], prec=case["prec"])
        return {"x": x, "info": info}
    if kind == "chol_mixed":
        x, info, _, _ = cf.posv_mixed(state["a"], state["b"], prec=case["prec"])
        return {"x": x, "info": info}
    plan = state["plan"]
    if kind == "batch_factor":
        plan.batch.data.copy_(state["source"])
        plan.run()
        return {"factors": plan.batch.data, "ipiv": plan.ipiv, "info": plan.info}
    plan.run()
    return {"x": plan.X, "info": plan.info}


def work(case):
    """One pass: every input read once, every output written once; the factorization's and the solve's operations."""
    if case["kind"].startswith("batch"):
        sizes = _sizes(case)
        n2 = float(sum(n * n for n in sizes))
        flops = sum((1 + i % 2) * n ** 3 / 3.0 for i, n in enumerate(sizes))
        if case["kind"] == "batch_factor":
            return {"bytes": 16.0 * n2, "flops": flops}
        return {"bytes": 8.0 * n2 + 16.0 * sum(sizes), "flops": flops + 2.0 * n2}
    n, nrhs = float(case["n"]), case["nrhs"]
    third = 2.0 if case["kind"].startswith("lu") else 1.0
    flops = third * n ** 3 / 3.0 + 2.0 * n * n * nrhs
    if case["kind"] in ("lu64", "chol64"):
        return {"bytes": 16.0 * n * n + 16.0 * n * nrhs, "flops": flops}
    return {"bytes": 8.0 * n * n + 16.0 * n * nrhs, "flops": flops}


# ---------------------------------------------------------------------------------------------------------------------
# The same in 64 bits without this library


def exact(case, seed):
    kind = case["kind"]
    if kind in ("lu_mixed", "chol_mixed"):
        return {"x": _normal(case["n"], case["nrhs"], seed), "info": None}
    if kind == "lu64":       # the factors depend on the pivoting rule, the solution does not
        return {"lu": None, "ipiv": None, "info": None, "x": _normal(case["n"], case["nrhs"], seed)}
    if kind == "chol64":
        a = _matrix(case, seed)
        return {"l": torch.linalg.cholesky(a) + a.triu(1), "info": None, "x": _normal(case["n"], case["nrhs"], seed)}
    batch = _batch(case, seed)
    if kind == "batch_mixed":
        return {"x": _batch_x(batch, seed), "info": None}
    data = batch.data.cpu()
    for i, n in enumerate(batch.sizes):     # partial pivoting: one block holds all candidate rows
        m = data[batch.offsets[i]:batch.offsets[i] + n * n].view(n, n).t()
        m.copy_(torch.linalg.lu_factor(m)[0] if i % 2 else torch.linalg.cholesky(m) + m.triu(1))
    return {"factors": data, "ipiv": None, "info": None}
