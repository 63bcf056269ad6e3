"""The workloads that this library's speed is measured on.

A case names one call of the public API (``paper_2305_19917_gb300.api``) with
its sizes and options: a plain FP64 / FP32 solve, a mixed-precision solve, a
batch of uneven solves, or a Cholesky factorisation.  ``listed`` gives the
fixed ones, ``draw`` further ones of the same ranges.

Inputs are synthetic, with the distributions of ``inputs.py``: the entries of
A off its diagonal U(-1, 1) / k (k = order of A), its diagonal U[1, 2), B
N(0, 1); Cholesky: symmetric with such entries, hence diagonally dominant.
The triangle that a solve does not reference holds numbers too, as it does
when A is one half of a factorisation.  All matrices are column-major.

A solve overwrites its right-hand side, so a pass copies the kept B (or A)
into the buffer that the call works on and then makes the call.
"""
import math
import random

import numpy as np
import torch

from paper_2305_19917_gb300 import api

LEFT, RIGHT = 0, 1
LOWER, UPPER = 0, 1
NOTRANS, TRANS = 0, 1
NONUNIT, UNIT = 0, 1


def _case(kind, dtype, side, uplo, trans, diag, m, n, alpha, name=None):
    c = dict(kind=kind, dtype=dtype, side=side, uplo=uplo, trans=trans, diag=diag, m=m, n=n, alpha=alpha)
    if name:
        c["name"] = name
    return c


def _batch(dtype, count, m_max, n_max, shape_seed, name=None):
    c = dict(kind="batched", dtype=dtype, count=count, m_max=m_max, n_max=n_max, shape_seed=shape_seed)
    if name:
        c["name"] = name
    return c


def _chol(dtype, uplo, n, name=None):
    c = dict(kind="potrf", dtype=dtype, uplo=uplo, n=n)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call of the benchmark's configurations: one diagonal
        # block's worth of work, where launches and latency are the time
        _case("plain", "f64", LEFT, LOWER, NOTRANS, NONUNIT, 256, 64, 1.0, "trsm_f64_256x64"),
        # an ordinary odd-sized solve from the right with a transposed factor
        # (whitening by a Cholesky factor, a block of a factorisation)
        _case("plain", "f64", RIGHT, UPPER, TRANS, NONUNIT, 300, 777, 1.5, "trsm_f64_right_300x777"),
        # a large factor and a few right-hand sides (back substitution)
        _case("plain", "f64", LEFT, UPPER, NOTRANS, NONUNIT, 4096, 256, 1.0, "trsm_f64_4096x256"),
        # the benchmark's plain solve at scale
        _case("plain", "f64", LEFT, LOWER, NOTRANS, NONUNIT, 8192, 8192, 1.5, "trsm_f64_8192"),
        # single precision, ordinary and odd, unit diagonal (an LU's L)
        _case("plain", "f32", LEFT, LOWER, TRANS, UNIT, 1000, 500, 1.0, "trsm_f32_1000x500"),
        # single precision at scale, from the right
        _case("plain", "f32", RIGHT, UPPER, NOTRANS, NONUNIT, 8192, 8192, 1.5, "trsm_f32_right_8192"),
        # mixed precision where its fixed costs count, odd sizes
        _case("bf16", "f64", RIGHT, LOWER, NOTRANS, NONUNIT, 700, 1500, 1.0, "mixed_bf16_right_700x1500"),
        # the benchmark's headline solve
        _case("bf16", "f64", LEFT, LOWER, NOTRANS, NONUNIT, 16384, 16384, 1.5, "mixed_bf16_16384"),
        # the benchmark's tall mixed solve, FP8 updates
        _case("fp8", "f64", LEFT, LOWER, NOTRANS, NONUNIT, 32768, 4096, 1.5, "mixed_fp8_32768x4096"),
        # the benchmark's batch of uneven solves (one plan, run many times)
        _batch("f64", 4096, 512, 256, 0, "batched_f64_4096"),
        _batch("f32", 4096, 512, 256, 0, "batched_f32_4096"),
        # Cholesky factorisation on the solver
        _chol("f64", LOWER, 8192, "potrf_f64_8192"),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi], odd ones among them."""
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["plain", "plain", "plain", "plain", "bf16", "bf16", "fp8", "batched", "batched", "potrf"])
    if kind == "batched":
        return _batch(rng.choice(["f64", "f32"]), _log_int(rng, 256, 4096), rng.randint(128, 512),
                      rng.randint(64, 256), rng.randrange(1 << 30))
    if kind == "potrf":
        return _chol("f64", rng.randint(0, 1), _log_int(rng, 512, 8192))
    side = rng.randint(0, 1)
    uplo, trans, diag = rng.randint(0, 1), rng.randint(0, 1), rng.randint(0, 1)
    alpha = rng.choice([1.0, 1.5])
    if kind == "plain":
        dtype = rng.choice(["f64", "f32"])
        k, cols = _log_int(rng, 256, 8192), _log_int(rng, 64, 8192)
    elif kind == "bf16":
        dtype = "f64"
        k, cols = _log_int(rng, 700, 16384), _log_int(rng, 700, 16384)
    else:
        dtype = "f64"
        k, cols = _log_int(rng, 700, 32768), _log_int(rng, 700, 4096)
    m, n = (k, cols) if side == LEFT else (cols, k)
    return _case(kind, dtype, side, uplo, trans, diag, m, n, alpha)


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _fill_triangle(a, k, g):
    """U(-1, 1) / k with the diagonal U[1, 2), in place on a k x k tensor."""
    a.uniform_(-1.0, 1.0, generator=g).div_(k)
    a.diagonal().uniform_(1.0, 2.0, generator=g)


def _order(case):
    return (case["m"], case["n"]) if case["side"] == LEFT else (case["n"], case["m"])


def _solve_inputs(case, seed):
    g = _generator(seed)
    dt = _dtype(case)
    k, _ = _order(case)
    A = torch.empty((k, k), dtype=dt, device="cuda").t()
    _fill_triangle(A, k, g)
    B = torch.empty((case["n"], case["m"]), dtype=dt, device="cuda").t()
    B.normal_(generator=g)
    return A, B


def _spd_input(case, seed):
    n = case["n"]
    A = torch.empty((n, n), dtype=_dtype(case), device="cuda").t()
    A.uniform_(-1.0, 1.0, generator=_generator(seed)).div_(n)
    A = (A + A.t()).mul_(0.5)  # symmetric, so its layout is column-major either way
    A.diagonal().uniform_(1.0, 2.0, generator=_generator(seed + 1))
    return A


def _batch_shapes(case):
    """(side, uplo, m, n) of every instance: the order m log-uniform, n uniform."""
    r = random.Random(case["shape_seed"])
    out = []
    for _ in range(case["count"]):
        m, n = _log_int(r, 16, case["m_max"]), r.randint(1, case["n_max"])
        out.append((r.randint(0, 1), r.randint(0, 1), m, n))
    return out


def _batch_inputs(case, seed):
    """One buffer with every A, one with every B, and the instances' places in them."""
    shapes = _batch_shapes(case)
    orders = [m if side == LEFT else n for side, _, m, n in shapes]
    a_off = np.concatenate([[0], np.cumsum([k * k for k in orders])])
    b_off = np.concatenate([[0], np.cumsum([m * n for _, _, m, n in shapes])])
    g = _generator(seed)
    a = torch.empty(int(a_off[-1]), dtype=_dtype(case), device="cuda").uniform_(-1.0, 1.0, generator=g)
    b = torch.empty(int(b_off[-1]), dtype=_dtype(case), device="cuda").normal_(generator=g)
    k_dev = torch.tensor(orders, device="cuda")
    a.div_(torch.repeat_interleave(k_dev, k_dev * k_dev).to(a.dtype))
    d_off = np.concatenate([o + (k + 1) * np.arange(k) for o, k in zip(a_off[:-1], orders)])
    d_idx = torch.from_numpy(d_off).cuda()
    a[d_idx] = torch.empty(len(d_off), dtype=a.dtype, device="cuda").uniform_(1.0, 2.0, generator=g)
    places = [(side, uplo, m, n, k, int(ao), int(bo))
              for (side, uplo, m, n), k, ao, bo in zip(shapes, orders, a_off, b_off)]
    return a, b, places


def prepare(case, seed):
    """What a program has before the call: its matrices and, for a batch, the plan."""
    if case["kind"] == "batched":
        a, b, places = _batch_inputs(case, seed)
        x = torch.empty_like(b)
        es = a.element_size()
        items = [dict(side=side, uplo=uplo, trans=NOTRANS, diag=NONUNIT, m=m, n=n, alpha=1.0,
                      A_ptr=a.data_ptr() + ao * es, lda=k, B_ptr=x.data_ptr() + bo * es, ldb=m)
                 for side, uplo, m, n, k, ao, bo in places]
        plan = api.BatchedPlan(0 if case["dtype"] == "f64" else 1, items,
                               stream=torch.cuda.current_stream().cuda_stream)
        return dict(case=case, A=a, B=b, X=x, plan=plan)
    if case["kind"] == "potrf":
        A = _spd_input(case, seed)
        return dict(case=case, A=A, X=torch.empty_strided(A.shape, A.stride(), dtype=A.dtype, device="cuda"))
    A, B = _solve_inputs(case, seed)
    return dict(case=case, A=A, B=B, X=torch.empty_strided(B.shape, B.stride(), dtype=B.dtype, device="cuda"))


def run(state):
    """One pass: the call's own buffer filled, then the call."""
    c, A, X = state["case"], state["A"], state["X"]
    if c["kind"] == "potrf":
        X.copy_(A)
        info = api.potrf(c["uplo"], X)
        return X, info
    X.copy_(state["B"])
    if c["kind"] == "batched":
        state["plan"].run(torch.cuda.current_stream().cuda_stream)
        return X
    if c["kind"] == "plain":
        return api.trsm(c["side"], c["uplo"], c["trans"], c["diag"], c["alpha"], A, X)
    prec = api.PREC_BF16 if c["kind"] == "bf16" else api.PREC_FP8
    status, _, _ = api.trsm_mixed(c["side"], c["uplo"], c["trans"], c["diag"], c["alpha"], A, X, tol=1e-11, prec=prec)
    return X, status


def work(case):
    """Bytes that have to move and multiply-add flops of one pass."""
    es = 8 if case["dtype"] == "f64" else 4
    if case["kind"] == "batched":
        bytes_, flops = 0, 0.0
        for side, _, m, n in _batch_shapes(case):
            k, cols = (m, n) if side == LEFT else (n, m)
            bytes_ += es * (k * (k + 1) // 2 + 2 * m * n)
            flops += float(k) * k * cols
        return {"bytes": bytes_, "flops": flops}
    if case["kind"] == "potrf":
        n = case["n"]
        return {"bytes": es * n * (n + 1), "flops": n ** 3 / 3.0}
    k, cols = _order(case)
    return {"bytes": es * (k * (k + 1) // 2 + 2 * k * cols), "flops": float(k) * k * cols}


def _solve64(side, uplo, trans, diag, alpha, A, B):
    """alpha op(A)^-1 B or alpha B op(A)^-1 in FP64."""
    A, B = A.double(), B.double()
    op = A.t() if trans == TRANS else A
    upper = (uplo == UPPER) != (trans == TRANS)
    return torch.linalg.solve_triangular(op, alpha * B, upper=upper, left=side == LEFT, unitriangular=diag == UNIT)


def exact(case, seed):
    if case["kind"] == "batched":
        a, b, places = _batch_inputs(case, seed)
        out = torch.empty(b.numel(), dtype=torch.float64, device="cuda")
        for side, uplo, m, n, k, ao, bo in places:
            X = _solve64(side, uplo, NOTRANS, NONUNIT, 1.0, a[ao:ao + k * k].view(k, k).t(),
                         b[bo:bo + m * n].view(n, m).t())
            out[bo:bo + m * n].view(n, m).copy_(X.t())
        return out
    if case["kind"] == "potrf":
        A = _spd_input(case, seed).double()
        if case["uplo"] == LOWER:
            return torch.linalg.cholesky(A).tril_() + A.triu(1), 0
        return torch.linalg.cholesky(A).t().triu() + A.tril(-1), 0
    A, B = _solve_inputs(case, seed)
    X = _solve64(case["side"], case["uplo"], case["trans"], case["diag"], case["alpha"], A, B)
    return X if case["kind"] == "plain" else (X, 0)
