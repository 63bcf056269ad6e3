"""The diagonal-block solve of many rows in one launch (the plain solves'
path for few right-hand sides), at the edges of its blocks (32 rows, 512 or
1024 rows), of its column counts per CTA, and at diagonals and couplings
whose scaled rows would leave the exponent range, against the CPU oracle.

Tolerance: substitution's backward error bound per entry, |alpha B - op(A) X|
<= (k + 4) u (|op(A)| |X| + |alpha B|) componentwise (each of the k terms one
rounding, the row's scaling by its inverse diagonal three more)."""
import numpy as np
import pytest

import oracle
from paper_2305_19917_gb300 import inputs
from tests.helpers import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


def _check(form, m, n, dtype, A, B, alpha=1.5, ldpad=0):
    side, uplo, trans, diag = form
    nt = np.float64 if dtype == "f64" else np.float32
    A, B = A.astype(nt).astype(np.float64), B.astype(nt).astype(np.float64)
    X, pad_ok = gpu_solve(side, uplo, trans, diag, alpha, A, B, dtype=dtype, ldpad=ldpad)
    assert pad_ok
    k = m if side == 0 else n
    R = np.abs(oracle.dresidual(side, uplo, trans, diag, alpha, A, B, X))
    T = np.abs(oracle.op_dense(uplo, trans, diag, A, k))
    S = (T @ np.abs(X) if side == 0 else np.abs(X) @ T) + abs(alpha) * np.abs(B)
    u = 2.0 ** (-53 if dtype == "f64" else -24)
    assert np.all(R <= (k + 4) * u * S)


FORMS = [(0, 0, 0, 0), (0, 1, 0, 0), (1, 0, 0, 0), (1, 1, 1, 1)]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k,cols", [(1, 1), (33, 2), (96, 305), (511, 3), (512, 5), (513, 1), (130, 609), (64, 1217),
                                    (95, 2433), (1023, 2), (1024, 1), (1025, 2)])
def test_edges(k, cols, dtype):
    for i, form in enumerate(FORMS):
        m, n = (k, cols) if form[0] == 0 else (cols, k)
        A, B = inputs.make_problem(*form, m, n, seed=k + i)
        _check(form, m, n, dtype, A, B, ldpad=i % 2)


@pytest.mark.parametrize("form", FORMS[:3])
def test_extreme_rows(form):
    """Rows whose entries divided by the diagonal overflow or underflow, in
    blocks beside ordinary ones: the solve multiplies by the inverse instead."""
    side, uplo, trans, diag = form
    k, cols = 130, 9
    low = uplo == side  # solved as a left-side lower (else upper) problem, or its transpose
    A, B = inputs.make_problem(0, 0 if low else 1, 0, 0, k, cols, seed=4)
    s = np.tril(np.ones((k, k)), -1) if low else np.triu(np.ones((k, k)), 1)
    A[40, :] = np.where(s[40, :] > 0, A[40, :] * 2.0 ** -700, A[40, :])
    A[40, 40] = 2.0 ** -700
    B[40, :] *= 2.0 ** -700
    A[100, :] = np.where(s[100, :] > 0, A[100, :] * 2.0 ** 350, A[100, :])
    A[:, 60] = np.where(s[:, 60] > 0, A[:, 60] * 2.0 ** -420, A[:, 60])
    if side == 1:
        A, B = np.asfortranarray(A.T), np.asfortranarray(B.T)
    _check(form, *B.shape, "f64", A, B)


@pytest.mark.parametrize("cols", [3, 310, 610, 1220])
@pytest.mark.parametrize("where", ["B", "diagonal", "triangle", "below"])
def test_nan_of_any_payload(where, cols):
    """FP64: a NaN in B reaches its own column from its row on, one in A every
    column from its row on, and nothing else, whatever its payload; the word
    that stands for an X not yet known is one of them."""
    k = 100
    A, B = inputs.make_problem(0, 0, 0, 0, k, cols, seed=7)
    want, _ = gpu_solve(0, 0, 0, 0, 1.5, A, B)
    at = {"B": (37, 1), "diagonal": (37, 37), "triangle": (37, 33), "below": (37, 3)}[where]
    for word in (0xFFF8DEADBEEF5A5A, 0x7FF8DEADBEEF5A5A, 0xFFF0DEADBEEF5A5A, 0x7FF8000000000000):
        An, Bn = A.copy(), B.copy()
        (Bn if where == "B" else An)[at] = np.array([word], dtype=np.uint64).view(np.float64)[0]
        X, _ = gpu_solve(0, 0, 0, 0, 1.5, An, Bn)
        hit = (slice(37, None), slice(1, 2) if where == "B" else slice(None))
        assert np.all(np.isnan(X[hit]))
        X[hit] = want[hit]
        # (a row with a NaN keeps its block from being scaled: rounding only)
        assert np.all(np.isfinite(X)) and np.all(np.abs(X - want) <= 1e-13 * np.abs(want).max())


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k,cols", [(1, 700), (8, 1), (15, 2500), (16, 33), (17, 608), (17, 609), (32, 609), (32, 65), (33, 1216),
                                    (33, 1217), (48, 2000), (64, 1300), (64, 5000)])
def test_small_orders(k, cols, dtype):
    """Orders of at most 64: the diagonal kernel and the panel kernel on both
    sides of the lines between them."""
    for i, form in enumerate(FORMS):
        m, n = (k, cols) if form[0] == 0 else (cols, k)
        A, B = inputs.make_problem(*form, m, n, seed=k + cols + i)
        _check(form, m, n, dtype, A, B, ldpad=i % 2)
