"""FP64 solves with more right-hand sides than the panels take (2433 on): the
64-row diagonal kernel in CTAs of 32 and of 64 right-hand sides, ragged orders
(rows past the block's end are solved to zero) and both directions.

Tolerance: the substitution's backward error, |A X - alpha B| <= (k + 4) u |A| |X|
entry by entry (k products, alpha, the diagonal's reciprocal and its product)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


@pytest.mark.parametrize("cols", [2433, 4864, 4865])
@pytest.mark.parametrize("k", [1, 16, 17, 33, 63, 64])
@pytest.mark.parametrize("side,uplo,trans", [(0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0), (1, 1, 0), (1, 0, 1)])
def test_substitution_bound(side, uplo, trans, k, cols):
    import torch
    from paper_2305_19917_gb300 import api
    r = np.random.default_rng(k * cols + side + 2 * uplo + 4 * trans)
    A = r.uniform(-1, 1, (k, k))
    A = (np.tril(A) if uplo == 0 else np.triu(A))
    A[np.arange(k), np.arange(k)] = r.uniform(1, 2, k)
    B = r.standard_normal((k, cols) if side == 0 else (cols, k))
    dA, dB = (api.to_device_colmajor(x, torch.float64) for x in (A, B))
    api.trsm(side, uplo, trans, 0, 1.5, dA, dB)
    X = dB.cpu().numpy()
    op = A.T if trans else A
    mul = (lambda m, x: m @ x) if side == 0 else (lambda m, x: x @ m)
    L = np.longdouble
    res = np.abs(mul(op.astype(L), X.astype(L)) - L(1.5) * B)
    assert np.all(res <= (k + 4) * 2.0 ** -53 * mul(np.abs(op), np.abs(X)))
