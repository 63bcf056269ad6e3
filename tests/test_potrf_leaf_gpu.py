"""The Cholesky leaf (orders to 64) at the edges of its roles: rows on both
panel warps, the last slot of the packed triangle, pivots whose exponents take
the reciprocal root's ordinary and its rare path, and the first pivot that is
not positive.

Tolerance: |A - L L^T| <= (n + 8) u |L| |L^T| entry by entry (the bound for
Cholesky with n + 1 roundings per entry; root and scaling add a few units)."""
import numpy as np
import pytest

from paper_2305_19917_gb300 import inputs

pytestmark = pytest.mark.gpu

ORDERS = [1, 2, 3, 31, 32, 33, 63, 64]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


def _factor(uplo, A):
    from paper_2305_19917_gb300 import api
    import torch
    dev = api.to_device_colmajor(A, torch.float64 if A.dtype == np.float64 else torch.float32)
    info = api.potrf(uplo, dev)
    return dev.cpu().numpy(), info


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("uplo", [0, 1])
@pytest.mark.parametrize("n", ORDERS)
def test_graded(n, uplo, dtype):
    far = 480 if dtype == np.float64 else 55
    scale = np.ldexp(1.0, np.resize([0, -far, far, 1, -3], n))
    A = (inputs.make_spd(n, seed=n) * scale[:, None] * scale[None, :]).astype(dtype)
    A = np.tril(A) + np.tril(A, -1).T
    F, info = _factor(uplo, A)
    assert info == 0
    L = (np.tril(F) if uplo == 0 else np.triu(F).T).astype(np.longdouble)
    u = np.finfo(dtype).eps / 2
    assert np.all(np.abs(A.astype(np.longdouble) - L @ L.T) <= (n + 8) * u * (np.abs(L) @ np.abs(L).T))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("bad", [0, 1, 2, 31, 32, 33, 62, 63])
@pytest.mark.parametrize("pivot", [0.0, -1.0, np.nan])
def test_first_bad_pivot(bad, pivot, dtype):
    A = np.diag(np.arange(1.0, 65.0)).astype(dtype)
    A[bad, bad] = pivot
    if bad < 63:
        A[63, 63] = -2.0  # a later one does not replace it
    F, info = _factor(0, A)
    assert info == bad + 1
    assert np.allclose(np.diag(F)[:bad], np.sqrt(np.arange(1.0, bad + 1)), rtol=2 * np.finfo(dtype).eps, atol=0)
