"""The leaf kernel's panel widths (32, 64 and 128 columns, by the width of the
problem: lines at 4864 and 9728 padded columns) at both sides of the lines, with
one leaf and a part of a second.

Tolerance: the refined solution's, 1e-10 of the FP64 solve, and the first
correction's size: a BF16 solve with two-term block inverses is within 1e-3."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


@pytest.mark.parametrize("m", [300, 1200])
@pytest.mark.parametrize("n", [100, 4864, 4865, 9728, 9729])
def test_widths(m, n):
    import torch
    from paper_2305_19917_gb300 import api
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n)
    A = torch.empty((m, m), dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g).div_(m).t()
    A.diagonal().uniform_(1, 2, generator=g)
    B = torch.empty((n, m), dtype=torch.float64, device="cuda").normal_(generator=g).t()
    X, Y = B.t().clone().t(), B.t().clone().t()
    api.trsm(0, 0, 0, 0, 1.5, A, X)
    st, it, est = api.trsm_mixed(0, 0, 0, 0, 1.5, A, Y, tol=1e-11)
    hist = api.gb_mixed_history()
    assert st == 0 and it <= 3 and hist[0][0] <= 1e-3, (st, it, hist)
    err = torch.linalg.vector_norm(Y - X, dim=0) / torch.linalg.vector_norm(X, dim=0)
    assert float(err.max()) <= 1e-10
