"""FP8 updates in 256-column tiles, chosen from 152 such tiles on: a width whose
last tile is half empty (1152 columns: the 8192-row solve's largest update has
32 x 5 tiles) and one just below the line (128-column tiles).

Tolerance: the refined solution's, 1e-10 of the FP64 solve; a wrong tile of the
low-precision solve leaves corrections of order one instead of 1e-3 (two FP8
mantissa steps of 2^-4 over sums of mostly cancelling products)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [1100, 1152, 900])
def test_wide_tiles(n):
    import torch
    from paper_2305_19917_gb300 import api
    m = 8192
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    A = torch.empty((m, m), dtype=torch.float64, device="cuda").uniform_(-1, 1, generator=g).div_(m).t()
    A.diagonal().uniform_(1, 2, generator=g)
    B = torch.empty((n, m), dtype=torch.float64, device="cuda").normal_(generator=g).t()
    X, Y = B.t().clone().t(), B.t().clone().t()
    api.trsm(0, 0, 0, 0, 1.5, A, X)
    st, it, est = api.trsm_mixed(0, 0, 0, 0, 1.5, A, Y, tol=1e-11, prec=api.PREC_FP8)
    hist = api.gb_mixed_history()
    assert st == 0 and it <= 4, (st, it, hist)
    assert hist[0][0] <= 1e-3, hist
    err = torch.linalg.vector_norm(Y - X, dim=0) / torch.linalg.vector_norm(X, dim=0)
    assert float(err.max()) <= 1e-10
