"""The batched solve at the edges of its teams (orders solved by one, two or
four warps), of its 32-row blocks and of its column chunks, in every form, with
padded leading dimensions, against the CPU oracle.

Tolerance: substitution's backward error bound per entry, |alpha B - op(A) X|
<= (k + 4) u (|op(A)| |X| + |alpha B|) componentwise (each of the k terms one
rounding, the product with the inverse diagonal and alpha three more)."""
import numpy as np
import pytest

import oracle
from paper_2305_19917_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("tile", [1, 2])
def test_team_edges(dtype, tile):
    import torch
    from paper_2305_19917_gb300 import api
    td, nt, u = [(torch.float64, np.float64, 2.0 ** -53), (torch.float32, np.float32, 2.0 ** -24)][dtype]
    items, keep = [], []
    for i, k in enumerate([1, 2, 31, 32, 33, 64, 65, 127, 128, 129, 255, 256, 257, 300, 511, 512]):
        for j, cols in enumerate([1, 16, 17, 33]):
            side, uplo, trans, diag = (i + j) & 1, (i >> 1 ^ j) & 1, (j >> 1) & 1, (i + j) % 3 == 0
            m, n = (k, cols) if side == 0 else (cols, k)
            A, B = inputs.make_problem(side, uplo, trans, int(diag), m, n, seed=100 * i + j, poison=True)
            A, B = A.astype(nt), B.astype(nt)
            pad = j  # odd and even leading dimensions
            Ad = torch.full((k, k + pad), float("nan"), dtype=td, device="cuda").t()
            Bd = torch.full((n, m + pad), 7.0, dtype=td, device="cuda").t()
            Ad[:k].copy_(torch.as_tensor(A))
            Bd[:m].copy_(torch.as_tensor(B))
            alpha = (1.0, -0.5)[j & 1]
            keep.append((Ad, Bd, A, B, (side, uplo, trans, int(diag)), m, n, alpha))
            items.append(dict(side=side, uplo=uplo, trans=trans, diag=int(diag), m=m, n=n, alpha=alpha,
                              A_ptr=Ad.data_ptr(), lda=k + pad, B_ptr=Bd.data_ptr(), ldb=m + pad))
    plan = api.BatchedPlan(dtype, items, tile=tile)
    plan.run(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    plan.close()
    for Ad, Bd, A, B, form, m, n, alpha in keep:
        assert bool(torch.all(Bd[m:] == 7.0))
        X = Bd[:m].double().cpu().numpy()
        A, B = np.nan_to_num(A.astype(np.float64), nan=0.0), B.astype(np.float64)
        k = m if form[0] == 0 else n
        R = np.abs(oracle.dresidual(*form, alpha, A, B, X))
        T = np.abs(oracle.op_dense(form[1], form[2], form[3], A, k))
        S = (T @ np.abs(X) if form[0] == 0 else np.abs(X) @ T) + abs(alpha) * np.abs(B)
        assert np.all(R <= (k + 4) * u * S), (form, m, n)
