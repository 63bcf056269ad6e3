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


@pytest.mark.parametrize("dtype", [0, 1])
def test_results_do_not_depend_on_the_batch(dtype):
    """An instance alone (FP64: units one right-hand side wide), in a batch of 40
    and in one of 1200 (wider ones), which differ in the width of the units and in
    the teams: the same bits, and the padding of B untouched."""
    import torch
    from paper_2305_19917_gb300 import api
    td = (torch.float64, torch.float32)[dtype]
    r = np.random.default_rng(5)
    probs = []
    for k, cols in [(1, 1), (5, 3), (31, 2), (33, 8), (40, 9), (64, 16), (70, 37), (100, 5), (129, 17), (200, 4), (300, 33), (512, 20)]:
        side, uplo, trans, diag = (int(x) for x in r.integers(0, 2, 4))
        m, n = (k, cols) if side == 0 else (cols, k)
        A, B = inputs.make_problem(side, uplo, trans, diag, m, n, seed=k, poison=True)
        a = torch.full((k, k + 1), float("nan"), dtype=td, device="cuda").t()
        a[:k].copy_(torch.as_tensor(A).to(td))
        probs.append((dict(side=side, uplo=uplo, trans=trans, diag=diag, m=m, n=n, alpha=-1.5, A_ptr=a.data_ptr(), lda=k + 1), a, B))

    def solve(which):
        bufs, items = [], []
        for i in which:
            item, _, B = probs[i]
            b = torch.full((item["n"], item["m"] + 2), 7.0, dtype=td, device="cuda").t()
            b[: item["m"]].copy_(torch.as_tensor(B).to(td))
            bufs.append(b)
            items.append(dict(item, B_ptr=b.data_ptr(), ldb=item["m"] + 2))
        plan = api.BatchedPlan(dtype, items)
        info = plan.info()
        plan.run(torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        plan.close()
        for i, b in zip(which, bufs):
            assert bool(torch.all(b[probs[i][0]["m"]:] == 7.0))
        return [b.cpu().numpy() for b in bufs], info["units"]

    alone = [solve([i])[0][0] for i in range(len(probs))]
    few, _ = solve([i % len(probs) for i in range(40)])
    many, units = solve([i % len(probs) for i in range(1200)])
    for i, x in enumerate(few + many):
        assert np.array_equal(x, alone[(i if i < 40 else i - 40) % len(probs)]), i
    if dtype == 0:  # the widths did differ
        one = [solve([i])[1] for i in range(len(probs))]
        assert one[6] == 37 and units < 100 * sum(one) // 2
    for i, (item, a, B) in enumerate(probs):
        form = (item["side"], item["uplo"], item["trans"], item["diag"])
        k = item["m"] if form[0] == 0 else item["n"]
        A = np.nan_to_num(a[:k].double().cpu().numpy(), nan=0.0)
        Bt = torch.as_tensor(B).to(td).double().numpy()
        X = alone[i][: item["m"]].astype(np.float64)
        R = np.abs(oracle.dresidual(*form, -1.5, A, Bt, X))
        T = np.abs(oracle.op_dense(form[1], form[2], form[3], A, k))
        S = (T @ np.abs(X) if form[0] == 0 else np.abs(X) @ T) + 1.5 * np.abs(Bt)
        assert np.all(R <= (k + 4) * 2.0 ** (-53 if dtype == 0 else -24) * S), i
