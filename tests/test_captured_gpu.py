"""Plain solves while their stream is being captured: no work space for digits
can be had then, so every update runs on the CUDA cores, in graphs that hold no
memory of the library and can be launched again on new contents.  Around the
lines at which the schedule changes (FP64 1216 right-hand sides, 512 rows) and
with explicit plans, against the CPU oracle (tolerance of the uncaptured solves,
10 k u normwise backward) and, with lookahead on and off, bit for bit."""
import numpy as np
import pytest

from paper_2305_19917_gb300 import inputs
from tests.helpers import U32, U64, bwd_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


def _captured(form, alpha, A, B, td, plan=None):
    """X of two launches of the captured solve, B restored before each."""
    import torch
    from paper_2305_19917_gb300 import api
    a, b = api.to_device_colmajor(A, td), api.to_device_colmajor(B, td)
    x = torch.empty_strided(b.shape, b.stride(), dtype=td, device="cuda")
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        x.copy_(b)
        api.trsm(*form, alpha, a, x, plan=plan, stream=s)
    out = []
    for _ in range(2):
        x.fill_(7.0)
        graph.replay()
        torch.cuda.synchronize()
        out.append(x.double().cpu().numpy())
    assert np.array_equal(out[0], out[1])
    return out[0]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k,cols", [(65, 1217), (300, 1216), (512, 1300), (513, 1217), (1100, 40), (1500, 1250)])
@pytest.mark.parametrize("form", [(0, 0, 0, 0), (1, 0, 0, 0), (0, 0, 1, 1)])
def test_captured_solve(form, k, cols, dtype):
    import torch
    m, n = (k, cols) if form[0] == 0 else (cols, k)
    A, B = inputs.make_problem(*form, m, n, seed=k)
    td, u = (torch.float64, U64) if dtype == "f64" else (torch.float32, U32)
    A, B = (np.asarray(torch.as_tensor(z).to(td).double()) for z in (A, B))
    X = _captured(form, 1.5, A, B, td)
    assert bwd_err(*form, 1.5, A, B, X) <= 10 * k * u


@pytest.mark.parametrize("plan", [dict(driver=0, nb=64, depth=0), dict(driver=1, nb=128, depth=2), dict(driver=2, nb=512, depth=0),
                                  dict(driver=0, nb=16, depth=0)])
def test_captured_plan_and_lookahead(plan):
    """Explicit plans, wide enough for 64-row blocks; the lookahead splits the
    CUDA-core updates between two streams and changes no bit."""
    import torch
    from paper_2305_19917_gb300 import api
    form, k, cols = (0, 0, 0, 0), 1200, 1300
    A, B = inputs.make_problem(*form, k, cols, seed=9)
    old = api.gb_set_lookahead(1)
    try:
        on = _captured(form, 1.5, A, B, torch.float64, plan)
        api.gb_set_lookahead(0)
        off = _captured(form, 1.5, A, B, torch.float64, plan)
    finally:
        api.gb_set_lookahead(old)
    assert np.array_equal(on, off)
    assert bwd_err(*form, 1.5, A, B, on) <= 10 * k * U64


def test_release_while_capturing():
    """With no work space of the mixed path kept there is nothing to free:
    the call returns 0 and leaves the capture as it is."""
    import torch
    from paper_2305_19917_gb300 import api
    A, B = inputs.make_problem(0, 0, 0, 0, 600, 100, seed=2)
    a, b = api.to_device_colmajor(A, torch.float64), api.to_device_colmajor(B, torch.float64)
    api.trsm(0, 0, 0, 0, 1.0, a, b)  # the digits' pool exists
    assert api.gb_mixed_workspace_release(torch.cuda.current_stream().cuda_stream) == 0
    x = torch.zeros(8, device="cuda")
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        x.add_(1.0)
        assert api.gb_mixed_workspace_release(s.cuda_stream) == 0
    graph.replay()
    torch.cuda.synchronize()
    assert bool(torch.all(x == 1.0))
