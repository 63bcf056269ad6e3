"""The lookahead where it does split updates (those on the CUDA cores: FP64 below
K = 64, FP32 below 128, and every one of a captured solve): more launches with it
than without, and the same bits."""
import numpy as np
import pytest

import oracle
from paper_2305_19917_gb300 import inputs
from tests.helpers import fwd_err, gpu_solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


def _launches(f):
    from paper_2305_19917_gb300 import api
    n = api.gb_kernel_launches()
    out = f()
    return out, api.gb_kernel_launches() - n


@pytest.mark.parametrize("side,uplo,trans", [(0, 0, 0), (0, 1, 0), (1, 0, 1), (1, 1, 1)])
@pytest.mark.parametrize("dtype,plan", [("f64", dict(driver=0, nb=16, depth=0)), ("f64", dict(driver=0, nb=32, depth=0)),
                                        ("f64", dict(driver=1, nb=32, depth=1)), ("f32", dict(driver=0, nb=64, depth=0))])
def test_split_updates_are_bitwise_neutral(side, uplo, trans, dtype, plan):
    from paper_2305_19917_gb300 import api
    m, n = (1100, 77) if side == 0 else (77, 1100)
    A, B = inputs.make_problem(side, uplo, trans, 0, m, n, seed=17 + side + 2 * uplo)
    got = []
    old = api.gb_set_lookahead(1)
    try:
        for on in (1, 0):
            api.gb_set_lookahead(on)
            got.append(_launches(lambda: gpu_solve(side, uplo, trans, 0, 1.5, A, B, dtype=dtype, plan=plan)[0]))
    finally:
        api.gb_set_lookahead(old)
    (x_on, l_on), (x_off, l_off) = got
    assert l_on > l_off
    assert np.array_equal(x_on, x_off)
    Xo = oracle.dtrsm(side, uplo, trans, 0, 1.5, A, B)
    assert fwd_err(x_on, Xo) <= (1e-12 if dtype == "f64" else 1e-4)


def test_digit_updates_are_not_split():
    """A solve whose updates all go to the tensor cores launches the same
    kernels with the lookahead on and off."""
    from paper_2305_19917_gb300 import api
    A, B = inputs.make_problem(0, 0, 0, 0, 2304, 70, seed=3)
    old = api.gb_set_lookahead(1)
    try:
        on = _launches(lambda: gpu_solve(0, 0, 0, 0, 1.0, A, B)[0])
        api.gb_set_lookahead(0)
        off = _launches(lambda: gpu_solve(0, 0, 0, 0, 1.0, A, B)[0])
    finally:
        api.gb_set_lookahead(old)
    assert on[1] == off[1]
    assert np.array_equal(on[0], off[0])
