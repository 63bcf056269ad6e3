"""The off-diagonal update by digit products on the tensor cores
(gb_gemm_update's path from K = 64 in FP64, from K = 128 in FP32) against
numpy in extended precision: tile and chunk edges, the split of K, both
factors' layouts (through the solve's other tests) and the inputs that the
digits must leave to the CUDA cores.

Tolerance, from the format: a factor is rounded at 2^-(8P+1) of its row's
(column's) scale, at most twice the largest entry (P = 7 digits FP64, 3
FP32), the pairs left out add (P - 1) 2^(14-8(P+2)) of the scales' product per
term at most, and the tiles taken by digits hold at least K/4 terms of 2^-10
of the largest product each: |error| <= 2^-41 (FP64), 2^-13 (FP32) of
sum |a||x| in the worst case.  Dense random factors stay far below it: the
factors' roundings are independent, about 2^-(8P) of sqrt(K) products, checked
as 2^-50 and 2^-21 of the factors' norms (CUDA-core sums round K times)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

WORST = {0: 2.0 ** -41, 1: 2.0 ** -13}
NORM = {0: 2.0 ** -50, 1: 2.0 ** -21}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2305_19917_gb300 import build
    build.build()


def _update(dtype, A, B, C, alpha):
    import torch
    from paper_2305_19917_gb300 import api
    td = torch.float64 if dtype == 0 else torch.float32
    dev = [api.to_device_colmajor(x, td) for x in (A, B, C)]
    (M, K), N = A.shape, B.shape[1]
    st = api.gb_gemm_update(dtype, M, N, K, dev[0].data_ptr(), M, dev[1].data_ptr(), K, dev[2].data_ptr(), M, alpha,
                            torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    return dev[2].cpu().numpy()


def _factors(dtype, M, N, K, seed):
    nt = np.float64 if dtype == 0 else np.float32
    r = np.random.default_rng(seed)
    return (r.uniform(-1, 1, (M, K)).astype(nt), r.standard_normal((K, N)).astype(nt),
            r.standard_normal((M, N)).astype(nt))


SIZES = [(1, 1, 128), (128, 128, 128), (129, 127, 191), (64, 300, 256), (127, 1, 257), (33, 65, 1000), (300, 260, 2100)]


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("M,N,K", SIZES + [(100, 77, 64), (70, 50, 17000)])
def test_dense_factors(dtype, M, N, K):
    A, B, C = _factors(dtype, M, N, K, seed=M + N + K)
    A *= np.exp2(np.arange(M) % 40 - 20).astype(A.dtype)[:, None]  # every row its own scale
    got = _update(dtype, A, B, C, 0.5)
    L = np.longdouble
    prod = A.astype(L) @ B.astype(L)
    bound = np.abs(A).astype(L) @ np.abs(B).astype(L)
    u = L(2.0) ** (-53 if dtype == 0 else -24)
    err = np.abs(got - (L(0.5) * C - prod))
    assert np.all(err <= WORST[dtype] * bound + 2 * u * np.abs(got))
    # sqrt(K) products: per row, |a_i| |B| in the 2-norms, and the old C
    rows = np.sqrt(np.sum(A.astype(L) ** 2, axis=1)) * np.sqrt(np.sum(B.astype(L) ** 2))
    rows += np.sqrt(np.sum(C.astype(L) ** 2, axis=1))
    assert np.all(np.sqrt(np.sum(err ** 2, axis=1)) <= NORM[dtype] * rows * max(1.0, K / 4096))


def _graded(A, B):
    A[:, ::2] *= 2.0 ** -30   # large entries of A meet ...
    B[1::2, :] *= 2.0 ** -30  # ... small ones of B: sum |a||x| is 2^-30 of the largest product


def _sparse(A, B):
    A[:, : A.shape[1] * 7 // 8] = 0


def _infinite(A, B):
    B[3, 5] = np.inf
    A[7, 11] = np.nan


def _huge(A, B):
    e = 500 if A.dtype == np.float64 else 60
    A *= A.dtype.type(2.0) ** e
    B *= A.dtype.type(2.0) ** -e


def _subnormal(A, B):
    A[9, :] = np.finfo(A.dtype).smallest_subnormal * 5


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("change", [_graded, _sparse, _infinite, _huge, _subnormal])
def test_what_digits_cannot_hold(dtype, change):
    """These tiles are computed by the CUDA cores: componentwise K u."""
    M, N, K = 200, 300, 520
    A, B, C = _factors(dtype, M, N, K, seed=5)
    change(A, B)
    C[:] = 0
    got = _update(dtype, A, B, C, 1.0)
    L = np.longdouble
    with np.errstate(all="ignore"):
        want = -(A.astype(L) @ B.astype(L))
        bound = np.abs(A).astype(L) @ np.abs(B).astype(L)
    ok = np.isfinite(want.astype(np.float64)) & np.isfinite(bound.astype(np.float64))
    # an infinity reaches its column (or row) and nothing else
    assert np.array_equal(np.isfinite(got), ok)
    u = 2.0 ** (-53 if dtype == 0 else -24)
    tiny = np.finfo(A.dtype).smallest_subnormal
    assert np.all(np.abs(got - want)[ok] <= K * (u * bound[ok] + tiny))


@pytest.mark.parametrize("M,N,K", [(1700, 1500, 64), (1700, 1500, 128), (1700, 1500, 129), (1700, 1500, 300)])
def test_schedules_by_share_of_k(M, N, K):
    """Enough tiles that K is not split: up to 128 of it the schedule with one
    accumulator per weight, from 129 the one for 256, with a last chunk of 44;
    entries of one sign, so that the sums come near their bounds."""
    A, B, C = _factors(0, M, N, K, seed=K)
    A, B = 1 - np.abs(A) / 64, 1 - np.abs(B) / 64
    got = _update(0, A, B, C, 1.0)
    L = np.longdouble
    rows, cols = np.r_[0:3, 126:131, M - 2:M], np.r_[0:2, 127:129, N - 2:N]
    want = C[np.ix_(rows, cols)].astype(L) - A[rows].astype(L) @ B[:, cols].astype(L)
    norms = np.linalg.norm(A[rows], axis=1)[:, None] * np.linalg.norm(B[:, cols], axis=0)[None, :]
    u = 2.0 ** -53
    assert np.all(np.abs(got[np.ix_(rows, cols)] - want) <= NORM[0] * norms + 2 * u * np.abs(want))


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("M,N,K", [(70, 50, 17000), (512, 64, 17000), (40, 40, 16385)])
def test_ragged_last_piece_of_k(M, N, K, dtype):
    """K beyond one piece on few tiles: the last piece is split by its own K.
    No wait runs out: those last two seconds, these updates a few hundred
    microseconds."""
    import torch
    from paper_2305_19917_gb300 import api
    A, B, C = _factors(dtype, M, N, K, seed=K)
    dev = [api.to_device_colmajor(x, torch.float64 if dtype == 0 else torch.float32) for x in (A, B, C)]
    t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    torch.cuda.synchronize()
    for _ in range(2):  # the first call may load the kernels
        t0.record()
        st = api.gb_gemm_update(dtype, M, N, K, dev[0].data_ptr(), M, dev[1].data_ptr(), K, dev[2].data_ptr(), M, 1.0,
                                torch.cuda.current_stream().cuda_stream)
        t1.record()
        torch.cuda.synchronize()
        assert st == 0
    assert t0.elapsed_time(t1) < 200.0
    L = np.longdouble
    want = C[:16].astype(L) - 2 * (A[:16].astype(L) @ B.astype(L))
    norms = np.linalg.norm(A[:16].astype(L), axis=1)[:, None] * np.linalg.norm(B.astype(L), axis=0)[None, :]
    u = 2.0 ** (-53 if dtype == 0 else -24)
    err = np.abs(dev[2].cpu().numpy()[:16] - want)
    assert np.all(err <= 2 * NORM[dtype] * norms * K / 4096 + 4 * u * (np.abs(want) + np.abs(C[:16])))


def _edge(kind, n, M, N, K, r):
    """Factors of which n products have both entries 2^-5 to 2^-4 of the scales;
    the other entries there meet ones 2^-12 smaller ("count": one entry per row is
    near the scale), or they are as large as the scale and meet ones of 2^-30
    ("big")."""
    def small(*size):
        return r.choice([-1.0, 1.0], size) * r.uniform(1 / 16, 1 / 8, size)

    def large(*size):
        return r.choice([-1.0, 1.0], size) * r.uniform(1, 1.99, size)
    A, B = small(M, K), small(K, N)
    rest = (K - n) // 2
    if kind == "count":
        A[:, :rest] *= 2.0 ** -12
        B[K - rest:] *= 2.0 ** -12
        A[:, 0] = B[-1, :] = 1.9
    else:
        A[:, :rest], A[:, K - rest:] = large(M, rest), A[:, K - rest:] * 2.0 ** -30
        B[K - rest:], B[:rest] = large(rest, N), B[:rest] * 2.0 ** -30
    return A, B


@pytest.mark.parametrize("dtype,K", [(0, 64), (0, 200), (0, 1000), (0, 2500), (0, 9000), (1, 128), (1, 500), (1, 2500)])
@pytest.mark.parametrize("kind", ["count", "big", "normal", "uniform"])
def test_error_below_the_cuda_core_sum(kind, dtype, K):
    """The claim itself, on both sides of the rule's edge: the root mean square
    error over a tile's entries is at most that of the CUDA-core sum of the same
    factors (the path taken while a stream is being captured; the same bits where
    the rule lists the tile).  Normal and uniform entries are the digits', and so
    are factors of which half of the products have a counted pair and no other
    entry is large."""
    import torch
    from paper_2305_19917_gb300 import api
    M = N = 130  # (FP32 takes digits from 16384 entries on)
    r = np.random.default_rng(K)
    nt = np.float64 if dtype == 0 else np.float32
    td = torch.float64 if dtype == 0 else torch.float32
    L = np.longdouble
    i, j = np.r_[0:15, 120:130], np.r_[0:10, 115:130]
    taken = []
    for part in ((64, 16, 8, 4, 2) if kind in ("count", "big") else (1,)):
        if kind in ("count", "big"):
            A, B = _edge(kind, max(K // part, 2), M, N, K, r)
        else:
            A = r.standard_normal((M, K)) if kind == "normal" else r.uniform(-1, 1, (M, K))
            B = r.standard_normal((K, N))
        A, B = A.astype(nt), B.astype(nt)
        a, b = api.to_device_colmajor(A, td), api.to_device_colmajor(B, td)
        got = _update(dtype, A, B, np.zeros((M, N), nt), 1.0)
        c = torch.zeros(N, M, dtype=td, device="cuda").t()
        s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            st = api.gb_gemm_update(dtype, M, N, K, a.data_ptr(), M, b.data_ptr(), K, c.data_ptr(), M, 1.0, s.cuda_stream)
        assert st == 0
        graph.replay()
        torch.cuda.synchronize()
        cuda = c.cpu().numpy()
        want = -(A[i].astype(L) @ B[:, j].astype(L))
        scale = np.abs(A[i]).astype(L) @ np.abs(B[:, j]).astype(L)
        rms = [float(np.sqrt(np.mean(((x[np.ix_(i, j)] - want) / scale) ** 2))) for x in (got, cuda)]
        assert rms[0] <= rms[1], (part, rms)
        taken.append(not np.array_equal(got, cuda))
    assert taken[-1] or kind == "big", taken


def test_weights_of_the_int64_sums():
    """FP64: the sums' weight W follows the factors' 2-norms, from 50 for the
    longest rows of large entries up to 62; one value too high would overflow.
    Tolerance as for dense factors."""
    seen = set()
    for K in (64, 129, 300, 1000, 4000, 9000, 16384):
        for f in (1.0, 0.5, 0.25, 0.125, 0.0625):
            r = np.random.default_rng(int(K / f))
            A, B = r.choice([-1.0, 1.0], (9, K)), r.choice([-1.0, 1.0], (K, 7))
            A, B = A * r.uniform(1.9, 1.999, A.shape), B * r.uniform(1.9, 1.999, B.shape)
            A[:, 1:] *= f
            B[1:] *= f
            n2 = [int(np.max(np.sum((np.round(np.abs(X) * 64) + 1) ** 2, axis=ax))) for X, ax in ((A, 1), (B, 0))]
            seen.add(min(62, int(78.95 - 0.5 * np.log2(float(n2[0]) * n2[1]))))
            got = _update(0, A, B, np.zeros((9, 7)), 1.0)
            L = np.longdouble
            want = -(A.astype(L) @ B.astype(L))
            norms = np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(B, axis=0)[None, :]
            assert np.all(np.abs(got - want) <= NORM[0] * norms + 2.0 ** -52 * np.abs(want)), (K, f)
    assert seen == set(range(50, 63)), seen


@pytest.mark.parametrize("dtype,K", [(0, 64), (0, 128), (0, 256), (0, 700), (1, 128), (1, 256), (1, 700)])
def test_digits_at_their_bounds(dtype, K):
    """All digits of all entries 127 (as far as the type's bits go) or all -128
    but the first, every product of one sign: the accumulators reach their
    bounds.  Tolerance: the last bits of T and the result's rounding."""
    n = 6 if dtype == 0 else 3
    up = sum(127 * 256.0 ** -(p + 1) for p in range(n))
    dn = 127 * 256.0 ** -1 - sum(128 * 256.0 ** -(p + 1) for p in range(1, n))
    nt = np.float64 if dtype == 0 else np.float32
    for a, x in ((up, up), (up, dn), (dn, dn)):
        A, B = np.full((130, K), 2 * a, nt), np.full((K, 130), 2 * x, nt)
        assert A[0, 0] == 2 * a and B[0, 0] == 2 * x
        got = _update(dtype, A, B, np.zeros((130, 130), nt), 1.0)
        want = -np.longdouble(2 * a) * np.longdouble(2 * x) * K
        u = 2.0 ** (-53 if dtype == 0 else -24)
        assert np.all(np.abs(got - want) <= 1.01 * u * abs(want))


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("M,N,K", [(1, 1, 512), (70, 300, 128), (130, 260, 512), (1000, 1100, 128), (1300, 2200, 130)])
def test_all_tiles_listed(M, N, K, dtype):
    """Half of A's columns zero, the other half meeting zeros of B: every tile is
    left to the CUDA cores, in parts of a quarter of their tiles where there are
    few and in whole ones, more parts than CTAs among them.  Componentwise K u,
    as for the CUDA-core sum."""
    A, B, C = _factors(dtype, M, N, K, seed=M + K)
    A[:, ::2] = 0
    B[1::4] = 0
    got = _update(dtype, A, B, C, 0.5)
    rows, cols = (np.unique(np.minimum(np.r_[0:5, n // 2, max(n - 70, 0):n], n - 1)) for n in (M, N))
    i = np.ix_(rows, cols)
    L = np.longdouble
    want = L(0.5) * C[i] - A[rows].astype(L) @ B[:, cols].astype(L)
    bound = np.abs(A[rows]).astype(L) @ np.abs(B[:, cols]).astype(L) + np.abs(C[i])
    u = 2.0 ** (-53 if dtype == 0 else -24)
    assert np.all(np.abs(got[i] - want) <= K * u * bound)
    assert np.all(np.isfinite(got))
    # and all of C: a probe against a product by another path
    full = 0.5 * C.astype(np.float64) - A.astype(np.float64) @ B.astype(np.float64)
    assert np.allclose(got, full, rtol=0, atol=(1e-11 if dtype == 0 else 1e-3))
