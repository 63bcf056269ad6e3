"""How an update by digit products is cut into pieces and shares of K
(csrc/digit_plan.cuh), on the CPU: the header is plain C++, compiled here with a
loop over sizes.  Every share of every piece holds some of K, the shares cover
it once, no piece needs more work space than was asked for, and K is not split
further than the work space was sized for."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "digit_plan.cuh"
using namespace gb::digits;
static long long bad = 0, pieces = 0, split_pieces = 0;
template <int P>
void check(int64_t M, int64_t N, int64_t K, int tri)
{
    const Piece pc = plan_piece<P>(M, N, K, tri);
    int64_t area = 0;
    for_pieces(pc, M, N, K, tri, [&](int64_t i, int64_t j, int64_t k, int64_t m, int64_t n, int64_t kk, int split) {
        pieces++;
        split_pieces += split > 1;
        area += m * n * kk;
        const int kt = int((kk + BK - 1) / BK);
        int at = 0;
        bool ok = split >= 1 && split <= pc.split && i + m <= M && j + n <= N && k + kk <= K;
        for (int sp = 0; sp < split; sp++) {
            int k0, k1;
            share_range(kt, split, sp, k0, k1);
            ok = ok && k0 == at && k1 > k0;
            at = k1;
        }
        ok = ok && at == kt && piece_bytes<P>(m, n, kk, tri, split) <= pc.bytes;
        if (!ok && bad++ < 5) printf("P %d: %ld x %ld x %ld tri %d: piece K %ld split %d\n", P, M, N, K, tri, kk, split);
        return 0;
    });
    if (area != M * N * K && bad++ < 5) printf("not covered: %ld x %ld x %ld\n", M, N, K);
}
int main()
{
    const int64_t mn[] = {1, 64, 70, 128, 129, 300, 512, 777, 1500, 4096, 9000, 40000};
    const int64_t ks[] = {64, 65, 127, 128, 129, 500, 1000, 4095, 4096, 4097, 4224, 5000, 8192, 8256, 12288, 16384, 16385, 16448,
                          16896, 17000, 20000, 32768, 33000, 49153, 100000};
    for (int64_t M : mn)
        for (int64_t N : mn)
            for (int64_t K : ks)
                for (int tri = 0; tri < 2; tri++) {
                    if (tri && N > M) continue;
                    check<3>(M, N, K, tri);
                    check<4>(M, N, K, tri);
                    check<7>(M, N, K, tri);
                    check<8>(M, N, K, tri);
                }
    printf("%lld pieces, %lld with K split, %lld bad\n", pieces, split_pieces, bad);
    return bad != 0 || split_pieces == 0;
}
"""


def test_no_share_of_k_is_empty(tmp_path):
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2305_19917_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
