// How a digit gemm is cut into launches and shares of K (internal header;
// gemm_digits.cu).  Integer arithmetic only, no CUDA: a test on the CPU
// compiles it and walks every share of many sizes.
#pragma once
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define GB_HD __host__ __device__ __forceinline__
#else
#define GB_HD inline
#endif

namespace gb {
namespace digits {

constexpr int BM = 128, BK = 64;  // tile of C, K of one load

// Largest piece of one launch sequence: the digits of both factors and the
// sums stay within the work space's cap, K within 16384, with eight digits (FP64)
// 8192, where the rounding of the sums' last bits still leaves room for normally
// distributed factors (gemm_digits.cu, "Accuracy").
constexpr size_t kWsCap = size_t(2) << 30;
template <int P>
constexpr int64_t kMaxK = P == 8 ? 8192 : 16384;

inline int64_t up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Tiles of C: all, or (tri) the trapezoid on and below its diagonal.
inline int64_t digit_tiles(int64_t nMt, int64_t nNt, int tri)
{
    return tri ? nNt * (nNt + 1) / 2 + (nMt - nNt) * nNt : nMt * nNt;
}

// Share sp of `split` of kt tiles of K: tiles [k0, k1).
GB_HD void share_range(int kt, int split, int sp, int &k0, int &k1)
{
    const int per = (kt + split - 1) / split;
    k0 = sp * per < kt ? sp * per : kt;
    k1 = k0 + per < kt ? k0 + per : kt;
}

// K is split over CTAs, down to 64 of it each, while the tiles alone leave SMs
// idle: 9 tiles of K = 512 on 72 CTAs instead of 9.  Beyond K = 2048 a share is at
// least a whole chunk of 256: every share rounds the sums' last bits once.  At most
// `most` shares, and none of them empty.
inline int pick_split(int64_t ntiles, int64_t K, int64_t most = 152)
{
    const int64_t kt = (K + BK - 1) / BK;
    int64_t s = 152 / ntiles;
    const int64_t least = K > 2048 ? 4 : 1;
    if (s > kt / least) s = kt / least;
    if (s > most) s = most;
    if (s < 2) return 1;
    const int64_t per = (kt + s - 1) / s;
    return int((kt + per - 1) / per);
}

struct Piece {
    int64_t mc, nc, kc;  // extents of one piece (mc, nc multiples of 128 unless whole)
    int split;           // of a whole piece
    size_t bytes;
};

// P: digits of a factor.
template <int P>
size_t piece_bytes(int64_t M, int64_t N, int64_t K, int tri, int split)
{
    const size_t mp = size_t(up(M, BM)), np = size_t(up(N, BM)), kp = size_t(up(K, BK));
    const size_t nt = size_t(digit_tiles(int64_t(mp / BM), int64_t(np / BM), tri));
    size_t b = 256 + 2 * P * mp * kp + (tri ? 0 : 2 * P * np * kp) + (split > 1 ? nt * BM * BM * 8 : 0);
    b += 4 * 4 * (mp + np) + 4 * (3 * nt + 3) + 12 * 256;
    return b;
}

template <int P>
Piece plan_piece(int64_t M, int64_t N, int64_t K, int tri)
{
    Piece p;
    p.kc = K < kMaxK<P> ? K : kMaxK<P>;
    p.mc = M;
    p.nc = N;
    // halve the longer of the two extents until the piece fits (of a triangle, K)
    while (!tri && piece_bytes<P>(p.mc, p.nc, p.kc, 0, 1) > kWsCap && (p.mc > 1024 || p.nc > 1024)) {
        if (p.nc >= p.mc) p.nc = up((p.nc + 1) / 2, BM);
        else p.mc = up((p.mc + 1) / 2, BM);
    }
    while (tri && piece_bytes<P>(M, N, p.kc, 1, 1) > kWsCap && p.kc > 1024) p.kc = up((p.kc + 1) / 2, BK);
    p.split = pick_split(digit_tiles(up(p.mc, BM) / BM, up(p.nc, BM) / BM, tri), p.kc);
    p.bytes = piece_bytes<P>(p.mc, p.nc, p.kc, tri, p.split);
    return p;
}

// Calls f(i, j, k, m, n, kk, split) for every piece: rows i.., columns j.., K k..,
// its extents, and the shares of its K.  The split is the piece's own: a ragged
// last piece of K with the split of the whole ones would have empty shares.
template <class F>
int for_pieces(const Piece &pc, int64_t M, int64_t N, int64_t K, int tri, F f)
{
    for (int64_t i = 0; i < M; i += pc.mc)
        for (int64_t j = 0; j < N; j += pc.nc)
            for (int64_t k = 0; k < K; k += pc.kc) {
                const int64_t m = M - i < pc.mc ? M - i : pc.mc, n = N - j < pc.nc ? N - j : pc.nc;
                const int64_t kk = K - k < pc.kc ? K - k : pc.kc;
                const int64_t nt = digit_tiles(up(m, BM) / BM, up(n, BM) / BM, tri);
                const int st = f(i, j, k, m, n, kk, pick_split(nt, kk, pc.split));
                if (st) return st;
            }
    return 0;
}

}  // namespace digits
}  // namespace gb
