// One C tile of the CUDA-core gemm task (internal header): C = alpha*C - Aop*Bop
// by DFMA / FFMA on one CTA.  Used by the update kernel of gemm_simt.cu and by
// the digit gemm's last pass, for the tiles that the digits cannot represent.
//
// Design: CTA tile BM x BN, k-slices of BK staged in shared memory with a
// register double buffer (global loads of slice k+1 are in flight while
// slice k is multiplied).  Each thread owns a TM x TN micro-tile split in two
// halves (rows ty*TM/2.. and BM/2 + ty*TM/2..) so that its shared-memory
// reads are conflict-free 16-byte vectors.  Global loads run along whichever
// dimension is contiguous (A normal or transposed; B/C column-major for
// side Left, row-major for side Right), and are transposed on the way into
// shared memory.  alpha is applied to C in the epilogue (first touch).
#pragma once
#include "common.cuh"

namespace gb {
namespace {

template <typename T>
struct GemmTile;
template <>
struct GemmTile<float> {  // FFMA: 128x128 tile, 8x8 per thread, 256 threads
    static constexpr int BM = 128, BN = 128, BK = 8, TM = 8, TN = 8, NT = 256;
};
template <>
struct GemmTile<double> {  // DFMA: 64x64 tile, 4x4 per thread, 256 threads
    static constexpr int BM = 64, BN = 64, BK = 16, TM = 4, TN = 4, NT = 256;
};

// A quarter of that by a quarter of the threads, the same micro-tiles: for
// updates of which the large tiles leave SMs idle.
template <typename T>
struct GemmTileSmall {
    static constexpr int BM = GemmTile<T>::BM / 2, BN = GemmTile<T>::BN / 2, BK = GemmTile<T>::BK;
    static constexpr int TM = GemmTile<T>::TM, TN = GemmTile<T>::TN, NT = GemmTile<T>::NT / 4;
};

template <typename T, int W>
struct VecT;
template <>
struct VecT<float, 4> {
    using type = float4;
};
template <>
struct VecT<double, 2> {
    using type = double2;
};

// AM: A-operand contiguous along M (Mv(i,k) = A(i,k), i.e. !mt).
// BC: Bop contiguous along K, else along N.  CL: C contiguous along M, else
// along N.  tri: only the entries on and below the diagonal of C.  smem: gemm_tile_smem<T, G>() elements, 16-byte aligned.
// Every thread of the CTA takes part; shared memory is free on return only
// after a barrier.
template <typename T, class G = GemmTile<T>>
constexpr int gemm_tile_smem()
{
    return 2 * G::BK * (G::BM + G::BN + G::TM);
}

template <typename T, bool AM, bool BC, bool CL, class G = GemmTile<T>>
__device__ __forceinline__ void gemm_tile(T *smem, int64_t m0, int64_t n0, int64_t M, int64_t N, int64_t K,
                                          const T *__restrict__ A, int64_t lda, const T *__restrict__ B, int64_t ldb,
                                          T *__restrict__ C, int64_t ldc, T alpha, int tri)
{
    constexpr int BM = G::BM, BN = G::BN, BK = G::BK;
    constexpr int TM = G::TM, TN = G::TN;
    constexpr int NTX = BN / TN, NTY = BM / TM;
    constexpr int NT = NTX * NTY;
    constexpr int VW = TM / 2;  // vector width of one half micro-tile
    static_assert(TM == TN, "square micro-tile");
    static_assert(VW * sizeof(T) == 16, "16-byte shared vectors");
    constexpr int PAD = VW;     // keeps rows 16-byte aligned, spreads banks
    constexpr int LDA_S = BM + PAD, LDB_S = BN + PAD;
    constexpr int A_PER = BM * BK / NT, B_PER = BN * BK / NT;
    static_assert(A_PER * NT == BM * BK && B_PER * NT == BN * BK, "tile split");
    using V = typename VecT<T, VW>::type;

    T (*As)[BK * LDA_S] = reinterpret_cast<T (*)[BK * LDA_S]>(smem);
    T (*Bs)[BK * LDB_S] = reinterpret_cast<T (*)[BK * LDB_S]>(smem + 2 * BK * LDA_S);

    const int tid = threadIdx.x;
    const int tx = tid % NTX, ty = tid / NTX;

    T ra[A_PER], rb[B_PER];

    // Global -> registers for k-slice starting at kk.
    auto load_tiles = [&](int64_t kk) {
#pragma unroll
        for (int p = 0; p < A_PER; p++) {
            int idx = tid + p * NT;
            int i, k;
            if (AM) { i = idx % BM; k = idx / BM; }
            else    { k = idx % BK; i = idx / BK; }
            int64_t gi = m0 + i, gk = kk + k;
            T v = T(0);
            if (gi < M && gk < K) v = AM ? A[gi + gk * lda] : A[gk + gi * lda];
            ra[p] = v;
        }
#pragma unroll
        for (int p = 0; p < B_PER; p++) {
            int idx = tid + p * NT;
            int k, j;
            if (BC) { k = idx % BK; j = idx / BK; }
            else    { j = idx % BN; k = idx / BN; }
            int64_t gk = kk + k, gj = n0 + j;
            T v = T(0);
            if (gk < K && gj < N) v = BC ? B[gk + gj * ldb] : B[gj + gk * ldb];
            rb[p] = v;
        }
    };
    auto store_tiles = [&](int buf) {
#pragma unroll
        for (int p = 0; p < A_PER; p++) {
            int idx = tid + p * NT;
            int i, k;
            if (AM) { i = idx % BM; k = idx / BM; }
            else    { k = idx % BK; i = idx / BK; }
            As[buf][k * LDA_S + i] = ra[p];
        }
#pragma unroll
        for (int p = 0; p < B_PER; p++) {
            int idx = tid + p * NT;
            int k, j;
            if (BC) { k = idx % BK; j = idx / BK; }
            else    { j = idx % BN; k = idx / BN; }
            Bs[buf][k * LDB_S + j] = rb[p];
        }
    };

    T acc[TM][TN];
#pragma unroll
    for (int r = 0; r < TM; r++)
#pragma unroll
        for (int c = 0; c < TN; c++) acc[r][c] = T(0);

    const int64_t nk = (K + BK - 1) / BK;
    if (nk > 0) {
        load_tiles(0);
        store_tiles(0);
        __syncthreads();
    }
    for (int64_t kt = 0; kt < nk; kt++) {
        const int cur = int(kt & 1);
        if (kt + 1 < nk) load_tiles((kt + 1) * BK);
#pragma unroll
        for (int k = 0; k < BK; k++) {
            T a[TM], b[TN];
            V a0 = *reinterpret_cast<const V *>(&As[cur][k * LDA_S + ty * VW]);
            V a1 = *reinterpret_cast<const V *>(&As[cur][k * LDA_S + BM / 2 + ty * VW]);
            V b0 = *reinterpret_cast<const V *>(&Bs[cur][k * LDB_S + tx * VW]);
            V b1 = *reinterpret_cast<const V *>(&Bs[cur][k * LDB_S + BN / 2 + tx * VW]);
            const T *pa0 = reinterpret_cast<const T *>(&a0), *pa1 = reinterpret_cast<const T *>(&a1);
            const T *pb0 = reinterpret_cast<const T *>(&b0), *pb1 = reinterpret_cast<const T *>(&b1);
#pragma unroll
            for (int e = 0; e < VW; e++) {
                a[e] = pa0[e]; a[VW + e] = pa1[e];
                b[e] = pb0[e]; b[VW + e] = pb1[e];
            }
#pragma unroll
            for (int r = 0; r < TM; r++)
#pragma unroll
                for (int c = 0; c < TN; c++) acc[r][c] = fma(a[r], b[c], acc[r][c]);
        }
        if (kt + 1 < nk) {
            store_tiles(cur ^ 1);
            __syncthreads();
        }
    }

    // ---- epilogue: C = alpha*C - acc ----------------------------------------
#pragma unroll
    for (int r = 0; r < TM; r++) {
        int64_t gi = m0 + (r < VW ? ty * VW + r : BM / 2 + ty * VW + (r - VW));
        if (gi >= M) continue;
#pragma unroll
        for (int c = 0; c < TN; c++) {
            int64_t gj = n0 + (c < VW ? tx * VW + c : BN / 2 + tx * VW + (c - VW));
            if (gj >= N || (tri && gj > gi)) continue;
            T *p = CL ? &C[gi + gj * ldc] : &C[gj + gi * ldc];
            *p = (alpha == T(1)) ? (*p - acc[r][c]) : (alpha * *p - acc[r][c]);
        }
    }
}

}  // namespace
}  // namespace gb
