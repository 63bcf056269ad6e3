// Off-diagonal update C = alpha*C - Aop*Bop on CUDA cores: the paper's gemm
// task (Section IV stage 2, b.low -= L.mid x.up; with many right-hand sides
// the gemv becomes a GEMM, Section V-A).  Used by the FP64 path (DFMA: the
// GB300 FP64 rate is set by the DFMA pipe, and tcgen05 has no f64 kind) and
// by the FP32 path (FFMA).
#include "common.cuh"
#include "gemm_digits.cuh"
#include "gemm_tile.cuh"

namespace gb {
namespace {

template <typename T, bool AM, bool LEFT>
__global__ void __launch_bounds__(GemmTile<T>::NT)
gemm_update_kernel(int64_t M, int64_t N, int64_t K, const T *__restrict__ A, int64_t lda,
                   const T *__restrict__ B, int64_t ldb, T *__restrict__ C, int64_t ldc, T alpha)
{
    __shared__ __align__(16) T smem[gemm_tile_smem<T>()];
    gemm_tile<T, AM, LEFT, LEFT>(smem, int64_t(blockIdx.y) * GemmTile<T>::BM, int64_t(blockIdx.x) * GemmTile<T>::BN,
                                 M, N, K, A, lda, B, ldb, C, ldc, alpha, 0);
}

// The trapezoid of C on and below its diagonal, Bop = the first N rows of
// Aop transposed: C(i, j) -= sum_k Aop(i, k) Aop(j, k).  AM: column-major
// operands, else both stored transposed.
template <typename T, bool AM>
__global__ void __launch_bounds__(GemmTile<T>::NT)
gemm_trapezoid_kernel(int64_t M, int64_t N, int64_t K, const T *__restrict__ P, int64_t ldp, T *__restrict__ C, int64_t ldc)
{
    constexpr int BM = GemmTile<T>::BM;
    __shared__ __align__(16) T smem[gemm_tile_smem<T>()];
    const int64_t m0 = int64_t(blockIdx.y) * BM, n0 = int64_t(blockIdx.x) * BM;
    if (n0 > m0 + BM - 1) return;
    gemm_tile<T, AM, !AM, AM>(smem, m0, n0, M, N, K, P, ldp, P, ldp, C, ldc, T(1), 1);
}

template <typename T, bool AM, bool LEFT>
int launch_cfg(int64_t M, int64_t N, int64_t K, const T *A, int64_t lda, const T *B,
               int64_t ldb, T *C, int64_t ldc, T alpha, cudaStream_t s)
{
    constexpr int BM = GemmTile<T>::BM, BN = GemmTile<T>::BN;
    constexpr int NT = GemmTile<T>::NT;
    int64_t gx = (N + BN - 1) / BN, gy = (M + BM - 1) / BM;
    if (gx > 0x7fffffff || gy > 65535) return GB_STATUS_CUDA_ERROR;
    LaunchScope ls(KK_GEMM_SIMT, s, 2.0 * M * N * K,
                   sizeof(T) * (double(M) * K + double(K) * N + 2.0 * M * N));
    gemm_update_kernel<T, AM, LEFT><<<dim3((unsigned)gx, (unsigned)gy), NT, 0, s>>>(
        M, N, K, A, lda, B, ldb, C, ldc, alpha);
    return check(cudaGetLastError());
}

}  // namespace

template <typename T>
int launch_gemm_update(const Canon<T> &c, int64_t ci0, int64_t M, int64_t ak0, int64_t K, T alpha)
{
    if (M <= 0 || c.ncols <= 0) return 0;
    if (K <= 0) {
        if (alpha == T(1)) return 0;
        K = 0;  // still scale C by alpha
    }
    const T *Ap = mv_ptr(c, ci0, ak0);
    const T *Bp = bv_ptr(c, ak0, 0);
    T *Cp = bv_ptr(c, ci0, 0);
    const bool am = !c.mt;
    if (am && c.left) return launch_cfg<T, true, true>(M, c.ncols, K, Ap, c.lda, Bp, c.ldb, Cp, c.ldb, alpha, c.stream);
    if (am && !c.left) return launch_cfg<T, true, false>(M, c.ncols, K, Ap, c.lda, Bp, c.ldb, Cp, c.ldb, alpha, c.stream);
    if (!am && c.left) return launch_cfg<T, false, true>(M, c.ncols, K, Ap, c.lda, Bp, c.ldb, Cp, c.ldb, alpha, c.stream);
    return launch_cfg<T, false, false>(M, c.ncols, K, Ap, c.lda, Bp, c.ldb, Cp, c.ldb, alpha, c.stream);
}

template <typename T>
int launch_gemm_trapezoid(bool am, int64_t M, int64_t N, int64_t K, const T *P, int64_t ldp, T *C, int64_t ldc, cudaStream_t s)
{
    if (M <= 0 || N <= 0 || K <= 0) return 0;
    constexpr int BM = GemmTile<T>::BM;
    const int64_t gx = (N + BM - 1) / BM, gy = (M + BM - 1) / BM;
    if (gx > 0x7fffffff || gy > 65535) return GB_STATUS_CUDA_ERROR;
    LaunchScope ls(KK_GEMM_SIMT, s, (2.0 * M - N) * N * K, sizeof(T) * (double(M) * K + (2.0 * M - N) * N));
    auto k = am ? gemm_trapezoid_kernel<T, true> : gemm_trapezoid_kernel<T, false>;
    k<<<dim3((unsigned)gx, (unsigned)gy), GemmTile<T>::NT, 0, s>>>(M, N, K, P, ldp, C, ldc);
    return check(cudaGetLastError());
}
template int launch_gemm_trapezoid<double>(bool, int64_t, int64_t, int64_t, const double *, int64_t, double *, int64_t, cudaStream_t);
template int launch_gemm_trapezoid<float>(bool, int64_t, int64_t, int64_t, const float *, int64_t, float *, int64_t, cudaStream_t);

template int launch_gemm_update<double>(const Canon<double> &, int64_t, int64_t, int64_t, int64_t, double);
template int launch_gemm_update<float>(const Canon<float> &, int64_t, int64_t, int64_t, int64_t, float);

// Column-major operands, by the kernels a solve would take for this size.
template <typename T>
static int gemm_update_colmajor(int64_t M, int64_t N, int64_t K, const T *A, int64_t lda, const T *B, int64_t ldb,
                                T *C, int64_t ldc, T alpha, cudaStream_t s)
{
    if (digit_gemm_wanted<T>(M, N, K, 0)) {
        DigitWorkspace w(s);
        char *ws = w.get(digit_gemm_bytes<T>(M, N, K, 0));
        if (ws) {
            const DigitGemm<T> g{M, N, K, A, lda, true, B, ldb, true, C, ldc, true, alpha, 0};
            return launch_digit_gemm<T>(g, ws, w.size(), s);
        }
    }
    return launch_cfg<T, true, true>(M, N, K, A, lda, B, ldb, C, ldc, alpha, s);
}

}  // namespace gb

// The gemm task on its own, column-major operands: C (M x N, ldc) =
// alpha*C - A (M x K, lda) * B (K x N, ldb), FP64 (dtype 0) or FP32 (1) --
// the kernel every plain solve uses for its off-diagonal updates.
extern "C" int gb_gemm_update(int dtype, int64_t M, int64_t N, int64_t K, const void *A, int64_t lda, const void *B,
                              int64_t ldb, void *C, int64_t ldc, double alpha, void *stream)
{
    if (dtype != 0 && dtype != 1) return -1;
    if (M < 0) return -2;
    if (N < 0) return -3;
    if (K < 0) return -4;
    if (A == nullptr && M * K > 0) return -5;
    if (lda < (M > 1 ? M : 1)) return -6;
    if (B == nullptr && K * N > 0) return -7;
    if (ldb < (K > 1 ? K : 1)) return -8;
    if (C == nullptr && M * N > 0) return -9;
    if (ldc < (M > 1 ? M : 1)) return -10;
    if (M == 0 || N == 0) return 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (dtype == 0)
        return gb::gemm_update_colmajor(M, N, K, static_cast<const double *>(A), lda, static_cast<const double *>(B),
                                        ldb, static_cast<double *>(C), ldc, alpha, s);
    return gb::gemm_update_colmajor(M, N, K, static_cast<const float *>(A), lda, static_cast<const float *>(B), ldb,
                                    static_cast<float *>(C), ldc, float(alpha), s);
}

namespace gb {

// ---- alpha == 0: Bv = 0 ------------------------------------------------------
namespace {
template <typename T>
__global__ void zero_kernel(T *B, int64_t ldb, int64_t rows, int64_t cols)
{
    // rows = contiguous extent, cols = strided extent
    int64_t total = rows * cols;
    for (int64_t idx = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; idx < total;
         idx += int64_t(gridDim.x) * blockDim.x) {
        int64_t r = idx % rows, c = idx / rows;
        B[r + c * ldb] = T(0);
    }
}
}  // namespace

template <typename T>
int launch_zero(const Canon<T> &c)
{
    // Bv column-major (Left): k rows contiguous, ncols strided; row-major
    // (Right): ncols contiguous, k strided.
    int64_t rows = c.left ? c.k : c.ncols, cols = c.left ? c.ncols : c.k;
    if (rows <= 0 || cols <= 0) return 0;
    int64_t total = rows * cols;
    int64_t blocks = (total + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    LaunchScope ls(KK_CONVERT, c.stream, 0.0, sizeof(T) * double(total));
    zero_kernel<T><<<(unsigned)blocks, 256, 0, c.stream>>>(c.B, c.ldb, rows, cols);
    return check(cudaGetLastError());
}

template int launch_zero<double>(const Canon<double> &);
template int launch_zero<float>(const Canon<float> &);

}  // namespace gb
