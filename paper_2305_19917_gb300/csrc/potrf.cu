// Cholesky factorisation on this triangular solver: the use the paper names
// for its TS machinery (Section VIII, future work), built with the same
// recursive computation model (Section V-A) as the solve, on panels that
// reach down to the last row:
//
//     panel of columns [c0, c1), rows [c0, n):
//         left half                                              (recursion)
//         right half -= L(rows, left) L(right rows, left)^T       (gemm task:
//                       its trapezoid on and below the diagonal)
//         right half                                             (recursion)
//
// down to leaves of at most 64 columns: the diagonal block factorised by one
// CTA in shared memory, the rows below it solved against it (TS task: the
// library's own TRSM, side Right, transposed).  So every column block meets
// one TS task, on all its rows at once: splitting the matrix in 2 x 2 blocks
// instead, with a TRSM of every order, ran 448 of them at n = 8192 instead of
// 127.  n = 8192 FP64: 128 -> 28.5 ms by the panels and the tasks' digit gemms, 23.7
// with the leaf below; n = 16384 87 ms (1.34 s before the digit gemms).  The upper form (A = U^T U) is the same with everything stored
// transposed.  Only the named triangle of A is read and written.
//
// A non-positive (or NaN) pivot stops the leaf that meets it; the leaf
// records info = (global column + 1) in a device word (the first failure
// wins, leaves run in order) and every later leaf returns without work.  As
// with LAPACK, the contents of A from that column on are then undefined.
#include <algorithm>
#include <cmath>
#include "common.cuh"
#include "driver.cuh"
#include "gemm_digits.cuh"
#include "mixed.cuh"

extern "C" int gb_dtrsm(int side, int uplo, int trans, int diag, int64_t m, int64_t n, double alpha,
                        const double *A, int64_t lda, double *B, int64_t ldb, void *stream);
extern "C" int gb_strsm(int side, int uplo, int trans, int diag, int64_t m, int64_t n, float alpha,
                        const float *A, int64_t lda, float *B, int64_t ldb, void *stream);

namespace gb {
namespace {

constexpr int kLeafNB = 64;
constexpr int kLeafThreads = 256;

// Exponent field and its largest value (tests on it are integer operations: a
// comparison of FP64 values takes 66 clocks as any operation of that unit).
__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ int expo(float x) { return (__float_as_int(x) >> 23) & 0xFF; }
template <typename T>
constexpr int kExpoMax = sizeof(T) == 8 ? 0x7FF : 0xFF;

// The rare cases by definition.  Out of line: inlined, the compiler evaluates
// a division beside every ordinary case and selects afterwards.
template <typename T>
__device__ __noinline__ void pivot_root_slow(T d, T &l, T &y)
{
    l = sqrt(d);
    y = T(1) / l;
}
template <typename T>
__device__ __noinline__ T pivot_scale_slow(T v, T l)
{
    return v / l;
}

// l = sqrt(d) and y = 1 / sqrt(d) of a pivot d > 0, the reciprocal square root
// corrected once against d.
template <typename T>
__device__ __forceinline__ void pivot_root(T d, T &l, T &y)
{
    const int e = expo(d);
    if (e < kExpoMax<T> / 8 || e == kExpoMax<T>) {  // where the corrections could leave the range
        pivot_root_slow(d, l, y);
        return;
    }
    y = rsqrt(d);
    const T h = T(0.5) * y;
    l = d * y;
    l = fma(fma(-l, l, d), h, l);
    y = fma(y, fma(-l, y, T(1)), y);
}
// v / l by the reciprocal y, corrected once: as exact as the division.
template <typename T>
__device__ __forceinline__ T pivot_scale(T v, T l, T y)
{
    T q = v * y;
    q = fma(fma(-q, l, v), y, q);
    if (expo(q) == kExpoMax<T>) q = pivot_scale_slow(v, l);
    return q;
}

// One diagonal block of order nr <= 64 at &A(r0, r0) (A0 points there),
// factorised right-looking in shared memory.  s[c][i] (i >= c) holds the
// block's lower triangle by columns: A(i, c) for the lower form, A(c, i) for
// the upper.  What bounds it is the chain of 64 pivots: a reciprocal square
// root, its corrections and the next pivot's update are about 18 operations
// of the FP64 unit, 66 clocks each.  Warp 0 does nothing else: while it forms
// pivot j + 1 from its own copy of that pivot's column entry, warps 1 and 2
// scale column j and then all but warps 0 and 4 (the one that shares warp 0's
// sub-partition) update the columns behind it.  One CTA barrier a column; a
// finished column goes to A at once.
// Measured (one 64-column block): FP64 70 us, FP32 27 (one thread's square
// root, a division per entry and three barriers a column: 107 and 48).
template <typename T>
__global__ void __launch_bounds__(kLeafThreads)
potrf_leaf_kernel(T *__restrict__ A0, int64_t lda, int nr, int upper, int64_t r0, int *info)
{
    __shared__ T s[kLeafNB][kLeafNB + 1];
    __shared__ T piv[2][2];           // l and y of the pivots, by parity of the column
    __shared__ T col[2][kLeafNB];     // scaled columns, likewise
    __shared__ int fail;
    if (*static_cast<volatile int *>(info) != 0) return;  // an earlier leaf failed
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // load the named triangle, reading A along its contiguous dimension
    // (every load before the first store)
    {
        constexpr int PER = kLeafNB * kLeafNB / kLeafThreads;
        T v[PER];
#pragma unroll
        for (int u = 0; u < PER; u++) {
            const int fast = tid % kLeafNB, slow = tid / kLeafNB + u * (kLeafThreads / kLeafNB);  // A(fast, slow)
            const int i = upper ? slow : fast, c = upper ? fast : slow;
            v[u] = (i < nr && c <= i) ? A0[fast + int64_t(slow) * lda] : T(0);
        }
#pragma unroll
        for (int u = 0; u < PER; u++) {
            const int fast = tid % kLeafNB, slow = tid / kLeafNB + u * (kLeafThreads / kLeafNB);
            s[upper ? fast : slow][upper ? slow : fast] = v[u];
        }
    }
    if (tid < 2 * kLeafNB) (&col[0][0])[tid] = T(0);
    if (tid == 0) fail = kLeafNB;
    __syncthreads();
    auto pivot = [&](int j, T d) {  // warp 0
        T l, y;
        pivot_root(d, l, y);
        if (lane == 0) {
            piv[j & 1][0] = l;
            piv[j & 1][1] = y;
            if (!(d > T(0))) fail = j;
            else A0[j + int64_t(j) * lda] = l;
        }
    };
    if (warp == 0) pivot(0, s[0][0]);
    for (int j = 0; j < nr; j++) {
        __syncthreads();
        if (fail <= j) break;
        const T l = piv[j & 1][0], y = piv[j & 1][1];
        if (warp == 0) {
            if (j + 1 < nr) {
                const T q = pivot_scale(s[j][j + 1], l, y);
                pivot(j + 1, fma(-q, q, s[j + 1][j + 1]));
            }
        } else if (warp != 4) {
            const int w = warp - 1 - (warp > 4);  // 0 .. 5
            T *q = col[j & 1];
            if (w < 2) {
                const int i = 32 * w + lane;
                if (i > j && i < nr) {
                    const T v = pivot_scale(s[j][i], l, y);
                    q[i] = v;
                    A0[upper ? j + int64_t(i) * lda : i + int64_t(j) * lda] = v;
                }
            }
            asm volatile("bar.sync 1, 192;" ::: "memory");
            // columns c > j, rows i >= c (but for the pivot (j + 1, j + 1): warp 0's)
            // (rows past nr hold zeros); columns below 32 in two pieces of
            // rows, two pieces at a time
            int c = j + 1 + w;
            for (; c < 32; c += 6) {
                const T f = q[c];
                const int i = c + lane, i2 = i + 32;
                const T a = s[c][i], b = i2 < kLeafNB ? s[c][i2] : T(0);
                const T qa = q[i], qb = i2 < kLeafNB ? q[i2] : T(0);
                const T ra = fma(-qa, f, a), rb = fma(-qb, f, b);
                if (i > j + 1) s[c][i] = ra;
                if (i2 < kLeafNB) s[c][i2] = rb;
            }
            for (; c < nr; c += 12) {
                const int i = c + lane, c2 = c + 6, i2 = c2 + lane;
                const bool in = i < kLeafNB, in2 = c2 < nr && i2 < kLeafNB;
                const T f = q[c], f2 = c2 < nr ? q[c2] : T(0);
                const T a = in ? s[c][i] : T(0), b = in2 ? s[c2][i2] : T(0);
                const T qa = in ? q[i] : T(0), qb = in2 ? q[i2] : T(0);
                const T ra = fma(-qa, f, a), rb = fma(-qb, f2, b);
                if (in && i > j + 1) s[c][i] = ra;
                if (in2) s[c2][i2] = rb;
            }
        }
    }
    if (tid == 0 && fail < nr) atomicCAS(info, 0, int(r0 + fail + 1));
}

int trsm_call(int side, int uplo, int trans, int64_t m, int64_t n, const double *A, int64_t lda, double *B,
              int64_t ldb, cudaStream_t s)
{
    return gb_dtrsm(side, uplo, trans, GB_NONUNIT, m, n, 1.0, A, lda, B, ldb, s);
}
int trsm_call(int side, int uplo, int trans, int64_t m, int64_t n, const float *A, int64_t lda, float *B,
              int64_t ldb, cudaStream_t s)
{
    return gb_strsm(side, uplo, trans, GB_NONUNIT, m, n, 1.0f, A, lda, B, ldb, s);
}

// Recursive model (Section V-A) on the panel of columns [c0, c1); an Exec
// either launches the tasks or finds their work space.
template <class E>
int potrf_rec(E &e, int64_t c0, int64_t c1)
{
    if (c1 - c0 <= kLeafNB) return e.leaf(c0, c1);
    const int64_t cm = c0 + rec_split(c1 - c0, kLeafNB);
    GB_TRY(potrf_rec(e, c0, cm));
    GB_TRY(e.update(c0, cm, c1));
    return potrf_rec(e, cm, c1);
}

template <typename T>
struct PotrfBytes {
    int64_t n;
    size_t bytes = 0;
    int leaf(int64_t, int64_t) { return 0; }
    int update(int64_t c0, int64_t cm, int64_t c1)
    {
        if (digit_gemm_wanted<T>(n - cm, c1 - cm, cm - c0, 1))
            bytes = std::max(bytes, digit_gemm_bytes<T>(n - cm, c1 - cm, cm - c0, 1));
        return 0;
    }
};

template <typename T>
struct PotrfExec {
    bool upper;
    int64_t n;
    T *A;
    int64_t lda;
    int *info;
    cudaStream_t s;
    size_t digit_bytes;
    DigitWorkspace ws;
    T *at(int64_t i, int64_t c) { return upper ? A + c + i * lda : A + i + c * lda; }
    int leaf(int64_t c0, int64_t c1)
    {
        const int64_t w = c1 - c0;
        {
            LaunchScope ls(KK_DIAG, s, double(w) * w * w / 3.0, sizeof(T) * double(w) * (w + 1));
            potrf_leaf_kernel<T><<<1, kLeafThreads, 0, s>>>(at(c0, c0), lda, int(w), upper, c0, info);
            GB_TRY(check(cudaGetLastError()));
        }
        if (c1 >= n) return 0;
        // L(c1.., c0..) = A(c1.., c0..) L11^-T, or U(c0.., c1..) = U11^-T A(c0.., c1..)
        if (upper) return trsm_call(GB_LEFT, GB_UPPER, GB_TRANS, w, n - c1, at(c0, c0), lda, at(c1, c0), lda, s);
        return trsm_call(GB_RIGHT, GB_LOWER, GB_TRANS, n - c1, w, at(c0, c0), lda, at(c1, c0), lda, s);
    }
    int update(int64_t c0, int64_t cm, int64_t c1)
    {
        const int64_t M = n - cm, N = c1 - cm, K = cm - c0;
        if (digit_gemm_wanted<T>(M, N, K, 1)) {
            if (char *p = ws.get(digit_bytes)) {
                const DigitGemm<T> g{M, N, K, at(cm, c0), lda, !upper, at(cm, c0), lda, upper, at(cm, cm), lda, !upper, T(1), 1};
                return launch_digit_gemm<T>(g, p, ws.size(), s);
            }
        }
        return launch_gemm_trapezoid<T>(!upper, M, N, K, at(cm, c0), lda, at(cm, cm), lda, s);
    }
};

template <typename T>
int potrf_impl(int uplo, int64_t n, T *A, int64_t lda, int64_t *info_out, void *stream)
{
    if (uplo != GB_LOWER && uplo != GB_UPPER) return -1;
    if (n < 0) return -2;
    if (A == nullptr && n > 0) return -3;
    if (lda < (n > 1 ? n : 1)) return -4;
    if (info_out == nullptr) return -5;
    *info_out = 0;
    if (n == 0) return 0;
    if (n > 0x7ffffffeLL) return -2;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaMemPool_t pool = mixed_pool();
    if (!pool) return GB_STATUS_CUDA_ERROR;
    int *dinfo = nullptr;
    GB_CUDA(cudaMallocFromPoolAsync(reinterpret_cast<void **>(&dinfo), sizeof(int), pool, s));
    int st = check(cudaMemsetAsync(dinfo, 0, sizeof(int), s));
    if (!st) {
        PotrfBytes<T> pb{n};
        potrf_rec(pb, 0, n);
        PotrfExec<T> e{uplo == GB_UPPER, n, A, lda, dinfo, s, pb.bytes, DigitWorkspace(s)};
        st = potrf_rec(e, 0, n);
    }
    int h = 0;
    if (!st) st = check(cudaMemcpyAsync(&h, dinfo, sizeof(int), cudaMemcpyDeviceToHost, s));
    cudaFreeAsync(dinfo, s);
    const int c = check(cudaStreamSynchronize(s));
    if (st) return st;
    if (c) return c;
    *info_out = h;
    return 0;
}

}  // namespace
}  // namespace gb

extern "C" int gb_dpotrf(int uplo, int64_t n, double *A, int64_t lda, int64_t *info, void *stream)
{
    return gb::potrf_impl<double>(uplo, n, A, lda, info, stream);
}

extern "C" int gb_spotrf(int uplo, int64_t n, float *A, int64_t lda, int64_t *info, void *stream)
{
    return gb::potrf_impl<float>(uplo, n, A, lda, info, stream);
}
