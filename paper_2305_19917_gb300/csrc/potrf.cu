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
// 127.  n = 8192 FP64: 128 -> 28.5 ms by the panels and the tasks' digit gemms, 18.0
// with the leaf below and overlapped launches; n = 16384 62 ms (1.34 s before the digit gemms).  The upper form (A = U^T U) is the same with everything stored
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
#include "tc_common.cuh"

extern "C" int gb_dtrsm(int side, int uplo, int trans, int diag, int64_t m, int64_t n, double alpha,
                        const double *A, int64_t lda, double *B, int64_t ldb, void *stream);
extern "C" int gb_strsm(int side, int uplo, int trans, int diag, int64_t m, int64_t n, float alpha,
                        const float *A, int64_t lda, float *B, int64_t ldb, void *stream);

namespace gb {
namespace {

constexpr int kLeafNB = 64;
constexpr int kLeafThreads = 384;

// Exponent field and its largest value (tests on it are integer operations: a
// comparison of FP64 values takes 66 clocks as any operation of that unit).
__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ int expo(float x) { return (__float_as_int(x) >> 23) & 0xFF; }
template <typename T>
constexpr int kExpoMax = sizeof(T) == 8 ? 0x7FF : 0xFF;
// where the corrections below could leave the range
template <typename T>
__device__ __forceinline__ bool extreme(T d)
{
    const int e = expo(d);
    return e < kExpoMax<T> / 8 || e == kExpoMax<T>;
}

// The rare cases by definition.  Out of line: inlined, the compiler evaluates
// a division beside every ordinary case and selects afterwards.
template <typename T>
__device__ __noinline__ T root_slow(T d)
{
    return sqrt(d);
}
template <typename T>
__device__ __noinline__ T ratio_slow(T v, T l)
{
    return v / l;
}

// 1 / sqrt(d) to about 22 bits, for d > 0 in the middle of the range: the FP32
// unit's approximation, FP64 exponents and mantissas moved by integer operations.
__device__ __forceinline__ float rsqrt_seed(float d)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
    return y;
}
__device__ __forceinline__ double rsqrt_seed(double d)
{
    const int hi = __double2hiint(d), k = ((hi >> 20) - 1023) >> 1;  // d = m 4^k, 1 <= m < 4
    const unsigned m = unsigned(hi - (k << 21) - (896 << 20));
    const unsigned y = __float_as_uint(rsqrt_seed(__uint_as_float(__funnelshift_l(__double2loint(d), m, 3))));
    return __hiloint2double(int((y >> 3) + (896 << 20)) - (k << 20), int(y << 29));
}
// y = 1 / sqrt(d) of a pivot d > 0: the seed's residual r = 1 - d y^2 through the
// series y (1 + r / 2 + 3 r^2 / 8), what follows is below 2^-63.
template <typename T>
__device__ __forceinline__ T root_rcp(T d)
{
    if (extreme(d)) return ratio_slow(T(1), root_slow(d));
    const T y = rsqrt_seed(d), r = fma(-(d * y), y, T(1));
    return fma(y * r, fma(r, T(0.375), T(0.5)), y);
}
// sqrt(d) by y, corrected once.
template <typename T>
__device__ __forceinline__ T root(T d, T y)
{
    if (extreme(d)) return root_slow(d);
    const T l = d * y;
    return fma(fma(-l, l, d), T(0.5) * y, l);
}
// v / l by the reciprocal y, corrected once: as exact as the division.
template <typename T>
__device__ __forceinline__ T pivot_scale(T v, T l, T y)
{
    T q = v * y;
    q = fma(fma(-q, l, v), y, q);
    if (expo(q) == kExpoMax<T>) q = ratio_slow(v, l);
    return q;
}

// One diagonal block of order nr <= 64 at &A(r0, r0) (A0 points there),
// factorised right-looking: A(i, c) is element (i, c) of the lower form,
// stored (c, i) for the upper.  What bounds it is the FP64 unit, 66 clocks an
// operation of a warp however many lanes take part: a chain of 64 pivots of 9
// operations each, and 43.7k multiply-adds behind them.  Roles, by step j (one CTA barrier each):
//   warp 0        pivot j + 1 and its reciprocal root, from the entries
//                 (j+1, j), (j+1, j+1) as of column j - 2 and what columns
//                 j - 1 and j add to them;
//   warps 1, 2    bring column j (as of column j - 2) up to date and scale it;
//   update warps  take column j - 1 off everything behind column j, and hand
//                 out column j + 1 and pivot entry j + 2.
// So nobody waits within a step.  The update warps hold the triangle in
// registers, packed by columns, 32 elements a slot: full lanes to the end
// (2080 / 32 slots at first; the columns one by one take 94), dealt out by what else
// a warp's sub-partition (warp mod 4) has to do.
// Measured (one 64-column block): FP64 46 us, FP32 24 (updates column by column
// in shared memory, CUDA's rsqrt() in the chain: 70 and 27; one thread's square
// root, a division per entry and three barriers a column: 107 and 48).
constexpr int kLeafSlots = kLeafNB * (kLeafNB + 1) / 2 / 32;  // 65
constexpr int kUpdWarps = 8, kUpdGroups = 3, kUpdPer = 3;     // slots: groups of three a warp
static_assert(kUpdWarps * kUpdGroups * kUpdPer >= kLeafSlots, "slots");

template <typename T>
__global__ void __launch_bounds__(kLeafThreads)
potrf_leaf_kernel(T *__restrict__ A0, int64_t lda, int nr, int upper, int64_t r0, int *info)
{
    __shared__ T cb[2][kLeafNB];  // column j as of column j - 2, by parity
    __shared__ T dg[2];           // pivot entry j + 1 as of column j - 2
    __shared__ T qb[2][kLeafNB];  // scaled columns
    __shared__ T pd[2], py[2];    // pivots and their reciprocal roots
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // update warps 3, 7, 11 | 5, 9 | 6, 10 | 4 (beside the pivots)
    const int uw = warp == 3 ? 0 : warp >= 4 && warp <= 7 ? warp - 3 : warp >= 9 ? warp - 4 : -1;
    T v[kUpdGroups][kUpdPer] = {};
    int col[kUpdGroups][kUpdPer], row[kUpdGroups][kUpdPer], last[kUpdGroups][kUpdPer];  // last: the slot's last column
    if (uw >= 0) {
#pragma unroll
        for (int g = 0; g < kUpdGroups; g++) {
#pragma unroll
            for (int u = 0; u < kUpdPer; u++) {
                const int slot = (g * kUpdPer + u) * kUpdWarps + uw;
                // element 32 slot + lane of the columns of 64, 63, 62, ... entries;
                // from the end column 63 - k starts at k (k + 1) / 2
                const int f = max(kLeafSlots * 32 - 1 - (32 * slot + lane), 0);
                const int k = int((sqrtf(8.0f * float(f) + 1.0f) - 1.0f) * 0.5f);
                const bool in = slot < kLeafSlots;
                const int c = in ? kLeafNB - 1 - k : 0, i = in ? kLeafNB - 1 - (f - k * (k + 1) / 2) : 0;
                col[g][u] = c;
                row[g][u] = i;
                last[g][u] = __shfl_sync(0xffffffffu, in ? c : -1, 31);
            }
        }
    }
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    const int before = *static_cast<volatile int *>(info);
    if (uw >= 0) {
#pragma unroll
        for (int g = 0; g < kUpdGroups; g++)
#pragma unroll
            for (int u = 0; u < kUpdPer; u++) {
                const int c = col[g][u], i = row[g][u];
                if (i < nr) v[g][u] = A0[upper ? c + int64_t(i) * lda : i + int64_t(c) * lda];
            }
#pragma unroll
        for (int u = 0; u < kUpdPer; u++) {  // (columns 0 and 1 lie in the first slots)
            const int c = col[0][u], i = row[0][u];
            if (c == 0) cb[0][i] = v[0][u];
            if (c == i && c < 2) dg[c] = v[0][u];
        }
    }
    if (before != 0) return;  // an earlier leaf failed
    __syncthreads();
    int fail = kLeafNB;  // first pivot that is not positive (warp 0; what follows it is undefined)
    auto pivot = [&](int j, T d) {
        const T y = root_rcp(d);
        if (lane == 0) {
            pd[j & 1] = d;
            py[j & 1] = y;
        }
        if (!(d > T(0))) fail = min(fail, j);
    };
    if (warp == 0) pivot(0, dg[0]);
    for (int j = 0; j < nr; j++) {
        __syncthreads();
        const T *q1 = qb[(j + 1) & 1];  // column j - 1
        if (warp == 0) {
            if (j + 1 < nr) {
                T x = cb[j & 1][j + 1], d = dg[(j + 1) & 1];
                if (j > 0) {
                    const T a = q1[j + 1];
                    x = fma(-a, q1[j], x);
                    d = fma(-a, a, d);
                }
                const T q = x * py[j & 1];
                pivot(j + 1, fma(-q, q, d));
            }
        } else if (warp < 3) {
            const int i = 32 * (warp - 1) + lane;
            if (32 * warp > j) {
                const T d = pd[j & 1], y = py[j & 1];
                T x = cb[j & 1][i];
                if (j > 0) x = fma(-q1[i], q1[j], x);
                const T l = root(d, y), q = pivot_scale(x, l, y);
                if (i > j) qb[j & 1][i] = q;
                if (i >= j && i < nr) A0[upper ? j + int64_t(i) * lda : i + int64_t(j) * lda] = i > j ? q : l;
            }
        } else if (uw >= 0) {
            T *cn = cb[(j + 1) & 1];
            auto publish = [&](int g, int u) {
                const int c = col[g][u], i = row[g][u];
                if (c == j + 1) cn[i] = v[g][u];
                if (c == j + 2 && i == c) dg[j & 1] = v[g][u];
            };
#pragma unroll
            for (int g = 0; g < kUpdGroups; g++) {
                if (sizeof(T) == 8) {
                    // slot by slot: an operation for a finished one costs as
                    // much as any, and loads in a batch gain nothing (52 us)
#pragma unroll
                    for (int u = 0; u < kUpdPer; u++)
                        if (last[g][u] > j) {
                            if (j > 0) v[g][u] = fma(-q1[row[g][u]], q1[col[g][u]], v[g][u]);
                            publish(g, u);
                        }
                } else if (max(last[g][0], max(last[g][1], last[g][2])) > j) {
                    // loads of a group at once
                    if (j > 0) {
                        T qi[kUpdPer], qc[kUpdPer];
#pragma unroll
                        for (int u = 0; u < kUpdPer; u++) {
                            qi[u] = q1[row[g][u]];
                            qc[u] = q1[col[g][u]];
                        }
#pragma unroll
                        for (int u = 0; u < kUpdPer; u++) v[g][u] = fma(-qi[u], qc[u], v[g][u]);
                    }
#pragma unroll
                    for (int u = 0; u < kUpdPer; u++) publish(g, u);
                }
            }
        }
    }
    if (threadIdx.x == 0 && fail < nr) atomicCAS(info, 0, int(r0 + fail + 1));
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
            GB_TRY(check(launch_pdl(potrf_leaf_kernel<T>, dim3(1), dim3(kLeafThreads), 0, s, at(c0, c0), lda, int(w), int(upper),
                                    c0, info)));
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
