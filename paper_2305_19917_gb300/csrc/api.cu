// C-ABI entry points of the plain FP64/FP32 solve: argument checking,
// canonicalisation of the 16 BLAS forms, plan choice and the kernel-launching
// executor for the decomposition drivers.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <mutex>
#include "common.cuh"
#include "driver.cuh"
#include "gemm_digits.cuh"
#include "panel.cuh"
#include "plan.cuh"

namespace gb {

static thread_local int tl_last_cuda_error = 0;
void set_cuda_error(cudaError_t e) { tl_last_cuda_error = (int)e; }

std::atomic<int> g_lookahead{1};

namespace {

std::mutex g_side_mu;
cudaStream_t g_side_stream[64] = {nullptr};

// A library stream per device for the trailing part of split updates.
int side_stream(cudaStream_t *out)
{
    int dev = 0;
    GB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return GB_STATUS_CUDA_ERROR;
    std::lock_guard<std::mutex> lk(g_side_mu);
    if (!g_side_stream[dev]) GB_CUDA(cudaStreamCreateWithFlags(&g_side_stream[dev], cudaStreamNonBlocking));
    *out = g_side_stream[dev];
    return 0;
}

// Rows of the largest TS task solved by one kernel: the panel kernel's (FP64
// 512, FP32 1024), halved while its multiply-adds outside the two halves (r^2 / 4
// per right-hand side, FP64 252 per clock on the whole chip, FP32 about 10000)
// take longer than the digit gemm that would replace them (50 and 30 us at
// these sizes).  FP64 beyond 2432 right-hand sides: the 64-row diagonal kernel
// (4096 rows: 1300 right-hand sides 4.5 ms with panels, 4.7 with it, 2400 4.84 and
// 4.90; beyond, panels of eight columns need a third round of CTAs).
template <typename T>
int64_t ts_rows(int64_t ncols)
{
    if (sizeof(T) == 8 && ncols > 2432) return 64;
    const double split = sizeof(T) == 8 ? 1.0e8 : 2.3e9;
    int64_t r = kPanelRows<T>;
    while (r > 64 && double(r) * double(r) * double(ncols) > split) r /= 2;
    return r;
}

// Whether a TS task of at most 64 rows goes to the diagonal kernel instead of the
// panel kernel, whose blocks are 32 rows whatever the task's: FP64 16 rows 4.3 us
// with any number of right-hand sides (panels 6.7 with 300, 12.8 with 1200, 21 with
// 2400); 32 rows 9.3 (6.8, 8.7 with 600, 12.8, 21); 64 rows 27.5 (11, 25 with 1200, 42).
// FP32 16 rows 2.5 us (2.9, 5.0 with 1200), 32 rows 5 (2.9, 4.9).
template <typename T>
bool diag_wanted(int64_t nr, int64_t ncols)
{
    if (sizeof(T) == 4) return nr <= 16;
    return nr <= 16 || ncols > (nr <= 32 ? 608 : 1216);
}

// FP64 right-hand sides from which updates on the CUDA cores (a stream that is
// being captured: no work space for digits) go with 64-row blocks, one update
// behind each, rather than with panels and the recursive model's small updates,
// whose few tiles leave SMs idle: captured, 1500 x 1500 4.47 ms (5.11 with panels),
// 700 x 2400 1.57 (2.09), 1024 x 3000 3.68 (4.18); 2048 x 1000 panels 5.08, blocks 6.5.
constexpr int64_t kBlockedColumns = 1216;

// A TS task larger than e.rows() is itself solved: by the recursive model down to
// such tasks, whose updates are wide enough for the digit gemm, or, for a plan
// that asks for smaller blocks or without digits, blocked.
template <class E, typename T>
void expand_ts(E &e, int64_t b0, int64_t nr, int64_t nb, T a, bool fwd)
{
    if (nb < 64 || e.blocked) drive_blocked(e, b0, b0 + nr, nb < nr ? nb : 64, a, fwd);
    else drive_recursive(e, b0, b0 + nr, 24, e.rows(), a, fwd);
}

// Executor that finds the work space of a schedule's largest digit gemm, and
// whether an update is tall enough that lookahead would split it: any, or one
// that goes to the CUDA cores although digits can be had.
template <typename T>
struct DigitBytesExec {
    int64_t nb, ncols;
    bool forward;
    bool blocked;
    size_t bytes = 0;
    bool tall = false, tall_cuda = false;
    bool ok() const { return true; }
    int64_t rows() const { return ts_rows<T>(ncols); }
    void ts(int64_t b0, int64_t nr, T a)
    {
        if (nr > rows()) expand_ts(*this, b0, nr, nb, a, forward);
    }
    void gemm(int64_t, int64_t M, int64_t, int64_t K, T)
    {
        const bool digits = !blocked && digit_gemm_wanted<T>(M, ncols, K, 0);
        if (digits) bytes = std::max(bytes, digit_gemm_bytes<T>(M, ncols, K, 0));
        tall = tall || M > 2 * nb;
        tall_cuda = tall_cuda || (!digits && M > 2 * nb);
    }
};

// Executor that launches the kernels of each task on the canonical view.
//
// A gemm task large enough goes to the digit gemm (gemm_digits.cu), in its
// work space; the others to the CUDA-core update, with lookahead:
//
// Lookahead (the overlap of the diagonal solve with the off-diagonal
// updates that the paper's blocked model aims at, Section V-C, and names as
// future work, Section VIII): a gemm task whose rows extend beyond the next
// diagonal block is split in two.  The head -- the next block's `nb` rows,
// the first ones the schedule needs -- runs on the caller's stream, so the
// next TS task can start at once; the tail -- every other row -- runs on a
// second stream at the same time.  Dependencies: the tail is ordered after
// everything issued on the caller's stream so far (an event: it reads the X
// rows just solved and writes rows those launches may have written), and
// any later launch on the caller's stream that touches rows written by an
// outstanding tail first waits for the latest tail (the tails run in order
// on their stream).  The solve joins the second stream before it returns.
template <typename T>
struct LaunchExec {
    const Canon<T> &c;
    int64_t nb;  // plan block size (inner blocking of large TS tasks)
    int status = 0;
    bool lookahead = false;
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_tail = nullptr;
    int64_t pend_lo = 0, pend_hi = 0;  // rows written by tails not yet waited for
    bool blocked = false;              // no digits, and wide (kBlockedColumns)
    size_t digit_bytes = 0;            // work space of the schedule's largest digit gemm (0: none)
    DigitWorkspace &dws;
    LaunchExec(const Canon<T> &c_, int64_t nb_, DigitWorkspace &dws_) : c(c_), nb(nb_), dws(dws_) {}
    ~LaunchExec()
    {
        if (ev_fork) cudaEventDestroy(ev_fork);
        if (ev_tail) cudaEventDestroy(ev_tail);
    }
    bool ok() const { return status == 0; }
    int64_t rows() const { return blocked ? 64 : ts_rows<T>(c.ncols); }
    int enable_lookahead()
    {
        GB_TRY(side_stream(&side));
        GB_CUDA(cudaEventCreateWithFlags(&ev_fork, cudaEventDisableTiming));
        GB_CUDA(cudaEventCreateWithFlags(&ev_tail, cudaEventDisableTiming));
        lookahead = true;
        return 0;
    }
    // Before a launch on the caller's stream that touches rows [r0, r1).
    void settle(int64_t r0, int64_t r1)
    {
        if (status || pend_hi <= pend_lo || r1 <= pend_lo || r0 >= pend_hi) return;
        status = check(cudaStreamWaitEvent(c.stream, ev_tail, 0));
        pend_lo = pend_hi = 0;
    }
    // End of the solve: the caller's stream waits for the last tail.
    int join()
    {
        if (lookahead && !status && pend_hi > pend_lo) status = check(cudaStreamWaitEvent(c.stream, ev_tail, 0));
        pend_lo = pend_hi = 0;
        return status;
    }
    void ts(int64_t b0, int64_t nr, T a)
    {
        if (status) return;
        if (nr <= rows()) {
            settle(b0, b0 + nr);
            if (status) return;
            status = nr <= 64 && diag_wanted<T>(nr, c.ncols) ? launch_diag_solve(c, b0, (int)nr, a)
                                                             : launch_panel_solve(c, b0, (int)nr, a);
            return;
        }
        expand_ts(*this, b0, nr, nb, a, c.forward);
    }
    void gemm(int64_t ci0, int64_t M, int64_t ak0, int64_t K, T a)
    {
        if (status) return;
        // (decided on the whole task, so that lookahead does not change it)
        if (digit_bytes && digit_gemm_wanted<T>(M, c.ncols, K, 0)) {
            char *ws = dws.get(digit_bytes);
            if (ws) {
                settle(ci0, ci0 + M);
                if (status) return;
                const DigitGemm<T> g{M, c.ncols, K, mv_ptr(c, ci0, ak0), c.lda, !c.mt, bv_ptr(c, ak0, 0), c.ldb, c.left,
                                     bv_ptr(c, ci0, 0), c.ldb, c.left, a, 0};
                status = launch_digit_gemm<T>(g, ws, dws.size(), c.stream);
                return;
            }
        }
        const int64_t h = nb;  // rows of the next diagonal block
        if (!lookahead || M <= 2 * h) {
            settle(ci0, ci0 + M);
            if (!status) status = launch_gemm_update(c, ci0, M, ak0, K, a);
            return;
        }
        // forward: the next block is at the top of the rows, backward at the bottom
        const int64_t head0 = c.forward ? ci0 : ci0 + M - h;
        const int64_t tail0 = c.forward ? ci0 + h : ci0;
        const int64_t tailM = M - h;
        // the head's rows may still be pending in an older tail
        settle(head0, head0 + h);
        if (status) return;
        // tail on the second stream, after everything issued so far
        if ((status = check(cudaEventRecord(ev_fork, c.stream)))) return;
        if ((status = check(cudaStreamWaitEvent(side, ev_fork, 0)))) return;
        Canon<T> cs = c;
        cs.stream = side;
        if ((status = launch_gemm_update(cs, tail0, tailM, ak0, K, a))) return;
        if ((status = check(cudaEventRecord(ev_tail, side)))) return;
        // the tail covers rows the fork already ordered; any earlier pending
        // tail is ordered before this one on the second stream
        pend_lo = pend_hi > pend_lo ? std::min(pend_lo, tail0) : tail0;
        pend_hi = std::max(pend_hi, tail0 + tailM);
        // head on the caller's stream: disjoint from the new tail's rows, and
        // ordered after any older tail that wrote them (settled above)
        status = launch_gemm_update(c, head0, h, ak0, K, a);
    }
};

template <typename T>
int trsm_impl(int side, int uplo, int trans, int diag, int64_t m, int64_t n, T alpha,
              const T *A, int64_t lda, T *B, int64_t ldb, const gb_plan *plan, void *stream)
{
    if (side != GB_LEFT && side != GB_RIGHT) return -1;
    if (uplo != GB_LOWER && uplo != GB_UPPER) return -2;
    if (trans != GB_NOTRANS && trans != GB_TRANS) return -3;
    if (diag != GB_NONUNIT && diag != GB_UNIT) return -4;
    if (m < 0) return -5;
    if (n < 0) return -6;
    const int64_t k = side == GB_LEFT ? m : n;
    const bool empty = (m == 0 || n == 0);
    if (A == nullptr && !empty && alpha != T(0)) return -8;
    if (lda < (k > 1 ? k : 1)) return -9;
    if (B == nullptr && !empty) return -10;
    if (ldb < (m > 1 ? m : 1)) return -11;
    gb_plan p;
    if (plan != nullptr) {
        if (!plan_valid(*plan)) return -12;
        p = *plan;
    }
    if (empty) return 0;

    Canon<T> c;
    c.A = A;
    c.lda = lda;
    c.mt = side == GB_LEFT ? (trans == GB_TRANS) : (trans == GB_NOTRANS);
    c.forward = (uplo == GB_LOWER) != c.mt;
    c.unit = diag == GB_UNIT;
    c.B = B;
    c.ldb = ldb;
    c.left = side == GB_LEFT;
    c.k = k;
    c.ncols = side == GB_LEFT ? n : m;
    c.alpha = alpha;
    c.stream = static_cast<cudaStream_t>(stream);

    if (alpha == T(0)) return launch_zero(c);
    DigitWorkspace dws(c.stream);
    const bool blocked = sizeof(T) == 8 && k > 64 && c.ncols > kBlockedColumns && !dws.usable();
    if (plan == nullptr || plan->driver == GB_DRIVER_AUTO)
        p = choose_plan(sizeof(T) == 8 ? GB_DTYPE_F64 : GB_DTYPE_F32, side, uplo, trans, m, n, blocked);
    LaunchExec<T> e(c, p.nb, dws);
    e.blocked = blocked;
    DigitBytesExec<T> db{p.nb, c.ncols, c.forward, blocked};
    drive_plan(db, p.driver, k, p.nb, p.depth, alpha, c.forward);
    e.digit_bytes = db.bytes;
    // lookahead where a split update can overlap the next diagonal block: the
    // blocked and recursive models on more than four blocks of rows, with
    // updates on the CUDA cores (digit gemms are not split)
    if (g_lookahead.load() && p.driver != GB_DRIVER_ITERATIVE && k > 4 * p.nb &&
        (db.tall_cuda || (db.tall && db.bytes && !dws.usable())))
        GB_TRY(e.enable_lookahead());
    drive_plan(e, p.driver, k, p.nb, p.depth, alpha, c.forward);
    if (e.status) {
        e.join();  // leave no work of this call on the second stream unordered
        return e.status;
    }
    return e.join();
}

// Executor that only counts the plan-level tasks.
struct CountExec {
    int64_t n_ts = 0, n_gemm = 0, n_blocks = 0;
    double madds = 0;
    int64_t nb = 1;
    bool ok() const { return true; }
    void ts(int64_t, int64_t, double) { n_ts++; }
    void gemm(int64_t, int64_t M, int64_t, int64_t K, double)
    {
        n_gemm++;
        madds += double(M) * double(K);
        n_blocks += ((M + nb - 1) / nb) * ((K + nb - 1) / nb);
    }
};

}  // namespace
}  // namespace gb

extern "C" {

int gb_dtrsm(int side, int uplo, int trans, int diag, int64_t m, int64_t n, double alpha,
             const double *A, int64_t lda, double *B, int64_t ldb, void *stream)
{
    return gb::trsm_impl<double>(side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb, nullptr, stream);
}

int gb_strsm(int side, int uplo, int trans, int diag, int64_t m, int64_t n, float alpha,
             const float *A, int64_t lda, float *B, int64_t ldb, void *stream)
{
    return gb::trsm_impl<float>(side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb, nullptr, stream);
}

int gb_dtrsm_plan(int side, int uplo, int trans, int diag, int64_t m, int64_t n, double alpha,
                  const double *A, int64_t lda, double *B, int64_t ldb, const gb_plan *plan,
                  void *stream)
{
    return gb::trsm_impl<double>(side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb, plan, stream);
}

int gb_strsm_plan(int side, int uplo, int trans, int diag, int64_t m, int64_t n, float alpha,
                  const float *A, int64_t lda, float *B, int64_t ldb, const gb_plan *plan,
                  void *stream)
{
    return gb::trsm_impl<float>(side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb, plan, stream);
}

int gb_plan_counts(const gb_plan *plan, int64_t k, int64_t *n_diag, int64_t *n_gemm,
                   int64_t *n_offdiag_blocks, double *gemm_madds_per_col)
{
    if (plan == nullptr || !gb::plan_valid(*plan) || plan->driver == GB_DRIVER_AUTO) return -1;
    if (k < 0) return -2;
    gb::CountExec e;
    e.nb = plan->nb;
    gb::drive_plan(e, plan->driver, k, (int64_t)plan->nb, plan->depth, 1.0, true);
    if (n_diag) *n_diag = e.n_ts;
    if (n_gemm) *n_gemm = e.n_gemm;
    if (n_offdiag_blocks) *n_offdiag_blocks = e.n_blocks;
    if (gemm_madds_per_col) *gemm_madds_per_col = e.madds;
    return 0;
}

const char *gb_status_string(int status)
{
    if (status < 0) return "invalid argument (status -i names argument i)";
    switch (status) {
    case GB_STATUS_OK: return "success";
    case GB_STATUS_NOT_CONVERGED: return "iterative refinement did not reach the tolerance";
    case GB_STATUS_CUDA_ERROR: return "CUDA error (see gb_last_cuda_error)";
    case GB_STATUS_TIMEOUT: return "device-side wait exceeded its iteration limit";
    case GB_STATUS_NO_MODEL: return "no cost model loaded";
    case GB_STATUS_SCRATCH_TOO_SMALL: return "problem too large for the fixed no-allocation scratch";
    case GB_STATUS_RANGE: return "operands outside the FP32 range of the low-precision solve";
    default: return "unknown status";
    }
}

int gb_last_cuda_error(void) { return gb::tl_last_cuda_error; }

int gb_set_lookahead(int on)
{
    const int old = gb::g_lookahead.load();
    if (on == 0 || on == 1) gb::g_lookahead.store(on);
    return old;
}

int gb_version(void) { return 100; }

}  // extern "C"
