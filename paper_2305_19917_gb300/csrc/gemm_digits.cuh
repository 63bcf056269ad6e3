// Off-diagonal update by exact digit products on the tensor cores (internal
// header; gemm_digits.cu).
#pragma once
#include <stddef.h>
#include <stdint.h>
#include <cuda_runtime.h>

namespace gb {

// One update C = alpha*C - Aop*Bop, C of M x N, K products per entry.
// am: Aop(i,k) = A[i + k lda] (else A[k + i lda]); bc: Bop(k,j) = B[k + j ldb]
// (else B[j + k ldb]); cl: C(i,j) = C[i + j ldc] (else C[j + i ldc]).
// tri: only the entries of C on and below its diagonal, with Bop = the first N
// rows of Aop, transposed (N <= M; the same digits serve both; B and bc say
// where the CUDA cores find it).
template <typename T>
struct DigitGemm {
    int64_t M, N, K;
    const T *A;
    int64_t lda;
    bool am;
    const T *B;
    int64_t ldb;
    bool bc;
    T *C;
    int64_t ldc;
    bool cl;
    T alpha;
    int tri;
};

// Whether the digit path is the faster one for this size (the rule and its
// measurements stand at the definition).
template <typename T>
bool digit_gemm_wanted(int64_t M, int64_t N, int64_t K, int tri);
// Work space of one update, at most about kWsCap (digit_plan.cuh; larger updates
// are done in pieces).
template <typename T>
size_t digit_gemm_bytes(int64_t M, int64_t N, int64_t K, int tri);
// The update on stream s, with `ws` at least digit_gemm_bytes<T> long and
// 256-byte aligned.
template <typename T>
int launch_digit_gemm(const DigitGemm<T> &g, char *ws, size_t ws_bytes, cudaStream_t s);

// Stream-ordered work space of one solve: taken on the first update that
// wants it (grown when a later one needs more), given back in stream order
// by release().  ok() is false while the stream is being captured or when
// the memory is not to be had: the caller then takes the CUDA-core update.
class DigitWorkspace {
public:
    explicit DigitWorkspace(cudaStream_t s) : s_(s) {}
    ~DigitWorkspace() { release(); }
    // The stream is not being captured.
    bool usable();
    char *get(size_t bytes);
    size_t size() const { return size_; }
    void release();

private:
    cudaStream_t s_;
    char *p_ = nullptr;
    size_t size_ = 0;
    int state_ = 0;  // 0 unknown, 1 usable, -1 not usable
};

// Gives the unused memory that the digit work spaces keep on the current
// device back to the driver.
void digit_pool_trim();

}  // namespace gb
