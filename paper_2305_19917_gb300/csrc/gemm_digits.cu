// Off-diagonal update C = alpha*C - Aop*Bop of the plain FP64 / FP32 solve on
// the tensor cores: the paper's gemm task (Section IV stage 2) by exact
// integer digit products.
//
// What bounds the CUDA-core update (gemm_simt.cu) is the FP64 unit: two DFMA
// per clock and SM, 1.26 TFLOP/s for the chip.  The BF16 tensor cores do
// about 1700 TFLOP/s, so cutting both factors into 8-bit digits and forming
// the digit products there is faster although 36 of them stand for one FP64
// product (10 for FP32).  Three launches per update:
//
//  1. digits_kernel: row i of Aop (column j of Bop) is scaled by the power of
//     two 2^-e that brings its largest entry below 1/2 and rounded to a
//     fixed-point number of 8 P - 1 bits and a sign, P = 8 (FP64) or 4 (FP32),
//     cut into P balanced base-256 digits, each an integer |d| <= 128 that BF16
//     holds exactly.  An entry keeps all its bits down to 2^-10 (FP32 2^-7) of
//     the largest one.
//  2. digit_mma_kernel: per 128 x 128 tile of C the digit products S_pq =
//     sum_k a_p x_q with p + q <= P + 1 (what is left out lies below 2^-60,
//     FP32 2^-30, of the scales' product).  K advances in chunks of 256, over
//     which the sums of one weight p + q are exact integers in the FP32
//     accumulators (the last two of FP64 nearly: Sched); so the pairs of one
//     weight share an accumulator (FP64: 36 pairs in ten accumulators, five
//     passes over the chunk, four where a CTA's share of K is at most 128), and
//     the chunk's sums are added into int64 sums T = sum 2^(W-8(p+q)) S_pq.
//     FP64's last weights lie below T's last bit: they are scaled and rounded
//     before they are added.  W is the largest weight for which T cannot
//     overflow, by the 2-norms of the tile's rows and columns, which pass 1
//     finds.  A pass multiplies slice a_p with [x_q; x_q+1] (N = 256: two
//     weights at a time, two accumulators of 128 x 256, one drained while the
//     other fills).
//     When a tile's sums are complete C = alpha C - 2^(e_i+f_j-W) T follows
//     in the same kernel, one rounding of T, while the tensor cores are at
//     the next tile.
//  3. digit_fallback_kernel: the tiles that pass 2 listed (usually none).
//
// Accuracy: what the digits leave out of a factor is below 2^-63 (FP32 2^-31) of
// its row's (column's) largest entry, what T's last bit leaves out of a chunk
// about 2^-62 of the factors' 2-norms, where the CUDA-core sum rounds every step
// at 2^-54 (2^-25) of the partial sum.  That is relative to the largest entries,
// not to each product: for a sum in which large entries of Aop meet only small
// ones of Bop it would be worse.  Pass 1 therefore counts the entries of every
// row and column within 2^-4 (and 2^-2) of its largest; where the counts of a row
// and a column add up to K + n, at least n products of the sum have both factors
// so near their scales, and n has to outweigh what is left out (kLeftOut,
// kLastBit).  A tile with a row and a column for which it does not, with an
// infinity or a NaN, or with exponents near the ends of the range, is listed for
// the last pass, which computes it with the CUDA-core tile of gemm_tile.cuh: the
// operations of gemm_simt.cu.  So is a tile whose bounded waits gave up.
//
// Measured, rms error over u sum |a||x|, digits / CUDA-core sum: uniform times
// normal entries 0.08 / 0.39 (FP64, K = 64), 0.016 / 0.38 (4096), 0.05 / 0.49 (FP32,
// K = 128).  At the edge of what the rule lets pass (n products at 2^-4 of the
// scales each, the other large entries against ones of 2^-30) 0.10 / 0.40 (FP64, K =
// 64, n = 32), 0.24 / 0.34 (1024, n = 512), 0.15 / 0.30 (FP32, 128, n = 64).  A rule of
// 5/4 K counted entries let pass, with a digit less (28 and 6 pairs: 4.95 instead of
// 5.9 ms for 4096 x 8192 x 4096 FP64, 1.49 instead of 2.14 FP32) and W at most 52,
// factors with 17 / 0.6 and 8.9 / 0.3; one of 3/2 K beyond K = 1024 listed tiles of
// exponential-kernel factors that the digits hold well (4096 x 4096 solve 33.8 ms,
// now 6.6).
#include <mutex>
#include <type_traits>
#include <cuda_bf16.h>
#include "common.cuh"
#include "digit_plan.cuh"
#include "fixed.cuh"
#include "gemm_digits.cuh"
#include "gemm_tile.cuh"
#include "tc_common.cuh"

namespace gb {

using namespace digits;

namespace {

constexpr int STAGES = 4;
constexpr int KC = 256;                        // K of one exact accumulation
constexpr uint32_t TILE_BYTES = BM * BK * 2;   // one digit tile of 128 rows
constexpr uint32_t STAGE_BYTES = 3 * TILE_BYTES;
constexpr int EPI_WARPS = 16;                  // four column groups of 32 times the four TMEM lane groups
constexpr int MMA_THREADS = 32 * (2 + EPI_WARPS);
constexpr uint32_t XP_BYTES = 32 * 5 * 8;      // a warp's transpose buffer (row-major C)
constexpr size_t MMA_SMEM = 1024 + STAGES * size_t(STAGE_BYTES) + EPI_WARPS * size_t(XP_BYTES) + 256;
constexpr int DROWS = 32;                      // rows of one digits_kernel CTA
constexpr int DTHREADS = 256;
constexpr int kMaxCluster = 8;
constexpr int kCntBad = -(1 << 28);            // a row the digits must not represent
// The rule for what the digits may take ("Accuracy" above; digit_item): entries
// within 2^-kNear (FP64 also: 2^-kNear2) of their row's largest are counted, and
// the products of two such must number kLeftOut sqrt(K) + kLastBit times T's last
// bit, in units of 2^-53 of the scales' product, times the root of how often it
// is rounded.  By rms: what the digits leave out is 0.0005 sqrt(K) (FP32 0.0022) of
// that unit, T's rounding 0.3 to 0.45 of its last bit; the CUDA-core sum's error 0.35
// to 0.6 of sum |a||x|, of which a product of two counted entries has 2^-8.8 of the
// scales' product (both within 2^-kNear2: 2^-4.8, one of them: 2^-6.8) if they are
// spread over their binades.
constexpr int kNear = 4, kNear2 = 2;
template <typename T>
constexpr float kLeftOut = sizeof(T) == 8 ? 0.8f : 3.0f;
constexpr float kLastBit = 640.f;

template <typename T>
struct Fmt;
template <>
struct Fmt<double> {
    static constexpr int P = 8;        // digits
    static constexpr int BIAS = 1023;
    static constexpr int EMAX = 400;   // |exponent of the largest entry| beyond which the CUDA cores take over
    __device__ static int field(double a) { return bexp(a); }
};
template <>
struct Fmt<float> {
    static constexpr int P = 4;
    static constexpr int BIAS = 127;
    static constexpr int EMAX = 45;
    __device__ static int field(float a) { return int((__float_as_uint(a) >> 23) & 0xFF); }
};

// a != 0 by its bits (a comparison of FP64 values takes 66 clocks of that unit).
__device__ __forceinline__ bool nonzero(double a) { return ((__double2hiint(a) << 1) | __double2loint(a)) != 0; }
__device__ __forceinline__ bool nonzero(float a) { return (__float_as_uint(a) << 1) != 0u; }

// Digits of a (exponent field of the row's largest entry: emax), most
// significant first, as the bit patterns of exact FP32 integers.
// e' = emax - BIAS + 1: |a| < 2^e', N = round(|a| 2^(8P - 1 - e')), so that every
// digit is at most 128; each with the sign of a.  Returns |d[0]|.
__device__ __forceinline__ int digits_of(double a, int emax, uint32_t (&d)[8])
{
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(a));
    const int E = int((b >> 52) & 0x7FF);
    const unsigned long long mant = E ? ((b & ((1ull << 52) - 1)) | (1ull << 52)) : 0ull;
    const uint32_t sign = uint32_t(b >> 32) & 0x80000000u;
    const int r = emax - E - 10;  // N = mant 2^-r
    unsigned long long n;
    if (r <= 0) n = mant << (-r);  // r >= -10
    else if (r >= 54) n = 0;
    else n = (mant + (1ull << (r - 1))) >> r;
    int x = int(uint32_t(n) & 0xFFFFFFu);
#pragma unroll
    for (int p = 7; p >= 5; p--) {
        const int q = bal8(x);
        d[p] = small_int_f32bits(q) ^ sign;
        x = (x - q) >> 8;
    }
    x += int(uint32_t(n >> 24) & 0xFFFFFFu);
#pragma unroll
    for (int p = 4; p >= 2; p--) {
        const int q = bal8(x);
        d[p] = small_int_f32bits(q) ^ sign;
        x = (x - q) >> 8;
    }
    x += int(uint32_t(n >> 48));  // at most 2^15
    const int q = bal8(x);
    d[1] = small_int_f32bits(q) ^ sign;
    x = (x - q) >> 8;
    d[0] = small_int_f32bits(x) ^ sign;
    return x;
}
__device__ __forceinline__ int digits_of(float a, int emax, uint32_t (&d)[4])
{
    const uint32_t b = __float_as_uint(a);
    const int E = int((b >> 23) & 0xFF);
    const uint32_t mant = E ? ((b & 0x7FFFFFu) | 0x800000u) : 0u;
    const uint32_t sign = b & 0x80000000u;
    const int r = emax - E - 7;
    uint32_t n;
    if (r <= 0) n = mant << (-r);  // r >= -7
    else if (r >= 25) n = 0;
    else n = (mant + (1u << (r - 1))) >> r;
    int x = int(n & 0xFFFFu);
#pragma unroll
    for (int p = 3; p >= 2; p--) {
        const int q = bal8(x);
        d[p] = small_int_f32bits(q) ^ sign;
        x = (x - q) >> 8;
    }
    x += int(n >> 16);  // at most 2^15
    const int q = bal8(x);
    d[1] = small_int_f32bits(q) ^ sign;
    x = (x - q) >> 8;
    d[0] = small_int_f32bits(x) ^ sign;
    return x;
}

// ---- pass 1: digits ----------------------------------------------------------

// One factor: R(r, k), r < rows, k < K; contiguous along k (kc) or along r.
template <typename T>
struct DigitSrc {
    const T *src;
    int64_t ld;
    int kc;
    int rows;             // valid rows; rp = padded to 128
    int rp;
    __nv_bfloat16 *out;   // P planes of rp x kp, row-major
    int *e;               // exponent e' + 1 per row
    int *cnt;             // entries within 2^-kNear of the largest; kCntBad; >= 2K for a zero or padding row
    int *cnt2;            // FP64: those within 2^-kNear2
    int *nrm;             // FP64: sum of (|d[0]| + 1)^2, above 2^16 times that of the squared entries over 2^(e' + 1)
};

// What bounds this kernel is the integer work of the digits (about half the
// issue slots) and the latency of its loads.  The next tile's loads go out before
// this one's digits are formed, and zeros are told by integer operations: the
// factors of 4096 x 8192 x 4096 take 370 us in FP64 (178 at the HBM rate), 208 in
// FP32 (with seven and three digits 362 and 181).  A CTA takes 32 rows
// and a share of K; the CTAs of one row block form a cluster along K (so that
// a few rows of a long K still fill the chip) and exchange the rows' largest
// exponents and counts through distributed shared memory.  The second read of
// the tile comes from L2.
template <typename T>
__global__ void __launch_bounds__(DTHREADS, sizeof(T) == 8 ? 3 : 4)
digits_kernel(DigitSrc<T> a, DigitSrc<T> x, int ablocks, int K, int kp, int *zero, int nzero, ulonglong2 *sums, int64_t nsums)
{
    constexpr int P = Fmt<T>::P;
    __shared__ T t[2][DROWS][65];
    __shared__ int key[DROWS];   // 2 * largest exponent field + (any nonzero entry)
    __shared__ int num[DROWS];
    __shared__ int sqs[DROWS];
    __shared__ int emx[DROWS];
    const int tid = threadIdx.x;
    const bool isa = int(blockIdx.x) < ablocks;
    const DigitSrc<T> s = isa ? a : x;
    const int r0 = (isa ? blockIdx.x : blockIdx.x - ablocks) * DROWS;
    const int rank = blockIdx.y, ncta = gridDim.y;  // the cluster is the grid's y extent
    const int ntile = kp / BK, per = (ntile + ncta - 1) / ncta;
    const int t0 = min(rank * per, ntile), t1 = min(t0 + per, ntile);

    if (tid < DROWS) {
        key[tid] = 0;
    }
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    // the tiles' words and sums of pass 2
    {
        const int64_t z0 = int64_t(blockIdx.x * gridDim.y + blockIdx.y) * DTHREADS + tid;
        const int64_t step = int64_t(gridDim.x) * gridDim.y * DTHREADS;
        for (int64_t z = z0; z < nzero; z += step) zero[z] = 0;
        for (int64_t z = z0; z < nsums; z += step) sums[z] = make_ulonglong2(0ull, 0ull);
    }
    __syncthreads();
    auto load = [&](int tile, T (&v)[8]) {
        const int kb = tile * BK;
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int r = s.kc ? (tid >> 6) + 4 * u : (tid & 31);
            const int k = kb + (s.kc ? (tid & 63) : (tid >> 5) + 8 * u);
            const bool in = r0 + r < s.rows && k < K;
            v[u] = in ? (s.kc ? s.src[k + int64_t(r0 + r) * s.ld] : s.src[r0 + r + int64_t(k) * s.ld]) : T(0);
        }
    };
    // largest exponent field of every row
    int mx[8];
#pragma unroll
    for (int u = 0; u < 8; u++) mx[u] = 0;
    T v[8];
#pragma unroll 2
    for (int tile = t0; tile < t1; tile++) {
        load(tile, v);
#pragma unroll
        for (int u = 0; u < 8; u++) mx[u] = max(mx[u], 2 * Fmt<T>::field(v[u]) + (nonzero(v[u]) ? 1 : 0));
    }
    if (s.kc) {  // a warp's lanes share the rows (tid >> 6) + 4u
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int w = __reduce_max_sync(0xffffffffu, mx[u]);
            if ((tid & 31) == 0) atomicMax(&key[(tid >> 6) + 4 * u], w);
        }
    } else {
#pragma unroll
        for (int u = 1; u < 8; u++) mx[0] = max(mx[0], mx[u]);
        atomicMax(&key[tid & 31], mx[0]);
    }
    auto cluster_sync = [&]() {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    // p of cluster CTA c's copy of a shared variable
    auto peer = [&](const int *p, int c) {
        uint32_t ad;
        int r;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ad) : "r"(tc::smem_u32(p)), "r"(c));
        asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(r) : "r"(ad) : "memory");
        return r;
    };
    cluster_sync();
    if (tid < DROWS) {
        int m = 0;
        for (int c = 0; c < ncta; c++) m = max(m, peer(&key[tid], c));
        emx[tid] = m;
    }
    __syncthreads();
    // digits, 8 consecutive k of one row per thread and tile
    const int row = tid >> 3, lk = (tid & 7) * 8;
    const int em = emx[row] >> 1;
    int near = 0, sq = 0;  // FP64: within 2^-kNear2 counted in the upper half of near
    const size_t plane = size_t(s.rp) * size_t(kp);
    // (backwards: the last tile is still in registers; the next one's loads go
    // out before the digits of this one are formed)
    for (int tile = t1 - 1; tile >= t0; tile--) {
        T(*tb)[65] = t[tile & 1];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int r = s.kc ? (tid >> 6) + 4 * u : (tid & 31);
            const int k = s.kc ? (tid & 63) : (tid >> 5) + 8 * u;
            tb[r][k] = v[u];
        }
        if (tile > t0) load(tile - 1, v);
        __syncthreads();
        uint32_t w[P][4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
            uint32_t d0[P], d1[P];
            const T a0 = tb[row][lk + u], a1 = tb[row][lk + u + 1];
            const int g0 = digits_of(a0, em, d0) + 1, g1 = digits_of(a1, em, d1) + 1;
            const int f0 = nonzero(a0) ? Fmt<T>::field(a0) - em : -kNear - 1, f1 = nonzero(a1) ? Fmt<T>::field(a1) - em : -kNear - 1;
            near += (f0 >= -kNear) + (f1 >= -kNear);
            if (sizeof(T) == 8) {
                near += ((f0 >= -kNear2) + (f1 >= -kNear2)) << 16;
                sq += g0 * g0 + g1 * g1;
            }
#pragma unroll
            for (int p = 0; p < P; p++) w[p][u >> 1] = pack_hi16(d0[p], d1[p]);
        }
        __nv_bfloat16 *o = s.out + size_t(r0 + row) * size_t(kp) + size_t(tile * BK + lk);
#pragma unroll
        for (int p = 0; p < P; p++)
            *reinterpret_cast<uint4 *>(o + p * plane) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        near += __shfl_xor_sync(0xffffffffu, near, o);
        if (sizeof(T) == 8) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    }
    if ((tid & 7) == 0) {
        num[row] = near;
        sqs[row] = sq;
    }
    cluster_sync();
    if (rank == 0 && tid < DROWS) {
        int c = 0, n2 = 0;
        for (int q = 0; q < ncta; q++) {
            c += peer(&num[tid], q);
            if (sizeof(T) == 8) n2 += peer(&sqs[tid], q);
        }
        const int k2 = emx[tid], f = k2 >> 1, e = f - Fmt<T>::BIAS;
        int c2 = c >> 16;
        c &= 0xFFFF;
        if (k2 == 0) c = c2 = 2 * K;                                    // a zero row: exact
        else if (f == 0 || e > Fmt<T>::EMAX || e < -Fmt<T>::EMAX) c = kCntBad;  // infinities and NaN too
        s.cnt[r0 + tid] = c;
        s.e[r0 + tid] = k2 == 0 ? 0 : e + 2;
        if (sizeof(T) == 8) {
            s.cnt2[r0 + tid] = c2;
            s.nrm[r0 + tid] = n2;
        }
    }
    cluster_sync();  // no CTA leaves while its shared memory may be read
}

// ---- pass 2: digit products ----------------------------------------------------

// The schedule of a chunk: products in order, grouped into passes (pass j:
// weight b = base(j) in the low half of the accumulator, b + 1 in the high
// half).  Product o takes A slice p(o) (0-based) with X slices q(o) = b - 2 - p
// and q(o) + 1 into both halves (two(o)), or slice b - 1 with X slice 0 alone
// into the high half.  With digits of at most 128 a pair's sum over K = 256 is at
// most 2^22.
//
// Full: a half holds at most four pairs of one weight, so that the sums of the
// weights up to 7 are exact integers of at most 2^24; weights 6 and 7 take two
// passes.  The seven and eight pairs of the last two weights share one: their
// sums may reach 2^25 and round at 2^-63 and below of the scales' product.  Thin,
// for shares of at most 128 of K: all pairs of a weight fit one half exactly,
// four passes are drained instead of five.
template <typename T>
struct Sched;
template <>
struct Sched<double> {
    static constexpr int THIN_K = 128;
    __device__ static int passes(bool thin) { return thin ? 4 : 5; }
    __device__ static int first(int j, bool thin) { return thin ? j * (j + 1) : int(0x140c0a060200ull >> (8 * j)) & 255; }
    __device__ static int base(int j, bool thin) { return thin ? 2 + 2 * j : (0x86642 >> (4 * j)) & 15; }
    __device__ static int p(int o, int j, bool thin) { return o - first(j, thin) + (!thin && j == 3 ? 4 : 0); }
};
template <>
struct Sched<float> {
    static constexpr int THIN_K = 0;
    __device__ static int passes(bool) { return 2; }
    __device__ static int first(int j, bool) { return j * (j + 1); }
    __device__ static int base(int j, bool) { return 2 + 2 * j; }
    __device__ static int p(int o, int j, bool) { return o - first(j, false); }
};

// The tiles' words, cleared by pass 1: number of listed tiles, how many parts of
// them the last pass has handed out, then per
// tile: partial sums stored (split > 1), listed or not, and the list; last the
// bounded waits' status (nobody reads it: a tile whose wait gave up is listed).
struct TileWords {
    int *count, *next, *done, *listed, *list;
};

template <typename T>
struct MmaArgs {
    DigitGemm<T> g;
    long long *Tg;      // split > 1: the tiles' sums (128 x 128, column-major), cleared by pass 1
    const int *cnt_a, *cnt_x, *cnt2_a, *cnt2_x, *nrm_a, *nrm_x, *e_a, *e_x;
    TileWords w;
    int kp, nMt, nNt, ntiles, split;
    int *status;
};

// Tile (m, n) number t of the launch: grouped rasterisation of the full
// grid, or of the trapezoid n <= m, its triangle first.
__device__ __forceinline__ void digit_tile(int t, int nMt, int nNt, int tri, int &m, int &n)
{
    if (tri) {
        const int head = nNt * (nNt + 1) / 2;
        if (t < head) {
            m = int((sqrtf(8.0f * float(t) + 1.0f) - 1.0f) * 0.5f);
            while (m * (m + 1) / 2 > t) m--;
            while ((m + 1) * (m + 2) / 2 <= t) m++;
            n = t - m * (m + 1) / 2;
            return;
        }
        tc::raster_grouped(t - head, nMt - nNt, nNt, 8, m, n);
        m += nNt;
        return;
    }
    tc::raster_grouped(t, nMt, nNt, 8, m, n);
}

__device__ __forceinline__ double scale_sum(double, long long t, int e) { return scaled_i64_to_f64(t, e); }
// |T| 2^e with a normal scale factor (EMAX bounds e): one rounding, of T
__device__ __forceinline__ float scale_sum(float, long long t, int e)
{
    return __ll2float_rn(t) * __int_as_float((e + 127) << 23);
}

// One work item of a CTA: a tile and a share [k0, k1) of K, taken in chunks of KC.
struct Item {
    int tile, i0, j0, sp, k0, k1;
    bool skip;  // the digits may not represent this tile
    bool thin;  // schedule
    int W;      // the sums are those of the products over the scales, times 2^W
};
// Evaluated by every warp for itself (all lanes).
template <typename T>
__device__ __forceinline__ Item digit_item(const MmaArgs<T> &a, int w, int lane)
{
    Item it;
    it.tile = w % a.ntiles;
    it.sp = w / a.ntiles;
    int m, n;
    digit_tile(it.tile, a.nMt, a.nNt, a.g.tri, m, n);
    it.i0 = m * BM;
    it.j0 = n * BM;
    share_range(a.kp / BK, a.split, it.sp, it.k0, it.k1);
    it.k0 *= BK;
    it.k1 *= BK;
    // (an empty share, of which the host makes none, runs no pass in any warp:
    // the other schedule's loops go over its chunks)
    it.thin = it.k0 < it.k1 && it.k1 - it.k0 <= Sched<T>::THIN_K;
    // four rows (columns) a lane, everything loaded before anything is reduced
    auto four = [&](const int *p, int at) { return reinterpret_cast<const int4 *>(p + at)[lane]; };
    auto least = [](int4 x) { return __reduce_min_sync(0xffffffffu, min(min(x.x, x.y), min(x.z, x.w))); };
    auto most = [](int4 x) { return __reduce_max_sync(0xffffffffu, max(max(x.x, x.y), max(x.z, x.w))); };
    const int K = int(a.g.K);
    const float need = kLeftOut<T> * sqrtf(float(K));
    const int4 va = four(a.cnt_a, it.i0), vx = four(a.cnt_x, it.j0);
    it.W = 40;  // FP32: every weight is an integer, |T| <= K 2^38
    bool skip;
    if constexpr (sizeof(T) == 8) {
        const int4 va2 = four(a.cnt2_a, it.i0), vx2 = four(a.cnt2_x, it.j0), wa = four(a.nrm_a, it.i0), wx = four(a.nrm_x, it.j0);
        // by the rows' and columns' 2-norms: |T| <= 2^(W - 16) sqrt(na nx) <= 2^62.95
        const float n2 = float(most(wa)) * float(most(wx));
        it.W = __reduce_max_sync(0xffffffffu, min(62, int(78.95f - 0.5f * log2f(n2))));
        // T's last bit: rounded once per chunk of every share
        const int per = (a.kp / BK + a.split - 1) / a.split, rounds = a.split * ((per * BK + KC - 1) / KC);
        const float last = kLastBit * __int_as_float((127 + 55 - it.W) << 23) * sqrtf(float(rounds));
        const int ca = least(va), cx = least(vx), ca2 = least(va2), cx2 = least(vx2);
        const float both = fmaxf(fmaxf(float(ca + cx - K), 4.f * float(max(ca2 + cx, ca + cx2) - K)), 16.f * float(ca2 + cx2 - K));
        skip = ca < 0 || cx < 0 || float(ca + cx - K) < need || both < need + last;
    } else {
        const int ca = least(va), cx = least(vx);
        skip = ca < 0 || cx < 0 || float(ca + cx - K) < need;
    }
    // (the reductions say to the compiler that all lanes agree: the loops over an
    // item keep their uniform registers, 1 % of the tensor time)
    it.skip = __reduce_max_sync(0xffffffffu, int(skip)) != 0;
    return it;
}

// S in FP32, |S| <= 2^26, rounded to an integer, as that integer + kIntBias modulo
// 2^32 (positive as a signed number): S is cut at bit 12, and each part added
// to 1.5 2^23 stands in the low bits of the sum.  Float-to-integer conversions
// run at a small fraction of the FP32 rate here: with them a drained
// accumulator pair took about 8000 clocks.
constexpr float kMagic = 12582912.0f;  // 1.5 2^23 = 0x4B400000
constexpr unsigned long long kIntBias = 0x4B400000ull;
__device__ __forceinline__ uint32_t biased_int(float S)
{
    const float h = fmaf(S, 1.0f / 4096.0f, kMagic);    // round(S / 2^12) + magic
    const float f = h - (kMagic + 3072.0f);             // round(S / 2^12) - 3072
    const float l = fmaf(f, -4096.0f, S);               // S - 2^12 round(S / 2^12) + magic
    // 2^12 times the magic's bits is 0 modulo 2^32
    return __float_as_uint(h) * 4096u + __float_as_uint(l);
}

// Persistent: one CTA per SM walks the items w = blockIdx.x, + gridDim.x, ...
// Warp 0 issues the TMA loads, warp 1 the MMAs, warps 2-17 drain the
// accumulators and finish C.  What bounds it: the tensor cores (36 x 2 flop
// per multiply-add of the product; 4096 x 8192 x 4096 alone 1800 TFLOP/s in FP64,
// 1440 in FP32), fed with 48 KB of digits per 512 clocks; the drains (ten half
// accumulators per 37k clocks of MMAs) go on beside them.
// Sixteen drain warps hide the latencies of the accumulators' loads.
// Issuing is close to the bound too: with the loops of warps 0 and 1 in a branch
// of one lane a stage's four MMAs, wait and commit took that lane about 700
// clocks, more than their 512 on the tensor cores (with seven and three digits,
// 4096 x 8192 x 4096: FP64 6.4 ms, FP32 1.94, so 4.96 and 1.52).  CTA pairs (256-row
// MMAs, cta_group::2) halve the X traffic but came out slower, 5.18 and 1.65 ms;
// loading the next chunk's slices into L2 ahead changed nothing.
template <typename T>
__global__ void __launch_bounds__(MMA_THREADS, 1)
digit_mma_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmX,
                 const __grid_constant__ MmaArgs<T> a)
{
    using S = Sched<T>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *xpose = base + STAGES * STAGE_BYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(xpose + EPI_WARPS * XP_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *accf = empty + STAGES;  // [2]
    uint64_t *acce = accf + 2;        // [2]
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acce + 2);
    __shared__ int abort_flag;
    __shared__ int last_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nitems = a.ntiles * a.split;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; s++) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);  // one MMA commit
        }
        for (int b = 0; b < 2; b++) {
            tc::mbar_init(&accf[b], 1);
            tc::mbar_init(&acce[b], EPI_WARPS);  // one arrival per epilogue warp
        }
        abort_flag = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) tc::tmem_alloc(tslot, 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tslot;
    volatile int *ab = &abort_flag;
    tc::pdl_wait();
    tc::pdl_launch_dependents();

    if (warp == 0) {
        if (lane == 0) {
            tc::tma_prefetch_desc(&tmA);
            tc::tma_prefetch_desc(&tmX);
        }
        // (No loop ends on a wait's result: after one that gave up nothing more
        // is issued, every further wait returns at once, and the tiles are
        // listed.  So the loops are the same for all lanes as far as the
        // compiler can tell, and addresses and descriptors stay in uniform
        // registers.)
        int n = 0;
        auto chunk = [&](auto thin, const Item &it, int kb, int ke) {
            constexpr bool TH = decltype(thin)::value;
#pragma unroll 1
            for (int j = 0; j < S::passes(TH); j++) {
                const int o1 = S::first(j + 1, TH);
                for (int o = S::first(j, TH); o < o1; o++) {
                    const int p = S::p(o, j, TH), b = S::base(j, TH);
                    const bool two = p < b - 1;
                    const int q = two ? b - 2 - p : 0;
                    for (int kk = kb; kk < ke; kk += BK, n++) {
                        const int s = n % STAGES;
                        const bool go = tc::mbar_pass(&empty[s], ((n / STAGES) & 1) ^ 1, ab, a.status, tc::TC_TIMEOUT_PRODUCER);
                        uint8_t *st = base + s * STAGE_BYTES;
                        if (tc::elect_one() && go) {
                            tc::mbar_arrive_expect_tx(&full[s], (two ? 3u : 2u) * TILE_BYTES);
                            tc::tma_load_3d(&tmA, &full[s], st, kk, it.i0, p);
                            tc::tma_load_3d(&tmX, &full[s], st + TILE_BYTES, kk, it.j0, q);
                            if (two) tc::tma_load_3d(&tmX, &full[s], st + 2 * TILE_BYTES, kk, it.j0, q + 1);
                        }
                    }
                }
            }
        };
        for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
            const Item it = digit_item(a, w, lane);
            if (it.skip) continue;
            if (S::THIN_K && it.thin) chunk(std::true_type(), it, it.k0, it.k1);
            else
                for (int kb = it.k0; kb < it.k1; kb += KC) chunk(std::false_type(), it, kb, min(kb + KC, it.k1));
        }
        __syncwarp();
        if (lane == 0) {
            // tail: wait until the MMAs released every stage, so that no
            // commit is still on its way to this CTA's barriers when it exits
            const int n0 = n;
            int ok = 1;
            for (int t = 0; t < STAGES && ok; t++, n++) {
                const int s = n % STAGES;
                const uint32_t ph = (n / STAGES) & 1;
                ok = tc::mbar_wait(&empty[s], ph ^ 1, ab, a.status, tc::TC_TIMEOUT_PRODUCER);
            }
            // after a wait that gave up: the copies still in flight land
            // before this CTA's shared memory is given away (bounded)
            if (*ab)
                for (int t = n0 > STAGES ? n0 - STAGES : 0; t < n0; t++)
                    for (int spin = 0; spin < (1 << 16) && !tc::mbar_try_wait(&full[t % STAGES], (t / STAGES) & 1); spin++) {
                    }
        }
    } else if (warp == 1) {
        const uint64_t d0 = tc::desc_kmajor_sw128(tc::smem_u32(base));
        const uint32_t idesc256 = tc::idesc_bf16_f32(BM, 256), idesc128 = tc::idesc_bf16_f32(BM, 128);
        int n = 0, cp = 0;
        auto chunk = [&](auto thin, int nk) {
            constexpr bool TH = decltype(thin)::value;
#pragma unroll 1
            for (int j = 0; j < S::passes(TH); j++, cp++) {
                const int buf = cp & 1;
                tc::mbar_pass(&acce[buf], ((cp >> 1) & 1) ^ 1, ab, a.status, tc::TC_TIMEOUT_MMA);
                tc::tc_fence_after();
                const uint32_t acc = tmem + uint32_t(buf * 256);
                const int o0 = S::first(j, TH), o1 = S::first(j + 1, TH);
                for (int o = o0; o < o1; o++) {
                    const bool two = S::p(o, j, TH) < S::base(j, TH) - 1;
                    const uint32_t d = two ? acc : acc + 128u;
                    const uint32_t idesc = two ? idesc256 : idesc128;
                    for (int kt = 0; kt < nk; kt++, n++) {
                        const int s = n % STAGES;
                        const bool go = tc::mbar_pass(&full[s], (n / STAGES) & 1, ab, a.status, tc::TC_TIMEOUT_MMA);
                        tc::tc_fence_after();
                        // the start address field counts 16-byte units: a
                        // 32-byte step along K adds 2
                        const uint64_t da = d0 + uint64_t(uint32_t(s) * (STAGE_BYTES >> 4));
                        const uint64_t db = da + uint64_t(TILE_BYTES >> 4);
                        if (tc::elect_one() && go) {
                            tc::mma_f16(d, da, db, idesc, o != o0 || kt != 0);
#pragma unroll
                            for (int kk = 1; kk < BK / 16; kk++)
                                tc::mma_f16(d, da + uint64_t(2 * kk), db + uint64_t(2 * kk), idesc, 1);
                            tc::mma_commit(&empty[s]);
                        }
                    }
                }
                if (tc::elect_one()) tc::mma_commit(&accf[buf]);
            }
        };
        for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
            const Item it = digit_item(a, w, lane);
            if (it.skip) continue;
            if (S::THIN_K && it.thin) chunk(std::true_type(), (it.k1 - it.k0) / BK);
            else
                for (int kb = it.k0; kb < it.k1; kb += KC) chunk(std::false_type(), (min(kb + KC, it.k1) - kb) / BK);
        }
        __syncwarp();
    } else {
        const int q = warp & 3;                 // TMEM lane group this warp may read
        const int cg = (warp - 2) >> 2;         // columns [32 cg, 32 cg + 32) of the tile
        const bool first = threadIdx.x == 64;   // speaks for the epilogue warps
        T *xp = reinterpret_cast<T *>(xpose + (warp - 2) * XP_BYTES);
        const uint32_t lbase = tmem + (uint32_t(q * 32) << 16) + uint32_t(cg * 32);
        int ok = 1, cp = 0;
        for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
            const Item it = digit_item(a, w, lane);
            if (it.skip || !ok) {
                if (first && atomicExch(&a.w.listed[it.tile], 1) == 0) a.w.list[atomicAdd(a.w.count, 1)] = it.tile;
                continue;
            }
            // Sums start at minus what the conversions below add: kIntBias 2^s
            // for every half accumulator of weight 2^s (modulo 2^64).
            long long T64[32];
            {
                unsigned long long bias = 0;
                for (int j = 0; j < S::passes(it.thin); j++)
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int s = it.W - 8 * (S::base(j, it.thin) + h);
                        if (s >= 0) bias += kIntBias << s;
                        else bias += h ? kIntBias : 0;
                    }
                bias *= (unsigned long long)((it.k1 - it.k0 + KC - 1) / KC);
#pragma unroll
                for (int c = 0; c < 32; c++) T64[c] = static_cast<long long>(0ull - bias);
            }
            // T += S 2^s over the 32 columns at tb
            auto add_half = [&](uint32_t tb, int s) {
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += 8) {
                    uint32_t r[8];
                    tc::tmem_ld8(tb + c0, r);
                    tc::tmem_ld_wait();
                    if (s >= 32) {
#pragma unroll
                        for (int e = 0; e < 8; e++)
                            T64[c0 + e] += static_cast<long long>(
                                static_cast<unsigned long long>(biased_int(__uint_as_float(r[e])) << (s - 32)) << 32);
                    } else {
                        const uint32_t m = 1u << s;
#pragma unroll
                        for (int e = 0; e < 8; e++)
                            T64[c0 + e] += static_cast<long long>(static_cast<unsigned long long>(biased_int(__uint_as_float(r[e]))) * m);
                    }
                }
            };
            for (int kb = it.k0; kb < it.k1 && ok; kb += KC) {
#pragma unroll 1
                for (int j = 0; j < S::passes(it.thin); j++, cp++) {
                    const int buf = cp & 1;
                    ok = tc::mbar_wait(&accf[buf], (cp >> 1) & 1, ab, a.status, tc::TC_TIMEOUT_EPILOGUE);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint32_t tb = lbase + uint32_t(buf * 256);
                    const int s1 = it.W - 8 * S::base(j, it.thin), s2 = s1 - 8;
                    if (sizeof(T) == 4 || s1 >= 0) add_half(tb, s1);
                    if (sizeof(T) == 4 || s2 >= 0) {
                        add_half(tb + 128, s2);
                    } else {
                        // a weight below the sums' last bit: scaled, and both
                        // halves rounded as one number when neither is above it
                        // (at most 2^23: W is at most 62)
                        const float m1 = s1 < 0 ? __int_as_float((127 + s1) << 23) : 0.f;
                        const float m2 = __int_as_float((127 + s2) << 23);
#pragma unroll
                        for (int c0 = 0; c0 < 32; c0 += 8) {
                            uint32_t r1[8], r2[8];
                            tc::tmem_ld8(tb + c0, r1);
                            tc::tmem_ld8(tb + 128 + c0, r2);
                            tc::tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 8; e++)
                                T64[c0 + e] += int(biased_int(fmaf(__uint_as_float(r1[e]), m1, __uint_as_float(r2[e]) * m2)));
                        }
                    }
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&acce[buf]);
                }
            }
            // one answer for all sixteen warps (a bounded wait that gave up in
            // any of them leaves the tile to the last pass): the barrier's own
            // AND, since warps 0 and 1, which take no part in it, may set the
            // flag while these read it
            ok = tc::bar_and(1, 32 * EPI_WARPS, ok && *ab == 0);
            if (!ok) {
                if (first && atomicExch(&a.w.listed[it.tile], 1) == 0) a.w.list[atomicAdd(a.w.count, 1)] = it.tile;
                continue;
            }
            const int row = q * 32 + lane;
            if (a.split > 1) {
                // the partial sums of this share are added into the tile's
                // (integers: in any order); the CTA that comes last finishes
                auto *o = reinterpret_cast<unsigned long long *>(a.Tg) + size_t(it.tile) * (BM * BM) + row + cg * 32 * BM;
#pragma unroll
                for (int c = 0; c < 32; c++) atomicAdd(o + c * BM, static_cast<unsigned long long>(T64[c]));
                __threadfence();
                asm volatile("bar.sync 1, %0;" ::"n"(32 * EPI_WARPS) : "memory");
                if (first) last_flag = atomicAdd(&a.w.done[it.tile], 1) == a.split - 1;
                asm volatile("bar.sync 1, %0;" ::"n"(32 * EPI_WARPS) : "memory");
                const bool last = last_flag != 0;
                if (!last) continue;
                __threadfence();
#pragma unroll
                for (int c = 0; c < 32; c++) T64[c] = static_cast<long long>(__ldcg(o + c * BM));
            }
            const DigitGemm<T> &g = a.g;
            const int64_t i = int64_t(it.i0) + row, jb = int64_t(it.j0) + cg * 32;
            const int ei = a.e_a[i] - it.W;
            if (g.cl) {
                // lanes hold consecutive rows: 256-byte accesses
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += 4) {
                    T old[4];
                    bool in[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int64_t j = jb + c0 + u;
                        in[u] = i < g.M && j < g.N && !(g.tri && j > i);
                        old[u] = in[u] ? g.C[i + j * g.ldc] : T(0);
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int64_t j = jb + c0 + u;
                        const T v = scale_sum(T(0), T64[c0 + u], ei + a.e_x[j]);
                        const T r = (g.alpha == T(1)) ? old[u] - v : g.alpha * old[u] - v;
                        if (in[u]) g.C[i + j * g.ldc] = r;
                    }
                }
            } else {
                // row-major: 32 bytes of a row at a time, through the warp's
                // transpose buffer
                constexpr int NC = int(32 / sizeof(T)), LX = NC + 1, LPR = 32 / NC;
                static_assert(32 * LX * sizeof(T) <= XP_BYTES, "transpose buffer");
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += NC) {
#pragma unroll
                    for (int u = 0; u < NC; u++)
                        xp[lane * LX + u] = scale_sum(T(0), T64[c0 + u], ei + a.e_x[jb + c0 + u]);
                    __syncwarp();
                    T old[NC];
                    const int64_t j = jb + c0 + lane % NC;
#pragma unroll
                    for (int u = 0; u < NC; u++) {
                        const int64_t ii = int64_t(it.i0) + q * 32 + lane / NC + u * LPR;
                        const bool in = ii < g.M && j < g.N && !(g.tri && j > ii);
                        old[u] = in ? g.C[j + ii * g.ldc] : T(0);
                    }
#pragma unroll
                    for (int u = 0; u < NC; u++) {
                        const int64_t ii = int64_t(it.i0) + q * 32 + lane / NC + u * LPR;
                        const bool in = ii < g.M && j < g.N && !(g.tri && j > ii);
                        const T v = xp[(lane / NC + u * LPR) * LX + lane % NC];
                        if (in) g.C[j + ii * g.ldc] = (g.alpha == T(1)) ? old[u] - v : g.alpha * old[u] - v;
                    }
                    __syncwarp();
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, 512);
    }
}

// ---- pass 3: the listed tiles on the CUDA cores ------------------------------------

// A listed tile is cut into parts of G::BM x G::BN, handed out one by one: with a
// fixed share per CTA the last round left half the SMs idle while others took two
// parts (512 x 8192 x 512 FP64, all tiles listed, 1024 parts: 4.22 ms instead of
// 3.66).
template <typename T, bool AM, bool BC, bool CL, class G>
__global__ void __launch_bounds__(G::NT)
digit_fallback_kernel(const T *__restrict__ A, const T *__restrict__ B, T *__restrict__ C, DigitGemm<T> g, TileWords w, int nMt, int nNt)
{
    constexpr int FB = G::BM, PER = BM / FB;
    __shared__ __align__(16) T smem[gemm_tile_smem<T, G>()];
    __shared__ int part;
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    const int n = *w.count * PER * PER;
    for (int t = blockIdx.x; t < n;) {
        const int tile = w.list[t / (PER * PER)], sub = t % (PER * PER);
        if (threadIdx.x == 0) part = int(gridDim.x) + atomicAdd(w.next, 1);
        int m_blk, n_blk;
        digit_tile(tile, nMt, nNt, g.tri, m_blk, n_blk);
        const int64_t i0 = int64_t(m_blk) * BM + (sub % PER) * FB, j0 = int64_t(n_blk) * BM + (sub / PER) * FB;
        if (i0 < g.M && j0 < g.N && !(g.tri && j0 > i0 + FB - 1))
            gemm_tile<T, AM, BC, CL, G>(smem, i0, j0, g.M, g.N, g.K, A, g.lda, B, g.ldb, C, g.ldc, g.alpha, g.tri);
        __syncthreads();
        t = part;
        __syncthreads();
    }
}

// ---- host ------------------------------------------------------------------------

// SMs of the current device.
inline int sm_count()
{
    static PerDeviceOnce n;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    int v = n.done[dev].load(std::memory_order_relaxed);
    if (!v && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) n.done[dev].store(v);
    return v > 0 ? v : 152;
}

// G: parts of the CUDA-core update's own tiles, or of a quarter of them where
// those would not fill the SMs (a part of 64 x 64 x 64 FP64 takes its SM 69 us
// whatever the others do).
template <typename T, class G>
int launch_fallback(const DigitGemm<T> &g, const TileWords &w, int nMt, int nNt, int64_t ntiles, cudaStream_t s)
{
    void (*k)(const T *, const T *, T *, DigitGemm<T>, TileWords, int, int) = nullptr;
    if (g.am && g.bc && g.cl) k = digit_fallback_kernel<T, true, true, true, G>;
    else if (g.am && !g.bc && !g.cl) k = digit_fallback_kernel<T, true, false, false, G>;
    else if (!g.am && g.bc && g.cl) k = digit_fallback_kernel<T, false, true, true, G>;
    else if (!g.am && !g.bc && !g.cl) k = digit_fallback_kernel<T, false, false, false, G>;
    else if (g.am && !g.bc && g.cl) k = digit_fallback_kernel<T, true, false, true, G>;    // P P^T
    else if (!g.am && g.bc && !g.cl) k = digit_fallback_kernel<T, false, true, false, G>;  // the same, stored transposed
    if (!k) return GB_STATUS_CUDA_ERROR;
    constexpr int PER = BM / G::BM;
    const int64_t parts = ntiles * PER * PER, most = int64_t(2) * sm_count() * (GemmTile<T>::NT / G::NT);
    return check(launch_pdl(k, dim3((unsigned)(parts < most ? parts : most)), dim3(G::NT), 0, s, g.A, g.B, g.C, g, w, nMt, nNt));
}

template <typename T>
int digit_piece(const DigitGemm<T> &g, char *ws, size_t ws_bytes, int split, cudaStream_t s)
{
    constexpr int P = Fmt<T>::P;
    const int64_t mp = up(g.M, BM), np = up(g.N, BM), kp = up(g.K, BK);
    const int nMt = int(mp / BM), nNt = int(np / BM);
    const int64_t nt = digit_tiles(nMt, nNt, g.tri);
    size_t off = 0;
    auto take = [&](size_t b) {
        char *p = ws + off;
        off += (b + 255) & ~size_t(255);
        return p;
    };
    __nv_bfloat16 *da = reinterpret_cast<__nv_bfloat16 *>(take(size_t(2) * P * mp * kp));
    __nv_bfloat16 *dx = g.tri ? da : reinterpret_cast<__nv_bfloat16 *>(take(size_t(2) * P * np * kp));
    long long *Tg = reinterpret_cast<long long *>(take(split > 1 ? size_t(nt) * BM * BM * 8 : 0));
    // (128-row arrays of int4 reads: each starts on a 256-byte boundary)
    int *ea = reinterpret_cast<int *>(take(4 * size_t(mp))), *ca = reinterpret_cast<int *>(take(4 * size_t(mp)));
    int *ca2 = reinterpret_cast<int *>(take(4 * size_t(mp))), *na = reinterpret_cast<int *>(take(4 * size_t(mp)));
    int *ex = g.tri ? ea : reinterpret_cast<int *>(take(4 * size_t(np)));
    int *cx = g.tri ? ca : reinterpret_cast<int *>(take(4 * size_t(np)));
    int *cx2 = g.tri ? ca2 : reinterpret_cast<int *>(take(4 * size_t(np)));
    int *nx = g.tri ? na : reinterpret_cast<int *>(take(4 * size_t(np)));
    int *words = reinterpret_cast<int *>(take(4 * (3 * size_t(nt) + 3)));
    const TileWords w{words, words + 1, words + 2, words + 2 + nt, words + 2 + 2 * nt};
    if (off > ws_bytes || nt * split > 0x3fffffff) return GB_STATUS_CUDA_ERROR;

    CUtensorMap ta, tx;
    {
        const uint32_t box[3] = {BK, BM, 1};
        uint64_t dims[3] = {uint64_t(kp), uint64_t(mp), uint64_t(P)};
        uint64_t strides[2] = {uint64_t(kp) * 2, uint64_t(mp) * uint64_t(kp) * 2};
        GB_TRY(encode_tmap(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, da, dims, strides, box));
        if (!g.tri) {
            dims[1] = uint64_t(np);
            strides[1] = uint64_t(np) * uint64_t(kp) * 2;
        }
        GB_TRY(encode_tmap(&tx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, dx, dims, strides, box));
    }
    {
        LaunchScope ls(KK_CONVERT, s, 0,
                       (sizeof(T) + 2.0 * P) * (double(g.M) + (g.tri ? 0.0 : double(g.N))) * double(g.K));
        DigitSrc<T> sa{g.A, g.lda, g.am ? 0 : 1, int(g.M), int(mp), da, ea, ca, ca2, na};
        DigitSrc<T> sx{g.B, g.ldb, g.bc ? 1 : 0, int(g.N), int(np), dx, ex, cx, cx2, nx};
        const int ab = int(mp / DROWS), xb = g.tri ? 0 : int(np / DROWS);
        const int64_t ktiles = kp / BK;
        int cl = 1;
        while (cl < kMaxCluster && ktiles >= (int64_t(ab + xb) * cl < 304 ? 2 : 4) * cl && int64_t(ab + xb) * cl < 1216) cl *= 2;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(ab + xb), (unsigned)cl);
        cfg.blockDim = dim3(DTHREADS);
        cfg.stream = s;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = 1;
        attr[1].val.clusterDim.y = (unsigned)cl;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        GB_CUDA(cudaLaunchKernelEx(&cfg, digits_kernel<T>, sa, sx, ab, int(g.K), int(kp), words, int(2 * nt + 2),
                                   reinterpret_cast<ulonglong2 *>(Tg), split > 1 ? nt * (BM * BM / 2) : int64_t(0)));
    }
    {
        static PerDeviceOnce attr;
        GB_TRY(smem_attr_once(attr, digit_mma_kernel<T>, MMA_SMEM));
        constexpr double pairs = P * (P + 1) / 2;
        LaunchScope ls(KK_GEMM_TC, s, 2.0 * pairs * double(nt) * BM * BM * double(kp), 8.0 * double(nt) * BM * BM);
        MmaArgs<T> a{g, Tg, ca, cx, ca2, cx2, na, nx, ea, ex, w, int(kp), nMt, nNt, int(nt), split, words + 3 * nt + 2};
        const int64_t items = nt * split;
        GB_CUDA(launch_pdl(digit_mma_kernel<T>, dim3((unsigned)(items < sm_count() ? items : sm_count())), dim3(MMA_THREADS),
                           MMA_SMEM, s, ta, tx, a));
    }
    LaunchScope ls(KK_GEMM_SIMT, s, 0, 0);
    constexpr int PER = BM / GemmTile<T>::BM;
    if (nt * PER * PER < 2 * sm_count()) return launch_fallback<T, GemmTileSmall<T>>(g, w, nMt, nNt, nt, s);
    return launch_fallback<T, GemmTile<T>>(g, w, nMt, nNt, nt, s);
}

cudaMemPool_t digit_pool()
{
    static cudaMemPool_t pool[64] = {nullptr};
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(mu);
    if (!pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p;
        if (cudaMemPoolCreate(&p, &props) != cudaSuccess) return nullptr;
        // freed work spaces up to this many bytes stay with the pool, the
        // rest goes back to the driver when the stream is next synchronised
        uint64_t thr = kWsCap + kWsCap / 4;
        cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &thr);
        pool[dev] = p;
    }
    return pool[dev];
}

}  // namespace

bool DigitWorkspace::usable()
{
    if (state_ == 0) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        state_ = cudaStreamIsCapturing(s_, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone ? -1 : 1;
    }
    return state_ > 0;
}

char *DigitWorkspace::get(size_t bytes)
{
    if (!usable()) return nullptr;
    if (size_ >= bytes) return p_;
    release();
    cudaMemPool_t pool = digit_pool();
    void *p = nullptr;
    if (!pool || cudaMallocFromPoolAsync(&p, bytes, pool, s_) != cudaSuccess) {
        cudaGetLastError();  // no memory: the CUDA-core update needs none
        state_ = -1;
        return nullptr;
    }
    p_ = static_cast<char *>(p);
    size_ = bytes;
    return p_;
}

void DigitWorkspace::release()
{
    if (p_) cudaFreeAsync(p_, s_);
    p_ = nullptr;
    size_ = 0;
}

void digit_pool_trim()
{
    cudaMemPool_t pool = digit_pool();
    if (pool) cudaMemPoolTrimTo(pool, 0);
}

// FP64: from K = 64 on at every M and N: measured, 64 x 32 x 64 takes 30 us
// (CUDA cores 70), 64 x 256 x 512 36 (527), 2048 x 8192 x 64 0.19 ms (1.78),
// 2048 x 8192 x 2048 1.59 ms (55).  FP32: from K = 128 and 64 x 256 outputs, or K =
// 512, where they are the faster ones: 64 x 256 x 128 29 us (31), 32 x 32 x 512
// 29 (68), 512 x 8192 x 128 43 (90), 2048 x 8192 x 2048 0.62 ms (2.6).
template <typename T>
bool digit_gemm_wanted(int64_t M, int64_t N, int64_t K, int)
{
    if (sizeof(T) == 8) return K >= 64;
    return K >= 128 && (double(M) * double(N) >= 16384.0 || K >= 512);
}

template <typename T>
size_t digit_gemm_bytes(int64_t M, int64_t N, int64_t K, int tri)
{
    return plan_piece<Fmt<T>::P>(M, N, K, tri).bytes;
}

template <typename T>
int launch_digit_gemm(const DigitGemm<T> &g, char *ws, size_t ws_bytes, cudaStream_t s)
{
    const Piece pc = plan_piece<Fmt<T>::P>(g.M, g.N, g.K, g.tri);
    return for_pieces(pc, g.M, g.N, g.K, g.tri, [&](int64_t i, int64_t j, int64_t k, int64_t m, int64_t n, int64_t kk, int split) {
        DigitGemm<T> d = g;
        d.M = m;
        d.N = n;
        d.K = kk;
        d.A = g.am ? g.A + i + k * g.lda : g.A + k + i * g.lda;
        d.B = g.bc ? g.B + k + j * g.ldb : g.B + j + k * g.ldb;
        d.C = g.cl ? g.C + i + j * g.ldc : g.C + j + i * g.ldc;
        if (k > 0) d.alpha = T(1);
        return digit_piece<T>(d, ws, ws_bytes, split, s);
    });
}

template bool digit_gemm_wanted<double>(int64_t, int64_t, int64_t, int);
template bool digit_gemm_wanted<float>(int64_t, int64_t, int64_t, int);
template size_t digit_gemm_bytes<double>(int64_t, int64_t, int64_t, int);
template size_t digit_gemm_bytes<float>(int64_t, int64_t, int64_t, int);
template int launch_digit_gemm<double>(const DigitGemm<double> &, char *, size_t, cudaStream_t);
template int launch_digit_gemm<float>(const DigitGemm<float> &, char *, size_t, cudaStream_t);

}  // namespace gb
