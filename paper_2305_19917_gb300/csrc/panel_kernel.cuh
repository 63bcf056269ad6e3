// (internal header) Diagonal-block solve of many rows in one launch: the paper's TS task
// (Section IV, stages 1 and 3) for a block of up to kPanelRows rows and any
// number of right-hand sides of the canonical view, each CTA with CW of them.
//
// Used where the right-hand sides are few enough that the chain of 64-row
// blocks (a diagonal kernel and an update launch each, on a handful of SMs)
// is the time: a CTA takes only CW = 1..8 right-hand sides, so that 64 of
// them already occupy 64 SMs, and walks the whole block by itself, without a
// launch or a grid-wide wait in between.
//
// Left-looking in 32-row blocks: warp w of the CTA owns the block rows w,
// w + NW, ...; lane l holds row l of the block, its CW right-hand sides and
// its row of the block's triangle in registers.  A block row takes its
// updates from the solved blocks in order (32 x 32 tiles of Mv streamed
// through a ring of asynchronous copies of its own), then solves its triangle
// by substitution, one step per row, x broadcast from its lane.  Each x goes
// to shared memory as soon as it is known and the next block row's warp takes
// it from there at once: X starts out as a pattern that stands for "not
// known yet", and a reader polls the value itself.  The pattern is a NaN, and
// FP64 arithmetic hands on the payload of a NaN in B or Mv: so one with this
// payload is replaced by another before it can get into X (once per block row
// where the triangle's entries are finite, else at every step).  So the critical chain is
// the substitution alone, the updates go on beside it, and the warps never
// meet at a barrier.
//
// What bounds it: FP64, the FP64 unit: one warp instruction takes 66 clocks of
// a sub-partition whatever its active lanes, dependent or not (measured; 19
// per instruction and SM with 16 warps), so a step with the multiplication by
// the inverse takes 190 clocks.  The multiplication is taken off the chain:
// the triangle's rows are scaled by the inverse beforehand (where no exponent
// is extreme) and a step is a shuffle and a multiply-add, 132 clocks.  FP32:
// 35 clocks a step, and shared-memory wavefronts.
#pragma once
#include "common.cuh"
#include "panel.cuh"
#include "tc_common.cuh"

namespace gb {
namespace {

constexpr int NB = 32;

template <typename T>
struct PanelCfg;
template <>
struct PanelCfg<double> {
    static constexpr int NW = 4, LD = NB + 2;  // warps, row stride of a tile
    static constexpr unsigned long long EMPTY = 0xFFF8DEADBEEF5A5Aull;  // X not known yet (a NaN)
    using Bits = unsigned long long;
    __device__ static Bits bits(double x) { return static_cast<Bits>(__double_as_longlong(x)); }
    __device__ static double from(Bits b) { return __longlong_as_double(static_cast<long long>(b)); }
    // x, or another NaN where its payload is EMPTY's (of either sign: arithmetic
    // may hand it on with the other one)
    __device__ static double other(double x)
    {
        const int lo = __double2loint(x), hi = __double2hiint(x);
        const bool is = lo == int(EMPTY & 0xFFFFFFFFu) && (hi & 0x7FFFFFFF) == int((EMPTY >> 32) & 0x7FFFFFFFu);
        return __hiloint2double(hi, is ? lo ^ 1 : lo);
    }
    __device__ static int field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
};
template <>
struct PanelCfg<float> {
    static constexpr int NW = 8, LD = NB + 4;
    __device__ static float other(float x) { return x; }
};

// Tiles in a warp's ring: two CTAs with their X share an SM.
template <typename T, int CW>
constexpr int panel_ring() { return sizeof(T) == 8 && CW >= 4 ? 2 : 3; }
constexpr int kSpins = 1 << 22;  // polls before a reader gives up

template <typename T, int CW>
constexpr size_t panel_smem(int nblk)
{
    using C = PanelCfg<T>;
    return sizeof(T) * (size_t(C::NW) * panel_ring<T, CW>() * NB * C::LD + size_t(nblk) * NB * CW);
}

__device__ __forceinline__ void cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
template <typename T>
__device__ __forceinline__ void cp1(T *dst, const T *src, bool in)
{
    const int n = in ? int(sizeof(T)) : 0;
    if (sizeof(T) == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(tc::smem_u32(dst)), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tc::smem_u32(dst)), "l"(src), "r"(n) : "memory");
}

// CW values of a row of X (CW sizeof(T) bytes, aligned to min(16, that)).
template <typename T, int CW>
__device__ __forceinline__ void load_x(const T *p, T (&x)[CW])
{
    constexpr int V = CW < int(16 / sizeof(T)) ? CW : int(16 / sizeof(T));
    struct alignas(V * sizeof(T)) Vec {
        T e[V];
    };
#pragma unroll
    for (int c = 0; c < CW; c += V) {
        const Vec q = *reinterpret_cast<const Vec *>(p + c);
#pragma unroll
        for (int u = 0; u < V; u++) x[c + u] = q.e[u];
    }
}
// The same once every value is there (the whole warp reads one address).
template <typename T, int CW>
__device__ __forceinline__ void await_x(const T *p, T (&x)[CW], bool &gave_up)
{
    for (int spin = 0;; spin++) {
        bool ok = true;
#pragma unroll
        for (int c = 0; c < CW; c++) {
            x[c] = *const_cast<const volatile T *>(p + c);
            ok = ok && PanelCfg<T>::bits(x[c]) != PanelCfg<T>::EMPTY;
        }
        if (ok || gave_up) return;
        if (spin > kSpins) gave_up = true;
    }
}

// AM: Mv(i,k) = M[i + k lda], else M[k + i lda]; Bv(i,c) = B[i si + c sc].
// M = &A(r0, r0), B = &Bv(r0, 0).  vec: off-diagonal tiles may be copied 16
// bytes at a time.
template <typename T, int CW, bool AM, bool FWD>
__global__ void __launch_bounds__(32 * PanelCfg<T>::NW)
panel_kernel(const T *__restrict__ M, int64_t lda, T *__restrict__ B, int64_t si, int64_t sc, int nr, int64_t ncols,
             T alpha, int unit, int vec)
{
    using C = PanelCfg<T>;
    constexpr int NW = C::NW, NS = panel_ring<T, CW>(), LD = C::LD, TILE = NB * LD, V = int(16 / sizeof(T));
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *ring = reinterpret_cast<T *>(smem_raw);
    T *Xs = ring + NW * NS * TILE;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nblk = (nr + NB - 1) / NB;
    ring += warp * NS * TILE;
    const int64_t c0 = int64_t(blockIdx.x) * CW;
    const int ncb = int(ncols - c0 < CW ? ncols - c0 : CW);

    __shared__ int solved;  // FP32: blocks whose X is in shared memory
    if constexpr (sizeof(T) == 8)
        for (int x = threadIdx.x; x < nblk * NB * CW; x += 32 * NW) Xs[x] = C::from(C::EMPTY);
    if (threadIdx.x == 0) solved = 0;
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    __syncthreads();

    // Tiles hold Mv in natural orientation (a backward solve reads them
    // mirrored): block b covers natural rows [nat(b), nat(b) + 32).
    auto nat = [&](int b) { return FWD ? b * NB : nr - (b + 1) * NB; };
    // element (row i, column k) of a tile
    auto at = [&](int i, int k) { return AM ? k * LD + i : i * LD + k; };
    auto load_tile = [&](int b, int kb, T *t) {
        const int ri = nat(b), ci = nat(kb);
        const T *src = AM ? M + ri + int64_t(ci) * lda : M + ci + int64_t(ri) * lda;
        if (vec && ri >= 0 && ri + NB <= nr) {
            constexpr int PER = NB / V;  // copies per contiguous run
#pragma unroll
            for (int q = 0; q < NB * PER / 32; q++) {
                const int idx = lane + 32 * q, f = (idx % PER) * V, s = idx / PER;
                cp16(t + s * LD + f, src + f + int64_t(s) * lda);
            }
            return;
        }
#pragma unroll 8
        for (int s = 0; s < NB; s++) {
            const int i = AM ? lane : s, k = AM ? s : lane;  // natural, inside the tile
            const bool in = ri + i >= 0 && ri + i < nr && ci + k >= 0;
            cp1(t + s * LD + lane, in ? src + lane + int64_t(s) * lda : M, in);
        }
    };

    // the warp's tiles in order: block rows warp, warp + NW, ...; in each kb = 0 .. b - 1
    int pb = warp ? warp : NW, pk = 0, pn = 0;  // next tile to load, its number
    auto prefetch = [&]() {
        if (pb < nblk) {
            load_tile(pb, pk, ring + (pn % NS) * TILE);
            if (++pk == pb) {
                pb += NW;
                pk = 0;
            }
        }
        pn++;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int q = 0; q < NS - 1; q++) prefetch();

    int n = 0;                                  // tile number
    int known = 0;                              // blocks known to be solved
    bool gave_up = false;
    const int ln = FWD ? lane : NB - 1 - lane;  // the lane's row inside a natural tile
    for (int b = warp; b < nblk; b += NW) {
        const int i = nat(b) + ln;  // the lane's natural row
        const bool live = i >= 0 && i < nr;
        // the row's right-hand sides, triangle entries (in solution order) and
        // inverse diagonal
        T t[CW], m[NB];
#pragma unroll
        for (int c = 0; c < CW; c++)
            t[c] = (live && c < ncb) ? B[i * si + (c0 + c) * sc] : T(0);
#pragma unroll
        for (int k = 0; k < NB - 1; k++) {
            const int col = nat(b) + (FWD ? k : NB - 1 - k);
            m[k] = (live && lane > k) ? (AM ? M[i + int64_t(col) * lda] : M[col + int64_t(i) * lda]) : T(0);
        }
        const T diag = (live && !unit) ? M[i + int64_t(i) * lda] : T(1);
        const T inv = T(1) / diag;
        bool scaled = false;
        if constexpr (sizeof(T) == 8) {
            // scaled rows: exponents within 2^+-400 of the diagonal's, the
            // diagonal's within 2^+-400 (so no infinity or NaN)
            const int fd = C::field(diag);
            bool ok = fd > 623 && fd < 1423;
#pragma unroll
            for (int k = 0; k < NB - 1; k++) {
                const int df = C::field(m[k]) - fd;
                ok = ok && (m[k] == T(0) || (df > -400 && df < 400));
            }
            scaled = __all_sync(0xffffffffu, ok);
            if (scaled && !unit) {
#pragma unroll
                for (int k = 0; k < NB - 1; k++) m[k] *= inv;
            }
        }
        // the updates' sum, kept apart from t: subtracted once, it does not
        // round at t's magnitude at every step
        T acc[CW];
#pragma unroll
        for (int c = 0; c < CW; c++) acc[c] = T(0);
        for (int kb = 0; kb < b; kb++, n++) {
            asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
            __syncwarp();
            prefetch();  // into the buffer of tile n - 1, which every lane has read
            const T *tile = ring + (n % NS) * TILE;
            const T *x0 = Xs + size_t(kb) * NB * CW;
            if constexpr (sizeof(T) == 4) {
                for (int spin = 0; known <= kb && !gave_up; spin++) {
                    known = *static_cast<volatile int *>(&solved);
                    if (spin > kSpins) gave_up = true;
                }
                __threadfence_block();
            } else if (kb >= known) {
                for (int k = 0; k < NB; k++) {
                    const T a = tile[at(ln, FWD ? k : NB - 1 - k)];
                    T x[CW];
                    await_x<T, CW>(x0 + k * CW, x, gave_up);
#pragma unroll
                    for (int c = 0; c < CW; c++) acc[c] = fma(a, x[c], acc[c]);
                }
                known = kb + 1;
                continue;
            }
            // KU steps' operands are loaded before they are used
            constexpr int KU = CW <= 4 ? 8 : 4;
#pragma unroll
            for (int k0 = 0; k0 < NB; k0 += KU) {
                T a[KU], x[KU][CW];
#pragma unroll
                for (int u = 0; u < KU; u++) {
                    a[u] = tile[at(ln, FWD ? k0 + u : NB - 1 - k0 - u)];
                    load_x<T, CW>(x0 + (k0 + u) * CW, x[u]);
                }
#pragma unroll
                for (int u = 0; u < KU; u++)
#pragma unroll
                    for (int c = 0; c < CW; c++) acc[c] = fma(a[u], x[u][c], acc[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < CW; c++) t[c] = C::other(alpha * t[c] - acc[c]);
        // a reader that gave up (it cannot unless the device is broken) says
        // so in every row from there on
        if (gave_up) {
#pragma unroll
            for (int c = 0; c < CW; c++) t[c] = T(NAN);
        }
        T *xb = Xs + size_t(b) * NB * CW;
        if (scaled) {
            if (!unit) {
#pragma unroll
                for (int c = 0; c < CW; c++) t[c] *= inv;
            }
#pragma unroll
            for (int k = 0; k < NB; k++) {
                T x[CW];
#pragma unroll
                for (int c = 0; c < CW; c++) x[c] = __shfl_sync(0xffffffffu, t[c], k);
                if (lane == k) {
#pragma unroll
                    for (int c = 0; c < CW; c++) *const_cast<volatile T *>(xb + k * CW + c) = x[c];
                }
                if (k < NB - 1) {
#pragma unroll
                    for (int c = 0; c < CW; c++) {
                        const T r = fma(-m[k], x[c], t[c]);
                        t[c] = lane > k ? r : t[c];
                    }
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < NB; k++) {
                const T d = __shfl_sync(0xffffffffu, inv, k);
                T x[CW];
#pragma unroll
                for (int c = 0; c < CW; c++) x[c] = C::other(__shfl_sync(0xffffffffu, t[c], k) * d);
                if (lane == k) {
#pragma unroll
                    for (int c = 0; c < CW; c++) *const_cast<volatile T *>(xb + k * CW + c) = x[c];
                }
#pragma unroll
                for (int c = 0; c < CW; c++) {
                    const T r = k < NB - 1 ? fma(-m[k < NB - 1 ? k : 0], x[c], t[c]) : t[c];
                    t[c] = lane == k ? x[c] : (lane > k ? r : t[c]);
                }
            }
        }
        if constexpr (sizeof(T) == 8) {
            known = b + 1;  // (its own rows: the next tile starts with a __syncwarp)
        } else {
            __syncwarp();
            if (lane == 0) {
                __threadfence_block();
                *static_cast<volatile int *>(&solved) = b + 1;
            }
        }
        if (live) {
#pragma unroll
            for (int c = 0; c < CW; c++)
                if (c < ncb) B[i * si + (c0 + c) * sc] = t[c];
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <typename T, int CW, bool AM, bool FWD>
int launch_form(const Canon<T> &c, const T *M, T *B, int nr, T alpha, int vec)
{
    static PerDeviceOnce attr;
    auto kern = panel_kernel<T, CW, AM, FWD>;
    GB_TRY(smem_attr_once(attr, kern, panel_smem<T, CW>(kPanelRows<T> / NB)));
    const int64_t grid = (c.ncols + CW - 1) / CW;
    if (grid > 0x7fffffff) return GB_STATUS_CUDA_ERROR;
    LaunchScope ls(KK_DIAG, c.stream, double(nr) * nr * c.ncols, sizeof(T) * (0.5 * nr * nr + 2.0 * nr * c.ncols));
    return check(launch_pdl(kern, dim3((unsigned)grid), dim3(32 * PanelCfg<T>::NW), panel_smem<T, CW>((nr + NB - 1) / NB),
                            c.stream, M, c.lda, B, c.left ? int64_t(1) : c.ldb, c.left ? c.ldb : int64_t(1), nr, c.ncols,
                            alpha, int(c.unit), vec));
}

}  // namespace

template <typename T, int CW>
int launch_panel_cw(const Canon<T> &c, int64_t r0, int nr, T alpha)
{
    const T *M = c.A + r0 + r0 * c.lda;
    T *B = bv_ptr(c, r0, 0);
    constexpr int V = int(16 / sizeof(T));
    // a tile's runs start at multiples of 32 rows from r0 (forward) or from
    // r0 + nr (backward)
    const int vec = reinterpret_cast<uintptr_t>(M) % 16 == 0 && c.lda % V == 0 && (c.forward || nr % V == 0);
    if (c.mt) return c.forward ? launch_form<T, CW, false, true>(c, M, B, nr, alpha, vec) : launch_form<T, CW, false, false>(c, M, B, nr, alpha, vec);
    return c.forward ? launch_form<T, CW, true, true>(c, M, B, nr, alpha, vec) : launch_form<T, CW, true, false>(c, M, B, nr, alpha, vec);
}

}  // namespace gb
