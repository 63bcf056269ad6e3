// Batched uneven triangular solves in one persistent launch: "n instances of
// TS" (Section IV, many right-hand sides) generalised to many independent
// problems of different order and width.
//
// Work units are (instance, chunk of right-hand sides), 32 wide in FP32, 16, 8, 4, 2
// or 1 in FP64 (width_of); sorted by cost (largest first), the first ones go to
// the teams by number, the others through a device-side work queue (atomic
// tickets; no CTA waits on another).  A unit is solved by the blocked model of
// Section V-C in left-looking order on 32-row blocks, X in shared memory, by a
// team of warps: warp w of n owns the block rows w, w + n, ..., each taking its
// updates from the solved blocks as these are published (no barrier inside a
// unit).  The more warps share a unit, the more of their time goes into waiting
// for its chain of blocks; but X has to stay in shared memory.  So teams are as
// small as that allows: the four warps of a CTA for orders above 256, two above
// 128, one below (half these orders with tile 2; FP32 batches that would leave SMs
// idle take larger teams, team_order), the CTA's X space divided among its teams.  Instances of order above KMAX are solved by the
// regular driver.
//
// A lane holds one right-hand side and its rows of the block in registers, so
// that the 32 x 32 triangle is solved by multiply-adds on independent rows,
// without shuffles of partial sums or lanes masked off: in FP64, where an
// instruction takes 66 clocks of its sub-partition whatever its active lanes
// and the multiply-adds are the time, a block's triangle takes 18 instructions
// per right-hand side instead of the 64 of a substitution with one row per
// lane.  FP64: 16 right-hand sides times the two halves of the rows (odd and
// even), or fewer times more parts, Mv read from L1 / L2 as it is needed (the
// loads hide behind the arithmetic, of narrow units behind each other).  FP32:
// 32 right-hand sides, tiles of Mv through a ring of asynchronous copies, packed
// multiply-adds (wide_tile.cuh); two CTAs of four warps fill an SM's shared
// memory, and the latencies that eight warps leave open are the time.  Measured,
// 4096 uneven instances (m log-uniform in [16, 512], n in [1, 256]): FP64 22.2 ->
// 16.0 ms (12.9 at the unit's peak), FP32 1.80 -> 1.29 ms.  With units always 16 wide
// small or narrow FP64 batches were up to 4.5 times slower than with one row per
// lane, 8 warps a unit (644 instances of order <= 128 and <= 5 right-hand sides 363 us
// against 81).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>
#include "common.cuh"
#include "wide_tile.cuh"

namespace gb {

namespace {

constexpr int KMAX = 512;  // largest order solved in shared memory
constexpr int NBB = 32;    // diagonal block
constexpr int NW = 4;      // warps per CTA
constexpr int NT = 32 * NW;

template <typename T>
constexpr int kChunk = sizeof(T) == 8 ? 16 : 32;  // right-hand sides per unit

template <typename T>
constexpr int kStride = sizeof(T) == 8 ? 16 : 33;  // row stride of X in shared memory (FP32: odd, read along rows too)

template <typename T>
struct Unit {
    const T *A;   // A of the instance
    T *B;         // B of the instance, offset to the chunk's first right-hand side
    int64_t lda, ldb;
    int k;        // order of the triangle
    int cw;       // right-hand sides in this chunk (<= CW)
    int flags;    // bit0 mt, bit1 rev (backward), bit2 unit diag, bit3 left
    T alpha;
};

// Who solves a unit: warp `wid` of `nwu`, X of the unit at Xs, blocks solved so
// far counted in *solved.
template <typename T>
struct Team {
    int wid, nwu;
    T *Xs;
    T *ring;       // FP32: the warp's two tiles
    T *inv;        // FP32: the warp's 32 inverse diagonal entries, and the entries
    int *solved;
};
// Until block kb of the unit is solved (bounded).
__device__ __forceinline__ void await_block(int *solved, int kb, int &known, bool &gave_up)
{
    for (int spin = 0; known <= kb && !gave_up; spin++) {
        known = *static_cast<volatile int *>(solved);
        if (spin > wide::kSpins) gave_up = true;
    }
    __threadfence_block();
}
__device__ __forceinline__ void publish_block(int *solved, int b)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        __threadfence_block();
        *static_cast<volatile int *>(solved) = b + 1;
    }
    __syncwarp();
}

constexpr int XLD = kStride<float>;

// FP32, in solution order (a backward problem by negative strides), so that
// one version of the unrolled steps serves every form: with one for each of
// the four (rows or columns of A contiguous, forward or backward) instruction
// fetch was the largest stall.
__device__ __forceinline__ void solve_unit(const Unit<float> &u, const Team<float> &tm)
{
    using namespace wide;
    const int lane = threadIdx.x & 31, k = u.k, nblk = (k + NB - 1) / NB;
    const bool mt = u.flags & 1, rev = u.flags & 2, unitd = u.flags & 4, left = u.flags & 8;
    int64_t sr = mt ? u.lda : 1, sc = mt ? 1 : u.lda, br = left ? 1 : u.ldb;
    const int64_t bc = left ? u.ldb : 1;
    const float *A = u.A;
    float *B = u.B;
    if (rev) {
        A += int64_t(k - 1) * (sr + sc);
        B += int64_t(k - 1) * br;
        sr = -sr;
        sc = -sc;
        br = -br;
    }
    // A tile's copies run along A's contiguous dimension: 32 rows of a column,
    // or (mt) 8 columns of 4 rows, which spreads the columns' stores over the
    // banks.  Lane's entry (li, lk) of copy (x, y): row li + 4 x, column lk + 8 y,
    // or row li, column x.
    const int li = mt ? lane >> 3 : lane, lk = mt ? lane & 7 : 0;
    const int64_t lsrc = li * sr + lk * sc;
    const int ldst = lk * WLD + li;
    auto load_tile = [&](int b, int kb, float *t) {
        const float *src = A + int64_t(b) * NB * sr + int64_t(kb) * NB * sc + lsrc;
        float *dst = t + ldst;
        if (kb < b && (b + 1) * NB <= k) {
            if (mt) {
#pragma unroll 4
                for (int y = 0; y < 4; y++)
#pragma unroll
                    for (int x = 0; x < 8; x++) cp4(dst + 8 * y * WLD + 4 * x, src + (4 * x * sr + 8 * y * sc), true);
            } else {
#pragma unroll 8
                for (int x = 0; x < NB; x++) cp4(dst + x * WLD, src + x * sc, true);
            }
            return;
        }
        // the last rows, and the strict triangle
        const int rows = k - b * NB;
        for (int s = 0; s < NB; s++) {
            const int x = mt ? 4 * (s & 7) : 0, y = mt ? 8 * (s >> 3) : s;
            const int i = li + x, c = lk + y;
            const bool in = i < rows && (kb < b || c < i);
            cp4(dst + y * WLD + x, in ? src + (x * sr + y * sc) : u.A, in);
        }
    };
    // the warp's tiles in order: block rows wid, wid + nwu, ...; in each kb = 0 .. b
    int pb = tm.wid, pk = 0, pn = 0;
    auto prefetch = [&]() {
        if (pb < nblk) {
            load_tile(pb, pk, tm.ring + (pn & 1) * TILE);
            if (pk == pb) {
                pb += tm.nwu;
                pk = 0;
            } else {
                pk++;
            }
        }
        pn++;
        commit();
    };
    prefetch();
    int n = 0, known = 0;
    bool gave_up = false;
    for (int b = tm.wid; b < nblk; b += tm.nwu) {
        const int r0 = b * NB, rows = min(NB, k - r0);
        // the rows' right-hand sides into their place in X
        float *xs = tm.Xs + size_t(b) * NB * XLD;
        {
            const float *src = B + int64_t(r0) * br + (left ? lane * br : lane * bc);
            const int64_t step = left ? bc : br;
            const int ds = left ? 1 : XLD;
            float *dst = xs + lane * (left ? XLD : 1);
            const int cnt = left ? u.cw : rows;
            const bool in = left ? lane < rows : lane < u.cw;
            // (what the copies leave out is zero)
#pragma unroll 8
            for (int x = 0; x < NB; x++) cp4(dst + x * ds, (in && x < cnt) ? src + x * step : u.A, in && x < cnt);
        }
        commit();
        {
            const float dg = (!unitd && lane < rows) ? A[int64_t(r0 + lane) * (sr + sc)] : 1.f;
            __syncwarp();
            tm.inv[lane] = 1.f / dg;
            tm.inv[NB + lane] = dg;
        }
        float *xb = xs + lane;
        Sum<true> sum;
        sum.clear();
        for (int kb = 0; kb < b; kb++, n++) {
            wait_all();
            __syncwarp();
            prefetch();  // into the buffer of tile n - 1, which every lane has read
            if (tm.nwu > 1) await_block(tm.solved, kb, known, gave_up);
            sum.update<XLD>(tm.ring + (n & 1) * TILE, tm.Xs + size_t(kb) * NB * XLD + lane);
        }
        wait_all();
        __syncwarp();
        prefetch();
        substitute<true, true, XLD>(sum.t, tm.ring + (n & 1) * TILE, tm.inv, xb, 1.f);
        n++;
        // a reader that gave up (it cannot unless the device is broken) says
        // so in every row from there on
        if (gave_up) {
            for (int i = 0; i < NB; i++) xb[i * XLD] = NAN;
        }
        publish_block(tm.solved, b);
        {
            float *dst = B + int64_t(r0) * br + (left ? lane * br : lane * bc);
            const int64_t step = left ? bc : br;
            const int ds = left ? 1 : XLD;
            const float *src = xs + lane * (left ? XLD : 1);
            const int cnt = left ? u.cw : rows;
            if (left ? lane < rows : lane < u.cw) {
#pragma unroll 8
                for (int x = 0; x < cnt; x++) dst[x * step] = u.alpha * src[x * ds];
            }
        }
    }
    wait_all();
    __syncwarp();  // X, the ring and the inverses are free for the next unit
}

// FP64, in solution order (a backward problem by negative strides): G lanes share
// a right-hand side, lane l holding rows G q + l / (32 / G) of the block for right-
// hand side l % (32 / G).  So a unit's instructions are as many as its right-hand
// sides are wide, 16, 8, 4 or 1 of them: G = 2, 4, 8, 32.
template <int G>
__device__ __forceinline__ void solve_unit(const Unit<double> &u, const Team<double> &tm)
{
    constexpr int CW = kChunk<double>, W = 32 / G, NQ = NBB / G;
    const int lane = threadIdx.x & 31, h = lane / W, col = lane % W;
    const int k = u.k, nblk = (k + NBB - 1) / NBB;
    const bool mt = u.flags & 1, rev = u.flags & 2, unitd = u.flags & 4, left = u.flags & 8;
    int64_t sr = mt ? u.lda : 1, sc = mt ? 1 : u.lda, br = left ? 1 : u.ldb;
    const double *A = u.A;
    double *B = u.B + col * (left ? u.ldb : 1);
    if (rev) {
        A += int64_t(k - 1) * (sr + sc);
        B += int64_t(k - 1) * br;
        sr = -sr;
        sc = -sc;
        br = -br;
    }
    const bool incol = col < u.cw;
    int known = 0;
    bool gave_up = false;
    for (int b = tm.wid; b < nblk; b += tm.nwu) {
        const int r0 = b * NBB, nv = min(NBB, k - r0), nq = (nv + G - 1) / G;
        // entry (row G q + h, column) of the block row; a row past the last one
        // reads the last one (its results are not used)
        const double *Ar = A + int64_t(r0 + h) * sr;
        auto row = [&](const double *p, int q) { return p[int64_t(min(G * q, nv - 1 - h)) * sr]; };
        if (G >= 8 && lane < nv) {
            // a narrow unit is a chain of latencies: the triangle's lines on their way
            const double *d = A + int64_t(r0) * (sr + sc) + lane * (mt ? sr : sc);
            asm volatile("prefetch.global.L1 [%0];" ::"l"(d));
            if (nv > 16) asm volatile("prefetch.global.L1 [%0];" ::"l"(d + 16 * (mt ? sc : sr)));
        }
        double t[NQ], acc[NQ];
#pragma unroll
        for (int q = 0; q < NQ; q++) {
            t[q] = (incol && G * q + h < nv) ? B[int64_t(r0 + G * q + h) * br] : 0.0;
            acc[q] = 0.0;
        }
        const double inv = (!unitd && lane < nv) ? 1.0 / A[int64_t(r0 + lane) * (sr + sc)] : 1.0;
        for (int kb = 0; kb < b; kb++) {
            if (tm.nwu > 1) await_block(tm.solved, kb, known, gave_up);
            const double *x0 = tm.Xs + size_t(kb) * NBB * CW + col;
            const double *ac = Ar + int64_t(kb) * NBB * sc;
            constexpr int U = G <= 4 ? 2 : 8;  // steps whose entries are loaded at once
            if (nv == NBB) {
#pragma unroll U
                for (int kk = 0; kk < NBB; kk++) {
                    const double x = x0[kk * CW];
                    double a[NQ];
#pragma unroll
                    for (int q = 0; q < NQ; q++) a[q] = ac[int64_t(G * q) * sr + kk * sc];
#pragma unroll
                    for (int q = 0; q < NQ; q++) acc[q] = fma(a[q], x, acc[q]);
                }
            } else if (G >= 8 || nv > 24) {
#pragma unroll 1
                for (int k0 = 0; k0 < NBB; k0 += U) {
                    double x[U], a[U][NQ];
#pragma unroll
                    for (int i = 0; i < U; i++) {
                        x[i] = x0[(k0 + i) * CW];
#pragma unroll
                        for (int q = 0; q < NQ; q++) a[i][q] = row(ac + (k0 + i) * sc, q);
                    }
#pragma unroll
                    for (int q = 0; q < NQ; q++)
                        if (q < nq) {
#pragma unroll
                            for (int i = 0; i < U; i++) acc[q] = fma(a[i][q], x[i], acc[q]);
                        }
                }
            } else {
                // few rows: their entries only
#pragma unroll 1
                for (int kk = 0; kk < NBB; kk++) {
                    const double x = x0[kk * CW];
                    const double *p = ac + kk * sc;
#pragma unroll
                    for (int g = 0; g < NQ; g += 4) {
                        if (g >= nq) break;
#pragma unroll
                        for (int q = g; q < (g + 4 < NQ ? g + 4 : NQ); q++)
                            if (q < nq) acc[q] = fma(row(p, q), x, acc[q]);
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NQ; q++) t[q] -= acc[q];
        // the triangle: x_k by the lanes of its row's group, the rows below it by all
        const double *ad = Ar + int64_t(r0) * sc;
        auto step = [&](int kk, auto entry) {
            const double v = t[kk / G] * __shfl_sync(0xffffffffu, inv, kk);
            const double x = __shfl_sync(0xffffffffu, v, (kk % G) * W + col);
            if (h == kk % G) t[kk / G] = x;
#pragma unroll
            for (int q = 0; q < NQ; q++) {
                if (G * q + G - 1 <= kk || q >= nq) continue;
                // this lane's row G q + h below kk
                const bool below = G * q > kk || G * q + h > kk;
                const double r = fma(-entry(kk, q, below), x, t[q]);
                t[q] = below ? r : t[q];
            }
        };
        if constexpr (G <= 4) {
#pragma unroll
            for (int kk = 0; kk < NBB; kk++)
                if (kk < nv) step(kk, [&](int kk, int q, bool below) { return below ? row(ad + kk * sc, q) : 0.0; });
        } else {
            // a step is short here: eight steps' entries are fetched at once
            constexpr int KS = 8;
#pragma unroll
            for (int k0 = 0; k0 < NBB; k0 += KS) {
                if (k0 < nv) {
                    double a[KS][NQ];
#pragma unroll
                    for (int i = 0; i < KS; i++)
#pragma unroll
                        for (int q = 0; q < NQ; q++)
                            a[i][q] = G * q + h > k0 + i && k0 + i < nv ? row(ad + (k0 + i) * sc, q) : 0.0;
#pragma unroll
                    for (int i = 0; i < KS; i++) step(k0 + i, [&](int kk, int q, bool) { return a[kk % KS][q]; });
                }
            }
        }
        // a reader that gave up (it cannot unless the device is broken) says
        // so in every row from there on
        if (gave_up) {
#pragma unroll
            for (int q = 0; q < NQ; q++) t[q] = NAN;
        }
        double *xb = tm.Xs + size_t(b) * NBB * CW + h * CW + col;
#pragma unroll
        for (int q = 0; q < NQ; q++) xb[G * q * CW] = t[q];
        publish_block(tm.solved, b);
        if (incol) {
#pragma unroll
            for (int q = 0; q < NQ; q++)
                if (G * q + h < nv) B[int64_t(r0 + G * q + h) * br] = u.alpha * t[q];
        }
    }
}
__device__ __forceinline__ void solve_unit(const Unit<double> &u, const Team<double> &tm)
{
    switch (u.flags >> 4) {
    case 0: solve_unit<2>(u, tm); break;
    case 1: solve_unit<4>(u, tm); break;
    case 2: solve_unit<8>(u, tm); break;
    case 3: solve_unit<16>(u, tm); break;
    default: solve_unit<32>(u, tm);
    }
}

// Shared memory: the warps' rings and inverse diagonals (FP32), then X: KMAX
// rows, divided among the CTA's teams.
template <typename T>
constexpr size_t batched_smem()
{
    return sizeof(T) * ((sizeof(T) == 4 ? size_t(NW) * (2 * wide::TILE + 2 * NBB) : 0) + size_t(KMAX) * kStride<T>);
}

// The units by the team that solves them: [0, n4) a CTA's four warps, [n4, n2)
// two warps, [n2, n1) one.
struct Queues {
    int n4, n2, n1;
};

// ticket[0..2]: the queues' counters.
template <typename T>
__global__ void __launch_bounds__(NT, sizeof(T) == 8 ? 3 : 2)
batched_kernel(const Unit<T> *__restrict__ units, Queues qs, unsigned *__restrict__ ticket)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int cur[NW], solved[NW];
    T *sm = reinterpret_cast<T *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Team<T> tm;
    tm.ring = tm.inv = nullptr;
    T *Xs = sm;
    if (sizeof(T) == 4) {
        tm.ring = sm + warp * 2 * wide::TILE;
        tm.inv = sm + NW * 2 * wide::TILE + warp * 2 * NBB;
        Xs = sm + NW * (2 * wide::TILE + 2 * NBB);
    }
#pragma unroll 1
    for (int c = 0; c < 3; c++) {
        const int nwu = NW >> c, team = warp / nwu;
        const int lo = c == 0 ? 0 : (c == 1 ? qs.n4 : qs.n2), hi = c == 0 ? qs.n4 : (c == 1 ? qs.n2 : qs.n1);
        if (lo == hi) continue;
        tm.nwu = nwu;
        tm.Xs = Xs + size_t(team) * (KMAX / NW) * nwu * kStride<T>;
        tm.solved = &solved[team];
        // a team's own barrier (the team of four: the CTA's)
        auto team_sync = [&]() {
            if (nwu == NW) __syncthreads();
            else if (nwu == 2) asm volatile("bar.sync %0, 64;" ::"r"(1 + team) : "memory");
            else __syncwarp();
        };
        __syncthreads();  // the other teams' X space is free
        // The first unit of every team by its number, the others by ticket; the
        // CTAs in turn from class to class, so that few units meet no busy one.
        const int grid = gridDim.x, nteams = grid << c;
        for (int t = lo + team * grid + (int(blockIdx.x) + grid - lo % grid) % grid; t < hi; t = cur[team]) {
            if (warp % nwu == 0 && lane == 0) solved[team] = 0;
            team_sync();
            const Unit<T> u = units[t];
            // (a warp is a sub-partition with its own FP64 unit, and the team's last
            // warps own the longest rows: they take turns)
            tm.wid = (warp + t + t / 152) % nwu;
            solve_unit(u, tm);
            team_sync();  // every warp of the team has left the unit
            if (warp % nwu == 0 && lane == 0) cur[team] = lo + nteams + int(atomicAdd(&ticket[c], 1u));
            team_sync();
        }
    }
}

}  // namespace

// ---- plan object ------------------------------------------------------------

struct BatchedPlan {
    int dtype = 0;                 // 0 FP64, 1 FP32
    int tile = 1;                  // split of the work over teams (see build_units)
    int64_t nunits = 0;
    Queues queues = {0, 0, 0};     // the units by team size
    void *units = nullptr;         // device array of Unit<T>
    unsigned *ticket = nullptr;    // the device work queues' counters
    int grid = 0;
    // instances too large for shared memory, solved by the regular driver
    struct Big {
        int side, uplo, trans, diag;
        int64_t m, n, lda, ldb;
        double alpha;
        const void *A;
        void *B;
    };
    std::vector<Big> big;
    cudaGraphExec_t exec = nullptr;
    uint64_t graph_kernels = 0;
    double flops = 0, bytes = 0;
};

namespace {

// FP64 unit of order k, w right-hand sides wide: FP64 warp instructions, those of
// its longest chain on a team of nt warps.
double unit_slots(int64_t k, int64_t w)
{
    const double nb = double((k + NBB - 1) / NBB);
    return nb * (nb - 1) / 2 * double(32 * w) + nb * double(48 + 15 * w);
}
double unit_chain(int64_t k, int64_t w, int nt)
{
    if (nt == 1) return unit_slots(k, w);
    const int nb = int((k + NBB - 1) / NBB);
    double load = 0;
    for (int i = 0; i < nt; i++) {
        double row = 0;
        for (int b = i; b < nb; b += nt) row += double(b * 32 * w + 48 + 15 * w);
        load = std::max(load, row);
    }
    return std::max(load, double(nb) * double(48 + 15 * w + (nb > 1 ? 32 * w : 0)));
}
// Width of the next unit of `rest` right-hand sides: the narrowest that holds
// them, at most cap.
int64_t width_of(int64_t rest, int64_t cap)
{
    int64_t w = 1;
    while (w < rest && w < cap) w *= 2;
    return w;
}
int sm_count()
{
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}
// FP64: the largest width of the batch's units.  Sixteen right-hand sides make
// the fewest instructions per right-hand side, narrower units a shorter chain and
// more of them: the width with the least of all instructions, spread over the
// sub-partitions, and the longest unit's chain (as a 1.5-norm: most of either
// hides behind the other; on 30 batches the widths so chosen were 1.6 % slower
// than the best ones on average).  Measured (orders x right-hand sides): 1125 of
// 169 x 200 6.5 ms (16 wide; 8.4 with four), 20 of 86 x 8 30 us (one wide; 92 with
// 16), 595 of up to 312 x 174 1.12 ms (8; 1.39 with 16).
int64_t unit_width(int64_t count, const int8_t *side, const int64_t *m, const int64_t *n, int one)
{
    const double parts = 4.0 * sm_count();
    int64_t best = 16;
    double least = 0;
    double chains[KMAX / NBB + 1][17] = {};  // by blocks and width (a block's orders share a team size)
    for (int64_t cap = 16; cap >= 1; cap /= 2) {
        double all = 0, chain = 0;
        for (int64_t i = 0; i < count; i++) {
            const int64_t k = side[i] == GB_LEFT ? m[i] : n[i], ncols = side[i] == GB_LEFT ? n[i] : m[i];
            if (k == 0 || ncols == 0 || k > KMAX) continue;
            const int nt = k > 2 * one ? 4 : (k > one ? 2 : 1);
            auto add = [&](int64_t w, double units) {
                all += units * unit_slots(k, w);
                double &c = chains[(k + NBB - 1) / NBB][w];
                if (c == 0) c = unit_chain(k, w, nt);
                chain = std::max(chain, c);
            };
            if (ncols / cap) add(cap, double(ncols / cap));
            for (int64_t rest = ncols % cap; rest > 0;) {
                const int64_t w = width_of(rest, cap);
                add(w, 1);
                rest -= std::min(rest, w);
            }
        }
        const double t = std::pow(all / parts, 1.5) + std::pow(chain, 1.5);
        if (cap == 16 || t < least) {
            least = t;
            best = cap;
        }
    }
    return best;
}
// FP32: the order up to which a unit is one warp's, 128, 64 or none.  Larger
// teams have shorter chains and idle warps (a unit of one warp: its tiles one after
// the other; of a team: 0.8 of a tile's time per block, or its busiest warp's
// tiles; two warps cost 1.3, four 1.7 times the work, eight warps of an SM take
// 1.5 times as long each as one alone): the order with the least of both (2-norm).
// 104 of up to 87 x 5 19.5 us (teams of four; 28.6 of one), 563 of up to 255 x 183
// 408 us (one; 509).
int team_order(int64_t count, const int8_t *side, const int64_t *m, const int64_t *n)
{
    const double warps = 8.0 * sm_count();
    int best = KMAX / 4;
    double least = 0;
    for (int one : {KMAX / 4, KMAX / 8, 0}) {
        double all = 0, chain = 0, chains[KMAX / NBB + 1] = {};
        for (int64_t i = 0; i < count; i++) {
            const int64_t k = side[i] == GB_LEFT ? m[i] : n[i], ncols = side[i] == GB_LEFT ? n[i] : m[i];
            if (k == 0 || ncols == 0 || k > KMAX) continue;
            const int nt = k > 2 * one ? 4 : (k > one ? 2 : 1), nb = int((k + NBB - 1) / NBB);
            const double tiles = nb * (nb + 1) / 2;
            double &c = chains[nb];
            if (c == 0) {
                double busiest = 0;
                for (int w = 0; w < nt; w++) {
                    double row = 0;
                    for (int b = w; b < nb; b += nt) row += b + 1;
                    busiest = std::max(busiest, row);
                }
                c = nt == 1 ? tiles : std::max(busiest, 0.8 * nb);
            }
            all += double((ncols + kChunk<float> - 1) / kChunk<float>) * tiles * (nt == 1 ? 1.0 : (nt == 2 ? 1.3 : 1.7));
            chain = std::max(chain, c);
        }
        const double t = std::hypot(1.5 * all / warps, chain);
        if (one == KMAX / 4 || t < least) {
            least = t;
            best = one;
        }
    }
    return best;
}

template <typename T>
void build_units(BatchedPlan &P, int64_t count, const int8_t *side, const int8_t *uplo, const int8_t *trans,
                 const int8_t *diag, const int64_t *m, const int64_t *n, const T *alpha, const void *const *A,
                 const int64_t *lda, void *const *B, const int64_t *ldb, std::vector<Unit<T>> &units)
{
    constexpr int CW = kChunk<T>;
    // orders up to which a unit is one warp's, two warps'
    const int one = P.tile == 2 ? KMAX / 8 : (sizeof(T) == 8 ? KMAX / 4 : team_order(count, side, m, n)), two = 2 * one;
    const int64_t cap = sizeof(T) == 8 ? unit_width(count, side, m, n, one) : CW;
    for (int64_t i = 0; i < count; i++) {
        if (m[i] == 0 || n[i] == 0) continue;
        const bool left = side[i] == GB_LEFT;
        const int64_t k = left ? m[i] : n[i];
        const int64_t ncols = left ? n[i] : m[i];
        P.flops += double(k) * double(k) * double(ncols);
        P.bytes += sizeof(T) * (double(k) * double(k) / 2 + 2.0 * double(k) * double(ncols));
        if (k > KMAX || alpha[i] == T(0)) {
            P.big.push_back({side[i], uplo[i], trans[i], diag[i], m[i], n[i], lda[i], ldb[i], double(alpha[i]), A[i],
                             B[i]});
            continue;
        }
        const bool mt = left ? (trans[i] == GB_TRANS) : (trans[i] == GB_NOTRANS);
        const bool fwd = (uplo[i] == GB_LOWER) != mt;
        const int flags = (mt ? 1 : 0) | (fwd ? 0 : 2) | (diag[i] == GB_UNIT ? 4 : 0) | (left ? 8 : 0);
        int64_t w = CW;
        for (int64_t c0 = 0; c0 < ncols; c0 += w) {
            int g = 0;  // FP64: the unit is 16 / 2^g wide
            if (sizeof(T) == 8) {
                w = width_of(ncols - c0, cap);
                while (16 >> g > w) g++;
            }
            Unit<T> u;
            u.A = static_cast<const T *>(A[i]);
            T *b = static_cast<T *>(B[i]);
            u.B = left ? b + c0 * ldb[i] : b + c0;
            u.lda = lda[i];
            u.ldb = ldb[i];
            u.k = int(k);
            u.cw = int(std::min<int64_t>(w, ncols - c0));
            u.flags = flags | g << 4;
            u.alpha = alpha[i];
            units.push_back(u);
        }
    }
    // by team size (warps per unit: X of a team of w warps is w KMAX / 4 rows),
    // largest first inside (longest-processing-time order for the queues)
    auto cls = [one, two](const Unit<T> &a) { return a.k > two ? 0 : (a.k > one ? 1 : 2); };
    std::stable_sort(units.begin(), units.end(), [&](const Unit<T> &a, const Unit<T> &b) {
        if (cls(a) != cls(b)) return cls(a) < cls(b);
        return a.k * a.cw > b.k * b.cw;
    });
    P.queues.n4 = int(std::count_if(units.begin(), units.end(), [&](const Unit<T> &a) { return cls(a) == 0; }));
    P.queues.n2 = P.queues.n4 + int(std::count_if(units.begin(), units.end(), [&](const Unit<T> &a) { return cls(a) == 1; }));
    P.queues.n1 = int(units.size());
}

template <typename T>
int upload_and_capture(BatchedPlan &P, std::vector<Unit<T>> &units, cudaStream_t s)
{
    P.nunits = int64_t(units.size());
    const size_t ub = units.size() * sizeof(Unit<T>);
    GB_CUDA(cudaMalloc(&P.units, ub > 0 ? ub : sizeof(Unit<T>)));
    GB_CUDA(cudaMalloc(&P.ticket, 3 * sizeof(unsigned)));
    if (ub) GB_CUDA(cudaMemcpyAsync(P.units, units.data(), ub, cudaMemcpyHostToDevice, s));
    GB_CUDA(cudaStreamSynchronize(s));
    static PerDeviceOnce attr;
    GB_TRY(smem_attr_once(attr, batched_kernel<T>, batched_smem<T>()));
    int dev = 0, sms = 0, per_sm = 0;
    GB_CUDA(cudaGetDevice(&dev));
    GB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    GB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batched_kernel<T>, NT, batched_smem<T>()));
    if (per_sm < 1) per_sm = 1;
    int64_t g = int64_t(sms) * per_sm;
    if (g > P.nunits) g = P.nunits;
    P.grid = int(g);
    if (P.nunits == 0) return 0;
    // CUDA graph: [reset the queue counters, persistent kernel]
    cudaStream_t cs;
    GB_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    const uint64_t before = capture_count();
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaMemsetAsync(P.ticket, 0, 3 * sizeof(unsigned), cs);
        {
            LaunchScope ls(KK_BATCHED, cs, P.flops, P.bytes);
            batched_kernel<T><<<P.grid, NT, batched_smem<T>(), cs>>>(
                static_cast<const Unit<T> *>(P.units), P.queues, P.ticket);
        }
        cudaGraph_t graph = nullptr;
        e = cudaStreamEndCapture(cs, &graph);
        if (e == cudaSuccess) {
            e = cudaGraphInstantiate(&P.exec, graph, 0);
            cudaGraphDestroy(graph);
        }
    }
    P.graph_kernels = capture_count() - before;
    cudaStreamDestroy(cs);
    return check(e);
}

}  // namespace

int batched_run(BatchedPlan &P, cudaStream_t s)
{
    if (P.nunits > 0) {
        LaunchScope ls(KK_BATCHED, s, P.flops, P.bytes, P.graph_kernels);
        GB_CUDA(cudaGraphLaunch(P.exec, s));
    }
    for (auto &b : P.big) {
        int st;
        if (P.dtype == 0)
            st = gb_dtrsm(b.side, b.uplo, b.trans, b.diag, b.m, b.n, b.alpha, static_cast<const double *>(b.A), b.lda,
                          static_cast<double *>(b.B), b.ldb, s);
        else
            st = gb_strsm(b.side, b.uplo, b.trans, b.diag, b.m, b.n, float(b.alpha), static_cast<const float *>(b.A),
                          b.lda, static_cast<float *>(b.B), b.ldb, s);
        if (st) return st;
    }
    return 0;
}

void batched_free(BatchedPlan *P)
{
    if (!P) return;
    if (P->exec) cudaGraphExecDestroy(P->exec);
    if (P->units) cudaFree(P->units);
    if (P->ticket) cudaFree(P->ticket);
    delete P;
}

int batched_create(int dtype, int64_t count, const int8_t *side, const int8_t *uplo, const int8_t *trans,
                   const int8_t *diag, const int64_t *m, const int64_t *n, const void *alpha, const void *const *A,
                   const int64_t *lda, void *const *B, const int64_t *ldb, cudaStream_t s, int tile, BatchedPlan **out)
{
    // argument checks (1-based argument numbers of gb_trsm_batched)
    if (dtype != 0 && dtype != 1) return -1;
    if (count < 0) return -2;
    if (count > 0) {
        const void *arrays[11] = {side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb};
        for (int a = 0; a < 11; a++)
            if (!arrays[a]) return -(3 + a);
    }
    for (int64_t i = 0; i < count; i++) {
        if (side[i] != GB_LEFT && side[i] != GB_RIGHT) return -3;
        if (uplo[i] != GB_LOWER && uplo[i] != GB_UPPER) return -4;
        if (trans[i] != GB_NOTRANS && trans[i] != GB_TRANS) return -5;
        if (diag[i] != GB_NONUNIT && diag[i] != GB_UNIT) return -6;
        if (m[i] < 0) return -7;
        if (n[i] < 0) return -8;
        const int64_t k = side[i] == GB_LEFT ? m[i] : n[i];
        const bool empty = m[i] == 0 || n[i] == 0;
        const double a = dtype == 0 ? static_cast<const double *>(alpha)[i] : static_cast<const float *>(alpha)[i];
        if (!empty && A[i] == nullptr && a != 0.0) return -10;
        if (lda[i] < (k > 1 ? k : 1)) return -11;
        if (!empty && B[i] == nullptr) return -12;
        if (ldb[i] < (m[i] > 1 ? m[i] : 1)) return -13;
    }
    BatchedPlan *P = new BatchedPlan;
    P->dtype = dtype;
    P->tile = tile;
    int st;
    if (dtype == 0) {
        std::vector<Unit<double>> units;
        build_units<double>(*P, count, side, uplo, trans, diag, m, n, static_cast<const double *>(alpha), A, lda, B,
                            ldb, units);
        st = upload_and_capture<double>(*P, units, s);
    } else {
        std::vector<Unit<float>> units;
        build_units<float>(*P, count, side, uplo, trans, diag, m, n, static_cast<const float *>(alpha), A, lda, B,
                           ldb, units);
        st = upload_and_capture<float>(*P, units, s);
    }
    if (st) {
        batched_free(P);
        return st;
    }
    *out = P;
    return 0;
}

}  // namespace gb

extern "C" {

int gb_batched_plan_create_tiled(int dtype, int64_t count, const int8_t *side, const int8_t *uplo,
                                 const int8_t *trans, const int8_t *diag, const int64_t *m, const int64_t *n,
                                 const void *alpha, const void *const *A, const int64_t *lda, void *const *B,
                                 const int64_t *ldb, int tile, void *stream, void **plan_out)
{
    if (!plan_out) return -17;
    *plan_out = nullptr;
    if (tile == 0) tile = 1;
    if (tile != 1 && tile != 2) return -15;
    gb::BatchedPlan *P = nullptr;
    int st = gb::batched_create(dtype, count, side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb,
                                static_cast<cudaStream_t>(stream), tile, &P);
    if (st) return st;
    *plan_out = P;
    return 0;
}

int gb_batched_plan_create(int dtype, int64_t count, const int8_t *side, const int8_t *uplo, const int8_t *trans,
                           const int8_t *diag, const int64_t *m, const int64_t *n, const void *alpha,
                           const void *const *A, const int64_t *lda, void *const *B, const int64_t *ldb,
                           void *stream, void **plan_out)
{
    if (!plan_out) return -15;
    const int st = gb_batched_plan_create_tiled(dtype, count, side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb,
                                                1, stream, plan_out);
    return st == -17 ? -15 : st;
}

int gb_batched_autotune(int dtype, int64_t count, const int8_t *side, const int8_t *uplo, const int8_t *trans,
                        const int8_t *diag, const int64_t *m, const int64_t *n, const void *alpha,
                        const void *const *A, const int64_t *lda, void *const *B, const int64_t *ldb, int reps,
                        void *stream, int *tile_out, double *ms_out)
{
    if (!tile_out) return -16;
    if (reps < 1 || reps > 100) return -14;
    *tile_out = 1;
    if (ms_out) ms_out[0] = ms_out[1] = 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the solves overwrite B: keep a device copy of every B and restore it
    // before each run and at the end
    const size_t esz = dtype == 0 ? 8 : 4;
    std::vector<size_t> off(count > 0 ? size_t(count) : 1, 0);
    size_t total = 0;
    for (int64_t i = 0; i < count; i++) {
        off[i] = total;
        if (m && n && m[i] > 0 && n[i] > 0) total += size_t(m[i]) * size_t(n[i]) * esz;
    }
    void *save = nullptr;
    if (total) GB_CUDA(cudaMallocAsync(&save, total, s));
    auto copy_all = [&](bool restore) {
        for (int64_t i = 0; i < count; i++) {
            if (m[i] <= 0 || n[i] <= 0) continue;
            char *sv = static_cast<char *>(save) + off[i];
            const cudaError_t e =
                restore ? cudaMemcpy2DAsync(B[i], esz * ldb[i], sv, esz * m[i], esz * m[i], n[i], cudaMemcpyDeviceToDevice, s)
                        : cudaMemcpy2DAsync(sv, esz * m[i], B[i], esz * ldb[i], esz * m[i], n[i], cudaMemcpyDeviceToDevice, s);
            if (e != cudaSuccess) return gb::check(e);
        }
        return 0;
    };
    int st = 0;
    double best = 1e300;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (!st) st = gb::check(cudaEventCreate(&e0));
    if (!st) st = gb::check(cudaEventCreate(&e1));
    if (!st && total) st = copy_all(false);
    for (int tile = 1; tile <= 2 && !st; tile++) {
        void *plan = nullptr;
        st = gb_batched_plan_create_tiled(dtype, count, side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb, tile,
                                          stream, &plan);
        if (st) break;
        std::vector<float> t(reps);
        for (int r = 0; r <= reps && !st; r++) {  // run 0 is a warm-up
            if (total) st = copy_all(true);
            if (st) break;
            cudaEventRecord(e0, s);
            st = gb_batched_plan_run(plan, stream);
            cudaEventRecord(e1, s);
            if (!st) st = gb::check(cudaEventSynchronize(e1));
            if (!st && r > 0) st = gb::check(cudaEventElapsedTime(&t[r - 1], e0, e1));
        }
        gb_batched_plan_destroy(plan);
        if (st) break;
        std::sort(t.begin(), t.end());
        const double ms = t[reps / 2];
        if (ms_out) ms_out[tile - 1] = ms;
        if (ms < best) {
            best = ms;
            *tile_out = tile;
        }
    }
    if (total && save) {
        const int c = copy_all(true);
        if (!st) st = c;
        cudaFreeAsync(save, s);
    }
    const int c = gb::check(cudaStreamSynchronize(s));
    if (!st) st = c;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    return st;
}

int gb_batched_plan_tile(const void *plan)
{
    if (!plan) return -1;
    return static_cast<const gb::BatchedPlan *>(plan)->tile;
}

int gb_batched_plan_run(void *plan, void *stream)
{
    if (!plan) return -1;
    return gb::batched_run(*static_cast<gb::BatchedPlan *>(plan), static_cast<cudaStream_t>(stream));
}

int gb_batched_plan_destroy(void *plan)
{
    gb::batched_free(static_cast<gb::BatchedPlan *>(plan));
    return 0;
}

int gb_batched_plan_info(const void *plan, int64_t *units, int *grid, int64_t *large_instances, double *flops)
{
    if (!plan) return -1;
    const gb::BatchedPlan *P = static_cast<const gb::BatchedPlan *>(plan);
    if (units) *units = P->nunits;
    if (grid) *grid = P->grid;
    if (large_instances) *large_instances = int64_t(P->big.size());
    if (flops) *flops = P->flops;
    return 0;
}

int gb_trsm_batched(int dtype, int64_t count, const int8_t *side, const int8_t *uplo, const int8_t *trans,
                    const int8_t *diag, const int64_t *m, const int64_t *n, const void *alpha, const void *const *A,
                    const int64_t *lda, void *const *B, const int64_t *ldb, void *stream)
{
    void *plan = nullptr;
    int st = gb_batched_plan_create(dtype, count, side, uplo, trans, diag, m, n, alpha, A, lda, B, ldb, stream, &plan);
    if (st) return st;
    st = gb_batched_plan_run(plan, stream);
    cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    gb_batched_plan_destroy(plan);
    if (st) return st;
    return gb::check(e);
}

}  // extern "C"
