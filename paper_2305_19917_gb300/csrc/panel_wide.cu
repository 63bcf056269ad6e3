// FP32 diagonal-block solve of many rows in one launch for many right-hand
// sides (the paper's TS task; panel_kernel.cuh has the form for few).
//
// As there, a CTA walks a block of up to 1024 rows by itself, left-looking in
// 32-row blocks, each warp owning every fourth block row and streaming its own
// tiles of Mv.  But a lane holds one right-hand side and the block's 32 rows of
// it, instead of one row and CW right-hand sides (wide_tile.cuh).  Bounded by
// the issue of one warp per sub-partition (two CTAs of 4 warps share an SM)
// and, for few CTAs, the chain of blocks.  Measured, 512 rows: 8192 right-hand sides
// 104 us (with one multiply-add an instruction 138, the other form 265).
#include <cmath>
#include "panel.cuh"
#include "wide_tile.cuh"

namespace gb {
namespace {

using namespace wide;
constexpr int NW = 4, NS = 2;

constexpr size_t wide_smem(int nblk) { return sizeof(float) * (size_t(NW) * (NS * TILE + NB) + size_t(nblk) * NB * CW); }

// AM: Mv(i,k) = M[i + k lda], else M[k + i lda]; Bv(i,c) = B[i si + c sc].
// vec: off-diagonal tiles 16 bytes at a time; vecb: si == 1 and columns of B
// 16 bytes at a time.  Rows inside a block are numbered in natural order; a
// backward solve takes the blocks from the bottom and the rows downwards.
template <bool AM, bool FWD>
__global__ void __launch_bounds__(32 * NW, 2)
panel_wide_kernel(const float *__restrict__ M, int64_t lda, float *__restrict__ B, int64_t si, int64_t sc, int nr,
                  int64_t ncols, float alpha, int unit, int vec, int vecb)
{
    extern __shared__ __align__(16) float smem[];
    __shared__ int solved;  // blocks whose X is in shared memory
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nblk = (nr + NB - 1) / NB;
    float *ring = smem + warp * NS * TILE;
    float *inv = smem + NW * NS * TILE + warp * NB;
    float *Xs = smem + NW * (NS * TILE + NB);
    const int64_t col = int64_t(blockIdx.x) * CW + lane;
    const bool incol = col < ncols;
    if (threadIdx.x == 0) solved = 0;
    tc::pdl_wait();
    tc::pdl_launch_dependents();
    __syncthreads();

    auto nat = [&](int b) { return FWD ? b * NB : nr - (b + 1) * NB; };
    // the warp's tiles in order: block rows warp, warp + NW, ...; in each kb = 0 .. b
    int pb = warp, pk = 0, pn = 0;
    auto prefetch = [&]() {
        if (pb < nblk) {
            load_block<AM>(M, lda, nr, nat(pb), nat(pk), pk < pb ? 0 : (FWD ? 1 : 2), vec, ring + (pn % NS) * TILE);
            if (pk == pb) {
                pb += NW;
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
    for (int b = warp; b < nblk; b += NW) {
        const int r0 = nat(b);
        Sum<AM> sum;
        sum.clear();
        // the rows' right-hand sides into their place in X (read again by the
        // lane that copied them)
        const float *bc = B + col * sc + int64_t(r0) * si;
        float *xb = Xs + size_t(b) * NB * CW + lane;
#pragma unroll 8
        for (int i = 0; i < NB; i++) {
            const bool in = incol && r0 + i >= 0 && r0 + i < nr;
            cp4(xb + i * CW, in ? bc + i * si : M, in);
        }
        commit();
        {
            const int i = r0 + lane;
            inv[lane] = (!unit && i >= 0 && i < nr) ? 1.f / M[i + int64_t(i) * lda] : 1.f;
        }
        for (int kb = 0; kb <= b; kb++, n++) {
            // everything committed (NS = 2: tile n, and the right-hand sides at kb = 0)
            wait_all();
            __syncwarp();
            prefetch();  // into the buffer of tile n - 1, which every lane has read
            const float *tile = ring + (n % NS) * TILE;
            if (kb < b) {
                for (int spin = 0; known <= kb && !gave_up; spin++) {
                    known = *static_cast<volatile int *>(&solved);
                    if (spin > kSpins) gave_up = true;
                }
                __threadfence_block();
                sum.update(tile, Xs + size_t(kb) * NB * CW + lane);
                continue;
            }
            // t = alpha B - the updates, then the triangle
            const bool whole = vecb && r0 >= 0 && r0 + NB <= nr;
            float2 t[NB / 2];
#pragma unroll
            for (int i = 0; i < NB; i++) at(t, i) = sum.row(i);
            substitute<FWD, false, CW>(t, tile, inv, xb, alpha);
            // a reader that gave up (it cannot unless the device is broken)
            // says so in every row from there on
            if (gave_up) {
#pragma unroll
                for (int i = 0; i < NB; i++) xb[i * CW] = at(t, i) = NAN;
            }
            __syncwarp();
            if (lane == 0) {
                __threadfence_block();
                *static_cast<volatile int *>(&solved) = b + 1;
            }
            if (!incol) continue;
            float *bo = B + col * sc + int64_t(r0) * si;
            if (whole) {
#pragma unroll
                for (int i = 0; i < NB; i += 4)
                    *reinterpret_cast<float4 *>(bo + i) = make_float4(t[i / 2].x, t[i / 2].y, t[i / 2 + 1].x, t[i / 2 + 1].y);
            } else {
#pragma unroll
                for (int i = 0; i < NB; i++)
                    if (r0 + i >= 0 && r0 + i < nr) bo[i * si] = at(t, i);
            }
        }
    }
    wait_all();
}

template <bool AM, bool FWD>
int launch_form(const Canon<float> &c, const float *M, float *B, int nr, float alpha, int vec, int vecb)
{
    static PerDeviceOnce attr;
    GB_TRY(smem_attr_once(attr, panel_wide_kernel<AM, FWD>, wide_smem(kPanelRows<float> / NB)));
    const int64_t grid = (c.ncols + CW - 1) / CW;
    if (grid > 0x7fffffff) return GB_STATUS_CUDA_ERROR;
    LaunchScope ls(KK_DIAG, c.stream, double(nr) * nr * c.ncols, 4.0 * (0.5 * nr * nr + 2.0 * nr * c.ncols));
    return check(launch_pdl(panel_wide_kernel<AM, FWD>, dim3((unsigned)grid), dim3(32 * NW), wide_smem((nr + NB - 1) / NB),
                            c.stream, M, c.lda, B, c.left ? int64_t(1) : c.ldb, c.left ? c.ldb : int64_t(1), nr, c.ncols,
                            alpha, int(c.unit), vec, vecb));
}

}  // namespace

int launch_panel_wide(const Canon<float> &c, int64_t r0, int nr, float alpha)
{
    const float *M = c.A + r0 + r0 * c.lda;
    float *B = bv_ptr(c, r0, 0);
    // runs start at multiples of 32 rows from r0 (forward) or from r0 + nr (backward)
    const bool rows4 = c.forward || nr % 4 == 0;
    const int vec = rows4 && reinterpret_cast<uintptr_t>(M) % 16 == 0 && c.lda % 4 == 0;
    const int vecb = rows4 && c.left && reinterpret_cast<uintptr_t>(B) % 16 == 0 && c.ldb % 4 == 0;
    if (c.mt) return c.forward ? launch_form<false, true>(c, M, B, nr, alpha, vec, vecb) : launch_form<false, false>(c, M, B, nr, alpha, vec, vecb);
    return c.forward ? launch_form<true, true>(c, M, B, nr, alpha, vec, vecb) : launch_form<true, false>(c, M, B, nr, alpha, vec, vecb);
}

}  // namespace gb
