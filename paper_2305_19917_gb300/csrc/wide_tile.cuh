// FP32 solve steps on 32 x 32 blocks with one right-hand side per lane
// (internal header): shared by the panel solve for many right-hand sides
// (panel_wide.cu) and the batched solve (batched.cu).
//
// A lane holds the 32 rows of a block row for its right-hand side in registers,
// as 16 pairs for the packed multiply-add (two FP32 multiply-adds an
// instruction, each rounded as by itself): an update step loads one X value
// per lane and the step's 32 Mv entries as eight broadcast vectors, nine
// shared-memory wavefronts and 26 instructions per 32 multiply-adds.  A
// substitution step needs no shuffle and has 31 independent multiply-adds
// behind it.  Tiles lie in shared memory in natural order, triangles by
// columns (entry (row i, column k) at k * WLD + i), other blocks as Mv is
// stored, so that 16-byte copies bring them in: by columns, the pairs being two
// rows, or by rows (i * WLD + k), the pairs being the sums over even and odd k.
#pragma once
#include <cmath>
#include "common.cuh"
#include "tc_common.cuh"

namespace gb {
namespace wide {

constexpr int NB = 32, WLD = NB + 4, TILE = NB * WLD, CW = 32;
constexpr int kSpins = 1 << 22;  // polls before a reader gives up

__device__ __forceinline__ void cp16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tc::smem_u32(dst)), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// One warp issues the copies of block (rows ri.., columns ci..) of the nr x nr
// triangle at M (AM: Mv(i,k) = M[i + k lda], else M[k + i lda]) into tile t;
// ri or ci may be negative or beyond nr (zeros there).  tri: 0 the whole
// block, 1 / 2 its strictly lower / upper triangle.  vec: 16 bytes at a time
// where the block lies inside.
template <bool AM>
__device__ __forceinline__ void load_block(const float *M, int64_t lda, int nr, int ri, int ci, int tri, bool vec, float *t)
{
    const int lane = threadIdx.x & 31;
    const float *src = AM ? M + ri + int64_t(ci) * lda : M + ci + int64_t(ri) * lda;
    if (vec && tri == 0 && ri >= 0 && ri + NB <= nr) {
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int idx = lane + 32 * q, f = (idx % 8) * 4, s = idx / 8;
            cp16(t + s * WLD + f, src + f + int64_t(s) * lda);
        }
        return;
    }
    const bool inside = tri == 0 && ri >= 0 && ri + NB <= nr && ci >= 0 && ci + NB <= nr;
#pragma unroll 8
    for (int s = 0; s < NB; s++) {
        const int i = AM ? lane : s, k = AM ? s : lane;
        bool in = inside || (ri + i >= 0 && ri + i < nr && ci + k >= 0 && ci + k < nr);
        if (tri) in = in && (tri == 1 ? k < i : k > i);
        cp4(t + ((AM || tri) ? k * WLD + i : i * WLD + k), in ? src + lane + int64_t(s) * lda : M, in);
    }
}

__device__ __forceinline__ float &at(float2 (&t)[NB / 2], int i) { return (i & 1) ? t[i / 2].y : t[i / 2].x; }

// The sum of a block row's updates.
template <bool AM>
struct Sum;
template <>
struct Sum<true> {  // tiles by columns
    float2 t[NB / 2];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < NB / 2; i++) t[i] = make_float2(0.f, 0.f);
    }
    // += (tile) x, x the 32 rows of a solved block (stride XLD)
    template <int XLD = CW>
    __device__ __forceinline__ void update(const float *tile, const float *x0)
    {
#pragma unroll 4
        for (int k = 0; k < NB; k++) {
            const float x = x0[k * XLD];
            const float2 xx = make_float2(x, x);
#pragma unroll
            for (int i = 0; i < NB; i += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(tile + k * WLD + i);
                t[i / 2] = __ffma2_rn(make_float2(a.x, a.y), xx, t[i / 2]);
                t[i / 2 + 1] = __ffma2_rn(make_float2(a.z, a.w), xx, t[i / 2 + 1]);
            }
        }
    }
    __device__ __forceinline__ float row(int i) { return at(t, i); }
};
template <>
struct Sum<false> {  // tiles by rows
    float2 t[NB];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < NB; i++) t[i] = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ void update(const float *tile, const float *x0)
    {
#pragma unroll 1
        for (int k = 0; k < NB; k += 4) {
            const float2 x01 = make_float2(x0[k * CW], x0[(k + 1) * CW]);
            const float2 x23 = make_float2(x0[(k + 2) * CW], x0[(k + 3) * CW]);
#pragma unroll
            for (int i = 0; i < NB; i++) {
                const float4 a = *reinterpret_cast<const float4 *>(tile + i * WLD + k);
                t[i] = __ffma2_rn(make_float2(a.x, a.y), x01, t[i]);
                t[i] = __ffma2_rn(make_float2(a.z, a.w), x23, t[i]);
            }
        }
    }
    __device__ __forceinline__ float row(int i) { return t[i].x + t[i].y; }
};

// Substitution with the block's strict triangle (tile) and inverse diagonal:
// t holds the rows' updates on entry and X on return, xb the right-hand sides
// (stride CW; times alpha) and then X.  The rows' sums go on inside the block
// and are subtracted once per row: x rounds at the right-hand side's magnitude
// once, not at every step.  EXACT: the product with the inverse is corrected
// once against the diagonal (inv[NB + k]), to the division's accuracy.
template <bool FWD, bool EXACT, int XLD>
__device__ __forceinline__ void substitute(float2 (&t)[NB / 2], const float *tile, const float *inv, float *xb, float alpha)
{
#pragma unroll
    for (int q = 0; q < NB; q++) {
        const int k = FWD ? q : NB - 1 - q;
        const float r = alpha * xb[k * XLD] - at(t, k);
        float x = r * inv[k];
        if (EXACT) {
            const float c = fmaf(fmaf(-inv[NB + k], x, r), inv[k], x);
            x = fabsf(x) < INFINITY ? c : x;
        }
        xb[k * XLD] = x;
        at(t, k) = x;
        const float2 xx = make_float2(x, x);
        const float *lk = tile + k * WLD;
#pragma unroll
        for (int i = 0; i < NB; i += 4) {
            if (!(FWD ? i + 3 > k : i < k)) continue;  // no row of the triangle's column k in this vector
            const float4 a = *reinterpret_cast<const float4 *>(lk + i);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int w = i + 2 * h;  // rows w, w + 1
                const float2 ah = h ? make_float2(a.z, a.w) : make_float2(a.x, a.y);
                const bool b0 = FWD ? w > k : w < k, b1 = FWD ? w + 1 > k : w + 1 < k;
                if (b0 && b1) t[w / 2] = __ffma2_rn(ah, xx, t[w / 2]);
                else if (b0) t[w / 2].x = fmaf(ah.x, x, t[w / 2].x);
                else if (b1) t[w / 2].y = fmaf(ah.y, x, t[w / 2].y);
            }
        }
    }
}

}  // namespace wide
}  // namespace gb
