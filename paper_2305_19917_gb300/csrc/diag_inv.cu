// Diagonal-block step of the mixed-precision low-precision solve, done by
// inversion: each 128 x 128 lower-triangular diagonal block L_b is inverted
// once per solve (FP32, one CTA per block) into a two-term BF16 split, and
// every TS task of the refinement then applies X_b = L_b^-1 Y_b as a product on
// the tensor cores (apply_tc.cu).  This turns the serial substitution on the
// critical path of the recursive model (Section V-A, the TS(i) leaves) into a
// fully parallel product.  Also here: the FP8 copy of a solved leaf.
//
// Storage ("band"): block b occupies band[(b*128 + c)*128 + i] = L_b(i, c),
// i.e. each block column-major with leading dimension 128.
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include "common.cuh"

namespace gb {
namespace {

constexpr int NBI = 128;
constexpr int LDI = NBI + 4;  // column stride in shared memory: columns stay 16-byte aligned, rows spread over banks
constexpr int NTI = 256;

// One CTA (8 warps) per block, by halves: the four 32 x 32 triangles by
// substitution on the unit vectors (a warp each, a lane per column, its 32 rows
// in registers), then twice
//     [A 0; C B]^-1 = [A^-1 0; -B^-1 C A^-1  B^-1]
// with a lane per row and eight columns per warp (the product C A^-1 of a
// warp's columns is used by that warp only).  Substitution over the whole block
// with a thread per column was one chain of 128 dot products, 167 us a launch;
// this is 20, mostly loads, stores and latencies.
__global__ void __launch_bounds__(NTI) invert_blocks_kernel(const float *__restrict__ band,
                                                            __nv_bfloat16 *__restrict__ inv16, int64_t kp)
{
    extern __shared__ __align__(16) float sm[];
    float *L = sm;               // L[c * LDI + i] = L_b(i, c)
    float *X = sm + NBI * LDI;   // X[c * LDI + i] = (L_b^-1)(i, c), zero above the diagonal
    float *T = X + NBI * LDI;    // the products C A^-1, 64 rows a column
    const float *Lb = band + size_t(blockIdx.x) * NBI * NBI;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll 8
    for (int idx = tid; idx < NBI * NBI / 4; idx += NTI) {
        const int i4 = (idx % (NBI / 4)) * 4, c = idx / (NBI / 4);
        *reinterpret_cast<float4 *>(L + c * LDI + i4) = reinterpret_cast<const float4 *>(Lb)[idx];
        *reinterpret_cast<float4 *>(X + c * LDI + i4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    if (warp < 4) {
        const int o = 32 * warp;
        const float *Ld = L + o * LDI + o;
        float x[32];
#pragma unroll
        for (int r = 0; r < 32; r++) x[r] = r == lane ? 1.f : 0.f;
#pragma unroll
        for (int k = 0; k < 32; k++) {
            x[k] /= Ld[k * LDI + k];
#pragma unroll
            for (int r = (k + 1) & ~3; r < 32; r += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(Ld + k * LDI + r);
                if (r > k) x[r] = fmaf(-a.x, x[k], x[r]);
                if (r + 1 > k) x[r + 1] = fmaf(-a.y, x[k], x[r + 1]);
                if (r + 2 > k) x[r + 2] = fmaf(-a.z, x[k], x[r + 2]);
                if (r + 3 > k) x[r + 3] = fmaf(-a.w, x[k], x[r + 3]);
            }
        }
        float *Xd = X + (o + lane) * LDI + o;
#pragma unroll
        for (int r = 0; r < 32; r++) Xd[r] = x[r];
    }
    __syncthreads();
    // halves of H rows at offset o: T = C A^-1, then X21 = -B^-1 T; RPL rows per lane
    auto combine = [&](auto rpl, int o, int c0) {
        constexpr int RPL = decltype(rpl)::value, H = 32 * RPL;
        float acc[RPL][8];
        float *Tc = T + warp * 8 * 64;
        auto product = [&](const float *A, const float *B, int ldb, int k0, float sign, float *out, int ldo) {
#pragma unroll
            for (int r = 0; r < RPL; r++)
#pragma unroll
                for (int c = 0; c < 8; c++) acc[r][c] = 0.f;
#pragma unroll 4
            for (int k = k0; k < H; k++) {
                float a[RPL];
#pragma unroll
                for (int r = 0; r < RPL; r++) a[r] = A[k * LDI + lane + 32 * r];
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const float b = B[c * ldb + k];
#pragma unroll
                    for (int r = 0; r < RPL; r++) acc[r][c] = fmaf(a[r], b, acc[r][c]);
                }
            }
#pragma unroll
            for (int r = 0; r < RPL; r++)
#pragma unroll
                for (int c = 0; c < 8; c++) out[c * ldo + lane + 32 * r] = sign * acc[r][c];
            __syncwarp();
        };
        // (rows above c0 of A^-1's columns c0.. are zero)
        product(L + o * LDI + o + H, X + (o + c0) * LDI + o, LDI, c0, 1.f, Tc, 64);
        product(X + (o + H) * LDI + o + H, Tc, 64, 0, -1.f, X + (o + c0) * LDI + o + H, LDI);
    };
    combine(std::integral_constant<int, 1>(), 64 * (warp >> 2), 8 * (warp & 3));
    __syncthreads();
    combine(std::integral_constant<int, 2>(), 0, 8 * warp);
    __syncthreads();
    // two-term BF16 split L^-1 = hi + lo, row-major (K-major for the tensor
    // cores): hi rows at block*128 + i, lo rows at kp + block*128 + i
    const int64_t r0 = int64_t(blockIdx.x) * NBI;
#pragma unroll 4
    for (int idx = tid; idx < NBI * NBI / 2; idx += NTI) {
        const int i = idx / (NBI / 2), k = (idx % (NBI / 2)) * 2;
        const float x0 = X[k * LDI + i], x1 = X[(k + 1) * LDI + i];
        const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
        const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - __low2float(h), x1 - __high2float(h));
        *reinterpret_cast<__nv_bfloat162 *>(inv16 + (r0 + i) * NBI + k) = h;
        *reinterpret_cast<__nv_bfloat162 *>(inv16 + (kp + r0 + i) * NBI + k) = l;
    }
}

constexpr size_t INV_SMEM = sizeof(float) * (2 * size_t(NBI) * LDI + 64 * 64);

// FP8 (E4M3) copy of the 128 x 64 block (blockIdx.y, blockIdx.x) of Y
// (column-major, ld), with one power-of-two scale s, amax / s <= 448; bound by
// memory (5 bytes per element).  A warp takes eight columns, a lane four
// consecutive rows of each.
__global__ void __launch_bounds__(256)
quantise_fp8_kernel(const float *__restrict__ Y, int64_t ld, uint8_t *__restrict__ Y8, float *__restrict__ scales,
                    int64_t lds)
{
    __shared__ float red[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t o = int64_t(blockIdx.y) * NBI + 4 * lane + (int64_t(blockIdx.x) * 64 + 8 * warp) * ld;
    float4 v[8];
#pragma unroll
    for (int c = 0; c < 8; c++) v[c] = *reinterpret_cast<const float4 *>(Y + o + c * ld);
    float mx = 0.f;
#pragma unroll
    for (int c = 0; c < 8; c++) mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v[c].x), fabsf(v[c].y)), fmaxf(fabsf(v[c].z), fabsf(v[c].w))));
    for (int s = 16; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    for (int w = 0; w < 8; w++) mx = fmaxf(mx, red[w]);
    const float sc = mx > 0.f ? exp2f(ceilf(log2f(mx / 448.f))) : 1.f;
    const float q = 1.f / sc;
    if (threadIdx.x == 0) scales[blockIdx.y * lds + blockIdx.x] = sc;
    auto cvt = [&](float x) { return uint32_t(__nv_cvt_float_to_fp8(x * q, __NV_SATFINITE, __NV_E4M3)); };
#pragma unroll
    for (int c = 0; c < 8; c++)
        *reinterpret_cast<uint32_t *>(Y8 + o + c * ld) = cvt(v[c].x) | (cvt(v[c].y) << 8) | (cvt(v[c].z) << 16) | (cvt(v[c].w) << 24);
}

}  // namespace

// Invert the nblocks diagonal blocks held in `band` into the two-term BF16
// split inv16 (2 x kp x 128, kp = 128 * nblocks rows of 128).
int launch_invert_blocks(const float *band, __nv_bfloat16 *inv16, int64_t nblocks, cudaStream_t s)
{
    if (nblocks <= 0) return 0;
    static PerDeviceOnce attr;
    GB_TRY(smem_attr_once(attr, invert_blocks_kernel, INV_SMEM));
    LaunchScope ls(KK_DIAG, s, double(nblocks) * NBI * NBI * NBI / 3.0, 8.0 * nblocks * NBI * NBI);
    invert_blocks_kernel<<<(unsigned)nblocks, NTI, INV_SMEM, s>>>(band, inv16, int64_t(nblocks) * NBI);
    return check(cudaGetLastError());
}

// The FP8 copy of nr rows (a multiple of 128) and np columns (of 64) of Y, and
// its block scales (row block i, column block j at scales[i * lds + j]).
int launch_quantise_fp8(const float *Y, int64_t ld, uint8_t *Y8, float *scales, int64_t lds, int64_t nr, int64_t np,
                        cudaStream_t s)
{
    if (nr <= 0 || np <= 0) return 0;
    if (nr % NBI || np % 64 || ld % 4 || np / 64 > 0x7fffffff || nr / NBI > 65535 ||
        (reinterpret_cast<uintptr_t>(Y) & 15) || (reinterpret_cast<uintptr_t>(Y8) & 3))
        return GB_STATUS_CUDA_ERROR;
    LaunchScope ls(KK_CONVERT, s, 0, 5.0 * double(nr) * double(np));
    quantise_fp8_kernel<<<dim3((unsigned)(np / 64), (unsigned)(nr / NBI)), 256, 0, s>>>(Y, ld, Y8, scales, lds);
    return check(cudaGetLastError());
}

}  // namespace gb
